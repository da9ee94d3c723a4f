"""The autotuner's choices for the two kinds of transport stages, axis-wise (H1) and spectral (H2, H3),
are measured and used apart (csrc/tune.cu); a context that changes between them takes the other kind's,
unless its caller has set the tiles or the launch mode."""
import math

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _config(n1, n2, regnorm):
    from paper_1503_00757_gb300.binding import Context
    ctx = Context(n1, n2, 2, regnorm=regnorm)
    cfg = ctx.tile_config()
    ctx.close()
    return cfg


def _solve(n1, n2, regnorm):
    import torch
    from paper_1503_00757_gb300.binding import default_opts, solve_batch
    z = lambda *s: torch.zeros(*s, device="cuda")
    solve_batch([dict(mT=z(n1, n2), mR=z(n1, n2), v=z(2, n1, n2), nt=2, regnorm=regnorm, beta=1e-2)],
                default_opts(maxit_newton=1), nworkers=1)


def test_each_kind_is_tuned_by_the_batch_that_needs_it():
    from paper_1503_00757_gb300.binding import Context, autotune
    n1, n2 = 32, 512  # used by no other test: both kinds start untuned in this process
    default = _config(n1, n2, 1)
    assert _config(n1, n2, 2) == default
    _solve(n1, n2, 1)
    axis = _config(n1, n2, 1)
    assert _config(n1, n2, 2) == default  # an H1 batch says nothing about the spectral stages
    _solve(n1, n2, 3)
    spectral = _config(n1, n2, 2)
    assert _config(n1, n2, 1) == axis and _config(n1, n2, 3) == spectral
    assert autotune(n1, n2, nt=2) == axis + (-1.0,)
    # a choice of its own per kind
    ctx = Context(n1, n2, 2, regnorm=1)
    ctx.set_params(2, regnorm=2)
    assert ctx.tile_config() == spectral
    ctx.set_params(2, regnorm=3, beta=1e-3)
    assert ctx.tile_config() == spectral
    ctx.set_params(2, regnorm=1, gamma=math.inf)
    assert ctx.tile_config() == axis
    ctx.set_tiles(8, 16, 0)
    ctx.set_pdl(False)
    ctx.set_params(2, regnorm=2)
    assert ctx.tile_config() == (8, 16, 0, 0)
    ctx.close()


@pytest.mark.parametrize("n1,n2", [(16, 16), (64, 64), (64, 1024)])
def test_choices_are_valid_on_every_kind_of_grid(n1, n2):
    """No valid tiles (16 x 16: the default rule), resident solves (P keeps its default), long rows."""
    from paper_1503_00757_gb300.binding import autotune
    from .test_gpu_tiles import valid_tiles
    before = _config(n1, n2, 1)
    R, C, P, D, ms = autotune(n1, n2, nt=2, concurrency=2, force=True)
    assert ms > 0.0 and D in (0, 1)
    assert (R, C, P) in valid_tiles(n1, n2) or ((n1, n2) == (16, 16) and (R, C, P) == before[:3])
    assert (n1, n2) != (64, 64) or P == before[2]
    assert _config(n1, n2, 1) == (R, C, P, D)
    s = _config(n1, n2, 2)
    assert s[:3] in valid_tiles(n1, n2) or (n1, n2) == (16, 16)
