"""Performance cases: the calls a user of the library makes, at the sizes they make them.

A case is one call (or the few calls that belong together) through
``paper_1503_00757_gb300.binding``:

  operator   a spectral operator on its own (gradient, divergence, projection, preconditioner);
  gradient   objective and reduced gradient at an iterate: the state and the adjoint solve;
  matvec     one Hessian product at a linearization point: what a Krylov iteration costs;
  measures   what is evaluated on a finished registration: det F, displacement, label overlap;
  solve      a registration from v = 0;
  batch      independent registrations through the batch executor;
  gradient3, matvec3   the same two in three dimensions;
  net        warm-start prediction;  train: loss and parameter gradients of one training batch.

Images are nested ellipses with smoothed edges (3-D: Gaussian bumps), the reference is the
template at displaced coordinates; velocities are band limited and within the explicit scheme's
CFL limit.  ``exact`` restates every path that is a fixed sequence of operations in FP64.
"""
import functools
import math

import numpy as np
import torch

from paper_1503_00757_gb300 import binding

TWO_PI = 2.0 * math.pi
WEIGHTS = "paper_1503_00757_gb300/weights/warmstart_n256.npy"
CHANNELS = (2, 32, 32, 32, 32, 32, 32, 32, 2)
DILATION = (1, 2, 4, 8, 8, 4, 2, 1)
EPS2 = 1.0e-6  # regularization of the viscosity, eps^2


def _c2(kind, n1, n2, nt, gamma=math.inf, beta=1e-3, regnorm=1, shear=0.0, stream=True, **more):
    return dict(kind=kind, n1=n1, n2=n2, nt=nt, gamma=gamma, beta=beta, regnorm=regnorm, shear=shear, stream=stream,
                **more)


def listed():
    return [
        # the smallest call: one derivative of a 64^2 image, on the default stream as in the README
        dict(name="grad-64", kind="operator", op="grad", n1=64, n2=64, beta=1e-3, gamma=math.inf, stream=False),
        # the mixed batch's most frequent problem, one outer iteration's gradient, mass source
        dict(name="gradient-128-mass", **_c2("gradient", 128, 128, 16, gamma=1e-3, beta=1e-2)),
        # a strongly anisotropic image (a slice stack) with an odd number of time steps, default stream
        dict(name="gradient-256x1024-nt7", **_c2("gradient", 256, 1024, 7, stream=False)),
        # the headline workload's Krylov iteration
        dict(name="matvec-512-nt32", **_c2("matvec", 512, 512, 32)),
        # shear control (sliding interfaces), middle size
        dict(name="matvec-256-shear", **_c2("matvec", 256, 256, 16, shear=-0.5, beta=1e-2)),
        # quality measures of a 512^2 registration
        dict(name="measures-512-nt32", **_c2("measures", 512, 512, 32)),
        # a registration on a budget of two Newton steps (a preview, or one level of a coarse-to-fine
        # series): Krylov iterations, line search and gradients, with iterates that rounding moves little
        dict(name="solve-256", **_c2("solve", 256, 256, 16, newton=2)),
        # volumes: a ragged box for the gradient, a cube for the Krylov iteration
        dict(name="gradient3-64x128x32-nt5", kind="gradient3", n1=64, n2=128, n3=32, nt=5, beta=1e-3, gamma=1e-3,
             stream=False),
        dict(name="matvec3-128-nt16", kind="matvec3", n1=128, n2=128, n3=128, nt=16, beta=1e-3, gamma=math.inf,
             stream=True),
        # warm-start network: prediction for a batch of pairs, one training batch
        dict(name="net-256-b8", kind="net", H=256, W=256, B=8),
        dict(name="train-256-b8", kind="train", H=256, W=256, B=8),
        # many small registrations at once (population studies)
        dict(name="batch-128-x8", kind="batch", n=128, nt=16, pairs=8, workers=8, newton=2),
    ]


def _log2(rng, lo, hi):
    """A power of two in [lo, hi]."""
    return 1 << rng.randint(lo.bit_length() - 1, hi.bit_length() - 1)


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(["operator", "gradient", "matvec", "measures", "solve", "gradient3", "matvec3", "net", "train",
                       "gradient", "matvec"])
    stream = rng.random() < 0.7
    if kind == "operator":
        return dict(kind=kind, op=rng.choice(["grad", "div", "proj", "precond"]), n1=_log2(rng, 16, 1024),
                    n2=_log2(rng, 16, 1024), beta=10.0 ** -rng.randint(2, 3),
                    gamma=rng.choice([math.inf, 1e-3]), stream=stream)
    if kind in ("gradient3", "matvec3"):
        while True:
            c = dict(kind=kind, n1=_log2(rng, 8, 128), n2=_log2(rng, 8, 128), n3=_log2(rng, 8, 128),
                     nt=_logint(rng, 2, 16), beta=1e-3, gamma=rng.choice([0.0, 1e-3, math.inf]), stream=stream)
            if c["n1"] * c["n2"] * c["n3"] >= 16 ** 3 and c["n1"] * c["n2"] * c["n3"] * c["nt"] < 128 ** 3 * 16:
                return c
    if kind in ("net", "train"):
        while True:
            c = dict(kind=kind, H=_log2(rng, 32, 512), W=_log2(rng, 32, 512), B=_logint(rng, 1, 16))
            if 4 * 32 * 32 <= c["H"] * c["W"] * c["B"] < 256 * 256 * 8:
                return c
    if kind == "solve":
        n = _log2(rng, 64, 256)
        return _c2(kind, n, n, _logint(rng, 8, 15), gamma=rng.choice([1e-3, math.inf]), regnorm=rng.randint(1, 2),
                   beta=1e-2, newton=2)
    while True:
        n1, n2, nt = _log2(rng, 32, 1024), _log2(rng, 32, 1024), _logint(rng, 3, 48)
        if n1 * n2 * nt < 512 * 512 * 32 and max(n1, n2) <= 16 * min(n1, n2):
            break
    if kind == "measures":
        return _c2(kind, n1, n2, nt, stream=stream)
    full = kind == "matvec" and rng.random() < 0.2  # the full Newton Hessian
    return _c2(kind, n1, n2, nt, gamma=rng.choice([0.0, 1e-3, math.inf]), beta=10.0 ** -rng.randint(2, 3),
               stream=stream, **(dict(full=True) if full else {}))


# ---------------------------------------------------------------------------
# inputs (FP64 on the device, then FP32), from the seed alone
# ---------------------------------------------------------------------------
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _axes(*n):
    return torch.meshgrid(*[TWO_PI * torch.arange(m, dtype=torch.float64, device=_dev()) / m for m in n],
                          indexing="ij")


def _modes(n1, n2, coef, d1, d2):
    """Real part of sum_k coef[k] (i k1)^d1 (i k2)^d2 exp(i k . x), |k_i| <= K, on the grid."""
    K = coef.shape[0] // 2
    ks = np.arange(-K, K + 1)
    C = coef * (1j * ks[:, None]) ** d1 * (1j * ks[None, :]) ** d2
    E1 = np.exp(1j * np.outer(TWO_PI * np.arange(n1) / n1, ks))
    E2 = np.exp(1j * np.outer(ks, TWO_PI * np.arange(n2) / n2))
    t = lambda a: torch.from_numpy(a).to(_dev())
    return (t(E1) @ t(C) @ t(E2)).real


def _velocity(rng, n1, n2, vmax, kmax=16):
    """Divergence-free velocity with modes |k| <= min(kmax, n/4), max |v| = vmax."""
    K = min(kmax, n1 // 4, n2 // 4)
    ks = np.arange(-K, K + 1)
    kk = ks[:, None] ** 2 + ks[None, :] ** 2
    coef = (rng.standard_normal(kk.shape) + 1j * rng.standard_normal(kk.shape)) / (1.0 + kk)
    coef[(kk == 0) | (kk > K * K)] = 0.0
    v = torch.stack([_modes(n1, n2, coef, 0, 1), -_modes(n1, n2, coef, 1, 0)])
    return v * (vmax / v.square().sum(0).sqrt().max())


def _wrap(d):
    return torch.remainder(d + math.pi, TWO_PI) - math.pi


def _ellipses(X1, X2, params, width):
    out, prev = torch.zeros_like(X1), 0.0
    for c1, c2, a, b, th, c in params:
        d1, d2 = _wrap(X1 - c1), _wrap(X2 - c2)
        p, q = math.cos(th) * d1 + math.sin(th) * d2, -math.sin(th) * d1 + math.cos(th) * d2
        r = torch.sqrt((p / a) ** 2 + (q / b) ** 2)
        out += (c - prev) * 0.5 * (1.0 + torch.tanh((1.0 - r) * math.sqrt(a * b) / width))
        prev = c
    return out


def _vmax(n, nt):
    """Velocity magnitude at CFL number 1/4, at most 0.5."""
    return min(0.5, 0.25 * TWO_PI * nt / n)


def _pair(rng, n1, n2, nt, far=None):
    """(m_T, m_R, v*): five nested ellipses (edges two cells wide), their displaced image and the
    displacement v*, within CFL; far: the image is displaced that far along v* instead (an early
    iterate, whose mismatch is still large)."""
    params = []
    c1, c2 = math.pi + rng.normal(0, 0.15), math.pi + rng.normal(0, 0.15)
    a, b, th = rng.uniform(0.55, 0.7) * math.pi, rng.uniform(0.45, 0.6) * math.pi, rng.uniform(0, math.pi)
    for _ in range(5):
        params.append((c1, c2, a, b, th, rng.uniform(0.1, 1.0)))
        s = rng.uniform(0.6, 0.8)
        a, b = a * s, b * s
        c1, c2, th = c1 + rng.normal(0, 0.1 * a), c2 + rng.normal(0, 0.1 * b), th + rng.normal(0, 0.3)
    v = _velocity(rng, n1, n2, _vmax(max(n1, n2), nt))
    X1, X2 = _axes(n1, n2)
    width = 2.0 * TWO_PI / min(n1, n2)
    d = v if far is None else v * (far / v.square().sum(0).sqrt().max())
    return _ellipses(X1, X2, params, width), _ellipses(X1 - d[0], X2 - d[1], params, width), v


def _smooth3(rng, X, kmax, amp):
    f = torch.zeros_like(X[0])
    for _ in range(8):
        k = rng.integers(-kmax, kmax + 1, size=3)
        f += rng.standard_normal() * torch.cos(sum(float(a) * x for a, x in zip(k, X)) + rng.uniform(0, TWO_PI))
    return amp * f / f.abs().max().clamp_min(1e-30)


def _volume(rng, case):
    """(m_T, m_R, v, v~) of a 3-D problem: bumps, displaced bumps, velocities within CFL."""
    n = (case["n1"], case["n2"], case["n3"])
    X = _axes(*n)
    mT, mR = torch.zeros_like(X[0]), torch.zeros_like(X[0])
    for _ in range(4):
        c, s, amp = rng.uniform(1.5, 4.8, size=3), rng.uniform(4.0, 16.0), rng.uniform(0.4, 1.0)
        d = rng.uniform(-0.2, 0.2, size=3)
        bump = lambda o: amp * torch.exp(-s * sum(torch.sin((x - float(o[i])) / 2) ** 2 for i, x in enumerate(X)))
        mT, mR = mT + bump(c), mR + bump(c + d)
    vmax = min(0.3, 0.5 * case["nt"] / (max(n) / 2))
    v = torch.stack([_smooth3(rng, X, 2, vmax) for _ in range(3)])
    return mT, mR, v, torch.stack([_smooth3(rng, X, min(8, min(n) // 4), 0.2) for _ in range(3)])


def _f32(x):
    return x.to(torch.float32).contiguous()


def _params(rng, trained):
    if trained:
        return np.load(WEIGHTS).astype(np.float32)
    out = []
    for cin, cout in zip(CHANNELS[:-1], CHANNELS[1:]):
        out += [rng.standard_normal(cout * cin * 9) * math.sqrt(2.0 / (9.0 * cin)), 0.01 * rng.standard_normal(cout)]
    return np.concatenate(out).astype(np.float32)


def _inputs(case, seed):
    """The FP32 inputs of a case, by name."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind in ("gradient3", "matvec3"):
        mT, mR, v, vt = _volume(rng, case)
        return dict(mT=_f32(mT), mR=_f32(mR), v=_f32(v), vt=_f32(vt))
    if kind in ("net", "train"):
        pairs = [_pair(rng, case["H"], case["W"], 16) for _ in range(case["B"])]
        return dict(images=_f32(torch.stack([torch.stack(p[:2]) for p in pairs])),
                    targets=_f32(torch.stack([p[2] for p in pairs])),
                    params=torch.from_numpy(_params(rng, kind == "net")).to(_dev()))
    if kind == "batch":
        return dict(pairs=[tuple(_f32(x) for x in _pair(rng, case["n"], case["n"], case["nt"])[:2])
                           for _ in range(case["pairs"])])
    mT, mR, v = _pair(rng, case["n1"], case["n2"], case.get("nt", 16),
                      far=0.2 if kind in ("gradient", "matvec") else None)
    vt = _velocity(rng, case["n1"], case["n2"], float(v.abs().max()))
    if kind == "operator":  # a vector field that is neither smooth nor divergence free, as a body force is
        return dict(mT=_f32(mT), mR=_f32(mR), v=_f32(torch.stack([mT, mR])))
    return dict(mT=_f32(mT), mR=_f32(mR), v=_f32(v if kind == "measures" else 0.5 * v), vt=_f32(vt))


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _stream():
    return torch.cuda.Stream()


def prepare(case, seed):
    x = _inputs(case, seed)
    kind, dev = case["kind"], _dev()
    # a program's contexts share its one working stream (or the default stream)
    stream = _stream() if case.get("stream") else None
    s = dict(case=case, x=x, stream=stream)
    if kind in ("solve", "batch"):
        s["opts"] = binding.default_opts(tol=1e-2, maxit_newton=case["newton"])
    torch.cuda.synchronize()
    if kind in ("net", "train"):
        s["net"] = binding.Net(case["H"], case["W"], case["B"])
        s["net"].set_params(x["params"])
        s["v"] = torch.empty_like(x["targets"])
        s["grads"] = torch.empty_like(x["params"])
    elif kind == "batch":
        # the mixed batch's settings: seminorm, weights and constraint vary from pair to pair
        opts = [(1, 1e-2, math.inf), (1, 1e-3, math.inf), (2, 1e-2, 1e-3), (1, 1e-2, 1e-3), (2, 1e-3, math.inf)]
        n = case["n"]
        s["items"] = [dict(mT=mT, mR=mR, v=torch.zeros(2, n, n, device=dev), nt=case["nt"], regnorm=o[0], beta=o[1],
                           gamma=o[2], shear=0.0) for (mT, mR), o in zip(x["pairs"], opts * case["pairs"])]
        s["executor"] = binding.Executor(case["workers"])
    elif kind in ("gradient3", "matvec3"):
        c = binding.Context3D(case["n1"], case["n2"], case["n3"], case["nt"], beta=case["beta"], gamma=case["gamma"],
                              stream=stream)
        s["ctx"], s["out"] = c, torch.empty_like(x["v"])
        c.set_images(x["mT"], x["mR"])
        if kind == "matvec3":
            c.gradient(x["v"], s["out"])
    else:
        c = binding.Context(case["n1"], case["n2"], case.get("nt", 1), regnorm=case.get("regnorm", 1),
                            beta=case["beta"], gamma=case["gamma"], shear=case.get("shear", 0.0), stream=stream)
        s["ctx"], s["out"] = c, torch.empty_like(x["v"])
        c.set_images(x["mT"], x["mR"])
        if case.get("full"):
            c.set_hessian(True)
        if kind == "matvec":
            c.gradient(x["v"], s["out"])
        if kind == "operator" and case["op"] == "div":
            s["out"] = torch.empty_like(x["mT"])
        if kind == "measures":
            s["detF"], s["labels"] = torch.empty_like(x["mT"]), torch.empty_like(x["mT"])
            s["LT"], s["LR"] = (x["mT"] > 0.3).float(), (x["mR"] > 0.3).float()
    torch.cuda.synchronize()
    return s


def run(s):
    case, x, kind = s["case"], s["x"], s["case"]["kind"]
    if kind == "operator":
        op, c = case["op"], s["ctx"]
        if op == "grad":
            c.spectral_grad(x["mT"], s["out"])
        else:
            dict(div=c.spectral_div, proj=c.apply_proj, precond=c.apply_precond)[op](x["v"], s["out"])
        return s["out"]
    if kind in ("gradient", "gradient3"):
        J = s["ctx"].gradient(x["v"], s["out"])
        return dict(g=s["out"], J=J)
    if kind in ("matvec", "matvec3"):
        s["ctx"].hessian_matvec(x["vt"], s["out"])
        return s["out"]
    if kind == "measures":
        c = s["ctx"]
        det = c.detgrad(x["v"], s["detF"])
        c.displacement(x["v"], s["out"])
        c.label_overlap(x["v"], s["LT"], s["LR"], s["labels"])
        return dict(detF=s["detF"], det=list(det), u=s["out"], labels=s["labels"])
    if kind == "solve":
        st = s["ctx"].solve(s["out"], s["opts"], check=False)
        return dict(v=s["out"], J=st["J"])
    if kind == "batch":
        s["executor"].solve(s["items"], s["opts"], check=False)
        return [it["v"] for it in s["items"]]
    if kind == "net":
        s["net"].forward(x["images"], s["v"])
        return s["v"]
    loss = s["net"].loss_grad(x["images"], x["targets"], s["grads"])
    return dict(loss=loss, grads=s["grads"])


def work(case):
    """Bytes: inputs and the stored state the call reads, outputs it writes, once each.  Flops:
    the real transforms of its derivatives (2.5 N log2 N each; 2-D: one forward, two inverse per
    Heun stage; 3-D: one and three), the convolutions' multiply-adds."""
    kind = case["kind"]
    if kind in ("net", "train"):
        px = case["B"] * case["H"] * case["W"]
        flops = sum(18.0 * a * b for a, b in zip(CHANNELS[:-1], CHANNELS[1:])) * px
        return dict(bytes=16.0 * px, flops=flops * (3 if kind == "train" else 1))
    if kind == "batch":
        N = case["n"] ** 2
        stages = 12 * 4 * case["nt"]  # two Newton steps are about 12 matvecs' worth of transport solves
        return dict(bytes=16.0 * N * case["pairs"], flops=case["pairs"] * stages * 7.5 * N * math.log2(N))
    if kind in ("gradient3", "matvec3"):
        N = case["n1"] * case["n2"] * case["n3"]
        hist = 12.0 * (case["nt"] + 1) * N if kind == "matvec3" else 0.0
        return dict(bytes=36.0 * N + hist, flops=4 * case["nt"] * 10.0 * N * math.log2(N))
    N = case["n1"] * case["n2"]
    stage = 7.5 * N * math.log2(N)
    if kind == "operator":
        return dict(bytes=(12.0 if case["op"] in ("grad", "div") else 16.0) * N, flops=stage)
    if kind == "measures":
        return dict(bytes=32.0 * N, flops=(8 + 4 + 2) * case["nt"] * stage)
    if kind == "solve":
        return dict(bytes=16.0 * N, flops=12 * 4 * case["nt"] * stage)
    hist = 8.0 * (case["nt"] + 1) * N if kind == "matvec" else 8.0 * N
    return dict(bytes=24.0 * N + hist, flops=4 * case["nt"] * stage)


# ---------------------------------------------------------------------------
# the same results in FP64 with torch alone
# ---------------------------------------------------------------------------
class _Box:
    """Spectral operators on a periodic box of any dimension: odd symbols with the Nyquist
    entry zero for first derivatives, the full even |k|^2 for the seminorm."""

    def __init__(self, shape):
        self.shape, self.d, self.dims = shape, len(shape), tuple(range(-len(shape), 0))
        odd, even = [], []
        for a, n in enumerate(shape):
            k = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device=_dev())
            o = k.clone()
            o[n // 2] = 0.0
            view = [1] * self.d
            view[a] = n
            odd.append(o.reshape(view))
            even.append(k.reshape(view))
        self.k = odd
        self.kk = sum(e * e for e in even)
        self.ko = sum(o * o for o in odd)
        self.h = math.prod(TWO_PI / n for n in shape)

    def fft(self, f):
        return torch.fft.fftn(f, dim=self.dims)

    def ifft(self, F):
        return torch.fft.ifftn(F, dim=self.dims).real

    def grad(self, f):
        F = self.fft(f)
        return torch.stack([self.ifft(1j * k * F) for k in self.k])

    def div(self, u):
        return self.ifft(1j * sum(k * self.fft(c) for k, c in zip(self.k, u)))

    def mult(self, m, u):
        return self.ifft(m * self.fft(u))

    def project(self, b, beta, gamma):
        if gamma == 0.0:
            return b
        den = self.ko if math.isinf(gamma) else self.ko + beta * self.kk / (gamma * (1.0 + self.kk))
        coef = torch.where(self.ko > 0, 1.0 / torch.where(self.ko > 0, den, 1.0), 0.0)
        B = [self.fft(c) for c in b]
        kb = coef * sum(k * c for k, c in zip(self.k, B))
        return torch.stack([self.ifft(c - k * kb) for k, c in zip(self.k, B)])


def _dot(g, v):
    return (g * v).sum(0)


def _state(box, m, v, nt):
    h, gm = 1.0 / nt, []
    for _ in range(nt):
        gm.append(box.grad(m))
        k1 = -_dot(gm[-1], v)
        k2 = -_dot(box.grad(m + h * k1), v)
        m = m + 0.5 * h * (k1 + k2)
    gm.append(box.grad(m))
    return m, gm


def _weights(nt):
    return [0.5 / nt if j in (0, nt) else 1.0 / nt for j in range(nt + 1)]


def _adjoint(box, lam, v, nt):
    h, out = 1.0 / nt, [None] * (nt + 1)
    out[nt] = lam
    for j in range(nt, 0, -1):
        k1 = box.div(out[j] * v)
        k2 = box.div((out[j] + h * k1) * v)
        out[j - 1] = out[j] + 0.5 * h * (k1 + k2)
    return out


def _strain(box, v):
    g0, g1 = box.grad(v[0]), box.grad(v[1])
    return torch.stack([g0[0], 0.5 * (g0[1] + g1[0]), g1[1]])


def _contract(E, F):
    return E[0] * F[0] + 2.0 * E[1] * F[1] + E[2] * F[2]


def _div_tensor(box, T):
    return torch.stack([box.div(T[:2]), box.div(T[1:])])


def _regular(box, case, v, vt=None):
    """beta_v A[v], or with vt the second variation beta_v B(v)[vt]."""
    beta, s = case["beta"], case.get("shear", 0.0)
    if s == 0.0:
        return box.mult(beta * box.kk ** case.get("regnorm", 1), v if vt is None else vt)
    nu = (1.0 + s) / (1.0 - s)
    E = _strain(box, v)
    ee = _contract(E, E) + EPS2
    eta = ee ** ((1.0 - nu) / (2.0 * nu))
    if vt is None:
        return -beta * _div_tensor(box, 2.0 * eta * E)
    Et = _strain(box, vt)
    q = ((1.0 - nu) / nu) * _contract(E, Et) / ee
    return -beta * _div_tensor(box, 2.0 * eta * (Et + q * E))


def _assemble(box, case, Av, b):
    if case.get("shear", 0.0) != 0.0:  # incompressible: the projection acts on the sum
        return box.project(Av + b, case["beta"], math.inf)
    return Av + box.project(b, case["beta"] if case.get("regnorm", 1) == 1 else 1.0, case["gamma"])


def _registration(case, x, want):
    shape = tuple(x["mT"].shape)
    box, nt = _Box(shape), case["nt"]
    mT, mR, v, vt = (x[k].double() for k in ("mT", "mR", "v", "vt"))
    m1, gm = _state(box, mT, v, nt)
    w = _weights(nt)
    if want == "gradient":
        lam = _adjoint(box, mR - m1, v, nt)
        b = sum(w[j] * lam[j] * gm[j] for j in range(nt + 1))
        Av = _regular(box, case, v)
        J = 0.5 * box.h * (mR - m1).square().sum()
        s = case.get("shear", 0.0)
        if s != 0.0:
            nu = (1.0 + s) / (1.0 - s)
            E = _strain(box, v)
            J = J + case["beta"] * 2.0 * nu / (nu + 1.0) * box.h * (
                (_contract(E, E) + EPS2) ** ((1.0 + nu) / (2.0 * nu))).sum()
        else:
            J = J + 0.5 * box.h * (Av * v).sum()
        if 0.0 < case["gamma"] < math.inf:
            d = box.div(v)
            J = J + 0.5 * case["gamma"] * box.h * (box.mult(1.0 + box.kk, d) * d).sum()
        return dict(g=_assemble(box, case, Av, b), J=float(J))
    h, mt, gmt, full = 1.0 / nt, torch.zeros_like(mT), [], case.get("full")
    for j in range(nt):
        g = box.grad(mt)
        gmt.append(g if full else None)
        k1 = -_dot(g, v) - _dot(gm[j], vt)
        k2 = -_dot(box.grad(mt + h * k1), v) - _dot(gm[j + 1], vt)
        mt = mt + 0.5 * h * (k1 + k2)
    if full:
        gmt.append(box.grad(mt))
        lam = _adjoint(box, mR - m1, v, nt)
        lt, b = -mt, w[nt] * (-mt * gm[nt] + lam[nt] * gmt[nt])
        for j in range(nt, 0, -1):
            k1 = box.div(lt * v) + box.div(lam[j] * vt)
            k2 = box.div((lt + h * k1) * v) + box.div(lam[j - 1] * vt)
            lt = lt + 0.5 * h * (k1 + k2)
            b = b + w[j - 1] * (lt * gm[j - 1] + lam[j - 1] * gmt[j - 1])
    else:
        lt = _adjoint(box, -mt, v, nt)
        b = sum(w[j] * lt[j] * gm[j] for j in range(nt + 1))
    return _assemble(box, case, _regular(box, case, v, vt), b)


def _measures(case, x):
    box, nt, h = _Box(tuple(x["mT"].shape)), case["nt"], 1.0 / case["nt"]
    v = x["v"].double()
    gv = torch.stack([box.grad(v[0]), box.grad(v[1])])
    F = torch.zeros((2, 2) + box.shape, dtype=torch.float64, device=v.device)
    F[0, 0] = F[1, 1] = 1.0

    def rhs(F):
        adv = torch.stack([torch.stack([_dot(box.grad(F[a, b]), v) for b in range(2)]) for a in range(2)])
        return torch.einsum("acxy,cbxy->abxy", gv, F) - adv

    u = torch.zeros_like(v)

    def move(u):
        return v - torch.stack([_dot(box.grad(c), v) for c in u])

    for _ in range(nt):
        k1 = rhs(F)
        F = F + 0.5 * h * (k1 + rhs(F + h * k1))
        k1 = move(u)
        u = u + 0.5 * h * (k1 + move(u + h * k1))
    det = F[0, 0] * F[1, 1] - F[0, 1] * F[1, 0]
    D = torch.sqrt((F[0, 0] - 1) ** 2 + F[0, 1] ** 2 + F[1, 0] ** 2 + (F[1, 1] - 1) ** 2)
    sigma = 3.0 * TWO_PI / case["n1"]
    labels = box.mult(torch.exp(-0.5 * sigma * sigma * box.kk), (x["mT"] > 0.3).double())
    stats = [float(t) for t in (det.min(), det.mean(), det.max(), D.max(), D.mean())]
    return dict(detF=det, det=stats, u=u, labels=_state(box, labels, v, nt)[0])


def _network(case, x, train):
    H, W = case["H"], case["W"]
    box = _Box((H, W))
    p = x["params"].double().requires_grad_(train)
    a, o = x["images"].double(), 0
    sigma = 2.0 * TWO_PI / max(H, W)
    low = torch.exp(-0.5 * sigma * sigma * box.kk)
    with torch.set_grad_enabled(train):
        for l, (cin, cout) in enumerate(zip(CHANNELS[:-1], CHANNELS[1:])):
            w, b = p[o:o + 9 * cin * cout].reshape(cout, cin, 3, 3), p[o + 9 * cin * cout:o + 9 * cin * cout + cout]
            o += 9 * cin * cout + cout
            d = max(1, min(DILATION[l], H // 8, W // 32))
            z = b.reshape(1, -1, 1, 1)
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    z = z + torch.einsum("oc,bcyx->boyx", w[:, :, dy + 1, dx + 1],
                                         torch.roll(a, (-d * dy, -d * dx), (-2, -1)))
            a = torch.relu(z) if l < 7 else z
        Z = low * torch.fft.fft2(a)
        coef = torch.where(box.ko > 0, 1.0 / torch.where(box.ko > 0, box.ko, 1.0), 0.0)
        kb = coef * (box.k[0] * Z[:, 0] + box.k[1] * Z[:, 1])
        v = torch.fft.ifft2(Z - torch.stack([box.k[0] * kb, box.k[1] * kb], 1)).real
        if not train:
            return v
        loss = 0.5 * (v - x["targets"].double()).square().mean()
        loss.backward()
    return dict(loss=float(loss.detach()), grads=p.grad)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "batch"):  # iterations that stop on a tolerance
        return None
    x = _inputs(case, seed)
    if kind == "operator":
        box = _Box((case["n1"], case["n2"]))
        if case["op"] == "grad":
            return box.grad(x["mT"].double())
        v = x["v"].double()
        if case["op"] == "div":
            return box.div(v)
        if case["op"] == "proj":
            return box.project(v, case["beta"], case["gamma"])
        return box.mult(1.0 / (case["beta"] * torch.where(box.kk > 0, box.kk, 1.0)), v)
    if kind in ("gradient", "gradient3"):
        return _registration(case, x, "gradient")
    if kind in ("matvec", "matvec3"):
        return _registration(case, x, "matvec")
    if kind == "measures":
        return _measures(case, x)
    return _network(case, x, kind == "train")
