"""Performance cases of the library: what its users have it do, at the sizes they do it.

Each case is one call (or one short run) through the public binding: deposits and gathers of
single precision and double precision, PIC runs with and without a width schedule, width
selection by cross-validation in the forms the library picks by itself, an ensemble step and a
batch of served requests.  Sizes and distributions are those of the repository's workloads
(`bench.py`, `kde_inputs`) and tests: 2^10 to 2^22 particles, grids of 64 to 4096 nodes,
uniform widths of 1 to 1e4 and particle-wise widths log-uniform in [5, 5e3].

Outputs.  Numbers are returned in the precision of the arithmetic that makes them: field
energies and CV curves, which the library reports in float64 containers but sums from FP32
terms (CV values to 2e-6 of their maximum, FP32 energies to 1e-5), come back as float32; FP64
runs return float64.  Positions come back as coordinates in [-L/2, L/2) (the 32-bit codes are
the fixed-point form of these), and a run of several steps returns its particles by label, since
the order inside a grid cell is the library's own.

`exact` evaluates the same formulas in 64 bits with plain torch: dense sums over nodes and
particles, Fourier series of the kernel where the sums run over pairs.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1804_11174_gb300 as kp

DEV = "cuda:0"
TWO32 = 4294967296.0
L4PI = 4 * math.pi
SCALES = 10.0 ** ((np.arange(16) - 8) / 8.0)  # the width factors of a served CV request


def listed():
    return [
        # the smallest calls: one density on a coarse grid, as in the cold Langmuir set-up
        {"name": "deposit_small", "kind": "deposit", "N": 4096, "Ng": 64, "kappa": 30.0, "weights": False, "f64": False},
        # weighted particles with a narrow uniform kernel (a few nodes wide), odd count
        {"name": "deposit_weights", "kind": "deposit", "N": 300007, "Ng": 512, "kappa": 2000.0, "weights": True,
         "f64": False},
        # the largest served deposit: particle-wise widths on the finest grid
        {"name": "deposit_request", "kind": "deposit", "N": 4000037, "Ng": 4096, "kappa": 0.0, "weights": False,
         "f64": False},
        # a double-precision density with particle-wise widths on a grid that is no power of two
        {"name": "deposit_f64", "kind": "deposit", "N": 65537, "Ng": 100, "kappa": 0.0, "weights": False, "f64": True},
        # a small field interpolation with one width
        {"name": "gather_small", "kind": "gather", "N": 5000, "Ng": 256, "kappa": 60.0, "f64": False},
        # a served gather: particle-wise widths
        {"name": "gather_request", "kind": "gather", "N": 1000003, "Ng": 1024, "kappa": 0.0, "f64": False},
        # the Landau-damping run: one width-update period (CV over 64 candidates, Silverman
        # widths, 50 steps) at the flagship size
        {"name": "pic_landau", "kind": "pic", "N": 1 << 20, "Ng": 256, "steps": 50, "kappa": 0.0, "f64": False},
        # the cold Langmuir wave in double precision, a short stretch of its many small steps
        {"name": "pic_langmuir_f64", "kind": "pic", "N": 4096, "Ng": 64, "steps": 20, "kappa": 100.0, "f64": True},
        # width selection on a clustered sample with leave-one-out densities
        {"name": "cv_sweep", "kind": "cv", "N": 1 << 18, "n_cand": 64, "scale": False},
        # a served width selection: factors on particle-wise widths
        {"name": "cv_scale", "kind": "cv", "N": 50021, "n_cand": 16, "scale": True},
        # one step of an ensemble of independent realisations of unequal sizes
        {"name": "ensemble", "kind": "ensemble", "R": 32, "log2_lo": 14.0, "log2_hi": 20.0},
        # a batch of mixed requests from host buffers through the request server
        {"name": "serve", "kind": "serve", "R": 24, "log2_hi": 18.0},
    ]


def _logint(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    """One more case: a kind as the listed ones stand for it, sizes log-uniform over its range."""
    kind = rng.choice(["deposit", "deposit", "gather", "gather", "pic", "pic", "cv", "cv_scale", "ensemble", "serve"])
    f64 = rng.random() < 0.25
    per = rng.random() < 0.5
    kappa = 0.0 if per else round(10.0 ** rng.uniform(0.0, 4.0), 3)
    Ng = _logint(rng, 64, 4096)
    if kind in ("deposit", "gather"):
        # FP64 exponentials are slow on this part: FP64 calls up to 2^17 particles
        c = {"kind": kind, "N": _logint(rng, 1 << 10, (1 << 17) if f64 else 4000000), "Ng": Ng, "kappa": kappa,
             "f64": f64}
        if kind == "deposit":
            c["weights"] = rng.random() < 0.3
        return c
    if kind == "pic":
        N = _logint(rng, 1 << 10, (1 << 16) if f64 else (1 << 20))
        if f64:
            return {"kind": "pic", "N": N, "Ng": _logint(rng, 64, 512), "steps": rng.randint(2, 10),
                    "kappa": kappa if kappa else 100.0, "f64": True}
        return {"kind": "pic", "N": N, "Ng": _logint(rng, 64, 2048), "steps": rng.randint(2, 50), "kappa": kappa,
                "f64": False}
    if kind == "cv":
        return {"kind": "cv", "N": _logint(rng, 1 << 9, 1 << 19), "n_cand": rng.randint(8, 64), "scale": False}
    if kind == "cv_scale":
        return {"kind": "cv", "N": _logint(rng, 1 << 10, 1 << 16), "n_cand": 16, "scale": True}
    if kind == "ensemble":
        lo = round(rng.uniform(11.0, 15.0), 2)
        return {"kind": "ensemble", "R": rng.randint(4, 32), "log2_lo": lo, "log2_hi": round(lo + rng.uniform(1, 4), 2)}
    return {"kind": "serve", "R": 4 * rng.randint(2, 6), "log2_hi": round(rng.uniform(13.0, 17.5), 2)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
_CTX = None


def _ctx():
    """The program's one context (a user keeps it for the life of the program)."""
    global _CTX
    if _CTX is None:
        _CTX = kp.Context(0)
    return _CTX


class _Rand:
    """Seeded draws on the device."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed) * 7919 + 12345)

    def uniform(self, n):
        return torch.rand(n, generator=self.g, device=DEV, dtype=torch.float64)

    def normal(self, n):
        return torch.randn(n, generator=self.g, device=DEV, dtype=torch.float64)

    def codes(self, t):
        """32-bit position codes of positions t in turns [0, 1), as the int32 tensors the binding takes."""
        c = torch.floor(torch.remainder(t, 1.0) * TWO32).to(torch.int64).clamp_(0, (1 << 32) - 1)
        return torch.where(c >= 1 << 31, c - (1 << 32), c).to(torch.int32)

    def landau(self, n, alpha=0.05, q=None):
        """Positions of 1 + alpha cos(2 pi t) by inverse CDF (Newton; q: the quantiles)."""
        q = self.uniform(n) if q is None else q
        t = q.clone()
        for _ in range(6):
            f = t + alpha / (2 * math.pi) * torch.sin(2 * math.pi * t) - q
            t = t - f / (1 + alpha * torch.cos(2 * math.pi * t))
        return self.codes(t)

    def mixture(self, n):
        """0.7 uniform + 0.3 clustered near the middle (a von Mises peak of kappa = 20)."""
        u = self.uniform(n)
        peak = 0.5 + self.normal(n) / (2 * math.pi * math.sqrt(20.0))
        return self.codes(torch.where(self.uniform(n) < 0.7, u, peak))

    def widths(self, n, dtype=torch.float32, lo=5.0, hi=5e3):
        return (lo * torch.exp(self.uniform(n) * math.log(hi / lo))).to(dtype)


def _candidates(n):
    return 1e4 ** (np.arange(n, dtype=np.float64) / max(n - 1, 1))


def _ens_sizes(case):
    R, lo, hi = case["R"], case["log2_lo"], case["log2_hi"]
    f = [((r * 0.6180339887498949) % 1.0) for r in range(R)]  # evenly spread sizes
    Ns = [int(round(2.0 ** (lo + (hi - lo) * x))) for x in f]
    Ngs = [(128, 256, 512, 1024)[r % 4] for r in range(R)]
    kap = [10.0 ** (3.0 * ((r * 0.7548776662466927) % 1.0)) for r in range(R)]
    return Ns, Ngs, kap


def _serve_requests(case, seed):
    """Kinds cycle deposit / gather / CV / 10-step PIC; N log-uniform from 2^12, CV up to 2^14."""
    rs = np.random.RandomState(int(seed) % (1 << 31))
    pin = lambda a: torch.from_numpy(a).pin_memory().numpy()
    out = []
    for q in range(case["R"]):
        kind = 1 + q % 4
        top = min(14.0, case["log2_hi"]) if kind == 3 else case["log2_hi"]
        N = int(2.0 ** (12.0 + (top - 12.0) * ((q * 0.6180339887498949) % 1.0)))
        Ng = int(round(64.0 * 64.0 ** ((q * 0.7548776662466927) % 1.0)))
        r = {"kind": kind, "N": N, "Ng": Ng, "u": pin(rs.randint(0, 1 << 32, N, dtype=np.uint32)),
             "kappa": pin((5.0 * 1e3 ** rs.random_sample(N)).astype(np.float32))}
        if kind == 2:
            g = np.arange(Ng) * (2 * math.pi / Ng)
            r["field"] = pin((np.sin(g) + 0.3 * np.cos(3 * g + q)).astype(np.float32))
        if kind == 4:
            r["v"] = pin(rs.standard_normal(N).astype(np.float32))
        out.append(r)
    return out


def _inputs(case, seed):
    """The arrays a user holds before the call."""
    kind, R, s = case["kind"], _Rand(seed), {}
    if kind == "ensemble":
        n = sum(_ens_sizes(case)[0])
        return {"u": R.landau(n), "v": R.normal(n).float()}
    N = case["N"]
    dt = torch.float64 if case.get("f64") else torch.float32
    if kind == "cv":
        s["L"] = L4PI if case["scale"] else 2 * math.pi
        s["u"] = R.landau(N) if case["scale"] else R.mixture(N)
        s["kr"] = R.widths(N) if case["scale"] else None
        s["cand"] = SCALES if case["scale"] else _candidates(case["n_cand"])
        return s
    if kind == "pic":
        if case["f64"]:  # quiet start, cold: the Langmuir wave
            q = (torch.arange(N, dtype=torch.float64, device=DEV) + R.uniform(1)) / N
            return {"u": R.landau(N, 0.01, q), "v": torch.zeros(N, dtype=dt, device=DEV)}
        return {"u": R.landau(N), "v": R.normal(N).to(dt)}
    s["u"] = R.landau(N)
    s["kappa"] = R.widths(N, dt, hi=500.0 if case["f64"] else 5e3) if case["kappa"] == 0.0 else None
    if kind == "deposit":
        s["w"] = (0.5 + R.uniform(N)).to(dt) if case["weights"] else None
    else:
        g = torch.arange(case["Ng"], dtype=torch.float64, device=DEV) * (2 * math.pi / case["Ng"])
        a = R.uniform(4)
        s["field"] = (torch.sin(g + 6 * a[0]) + 0.3 * torch.cos(3 * g + 6 * a[1]) + 0.1 * a[2]
                      + 0.02 * R.normal(case["Ng"])).to(dt)
    return s


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        s = {"reqs": _serve_requests(case, seed)}
        pin = lambda n, dt: torch.empty(n, dtype=dt).pin_memory().numpy()
        for r in s["reqs"]:
            k = r["kind"]
            r["out"] = pin(r["Ng"] if k == 1 else r["N"], torch.float32) if k in (1, 2) else None
            r["out64"] = pin(16 if k == 3 else 10, torch.float64) if k in (3, 4) else None
        s["server"] = kp.Server(0, n_slots=4, hbm_budget_bytes=100 << 30)
        return {"case": case, "ctx": _ctx(), **s}
    s = {"case": case, "ctx": _ctx(), **_inputs(case, seed)}
    if kind == "ensemble":
        Ns, Ngs, kap = _ens_sizes(case)
        s["u0"], s["v0"] = s["u"].clone(), s["v"].clone()
        s["energy"] = torch.zeros(len(Ns), dtype=torch.float64, device=DEV)
        s["ens"] = kp.Ensemble(s["ctx"], Ns, Ngs, kap, L4PI, 0.1, s["u"], s["v"])
    elif kind == "cv":
        s["loo"] = torch.empty(case["N"], device=DEV)
    elif kind == "pic":
        N, kw = case["N"], {}
        if case["kappa"] == 0.0:  # the width schedule: an update at step 0 and every 50 steps
            kw = dict(kappa=torch.ones(N, device=DEV), width_every=50, cand=_candidates(64), alpha=0.5, kappa_min=1.0,
                      kappa_max=1e5)
        s["st"] = kp.PicState(s["u"], s["v"], L4PI, case["Ng"], 0.1, kappa_uniform=case["kappa"],
                              ids=torch.arange(N, dtype=torch.int32, device=DEV), max_steps=case["steps"], **kw)
        s["snap"] = s["st"].snapshot()
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _coords(u, L, dtype):
    """Coordinates in [-L/2, L/2) of position codes (int32: the upper half of the box is negative)."""
    return u.to(dtype) * (L / TWO32)


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "deposit":
        return ctx.deposit(s["u"], case["Ng"], L4PI, kappa=s["kappa"], kappa_uniform=case["kappa"], weight=s["w"],
                           dtype=torch.float64 if case["f64"] else torch.float32)
    if kind == "gather":
        return ctx.gather(s["u"], s["field"], L4PI, kappa=s["kappa"], kappa_uniform=case["kappa"])
    if kind == "pic":
        st = s["st"]
        st.restore(s["snap"])
        ctx.pic_step(st, case["steps"])
        # the particles by label
        at = st.id.long()
        dt = st.v.dtype
        out = {"x": torch.empty_like(st.v).index_copy_(0, at, _coords(st.u, L4PI, dt)),
               "v": torch.empty_like(st.v).index_copy_(0, at, st.v), "energy": st.energy.to(dt)}
        if st.kappa is not None:
            out["kappa"] = torch.empty_like(st.kappa).index_copy_(0, at, st.kappa)
            out["kappa_star"] = st.kappa_star.clone()
        return out
    if kind == "cv":
        cv, am, loo = ctx.cv(s["u"], s["L"], s["cand"], kappa_rel=s["kr"], loo=s["loo"])
        return {"cv": cv.astype(np.float32), "argmin": am, "loo": loo}
    if kind == "ensemble":
        s["u"].copy_(s["u0"])
        s["v"].copy_(s["v0"])
        s["ens"].run(1, s["energy"])
        return {"x": _coords(s["u"], L4PI, torch.float32), "v": s["v"], "energy": s["energy"].float()}
    srv = s["server"]
    tickets = [srv.submit(r["kind"], r["u"], L4PI, Ng=r["Ng"], kappa=r["kappa"], v=r.get("v"), field=r.get("field"),
                          cand=SCALES if r["kind"] == 3 else None, n_steps=10 if r["kind"] == 4 else 0, dt=0.1,
                          out=r["out"], out64=r["out64"]) for r in s["reqs"]]
    done = [srv.wait(t) for t in tickets]
    return [[r["out"] if r["out"] is not None else r["out64"].astype(np.float32), d[2] if r["kind"] == 3 else 0]
            for r, d in zip(s["reqs"], done)]


def work(case):
    """Every input read once and every output written once; a pass over a particle cannot do
    with fewer operations than forming its kernel's value and adding it (about ten)."""
    kind = case["kind"]
    if kind == "serve":
        b = f = 0
        for r in range(case["R"]):
            k = 1 + r % 4
            top = min(14.0, case["log2_hi"]) if k == 3 else case["log2_hi"]
            N = int(2.0 ** (12.0 + (top - 12.0) * ((r * 0.6180339887498949) % 1.0)))
            b += N * (8 + (4 if k in (2, 4) else 0))
            f += 10 * N
        return {"bytes": b, "flops": f}
    if kind == "ensemble":
        n = sum(_ens_sizes(case)[0])
        return {"bytes": n * 16, "flops": 20 * n}
    N, el = case["N"], 8 if case.get("f64") else 4
    if kind == "cv":
        return {"bytes": N * (8 + (4 if case["scale"] else 0)), "flops": 10 * N * case["n_cand"]}
    if kind == "pic":
        per = case["kappa"] == 0.0
        return {"bytes": case["steps"] * N * (8 + 2 * el + (el if per else 0)), "flops": 20 * N * case["steps"]}
    b = N * 4 + case["Ng"] * el + (N * el if case["kappa"] == 0.0 else 0)
    if kind == "deposit":
        b += N * el if case["weights"] else 0
    else:
        b += N * el
    return {"bytes": b, "flops": 10 * N}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _i0e(k):
    """exp(-k) I0(k) in FP64 (torch's, good to a few ulp)."""
    return torch.special.i0e(k)


def _theta(u):
    return u.to(torch.int64).remainder(1 << 32).double() * (2 * math.pi / TWO32)


def _dense(th, kap, Ng, w=None, field=None):
    """sum_i w_i norm_i e^(kappa_i (cos - 1)) at the nodes, or for a field the particles' sums."""
    half = torch.arange(Ng, dtype=torch.float64, device=DEV) * (math.pi / Ng)
    S, C = torch.sin(half), torch.cos(half)
    norm = 1.0 / (2 * math.pi * _i0e(kap))
    out = torch.zeros(Ng, dtype=torch.float64, device=DEV) if field is None else torch.empty_like(th)
    step = max(1, (1 << 26) // Ng)
    for a in range(0, th.numel(), step):
        t, k, n = th[a:a + step] / 2, kap[a:a + step], norm[a:a + step]
        e = torch.outer(torch.cos(t), S)
        e -= torch.outer(torch.sin(t), C)
        e.square_().mul_((-2.0 * k)[:, None]).exp_()
        if field is None:
            out += (n * w[a:a + step]) @ e
        else:
            out[a:a + step] = (e @ field) * n
    return out


def _poisson(rho, L):
    """E with dE/dx = 1 - rho on the periodic grid (no mean, no Nyquist mode)."""
    Ng = rho.numel()
    r = torch.fft.rfft(1.0 - rho)
    m = torch.arange(r.numel(), dtype=torch.float64, device=DEV)
    keep = (m > 0) & (2 * m != Ng)
    e = torch.where(keep, r / (1j * torch.where(keep, m, 1.0) * (2 * math.pi / L)), 0.0)
    return torch.fft.irfft(e, n=Ng)


def _ratios(k, M):
    """A_m(k) = I_m / I_0 for m = 0..M (k: any shape), stacked along a new first axis: the
    backward recurrence of I_m / I_(m-1)."""
    start = M + 64 + int(2.0 * math.sqrt(float(k.max())))
    r = k / (start + 0.5 + torch.sqrt((start + 0.5) ** 2 + k * k))
    A = torch.empty((M + 1,) + tuple(k.shape), dtype=torch.float64, device=k.device)
    for m in range(start, 0, -1):
        r = 1.0 / (2.0 * m / k + r)
        if m <= M:
            A[m] = r
    A[0] = 1.0
    for m in range(1, M + 1):
        A[m] *= A[m - 1]
    return A


def _modes(k):
    return int(math.ceil(math.sqrt(78.4 * k))) + 8


def _phase(u, m):
    """e^(i m theta) with the exact integer phase m u mod 2^32."""
    t = (u * m).remainder(1 << 32).double() * (2 * math.pi / TWO32)
    return torch.cos(t), torch.sin(t)


def _cv_uniform(u, L, cand, want_loo=True):
    """CV curve, argmin and leave-one-out densities for uniform widths by the Fourier series."""
    uu = u.to(torch.int64).remainder(1 << 32)
    n, M = float(uu.numel()), _modes(max(cand))
    S = torch.empty(M + 1, 2, dtype=torch.float64, device=DEV)
    for m in range(1, M + 1):
        c, s = _phase(uu, m)
        S[m, 0], S[m, 1] = c.sum(), s.sum()
    P = S[1:].square().sum(1)
    k = torch.tensor(cand, dtype=torch.float64, device=DEV)
    A = _ratios(k, M)[1:]  # [M, n_cand]
    f2 = (n * n + 2 * (A * A * P[:, None]).sum(0)) / (2 * math.pi * n * n)
    pairs = (n * n + 2 * (A * P[:, None]).sum(0)) / (2 * math.pi) - n / (2 * math.pi * _i0e(k))
    cv = (2 * math.pi / L) * (f2 - 2 * pairs / (n * (n - 1)))
    am = int(cv.argmin())
    loo = None
    if want_loo:
        acc = torch.full_like(uu, n, dtype=torch.float64)
        for m in range(1, _modes(cand[am]) + 1):
            c, s = _phase(uu, m)
            acc += 2 * float(A[m - 1, am]) * (c * S[m, 0] + s * S[m, 1])
        loo = (2 * math.pi / L) * (acc / (2 * math.pi) - 1 / (2 * math.pi * _i0e(k[am]))) / (n - 1)
    return cv, am, loo


def _cv_scaled(u, kr, L, cand):
    """The same for widths cand[c] kappa_j: F_m = sum_j A_m(cand kappa_j) e^(i m theta_j)."""
    uu = u.to(torch.int64).remainder(1 << 32)
    k = torch.tensor(cand, dtype=torch.float64, device=DEV)[:, None] * kr.double()  # [n_cand, N]
    n, M = float(uu.numel()), _modes(float(k.max()))
    A = _ratios(k, M)
    S = torch.empty(M + 1, 2, dtype=torch.float64, device=DEV)
    F = torch.zeros(len(cand), M + 1, 2, dtype=torch.float64, device=DEV)
    for m in range(1, M + 1):
        e = torch.stack(_phase(uu, m), 1)
        S[m] = e.sum(0)
        F[:, m] = A[m] @ e
    del A
    f2 = (n * n + 2 * F.square().sum((1, 2))) / (2 * math.pi * n * n)
    own = 1 / (2 * math.pi * _i0e(k))
    pairs = (n * n + 2 * (F[:, 1:] * S[1:]).sum((1, 2))) / (2 * math.pi) - own.sum(1)
    cv = (2 * math.pi / L) * (f2 - 2 * pairs / (n * (n - 1)))
    am = int(cv.argmin())
    acc = torch.full((uu.numel(),), n, dtype=torch.float64, device=DEV)
    for m in range(1, M + 1):
        c, s = _phase(uu, m)
        acc += 2 * (c * F[am, m, 0] + s * F[am, m, 1])
    loo = (2 * math.pi / L) * (acc / (2 * math.pi) - own[am]) / (n - 1)
    return cv, am, loo


def _pic(u, v, L, Ng, dt, steps, kap, sched=None):
    """Leap-frog steps in 64 bits on 32-bit position codes (half kick on the first); sched: the
    candidates of the width update at step 0."""
    uu, v = u.to(torch.int64).remainder(1 << 32), v.double().clone()
    N = uu.numel()
    kap = kap.double().expand(N).clone()
    star = None
    if sched is not None:
        _, am, loo = _cv_uniform(uu, L, sched)
        star = sched[am]
        K0 = (2 * math.pi / L) / (2 * math.pi * float(_i0e(torch.tensor(star, dtype=torch.float64))))
        f = ((N - 1) * loo + K0) / N
        lg = f.log()
        kap = (star * torch.exp(lg - lg.mean())).clamp(1.0, 1e5)
    w = torch.full((N,), L / N * 2 * math.pi / L, dtype=torch.float64, device=DEV)
    en = torch.empty(steps, dtype=torch.float64)
    for s in range(steps):
        th = uu.double() * (2 * math.pi / TWO32)
        E = _poisson(_dense(th, kap, Ng, w=w), L)
        en[s] = 0.5 * float(E.square().sum()) * L / Ng
        Ei = _dense(th, kap, Ng, field=E) * (2 * math.pi / Ng)
        v = v - (0.5 if s == 0 else 1.0) * dt * Ei
        uu = (uu + torch.round(v * (dt * TWO32 / L)).to(torch.int64)).remainder(1 << 32)
    x = torch.where(uu >= 1 << 31, uu - (1 << 32), uu).double() * (L / TWO32)
    return {"x": x, "v": v, "energy": en, "kappa": kap, "star": star}


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        out = []
        for r in _serve_requests(case, seed):
            u = torch.from_numpy(r["u"].astype(np.int64)).to(DEV)
            k = torch.from_numpy(r["kappa"]).to(DEV).double()
            th = _theta(u)
            if r["kind"] == 1:
                w = torch.full_like(th, 2 * math.pi / r["N"])
                out.append([_dense(th, k, r["Ng"], w=w), 0])
            elif r["kind"] == 2:
                f = torch.from_numpy(r["field"]).to(DEV).double()
                out.append([_dense(th, k, r["Ng"], field=f) * (2 * math.pi / r["Ng"]), 0])
            elif r["kind"] == 3:
                cv, am, _ = _cv_scaled(u, k, L4PI, list(SCALES))
                out.append([cv, am])
            else:
                p = _pic(u, torch.from_numpy(r["v"]).to(DEV), L4PI, r["Ng"], 0.1, 10, k)
                out.append([p["energy"], 0])
        return out
    s = _inputs(case, seed)
    if kind == "cv":
        if case["scale"]:
            cv, am, loo = _cv_scaled(s["u"], s["kr"], s["L"], list(s["cand"]))
        else:
            cv, am, loo = _cv_uniform(s["u"], s["L"], list(s["cand"]))
        return {"cv": cv, "argmin": am, "loo": loo}
    if kind == "ensemble":
        Ns, Ngs, kap = _ens_sizes(case)
        xs, vs, es, a = [], [], [], 0
        for N, Ng, k in zip(Ns, Ngs, kap):
            u, v = s["u"][a:a + N], s["v"][a:a + N]
            cell = (u.to(torch.int64).remainder(1 << 32) * Ng) >> 32
            order = torch.sort(cell, stable=True)[1]  # a step leaves the particles in cell order
            p = _pic(u[order], v[order], L4PI, Ng, 0.1, 1, torch.tensor([k], dtype=torch.float64, device=DEV))
            xs.append(p["x"])
            vs.append(p["v"])
            es.append(p["energy"])
            a += N
        return {"x": torch.cat(xs), "v": torch.cat(vs), "energy": torch.cat(es)}
    if kind == "pic":
        per = case["kappa"] == 0.0
        k = torch.tensor([1.0 if per else case["kappa"]], dtype=torch.float64, device=DEV)
        p = _pic(s["u"], s["v"], L4PI, case["Ng"], 0.1, case["steps"], k, list(_candidates(64)) if per else None)
        out = {"x": p["x"], "v": p["v"], "energy": p["energy"]}
        if per:
            out["kappa"] = p["kappa"]
            out["kappa_star"] = torch.full((case["steps"],), p["star"], dtype=torch.float64)
        return out
    th = _theta(s["u"])
    k = s["kappa"].double() if s["kappa"] is not None else torch.full_like(th, case["kappa"])
    if kind == "deposit":
        w = s["w"].double() * (2 * math.pi / L4PI) if s["w"] is not None else torch.full_like(th, 2 * math.pi / case["N"])
        return _dense(th, k, case["Ng"], w=w)
    return _dense(th, k, case["Ng"], field=s["field"].double()) * (2 * math.pi / case["Ng"])
