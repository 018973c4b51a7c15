"""Compressed deposit and gather (particles summed into, or interpolated from, Chebyshev proxy
particles) against the oracle and against the sweep over the particles themselves.

Tolerance.  Each interpolant is below 2e-8 of the kernel's peak, times the Lebesgue constants
of both directions (about 3 each): 2e-7; FP32 rounding of the sums stays below 5e-7 in L2 (the
bound the direct sweep's own tests use is 2e-6).  1e-6 relative L2 covers both.  The direct
sweep is reached by a truncation cut other than the default (2^-25: a wider window only).
"""
import math

import numpy as np
import pytest

import kde_inputs as I
from conftest import rel_l2, to_dev, to_dev_u

pytestmark = pytest.mark.gpu
L = 4 * math.pi
TOL = 1e-6


def widths(kind, seed, N):
    if kind == "one":  # particle-wise widths that are all the same
        return np.full(N, 40.0, np.float32)
    lo, hi = {"narrow": (13.0, 16.0), "ten": (5.0, 50.0), "wide": (5.0, 5e3), "widest": (0.5, 4e4)}[kind]
    return I.log_uniform(seed, I.STREAM_KAPPA, N, lo, hi).astype(np.float32)


def positions(seed, N, where):
    u, _ = I.landau_load(seed, N, L, 0.05, 1.0)
    if where == "spike":  # half of them in one cell next to the wrap-around point
        u[::2] = np.uint32(0xFFFFFFFF) - (u[::2] >> np.uint32(14))
    return u


CASES = [  # N, Ng, uniform width or distribution, positions
    (20000, 256, 0.3, "box"), (70001, 256, 3.0, "box"), (70001, 256, 14.0, "box"), (70001, 100, 60.0, "box"),
    (70001, 1000, 300.0, "box"), (50000, 64, 800.0, "box"), (70001, 512, 5000.0, "spike"), (3000, 33, 2.0, "box"),
    (5000, 1, 4.0, "box"), (5000, 2, 4.0, "box"), (400, 4096, 1.5, "box"),
    (70001, 256, "one", "box"), (70001, 256, "narrow", "box"), (20000, 100, "narrow", "spike"),
    (70001, 1000, "ten", "box"), (70001, 256, "wide", "box"), (70001, 3001, "wide", "spike"), (70001, 512, "widest", "box"),
]


@pytest.mark.parametrize("weights", [False, True])
@pytest.mark.parametrize("N,Ng,kap,where", CASES)
def test_deposit_compressed(ctx, oracle, N, Ng, kap, where, weights):
    u = positions(N + Ng, N, where)
    k = widths(kap, Ng, N) if isinstance(kap, str) else None
    w = (0.5 + I.uniforms(7, 9, N)).astype(np.float32) if weights else None
    kw = dict(kappa=to_dev(k)) if k is not None else dict(kappa_uniform=kap)
    if w is not None:
        kw["weight"] = to_dev(w)
    ud = to_dev_u(u)
    rho = ctx.deposit(ud, Ng, L, **kw).cpu().numpy()
    okw = dict(kappa=k.astype(np.float64)) if k is not None else dict(kappa_u=kap)
    if w is not None:
        okw["w"] = w.astype(np.float64)
    assert rel_l2(rho, oracle.deposit(I.from_fixed(u, L), Ng, L, **okw)) <= TOL
    try:
        ctx.set_truncation(25.0)
        direct = ctx.deposit(ud, Ng, L, **kw).cpu().numpy()
    finally:
        ctx.set_truncation(0.0)
    assert rel_l2(rho, direct) <= 2 * TOL


@pytest.mark.parametrize("N,Ng,kap,where", CASES + [(20000, 4096, 2e5, "box"), (1, 64, 30.0, "box"),
                                                    (1025, 300, "extreme", "spike")])
def test_gather_from_tables(ctx, oracle, N, Ng, kap, where):
    u = positions(N + Ng, N, where)
    k = None
    if kap == "extreme":  # every band, the widths below 1/2 and those beyond the bands
        k = np.exp(np.linspace(math.log(1e-6), math.log(1e6), N)).astype(np.float32)
        k[-1] = 1e6
    elif isinstance(kap, str):
        k = widths(kap, Ng, N)
    g = 2 * math.pi * np.arange(Ng) / Ng
    f = (np.sin(g) + 0.3 * np.cos(3 * g) + 0.2 * (I.uniforms(5, 3, Ng) - 0.5)).astype(np.float32)
    kw = dict(kappa=to_dev(k)) if k is not None else dict(kappa_uniform=kap)
    ud, fd = to_dev_u(u), to_dev(f)
    out = ctx.gather(ud, fd, L, **kw).cpu().numpy()
    okw = dict(kappa=k.astype(np.float64)) if k is not None else dict(kappa_u=kap)
    assert rel_l2(out, oracle.gather(I.from_fixed(u, L), f.astype(np.float64), L, **okw)) <= TOL
    try:
        ctx.set_truncation(25.0)
        direct = ctx.gather(ud, fd, L, **kw).cpu().numpy()
    finally:
        ctx.set_truncation(0.0)
    # the direct sweep's half-angle form has its own error, about sqrt(8 kappa x) 6e-8 e^-x per value
    kmax = float(k.max()) if k is not None else kap
    assert rel_l2(out, direct) <= 2 * TOL + 6e-8 * math.sqrt(kmax)


@pytest.mark.parametrize("N,Ng,kap", [(20000, 256, "one"), (70001, 256, "narrow"), (130, 256, "narrow"),
                                      (70001, 1000, "ten"), (20000, 300, "wide"), (70001, 33, 2.0), (70001, 512, 300.0),
                                      (40000, 1024, 40.0), (33, 64, 5.0), (3000, 4096, 3.0), (300, 2, 4.0)])
def test_pic_step_through_proxies(ctx, kp, oracle, N, Ng, kap):
    # deposit and gather + push of two steps, every form of their tiles
    dt = 0.1
    u, v = I.landau_load(N + Ng, N, L, 0.05, 1.0)
    v32 = v.astype(np.float32)
    k = widths(kap, Ng, N) if isinstance(kap, str) else None
    import torch
    st = kp.PicState(to_dev_u(u), to_dev(v32), L, Ng, dt, kappa=None if k is None else to_dev(k),
                     kappa_uniform=0.0 if k is not None else kap, max_steps=2,
                     ids=torch.arange(N, dtype=torch.int32, device="cuda:0"))
    ctx.pic_step(st, 2)
    ctx.sync()
    r = oracle.pic_run(I.from_fixed(u, L), v32, L, Ng, dt, 2, kappa=None if k is None else k.astype(np.float64),
                       kappa_u=0.0 if k is not None else kap)
    e = st.energy.cpu().numpy()[:2]
    np.testing.assert_allclose(e, r["energy"], rtol=1e-5, atol=1e-12 * max(1.0, float(np.max(r["energy"]))))
    at = np.argsort(st.id.cpu().numpy())
    x = I.from_fixed(st.u.cpu().numpy().view(np.uint32), L)[at]
    assert np.max(np.abs((x - r["x"] + L / 2) % L - L / 2)) <= 1e-6 * L
    assert rel_l2(st.v.cpu().numpy()[at], r["v"]) <= 1e-5


@pytest.mark.parametrize("N,Ng,kap", [(1, 64, 30.0), (15, 33, 5.0), (17, 100, 200.0), (33, 1, 2.0), (700, 2, 40.0),
                                      (5000, 300, "ten"), (3000, 1030, "wide"), (1300, 4096, 3.0), (90000, 64, 100.0),
                                      (2000, 129, "extreme")])
def test_fp64_deposit_and_gather(ctx, oracle, N, Ng, kap):
    # tolerance: a few FP64 roundings a value (the exponential within 2e-16, exponents up to
    # 2 kappa sin^2 log2 e with kappa to 1e6 known to 1e-16 of 1e6: 1e-10 there, else 1e-12)
    import torch
    u = positions(N + Ng, N, "box")
    k = None
    if kap == "extreme":
        k = np.exp(np.linspace(math.log(1e-6), math.log(1e6), N))
        k[-1] = 1e6
    elif isinstance(kap, str):
        k = widths(kap, Ng, N).astype(np.float64)
    tol = 1e-10 if kap == "extreme" else 1e-12
    x, ud = I.from_fixed(u, L), to_dev_u(u)
    w = 0.5 + I.uniforms(7, 9, N)
    kw = dict(kappa=to_dev(k, torch.float64)) if k is not None else dict(kappa_uniform=kap)
    okw = dict(kappa=k) if k is not None else dict(kappa_u=kap)
    rho = ctx.deposit(ud, Ng, L, weight=to_dev(w, torch.float64), dtype=torch.float64, **kw).cpu().numpy()
    assert rel_l2(rho, oracle.deposit(x, Ng, L, w=w, **okw)) <= tol
    f = np.cos(2 * math.pi * np.arange(Ng) / Ng) + 0.3 * I.uniforms(5, 3, Ng)
    out = ctx.gather(ud, to_dev(f, torch.float64), L, **kw).cpu().numpy()
    assert rel_l2(out, oracle.gather(x, f, L, **okw)) <= tol


@pytest.mark.parametrize("kind", ["top", "edges", "extreme"])
def test_gather_tables_at_the_band_edges(ctx, oracle, kind):
    # enough pairs for the tables (range, bands, evaluation: three launches), widths at the ends of
    # the half-octave bands, in the band below 1/2 and beyond the last one.  Tolerance: TOL, per
    # width group, since a wrong band is a wrong kernel for that group alone
    N, Ng = 16500, 4096
    if kind == "top":
        ks = np.array([65535.0, 65535.93, 65535.95, 65535.96, 65535.996, 65536.0, 65536.01, 65537.0], np.float32)
    elif kind == "edges":
        e = 0.5 * 2.0 ** (0.5 * np.arange(0, 35))
        ks = np.concatenate([e * (1 - 2e-7), e, e * (1 + 2e-7)]).astype(np.float32)
    else:
        ks = np.exp(np.linspace(math.log(1e-6), math.log(1e6), 97)).astype(np.float32)
    k = ks[np.arange(N) % ks.size]
    u = positions(77, N, "box")
    g = 2 * math.pi * np.arange(Ng) / Ng
    f = (1 + np.sin(g) + 0.3 * np.cos(3 * g) + 0.2 * (I.uniforms(5, 3, Ng) - 0.5)).astype(np.float32)
    ctx.profile_enable(True)
    out = ctx.gather(to_dev_u(u), to_dev(f), L, kappa=to_dev(k)).cpu().numpy()
    launches = ctx.profile_read("all")[1]
    ctx.profile_enable(False)
    ref = oracle.gather(I.from_fixed(u, L), f.astype(np.float64), L, kappa=k.astype(np.float64))
    for i, kv in enumerate(ks):
        at = np.arange(i, N, ks.size)
        assert rel_l2(out[at], ref[at]) <= TOL, kv
    assert launches == 3


@pytest.mark.parametrize("lo", [2047.9998])
def test_deposit_of_nearly_equal_widths(ctx, lo):
    # widths of two neighbouring floats: a CTA's range of widths is one rounding long, and a value
    # from elsewhere mapped into it would be 1e7 half-lengths away.  Against one width for all:
    # both deposits are within TOL of the exact one, whose own difference is below 1e-7
    N, Ng = 1000003, 4096
    u = positions(31, N, "box")
    k = np.full(N, lo, np.float32)
    k[::3] = np.nextafter(np.float32(lo), np.float32(1e6))
    ud = to_dev_u(u)
    rho = ctx.deposit(ud, Ng, L, kappa=to_dev(k)).cpu().numpy()
    one = ctx.deposit(ud, Ng, L, kappa_uniform=float(k[0])).cpu().numpy()
    ctx.sync()
    assert np.all(np.isfinite(rho)) and rel_l2(rho, one) <= 2 * TOL


@pytest.mark.parametrize("lo,ulps", [(1e-39, 1), (1e-30, 1), (14.0, 1), (14.0, 3), (300.0, 1), (300.0, 2)])
def test_deposit_of_widths_a_few_roundings_apart(ctx, lo, ulps):
    # the middle of such a range is rounded by a large part of its length.  Against one width for
    # all, both within TOL of the exact density, whose own difference is below 4e-7
    N, Ng = 1000003, 4096
    u = positions(31, N, "box")
    k = np.full(N, lo, np.float32)
    hi = k[:1].copy()
    for _ in range(ulps):
        hi = np.nextafter(hi, np.float32(1e6))
    k[::3] = hi
    ud = to_dev_u(u)
    rho = ctx.deposit(ud, Ng, L, kappa=to_dev(k)).cpu().numpy()
    one = ctx.deposit(ud, Ng, L, kappa_uniform=float(k[0])).cpu().numpy()
    ctx.sync()
    assert rel_l2(rho, one) <= 2 * TOL


@pytest.mark.parametrize("N,kap", [(60000000, 14.0), (60000000, "narrow"), (30000000, "wide"), (1 << 24, "outliers")])
def test_deposit_mass_of_large_samples(ctx, N, kap):
    # one weight for all: the zeroth moment adds the same number N / (CTAs x threads) times, and
    # its rounding would be one factor on the whole density.  The grid's mean is exactly 1 (the
    # kernels' modes beyond the grid are below 1e-17); TOL covers norms (5e-7) and interpolation
    import torch
    Ng = 1024 if kap == "wide" else 256
    g = torch.Generator(device="cuda:0")
    g.manual_seed(3)
    u = torch.randint(-(1 << 31), 1 << 31, (N,), generator=g, device="cuda:0", dtype=torch.int64).to(torch.int32)
    if kap == "outliers":  # one width but for a few
        k = torch.full((N,), 40.0, device="cuda:0")
        k[::1000] = 400.0
        kw = dict(kappa=k)
    elif isinstance(kap, str):
        lo, hi = {"narrow": (13.0, 16.0), "wide": (5.0, 2e3)}[kap]
        kw = dict(kappa=lo * torch.exp(math.log(hi / lo) * torch.rand(N, generator=g, device="cuda:0")))
    else:
        kw = dict(kappa_uniform=kap)
    rho = ctx.deposit(u, Ng, L, **kw)
    ctx.sync()
    assert abs(float(rho.double().mean()) - 1) <= TOL


@pytest.mark.parametrize("N,low", [(33023, False), (33001, True), (33025, False)])
def test_width_range_of_a_partial_warp(ctx, kp, oracle, N, low):
    # the widths that end the range belong to the last warp of the pass over the state, which has
    # lanes without a particle: the range holds them.  They sit on one spot, so that a range without
    # them (one width for all, then) would change the field by 1e-4
    import torch
    Ng, dt, n = 512, 0.1, N % 32
    u, v = I.landau_load(N, N, L, 0.05, 1.0)
    u[-n:] = np.uint32(0x52345678)
    k = np.full(N, 16.4 if low else 13.0, np.float32)
    k[-n:] = 13.0 if low else 16.4
    st = kp.PicState(to_dev_u(u), to_dev(v.astype(np.float32)), L, Ng, dt, kappa=to_dev(k), max_steps=1,
                     ids=torch.arange(N, dtype=torch.int32, device="cuda:0"))
    ctx.pic_step(st, 1)
    ctx.sync()
    r = oracle.pic_run(I.from_fixed(u, L), v.astype(np.float32), L, Ng, dt, 1, kappa=k.astype(np.float64))
    np.testing.assert_allclose(st.energy.cpu().numpy()[:1], r["energy"], rtol=1e-5)
    assert rel_l2(st.v.cpu().numpy()[np.argsort(st.id.cpu().numpy())], r["v"]) <= 1e-5


# Scheduled widths of 2^16 particles and more, whose gather takes its tiles' interpolants: Silverman widths of
# one candidate, so that the widths' law is the oracle's.  The tiles have P <= 6 ("six") or P = 7, 8
# ("eight"); the widths of the box vary by a few per cent or, with half the density modulated, by a
# factor of three, and then over a tile by a few per cent; widths of a noisy pilot (alpha = 2) vary
# by much in every tile, which then sweeps its nodes
@pytest.mark.parametrize("N,Ng,amp,kstar,alpha", [
    (131072, 256, 0.05, 14.0, 0.5), (70001, 256, 0.05, 14.0, 0.5), (131072, 256, 0.5, 14.0, 0.5),
    (70001, 256, 0.5, 14.0, 0.5), (131077, 1000, 0.5, 40.0, 0.5), (70001, 1024, 0.5, 14.0, 0.5),
    (70001, 256, 0.5, 3000.0, 2.0), (65537, 4096, 0.5, 300.0, 2.0)],
    ids=["narrow six", "narrow eight", "tile six", "tile eight", "tile, odd grid", "tile eight, fine grid", "noisy",
         "noisy, fine grid"])
def test_scheduled_step_against_oracle(ctx, kp, oracle, N, Ng, amp, kstar, alpha):
    # particles at rest: the velocity after a step is half a kick, the field at the particle.
    # Tolerance: deposit and gather within TOL of the density's norm and the field's; the density's
    # modulated part, whose field this is, is a 28th (5%) or a third (50%) of that norm, and noise
    # of the kernels' widths adds about as much as the modulation at alpha = 2
    import torch
    dt = 1.0
    u, _ = I.landau_load(N + Ng, N, L, amp, 1.0)
    v = np.zeros(N, np.float32)
    cand = np.array([kstar])
    kw = dict(width_every=10, alpha=alpha, kappa_min=1.0, kappa_max=1e5)
    st = kp.PicState(to_dev_u(u), to_dev(v), L, Ng, dt, kappa=torch.ones(N, device="cuda:0"), cand=cand, max_steps=1,
                     ids=torch.arange(N, dtype=torch.int32, device="cuda:0"), **kw)
    ctx.pic_step(st, 1)
    ctx.sync()
    r = oracle.pic_run(I.from_fixed(u, L), v, L, Ng, dt, 1, kappa=np.ones(N), cands=cand, width_every=10, alpha=alpha,
                       kmin=1.0, kmax=1e5)
    at = np.argsort(st.id.cpu().numpy())
    k = st.kappa.double().cpu().numpy()[at]
    print("widths from %g to %g" % (k.min(), k.max()))
    tol = TOL * (28 if amp < 0.1 else 3)
    assert rel_l2(k, r["kappa"]) <= 4 * TOL
    np.testing.assert_allclose(st.energy.cpu().numpy()[:1], r["energy"], rtol=2 * tol)
    vg = st.v.double().cpu().numpy()[at]
    assert rel_l2(vg, r["v"]) <= tol
    assert np.max(np.abs(vg - r["v"])) <= 3 * tol * np.max(np.abs(r["v"]))


@pytest.mark.parametrize("weights", [False, True])
@pytest.mark.parametrize("kap", [0.3, 3.0, 14.0, 60.0, 300.0, 800.0, "one", "narrow", "hundred", "ten"])
def test_deposit_of_every_compressed_form(ctx, oracle, kap, weights):
    # more pairs than the unsorted sweep takes, and particles enough for the compressed forms to
    # pay: one width with P <= 8 (up to 60) and <= 16, narrow ranges with P <= 6 and P = 7, 8
    # ("hundred"), and the matrix product ("ten")
    N, Ng = 500009, 256
    u = positions(N, N, "box")
    k = None
    if kap == "hundred":
        k = I.log_uniform(Ng, I.STREAM_KAPPA, N, 100.0, 115.0).astype(np.float32)
    elif isinstance(kap, str):
        k = widths(kap, Ng, N)
    w = (0.5 + I.uniforms(7, 9, N)).astype(np.float32) if weights else None
    kw = dict(kappa=to_dev(k)) if k is not None else dict(kappa_uniform=kap)
    okw = dict(kappa=k.astype(np.float64)) if k is not None else dict(kappa_u=kap)
    rho = ctx.deposit(to_dev_u(u), Ng, L, weight=None if w is None else to_dev(w), **kw).cpu().numpy()
    ctx.sync()
    assert rel_l2(rho, oracle.deposit(I.from_fixed(u, L), Ng, L, w=None if w is None else w.astype(np.float64), **okw)) <= TOL


@pytest.mark.parametrize("N,Ng,lo,hi", [(60001, 100, 0.1, 1e5), (80001, 64, 5.0, 5e3), (160003, 65, 2.0, 2e4), (320001, 17, 0.5, 3e3),
                                        (70001, 700, 1e4, 6e4), (70001, 1001, 100.0, 2e4), (200003, 256, 300.0, 5e3)])
def test_gather_sweeps_and_short_intervals(ctx, oracle, N, Ng, lo, hi):
    # calls swept in rounds of four particles a warp (one to eight rounds, with particles past the
    # end in the last), and tables whose bands' windows are at most 32 nodes, some or all of them
    u = positions(N, N, "spike")
    k = I.log_uniform(N, I.STREAM_KAPPA, N, lo, hi).astype(np.float32)
    g = 2 * math.pi * np.arange(Ng) / Ng
    f = (np.sin(g) + 0.3 * np.cos(3 * g) + 0.2 * (I.uniforms(5, 3, Ng) - 0.5)).astype(np.float32)
    out = ctx.gather(to_dev_u(u), to_dev(f), L, kappa=to_dev(k)).cpu().numpy()
    ctx.sync()
    ref = oracle.gather(I.from_fixed(u, L), f.astype(np.float64), L, kappa=k.astype(np.float64))
    assert rel_l2(out, ref) <= TOL
    assert np.max(np.abs(out - ref)) <= 1e-5 * np.max(np.abs(ref))
