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
