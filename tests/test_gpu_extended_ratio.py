"""The K_e/I_e histogram and maximum where FP32 cannot decide them alone.

Bins and maximum are those of FP64 arithmetic; the kernel decides from an FP32
value where that is clear.  The states here make it unclear: ratios planted on
within 1e-9 to 1e-7 of bin edges (FP32 tells nothing there, FP64 everything),
ratios below the FP32 range, a maximum shared by nodes that differ in the
last bits, nodes at rest.  Counts equal the oracle's, and the maximum is
within one rounding (2^-52).
"""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,nbins,lo,hi", [(64, 9, 40, -8.0, 0.0), (33, 17, 7, -5.5, -1.25), (300, 12, 1024, -3.0, -1.0),
                                               (40, 7, 16, -70.0, 0.0), (257, 6, 1, -4.0, 0.0)])
@pytest.mark.parametrize("kind", ["edges", "tiny", "ties", "rest"])
def test_ratio_counts_equal_float64(nx, nz, nbins, lo, hi, kind):
    import paper_2411_10372_gb300 as cm
    cfg = O.Config(nx=nx, nz=nz, Ra=1e5)
    X = O.init(cfg)
    rng = np.random.default_rng(nx + nbins)
    b = cfg.gamma * cfg.eps * cfg.D
    shape = X[0].shape
    rho = X[0]
    z = np.linspace(0.0, 1.0, nz)[:, None]
    if kind == "edges":
        q = rng.integers(0, nbins + 1, shape)
        r = 10.0 ** (lo + q * (hi - lo) / nbins)
        r = r * (1.0 + rng.choice([-1.0, 1.0], shape) * 10.0 ** rng.uniform(-9.0, -7.0, shape))
    elif kind == "tiny":
        r = 10.0 ** rng.uniform(-200.0, -30.0, shape)
    elif kind == "ties":
        r = 1.3e-2 * (1.0 + rng.integers(-3, 4, shape) * 2.0 ** -51)
    else:
        r = np.where(rng.random(shape) < 0.5, 0.0, 10.0 ** rng.uniform(lo, hi, shape))
    T = np.ones(shape) - (cfg.eps + cfg.D) * z
    u = np.sqrt(2.0 * r * T / b)
    u[0] = u[-1] = 0.0
    X[1], X[2] = rho * u, 0.0
    X[3] = rho * (0.5 * u * u + T / b + z / cfg.eps)
    X = np.ascontiguousarray(X)
    s = cm.Solver(nx, nz, cfg.Ra, cfg.Pr, cfg.gamma, precision="fp64")
    s.set_state(X)
    ext, hist = s.extended(nbins, lo, hi)
    s.close()
    want, want_hist = O.extended(cfg, X, nbins, lo, hi)
    assert abs(ext["r_max"] - want["r_max"]) <= 2.0 ** -52 * want["r_max"]
    assert np.array_equal(hist, want_hist)
