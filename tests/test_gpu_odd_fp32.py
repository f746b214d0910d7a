"""FP32 sweeps with two columns per lane on boxes of an odd number of columns.

The strips are 60 columns wide, and a lane at the periodic seam holds two
columns that are not neighbours in memory; the sizes sit around one, two and
three strips, and below one.  Each sweep against the oracle on the same
float32 state (2e-6 of the field, the bar of the even sizes), the time step
reduced in the last sweep against the oracle's rule on the stored state
(1e-6: float32 speeds), and shifts in x: every column goes through the same
operations wherever it sits in its lane, so a shifted state steps to the
shifted result bit for bit.
"""
import numpy as np
import pytest

import oracle as O
from test_gpu_3d import stirred_state_3d
from test_gpu_parity import rel_l2, stirred_state

pytestmark = pytest.mark.gpu


def _solver(cfg, **kw):
    import paper_2411_10372_gb300 as cm
    return cm.Solver(cfg.nx, cfg.nz, cfg.Ra, cfg.Pr, cfg.gamma, ny=cfg.ny, ndim=cfg.ndim, precision="fp32",
                     zstretch=cfg.zstretch, **kw)


def _rounded(X):
    return X.astype(np.float32).astype(np.float64)


def _check(got, want, tol):
    """rho and E by their relative L2, the momenta against the scale rho c (c = 3.65)."""
    for f in (0, -1):
        assert rel_l2(got[f], want[f]) <= tol, f
    for f in range(1, got.shape[0] - 1):
        assert np.linalg.norm(got[f] - want[f]) / (3.65 * np.linalg.norm(want[0])) <= tol, f


@pytest.mark.parametrize("zstretch", [0.0, 1.4])
@pytest.mark.parametrize("nx,nz", [(5, 5), (57, 9), (59, 40), (61, 12), (63, 23), (65, 31), (119, 6), (121, 70), (123, 17),
                                   (181, 33), (1001, 21)])
def test_2d(nx, nz, zstretch):
    cfg = O.Config(nx=nx, nz=nz, Ra=1e6, zstretch=zstretch)
    X = _rounded(stirred_state(cfg, seed=nx * 7 + nz))
    s = _solver(cfg)
    hmin = min(cfg.aspect / nx, float(np.min(np.diff(s.z))))
    for direction in (2, 0):
        s.set_state(X)
        s.sweep(direction, 0.05 * hmin)
        _check(s.state(), O.sweep(cfg, X, direction, 0.05 * hmin), 2e-6)
    s.set_state(X)
    s.step(1)
    Y = s.state()
    assert abs(s.dt() / O.dt(cfg, Y) - 1.0) <= 1e-6
    for shift in (1, nx // 2):
        s.set_state(np.roll(X, shift, axis=-1))
        s.step(1)
        assert np.array_equal(s.state(), np.roll(Y, shift, axis=-1)), shift
    s.close()


@pytest.mark.parametrize("zstretch", [0.0, 1.4])
@pytest.mark.parametrize("nx,ny,nz", [(5, 4, 5), (59, 9, 7), (61, 8, 12), (63, 17, 9), (121, 10, 14)])
def test_3d(nx, ny, nz, zstretch):
    cfg = O.Config(nx=nx, ny=ny, nz=nz, ndim=3, Ra=1e6, zstretch=zstretch)
    X = _rounded(stirred_state_3d(cfg, seed=nx + ny + nz))
    s = _solver(cfg)
    hmin = min(cfg.aspect / nx, cfg.aspect / ny, float(np.min(np.diff(s.z))))
    for direction in (2, 1, 0):
        s.set_state(X)
        s.sweep(direction, 0.05 * hmin)
        _check(s.state(), O.sweep(cfg, X, direction, 0.05 * hmin), 2e-6)
    s.set_state(X)
    s.step(1)
    Y = s.state()
    assert abs(s.dt() / O.dt(cfg, Y) - 1.0) <= 1e-6
    s.set_state(np.roll(X, 1, axis=-1))
    s.step(1)
    assert np.array_equal(s.state(), np.roll(Y, 1, axis=-1))
    s.close()
