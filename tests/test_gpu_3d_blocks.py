"""The packed FP32 3D sweeps where their blocks and their two-row loop end.

A block stores 10 rows of the direction across its warps (y for L_z and L_x, z
for L_y) between two halo warps, and marches two rows a trip.  Row counts sit
at and next to one and two blocks, with planes left over either way; segments
are of odd and even length and of one row more than a trip.  Each sweep against
the oracle on the same float32 state (2e-6, the bar of the other packed
sweeps).  Every row goes through the same operations whichever half of a trip,
segment or warp it falls on, so segment lengths and shifts along y leave the
result of a step as it is, bit for bit.
"""
import numpy as np
import pytest

import oracle as O
from test_gpu_3d import stirred_state_3d
from test_gpu_odd_fp32 import _check, _rounded, _solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("zstretch", [0.0, 1.4])
@pytest.mark.parametrize("nx,ny,nz", [(60, 4, 11), (62, 9, 10), (62, 10, 12), (63, 11, 13), (122, 20, 22), (121, 21, 21)])
def test_blocks_and_rows(nx, ny, nz, zstretch, monkeypatch):
    cfg = O.Config(nx=nx, ny=ny, nz=nz, ndim=3, Ra=1e6, zstretch=zstretch)
    X = _rounded(stirred_state_3d(cfg, seed=nx + ny + nz))
    s = _solver(cfg)
    hmin = min(cfg.aspect / nx, cfg.aspect / ny, float(np.min(np.diff(s.z))))
    for direction in (2, 1, 0):
        s.set_state(X)
        s.sweep(direction, 0.05 * hmin)
        _check(s.state(), O.sweep(cfg, X, direction, 0.05 * hmin), 2e-6)
    s.set_state(X)
    s.step(2)
    Y = s.state()
    for shift in (1, 4):
        s.set_state(np.roll(X, shift, axis=-2))
        s.step(2)
        assert np.array_equal(s.state(), np.roll(Y, shift, axis=-2)), shift
    s.close()
    for rows in ("4", "5", "7", "64"):
        monkeypatch.setenv("CM_SEG_ROWS", rows)
        s = _solver(cfg)
        s.set_state(X)
        s.step(2)
        assert np.array_equal(s.state(), Y), rows
        s.close()
