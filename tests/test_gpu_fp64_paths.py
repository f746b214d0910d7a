"""FP64 sweeps at the edges of their quotients: bit for bit the oracle's.

The FP64 kernels form quotients from a reciprocal and two multiply-adds while
the operands stay in a range where that rounds as a division, and divide
plainly out of it; comparisons work on the bits.
The states here hold what takes each of those branches: exact zeros (at rest,
uniform along a direction), values near the ends of the double range and
below it, and both signs of zero.  Every operation rounds as the oracle's
does, so the results are equal, not close.  Both forms of the sweeps take
them: the staged kernels, and the marching ones that need no scratch.
"""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


def _state(cfg, kind, seed):
    rng = np.random.default_rng(seed)
    X = O.init(cfg)
    m = X[1:-1]
    shape = m[0][1:-1].shape
    for f in range(m.shape[0]):
        v = rng.uniform(-0.3, 0.3, shape)
        if kind == "rest":
            v[:] = 0.0
        elif kind == "signed_zeros":
            v[rng.random(shape) < 0.5] = 0.0
            v[rng.random(shape) < 0.3] *= -0.0
        elif kind == "tiny":
            v *= 10.0 ** rng.uniform(-322.0, -100.0, shape)
        elif kind == "mixed":
            v *= 10.0 ** rng.uniform(-180.0, 0.0, shape)
            v[rng.random(shape) < 0.2] = 0.0
        elif kind == "x_uniform":
            v[...] = v[..., :1]
        m[f][1:-1] = v * X[0][1:-1]
    if kind == "x_uniform":
        X[0] = X[0][..., :1]
        X[-1] = X[-1][..., :1]
    X[-1][1:-1] += (0.5 * sum(q * q for q in m) / X[0])[1:-1]
    return np.ascontiguousarray(X)


@pytest.mark.parametrize("kind", ["rest", "signed_zeros", "tiny", "mixed", "x_uniform", "stirred"])
@pytest.mark.parametrize("shape", [(33, 1, 6), (5, 1, 37), (130, 1, 9), (29, 7, 5)])
@pytest.mark.parametrize("zstretch", [0.0, 1.3])
@pytest.mark.parametrize("form", ["staged", "march"])
def test_sweeps_equal_oracle(kind, shape, zstretch, form, monkeypatch):
    import paper_2411_10372_gb300 as cm
    if form == "march":
        monkeypatch.setenv("CM_F64_MARCH", "1")
    nx, ny, nz = shape
    nd = 3 if ny > 1 else 2
    cfg = O.Config(nx=nx, ny=ny, nz=nz, ndim=nd, Ra=3e5, zstretch=zstretch, pert_amp=1e-2, seed=3)
    X = _state(cfg, kind, nx + nz)
    s = cm.Solver(nx, nz, cfg.Ra, cfg.Pr, cfg.gamma, ny=ny, ndim=nd, precision="fp64", zstretch=zstretch)
    for direction in ((2, 0) if nd == 2 else (2, 1, 0)):
        s.set_state(X)
        s.sweep(direction, 1e-3)
        assert np.array_equal(s.state(), O.sweep(cfg, X, direction, 1e-3)), (kind, shape, direction)
    s.close()


@pytest.mark.parametrize("shape,zstretch", [((1025, 1, 1100), 0.0), ((1000, 1, 1061), 1.5), ((300, 260, 30), 1.2)])
def test_chunks_equal_march(shape, zstretch, monkeypatch):
    """Boxes larger than the scratch: several chunks of planes, the last one short, equal the marching kernels."""
    import paper_2411_10372_gb300 as cm
    nx, ny, nz = shape
    got = []
    for form in ("staged", "march"):
        if form == "march":
            monkeypatch.setenv("CM_F64_MARCH", "1")
        s = cm.Solver(nx, nz, 1e10, ny=ny, ndim=3 if ny > 1 else 2, precision="fp64", zstretch=zstretch, pert_amp=1e-2)
        s.step(2)
        got.append((s.state(), s.dt(), s.time()))
        s.close()
    assert np.array_equal(got[0][0], got[1][0]) and got[0][1:] == got[1][1:]
