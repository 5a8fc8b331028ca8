"""Kernels chosen by size, at the sizes where they change shape, against the oracle.

* the residual's penalty with a velocity per surface point (a warp per host element): elements
  hosting fewer than 8, a few and several hundred points, slots and atomics.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.oracle import OracleMesh
from paper_2009_00706_gb300 import _lib, api
from paper_2009_00706_gb300 import inputs as I

C = (0.5, 0.5, 0.5)


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    _lib.build()
    return torch.device("cuda:0")


def T(a, dev):
    return torch.from_numpy(np.ascontiguousarray(a)).to(dev)


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def pair(tri, level, radius=0.2, lmax=2):
    reg = [I.Region(I.REGION_SPHERE_BAND, level, (*C, radius, 0.05))]
    args = ((0.0, 0.0, 0.0), (1.0, 1.0, 1.0), 3, reg, tri, lmax)
    return api.Mesh(*args), OracleMesh(*args)


# float64 sums of at most a few hundred terms of one sign: well below 1e-12 of the result
TOL64 = 1e-12


@pytest.mark.parametrize("triangles,level", [(0, 5), (2, 4), (4, 4)])
@pytest.mark.parametrize("deterministic", [True, False])
def test_penalty_with_point_velocities(dev, triangles, level, deterministic):
    g, o = pair(I.icosphere(triangles, 0.2, C, 1e-3, 3), level)
    g.deterministic(deterministic)
    sq = g.surface_points()
    per = np.unique(sq[:, 8], return_counts=True)[1]
    assert {0: per.min() < 8, 2: per.max() > 8, 4: per.max() > 64}[triangles]
    vel = 0.3 * np.sin(7.0 * sq[:, :3] + np.array([0.0, 1.0, 2.0]))
    ph = I.Physics(mu=0.5, dt=1.0, scheme=I.SCHEME_CN, g=(0.1, -0.2, 0.05))   # the penalty dominates
    u, up, _ = I.state(g.n_nodes, 9)
    o.set_surface_velocity(0.3 * np.sin(7.0 * o.surface_points()[:, :3] + np.array([0.0, 1.0, 2.0])))
    try:
        want = o.residual_jvp(ph, u, up, v=up)[0]
    finally:
        o.set_surface_velocity(None)
    got = g.residual(ph, T(u, dev), T(up, dev), g_points=T(vel, dev)).cpu().numpy()
    assert rel(got, want) <= TOL64
