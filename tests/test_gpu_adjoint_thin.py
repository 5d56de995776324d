"""The adjoint of thin grids on a tilted detector whose rays spread strongly
along z: one row's end must not pass for the next row's start where a warp's
rays hand their taps on.  Against the FP64 oracle's transpose."""
import math

import numpy as np
import pytest

import oracle
from synth.geometry import ConeGeometry, VolumeGeometry

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL32 = 1e-5


@pytest.fixture(scope="module")
def gjp():
    from paper_1609_00958_gb300 import build
    build.build()
    import paper_1609_00958_gb300 as m
    return m


def _scan(nz, tilt, flip):
    """A source above the grid, a quarter of its length from one end: rays 1.5 voxels apart on the centre plane
    are 4 apart at the other end."""
    t = tilt
    eu = np.array([0.0, math.cos(t), -math.sin(t)]) * 3.0
    ev = np.array([0.0, math.sin(t), math.cos(t)]) * (-8.0 if flip else 8.0)
    nu, nv = 24, 32
    src, centre = np.array([-60.0, 0.0, 30.0]), np.array([240.0, 0.0, -30.0])
    org = centre - 0.5 * (nu - 1) * eu - 0.5 * (nv - 1) * ev
    return VolumeGeometry.centred((200, 60, nz)), ConeGeometry(src[None], org[None], eu[None], ev[None], nu, nv)


@pytest.mark.parametrize("flip", [False, True])
@pytest.mark.parametrize("tilt", [0.29, -0.29])
@pytest.mark.parametrize("nz", [4, 5, 6, 8])
def test_thin_grid(gjp, nz, tilt, flip):
    vg, cg = _scan(nz, tilt, flip)
    y = np.random.default_rng(5).standard_normal((1, cg.nv, cg.nu)).astype(np.float32)
    back = gjp.adjoint(torch.from_numpy(y).cuda(), gjp.Geometry.from_cone(cg), vg.n, vg.h, vg.origin)
    gjp.stream_status()
    ref = oracle.adjoint(y.astype(np.float64), vg, cg)
    assert np.abs(ref).max() > 0
    assert np.abs(back.cpu().numpy() - ref).max() <= TOL32 * np.abs(ref).max()
