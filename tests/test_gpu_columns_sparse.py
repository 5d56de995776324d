"""The column form of the adjoint on projections that are mostly zero (a
masked sinogram, a metal trace, missing views): rays of zeros cost little, as
in the scatter, and what is left out is nothing but zeros."""
import numpy as np
import pytest

import oracle
import synth
from synth.geometry import VolumeGeometry

from .column_family import takes_columns

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL32 = 1e-5


@pytest.fixture(scope="module")
def gjp():
    from paper_1609_00958_gb300 import build
    build.build()
    import paper_1609_00958_gb300 as m
    return m


def _mask(name, shape):
    views, nv, nu = shape
    keep = np.zeros(shape, dtype=bool)
    if name == "one_row":
        keep[:, nv // 3] = True
    elif name == "ends":                               # the lines' first and last rows
        keep[:, 0, ::3] = keep[:, -1, 1::3] = True
    elif name == "one_column":
        keep[:, :, nu // 2] = True
    elif name == "trace":
        keep[:, nv // 2 - 3:nv // 2 + 4, nu // 4:nu // 4 + 5] = True
    elif name == "missing_views":
        keep[::4] = True
    elif name == "scattered":
        keep[:] = np.random.default_rng(1).random(shape) < 0.003
    return keep


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("name", ["one_row", "ends", "one_column", "trace", "missing_views", "scattered", "none"])
def test_sparse_projections_match_oracle(gjp, name, sign):
    vg = VolumeGeometry.centred((92, 85, 250))
    cg = synth.circular(9, 70, 270, 300.0, 600.0, 2.1, angles=0.1 + 0.77 * np.arange(9))
    if sign < 0:
        cg.det_origin, cg.det_v = cg.det_origin + (cg.nv - 1) * cg.det_v, -cg.det_v
    y = np.random.default_rng(2).standard_normal((9, 270, 70)).astype(np.float32) * _mask(name, (9, 270, 70))
    g = gjp.Geometry.from_cone(cg)
    d = torch.from_numpy(y.astype(np.float32)).cuda()
    back = gjp.adjoint(d, g, vg.n, vg.h)
    gjp.stream_status()
    ref = oracle.adjoint(y.astype(np.float64), vg, cg)
    assert np.abs(back.cpu().numpy() - ref).max() <= TOL32 * np.abs(ref).max()
    assert takes_columns(gjp, d, g, vg)


def _ms(f):
    best = 1e9
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        for _ in range(3):
            f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / 3)
    return best


@pytest.mark.parametrize("name", ["none", "trace", "one_column"])
def test_sparse_projections_cost_little(gjp, name):
    """A quarter of what dense ones take, at most."""
    vg = VolumeGeometry.centred((256, 256, 256))
    cg = synth.cone_angle_geometry(256, 256, 90, 10.0, angles=0.01 + np.arange(90) * np.pi / 45)
    g = gjp.Geometry.from_cone(cg)
    y = torch.randn(g.proj_shape, device="cuda")
    sparse = y * torch.from_numpy(_mask(name, g.proj_shape)).cuda()
    out = torch.empty(vg.n, device="cuda")
    dense = _ms(lambda: gjp.adjoint(y, g, vg.n, vg.h, out=out))
    little = _ms(lambda: gjp.adjoint(sparse, g, vg.n, vg.h, out=out))
    assert little <= 0.25 * dense, (little, dense)
