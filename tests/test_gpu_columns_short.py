"""The column form of the adjoint where the detector covers a part of the z
lines only, so that a chunk of voxels meets the rows with its uppermost or
lowermost part: against the FP64 oracle's transpose."""
import math

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


def _scan(n, views, nu, nv, half, pitch, shift, sign):
    """Views at right angles from 0 on; rows `pitch` voxels apart on the axis, moved along z by `shift` rows."""
    a = math.radians(half)
    d = 0.5 * max(n[:2]) / math.sin(a)
    cg = synth.circular(views, nu, nv, d, 2.0 * d, 4.0 * d * math.tan(a) / nu, pitch_v=2.0 * pitch,
                        angles=0.5 * np.pi * np.arange(views), det_shift_v=shift)
    if sign < 0:
        cg.det_origin, cg.det_v = cg.det_origin + (nv - 1) * cg.det_v, -cg.det_v
    return VolumeGeometry.centred(n), cg


def _check(gjp, vg, cg):
    y = np.random.default_rng(21).standard_normal((cg.n_views, cg.nv, cg.nu)).astype(np.float32)
    g = gjp.Geometry.from_cone(cg)
    d = torch.from_numpy(y).cuda()
    back = gjp.adjoint(d, g, vg.n, vg.h, vg.origin)
    gjp.stream_status()
    ref = oracle.adjoint(y.astype(np.float64), vg, cg)
    assert np.abs(back.cpu().numpy() - ref).max() <= TOL32 * np.abs(ref).max()
    return d, g


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("shift", [0.0, -200.0, 230.0])
def test_few_rows(gjp, shift, sign):
    _check(gjp, *_scan((100, 100, 512), 4, 60, 32, 4.0, 1.0, shift, sign))


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("shift", [0.0, -65.0, 65.0])
def test_rows_of_half_the_height(gjp, shift, sign):
    vg, cg = _scan((108, 100, 512), 4, 60, 130, 4.0, 2.0, shift, sign)
    d, g = _check(gjp, vg, cg)
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


@pytest.mark.parametrize("nv,pitch", [(16, 1.0), (64, 1.0), (61, 0.5), (24, 2.0)])
def test_few_rows_cost_no_more_than_the_scatter(gjp, nv, pitch):
    vg, cg = _scan((256, 256, 256), 4, 256, nv, 8.0, pitch, 0.0, 1)
    cg = synth.ConeGeometry(*(np.tile(x, (23, 1)) for x in (cg.src, cg.det_origin, cg.det_u, cg.det_v)), cg.nu, cg.nv)
    g = gjp.Geometry.from_cone(cg)
    y = torch.randn(g.proj_shape, device="cuda")
    out = torch.empty(vg.n, device="cuda")
    t = [_ms(lambda: gjp.adjoint(y, g, vg.n, vg.h, out=out, path=p)) for p in ("auto", "combine")]
    assert t[0] <= 1.3 * t[1], t
