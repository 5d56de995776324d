"""Scans whose detector reaches far beyond the grid along z: the rays outside
cost the gather next to nothing, so the default forward stays with it, bit
for bit; with enough rows inside it takes the column form."""
import numpy as np
import pytest

import oracle
import synth
from synth.geometry import VolumeGeometry

from . import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL32 = 1e-5


@pytest.fixture(scope="module")
def gjp():
    from paper_1609_00958_gb300 import build
    build.build()
    import paper_1609_00958_gb300 as m
    return m


@pytest.mark.parametrize("nv,pitch,shift,columns", [
    (128, 1.0, 0.0, True), (128, 1.0, 20.0, True), (128, 1.0, -20.0, True), (156, 1.0, 0.0, True), (256, 1.0, 0.0, False),
    (128, 1.0, 100.0, False), (128, 1.0, -100.0, False), (384, 0.5, 200.0, False), (128, 3.0, 0.0, False)])
@pytest.mark.parametrize("sign", [1, -1])
def test_rows_beyond_the_grid(gjp, nv, pitch, shift, columns, sign):
    vg = VolumeGeometry.centred((190, 180, 128))
    cg = synth.circular(20, 110, nv, 800.0, 1600.0, 2.3, pitch_v=2.0 * pitch, angles=0.1 + 0.31 * np.arange(20), det_shift_v=shift)
    if sign < 0:
        cg.det_origin, cg.det_v = cg.det_origin + (nv - 1) * cg.det_v, -cg.det_v
    vol = synth.random_field(vg.n, seed=3)
    v = torch.from_numpy(vol).cuda()
    g = gjp.Geometry.from_cone(cg)
    out = gjp.forward(v, g, vg.h)
    assert torch.equal(out, gjp.forward(v, g, vg.h, path="gather")) == (not columns)
    gjp.stream_status()
    rays = parity.sampled_rays(cg, 4000, seed=1)
    ref = oracle.rays(vol, vg, cg, *rays)
    got = out.cpu().numpy().astype(np.float64)[rays[0], rays[2], rays[1]]
    parity.check_rays(got, vol, vg, cg, *rays, np.abs(ref).max(), TOL32, ref=ref)


@pytest.mark.parametrize("offset", [1e8, -1e8])
def test_rows_far_beyond_the_grid(gjp, offset):
    """A source and detector 1e8 voxels up or down, rows a fiftieth of a voxel apart: nothing is projected."""
    vg = VolumeGeometry.centred((190, 180, 128))
    cg = synth.circular(20, 110, 256, 800.0, 1600.0, 2.3, pitch_v=0.04, angles=0.1 + 0.31 * np.arange(20))
    cg.src[:, 2] += offset
    cg.det_origin[:, 2] += offset
    v = torch.ones(vg.n, device="cuda")
    g = gjp.Geometry.from_cone(cg)
    out = gjp.forward(v, g, vg.h)
    assert torch.equal(out, gjp.forward(v, g, vg.h, path="gather"))
    assert float(out.abs().max()) == 0.0
