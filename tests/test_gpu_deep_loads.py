"""The gather forward with deeper load batches, which launches of few views
and of grids beyond the L2 take: bit for bit the default kernel, which a
launch shape of 8 detector columns selects."""
import numpy as np
import pytest

import synth
from synth.geometry import VolumeGeometry

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gjp():
    from paper_1609_00958_gb300 import build
    build.build()
    import paper_1609_00958_gb300 as m
    return m


def _check(gjp, v, cg, h, path, weight):
    g = gjp.Geometry.from_cone(cg, weight=weight)
    got = gjp.forward(v, g, h, path=path)
    g.set_launch(8, 1)
    want = gjp.forward(v, g, h, path=path)
    gjp.stream_status()
    assert torch.equal(got, want)
    assert float(got.abs().max()) > 0


@pytest.mark.parametrize("weight", ["lin", "spl"])
@pytest.mark.parametrize("dt", ["float32", "bfloat16", "float16"])
@pytest.mark.parametrize("n", [(9, 7, 40), (45, 45, 45), (70, 66, 20), (130, 37, 64)])
def test_few_views(gjp, n, dt, weight):
    """Fewer planes than one load batch, several table windows, ragged
    detectors and lanes that leave the grid at different planes."""
    vg = VolumeGeometry.centred(n, h=(1.0, 1.1, 0.9))
    w = float(max(n[:2]))
    cg = synth.circular(5, 37, 64, 1.3 * w, 2.6 * w, 0.09 * w, angles=[0.03, 0.7, 1.5708, 2.3, 3.9], det_shift_v=0.3)
    v = torch.from_numpy(synth.random_field(n, seed=5)).cuda().to(getattr(torch, dt))
    _check(gjp, v, cg, vg.h, "gather", weight)


@pytest.mark.parametrize("weight", ["lin", "spl"])
@pytest.mark.parametrize("dt", ["bfloat16", "float16"])
def test_paired_copy_of_a_large_grid(gjp, dt, weight):
    """A z-paired copy beyond the L2, views too far apart to share it."""
    n = (420, 410, 400)
    cg = synth.cone_angle_geometry(420, 96, 3, 10.0, angles=[0.2, 1.7, 3.3])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    v = torch.rand(n, device="cuda", generator=gen).to(getattr(torch, dt))
    _check(gjp, v, cg, (1.0, 1.0, 1.0), "pairs", weight)


def test_large_float32_grid(gjp):
    """More than 16 views of a grid beyond the L2."""
    n = (480, 470, 460)
    cg = synth.cone_angle_geometry(480, 64, 18, 10.0, angles=np.radians(3.0 * np.arange(18)))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)
    _check(gjp, torch.rand(n, device="cuda", generator=gen), cg, (1.0, 1.0, 1.0), "gather", "lin")
