"""The column form of the adjoint with the source far away (a nearly parallel
beam written as a cone): no ray of a column may be missed, whatever the
distance.  Against the FP64 oracle's transpose."""
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


@pytest.mark.parametrize("distance", [1e5, 1e7, 2e7, 5e7, 1e9])
def test_far_source(gjp, distance):
    vg = VolumeGeometry.centred((128, 120, 128))
    cg = synth.circular(10, 131, 133, distance, 2.0 * distance, 2.03, angles=0.4 + 0.61 * np.arange(10))
    y = np.random.default_rng(4).standard_normal((cg.n_views, cg.nv, cg.nu)).astype(np.float32)
    g = gjp.Geometry.from_cone(cg)
    d = torch.from_numpy(y).cuda()
    back = gjp.adjoint(d, g, vg.n, vg.h, vg.origin)
    gjp.stream_status()
    ref = oracle.adjoint(y.astype(np.float64), vg, cg)
    assert np.abs(back.cpu().numpy() - ref).max() <= TOL32 * np.abs(ref).max()
    assert takes_columns(gjp, d, g, vg)
