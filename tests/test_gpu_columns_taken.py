"""Which default adjoints take the column form: every scan that
test_gpu_columns compares with the oracle does (but the one whose detector is
short against the z lines), so that those tests are of its kernel."""
import numpy as np
import pytest

import synth
from synth.geometry import VolumeGeometry

from . import test_gpu_columns
from .column_family import takes_columns

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gjp():
    from paper_1609_00958_gb300 import build
    build.build()
    import paper_1609_00958_gb300 as m
    return m


def _takes(gjp, vg, cg, weight="lin"):
    g = gjp.Geometry.from_cone(cg, weight=weight)
    return takes_columns(gjp, torch.zeros(g.proj_shape, device="cuda"), g, vg)


@pytest.mark.parametrize("weight", ["lin", "spl"])
@pytest.mark.parametrize("case", [c for c in test_gpu_columns.CASES if c != "short_detector"])
def test_the_compared_scans_take_columns(gjp, case, weight):
    assert _takes(gjp, *test_gpu_columns._scan(case), weight)


def test_scans_that_do_not(gjp):
    vg = VolumeGeometry.centred((128, 128, 128))
    full = lambda views, nv=140, **kw: synth.circular(views, 130, nv, 500.0, 1000.0, 2.0, angles=0.1 + 0.5 * np.arange(views), **kw)
    assert _takes(gjp, vg, full(12))
    assert not _takes(gjp, vg, full(7))                              # less than 2^24 view-voxels
    assert not _takes(gjp, vg, full(12, nv=30))                      # few rows
    assert not _takes(gjp, vg, full(12, nv=48, pitch_v=6.4))         # rows 3.2 voxels apart
    assert not _takes(gjp, *test_gpu_columns._scan("short_detector"))
    tilted = full(12)
    tilted.det_v = tilted.det_v + 1e-3 * tilted.det_u
    assert not _takes(gjp, vg, tilted)
    assert not _takes(gjp, VolumeGeometry.centred((192, 192, 64)), full(12))   # short z lines


@pytest.mark.parametrize("offset", [500.0, 1e8, -1e8])
def test_rows_beyond_the_grid(gjp, offset):
    """No row meets the grid: nothing is projected back, and no column form is built."""
    vg = VolumeGeometry.centred((128, 128, 128))
    cg = synth.circular(12, 130, 140, 500.0, 1000.0, 2.0, angles=0.1 + 0.5 * np.arange(12))
    cg.src[:, 2] += offset
    cg.det_origin[:, 2] += offset
    g = gjp.Geometry.from_cone(cg)
    y = torch.ones(g.proj_shape, device="cuda")
    assert float(gjp.adjoint(y, g, vg.n, vg.h).abs().max()) == 0.0
    assert not takes_columns(gjp, y, g, vg)
