"""The column form of the adjoint is no further from 64-bit values than the
scatter that it stands in for: rms error on white noise, which shows every
weight's error by itself, over the row distances that it takes."""
import math

import numpy as np
import pytest

import oracle
import synth
from synth.geometry import VolumeGeometry

from .column_family import takes_columns

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gjp():
    from paper_1609_00958_gb300 import build
    build.build()
    import paper_1609_00958_gb300 as m
    return m


@pytest.mark.parametrize("weight", ["lin", "spl"])
@pytest.mark.parametrize("pitch", [0.45, 0.6, 0.8, 1.0, 1.4, 2.0, 2.5])
def test_error_against_64_bits(gjp, pitch, weight):
    vg = VolumeGeometry.centred((192, 190, 256))
    a = math.radians(6.0)
    d = 96.0 / math.sin(a)
    cg = synth.circular(2, 192, int(300 / pitch), d, 2.0 * d, 4.0 * d * math.tan(a) / 192, pitch_v=2.0 * pitch,
                        angles=[0.1, 0.8], det_shift_v=0.3)
    y = np.random.default_rng(12).standard_normal((2, cg.nv, cg.nu)).astype(np.float32)
    g = gjp.Geometry.from_cone(cg, weight=weight)
    dev = torch.from_numpy(y).cuda()
    ref = oracle.adjoint(y.astype(np.float64), vg, cg, wfun=1 if weight == "spl" else 0)
    err = [np.linalg.norm(gjp.adjoint(dev, g, vg.n, vg.h, path=p).double().cpu().numpy() - ref) / np.linalg.norm(ref)
           for p in ("auto", "combine")]
    assert err[0] <= 1.02 * err[1], err
    assert takes_columns(gjp, dev, g, vg)
