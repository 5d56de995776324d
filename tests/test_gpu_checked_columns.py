"""The debug build (GJP_CHECK_TAPS=1) over the column forms: the volume reads
and shared-memory taps of the forward, and the line reads of the adjoint, are
range-checked.  No call may report one out of range, and the results match
the FP64 oracle."""
import numpy as np
import pytest

import oracle

from . import parity, test_gpu_columns, test_gpu_columns_short, test_gpu_forward_columns

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL32 = 1e-5


@pytest.fixture(scope="module")
def gjp():
    """The package with the checked library swapped in for this module."""
    from paper_1609_00958_gb300 import build, _capi
    path = build.build_checked()
    saved = _capi._lib
    _capi._lib = _capi.load(path)
    import paper_1609_00958_gb300 as pkg
    yield pkg
    import gc
    gc.collect()                   # geometries made here are released by the checked library
    _capi._lib = saved


def _status():
    from paper_1609_00958_gb300 import _capi
    return _capi.gjp_stream_status(torch.cuda.current_stream().cuda_stream) == _capi.GJP_OK


def _adjoint(gjp, vg, cg, weight):
    y = np.random.default_rng(17).standard_normal((cg.n_views, cg.nv, cg.nu)).astype(np.float32)
    back = gjp.adjoint(torch.from_numpy(y).cuda(), gjp.Geometry.from_cone(cg, weight=weight), vg.n, vg.h, vg.origin)
    assert _status()
    ref = oracle.adjoint(y.astype(np.float64), vg, cg, wfun=1 if weight == "spl" else 0)
    assert np.abs(back.cpu().numpy() - ref).max() <= TOL32 * np.abs(ref).max()


@pytest.mark.parametrize("case", ["nz133", "nz256", "pitch_0.33", "pitch_0.5", "pitch_2.5", "helix_off_centre"])
def test_checked_adjoint(gjp, case):
    _adjoint(gjp, *test_gpu_columns._scan(case), "spl" if case == "nz133" else "lin")


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("shift", [0.0, -65.0, 65.0])
def test_checked_adjoint_of_short_detectors(gjp, shift, sign):
    _adjoint(gjp, *test_gpu_columns_short._scan((108, 100, 512), 4, 60, 130, 4.0, 2.0, shift, sign), "lin")


@pytest.mark.parametrize("case", test_gpu_forward_columns.CASES)
def test_checked_forward(gjp, case):
    vg, cg = test_gpu_forward_columns._scan(case)
    vol = np.random.default_rng(18).random(vg.n, dtype=np.float32)
    out = gjp.forward(torch.from_numpy(vol).cuda(), gjp.Geometry.from_cone(cg), vg.h, vg.origin)
    assert _status()
    ref = oracle.forward(vol, vg, cg)
    views, ius, ivs = parity.all_rays(cg)
    got = out.cpu().numpy().astype(np.float64)
    parity.check_rays(got[views, ivs, ius], vol, vg, cg, views, ius, ivs, np.abs(ref).max(), TOL32, ref=ref[views, ivs, ius])
