"""The column form of the adjoint (scans with detector rows along z, z lines
of about 100 voxels and more, 2^24 view-voxels) against the FP64 oracle's transpose: chunk
sizes and remainders along z, ragged strips and planes, ray pitches from a
quarter of a voxel to several, both row directions, every option that the
adjoint takes, non-finite values, and the calls that fall back to the
warp-combined scatter."""
import numpy as np
import pytest

import oracle
import synth
from synth.geometry import VolumeGeometry

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL32 = 1e-5


@pytest.fixture(scope="module")
def gjp():
    from paper_1609_00958_gb300 import build
    build.build()
    import paper_1609_00958_gb300 as m
    return m


def _scan(name):
    """(volume grid, scan) of one case."""
    if name.startswith("nz"):                          # 64, 128, 192 and 256 voxel chunks, with remainders
        nz = int(name[2:])
        vg = VolumeGeometry.centred((109, 122, nz))
        return vg, synth.circular(14, 61, nz + 9, 600.0, 1200.0, 2.1, angles=0.1 + 0.437 * np.arange(14))
    if name == "many_views":                           # several passes of 32 views, several view groups
        vg = VolumeGeometry.centred((42, 44, 128))
        return vg, synth.circular(75, 23, 40, 200.0, 400.0, 2.0, pitch_v=4.5)
    if name == "one_view":
        vg = VolumeGeometry.centred((361, 353, 132))
        return vg, synth.circular(1, 137, 131, 700.0, 1400.0, 2.0, angles=[0.4])
    if name in ("pitch_0.33", "pitch_0.5", "pitch_0.8", "pitch_2.5"):
        p = float(name[6:])
        vg = VolumeGeometry.centred((119, 122, 128))
        return vg, synth.circular(10, 59, int(140 / p), 600.0, 1200.0, 2.0, pitch_v=2.0 * p,
                                  angles=0.3 + 0.62 * np.arange(10))
    if name == "short_detector":                       # rays cover part of the z lines only
        vg = VolumeGeometry.centred((100, 97, 256))
        return vg, synth.circular(8, 61, 40, 300.0, 600.0, 2.0, angles=0.1 + 0.77 * np.arange(8), det_shift_v=20.0)
    if name == "rows_along_minus_z":
        vg = VolumeGeometry.centred((125, 122, 150))
        cg = synth.cone_angle_geometry(150, 70, 9, 12.0)
        cg.det_origin = cg.det_origin + (cg.nv - 1) * cg.det_v
        cg.det_v = -cg.det_v
        return vg, cg
    if name == "helix_off_centre":                     # anisotropic voxels, an origin, a source that moves along z
        vg = VolumeGeometry((127, 131, 141), (0.9, 1.1, 1.3), (-55.0, -74.0, -83.0))
        cg = synth.circular(9, 73, 150, 400.0, 810.0, 2.1, pitch_v=2.7, det_shift_u=2.3)
        dz = np.linspace(-30.0, 30.0, 9)
        cg.src[:, 2] += dz
        cg.det_origin[:, 2] += dz
        return vg, cg
    raise KeyError(name)


CASES = ["nz99", "nz128", "nz133", "nz192", "nz256", "nz300", "nz517", "many_views", "one_view", "pitch_0.33", "pitch_0.5",
         "pitch_0.8", "pitch_2.5", "short_detector", "rows_along_minus_z", "helix_off_centre"]


def _rows(cg, seed=3):
    return np.random.default_rng(seed).standard_normal((cg.n_views, cg.nv, cg.nu)).astype(np.float32)


def _check(back, ref):
    err = np.abs(back.double().cpu().numpy() - ref).max() / np.abs(ref).max()
    assert err <= TOL32, err


@pytest.mark.parametrize("weight", ["lin", "spl"])
@pytest.mark.parametrize("case", CASES)
def test_column_adjoint_matches_oracle(gjp, case, weight):
    vg, cg = _scan(case)
    y = _rows(cg)
    g = gjp.Geometry.from_cone(cg, weight=weight)
    back = gjp.adjoint(torch.from_numpy(y).cuda(), g, vg.n, vg.h, vg.origin)
    gjp.stream_status()
    _check(back, oracle.adjoint(y.astype(np.float64), vg, cg, wfun=1 if weight == "spl" else 0))


def test_column_adjoint_field_of_view(gjp):
    """Clipped rays: the same planes as the general scatter drops (which the
    parity tests pin against the oracle)."""
    vg, cg = _scan("helix_off_centre")
    g = gjp.Geometry.from_cone(cg)
    g.set_fov(52.3)
    y = torch.from_numpy(_rows(cg)).cuda()
    ref = gjp.adjoint(y, g, vg.n, vg.h, vg.origin, path="gather")
    back = gjp.adjoint(y, g, vg.n, vg.h, vg.origin)
    gjp.stream_status()
    _check(back, ref.double().cpu().numpy())


def test_column_adjoint_accumulates(gjp):
    vg, cg = _scan("nz133")
    y = _rows(cg)
    g = gjp.Geometry.from_cone(cg)
    out = torch.full(vg.n, 2.5, device="cuda")
    gjp.adjoint(torch.from_numpy(y).cuda(), g, vg.n, vg.h, vg.origin, out=out, accumulate=True)
    gjp.stream_status()
    _check(out, oracle.adjoint(y.astype(np.float64), vg, cg) + 2.5)


@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_column_adjoint_non_finite_values(gjp, value):
    """A non-finite pixel reaches the voxels of its own ray and no others."""
    vg, cg = _scan("nz128")
    y = _rows(cg)
    y[2, 70, 33] = value
    g = gjp.Geometry.from_cone(cg)
    d = torch.from_numpy(y).cuda()
    ref = gjp.adjoint(d, g, vg.n, vg.h, vg.origin, path="gather")
    back = gjp.adjoint(d, g, vg.n, vg.h, vg.origin)
    gjp.stream_status()
    ok = torch.isfinite(ref)
    assert 0 < int((~ok).sum()) < ok.numel() // 10
    assert torch.equal(torch.isfinite(back), ok)
    _check(back[ok], ref[ok].double().cpu().numpy())


def test_column_adjoint_without_workspace(gjp):
    """No room for the transposed projections, or a stream being captured:
    the warp-combined scatter does the work."""
    from paper_1609_00958_gb300 import _capi
    vg, cg = _scan("nz128")
    y = torch.from_numpy(_rows(cg)).cuda()
    ref = oracle.adjoint(y.double().cpu().numpy(), vg, cg)
    g = gjp.Geometry.from_cone(cg)
    out = gjp.adjoint(y, g, vg.n, vg.h, vg.origin)             # builds the tables
    try:
        assert _capi.gjp_debug_fail_allocations(1) == _capi.GJP_OK
        _check(gjp.adjoint(y, g, vg.n, vg.h, vg.origin), ref)
        gjp.Geometry.from_cone(cg)
        gjp.forward(torch.zeros(vg.n, device="cuda"), gjp.Geometry.from_cone(cg), vg.h, vg.origin)   # the failure is used up
    finally:
        _capi.gjp_debug_fail_allocations(0)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        gjp.adjoint(y, g, vg.n, vg.h, vg.origin, out=out)
    out.fill_(7.0)
    graph.replay()
    torch.cuda.synchronize()
    _check(out, ref)
