"""The warp-combined adjoint on detectors tilted against the rotation axis:
a warp's rays follow one another along z without sharing a row, so a ray's
upper taps join its neighbour's lower ones only where both lie on one row.
Against the FP64 oracle's transpose, under every option the adjoint takes."""
import math

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


def _tilt(cg, degrees, lean=0.0):
    """The scan with its detector turned in its plane and leaned towards the source about its centre."""
    t, b = math.radians(degrees), math.radians(lean)
    cu, cv = 0.5 * (cg.nu - 1), 0.5 * (cg.nv - 1)
    centre = cg.det_origin + cu * cg.det_u + cv * cg.det_v
    pu = np.linalg.norm(cg.det_u, axis=1, keepdims=True)
    pv = np.linalg.norm(cg.det_v, axis=1, keepdims=True)
    eu, ev = cg.det_u / pu, cg.det_v / pv
    nrm = np.cross(eu, ev)
    eu, ev = math.cos(t) * eu + math.sin(t) * ev, -math.sin(t) * eu + math.cos(t) * ev
    ev = math.cos(b) * ev + math.sin(b) * nrm
    cg.det_u, cg.det_v = eu * pu, ev * pv
    cg.det_origin = centre - cu * cg.det_u - cv * cg.det_v
    return cg


def _scan(case):
    angles = [0.13, 0.7, 1.6, 2.9, 4.0, 5.3]
    if case == "slight":
        vg = VolumeGeometry.centred((41, 38, 45))
        return vg, _tilt(synth.circular(6, 43, 64, 140.0, 280.0, 1.9, angles=angles), 0.6, 0.3)
    if case == "ragged_off_centre":                    # a part-empty last warp, anisotropic voxels, an origin
        vg = VolumeGeometry((37, 42, 50), (0.9, 1.1, 1.2), (-14.0, -25.0, -31.0))
        return vg, _tilt(synth.circular(6, 39, 77, 150.0, 300.0, 2.0, angles=angles, det_shift_v=3.2), 1.5)
    if case == "rows_along_minus_z":
        vg = VolumeGeometry.centred((40, 36, 40))
        cg = synth.circular(6, 41, 64, 140.0, 280.0, 1.8, angles=angles)
        cg.det_origin = cg.det_origin + (cg.nv - 1) * cg.det_v
        cg.det_v = -cg.det_v
        return vg, _tilt(cg, -0.9, 0.5)
    if case == "dense_rows":                           # two and three rays per voxel: tap by tap
        vg = VolumeGeometry.centred((30, 30, 24))
        return vg, _tilt(synth.circular(6, 33, 96, 90.0, 180.0, 1.4, pitch_v=0.5, angles=angles), 1.0)
    if case == "rows_just_apart":                      # ray distances around a half and 1.6 voxels
        vg = VolumeGeometry.centred((30, 34, 60))
        return vg, _tilt(synth.circular(6, 31, 64, 120.0, 240.0, 2.0, pitch_v=2.9, angles=angles), 0.8)
    if case == "strong":                               # rows cross several voxels within a warp
        vg = VolumeGeometry.centred((36, 36, 36))
        return vg, _tilt(synth.circular(6, 45, 64, 130.0, 260.0, 1.8, angles=angles), 20.0, 4.0)
    if case == "thin":                                 # z lines of 3 voxels
        vg = VolumeGeometry.centred((36, 36, 3))
        return vg, _tilt(synth.circular(6, 45, 64, 130.0, 260.0, 1.8, angles=angles), 0.7)
    raise KeyError(case)


CASES = ["slight", "ragged_off_centre", "rows_along_minus_z", "dense_rows", "rows_just_apart", "strong", "thin"]


@pytest.mark.parametrize("weight", ["lin", "spl"])
@pytest.mark.parametrize("case", CASES)
def test_tilted_adjoint_matches_oracle(gjp, case, weight):
    vg, cg = _scan(case)
    y = np.random.default_rng(6).standard_normal((cg.n_views, cg.nv, cg.nu)).astype(np.float32)
    y[:, 10:14, 5:9] = 0.0                             # rays that add nothing themselves
    g = gjp.Geometry.from_cone(cg, weight=weight)
    back = gjp.adjoint(torch.from_numpy(y).cuda(), g, vg.n, vg.h, vg.origin)
    gjp.stream_status()
    ref = oracle.adjoint(y.astype(np.float64), vg, cg, wfun=1 if weight == "spl" else 0)
    assert np.abs(back.cpu().numpy() - ref).max() <= TOL32 * np.abs(ref).max()


def test_tilted_adjoint_field_of_view(gjp):
    """Clipped rays drop the same planes as in the tap-by-tap scatter."""
    vg, cg = _scan("slight")
    g = gjp.Geometry.from_cone(cg)
    g.set_fov(15.4)
    y = torch.from_numpy(np.random.default_rng(8).standard_normal((cg.n_views, cg.nv, cg.nu)).astype(np.float32)).cuda()
    ref = gjp.adjoint(y, g, vg.n, vg.h, vg.origin, path="gather")
    back = gjp.adjoint(y, g, vg.n, vg.h, vg.origin)
    gjp.stream_status()
    assert (back - ref).abs().max().item() <= TOL32 * ref.abs().max().item()


@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_tilted_adjoint_non_finite_values(gjp, value):
    vg, cg = _scan("slight")
    y = np.random.default_rng(9).standard_normal((cg.n_views, cg.nv, cg.nu)).astype(np.float32)
    y[2, 30, 17] = value
    g = gjp.Geometry.from_cone(cg)
    d = torch.from_numpy(y).cuda()
    ref = gjp.adjoint(d, g, vg.n, vg.h, vg.origin, path="gather")
    back = gjp.adjoint(d, g, vg.n, vg.h, vg.origin)
    gjp.stream_status()
    ok = torch.isfinite(ref)
    assert 0 < int((~ok).sum()) < ok.numel() // 10
    assert torch.equal(torch.isfinite(back), ok)
    assert (back[ok] - ref[ok]).abs().max().item() <= TOL32 * ref[ok].abs().max().item()
