"""The column form of the forward (scans with detector rows along z, z lines
of whole 16-byte words, more than 2^22 voxels, enough columns to fill the GPU) against the FP64
oracle: block shapes and remainders along z and the detector rows, both row
directions, every option, all entry points that take it, and volumes that it
leaves to the gather."""
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


def _orbit(views, nu, nv, d, pitch, **more):
    return synth.circular(views, nu, nv, d, 2.0 * d, pitch, angles=0.1 + 2.0 * np.pi * np.arange(views) / views, **more)


def _scan(case):
    if case == "one_warp":                 # 32 threads of 4 rays
        return VolumeGeometry.centred((190, 176, 128)), _orbit(48, 48, 128, 700.0, 2.2)
    if case == "ragged_lines":             # 31 quads of z, the last rays missing
        return VolumeGeometry.centred((181, 190, 124)), _orbit(48, 50, 126, 700.0, 2.1)
    if case == "two_warps":
        return VolumeGeometry.centred((131, 130, 256)), _orbit(30, 40, 250, 800.0, 2.3)
    if case == "five_rays":
        return VolumeGeometry.centred((190, 181, 128)), _orbit(48, 48, 160, 700.0, 1.9)
    if case == "two_blocks_of_six_rays":   # rays that miss the grid above and below
        return VolumeGeometry.centred((187, 181, 128)), _orbit(30, 40, 380, 800.0, 1.4)
    if case == "minus_z":
        cg = _orbit(48, 48, 128, 700.0, 2.2)
        cg.det_origin = cg.det_origin + (cg.nv - 1) * cg.det_v
        cg.det_v = -cg.det_v
        return VolumeGeometry.centred((176, 190, 128)), cg
    if case == "helix_off_centre":
        vg = VolumeGeometry((190, 183, 128), (0.9, 1.1, 1.3), (-80.0, -111.0, -79.0))
        cg = _orbit(48, 48, 128, 800.0, 4.4, pitch_v=2.9, det_shift_u=1.7, det_shift_v=-2.4)
        dz = np.linspace(-40.0, 40.0, 48)
        cg.src[:, 2] += dz
        cg.det_origin[:, 2] += dz
        return vg, cg
    raise KeyError(case)


CASES = ["one_warp", "ragged_lines", "two_warps", "five_rays", "two_blocks_of_six_rays", "minus_z", "helix_off_centre"]


def _noalloc(gjp, v, g, vg, dtype_code):
    from paper_1609_00958_gb300 import _capi
    out = torch.empty(g.proj_shape, device="cuda")
    st = _capi.gjp_forward_noalloc(v.data_ptr(), dtype_code, *vg.n, vg.h, vg.origin, g.handle, out.data_ptr(),
                                   torch.cuda.current_stream().cuda_stream)
    assert st == _capi.GJP_OK
    return out


@pytest.mark.parametrize("weight", ["lin", "spl"])
@pytest.mark.parametrize("case", CASES)
def test_column_forward_matches_oracle(gjp, case, weight):
    vg, cg = _scan(case)
    vol = synth.random_field(vg.n, seed=11)
    g = gjp.Geometry.from_cone(cg, weight=weight)
    v = torch.from_numpy(vol).cuda()
    out = gjp.forward(v, g, vg.h, vg.origin)
    batch = gjp.Batch([(v, g, vg.h, vg.origin, torch.empty(g.proj_shape, device="cuda"))])
    assert torch.equal(batch.forward()[0], out)
    assert torch.equal(_noalloc(gjp, v, g, vg, 0), out)
    gjp.stream_status()
    assert not torch.equal(gjp.forward(v, g, vg.h, vg.origin, path="gather"), out)   # another order of sums
    wfun = 1 if weight == "spl" else 0
    ref = oracle.forward(vol, vg, cg, wfun=wfun)
    views, ius, ivs = parity.all_rays(cg)
    got = out.cpu().numpy().astype(np.float64)
    if weight == "spl":
        assert np.abs(got - ref).max() <= TOL32 * np.abs(ref).max()
    else:
        parity.check_rays(got[views, ivs, ius], vol, vg, cg, views, ius, ivs, np.abs(ref).max(), TOL32,
                          ref=ref[views, ivs, ius])


def test_column_forward_field_of_view(gjp):
    vg, cg = _scan("one_warp")
    radius = 70.3
    x = np.arange(vg.n[0]) - 0.5 * (vg.n[0] - 1)
    y = np.arange(vg.n[1]) - 0.5 * (vg.n[1] - 1)
    mask = (x[:, None] ** 2 + y[None, :] ** 2 <= (radius - 2.5) ** 2)[:, :, None]
    vol = (synth.random_field(vg.n, seed=12) * mask).astype(np.float32)
    g = gjp.Geometry.from_cone(cg)
    g.set_fov(radius)
    out = gjp.forward(torch.from_numpy(vol).cuda(), g, vg.h, vg.origin).cpu().numpy().astype(np.float64)
    gjp.stream_status()
    ref = oracle.forward(vol, vg, cg, fov=radius)
    assert np.abs(out - ref).max() <= TOL32 * np.abs(ref).max()


@pytest.mark.parametrize("dt", ["bfloat16", "float16"])
def test_column_forward_16bit(gjp, dt):
    """A grid of more than 2^25 voxels: sampled rays against the oracle on
    the stored values, and the other entry points bit for bit."""
    n = (300, 310, 384)
    vg = VolumeGeometry.centred(n)
    cg = _orbit(90, 16, 384, 1100.0, 2.0)
    v = torch.from_numpy(synth.random_field(n, seed=13)).cuda().to(getattr(torch, dt))
    g = gjp.Geometry.from_cone(cg)
    out = gjp.forward(v, g, vg.h, vg.origin)
    assert torch.equal(_noalloc(gjp, v, g, vg, {"bfloat16": 1, "float16": 2}[dt]), out)
    assert torch.equal(gjp.Batch([(v, g, vg.h, vg.origin, torch.empty(g.proj_shape, device="cuda"))]).forward()[0], out)
    gjp.stream_status()
    stored = v.float().cpu().numpy()
    rays = parity.sampled_rays(cg, 3000, seed=2)
    ref = oracle.rays(stored, vg, cg, *rays)
    got = out.cpu().numpy().astype(np.float64)[rays[0], rays[2], rays[1]]
    parity.check_rays(got, stored, vg, cg, *rays, np.abs(ref).max(), TOL32, ref=ref)


def test_column_forward_leaves_unaligned_volumes_to_the_gather(gjp):
    vg, cg = _scan("one_warp")
    flat = torch.empty(int(np.prod(vg.n)) + 1, device="cuda")
    v = flat[1:].view(vg.n)
    v.copy_(torch.from_numpy(synth.random_field(vg.n, seed=14)))
    assert v.data_ptr() % 16 != 0
    g = gjp.Geometry.from_cone(cg)
    assert torch.equal(gjp.forward(v, g, vg.h), gjp.forward(v, g, vg.h, path="gather"))


@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_column_forward_non_finite_voxels(gjp, value):
    """A non-finite voxel reaches the rays that read it and no others."""
    vg, cg = _scan("one_warp")
    vol = synth.random_field(vg.n, seed=15)
    vol[97, 80, 60] = vol[83, 90, 127] = vol[0, 85, 0] = value
    v = torch.from_numpy(vol).cuda()
    g = gjp.Geometry.from_cone(cg)
    ok = torch.isfinite(gjp.forward(v, g, vg.h, path="gather"))
    out = gjp.forward(v, g, vg.h)
    gjp.stream_status()
    assert 0 < int((~ok).sum()) < ok.numel() // 10
    assert torch.equal(torch.isfinite(out), ok)
