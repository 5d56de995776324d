"""Where the column form of the adjoint reads its lines, on the host: the
table entries and search positions of csrc/gjp_column_index.h, compiled here
as plain C++, over whole scans.  Every element that any lane loads has to lie
in the line of the entry's own detector column."""
import ctypes
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

import synth
from synth.geometry import VolumeGeometry

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1609_00958_gb300", "csrc")

HARNESS = r"""
#include <climits>
#include "gjp_column_index.h"
using namespace gjp_detail;

// least and greatest line element (from the line's first one) that entries
// of the columns load, and the number of entries
template <int K2>
static void sweep(const long long *r, int n_cols, int nx, int ny, int nz, int nv, double pitch, long long *out)
{
    const int pad = line_pad(K2, pitch), nvp = line_length(nv, pad);
    out[0] = LLONG_MAX;
    out[1] = LLONG_MIN;
    out[2] = 0;
    out[3] = nvp;
    for (int k = 0; k < n_cols; ++k, r += 5) {
        Column c{0, 0, r[0], r[1], r[2], r[3], (int)r[4], 0};
        const int nm = c.m == 0 ? nx : ny, line = k * nvp;
        for (int i = 0; i < nm; ++i)
            for (int zc = 0; zc < nz; zc += chunk_of(K2)) {
                ColumnEntry e;
                if (!column_place<K2>(c, i - ((nm - 1) >> 1), zc, nv, pad, line, 0, nv, e)) continue;
                ++out[2];
                for (int lane = 0; lane < 32; lane += 31) {
                    long long pos = column_position(e, lane);
                    for (int p = 0; p < K2; ++p)
                        for (int s = 0; s < 2; ++s, pos += column_half(e)) {
                            const long long first = column_element(pos);
                            if (first - line < out[0]) out[0] = first - line;
                            if (first + (e.code >> 4) - 1 - line > out[1]) out[1] = first + (e.code >> 4) - 1 - line;
                        }
                }
            }
    }
}

extern "C" int pitch_bits() { return kPitchBits; }

// position of the chunk's first voxel above the line's first ray, in rays (N > 2: of the voxel below it)
extern "C" double first_position(const long long *r, int nm, int i, int zc, int nv, int *rays)
{
    ColumnEntry e;
    column_place<4>(Column{0, 0, r[0], r[1], r[2], r[3], (int)r[4], 0}, i - ((nm - 1) >> 1), zc, nv, 0, 0, 0, nv, e);
    *rays = e.code >> 4;
    return (double)(e.pos >> 32) + (double)(e.pos & 0xffffffffLL) / 4294967296.0;
}

extern "C" void sweep_scan(const long long *r, int n_cols, int nx, int ny, int nz, int nv, int k2, double pitch, long long *out)
{
    switch (k2) {
    case 1: sweep<1>(r, n_cols, nx, ny, nz, nv, pitch, out); break;
    case 2: sweep<2>(r, n_cols, nx, ny, nz, nv, pitch, out); break;
    case 3: sweep<3>(r, n_cols, nx, ny, nz, nv, pitch, out); break;
    default: sweep<4>(r, n_cols, nx, ny, nz, nv, pitch, out);
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("column_index")
    src, so = d / "harness.cpp", d / "harness.so"
    src.write_text(HARNESS)
    subprocess.check_call([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(so), str(src)])
    return ctypes.CDLL(str(so))


def _columns(vg, cg, bits):
    """Records Z0, Z1, Y0, Y1, m of every (view, column), and the least pitch on the grid's end planes."""
    n, h, o = (np.array(v, float) for v in (vg.n, vg.h, vg.origin))
    src = (cg.src - o) / h
    du, dv = cg.det_u / h, cg.det_v / h
    mid = (cg.det_origin - cg.src) / h + 0.5 * (cg.nv - 1) * dv
    r = mid[:, None, :] + np.arange(cg.nu)[None, :, None] * du[:, None, :]
    m = (np.abs(r[..., 1]) > np.abs(r[..., 0])).astype(int)
    rm = np.take_along_axis(r, m[..., None], 2)[..., 0]
    sm = np.take_along_axis(np.broadcast_to(src[:, None, :], r.shape), m[..., None], 2)[..., 0]
    nm = n[m]
    t = (np.floor((nm - 1) / 2) - sm) / rm
    ends = np.abs(np.stack([(0 - sm) / rm, (nm - 1 - sm) / rm]) * dv[:, 2][:, None])
    z, y = float(1 << 32), float(1 << bits)
    rec = [(src[:, 2][:, None] + t * r[..., 2]) * z, r[..., 2] / rm * z, t * dv[:, 2][:, None] * y, dv[:, 2][:, None] / rm * y]
    rec = np.stack([np.rint(a).astype(np.int64) for a in rec] + [m.astype(np.int64)], -1)
    return np.ascontiguousarray(rec.reshape(-1, 5)), float(ends.min())


def _sweep(lib, vg, cg, k2):
    rec, pitch = _columns(vg, cg, lib.pitch_bits())
    out = (ctypes.c_longlong * 4)()
    lib.sweep_scan(rec.ctypes.data_as(ctypes.c_void_p), len(rec), *[int(v) for v in vg.n], cg.nv, k2, ctypes.c_double(pitch), out)
    return pitch, list(out)


LEAST = {1: 0.26, 2: 0.26, 3: 0.42, 4: 0.55}         # the least row pitch (voxels) for which a chunk is taken


def _check(lib, vg, cg):
    entries = 0
    for k2, least in LEAST.items():
        pitch, (low, high, count, nvp) = _sweep(lib, vg, cg, k2)
        if pitch <= least or not count:
            continue
        entries += count
        assert 0 <= low and high < nvp, (k2, low, high, nvp)
    return entries


def _cone(n, views, nu, nv, half_angle, pitch, shift=0.0, pitch_u=None):
    """A scan of the grid's inscribed cylinder whose rows are `pitch` voxels apart on the axis."""
    a = math.radians(half_angle)
    d = 0.5 * max(n[:2]) / math.sin(a)
    pu = 4.0 * d * math.tan(a) / nu if pitch_u is None else pitch_u
    return synth.circular(views, nu, nv, d, 2.0 * d, pu, pitch_v=2.0 * pitch, det_shift_v=shift)


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("n,views,nu,nv,half,pitch,shift", [
    ((100, 100, 512), 4, 60, 32, 4.0, 1.0, 0.0),
    ((100, 100, 512), 4, 60, 32, 4.0, 1.0, -200.0),
    ((100, 100, 512), 4, 60, 32, 4.0, 1.0, 230.0),
    ((512, 512, 512), 1, 512, 32, 10.0, 1.0, 0.0),
    ((512, 512, 512), 4, 64, 32, 10.0, 1.0, 0.0),
    ((512, 512, 512), 8, 64, 24, 4.0, 1.5, 0.0),
    ((512, 512, 512), 8, 64, 24, 4.0, 2.0, 0.0),
    ((256, 256, 256), 32, 16, 16, 4.0, 2.0, 60.0),
])
def test_short_detectors_stay_in_their_lines(lib, n, views, nu, nv, half, pitch, shift, sign):
    vg, cg = VolumeGeometry.centred(n), _cone(n, views, nu, nv, half, pitch, shift)
    if sign < 0:
        cg.det_origin, cg.det_v = cg.det_origin + (nv - 1) * cg.det_v, -cg.det_v
    assert _check(lib, vg, cg) > 0


def test_loads_stay_in_their_lines_over_the_range(lib):
    """Chunks, pitches, rows and shifts at random, helices among them."""
    rng = np.random.default_rng(71)
    entries = 0
    for _ in range(150):
        nz = int(np.exp(rng.uniform(np.log(64), np.log(1100))))
        n = (int(rng.integers(24, 90)), int(rng.integers(24, 90)), nz)
        pitch = float(np.exp(rng.uniform(np.log(0.34), np.log(2.6))))
        nv = int(np.exp(rng.uniform(np.log(2), np.log(1.3 * nz / pitch + 2))))
        views = int(rng.integers(1, 5))
        cg = _cone(n, views, int(rng.integers(4, 40)), nv, float(rng.uniform(3.0, 14.0)), pitch,
                   shift=float(rng.uniform(-0.5, 0.5)) * nz / pitch)
        if rng.random() < 0.4:
            dz = rng.uniform(-0.3, 0.3, views) * nz
            cg.src[:, 2] += dz
            cg.det_origin[:, 2] += dz
        if rng.random() < 0.3:
            cg.det_origin, cg.det_v = cg.det_origin + (nv - 1) * cg.det_v, -cg.det_v
        entries += _check(lib, VolumeGeometry.centred(n, (1.0, 1.0, float(rng.uniform(0.6, 1.6)))), cg)
    assert entries > 100000


def test_positions_on_a_tall_detector(lib):
    """Many fine rows far from the centre plane: positions within 4e-7 voxel of float64's (increments per plane hold
    2^-33 voxel, times 512 planes, and as much for the rows; with 40 fraction bits of the rows' distance 2e-6)."""
    n, nv = (1024, 24, 4096), 12000
    vg, cg = VolumeGeometry.centred(n), _cone(n, 2, 3, nv, 4.0, 0.33)
    rec, _ = _columns(vg, cg, lib.pitch_bits())
    lib.first_position.restype = ctypes.c_double
    src = cg.src - np.array(vg.origin)
    for col, row in enumerate(rec):
        k, u = divmod(col, cg.nu)
        r = cg.det_origin[k] + u * cg.det_u[k] - cg.src[k]                 # to row 0, the lowest one
        m = int(row[4])
        for i in (0, 100, n[m] // 2, n[m] - 1):
            t = (i - src[k, m]) / r[m]
            low, pitch = src[k, 2] + t * r[2], t * cg.det_v[k, 2]
            for zc in (0, 256, 2048, 3840):
                rays = ctypes.c_int()
                got = lib.first_position(row.ctypes.data_as(ctypes.c_void_p), n[m], i, zc, nv, ctypes.byref(rays))
                below = 1 if rays.value > 2 else 0                         # the element is counted one up there
                assert abs((got - below) * pitch - (zc - below - low)) <= 4e-7, (col, i, zc)
