// gjp_column_index.h -- where the column form of the adjoint reads its
// lines: the record of a detector column, the entry that a tile of voxels
// makes of it, and the line elements that a lane then loads.  Plain C++, so
// that the bounds are also checked on the host without a GPU.
#pragma once
#include <cmath>

#if defined(__CUDACC__)
#define GJP_HD __host__ __device__ __forceinline__
#else
#define GJP_HD inline
#endif

namespace gjp_detail {

// Fraction bits of the row pitch B in Column (z positions have 32).  The
// pitch is multiplied by up to kMostRows / 2 rows and as many planes: 46 bits
// keep 1024 planes of 32768 rows to 2^-24 voxel, what a ray's own increment
// per plane has.  Rows spread over kMostSpread voxels at most, so that their
// product fits 64 bits.
constexpr int kPitchBits = 46;
constexpr float kPitchScale = (float)(1LL << kPitchBits), kPitchUnit = 1.0f / kPitchScale;
constexpr int kMostRows = 1 << 15;
constexpr double kMostSpread = 32768.0;

// One detector column of one view: the (x, y) path its rays share and their
// z positions, in fixed point (32 fraction bits; the pitch kPitchBits).
struct Column {
    long long Pa, Ga;       // transverse position on plane ic, increment per plane (as Ray)
    long long Z0, Z1;       // z of the middle row on plane ic, increment per plane
    long long Y0, Y1;       // z pitch per detector row on plane ic, increment per plane
    int m, pad;             // driving axis (0 or 1)
};

GJP_HD constexpr int chunk_of(int K2) { return 64 * K2; }
// Zeros before and after a line's values: a tile whose z range only touches
// the detector's reads this far beyond it.
inline int line_pad(int K2, double pitch) { return (int)std::ceil(chunk_of(K2) / pitch) + 16; }
inline int line_length(int nv, int pad) { return (nv + 2 * pad + 31) / 32 * 32; }

// What a tile needs of one column on its plane, shared by the lanes.  The
// first of the rays that reach a voxel is found in fixed point: line element
// and 32 fraction bits of a ray, as many as the sample positions of the
// scatter have.
struct alignas(16) ColumnEntry {
    long long pos;                     // position of the chunk's first voxel: element of the lines << 32 | fraction
    long long step;                    // its increment per voxel
    float pitch;                       // B
    float w1;                          // weight of the upper row
    int code;                          // row + 1 | rays << 4
    int line;                          // the line's first element (debug build)
};

GJP_HD long long column_fixed(float x)             // round(x 2^32)
{
#if defined(__CUDA_ARCH__)
    return __float2ll_rn(x * 4294967296.0f);
#else
    return llrintf(x * 4294967296.0f);
#endif
}

// Position, step, pitch and ray count of column c, di planes from the
// centre plane, for the chunk of chunk_of(K2) voxels from zc on; `line` is
// the first element of the column's line, and only its rows first .. end - 1
// (counted upwards in z) hold anything but zeros.  False when none of these
// comes near the chunk.
template <int K2>
GJP_HD bool column_place(const Column &c, int di, int zc, int nv, int pad, int line, int first, int end, ColumnEntry &e)
{
    const float inv32 = 2.3283064365386963e-10f, invp = kPitchUnit;                // 2^-32, 2^-kPitchBits
    const long long bs = c.Y0 + (long long)di * c.Y1;
    const long long bq = bs < 0 ? -bs : bs;
    const float b = (float)bq * invp;
    const float b_lo = (float)(bq - (long long)(b * kPitchScale)) * invp;     // exact: b has 24 bits
    const float x = 1.0f / b;
    const float x_lo = fmaf(-b, x, 1.0f) * x - b_lo * x * x;           // 1 / B = x + x_lo
    const int n = b >= 1.0f ? 2 : (int)ceilf(2.0001f * x);
    // the chunk's first voxel (the one below it for N > 2) from the line's
    // first ray, which is the detector row lowest in z
    const long long z = ((long long)(zc - (n > 2 ? 1 : 0)) << 32) - c.Z0 - (long long)di * c.Z1 +
                        (((long long)(nv - 1) * bq) >> (kPitchBits - 31));
    const int ray = (int)floorf((float)z * inv32 * x);
    // some such ray of the column near the tile
    const bool near = ray < end + 2 && ray + (int)((float)chunk_of(K2) * x) + n + 2 >= first;
    // what is left of z, in rays: the product of two pairs (a float that is
    // a ray off still is the same position)
    const long long rest = z - (((long long)ray * bq) >> (kPitchBits - 32));
    const float r = (float)rest * inv32, r_lo = (float)(rest - column_fixed(r)) * inv32;
    const float q = r * x, q_lo = fmaf(r, x, -q) + fmaf(r, x_lo, r_lo * x);
    e.pos = ((long long)(line + pad + ray + (n > 2 ? 1 : 0)) << 32) + column_fixed(q) + column_fixed(q_lo);
    e.step = column_fixed(x) + column_fixed(x_lo);
    e.pitch = b;
    e.code = n << 4;
    return near;
}

// The lane's position for its first voxel, its step to the voxel 32 further
// up, and the first line element that a position's rays are loaded from.
GJP_HD long long column_position(const ColumnEntry &e, int lane) { return e.pos + (long long)lane * e.step; }
GJP_HD long long column_half(const ColumnEntry &e) { return e.step << 5; }
GJP_HD int column_element(long long position) { return (int)(position >> 32); }

}  // namespace gjp_detail
