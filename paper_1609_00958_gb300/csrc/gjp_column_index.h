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

// Fraction bits of the row pitch B in Column (z positions have 32).
constexpr int kPitchBits = 40;

// One detector column of one view: the (x, y) path its rays share and their
// z positions, in fixed point (32 fraction bits; the pitch kPitchBits).
struct Column {
    long long Pa, Ga;       // transverse position on plane ic, increment per plane (as Ray)
    long long Z0, Z1;       // z of the middle row on plane ic, increment per plane
    long long Y0, Y1;       // z pitch per detector row on plane ic, increment per plane
    int m, pad;             // driving axis (0 or 1)
};

// The line index of a voxel's rays is found in fixed point: 9 integer and 23
// fraction bits, the entry's position for the voxel at lane 16 of the first
// 32 plus the lane's share (29 fraction bits, the upper half of a product) and
// that of whole pairs and halves of 64 voxels.  Weights then are good to 1e-7
// (rms), with no bias.  kBias keeps the position positive.
constexpr int kBias = 64;
GJP_HD constexpr int chunk_of(int K2) { return 64 * K2; }
// Zeros before and after a line's values: a tile whose z range only touches
// the detector's reads this far beyond it.
inline int line_pad(int K2, double pitch) { return (int)std::ceil(chunk_of(K2) / pitch) + 16; }
inline int line_length(int nv, int pad) { return (nv + 2 * pad + 31) / 32 * 32; }

// What a tile needs of one column on its plane, shared by the lanes.  `base`
// has a sign: a line's element 0 is up to kBias elements above position 0,
// and the first line has nothing below it.
struct alignas(16) ColumnEntry {
    int c, inv;                        // search position (2^-23 rays), its increment per 64 voxels (per voxel: 2^-29)
    float pitch;                       // B
    float w1;                          // weight of the upper row
    int base;                          // element of search position 0 in the lines
    int code;                          // row + 1 | rays << 4
    int line, length;                  // the line's first element and its length (debug build)
};

GJP_HD int column_round(float x)
{
#if defined(__CUDA_ARCH__)
    return __float2int_rn(x);
#else
    return (int)lrintf(x);
#endif
}

GJP_HD int column_mulhi(int a, int b)
{
#if defined(__CUDA_ARCH__)
    return __mulhi(a, b);
#else
    return (int)(((long long)a * b) >> 32);
#endif
}

// Search position, pitch, ray count and base of column c, di planes from the
// centre plane, for the chunk of chunk_of(K2) voxels from zc on; `line` is
// the first element of the column's line, and only its rows first .. end - 1
// (counted upwards in z) hold anything but zeros.  False when none of these
// comes near the chunk.
template <int K2>
GJP_HD bool column_place(const Column &c, int di, int zc, int nv, int pad, int line, int first, int end, ColumnEntry &e)
{
    const float inv32 = 2.3283064365386963e-10f, invp = 9.094947017729282e-13f;   // 2^-32, 2^-kPitchBits
    const long long bs = c.Y0 + (long long)di * c.Y1;
    const long long bq = bs < 0 ? -bs : bs;
    const float b = (float)bq * invp;
    const float b_lo = (float)(bq - (long long)(b * 1099511627776.0f)) * invp;     // exact: b has 24 bits
    const float x = 1.0f / b;
    const float x_lo = fmaf(-b, x, 1.0f) * x - b_lo * x * x;           // 1 / B = x + x_lo
    const int n = b >= 1.0f ? 2 : (int)ceilf(2.0001f * x);
    // the tile's 17th voxel (the one below it for N > 2) from the
    // line's first ray, which is the detector row lowest in z
    const long long z16 = ((long long)(zc + 16 - (n > 2 ? 1 : 0)) << 32) - c.Z0 - (long long)di * c.Z1 +
                          (((long long)(nv - 1) * bq) >> (kPitchBits - 31));
    const int ray = (int)floorf((float)z16 * inv32 * x);
    // some such ray of the column near the tile
    const float reach = (float)(chunk_of(K2) - 16) * x;
    const bool near = ray - (int)(16.0f * x) < end + 2 && ray + (int)reach + n + 2 >= first;
    const float rest = (float)(z16 - (((long long)ray * bq) >> (kPitchBits - 32))) * inv32;
    // (+ 1/2: the lane's share is rounded down)
    e.c = column_round(fmaf(rest * x + rest * x_lo, 8388608.0f, 0.5f)) + (kBias << 23);
    e.inv = column_round(x * 536870912.0f) + column_round(x_lo * 536870912.0f);
    e.pitch = b;
    e.base = line + pad + ray - kBias + (n > 2 ? 1 : 0);
    e.code = n << 4;
    return near;
}

// The search position of the lane's first voxel (lane16: its lane - 16), its
// step to the voxel 32 further up, and the first line element that a
// position's rays are loaded from, counted from the entry's base.
GJP_HD unsigned column_position(const ColumnEntry &e, int lane16)
{
    return (unsigned)(e.c + column_mulhi(lane16 * (1 << 26), e.inv));
}
GJP_HD unsigned column_half(const ColumnEntry &e) { return (unsigned)(e.inv + 1) >> 1; }
GJP_HD int column_element(unsigned position) { return (int)(position >> 23); }

}  // namespace gjp_detail
