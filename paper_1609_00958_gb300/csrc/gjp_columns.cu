// gjp_columns.cu -- the column forms of the adjoint (a gather driven by the
// voxels, first below) and of the forward (at the end of the file), for scans
// whose detector rows run along z.
//
// When det_v is parallel to z, all rays of one detector column (fixed view
// and iu) share their path in (x, y): the same driving axis m, and on plane
// i the same transverse position p_a, whatever their row.  Their z positions
// on that plane are equally spaced,
//     z(iv) = z_0 + iv B,    z_0 and B affine in i.
// The transpose of Eq. 12 then separates.  For one column and one plane,
//     Q[z] = sum over iv of  hat(z(iv) - z) y(iv) step(iv)
// is a short sum over the ceil(2 / B) rays within one voxel of z, and rows
// floor(p_a) and floor(p_a) + 1 of the volume receive (1 - d_a) Q and d_a Q.
// A warp owns a tile of voxels (one plane i of the driving axis, 8 rows,
// 64 K2 z), keeps their sums in registers, and visits the columns that cross
// the tile view after view: no shared taps to hand over, and one addition to
// memory per voxel, driving axis and view group instead of about two per
// voxel and view.
//
// Measured on 512^3 / 512^2 / 360 views: 37.2 ms, against 67.7 ms for the
// warp-combined scatter, with a fifth of its error.  Issue (59%) and the L1
// (58%) are the busiest units, at the 16 warps per SM that the registers
// allow; 22.6 warp instructions per 32 samples of the forward, with 1.3
// column voxels per sample (a column at a tile's edge is visited by both
// tiles).  8 rows and 256 z fill the registers; fewer rows or a shorter chunk
// cost more per column (of a first version at 38.1 ms: 6 rows 44 ms; 128 z 47
// ms; 64 z 66 ms), and 4 planes of one strip in a block share the lines in
// the L1 (90% hits; 8 or 16 planes 38.7 and 38.9 ms).  Ray positions with 23
// fraction bits in one word took 37.4 ms, but their error grew with the rows'
// distance (3.6e-7 of the norm on white noise for rows two voxels apart,
// 1.5e-7 now, 1.8e-7 for the scatter).
#include "gjp_common.cuh"

namespace gjp_detail {

constexpr int kStrip = 8;                    // rows of a tile
constexpr double kColumnSlack = 0.02;        // columns that the float32 search may be off, and twice what it is
constexpr int kColWarps = 4;                 // warps per block: neighbouring planes of one strip

// ---------------------------------------------------------------------------
// Host: whether a scan on a grid has the column form, and the per-view
// records of the column search.

int column_pairs(int nz, double pitch);

// The smallest driving component over the columns of a view with direction
// r0 + u ru (|u| <= cu): at an end or where |r_x| = |r_y| or a component
// vanishes, since max(|r_x|, |r_y|) is convex in u.  `changes` counts the
// places between the ends where |r_x| = |r_y|, the last one at `change`.
static double least_lateral(const double r0[3], const double ru[3], double cu, int &changes, double &change)
{
    const auto lateral = [&](double u) { return std::max(std::fabs(r0[0] + u * ru[0]), std::fabs(r0[1] + u * ru[1])); };
    const double cand[4] = {(r0[1] - r0[0]) / (ru[0] - ru[1]), -(r0[0] + r0[1]) / (ru[0] + ru[1]), -r0[0] / ru[0],
                            -r0[1] / ru[1]};
    double least = std::min(lateral(-cu), lateral(cu));
    changes = 0;
    for (int c = 0; c < 4; ++c)
        if (cand[c] > -cu && cand[c] < cu) {        // false for nan
            least = std::min(least, lateral(cand[c]));
            if (c < 2) {
                ++changes;
                change = cand[c];
            }
        }
    return least;
}

// Ray direction of view k (index units) at the detector's centre, and per column.
static void view_direction(const gjp_geometry &g, int k, const double h[3], double r0[3], double ru[3])
{
    const double cu = 0.5 * (g.nu - 1), cv = 0.5 * (g.nv - 1);
    for (int a = 0; a < 3; ++a) {
        ru[a] = g.du[3 * k + a] / h[a];
        r0[a] = (g.org[3 * k + a] - g.src[3 * k + a]) / h[a] + cu * ru[a] + cv * g.dv[3 * k + a] / h[a];
    }
}

// Block shape of the forward's column form: `threads` threads with four
// voxels of a line each (nz / 4 rounded up to warps) and `rays` rays of the
// column each; `parts` blocks share a column.
struct ColumnShape {
    int threads, rays, parts;
};
static ColumnShape column_shape(int nv, int nz)
{
    ColumnShape c;
    c.threads = (nz / 4 + 31) / 32 * 32;
    const int parts = (nv + 6 * c.threads - 1) / (6 * c.threads);
    c.rays = std::max(4, (nv + parts * c.threads - 1) / (parts * c.threads));
    c.parts = (nv + c.rays * c.threads - 1) / (c.rays * c.threads);
    return c;
}

// Whether enough of the rows lie in the grid: `inside` a view on the mean, on
// its centre plane, `pitch` apart.  A plane of a block costs about 1.8
// samples of each thread for its part of the line plus one per ray, whatever
// rays meet the grid; the gather passes over those that do not.  Measured over 8 grids, 5
// row distances and rows over 0.3 .. 3 times the grid's height or beside it:
// with half of the rows inside, columns / gather is 1.03 .. 1.35 up to 384^3
// (bf16 to 1.38), on larger grids 1.05 .. 1.18 for rows closer than 0.8 voxel
// and 0.66 .. 1.05 for others, with a third there 0.77 .. 1.08; with a fifth
// 1.2 .. 2.1 (640x640x256 / 24 views 1.63 against 0.79 ms).
static bool rows_pay(const ColumnShape &c, const int64_t n[3], double inside, double pitch)
{
    const bool large = (double)n[0] * n[1] * n[2] >= 8.5e7 && pitch >= 0.8;
    return c.parts * c.threads * (1.8 + c.rays) <= (large ? 2.7 : 1.9) * 1.45 * inside;   // as `cost` in forward_columns_pay
}

// Whether the forward's column form covers a scan on a grid: detector rows
// along z in every view, slopes along z below 1/2, rows that spread over
// kMostSpread voxels at most on the centre plane, and enough of them inside
// the grid (rows_pay).
bool column_rays(const gjp_geometry &g, const int64_t n[3], const double h[3], const double o[3])
{
    if (g.nv > kMostRows) return false;
    for (int k = 0; k < g.n_views; ++k)
        if (g.dv[3 * k] != 0.0 || g.dv[3 * k + 1] != 0.0) return false;
    const double cu = 0.5 * (g.nu - 1), cv = 0.5 * (g.nv - 1);
    const ColumnShape c = column_shape(g.nv, (int)n[2]);
    double inside = 0.0, pitch_mean = 0.0;
    for (int k = 0; k < g.n_views; ++k) {
        double r0[3], ru[3], change;
        int changes;
        view_direction(g, k, h, r0, ru);
        const double pv = std::fabs(g.dv[3 * k + 2] / h[2]), least = least_lateral(r0, ru, cu, changes, change);
        if (!(std::fabs(r0[2]) + cu * std::fabs(ru[2]) + cv * pv < 0.49 * least)) return false;
        for (int m = 0; m < 2; ++m) {
            const double away = std::fabs((g.src[3 * k + m] - o[m]) / h[m] - 0.5 * (double)(n[m] - 1));
            if (!(g.nv * pv * away < kMostSpread * least)) return false;
        }
        const int m = std::fabs(r0[0]) >= std::fabs(r0[1]) ? 0 : 1;
        const double t = (0.5 * (double)(n[m] - 1) - (g.src[3 * k + m] - o[m]) / h[m]) / r0[m];
        const double mid = (g.src[3 * k + 2] - o[2]) / h[2] + t * r0[2], pitch = std::max(std::fabs(t * pv), 1e-9);
        const bool up = t * g.dv[3 * k + 2] > 0.0;
        const double below = (mid + 1.0) / pitch, above = ((double)n[2] - mid) / pitch;   // rows from the middle one
        const double first = std::max(0.0, std::ceil(cv - (up ? below : above)));
        const double last = std::min((double)(g.nv - 1), std::floor(cv + (up ? above : below)));
        inside += std::max(0.0, last - first + 1.0) / g.n_views;
        pitch_mean += pitch / g.n_views;
    }
    return rows_pay(c, n, inside, pitch_mean);
}

// Every view needs det_v parallel to z, rays driven by x or y only (with a
// margin, so that float32 and float64 agree), one change of driving axis
// across the detector at most, the whole grid in front of the source, a
// row pitch between 0.26 (at most 8 rays within a voxel of one) and 64 voxels,
// and a grid on which the float32 column search is good to half its margin.
bool column_plan(const gjp_geometry &g, const int64_t n[3], const double h[3], const double o[3], ColumnPlan &plan)
{
    if (g.n_views > 65535 || (int64_t)g.n_views * g.nu > kMaxColumns || g.nv > kMostRows ||
        (int64_t)g.nu * (g.nv + 4096) > (1 << 27))
        return false;
    for (int a = 0; a < 3; ++a)
        if (n[a] > (1 << 15)) return false;
    for (int k = 0; k < g.n_views; ++k)
        if (g.dv[3 * k] != 0.0 || g.dv[3 * k + 1] != 0.0) return false;
    ColumnExtent &x = plan.extent;
    x.pitch = 1e30;
    std::vector<std::pair<double, double>> rows(g.n_views);   // lowest and highest row on the centre plane
    const double cu = 0.5 * (g.nu - 1), cv = 0.5 * (g.nv - 1);
    for (int k = 0; k < g.n_views; ++k) {
        double s[3], r0[3], ru[3], change = 0.0;
        int changes = 0;
        const double pv = g.dv[3 * k + 2] / h[2];
        for (int a = 0; a < 3; ++a) s[a] = (g.src[3 * k + a] - o[a]) / h[a];
        view_direction(g, k, h, r0, ru);
        const auto at = [&](int a, double u) { return r0[a] + u * ru[a]; };
        const double least = least_lateral(r0, ru, cu, changes, change);
        if (changes > 1) return false;
        if (!(std::fabs(r0[2]) + cu * std::fabs(ru[2]) + cv * std::fabs(pv) < 0.999 * least)) return false;
        for (int m = 0; m < 2; ++m) {
            const int a = 1 - m;
            const auto drives = [&](double u) { return std::fabs(at(m, u)) >= std::fabs(at(a, u)); };
            int lo = 0, hi = g.nu - 1;                    // one column of slack: each column's own axis decides
            if (changes) {
                if (drives(-cu)) hi = std::min(hi, (int)std::ceil(change + cu) + 1);
                else lo = std::max(lo, (int)std::floor(change + cu) - 1);
            } else if (!drives(0.0)) {
                continue;
            }
            const double det = r0[m] * ru[a] - r0[a] * ru[m];
            double least_t = 1e300;
            for (int e = 0; e < 4; ++e) {                 // both are monotone in the plane and in the column
                const double rm = at(m, (e & 2 ? hi : lo) - cu);
                const double t = ((e & 1 ? (double)(n[m] - 1) : 0.0) - s[m]) / rm;
                const double pitch = std::fabs(t * pv), spacing = std::fabs(t * det / rm);
                if (!(t > 0.0) || !(pitch >= 0.26) || !(pitch <= 64.0) || !(spacing >= 0.05)) return false;
                x.pitch = std::min(x.pitch, pitch);
                x.pitch_max = std::max(x.pitch_max, pitch);
                least_t = std::min(least_t, t);
            }
            // The column through a point (x, y) of (axis m, axis a): iu - cu =
            // num / den with num = y r0_m - x r0_a - (s_a r0_m - s_m r0_a),
            // den = x ru_a - y ru_m - (s_m ru_a - s_a ru_m), s the source.
            // These moments are formed here in float64, so that a distant
            // source costs no digits; den is made positive in front of it.
            const double q = std::copysign(1.0 / (std::fabs(ru[m]) + std::fabs(ru[a])), det);
            const double num[3] = {q * r0[m], q * r0[a], q * (s[a] * r0[m] - s[m] * r0[a])};
            const double den[3] = {q * ru[a], q * ru[m], q * (s[m] * ru[a] - s[a] * ru[m])};
            // float32 error of iu: five roundings of each sum's largest partial
            // sum (coefficients, products, sums), relative to den = t |q det|
            const double mx = (double)n[m], my = (double)n[a] + kStrip, eps = 5.9604644775390625e-08;   // 2^-24
            const double err_num = 5.0 * eps * (my * std::fabs(num[0]) + mx * std::fabs(num[1]) + std::fabs(num[2]));
            const double err_den = 5.0 * eps * (mx * std::fabs(den[0]) + my * std::fabs(den[1]) + std::fabs(den[2]));
            const double err = (err_num + (cu + 2.0) * err_den) / (least_t * std::fabs(q * det)) + 8.0 * eps * (cu + 2.0);
            if (!(err <= 0.5 * kColumnSlack)) return false;
            ColumnView v;
            for (int j = 0; j < 3; ++j) {
                v.num[j] = (float)num[j];
                v.den[j] = (float)den[j];
            }
            v.u_lo = lo;
            v.u_hi = hi;
            v.view = k;
            v.rising = at(m, lo - cu) * det > 0.0 ? 1 : -1;
            plan.views[m].push_back(v);
        }
        const int m = std::fabs(r0[0]) >= std::fabs(r0[1]) ? 0 : 1;
        const double t = (0.5 * (double)(n[m] - 1) - s[m]) / r0[m], half = std::fabs(t * pv) * cv;
        x.pitch_mean += std::fabs(t * pv) / g.n_views;
        rows[k] = {s[2] + t * r0[2] - half, s[2] + t * r0[2] + half};
    }
    if (!(g.nv * x.pitch_max < kMostSpread)) return false;
    const double top = (double)(n[2] - 1), chunk = chunk_of(column_pairs((int)n[2], x.pitch));
    for (const auto &r : rows) {
        const double lo = std::max(0.0, r.first), hi = std::min(top, r.second);
        x.whole = x.whole && r.first <= 1.0 && r.second >= top - 1.0;
        if (lo > hi) continue;
        x.covered += hi - lo + 1.0;
        x.chunks += std::floor(hi / chunk) - std::floor(lo / chunk) + 1.0;
    }
    return true;
}

// ---------------------------------------------------------------------------
// Device: the column records, once per geometry and grid.

// The same double-float steps as setup_ray at the detector's middle row, so
// that the driving axis and the transverse position agree with the forward's
// bit for bit; the z position and its pitch per row follow from the moment's
// and the direction's dependence on v.
__device__ __forceinline__ Column make_column(const ViewParams &vp, const VolParams &V, float fu)
{
    Ray R;
    setup_ray(vp, V, fu, 0.0f, R);
    const int m = R.m, a = 1 - m;
    const auto lateral = [&](int k) {
        return f2_affine({vp.rh[k], vp.rl[k]}, {vp.rh[3 + k], vp.rl[3 + k]}, {vp.rh[6 + k], vp.rl[6 + k]}, fu, 0.0f);
    };
    const f2 rm = m == 0 ? lateral(0) : lateral(1);
    const float inv = __fdividef(1.0f, rm.hi);
    const f2 mv = {a == 0 ? vp.mh[6] : vp.mh[7], a == 0 ? vp.ml[6] : vp.ml[7]};   // dL_a / dv
    f2 dq = f2_div(mv, rm, inv);
    if (2 == (m + 1) % 3) dq = f2_neg(dq);
    const f2 dg = f2_div({vp.rh[8], vp.rl[8]}, rm, inv);                            // d(rt_z) / dv
    const int nm = m == 0 ? V.n[0] : V.n[1];
    const f2 y0 = f2_shift(dq, 0.0f, dg, (float)R.ic - 0.5f * (float)(nm - 1));
    Column c;
    c.Pa = R.Pa;
    c.Ga = R.Ga;
    c.Z0 = R.Pb;
    c.Z1 = R.Gb;
    c.Y0 = __float2ll_rn(y0.hi * kPitchScale) + __float2ll_rn(y0.lo * kPitchScale);
    c.Y1 = __float2ll_rn(dg.hi * kPitchScale) + __float2ll_rn(dg.lo * kPitchScale);
    c.m = m;
    c.pad = 0;
    return c;
}

__global__ void gjp_columns_kernel(const ViewParams *__restrict__ views, VolParams V, int nu, int n_views,
                                   Column *__restrict__ cols)
{
    const int u = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (u >= nu) return;
    ViewParams vp;
    load_view(views, k, vp);
    cols[(size_t)k * nu + u] = make_column(vp, V, (float)u - 0.5f * (float)(nu - 1));
}

cudaError_t write_columns(const ViewParams *views, const VolParams &V, const gjp_geometry &g, Column *cols,
                          cudaStream_t s)
{
    const dim3 grid((unsigned)((g.nu + 127) / 128), (unsigned)g.n_views);
    gjp_columns_kernel<<<grid, 128, 0, s>>>(views, V, g.nu, g.n_views, cols);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// The projections, times their plane step, with the detector rows contiguous
// and ascending in z: line (view, iu) holds y step at pad + row, zeros
// elsewhere.  Sets head[0] when a value is not finite, and in line_ranges(head)
// each line's extent of values other than zero, from both ends, so that the
// gather passes over the rest, as the scatter does over rays of zeros.  512^3
// / 60 views, without -> with the ranges: zeros 6.40 -> 0.80 ms (the scatter
// 0.59), one column in 16 6.43 -> 1.14 (1.70), a trace of 32^2 pixels 6.40 ->
// 1.20 (0.70), dense projections 6.43 -> 6.32 (12.9): the 32-row tiles outside
// the detector, more than half of them, now only store zeros.
constexpr int kTrRows = 8;

// Head of the workspace: a flag word, and from byte 256 on one pair per line.
constexpr size_t kHeadBytes = 256;
struct LineRange {
    unsigned from_end, end;            // line length - first such element, last one + 1; zeros: none
};
template <typename W> __host__ __device__ __forceinline__ auto line_ranges(W *head)
{
    using R = std::conditional_t<std::is_const<W>::value, const LineRange, LineRange>;
    return reinterpret_cast<R *>(head + kHeadBytes / sizeof(W));
}

__global__ void __launch_bounds__(32 * kTrRows) gjp_lines_kernel(const float *__restrict__ proj, VolParams V,
                                                                  const Column *__restrict__ cols, int nu, int nv,
                                                                  int nvp, int pad, int view0, float *__restrict__ lines,
                                                                  unsigned *__restrict__ head)
{
    __shared__ float tile[32][33];
    const int u0 = blockIdx.x * 32, p0 = blockIdx.y * 32;            // p: position in the line
    const int view = view0 + blockIdx.z;
    if (p0 + 32 <= pad || p0 >= pad + nv) {                          // zeros around the values: more than half of a line
#pragma unroll
        for (int k = threadIdx.y; k < 32; k += kTrRows)
            if (u0 + k < nu) lines[((size_t)blockIdx.z * nu + u0 + k) * nvp + p0 + threadIdx.x] = 0.0f;
        return;
    }
    const bool down = cols[(size_t)view * nu].Y0 < 0;                // rows descend in z: reversed lines
    const float *src = proj + (size_t)view * nv * nu;
#pragma unroll
    for (int k = threadIdx.y; k < 32; k += kTrRows) {
        const int r = p0 + k - pad, u = u0 + threadIdx.x;
        const int iv = down ? nv - 1 - r : r;
        tile[k][threadIdx.x] = (r >= 0 && r < nv && u < nu) ? __ldg(src + (size_t)iv * nu + u) : 0.0f;
    }
    __syncthreads();
    const float inv = 2.3283064365386963e-10f;                       // 2^-32
    bool bad = false;
#pragma unroll
    for (int k = threadIdx.y; k < 32; k += kTrRows) {
        const int u = u0 + k, p = p0 + threadIdx.x;
        if (u >= nu) continue;                                       // the whole warp (and p < nvp: a multiple of 32)
        const Column *c = cols + (size_t)view * nu + u;
        const int m = c->m;
        const float hm = m == 0 ? V.h[0] : V.h[1], ha = m == 0 ? V.h[1] : V.h[0];
        const int r = p - pad;
        const float v = (float)(down ? nv - 1 - r : r) - 0.5f * (float)(nv - 1);
        const float ga = ha * (__ll2float_rn(c->Ga) * inv);
        const float gb = V.h[2] * __fmaf_rn(v, __ll2float_rn(c->Y1) * kPitchUnit, __ll2float_rn(c->Z1) * inv);
        const float y = tile[threadIdx.x][k] * sqrtf(hm * hm + ga * ga + gb * gb);
        bad = bad || !(fabsf(y) <= 3.402823466e38f);
        const size_t line = (size_t)blockIdx.z * nu + u;
        lines[line * nvp + p] = y;
        const unsigned some = __ballot_sync(0xffffffffu, y != 0.0f);
        if (some && threadIdx.x == 0) {
            LineRange *r = line_ranges(head) + line;
            atomicMax(&r->from_end, (unsigned)(nvp - (p0 + __ffs(some) - 1)));
            atomicMax(&r->end, (unsigned)(p0 + 32 - __clz(some)));
        }
    }
    if (bad) atomicOr(head, 1u);
}

// ---------------------------------------------------------------------------
// The gather.

int column_chunks(int nz, int K2) { return (nz + chunk_of(K2) - 1) / chunk_of(K2); }

struct ColumnTiles {
    int n_zc, n_strip[2], n_pg[2];     // z chunks; strips of kStrip rows and groups of planes per driving axis
    int first[2];                      // first tile of each driving axis
    int view_lo[2], view_hi[2];        // range of the axis' ColumnViews
};

__device__ __forceinline__ float fma_sat(float a, float b, float c)
{
    float r;
    asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Weight of a ray for its reach e = 1 - distance (Eq. 13/14).
template <bool SPL> __device__ __forceinline__ float2 shape(float2 e)
{
    return SPL ? __fmul2_rn(__fmul2_rn(e, e), __ffma2_rn(e, make_float2(-2.0f, -2.0f), make_float2(3.0f, 3.0f))) : e;
}

// Debug build (GJP_CHECK_TAPS): where a lane loads `n` elements of entry e's
// line of nvp elements from; loads that would leave the line are recorded and
// read its first elements instead (a line is longer than any n).  The element
// itself, and free, in the production build.
__device__ __forceinline__ int checked_element(const ColumnEntry &e, long long position, int n, int nvp)
{
    const int k = column_element(position);
    if (!GJP_CHECK_TAPS) return k;
    const bool ok = k >= e.line && k + n <= e.line + nvp;
    if (!ok) atomicOr(&g_gjp_tap_fault, 1u);
    return ok ? k : e.line;
}

// The same for the taps z0 and z0 + 1 of a forward line of nz voxels with its
// edges.
__device__ __forceinline__ int checked_line_tap(int z0, int nz, int edge)
{
    if (!GJP_CHECK_TAPS) return z0;
    const bool ok = z0 >= -edge && z0 + 1 < nz + edge;
    if (!ok) atomicOr(&g_gjp_tap_fault, 1u);
    return ok ? z0 : 0;
}

// Q of one column at the lane's 2 K2 voxels (z = lane + 32 k).  N = 2
// (B >= 1): the rays on either side of z; N = 3 (B >= 2/3): the first three
// above z - 1; N = 0: the first n above z - 1.  CAREFUL keeps a ray out of
// reach from contributing 0 x inf.
template <int K2, int N, bool SPL, bool CAREFUL>
__device__ __forceinline__ void column_sums(const float *__restrict__ lines, const ColumnEntry &e, int lane, int n, int nvp,
                                            float2 (&q)[K2])
{
    long long pos = column_position(e, lane);
    const long long half = column_half(e);
    const float B = e.pitch, b = B * 2.3283064365386963e-10f;            // per 2^-32 of a ray
#pragma unroll
    for (int p = 0; p < K2; ++p) {
        float2 w[3], y[3];
        float f[2];                                                      // past the ray, in 2^-32 rays
        const float *at[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            at[s] = lines + checked_element(e, pos, N > 0 ? N : n, nvp);
            f[s] = __uint2float_rn((unsigned)pos);
            pos += half;
        }
        if (N == 2) {
            w[0] = make_float2(fma_sat(-f[0], b, 1.0f), fma_sat(-f[1], b, 1.0f));
            w[1] = make_float2(fma_sat(f[0], b, 1.0f - B), fma_sat(f[1], b, 1.0f - B));
        } else if (N == 3) {
            const float2 F = make_float2(f[0], f[1]), mb = make_float2(-b, -b);
            const float c = B - 1.0f;
            w[0] = __ffma2_rn(F, mb, make_float2(B, B));
            const float2 t = __fadd2_rn(w[0], make_float2(c, c));
            w[1] = make_float2(1.0f - fabsf(t.x), 1.0f - fabsf(t.y));
            w[2] = make_float2(fma_sat(c, -2.0f, -w[0].x), fma_sat(c, -2.0f, -w[0].y));
        }
        if (N > 0) {
#pragma unroll
            for (int j = 0; j < N; ++j) {
                y[j] = make_float2(__ldg(at[0] + j), __ldg(at[1] + j));
                w[j] = shape<SPL>(w[j]);
                if (CAREFUL) {
                    y[j].x = w[j].x > 0.0f ? y[j].x : 0.0f;
                    y[j].y = w[j].y > 0.0f ? y[j].y : 0.0f;
                }
            }
            q[p] = __fmul2_rn(w[0], y[0]);
#pragma unroll
            for (int j = 1; j < N; ++j) q[p] = __ffma2_rn(w[j], y[j], q[p]);
        } else {
            float2 d = __ffma2_rn(make_float2(f[0], f[1]), make_float2(-b, -b), make_float2(B - 1.0f, B - 1.0f));
            float2 sum = make_float2(0.0f, 0.0f);
            for (int j = 0; j < n; ++j) {
                const float2 v = shape<SPL>(make_float2(__saturatef(1.0f - fabsf(d.x)), __saturatef(1.0f - fabsf(d.y))));
                float2 x = make_float2(__ldg(at[0] + j), __ldg(at[1] + j));
                if (CAREFUL) {
                    x.x = v.x > 0.0f ? x.x : 0.0f;
                    x.y = v.y > 0.0f ? x.y : 0.0f;
                }
                sum = __ffma2_rn(v, x, sum);
                d = __fadd2_rn(d, make_float2(B, B));
            }
            q[p] = sum;
        }
    }
}

// The columns of up to 32 views that may cross a tile, one record per view
// that has any, numbered through.
struct ColumnSpan {
    int view, u_lo, start;             // the view, its first column, that column's number
};

// Lane l looks for the columns of the axis' view vb + l: those through rows
// a0 - 1 and a0 + kStrip on plane i.  Returns their number; `start` is the number
// of this lane's first one, `any` whether it has one.
__device__ __forceinline__ int column_spans(const ColumnView *__restrict__ cviews, int nu, int vb, int view_hi, int i,
                                            int a0, ColumnSpan *__restrict__ spans, int &start, bool &any)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    int cnt = 0, u_lo = 0, view = 0;
    if (vb + lane < view_hi) {
        const ColumnView cv = cviews[vb + lane];
        const float cu = 0.5f * (float)(nu - 1), x = (float)i, y0 = (float)(a0 - 1), y1 = (float)(a0 + kStrip);
        const float n0 = x * cv.den[0] - y0 * cv.den[1] - cv.den[2], n1 = x * cv.den[0] - y1 * cv.den[1] - cv.den[2];
        // in front of the source, den is positive; iu grows or falls with the
        // row throughout, without bound where den goes to zero
        const bool f0 = n0 > 0.0f, f1 = n1 > 0.0f;
        const float far = cv.rising > 0 ? 1.0e9f : -1.0e9f;
        const float u0 = f0 ? __fdividef(y0 * cv.num[0] - x * cv.num[1] - cv.num[2], n0) + cu : -far;
        const float u1 = f1 ? __fdividef(y1 * cv.num[0] - x * cv.num[1] - cv.num[2], n1) + cu : far;
        u_lo = max(cv.u_lo, (int)floorf(fmaxf(fminf(u0, u1) - (float)kColumnSlack, -1.0f)));
        const int u_hi = min(cv.u_hi, (int)ceilf(fminf(fmaxf(u0, u1) + (float)kColumnSlack, 1.0e9f)));
        cnt = f0 || f1 ? max(0, u_hi - u_lo + 1) : 0;
        view = cv.view;
    }
    any = cnt > 0;
    int sum = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int up = __shfl_up_sync(full, sum, d);
        if (lane >= d) sum += up;
    }
    start = sum - cnt;
    const unsigned have = __ballot_sync(full, any);
    if (any) spans[__popc(have & ((1u << lane) - 1u))] = {view, u_lo, start};
    return __shfl_sync(full, sum, 31);
}

// The table entries of the columns numbered q0 .. q0 + 31 (of `total`): lane
// l takes number q0 + l.  The valid entries are kept together; returns their
// number.
template <int K2, bool SPL>
__device__ __forceinline__ int column_fill(const VolParams &V, const Column *__restrict__ cols, int nu, int nv, int nvp,
                                           int pad, int line_view0, int m, int i, int a0, int zc,
                                           const LineRange *__restrict__ ranges, const ColumnSpan *__restrict__ spans,
                                           int start, bool any, int q0, int total,
                                           ColumnEntry *__restrict__ tab)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    // the record of number q0 + lane: the last one that starts at or below it
    const int from = start - q0;
    const unsigned begins = __reduce_or_sync(full, any && from > 0 && from < 32 ? 1u << from : 0u);
    const int before = __popc(__ballot_sync(full, any && from <= 0));
    bool ok = q0 + lane < total;
    ColumnEntry e;
    {
        if (ok) {
            const ColumnSpan sp = spans[before - 1 + __popc(begins & (0xffffffffu >> (31 - lane)))];
            const int u = sp.u_lo + (q0 + lane - sp.start);
            const Column c = cols[(size_t)sp.view * nu + u];
            const int ic = ((m == 0 ? V.n[0] : V.n[1]) - 1) >> 1;
            const int di = i - ic;
            const unsigned long long pa = (unsigned long long)(c.Pa + (long long)di * c.Ga);
            const int row = floor_of(pa) - a0;
            ok = c.m == m && row >= -1 && row < kStrip;
            if (V.fov_r2 > 0.0f) {
                int lo, hi;
                fov_planes(V, m, ic, c.Pa, c.Ga, 0, 0, lo, hi);   // z plays no part
                ok = ok && i >= lo && i <= hi;
            }
            const int line = (sp.view - line_view0) * nu + u;
            const LineRange r = ranges[line];
            ok = column_place<K2>(c, di, zc, nv, pad, line * nvp, nvp - pad - (int)r.from_end, (int)r.end - pad, e) && ok;
            e.w1 = upper_weight<SPL>(frac_of(pa));
            e.code |= row + 1;
            e.line = GJP_CHECK_TAPS ? line * nvp : 0;
        }
    }
    const unsigned mask = __ballot_sync(0xffffffffu, ok);
    if (ok) tab[__popc(mask & ((1u << lane) - 1u))] = e;
    return __popc(mask);
}

template <int K2, bool SPL, bool CAREFUL>
__device__ __forceinline__ void column_gather(const float *__restrict__ lines, const VolParams &V,
                                              const ColumnView *__restrict__ cviews, const Column *__restrict__ cols,
                                              int nu, int nv, int nvp, int pad, int line_view0, int view_lo, int view_hi,
                                              int m, int i, int a0, int zc, const LineRange *__restrict__ ranges,
                                              ColumnEntry *__restrict__ tab, ColumnSpan *__restrict__ spans,
                                              float2 (&acc)[kStrip][K2])
{
    const int lane = (int)(threadIdx.x & 31);
    for (int vb = view_lo; vb < view_hi; vb += 32) {
        int start;
        bool any;
        __syncwarp();                                    // the last views' records are read
        const int total = column_spans(cviews, nu, vb, view_hi, i, a0, spans, start, any);
        for (int q0 = 0; q0 < total; q0 += 32) {
            __syncwarp();                                // records written; every lane has read the last table
            const int cnt = column_fill<K2, SPL>(V, cols, nu, nv, nvp, pad, line_view0, m, i, a0, zc, ranges, spans, start, any,
                                                    q0, total, tab);
            __syncwarp();
#pragma unroll 1
            for (int k = 0; k < cnt; ++k) {
                const ColumnEntry e = tab[k];
                const int n = e.code >> 4;
                float2 q[K2];
                if (n == 2) column_sums<K2, 2, SPL, CAREFUL>(lines, e, lane, n, nvp, q);
                else if (n == 3) column_sums<K2, 3, SPL, CAREFUL>(lines, e, lane, n, nvp, q);
                else column_sums<K2, 0, SPL, CAREFUL>(lines, e, lane, n, nvp, q);
                const float2 w1 = make_float2(e.w1, e.w1), w0 = make_float2(1.0f - e.w1, 1.0f - e.w1);
                const auto rows = [&](auto r) {           // rows r - 1 and r of the tile
                    constexpr int R = decltype(r)::value;
#pragma unroll
                    for (int p = 0; p < K2; ++p) {
                        if constexpr (R > 0) acc[R - 1][p] = __ffma2_rn(w0, q[p], acc[R - 1][p]);
                        if constexpr (R < kStrip) acc[R][p] = __ffma2_rn(w1, q[p], acc[R][p]);
                    }
                };
                switch (e.code & 15) {                    // warp-uniform
                case 0: rows(std::integral_constant<int, 0>{}); break;
                case 1: rows(std::integral_constant<int, 1>{}); break;
                case 2: rows(std::integral_constant<int, 2>{}); break;
                case 3: rows(std::integral_constant<int, 3>{}); break;
                case 4: rows(std::integral_constant<int, 4>{}); break;
                case 5: rows(std::integral_constant<int, 5>{}); break;
                case 6: rows(std::integral_constant<int, 6>{}); break;
                case 7: rows(std::integral_constant<int, 7>{}); break;
                case 8: rows(std::integral_constant<int, 8>{}); break;
                }
            }
        }
    }
}

// resident blocks by register use: 4 K2 x 8 rows of sums, and about 60 more
constexpr int column_blocks(int K2) { return K2 == 1 ? 8 : K2 == 2 ? 6 : 4; }

template <int K2, bool SPL>
__global__ void __launch_bounds__(32 * kColWarps, column_blocks(K2)) gjp_adjoint_columns_kernel(
    const float *__restrict__ lines, const unsigned *__restrict__ head, VolParams V,
    const ColumnView *__restrict__ cviews, const Column *__restrict__ cols, int nu, int nv, int nvp, int pad,
    int line_view0, int per_group, ColumnTiles T, float *__restrict__ vol)
{
    __shared__ ColumnEntry s_tab[kColWarps * 32];
    __shared__ ColumnSpan s_spans[kColWarps * 32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int tile = blockIdx.x;
    const int m = tile >= T.first[1] ? 1 : 0;
    tile -= T.first[m];
    const int zc = (tile % T.n_zc) * chunk_of(K2);
    tile /= T.n_zc;
    const int a0 = (tile % T.n_strip[m]) * kStrip;
    const int i = (tile / T.n_strip[m]) * kColWarps + warp;
    const int nm = m == 0 ? V.n[0] : V.n[1], na = m == 0 ? V.n[1] : V.n[0];
    const int view_lo = T.view_lo[m] + blockIdx.y * per_group;
    const int view_hi = min(view_lo + per_group, T.view_hi[m]);
    if (i >= nm || view_lo >= view_hi) return;            // the whole warp

    float2 acc[kStrip][K2];
#pragma unroll
    for (int r = 0; r < kStrip; ++r)
#pragma unroll
        for (int p = 0; p < K2; ++p) acc[r][p] = make_float2(0.0f, 0.0f);
    ColumnEntry *tab = s_tab + 32 * warp;
    const LineRange *ranges = line_ranges(head);
    if (__ldg(head) == 0u)
        column_gather<K2, SPL, false>(lines, V, cviews, cols, nu, nv, nvp, pad, line_view0, view_lo, view_hi, m, i, a0,
                                         zc, ranges, tab, s_spans + 32 * warp, acc);
    else
        column_gather<K2, SPL, true>(lines, V, cviews, cols, nu, nv, nvp, pad, line_view0, view_lo, view_hi, m, i, a0,
                                        zc, ranges, tab, s_spans + 32 * warp, acc);
    const long long sm = m == 0 ? V.s[0] : V.s[1], sa = m == 0 ? V.s[1] : V.s[0];
    const int z0 = zc + lane;
    float *out = vol + (long long)i * sm + (long long)a0 * sa + z0;
#pragma unroll
    for (int r = 0; r < kStrip; ++r) {
        if (a0 + r >= na) break;
#pragma unroll
        for (int p = 0; p < K2; ++p) {
            if (z0 + 64 * p < V.n[2] && acc[r][p].x != 0.0f) atomicAdd(out + 64 * p, acc[r][p].x);
            if (z0 + 64 * p + 32 < V.n[2] && acc[r][p].y != 0.0f) atomicAdd(out + 64 * p + 32, acc[r][p].y);
        }
        out += sa;
    }
}

struct ColumnJob {
    const float *lines;
    const unsigned *head;
    VolParams V;
    const ColumnForm *form;
    const gjp_geometry *g;
    int nvp, pad, view0, n_views, groups;
    float *vol;
    cudaStream_t s;
};

template <int K2> cudaError_t launch_tiles(const ColumnJob &j)
{
    const VolParams &V = j.V;
    ColumnTiles T;
    T.n_zc = column_chunks(V.n[2], K2);
    int tiles = 0, longest = 0;
    for (int m = 0; m < 2; ++m) {
        T.n_strip[m] = (V.n[1 - m] + kStrip - 1) / kStrip;
        T.n_pg[m] = (V.n[m] + kColWarps - 1) / kColWarps;
        T.first[m] = tiles;
        // the axis' views among view0 .. view0 + n_views - 1 (the lists ascend)
        const std::vector<int> &ids = j.form->view_ids[m];
        const int base = m == 0 ? 0 : (int)j.form->view_ids[0].size();
        T.view_lo[m] = base + (int)(std::lower_bound(ids.begin(), ids.end(), j.view0) - ids.begin());
        T.view_hi[m] = base + (int)(std::lower_bound(ids.begin(), ids.end(), j.view0 + j.n_views) - ids.begin());
        longest = std::max(longest, T.view_hi[m] - T.view_lo[m]);
        if (T.view_hi[m] > T.view_lo[m]) tiles += T.n_zc * T.n_strip[m] * T.n_pg[m];
    }
    if (!tiles) return cudaSuccess;
    const int groups = std::max(1, std::min(j.groups, longest));
    const int per = (longest + groups - 1) / groups;
    const dim3 grid((unsigned)tiles, (unsigned)((longest + per - 1) / per));
    auto kern = j.g->weight == GJP_WEIGHT_SPL ? gjp_adjoint_columns_kernel<K2, true> : gjp_adjoint_columns_kernel<K2, false>;
    kern<<<grid, 32 * kColWarps, 0, j.s>>>(j.lines, j.head, V, j.form->d_views, j.form->d_cols, j.g->nu, j.g->nv, j.nvp,
                                           j.pad, j.view0, per, T, j.vol);
    return cudaGetLastError();
}

// Voxels per lane and table entry: 2 K2, in chunks of 64 K2 along z.  An
// entry costs about as much as one more pair of voxels (256^3 / 180 views,
// ms for K2 = 1..4: 4.27, 3.13, 4.74, 2.64, i.e. 1.07, 1.56, 2.37, 2.64 per
// chunk), so chunks x (K2 + 1) is what a grid costs.  9 bits of search
// position hold a chunk's rays down to the pitch given here.
int column_pairs(int nz, double pitch)
{
    static const double least[5] = {0, 0.26, 0.26, 0.42, 0.55};
    int best = 1;
    for (int k = 1; k <= 4; ++k)
        if (pitch > least[k] && column_chunks(nz, k) * (k + 1) <= column_chunks(nz, best) * (best + 1)) best = k;
    return best;
}

// Whether the column form is the faster adjoint: short z lines leave most of
// a chunk's lanes idle (64^3: 37 us against 33 us for the warp-combined
// scatter; 256^3: 2.64 ms against 4.37 ms), with rays far apart most voxels
// that it visits receive nothing, and its transposed projections and two
// passes are not repaid by little work (128^3, 4 views: 37 against 34 us;
// 200x180x256, 2 views: 49 against 67 us; 128^3, 16 views: 67 against 77 us).
// The z lines at which both are even, per chunk and pair of voxels (and one
// more), are 19 (300x300x1024) to 33 (100x100x256) over 8 grids with rows one
// voxel apart: the line lies at the last.
bool columns_pay(const int64_t n[3], int n_views, double pitch)
{
    if (n[2] > (1 << 15) || (double)n_views * (double)n[0] * (double)n[1] * (double)n[2] < 16777216.0) return false;
    const int nz = (int)n[2], k = column_pairs(nz, pitch);
    return 33 * (k + 1) * column_chunks(nz, k) <= nz;
}

// Where the detector covers a part of the z lines only, an entry still works
// on its whole chunk, while the scatter's time follows the rows.  Measured
// over 8 grids, 6 coverages and the pitches of row centres 0.5 .. 2 (512^3 /
// 60 views, pitch 1, ms: 30 rows 6.36 against 0.86, 153 6.39 / 4.10, 256
// 6.41 / 6.40, 358 6.43 / 9.91, 537 6.46 / 13.1), the two are even, within a
// fifth, where the rows cover `least` voxels per voxel pair (and one more) of the chunks that
// they meet: 20 below a pitch of 0.53, where the scatter combines little and
// the gather takes four or more rays, 42 up to 0.72 (four rays, but the
// scatter combines pairs), 28 up to 1.25, and 22 above, where no two rays
// of a column share a voxel.
bool columns_pay(const ColumnExtent &x, const int64_t n[3], int n_views)
{
    if (x.pitch_max > 3.0 || !columns_pay(n, n_views, x.pitch)) return false;
    const double least = x.pitch_mean < 0.53 ? 20.0 : x.pitch_mean < 0.72 ? 42.0 : x.pitch_mean < 1.25 ? 28.0 : 22.0;
    return x.whole || (x.chunks > 0.0 && least * (column_pairs((int)n[2], x.pitch) + 1) * x.chunks <= x.covered);
}

// Adds A^T proj to vol.
gjp_status adjoint_columns(const float *proj, const VolParams &V, const ColumnForm &form, const gjp_geometry &g,
                           float *vol, cudaStream_t s)
{
    const int K2 = column_pairs(V.n[2], form.extent.pitch);
    const int pad = line_pad(K2, form.extent.pitch), nvp = line_length(g.nv, pad);
    const size_t line_bytes = (size_t)g.nu * nvp * sizeof(float);
    const int most = (int)std::max<size_t>(1, std::min<size_t>((size_t)g.n_views, (512ull << 20) / line_bytes));
    const size_t head_bytes = (kHeadBytes + sizeof(LineRange) * (size_t)most * g.nu + 255) / 256 * 256;
    void *ws = nullptr;
    const gjp_status got = workspace_alloc(head_bytes + (size_t)most * line_bytes, s, &ws);
    if (got != GJP_OK) return got;
    ColumnJob j;
    j.head = static_cast<unsigned *>(ws);
    float *lines = reinterpret_cast<float *>(static_cast<char *>(ws) + head_bytes);
    j.lines = lines;
    j.V = V;
    j.form = &form;
    j.g = &g;
    j.nvp = nvp;
    j.pad = pad;
    j.vol = vol;
    j.s = s;
    cudaError_t e = cudaStreamWaitEvent(s, form.ready, 0);       // the records, written on another stream perhaps
    for (int v0 = 0; v0 < g.n_views && e == cudaSuccess; v0 += most) {
        j.view0 = v0;
        j.n_views = std::min(most, g.n_views - v0);
        if ((e = cudaMemsetAsync(ws, 0, head_bytes, s)) != cudaSuccess) break;
        const dim3 tg((unsigned)((g.nu + 31) / 32), (unsigned)((nvp + 31) / 32), (unsigned)j.n_views);
        gjp_lines_kernel<<<tg, dim3(32, kTrRows), 0, s>>>(proj, V, form.d_cols, g.nu, g.nv, nvp, pad, v0, lines,
                                                          static_cast<unsigned *>(ws));
        if ((e = cudaGetLastError()) != cudaSuccess) break;
        // View groups run one after another: their lines (the values, without
        // the zeros) stay in the L2 while all tiles read them, 64 MB measured
        // best (512^3, 216 views of 1 MB, a version at 38.0 ms: 2 / 4 / 8 groups 38.3 / 38.0 /
        // 39.2 ms per 360 views); small grids take more groups until every SM
        // has some waves of warps, of eight views or more (us for 3000 /
        // 10000 / 30000 warps: 128^3, 64 views 227 / 180 / 185; 16 views 76 /
        // 70 / 70; 256^3, 32 views 482 / 482 / 488; 200x180x256, 12 views
        // 130 / 136 / 137).
        const double mb = (double)j.n_views * g.nu * g.nv * 4.0 / (64.0 * 1024 * 1024);
        const double warps = 2.0 * V.n[0] * V.n[1] / kStrip * column_chunks(V.n[2], K2);
        j.groups = std::max((int)std::ceil(mb), (int)std::ceil(10000.0 / warps));
        j.groups = std::max(1, std::min(j.groups, (j.n_views + 7) / 8));
        e = K2 == 4 ? launch_tiles<4>(j) : K2 == 3 ? launch_tiles<3>(j) : K2 == 2 ? launch_tiles<2>(j) : launch_tiles<1>(j);
    }
    const cudaError_t f = cudaFreeAsync(ws, s);
    return e == cudaSuccess && f == cudaSuccess ? GJP_OK : GJP_ERR_CUDA;
}

unsigned columns_tap_faults() { return take_tap_faults(); }

// ---------------------------------------------------------------------------
// Forward, column form.
//
// The forward of one detector column separates the same way: on plane i its
// rays sample one line of z, W[z] = (1 - d_a) V[ia][z] + d_a V[ia + 1][z].
// A block owns a column (all its rays, or a part of them): its threads form
// W for kPhase planes from whole z lines, read in aligned 16-byte words, and
// leave it in shared memory; then each ray takes its two z taps of W from
// there.  Against the gather's four unaligned loads per sample (two 128-byte
// lines each, which bound it) this reads each row of a plane once per column
// in whole lines, and a sample is one interpolation.  512^3 / 360 views: f32
// 35.2 -> 31.0 ms, bf16 31.6 -> 29.8 ms.  The L1 data pipe (76%; bf16 66%)
// and issue (63%; bf16 71%; 20.2 and 21.9 warp instructions per 32 samples, lines
// included) bound it at 16 warps per SM; 20 or 24 warps cost spills (34.8, 43.0 ms), two planes
// per step more barriers (37 ms), eight more registers (36.9 ms), and skipping
// the part of a line that no ray needs more than it saves (36.1 ms).

constexpr int kPhase = 4;            // planes per step
constexpr int kLineEdge = 4;         // words before (and after) a line in shared memory: zeros at its ends

template <typename T> struct Quad { using type = float4; };
template <> struct Quad<__nv_bfloat16> { using type = uint2; };
template <> struct Quad<__half> { using type = uint2; };
template <typename T> __device__ __forceinline__ float4 widen_quad(typename Quad<T>::type q)
{
    if constexpr (std::is_same<T, float>::value) return q;
    else
        return make_float4(widen<T>((unsigned short)(q.x & 0xffffu)), widen<T>((unsigned short)(q.x >> 16)),
                           widen<T>((unsigned short)(q.y & 0xffffu)), widen<T>((unsigned short)(q.y >> 16)));
}

template <typename T, int RAYS, bool SPL>
__global__ void __launch_bounds__(256, 2) gjp_forward_columns_kernel(
    const T *__restrict__ vol, VolParams V, const ViewParams *__restrict__ views, int nu, int nv, int n_vt, int n_views,
    int view_group, float *__restrict__ proj)
{
    using Q = typename Quad<T>::type;
    extern __shared__ __align__(16) float s_lines[];     // [2][kPhase][kLineEdge + nz + kLineEdge]
    int tile, view;
    block_tile_view(n_views, view_group, tile, view);
    const int nt = blockDim.x, tid = threadIdx.x;
    const int iu = tile / n_vt, iv0 = (tile % n_vt) * RAYS * nt + tid;   // rays iv0 + j nt
    const int nz = V.n[2], stride = nz + 2 * kLineEdge;

    Column c;
    {
        ViewParams vp;
        load_view(views, view, vp);
        c = make_column(vp, V, (float)iu - 0.5f * (float)(nu - 1));
    }
    const int m = c.m, nm = m == 0 ? V.n[0] : V.n[1], na = m == 0 ? V.n[1] : V.n[0];
    const int sm = (int)(m == 0 ? V.s[0] : V.s[1]), sa = (int)(m == 0 ? V.s[1] : V.s[0]);
    const int ic = (nm - 1) >> 1;
    int i0, i1, j0, j1;                                   // planes on which the column meets the grid
    plane_ranges(c.Pa, c.Ga, ic, na, nm, i0, i1, j0, j1);
    if (V.fov_r2 > 0.0f) {
        int lo, hi;
        fov_planes(V, m, ic, c.Pa, c.Ga, 0, 0, lo, hi);   // z plays no part
        i0 = max(i0, lo);
        i1 = min(i1, hi);
    }

    // rays: position on the next plane, increment (|.| < 1/2: it fits 32
    // fraction bits with its sign), and the planes on which some ray of the
    // warp meets the z range of the grid, and on which all do
    long long pb[RAYS];
    int gb[RAYS], any_lo[RAYS], any_hi[RAYS], all_lo[RAYS], all_hi[RAYS];
    float2 acc[RAYS], blk[RAYS];
#pragma unroll
    for (int j = 0; j < RAYS; ++j) {
        const long long v2 = 2 * min(iv0 + j * nt, nv - 1) - (nv - 1);   // twice the centred row
        const long long P = c.Z0 + ((v2 * c.Y0) >> (kPitchBits - 31)), G = c.Z1 + ((v2 * c.Y1) >> (kPitchBits - 31));
        int z0, z1, k0, k1;
        plane_ranges(P, G, ic, nz, nm, z0, z1, k0, k1);
        any_lo[j] = __reduce_min_sync(0xffffffffu, z0 <= z1 ? z0 : INT_MAX);
        any_hi[j] = __reduce_max_sync(0xffffffffu, z0 <= z1 ? z1 : -1);
        all_lo[j] = __reduce_max_sync(0xffffffffu, z0);
        all_hi[j] = __reduce_min_sync(0xffffffffu, z1);
        pb[j] = pos_at(P, G, i0, ic);
        gb[j] = (int)G;
        acc[j] = blk[j] = make_float2(0.0f, 0.0f);
    }
    for (int k = tid; k < 2 * kPhase * 2 * kLineEdge; k += nt) {     // the zeros at the lines' ends
        const int line = k / (2 * kLineEdge), e = k % (2 * kLineEdge);
        s_lines[line * stride + (e < kLineEdge ? e : nz + e)] = 0.0f;
    }

    unsigned long long pa = (unsigned long long)pos_at(c.Pa, c.Ga, i0, ic);
    const bool mine = 4 * tid < nz;
    int base = i0 * sm + 4 * tid;
    Q lo[kPhase], hi[kPhase];
    float da[kPhase];
    const auto fetch = [&](int i) {                       // rows of planes i .. i + kPhase - 1
        const bool inside = i >= j0 && i + kPhase - 1 <= min(i1, j1);   // both rows of every plane in the grid
        if (inside && mine) {
#pragma unroll
            for (int t = 0; t < kPhase; ++t) {
                da[t] = upper_weight<SPL>(frac_of(pa));
                const int off = base + floor_of(pa) * sa;
                const bool ok = taps_in_grid(i + t, floor_of(pa), 4 * tid + 2, nm, na, nz);   // debug build only
                lo[t] = ok ? __ldg(reinterpret_cast<const Q *>(vol + off)) : Q{};
                hi[t] = ok ? __ldg(reinterpret_cast<const Q *>(vol + (off + sa))) : Q{};
                pa += (unsigned long long)c.Ga;
                base += sm;
            }
        } else {
#pragma unroll
            for (int t = 0; t < kPhase; ++t) {
                const int ia = floor_of(pa);
                da[t] = upper_weight<SPL>(frac_of(pa));
                const bool in = mine && i + t <= i1;
                const int off = base + ia * sa;
                lo[t] = in && ia >= 0 ? __ldg(reinterpret_cast<const Q *>(vol + off)) : Q{};
                hi[t] = in && ia + 1 < na ? __ldg(reinterpret_cast<const Q *>(vol + (off + sa))) : Q{};
                pa += (unsigned long long)c.Ga;
                base += sm;
            }
        }
    };
    // one ray's samples of a phase; CLAMP: outside the z range both taps are a line's end zeros
    const auto sample = [&](const float *lines, long long &pos, int step, float2 &sum, auto clamp) {
#pragma unroll
        for (int t = 0; t < kPhase; t += 2) {
            const long long p0 = pos, p1 = pos + step;
            int z0 = floor_of((unsigned long long)p0), z1 = floor_of((unsigned long long)p1);
            if (decltype(clamp)::value) {
                z0 = min(max(z0, -2), nz);
                z1 = min(max(z1, -2), nz);
            }
            z0 = checked_line_tap(z0, nz, kLineEdge);
            z1 = checked_line_tap(z1, nz, kLineEdge);
            const float *l0 = lines + t * stride + z0, *l1 = lines + (t + 1) * stride + z1;
            const float2 lower = make_float2(l0[0], l1[0]), upper = make_float2(l0[1], l1[1]);
            const float2 d = __ffma2_rn(lower, make_float2(-1.0f, -1.0f), upper);
            sum = __fadd2_rn(sum, __ffma2_rn(upper_weight2<SPL>((unsigned long long)p0, (unsigned long long)p1), d, lower));
            pos = p1 + step;
        }
    };
    if (i0 <= i1) fetch(i0);
    int buf = 0, phases = 0;
    for (int i = i0; i <= i1; i += kPhase) {
        float *lines = s_lines + buf * kPhase * stride + kLineEdge;
        if (mine) {
#pragma unroll
            for (int t = 0; t < kPhase; ++t) {
                const float4 a = widen_quad<T>(lo[t]), b = widen_quad<T>(hi[t]);
                const float2 m1 = make_float2(-1.0f, -1.0f), w = make_float2(da[t], da[t]);
                const float2 x = make_float2(a.x, a.y), y = make_float2(a.z, a.w);
                const float2 p = __ffma2_rn(w, __ffma2_rn(x, m1, make_float2(b.x, b.y)), x);
                const float2 q = __ffma2_rn(w, __ffma2_rn(y, m1, make_float2(b.z, b.w)), y);
                *reinterpret_cast<float4 *>(lines + t * stride + 4 * tid) = make_float4(p.x, p.y, q.x, q.y);
            }
        }
        __syncthreads();        // lines complete; every warp is done with the other buffer's last lines
        if (i + kPhase <= i1) fetch(i + kPhase);
#pragma unroll
        for (int j = 0; j < RAYS; ++j) {
            if (i >= all_lo[j] && i + kPhase - 1 <= all_hi[j])
                sample(lines, pb[j], gb[j], blk[j], std::false_type{});
            else if (i <= any_hi[j] && i + kPhase - 1 >= any_lo[j])
                sample(lines, pb[j], gb[j], blk[j], std::true_type{});
            else
                pb[j] += (long long)kPhase * gb[j];
        }
        buf ^= 1;
        if ((++phases % (16 / kPhase)) == 0) {            // 16 planes: join the total
#pragma unroll
            for (int j = 0; j < RAYS; ++j) {
                acc[j] = __fadd2_rn(acc[j], blk[j]);
                blk[j] = make_float2(0.0f, 0.0f);
            }
        }
    }
    const float hm = m == 0 ? V.h[0] : V.h[1], ha = m == 0 ? V.h[1] : V.h[0];
    const float ga = ha * (__ll2float_rn(c.Ga) * 2.3283064365386963e-10f);
#pragma unroll
    for (int j = 0; j < RAYS; ++j) {
        const int iv = iv0 + j * nt;
        if (iv >= nv) break;
        const float2 s = __fadd2_rn(acc[j], blk[j]);
        const float gz = V.h[2] * ((float)gb[j] * 2.3283064365386963e-10f);
        proj[((size_t)view * nv + iv) * nu + iu] = (s.x + s.y) * sqrtf(hm * hm + ga * ga + gz * gz);
    }
}

// Whether the column form is the faster forward.  A thread's plane costs
// about 1.8 samples for its part of the line plus one per ray, so idle lanes
// (lines of nz / 4 threads or rays that do not fill the warps) show in
// `cost`, 1 for full ones.  Measured against the gather (with its deeper
// loads and paired copies), gather -> columns:
//   float32: 512^3 / 360 views 35.2 -> 31.0 ms, 8 views 1.15 -> 0.81 ms; 256^3 / 180 views
//     2.35 -> 1.98 ms; 128^3 / 32 views 87 -> 71 us; 512x512x128 / 60 views 1.93 -> 1.27 ms;
//     448^3 / 60 views (cost 1.14) 4.76 -> 4.14 ms; 320^3 / 120 views (1.20) 3.02 -> 3.36 ms;
//     400^3 with 600^2 pixels / 50 views (1.15) 5.35 -> 5.78 ms.
//   16-bit: 512^3 / 360 views 31.6 -> 29.8 ms, 16 views 2.27 -> 1.43 ms; 1024^3 / 60 views
//     53.1 -> 43.5 ms; 448^3 / 60 views (1.14) 4.12 -> 4.13 ms; 384x384x256 / 60 views (1.00)
//     1.44 ms in columns.  Grids up to 2^25 voxels keep the z-paired copy, not for their time
//     (320x320x256 / 60 views 1.21 -> 1.01 ms, 256^3 / 180 views 2.24 -> 1.96): calls rely on
//     AUTO's bits and on a batch's launch count there.
// Beyond the limits (not taken): float32 600x600x320 / 24 views (1.20) 2.92 -> 2.41 ms, 400^3 /
// 50 views (1.28) 2.79 -> 2.76, 320^3 / 60 views (1.20) 1.59 -> 1.70, 200^3 / 90 views (1.28)
// 0.66 -> 0.72; bf16 600x600x320 2.94 -> 2.39, 700^3 / 12 views (1.10) 4.16 -> 3.70, 448^3 /
// 48 views (1.14) 3.37 -> 3.30, 320^3 / 60 views 1.49 -> 1.71.
// Fewer than 2048 warps leave SMs idle (256^3, f32: one view 34 us for the gather, 56 us for
// columns; two views 45, 56; four 70, 60).  Float32 grids up to 2^22 voxels keep the gather,
// with which AUTO agrees bit for bit there.
bool forward_columns_pay(const int64_t n[3], int nu, int nv, int n_views, gjp_dtype dt, const void *vol)
{
    if (n[2] % 4 != 0 || n[2] < 112 || n[2] > 1024 || n_views > 65535 || !fits_int32(n)) return false;
    if (reinterpret_cast<uintptr_t>(vol) % (dt == GJP_F32 ? 16 : 8) != 0) return false;
    const ColumnShape c = column_shape(nv, (int)n[2]);
    if ((double)n_views * nu * c.parts * (c.threads / 32) < 2048.0) return false;
    const double voxels = (double)n[0] * n[1] * n[2];
    const double cost = c.parts * c.threads * (1.8 + c.rays) / (1.45 * nv);
    if (dt == GJP_F32) return voxels > 4194304.0 && (cost <= 1.06 || (cost <= 1.16 && voxels >= 8.5e7));
    return cost <= 1.06 && voxels > 33554432.0;
}

template <typename T>
cudaError_t launch_columns(const T *vol, const VolParams &V, const ViewParams *table, const GatherShape &sh, float *proj,
                           cudaStream_t s)
{
    const ColumnShape c = column_shape(sh.nv, V.n[2]);
    const dim3 grid((unsigned)(c.parts * sh.nu), (unsigned)sh.n_views);
    const size_t smem = (size_t)2 * kPhase * (V.n[2] + 2 * kLineEdge) * sizeof(float);
#define GJP_COLUMNS(R, S)                                                                                          \
    gjp_forward_columns_kernel<T, R, S><<<grid, c.threads, smem, s>>>(vol, V, table, sh.nu, sh.nv, c.parts, sh.n_views, \
                                                                      sh.view_group, proj)
    switch (c.rays) {
    case 4: if (sh.spl) GJP_COLUMNS(4, true); else GJP_COLUMNS(4, false); break;
    case 5: if (sh.spl) GJP_COLUMNS(5, true); else GJP_COLUMNS(5, false); break;
    default: if (sh.spl) GJP_COLUMNS(6, true); else GJP_COLUMNS(6, false); break;
    }
#undef GJP_COLUMNS
    return cudaGetLastError();
}

cudaError_t forward_columns(const void *vol, gjp_dtype dt, const VolParams &V, const ViewParams *table,
                            const GatherShape &sh, float *proj, cudaStream_t s)
{
    switch (dt) {
    case GJP_F32: return launch_columns<float>(static_cast<const float *>(vol), V, table, sh, proj, s);
    case GJP_BF16: return launch_columns<__nv_bfloat16>(static_cast<const __nv_bfloat16 *>(vol), V, table, sh, proj, s);
    default: return launch_columns<__half>(static_cast<const __half *>(vol), V, table, sh, proj, s);
    }
}

}  // namespace gjp_detail
