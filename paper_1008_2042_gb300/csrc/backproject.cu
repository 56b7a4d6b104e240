// Exact adjoint P^T of the Siddon projector: f_j = sum_i a_ij g_i with the same a_ij.
//
// The paper replaces the adjoint by the closed form of Eq. (3) because a ray-driven
// scatter would make threads collide on voxels (Section 2.2.2). Here the exact transpose
// is computed as a gather: each thread owns one (x, y) voxel column and a chunk of ZC
// consecutive z voxels and, for every view, visits exactly the rays that can cross it.
// The geometry separates: ray (u, v) meets column (ix, iy) over a tau interval [ta, tb]
// that depends on u only, and meets z slab k over an interval that depends on v only, so
//   a_ij = |D - S| * max(0, min(tb, tz1(v)) - max(ta, tz0(v))).
// Candidate imager columns u come from the shadow of the voxel column's corners. For one
// u, almost every row whose ray reaches slab k stays inside it across the whole column
// and so has weight (tb - ta): those rows form a contiguous range and are summed at once
// from per-column prefix sums over rows (k_row_prefix); only the rows whose ray crosses
// a z plane inside the column (about 0.1 per plane at the paper's sizes) are evaluated
// one by one. The factor |D - S| is folded into the table, which holds for every row m
// the pair (prefix of the rows below m, value of row m): one 8-byte load per plane gives
// both the window's prefix and its straddling row. The crossing parameters come from the
// same plane coordinates and reciprocals as the projector's, so both operators use the same
// weights to FP32 rounding. No atomics: the result is independent of scheduling.
//
// What bounds it on the paper's finest grid (512x512x70, 40 views, 1.18 ms, 14 voxels per
// thread): issue slots 80% (1.14e9 warp instructions, three fifths of them the plane loop's) and
// L1 data wavefronts 67% (the table's lines: lanes of a patch read about ten sectors). Before the
// straddling row became one saturating multiply and the chunks whole it took 1.63 ms, with
// the plane heights computed for each plane 1.25 ms; with the warps of a block on the same
// patch taking turns at the views, 128x128x18 takes 103 us (200 before), 64x64x16 21 us (61).
// Chunks that begin or end at z = 0 take the loops of one side where the middle plane rounds to 0 (see bp_plan):
// 256x256x64 457 -> 395 us, 128x128x32 145 -> 119 us.
#include "cbct_internal.cuh"

#include <math_constants.h>

#include <cmath>

namespace cbct {

// Thread mapping: each warp takes an 8 x 4 patch of voxel columns and a block stacks patches two
// wide. Lanes whose columns are close in both x and y read nearby table entries in every view
// (a voxel's imager column moves with x at some views and with y at others): an 8 x 4 patch
// touches 10 sectors per table request where a 32 x 1 row touched 16, and the warps of a
// block share their lines in L1. Where the grid has too few columns to fill the chip, the
// warps of a block also split the views: `slices` warps take the same patch and every
// slices-th view each, and their sums are added in a fixed order through shared memory.
constexpr int BP_WX = 8, BP_WY = 4; // warp patch

// A launch: zc voxels per thread (an instantiation), warps per block and view slices per patch; a
// block holds warps / slices patches, two wide. The last chunk of a
// column ends at its top and so may overlap the one before, which keeps the voxels they share:
// every chunk is whole, and the plane loop needs no test of where it ends.
struct BpPlan {
    int zc, warps, slices;
    int bx, by; // columns of a block's tile
    dim3 grid;
};
constexpr int BP_MAX_WARPS = 16;
constexpr int BP_ZC[] = {8, 12, 14, 16, 18};

// The voxels per thread that cover a column at the least cost: its planes, two more per chunk for
// its first plane and set-up, a sixteenth more for a chunk that z = 0 cuts (its rows are tested one by
// one) and 3% more for chunks of 16 and 18, which spill. Measured (8 | 12 | 14 | 16 | 18): 512x512x70
// 1464 | 1241 | 1177 | 1286 | 1241 us, 256x256x64 (meeting at z = 0 for 8 and 16 only) 507 | 490 | 462 | 393 | 487 us,
// 256x256x48 397 | 321 | 374 | 333 | 395 us, 512x512x30 356 | 342 | 380 | 327 | 358 us (20 views), 1000x1000x20 542 | 479 |
// 524 | 567 | 612 us (12 views). Where even 8 slices leave few warps, 8 voxels
// (64x64x16: 24.6 us, with 16 32.8 us). Slices double until the chip has about 96 warps per
// SM to draw from: 256x256x35 with 1 | 2 | 4 | 8 slices 403 | 354 | 339 | 356 us, 128x128x18 456 |
// 240 | 131 | 104 us, 512x512x70 1254 | 1311 | 1393 | 1583 us (less of the table is shared in L1).
//
// An even volume's middle plane is 0 only where nz / 2 dz and the corner round alike (always for pitches
// of few bits, for about a third of the usual ones). Elsewhere it is +-1e-6 mm, and one or both of the
// chunks that meet there count as cut: 256x256x56 360 us with dz = 1.0, 401 us with 1.7.
static BpPlan bp_plan(const GeomDev &G)
{
    BpPlan p{};
    const long long patches = (long long)((G.nx + BP_WX - 1) / BP_WX) * ((G.ny + BP_WY - 1) / BP_WY);
    const long long sms = device_sm_count();
    int chunks = 0;
    double best = 1e30;
    for (int zc : BP_ZC) {
        const int n = (G.nz + zc - 1) / zc;
        double cost = 0.0;
        for (int c = 0; c < n; ++c) {
            const int z = G.nz < zc ? 0 : c * zc < G.nz - zc ? c * zc : G.nz - zc;
            // (the kernel's own planes; it takes a lowest plane just above 0 for a cut one)
            const float bot = std::fmaf((float)z, G.dz, G.z0), top = std::fmaf((float)(z + zc), G.dz, G.z0);
            const bool cut = top > 0.0f && bot != 0.0f && bot < 1e-2f * G.dz;
            cost += (zc + 2.0) * (cut ? 17.0 / 16.0 : 1.0) * (zc >= 16 ? 1.03 : 1.0);
        }
        if (cost < best) {
            best = cost;
            p.zc = zc;
            chunks = n;
        }
    }
    if (patches * chunks * 8 < 16 * sms) {
        p.zc = BP_ZC[0];
        chunks = (G.nz + p.zc - 1) / p.zc;
    }
    p.warps = BP_MAX_WARPS;
    p.slices = 1;
    while (p.slices < 8 && patches * chunks * p.slices < 96 * sms && 2 * p.slices <= G.nviews) p.slices *= 2;
    const int patches_block = p.warps / p.slices;
    p.bx = 2 * BP_WX;
    p.by = patches_block / 2 * BP_WY;
    p.grid = dim3((G.nx + p.bx - 1) / p.bx, (G.ny + p.by - 1) / p.by, chunks);
    return p;
}

size_t prefix_table_bytes(const GeomDev &G) { return sizeof(float2) * (size_t)G.nviews * G.nu * ((size_t)G.nv + 1); }

int backproject_max_blocks(const GeomDev &G)
{
    // the smallest tile is two patches (8 slices of 16 warps), the smallest chunk 8 voxels
    return ((G.nx + 2 * BP_WX - 1) / (2 * BP_WX)) * ((G.ny + BP_WY - 1) / BP_WY) * ((G.nz + BP_ZC[0] - 1) / BP_ZC[0]);
}

// Rows whose ray, while inside the column (tau in [ta, tb], 1/(tc+ta) = A, 1/(tc+tb) = B),
// reaches the plane z = zp: v (tc + tau) = zp for some tau, i.e. v between zp*A and zp*B.
// Returned as a widened integer row range (may extend outside [0, nv-1]).
__device__ __forceinline__ void straddle_rows(const GeomDev &G, float zp, float A, float B, int &lo, int &hi)
{
    const float v0 = zp * A, v1 = zp * B;
    const float lim = (float)(G.nv + 1);
    const float flo = fminf(fmaxf(fmaf(fminf(v0, v1) - G.v_first, G.inv_dv, -1e-3f), -2.0f), lim);
    const float fhi = fminf(fmaxf(fmaf(fmaxf(v0, v1) - G.v_first, G.inv_dv, 1e-3f), -2.0f), lim);
    lo = (int)ceilf(flo);
    hi = (int)floorf(fhi);
}

// The planes of one visit to a voxel column: the ray column's entries of the prefix table `tab`
// (entry m at row_bytes * m, biased by ROUND_BIAS rows), 1 / v of the rows at shared address `iv`
// (biased likewise), the column's interval [ta, tb] with A = 1 / (tc + ta), B = 1 / (tc + tb).
constexpr int ROUND_BIAS = 0x4B400000; // bits of 1.5 * 2^23: what ceil by the FP adder leaves on top
struct BpVisit {
    const char *tab;
    unsigned iv;
    int row_bytes;
    float ta, tb, A, B;
};
// The chunk: its lowest plane (and in rows at unit scale), the plane pitch in rows at unit scale,
// the row coordinate of v = 0 minus the windows' margin, its voxels (ZC, or all nz < ZC).
struct BpChunk {
    float zbot, zs_bot, dzs, c0;
    int nzc;
    unsigned zpairs; // shared address of the heights of planes 1, 2, ..., ZC times SIDE
};

// Adds this visit's share of every voxel of the chunk. The rows that reach plane zp inside the
// column lie in the window [zp B, zp A] of v (zp >= 0; [zp A, zp B] below) and are at most one
// (the caller's `simple` test): row a, the first at or above the window's start. With the prefix
// P[a] of the rows below, plane z is passed by
//     (tb - ta) P[a_z] + below_z,   below_z = g_a * (part of [ta, tb] with row a below the plane),
// and slab z receives the difference of its two planes,
//     (tb - ta) ((P[a_{z+1}] - P[a_z]) + g_{z+1} f_{z+1} - g_z f_z),
// with f the fraction of [ta, tb] that row a spends below the plane. f comes from the
// crossing tau = zp / v - tc (rounded as the projector rounds it: subtracting tc + ta at once saves 1% of
// the time, but its error grows by a tenth) by one saturating multiply: where row a lies beyond the window, tau lies
// beyond [ta, tb] on the side where f is 0, so no test of the window's end is needed.
// SIDE +1 / -1: row a of every plane has v > 0 / v < 0 (it rises / falls); 0: tested per row.
// CLAMP: windows may leave the imager (rows clamped to [0, nv]; entry nv has value 0).
// FULL: the chunk has ZC voxels.
template <int ZC, int SIDE, bool CLAMP, bool FULL>
__device__ __forceinline__ void bp_planes(const GeomDev &G, const BpVisit &q, const BpChunk &c, float (&acc)[ZC])
{
    const float w = q.tb - q.ta, winv = __fdividef(1.0f, w);
    const float lo = SIDE < 0 ? q.A : q.B, x0 = fmaf(c.zs_bot, lo, c.c0), xs = c.dzs * lo;
    auto plane = [&](int z, float &P, float &g, float &f) {
        const float zp = fmaf((float)z, G.dz, c.zbot);
        float x;
        if (SIDE != 0) {
            x = fmaf((float)z, xs, x0);
        } else {
            const float zs = fmaf((float)z, c.dzs, c.zs_bot);
            x = fmaf(zs, zs >= 0.0f ? q.B : q.A, c.c0);
        }
        if (CLAMP) x = fminf(fmaxf(x, 0.0f), (float)G.nv);
        const int a = __float_as_int(__fadd_ru(x, 12582912.0f)); // ROUND_BIAS + ceil(x)
        const float2 T = __ldg(reinterpret_cast<const float2 *>(q.tab + (long long)a * q.row_bytes));
        const float iw = lds_float(q.iv + 4u * (unsigned)a);
        if (SIDE < 0) {
            f = __saturatef((q.tb - fmaf(zp, iw, -G.tc)) * winv);
        } else {
            f = __saturatef((fmaf(zp, iw, -G.tc) - q.ta) * winv);
        }
        if (SIDE == 0) {
            if (!(iw > 0.0f)) f = 1.0f - f;
        }
        P = T.x;
        g = f > 0.0f ? T.y : 0.0f; // (a row outside the window is not touched, whatever its value)
    };
    float P0, g0, f0;
    plane(0, P0, g0, f0);
    if constexpr (SIDE != 0 && FULL && !CLAMP) {
        static_assert(ZC % 2 == 0);
        constexpr bool LOOKUP = ZC > BP_ZC[0];
        // Two planes at a time. Longer chunks read the pair's heights from shared memory, one load
        // for both: the heights' arithmetic costs them issue slots and registers (512x512x70, 14
        // voxels: 1181 us, computed 1251 us; 512x512x128: 1991 | 2166 us). Chunks of 8 have the
        // registers and little to hide the load behind (64x64x16: 24.6 us, computed 22.6 us).
        const float tc = SIDE > 0 ? -G.tc : G.tc, edge = SIDE > 0 ? q.ta : -q.tb;
#pragma unroll
        for (int z = 0; z < ZC; z += 2) {
            const int a1 = __float_as_int(__fadd_ru(fmaf((float)(z + 1), xs, x0), 12582912.0f));
            const int a2 = __float_as_int(__fadd_ru(fmaf((float)(z + 2), xs, x0), 12582912.0f));
            const float2 T1 = __ldg(reinterpret_cast<const float2 *>(q.tab + (long long)a1 * q.row_bytes));
            const float2 T2 = __ldg(reinterpret_cast<const float2 *>(q.tab + (long long)a2 * q.row_bytes));
            float2 zp;
            if constexpr (LOOKUP) zp = lds_float2(c.zpairs + 4u * (unsigned)z);
            else zp = make_float2(SIDE * fmaf((float)(z + 1), G.dz, c.zbot), SIDE * fmaf((float)(z + 2), G.dz, c.zbot));
            const float t1 = fmaf(zp.x, lds_float(q.iv + 4u * (unsigned)a1), tc);
            const float t2 = fmaf(zp.y, lds_float(q.iv + 4u * (unsigned)a2), tc);
            const float f1 = __saturatef((t1 - edge) * winv), f2 = __saturatef((t2 - edge) * winv);
            const float g1 = f1 > 0.0f ? T1.y : 0.0f, g2 = f2 > 0.0f ? T2.y : 0.0f;
            acc[z] = fmaf(w, fmaf(-g0, f0, fmaf(g1, f1, T1.x - P0)), acc[z]);
            acc[z + 1] = fmaf(w, fmaf(-g1, f1, fmaf(g2, f2, T2.x - T1.x)), acc[z + 1]);
            P0 = T2.x;
            g0 = g2;
            f0 = f2;
        }
        return;
    }
#pragma unroll
    for (int z = 0; z < ZC; ++z) {
        if (!FULL && z >= c.nzc) break;
        float P1, g1, f1;
        plane(z + 1, P1, g1, f1);
        acc[z] = fmaf(w, fmaf(-g0, f0, fmaf(g1, f1, P1 - P0)), acc[z]);
        P0 = P1;
        g0 = g1;
        f0 = f1;
    }
}

// Register budget: 64, two resident blocks of 512 threads (chunks of 18 voxels spill 56-64 bytes, those of 16 four).
// FLAT: each lane walks its own list of candidates (view, imager column), so a warp runs for the
// longest per-lane total instead of the widest shadow in every view: fewer idle lanes where
// shadows are about one column wide.
template <int ZC, bool FLAT>
__global__ void __launch_bounds__(32 * BP_MAX_WARPS, 2)
k_backproject(GeomDev G, const float2 *__restrict__ ps, float *__restrict__ out, int sx, int sy, int sz, int slices, float span_lim,
              float *__restrict__ out2, double *__restrict__ partials, Scalars *__restrict__ sc, int fin_op, int scale_q)
{
    // 1 / v per imager row (one more for entry nv); the same with -inf where v >= 0, for falling chunks; the slices' sums
    extern __shared__ float smem[];
    __shared__ double s_warp[BP_MAX_WARPS];
    float *s_invv = smem, *s_sum = smem + 2 * (G.nv + 1);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i <= G.nv; i += blockDim.x) {
        const float v = imager_v(G, i);
        s_invv[i] = v != 0.0f ? __frcp_rn(v) : 1e30f;
        s_invv[G.nv + 1 + i] = v < 0.0f ? __frcp_rn(v) : -CUDART_INF_F;
    }

    const int npatch = (blockDim.x >> 5) / slices, slice = warp / npatch, patch = warp - slice * npatch;
    const int bx = 2 * BP_WX, by = npatch / 2 * BP_WY;
    const int ix = blockIdx.x * bx + (patch & 1) * BP_WX + lane % BP_WX;
    const int iy = blockIdx.y * by + (patch >> 1) * BP_WY + lane / BP_WX;
    const int iz0 = max(0, min((int)blockIdx.z * ZC, G.nz - ZC)), iz_own = blockIdx.z * ZC; // first voxel; first that is stored
    const bool ok = ix < G.nx && iy < G.ny;
    float acc[ZC];
#pragma unroll
    for (int z = 0; z < ZC; ++z) acc[z] = 0.0f;

    const float xl = plane_at(ix, G.dx, G.x0), xh = plane_at(ix + 1, G.dx, G.x0);
    const float yl = plane_at(iy, G.dy, G.y0), yh = plane_at(iy + 1, G.dy, G.y0);
    BpChunk ch;
    ch.nzc = min(ZC, G.nz);
    ch.zbot = plane_at(iz0, G.dz, G.z0);
    ch.zs_bot = ch.zbot * G.inv_dv;
    ch.dzs = G.dz * G.inv_dv;
    ch.c0 = fmaf(-G.v_first, G.inv_dv, -1e-3f);
    __shared__ __align__(8) float s_z[2][ZC];
    if (tid < ZC) {
        const float z = plane_at(iz0 + 1 + tid, G.dz, G.z0);
        s_z[0][tid] = z;
        s_z[1][tid] = -z;
    }
    const float ztop = plane_at(iz0 + ch.nzc, G.dz, G.z0), zs_top = ztop * G.inv_dv;
    const float zabs = fmaxf(fabsf(ch.zbot), fabsf(ztop));
    const float c1 = fmaf(-G.v_first, G.inv_dv, 1e-3f);
    const size_t view_stride = ((size_t)G.nv + 1) * G.nu;
    const unsigned iv0 = smem_u32(s_invv) - 4u * (unsigned)ROUND_BIAS;
    // Side +1: the window of the lowest plane, hence of every plane, starts at a row with
    // v / dv >= zs B - 1e-3; where the first row from -1e-3 on has v > 0, z = 0 will do.
    const float zs_rise = ch.zs_bot == 0.0f && imager_v(G, (int)ceilf(ch.c0)) > 0.0f ? 1.0f : ch.zs_bot;

    // imager columns in the shadow of the voxel column in view k (its corners' u); the least and
    // greatest u / sdd, scaled once (scaled corner by corner 1181 us at 512x512x70, so 1163)
    auto shadow = [&](int k, int &lo, int &hi) {
        const float2 cs = G.cs[k];
        float umin = 3.0e38f, umax = -3.0e38f;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float px = (c & 1) ? xh : xl, py = (c & 2) ? yh : yl;
            const float a = fmaf(-px, cs.y, py * cs.x);
            const float w = fmaf(-px, cs.x, fmaf(-py, cs.y, G.sad));
            const float t = __fdividef(a, w);
            umin = fminf(umin, t);
            umax = fmaxf(umax, t);
        }
        lo = max(0, (int)ceilf(fmaf(fmaf(umin, G.sdd, -G.u_first), G.inv_du, -1e-3f)));
        hi = min(G.nu - 1, (int)floorf(fmaf(fmaf(umax, G.sdd, -G.u_first), G.inv_du, 1e-3f)));
    };
    // all rows of imager column iu in view k that cross this voxel column
    auto visit = [&](int k, int iu) {
        const float4 r4 = __ldg(G.ray4 + k * G.nu + iu); // (dxr, dyr, qx, qy)
        const float2 r2 = __ldg(G.ray2 + k * G.nu + iu); // (1/dxr, 1/dyr)
        const float t0 = tau_plane(xl, r4.z, r2.x), t1 = tau_plane(xh, r4.z, r2.x);
        const float t2 = tau_plane(yl, r4.w, r2.y), t3 = tau_plane(yh, r4.w, r2.y);
        const float ta = fmaxf(fminf(t0, t1), fminf(t2, t3));
        const float tb = fminf(fmaxf(t0, t1), fmaxf(t2, t3));
        if (!(tb > ta)) return;
        const float A = __fdividef(1.0f, G.tc + ta), B = __fdividef(1.0f, G.tc + tb);
        const size_t entry = (size_t)k * view_stride + iu; // row m's entry: ps[entry + m * nu]
        // Plane z = zp is reached by the rows with v between zp*A and zp*B. While that
        // window is shorter than a row pitch and adjacent planes' windows are apart,
        // every row crosses at most one plane inside the column (the usual case; span_lim is 1
        // row, or 0 where the plane loop's row step does not fit, see the launcher).
        const float span = zabs * (A - B) * G.inv_dv;
        if (span + 3e-3f < span_lim && fmaf(G.dz * B, G.inv_dv, -span) > 3e-3f) {
            BpVisit q;
            q.iv = iv0;
            q.ta = ta;
            q.tb = tb;
            q.A = A;
            q.B = B;
            // row-window bounds at the lowest and highest plane of the chunk (monotone
            // in the plane height, so these bound every plane's window)
            const bool inside = fmaf(ch.zs_bot, ch.zs_bot >= 0.0f ? B : A, ch.c0) >= 0.0f &&
                                fmaf(zs_top, zs_top >= 0.0f ? A : B, c1) <= (float)(G.nv - 1);
            // Side -1: every plane has z <= 0. A row at a window's start then has v < 0, or lies beyond the
            // window with v >= 0, where -inf instead of 1 / v gives it no part (at z = 0 as well: 0 * inf
            // saturates to 0).
            const int side = !inside ? 0 : zs_rise * B > 2e-3f ? 1 : zs_top <= 0.0f ? -1 : 0;
            q.row_bytes = 8 * G.nu;
            q.tab = reinterpret_cast<const char *>(ps + entry) - (long long)ROUND_BIAS * q.row_bytes;
            if (ch.nzc == ZC) {
                if (side > 0) {
                    ch.zpairs = smem_u32(s_z[0]);
                    bp_planes<ZC, 1, false, true>(G, q, ch, acc);
                } else if (side < 0) {
                    ch.zpairs = smem_u32(s_z[1]);
                    q.iv += 4u * (unsigned)(G.nv + 1);
                    bp_planes<ZC, -1, false, true>(G, q, ch, acc);
                } else {
                    bp_planes<ZC, 0, true, true>(G, q, ch, acc);
                }
            } else {
                bp_planes<ZC, 0, true, false>(G, q, ch, acc);
            }
        } else {
            const float2 *col = ps + entry;
            const float wfull = tb - ta;
            int lo_p, hi_p;
            straddle_rows(G, ch.zbot, A, B, lo_p, hi_p);
#pragma unroll
            for (int z = 0; z < ZC; ++z) {
                if (z >= ch.nzc) break;
                const float z0 = plane_at(iz0 + z, G.dz, G.z0), z1 = plane_at(iz0 + z + 1, G.dz, G.z0);
                int lo_n, hi_n;
                straddle_rows(G, z1, A, B, lo_n, hi_n);
                float a = acc[z];
                const int f0 = max(hi_p + 1, 0), f1 = min(lo_n - 1, G.nv - 1);
                if (f0 <= f1) {
                    const float P1 = __ldg(col + (f1 + 1) * G.nu).x, P0 = __ldg(col + f0 * G.nu).x;
                    a = fmaf(wfull, P1 - P0, a);
                }
                // rows that cross a z plane inside the column: exact overlap
                const int r0 = max(lo_p, 0), r1 = min(hi_n, G.nv - 1);
                for (int iv = r0; iv <= r1; ++iv) {
                    if (iv == f0 && f0 <= f1) { // already counted
                        iv = f1;
                        continue;
                    }
                    const float iw = s_invv[iv];
                    const float s0 = tau_zplane(z0, iw, G.tc), s1 = tau_zplane(z1, iw, G.tc);
                    const float lo = fmaxf(ta, fminf(s0, s1)), hi = fminf(tb, fmaxf(s0, s1));
                    if (hi > lo) a = fmaf(__ldg(col + iv * G.nu).y, hi - lo, a);
                }
                acc[z] = a;
                lo_p = lo_n;
                hi_p = hi_n;
            }
        }
    };

    chain_wait();
    __syncthreads();
    if (ok && FLAT) {
        // (the lane's list goes on across all views of its slice)
        int k = slice - slices, iu = 0, iu_hi = -1;
        for (;;) {
            while (iu > iu_hi && k < G.nviews) // next view with a non-empty shadow
                if ((k += slices) < G.nviews) shadow(k, iu, iu_hi);
            if (k >= G.nviews) break;
            visit(k, iu++);
        }
    } else if (ok) {
        for (int k = slice; k < G.nviews; k += slices) {
            int lo, hi;
            shadow(k, lo, hi);
            for (int iu = lo; iu <= hi; ++iu) visit(k, iu);
        }
    }

    // the slices' sums, in the slices' order
    if (slices > 1) {
        const int per = npatch * 32, at = patch * 32 + lane;
        if (slice > 0)
#pragma unroll
            for (int z = 0; z < ZC; ++z)
                s_sum[((slice - 1) * ZC + z) * per + at] = acc[z];
        __syncthreads();
        if (slice == 0)
            for (int q = 0; q + 1 < slices; ++q)
#pragma unroll
                for (int z = 0; z < ZC; ++z)
                    acc[z] += s_sum[(q * ZC + z) * per + at];
    }
    double red = 0.0;
    if (ok && slice == 0) {
        const long long base = (long long)ix * sx + (long long)iy * sy;
#pragma unroll
        for (int z = 0; z < ZC; ++z) {
            if (iz0 + z >= iz_own && iz0 + z < G.nz) {
                const long long o = base + (long long)(iz0 + z) * sz;
                out[o] = acc[z];
                if (out2) out2[o] = acc[z];
                red += (double)acc[z] * (double)acc[z];
            }
        }
    }
    if (partials) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) red += __shfl_down_sync(0xffffffffu, red, o);
        if ((tid & 31) == 0) s_warp[tid >> 5] = red;
        __syncthreads();
        const unsigned blocks = gridDim.x * gridDim.y * gridDim.z;
        bool last = false;
        if (tid == 0) {
            double t = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += s_warp[w];
            partials[((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = t;
            last = last_to_arrive(sc, blocks);
        }
        if (__syncthreads_or(last)) {
            double t = sum_partials(partials, blocks, tid, blockDim.x);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
            if ((tid & 31) == 0) s_warp[tid >> 5] = t;
            __syncthreads();
            if (tid == 0) {
                double sum = 0.0;
                for (int w = 0; w < (int)(blockDim.x >> 5); ++w) sum += s_warp[w];
                apply_sum(sc, sum, fin_op, scale_q);
            }
        }
    }
}

static const void *bp_kernel(int zc, bool flat)
{
    switch (zc) {
    case 18: return flat ? (const void *)&k_backproject<18, true> : (const void *)&k_backproject<18, false>;
    case 16: return flat ? (const void *)&k_backproject<16, true> : (const void *)&k_backproject<16, false>;
    case 14: return flat ? (const void *)&k_backproject<14, true> : (const void *)&k_backproject<14, false>;
    case 12: return flat ? (const void *)&k_backproject<12, true> : (const void *)&k_backproject<12, false>;
    default: return flat ? (const void *)&k_backproject<8, true> : (const void *)&k_backproject<8, false>;
    }
}

// The shared-memory opt-in of every instantiation, once per device: at most 66 KB of rows (nv <= 8192)
// and 34 KB of the slices' sums (7/8 of 512 threads, 18 voxels).
constexpr int BP_SMEM_LIMIT = 104 * 1024;
cbct_status backproject_prepare()
{
    static std::atomic<unsigned long long> done[sizeof(BP_ZC) / sizeof(int)][2];
    for (int i = 0; i < (int)(sizeof(BP_ZC) / sizeof(int)); ++i)
        for (int flat = 0; flat < 2; ++flat) {
            const cudaError_t e = smem_optin_once(bp_kernel(BP_ZC[i], flat != 0), BP_SMEM_LIMIT, done[i][flat]);
            if (e != cudaSuccess) return check_cuda(e, "backproject attribute");
        }
    return CBCT_OK;
}

cbct_status launch_backproject(const GeomDev &G, const float2 *ps, float *out, long long sx, long long sy,
                               long long sz, float *out2, double *partials, cudaStream_t st, Scalars *sc, int fin_op,
                               int scale_q)
{
    BpPlan p = bp_plan(G);
    // flatten the candidate loop where a voxel column's shadow spans about one imager
    // column (its diagonal, magnified at the rotation axis, below 1.5 pixels)
    const bool flat = sqrtf(G.dx * G.dx + G.dy * G.dy) * (G.sdd / G.sad) < 1.5f * G.du;
    const cbct_status r = backproject_prepare();
    if (r != CBCT_OK) return r;
    const size_t smem = sizeof(float) * (2 * ((size_t)G.nv + 1) + (size_t)(p.slices - 1) * p.zc * (p.warps / p.slices) * 32);
    // The plane loop steps through the table by rows of 8 nu bytes held in 32 bits. Rows of 2 GiB or
    // more take the row-by-row loop at every visit, whose offsets count entries ((nv + 1) nu of them).
    float span_lim = G.nu < 1 << 28 ? 1.0f : 0.0f;
    GeomDev g = G;
    int isx = (int)sx, isy = (int)sy, isz = (int)sz;
    void *args[] = {&g, &ps, &out, &isx, &isy, &isz, &p.slices, &span_lim, &out2, &partials, &sc, &fin_op, &scale_q};
    ProfToken tok = prof_start(CBCT_KERNEL_BACKPROJECT, st);
    const cudaError_t e = launch_chained(bp_kernel(p.zc, flat), p.grid, dim3(32u * p.warps), args, smem, st);
    prof_stop(tok, st);
    note_launch();
    if (e != cudaSuccess) cudaGetLastError(); // the error is returned, not left pending
    return check_cuda(e, "backproject launch");
}

// Prefix sums over imager rows of every (view k, imager column iu), stored row-major like
// the projections so that neighbouring lanes (columns) touch neighbouring addresses:
// ps[k][m][iu] = (P_m, w(m) g[k][m][iu]) for m = 0..nv, where P_m = sum_{iv < m} w(iv)
// g[k][iv][iu] and the second member is row m's own weighted value (0 at m = nv), with
// w = |D - S| if `prescale` (folds the ray length into the adjoint's input) and 1
// otherwise. The running sums are compensated (Neumaier) and rounded to FP32 once per
// entry, so a difference of two prefixes carries at most two roundings of the prefixes'
// magnitude. A block covers 32 columns (lanes, coalesced reads) of one view; its 16 warps
// take consecutive row chunks: pass 1 sums each chunk, the chunk offsets come from shared
// memory, pass 2 writes.
constexpr int PREFIX_WARPS = 16;

// Compensated FP32 summation (Neumaier): s + c carries the running sum to about twice
// FP32's precision. (FP64 arithmetic is much slower on this part.)
__device__ __forceinline__ void comp_add(float &s, float &c, float v)
{
    const float t = s + v;
    const bool s_big = fabsf(s) >= fabsf(v);
    c += ((s_big ? s : v) - t) + (s_big ? v : s);
    s = t;
}

// UPDATE: g is the CGLS residual r and first becomes r - alpha q (q stored as kappa q; FP32
// arithmetic, one rounding to the storage type), which saves a pass over r and q of its own.
template <typename T, bool UPDATE>
__global__ void __launch_bounds__(32 * PREFIX_WARPS)
k_row_prefix(GeomDev G, T *g, const T *__restrict__ q, const Scalars *__restrict__ sc, float2 *__restrict__ ps, int prescale)
{
    chain_wait();
    __shared__ float2 s_tot[PREFIX_WARPS][32];
    const int lane = threadIdx.x, w = threadIdx.y;
    const int k = blockIdx.y, iu = blockIdx.x * 32 + lane;
    const bool ok = iu < G.nu;
    const int chunk = (G.nv + PREFIX_WARPS - 1) / PREFIX_WARPS;
    const int r0 = min(G.nv, w * chunk), r1 = min(G.nv, r0 + chunk);
    float dxr = 0.f, dyr = 0.f;
    if (prescale && ok) {
        const float4 r4 = __ldg(G.ray4 + k * G.nu + iu);
        dxr = r4.x;
        dyr = r4.y;
    }
    const float step = UPDATE ? (float)(sc->alpha / sc->kappa) : 0.0f;
    const size_t first = (size_t)k * G.nv * G.nu + iu;
    T *src = g + first;
    float ts = 0.0f, tc = 0.0f;
    if (ok)
        for (int i0 = r0; i0 < r1; i0 += 4) { // four rows at a time: their loads go out together
            float val[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const size_t at = (size_t)min(i0 + i, r1 - 1) * G.nu;
                val[i] = UPDATE ? as_float(src[at]) : load_as_float(src + at);
                if (UPDATE) val[i] = fmaf(-step, load_as_float(q + first + at), val[i]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (i0 + i >= r1) break;
                if (UPDATE) {
                    T *at = src + (size_t)(i0 + i) * G.nu;
                    store_from_float(at, val[i]);
                    val[i] = as_float(*at);
                }
                if (prescale) val[i] *= ray_length(dxr, dyr, imager_v(G, i0 + i));
                comp_add(ts, tc, val[i]);
            }
        }
    s_tot[w][lane] = make_float2(ts, tc);
    __syncthreads();
    float rs = 0.0f, rc = 0.0f; // the chunks before this warp's
    for (int c = 0; c < w; ++c) {
        const float2 t = s_tot[c][lane];
        comp_add(rs, rc, t.x);
        rc += t.y;
    }
    if (!ok) return;
    float2 *dst = ps + (size_t)k * ((size_t)G.nv + 1) * G.nu + iu; // entry m at dst[m * nu]
#pragma unroll 4
    for (int iv = r0; iv < r1; ++iv) {
        float val = UPDATE ? as_float(src[(size_t)iv * G.nu]) : load_as_float(src + (size_t)iv * G.nu);
        if (prescale) val *= ray_length(dxr, dyr, imager_v(G, iv));
        dst[(size_t)iv * G.nu] = make_float2(rs + rc, val);
        comp_add(rs, rc, val);
    }
    if (w == PREFIX_WARPS - 1) dst[(size_t)G.nv * G.nu] = make_float2(rs + rc, 0.0f); // all rows
}

template <typename T>
static void row_prefix(const GeomDev &G, void *g, const void *q, const Scalars *sc, float2 *ps, int prescale, cudaStream_t st)
{
    const dim3 grid((G.nu - 1) / 32 + 1, G.nviews), block(32, PREFIX_WARPS); // (nu + 31 may pass 2^31)
    if (q)
        CBCT_TIMED(CBCT_KERNEL_OTHER, st,
                   launch_chained(k_row_prefix<T, true>, grid, block, 0, st, G, static_cast<T *>(g), static_cast<const T *>(q), sc, ps, prescale));
    else
        CBCT_TIMED(CBCT_KERNEL_OTHER, st,
                   launch_chained(k_row_prefix<T, false>, grid, block, 0, st, G, static_cast<T *>(g), nullptr, nullptr, ps, prescale));
}

cbct_status launch_update_prefix(const GeomDev &G, void *r, const void *q, const Scalars *sc, float2 *ps, int prescale,
                                 cudaStream_t st, int storage)
{
    if (storage == ST_BF16) row_prefix<__nv_bfloat16>(G, r, q, sc, ps, prescale, st);
    else if (storage == ST_F16) row_prefix<__half>(G, r, q, sc, ps, prescale, st);
    else row_prefix<float>(G, r, q, sc, ps, prescale, st);
    return check_cuda(cudaGetLastError(), "row prefix launch");
}

cbct_status launch_row_prefix(const GeomDev &G, const void *g, float2 *ps, int prescale, cudaStream_t st, int storage)
{
    return launch_update_prefix(G, const_cast<void *>(g), nullptr, nullptr, ps, prescale, st, storage); // (g is only read)
}

// The paper's own backprojector, Eq. (3): voxel-driven, for every view the imager value at
// the point u* where the ray through the voxel centre x meets the imager is taken by
// bilinear interpolation (zero outside the imager) and weighted by
// (dx dy dz / (du dv)) L^3(u*) / (L0 l^2(x)) with L0 = sdd, l = |x - S|, L = |u* - S|.
// With w the distance of x from the source along the central ray, L = l sdd / w, so the
// weight is (dx dy dz / (du dv)) l sdd^2 / w^3. It approximates the exact adjoint
// (Appendix 2). Thread per voxel, lanes along x (public x-fastest layout).
__global__ void __launch_bounds__(128)
k_backproject_eq3(GeomDev G, const float *__restrict__ g, float *__restrict__ f, float pref)
{
    const int ix = blockIdx.x * 32 + threadIdx.x, iy = blockIdx.y * 4 + threadIdx.y, iz = blockIdx.z;
    if (ix >= G.nx || iy >= G.ny) return;
    const float px = fmaf((float)ix + 0.5f, G.dx, G.x0);
    const float py = fmaf((float)iy + 0.5f, G.dy, G.y0);
    const float pz = fmaf((float)iz + 0.5f, G.dz, G.z0);
    const float sdd2 = G.sdd * G.sdd;
    float acc = 0.0f;
    for (int k = 0; k < G.nviews; ++k) {
        const float2 cs = G.cs[k];
        const float w = G.sad - fmaf(px, cs.x, py * cs.y);
        const float inv_w = 1.0f / w;
        const float u = G.sdd * fmaf(-px, cs.y, py * cs.x) * inv_w;
        const float v = G.sdd * pz * inv_w;
        const float fu = (u - G.u_first) * G.inv_du, fv = (v - G.v_first) * G.inv_dv;
        const float flu = floorf(fu), flv = floorf(fv);
        const int i0 = (int)flu, j0 = (int)flv;
        const float wu = fu - flu, wv = fv - flv;
        const float *gk = g + (size_t)k * G.nv * G.nu;
        float val = 0.0f;
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const int iu = i0 + a, iv = j0 + b;
                if (iu >= 0 && iu < G.nu && iv >= 0 && iv < G.nv)
                    val = fmaf((a ? wu : 1.0f - wu) * (b ? wv : 1.0f - wv), __ldg(gk + (size_t)iv * G.nu + iu), val);
            }
        const float dxs = fmaf(-G.sad, cs.x, px), dys = fmaf(-G.sad, cs.y, py);
        const float l = sqrtf(fmaf(dxs, dxs, fmaf(dys, dys, pz * pz)));
        acc = fmaf(pref * l * sdd2 * inv_w * inv_w * inv_w, val, acc);
    }
    f[((size_t)iz * G.ny + iy) * G.nx + ix] = acc;
}

cbct_status launch_backproject_eq3(const GeomDev &G, const float *g, float *f, float pref, cudaStream_t st)
{
    dim3 grid((G.nx + 31) / 32, (G.ny + 3) / 4, G.nz), block(32, 4);
    CBCT_TIMED(CBCT_KERNEL_BACKPROJECT, st, k_backproject_eq3<<<grid, block, 0, st>>>(G, g, f, pref));
    return check_cuda(cudaGetLastError(), "backproject_eq3 launch");
}

} // namespace cbct
