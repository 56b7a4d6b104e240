// Forward projector P (Eq. (1), Section 2.2.1: one ray per imager pixel, Siddon's exact
// ray tracing, g_i = sum_j a_ij f_j with a_ij the length of ray i inside voxel j).
//
// GB300 mapping. All rays of one view that hit the same imager column u share their
// transverse path through the (x, y) voxel columns; the imager row v only tilts them in
// z. The path of every (view, column) is a record of the grid's trace table
// (project_trace.cu). Along it the integral of slab k up to tau,
//     C_k(tau) = int f(column at tau', slab k) dtau',
// is piecewise linear, and a ray that leaves slab k for slab k' at tau contributes
// C_k(tau) - C_k'(tau): a row does work only where it crosses a z plane (about five times
// per ray at the paper's sizes), and the per-column work is done once per slab instead of
// once per row. So, group by group of SG columns, a block tabulates C_k at the column
// boundaries, and every row interpolates it at its crossings.
//
// A block is one producer warp and up to six consumer warps (whose threads own the imager
// rows), and works through several (view, column) items. The producer brings each group's
// z-lines by TMA, one group ahead and across items: the volume is a matrix of nx ny lines,
// and one gather4 instruction fetches the lines of four columns, so the copies cost no
// issue slots and no load/store wavefronts and their latency is hidden. The consumers turn
// the lines into the table in place: each lane takes a quad of slabs (16-byte shared
// accesses) and nb consecutive columns of the group; the 32 / QW parts of a quad sit in one
// warp, which turns the parts' sums into offsets with shuffles. Pairs of slabs share one
// instruction (fma.rn.f32x2; each half rounds like a scalar FMA).
// Accumulation is FP32; the epilogue can scale by |D - S|, form the CGLS residual and
// reduce squared norms in FP64 into one partial per block; the output is stored as FP32,
// BF16 or FP16.
//
// This header holds the kernel template; it is instantiated for each QW in the
// project_q*.cu units (compiled in parallel) and launched from project.cu.
#pragma once
#include "async.cuh"
#include "f32x2.cuh"
#include "project.cuh"

namespace cbct {

// Shared-memory accesses by 32-bit address (byte offsets are added to it in one instruction).
__device__ __forceinline__ ulonglong2 lds_quad(unsigned a)
{
    ulonglong2 v;
    asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts_quad(unsigned a, ulonglong2 v)
{
    asm volatile("st.shared.v2.u64 [%0], {%1, %2};" ::"r"(a), "l"(v.x), "l"(v.y) : "memory");
}
__device__ __forceinline__ f32x2 lds_pair(unsigned a)
{
    f32x2 v;
    asm volatile("ld.shared.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}

// The transverse ray shared by every row of imager column iu in a view, and the tau
// interval in which it crosses the volume's (x, y) footprint.
struct ColumnRay {
    float dxr, dyr, qx, qy, inv_x, inv_y, tau_in, tau_out;
    int sxs, sys;
    bool hit;
};
__device__ __forceinline__ ColumnRay column_ray(const GeomDev &G, int view, int iu)
{
    ColumnRay c;
    const float2 cs = G.cs[view];
    ray_xy(G, cs.x, cs.y, imager_u(G, iu), c.dxr, c.dyr, c.qx, c.qy);
    c.inv_x = safe_rcp(c.dxr);
    c.inv_y = safe_rcp(c.dyr);
    const float xa = tau_plane(G.x0, c.qx, c.inv_x), xb = tau_plane(plane_at(G.nx, G.dx, G.x0), c.qx, c.inv_x);
    const float ya = tau_plane(G.y0, c.qy, c.inv_y), yb = tau_plane(plane_at(G.ny, G.dy, G.y0), c.qy, c.inv_y);
    c.tau_in = fmaxf(fmaxf(fminf(xa, xb), fminf(ya, yb)), -G.tc);
    c.tau_out = fminf(fminf(fmaxf(xa, xb), fmaxf(ya, yb)), 1.0f - G.tc);
    c.hit = c.tau_in < c.tau_out;
    c.sxs = c.dxr > 0.0f ? 1 : -1;
    c.sys = c.dyr > 0.0f ? 1 : -1;
    return c;
}

// Phase 1 of a column (whole block, one barrier inside): the crossings of the ray with
// each plane family are increasing in tau, so every crossing's position in the merged order
// is its own index plus the number of crossings of the other family before it. Writes, for
// the nseg = nA + nB + 1 segments the ray spends in (x, y) voxel columns, sEnd[j] (the tau at
// which segment j ends) and sCol[j] (its column iy * nx + ix); sA (nx + 1
// floats), sB (ny + 1) and s_cnt (4 per warp) are scratch. Returns (nA, nB, ix_e, iy_e): the
// x- and y-plane crossings inside the volume and the column entered first.
__device__ __forceinline__ int4 trace_column(const GeomDev &G, const ColumnRay &ray, float *sA,
                                             float *sB, unsigned *s_cnt, float *sEnd, int *sCol, int tid, int nthr)
{
    const float dxr = ray.dxr, dyr = ray.dyr, qx = ray.qx, qy = ray.qy, inv_x = ray.inv_x, inv_y = ray.inv_y;
    const float tau_in = ray.tau_in, tau_out = ray.tau_out;
    const bool hit = ray.hit;
    const int sxs = ray.sxs, sys = ray.sys;
    // counts of the crossings before the entry point and inside the volume: per thread, then
    // one block-wide sum (the lists are written before the barrier of that sum)
    unsigned cnt4[4] = {0u, 0u, 0u, 0u}; // a_le, a_in, b_le, b_in
    for (int a = tid; a <= G.nx; a += nthr) {
        if (hit && dxr != 0.0f) {
            const float t = tau_plane(plane_at(dxr > 0.0f ? a : G.nx - a, G.dx, G.x0), qx, inv_x);
            sA[a] = t;
            cnt4[0] += t <= tau_in;
            cnt4[1] += t > tau_in && t < tau_out;
        }
    }
    for (int b = tid; b <= G.ny; b += nthr) {
        if (hit && dyr != 0.0f) {
            const float t = tau_plane(plane_at(dyr > 0.0f ? b : G.ny - b, G.dy, G.y0), qy, inv_y);
            sB[b] = t;
            cnt4[2] += t <= tau_in;
            cnt4[3] += t > tau_in && t < tau_out;
        }
    }
    // per-warp sums
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const unsigned v = __reduce_add_sync(0xffffffffu, cnt4[q]);
        if ((tid & 31) == 0) s_cnt[4 * (tid >> 5) + q] = v;
    }
    __syncthreads();
    int a_le = 0, a_in = 0, b_le = 0, b_in = 0;
    for (int wq = 0; wq < (nthr + 31) / 32; ++wq) {
        a_le += (int)s_cnt[4 * wq + 0];
        a_in += (int)s_cnt[4 * wq + 1];
        b_le += (int)s_cnt[4 * wq + 2];
        b_in += (int)s_cnt[4 * wq + 3];
    }
    const float *LA = sA + a_le, *LB = sB + b_le;
    const int nA = a_in, nB = b_in, nseg = nA + nB + 1;
    // the column entered first contains the midpoint of the first segment
    float e0 = tau_out;
    if (nA) e0 = fminf(e0, LA[0]);
    if (nB) e0 = fminf(e0, LB[0]);
    const float tm = 0.5f * (tau_in + e0);
    const int ix_e = min(max((int)floorf((fmaf(tm, dxr, qx) - G.x0) / G.dx), 0), G.nx - 1);
    const int iy_e = min(max((int)floorf((fmaf(tm, dyr, qy) - G.y0) / G.dy), 0), G.ny - 1);
    // The rank of a crossing in the other family's list: the planes of that family the ray has
    // passed at t, estimated from its transverse position and then moved to the exact count
    // (# LB[j] < t for an x crossing, # LA[i] <= t for a y crossing), which the lists decide.
    auto passed = [&](float pos, float o, float inv_h, int n, int sgn, int le) {
        const int k = (int)floorf((pos - o) * inv_h); // the plane at or below pos
        return sgn > 0 ? k + 1 - le : n - k - le;
    };
    const float inv_dx = 1.0f / G.dx, inv_dy = 1.0f / G.dy;
    for (int i = tid; i < nA; i += nthr) {
        const float t = LA[i];
        int nb = 0;
        if (nB) {
            nb = min(max(passed(fmaf(t, dyr, qy), G.y0, inv_dy, G.ny, sys, b_le), 0), nB);
            while (nb > 0 && !(LB[nb - 1] < t)) --nb;
            while (nb < nB && LB[nb] < t) ++nb;
        }
        const int r = i + nb;
        const int cx = min(max(ix_e + sxs * (i + 1), 0), G.nx - 1), cy = min(max(iy_e + sys * nb, 0), G.ny - 1);
        sEnd[r] = t;
        sCol[r + 1] = cy * G.nx + cx;
    }
    for (int j = tid; j < nB; j += nthr) {
        const float t = LB[j];
        int na = 0;
        if (nA) {
            na = min(max(passed(fmaf(t, dxr, qx), G.x0, inv_dx, G.nx, sxs, a_le), 0), nA);
            while (na > 0 && LA[na - 1] > t) --na;
            while (na < nA && LA[na] <= t) ++na;
        }
        const int r = j + na;
        const int cx = min(max(ix_e + sxs * na, 0), G.nx - 1), cy = min(max(iy_e + sys * (j + 1), 0), G.ny - 1);
        sEnd[r] = t;
        sCol[r + 1] = cy * G.nx + cx;
    }
    if (tid == 0) {
        sCol[0] = iy_e * G.nx + ix_e;
        sEnd[nseg - 1] = tau_out;
    }
    return make_int4(nA, nB, ix_e, iy_e);
}


// TMA gather of the z-lines of four columns (rows y.x .. y.w of the line matrix) into four
// consecutive line slots; dst is a 128-byte aligned shared address.
__device__ __forceinline__ void gather4_g2s(unsigned dst, const CUtensorMap *map, int4 y, unsigned long long *bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cta.global.tile::gather4.mbarrier::complete_tx::bytes "
                 "[%0], [%1, {%2, %3, %4, %5, %6}], [%7];\n" ::"r"(dst),
                 "l"(map), "r"(0), "r"(y.x), "r"(y.y), "r"(y.z), "r"(y.w), "r"(smem_u32(bar))
                 : "memory");
}
// one line by a bulk copy (bytes a multiple of 16, both addresses 16-byte aligned)
__device__ __forceinline__ void bulk_g2s(unsigned dst, const float *src, int bytes, unsigned long long *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// one value by an asynchronous copy; copies_arrive: this thread's arrival once its copies landed
__device__ __forceinline__ void copy4_async(unsigned dst, const float *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_arrive(unsigned long long *bar)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared.b64 [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
// barrier of the n consumer threads that also tells whether any of them passed `v`
__device__ __forceinline__ bool consumer_or(bool v, int n)
{
    unsigned r;
    asm volatile("{\n .reg .pred p, q;\n setp.ne.u32 q, %1, 0;\n bar.red.or.pred p, 1, %2, q;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(r)
                 : "r"((unsigned)v), "r"(n)
                 : "memory");
    return r != 0;
}

// tau at which a row (1 / v = inv_v) in slab k leaves it; never if k is outside the volume
__device__ __forceinline__ float next_crossing(const GeomDev &G, int k, float inv_v)
{
    return (unsigned)k < (unsigned)G.nz ? tau_zplane(plane_at(k + (inv_v > 0.0f), G.dz, G.z0), inv_v, G.tc) : P_INF;
}

// The table build of one lane's part of NB columns (an even number): lines at `at`, pitch lp4
// bytes, the lengths of the columns in pairs at `al`; p becomes the part's sums.
template <int NB>
__device__ __forceinline__ void build_part(unsigned at, unsigned lp4, unsigned al, bool store, ulonglong2 &p)
{
#pragma unroll
    for (int i0 = 0; i0 < NB; i0 += BUILD_BATCH) {
        ulonglong2 v[BUILD_BATCH], l4[BUILD_BATCH / 2]; // lines; the lengths of two columns each
#pragma unroll
        for (int i = 0; i < BUILD_BATCH; ++i)
            if (i0 + i < NB) v[i] = lds_quad(at + i * lp4);
#pragma unroll
        for (int i = 0; i < BUILD_BATCH / 2; ++i)
            if (i0 + 2 * i < NB) l4[i] = lds_quad(al + 8 * i0 + 16 * i);
#pragma unroll
        for (int i = 0; i < BUILD_BATCH; ++i)
            if (i0 + i < NB) {
                const f32x2 l2 = i & 1 ? l4[i / 2].y : l4[i / 2].x;
                p.x = fma2(v[i].x, l2, p.x);
                p.y = fma2(v[i].y, l2, p.y);
                if (store) sts_quad(at + i * lp4, p);
            }
        at += BUILD_BATCH * lp4;
    }
}

// Items (view, imager column, chunk of rows) first_item + blockIdx.x, + gridDim.x, ...: item i is
// chunk i / ncols of column col_first + i % ncols, whose record is rec[i % ncols]. (Unsigned: the last
// step of a block may pass 2^31.)
// Per group of sg segments of an item's trace the lines become the table in place,
// T[c][k] = sum of f(column, slab k) * length over the columns of c's part up to and
// including c, with the sums of the parts before in O[part][k] (O[PARTS] is the group's
// total); then each consumer thread (R imager rows) adds, for every z crossing of its rows
// inside the group, the interpolated table value of the slab left minus that of the slab
// entered, and at the group's end the total of the slab the row is in (every group starts
// from zero). One barrier of the consumers per group; two line buffers.
// QW: quads of slabs per warp in the table build (PARTS = 32 / QW parts of nb columns each).
// FILL_GATHER: lines by gather4; FILL_BULK: one bulk copy per line; FILL_PACKED: 4-byte copies
// by the producer's lanes.
template <int MODE, typename TP, int QW, int R, int FILL>
__global__ void __launch_bounds__(PROJ_THREADS + 32, CBCT_PROJ_MIN_BLOCKS)
k_project(GeomDev G, const __grid_constant__ CUtensorMap lines, const float *__restrict__ f, int zpitch, ProjPlan pl,
          const float *__restrict__ y, TP *__restrict__ out, double *__restrict__ partials, Scalars *__restrict__ sc,
          const float *__restrict__ rec, int col_first, unsigned ncols, unsigned nitems)
{
    constexpr int PARTS = 32 / QW;
    extern __shared__ __align__(128) float smem[];
    __shared__ double s_warp[PROJ_THREADS / 32];
    __shared__ __align__(16) float s_hdr[2][TRACE_HDR / 2]; // headers of the items in work
    __shared__ float s_gend[2];                              // tau at which a group ends
    __shared__ __align__(8) unsigned long long s_full[2], s_empty[2];
    __shared__ int s_give_up;
    const int sg = pl.sg, lp = pl.pitch, bsh = pl.nbuf - 1; // group s uses buffer s & bsh, its use number s >> bsh
    // a line of room (the line before a buffer's first may be read, not used), then [nbuf][sg][lp]
    // lines, then table
    float *sBuf = smem + (lp + 31) / 32 * 32;
    float2 *sLen = reinterpret_cast<float2 *>(sBuf + pl.nbuf * sg * lp); // [nbuf][sg] (length, length) of a column's segment
    float2 *sSeg = sLen + pl.nbuf * sg;                                  // [nbuf][sg] (tau at its start, 1 / length)
    float *sOff = reinterpret_cast<float *>(sSeg + pl.nbuf * sg);        // [nbuf][PARTS + 1][zp] part offsets
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nthr = blockDim.x - 32, nwarps = nthr >> 5; // consumers; the last warp is the producer
    const int tcap = trace_cap(G), rwords = trace_words(G);
    if (tid == 0) {
        s_give_up = 0;
        for (int b = 0; b < 2; ++b) {
            // the copies' transactions and the producer's own stores (and its lanes' 4-byte copies)
            mbar_init(&s_full[b], FILL == FILL_PACKED ? 34u : 2u);
            mbar_init(&s_empty[b], (unsigned)nwarps);
        }
    }
    chain_wait();
    __syncthreads();

    if (warp == nwarps) {
        // ---- producer: one group ahead of the consumers, through all items ----
        unsigned item = blockIdx.x;
        int g = 0, nitem = 0, nseg = 0;
        const float *r = nullptr;
        int4 col = make_int4(0, 0, 0, 0);          // four columns of the next group ...
        float4 end = make_float4(0.f, 0.f, 0.f, 0.f); // ... the tau at which they end ...
        float start = 0.0f;                        // ... and where the first begins
        float hdr = 0.0f;                          // lane's word of the item's header
        auto next_columns = [&]() { // (past the trace's end: unused values of the record)
            if (4 * lane < min(sg, tcap - g * sg)) {
                const float *e = r + TRACE_HDR + g * sg + 4 * lane;
                end = __ldg(reinterpret_cast<const float4 *>(e));
                start = __ldg(e - 1);
                col = __ldg(reinterpret_cast<const int4 *>(e + tcap));
            }
        };
        auto next_item = [&]() {
            r = rec + (size_t)(item % ncols) * rwords;
            if (lane < TRACE_HDR / 2) hdr = __ldg(r + lane);
        };
        next_item();
        next_columns();
        nseg = __shfl_sync(0xffffffffu, __float_as_int(hdr), 0);
        for (int s = 0;; ++s) {
            const int b = s & bsh, n = min(sg, nseg - g * sg), quads = (n + 3) / 4;
            if (s > bsh && !mbar_wait(&s_empty[b], ((s >> bsh) - 1) & 1, &s_give_up)) break;
            const unsigned dst = smem_u32(sBuf) + 4u * (unsigned)(b * sg * lp);
            if (lane == 0)
                mbar_arrive_expect_tx(&s_full[b], FILL == FILL_GATHER ? 16u * (unsigned)(quads * lp)
                                                  : FILL == FILL_BULK ? 16u * (unsigned)(quads * G.zp) : 0u);
            if (g == 0 && lane < TRACE_HDR / 2) s_hdr[nitem & 1][lane] = hdr;
            __syncwarp();
            const unsigned to = dst + (unsigned)lane * 16u * (unsigned)lp; // this lane's four line slots
            if (FILL == FILL_GATHER) {
                if (lane < quads) gather4_g2s(to, &lines, col, &s_full[b]);
            } else if (FILL == FILL_BULK) {
                if (lane < quads) {
                    bulk_g2s(to, f + (size_t)col.x * zpitch, 4 * G.zp, &s_full[b]);
                    bulk_g2s(to + 4 * lp, f + (size_t)col.y * zpitch, 4 * G.zp, &s_full[b]);
                    bulk_g2s(to + 8 * lp, f + (size_t)col.z * zpitch, 4 * G.zp, &s_full[b]);
                    bulk_g2s(to + 12 * lp, f + (size_t)col.w * zpitch, 4 * G.zp, &s_full[b]);
                }
            } else {
                for (int u = 0; u < n; ++u) {
                    const int c4 = u & 3, cu = c4 == 0 ? col.x : c4 == 1 ? col.y : c4 == 2 ? col.z : col.w;
                    const float *line = f + (size_t)__shfl_sync(0xffffffffu, cu, u >> 2) * zpitch;
                    for (int k = lane; k < G.nz; k += 32) copy4_async(dst + 4 * (u * lp + k), line + k);
                }
                copies_arrive(&s_full[b]);
            }
            if (lane == quads - 1) s_gend[b] = end.w; // (a record's tail repeats its last segment)
            if (lane < quads) {
                const float l0 = end.x - start, l1 = end.y - end.x, l2 = end.z - end.y, l3 = end.w - end.z;
                float4 *len = reinterpret_cast<float4 *>(sLen + b * sg + 4 * lane);
                len[0] = make_float4(l0, l0, l1, l1);
                len[1] = make_float4(l2, l2, l3, l3);
                float4 *seg = reinterpret_cast<float4 *>(sSeg + b * sg + 4 * lane);
                seg[0] = make_float4(start, __fdividef(1.0f, l0), end.x, __fdividef(1.0f, l1));
                seg[1] = make_float4(end.y, __fdividef(1.0f, l2), end.z, __fdividef(1.0f, l3));
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_full[b]);
            if (++g * sg >= nseg) {
                g = 0;
                ++nitem;
                item += gridDim.x;
                if (item >= nitems) break;
                next_item();
            }
            next_columns();
            if (g == 0) nseg = __shfl_sync(0xffffffffu, __float_as_int(hdr), 0);
        }
        return;
    }

    // ---- consumers ----
    const int h = lane / QW, qs = lane - h * QW; // this lane's part and quad of a warp's QW quads
    const int nq = G.zp >> 2;
    const unsigned a_buf = smem_u32(sBuf), a_len = smem_u32(sLen), a_seg = smem_u32(sSeg), a_off = smem_u32(sOff);
    const unsigned lp4 = 4 * lp, zp4 = 4 * G.zp, b_buf = sg * lp4, b_seg = 8 * sg, b_off = (PARTS + 1) * zp4;
    const float inv_dz = 1.0f / G.dz;
    const float kappa = (MODE == PM_Q_SCALED) ? (float)sc->kappa : 1.0f;
    constexpr bool PRESCALE = sizeof(TP) == 4;
    double red = 0.0;
    bool lost = false; // a wait of the block ran out: NaN rows from here on
    int s = 0, nitem = 0; // groups and items so far
    for (unsigned item = blockIdx.x; item < nitems; item += gridDim.x, ++nitem) {
        const int chunk = item / ncols;
        int kz[R];
        float inv_v[R], tzn[R], acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = 0.0f;
        int nseg = 0;
        float mx = 0.f, my = 0.f, cx = 0.f, cy = 0.f, dxy2 = 0.f;
        for (int g = 0; !lost && (g == 0 || g * sg < nseg); ++g, ++s) {
            const int j0 = g * sg, b = s & bsh;
            lost = !mbar_wait(&s_full[b], (s >> bsh) & 1, &s_give_up);
            if (g == 0) {
                // the item's trace (see k_trace_table) and the rows' z state
                const float4 a = *reinterpret_cast<const float4 *>(s_hdr[nitem & 1]);
                const float4 d = *reinterpret_cast<const float4 *>(s_hdr[nitem & 1] + 4);
                nseg = __float_as_int(a.x);
                const float tau_in = a.y;
                dxy2 = a.z;
                mx = d.x;
                my = d.y;
                cx = d.z;
                cy = d.w;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int iv = chunk * (R * nthr) + r * nthr + tid;
                    const float v = imager_v(G, iv);
                    inv_v[r] = v != 0.0f ? __frcp_rn(v) : 1e30f;
                    kz[r] = (int)floorf((v * (G.tc + tau_in) - G.z0) * inv_dz);
                    if (nseg == 0 || iv >= G.nv) kz[r] = -1;
                    tzn[r] = next_crossing(G, kz[r], inv_v[r]);
                    if (tzn[r] <= tau_in) { // the entry point already lies past that plane
                        kz[r] += inv_v[r] > 0.0f ? 1 : -1;
                        tzn[r] = next_crossing(G, kz[r], inv_v[r]);
                    }
                }
            }
            const int clast = min(sg, nseg - j0) - 1; // the group's last column
            const unsigned aT = a_buf + b * b_buf, aO = a_off + b * b_off, aLen = a_len + b * b_seg, aSeg = a_seg + b * b_seg;
            const int nb = pl.nb, inv_nb = pl.inv_nb;
            for (int qg = warp; qg * QW < nq && !lost; qg += nwarps) {
                const int q = min(qg * QW + qs, nq - 1);
                const bool mine = qg * QW + qs < nq;
                unsigned at = aT + h * nb * lp4 + 16 * q, al = aLen + 8 * h * nb;
                ulonglong2 p = make_ulonglong2(0ull, 0ull); // running sums of the quad (all bits 0: 0.0f)
                if (clast + 1 == 80 && nb == 80 / PARTS) {
                    build_part<80 / PARTS>(at, lp4, al, mine, p);
                } else if (clast + 1 == 112 && nb == 112 / PARTS) {
                    build_part<112 / PARTS>(at, lp4, al, mine, p);
                } else {
                    const int n = min(nb, clast + 1 - h * nb); // columns of this lane's part
                    for (int i = 0; i < n; ++i, at += lp4, al += 8) {
                        const ulonglong2 v = lds_quad(at);
                        const f32x2 l2 = lds_pair(al);
                        p.x = fma2(v.x, l2, p.x);
                        p.y = fma2(v.y, l2, p.y);
                        if (mine) sts_quad(at, p);
                    }
                }
                // sums of the parts before this one: shift by a part, then scan
                ulonglong2 x;
                x.x = __shfl_up_sync(0xffffffffu, p.x, QW);
                x.y = __shfl_up_sync(0xffffffffu, p.y, QW);
                if (h == 0) x = make_ulonglong2(0ull, 0ull);
#pragma unroll
                for (int d = QW; d < 32; d *= 2) {
                    const f32x2 tx = __shfl_up_sync(0xffffffffu, x.x, d), ty = __shfl_up_sync(0xffffffffu, x.y, d);
                    if (lane >= d) {
                        x.x = add2(x.x, tx);
                        x.y = add2(x.y, ty);
                    }
                }
                const unsigned ao = aO + h * zp4 + 16 * q;
                if (mine) sts_quad(ao, x);
                if (mine && h == PARTS - 1) sts_quad(ao + zp4, make_ulonglong2(add2(x.x, p.x), add2(x.y, p.y))); // the group's total
            }
            lost = consumer_or(lost, nthr); // the table is built
            if (lost) break;
            const float gend = s_gend[b];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if ((unsigned)kz[r] >= (unsigned)G.nz) continue; // not in the volume, or out of it
                const int dir = inv_v[r] > 0.0f ? 1 : -1;
                float a = acc[r];
                // The segment that holds a crossing: the x and y planes the ray has passed there,
                // from its transverse position (no search). At a near tie this may name the
                // neighbouring segment, which only moves a rounding-sized piece of length between
                // two adjacent columns.
                while (tzn[r] < gend) { // a z crossing inside this group
                    const float t = tzn[r];
                    const int c = min(max(floor_small(fmaf(t, mx, cx)) + floor_small(fmaf(t, my, cy)) - j0, 0), clast);
                    const float2 sl = lds_float2(aSeg + 8 * c);
                    const float w = __saturatef((t - sl.x) * sl.y); // (a 0 x inf of an empty segment saturates to 0)
                    const int part = (c * inv_nb) >> 16;
                    const bool first = c == part * nb; // of its part: the sums before it are zero
                    const unsigned at = aT + c * lp4 + 4 * kz[r], ao = aO + part * zp4 + 4 * kz[r]; // slab left
                    kz[r] += dir;
                    const bool in = (unsigned)kz[r] < (unsigned)G.nz;
                    const unsigned st = in ? 4 * dir : 0; // to the slab entered
                    float d0 = lds_float(at - lp4), d1 = lds_float(at), o = lds_float(ao);
                    const float e0 = lds_float(at - lp4 + st), e1 = lds_float(at + st), eo = lds_float(ao + st);
                    d0 -= in ? e0 : 0.0f;
                    d1 -= in ? e1 : 0.0f;
                    o -= in ? eo : 0.0f;
                    if (first) d0 = 0.0f;
                    a += fmaf(w, d1 - d0, d0) + o;
                    tzn[r] = next_crossing(G, kz[r], inv_v[r]);
                }
                if ((unsigned)kz[r] < (unsigned)G.nz) a += lds_float(aO + PARTS * zp4 + 4 * kz[r]);
                acc[r] = a;
            }
            // this warp is done with the buffer
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_empty[b]);
        }

        // ---- epilogue of the item ----
        const int column = col_first + (int)(item - chunk * ncols), view = column / G.nu, iu = column - view * G.nu;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int iv = chunk * (R * nthr) + r * nthr + tid;
            if (iv >= G.nv) continue;
            const size_t idx = ((size_t)view * G.nv + iv) * G.nu + iu;
            const float v = imager_v(G, iv), len = sqrtf(fmaf(v, v, dxy2));
            // rows whose lines never arrived are NaN (reported through sc)
            const float q = lost ? __int_as_float(0x7fc00000) : acc[r] * len;
            // FP32 storage keeps |D - S| folded into r and q (the adjoint then needs no
            // per-sample rescale); 16-bit storage keeps the bare values
            const float scl = PRESCALE ? len : 1.0f;
            if (MODE == PM_PLAIN) {
                store_from_float(out + idx, q);
            } else if (MODE == PM_Q_SCALED) {
                store_from_float(out + idx, q * scl * kappa);
                red += (double)q * (double)q;
            } else if (MODE == PM_RESID) {
                const float rr = __ldg(y + idx) - q;
                store_from_float(out + idx, rr * scl);
                red += (double)rr * (double)rr;
            }
        }
    }
    if (lost) { // once more with a limit for the two groups that may still be in flight
        if (tid == 0 && sc) atomicOr(&sc->flags, 2u);
        int waiting = 0;
        mbar_wait(&s_full[s & bsh], (s >> bsh) & 1, &waiting);
        if (bsh) mbar_wait(&s_full[(s + 1) & 1], ((s + 1) >> 1) & 1, &waiting);
    }
    if (MODE != PM_PLAIN) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) red += __shfl_down_sync(0xffffffffu, red, o);
        if (lane == 0) s_warp[warp] = red;
        consumer_or(false, nthr);
        bool last = false;
        if (tid == 0) {
            double t = 0.0;
            for (int w = 0; w < nwarps; ++w) t += s_warp[w];
            partials[blockIdx.x] = t;
            last = last_to_arrive(sc, gridDim.x);
        }
        if (consumer_or(last, nthr)) {
            double t = sum_partials(partials, gridDim.x, tid, nthr);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
            if (lane == 0) s_warp[warp] = t;
            consumer_or(false, nthr);
            if (tid == 0) {
                double sum = 0.0;
                for (int w = 0; w < nwarps; ++w) sum += s_warp[w];
                apply_sum(sc, sum, MODE == PM_RESID ? FIN_RR : FIN_ALPHA, 0);
            }
        }
    }
}

template <int MODE, typename TP, int QW> static const void *kernel_ptr(int rows, int fill)
{
    if (fill == FILL_GATHER)
        return rows == 2 ? reinterpret_cast<const void *>(&k_project<MODE, TP, QW, 2, FILL_GATHER>)
                         : reinterpret_cast<const void *>(&k_project<MODE, TP, QW, 1, FILL_GATHER>);
    if (fill == FILL_BULK) return reinterpret_cast<const void *>(&k_project<MODE, TP, QW, 2, FILL_BULK>);
    if constexpr (MODE == PM_PLAIN && sizeof(TP) == 4)
        return reinterpret_cast<const void *>(&k_project<MODE, TP, QW, 2, FILL_PACKED>);
    return nullptr;
}

template <int QW> const void *project_kernel(int mode, int storage, int rows, int fill)
{
    const int s = storage == ST_BF16 ? 1 : storage == ST_F16 ? 2 : 0;
    switch (mode * 3 + s) {
    case PM_PLAIN * 3 + 0: return kernel_ptr<PM_PLAIN, float, QW>(rows, fill);
    case PM_PLAIN * 3 + 1: return kernel_ptr<PM_PLAIN, __nv_bfloat16, QW>(rows, fill);
    case PM_PLAIN * 3 + 2: return kernel_ptr<PM_PLAIN, __half, QW>(rows, fill);
    case PM_Q_SCALED * 3 + 0: return kernel_ptr<PM_Q_SCALED, float, QW>(rows, fill);
    case PM_Q_SCALED * 3 + 1: return kernel_ptr<PM_Q_SCALED, __nv_bfloat16, QW>(rows, fill);
    case PM_Q_SCALED * 3 + 2: return kernel_ptr<PM_Q_SCALED, __half, QW>(rows, fill);
    case PM_RESID * 3 + 0: return kernel_ptr<PM_RESID, float, QW>(rows, fill);
    case PM_RESID * 3 + 1: return kernel_ptr<PM_RESID, __nv_bfloat16, QW>(rows, fill);
    case PM_RESID * 3 + 2: return kernel_ptr<PM_RESID, __half, QW>(rows, fill);
    default: return nullptr;
    }
}

} // namespace cbct
