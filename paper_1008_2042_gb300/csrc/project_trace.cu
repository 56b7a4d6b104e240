// The projector's trace table: phase 1 of every (view, imager column), stored so that the
// projections of a reconstruction read it instead of recomputing it (Section 2.2.1: the
// transverse part of every ray of an imager column is the same Siddon trace).
#include "project_kernel.cuh"

namespace cbct {

// The grid's trace table: one record per (view, imager column), a header (segments as an
// integer, 0 where the rays miss the volume; tau where the trace starts; |d|^2 of the transverse
// direction; mx, my, cx, cy of the segment index, below; the start again in the last word, so
// that it precedes the first end), then End[trace_cap] floats and Col[trace_cap] ints, of which
// the first nseg rounded up to 4 are written (the rounding tail with the last segment's values).
// The segment that holds tau is floor(tau mx + cx) + floor(tau my + cy): the x and y planes the
// ray has passed there. The trace depends on the geometry only, so a reconstruction builds it
// once per level and every projection of that level reads it.
__global__ void __launch_bounds__(PROJ_THREADS) k_trace_table(GeomDev G, float *__restrict__ traces, int col_first)
{
    chain_wait();
    extern __shared__ __align__(16) float smem[];
    const int cap = trace_cap(G);
    float *sEnd = smem;
    int *sCol = reinterpret_cast<int *>(sEnd + cap);
    unsigned *s_cnt = reinterpret_cast<unsigned *>(sCol + cap); // 4 per warp
    float *sA = reinterpret_cast<float *>(s_cnt + 4 * (PROJ_THREADS / 32));
    float *sB = sA + (G.nx + 1);
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int column = col_first + blockIdx.x, view = column / G.nu, iu = column - view * G.nu;
    const ColumnRay ray = column_ray(G, view, iu);
    const int4 tr = trace_column(G, ray, sA, sB, s_cnt, sEnd, sCol, tid, nthr);
    __syncthreads();
    const int nseg = ray.hit ? tr.x + tr.y + 1 : 0, n4 = (nseg + 3) & ~3;
    float *rec = traces + (size_t)blockIdx.x * trace_words(G);
    float *E = rec + TRACE_HDR;
    int *C = reinterpret_cast<int *>(E + cap);
    // streaming stores: the table is read back once per projection, not kept in L2
    for (int q = tid; q < n4; q += nthr) {
        __stcs(E + q, sEnd[min(q, nseg - 1)]);
        __stcs(C + q, sCol[min(q, nseg - 1)]);
    }
    if (tid == 0) {
        const float inv_dx = 1.0f / G.dx, inv_dy = 1.0f / G.dy;
        const float fx = (ray.qx - G.x0) * inv_dx - (float)tr.z, fy = (ray.qy - G.y0) * inv_dy - (float)tr.w;
        const bool sx = ray.dxr != 0.0f, sy = ray.dyr != 0.0f; // a ray along an axis passes no plane of it
        float4 *hd = reinterpret_cast<float4 *>(rec);
        __stcs(hd, make_float4(__int_as_float(nseg), ray.tau_in, fmaf(ray.dxr, ray.dxr, ray.dyr * ray.dyr), 0.0f));
        __stcs(hd + 1, make_float4(sx ? (float)ray.sxs * ray.dxr * inv_dx : 0.0f, sy ? (float)ray.sys * ray.dyr * inv_dy : 0.0f,
                                   !sx ? 0.5f : ray.sxs > 0 ? fx : 1.0f - fx, !sy ? 0.5f : ray.sys > 0 ? fy : 1.0f - fy));
        __stcs(hd + 2, make_float4(0.0f, 0.0f, 0.0f, 0.0f));
        __stcs(hd + 3, make_float4(0.0f, 0.0f, 0.0f, ray.tau_in));
    }
}

size_t trace_table_bytes(const GeomDev &G)
{
    return (size_t)G.nviews * G.nu * sizeof(float) * trace_words(G);
}

static std::atomic<unsigned long long> g_trace_optin{0};

cbct_status trace_table_prepare()
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return check_cuda(e, "trace table device");
    const unsigned long long bit = 1ull << (dev & 63);
    if (g_trace_optin.load() & bit) return CBCT_OK;
    e = cudaFuncSetAttribute(k_trace_table, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PROJECT_SMEM_LIMIT);
    if (e != cudaSuccess) return check_cuda(e, "trace table attribute");
    g_trace_optin.fetch_or(bit);
    return CBCT_OK;
}

cbct_status launch_trace_table(const GeomDev &G, void *tab, cudaStream_t st, int col_first, int ncols)
{
    const size_t smem = trace_smem(G);
    if (smem > PROJECT_SMEM_LIMIT) return set_error(CBCT_ERR_UNSUPPORTED, "trace table: grid too large (nx + ny)");
    cbct_status r = trace_table_prepare();
    if (r != CBCT_OK) return r;
    if (ncols == 0) ncols = G.nviews * G.nu;
    launch_chained(k_trace_table, (unsigned)ncols, PROJ_THREADS, smem, st, G, static_cast<float *>(tab), col_first);
    note_launch();
    return check_cuda(cudaGetLastError(), "trace table launch");
}

// Non-zeros of P: every row of a block's (view, imager column) walks the trace and counts its
// segments longer than count_thr, splitting them at the z planes it crosses.
__global__ void __launch_bounds__(PROJ_THREADS) k_project_count(GeomDev G, double *__restrict__ partials,
                                                                float count_thr, int tcap, int rows)
{
    extern __shared__ __align__(16) float smem[];
    __shared__ double s_warp[PROJ_THREADS / 32];
    float *sEnd = smem;
    int *sCol = reinterpret_cast<int *>(sEnd + tcap);
    unsigned *s_cnt = reinterpret_cast<unsigned *>(sCol + tcap); // 4 per warp
    float *sA = reinterpret_cast<float *>(s_cnt + 4 * (PROJ_THREADS / 32));
    float *sB = sA + (G.nx + 1);
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int view = blockIdx.x / G.nu, iu = blockIdx.x - view * G.nu;
    const ColumnRay ray = column_ray(G, view, iu);
    const int4 tr = trace_column(G, ray, sA, sB, s_cnt, sEnd, sCol, tid, nthr);
    __syncthreads();
    const int nseg = tr.x + tr.y + 1;
    int cnt = 0;
    for (int r = 0; r < rows && ray.hit; ++r) {
        const int iv = blockIdx.y * (rows * nthr) + r * nthr + tid;
        const float v = imager_v(G, iv);
        const float inv_v = v != 0.0f ? __frcp_rn(v) : 1e30f;
        const int skz = v >= 0.0f ? 1 : -1;
        int kz = (int)floorf((v * (G.tc + ray.tau_in) - G.z0) / G.dz);
        bool active = iv < G.nv && kz >= 0 && kz < G.nz;
        auto next = [&]() { return active ? tau_zplane(plane_at(kz + (skz > 0), G.dz, G.z0), inv_v, G.tc) : P_INF; };
        float tzn = next();
        if (active && tzn <= ray.tau_in) { // the entry point already lies past that plane
            kz += skz;
            active = (unsigned)kz < (unsigned)G.nz;
            tzn = next();
        }
        const float thr_tau = count_thr / ray_length(ray.dxr, ray.dyr, v);
        float s0 = ray.tau_in;
        for (int j = 0; j < nseg; ++j) {
            const float e = sEnd[j];
            float sl = s0;
            while (tzn < e) {
                cnt += (tzn - sl) > thr_tau;
                sl = tzn;
                kz += skz;
                active = (unsigned)kz < (unsigned)G.nz;
                tzn = next();
            }
            if (active) cnt += (e - sl) > thr_tau;
            s0 = e;
        }
    }
    double red = (double)cnt;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) red += __shfl_down_sync(0xffffffffu, red, o);
    if ((tid & 31) == 0) s_warp[tid >> 5] = red;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < nthr / 32; ++w) t += s_warp[w];
        partials[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = t;
    }
}

static std::atomic<unsigned long long> g_count_optin{0};

cbct_status launch_project_count(const GeomDev &G, double *partials, float count_thr, cudaStream_t st)
{
    const size_t smem = trace_smem(G);
    if (smem > PROJECT_SMEM_LIMIT) return set_error(CBCT_ERR_UNSUPPORTED, "count_nnz: grid too large (nx + ny)");
    const cudaError_t e = smem_optin_once(k_project_count, (int)PROJECT_SMEM_LIMIT, g_count_optin);
    if (e != cudaSuccess) return check_cuda(e, "count_nnz attribute");
    const int threads = proj_threads(G), rows = proj_rows_per_thread(G);
    const dim3 grid((unsigned)(G.nviews * G.nu), (unsigned)((G.nv + rows * threads - 1) / (rows * threads)));
    CBCT_TIMED(CBCT_KERNEL_PROJECT, st,
               k_project_count<<<grid, threads, smem, st>>>(G, partials, count_thr, trace_cap(G), rows));
    return check_cuda(cudaGetLastError(), "count_nnz launch");
}

} // namespace cbct
