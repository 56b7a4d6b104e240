// Internal declarations of the cbcttf CUDA library (not part of the C ABI).
//
// Internal data layouts (the public ABI converts at its boundary):
//   volumes inside the iteration are z-fastest, [ny][nx][zp], so that a voxel column's
//   z-line is contiguous; zp = nz rounded up to a multiple of 4, so that every line starts
//   on a 16-byte boundary and is read in 16-byte pieces (the up to 3 padding values of a
//   line are never part of a result). Public volumes are x-fastest [nz][ny][nx]. Kernels
//   that touch volumes take the element strides (sx, sy, sz) so they serve both layouts.
//   projection stacks are always [n_views][nv][nu].
#pragma once

#include <atomic>

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "../../include/cbcttf.h"

namespace cbct {

// Geometry of one multigrid level as the kernels see it (FP32, derived from the FP64
// description on the host). All rays of view k at imager column u share their
// transverse (x, y) path; the v coordinate only tilts the ray in z (Section 2.1 geometry:
// the source orbit lies in the plane z = 0 and the imager's v axis is z).
struct GeomDev {
    int nx, ny, nz;
    int zp;                 // floats per z-line of the internal layout: nz rounded up to 4
    float dx, dy, dz;
    float x0, y0, z0;       // volume corner, -n * d / 2
    int nu, nv, nviews;
    float du, dv;
    float u_first, v_first; // coordinates of pixel 0
    float inv_du, inv_dv;
    float sad, sdd;
    float tc;               // sad / sdd: ray parameter of the isocentre plane
    const float2 *cs;       // (cos t_k, sin t_k) per view, device memory
    const float4 *ray4;     // per (view, imager column): (dxr, dyr, qx, qy) of ray_xy
    const float2 *ray2;     // per (view, imager column): (1/dxr, 1/dyr) of safe_rcp
};

// Rays are parametrised as X(tau) = Q + tau * d, d = D - S (source to pixel centre) and
// Q = S + tc * d, the point where the ray crosses the plane through the rotation axis
// parallel to the imager. For the circular orbit Q = tc * (u e_u + v e_z), so Q and the
// plane offsets stay small numbers and FP32 keeps ~1e-5 mm resolution along the ray.
// tau runs from -tc (source) to 1 - tc (pixel); the volume lies strictly inside.

// Coordinate of plane i of an axis with origin o and spacing h. P and P^T both use this
// exact expression so that both compute bit-identical crossing parameters.
__device__ __forceinline__ float plane_at(int i, float h, float o) { return fmaf((float)i, h, o); }

// Transverse part of ray (view with cos/sin c, s; imager coordinate u).
__device__ __forceinline__ void ray_xy(const GeomDev &G, float c, float s, float u, float &dxr,
                                       float &dyr, float &qx, float &qy)
{
    dxr = fmaf(-u, s, -G.sdd * c);
    dyr = fmaf(u, c, -G.sdd * s);
    float tu = G.tc * u;
    qx = -tu * s;
    qy = tu * c;
}

// 1 / d with a finite stand-in for d == 0 (such a ray never crosses that plane family).
__device__ __forceinline__ float safe_rcp(float d) { return d != 0.0f ? __frcp_rn(d) : 1e30f; }

// tau at which a ray with transverse offset q and reciprocal direction inv crosses plane p.
__device__ __forceinline__ float tau_plane(float p, float q, float inv) { return (p - q) * inv; }

// tau at which the ray through imager row v (1/v = inv_v) crosses the plane z = p:
// z(tau) = v (tc + tau) for every ray of the orbit, hence tau = p / v - tc.
__device__ __forceinline__ float tau_zplane(float p, float inv_v, float tc) { return fmaf(p, inv_v, -tc); }

__device__ __forceinline__ float imager_u(const GeomDev &G, int iu) { return fmaf((float)iu, G.du, G.u_first); }
__device__ __forceinline__ float imager_v(const GeomDev &G, int iv) { return fmaf((float)iv, G.dv, G.v_first); }

// Exact floor of |x| < 2^22 through the FP adder (no conversion instruction):
// adding 1.5 * 2^23 with rounding down leaves the integer in the low mantissa bits.
__device__ __forceinline__ int floor_small(float x) { return __float_as_int(__fadd_rd(x, 12582912.0f)) - 0x4B400000; }

// The kernels of a reconstruction are set up while the one they follow still runs (launch_chained):
// each waits here, before it touches anything in global memory, until every kernel before it has
// ended. Every block waits, so a kernel that has ended implies that all before it have. Launched
// plainly, the wait does nothing.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Shared memory by 32-bit address.
__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ float lds_float(unsigned a)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float2 lds_float2(unsigned a)
{
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}

// Length of ray (d) per unit tau: |D - S|.
__device__ __forceinline__ float ray_length(float dxr, float dyr, float v)
{
    return sqrtf(fmaf(dxr, dxr, fmaf(dyr, dyr, v * v)));
}

// Storage type of the projection-domain working vectors (y, r, q) and of stored frame
// coefficients: FP32, BF16 or FP16. Arithmetic is always FP32 (FP64 for inner products).
enum StorageType { ST_F32 = 0, ST_BF16 = 1, ST_F16 = 2 };

template <typename T> __device__ __forceinline__ float load_as_float(const T *p);
template <> __device__ __forceinline__ float load_as_float<float>(const float *p) { return __ldg(p); }
template <> __device__ __forceinline__ float load_as_float<__nv_bfloat16>(const __nv_bfloat16 *p)
{
    return __bfloat162float(__ldg(p));
}
template <> __device__ __forceinline__ float load_as_float<__half>(const __half *p) { return __half2float(__ldg(p)); }
__device__ __forceinline__ float as_float(float v) { return v; }
__device__ __forceinline__ float as_float(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float as_float(__half v) { return __half2float(v); }
template <typename T> __device__ __forceinline__ void store_from_float(T *p, float v);
template <> __device__ __forceinline__ void store_from_float<float>(float *p, float v) { *p = v; }
template <> __device__ __forceinline__ void store_from_float<__nv_bfloat16>(__nv_bfloat16 *p, float v)
{
    *p = __float2bfloat16_rn(v);
}
template <> __device__ __forceinline__ void store_from_float<__half>(__half *p, float v) { *p = __float2half_rn(v); }

// streaming (evict-first) store of a value that is not read again by this kernel
template <typename T> __device__ __forceinline__ void store_stream(T *p, float v);
template <> __device__ __forceinline__ void store_stream<float>(float *p, float v) { __stcs(p, v); }
template <> __device__ __forceinline__ void store_stream<__nv_bfloat16>(__nv_bfloat16 *p, float v)
{
    __stcs(p, __float2bfloat16_rn(v));
}
template <> __device__ __forceinline__ void store_stream<__half>(__half *p, float v) { __stcs(p, __float2half_rn(v)); }

// Opts a kernel into more than 48 KB of dynamic shared memory. The attribute belongs to
// the function on one device, so it is set once per device (`done` holds one bit each).
template <typename Kernel>
inline cudaError_t smem_optin_once(Kernel fn, int bytes, std::atomic<unsigned long long> &done)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (done.load() & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done.fetch_or(bit);
    return e;
}

// Device-resident scalars of CGLS (Appendix 1), FP64.
struct Scalars {
    double gamma;    // ||s||^2
    double delta;    // ||q||^2
    double alpha;    // gamma / delta
    double beta;     // gamma' / gamma
    double rr;       // ||r||^2 (monitoring)
    double kappa;    // q is stored as kappa * q, kappa = 1 / sqrt(gamma): keeps FP16 in range
    unsigned int flags; // bit 0: a reduction was not finite; bit 1: a projector block's wait timed out
    unsigned int arrived; // blocks of the running reduction that have written their partial sum (0 between kernels)
};

// What the sum of a kernel's partials becomes. scale_q: q is about to be stored in FP16, so keep
// kappa = 1 / sqrt(gamma) (||kappa p|| >= 1 and kappa q stays O(1)); otherwise kappa = 1.
enum FinalizeOp { FIN_NONE = -1, FIN_GAMMA = 0, FIN_ALPHA = 1, FIN_BETA = 2, FIN_RR = 3 };

// After thread 0 of a block has stored partials[block]: true in the block that is the last of
// `blocks` to do so (thread 0 only).
__device__ __forceinline__ bool last_to_arrive(Scalars *sc, unsigned blocks)
{
    __threadfence();
    return atomicAdd(&sc->arrived, 1u) == blocks - 1u;
}
// The last block's share: thread t of nthr sums partials t, t + nthr, ... (a fixed order, so the
// result does not depend on scheduling).
__device__ __forceinline__ double sum_partials(const double *partials, unsigned n, int t, int nthr)
{
    __threadfence();
    double v = 0.0;
    for (unsigned i = t; i < n; i += nthr) v += __ldcg(partials + i);
    return v;
}
// Thread 0 of the last block: the scalars of CGLS from the whole sum.
__device__ __forceinline__ void apply_sum(Scalars *sc, double sum, int op, int scale_q)
{
    if (!isfinite(sum)) atomicOr(&sc->flags, 1u);
    if (op == FIN_GAMMA || op == FIN_BETA) {
        if (op == FIN_BETA) sc->beta = sc->gamma > 0.0 ? sum / sc->gamma : 0.0;
        sc->gamma = sum;
        sc->kappa = (scale_q && sum > 0.0 && isfinite(sum)) ? 1.0 / sqrt(sum) : 1.0;
    } else if (op == FIN_ALPHA) {
        sc->delta = sum;
        sc->alpha = (sc->gamma > 0.0 && sum > 0.0) ? sc->gamma / sum : 0.0;
    } else {
        sc->rr = sum;
    }
    sc->arrived = 0u;
}

// Projector epilogues (q = |D - S| * sum of f * dtau is the projection of the ray).
enum ProjectMode {
    PM_PLAIN = 0,      // out = q                                     (public P)
    PM_Q_SCALED = 1,   // out = kappa * q (stored type), partial sums of q^2
    PM_RESID = 2,      // out = y - q (stored type), partial sums of (y - q)^2
    PM_COUNT = 3       // count segments longer than a threshold
};

// ---- host side ----------------------------------------------------------------------

// Optional per-launch timing (cbct_profiling_enable): events around each launch.
struct ProfToken {
    cudaEvent_t start;
    int kind;
};
ProfToken prof_start(int kind, cudaStream_t st);
void prof_stop(const ProfToken &t, cudaStream_t st);

// Launch a kernel with optional timing and the launch counter:
//   CBCT_TIMED(kind, stream, kernel<<<grid, block, smem, stream>>>(args...));
#define CBCT_TIMED(kind, st, ...)                                                                  \
    do {                                                                                           \
        ::cbct::ProfToken _cbct_tok = ::cbct::prof_start((kind), (st));                            \
        __VA_ARGS__;                                                                               \
        ::cbct::prof_stop(_cbct_tok, (st));                                                        \
        ::cbct::note_launch();                                                                     \
    } while (0)

// Launches a kernel that calls chain_wait(): its launch overlaps the end of the kernel before it. An iteration of
// short kernels gains most: 64x64x16, 20 iterations 4.13 -> 3.48 ms, 256x256x64 in three levels 49.0 -> 48.0 ms,
// 512x512x70 135.6 -> 134.5 ms. (Letting the next kernel's blocks in as soon as all of this one's are
// placed loses: 4.40, 54.4 and 156 ms; they take room from this kernel's second block per SM.)
cudaError_t launch_chained(const void *kernel, dim3 grid, dim3 block, void **args, size_t smem, cudaStream_t st);
template <typename T> struct AsIs { using type = T; };
template <typename... P>
inline void launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                           typename AsIs<P>::type... a)
{
    void *args[] = {static_cast<void *>(&a)...};
    launch_chained(reinterpret_cast<const void *>(kernel), grid, block, args, smem, st);
}

cbct_status set_error(cbct_status st, const char *fmt, ...);
cbct_status check_cuda(cudaError_t e, const char *what);
void note_launch(unsigned n = 1);
int device_sm_count();

// Launchers (all asynchronous on `st`; return CBCT_ERR_CUDA on launch failure).
// Volume element (ix, iy, iz) lives at ix*sx + iy*sy + iz*sz.
int project_num_blocks(const GeomDev &G);
// Elements of a volume in the internal layout.
static inline size_t internal_elems(const GeomDev &G) { return (size_t)G.nx * G.ny * G.zp; }
// Dynamic shared memory a projector block may use (opted in per kernel).
constexpr size_t PROJECT_SMEM_LIMIT = 200 * 1024;

// out holds `storage`-typed values (PM_COUNT: none); y is FP32; sc supplies kappa in
// PM_Q_SCALED and, when given, receives bit 1 of its flags if a block's wait for its copies
// ran out (its rows are NaN). With FP32 storage the CGLS modes store |D - S| r and |D - S| q.
// f is in the internal layout with z-lines of zpitch floats: G.zp, or G.nz for a volume without
// padding (PM_PLAIN with FP32 storage only; the same results from narrower loads). traces: the
// trace table from launch_trace_table (PM_COUNT: none); only the (view, imager column) pairs
// [col_first, col_first + ncols) are projected, whose records are its first (ncols = 0: all).
// In the CGLS modes the last block to finish also sums the blocks' partials (at most
// project_num_blocks(G) of them) into sc: ||y - q||^2 (PM_RESID), ||q||^2 and alpha (PM_Q_SCALED).
cbct_status launch_project(const GeomDev &G, const float *f, int zpitch, const float *y, void *out, int mode,
                           double *partials, float count_thr, cudaStream_t st, int storage, Scalars *sc,
                           const void *traces, int col_first = 0, int ncols = 0);
// The projector's trace table of a grid (trace_table_bytes(G) bytes for all columns, 16-byte
// aligned): the transverse trace of the (view, imager column) pairs [col_first, col_first + ncols)
// (ncols = 0: all).
size_t trace_table_bytes(const GeomDev &G);
cbct_status launch_trace_table(const GeomDev &G, void *tab, cudaStream_t st, int col_first = 0, int ncols = 0);
cbct_status trace_table_prepare();
// Upper bound of the blocks of an adjoint launch over every grid no larger than G's.
int backproject_max_blocks(const GeomDev &G);
// ps: per-(view, imager column) prefix sums over rows of the |D - S|-weighted stack,
// [n_views][nv + 1][nu] float2 (prefix of the rows below m, value of row m), prefix_table_bytes(G)
// bytes, built by launch_row_prefix. With partials, the last block to finish sums them into sc by
// fin_op (FinalizeOp).
size_t prefix_table_bytes(const GeomDev &G);
cbct_status launch_backproject(const GeomDev &G, const float2 *ps, float *out, long long sx,
                               long long sy, long long sz, float *out2, double *partials,
                               cudaStream_t st, Scalars *sc = nullptr, int fin_op = FIN_NONE, int scale_q = 0);
cbct_status launch_row_prefix(const GeomDev &G, const void *g, float2 *ps, int prescale,
                              cudaStream_t st, int storage = ST_F32);
// The same of the CGLS residual after its update r -= alpha q, which is written back to r.
cbct_status launch_update_prefix(const GeomDev &G, void *r, const void *q, const Scalars *sc, float2 *ps, int prescale,
                                 cudaStream_t st, int storage);
cbct_status launch_backproject_eq3(const GeomDev &G, const float *g, float *f, float pref,
                                   cudaStream_t st);

// alpha holds `storage`-typed coefficients (FP32, BF16 or FP16); arithmetic is FP32
cbct_status launch_tf_analyze(int n0, int n1, int n2, const float *f, void *alpha,
                              cudaStream_t st, int storage = ST_F32);
cbct_status launch_tf_synth_shrink(int n0, int n1, int n2, const void *alpha, float mu,
                                   int positivity, float *f, cudaStream_t st, int storage = ST_F32);
// Fused f_new = H(W^T T_mu W x) and, if vout != nullptr, v = f_new + coef (f_new - f_old).
// p0 >= n0: elements from one row along axis 0 to the next, of every array.
cbct_status launch_tf_shrink_fused(int n0, int n1, int n2, int p0, const float *x, float mu, int positivity,
                                   float *fnew, const float *fold, float coef, float *vout,
                                   cudaStream_t st);
// Public x-fastest [nz][ny][nx] <-> internal z-fastest [ny][nx][zpitch] volume layout.
cbct_status transpose(const float *in, float *out, int nx, int ny, int nz, int zpitch, bool to_internal,
                      cudaStream_t st);

} // namespace cbct

// Library-owned geometry handle.
struct cbct_geometry {
    cbct_geometry_desc desc; // angles points into `angles`
    double *angles;          // host copy
    int device;
    float2 *d_cs;            // per-view (cos, sin)
    float4 *d_ray4;          // per (view, imager column) transverse ray (ray_xy)
    float2 *d_ray2;          // per (view, imager column) reciprocal directions
    float *d_scratch;        // public project/backproject scratch (lazily allocated)
    size_t scratch_bytes;
    void *d_ws;              // reconstruction workspace (lazily allocated)
    size_t ws_bytes;
};

namespace cbct {
constexpr int MAX_LEVELS = 8; // multigrid levels a reconstruction may use
GeomDev level_geom(const cbct_geometry *g, int level);
cbct_status ensure_scratch(cbct_geometry *g, size_t bytes);

// Geometry pieces for callers that build a cbct_geometry in memory they own (the request
// server): argument checks, the host view table (angles and FP32 cos/sin), and the
// stream-ordered ray-table kernel.
cbct_status validate_geometry_desc(const cbct_geometry_desc &d);
// Shared memory one projector block needs on the finest grid (the largest level).
size_t project_smem_bytes(const GeomDev &G);
// Force the projector's column-group size (0: choose per launch); the size a PM_PLAIN FP32
// launch on G uses.
cbct_status project_set_group(int sg);
cbct_status project_group_of(const GeomDev &G, int *sg);
// UNSUPPORTED when the projector's per-block shared memory for this geometry exceeds what
// it may use (its staged z-lines and tables grow with nz, its segment lists with nx + ny).
cbct_status check_projector_fits(const cbct_geometry_desc &d);
void view_table(const cbct_geometry_desc &d, double *angles, float2 *cs);
cbct_status launch_ray_table(const cbct_geometry *g, cudaStream_t st);

// The reconstruction as pure stream work: no allocation, no synchronisation, nothing read
// back (capturable into a CUDA graph). ws must hold reconstruct_ws_bytes(g) bytes, 256-byte
// aligned; the iteration's status word (bit 0: a non-finite inner product) is at
// reconstruct_flags_address(g, ws) once the work has run.
cbct_status validate_recon_args(float mu, float lambda, int levels, const int *iters, const cbct_recon_opts &o);
size_t reconstruct_ws_bytes(const cbct_geometry *g);
cbct_status reconstruct_enqueue(const float *y, cbct_geometry *g, float mu, int levels, const int *iters,
                                const cbct_recon_opts &o, void *ws, size_t ws_bytes, float *f_out, cudaStream_t st);
const unsigned int *reconstruct_flags_address(const cbct_geometry *g, void *ws);

// The same reconstruction enqueued one step at a time (one A2 iteration per step; the
// set-up of a level rides on its first step, the change back to the public layout on the
// last). Consecutive steps may go to different streams if the caller orders them (an
// event recorded after one step, waited on by the stream of the next). The cursor keeps
// iters; the buffers must outlive the last step.
struct ReconCursor;
cbct_status reconstruct_cursor_create(const float *y, cbct_geometry *g, float mu, int levels, const int *iters,
                                      const cbct_recon_opts &o, void *ws, size_t ws_bytes, float *f_out,
                                      ReconCursor **out);
cbct_status reconstruct_cursor_step(ReconCursor *c, cudaStream_t st);
bool reconstruct_cursor_finished(const ReconCursor *c);
void reconstruct_cursor_destroy(ReconCursor *c);

// Sets every kernel attribute the launchers would otherwise set on first use (shared
// memory opt-ins) on the current device, so that later launches can be graph-captured.
cbct_status project_prepare();
cbct_status backproject_prepare();
cbct_status tf_prepare();
}
