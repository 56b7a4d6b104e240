// Piecewise-linear tight frame (Section 2.1): analysis W, and vector shrinkage T_mu
// (Eq. (2)) + synthesis W^T + positivity H.
//
// The 3-D filters are tensor products of h0 = [1,2,1]/4, h1 = sqrt(2)/4 [1,0,-1],
// h2 = [-1,2,-1]/4, so both transforms run as three 3-tap passes. Arrays are addressed as
// (i2 * n1 + i1) * n0 + i0 with i0 the contiguous axis; channel i = l + 3m + 9n applies
// h_l along axis 0, h_m along axis 1 and h_n along axis 2. The boundary is periodic.
//
// GB300 mapping. Every kernel marches along axis 2 so that each input value is read from
// DRAM once and each output written once, with warps reading and writing rows along the
// contiguous axis. The analysis W marches a tile of the (axis 0, axis 1) plane that is read
// through shared memory (with a one-voxel halo). The shrink +
// synthesis and the fused step give each lane whole positions and pass neighbour values by
// warp shuffles (axis 0), a shared exchange (axis 1) and registers (axis 2); they are
// described at their kernels. The public transforms are bandwidth bound: 4 B in + 108 B
// out per voxel for W, 108 B in + 4 B out for the shrink/synthesis (FP32 coefficients).
#include "cbct_internal.cuh"
#include "f32x2.cuh"

namespace cbct {

constexpr int TA = 32, TB = 8, TF_THREADS = TA * TB;
constexpr int MAX_GRID_Y = 65535;
constexpr float R2_4 = 0.35355339059327373f; // sqrt(2) / 4

__device__ __forceinline__ int wrapi(int i, int n)
{
    i %= n;
    return i < 0 ? i + n : i;
}

// Analysis along one axis for the window (f(x-1), f(x), f(x+1)) = (p, c, n):
// alpha_l(x) = h_l[-1] f(x+1) + h_l[0] f(x) + h_l[1] f(x-1).
__device__ __forceinline__ void ana3(float p, float c, float n, float &o0, float &o1, float &o2)
{
    const float s = n + p;
    o0 = fmaf(0.25f, s, 0.5f * c);
    o1 = __fmul_rn(R2_4, n - p); // (not contracted into the next pass: the packed form's bits)
    o2 = fmaf(-0.25f, s, 0.5f * c);
}

__device__ __forceinline__ void ana3(f32x2 p, f32x2 c, f32x2 n, f32x2 &o0, f32x2 &o1, f32x2 &o2)
{
    const f32x2 s = add2(n, p), h = mul2(splat(0.5f), c);
    o0 = fma2(splat(0.25f), s, h);
    o1 = mul2(splat(R2_4), sub2(n, p));
    o2 = fma2(splat(-0.25f), s, h);
}

// Two adjacent values of the contiguous axis as stored.
template <typename T> struct Pair;
template <> struct Pair<float> {
    using T2 = float2;
    static __device__ __forceinline__ f32x2 get(T2 v) { return pk(v.x, v.y); }
    static __device__ __forceinline__ T2 put(f32x2 v) { return make_float2(lo2(v), hi2(v)); }
};
template <> struct Pair<__nv_bfloat16> {
    using T2 = __nv_bfloat162;
    static __device__ __forceinline__ f32x2 get(T2 v)
    {
        const float2 f = __bfloat1622float2(v);
        return pk(f.x, f.y);
    }
    static __device__ __forceinline__ T2 put(f32x2 v) { return __floats2bfloat162_rn(lo2(v), hi2(v)); }
};
template <> struct Pair<__half> {
    using T2 = __half2;
    static __device__ __forceinline__ f32x2 get(T2 v)
    {
        const float2 f = __half22float2(v);
        return pk(f.x, f.y);
    }
    static __device__ __forceinline__ T2 put(f32x2 v) { return __floats2half2_rn(lo2(v), hi2(v)); }
};

template <typename TA_T>
__global__ void __launch_bounds__(TF_THREADS)
k_tf_analyze(int n0, int n1, int n2, int chunk, const float *__restrict__ f, TA_T *__restrict__ alpha)
{
    __shared__ float s[3][TB + 2][TA + 2];
    const int a0 = blockIdx.x * TA, b0 = blockIdx.y * TB;
    const int c_begin = blockIdx.z * chunk;
    const int c_end = min(n2, c_begin + chunk);
    if (c_begin >= c_end) return;
    const int tid = threadIdx.y * TA + threadIdx.x;
    const size_t N = (size_t)n0 * n1 * n2;

    int off[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int pos = tid + k * TF_THREADS;
        if (pos < (TA + 2) * (TB + 2)) {
            const int r = pos / (TA + 2), q = pos - r * (TA + 2);
            off[k] = wrapi(b0 + r - 1, n1) * n0 + wrapi(a0 + q - 1, n0);
        } else {
            off[k] = -1;
        }
    }
    // the haloed tile of plane c: this thread's (at most two) values
    float nxt[2] = {0.0f, 0.0f};
    auto fetch = [&](int c) {
        const float *src = f + (size_t)wrapi(c, n2) * n1 * n0;
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (off[k] >= 0) nxt[k] = __ldg(src + off[k]);
    };
    auto put = [&](int slot) {
        float *d = &s[slot][0][0];
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (off[k] >= 0) d[tid + k * TF_THREADS] = nxt[k];
    };
    fetch(c_begin - 1);
    put(0);
    fetch(c_begin);
    put(1);
    fetch(c_begin + 1);
    const int ta = threadIdx.x, tb = threadIdx.y;
    const bool inside = a0 + ta < n0 && b0 + tb < n1;
    for (int c = c_begin; c < c_end; ++c) {
        const int j = c - c_begin;
        put((j + 2) % 3); // plane c + 1, loaded during the previous plane
        __syncthreads();
        if (c + 1 < c_end) fetch(c + 2); // lands while this plane is computed and stored
        if (inside) {
            const int sl[3] = {j % 3, (j + 1) % 3, (j + 2) % 3}; // planes c-1, c, c+1
            // axis 0 then axis 1: u[cc][m][l]
            float u[3][3][3];
#pragma unroll
            for (int cc = 0; cc < 3; ++cc) {
                float t[3][3]; // [bb][l]
#pragma unroll
                for (int bb = 0; bb < 3; ++bb)
                    ana3(s[sl[cc]][tb + bb][ta], s[sl[cc]][tb + bb][ta + 1], s[sl[cc]][tb + bb][ta + 2],
                         t[bb][0], t[bb][1], t[bb][2]);
#pragma unroll
                for (int l = 0; l < 3; ++l) ana3(t[0][l], t[1][l], t[2][l], u[cc][0][l], u[cc][1][l], u[cc][2][l]);
            }
            const size_t o = ((size_t)c * n1 + (b0 + tb)) * n0 + (a0 + ta);
#pragma unroll
            for (int m = 0; m < 3; ++m)
#pragma unroll
                for (int l = 0; l < 3; ++l) {
                    float w0, w1, w2;
                    ana3(u[0][m][l], u[1][m][l], u[2][m][l], w0, w1, w2);
                    store_stream(alpha + (size_t)(l + 3 * m) * N + o, w0);
                    store_stream(alpha + (size_t)(l + 3 * m + 9) * N + o, w1);
                    store_stream(alpha + (size_t)(l + 3 * m + 18) * N + o, w2);
                }
        }
        __syncthreads();
    }
}

// The same with two adjacent positions per lane (an even n0, so that every pair is aligned): one
// store of a pair per channel, packed arithmetic with the bits of the general kernel's, and the axis-0
// and axis-1 passes of each plane done once (those of the two planes before stay in registers).
// Bound by the 27 written channels: 512x512x70 FP32 334 us (6.2 TB/s; one position per lane and three
// planes in shared memory 360 us), BF16 198 us (240), 256x256x64 74 (76) and 44 us (62). Blocks of
// 4 rows, 96 registers, five per SM; with 80 registers 336 | 245 us, blocks of 8 rows 330 | 221 us but
// 84 us at 256x256x64 FP32 (the last wave), 2 rows 341 | 256 us. An odd n0 takes the general kernel, and so do the
// widths that leave too much of its tiles idle (rule at the launcher).
constexpr int AP_B = 4, AP_THREADS = 32 * AP_B, AP_BLOCKS = 5;
template <typename T>
__global__ void __launch_bounds__(AP_THREADS, AP_BLOCKS)
k_tf_analyze_pair(int n0, int n1, int n2, int chunk, const float *__restrict__ f, T *__restrict__ alpha)
{
    using P = Pair<T>;
    using T2 = typename P::T2;
    constexpr int W = 66, SIZE = W * (AP_B + 2), PER = (SIZE + AP_THREADS - 1) / AP_THREADS;
    __shared__ __align__(8) float s[2][SIZE]; // a plane of the tile with its halo
    const int a0 = blockIdx.x * 64, b0 = blockIdx.y * AP_B;
    const int c_begin = blockIdx.z * chunk;
    const int c_end = min(n2, c_begin + chunk);
    if (c_begin >= c_end) return;
    const int tid = threadIdx.y * 32 + threadIdx.x;
    const size_t plane = (size_t)n0 * n1, N = plane * n2;

    int off[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int pos = tid + k * AP_THREADS, r = pos / W, q = pos - r * W;
        off[k] = pos < SIZE ? wrapi(b0 + r - 1, n1) * n0 + wrapi(a0 + q - 1, n0) : -1;
    }
    float nxt[PER];
    auto fetch = [&](int c) {
        const float *src = f + (size_t)wrapi(c, n2) * plane;
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if (off[k] >= 0) nxt[k] = __ldg(src + off[k]);
    };
    fetch(c_begin - 1);
    const int pa = a0 + 2 * threadIdx.x, pb = b0 + threadIdx.y;
    const bool inside = pa < n0 && pb < n1;
    f32x2 um[3][3], u0[3][3]; // [m][l] of planes cp - 2 and cp - 1
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
        for (int l = 0; l < 3; ++l) um[m][l] = u0[m][l] = 0ull;
    int buf = 0;
    for (int cp = c_begin - 1; cp <= c_end; ++cp, buf ^= 1) {
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if (off[k] >= 0) s[buf][tid + k * AP_THREADS] = nxt[k];
        __syncthreads();
        if (cp < c_end) fetch(cp + 1);
        f32x2 t[3][3], up[3][3];
#pragma unroll
        for (int bb = 0; bb < 3; ++bb) {
            const float2 *row = reinterpret_cast<const float2 *>(&s[buf][(threadIdx.y + bb) * W + 2 * threadIdx.x]);
            const float2 v0 = row[0], v1 = row[1];
            ana3(pk(v0.x, v0.y), pk(v0.y, v1.x), pk(v1.x, v1.y), t[bb][0], t[bb][1], t[bb][2]);
        }
#pragma unroll
        for (int l = 0; l < 3; ++l) ana3(t[0][l], t[1][l], t[2][l], up[0][l], up[1][l], up[2][l]);
        if (inside && cp > c_begin) {
            T2 *q = reinterpret_cast<T2 *>(alpha + (size_t)(cp - 1) * plane + (size_t)pb * n0 + pa);
            const size_t ch = N / 2; // (N is even)
#pragma unroll
            for (int m = 0; m < 3; ++m)
#pragma unroll
                for (int l = 0; l < 3; ++l) {
                    f32x2 w[3];
                    ana3(um[m][l], u0[m][l], up[m][l], w[0], w[1], w[2]);
#pragma unroll
                    for (int n = 0; n < 3; ++n) __stcs(q + (l + 3 * m + 9 * n) * ch, P::put(w[n]));
                }
        }
#pragma unroll
        for (int m = 0; m < 3; ++m)
#pragma unroll
            for (int l = 0; l < 3; ++l) {
                um[m][l] = u0[m][l];
                u0[m][l] = up[m][l];
            }
    }
}

// Resident blocks of a kernel on the whole device. The kernel's occupancy is asked for once per
// device (`cache`, one per kernel): the query costs about as much host time as a launch.
using Residency = std::atomic<int>[64];
static cudaError_t resident_blocks(const void *kernel, int threads, Residency &cache, int *slots)
{
    int dev = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 64) per_sm = cache[dev].load(std::memory_order_relaxed);
    if (!per_sm) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
        if (dev < 64) cache[dev].store(per_sm, std::memory_order_relaxed);
    }
    *slots = per_sm * device_sm_count();
    return cudaSuccess;
}

// Planes per block along axis 2: the split whose blocks fill whole waves of the resident slots best, counting the
// two extra planes each block computes at its ends as `extra` (a block's cost grows with chunk + extra).
// *cost, if given: the waves times the planes of a block.
static int fused_chunk(long long tiles, int n2, int slots, double extra = 2.0, long long *cost = nullptr)
{
    int best = n2;
    double best_eff = -1.0;
    // (every split into equal chunks once: from one length to the next shorter one)
    for (int nch = 1, chunk = n2;; nch = (n2 + chunk - 2) / (chunk - 1)) {
        chunk = (n2 + nch - 1) / nch;
        const long long nb = tiles * ((n2 + chunk - 1) / chunk);
        const long long waves = (nb + slots - 1) / slots;
        const double eff = (double)n2 / ((double)((n2 + chunk - 1) / chunk) * (chunk + extra)) * (double)nb /
                           ((double)waves * slots);
        if (eff > best_eff + 1e-9) {
            best_eff = eff;
            best = chunk;
            if (cost) *cost = waves * (chunk + 2);
        }
        if (chunk == 1) break;
    }
    return best;
}

// ------------------------------------------------------------------------------------
// Shrink + synthesis f = H(W^T T_mu alpha) of the public entry point.
//
// A warp covers 32 consecutive positions of one row along axis 0 (the 30 positions of the
// tile plus one halo position on either side); a block stacks SY_ROWS + 2 such warps along
// axis 1 (its SY_ROWS rows plus one halo row on either side) and marches along axis 2.
// Every lane reads the 27 coefficients of its own position (coalesced 128-byte rows per
// channel), the next plane's while the current one is computed, and shrinks them in
// registers (Eq. (2)). The separable synthesis then splits each 3-tap sum into what a
// position gives its neighbours: along axis 1 of the filter triple (a_0, a_1, a_2) at
// position p, p + 1 receives a_0/4 + (sqrt(2)/4) a_1 - a_2/4, p itself (a_0 + a_2)/2 and
// p - 1 a_0/4 - (sqrt(2)/4) a_1 - a_2/4. Axis 0 passes those shares between lanes with
// two shuffles per channel group, axis 1 between warps through shared memory (one
// barrier per plane, double buffered), and axis 2 between planes in registers.
// HBM traffic: 27 coefficients read and one value written per voxel; the halo positions
// (32/30 along axis 0, (SY_ROWS + 2)/SY_ROWS along axis 1) are re-read from L2, and a warp's
// row touches five sectors of each channel, not four. 512x512x70 FP32: 411 us, 2.10 GB from
// DRAM (5.3 TB/s), 3.58 GB from L2 (8.8 TB/s), issue 60%. Two positions per lane 420 us, 16 or 20 warps
// in one block 414 | 411 us, a second plane of coefficients under way 413 us.
// ------------------------------------------------------------------------------------
constexpr int SY_ROWS = 8;
constexpr int SY_OUT = 30;                       // output positions per warp along axis 0
constexpr int SY_WARPS = SY_ROWS + 2;
constexpr int SY_THREADS = 32 * SY_WARPS;

// Each pass leaves out a factor 1/4 of its taps: shares a_0 - a_2 +- sqrt(2) a_1 and 2 (a_0 + a_2), of
// coefficients that enter as 64ths (which rounds nothing, but for values below 2^-114, and leaves no intermediate
// larger than the taps would). The shrinkage factor is applied to a triple's sum and difference.
// Kernels for pairs of positions take the same operations and leave the same bits.
constexpr float SYN_R = 4.0f * R2_4;

template <typename TA_T>
__global__ void __launch_bounds__(SY_THREADS, 2)
k_tf_synth_shrink(int n0, int n1, int n2, int chunk, const TA_T *__restrict__ alpha, float mu,
                  int positivity, float *__restrict__ f)
{
    __shared__ float s_up[2][SY_WARPS][3][32], s_dn[2][SY_WARPS][3][32];
    const int lane = threadIdx.x, w = threadIdx.y;
    const int a_out = blockIdx.x * SY_OUT;           // first output position along axis 0
    const int b_out = blockIdx.y * SY_ROWS;          // first output row along axis 1
    const int c_begin = blockIdx.z * chunk;
    const int c_end = min(n2, c_begin + chunk);
    if (c_begin >= c_end) return;
    const size_t N = (size_t)n0 * n1 * n2;
    const size_t plane = (size_t)n0 * n1;
    const int pa = a_out + lane - 1, pb = b_out + w - 1; // this lane's position (unwrapped)
    const size_t inplane = (size_t)wrapi(pb, n1) * n0 + wrapi(pa, n0);
    const bool out_lane = lane >= 1 && lane <= SY_OUT && pa < n0;
    const bool out_row = w >= 1 && w <= SY_ROWS && pb < n1;

    TA_T nxt[27];
    auto fetch = [&](int c) {
        const TA_T *src = alpha + (size_t)wrapi(c, n2) * plane + inplane;
#pragma unroll
        for (int ch = 0; ch < 27; ++ch) nxt[ch] = src[(size_t)ch * N];
    };
    fetch(c_begin - 1);
    float w_m2[3] = {0.f, 0.f, 0.f}, w_m1[3] = {0.f, 0.f, 0.f}; // axis-2 inputs at planes cp-2, cp-1
    int buf = 0;
    for (int cp = c_begin - 1; cp <= c_end; ++cp, buf ^= 1) {
        float a[27];
#pragma unroll
        for (int ch = 0; ch < 27; ++ch) a[ch] = as_float(nxt[ch]);
        if (cp < c_end) fetch(cp + 1);
        // vector shrinkage, Eq. (2)
        float s2 = 0.0f;
#pragma unroll
        for (int ch = 1; ch < 27; ++ch) s2 = fmaf(a[ch], a[ch], s2);
        const float nrm = sqrtf(s2);
        const float scale = (nrm > mu ? 1.0f - mu / nrm : 0.0f) * (1.0f / 64.0f);
        const float sc2 = scale + scale, scr = SYN_R * scale, scn = -SYN_R * scale;
        // axis 0 (lanes): u[m + 3n] = sum over l and the lane's neighbours
        float u[9];
#pragma unroll
        for (int mn = 0; mn < 9; ++mn) {
            // (channel 0 is not shrunk)
            const float a0 = mn ? a[3 * mn] : a[0] * (1.0f / 64.0f), a2 = mn ? a[3 * mn + 2] : __fmul_rn(scale, a[2]);
            const float q = mn ? __fmul_rn(scale, a0 - a2) : a0 - a2;
            const float up = fmaf(scr, a[3 * mn + 1], q), dn = fmaf(scn, a[3 * mn + 1], q);
            u[mn] = fmaf(mn ? sc2 : 2.0f, a0 + a2, __shfl_up_sync(0xffffffffu, up, 1)) + __shfl_down_sync(0xffffffffu, dn, 1);
        }
        // axis 1 (warps): shares of rows to the rows above and below through shared memory
        float mid[3];
#pragma unroll
        for (int n = 0; n < 3; ++n) {
            const float q = u[3 * n] - u[3 * n + 2];
            mid[n] = u[3 * n] + u[3 * n + 2];
            s_up[buf][w][n][lane] = fmaf(SYN_R, u[3 * n + 1], q);
            s_dn[buf][w][n][lane] = fmaf(-SYN_R, u[3 * n + 1], q);
        }
        __syncthreads();
        if (out_row) {
            float wv[3];
#pragma unroll
            for (int n = 0; n < 3; ++n) wv[n] = fmaf(2.0f, mid[n], s_up[buf][w - 1][n][lane]) + s_dn[buf][w + 1][n][lane];
            // axis 2 (planes): plane cp - 1 from planes cp - 2, cp - 1, cp
            if (cp >= c_begin + 1 && out_lane) {
                const float ends = (w_m2[0] + wv[0]) - (w_m2[2] + wv[2]);
                float o = fmaf(2.0f, w_m1[0] + w_m1[2], SYN_R * (w_m2[1] - wv[1])) + ends;
                if (positivity && o < 0.0f) o = 0.0f;
                f[(size_t)(cp - 1) * plane + (size_t)pb * n0 + pa] = o;
            }
#pragma unroll
            for (int n = 0; n < 3; ++n) {
                w_m2[n] = w_m1[n];
                w_m1[n] = wv[n];
            }
        }
    }
}

template <typename TA_T>
static cbct_status launch_tf_analyze_t(int n0, int n1, int n2, const float *f, TA_T *alpha, cudaStream_t st)
{
    // The pair kernel's tiles are twice as wide, so that a row's last tile may do twice the columns in vain: taken
    // up to 4/3 of the general kernel's (all widths above 32), and of FP32 rows of whole sectors, which the general
    // kernel also writes well, up to 5/4 (pair | general: 18x512x64 24.6 | 18.9 us, 96x256x100 57.4 | 47.1 us, 160x256x100
    // 72.4 | 82.5 us, 98x256x100 105 | 119 us; BF16 96x256x100 35.0 | 41.2 us). (Its AP_B rows reach the grid's limit along y at half the rows that are accepted.)
    const int cols = (n0 + 63) / 64 * 64, general_cols = (n0 + TA - 1) / TA * TA;
    const bool pair = n0 % 2 == 0 && (reinterpret_cast<uintptr_t>(alpha) & (2 * sizeof(TA_T) - 1)) == 0 &&
                      (sizeof(TA_T) == 4 && n0 % 8 == 0 ? 4LL * cols <= 5LL * general_cols : 3LL * cols <= 4LL * general_cols) &&
                      (n1 + AP_B - 1) / AP_B <= MAX_GRID_Y;
    const auto kernel = pair ? k_tf_analyze_pair<TA_T> : k_tf_analyze<TA_T>;
    const int ta = pair ? 64 : TA, tb = pair ? AP_B : TB;
    static Residency residency[2];
    int slots = 0;
    const cudaError_t e = resident_blocks(reinterpret_cast<const void *>(kernel), 32 * tb, residency[pair], &slots);
    if (e != cudaSuccess) return check_cuda(e, "tf_analyze occupancy");
    const long long tiles = (long long)((n0 + ta - 1) / ta) * ((n1 + tb - 1) / tb);
    // The extra planes of the pair kernel are read and passed along two axes but not stored, which is what an FP32
    // plane costs: 0.6 of one (with 2 | 0.6: 288x512x64 218 | 171 us, 82x256x100 95 | 71 us, 256x256x20 28.7 |
    // 25.9 us, 512x512x70 328 | 322 us). 16-bit planes cost as much to compute as to store (256x256x20 BF16 16.9 | 18.2 us).
    const int chunk = fused_chunk(tiles, n2, slots, pair && sizeof(TA_T) == 4 ? 0.6 : 2.0);
    dim3 grid((n0 + ta - 1) / ta, (n1 + tb - 1) / tb, (n2 + chunk - 1) / chunk);
    CBCT_TIMED(CBCT_KERNEL_TF_ANALYZE, st, kernel<<<grid, dim3(32, tb), 0, st>>>(n0, n1, n2, chunk, f, alpha));
    return check_cuda(cudaGetLastError(), "tf_analyze launch");
}

cbct_status launch_tf_analyze(int n0, int n1, int n2, const float *f, void *alpha, cudaStream_t st, int storage)
{
    if (storage == ST_BF16) return launch_tf_analyze_t(n0, n1, n2, f, static_cast<__nv_bfloat16 *>(alpha), st);
    if (storage == ST_F16) return launch_tf_analyze_t(n0, n1, n2, f, static_cast<__half *>(alpha), st);
    return launch_tf_analyze_t(n0, n1, n2, f, static_cast<float *>(alpha), st);
}

// The same step for 16-bit coefficients with two adjacent positions per lane: each
// channel is one 4-byte load of the pair, and one pair of shuffles per channel group
// serves both positions (the pair's inner shares stay in the lane). A warp covers 64
// positions: 60 outputs, the halo position on either side and one unused position at each
// end, so that every pair starts on an even position (4-byte aligned when the contiguous
// extent n0 is even, which the launcher requires; an even n0 also keeps a pair from
// straddling the periodic wrap).
constexpr int SP_OUT = 60;
// Output rows per block: one block of 16 warps per SM (126 registers, 48 KB of shared memory)
// takes 313 us at 512x512x70 BF16 in packed arithmetic (329 us position by position), two blocks of
// 6 rows 329 us, 10 warps 366 us; 18 and 20 warps spill (507 us), and so does a second plane of
// coefficients under way (383 us).
constexpr int SP_ROWS = 14, SP_WARPS = SP_ROWS + 2;

template <typename T>
__global__ void __launch_bounds__(32 * SP_WARPS, 1)
k_tf_synth_shrink_pair(int n0, int n1, int n2, int chunk, const T *__restrict__ alpha, float mu, int positivity,
                       float *__restrict__ f)
{
    using P = Pair<T>;
    using T2 = typename P::T2;
    __shared__ f32x2 s_up[2][SP_WARPS][3][32], s_dn[2][SP_WARPS][3][32];
    const int lane = threadIdx.x, w = threadIdx.y;
    const int a_out = blockIdx.x * SP_OUT, b_out = blockIdx.y * SP_ROWS;
    const int c_begin = blockIdx.z * chunk;
    const int c_end = min(n2, c_begin + chunk);
    if (c_begin >= c_end) return;
    const size_t N = (size_t)n0 * n1 * n2;
    const size_t plane = (size_t)n0 * n1;
    const int pa = a_out - 2 + 2 * lane, pb = b_out + w - 1; // the pair (pa, pa + 1), unwrapped
    const size_t inplane = (size_t)wrapi(pb, n1) * n0 + wrapi(pa, n0);
    const bool out_lane = lane >= 1 && lane <= SP_OUT / 2 && pa < n0; // n0 even: pa + 1 < n0 too
    const bool out_row = w >= 1 && w <= SP_ROWS && pb < n1;

    T2 nxt[27];
    auto fetch = [&](int c) {
        const T2 *src = reinterpret_cast<const T2 *>(alpha + (size_t)wrapi(c, n2) * plane + inplane);
        const size_t stride = N / 2; // channels in pairs (N is even)
#pragma unroll
        for (int ch = 0; ch < 27; ++ch) nxt[ch] = src[(size_t)ch * stride];
    };
    fetch(c_begin - 1);
    f32x2 w_m2[3] = {0ull, 0ull, 0ull}, w_m1[3] = {0ull, 0ull, 0ull}; // axis-2 inputs at planes cp-2, cp-1
    int buf = 0;
    for (int cp = c_begin - 1; cp <= c_end; ++cp, buf ^= 1) {
        T2 cur[27];
#pragma unroll
        for (int ch = 0; ch < 27; ++ch) cur[ch] = nxt[ch];
        if (cp < c_end) fetch(cp + 1);
        // vector shrinkage, Eq. (2), for both positions
        f32x2 s2 = 0ull;
#pragma unroll
        for (int ch = 1; ch < 27; ++ch) {
            const f32x2 a = P::get(cur[ch]);
            s2 = fma2(a, a, s2);
        }
        const float na = sqrtf(lo2(s2)), nb = sqrtf(hi2(s2));
        const f32x2 sc = mul2(pk(na > mu ? 1.0f - mu / na : 0.0f, nb > mu ? 1.0f - mu / nb : 0.0f), splat(1.0f / 64.0f));
        const f32x2 sc2 = add2(sc, sc), scr = mul2(splat(SYN_R), sc), scn = mul2(splat(-SYN_R), sc);
        // axis 0: the even position takes lane - 1's odd one and its own odd one; the odd position takes
        // its own even one and lane + 1's even one
        f32x2 u[9];
#pragma unroll
        for (int mn = 0; mn < 9; ++mn) {
            f32x2 a0 = P::get(cur[3 * mn]), a1 = P::get(cur[3 * mn + 1]), a2 = P::get(cur[3 * mn + 2]);
            if (mn == 0) { // (channel 0 is not shrunk)
                a0 = mul2(splat(1.0f / 64.0f), a0);
                a2 = mul2(sc, a2);
            }
            const f32x2 q = mn ? mul2(sc, sub2(a0, a2)) : sub2(a0, a2);
            const f32x2 up = fma2(scr, a1, q), dn = fma2(scn, a1, q);
            u[mn] = add2(fma2(mn ? sc2 : splat(2.0f), add2(a0, a2), pk(__shfl_up_sync(0xffffffffu, hi2(up), 1), lo2(up))),
                         pk(hi2(dn), __shfl_down_sync(0xffffffffu, lo2(dn), 1)));
        }
        // axis 1 (warps) through shared memory
        f32x2 mid[3];
#pragma unroll
        for (int n = 0; n < 3; ++n) {
            const f32x2 q = sub2(u[3 * n], u[3 * n + 2]);
            mid[n] = add2(u[3 * n], u[3 * n + 2]);
            s_up[buf][w][n][lane] = fma2(splat(SYN_R), u[3 * n + 1], q);
            s_dn[buf][w][n][lane] = fma2(splat(-SYN_R), u[3 * n + 1], q);
        }
        __syncthreads();
        if (out_row) {
            f32x2 wv[3];
#pragma unroll
            for (int n = 0; n < 3; ++n)
                wv[n] = add2(fma2(splat(2.0f), mid[n], s_up[buf][w - 1][n][lane]), s_dn[buf][w + 1][n][lane]);
            if (cp >= c_begin + 1 && out_lane) {
                const f32x2 ends = sub2(add2(w_m2[0], wv[0]), add2(w_m2[2], wv[2]));
                const f32x2 o2 = add2(fma2(splat(2.0f), add2(w_m1[0], w_m1[2]), mul2(splat(SYN_R), sub2(w_m2[1], wv[1]))), ends);
                float2 o = make_float2(lo2(o2), hi2(o2));
                if (positivity) {
                    o.x = o.x < 0.0f ? 0.0f : o.x;
                    o.y = o.y < 0.0f ? 0.0f : o.y;
                }
                *reinterpret_cast<float2 *>(f + (size_t)(cp - 1) * plane + (size_t)pb * n0 + pa) = o;
            }
#pragma unroll
            for (int n = 0; n < 3; ++n) {
                w_m2[n] = w_m1[n];
                w_m1[n] = wv[n];
            }
        }
    }
}

template <typename T>
static cbct_status launch_tf_synth_shrink_pair(int n0, int n1, int n2, const T *alpha, float mu, int positivity,
                                               float *f, cudaStream_t st)
{
    constexpr int rows = SP_ROWS;
    static Residency residency;
    int slots = 0;
    const cudaError_t e = resident_blocks(reinterpret_cast<const void *>(k_tf_synth_shrink_pair<T>), 32 * SP_WARPS, residency, &slots);
    if (e != cudaSuccess) return check_cuda(e, "tf_synth_shrink occupancy");
    const long long tiles = (long long)((n0 + SP_OUT - 1) / SP_OUT) * ((n1 + rows - 1) / rows);
    const int chunk = fused_chunk(tiles, n2, slots);
    dim3 grid((n0 + SP_OUT - 1) / SP_OUT, (n1 + rows - 1) / rows, (n2 + chunk - 1) / chunk);
    CBCT_TIMED(CBCT_KERNEL_TF_SYNTH, st,
               k_tf_synth_shrink_pair<T><<<grid, dim3(32, SP_WARPS), 0, st>>>(n0, n1, n2, chunk, alpha, mu, positivity, f));
    return check_cuda(cudaGetLastError(), "tf_synth_shrink launch");
}

template <typename TA_T>
static cbct_status launch_tf_synth_shrink_t(int n0, int n1, int n2, const TA_T *alpha, float mu, int positivity,
                                            float *f, cudaStream_t st)
{
    // 16-bit coefficients of an even contiguous extent: two positions per lane (aligned pairs;
    // the array's base is at least 4-byte aligned, as for any 16-bit tensor the API accepts)
    if constexpr (sizeof(TA_T) == 2)
        if (n0 % 2 == 0 && (reinterpret_cast<uintptr_t>(alpha) & 3) == 0 && (reinterpret_cast<uintptr_t>(f) & 7) == 0)
            return launch_tf_synth_shrink_pair(n0, n1, n2, alpha, mu, positivity, f, st);
    static Residency residency;
    int slots = 0;
    const cudaError_t e = resident_blocks(reinterpret_cast<const void *>(k_tf_synth_shrink<TA_T>), SY_THREADS, residency, &slots);
    if (e != cudaSuccess) return check_cuda(e, "tf_synth_shrink occupancy");
    const long long tiles = (long long)((n0 + SY_OUT - 1) / SY_OUT) * ((n1 + SY_ROWS - 1) / SY_ROWS);
    const int chunk = fused_chunk(tiles, n2, slots);
    dim3 grid((n0 + SY_OUT - 1) / SY_OUT, (n1 + SY_ROWS - 1) / SY_ROWS, (n2 + chunk - 1) / chunk);
    CBCT_TIMED(CBCT_KERNEL_TF_SYNTH, st,
               k_tf_synth_shrink<TA_T><<<grid, dim3(32, SY_WARPS), 0, st>>>(n0, n1, n2, chunk, alpha, mu, positivity, f));
    return check_cuda(cudaGetLastError(), "tf_synth_shrink launch");
}

cbct_status launch_tf_synth_shrink(int n0, int n1, int n2, const void *alpha, float mu,
                                   int positivity, float *f, cudaStream_t st, int storage)
{
    if (storage == ST_BF16)
        return launch_tf_synth_shrink_t(n0, n1, n2, static_cast<const __nv_bfloat16 *>(alpha), mu, positivity, f, st);
    if (storage == ST_F16)
        return launch_tf_synth_shrink_t(n0, n1, n2, static_cast<const __half *>(alpha), mu, positivity, f, st);
    return launch_tf_synth_shrink_t(n0, n1, n2, static_cast<const float *>(alpha), mu, positivity, f, st);
}

} // namespace cbct

namespace cbct {

// ------------------------------------------------------------------------------------
// Fused shrinkage step of Algorithm A2 (steps 3-4, then step 1 of the next iteration):
//   f_new = H(W^T T_mu W x)   and optionally   v = f_new + c (f_new - f_old).
// The 27 coefficients never leave the SM: HBM traffic is one read of x (halo re-reads hit
// L2) and the writes of f_new (and v, with one read of f_old).
//
// A warp covers 32 consecutive positions along axis 0 (28 outputs and two halo positions on
// either side: the coefficients of the outputs' neighbours need x one position further out)
// of two adjacent rows, whose values a lane holds as pairs and treats with one instruction
// (fma.rn.f32x2 and its kind: each half rounds like the scalar operation). A block stacks
// FR_WARPS such pairs along axis 1, the first and last of them halo rows, and marches along
// axis 2. Per plane every lane
//   1. analyses along axis 2 from the three x planes it holds in registers (the next plane
//      is loaded while this one is computed),
//   2. along axis 1: each row's neighbour is the pair's other row or, through shared memory,
//      the adjacent warp's near row,
//   3. along axis 0 from its neighbour lanes by shuffles, giving its positions' 27
//      coefficients, which it shrinks in registers (Eq. (2)),
// and then synthesises back as the shrink + synthesis kernel does: shares of neighbouring
// lanes by shuffles, of neighbouring rows within the pair or through shared memory, of
// neighbouring planes in registers, finishing the output plane one behind the analysed one.
//
// Bound by instruction issue (57%), the packed-FP32 pipe and the shuffles; 16 warps (120
// registers) per SM. 512x512x70: 333 us (one row per warp, 22 warps: 377 us), z-fastest as in
// the iteration 358 us (416 us). Volumes whose tiles of 16 warps end in a poor last wave take 12 warps (rule at
// the launcher).
// ------------------------------------------------------------------------------------
constexpr int FR_OUT = 28; // output positions per warp along axis 0
constexpr int fr_rows(int warps) { return 2 * warps - 4; } // output rows per block along axis 1

// The frame with plain taps: [1, 2, 1], [1, 0, -1] and [1, -2, 1] stand for 4 h_0, (4 / sqrt(2)) h_1
// and -4 h_2, so that a triple takes four operations. Of x / 64, a coefficient with j factors h_1 is then
// 1 / sqrt(2)^j times the frame's (its sign is its own on both ways), the squared norm is the sum of
// 2^j A^2, and synthesis counts the middle tap triple twice, of A / 64: all powers of two, which
// round nothing (values below 2^-114 lose their last bits), and no intermediate is larger than the frame's.
__device__ __forceinline__ void ana3_plain(f32x2 p, f32x2 c, f32x2 n, f32x2 &o0, f32x2 &o1, f32x2 &o2)
{
    const f32x2 s = add2(n, p);
    o0 = fma2(splat(2.0f), c, s);
    o1 = sub2(n, p);
    o2 = fma2(splat(-2.0f), c, s);
}
// shares of a triple: to p + 1, half of that to p itself, to p - 1
__device__ __forceinline__ void syn_shares_plain(f32x2 a0, f32x2 a1, f32x2 a2, f32x2 &up, f32x2 &half, f32x2 &dn)
{
    const f32x2 q = add2(a0, a2);
    up = fma2(splat(2.0f), a1, q);
    dn = fma2(splat(-2.0f), a1, q);
    half = sub2(a0, a2);
}

template <int FR_WARPS>
__global__ void __launch_bounds__(32 * FR_WARPS, 1)
k_tf_shrink_fused(int n0, int n1, int n2, int p0, int chunk, const float *__restrict__ x, float mu, int positivity,
                  float *__restrict__ fnew, const float *__restrict__ fold, float coef, float *__restrict__ vout)
{
    constexpr int FR_ROWS = fr_rows(FR_WARPS);
    chain_wait();
    __shared__ f32x2 s_t[2][FR_WARPS][3][32];                      // axis-2 analysis of each pair
    __shared__ float s_up[2][FR_WARPS][3][32], s_dn[2][FR_WARPS][3][32]; // axis-1 synthesis shares to the pairs beside
    const int lane = threadIdx.x, w = threadIdx.y;
    const int a_out = blockIdx.x * FR_OUT, b_out = blockIdx.y * FR_ROWS;
    const int c_begin = blockIdx.z * chunk;
    const int c_end = min(n2, c_begin + chunk);
    if (c_begin >= c_end) return;
    const size_t plane = (size_t)p0 * n1;
    const int pa = a_out + lane - 2, pb = b_out + 2 * w - 2;  // this lane's position and first row (unwrapped)
    const size_t in0 = (size_t)wrapi(pb, n1) * p0 + wrapi(pa, n0), in1 = (size_t)wrapi(pb + 1, n1) * p0 + wrapi(pa, n0);
    const bool out_pair = w >= 1 && w <= FR_WARPS - 2 && pb < n1;
    const bool out_lane = lane >= 2 && lane < 2 + FR_OUT && pa < n0;
    const int wu = w > 0 ? w - 1 : 0, wd = w < FR_WARPS - 1 ? w + 1 : w; // (the outermost halo rows' coefficients are not used)
    auto load = [&](int c) {
        const float *src = x + (size_t)wrapi(c, n2) * plane;
        return pk(__ldg(src + in0), __ldg(src + in1));
    };
    const f32x2 r64 = splat(1.0f / 64.0f);

    // x / 64 of these positions at planes cp - 1, cp, cp + 1 (cp: the analysed plane)
    f32x2 xm = mul2(load(c_begin - 2), r64), x0 = mul2(load(c_begin - 1), r64), xp = mul2(load(c_begin), r64);
    f32x2 w_m2[3] = {0ull, 0ull, 0ull}, w_m1[3] = {0ull, 0ull, 0ull}; // axis-2 synthesis inputs at cp-2, cp-1
    int buf = 0;
    for (int cp = c_begin - 1; cp <= c_end; ++cp, buf ^= 1) {
        const f32x2 xn = cp < c_end ? load(cp + 2) : 0ull;
        // 1. analysis along axis 2
        f32x2 t[3];
        ana3_plain(xm, x0, xp, t[0], t[1], t[2]);
#pragma unroll
        for (int n = 0; n < 3; ++n) s_t[buf][w][n][lane] = t[n];
        __syncthreads();
        // 2. along axis 1: u[m][n]
        f32x2 u[3][3];
#pragma unroll
        for (int n = 0; n < 3; ++n) {
            const float above = hi2(s_t[buf][wu][n][lane]), below = lo2(s_t[buf][wd][n][lane]);
            ana3_plain(pk(above, lo2(t[n])), t[n], pk(hi2(t[n]), below), u[0][n], u[1][n], u[2][n]);
        }
        // 3. along axis 0: alpha[l + 3m + 9n]
        f32x2 al[27];
#pragma unroll
        for (int m = 0; m < 3; ++m)
#pragma unroll
            for (int n = 0; n < 3; ++n) {
                const f32x2 pv = __shfl_up_sync(0xffffffffu, u[m][n], 1);
                const f32x2 nv = __shfl_down_sync(0xffffffffu, u[m][n], 1);
                ana3_plain(pv, u[m][n], nv, al[3 * m + 9 * n], al[1 + 3 * m + 9 * n], al[2 + 3 * m + 9 * n]);
            }
        // vector shrinkage, Eq. (2): squares summed by their number j of factors h_1
        f32x2 sj[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
        for (int ch = 1; ch < 27; ++ch) {
            const int j = (ch % 3 == 1) + (ch / 3 % 3 == 1) + (ch / 9 == 1);
            sj[j] = fma2(al[ch], al[ch], sj[j]);
        }
        const f32x2 s2 = fma2(splat(2.0f), fma2(splat(2.0f), fma2(splat(2.0f), sj[3], sj[2]), sj[1]), sj[0]);
        const float na = sqrtf(lo2(s2)), nb = sqrtf(hi2(s2));
        const f32x2 scale = mul2(pk(na > mu ? 1.0f - mu / na : 0.0f, nb > mu ? 1.0f - mu / nb : 0.0f), r64);
        al[0] = mul2(al[0], r64);
#pragma unroll
        for (int ch = 1; ch < 27; ++ch) al[ch] = mul2(al[ch], scale);
        // synthesis along axis 0 (lanes), then the shares along axis 1
        f32x2 us[9];
#pragma unroll
        for (int mn = 0; mn < 9; ++mn) {
            f32x2 up, half, dn;
            syn_shares_plain(al[3 * mn], al[3 * mn + 1], al[3 * mn + 2], up, half, dn);
            us[mn] = add2(fma2(splat(2.0f), half, __shfl_up_sync(0xffffffffu, up, 1)), __shfl_down_sync(0xffffffffu, dn, 1));
        }
        f32x2 up[3], half[3], dn[3];
#pragma unroll
        for (int n = 0; n < 3; ++n) {
            syn_shares_plain(us[3 * n], us[3 * n + 1], us[3 * n + 2], up[n], half[n], dn[n]);
            s_up[buf][w][n][lane] = hi2(up[n]);
            s_dn[buf][w][n][lane] = lo2(dn[n]);
        }
        __syncthreads();
        if (out_pair) {
            f32x2 wv[3];
#pragma unroll
            for (int n = 0; n < 3; ++n)
                wv[n] = add2(fma2(splat(2.0f), half[n], pk(s_up[buf][wu][n][lane], lo2(up[n]))),
                             pk(hi2(dn[n]), s_dn[buf][wd][n][lane]));
            // synthesis along axis 2: plane cp - 1 from planes cp - 2, cp - 1, cp
            if (cp >= c_begin + 1 && out_lane) {
                const size_t idx = (size_t)(cp - 1) * plane + (size_t)pb * p0 + pa;
                const f32x2 ends = add2(add2(w_m2[0], w_m2[2]), add2(wv[0], wv[2]));
                const f32x2 o2 = fma2(splat(2.0f), add2(sub2(w_m1[0], w_m1[2]), sub2(w_m2[1], wv[1])), ends);
                float o[2] = {lo2(o2), hi2(o2)};
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    if (pb + r >= n1) break; // an odd number of rows
                    if (positivity && o[r] < 0.0f) o[r] = 0.0f;
                    const size_t at = idx + (size_t)r * p0;
                    fnew[at] = o[r];
                    if (vout) vout[at] = fmaf(coef, o[r] - __ldg(fold + at), o[r]);
                }
            }
#pragma unroll
            for (int n = 0; n < 3; ++n) {
                w_m2[n] = w_m1[n];
                w_m1[n] = wv[n];
            }
        }
        xm = x0;
        x0 = xp;
        xp = mul2(xn, r64); // (here and not at the load, which this plane's work hides)
    }
}

cbct_status tf_prepare() { return CBCT_OK; }

// A launch of the fused step with WARPS warps per block, and its cost in planes of a block, one after another.
struct FusedPlan {
    dim3 grid;
    int chunk;
    long long cost;
};
template <int WARPS> static cudaError_t fused_plan(int n0, int n1, int n2, FusedPlan *p)
{
    static Residency residency;
    int slots = 0;
    const cudaError_t e = resident_blocks(reinterpret_cast<const void *>(k_tf_shrink_fused<WARPS>), 32 * WARPS, residency, &slots);
    if (e != cudaSuccess) return e;
    const int tx = (n0 + FR_OUT - 1) / FR_OUT, ty = (n1 + fr_rows(WARPS) - 1) / fr_rows(WARPS);
    p->chunk = fused_chunk((long long)tx * ty, n2, slots, 2.0, &p->cost);
    p->grid = dim3(tx, ty, (n2 + p->chunk - 1) / p->chunk);
    return cudaSuccess;
}

// 16 warps share their halo rows best, but their few large blocks may leave most of a wave empty (256x256x8: 100
// blocks on 152 SMs). A plane costs a block of 16 warps 1.85 us and one of 12 warps 1.40 us (nearly the same at every
// size), so 12 warps where their planes are fewer than 1.32 times as many. Measured (16 | 12 warps, planes): 256x256x8 19.2 | 15.0 us (10 |
// 10), 256x256x20 33.9 | 31.3 us (18 | 22), 450x430x60 223.7 | 220.5 us (124 | 160), 512x512x20 110 | 118 us (60 | 84),
// 512x512x70 332 | 354 us (185 | 259). 8, 10, 11 and 14 warps were no better where 12 win, but for a few per cent.
cbct_status launch_tf_shrink_fused(int n0, int n1, int n2, int p0, const float *x, float mu, int positivity, float *fnew,
                                   const float *fold, float coef, float *vout, cudaStream_t st)
{
    FusedPlan p{}, q{};
    cudaError_t e = fused_plan<16>(n0, n1, n2, &p);
    if (e == cudaSuccess) e = fused_plan<12>(n0, n1, n2, &q);
    if (e != cudaSuccess) return check_cuda(e, "tf_shrink_fused occupancy");
    const bool few = 100 * q.cost < 132 * p.cost;
    const auto kernel = few ? k_tf_shrink_fused<12> : k_tf_shrink_fused<16>;
    if (few) p = q;
    CBCT_TIMED(CBCT_KERNEL_TF_SYNTH, st,
               launch_chained(kernel, p.grid, dim3(32, few ? 12 : 16), 0, st, n0, n1, n2, p0, p.chunk, x, mu, positivity, fnew,
                              fold, coef, vout));
    return check_cuda(cudaGetLastError(), "tf_shrink_fused launch");
}

} // namespace cbct
