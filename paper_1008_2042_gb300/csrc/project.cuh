// Forward projector P: launch geometry and shared-memory sizing common to the host
// dispatcher (project.cu) and the kernel's instantiations (project_kernel.cuh).
#pragma once
#include <cuda.h>

#include <cstddef>

#include "cbct_internal.cuh"

namespace cbct {

constexpr int PROJ_THREADS = 192; // consumer threads per block at most; each owns one or two imager rows
#ifndef CBCT_PROJ_MIN_BLOCKS
// resident blocks per SM the register budget is sized for (72 registers a thread; the kernels with 8 quads per warp
// and two rows per thread spill 24 bytes, in the modes of CGLS up to 44)
#define CBCT_PROJ_MIN_BLOCKS 4
#endif
// fewest threads of a block: short imagers would leave the table build to one warp
constexpr int PROJ_MIN_THREADS = 64;
constexpr float P_INF = 3.0e38f;

// imager rows per thread, threads of a block (a multiple of 32, every lane present for warp
// votes and shuffles) and so the imager rows one block covers
static inline int proj_rows_per_thread(const GeomDev &G) { return G.nv > PROJ_THREADS ? 2 : 1; }
static inline int proj_threads(const GeomDev &G)
{
    const int r = proj_rows_per_thread(G);
    const int t = (((G.nv + r - 1) / r + 31) / 32) * 32;
    return t < PROJ_MIN_THREADS ? PROJ_MIN_THREADS : t < PROJ_THREADS ? t : PROJ_THREADS;
}

// How a block gets the z-lines of a group: TMA gathers of four lines, a bulk copy per line (lines
// longer than a TMA box), or 4-byte copies (z-lines without padding).
enum ProjFill { FILL_GATHER = 0, FILL_BULK = 1, FILL_PACKED = 2 };
constexpr int TMA_BOX_MAX = 256; // elements along one dimension of a TMA box

// A launch's group of columns (one table) and shared-memory layout.
struct ProjPlan {
    int sg;     // columns per table
    int nbuf;   // line buffers, 1 or 2
    int nb;     // columns per part of the table build, ceil(sg / (32 / QW))
    int inv_nb; // ceil(2^16 / nb): column / nb = column * inv_nb >> 16 for every column < 128
    int pitch;  // floats from one line slot to the next
};
constexpr int BUILD_BATCH = 4; // lines a lane holds at once in the unrolled table build

// The trace table (k_trace_table): a record of 64 + 8 trace_cap bytes per (view, imager
// column), trace_cap = nx + ny + 2 rounded up to 4: a header of TRACE_HDR words, then the tau at
// which each segment ends and its voxel column iy * nx + ix.
constexpr int TRACE_HDR = 16;
static inline __host__ __device__ int trace_cap(const GeomDev &G) { return ((G.nx + G.ny + 2 + 3) / 4) * 4; }
static inline __host__ __device__ int trace_words(const GeomDev &G) { return TRACE_HDR + 2 * trace_cap(G); }
static inline size_t trace_smem(const GeomDev &G)
{
    return sizeof(float) * (2 * (size_t)trace_cap(G) + 4 * (PROJ_THREADS / 32) + (size_t)G.nx + G.ny + 2);
}

// The plan for groups of sg columns: qw quads of slabs per warp in the table build. The pitch is
// a multiple of 8 floats (four line slots are one 128-byte aligned TMA destination) and, where
// possible, puts the parts' 16-byte accesses of a quarter warp on distinct banks.
static inline ProjPlan project_plan(const GeomDev &G, int sg, int qw, int nbuf)
{
    ProjPlan p;
    p.sg = sg;
    p.nbuf = nbuf;
    p.nb = (sg * qw + 31) / 32;
    p.inv_nb = (65536 + p.nb - 1) / p.nb;
    p.pitch = (G.zp + 7) / 8 * 8;
    for (int t = p.pitch; t < p.pitch + 32 && t <= TMA_BOX_MAX; t += 8) {
        const int o = p.nb * t % 32;
        if (qw >= 8 || o == 16) {
            p.pitch = t;
            break;
        }
    }
    return p;
}
// Shared memory of one block: a line of room, and per buffer its lines, the lengths, starts and
// reciprocal lengths of their segments, and the part offsets.
static inline size_t project_smem(const GeomDev &G, const ProjPlan &p, int qw)
{
    return sizeof(float) * ((p.pitch + 31) / 32 * 32) +
           p.nbuf * sizeof(float) * ((size_t)p.sg * (p.pitch + 4) + (size_t)(32 / qw + 1) * G.zp);
}

// Column segments per group; the dispatcher (project.cu) picks one per launch. A table holds one
// group, or two groups of 56.
constexpr int PROJECT_GROUP_SIZES[] = {16, 24, 32, 40, 48, 56, 64, 80, 96};
constexpr int PROJECT_N_GROUP_SIZES = (int)(sizeof(PROJECT_GROUP_SIZES) / sizeof(int));

// The instantiation of k_project for a mode, storage type, rows per thread and ProjFill (host
// address for cudaLaunchKernel and the attribute and occupancy queries), or nullptr where it
// is not compiled. Defined for QW = 4, 8 in the project_q*.cu units.
template <int QW> const void *project_kernel(int mode, int storage, int rows, int fill);

// PM_COUNT: segments longer than count_thr (mm), one partial per block (project_trace.cu).
cbct_status launch_project_count(const GeomDev &G, double *partials, float count_thr, cudaStream_t st);

} // namespace cbct
