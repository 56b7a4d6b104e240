// Forward projector P (Eq. (1), Section 2.2.1): host dispatcher. Chooses the column-group
// size of each launch, opts the kernel into its shared memory and launches it. The kernel
// itself is in project_kernel.cuh.
#include <atomic>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <tuple>

#include "async.cuh"
#include "project.cuh"

namespace cbct {

int project_num_blocks(const GeomDev &G)
{
    const int rows = proj_rows_per_thread(G) * proj_threads(G);
    return G.nviews * G.nu * ((G.nv + rows - 1) / rows);
}

// The documented limit of the accepted grids: 16 bytes per possible segment (in groups of
// 16) and per slab 16 staged values, 17 table entries and two totals. The kernel's own need
// with the smallest group (project_smem) is below it for every grid.
size_t project_smem_bytes(const GeomDev &G)
{
    const size_t segs = ((size_t)G.nx + G.ny + 2 + 15) / 16 * 16;
    const size_t lists = ((size_t)G.nx + G.ny + 2 + 3) / 4 * 4, lines = 16 * (((size_t)G.nz + 9) / 4 * 4);
    return 16 * segs + sizeof(float) * ((lines > lists ? lines : lists) + (size_t)G.nz * 19);
}

// Quads of slabs per warp in the table build, 4 or 8: with 8 there are half the parts, of twice
// the columns, so fewer passes end in a scan (each pass costs about 8 instructions per column
// and 60 around them), but the longest chain doubles. The split with the least total work plus
// longest chain. Measured with groups of 80 (4 | 8): 18 quads on 6 warps 661 | 703 us, 16 quads
// 206 | 187 us, 9 quads 315 | 355 us, 5 quads 185 | 211 us, as the costs order them; in between
// the costs may lie within 3-6% of each other, and the order was not measured there.
static int quads_per_warp(const GeomDev &G, int threads, int sg)
{
    const int nq = G.zp / 4, warps = threads / 32;
    int best = 8, best_cost = 1 << 30;
    for (int qw = 8; qw >= 4; qw /= 2) {
        if (nq > 16 * qw && qw < 8) break; // more parts take more shared memory for their offsets
        const int passes = (nq + qw - 1) / qw, rounds = (passes + warps - 1) / warps;
        const int cost = (passes + rounds) * (8 * ((sg * qw + 31) / 32) + 60);
        if (cost < best_cost) {
            best_cost = cost;
            best = qw;
        }
    }
    return best;
}

static const void *kernel_for(int qw, int mode, int storage, int rows, int fill)
{
    return qw == 4 ? project_kernel<4>(mode, storage, rows, fill) : project_kernel<8>(mode, storage, rows, fill);
}

static int group_index(int sg)
{
    for (int i = 0; i < PROJECT_N_GROUP_SIZES; ++i)
        if (PROJECT_GROUP_SIZES[i] == sg) return i;
    return -1;
}

// per-device record of the shared-memory opt-in, one per instantiation
static std::atomic<unsigned long long> g_optin[2][3][3][2][3];

static cbct_status optin(int qw, int mode, int storage, int rows, int fill, const void **fn)
{
    *fn = kernel_for(qw, mode, storage, rows, fill);
    if (!*fn) return set_error(CBCT_ERR_UNSUPPORTED, "project: no kernel for mode %d, storage %d", mode, storage);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return check_cuda(e, "project device");
    std::atomic<unsigned long long> &done =
        g_optin[qw / 8][mode][storage == ST_BF16 ? 1 : storage == ST_F16 ? 2 : 0][rows - 1][fill];
    const unsigned long long bit = 1ull << (dev & 63);
    if (done.load() & bit) return CBCT_OK;
    e = cudaFuncSetAttribute(*fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PROJECT_SMEM_LIMIT);
    if (e != cudaSuccess) return check_cuda(e, "project attribute");
    done.fetch_or(bit);
    return CBCT_OK;
}

static std::atomic<int> g_forced_group{0}; // 0: automatic

static int fill_of(const GeomDev &G, int zpitch)
{
    return zpitch % 4 ? FILL_PACKED : G.zp <= TMA_BOX_MAX ? FILL_GATHER : FILL_BULK;
}

struct GroupChoice {
    int sg, qw, grid; // columns per group, quads per warp, resident blocks on the device
    ProjPlan plan;
    size_t smem;
};

// Tables of `groups` groups of sg columns; one line buffer where two do not fit.
static bool make_plan(const GeomDev &G, int threads, int sg, int groups, GroupChoice *c)
{
    c->sg = sg;
    c->qw = quads_per_warp(G, threads, sg * groups);
    for (int nbuf = 2; nbuf >= 1; --nbuf) {
        c->plan = project_plan(G, sg * groups, c->qw, nbuf);
        c->smem = project_smem(G, c->plan, c->qw);
        if (c->smem <= PROJECT_SMEM_LIMIT) return true;
    }
    return false;
}

// The group size of a launch. A table costs its block about as much as building and walking 60
// columns (the waits, the barrier, the scans, the rows' set-up), which a larger table spreads
// over more columns; but it takes more shared memory, so fewer blocks stay resident to fill
// each other's waits:
//     (1 + TABLE_COST / columns) * (REF_WARPS / resident warps)^OCC_EXP,
// a tenth more where the build's accesses share banks, a twentieth more where it is not unrolled
// (tables other than 80 and 112 columns). Measured (us, columns: 48 | 80 | 112):
// the paper's finest grid 857 | 647 | 660 (4, 4, 3 blocks), its level 1 395 | 302 | 271, its level
// 2 247 | 179 | 168, 256x256x64 240 | 186 | 201, 512x512x128 971 | 1014 | 1680 (4, 2, 1 blocks).
constexpr double TABLE_COST = 60.0, REF_WARPS = 24.0, OCC_EXP = 0.6;

static cbct_status choose_group(const GeomDev &G, int threads, int mode, int storage, int fill, GroupChoice *out)
{
    const int forced = g_forced_group.load();
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return check_cuda(e, "project device");
    const int rows = fill == FILL_GATHER ? proj_rows_per_thread(G) : 2;
    using Key = std::tuple<int, int, int, int, int, int, int, int>; // all that the occupancy and the plans depend on
    static std::mutex mu;
    static std::map<Key, GroupChoice> cache;
    const Key key{dev, mode, storage, threads, rows, G.nz, fill, forced};
    {
        std::lock_guard<std::mutex> lk(mu);
        auto it = cache.find(key);
        if (it != cache.end()) {
            *out = it->second;
            return CBCT_OK;
        }
    }
    GroupChoice best{}, c{};
    const bool use_forced = forced && make_plan(G, threads, forced, 1, &c);
    double best_cost = 1e300;
    for (int i = 0; i <= PROJECT_N_GROUP_SIZES; ++i) {
        const int groups = i < PROJECT_N_GROUP_SIZES ? 1 : 2, sg = groups == 1 ? PROJECT_GROUP_SIZES[i] : 56;
        if ((use_forced && (sg != forced || groups > 1)) || !make_plan(G, threads, sg, groups, &c)) continue;
        const void *fn = nullptr;
        cbct_status r = optin(c.qw, mode, storage, rows, fill, &fn);
        if (r != CBCT_OK) return r;
        int nb = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, threads + 32, c.smem);
        if (e != cudaSuccess) return check_cuda(e, "project occupancy");
        if (nb < 1) continue;
        c.grid = nb * device_sm_count();
        const double warps = (double)nb * (threads / 32);
        const bool banks = c.qw == 4 && c.plan.nb * c.plan.pitch % 32 != 16;
        const bool unrolled = c.plan.sg == 80 || c.plan.sg == 112;
        const double cost = (1.0 + TABLE_COST / c.plan.sg) * std::pow(REF_WARPS / warps, OCC_EXP) * (banks ? 1.1 : 1.0) *
                            (unrolled ? 1.0 : 1.05);
        if (cost <= best_cost) {
            best_cost = cost;
            best = c;
        }
    }
    if (!best.sg) return set_error(CBCT_ERR_UNSUPPORTED, "project: grid too large for the projector's shared memory (nx + ny and nz)");
    std::lock_guard<std::mutex> lk(mu);
    cache[key] = best;
    *out = best;
    return CBCT_OK;
}

cbct_status project_set_group(int sg)
{
    if (sg != 0 && group_index(sg) < 0)
        return set_error(CBCT_ERR_INVALID_ARG, "set_project_group: %d is not one of the compiled group sizes", sg);
    g_forced_group.store(sg);
    return CBCT_OK;
}

cbct_status project_group_of(const GeomDev &G, int *sg)
{
    GroupChoice c{};
    const cbct_status st = choose_group(G, proj_threads(G), PM_PLAIN, ST_F32, fill_of(G, G.zp), &c);
    *sg = c.sg;
    return st;
}

cbct_status project_prepare()
{
    cbct_status t = trace_table_prepare();
    if (t != CBCT_OK) return t;
    for (int qw = 4; qw <= 8; qw *= 2)
        for (int mode = PM_PLAIN; mode < PM_COUNT; ++mode)
            for (int storage = ST_F32; storage <= ST_F16; ++storage)
                for (int rows = 1; rows <= 2; ++rows)
                    for (int fill = FILL_GATHER; fill <= FILL_BULK; ++fill) {
                        const void *fn = nullptr;
                        cbct_status r = optin(qw, mode, storage, rows, fill, &fn);
                        if (r != CBCT_OK) return r;
                    }
    return CBCT_OK;
}

EncodeTiled encode_tiled()
{
    static const EncodeTiled fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess || q != cudaDriverEntryPointSuccess) p = nullptr;
        return reinterpret_cast<EncodeTiled>(p);
    }();
    return fn;
}

// The volume as a matrix of nx ny lines of zp values; a box is one line of `pitch` slots (the
// slots past zp are filled with zeros).
static cbct_status line_map(const GeomDev &G, const float *f, int pitch, CUtensorMap *map)
{
    const EncodeTiled enc = encode_tiled();
    if (!enc) return set_error(CBCT_ERR_CUDA, "project: the driver has no cuTensorMapEncodeTiled");
    const cuuint64_t dims[2] = {(cuuint64_t)G.zp, (cuuint64_t)G.nx * G.ny}, strides[1] = {(cuuint64_t)G.zp * 4};
    const cuuint32_t box[2] = {(cuuint32_t)pitch, 1}, step[2] = {1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float *>(f), dims, strides, box, step,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(CBCT_ERR_CUDA, "project: tensor map of the volume (%d)", (int)r);
    return CBCT_OK;
}

cbct_status launch_project(const GeomDev &G, const float *f, int zpitch, const float *y, void *out, int mode,
                           double *partials, float count_thr, cudaStream_t st, int storage, Scalars *sc,
                           const void *traces, int col_first, int ncols)
{
    if (project_smem_bytes(G) > PROJECT_SMEM_LIMIT)
        return set_error(CBCT_ERR_UNSUPPORTED, "project: grid too large for the projector's shared memory (nx + ny and nz)");
    if (mode == PM_COUNT) return launch_project_count(G, partials, count_thr, st);
    const int threads = proj_threads(G), fill = fill_of(G, zpitch);
    const int rows = fill == FILL_GATHER ? proj_rows_per_thread(G) : 2;
    if (ncols == 0) ncols = G.nviews * G.nu;
    // (views x columns < 2^31 / nv, so the items fit 31 bits)
    unsigned nitems = (unsigned)ncols * ((G.nv + rows * threads - 1) / (rows * threads));
    // the packed layout takes the padded one's plan: the same tables, hence the same sums
    GroupChoice c{};
    cbct_status r = choose_group(G, threads, mode, storage, fill_of(G, G.zp), &c);
    if (r != CBCT_OK) return r;
    const void *fn = nullptr;
    r = optin(c.qw, mode, storage, rows, fill, &fn);
    if (r != CBCT_OK) return r;
    if (fill == FILL_PACKED) {
        int nb = 0;
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, threads + 32, c.smem);
        if (e != cudaSuccess) return check_cuda(e, "project occupancy");
        c.grid = (nb > 0 ? nb : 1) * device_sm_count();
    }
    alignas(64) CUtensorMap map;
    memset(&map, 0, sizeof(map));
    if (fill == FILL_GATHER) {
        r = line_map(G, f, c.plan.pitch, &map);
        if (r != CBCT_OK) return r;
    }
    const unsigned grid = nitems < (unsigned)c.grid ? nitems : (unsigned)c.grid;
    unsigned ucols = (unsigned)ncols;
    GeomDev g = G;
    const float *rec = static_cast<const float *>(traces);
    void *args[] = {&g, &map, &f, &zpitch, &c.plan, &y, &out, &partials, &sc, &rec, &col_first, &ucols, &nitems};
    ProfToken tok = prof_start(CBCT_KERNEL_PROJECT, st);
    cudaError_t e = launch_chained(fn, dim3(grid), dim3((unsigned)threads + 32), args, c.smem, st);
    prof_stop(tok, st);
    note_launch();
    if (e != cudaSuccess) cudaGetLastError(); // the error is returned, not left pending
    return check_cuda(e, "project launch");
}

} // namespace cbct
