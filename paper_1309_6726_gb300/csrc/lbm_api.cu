// lbm_api.cu -- the C ABI declared in include/lbm.h: handle life cycle,
// packed ragged layout of a batch, stepping, observables, field access,
// checkpoints.  All arithmetic of the method runs in the kernels of
// lbm_step_tma.cu, lbm_step_cluster.cu, lbm_step.cu and lbm_aux.cu; this file
// sizes, allocates, copies, deals the tiles and launches.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include <cuda.h>
#include <cudaTypedefs.h>

#include "../../include/lbm.h"
#include "lbm_device.cuh"

namespace lbmk {
// store: 0 FP32, 1 FP16, 2 BF16 storage
cudaError_t launch_step_direct(const StepArgs &a, int ntiles, int tx,
                               int ty, int store, cudaStream_t s);
cudaError_t launch_step_tma(const StepArgs &a, const CUtensorMap *pop_maps,
                            const CUtensorMap *mask_maps,
                            const CUtensorMap *out_maps, const TileRec *sched,
                            int nslots, int grid, int tx, int ty, int store,
                            int *err, cudaStream_t s);
cudaError_t grid_step_tma(int tx, int ty, int store, int *grid);
bool plan_cluster(const int32_t *nx, const int32_t *ny, int count, int *tx,
                  int *ty, int *csize);
int active_clusters(int tx, int ty, int store, int csize);
cudaError_t launch_step_cluster(const StepArgs &a, int count, int nsteps,
                                int tx, int ty, int csize, int store,
                                cudaStream_t s);
int tma_box_x(int tx);
int tma_mask_box_x(int tx);
__global__ void k_unstream(const LatDesc *, int, const float *,
                           const uint8_t *, uint8_t, void *, bool);
__global__ void k_export(const LatDesc *, int, const void *, const uint8_t *,
                         const double *, long long, bool, float *, float *,
                         double *);
__global__ void k_settle(const LatDesc *, int, const void *, uint8_t *,
                         double *, LatState *, long long, bool);
__global__ void k_mask_agree(const LatDesc *, int, uint8_t *, long long);
__global__ void k_solid_mask(const LatDesc *, int, const uint8_t *, uint8_t,
                             uint8_t *);
__global__ void k_gather_inputs(const InPtrs *, int, const int64_t *, float *,
                                uint8_t *);
__global__ void k_mask_init_all(const LatDesc *, int, const int64_t *,
                                const int64_t *, const uint8_t *, uint8_t *);
__global__ void k_col_init_all(const LatDesc *, int, const int64_t *,
                               const int64_t *, const uint8_t *, int32_t *,
                               int16_t *, LatState *);
__global__ void k_init_rest_all(const LatDesc *, int, const int64_t *,
                                const int64_t *, const float *, const uint8_t *,
                                void *, bool);
__global__ void k_solid_mask_all(const LatDesc *, int, const int64_t *,
                                 const int64_t *, const uint8_t *, uint8_t,
                                 uint8_t *);
void launch_obs_columns(bool summed, int store, int nb, int ncols,
                        const LatDesc *desc, const int32_t *col_lat,
                        const int64_t *col_base, const void *fin,
                        const uint8_t *mask, const double *m, long long t,
                        ColObs *out, cudaStream_t s);
struct LbmObsDev;
__global__ void k_obs_reduce(const LatDesc *, const int64_t *,
                             const ColObs *, const int16_t *,
                             const LatState *, const double *, long long,
                             LbmObsDev *);
}  // namespace lbmk

using namespace lbmk;

static_assert(sizeof(lbm_obs) == 8 * 16 + 4 * 2 + 8, "lbm_obs layout");

struct lbm_handle {
    int count = 0;
    bool half = false;  // 16-bit storage (FP16 or BF16): the 15-word layout
    bool bf16 = false;  // its format
    // 0 FP32, 1 FP16, 2 BF16 (the step kernels' storage policy)
    int store() const { return half ? (bf16 ? 2 : 1) : 0; }
    // tile of the step kernel (LBM_TILE overrides, lbm_autotune picks per
    // workload); set by pick_tile
    int tx = 64, ty = 4;
    bool use_tma = true;
    // small lattices advance several steps per launch, one thread block
    // cluster of csize tiles of ctx by cty nodes each (0: they do not)
    int csize = 0, ctx = 0, cty = 0;
    std::vector<LatDesc> desc;
    std::vector<int64_t> col_base;   // first column of lattice l (all columns)
    std::vector<int64_t> in_off_host;  // first node of lattice l, unpadded (count + 1)
    int64_t ncols = 0;               // columns of all lattices
    int64_t nsec = 0;                // section columns of all lattices
    int ntiles = 0;
    int64_t pop_elems = 0, node_elems = 0;  // 32-bit words, mask bytes
    size_t max_nodes = 0;            // largest nx*ny
    // device
    void *d_arena = nullptr;       // what follows, but for what is said to be apart
    LatDesc *d_desc = nullptr;
    int32_t *d_tile_lat = nullptr; // direct kernel's tiles (apart)
    int32_t *d_col_lat = nullptr;
    int64_t *d_col_base = nullptr;
    int64_t *d_in_off = nullptr;       // node then row prefixes, 2 (count + 1)
    int64_t total_rows = 0;
    uint8_t *d_masks = nullptr;        // all solid masks, unpadded (apart, on first use)
    void *d_pop[2] = {nullptr, nullptr};
    uint8_t *d_mask = nullptr;
    double *d_m = nullptr;
    int32_t *d_col_fluid = nullptr;
    int16_t *d_wall0 = nullptr;
    LatState *d_st = nullptr;
    int64_t *d_step = nullptr;     // step count, one slot per population buffer
    ColObs *d_cols = nullptr;
    void *d_obs = nullptr;
    // [count][3] A, B and solute totals that the last launch of each
    // lbm_step call adds up, valid for step count sums_step
    double *d_sums = nullptr;
    int64_t sums_step = -1;
    float *d_canon = nullptr;      // [22][ny][nx] scratch of one lattice
    float *d_dens = nullptr;       // [3][ny][nx]
    double *d_dep = nullptr;       // [ny][nx]
    // [2 buffers][count] population maps over the ghost band for the tile
    // copies, then [2 buffers][count] over the lattice itself for the
    // output stores
    CUtensorMap *d_maps = nullptr;
    CUtensorMap *d_mask_maps = nullptr; // [count] mask maps
    TileRec *d_sched = nullptr;        // TMA kernel: tiles of each block (apart)
    int sched_grid = 0, sched_slots = 0;
    // kGraphSteps steps from cur == 0; [1]: the last launch sums the
    // lattice totals (the replay that ends an lbm_step call)
    cudaGraphExec_t graph[2] = {nullptr, nullptr};
    bool use_graph = true;
    int stall_tx = 0;  // test hook, see pick_tile
    int *d_err = nullptr;              // kernel error flags
    int cur = 0;
    int64_t steps = 0;
    cudaStream_t own = nullptr, stream = nullptr;
    bool dead = false;
    std::string err;
};

static thread_local std::string g_create_err;

static lbm_status fail(lbm_handle *h, lbm_status st, const std::string &msg) {
    // the message below reports the error: left pending it would be taken for
    // one of the next launch, of this or of another handle
    if (st == LBM_ECUDA || st == LBM_ENOMEM) cudaGetLastError();
    if (h) {
        h->err = msg;
        if (st == LBM_ECUDA) h->dead = true;
    } else {
        g_create_err = msg;
    }
    return st;
}

#define CK(h, call)                                                        \
    do {                                                                   \
        cudaError_t e_ = (call);                                           \
        if (e_ != cudaSuccess)                                             \
            return fail((h), LBM_ECUDA,                                    \
                        std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

template <class T>
static cudaError_t dalloc(T **p, size_t n) {
    return cudaMalloc((void **)p, std::max<size_t>(n, 1) * sizeof(T));
}

// Buffers of one device allocation: each is registered with its size, then
// all are placed, 256 bytes apart at least.  (One allocation per buffer and
// its release were 0.25 of the 0.41 ms that creating and destroying a 131 x 13
// lattice took.)
struct Arena {
    struct Item { void **p; size_t at; };
    std::vector<Item> items;
    size_t bytes = 0;
    template <class T>
    size_t add(T **p, size_t n) {
        const size_t at = bytes;
        items.push_back({(void **)p, at});
        bytes += (std::max<size_t>(n, 1) * sizeof(T) + 255) / 256 * 256;
        return at;
    }
    cudaError_t place(void **base) {
        cudaError_t e = cudaMalloc(base, std::max<size_t>(bytes, 256));
        if (e == cudaSuccess)
            for (Item &i : items) *i.p = (char *)*base + i.at;
        return e;
    }
};

static void free_all(lbm_handle *h) {
    void *ps[] = {h->d_arena, h->d_tile_lat, h->d_masks, h->d_sched};
    for (void *p : ps)
        if (p) cudaFree(p);
    for (cudaGraphExec_t g : h->graph)
        if (g) cudaGraphExecDestroy(g);
    if (h->own) cudaStreamDestroy(h->own);
}

static bool valid_params(const lbm_params &p, std::string &why) {
    if (!(p.tau_a > 0.5 && p.tau_b > 0.5 && p.tau_d > 0.5)) {
        why = "relaxation times must exceed 1/2";
        return false;
    }
    if (!(p.k_r >= 0.0) || !std::isfinite(p.k_r)) {
        why = "k_r must be finite and >= 0";
        return false;
    }
    if (!std::isfinite(p.g_coh) || !std::isfinite(p.g_ads) ||
        !std::isfinite(p.c_in) || !std::isfinite(p.body_force_x) ||
        std::isnan(p.m_threshold)) {
        why = "non-finite constant";
        return false;
    }
    // Deposit only grows, by the reaction: with a positive threshold a node
    // can only reach it in a step in which it reacts, which is where the
    // step kernel tests it.
    if (!(p.m_threshold > 0.0)) {
        why = "m_threshold must be > 0";
        return false;
    }
    if (p.precision != LBM_FP32 && p.precision != LBM_FP16 &&
        p.precision != LBM_BF16) {
        why = "unknown precision";
        return false;
    }
    return true;
}

// The address under which this device reads a caller's array, or null if
// it cannot: pinned or registered host memory is mapped into the device's
// address space (its device pointer), managed memory and this device's
// memory are used as they are, and so is pageable host memory where the
// device walks the host's page tables (pageable; it then reads such memory
// at the link's rate, where a copy per array cost 1.6 ms for the 128 arrays
// of 32 capillaries).  Null: another device's memory, pageable memory on a
// device that cannot address it, or an address that is no multiple of the
// element's size (a view into a byte buffer, a file mapped behind an odd
// header): the host may read and copy such an array, a device load faults.
template <class T>
static const T *device_view(const T *p, bool pageable) {
    if (!p || reinterpret_cast<uintptr_t>(p) % sizeof(T) != 0) return nullptr;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    const T *mapped = static_cast<const T *>(a.devicePointer);
    switch (a.type) {
    case cudaMemoryTypeHost:
        return mapped;
    case cudaMemoryTypeDevice:
        return a.device == dev ? mapped : nullptr;
    case cudaMemoryTypeManaged:
        return mapped ? mapped : p;
    default:
        return pageable ? p : nullptr;
    }
}
// Whether this device addresses pageable host memory as the host does.
static bool reads_pageable() {
    int dev = 0, on = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&on, cudaDevAttrPageableMemoryAccessUsesHostPageTables,
                               dev) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return on != 0;
}

// Share of solid nodes inside the lattices of a batch of `nodes` nodes, from
// evenly spaced rows, about 64k nodes in all (the outermost rows, walls of a
// capillary, are left out).  Device arrays: one strided copy for each of 32
// lattices at most.
static double solid_share(const lbm_geometry *g, int count, int64_t nodes) {
    const int64_t step = std::max<int64_t>(16, nodes >> 16);
    int64_t solid = 0, seen = 0, copies = 0;
    std::vector<uint8_t> rows;
    for (int l = 0; l < count; ++l) {
        const int64_t nx = g[l].nx, ny = g[l].ny, y0 = std::min(step, ny) / 2;
        const int64_t n = (ny - 2 - y0) / step + 1;  // rows y0, y0 + step, ... < ny - 1
        const uint8_t *src = g[l].solid + y0 * nx;
        int64_t pitch = step * nx;
        cudaPointerAttributes a;
        if (cudaPointerGetAttributes(&a, src) != cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        if (a.type == cudaMemoryTypeDevice) {
            if (l * 32LL / count < copies) continue;
            ++copies;
            rows.resize(n * nx);
            if (cudaMemcpy2D(rows.data(), nx, src, pitch, nx, n, cudaMemcpyDeviceToHost) !=
                cudaSuccess) {
                cudaGetLastError();
                continue;
            }
            src = rows.data();
            pitch = nx;
        }
        for (int64_t r = 0; r < n; ++r)
            for (int64_t x = 0; x < nx; ++x) solid += src[r * pitch + x] != 0;
        seen += n * nx;
    }
    return seen > 0 ? (double)solid / (double)seen : 0.0;
}

static void pick_tile(lbm_handle *h, const lbm_geometry *g) {
    // Measured, us per step.  FP16: 64 x 4, two 256-thread blocks per SM, on
    // every workload (sweep of 40 lattices 248 at 64 x 8, 241 at 64 x 4).
    // FP32: the same where it wins, in lattices up to 640k nodes of batches up
    // to 24M (64 x 8 / 64 x 4: 4096 x 128 20.8 / 18.7, sweep of 40 lattices
    // 252 / 244, of 100 644 / 638); its stores go to 22 planes at once, and in
    // larger planes or batches one 512-thread block of 64 x 8 with an output
    // tile is ahead (sweep of 192 lattices 1175 / 1270, of 512 3118 / 3521;
    // 2048 x 2048 box 137 / 154, preform 142 / 242).  640k nodes: both buffers
    // take 113 MB, about what L2 holds; beyond, the stores reach memory.  24M:
    // the line lies between the sweeps of 100 lattices (20M) and of 192 (38M);
    // what turns there was not isolated.  (Solid-free boxes of 6M nodes in
    // batches are past it already: 24 of 512 x 512 220 / 235.)
    constexpr int kSms = 152;
    constexpr int64_t kLargeLattice = 640000, kLargeBatch = 24000000;
    // FP32 batches with solid nodes inside, of more than L2 holds of both
    // buffers (1.2M nodes, 210 MB): 64 x 8 too.  64 x 4 stores node by node,
    // and rows with solid nodes leave holes in the sectors on their way to
    // memory; the more of them turn solid, the more it loses.  64 x 8 / 64 x 4:
    // 16 preforms of 512 x 512, 5 % solid 147 / 165, 25 % 150 / 207; random
    // solid nodes, 24 of 512 x 512, 3 % 290 / 311, and when growth has filled
    // half 227 / 346; 15 % 306 / 382; four of 4096 x 128, 3 % 101 / 101 and 79 /
    // 105; two of 790 x 800 (1.26M), 3 % 72.0 / 69.4 and 58.8 / 69.6.  At 1 %
    // 64 x 4 is ahead (24 of 512 x 512 269 / 251), as in smaller batches (four
    // preforms of 512 x 512 44.9 / 41.2, one of 790 x 800 45.2 / 42.6).
    constexpr int64_t kSolidBatch = 1200000;
    constexpr double kSolidInside = 0.02;
    int64_t small = 0, nodes = 0, most = 0;
    for (int l = 0; l < h->count; ++l) {
        const int64_t n = (int64_t)g[l].nx * g[l].ny;
        small += (int64_t)((g[l].nx + 31) / 32) * ((g[l].ny + 3) / 4);
        nodes += n;
        most = std::max(most, n);
    }
    h->tx = 64;
    h->ty = 4;
    if (!h->half &&
        (most > kLargeLattice || nodes > kLargeBatch ||
         (h->count > 1 && nodes > kSolidBatch &&
          solid_share(g, h->count, nodes) >= kSolidInside)))
        h->ty = 8;
    // Where 32 x 4 tiles leave no SM more than one tile, a step is one tile's
    // latency, which the smaller block shortens: 256 x 32 (64 tiles) 64 x 4 /
    // 32 x 4: FP32 5.5 / 4.3, FP16 5.3 / 4.5; beyond (1000 x 60, 480 tiles)
    // 5.6 / 6.6.
    if (small <= kSms) {
        h->tx = 32;
        h->ty = 4;
    }
    // One FP32 lattice of that size up to 1.5M nodes, a quarter or more of it
    // solid: 32 x 8 (preform, 64 x 8 / 32 x 8: 1024 x 1024 44.8 / 40.6, 1448 x
    // 1448 75.4 / 80.5, 2048 x 2048 142 / 170).
    if (h->ty == 8 && h->count == 1 && nodes <= 1500000 &&
        solid_share(g, 1, nodes) >= 0.25)
        h->tx = 32;
    const char *e = getenv("LBM_TILE");
    if (e) {
        int a = 0, b = 0;
        if (sscanf(e, "%dx%d", &a, &b) == 2) {
            h->tx = a;
            h->ty = b;
        }
    }
    const char *k = getenv("LBM_KERNEL");
    if (k && strcmp(k, "direct") == 0) h->use_tma = false;
    // The clusters of all lattices have to fit the device at once, so that
    // the handle advances at one tile's latency per step (figures at
    // k_step_cluster).  (A tile or kernel asked for by name is used for every
    // step.)
    if (!e && h->use_tma) {
        std::vector<int32_t> nx(h->count), ny(h->count);
        for (int l = 0; l < h->count; ++l) {
            nx[l] = g[l].nx;
            ny[l] = g[l].ny;
        }
        int c = 0;
        if (plan_cluster(nx.data(), ny.data(), h->count, &h->ctx, &h->cty, &c) &&
            active_clusters(h->ctx, h->cty, h->store(), c) >= h->count)
            h->csize = c;
    }
    const char *gr = getenv("LBM_GRAPH");
    if (gr && strcmp(gr, "0") == 0) h->use_graph = false;
    // test hook of the failure path: the first step's first tile of block 0
    // waits for bytes that never arrive (the bounded wait runs out and the
    // step reports LBM_ETIMEOUT); never set in normal use
    const char *st = getenv("LBM_TEST_STALL");
    if (st) h->stall_tx = std::min(std::max(atoi(st), 0), 1 << 20);
}

static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

// One 3-D tensor map per lattice and buffer: (x, y, plane) over the
// lattice's planes of 32-bit words including the ghost band (box = the
// kernel's tile plus halo, all planes), and one over the lattice's own nodes
// (box = the tile) for the output stores; coordinates beyond read as zeros.
// (`up` holds what is uploaded; the caller keeps it until the stream has it.)
static bool make_maps(lbm_handle *h, std::vector<CUtensorMap> &up, std::string &why) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc) {
        why = "cuTensorMapEncodeTiled unavailable";
        return false;
    }
    const int count = h->count;
    const size_t esz = 4;
    up.resize(5 * (size_t)count);
    CUtensorMap *maps = up.data(), *mmaps = maps + 4 * (size_t)count;
    const cuuint64_t npl = h->half ? NW16 : NPOP;
    const CUtensorMapDataType pty = CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    for (int b = 0; b < 2; ++b) {
        for (int l = 0; l < count; ++l) {
            const LatDesc &d = h->desc[l];
            const cuuint64_t rows = (cuuint64_t)(d.ny + 2 * GHOST);
            cuuint64_t dims[3] = {(cuuint64_t)d.pitch, rows, npl};
            cuuint64_t strides[2] = {(cuuint64_t)d.pitch * esz, (cuuint64_t)d.plane * esz};
            cuuint32_t box[3] = {(cuuint32_t)tma_box_x(h->tx),
                                 (cuuint32_t)(h->ty + 4), (cuuint32_t)npl};
            cuuint32_t es[3] = {1, 1, 1};
            void *base = (char *)h->d_pop[b] +
                         (size_t)(d.pop_off - GHOST * d.pitch - XGHOST) * esz;
            CUresult r = enc(&maps[b * count + l], pty, 3, base, dims, strides, box, es,
                             CU_TENSOR_MAP_INTERLEAVE_NONE,
                             CU_TENSOR_MAP_SWIZZLE_NONE,
                             CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) {
                why = "cuTensorMapEncodeTiled failed for populations, code " +
                      std::to_string((int)r);
                return false;
            }
            // output: the lattice's own nodes, logical (0, 0) at the base
            // (16-byte aligned: the ghost band is 16 columns wide)
            cuuint64_t odims[3] = {(cuuint64_t)d.nx, (cuuint64_t)d.ny, npl};
            cuuint32_t obox[3] = {(cuuint32_t)h->tx, (cuuint32_t)h->ty, (cuuint32_t)npl};
            r = enc(&maps[(2 + b) * count + l], pty, 3,
                    (char *)h->d_pop[b] + (size_t)d.pop_off * esz, odims, strides,
                    obox, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) {
                why = "cuTensorMapEncodeTiled failed for the output, code " +
                      std::to_string((int)r);
                return false;
            }
        }
    }
    for (int l = 0; l < count; ++l) {
        const LatDesc &d = h->desc[l];
        cuuint64_t dims[2] = {(cuuint64_t)d.pitch, (cuuint64_t)(d.ny + 2 * GHOST)};
        cuuint64_t strides[1] = {(cuuint64_t)d.pitch};
        cuuint32_t box[2] = {(cuuint32_t)tma_mask_box_x(h->tx), (cuuint32_t)(h->ty + 4)};
        cuuint32_t es[2] = {1, 1};
        CUresult r = enc(&mmaps[l], CU_TENSOR_MAP_DATA_TYPE_UINT8, 2,
                         h->d_mask + d.node_off - GHOST * d.pitch - XGHOST, dims,
                         strides, box, es,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) {
            why = "cuTensorMapEncodeTiled failed for the mask, code " +
                  std::to_string((int)r);
            return false;
        }
    }
    if (cudaMemcpyAsync(h->d_maps, up.data(), up.size() * sizeof(CUtensorMap),
                        cudaMemcpyHostToDevice, h->stream) != cudaSuccess) {
        why = "tensor map upload";
        return false;
    }
    return true;
}

struct Strip { int lat, col, row0, rows; };

// Deals strips, longest first, to the block with the least work so far (ties
// to the lower index).
static void deal_strips(std::vector<Strip> &strips, int grid,
                        std::vector<std::vector<int>> &lists,
                        std::vector<long long> &load) {
    std::stable_sort(strips.begin(), strips.end(),
                     [](const Strip &a, const Strip &b) { return a.rows > b.rows; });
    lists.assign(grid, {});
    load.assign(grid, 0);
    std::vector<int> heap(grid);
    for (int b = 0; b < grid; ++b) heap[b] = b;
    auto less = [&](int a, int b) { return load[a] > load[b] || (load[a] == load[b] && a > b); };
    std::make_heap(heap.begin(), heap.end(), less);
    for (size_t i = 0; i < strips.size(); ++i) {
        std::pop_heap(heap.begin(), heap.end(), less);
        const int b = heap.back();
        lists[b].push_back((int)i);
        load[b] += strips[i].rows;
        std::push_heap(heap.begin(), heap.end(), less);
    }
}

// The tiles of dealt strips as the kernel's table; returns the slots per block.
static size_t lay_strips(const std::vector<Strip> &strips, int tx, int ty, int grid,
                         const std::vector<std::vector<int>> &lists,
                         const std::vector<long long> &load,
                         std::vector<TileRec> &sched) {
    size_t slots = 0;
    for (long long n : load) slots = std::max(slots, (size_t)n);
    sched.assign((size_t)grid * slots, TileRec{-1, 0, 0, 0});
    for (int b = 0; b < grid; ++b) {
        size_t k = 0;
        for (int i : lists[b]) {
            const Strip &st = strips[i];
            for (int r = st.row0; r < st.row0 + st.rows; ++r)
                sched[b + k++ * grid] = TileRec{st.lat, st.col * tx, r * ty, 0};
        }
    }
    return slots;
}

// Most tiles of a strip of plan_tiles.
static long long strip_rows(long long total, int grid) {
    return std::max(4LL, (total + 4LL * grid - 1) / (4LL * grid));
}

// Tile schedule of the persistent TMA kernel, host arithmetic only.  A
// strip is a run of tiles down one tile column of a lattice (the halo rows
// each tile copies were just copied by the tile above it).  Columns taller
// than a quarter of a block's share (at least 4 tiles) are cut into strips
// of that length, so that a few tall lattices (a 2048-row preform: 32
// columns of 256 tiles) still spread over every block.  Strips go, longest
// first, to the block with the least work so far; block b then walks its
// strips top to bottom, its k-th tile at sched[b + k * grid] (lattice -1 =
// done).  Returns the slots per block.
static size_t plan_tiles(const int32_t *nx, const int32_t *ny, int count,
                         int tx, int ty, int grid, std::vector<TileRec> &sched) {
    long long total = 0;
    for (int l = 0; l < count; ++l)
        total += (long long)((nx[l] + tx - 1) / tx) * ((ny[l] + ty - 1) / ty);
    const long long seg = strip_rows(total, grid);
    std::vector<Strip> strips;
    for (int l = 0; l < count; ++l) {
        const int cols = (nx[l] + tx - 1) / tx, rows = (ny[l] + ty - 1) / ty;
        for (int c = 0; c < cols; ++c)
            for (int r0 = 0; r0 < rows; r0 += (int)seg)
                strips.push_back({l, c, r0, (int)std::min<long long>(seg, rows - r0)});
    }
    std::vector<std::vector<int>> lists;
    std::vector<long long> load;
    deal_strips(strips, grid, lists, load);
    return lay_strips(strips, tx, ty, grid, lists, load, sched);
}

// The schedule of a handle.  Batches of many tiles per block are dealt in
// strips (plan_tiles): adjacent tile columns then run at about the same time
// on different blocks, so their shared halo columns are read from L2.  With
// few tiles per block the strips (4 tiles at least) are too coarse: 256 x 32
// at 64 x 8 is 16 tiles on 4 of 152 blocks, and 4096 x 128 leaves some blocks
// 8 tiles and others 4 where 6.7 is the mean.  There each block takes one
// run of consecutive tiles in (lattice, tile column, row) order, lists that
// differ by one tile at most.  Step time at 64 x 8 FP32, strips / runs:
// 256 x 32 16.0 / 6.3 us, 1000 x 60 15.0 / 6.3 us, 4096 x 128 24.6 / 22.7 us
// (6.7 tiles per block); above that the lost halo sharing costs more than the balance
// gives: a 1024 x 1024 preform (13.5 tiles) 52.1 / 57.2 us, three 4096 x 128
// lattices FP16 (20.2 tiles) 51.8 / 53.3 us, so the line is at 8.
constexpr int kRunTiles = 8;  // most tiles per block dealt as runs
// From 16 to 32 tiles per block, in lattices of at most 64 tiles a column, the
// strips are evened out (even_strips) where that takes a sixteenth off the
// fullest block.  us per step, plan_tiles / even_strips: three 4096 x 128
// lattices FP32 54.9 / 51.6, FP16 50.0 / 48.5, three of 4600 x 160 FP32 76.4 /
// 70.4, FP16 72.7 / 65.9, five of the sweep FP32 52.9 / 49.9.  Where less is to
// be had the shorter strips cost as much (four 4096 x 128 lattices, 29 tiles
// against 28: FP32 68.7 / 70.8, FP16 65.8 / 62.8; ten of the sweep FP32 72.8 /
// 73.7), fewer tiles per block gain nothing (three of 3001 x 97, 11.6: FP32
// 32.9 / 33.6), and tall lattices lose more halo sharing than the balance
// gives (1024 x 1024 preform BF16 42.5 / 44.5).
constexpr int kEvenFrom = 16, kEvenTo = 32, kEvenRows = 64;

// Tiles of the fullest block when strips, `by_rows` of each length, are dealt
// as deal_strips deals them: which of the emptiest blocks takes a strip makes
// no difference to the loads, so blocks and strips are counted, not listed.
static long long fullest_block(const std::map<int, long long> &by_rows, int grid) {
    std::map<long long, long long> blocks{{0, grid}};  // blocks of each load
    for (auto r = by_rows.rbegin(); r != by_rows.rend(); ++r)
        for (long long left = r->second; left > 0;) {
            const auto low = blocks.begin();
            const long long load = low->first, n = std::min(left, low->second);
            if ((low->second -= n) == 0) blocks.erase(low);
            blocks[load + r->first] += n;
            left -= n;
        }
    return blocks.rbegin()->first;
}

// Strips as plan_tiles, but each tile column cut into equal pieces (their
// lengths differ by one), of the length 3 to 8 that leaves the fullest block
// the least, the longest such.  Returns the slots per block, or 0 where that
// is not a sixteenth below `plain`; the strips are listed and dealt once, when
// it is known that they are taken.
static size_t even_strips(const int32_t *nx, const int32_t *ny, int count, int tx,
                          int ty, int grid, long long plain, std::vector<TileRec> &sched) {
    long long top = 0;
    int seg = 0;
    for (int len = 8; len >= 3; --len) {
        std::map<int, long long> by_rows;
        for (int l = 0; l < count; ++l) {
            const int cols = (nx[l] + tx - 1) / tx, rows = (ny[l] + ty - 1) / ty;
            const int n = (rows + len - 1) / len;
            by_rows[rows / n] += (long long)cols * (n - rows % n);
            if (rows % n) by_rows[rows / n + 1] += (long long)cols * (rows % n);
        }
        const long long t = fullest_block(by_rows, grid);
        if (seg == 0 || t < top) {
            top = t;
            seg = len;
        }
    }
    if (16 * top > 15 * plain) return 0;
    std::vector<Strip> strips;
    for (int l = 0; l < count; ++l) {
        const int cols = (nx[l] + tx - 1) / tx, rows = (ny[l] + ty - 1) / ty;
        const int n = (rows + seg - 1) / seg;
        for (int c = 0; c < cols; ++c)
            for (int k = 0; k < n; ++k) {
                const int r0 = (int)((long long)k * rows / n);
                strips.push_back({l, c, r0, (int)((long long)(k + 1) * rows / n) - r0});
            }
    }
    std::vector<std::vector<int>> lists;
    std::vector<long long> load;
    deal_strips(strips, grid, lists, load);
    return lay_strips(strips, tx, ty, grid, lists, load, sched);
}

static size_t deal_tiles(const int32_t *nx, const int32_t *ny, int count,
                         int tx, int ty, int grid, std::vector<TileRec> &sched) {
    long long total = 0;
    for (int l = 0; l < count; ++l)
        total += (long long)((nx[l] + tx - 1) / tx) * ((ny[l] + ty - 1) / ty);
    if (total > (long long)kRunTiles * grid) {
        int tall = 0;
        for (int l = 0; l < count; ++l) tall = std::max(tall, (ny[l] + ty - 1) / ty);
        if (total > (long long)kEvenFrom * grid && total <= (long long)kEvenTo * grid &&
            tall <= kEvenRows) {
            const int seg = (int)strip_rows(total, grid);
            std::map<int, long long> by_rows;
            for (int l = 0; l < count; ++l) {
                const int cols = (nx[l] + tx - 1) / tx, rows = (ny[l] + ty - 1) / ty;
                if (rows / seg) by_rows[seg] += (long long)cols * (rows / seg);
                if (rows % seg) by_rows[rows % seg] += cols;
            }
            const size_t n = even_strips(nx, ny, count, tx, ty, grid,
                                         fullest_block(by_rows, grid), sched);
            if (n > 0) return n;
        }
        return plan_tiles(nx, ny, count, tx, ty, grid, sched);
    }
    const size_t slots = (size_t)((total + grid - 1) / grid);
    sched.assign((size_t)grid * slots, TileRec{-1, 0, 0, 0});
    // block b: tiles [first, end), end = ceil((b + 1) total / grid)
    long long t = 0, first = 0, end = (total + grid - 1) / grid;
    int b = 0;
    for (int l = 0; l < count; ++l)
        for (int x = 0; x < nx[l]; x += tx)
            for (int y = 0; y < ny[l]; y += ty, ++t) {
                while (t >= end) {
                    ++b;
                    first = end;
                    end = ((b + 1) * total + grid - 1) / grid;
                }
                sched[b + (size_t)(t - first) * grid] = TileRec{l, x, y, 0};
            }
    return slots;
}

static bool make_schedule(lbm_handle *h, std::vector<TileRec> &sched, std::string &why) {
    int grid = 0;
    cudaError_t e = grid_step_tma(h->tx, h->ty, h->store(), &grid);
    if (e != cudaSuccess || grid <= 0) {
        why = std::string("TMA kernel setup: ") + cudaGetErrorString(e);
        return false;
    }
    std::vector<int32_t> nx(h->count), ny(h->count);
    for (int l = 0; l < h->count; ++l) {
        nx[l] = h->desc[l].nx;
        ny[l] = h->desc[l].ny;
    }
    const size_t slots = deal_tiles(nx.data(), ny.data(), h->count, h->tx, h->ty, grid, sched);
    if (cudaMalloc(&h->d_sched, std::max<size_t>(sched.size(), 1) * sizeof(TileRec)) != cudaSuccess ||
        cudaMemcpyAsync(h->d_sched, sched.data(), sched.size() * sizeof(TileRec),
                        cudaMemcpyHostToDevice, h->stream) != cudaSuccess) {
        why = "schedule upload";
        return false;
    }
    h->sched_grid = grid;
    h->sched_slots = (int)slots;
    return true;
}

// The direct kernel's table of each tile's lattice, for the tile counts in
// the descriptors.
static cudaError_t make_tile_table(lbm_handle *h) {
    std::vector<int32_t> tile_lat(h->ntiles);
    for (int l = 0; l < h->count; ++l) {
        const LatDesc &d = h->desc[l];
        const int nt = d.tiles_x * ((d.ny + h->ty - 1) / h->ty);
        for (int k = 0; k < nt; ++k) tile_lat[d.tile_base + k] = l;
    }
    if (h->d_tile_lat) cudaFree(h->d_tile_lat);
    h->d_tile_lat = nullptr;
    cudaError_t e = dalloc(&h->d_tile_lat, h->ntiles);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(h->d_tile_lat, tile_lat.data(), h->ntiles * sizeof(int32_t),
                            cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    return e;
}

// Re-tiles every lattice for another step kernel or tile shape: tile
// counts in the descriptors, the tile -> lattice table and, for the TMA
// kernel, the tensor maps and the block schedule.  Drops the captured graph.
static lbm_status retile(lbm_handle *h, bool tma, int tx, int ty) {
    for (cudaGraphExec_t &g : h->graph) {
        if (g) cudaGraphExecDestroy(g);
        g = nullptr;
    }
    h->use_tma = tma;
    h->tx = tx;
    h->ty = ty;
    int tiles = 0;
    for (auto &d : h->desc) {
        d.tiles_x = (d.nx + tx - 1) / tx;
        d.tile_base = tiles;
        tiles += d.tiles_x * ((d.ny + ty - 1) / ty);
    }
    CK(h, cudaMemcpyAsync(h->d_desc, h->desc.data(), h->count * sizeof(LatDesc),
                          cudaMemcpyHostToDevice, h->stream));
    CK(h, cudaStreamSynchronize(h->stream));
    h->ntiles = tiles;
    if (h->d_sched) cudaFree(h->d_sched);
    h->d_sched = nullptr;
    if (tma) {
        std::string why;
        std::vector<CUtensorMap> maps;
        std::vector<TileRec> sched;
        if (!make_maps(h, maps, why) || !make_schedule(h, sched, why)) {
            cudaStreamSynchronize(h->stream);  // (what was issued reads the vectors)
            cudaGetLastError();
            return fail(h, LBM_EINVAL, "tile shape not supported: " + why);
        }
        CK(h, cudaStreamSynchronize(h->stream));
        return LBM_OK;
    }
    CK(h, make_tile_table(h));
    return LBM_OK;
}

extern "C" lbm_status lbm_create_batch(const lbm_geometry *g,
                                       const lbm_params *p, int32_t count,
                                       lbm_handle **out) {
    if (!out) return fail(nullptr, LBM_EINVAL, "out is NULL");
    *out = nullptr;
    if (!g || !p || count < 1)
        return fail(nullptr, LBM_EINVAL, "geometry/params NULL or count < 1");
    std::string why;
    for (int l = 0; l < count; ++l) {
        const lbm_geometry &G = g[l];
        if (G.nx < 1 || G.ny < 3 || !G.solid || !G.rho_a || !G.rho_b ||
            !G.conc)
            return fail(nullptr, LBM_EINVAL,
                        "lattice " + std::to_string(l) +
                            ": need nx >= 1, ny >= 3 and all arrays");
        // 32-bit offsets inside a lattice: 22 planes of ny * pitch elements
        if ((int64_t)NPOP * (G.ny + 2 * GHOST) * ((G.nx + 2 * XGHOST + 31) / 32 * 32) >=
            ((int64_t)1 << 31))
            return fail(nullptr, LBM_EINVAL, "lattice too large");
        if (!(0 <= G.cap_x0 && G.cap_x0 < G.cap_x1 && G.cap_x1 <= G.nx))
            return fail(nullptr, LBM_EINVAL,
                        "lattice " + std::to_string(l) + ": bad section");
        if (!valid_params(p[l], why))
            return fail(nullptr, LBM_EINVAL,
                        "lattice " + std::to_string(l) + ": " + why);
        if (p[l].precision != p[0].precision)
            return fail(nullptr, LBM_EINVAL, "mixed precision in a batch");
    }
    lbm_handle *h = new (std::nothrow) lbm_handle();
    if (!h) return fail(nullptr, LBM_ENOMEM, "host allocation");
    h->count = count;
    h->half = p[0].precision != LBM_FP32;
    h->bf16 = p[0].precision == LBM_BF16;
    pick_tile(h, g);

    // ---- packed ragged layout ------------------------------------------
    h->desc.resize(count);
    h->col_base.resize(count);
    h->in_off_host.assign(count + 1, 0);
    int64_t pop = 0, node = 0, cols = 0, sec = 0;
    int tiles = 0;
    for (int l = 0; l < count; ++l) {
        const lbm_geometry &G = g[l];
        const lbm_params &P = p[l];
        LatDesc &d = h->desc[l];
        d.nx = G.nx;
        d.ny = G.ny;
        d.pitch = (G.nx + 2 * XGHOST + 31) / 32 * 32;
        d.tiles_x = (G.nx + h->tx - 1) / h->tx;
        d.tile_base = tiles;
        tiles += d.tiles_x * ((G.ny + h->ty - 1) / h->ty);
        d.cap_x0 = G.cap_x0;
        d.cap_x1 = G.cap_x1;
        d.inlet = P.inlet ? 1 : 0;
        // planes include GHOST rows on both sides; offsets point at row 0
        d.plane = (int64_t)(d.ny + 2 * GHOST) * d.pitch;
        d.node_off = node + GHOST * d.pitch + XGHOST;
        d.pop_off = pop + GHOST * d.pitch + XGHOST;
        d.pad64_ = 0;
        d.col_off = sec;
        node += d.plane;
        pop += (h->half ? NW16 : NPOP) * d.plane;
        h->col_base[l] = cols;
        cols += d.nx;
        sec += G.cap_x1 - G.cap_x0;
        d.tau_a = (float)P.tau_a;
        d.tau_b = (float)P.tau_b;
        d.inv_tau_a = (float)(1.0 / P.tau_a);
        d.inv_tau_b = (float)(1.0 / P.tau_b);
        d.inv_tau_d = (float)(1.0 / P.tau_d);
        d.g_coh = (float)P.g_coh;
        d.g_ads = (float)P.g_ads;
        d.k_r = (float)P.k_r;
        d.c_in = (float)P.c_in;
        d.body_x = (float)P.body_force_x;
        d.m_th = P.m_threshold;
        d.index = l;
        d.bf16 = h->bf16 ? 1 : 0;
        h->max_nodes = std::max(h->max_nodes, (size_t)G.nx * G.ny);
        h->in_off_host[l + 1] = h->in_off_host[l] + (int64_t)G.nx * G.ny;
    }
    h->ntiles = tiles;
    h->pop_elems = pop;
    h->node_elems = node;
    h->ncols = cols;
    h->nsec = sec;

    // prefixes over the lattices (count + 1 entries each): nodes (staging
    // offsets), rows, rows with the ghost band, section columns
    const int C1 = count + 1;
    std::vector<int64_t> pre_h(4 * C1, 0);
    for (int l = 0; l < count; ++l) {
        pre_h[l + 1] = h->in_off_host[l + 1];
        pre_h[C1 + l + 1] = pre_h[C1 + l] + h->desc[l].ny;
        pre_h[2 * C1 + l + 1] = pre_h[2 * C1 + l] + h->desc[l].ny + 2 * GHOST;
        pre_h[3 * C1 + l] = h->desc[l].col_off;
    }
    pre_h[3 * C1 + count] = h->nsec;
    h->total_rows = pre_h[C1 + count];

    // ---- device allocation ------------------------------------------------
    const size_t esz = 4;  // 32-bit words in both storages
    const int64_t total = h->in_off_host.back();
    Arena ar;
    // zeroed in one go
    uint32_t *pop_w[2];
    ar.add(&pop_w[0], (size_t)pop);
    ar.add(&pop_w[1], (size_t)pop);
    ar.add(&h->d_mask, (size_t)node);
    ar.add(&h->d_m, (size_t)node);
    ar.add(&h->d_step, 2);
    ar.add(&h->d_err, 1);
    const size_t zeroed = ar.bytes;
    // uploaded in one go
    int64_t *pre = nullptr;
    const size_t tab = ar.bytes;
    const size_t at_desc = ar.add(&h->d_desc, count) - tab;
    const size_t at_col_lat = ar.add(&h->d_col_lat, cols) - tab;
    const size_t at_col_base = ar.add(&h->d_col_base, count) - tab;
    const size_t at_pre = ar.add(&pre, 4 * C1) - tab;
    const size_t at_st = ar.add(&h->d_st, count) - tab;
    const size_t tab_bytes = ar.bytes - tab;
    ar.add(&h->d_maps, 5 * (size_t)count);
    ar.add(&h->d_col_fluid, sec);
    ar.add(&h->d_wall0, 2 * sec);
    ar.add(&h->d_cols, cols);
    lbm_obs *obs = nullptr;
    ar.add(&obs, count);
    ar.add(&h->d_sums, 3 * (size_t)count);
    ar.add(&h->d_canon, NPOP * h->max_nodes);
    ar.add(&h->d_dens, 3 * h->max_nodes);
    ar.add(&h->d_dep, h->max_nodes);
    cudaError_t e = ar.place(&h->d_arena);
    if (e != cudaSuccess) {
        std::string msg = std::string("device allocation: ") + cudaGetErrorString(e);
        free_all(h);
        delete h;
        return fail(nullptr, e == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA, msg);
    }
    h->d_pop[0] = pop_w[0];
    h->d_pop[1] = pop_w[1];
    h->d_obs = obs;
    h->d_in_off = pre;
    h->d_mask_maps = h->d_maps + 4 * (size_t)count;
    lbm_status st = LBM_OK;
    auto bad = [&](cudaError_t ce, const char *what) {
        if (ce != cudaSuccess && st == LBM_OK) {
            g_create_err = std::string(what) + ": " + cudaGetErrorString(ce);
            st = LBM_ECUDA;
        }
    };
    bad(cudaStreamCreateWithFlags(&h->own, cudaStreamNonBlocking), "stream");
    h->stream = h->own;
    cudaStream_t s = h->stream;
    // the zeroed buffers on a stream of their own, behind nothing, so that
    // they run beside the gather
    cudaStream_t s2 = nullptr;
    cudaEvent_t zero_done = nullptr;
    bad(cudaStreamCreateWithFlags(&s2, cudaStreamNonBlocking), "stream");
    bad(cudaEventCreateWithFlags(&zero_done, cudaEventDisableTiming), "event");
    if (st == LBM_OK) {
        bad(cudaMemsetAsync(h->d_arena, 0, zeroed, s2), "memset");
        bad(cudaEventRecord(zero_done, s2), "event");
    }
    // tables the kernels read
    std::vector<uint8_t> tabs(tab_bytes, 0);
    memcpy(&tabs[at_desc], h->desc.data(), count * sizeof(LatDesc));
    int32_t *col_lat = reinterpret_cast<int32_t *>(&tabs[at_col_lat]);
    for (int l = 0; l < count; ++l)
        for (int x = 0; x < h->desc[l].nx; ++x) col_lat[h->col_base[l] + x] = l;
    memcpy(&tabs[at_col_base], h->col_base.data(), count * sizeof(int64_t));
    memcpy(&tabs[at_pre], pre_h.data(), pre_h.size() * sizeof(int64_t));
    for (int l = 0; l < count; ++l)
        reinterpret_cast<LatState *>(&tabs[at_st])[l].closure = ~0ull;
    if (st == LBM_OK)
        bad(cudaMemcpyAsync((char *)h->d_arena + tab, tabs.data(), tab_bytes,
                            cudaMemcpyHostToDevice, s),
            "tables");
    // Initial state of the whole batch: every lattice's inputs go into one
    // device staging area -- read in place by one gather kernel where the
    // device can address the caller's arrays, else copied by the host (one
    // copy per array) -- issued on the handle's stream and landing while the
    // host builds the tensor maps and the schedule below; then one launch per
    // set-up kernel covers all lattices.  (Mask bytes, section-column counts
    // and initial wall thicknesses are built on the device from the solid
    // arrays.)
    float *rho3 = nullptr;
    uint8_t *sol = nullptr;
    InPtrs *d_ptrs = nullptr;
    void *staging = nullptr;
    Arena sg;
    sg.add(&rho3, 3 * (size_t)total);
    sg.add(&sol, (size_t)total);
    sg.add(&d_ptrs, (size_t)count);
    if (st == LBM_OK) bad(sg.place(&staging), "alloc");
    std::vector<InPtrs> ptrs(count);
    // Pageable arrays are read in place up to 4 MB each; larger ones the driver
    // copies faster, and far faster where their pages are not present yet
    // (zeros never written): each is a fault of the device then.  Creating one
    // lattice from pageable arrays, copied / in place: 1024 x 1024 694 / 644 us,
    // 2048 x 2048 1117 / 1735, 4096 x 4096 2730 / 5853, with two arrays of
    // unwritten zeros 9.0 / 71.6 ms; 8 of 512 x 512 1192 / 688 us.
    constexpr int64_t kInPlaceBytes = 4 << 20;
    const bool can_read = reads_pageable();
    if (st == LBM_OK) {
        bool any = false;
        for (int l = 0; l < count && st == LBM_OK; ++l) {
            const int64_t N = (int64_t)h->desc[l].nx * h->desc[l].ny, o = h->in_off_host[l];
            const bool pageable = can_read && N * (int64_t)sizeof(float) <= kInPlaceBytes;
            InPtrs &q = ptrs[l];
            q.rho_a = device_view(g[l].rho_a, pageable);
            q.rho_b = device_view(g[l].rho_b, pageable);
            q.conc = device_view(g[l].conc, pageable);
            q.solid = device_view(g[l].solid, pageable);
            any = any || q.rho_a || q.rho_b || q.conc || q.solid;
            // (the copy direction is inferred: host memory, or another
            // device's)
            if (!q.rho_a)
                bad(cudaMemcpyAsync(rho3 + 3 * o, g[l].rho_a, N * 4, cudaMemcpyDefault, s), "rho_a");
            if (!q.rho_b)
                bad(cudaMemcpyAsync(rho3 + 3 * o + N, g[l].rho_b, N * 4, cudaMemcpyDefault, s), "rho_b");
            if (!q.conc)
                bad(cudaMemcpyAsync(rho3 + 3 * o + 2 * N, g[l].conc, N * 4, cudaMemcpyDefault, s), "conc");
            if (!q.solid)
                bad(cudaMemcpyAsync(sol + o, g[l].solid, N, cudaMemcpyDefault, s), "solid");
        }
        if (any && st == LBM_OK) {
            bad(cudaMemcpyAsync(d_ptrs, ptrs.data(), count * sizeof(InPtrs),
                                cudaMemcpyHostToDevice, s), "pointers");
            // at most 65535 lattices per launch (grid y)
            for (int l0 = 0; l0 < count && st == LBM_OK; l0 += 65535) {
                const unsigned ny_ = (unsigned)std::min(count - l0, 65535);
                k_gather_inputs<<<dim3(16, ny_), 256, 0, s>>>(d_ptrs, l0, h->d_in_off,
                                                              rho3, sol);
                bad(cudaGetLastError(), "gather");
            }
        }
    }
    std::vector<CUtensorMap> maps;
    std::vector<TileRec> sched;
    if (st == LBM_OK && h->use_tma) {
        std::string why;
        if (!make_maps(h, maps, why) || !make_schedule(h, sched, why)) {
            g_create_err = why;
            st = LBM_ECUDA;
        }
    } else if (st == LBM_OK) {
        bad(make_tile_table(h), "tiles");
    }
    // the zeroing lands before the set-up kernels
    if (st == LBM_OK) bad(cudaStreamWaitEvent(s, zero_done, 0), "sync");
    if (st == LBM_OK) {
        k_mask_init_all<<<(unsigned)pre_h[2 * C1 + count], 128, 0, s>>>(
            h->d_desc, count, pre + 2 * C1, pre, sol, h->d_mask);
        if (h->nsec > 0)
            k_col_init_all<<<(unsigned)((h->nsec + 255) / 256), 256, 0, s>>>(
                h->d_desc, count, pre + 3 * C1, pre, sol, h->d_col_fluid,
                h->d_wall0, h->d_st);
        k_init_rest_all<<<(unsigned)h->total_rows, 128, 0, s>>>(
            h->d_desc, count, pre + C1, pre, rho3, h->d_mask, h->d_pop[0], h->half);
        bad(cudaGetLastError(), "init kernels");
    }
    // (also after a failure: what was issued reads the arrays above)
    if (s2) bad(cudaStreamSynchronize(s2), "init sync");
    if (s) bad(cudaStreamSynchronize(s), "init sync");
    if (zero_done) cudaEventDestroy(zero_done);
    if (s2) cudaStreamDestroy(s2);
    if (staging) cudaFree(staging);
    if (st != LBM_OK) {
        free_all(h);
        delete h;
        cudaGetLastError();  // (as fail does)
        return st;
    }
    *out = h;
    return LBM_OK;
}

extern "C" lbm_status lbm_create(const lbm_geometry *g, const lbm_params *p,
                                 lbm_handle **out) {
    return lbm_create_batch(g, p, 1, out);
}

extern "C" void lbm_destroy(lbm_handle *h) {
    if (!h) return;
    if (h->stream) cudaStreamSynchronize(h->stream);
    free_all(h);
    delete h;
}

extern "C" const char *lbm_last_error(const lbm_handle *h) {
    if (!h) return g_create_err.c_str();
    return h->err.c_str();
}

extern "C" int64_t lbm_step_count(const lbm_handle *h) { return h ? h->steps : -1; }
extern "C" int32_t lbm_count(const lbm_handle *h) { return h ? h->count : 0; }

extern "C" lbm_status lbm_set_stream(lbm_handle *h, void *cuda_stream) {
    if (!h) return LBM_EINVAL;
    if (h->dead) return fail(h, LBM_ECUDA, "handle is dead: " + h->err);
    CK(h, cudaStreamSynchronize(h->stream));
    h->stream = cuda_stream ? (cudaStream_t)cuda_stream : h->own;
    return LBM_OK;
}

static StepArgs step_args(lbm_handle *h) {
    StepArgs a;
    a.desc = h->d_desc;
    a.tile_lat = h->d_tile_lat;
    a.fin = h->d_pop[h->cur];
    a.fout = h->d_pop[h->cur ^ 1];
    a.mask = h->d_mask;
    a.m = h->d_m;
    a.col_fluid = h->d_col_fluid;
    a.st = h->d_st;
    a.step = h->d_step + h->cur;
    a.step_next = h->d_step + (h->cur ^ 1);
    a.stall_tx = h->stall_tx;
    a.sums = nullptr;
    return a;
}

// One launch of the step kernel reading buffer cur, writing cur ^ 1.  sum:
// the launch also adds up the lattice totals (zeroed first, on the stream)
// that lbm_observables then reads instead of the whole state.
static cudaError_t launch_one(lbm_handle *h, bool sum) {
    StepArgs a = step_args(h);
    if (sum) {
        cudaError_t e = cudaMemsetAsync(h->d_sums, 0, 3 * h->count * sizeof(double),
                                        h->stream);
        if (e != cudaSuccess) return e;
        a.sums = h->d_sums;
    }
    if (!h->use_tma)
        return launch_step_direct(a, h->ntiles, h->tx, h->ty, h->store(), h->stream);
    const int c = h->count, in = h->cur, out = h->cur ^ 1;
    return launch_step_tma(a, h->d_maps + in * c, h->d_mask_maps,
                           h->d_maps + (2 + out) * c, h->d_sched, h->sched_slots,
                           h->sched_grid, h->tx, h->ty, h->store(), h->d_err,
                           h->stream);
}

// Steps per captured graph: even, so a replay starts and ends with the
// same population buffer as input.
static const int kGraphSteps = 16;
// Steps per cluster launch at most (a launch stays around a millisecond), and
// the shortest call that uses them: a launch also loads and stores the state,
// about 17 us (a call of 16 steps of 256 x 32 FP32 69 us with it and 66
// without, of 24 steps 90 and 100, of 64 steps 204 and 245).
static const int kClusterSteps = 512, kClusterMin = 24;

// Captures kGraphSteps launches starting from buffer 0 into h->graph[sum];
// sum: the last one adds up the lattice totals.
static lbm_status capture_graph(lbm_handle *h, int sum) {
    const int cur0 = h->cur;
    h->cur = 0;
    cudaGraph_t g = nullptr;
    CK(h, cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < kGraphSteps && e == cudaSuccess; ++k) {
        e = launch_one(h, sum && k == kGraphSteps - 1);
        h->cur ^= 1;
    }
    cudaError_t e2 = cudaStreamEndCapture(h->stream, &g);
    h->cur = cur0;
    CK(h, e);
    CK(h, e2);
    cudaError_t e3 = cudaGraphInstantiate(&h->graph[sum], g, 0);
    cudaGraphDestroy(g);
    CK(h, e3);
    return LBM_OK;
}

extern "C" lbm_status lbm_step(lbm_handle *h, int64_t n) {
    if (!h || n < 0) return fail(h, LBM_EINVAL, "bad handle or n < 0");
    if (h->dead) return fail(h, LBM_ECUDA, "handle is dead: " + h->err);
    // The last launch of the call adds up the lattice totals of the state it
    // leaves (a replay that ends the call uses the graph whose last launch
    // sums).
    // Lattices that fit a cluster: all but the last steps on chip, up to
    // kClusterSteps per launch.  A launch moves the state to the other buffer
    // whatever its step count, and a graph that the caller captured around
    // lbm_step reads the buffer it was captured with.  So none are captured,
    // and a call moves the state as often as n single steps would, give or
    // take an even number: the steps left for single launches, one to three,
    // see to it.
    if (h->csize > 0 && h->stall_tx == 0 && n >= kClusterMin) {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(h->stream, &cap) != cudaSuccess) {
            cudaGetLastError();
            cap = cudaStreamCaptureStatusActive;
        }
        int64_t single = 1;
        while (((n - single + kClusterSteps - 1) / kClusterSteps + single - n) % 2 != 0)
            ++single;
        while (cap == cudaStreamCaptureStatusNone && n > single) {
            const int m = (int)std::min<int64_t>(n - single, kClusterSteps);
            CK(h, launch_step_cluster(step_args(h), h->count, m, h->ctx, h->cty,
                                      h->csize, h->store(), h->stream));
            h->cur ^= 1;
            h->steps += m;
            n -= m;
        }
    }
    // Whole groups of kGraphSteps steps replay one captured graph (the
    // step count lives on the device, so the graph needs no new arguments)
    // (a pending test stall is never captured into the graph)
    if (n > 0) h->sums_step = -1;
    while (h->use_graph && h->stall_tx == 0 &&
           n >= kGraphSteps + (h->cur ? 1 : 0)) {
        if (h->cur) {  // one plain step to get back to buffer 0
            CK(h, launch_one(h, false));
            h->cur ^= 1;
            h->steps += 1;
            n -= 1;
        }
        const int sum = n == kGraphSteps;
        if (!h->graph[sum]) {
            lbm_status st = capture_graph(h, sum);
            if (st != LBM_OK) return st;
        }
        CK(h, cudaGraphLaunch(h->graph[sum], h->stream));
        h->steps += kGraphSteps;
        n -= kGraphSteps;
        if (sum) h->sums_step = h->steps;
    }
    for (int64_t k = 0; k < n; ++k) {
        cudaError_t e = launch_one(h, k == n - 1);
        if (e == cudaErrorInvalidValue && k == 0)
            return fail(h, LBM_EINVAL, "unsupported tile shape");
        CK(h, e);
        h->stall_tx = 0;  // the test stall applies to one launch
        h->cur ^= 1;
        h->steps += 1;
        if (k == n - 1) h->sums_step = h->steps;
    }
    return LBM_OK;
}

extern "C" lbm_status lbm_observables(lbm_handle *h, lbm_obs *out) {
    if (!h || !out) return fail(h, LBM_EINVAL, "NULL argument");
    if (h->dead) return fail(h, LBM_ECUDA, "handle is dead: " + h->err);
    // 32 columns per block, OBS_ROWS warps splitting their rows
    // the last step launch summed the stored totals: the column pass then
    // reads the mask and the nodes that turned solid, not the whole state
    const bool summed = h->sums_step == h->steps;
    const int nb = (int)((h->ncols + 31) / 32);
    launch_obs_columns(summed, h->store(), nb, (int)h->ncols, h->d_desc,
                       h->d_col_lat, h->d_col_base, h->d_pop[h->cur], h->d_mask,
                       h->d_m, h->steps, h->d_cols, h->stream);
    k_obs_reduce<<<h->count, 256, 0, h->stream>>>(
        h->d_desc, h->d_col_base, h->d_cols, h->d_wall0, h->d_st,
        summed ? h->d_sums : nullptr, h->steps, (LbmObsDev *)h->d_obs);
    CK(h, cudaGetLastError());
    CK(h, cudaMemcpyAsync(out, h->d_obs, h->count * sizeof(lbm_obs),
                          cudaMemcpyDeviceToHost, h->stream));
    CK(h, cudaStreamSynchronize(h->stream));
    int kerr = 0;
    CK(h, cudaMemcpy(&kerr, h->d_err, sizeof(int), cudaMemcpyDeviceToHost));
    if (kerr) {
        h->dead = true;
        return fail(h, LBM_ETIMEOUT, "a bounded wait in the step kernel ran out");
    }
    for (int l = 0; l < h->count; ++l)
        if (out[l].nonfinite)
            return fail(h, LBM_ENAN, "non-finite density in lattice " + std::to_string(l));
    return LBM_OK;
}

extern "C" lbm_status lbm_get_solid_mask(lbm_handle *h, int32_t k,
                                         uint8_t *host, size_t n) {
    if (!h || !host || k < 0 || k >= h->count) return fail(h, LBM_EINVAL, "bad argument");
    if (h->dead) return fail(h, LBM_ECUDA, "handle is dead: " + h->err);
    const LatDesc &d = h->desc[k];
    if (n != (size_t)d.nx * d.ny) return fail(h, LBM_EINVAL, "size mismatch");
    // extracted on the device into the export scratch (max_nodes floats)
    const MaskBits mb(h->steps);
    uint8_t *tmp = reinterpret_cast<uint8_t *>(h->d_canon);
    k_solid_mask<<<dim3((d.nx + 127) / 128, d.ny), 128, 0, h->stream>>>(
        h->d_desc, k, h->d_mask, mb.force, tmp);
    CK(h, cudaGetLastError());
    CK(h, cudaMemcpyAsync(host, tmp, n, cudaMemcpyDeviceToHost, h->stream));
    CK(h, cudaStreamSynchronize(h->stream));
    return LBM_OK;
}

extern "C" lbm_status lbm_get_solid_masks(lbm_handle *h, uint8_t *host,
                                          size_t n) {
    if (!h || !host) return fail(h, LBM_EINVAL, "bad argument");
    if (h->dead) return fail(h, LBM_ECUDA, "handle is dead: " + h->err);
    const int64_t total = h->in_off_host.back();
    if (n != (size_t)total) return fail(h, LBM_EINVAL, "size mismatch");
    // device scratch, then one copy (into pinned memory the copy runs at
    // the link's rate; the kernel writing pinned memory itself measured
    // slower, 1.07 against 0.77 ms for 105 MB)
    if (!h->d_masks) CK(h, dalloc(&h->d_masks, (size_t)total));
    const MaskBits mb(h->steps);
    k_solid_mask_all<<<(unsigned)h->total_rows, 128, 0, h->stream>>>(
        h->d_desc, h->count, h->d_in_off + h->count + 1, h->d_in_off, h->d_mask,
        mb.force, h->d_masks);
    CK(h, cudaGetLastError());
    CK(h, cudaMemcpyAsync(host, h->d_masks, n, cudaMemcpyDefault, h->stream));
    CK(h, cudaStreamSynchronize(h->stream));
    return LBM_OK;
}

extern "C" lbm_status lbm_get_fields(lbm_handle *h, int32_t k, int32_t which,
                                     void *host, size_t bytes) {
    if (!h || !host || k < 0 || k >= h->count) return fail(h, LBM_EINVAL, "bad argument");
    if (h->dead) return fail(h, LBM_ECUDA, "handle is dead: " + h->err);
    const LatDesc &d = h->desc[k];
    const size_t N = (size_t)d.nx * d.ny;
    size_t need = which == LBM_FIELD_POPS ? NPOP * N * 4
                : which == LBM_FIELD_DEPOSIT ? N * 8
                : which == LBM_FIELD_DENSITY ? 3 * N * 4 : 0;
    if (need == 0) return fail(h, LBM_EINVAL, "unknown field");
    if (bytes != need) return fail(h, LBM_EINVAL, "size mismatch");
    dim3 grid((d.nx + 127) / 128, d.ny), blk(128);
    k_export<<<grid, blk, 0, h->stream>>>(
        h->d_desc, k, h->d_pop[h->cur], h->d_mask, h->d_m, h->steps, h->half, which == LBM_FIELD_POPS ? h->d_canon : nullptr,
        which == LBM_FIELD_DENSITY ? h->d_dens : nullptr,
        which == LBM_FIELD_DEPOSIT ? h->d_dep : nullptr);
    CK(h, cudaGetLastError());
    const void *src = which == LBM_FIELD_POPS ? (const void *)h->d_canon
                    : which == LBM_FIELD_DENSITY ? (const void *)h->d_dens
                    : (const void *)h->d_dep;
    CK(h, cudaMemcpyAsync(host, src, need, cudaMemcpyDeviceToHost, h->stream));
    CK(h, cudaStreamSynchronize(h->stream));
    return LBM_OK;
}

// Folds pending flips of lattice k into its ledger and aligns its mask bits.
static lbm_status settle(lbm_handle *h, int k) {
    const LatDesc &d = h->desc[k];
    dim3 grid((d.nx + 127) / 128, d.ny), blk(128);
    k_settle<<<grid, blk, 0, h->stream>>>(h->d_desc, k, h->d_pop[h->cur],
                                         h->d_mask, h->d_m, h->d_st, h->steps,
                                         h->half);
    k_mask_agree<<<grid, blk, 0, h->stream>>>(h->d_desc, k, h->d_mask, h->steps);
    CK(h, cudaGetLastError());
    return LBM_OK;
}

extern "C" lbm_status lbm_set_fields(lbm_handle *h, int32_t k, int32_t which,
                                     const void *host, size_t bytes) {
    if (!h || !host || k < 0 || k >= h->count) return fail(h, LBM_EINVAL, "bad argument");
    if (h->dead) return fail(h, LBM_ECUDA, "handle is dead: " + h->err);
    const LatDesc &d = h->desc[k];
    const size_t N = (size_t)d.nx * d.ny;
    h->sums_step = -1;  // the last step's lattice totals no longer hold
    if (which == LBM_FIELD_POPS) {
        if (bytes != NPOP * N * 4) return fail(h, LBM_EINVAL, "size mismatch");
        lbm_status s = settle(h, k);
        if (s != LBM_OK) return s;
        CK(h, cudaMemcpyAsync(h->d_canon, host, bytes, cudaMemcpyHostToDevice, h->stream));
        dim3 grid((d.nx + 127) / 128, d.ny), blk(128);
        const MaskBits mb(h->steps);
        k_unstream<<<grid, blk, 0, h->stream>>>(h->d_desc, k, h->d_canon, h->d_mask,
                                               mb.force, h->d_pop[h->cur],
                                               h->half);
        CK(h, cudaGetLastError());
        CK(h, cudaStreamSynchronize(h->stream));
        return LBM_OK;
    }
    if (which == LBM_FIELD_DEPOSIT) {
        if (bytes != N * 8) return fail(h, LBM_EINVAL, "size mismatch");
        lbm_status s = settle(h, k);
        if (s != LBM_OK) return s;
        const size_t rows_n = (size_t)d.ny * d.pitch;
        std::vector<uint8_t> raw(rows_n);
        CK(h, cudaMemcpyAsync(raw.data(), h->d_mask + d.node_off, rows_n,
                              cudaMemcpyDeviceToHost, h->stream));
        CK(h, cudaStreamSynchronize(h->stream));
        std::vector<double> m(rows_n, 0.0);
        const double *src = static_cast<const double *>(host);
        for (int y = 0; y < d.ny; ++y)
            for (int x = 0; x < d.nx; ++x)
                if (!(raw[(size_t)y * d.pitch + x] & 7)) {
                    const double v = src[(size_t)y * d.nx + x];
                    // a fluid node at or above the threshold would have
                    // turned solid when its deposit crossed it
                    if (!(v >= 0.0 && v < d.m_th))
                        return fail(h, LBM_EINVAL,
                                    "deposit outside [0, m_threshold) at a fluid node");
                    m[(size_t)y * d.pitch + x] = v;
                }
        CK(h, cudaMemcpyAsync(h->d_m + d.node_off, m.data(), rows_n * 8,
                              cudaMemcpyHostToDevice, h->stream));
        CK(h, cudaStreamSynchronize(h->stream));
        return LBM_OK;
    }
    return fail(h, LBM_EINVAL, "field cannot be set");
}

// ---- checkpoints -----------------------------------------------------------

static const char kMagic[8] = {'L', 'B', 'M', 'C', 'K', 'P', 'T', '5'};

struct CkptHeader {
    char magic[8];
    int32_t count, half;  // half: the storage, 0 FP32, 1 FP16, 2 BF16
    int64_t pop_elems, node_elems, nsec, steps;
    int32_t cur, pad;
};

extern "C" lbm_status lbm_save(lbm_handle *h, const char *path) {
    if (!h || !path) return fail(h, LBM_EINVAL, "NULL argument");
    if (h->dead) return fail(h, LBM_ECUDA, "handle is dead: " + h->err);
    CK(h, cudaStreamSynchronize(h->stream));
    const size_t esz = 4;
    CkptHeader hd;
    memcpy(hd.magic, kMagic, 8);
    hd.count = h->count;
    hd.half = h->store();
    hd.pop_elems = h->pop_elems;
    hd.node_elems = h->node_elems;
    hd.nsec = h->nsec;
    hd.steps = h->steps;
    hd.cur = 0;
    hd.pad = 0;
    FILE *f = fopen(path, "wb");
    if (!f) return fail(h, LBM_EIO, std::string("cannot open ") + path);
    bool ok = fwrite(&hd, sizeof(hd), 1, f) == 1;
    ok = ok && fwrite(h->desc.data(), sizeof(LatDesc), h->count, f) == (size_t)h->count;
    auto dump = [&](const void *dptr, size_t bytes) {
        if (!ok) return;
        std::vector<uint8_t> buf(std::min<size_t>(bytes, (size_t)1 << 28));
        size_t done = 0;
        while (ok && done < bytes) {
            const size_t n = std::min(buf.size(), bytes - done);
            if (cudaMemcpy(buf.data(), (const uint8_t *)dptr + done, n, cudaMemcpyDeviceToHost) != cudaSuccess) {
                ok = false;
                return;
            }
            ok = fwrite(buf.data(), 1, n, f) == n;
            done += n;
        }
    };
    dump(h->d_pop[h->cur], h->pop_elems * esz);
    dump(h->d_mask, h->node_elems);
    dump(h->d_m, h->node_elems * 8);
    dump(h->d_col_fluid, h->nsec * 4);
    dump(h->d_st, h->count * sizeof(LatState));
    dump(h->d_step + h->cur, 8);
    ok = (fclose(f) == 0) && ok;
    if (!ok) return fail(h, LBM_EIO, std::string("write failed: ") + path);
    return LBM_OK;
}

extern "C" lbm_status lbm_load(lbm_handle *h, const char *path) {
    if (!h || !path) return fail(h, LBM_EINVAL, "NULL argument");
    if (h->dead) return fail(h, LBM_ECUDA, "handle is dead: " + h->err);
    CK(h, cudaStreamSynchronize(h->stream));
    FILE *f = fopen(path, "rb");
    if (!f) return fail(h, LBM_EIO, std::string("cannot open ") + path);
    CkptHeader hd;
    bool ok = fread(&hd, sizeof(hd), 1, f) == 1 && memcmp(hd.magic, kMagic, 8) == 0;
    ok = ok && hd.count == h->count && hd.half == h->store() &&
         hd.pop_elems == h->pop_elems && hd.node_elems == h->node_elems &&
         hd.nsec == h->nsec;
    std::vector<LatDesc> dsc(h->count);
    ok = ok && fread(dsc.data(), sizeof(LatDesc), h->count, f) == (size_t)h->count;
    // the tiles are how a handle launches, not part of the state: they depend
    // on the storage, the sizes and the solid share at create
    for (int l = 0; ok && l < h->count; ++l) {
        LatDesc mine = h->desc[l];
        mine.tiles_x = dsc[l].tiles_x;
        mine.tile_base = dsc[l].tile_base;
        ok = memcmp(&dsc[l], &mine, sizeof(LatDesc)) == 0;
    }
    if (!ok) {
        fclose(f);
        return fail(h, LBM_EINVAL, "checkpoint does not match this handle");
    }
    const size_t esz = 4;
    auto slurp = [&](void *dptr, size_t bytes) {
        if (!ok) return;
        std::vector<uint8_t> buf(std::min<size_t>(bytes, (size_t)1 << 28));
        size_t done = 0;
        while (ok && done < bytes) {
            const size_t n = std::min(buf.size(), bytes - done);
            ok = fread(buf.data(), 1, n, f) == n;
            // on the handle's stream: a plain copy from pageable memory may
            // return before it has landed, and nothing orders the handle's
            // next launch behind it
            if (ok && (cudaMemcpyAsync((uint8_t *)dptr + done, buf.data(), n,
                                       cudaMemcpyHostToDevice, h->stream) != cudaSuccess ||
                       cudaStreamSynchronize(h->stream) != cudaSuccess))
                ok = false;
            done += n;
        }
    };
    h->cur = 0;
    slurp(h->d_pop[0], h->pop_elems * esz);
    slurp(h->d_mask, h->node_elems);
    slurp(h->d_m, h->node_elems * 8);
    slurp(h->d_col_fluid, h->nsec * 4);
    slurp(h->d_st, h->count * sizeof(LatState));
    slurp(h->d_step, 8);
    fclose(f);
    if (!ok) return fail(h, LBM_EIO, std::string("read failed: ") + path);
    h->steps = hd.steps;
    h->sums_step = -1;
    return LBM_OK;
}

// Host entry of a way of dealing tiles: checks, the schedule, its table.
using Dealing = size_t (*)(const int32_t *, const int32_t *, int, int, int, int,
                           std::vector<TileRec> &);
static lbm_status export_schedule(Dealing deal, const int32_t *nx, const int32_t *ny,
                                  int32_t count, int32_t tx, int32_t ty, int32_t grid,
                                  int32_t *out, int64_t cap, int32_t *slots) {
    if (!nx || !ny || !slots || count < 1 || tx < 1 || ty < 1 || grid < 1)
        return fail(nullptr, LBM_EINVAL, "plan_tiles: NULL array, count, tile or grid < 1");
    for (int l = 0; l < count; ++l)
        if (nx[l] < 1 || ny[l] < 1)
            return fail(nullptr, LBM_EINVAL, "plan_tiles: lattice size < 1");
    std::vector<TileRec> sched;
    const size_t n = deal(nx, ny, count, tx, ty, grid, sched);
    *slots = (int32_t)n;
    if (!out) return LBM_OK;
    if ((int64_t)sched.size() * 3 > cap)
        return fail(nullptr, LBM_EINVAL, "plan_tiles: output holds fewer than 3 * grid * slots values");
    for (size_t k = 0; k < sched.size(); ++k) {
        out[3 * k] = sched[k].lat;
        out[3 * k + 1] = sched[k].lat >= 0 ? sched[k].x0 : 0;
        out[3 * k + 2] = sched[k].lat >= 0 ? sched[k].y0 : 0;
    }
    return LBM_OK;
}

extern "C" lbm_status lbm_plan_tiles(const int32_t *nx, const int32_t *ny,
                                     int32_t count, int32_t tx, int32_t ty,
                                     int32_t grid, int32_t *out, int64_t cap,
                                     int32_t *slots) {
    return export_schedule(plan_tiles, nx, ny, count, tx, ty, grid, out, cap, slots);
}

extern "C" lbm_status lbm_plan_schedule(const int32_t *nx, const int32_t *ny,
                                        int32_t count, int32_t tx, int32_t ty,
                                        int32_t grid, int32_t *out, int64_t cap,
                                        int32_t *slots) {
    return export_schedule(deal_tiles, nx, ny, count, tx, ty, grid, out, cap, slots);
}

extern "C" lbm_status lbm_fit_reff(const double *t, const double *z,
                                   int32_t n, double gamma, double mu,
                                   double length, double cos_theta0,
                                   double *r_eff) {
    if (!t || !z || !r_eff || n < 2 || !(gamma > 0) || !(cos_theta0 != 0))
        return LBM_EINVAL;
    double st = 0, sz = 0;
    for (int i = 0; i < n; ++i) { st += t[i]; sz += z[i]; }
    const double mt = st / n, mz = sz / n;
    double num = 0, den = 0;
    for (int i = 0; i < n; ++i) {
        num += (t[i] - mt) * (z[i] - mz);
        den += (t[i] - mt) * (t[i] - mt);
    }
    if (!(den > 0)) return LBM_EINVAL;
    const double v = num / den;
    *r_eff = 3.0 * mu * length * v / (gamma * cos_theta0);
    return LBM_OK;
}

// ---- autotuner ---------------------------------------------------------------

extern "C" lbm_status lbm_get_tuning(const lbm_handle *h, lbm_tuning *out) {
    if (!h || !out) return LBM_EINVAL;
    out->kernel = h->use_tma ? 1 : 0;
    out->tx = h->tx;
    out->ty = h->ty;
    out->ms_per_step = 0.0;
    return LBM_OK;
}

extern "C" int32_t lbm_get_on_chip(const lbm_handle *h, int32_t *tx, int32_t *ty) {
    if (!h) return -1;
    if (h->csize > 0) {
        if (tx) *tx = h->ctx;
        if (ty) *ty = h->cty;
    }
    return h->csize;
}

extern "C" lbm_status lbm_autotune(lbm_handle *h, int32_t steps,
                                   lbm_tuning *out) {
    if (!h || steps < 1) return fail(h, LBM_EINVAL, "bad handle or steps < 1");
    if (h->dead) return fail(h, LBM_ECUDA, "handle is dead: " + h->err);
    CK(h, cudaStreamSynchronize(h->stream));
    // snapshot of everything a step changes
    const size_t esz = 4;
    struct Piece { void *dev; size_t bytes; };
    const int cur0 = h->cur;
    const int64_t steps0 = h->steps;
    std::vector<Piece> parts = {
        {h->d_pop[cur0], (size_t)h->pop_elems * esz},
        {h->d_mask, (size_t)h->node_elems},
        {h->d_m, (size_t)h->node_elems * 8},
        {h->d_col_fluid, (size_t)h->nsec * 4},
        {h->d_st, (size_t)h->count * sizeof(LatState)},
        {h->d_step + cur0, 8}};
    size_t total = 0;
    for (auto &p : parts) total += (p.bytes + 255) / 256 * 256;
    char *snap = nullptr;
    if (cudaMalloc(&snap, total) != cudaSuccess) {
        return fail(h, LBM_ENOMEM, "autotune: no room for a state copy");
    }
    auto copy_all = [&](bool save) -> cudaError_t {
        size_t off = 0;
        for (auto &p : parts) {
            cudaError_t e = save ? cudaMemcpyAsync(snap + off, p.dev, p.bytes,
                                                   cudaMemcpyDeviceToDevice, h->stream)
                                 : cudaMemcpyAsync(p.dev, snap + off, p.bytes,
                                                   cudaMemcpyDeviceToDevice, h->stream);
            if (e != cudaSuccess) return e;
            off += (p.bytes + 255) / 256 * 256;
        }
        return cudaStreamSynchronize(h->stream);
    };
    struct Cand { bool tma; int tx, ty; };
    const Cand cands[] = {{true, 32, 16}, {true, 32, 8},  {true, 64, 4},
                          {true, 64, 8},  {true, 32, 4},  {true, 128, 4},
                          {false, 32, 8}, {false, 32, 4}, {false, 64, 4},
                          {false, 128, 4}};
    const Cand orig = {h->use_tma, h->tx, h->ty};
    // the variants are what a single step uses; steps on chip are set aside
    const int csize0 = h->csize;
    h->csize = 0;
    Cand best = orig;
    double best_ms = 1e300;
    lbm_status st = LBM_OK;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t ce = copy_all(true);
    if (ce == cudaSuccess) ce = cudaEventCreate(&e0);
    if (ce == cudaSuccess) ce = cudaEventCreate(&e1);
    for (const Cand &c : cands) {
        if (ce != cudaSuccess || st != LBM_OK) break;
        if (retile(h, c.tma, c.tx, c.ty) != LBM_OK) {
            st = LBM_OK;  // shape not available on this device: skip it
            h->err.clear();
            continue;
        }
        st = lbm_step(h, kGraphSteps + 2);  // warm-up, graph capture
        if (st != LBM_OK) break;
        const int n = (steps + kGraphSteps - 1) / kGraphSteps * kGraphSteps;
        ce = cudaEventRecord(e0, h->stream);
        if (ce == cudaSuccess) st = lbm_step(h, n);
        if (ce == cudaSuccess && st == LBM_OK) ce = cudaEventRecord(e1, h->stream);
        if (ce == cudaSuccess && st == LBM_OK) ce = cudaEventSynchronize(e1);
        float ms = 0.f;
        if (ce == cudaSuccess && st == LBM_OK) ce = cudaEventElapsedTime(&ms, e0, e1);
        if (ce == cudaSuccess && st == LBM_OK && ms / n < best_ms) {
            best_ms = ms / n;
            best = c;
        }
        // back to the saved state (its lattice totals are not kept)
        if (ce == cudaSuccess) ce = copy_all(false);
        h->cur = cur0;
        h->steps = steps0;
        h->sums_step = -1;
    }
    h->csize = csize0;
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(snap);
    if (st != LBM_OK) return st;
    CK(h, ce);
    lbm_status r = retile(h, best.tma, best.tx, best.ty);
    if (r != LBM_OK) return r;
    if (out) {
        out->kernel = best.tma ? 1 : 0;
        out->tx = best.tx;
        out->ty = best.ty;
        out->ms_per_step = best_ms;
    }
    return LBM_OK;
}
