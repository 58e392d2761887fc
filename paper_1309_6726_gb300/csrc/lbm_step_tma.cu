// lbm_step_tma.cu -- the fused reactive step with TMA-staged tiles
// (sm_103a).  Same per-node work as the direct kernel in lbm_step.cu; what
// differs is how the populations reach the SM:
//
//   * the kernel is persistent: a grid of (SM count x resident blocks)
//     walks the tiles of every lattice of the batch;
//   * for each tile of TX x TY nodes, one thread issues a 3-D bulk tensor
//     copy (cp.async.bulk.tensor) of the population planes (32-bit words:
//     22 FP32 values, or the 15 words of FP16 storage) over the tile plus
//     a halo of 2 rows and 4 columns -- the x start stays 16-byte aligned
//     -- into shared memory, completing on an mbarrier; the mask box and
//     the lattice descriptor come with it;
//   * two stages: the copy of the next tile is in flight while the current
//     one is computed;
//   * all pulls -- the tile's own nodes and the one-node density ring the
//     cohesion stencil needs -- then read shared memory at fixed offsets;
//   * the post-collision values of tiles up to 256 nodes are stored node by
//     node; larger tiles, and FP32 32 x 8, write them to a shared output tile
//     that one bulk tensor store copies out (TmaTile::NOUT);
//   * the lattice planes carry a two-node periodic ghost band (rows and
//     columns), so every copy reads valid neighbours and nothing needs
//     patching;
//   * every wait on an mbarrier is bounded; on time-out the kernel records
//     an error, lets its copies in flight land and returns.
#include <cuda.h>

#include "lbm_tile.cuh"

namespace lbmk {

// ---- PTX wrappers ----------------------------------------------------------

__device__ __forceinline__ unsigned smem_u32(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(count)
                 : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                     smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Waits for the phase with the given parity to complete; gives up after
// about two seconds (or 2^26 polls) and returns false.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar,
                                                  unsigned parity) {
    const long long t0 = clock64();
    for (unsigned it = 0; it < (1u << 26); ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if (clock64() - t0 > 4000000000LL) break;
    }
    return false;
}

__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap *m) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
// Programmatic dependent launch: lets the next launch of the stream start
// its blocks where there is room, and waits for the previous launch to end
// and its writes to be visible (both no-ops for a plain launch).
__device__ __forceinline__ void launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void grid_dependency_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map,
                                            int c0, int c1, int c2,
                                            uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::"
        "bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2),
        "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map,
                                            int c0, int c1, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::"
        "bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1),
        "r"(smem_u32(bar))
        : "memory");
}

// Bulk tensor store of a shared-memory box to global memory (elements
// outside the tensor are skipped), committed as one bulk group.
__device__ __forceinline__ void tma_store_3d(const CUtensorMap *map,
                                             const void *src, int c0, int c1,
                                             int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.global.shared::cta.bulk_group "
        "[%0, {%1, %2, %3}], [%4];" ::"l"(reinterpret_cast<uint64_t>(map)),
        "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(src))
        : "memory");
}
__device__ __forceinline__ void bulk_commit() {
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// The shared memory of every committed store has been read.
__device__ __forceinline__ void bulk_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
// Every committed store has completed.
__device__ __forceinline__ void bulk_wait_all() {
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ void bulk_load(void *dst, const void *src,
                                          unsigned bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// Tensor maps of one launch, per lattice: the tile copies (populations,
// mask) and the output stores.
struct TmaMaps {
    const CUtensorMap *pop, *mask, *out;
};

// SUM: the launch also adds up the lattice totals (StepArgs::sums).
template <class S, int TX, int TY, bool SUM>
__global__ void __launch_bounds__(TX *TY, (TmaTile<S, TX, TY>::MINB))
    k_step_tma(StepArgs a, TmaMaps mp, const TileRec *__restrict__ sched,
               int nslots, int *__restrict__ err) {
    using TT = TmaTile<S, TX, TY>;
    using T = typename S::T;
    extern __shared__ __align__(128) unsigned char smem[];
    auto stage_pop = [&](int s) { return reinterpret_cast<T *>(smem + s * TT::STAGE); };
    auto stage_mask = [&](int s) { return smem + s * TT::STAGE + TT::MASK_OFF; };
    auto sdesc = [&](int slot) {
        return reinterpret_cast<LatDesc *>(smem + TT::DESC_OFF + 128 * slot);
    };
    auto srho = [&](int f) {
        return reinterpret_cast<float *>(smem + TT::RHO_OFF + f * TT::RHO_AL);
    };
    constexpr int NS = TT::NS, NSL = TT::NSL;
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + TT::BAR_OFF);  // NS
    long long *s_t = reinterpret_cast<long long *>(bar + 3);
    TileRec *s_rec = reinterpret_cast<TileRec *>(bar + 4);  // tile of each desc slot

    // This block's tiles: sched[blockIdx.x + k * gridDim.x], k = 0, 1, ...,
    // until the first -1; consecutive entries mostly walk down one tile
    // column of a lattice, so the halo rows a tile copies were copied by the
    // previous tile of the same block and come from L2.
    auto sched_at = [&](int k) {
        return k < nslots ? sched[blockIdx.x + (size_t)k * gridDim.x]
                          : TileRec{-1, 0, 0, 0};
    };

    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;

    // Copies tile r into stage s and its lattice descriptor into `slot`.
    auto issue = [&](const TileRec &r, int s, int slot, int extra_tx) {
        const int l = r.lat;
        // physical coordinates: column x0 - XO and row y0 - 2 of the lattice
        const int x0 = r.x0 + XGHOST;
        const int y0 = r.y0;
        fence_proxy_async();
        mbar_expect_tx(&bar[s], TT::TX_BYTES + extra_tx);
        bulk_load(sdesc(slot), a.desc + l, 128, &bar[s]);
        tma_load_3d(stage_pop(s), &mp.pop[l], x0 - TT::XO, y0, 0, &bar[s]);
        tma_load_2d(stage_mask(s), &mp.mask[l], x0 - TT::MXO, y0, &bar[s]);
    };

    // What the previous launch does not write comes before the wait for it:
    // the barriers, the schedule, the tensor maps.
    if (tid == 0) {
        for (int j = 0; j < NS; ++j) mbar_init(&bar[j], 1);
        fence_mbar_init();
        bool more = true;
        for (int j = 0; j < NSL; ++j) {
            const TileRec r = more && j < NS ? sched_at(j) : TileRec{-1, 0, 0, 0};
            s_rec[j] = r;
            more = r.lat >= 0;
        }
        if (s_rec[0].lat >= 0) {
            prefetch_map(&mp.pop[s_rec[0].lat]);
            prefetch_map(&mp.mask[s_rec[0].lat]);
        }
    }
    launch_dependents();
    grid_dependency_wait();
    if (tid == 0) {
        for (int j = 0; j < NS && s_rec[j].lat >= 0; ++j)
            // (the test hook: block 0's first tile waits for bytes that
            // never come, so its bounded wait runs out)
            issue(s_rec[j], j, j, j == 0 && blockIdx.x == 0 ? a.stall_tx : 0);
    }
    if (tid == 32) *s_t = *a.step;  // (beside thread 0's chain of loads)
    __syncthreads();
    const long long t = *s_t;
    const MaskBits mb(t);

    // output tiles in shared memory (TS): node lid = ly * TX + lx of plane q
    // at sout(b)[q * NT + lid]
    auto sout = [&](int b) {
        return reinterpret_cast<T *>(smem + TT::OUT_OFF +
                                     (TT::NOUT == 2 ? (b & 1) : 0) * TT::OUT_BYTES);
    };
    // bulk tensor store of output tile b (thread 0; every thread fenced its
    // writes and passed a barrier since)
    auto store_out = [&](const TileRec &r, int b) {
        tma_store_3d(&mp.out[r.lat], sout(b), r.x0, r.y0, 0);
        bulk_commit();
    };
    // thread 0: the tile whose output awaits its store, and its output tile
    TileRec prev{-1, 0, 0, 0};
    int prev_buf = 0;
    bool failed = false;
    // gives up after a bounded wait ran out: lets the copies still in
    // flight land before exiting
    auto give_up = [&](int k, unsigned par) {
        if (tid == 0) {
            atomicOr(err, 1);
            for (int j = 1; j < NS; ++j) {
                if (s_rec[(k + j) % NSL].lat < 0) break;
                const int sj = (k + j) % NS;
                mbar_wait_bounded(&bar[sj], (par >> sj) & 1u);
            }
        }
    };

    unsigned parity = 0u;  // bit s: phase parity of stage s
    TotAcc acc;
    if constexpr (SUM) tot_reset(acc, -1);
    for (int k = 0; s_rec[k % NSL].lat >= 0; ++k) {
        // the record of the tile NS ahead, fetched now so that its load
        // latency hides behind this tile's work
        TileRec nxt{-1, 0, 0, 0};
        if (tid == 0 && s_rec[(k + NS - 1) % NSL].lat >= 0) nxt = sched_at(k + NS);
        const int s = k % NS;
        const int slot = k % NSL;
        const bool ok = mbar_wait_bounded(&bar[s], (parity >> s) & 1u);
        parity ^= 1u << s;
        if constexpr (!TT::ONE_BAR) {
            if (__syncthreads_or(!ok)) {
                give_up(k, parity);
                failed = true;
                break;
            }
            // every thread finished the previous tile's output
            if (TT::TS && tid == 0 && prev.lat >= 0) store_out(prev, 0);
        }
        // (ONE_BAR: a thread whose wait ran out still reads the stage --
        // shared memory at fixed offsets, results discarded -- and the
        // failure is taken at the barrier below)
        const TileRec rc = s_rec[slot];
        const LatDesc &d = *sdesc(slot);
        const int l = rc.lat;
        const int nx = d.nx, ny = d.ny;
        const int tx0 = rc.x0, ty0 = rc.y0;
        // rows / columns of the tile that hold lattice nodes; frame
        // positions further out are never a node's neighbour
        const int n_act = min(TY, ny - ty0), m_act = min(TX, nx - tx0);
        T *tp = stage_pop(s);
        uint8_t *sm = stage_mask(s);

        // own node: mask bits, pull, density
        const int lx = tid % TX, ly = tid / TX;
        const int x = tx0 + lx, y = ty0 + ly;
        const bool active = (x < nx) && (y < ny);
        const bool in_frame = lx <= m_act && ly <= n_act;  // neighbour of a node
        const int pc = (ly + 2) * TT::BX + lx + TT::XO;    // stage cell
        const int mc = (ly + 2) * TT::MBX + lx + TT::MXO;  // mask cell
        const uint8_t s_own = in_frame ? sm[mc] : (uint8_t)0xFF;
        const bool own_pull_fluid = !(s_own & mb.pull);
        // warps whose rows and their neighbours hold no solid node skip the
        // neighbour bits (all zero) and the bounce-back selects
        const bool clean = warp_clean<TT>(sm, ly, lx & ~31, lane,
                                          (uint8_t)(mb.pull | mb.force));
        const unsigned bb = clean ? 0u : nb_bits<TT, -1>(sm, mc, mb.pull);   // sources solid
        const unsigned snb = clean ? 0u : nb_bits<TT, +1>(sm, mc, mb.force); // neighbours solid
        float fA[Q], fB[Q], g[QS];
        float2 f2[Q];  // FP16 storage: scaled {A, B} pairs
        float *fr = srho(k & 1);
        float2 rho = make_float2(0.f, 0.f);
        {
            if (own_pull_fluid) {
                spull22<S, TT>(tp, pc, bb, clean, fA, fB, f2, g);
                if constexpr (S::kHalf) {
                    rho = dens2(f2);
                } else {
#pragma unroll
                    for (int i = 0; i < Q; ++i) { rho.x += fA[i]; rho.y += fB[i]; }
                }
            }
            const bool force_solid = s_own & mb.force;
            const int fc = (ly + 1) * TT::RX + lx + 1;
            if constexpr (S::kHalf) {
                reinterpret_cast<float2 *>(fr)[fc] =
                    force_solid ? make_float2(0.f, 0.f) : rho;
            } else {
                fr[fc] = force_solid ? 0.f : rho.x;
                fr[TT::RX * TT::RY + fc] = force_solid ? 0.f : rho.y;
            }
        }
        // ring of the density frame: the lanes of the first warps take
        // RW consecutive ring cells each (consecutive addresses, no
        // shared-memory bank conflicts).  When the previous tile of this
        // block is the one just above (a strip walks down a
        // tile column), the top ring row is that tile's last frame row
        // (its last row of nodes and their side ring cells, same step),
        // copied instead of pulled again.
        {
            const TileRec rp = s_rec[(k + NSL - 1) % NSL];
            const bool above = k > 0 && rp.lat == rc.lat && rp.x0 == tx0 &&
                               rp.y0 + TY == ty0;
            const int r = warp * TT::RW + lane;
            if (lane < TT::RW && r < TT::NRING) {
                int ry, rx;
                if (r < TT::RX) { ry = 0; rx = r; }
                else if (r < 2 * TT::RX) { ry = TT::RY - 1; rx = r - TT::RX; }
                else if (r < 2 * TT::RX + TY) { ry = 1 + r - 2 * TT::RX; rx = 0; }
                else { ry = 1 + r - 2 * TT::RX - TY; rx = TT::RX - 1; }
                const int rmc = (ry + 1) * TT::MBX + rx - 1 + TT::MXO;
                const int rpc = (ry + 1) * TT::BX + rx - 1 + TT::XO;
                float2 q = make_float2(0.f, 0.f);
                if (above && ry == 0) {
                    const float *fp = srho((k + 1) & 1);
                    const int pf = TY * TT::RX + rx;
                    q = S::kHalf ? reinterpret_cast<const float2 *>(fp)[pf]
                                 : make_float2(fp[pf], fp[TT::RX * TT::RY + pf]);
                } else if (!(sm[rmc] & mb.force)) {
                    // per lane: a warp-uniform choice here measured slower
                    const unsigned rbb = nb_bits<TT, -1>(sm, rmc, mb.pull);
                    q = sdens<S, TT>(tp, rpc, rbb, rbb == 0u);
                }
                const int fc = ry * TT::RX + rx;
                if constexpr (S::kHalf) {
                    reinterpret_cast<float2 *>(fr)[fc] = q;
                } else {
                    fr[fc] = q.x;
                    fr[TT::RX * TT::RY + fc] = q.y;
                }
            }
        }
        fence_proxy_async();
        // Output through shared memory and a bulk tensor store, except for
        // tiles that end past the lattice's last column: a store box that
        // crosses x = nx was measured to overwrite the ghost columns there
        // (partial 16-byte rows are not clipped element by element), so
        // those tiles store their nodes directly.
        const bool ts_tile = TT::TS && tx0 + TX <= nx;
        if constexpr (TT::TS) {
            // the output tile written below must have been read by its last
            // store (ONE_BAR: the store of two tiles ago)
            if (tid == 0) bulk_wait_read();
        }
        if constexpr (TT::ONE_BAR) {
            if (__syncthreads_or(!ok)) {
                give_up(k, parity);
                failed = true;
                break;
            }
            // every thread finished the previous tile's output
            if (tid == 0) {
                if (prev.lat >= 0) store_out(prev, prev_buf);
                prev = ts_tile ? rc : TileRec{-1, 0, 0, 0};
                prev_buf = k & 1;
            }
        } else {
            if (TT::TS && tid == 0) prev = ts_tile ? rc : TileRec{-1, 0, 0, 0};
            __syncthreads();
        }
        // stage s is free: start the copy of the tile NS ahead into it
        if (tid == 0) {
            s_rec[(k + NS) % NSL] = nxt;
            if (nxt.lat >= 0) issue(nxt, s, (k + NS) % NSL, 0);
        }

        constexpr bool want = SUM;
        NodeTot tot{0.f, 0.f, 0.f};
        if (active) {
            const int own = y * d.pitch + x;
            const int lid = ly * TX + lx;
            if (s_own & mb.force) {
                if (own_pull_fluid) {
                    if constexpr (S::kHalf)
                        retire_node16(a, d, l, own, f2, g);
                    else
                        retire_node(a, d, l, own, fA, fB, g);
                }
                const uint8_t nb = s_own | mb.next;
                if (nb != s_own) mask_store(a.mask + d.node_off, own, x, y, nx, ny, d.pitch, nb);
            } else {
                const int ns = __popc(snb & 0x1Eu);
                bool flagged;
                if constexpr (S::kHalf) {
                    float2 nbv[Q];
#pragma unroll
                    for (int i = 1; i < Q; ++i)
                        nbv[i] = reinterpret_cast<const float2 *>(fr)[
                            (ly + 1 + cy(i)) * TT::RX + lx + 1 + cx(i)];
                    flagged = fluid_update16<typename S::Fmt>(
                        a, d, l, t, x, y, own, f2, g, rho, nbv, snb, ns,
                        [&](const uint32_t *v) {
                            if (ts_tile)
                                store_words16(sout(k) + lid, TT::NT, v);
                            else
                                store_words16(static_cast<uint32_t *>(a.fout) +
                                                  d.pop_off + own,
                                              (int)d.plane, v);
                            store_ghosts16(a, d, x, y, own, v);
                        },
                        want, tot);
                } else {
                    float rAn[Q], rBn[Q];
#pragma unroll
                    for (int i = 1; i < Q; ++i) {
                        const int fc = (ly + 1 + cy(i)) * TT::RX + lx + 1 + cx(i);
                        rAn[i] = fr[fc];
                        rBn[i] = fr[TT::RX * TT::RY + fc];
                    }
                    flagged = fluid_update(
                        a, d, l, t, x, y, own, fA, fB, g, rAn, rBn, snb, ns,
                        [&](const float *pa, const float *pb, const float *pg) {
                            if (ts_tile)
                                store22_f32(reinterpret_cast<float *>(sout(k)) + lid,
                                            TT::NT, pa, pb, pg);
                            else
                                store_node22(a, d, own, pa, pb, pg);
                            store_ghosts22(a, d, x, y, own, pa, pb, pg);
                        },
                        want, tot);
                }
                if (flagged)
                    mask_store(a.mask + d.node_off, own, x, y, nx, ny, d.pitch, s_own | mb.next);
            }
        }
        if constexpr (SUM) tot_add(acc, tot, l, a.sums, lane);
        if constexpr (TT::TS) fence_proxy_async();  // before the next barrier
    }
    if constexpr (TT::TS) {
        __syncthreads();
        if (tid == 0) {
            if (!failed && prev.lat >= 0) store_out(prev, prev_buf);
            bulk_wait_all();
        }
    }
    if constexpr (SUM) tot_flush(acc, a.sums, lane);
    next_step(a, t);
}

constexpr int kOverlapTiles = 8;  // most tiles per block of such launches

// ---- host side ---------------------------------------------------------------

template <class S, int TX, int TY>
static cudaError_t grid_tma_t(int *grid) {
    using TT = TmaTile<S, TX, TY>;
    cudaError_t e = cudaFuncSetAttribute(
        k_step_tma<S, TX, TY, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
        TT::SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_step_tma<S, TX, TY, true>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 TT::SMEM);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_step_tma<S, TX, TY, false>,
                                                      TX * TY, TT::SMEM);
    if (e != cudaSuccess) return e;
    *grid = sms * (per > 0 ? per : 1);
    return cudaSuccess;
}

template <class S, int TX, int TY>
static cudaError_t launch_tma_t(const StepArgs &a, const TmaMaps &mp,
                                const TileRec *sched, int nslots, int grid,
                                int *err, cudaStream_t s) {
    using TT = TmaTile<S, TX, TY>;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(TX * TY);
    c.dynamicSmemBytes = TT::SMEM;
    c.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    // Blocks of few tiles: the next launch starts under this one's tail and
    // waits in the kernel.  256 x 32 4.55 -> 4.15 us per step FP32, 4.75 ->
    // 4.1 FP16, 1000 x 60 5.95 -> 5.3, 4096 x 128 (6.7 tiles per block) 20.2
    // -> 19.9; with more tiles per block it costs (1024 x 1024 preform, 13.5:
    // 51.6 -> 52.7; sweep of 40 lattices 251.3 -> 254.4).
    c.numAttrs = nslots <= kOverlapTiles ? 1 : 0;
    return a.sums ? cudaLaunchKernelEx(&c, k_step_tma<S, TX, TY, true>, a, mp, sched, nslots, err)
                  : cudaLaunchKernelEx(&c, k_step_tma<S, TX, TY, false>, a, mp, sched, nslots, err);
}

#define LBM_TMA_SHAPES(M) M(32, 8) M(32, 4) M(64, 4) M(32, 16) M(64, 8) M(128, 4)

// Persistent grid of the TMA step kernel for a tile shape (also sets its
// shared-memory limit); 0 on an unsupported shape.
// store: 0 FP32, 1 FP16, 2 BF16 storage
cudaError_t grid_step_tma(int tx, int ty, int store, int *grid) {
    *grid = 0;
#define LBM_TMA_GRID(X, Y)                                                   \
    if (tx == X && ty == Y)                                                  \
        return store == 2   ? grid_tma_t<Store16<BF16>, X, Y>(grid)          \
               : store == 1 ? grid_tma_t<Store16<F16>, X, Y>(grid)           \
                            : grid_tma_t<Store32, X, Y>(grid);
    LBM_TMA_SHAPES(LBM_TMA_GRID)
#undef LBM_TMA_GRID
    return cudaErrorInvalidValue;
}

cudaError_t launch_step_tma(const StepArgs &a, const CUtensorMap *pop_maps,
                            const CUtensorMap *mask_maps,
                            const CUtensorMap *out_maps, const TileRec *sched,
                            int nslots, int grid, int tx, int ty, int store,
                            int *err, cudaStream_t s) {
    const TmaMaps mp{pop_maps, mask_maps, out_maps};
#define LBM_TMA_CASE(X, Y)                                                   \
    if (tx == X && ty == Y)                                                  \
        return store == 2                                                    \
                   ? launch_tma_t<Store16<BF16>, X, Y>(a, mp, sched, nslots, \
                                                       grid, err, s)         \
               : store == 1                                                  \
                   ? launch_tma_t<Store16<F16>, X, Y>(a, mp, sched, nslots,  \
                                                      grid, err, s)          \
                   : launch_tma_t<Store32, X, Y>(a, mp, sched, nslots, grid, \
                                                 err, s);
    LBM_TMA_SHAPES(LBM_TMA_CASE)
#undef LBM_TMA_CASE
    return cudaErrorInvalidValue;
}

// Tensor map geometry must match TmaTile: box (TX + 8) x (TY + 4) x
// planes of 32-bit words for the populations, (TX + 32) x (TY + 4) for the
// mask; the output maps span the lattice itself with box TX x TY x planes.
int tma_box_x(int tx) { return tx + 8; }
int tma_mask_box_x(int tx) { return tx + 32; }

}  // namespace lbmk
