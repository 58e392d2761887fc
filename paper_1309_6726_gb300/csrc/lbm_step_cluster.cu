// lbm_step_cluster.cu -- many steps of a small lattice in one launch, its
// state on chip.  A lattice of at most 16 tiles is advanced by one thread
// block cluster, one block per tile: the tile's populations (two buffers, with
// the two-node halo the pulls reach into) and its mask stay in the block's
// shared memory from the first step to the last.  A node writes its
// post-collision values to its own cell and, next to the tile's edge, to the
// halo cells of the neighbouring tiles through distributed shared memory; the
// periodic images are the halos of the tiles across the lattice.  One cluster
// barrier per step is all the synchronisation there is.  Device memory is
// read once, written once, and in between only for deposits, ledgers and
// flags.  Per node the step is that of lbm_step_tma.cu, in the same order, so
// the results are the same bit for bit.
//
// What bounds it: the latency of one tile's step.  Stamped per warp (256 x 32,
// FP32, 64 x 8 tiles): pull and density ring 960 cycles (1580 in the warps that
// take the ring), update with the stores to other blocks 3090, cluster barrier
// 1270 to arrive (its release waits for those stores) and 860 to pass; issue
// slots 38 % busy, top stalls barrier 1.9 and membar 1.5 per issue.  Against
// one launch per step (which adds the launch, the reload from L2 and the drain
// of the stores): 256 x 32 FP32 3.9 -> 2.7 us per step, FP16 3.9 -> 3.05, 131 x
// 13 FP16 3.8 -> 3.3.  Stores to other blocks are what the halo costs: sending
// every value of the two edge rows and columns, from the registers or copied
// from shared memory afterwards in 16-byte words, measured 3.3 and 3.5 us;
// only what the other tile reads goes out.
#include "lbm_tile.cuh"

namespace lbmk {

constexpr int kClusterTiles = 16;  // most tiles of a lattice

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n"
                 "barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Shared-memory address `p` of this block, in block `rank` of the cluster.
__device__ __forceinline__ unsigned peer_addr(unsigned p, unsigned rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(p), "r"(rank));
    return r;
}
__device__ __forceinline__ void peer_st32(unsigned addr, unsigned v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void peer_st8(unsigned addr, unsigned v) {
    asm volatile("st.shared::cluster.u8 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

template <class S, int TX, int TY>
struct ClusterTile : TmaTile<S, TX, TY> {
    using B = TmaTile<S, TX, TY>;
    static constexpr int POPS = B::NPL * B::PL;  // words of a buffer
    static constexpr int MASK_AT = (2 * POPS * 4 + 127) / 128 * 128;
    static constexpr int RHO_AT = MASK_AT + B::MASK_BYTES;
    static constexpr int DESC_AT = RHO_AT + B::RHO_AL;
    static constexpr int BYTES = DESC_AT + 128;
    static_assert(BYTES <= 232448, "shared memory per block");
};

template <class S, int TX, int TY>
__global__ void __launch_bounds__(TX *TY, 1)
    k_step_cluster(StepArgs a, int nsteps, int csize) {
    using TT = ClusterTile<S, TX, TY>;
    using T = typename S::T;
    extern __shared__ __align__(128) unsigned char smem[];
    T *const pops = reinterpret_cast<T *>(smem);  // buffer b at b * TT::POPS
    uint8_t *const sm = smem + TT::MASK_AT;
    float *const fr = reinterpret_cast<float *>(smem + TT::RHO_AT);
    LatDesc &d = *reinterpret_cast<LatDesc *>(smem + TT::DESC_AT);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int l = blockIdx.x / csize, rank = (int)cluster_rank();
    if (tid < 32)
        reinterpret_cast<uint32_t *>(&d)[tid] =
            reinterpret_cast<const uint32_t *>(a.desc + l)[tid];
    __syncthreads();
    const int nx = d.nx, ny = d.ny;
    const int tiles_x = (nx + TX - 1) / TX, tiles_y = (ny + TY - 1) / TY;
    const bool mine = rank < tiles_x * tiles_y;  // (a smaller lattice of the batch)
    const int cxt = rank % tiles_x, cyt = rank / tiles_x;
    const int tx0 = cxt * TX, ty0 = cyt * TY;
    const long long t0 = *a.step;

    // ---- load the tile with its halo --------------------------------------
    if (mine) {
        const T *in = static_cast<const T *>(a.fin) + d.pop_off;
        const uint8_t *mk = a.mask + d.node_off;
        for (int e = tid; e < TT::PL; e += TT::NT) {
            const int r = e / TT::BX, c = e - r * TT::BX;
            const int x = tx0 - TT::XO + c, y = ty0 - 2 + r;
            const bool ok = x >= -GHOST && x < nx + GHOST && y >= -GHOST && y < ny + GHOST;
            const int off = y * d.pitch + x;
            for (int q = 0; q < TT::NPL; ++q) {
                pops[q * TT::PL + e] = ok ? in[q * d.plane + off] : T(0);
                pops[TT::POPS + q * TT::PL + e] = T(0);
            }
        }
        for (int e = tid; e < TT::BY * TT::MBX; e += TT::NT) {
            const int r = e / TT::MBX, c = e - r * TT::MBX;
            const int x = tx0 - TT::MXO + c, y = ty0 - 2 + r;
            const bool ok = x >= -GHOST && x < nx + GHOST && y >= -GHOST && y < ny + GHOST;
            sm[e] = ok ? mk[y * d.pitch + x] : (uint8_t)0;
        }
    }

    // ---- this thread's node and where else its values are read --------------
    const int lx = tid % TX, ly = tid / TX;
    const int x = tx0 + lx, y = ty0 + ly;
    const bool active = mine && x < nx && y < ny;
    const int own = y * d.pitch + x;
    const int pc = (ly + 2) * TT::BX + lx + TT::XO;    // stage cell
    const int mc = (ly + 2) * TT::MBX + lx + TT::MXO;  // mask cell
    const int n_act = min(TY, ny - ty0), m_act = min(TX, nx - tx0);
    const bool in_frame = mine && lx <= m_act && ly <= n_act;
    // Per axis: the node's cell in the previous tile's far halo (its first
    // two columns or rows) and in the next tile's near halo (its last two).
    // Tiles are at least two wide (the host's rule), so no other tile sees
    // it; the first tile's previous one is the last across the period.
    const int wl = tiles_x > 1 && cxt == 0 ? nx - (tiles_x - 1) * TX : TX;  // its width
    const int hd = tiles_y > 1 && cyt == 0 ? ny - (tiles_y - 1) * TY : TY;
    const bool left = active && lx < 2, right = active && lx >= m_act - 2;
    const bool down = active && ly < 2, up = active && ly >= n_act - 2;
    const int prev_w = tiles_x == 1 ? nx : wl, prev_h = tiles_y == 1 ? ny : hd;
    const int tl = cxt == 0 ? tiles_x - 1 : cxt - 1, tr = cxt + 1 == tiles_x ? 0 : cxt + 1;
    const int td = cyt == 0 ? tiles_y - 1 : cyt - 1, tu = cyt + 1 == tiles_y ? 0 : cyt + 1;
    // Calls f(rank, dx, dy, sx, sy) for each of them: (dx, dy) from this node's
    // position in its tile to that in the other one; sx, sy the side of this
    // tile that the other one lies on (-1, 0, 1), doubled where the node is the
    // second from that side.
    const int sl = lx == 0 ? -1 : -2, sr = lx == m_act - 1 ? 1 : 2;
    const int sd = ly == 0 ? -1 : -2, su = ly == n_act - 1 ? 1 : 2;
    auto images = [&](auto f) {
        if (left) f(cyt * tiles_x + tl, prev_w, 0, sl, 0);
        if (right) f(cyt * tiles_x + tr, -m_act, 0, sr, 0);
        if (down) {
            f(td * tiles_x + cxt, 0, prev_h, 0, sd);
            if (left) f(td * tiles_x + tl, prev_w, prev_h, sl, sd);
            if (right) f(td * tiles_x + tr, -m_act, prev_h, sr, sd);
        }
        if (up) {
            f(tu * tiles_x + cxt, 0, -n_act, 0, su);
            if (left) f(tu * tiles_x + tl, prev_w, -n_act, sl, su);
            if (right) f(tu * tiles_x + tr, -m_act, -n_act, sr, su);
        }
    };
    // What the other tile reads of the node: next to it, every D2Q9 value (its
    // nodes pull the ones that come towards them, its density ring the others)
    // and, straight across, the solute that comes towards it; one node further
    // off, only what the ring pulls from there, the directions that point to
    // the other tile along each such axis.
    auto q9_read = [](int i, int sx, int sy) {
        return (abs(sx) < 2 || 2 * cx(i) == sx) && (abs(sy) < 2 || 2 * cy(i) == sy);
    };
    auto q4_read = [](int k, int sx, int sy) {
        return sy == 0 ? sx == lbmk::sx(k) && sx != 0 : sx == 0 && sy == lbmk::sy(k);
    };
    const unsigned pops_a = (unsigned)__cvta_generic_to_shared(pops);
    const unsigned mask_a = (unsigned)__cvta_generic_to_shared(sm);
    auto put_mask = [&](uint8_t v) {
        sm[mc] = v;
        images([&](int rk, int dx, int dy, int, int) {
            peer_st8(peer_addr(mask_a + mc + dy * TT::MBX + dx, rk), v);
        });
    };
    cluster_sync();
    const uint8_t s_first = in_frame ? sm[mc] : (uint8_t)0;

    for (int step = 0; step < nsteps; ++step) {
        const long long t = t0 + step;
        const MaskBits mb(t);
        const T *tp = pops + (step & 1) * TT::POPS;
        const unsigned np_a = pops_a + ((step & 1) ^ 1) * TT::POPS * 4 + 4 * pc;
        T *np = pops + ((step & 1) ^ 1) * TT::POPS;
        uint8_t s_own = 0xFF;
        bool own_pull_fluid = false;
        unsigned snb = 0;
        float fA[Q], fB[Q], g[QS];
        float2 f2[Q];
        float2 rho = make_float2(0.f, 0.f);
        if (mine) {
            if (in_frame) s_own = sm[mc];
            own_pull_fluid = !(s_own & mb.pull);
            const bool clean = warp_clean<TT>(sm, ly, lx & ~31, lane,
                                              (uint8_t)(mb.pull | mb.force));
            const unsigned bb = clean ? 0u : nb_bits<TT, -1>(sm, mc, mb.pull);
            snb = clean ? 0u : nb_bits<TT, +1>(sm, mc, mb.force);
            if (own_pull_fluid) {
                spull22<S, TT>(tp, pc, bb, clean, fA, fB, f2, g);
                if constexpr (S::kHalf) {
                    rho = dens2(f2);
                } else {
#pragma unroll
                    for (int i = 0; i < Q; ++i) { rho.x += fA[i]; rho.y += fB[i]; }
                }
            }
            const float2 q = s_own & mb.force ? make_float2(0.f, 0.f) : rho;
            const int fc = (ly + 1) * TT::RX + lx + 1;
            if constexpr (S::kHalf) {
                reinterpret_cast<float2 *>(fr)[fc] = q;
            } else {
                fr[fc] = q.x;
                fr[TT::RX * TT::RY + fc] = q.y;
            }
            // ring of the density frame
            const int r = warp * TT::RW + lane;
            if (r < TT::NRING) {
                int ry, rx;
                if (r < TT::RX) { ry = 0; rx = r; }
                else if (r < 2 * TT::RX) { ry = TT::RY - 1; rx = r - TT::RX; }
                else if (r < 2 * TT::RX + TY) { ry = 1 + r - 2 * TT::RX; rx = 0; }
                else { ry = 1 + r - 2 * TT::RX - TY; rx = TT::RX - 1; }
                const int rmc = (ry + 1) * TT::MBX + rx - 1 + TT::MXO;
                const int rpc = (ry + 1) * TT::BX + rx - 1 + TT::XO;
                float2 p = make_float2(0.f, 0.f);
                if (!(sm[rmc] & mb.force)) {
                    const unsigned rbb = nb_bits<TT, -1>(sm, rmc, mb.pull);
                    p = sdens<S, TT>(tp, rpc, rbb, rbb == 0u);
                }
                const int rc = ry * TT::RX + rx;
                if constexpr (S::kHalf) {
                    reinterpret_cast<float2 *>(fr)[rc] = p;
                } else {
                    fr[rc] = p.x;
                    fr[TT::RX * TT::RY + rc] = p.y;
                }
            }
        }
        __syncthreads();
        if (active) {
            if (s_own & mb.force) {
                if (own_pull_fluid) {
                    if constexpr (S::kHalf)
                        retire_node16(a, d, l, own, f2, g);
                    else
                        retire_node(a, d, l, own, fA, fB, g);
                }
                const uint8_t nb = s_own | mb.next;
                if (nb != s_own) put_mask(nb);
            } else {
                const int ns = __popc(snb & 0x1Eu);
                NodeTot tot;
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
                            store_words16(np + pc, TT::PL, v);
                            images([&](int rk, int dx, int dy, int sx, int sy) {
                                const unsigned p = peer_addr(np_a + 4 * (dy * TT::BX + dx), rk);
#pragma unroll
                                for (int i = 1; i < Q; ++i)
                                    if (q9_read(i, sx, sy)) peer_st32(p + 4 * (i - 1) * TT::PL, v[i - 1]);
                                const bool s01 = q4_read(0, sx, sy) || q4_read(1, sx, sy);
                                const bool s23 = q4_read(2, sx, sy) || q4_read(3, sx, sy);
                                if (s01) peer_st32(p + 4 * W16_SOL * TT::PL, v[W16_SOL]);
                                if (s23) peer_st32(p + 4 * (W16_SOL + 1) * TT::PL, v[W16_SOL + 1]);
                                if (s01 || s23) peer_st32(p + 4 * (W16_REF + 2) * TT::PL, v[W16_REF + 2]);
#pragma unroll
                                for (int w = W16_VEL; w < W16_REF + 2; ++w)
                                    peer_st32(p + 4 * w * TT::PL, v[w]);
                            });
                        },
                        false, tot);
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
                            store22_f32(reinterpret_cast<float *>(np) + pc, TT::PL, pa, pb, pg);
                            images([&](int rk, int dx, int dy, int sx, int sy) {
                                const unsigned p = peer_addr(np_a + 4 * (dy * TT::BX + dx), rk);
#pragma unroll
                                for (int i = 0; i < Q; ++i)
                                    if (q9_read(i, sx, sy)) {
                                        peer_st32(p + 4 * i * TT::PL, __float_as_uint(pa[i]));
                                        peer_st32(p + 4 * (Q + i) * TT::PL, __float_as_uint(pb[i]));
                                    }
#pragma unroll
                                for (int k = 0; k < QS; ++k)
                                    if (q4_read(k, sx, sy))
                                        peer_st32(p + 4 * (2 * Q + k) * TT::PL, __float_as_uint(pg[k]));
                            });
                        },
                        false, tot);
                }
                if (flagged) put_mask(s_own | mb.next);
            }
        }
        cluster_sync();
    }

    // ---- write the state back -----------------------------------------------
    if (active) {
        const uint8_t s = sm[mc];
        const T *fin = pops + (nsteps & 1) * TT::POPS + pc;
        if (!(s & MaskBits(t0 + nsteps - 1).force)) {  // updated in the last step
            T *out = static_cast<T *>(a.fout) + d.pop_off;
            auto put = [&](int off) {
#pragma unroll
                for (int q = 0; q < TT::NPL; ++q) out[q * (int)d.plane + off] = fin[q * TT::PL];
            };
            put(own);
            for_ghosts(x, y, nx, ny, d.pitch, own, put);
        }
        if (s != s_first) mask_store(a.mask + d.node_off, own, x, y, nx, ny, d.pitch, s);
    }
    if (blockIdx.x == 0 && tid == 0) *a.step_next = t0 + nsteps;
}

// ---- host side ---------------------------------------------------------------

// smallest first: fewer warps share an SM, and a step is one tile's latency
#define LBM_CLUSTER_SHAPES(M) M(32, 4) M(64, 4) M(64, 8)

template <class S, int TX, int TY>
static cudaError_t config_cluster(cudaLaunchConfig_t *c, cudaLaunchAttribute *at,
                                  int count, int csize, cudaStream_t s) {
    *c = {};
    c->gridDim = dim3(count * csize);
    c->blockDim = dim3(TX * TY);
    c->dynamicSmemBytes = ClusterTile<S, TX, TY>::BYTES;
    c->stream = s;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = csize;
    at->val.clusterDim.y = 1;
    at->val.clusterDim.z = 1;
    c->attrs = at;
    c->numAttrs = 1;
    cudaError_t e = cudaFuncSetAttribute(k_step_cluster<S, TX, TY>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         ClusterTile<S, TX, TY>::BYTES);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_step_cluster<S, TX, TY>,
                                 cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

// The tile with which lattices of these sizes can be advanced on chip, and
// the blocks per cluster; false where none can.  Every lattice needs at most
// 16 tiles, each at least two nodes wide and high.
bool plan_cluster(const int32_t *nx, const int32_t *ny, int count, int *tx,
                  int *ty, int *csize) {
#define LBM_CLUSTER_FIT(X, Y)                                                  \
    {                                                                          \
        int most = 0;                                                          \
        bool ok = true;                                                        \
        for (int l = 0; l < count && ok; ++l) {                                \
            const int tiles = ((nx[l] + X - 1) / X) * ((ny[l] + Y - 1) / Y);   \
            ok = tiles <= kClusterTiles && nx[l] >= 4 && ny[l] >= 4 &&         \
                 (nx[l] - 1) % X >= 1 && (ny[l] - 1) % Y >= 1;                 \
            most = tiles > most ? tiles : most;                                \
        }                                                                      \
        if (ok) {                                                              \
            *tx = X;                                                           \
            *ty = Y;                                                           \
            for (*csize = 1; *csize < most;) *csize *= 2;                      \
            return true;                                                       \
        }                                                                      \
    }
    LBM_CLUSTER_SHAPES(LBM_CLUSTER_FIT)
#undef LBM_CLUSTER_FIT
    return false;
}

template <class S, int TX, int TY>
static int active_clusters_t(int csize) {
    cudaLaunchConfig_t c;
    cudaLaunchAttribute at;
    int n = 0;
    if (config_cluster<S, TX, TY>(&c, &at, 1, csize, nullptr) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, k_step_cluster<S, TX, TY>, &c) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

template <class S, int TX, int TY>
static cudaError_t launch_cluster_t(const StepArgs &a, int count, int nsteps,
                                    int csize, cudaStream_t s) {
    cudaLaunchConfig_t c;
    cudaLaunchAttribute at;
    cudaError_t e = config_cluster<S, TX, TY>(&c, &at, count, csize, s);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&c, k_step_cluster<S, TX, TY>, a, nsteps, csize);
}

#define LBM_CLUSTER_STORE(F, X, Y, ...)                        \
    (store == 2   ? F<Store16<BF16>, X, Y>(__VA_ARGS__)        \
     : store == 1 ? F<Store16<F16>, X, Y>(__VA_ARGS__)         \
                  : F<Store32, X, Y>(__VA_ARGS__))

// Clusters of that tile and size that fit the device at once (0: none).
int active_clusters(int tx, int ty, int store, int csize) {
#define LBM_CLUSTER_CASE(X, Y) \
    if (tx == X && ty == Y) return LBM_CLUSTER_STORE(active_clusters_t, X, Y, csize);
    LBM_CLUSTER_SHAPES(LBM_CLUSTER_CASE)
#undef LBM_CLUSTER_CASE
    return 0;
}

// nsteps >= 1 steps of `count` lattices from a.fin to a.fout.
cudaError_t launch_step_cluster(const StepArgs &a, int count, int nsteps,
                                int tx, int ty, int csize, int store,
                                cudaStream_t s) {
#define LBM_CLUSTER_CASE(X, Y)     \
    if (tx == X && ty == Y)        \
        return LBM_CLUSTER_STORE(launch_cluster_t, X, Y, a, count, nsteps, csize, s);
    LBM_CLUSTER_SHAPES(LBM_CLUSTER_CASE)
#undef LBM_CLUSTER_CASE
    return cudaErrorInvalidValue;
}

}  // namespace lbmk
