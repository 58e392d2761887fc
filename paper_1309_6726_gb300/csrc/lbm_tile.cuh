// lbm_tile.cuh -- a tile of a lattice in shared memory, as the step kernels
// that work from there hold it (TMA-staged tiles in lbm_step_tma.cu, tiles
// that stay on chip for many steps in lbm_step_cluster.cu): its geometry and
// the pulls, densities and mask bits read from it.
#pragma once

#include "lbm_node.cuh"

namespace lbmk {

// ---- tile geometry -----------------------------------------------------------

template <class S, int TX_, int TY_>
struct TmaTile {
    using T = typename S::T;  // 32-bit words: FP32 values or 16-bit pairs
    using Fmt = typename S::Fmt;  // 16-bit format (16-bit storage)
    static constexpr int TX = TX_, TY = TY_;
    static constexpr int NT = TX * TY;
    static constexpr int NW = NT / 32;            // warps
    static constexpr int XO = 4;                  // halo columns copied (16 B)
    static constexpr int BX = TX + 2 * XO;        // box width
    static constexpr int BY = TY + 4;             // box height (halo 2)
    static constexpr int PL = BX * BY;            // words per plane
    static constexpr int MXO = 16;                // mask box: 16-byte aligned
    static constexpr int MBX = TX + 2 * MXO;
    // population planes of a stage: 22 FP32, or the 15 words of FP16 storage
    static constexpr int NPL = S::kPlanes;
    static constexpr int POP_BYTES = NPL * PL * 4;
    static constexpr int MASK_BYTES = (MBX * BY + 127) / 128 * 128;
    static constexpr int STAGE = ((POP_BYTES + 127) / 128 * 128) + MASK_BYTES;
    static constexpr int MASK_OFF = STAGE - MASK_BYTES;  // within a stage
    static constexpr int TX_BYTES = POP_BYTES + MBX * BY + 128;
    static constexpr int RX = TX + 2, RY = TY + 2;  // density frame
    static constexpr int NRING = 2 * RX + 2 * TY;
    // FP32: two planes rho_A, rho_B; FP16: one plane of {rho_A, rho_B}
    static constexpr int RHO_BYTES = 2 * RX * RY * 4;
    static constexpr int RHO_AL = (RHO_BYTES + 127) / 128 * 128;
    // Two stages: the copy of the next tile lands while this one is
    // computed (a third stage measured no faster).  One descriptor slot
    // more than stages: the current tile's stays readable while the next
    // copies land.
    static constexpr int NS = 2;
    static constexpr int NSL = NS + 1;
    static constexpr int DESC_OFF = NS * STAGE;                // NSL x 128
    static constexpr int RHO_OFF = DESC_OFF + NSL * 128;       // 2 frames
    // The tile's post-collision output, [NPL][TY][TX] words, written by
    // bulk tensor stores, or (NOUT 0) stored node by node in coalesced
    // 32-bit stores.  Tiles of up to 256 nodes run two blocks per SM at 128
    // registers, which hide each other's latencies; they store node by node,
    // without an output tile, and take one block barrier per tile (ONE_BAR).
    // For FP32 an output tile of 64 x 4 leaves room for one block only
    // (sweep of 40 lattices: one 512-thread block of 64 x 8 with an output
    // tile 267 us per step, two of 64 x 4 with direct stores 252; 4096 x 128:
    // 22.4 and 19.8; larger planes and batches the other way round, see
    // pick_tile).  FP32 32 x 8 fits two blocks with its output tile, and
    // keeps it: slower on capillaries (308 us on the sweep) but the fastest
    // where solid nodes are everywhere (1024 x 1024 preform: 44.0 us against
    // 50.9 without it and 48.4 at 64 x 4).  (FP16: the budget of three
    // blocks, 80 registers, spilled and measured 10 % slower on the batched
    // sweep at 64 x 4, whose stages leave room for two blocks only.)  Larger
    // FP16 tiles keep two output tiles, so that the store of one is issued
    // while the next is written; FP32 ones one, with two barriers per tile.
    static constexpr int OUT_BYTES = (NPL * NT * 4 + 127) / 128 * 128;
    static constexpr int OUT_OFF = RHO_OFF + 2 * RHO_AL;
    static constexpr int NOUT =
        S::kHalf ? (NT <= 256 ? 0 : (OUT_OFF + 2 * OUT_BYTES + 128 <= 232448 ? 2 : 0))
        : NT <= 256 ? (TX == 32 && TY == 8 ? 1 : 0)
                    : (OUT_OFF + OUT_BYTES + 128 <= 232448 ? 1 : 0);
    static constexpr bool TS = NOUT > 0;
    static constexpr bool ONE_BAR = S::kHalf || !TS;
    // blocks per SM the register budget is set for
    static constexpr int MINB = NT <= 256 ? 2 : 1;
    static constexpr int BAR_OFF = OUT_OFF + NOUT * OUT_BYTES;
    static constexpr int SMEM = BAR_OFF + 128;
    static_assert(SMEM <= 232448, "shared memory per block");
    static_assert((TX * 4) % 16 == 0, "store box row");
    static_assert(POP_BYTES % 16 == 0, "stage alignment");
    static_assert((BX * 4) % 16 == 0, "TMA box row");
    // ring cells per warp: whole warps take the ring (5 of 8 at 64 x 4),
    // since a warp costs the same issue slots with 10 lanes active as with
    // 32 (spreading it thinly over every warp measured 4 % slower for FP16)
    static constexpr int RW = 32;
    static_assert(NRING <= NT && RW <= 32, "ring spread");
    static_assert(TX % 32 == 0, "a warp covers 32 columns of one row");
};

// The 9 populations of component `comp` pulled into the node at stage cell
// `c`, from shared memory (bb: bounce-back bits), FP32 storage.  BB = false:
// no source is solid, every address is the node's cell plus a constant.
template <class TT, bool BB>
__device__ __forceinline__ void spull9(const float *tile, int comp, int c,
                                       unsigned bb, float f[Q]) {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const bool b = BB && ((bb >> i) & 1u);
        const int cell = b ? c : c - cy(i) * TT::BX - cx(i);
        const int qi = b ? opp(i) : i;
        f[i] = tile[(comp * Q + qi) * TT::PL + cell];
    }
}

template <class TT, bool BB>
__device__ __forceinline__ void spull4(const float *tile, int c, unsigned bb4,
                                       float g[QS]) {
#pragma unroll
    for (int k = 0; k < QS; ++k) {
        const bool b = BB && ((bb4 >> k) & 1u);
        const int cell = b ? c : c - sy(k) * TT::BX - sx(k);
        g[k] = tile[(2 * Q + (b ? sopp(k) : k)) * TT::PL + cell];
    }
}

// FP16 storage: the scaled {A, B} populations pulled into the node at
// stage cell c -- per direction one packed deviation word, the source's two
// FP32 references and its one or two linear-reference words; the rest
// populations are the node's own references.
template <class TT, bool BB>
__device__ __forceinline__ void spull16ab(const uint32_t *tile, int c,
                                          unsigned bb, float2 f[Q]) {
    const float *ref = reinterpret_cast<const float *>(tile) + W16_REF * TT::PL;
    f[0] = make_float2(ref[c], ref[TT::PL + c]);
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const bool b = BB && ((bb >> i) & 1u);
        const int cell = b ? c : c - cy(i) * TT::BX - cx(i);
        const int qi = b ? opp(i) : i;
        const uint32_t wx = cx(i) != 0 ? tile[W16_VEL * TT::PL + cell] : 0u;
        const uint32_t wy = cy(i) != 0 ? tile[(W16_VEL + 1) * TT::PL + cell] : 0u;
        f[i] = dec_pair<typename TT::Fmt>(i, b, tile[(qi - 1) * TT::PL + cell],
                        make_float2(ref[cell], ref[TT::PL + cell]), wx, wy);
    }
}

// FP16 storage: the 4 scaled solute populations (bb: the D2Q9 bounce-back
// bits; D2Q4 direction k is D2Q9 direction k + 1).
template <class TT, bool BB>
__device__ __forceinline__ void spull16s(const uint32_t *tile, int c,
                                         unsigned bb, float g[QS]) {
    const float *ref = reinterpret_cast<const float *>(tile) + (W16_REF + 2) * TT::PL;
#pragma unroll
    for (int k = 0; k < QS; ++k) {
        const bool b = BB && ((bb >> (k + 1)) & 1u);
        const int cell = b ? c : c - sy(k) * TT::BX - sx(k);
        const int qk = b ? sopp(k) : k;
        g[k] = dec_sol16<typename TT::Fmt>(tile[(W16_SOL + (qk >> 1)) * TT::PL + cell], qk,
                                           ref[cell]);
    }
}

// The 22 populations of the node at stage cell c, FP32 storage (fA, fB, g)
// or FP16 storage (scaled {A, B} pairs in fA2, solute in g).  `fast`
// (bb == 0 on every lane that calls) takes the path without bounce-back
// selects; the other path gives the same values for bb == 0, so a warp with
// any bounce-back lane runs that one alone.
template <class S, class TT>
__device__ __forceinline__ void spull22(const typename S::T *tile, int c,
                                        unsigned bb, bool fast, float fA[Q],
                                        float fB[Q], float2 fA2[Q],
                                        float g[QS]) {
    if constexpr (!S::kHalf) {
        if (fast) {
            spull9<TT, false>(tile, 0, c, 0u, fA);
            spull9<TT, false>(tile, 1, c, 0u, fB);
            spull4<TT, false>(tile, c, 0u, g);
        } else {
            spull9<TT, true>(tile, 0, c, bb, fA);
            spull9<TT, true>(tile, 1, c, bb, fB);
            spull4<TT, true>(tile, c, (bb >> 1) & 0xFu, g);
        }
    } else {
        if (fast) {
            spull16ab<TT, false>(tile, c, 0u, fA2);
            spull16s<TT, false>(tile, c, 0u, g);
        } else {
            spull16ab<TT, true>(tile, c, bb, fA2);
            spull16s<TT, true>(tile, c, bb, g);
        }
    }
}

// Densities of both components at stage cell c (`fast` as for spull22),
// formed as the node's own update forms them.
template <class S, class TT>
__device__ __forceinline__ float2 sdens(const typename S::T *tile, int c,
                                        unsigned bb, bool fast) {
    if constexpr (!S::kHalf) {
        float f[Q];
        float ra = 0.f, rb = 0.f;
        if (fast) {
            spull9<TT, false>(tile, 0, c, 0u, f);
#pragma unroll
            for (int i = 0; i < Q; ++i) ra += f[i];
            spull9<TT, false>(tile, 1, c, 0u, f);
#pragma unroll
            for (int i = 0; i < Q; ++i) rb += f[i];
        } else {
            spull9<TT, true>(tile, 0, c, bb, f);
#pragma unroll
            for (int i = 0; i < Q; ++i) ra += f[i];
            spull9<TT, true>(tile, 1, c, bb, f);
#pragma unroll
            for (int i = 0; i < Q; ++i) rb += f[i];
        }
        return make_float2(ra, rb);
    } else {
        float2 f[Q];
        if (fast)
            spull16ab<TT, false>(tile, c, 0u, f);
        else
            spull16ab<TT, true>(tile, c, bb, f);
        return dens2(f);
    }
}

// True when no node in rows ly - 1 .. ly + 1, columns c0 - 1 .. c0 + 32 of
// the tile (c0 = this warp's first column) has `bits` set in the mask box:
// then every node of the warp has no solid neighbour and no solid source.
// The 34 bytes of a row lie in 10 aligned words; lane j < 30 tests one.
template <class TT>
__device__ __forceinline__ bool warp_clean(const uint8_t *sm, int ly, int c0,
                                           int lane, uint8_t bits) {
    bool dirty = false;
    if (lane < 30) {
        const int row = lane / 10, w = lane % 10;
        const int off = (ly + 1 + row) * TT::MBX + TT::MXO + c0 - 4 + 4 * w;
        unsigned keep = 0xFFFFFFFFu;
        if (w == 0) keep = 0xFF000000u;  // column c0 - 1 only
        if (w == 9) keep = 0x000000FFu;  // column c0 + 32 only
        const unsigned v = *reinterpret_cast<const unsigned *>(sm + off);
        dirty = (v & keep & (bits * 0x01010101u)) != 0u;
    }
    return !__any_sync(0xFFFFFFFFu, dirty);
}

// Mask bits around the node at mask-box cell mc: bit i of the result is set
// when the node at mc + e_i (sign = +1) or mc - e_i (sign = -1) has `bit`.
template <class TT, int SIGN>
__device__ __forceinline__ unsigned nb_bits(const uint8_t *sm, int mc,
                                            uint8_t bit) {
    unsigned r = 0;
#pragma unroll
    for (int i = 1; i < Q; ++i)
        if (sm[mc + SIGN * (cy(i) * TT::MBX + cx(i))] & bit) r |= 1u << i;
    return r;
}

}  // namespace lbmk
