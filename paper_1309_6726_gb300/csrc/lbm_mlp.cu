// lbm_mlp.cu -- the surrogate network of lbm_mlp.h.  A pass over the network
// is one launch: a block carries 16, 32 or 64 rows of the batch through all
// layers, forward (k_net<., false>) or forward, loss and back to the first
// layer (k_net<., true>), with the activations in shared memory.  The weight
// gradients of all layers are one launch (k_dweight) and so is what follows
// them (k_finish: the sums over the parts, and Adam).  Products run on the
// tensor cores with BF16 operands and FP32 accumulation.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "../../include/lbm_mlp.h"

namespace lbmmlp {

constexpr int kMaxLayers = 9;      // L hidden + output
// warps of a k_net block, side by side along the units: 16 for 16 rows, where
// latency is all there is (8 -> 16: 256 rows forward 10.1 -> 8.6 us, a
// training step on 1024 rows 36.9 -> 32.6), else 8
__host__ __device__ constexpr int net_warps(int mt) { return mt == 1 ? 16 : 8; }
constexpr int kMaxBlocks = 608;    // most blocks of k_net (4 x 152 SMs)
constexpr int DT = 64, DR = 64;    // k_dweight: tile side, batch rows a stage
constexpr int DLD = DT + 8;        // padded row
constexpr int kDwThreads = 128;    // 2 x 2 warps
constexpr int kParts = 8;          // parts below which the sums are folded,
constexpr int kChains = 16;        // into that many chains

__host__ __device__ constexpr int pad32(int d) { return (d + 31) & ~31; }

// Layer l maps dim[l] inputs to dim[l + 1] units (dim[0] = n_in, the output
// layer is layer L).  Activations and gradients kept for k_dweight have rows
// of pad32(dim) BF16 values, zero beyond dim.
//
// Weights in BF16 are kept in the order the tensor-core operand wants them:
// for a tile of 8 units and 32 inputs, lane 4 g + t of a warp owns the 8
// values of unit g at inputs 2 t, 2 t + 1, 2 t + 8, 2 t + 9 and those 16
// further, as one 16-byte word, the 32 lanes' words back to back.  wf holds
// W (the forward products), wt its transpose (the gradients of the
// activations); both are zero beyond the layer's sizes.
struct Net {
    int L;                          // hidden layers
    int dim[kMaxLayers + 1];
    long off_w[kMaxLayers], off_b[kMaxLayers];  // in the packed parameters
    long off_f[kMaxLayers], off_t[kMaxLayers];  // in wf and wt
    int off_db[kMaxLayers];         // in a block's partial bias gradients
    int ndb;                        // length of those
    long np;
    float *w;
    __nv_bfloat16 *wf, *wt;
    float *hs[kMaxLayers];          // FP32 hidden activations of the rows that the
                                    // blocks work on, [block][16 MT][H]
    __nv_bfloat16 *act[kMaxLayers]; // inputs of layer l in BF16
    __nv_bfloat16 *dz[kMaxLayers];  // gradients at layer l's pre-activation
    float *db;                      // [blocks of k_net][ndb]
    double *loss;                   // [blocks of k_net]
    float *parts;                   // [split][np] partial weight gradients
};

// Place of weight (unit j, input i) of a layer with `in` inputs in wf; the
// same with the roles swapped in wt.
__device__ __forceinline__ long frag_at(int j, int i, int in) {
    const int r = i & 15;
    return (((long)(j >> 3) * (pad32(in) >> 5) + (i >> 5)) * 32 + (j & 7) * 4 +
            ((r & 7) >> 1)) * 8 + ((i >> 4) & 1) * 4 + (r >> 3) * 2 + (r & 1);
}

__device__ __forceinline__ void mma_bf16(float d[4], const unsigned a[4],
                                         unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
        "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm4(unsigned r[4], const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
}
__device__ __forceinline__ void ldsm4t(unsigned r[4], const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
}
__device__ __forceinline__ void st_bf2(__nv_bfloat16 *p, float a, float b) {
    *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(a, b);
}

// Programmatic dependent launch of the inference pass: its blocks start under
// the tail of the launch before it in the stream, let the next one start at
// once and wait here for the previous launch to end before they touch memory
// (back to back: 256 rows forward 8.7 -> 8.6 us, 1024 rows 9.1 -> 8.7, 8192
// rows 18.9 -> 18.5).
// Training's three launches are plain: with the weight gradients' blocks
// waiting on the SMs a step on 8192 rows took 102 us instead of 89.
__device__ __forceinline__ void start_after_previous() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// One product of a block: its rows (in shared memory, K columns) times a
// fragment-ordered matrix of N columns, in passes of up to 256 columns; warp
// v takes `ntw` neighbouring 8-column tiles of a pass.  Every weight is read
// once per block, from L2 straight into the register that feeds the tensor
// core: PF words of 32 inputs ahead, and the first PF of the next product
// before the current one's epilogue.
template <int MT, int PF>
struct Product {
    static constexpr int NW = net_warps(MT);
    static constexpr int TW = 32 / NW;  // most tiles of a warp
    const uint4 *bp;  // this lane's words of the warp's first tile
    int kt, cnt;      // words of 32 inputs; tiles of this warp, 0..TW
    int n0;           // first column of the warp
    uint4 q[PF][TW];

    __device__ __forceinline__ void start(const __nv_bfloat16 *wp, int K, int N,
                                          int pass, int warp, int lane) {
        kt = pad32(K) >> 5;
        const int left = min(32, (pad32(N) >> 3) - 32 * pass);
        const int ntw = (left + NW - 1) / NW;
        const int t0 = 32 * pass + warp * ntw;
        cnt = max(0, min(ntw, left - warp * ntw));
        n0 = 8 * t0;
        bp = reinterpret_cast<const uint4 *>(wp) + (long)t0 * kt * 32 + lane;
#pragma unroll
        for (int p = 0; p < PF; ++p) load(p, p);
    }
    __device__ __forceinline__ void load(int p, int k) {
        if (k >= kt) return;
#pragma unroll
        for (int j = 0; j < TW; ++j)
            if (j < cnt) q[p][j] = __ldg(bp + ((long)j * kt + k) * 32);
    }
    __device__ __forceinline__ void run(const __nv_bfloat16 *as, int ld, int lane,
                                        float acc[MT][TW][4]) {
#pragma unroll
        for (int mi = 0; mi < MT; ++mi)
#pragma unroll
            for (int j = 0; j < TW; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[mi][j][e] = 0.f;
        if (cnt == 0) return;
        const __nv_bfloat16 *ap = as + (lane & 15) * ld + (lane >> 4) * 8;
        for (int k0 = 0; k0 < kt; k0 += PF) {
#pragma unroll
            for (int p = 0; p < PF; ++p) {
                if (k0 + p >= kt) break;
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    unsigned af[MT][4];
#pragma unroll
                    for (int mi = 0; mi < MT; ++mi)
                        ldsm4(af[mi], ap + mi * 16 * ld + (k0 + p) * 32 + s * 16);
#pragma unroll
                    for (int j = 0; j < TW; ++j)
                        if (j < cnt) {
                            const unsigned b0 = s ? q[p][j].z : q[p][j].x;
                            const unsigned b1 = s ? q[p][j].w : q[p][j].y;
#pragma unroll
                            for (int mi = 0; mi < MT; ++mi) mma_bf16(acc[mi][j], af[mi], b0, b1);
                        }
                }
                load(p, k0 + p + PF);
            }
        }
    }
};

// A pass over the network for rows [16 MT blockIdx.x, + 16 MT) and every
// gridDim.x-th such tile after it.  TRAIN: also the loss, the gradients at
// every pre-activation (in BF16 for k_dweight) and the block's share of the
// bias gradients and of the loss; without it y receives the output.
//
// Bound by latency: the chain of products, each with 128 KB of weights from L2
// per block, and the epilogues' tanh (tensor pipe 4 % busy in training on 1024
// rows, 23 % forward on 8192).  One launch per product took 133 us forward on
// 256 rows and 158 on 8192; this 8.6 and 18.5.
template <int MT, bool TRAIN>
__global__ void __launch_bounds__(32 * net_warps(MT))
    k_net(const __grid_constant__ Net net, const float *__restrict__ x,
          const float *__restrict__ target, int batch, float *__restrict__ y,
          int ld, float inv_count) {
    constexpr int BM = 16 * MT;
    constexpr int PF = MT == 1 ? 8 : MT == 2 ? 4 : 3;
    constexpr int NT = 32 * net_warps(MT), TW = 32 / net_warps(MT);
    extern __shared__ __align__(16) __nv_bfloat16 sm[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t4 = lane & 3;
    const int L = net.L;
    // row of hs for row m = m0 + r of the batch: the block's own rows.  (Tiles
    // of 16 rows never outnumber the blocks, see pick_mt: there these are the
    // batch's rows, and indexing by m keeps 0.3 us of a training step's 32.)
    auto hrow = [&](int r, int m) -> long {
        return MT == 1 ? (long)m : (long)blockIdx.x * BM + r;
    };
    __nv_bfloat16 *cur = sm, *nxt = sm + BM * ld;
    if constexpr (!TRAIN) start_after_previous();
    double lsum = 0.0;
    Product<MT, PF> pr;
    float acc[MT][TW][4];

    for (int tile = blockIdx.x; tile * BM < batch; tile += gridDim.x) {
        const int m0 = tile * BM;
        const bool first = tile == (int)blockIdx.x;
        pr.start(net.wf + net.off_f[0], net.dim[0], net.dim[1], 0, warp, lane);
        {  // the inputs, rounded to BF16, zero beyond the batch and n_in
            const int n_in = net.dim[0], kp = pad32(n_in);
            for (int e = tid; e < BM * kp; e += NT) {
                const int r = e / kp, c = e - r * kp;
                const bool in = c < n_in && m0 + r < batch;
                const __nv_bfloat16 v =
                    __float2bfloat16_rn(in ? x[(long)(m0 + r) * n_in + c] : 0.f);
                cur[r * ld + c] = v;
                if (TRAIN && m0 + r < batch) net.act[0][(long)(m0 + r) * kp + c] = v;
            }
        }
        __syncthreads();
        // ---- forward ------------------------------------------------------
        for (int l = 0; l <= L; ++l) {
            const int N = net.dim[l + 1], np32 = pad32(N);
            const int passes = (np32 + 255) / 256;
            const float *bias = net.w + net.off_b[l];
            for (int ps = 0; ps < passes; ++ps) {
                pr.run(cur, ld, lane, acc);
                const int n0 = pr.n0, cnt = pr.cnt;
                if (ps + 1 < passes)
                    pr.start(net.wf + net.off_f[l], net.dim[l], N, ps + 1, warp, lane);
                else if (l < L)
                    pr.start(net.wf + net.off_f[l + 1], N, net.dim[l + 2], 0, warp, lane);
                else if (TRAIN && L > 0)
                    pr.start(net.wt + net.off_t[L], N, net.dim[L], 0, warp, lane);
#pragma unroll
                for (int j = 0; j < TW; ++j) {
                    if (j >= cnt) break;
                    const int n = n0 + 8 * j + 2 * t4;
                    const float b0 = n < N ? bias[n] : 0.f;
                    const float b1 = n + 1 < N ? bias[n + 1] : 0.f;
                    float d0 = 0.f, d1 = 0.f;  // column sums of the gradient
#pragma unroll
                    for (int mi = 0; mi < MT; ++mi)
#pragma unroll
                        for (int hf = 0; hf < 2; ++hf) {
                            const int r = mi * 16 + hf * 8 + g, m = m0 + r;
                            float v0 = acc[mi][j][2 * hf] + b0;
                            float v1 = acc[mi][j][2 * hf + 1] + b1;
                            if (l < L) {
                                v0 = n < N ? tanhf(v0) : 0.f;
                                v1 = n < N ? tanhf(v1) : 0.f;  // N is even here
                                st_bf2(nxt + r * ld + n, v0, v1);
                                if (TRAIN && m < batch) {
                                    st_bf2(net.act[l + 1] + (long)m * np32 + n, v0, v1);
                                    if (n < N)
                                        *reinterpret_cast<float2 *>(net.hs[l] + hrow(r, m) * N + n) =
                                            make_float2(v0, v1);
                                }
                            } else if (!TRAIN) {
                                if (m < batch && n < N) y[(long)m * N + n] = v0;
                                if (m < batch && n + 1 < N) y[(long)m * N + n + 1] = v1;
                            } else {
                                // d loss / d y = 2 (y - t) / (rows * outputs), 0
                                // where the target is unknown (NaN)
                                float e0 = 0.f, e1 = 0.f;
                                if (m < batch && n < N) {
                                    const float tv = target[(long)m * N + n];
                                    if (!isnan(tv)) e0 = v0 - tv;
                                }
                                if (m < batch && n + 1 < N) {
                                    const float tv = target[(long)m * N + n + 1];
                                    if (!isnan(tv)) e1 = v1 - tv;
                                }
                                lsum += (double)e0 * e0 + (double)e1 * e1;
                                e0 = 2.0f * e0 * inv_count;
                                e1 = 2.0f * e1 * inv_count;
                                d0 += e0;
                                d1 += e1;
                                st_bf2(nxt + r * ld + n, e0, e1);
                                if (m < batch) st_bf2(net.dz[L] + (long)m * np32 + n, e0, e1);
                            }
                        }
                    if (TRAIN && l == L) {
#pragma unroll
                        for (int o = 4; o < 32; o <<= 1) {
                            d0 += __shfl_xor_sync(0xffffffffu, d0, o);
                            d1 += __shfl_xor_sync(0xffffffffu, d1, o);
                        }
                        if (g == 0) {
                            float *q = net.db + (long)blockIdx.x * net.ndb + net.off_db[l] + n;
                            if (n < N) q[0] = first ? d0 : q[0] + d0;
                            if (n + 1 < N) q[1] = first ? d1 : q[1] + d1;
                        }
                    }
                }
            }
            __syncthreads();
            __nv_bfloat16 *sw = cur;
            cur = nxt;
            nxt = sw;
        }
        if constexpr (TRAIN) {
            // ---- back: the gradient at layer l - 1's pre-activation is
            // (dz_l W_l) (1 - h^2); a thread meets the h that it wrote
            for (int l = L; l >= 1; --l) {
                const int N = net.dim[l], np32 = pad32(N);
                const int passes = (np32 + 255) / 256;
                const float *hp = net.hs[l - 1];
                for (int ps = 0; ps < passes; ++ps) {
                    pr.run(cur, ld, lane, acc);
                    const int n0 = pr.n0, cnt = pr.cnt;
                    if (ps + 1 < passes)
                        pr.start(net.wt + net.off_t[l], net.dim[l + 1], N, ps + 1, warp, lane);
                    else if (l > 1)
                        pr.start(net.wt + net.off_t[l - 1], N, net.dim[l - 1], 0, warp, lane);
#pragma unroll
                    for (int j = 0; j < TW; ++j) {
                        if (j >= cnt) break;
                        const int n = n0 + 8 * j + 2 * t4;
                        float d0 = 0.f, d1 = 0.f;
#pragma unroll
                        for (int mi = 0; mi < MT; ++mi)
#pragma unroll
                            for (int hf = 0; hf < 2; ++hf) {
                                const int r = mi * 16 + hf * 8 + g, m = m0 + r;
                                float v0 = 0.f, v1 = 0.f;
                                if (m < batch && n < N) {
                                    const float2 h = *reinterpret_cast<const float2 *>(
                                        hp + hrow(r, m) * N + n);
                                    v0 = acc[mi][j][2 * hf] * (1.0f - h.x * h.x);
                                    v1 = acc[mi][j][2 * hf + 1] * (1.0f - h.y * h.y);
                                }
                                d0 += v0;
                                d1 += v1;
                                st_bf2(nxt + r * ld + n, v0, v1);
                                if (m < batch)
                                    st_bf2(net.dz[l - 1] + (long)m * np32 + n, v0, v1);
                            }
#pragma unroll
                        for (int o = 4; o < 32; o <<= 1) {
                            d0 += __shfl_xor_sync(0xffffffffu, d0, o);
                            d1 += __shfl_xor_sync(0xffffffffu, d1, o);
                        }
                        if (g == 0 && n < N) {
                            float *q = net.db + (long)blockIdx.x * net.ndb + net.off_db[l - 1] + n;
                            q[0] = first ? d0 : q[0] + d0;
                            q[1] = first ? d1 : q[1] + d1;
                        }
                    }
                }
                __syncthreads();
                __nv_bfloat16 *sw = cur;
                cur = nxt;
                nxt = sw;
            }
        }
    }
    if constexpr (TRAIN) {
        __shared__ double sl[net_warps(MT)];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        if (lane == 0) sl[warp] = lsum;
        __syncthreads();
        if (tid == 0) {
            double s = 0.0;
            for (int v = 0; v < net_warps(MT); ++v) s += sl[v];
            net.loss[blockIdx.x] = s;
        }
    }
}

__device__ __forceinline__ void cp16(void *dst, const void *src, bool in) {
    const int n = in ? 16 : 0;  // 0: the 16 bytes are zeroed
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(n));
}

// Weight gradients of every layer, dW_l[n][k] = sum over the batch of
// dz_l[b][n] act_l[b][k]: block x takes a DT x DT tile of one layer, block y
// `rows` rows of the batch (a multiple of DR), and writes its part to
// parts[y].  Both operands lie batch-major; ldmatrix transposes them.  FOLD:
// every `chain` rows (a multiple of DR) the sums so far are added to a second
// set and start anew, for networks with so many tiles that the batch has fewer
// than kParts parts: the tensor core truncates its running sum at each step,
// and over 65536 rows of two layers of 1024 units one chain left errors of
// 4.3e-4 of the gradient, eight 4.4e-5, sixteen 1.8e-5 (ten parts, as 256 units
// have, 2.8e-5); a training step there 2896 and 2905 us.  About
// 450 blocks, each waiting for its operands from L2: 8.7 us for 1024 rows of
// the 5-256-256-256-65 network, where the layers' products and column sums
// took 36 and 59 us each.
template <bool FOLD>
__global__ void __launch_bounds__(kDwThreads)
    k_dweight(const __grid_constant__ Net net, int batch, int rows, int chain) {
    __shared__ __align__(16) __nv_bfloat16 sa[2][DR][DLD], sb[2][DR][DLD];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = warp >> 1, wn = warp & 1;
    int l = 0, t = blockIdx.x, kx = 0;
    for (;; ++l) {
        kx = (net.dim[l] + DT - 1) / DT;
        const int n = kx * ((net.dim[l + 1] + DT - 1) / DT);
        if (t < n) break;
        t -= n;
    }
    const int N = net.dim[l + 1], K = net.dim[l], lda = pad32(N), ldb = pad32(K);
    const int n0 = t / kx * DT, k0 = t % kx * DT;
    const int b0 = blockIdx.y * rows, b1 = min(batch, b0 + rows);
    const __nv_bfloat16 *A = net.dz[l], *B = net.act[l];
    float acc[2][4][4] = {};
    float sum[2][4][4] = {};
    int next = b0 + chain;  // row at which the sums are folded
    auto fold = [&] {
#pragma unroll
        for (int mi = 0; mi < 2; ++mi)
#pragma unroll
            for (int ni = 0; ni < 4; ++ni)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    sum[mi][ni][q] += acc[mi][ni][q];
                    acc[mi][ni][q] = 0.f;
                }
    };
    auto stage = [&](int s, int r0) {
#pragma unroll
        for (int j = 0; j < DR * DT / 8 / kDwThreads; ++j) {
            const int e = tid + j * kDwThreads, r = e >> 3, c = (e & 7) * 8;
            const bool row = r0 + r < b1;
            const bool ia = row && n0 + c < lda, ib = row && k0 + c < ldb;
            cp16(&sa[s][r][c], ia ? A + (long)(r0 + r) * lda + n0 + c : A, ia);
            cp16(&sb[s][r][c], ib ? B + (long)(r0 + r) * ldb + k0 + c : B, ib);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    stage(0, b0);
    for (int r0 = b0, s = 0; r0 < b1; r0 += DR, s ^= 1) {
        if (r0 + DR < b1) {
            stage(s ^ 1, r0 + DR);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < DR; kk += 16) {
            unsigned af[2][4], bf[2][4];
            const int mr = (lane & 7) + (lane >> 4) * 8, mc = ((lane >> 3) & 1) * 8;
            const int br = (lane & 7) + ((lane >> 3) & 1) * 8, bc = (lane >> 4) * 8;
#pragma unroll
            for (int mi = 0; mi < 2; ++mi)
                ldsm4t(af[mi], &sa[s][kk + mr][wm * 32 + mi * 16 + mc]);
#pragma unroll
            for (int nj = 0; nj < 2; ++nj)
                ldsm4t(bf[nj], &sb[s][kk + br][wn * 32 + nj * 16 + bc]);
#pragma unroll
            for (int mi = 0; mi < 2; ++mi)
#pragma unroll
                for (int ni = 0; ni < 4; ++ni)
                    mma_bf16(acc[mi][ni], af[mi], bf[ni >> 1][(ni & 1) * 2],
                             bf[ni >> 1][(ni & 1) * 2 + 1]);
        }
        if constexpr (FOLD) {
            if (r0 + DR >= next) {
                fold();
                next += chain;
            }
        }
        __syncthreads();
    }
    if constexpr (FOLD) fold();
    float *c = net.parts + blockIdx.y * net.np + net.off_w[l];
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int ni = 0; ni < 4; ++ni)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int n = n0 + wm * 32 + mi * 16 + (lane >> 2) + (q >> 1) * 8;
                const int k = k0 + wn * 32 + ni * 8 + 2 * (lane & 3) + (q & 1);
                if (n < N && k < K)
                    c[(long)n * K + k] = FOLD ? sum[mi][ni][q] : acc[mi][ni][q];
            }
}

// Layer of parameter i, and whether it is a weight (else a bias).
__device__ __forceinline__ int layer_of(const Net &net, long i, bool &weight) {
    int l = net.L;
    while (l > 0 && i < net.off_w[l]) --l;
    weight = i < net.off_b[l];
    return l;
}
// The BF16 copies of weight i of layer l.
__device__ __forceinline__ void put_weight(const Net &net, int l, long i, float v) {
    const int K = net.dim[l], N = net.dim[l + 1];
    const int e = (int)(i - net.off_w[l]), j = e / K, k = e - j * K;
    const __nv_bfloat16 b = __float2bfloat16_rn(v);
    net.wf[net.off_f[l] + frag_at(j, k, K)] = b;
    if (l > 0) net.wt[net.off_t[l] + frag_at(k, j, N)] = b;
}

// Adam with bias correction on parameter i, and the refreshed BF16 copies.
struct AdamArgs {
    float *m1, *m2;
    float lr, c1, c2;
};
__device__ __forceinline__ float adam(const Net &net, const AdamArgs &o, long i, float gv) {
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float a = b1 * o.m1[i] + (1.0f - b1) * gv;
    const float v = b2 * o.m2[i] + (1.0f - b2) * gv * gv;
    o.m1[i] = a;
    o.m2[i] = v;
    const float wv = net.w[i] - o.lr * (a * o.c1) / (sqrtf(v * o.c2) + eps);
    net.w[i] = wv;
    return wv;
}

// After the parts: sums them, in order, into the gradient (grad, when not
// null) and, with ADAM, updates the parameters.  Blocks x < nwb take 256
// parameters each and do the weights among them; the others take 32 bias
// entries each, 8 threads sharing the k_net blocks' shares of an entry; the
// last of them also adds up the loss.  Latency of the parts' loads: 7.8 us
// for 149,000 parameters in 8 parts.
template <bool ADAM>
__global__ void __launch_bounds__(256)
    k_finish(const __grid_constant__ Net net, int split, int nblk, int nwb,
             float *__restrict__ grad, AdamArgs o, float inv_count,
             double *__restrict__ loss) {
    const int tid = threadIdx.x;
    if ((int)blockIdx.x < nwb) {
        const long i = blockIdx.x * 256L + tid;
        if (i >= net.np) return;
        bool weight;
        const int l = layer_of(net, i, weight);
        if (!weight) return;
        float v = 0.f;
#pragma unroll 8
        for (int z = 0; z < split; ++z) v += net.parts[z * net.np + i];
        if (grad) grad[i] = v;
        if (ADAM) put_weight(net, l, i, adam(net, o, i, v));
        return;
    }
    __shared__ float sv[8][32];
    __shared__ double sd[256];
    const int c = (blockIdx.x - nwb) * 32 + (tid & 31), z0 = tid >> 5;
    float v = 0.f;
    if (c < net.ndb) {
#pragma unroll 8
        for (int z = z0; z < nblk; z += 8) v += net.db[(long)z * net.ndb + c];
    }
    sv[z0][tid & 31] = v;
    __syncthreads();
    if (z0 == 0 && c < net.ndb) {
        v = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) v += sv[k][tid];
        int l = 0;
        while (l < net.L && c >= net.off_db[l + 1]) ++l;
        const long i = net.off_b[l] + (c - net.off_db[l]);
        if (grad) grad[i] = v;
        if (ADAM) adam(net, o, i, v);
    }
    if (blockIdx.x == gridDim.x - 1) {
        double s = 0.0;
        for (int z = tid; z < nblk; z += 256) s += net.loss[z];
        sd[tid] = s;
        __syncthreads();
        for (int w = 128; w > 0; w >>= 1) {
            if (tid < w) sd[tid] += sd[tid + w];
            __syncthreads();
        }
        if (tid == 0) *loss = sd[0] * inv_count;
    }
}

// The BF16 copies of every weight.
__global__ void k_pack(const __grid_constant__ Net net) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < net.np;
         i += (long)gridDim.x * blockDim.x) {
        bool weight;
        const int l = layer_of(net, i, weight);
        if (weight) put_weight(net, l, i, net.w[i]);
    }
}

}  // namespace lbmmlp

using namespace lbmmlp;

struct lbm_mlp {
    lbm_mlp_shape sh{};
    Net net{};
    void *arena = nullptr;  // every device buffer
    float *m1 = nullptr, *m2 = nullptr;
    double *d_loss = nullptr;
    int tiles = 0;       // k_dweight tiles of all layers
    int max_split = 1;   // parts of the weight gradients
    cudaStream_t own = nullptr, stream = nullptr;
    cudaEvent_t moved = nullptr;  // end of the work queued before a change of stream
    bool queued = false;          // the stream holds work that no call waited for
    long adam_t = 0;
    std::string err;
    bool dead = false;
};

namespace {
std::string g_create_err;

lbm_status fail(lbm_mlp *h, lbm_status st, const std::string &msg) {
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

#define MCK(h, call)                                                         \
    do {                                                                     \
        cudaError_t e_ = (call);                                             \
        if (e_ != cudaSuccess)                                               \
            return fail(h, LBM_ECUDA, std::string(#call) + ": " +            \
                                          cudaGetErrorString(e_));           \
    } while (0)

constexpr int kSmemMax = 232448 - 1024;

// Row length of a block's activations in shared memory: 8 values beyond the
// widest layer, so that the 8 rows an ldmatrix reads lie in different banks.
int row_len(const lbm_mlp *h) {
    int d = 0;
    for (int l = 0; l <= h->net.L + 1; ++l) d = std::max(d, pad32(h->net.dim[l]));
    return d + 8;
}
size_t net_smem(const lbm_mlp *h, int mt) {
    return (size_t)2 * 16 * mt * row_len(h) * sizeof(__nv_bfloat16);
}

// 16-row units per block.  Small blocks cut the latency of a pass, which every
// block pays in full (one block: 8.8 us forward with 16 rows, 14.4 with 32,
// 20.7 with 64), until the blocks no longer run at once: 16 rows while each SM
// has one block, 32 while it has one (training) or two (inference, which fits
// two at 128 registers: 8192 rows 19.1 us with 32, 21.5 with 64, 35.3 with
// 16; a training step on 8192 rows 97.6 with 32, 88.6 with 64).
int pick_mt(const lbm_mlp *h, int batch, bool train) {
    const int sms = 152;
    int mt = batch <= 16 * sms ? 1 : batch <= 32 * sms * (train ? 1 : 2) ? 2 : 4;
    while (mt > 1 && net_smem(h, mt) > (size_t)kSmemMax) mt >>= 1;
    return mt;
}

template <bool TRAIN>
cudaError_t launch_net(lbm_mlp *h, const float *x, const float *target, int batch,
                       float *y, float inv_count, int *blocks) {
    h->queued = true;
    const int mt = pick_mt(h, batch, TRAIN);
    const int grid = std::min((batch + 16 * mt - 1) / (16 * mt), kMaxBlocks);
    const size_t sm = net_smem(h, mt);
    *blocks = grid;
    const int ld = row_len(h);
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.dynamicSmemBytes = sm;
    c.stream = h->stream;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = TRAIN ? 0 : 1;  // start_after_previous
    auto go = [&](auto *k, int warps) {
        c.blockDim = dim3(32 * warps);
        return cudaLaunchKernelEx(&c, k, h->net, x, target, batch, y, ld, inv_count);
    };
    return mt == 1   ? go(k_net<1, TRAIN>, net_warps(1))
           : mt == 2 ? go(k_net<2, TRAIN>, net_warps(2))
                     : go(k_net<4, TRAIN>, net_warps(4));
}

// Gradient of the loss into grad (when not null); adam: also the update.
cudaError_t train(lbm_mlp *h, const float *x, const float *target, int batch,
                  float *grad, const AdamArgs *adam) {
    const float inv = 1.0f / (float)((long)batch * h->sh.n_out);
    int blocks = 0;
    cudaError_t e = launch_net<true>(h, x, target, batch, nullptr, inv, &blocks);
    if (e != cudaSuccess) return e;
    // parts of equal, whole stages of rows
    const int stages = (batch + DR - 1) / DR;
    const int per = (stages + h->max_split - 1) / h->max_split;
    const int split = (stages + per - 1) / per;
    const int chain = (stages + kChains - 1) / kChains;
    const dim3 dw(h->tiles, split);
    if (h->max_split < kParts && per > chain)
        k_dweight<true><<<dw, kDwThreads, 0, h->stream>>>(h->net, batch, per * DR, chain * DR);
    else
        k_dweight<false><<<dw, kDwThreads, 0, h->stream>>>(h->net, batch, per * DR, 0);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int nwb = (int)((h->net.np + 255) / 256), nbb = (h->net.ndb + 31) / 32;
    if (adam)
        k_finish<true><<<nwb + nbb, 256, 0, h->stream>>>(h->net, split, blocks, nwb, grad,
                                                         *adam, inv, h->d_loss);
    else
        k_finish<false><<<nwb + nbb, 256, 0, h->stream>>>(h->net, split, blocks, nwb, grad,
                                                          AdamArgs{}, inv, h->d_loss);
    return cudaGetLastError();
}

lbm_status check_batch(lbm_mlp *h, int batch) {
    if (!h) return LBM_EINVAL;
    if (h->dead) return LBM_ECUDA;
    if (batch < 1 || batch > h->sh.max_batch)
        return fail(h, LBM_EINVAL, "batch outside 1..max_batch");
    return LBM_OK;
}

bool capturing(cudaStream_t s) {
    cudaStreamCaptureStatus c = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &c) != cudaSuccess) {  // (the legacy stream during a capture)
        cudaGetLastError();
        return true;
    }
    return c != cudaStreamCaptureStatusNone;
}

lbm_status read_loss(lbm_mlp *h, double *loss) {
    if (!loss) return LBM_OK;
    MCK(h, cudaMemcpyAsync(loss, h->d_loss, sizeof(double),
                           cudaMemcpyDeviceToHost, h->stream));
    MCK(h, cudaStreamSynchronize(h->stream));
    h->queued = false;
    return LBM_OK;
}
}  // namespace

extern "C" {

lbm_status lbm_mlp_create(const lbm_mlp_shape *shape, lbm_mlp **out) {
    if (!shape || !out) return fail(nullptr, LBM_EINVAL, "NULL argument");
    *out = nullptr;
    const lbm_mlp_shape s = *shape;
    if (s.n_in < 1 || s.n_in > 256 || s.n_hidden < 16 || s.n_hidden > 1024 ||
        s.n_hidden % 16 != 0 || s.n_layers < 1 || s.n_layers > 8 ||
        s.n_out < 1 || s.n_out > 1024 || s.max_batch < 1 ||
        s.max_batch > (1 << 24))
        return fail(nullptr, LBM_EINVAL, "shape outside the supported ranges");
    lbm_mlp *h = new (std::nothrow) lbm_mlp();
    if (!h) return fail(nullptr, LBM_ENOMEM, "host allocation");
    h->sh = s;
    Net &net = h->net;
    net.L = s.n_layers;
    net.dim[0] = s.n_in;
    for (int l = 1; l <= s.n_layers; ++l) net.dim[l] = s.n_hidden;
    net.dim[s.n_layers + 1] = s.n_out;
    long np = 0, nf = 0, nt = 0;
    for (int l = 0; l <= s.n_layers; ++l) {
        const int K = net.dim[l], N = net.dim[l + 1];
        net.off_w[l] = np;
        np += (long)N * K;
        net.off_b[l] = np;
        np += N;
        net.off_f[l] = nf;
        nf += (long)pad32(N) * pad32(K);
        net.off_t[l] = nt;
        if (l > 0) nt += (long)pad32(N) * pad32(K);
        net.off_db[l] = net.ndb;
        net.ndb += N;
        h->tiles += ((N + DT - 1) / DT) * ((K + DT - 1) / DT);
    }
    net.np = np;
    // parts of a weight gradient: about three blocks per SM
    h->max_split = std::min(std::max(456 / h->tiles, 1), 16);
    // one allocation: each buffer's place in it, then the buffers
    struct Item { void **p; size_t at; };
    std::vector<Item> items;
    size_t bytes = 0;
    auto al = [&](auto **p, size_t n) {
        items.push_back({(void **)p, bytes});
        bytes += (std::max<size_t>(n, 1) * sizeof(**p) + 255) / 256 * 256;
    };
    al(&net.w, np);
    al(&h->m1, np);
    al(&h->m2, np);
    al(&net.wf, nf);
    al(&net.wt, nt);
    const size_t zeroed = bytes;
    for (int l = 0; l <= s.n_layers; ++l) {
        // (the blocks' rows, 64 each at most: a block is done with a tile's
        // hidden activations before it goes on to its next tile)
        if (l < s.n_layers)
            al(&net.hs[l], std::min((size_t)s.max_batch, (size_t)kMaxBlocks * 64) * s.n_hidden);
        al(&net.act[l], (size_t)s.max_batch * pad32(net.dim[l]));
        al(&net.dz[l], (size_t)s.max_batch * pad32(net.dim[l + 1]));
    }
    const size_t blocks = std::min(((size_t)s.max_batch + 15) / 16, (size_t)kMaxBlocks);
    al(&net.db, blocks * net.ndb);
    al(&net.loss, blocks);
    al(&net.parts, (size_t)h->max_split * np);
    al(&h->d_loss, 1);
    bool ok = cudaMalloc(&h->arena, bytes) == cudaSuccess;
    if (ok)
        for (const Item &i : items) *i.p = (char *)h->arena + i.at;
    if (ok && (cudaStreamCreateWithFlags(&h->own, cudaStreamNonBlocking) != cudaSuccess ||
               cudaEventCreateWithFlags(&h->moved, cudaEventDisableTiming) != cudaSuccess))
        ok = false;
    h->stream = h->own;
    if (ok) {
        // (on the handle's stream, which the default stream's queue does not
        // order, and waited for: the next call may come on any stream)
        ok = cudaMemsetAsync(h->arena, 0, zeroed, h->own) == cudaSuccess &&
             cudaStreamSynchronize(h->own) == cudaSuccess;
        const int a = (int)cudaFuncAttributeMaxDynamicSharedMemorySize;
        for (const void *f : {(const void *)k_net<1, false>, (const void *)k_net<1, true>,
                              (const void *)k_net<2, false>, (const void *)k_net<2, true>,
                              (const void *)k_net<4, false>, (const void *)k_net<4, true>})
            ok = ok && cudaFuncSetAttribute(f, (cudaFuncAttribute)a, kSmemMax) == cudaSuccess;
    }
    if (!ok) {
        lbm_mlp_destroy(h);
        return fail(nullptr, LBM_ENOMEM, "device allocation");
    }
    *out = h;
    return LBM_OK;
}

int64_t lbm_mlp_param_count(const lbm_mlp *h) { return h ? h->net.np : -1; }

lbm_status lbm_mlp_set_params(lbm_mlp *h, const float *host, int64_t n) {
    if (!h || !host) return LBM_EINVAL;
    if (h->dead) return LBM_ECUDA;
    if (n != h->net.np) return fail(h, LBM_EINVAL, "parameter count mismatch");
    MCK(h, cudaMemcpyAsync(h->net.w, host, n * sizeof(float), cudaMemcpyHostToDevice,
                           h->stream));
    MCK(h, cudaMemsetAsync(h->m1, 0, n * sizeof(float), h->stream));
    MCK(h, cudaMemsetAsync(h->m2, 0, n * sizeof(float), h->stream));
    k_pack<<<(int)std::min<long>((n + 255) / 256, 4096), 256, 0, h->stream>>>(h->net);
    MCK(h, cudaGetLastError());
    // the host array may be reused as soon as this returns
    MCK(h, cudaStreamSynchronize(h->stream));
    h->queued = false;
    h->adam_t = 0;
    return LBM_OK;
}

lbm_status lbm_mlp_get_params(lbm_mlp *h, float *host, int64_t n) {
    if (!h || !host) return LBM_EINVAL;
    if (h->dead) return LBM_ECUDA;
    if (n != h->net.np) return fail(h, LBM_EINVAL, "parameter count mismatch");
    MCK(h, cudaMemcpyAsync(host, h->net.w, n * sizeof(float), cudaMemcpyDeviceToHost,
                           h->stream));
    MCK(h, cudaStreamSynchronize(h->stream));
    h->queued = false;
    return LBM_OK;
}

lbm_status lbm_mlp_set_stream(lbm_mlp *h, void *cuda_stream) {
    if (!h) return LBM_EINVAL;
    const cudaStream_t to = cuda_stream ? static_cast<cudaStream_t>(cuda_stream) : h->own;
    if (to == h->stream) return LBM_OK;
    // weights, moments and activations are shared by all calls: what the next
    // ones queue on the new stream waits for what is queued on the old one.
    // (A stream that is being captured can neither wait for work outside the
    // capture nor be waited for from outside: there the caller orders the
    // replays, as with any captured work.)
    if (h->queued && !h->dead && !capturing(h->stream) && !capturing(to)) {
        MCK(h, cudaEventRecord(h->moved, h->stream));
        MCK(h, cudaStreamWaitEvent(to, h->moved, 0));
    }
    h->stream = to;
    return LBM_OK;
}

lbm_status lbm_mlp_forward(lbm_mlp *h, const float *x, int32_t batch, float *y) {
    lbm_status st = check_batch(h, batch);
    if (st != LBM_OK) return st;
    if (!x || !y) return fail(h, LBM_EINVAL, "NULL argument");
    int blocks = 0;
    MCK(h, launch_net<false>(h, x, nullptr, batch, y, 0.f, &blocks));
    return LBM_OK;
}

lbm_status lbm_mlp_grad(lbm_mlp *h, const float *x, const float *target,
                        int32_t batch, float *grad, double *loss) {
    lbm_status st = check_batch(h, batch);
    if (st != LBM_OK) return st;
    if (!x || !target || !grad) return fail(h, LBM_EINVAL, "NULL argument");
    MCK(h, train(h, x, target, batch, grad, nullptr));
    return read_loss(h, loss);
}

lbm_status lbm_mlp_train_step(lbm_mlp *h, const float *x, const float *target,
                              int32_t batch, float lr, double *loss) {
    lbm_status st = check_batch(h, batch);
    if (st != LBM_OK) return st;
    if (!x || !target) return fail(h, LBM_EINVAL, "NULL argument");
    if (!(lr > 0.f)) return fail(h, LBM_EINVAL, "learning rate must be > 0");
    ++h->adam_t;
    const AdamArgs o{h->m1, h->m2, lr,
                     (float)(1.0 / (1.0 - std::pow(0.9, (double)h->adam_t))),
                     (float)(1.0 / (1.0 - std::pow(0.999, (double)h->adam_t)))};
    MCK(h, train(h, x, target, batch, nullptr, &o));
    return read_loss(h, loss);
}

void lbm_mlp_destroy(lbm_mlp *h) {
    if (!h) return;
    if (h->stream) cudaStreamSynchronize(h->stream);
    if (h->arena) cudaFree(h->arena);
    if (h->moved) cudaEventDestroy(h->moved);
    if (h->own) cudaStreamDestroy(h->own);
    delete h;
}

const char *lbm_mlp_last_error(const lbm_mlp *h) {
    return h ? h->err.c_str() : g_create_err.c_str();
}

}  // extern "C"
