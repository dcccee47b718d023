// surrogate.cu -- a small MLP that learns the NCI growth rate from the root
// solver's data (forward, backward and Adam written here; BF16 weights and
// activations as tensor-core operands, FP32 accumulation, FP32 master
// weights).  Architecture: n_in -> width x depth (tanh) -> 1 (linear).
//
// The GEMMs run on the fifth-generation tensor cores: tcgen05.mma (kind::f16,
// BF16 operands) into FP32 accumulators in tensor memory, 128 x 32 output tiles
// per CTA (narrow, so that the small products still give each SM a dozen warps), operands loaded into the canonical K-major shared-memory layout with
// 16-byte vector loads: every operand is stored with its K index contiguous
// (the epilogues write the activations and dH both batch-major and
// feature-major, and the weights are kept in BF16 both ways).  The network is
// small (widths 16..256), so this is not a roofline-bound path.  The
// elementwise work sits in the GEMM epilogues (bias and tanh; loss, output dH
// and its bias gradient; tanh' and the bias gradient of the layer below), and
// the Adam step sums the gradient parts and writes the BF16 weight copies: a
// training step is 3 launches per layer (forward, dW, dX; no dX below the first
// layer) plus the Adam step.  Networks wider than 64 run the forward and backward products of a tile
// of the batch in one kernel (k_mlp_chain) and all weight gradients in another: 3 launches a step.  No sum is taken with atomics: the weight
// gradients (K = batch, split over up to 64 CTAs per tile), the bias gradients
// and the loss are written as per-CTA parts and added in a fixed order, so a
// training run is bit-reproducible.
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "hyb_internal.cuh"
#include "tm_dev.cuh"

namespace hyb {
// per-layer offsets and sizes for the gradient sums and the Adam step (passed by value)
constexpr int kMaxLayers = 17;
struct LayerTab {
    int L;
    int nrb;                                          // row blocks of the batch (parts of a bias gradient)
    int nrc;                                          // 64-row blocks of the batch (k_mlp_chain: the halves of nrb's)
    int64_t wk_off[kMaxLayers];                       // k_mlp_chain: BF16 weights of a layer, rows of its tile
    int rows[kMaxLayers];
    int64_t w_off[kMaxLayers], wb_off[kMaxLayers];    // parameters; BF16 weight copies
    int64_t ws_w[kMaxLayers], ws_b[kMaxLayers];       // parts of the weight and bias gradients
    int fo[kMaxLayers], fi[kMaxLayers], fop[kMaxLayers], fip[kMaxLayers], split[kMaxLayers];
};
}  // namespace hyb

struct hyb_mlp {
    int n_in = 0, width = 0, depth = 0;   // hidden layers of `width`
    int L = 0;                            // layers = depth + 1
    hyb::LayerTab tab{};
    float* master = nullptr;              // FP32 weights and biases, all layers
    float* adam_m = nullptr;
    float* adam_v = nullptr;
    __nv_bfloat16* wbf = nullptr;         // BF16 weights [fout_pad][fin_pad] per layer
    __nv_bfloat16* wbt = nullptr;         // BF16 weights transposed [fin_pad][fout_pad] per layer
    float* grad = nullptr;                // FP32 gradients (same layout as master)
    std::vector<size_t> w_off, b_off, wb_off;
    size_t n_params = 0;
    int64_t cap = 0;                      // batch capacity of the activations
    __nv_bfloat16* act = nullptr;         // [L-1][cap][256] BF16 inputs X_l of layers l >= 1
    __nv_bfloat16* actT = nullptr;        // [L-1][256][cap] the same, feature-major
    float* pre = nullptr;                 // [L-1][cap][256] FP32 pre-activations of the hidden layers
    __nv_bfloat16* dhb = nullptr;         // [2][cap][256] BF16 dH (two layers' worth)
    __nv_bfloat16* dhT = nullptr;         // [2][256][cap] the same, feature-major
    float* ws = nullptr;                  // gradient parts: weights (split x fo x fi per layer), biases, loss
    size_t ws_w_size = 0;
    float* loss = nullptr;                // device scalar
    int* err = nullptr;                   // device flag: bit 1 = a bounded wait in a GEMM gave up
    // networks wider than kNarrow (k_mlp_chain): BF16 weights in the order the kernel's shared memory
    // holds them; every layer's input (actT) and dH (dhT) in the order of k_dw_tiles, tanh of the hidden layers (pre)
    bool chain = false;
    __nv_bfloat16* wk = nullptr;          // [fin/8][rows][8] per layer (rows: outputs, padded)
    __nv_bfloat16* wkt = nullptr;         // [fout/8][rows][8] of the transposed weights (rows: inputs, padded)
    int64_t step = 0;
    int64_t launches = 0;                 // kernels launched so far (hyb_mlp_launch_count)
};

namespace hyb {

// GEMM tiles: 128 x 32 outputs per CTA (tcgen05.mma M = 128, N = 32), K in chunks of 64
constexpr int TM = 128, TN = 32, TKC = 64, GT = 128;
constexpr int LBO_A = TM * 16 + 16, LBO_B = TN * 16 + 16;     // K-group strides (16-byte slots spread)
constexpr int kMaxSplit = 64;
// Networks up to this width run a product per launch (3 launches per layer, as hyb_mlp_launch_count states),
// wider ones k_mlp_chain
constexpr int kNarrow = 64;
constexpr int CB = 64, CT = 512;         // k_mlp_chain: rows of the batch per CTA, threads

// Epilogues of the GEMM (what happens to an accumulator value v of output (row, col)):
//   EP_PART    part z of a split K: P[z][row][col] = v (row stride N); a CTA with an empty K
//              range writes zeros
//   EP_HIDDEN  h = v + b[col]; pre[row][col] = h; X[row][col] = XT[col][row] = BF16(tanh h)
//              (0 for col >= n)
//   EP_OUTPUT  y = v + b[0] (column 0); out[row] = y; with a target t: d = 2 (y - t) / B,
//              dH[row] = (d, 0, ..., 0) and dHT[0][row] = d in BF16, and per CTA the parts
//              sum (y - t)^2 / B and sum d (loss and bias gradient) at index blockIdx.y
//   EP_DX      dH'[row][col] = dH'T[col][row] = BF16(v (1 - tanh(pre[row][col])^2)) for
//              col < n (else 0), and per CTA the column sums of dH' (bias gradient of the
//              layer below) at [blockIdx.y][col]
enum : int { EP_PART = 0, EP_HIDDEN, EP_OUTPUT, EP_DX };
struct Epi {
    float* c = nullptr;                  // EP_PART output
    const float* bias = nullptr;         // EP_HIDDEN, EP_OUTPUT
    float* pre = nullptr;                // EP_HIDDEN: written; EP_DX: read (pre-activations below)
    __nv_bfloat16* act = nullptr;        // EP_HIDDEN: X (row stride 256); EP_OUTPUT, EP_DX: dH
    __nv_bfloat16* actT = nullptr;       // the same, feature-major (row stride ldT)
    int64_t ldT = 0;
    float* out = nullptr;                // EP_OUTPUT: y (nullable)
    const float* tgt = nullptr;          // EP_OUTPUT: targets (nullable: forward only)
    float* loss_part = nullptr;          // EP_OUTPUT: [row blocks]
    float* db_part = nullptr;            // EP_OUTPUT: [row blocks]; EP_DX: [row blocks][n]
    int n = 0;                           // live columns
    float invB = 0.f;
};

__device__ __forceinline__ uint32_t bf16_bits(float x) { return (uint32_t)__bfloat16_as_ushort(__float2bfloat16(x)); }
__device__ __forceinline__ uint32_t bf16_bits(__nv_bfloat16 x) { return (uint32_t)__bfloat16_as_ushort(x); }

// 16-byte slots (row r, group g of 8 k values) of a ROWS x 64 tile: ROWS x 8 slots, ROWS * 8 / GT
// per thread.  All of a thread's global loads are issued before its shared-memory stores, so
// that their latencies overlap (a store between two loads would serialise them).  A source
// whose k index is contiguous is read 16 bytes at a time; the network input (FP32, 6 columns)
// is read element by element and rounded to BF16.
template <int ROWS, typename TA>
__device__ __forceinline__ void gemm_fill(uint32_t dst, int lbo, int rmax, int r0, int k0, int kmax,
                                          const TA* __restrict__ src, int64_t sr, int64_t sk, int tid) {
    constexpr int IT = ROWS * 8 / GT;
    constexpr bool kBF = sizeof(TA) == 2;
    const bool kfast = sk == 1 && (sr & 7) == 0;
    uint4 v[IT];
    uint32_t off[IT];
#pragma unroll
    for (int q = 0; q < IT; q++) {
        const int i = tid + q * GT;
        const int r = kfast ? i >> 3 : i % ROWS, g = kfast ? i & 7 : i / ROWS;
        const int row = r0 + r, k = k0 + 8 * g;
        off[q] = (uint32_t)(g * lbo + 16 * r);
        v[q] = make_uint4(0u, 0u, 0u, 0u);
        if (row < rmax) {
            if (kBF && kfast && k + 8 <= kmax) {
                v[q] = __ldg(reinterpret_cast<const uint4*>(src + (int64_t)row * sr + k));
            } else {
                uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int e = 0; e < 8; e++) {
                    const uint32_t x = (k + e < kmax) ? bf16_bits(__ldg(src + (int64_t)row * sr + (int64_t)(k + e) * sk)) : 0u;
                    w[e >> 1] |= x << (16 * (e & 1));
                }
                v[q] = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < IT; q++)
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                     :: "r"(dst + off[q]), "r"(v[q].x), "r"(v[q].y), "r"(v[q].z), "r"(v[q].w) : "memory");
}

// sum of v over the 32 lanes of a warp (the same butterfly order in every lane)
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// C[m][n] (FP32) = sum_k A(m,k) B(k,n), A(m,k) = a[m*sam + k*sak], B(k,n) = b[k*sbk + n*sbn]
// (BF16, or FP32 rounded to BF16 on the way in: the network input), K a multiple of 16,
// entries with k >= kmax read as zero.  Split K (EP_PART only): block z handles k in
// [z*kchunk, (z+1)*kchunk).
// Per 64-wide K chunk the 128 threads load the A and B tiles into shared memory in the
// canonical K-major layout without swizzle (8 x 16-byte core matrices; 16-byte slots (row, k/8)),
// one thread issues the k-steps of tcgen05.mma into the 128 x 32 FP32 accumulator in TMEM and
// commits them to an mbarrier, and after the last chunk each warp reads its 32 rows with
// tcgen05.ld into the epilogue.  Waits are bounded: on time-out bit 1 of *err is set and the
// CTA skips the rest, drains and frees its TMEM.
template <int EP, typename TA, typename TB>
__global__ void __launch_bounds__(GT) k_gemm_tc(int M, int N, int K, int kmax, const TA* __restrict__ a, int64_t sam, int64_t sak,
                                                const TB* __restrict__ b, int64_t sbk, int64_t sbn, Epi ep, int kchunk, int* err) {
    __shared__ __align__(128) unsigned char sbuf[8 * LBO_A + 8 * LBO_B];
    __shared__ uint64_t bar;
    __shared__ uint32_t s_taddr;
    __shared__ int s_abort;
    __shared__ float s_red[4][TN];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sA = smem_addr(sbuf), sB = sA + 8 * LBO_A, mb = smem_addr(&bar);
    if (warp == 0) {
        tm_alloc(smem_addr(&s_taddr), TN);
        tm_relinquish();
    }
    if (tid == 0) {
        mbar_init(mb, 1);
        mbar_fence_init();
        s_abort = 0;
    }
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    const uint32_t tbase = s_taddr;
    const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
    const int kb = blockIdx.z * kchunk, ke = min(K, kb + kchunk);
    uint32_t ph = 0;
    bool pend = false, abort = false, any = false;
    for (int k0 = kb; k0 < ke && !abort; k0 += TKC) {
        gemm_fill<TM, TA>(sA, LBO_A, M, m0, k0, kmax, a, sam, sak, tid);
        gemm_fill<TN, TB>(sB, LBO_B, N, n0, k0, kmax, b, sbn, sbk, tid);
        fence_proxy_async_smem();
        tm_fence_before();
        __syncthreads();
        if (tid == 0) {
            tm_fence_after();
            const int nks = min(TKC, ke - k0) / 16;
            for (int ks = 0; ks < nks; ks++)
                mma_bf16(tbase, smem_desc(sA + 2 * ks * LBO_A, LBO_A, 128), smem_desc(sB + 2 * ks * LBO_B, LBO_B, 128),
                         idesc_bf16(TN), (k0 > kb || ks > 0) ? 1u : 0u);
            mma_commit(mb);
            pend = true;
            mbar_wait(mb, ph, err, &s_abort);
            if (!s_abort) {
                ph ^= 1;
                pend = false;
            }
        }
        __syncthreads();
        abort = s_abort != 0;
        any = true;
    }
    if (!abort) {
        if (any) tm_fence_after();
        const int row = m0 + 32 * warp + lane;
        const bool live = row < M;
        const int nchunk = EP == EP_OUTPUT ? 1 : TN / 16;
        for (int u = 0; u < nchunk; u++) {
            float t[16];
            if (any) {
                tm_ld16(tbase + ((uint32_t)(32 * warp) << 16) + (uint32_t)(16 * u), t);
                tm_wait_ld();
            } else {
#pragma unroll
                for (int j = 0; j < 16; j++) t[j] = 0.f;
            }
            const int c0 = n0 + 16 * u;
            if (EP == EP_PART) {
                if (live && c0 < N) {
                    float* p = ep.c + (int64_t)blockIdx.z * M * N + (int64_t)row * N + c0;
                    if ((N & 3) == 0 && c0 + 16 <= N) {
#pragma unroll
                        for (int j = 0; j < 4; j++)
                            reinterpret_cast<float4*>(p)[j] = make_float4(t[4 * j], t[4 * j + 1], t[4 * j + 2], t[4 * j + 3]);
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; j++)
                            if (c0 + j < N) p[j] = t[j];
                    }
                }
            } else if (EP == EP_HIDDEN) {
                if (live && c0 < N) {
                    float h[16];
                    uint32_t q[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll
                    for (int j = 0; j < 16; j++) {
                        const int col = c0 + j;
                        h[j] = t[j] + (col < ep.n ? __ldg(ep.bias + col) : 0.f);
                        q[j >> 1] |= (col < ep.n ? bf16_bits(tanhf(h[j])) : 0u) << (16 * (j & 1));
                    }
                    float4* pp = reinterpret_cast<float4*>(ep.pre + (int64_t)row * 256 + c0);
#pragma unroll
                    for (int j = 0; j < 4; j++) pp[j] = make_float4(h[4 * j], h[4 * j + 1], h[4 * j + 2], h[4 * j + 3]);
                    uint4* pa = reinterpret_cast<uint4*>(ep.act + (int64_t)row * 256 + c0);
                    pa[0] = make_uint4(q[0], q[1], q[2], q[3]);
                    pa[1] = make_uint4(q[4], q[5], q[6], q[7]);
                    unsigned short* pt = reinterpret_cast<unsigned short*>(ep.actT) + (int64_t)c0 * ep.ldT + row;
#pragma unroll
                    for (int j = 0; j < 16; j++) pt[(int64_t)j * ep.ldT] = (unsigned short)(q[j >> 1] >> (16 * (j & 1)));
                }
            } else if (EP == EP_OUTPUT) {
                const float y = t[0] + __ldg(ep.bias);
                if (live && ep.out) ep.out[row] = y;
                if (ep.tgt) {
                    const float dd = live ? y - ep.tgt[row] : 0.f;
                    const float d = 2.f * dd * ep.invB;
                    if (live) {
                        const uint32_t db = bf16_bits(d);
                        uint4* pa = reinterpret_cast<uint4*>(ep.act + (int64_t)row * 256);
                        pa[0] = make_uint4(db, 0u, 0u, 0u);
                        pa[1] = make_uint4(0u, 0u, 0u, 0u);
                        reinterpret_cast<unsigned short*>(ep.actT)[row] = (unsigned short)db;
                    }
                    const float l = warp_sum(dd * dd * ep.invB), sd = warp_sum(d);
                    if (lane == 0) { s_red[warp][0] = l; s_red[warp][1] = sd; }
                    __syncthreads();
                    if (tid == 0) {
                        ep.loss_part[blockIdx.y] = (s_red[0][0] + s_red[1][0]) + (s_red[2][0] + s_red[3][0]);
                        ep.db_part[blockIdx.y] = (s_red[0][1] + s_red[1][1]) + (s_red[2][1] + s_red[3][1]);
                    }
                }
            } else {   // EP_DX
                if (c0 < N) {
                    float d[16];
                    uint32_t q[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
                    if (live) {
                        const float4* pp = reinterpret_cast<const float4*>(ep.pre + (int64_t)row * 256 + c0);
#pragma unroll
                        for (int j = 0; j < 4; j++) {
                            const float4 h = pp[j];
                            const float hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
                            for (int i = 0; i < 4; i++) {
                                const float th = tanhf(hv[i]);
                                d[4 * j + i] = (c0 + 4 * j + i < ep.n) ? t[4 * j + i] * (1.f - th * th) : 0.f;
                            }
                        }
#pragma unroll
                        for (int j = 0; j < 16; j++) q[j >> 1] |= bf16_bits(d[j]) << (16 * (j & 1));
                        uint4* pa = reinterpret_cast<uint4*>(ep.act + (int64_t)row * 256 + c0);
                        pa[0] = make_uint4(q[0], q[1], q[2], q[3]);
                        pa[1] = make_uint4(q[4], q[5], q[6], q[7]);
                        unsigned short* pt = reinterpret_cast<unsigned short*>(ep.actT) + (int64_t)c0 * ep.ldT + row;
#pragma unroll
                        for (int j = 0; j < 16; j++) pt[(int64_t)j * ep.ldT] = (unsigned short)(q[j >> 1] >> (16 * (j & 1)));
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; j++) d[j] = 0.f;
                    }
#pragma unroll
                    for (int j = 0; j < 16; j++) {
                        const float sj = warp_sum(d[j]);
                        if (lane == 0) s_red[warp][16 * u + j] = sj;
                    }
                }
            }
        }
        if (EP == EP_DX) {
            __syncthreads();
            if (tid < TN && n0 + tid < ep.n)
                ep.db_part[(int64_t)blockIdx.y * ep.n + n0 + tid] = (s_red[0][tid] + s_red[1][tid]) + (s_red[2][tid] + s_red[3][tid]);
        }
    }
    if (tid == 0 && pend) mbar_drain(mb, ph);
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    if (warp == 0) tm_dealloc(tbase, TN);
}

// K is rounded up to 16 (the MMA depth); entries with k >= K read as zero.
static int split_of(int M, int N, int K) {
    const int Kp = (K + 15) & ~15;
    const int tiles = ((N + TN - 1) / TN) * ((M + TM - 1) / TM);
    int split = 1;
    while (split < kMaxSplit && tiles * split < 600 && Kp / (split * 2) >= 256) split *= 2;
    return split;
}
// Few output tiles and a long K (the weight gradients: K = batch) are split along K into
// parts that the caller adds up (EP_PART).
template <int EP, typename TA, typename TB>
static void gemm(int M, int N, int K, const TA* a, int64_t sam, int64_t sak, const TB* b, int64_t sbk, int64_t sbn,
                 const Epi& ep, cudaStream_t s, int64_t& launches, int* err) {
    const int Kp = (K + 15) & ~15;
    const int split = EP == EP_PART ? split_of(M, N, K) : 1;
    const int kchunk = (((Kp + split - 1) / split + 15) & ~15);     // the parts cover all of K
    dim3 grid((N + TN - 1) / TN, (M + TM - 1) / TM, split);
    k_gemm_tc<EP, TA, TB><<<grid, GT, 0, s>>>(M, N, Kp, K, a, sam, sak, b, sbk, sbn, ep, kchunk, err);
    launches++;
}

// k_mlp_chain's order of a weight matrix: element (row, k) of [K/8][rows][8], the canonical K-major layout of a
// tcgen05 operand without swizzle, so that a layer is one contiguous copy
__host__ __device__ __forceinline__ int64_t chain_at(int row, int k, int rows) { return ((int64_t)(k >> 3) * rows + row) * 8 + (k & 7); }

// Gradient sums in a fixed order (the split-K parts of a weight gradient, the row-block parts of
// a bias gradient, the loss parts); with update != 0 also the Adam step on every parameter and
// the BF16 copies of the updated weights (zero-padded, both layouts; the padding was written by
// refresh()).  Without it the sums go to g (the gradients of hyb_mlp_gradients).
__global__ void k_grad_adam(float* __restrict__ w, float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                            const float* __restrict__ ws, const float* __restrict__ loss_part, float* __restrict__ loss,
                            int64_t n, int update, float lr, float b1, float b2, float eps, float c1, float c2, LayerTab tab,
                            __nv_bfloat16* __restrict__ wb, __nv_bfloat16* __restrict__ wt) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i == 0) {
        float s = 0.f;
        for (int y = 0; y < tab.nrb; y++) s += loss_part[y];
        *loss = s;
    }
    if (i >= n) return;
    int l = 0;
    while (l + 1 < tab.L && i >= tab.w_off[l + 1]) l++;
    const int64_t loc = i - tab.w_off[l];
    const int64_t nw = (int64_t)tab.fo[l] * tab.fi[l];
    float gi = 0.f;
    if (loc < nw) {
        const float* p = ws + tab.ws_w[l] + loc;
        for (int z = 0; z < tab.split[l]; z++) gi += p[z * nw];
    } else {
        const float* p = ws + tab.ws_b[l] + (loc - nw);
        for (int y = 0; y < tab.nrb; y++) gi += p[(int64_t)y * tab.fo[l]];
    }
    if (!update) {
        g[i] = gi;
        return;
    }
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    if (loc < nw) {
        const int r = (int)(loc / tab.fi[l]), c = (int)(loc % tab.fi[l]);
        const __nv_bfloat16 q = __float2bfloat16(wi);
        wb[tab.wb_off[l] + (int64_t)r * tab.fip[l] + c] = q;
        wt[tab.wb_off[l] + (int64_t)c * tab.fop[l] + r] = q;
    }
}

// ------------------------------------------------------------------ the chain of a batch tile
// A training step's forward and backward products of CB = 64 rows of the batch in one CTA, layer by layer
// without leaving the SM (before: a launch per layer and direction, 10 to 20 us each, latency-bound).  The
// products are taken transposed, D^T[features][rows] = W X^T: A is the weight matrix (128-row tiles, K-major, in
// shared memory as it lies in global memory: one bulk copy per layer, which runs while the previous
// layer's epilogue does), B the tile of activations [64 rows][K].  A TMEM lane is then a feature and
// its columns the rows of the batch: bias, tanh and tanh' are lane-local, the copies that the weight gradients
// read are written in their operands' order, a warp's 512 bytes at a time, and the epilogue writes the
// next product's B operand straight into shared memory.  The output layer's product is taken the other way round (a lane per row:
// loss and dH of a row), and its dX, one product per element, needs no MMA.  Bound by the epilogues (16384
// values per layer and tile, an accurate tanhf each): 16 warps, and 64 rows so that a batch of 8192 is 128 CTAs.
// 8192 x (6 -> 256 x 4 -> 1): a step took 262 us with a launch per product, 80 us now (40 chain, 16 dW, 13 Adam).
// Sums and roundings are those of the launch-per-product form (same products in the same K order, the same
// trees of partial sums), so both give the same gradients.
struct ChainArgs {
    int n_in, width, depth;
    int64_t B, cap;
    const float* x;
    const float* tgt;                                  // null: forward only
    float* y;                                          // nullable
    const __nv_bfloat16* wk[kMaxLayers];
    const __nv_bfloat16* wkt[kMaxLayers];
    const float* bias[kMaxLayers];
    __nv_bfloat16* act;                                // per layer 256 cap values: its input as [cap/8][rows][8] (rows:
                                                       // pad16(n_in), then those of a weight tile)
    __nv_bfloat16* dh;                                 // per layer its dH the same way (16 rows for the output layer)
    float* th;                                         // tanh of the hidden layers, per layer [cap/4][rows][4]
    float* db_part[kMaxLayers];                        // [64-row blocks][fo]
    float* loss_part;                                  // [64-row blocks]
    float invB;
    int* err;
};
constexpr int LBO_X = CB * 16 + 16;                    // K-group stride of the activations (spread over the banks)
__host__ __device__ constexpr int pad16c(int v) { return (v + 15) & ~15; }
__host__ __device__ constexpr int chain_kmax(int n_in, int width) { return pad16c(n_in > width ? n_in : width); }
// weights | activations (+ 1 KB: the output product's A rows 64..127, which nothing reads, lie beyond) | output weights
__host__ __device__ constexpr size_t chain_w_bytes(int n_in, int width) { return (size_t)((width + 127) / 128 * 128) * chain_kmax(n_in, width) * 2; }
__host__ __device__ constexpr size_t chain_x_bytes(int n_in, int width) { return (size_t)(chain_kmax(n_in, width) / 8) * LBO_X + 1024; }
__host__ __device__ constexpr size_t chain_smem(int n_in, int width) {
    return chain_w_bytes(n_in, width) + chain_x_bytes(n_in, width) + (size_t)pad16c(width) * 32;
}

// sum of 32 values in the order of warp_sum's butterfly
__device__ __forceinline__ float tree_sum(const float (&v)[32]) {
    float a[16];
#pragma unroll
    for (int i = 0; i < 16; i++) a[i] = v[i] + v[i + 16];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < o; i++) a[i] = a[i] + a[i + o];
    return a[0];
}

__global__ void __launch_bounds__(CT, 1) k_mlp_chain(__grid_constant__ const ChainArgs g) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ uint64_t bars[2];                       // weights, products
    __shared__ uint32_t s_taddr;
    __shared__ int s_abort;
    __shared__ float s_red[2][256];
    __shared__ float s_d[CB];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int width = g.width, depth = g.depth;
    const int K0 = pad16c(g.n_in), Kh = pad16c(width), rows = (width + 127) / 128 * 128;
    const bool train = g.tgt != nullptr;
    const uint32_t sW = smem_addr(smem), sX = sW + (uint32_t)chain_w_bytes(g.n_in, width);
    const uint32_t sO = sX + (uint32_t)chain_x_bytes(g.n_in, width);
    const uint32_t wb = smem_addr(&bars[0]), mb = smem_addr(&bars[1]);
    const int64_t b0 = (int64_t)blockIdx.x * CB;
    // this thread's part of an accumulator: feature f (TMEM lane), rows 32 ch .. 32 ch + 31 of the tile
    const int half = (warp >> 2) & 1, ch = warp >> 3, f = 128 * half + 32 * (warp & 3) + lane;
    const bool mine = 128 * half < rows, live = f < width;
    if (warp == 0) {
        tm_alloc(smem_addr(&s_taddr), 256);
        tm_relinquish();
    }
    if (tid == 0) {
        mbar_init(wb, 1);
        mbar_init(mb, 1);
        mbar_fence_init();
        s_abort = 0;
    }
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    const uint32_t tbase = s_taddr, tacc = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(64 * half + 32 * ch);
    uint32_t wph = 0, mph = 0;
    bool wpend = false, mpend = false;                 // (thread 0) copies and products in flight
    auto load_w = [&](const __nv_bfloat16* src, int K, bool out_too) {
        const uint32_t bytes = (uint32_t)rows * (uint32_t)K * 2u, ob = out_too ? (uint32_t)Kh * 32u : 0u;
        mbar_expect_tx(wb, bytes + ob);
        if (out_too) bulk_load(sO, g.wk[depth], ob, wb);
        for (uint32_t o = 0; o < bytes; o += 16384u) bulk_load(sW + o, reinterpret_cast<const unsigned char*>(src) + o, min(16384u, bytes - o), wb);
        wpend = true;
    };
    if (tid == 0) load_w(g.wk[0], K0, true);
    // the network's input in BF16: this tile's B operand and the feature-major copy
    for (int i = tid; i < CB * K0; i += CT) {
        const int n = i & (CB - 1), k = i / CB;
        const int64_t b = b0 + n;
        const uint32_t v = (b < g.B && k < g.n_in) ? bf16_bits(__ldg(g.x + b * g.n_in + k)) : 0u;
        asm volatile("st.shared.u16 [%0], %1;" :: "r"(sX + (uint32_t)((k >> 3) * LBO_X + n * 16 + (k & 7) * 2)), "h"((unsigned short)v) : "memory");
        if (train) reinterpret_cast<unsigned short*>(g.act)[chain_at(k, (int)b, K0)] = (unsigned short)v;
    }
    fence_proxy_async_smem();
    __syncthreads();
    // D^T = A X^T over K: issued by thread 0 once the weights are there; every thread waits for the products
    auto product = [&](int K) {
        if (tid == 0 && !s_abort) {
            mbar_wait(wb, wph, g.err, &s_abort);
            if (!s_abort) {
                wph ^= 1;
                wpend = false;
                tm_fence_after();
                for (int h = 0; h < rows / 128; h++)
                    for (int ks = 0; ks < K / 16; ks++)
                        mma_bf16(tbase + 64 * h, smem_desc(sW + h * 2048 + 2 * ks * rows * 16, rows * 16, 128),
                                 smem_desc(sX + 2 * ks * LBO_X, LBO_X, 128), idesc_bf16(CB), ks > 0 ? 1u : 0u);
                mma_commit(mb);
                mpend = true;
            }
        }
    };
    auto wait_product = [&]() {
        mbar_wait_next(mb, mph, g.err, &s_abort);
        tm_fence_after();
    };
    auto abort_now = [&]() {                            // the same answer in every thread
        __syncthreads();
        return s_abort != 0;
    };
    // an epilogue's 32 BF16 values (bits in pairs) into the B operand and the feature-major copy
    auto put = [&](const uint32_t (&q)[16], bool operand, __nv_bfloat16* copy) {
        if (operand && f < Kh) {
            const uint32_t at = sX + (uint32_t)((f >> 3) * LBO_X + 32 * ch * 16 + (f & 7) * 2);
#pragma unroll
            for (int n = 0; n < 32; n++)
                asm volatile("st.shared.u16 [%0], %1;" :: "r"(at + 16 * n), "h"((unsigned short)(q[n >> 1] >> (16 * (n & 1)))) : "memory");
        }
        if (copy && mine) {
#pragma unroll
            for (int e = 0; e < 4; e++)
                *reinterpret_cast<uint4*>(copy + ((b0 / 8 + 4 * ch + e) * rows + f) * 8) = make_uint4(q[4 * e], q[4 * e + 1], q[4 * e + 2], q[4 * e + 3]);
        }
    };
    bool stop = false;
    // ---- forward
    for (int l = 0; l < depth && !stop; l++) {
        product(l == 0 ? K0 : Kh);
        wait_product();
        if (tid == 0 && !s_abort) {
            mpend = false;
            if (l + 1 < depth) load_w(g.wk[l + 1], Kh, false);
            else if (train && depth > 1) load_w(g.wkt[depth - 1], Kh, false);
        }
        if (mine && !s_abort) {
            float t[32];
            tm_ld16(tacc, reinterpret_cast<float(&)[16]>(t[0]));
            tm_ld16(tacc + 16, reinterpret_cast<float(&)[16]>(t[16]));
            tm_wait_ld();
            const float bias = live ? __ldg(g.bias[l] + f) : 0.f;
            uint32_t q[16];
#pragma unroll
            for (int n = 0; n < 32; n++) t[n] = live ? tanhf(t[n] + bias) : 0.f;
#pragma unroll
            for (int n = 0; n < 16; n++) q[n] = bf16_bits(t[2 * n]) | (bf16_bits(t[2 * n + 1]) << 16);
            if (train && live) {
                float4* o = reinterpret_cast<float4*>(g.th + (int64_t)l * 256 * g.cap) + (b0 / 4 + 8 * ch) * rows + f;
#pragma unroll
                for (int e = 0; e < 8; e++) o[e * rows] = make_float4(t[4 * e], t[4 * e + 1], t[4 * e + 2], t[4 * e + 3]);
            }
            put(q, true, train ? g.act + (int64_t)(l + 1) * 256 * g.cap : nullptr);
        }
        tm_fence_before();
        fence_proxy_async_smem();
        stop = abort_now();
    }
    // ---- output layer: a lane per row
    if (!stop) {
        if (tid == 0) {
            tm_fence_after();
            for (int ks = 0; ks < Kh / 16; ks++)
                mma_bf16(tbase + 128, smem_desc(sX + 2 * ks * LBO_X, LBO_X, 128), smem_desc(sO + 2 * ks * 256, 256, 128), idesc_bf16(16),
                         ks > 0 ? 1u : 0u);
            mma_commit(mb);
            mpend = true;
        }
        wait_product();
        if (tid == 0 && !s_abort) mpend = false;
        if (warp < 2 && !s_abort) {
            float t[16];
            tm_ld16(tbase + ((uint32_t)(32 * warp) << 16) + 128, t);
            tm_wait_ld();
            const int64_t b = b0 + 32 * warp + lane;
            const bool in = b < g.B;
            const float y = t[0] + __ldg(g.bias[depth]);
            if (in && g.y) g.y[b] = y;
            if (train) {
                const float dd = in ? y - g.tgt[b] : 0.f;
                const float d = 2.f * dd * g.invB;
                const __nv_bfloat16 db = __float2bfloat16(d);
                g.dh[(int64_t)depth * 256 * g.cap + chain_at(0, (int)b, 16)] = db;
                s_d[32 * warp + lane] = __bfloat162float(db);
                const float ls = warp_sum(dd * dd * g.invB), sd = warp_sum(d);
                if (lane == 0) { s_red[0][warp] = ls; s_red[1][warp] = sd; }
            }
        }
        tm_fence_before();
        stop = abort_now();
        if (train && !stop) {
            if (tid == 0) {
                g.loss_part[blockIdx.x] = s_red[0][0] + s_red[0][1];
                g.db_part[depth][blockIdx.x] = s_red[1][0] + s_red[1][1];
            }
            __syncthreads();
        }
    }
    // ---- backward: dH of hidden layer l from that of the layer above
    for (int l = depth - 1; train && l >= 0 && !stop; l--) {
        float th[32];
        if (live) {
            const float4* o = reinterpret_cast<const float4*>(g.th + (int64_t)l * 256 * g.cap) + (b0 / 4 + 8 * ch) * rows + f;
#pragma unroll
            for (int e = 0; e < 8; e++) {
                const float4 v = o[e * rows];
                th[4 * e] = v.x; th[4 * e + 1] = v.y; th[4 * e + 2] = v.z; th[4 * e + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int e = 0; e < 32; e++) th[e] = 0.f;
        }
        float t[32];
        if (l == depth - 1) {                           // dX of the output layer: one product per element
            const float w = live ? __bfloat162float(g.wk[depth][chain_at(0, f, 16)]) : 0.f;
#pragma unroll
            for (int n = 0; n < 32; n++) t[n] = s_d[32 * ch + n] * w;
        } else {
            product(Kh);
            wait_product();
            if (tid == 0 && !s_abort) {
                mpend = false;
                if (l > 0) load_w(g.wkt[l], Kh, false);
            }
            if (mine && !s_abort) {
                tm_ld16(tacc, reinterpret_cast<float(&)[16]>(t[0]));
                tm_ld16(tacc + 16, reinterpret_cast<float(&)[16]>(t[16]));
                tm_wait_ld();
            } else {
#pragma unroll
                for (int n = 0; n < 32; n++) t[n] = 0.f;
            }
        }
        uint32_t q[16];
#pragma unroll
        for (int n = 0; n < 32; n++) t[n] = live ? t[n] * (1.f - th[n] * th[n]) : 0.f;
#pragma unroll
        for (int n = 0; n < 16; n++) q[n] = bf16_bits(t[2 * n]) | (bf16_bits(t[2 * n + 1]) << 16);
        put(q, l > 0, g.dh + (int64_t)l * 256 * g.cap);
        s_red[ch][f] = tree_sum(t);
        tm_fence_before();
        fence_proxy_async_smem();
        stop = abort_now();
        if (!stop && ch == 0 && live) g.db_part[l][(int64_t)blockIdx.x * width + f] = s_red[0][f] + s_red[1][f];
        __syncthreads();                                // s_red is read before the next layer writes it
    }
    if (tid == 0) {
        if (wpend) mbar_drain(wb, wph);
        if (mpend) mbar_drain(mb, mph);
    }
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    if (warp == 0) tm_dealloc(tbase, 256);
}

// ------------------------------------------------------------------ the weight gradients after the chain
// dW parts of every layer in one launch: dW[fo][fi] = dH^T X, K = batch, split as in the launch-per-product form (the
// same parts, the same bits).  A CTA takes one part of one 128-row tile: both operands lie in global memory in
// the order of the tensor core's K-major layout (k_mlp_chain wrote them so), so a chunk of 64 rows of the batch is one bulk
// copy for X and one per K group for the tile's rows of dH; two chunks in flight.  The parts are written
// [part][column][row], a warp's rows contiguous.  The six launches this replaces loaded their operands through
// registers, 32 columns a CTA: 33 us for 8192 x (6 -> 256 x 4 -> 1), 15.5 us now.
constexpr int DT = 256, DK = 64;                       // threads; rows of the batch per chunk
struct DwTab {
    int L;
    int first[kMaxLayers + 1];                         // first block of a layer
    int M[kMaxLayers], N[kMaxLayers];                  // dW's rows (outputs) and columns (inputs)
    int ra[kMaxLayers], rb[kMaxLayers];                // rows of the stored dH and X
    int kchunk[kMaxLayers];
    const __nv_bfloat16* a[kMaxLayers];
    const __nv_bfloat16* b[kMaxLayers];
    float* c[kMaxLayers];
};
constexpr int kDwA = 128 * DK * 2, kDwB = 256 * DK * 2, kDwSmem = 2 * (kDwA + kDwB);
__global__ void __launch_bounds__(DT, 2) k_dw_tiles(const __grid_constant__ DwTab t, int K, int* err) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ uint64_t bars[3];                       // two chunks, the products
    __shared__ uint32_t s_taddr;
    __shared__ int s_abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int l = 0;
    while (l + 1 < t.L && (int)blockIdx.x >= t.first[l + 1]) l++;
    const int M = t.M[l], N = t.N[l], Np = (N + 15) & ~15, ny = (M + 127) / 128;
    const int r = blockIdx.x - t.first[l], m0 = (r % ny) * 128, z = r / ny;
    const int kb = z * t.kchunk[l], ke = min(K, kb + t.kchunk[l]), nc = kb < ke ? (ke - kb + DK - 1) / DK : 0;
    const int ra = t.ra[l], rb = t.rb[l], ma = min(128, ra - m0);       // rows of dH loaded per K group
    if (warp == 0) {
        tm_alloc(smem_addr(&s_taddr), 256);
        tm_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < 3; i++) mbar_init(smem_addr(&bars[i]), 1);
        mbar_fence_init();
        s_abort = 0;
    }
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    const uint32_t tbase = s_taddr, mb = smem_addr(&bars[2]);
    if (tid == 0 && nc > 0) {
        auto load = [&](int c) {
            const int s = c & 1, k0 = kb + c * DK, g8 = (min(ke, k0 + DK) - k0) / 8;
            const uint32_t sa = smem_addr(smem) + s * (kDwA + kDwB), sb = sa + kDwA, bar = smem_addr(&bars[s]);
            mbar_expect_tx(bar, (uint32_t)g8 * (uint32_t)(ma + rb) * 16u);
            for (int g = 0; g < g8; g++)
                bulk_load(sa + g * ma * 16, t.a[l] + ((int64_t)(k0 / 8 + g) * ra + m0) * 8, (uint32_t)ma * 16u, bar);
            bulk_load(sb, t.b[l] + (int64_t)(k0 / 8) * rb * 8, (uint32_t)g8 * (uint32_t)rb * 16u, bar);
        };
        int loaded = 0, done = 0;
        uint32_t mph = 0;
        for (; loaded < min(2, nc); loaded++) load(loaded);
        for (int c = 0; c < nc && !s_abort; c++) {
            const int s = c & 1, k0 = kb + c * DK, ks_n = (min(ke, k0 + DK) - k0) / 16;
            mbar_wait(smem_addr(&bars[s]), (c >> 1) & 1, err, &s_abort);
            if (s_abort) break;
            done = c + 1;
            tm_fence_after();
            const uint32_t sa = smem_addr(smem) + s * (kDwA + kDwB), sb = sa + kDwA;
            for (int ks = 0; ks < ks_n; ks++)
                mma_bf16(tbase, smem_desc(sa + 2 * ks * ma * 16, ma * 16, 128), smem_desc(sb + 2 * ks * rb * 16, rb * 16, 128), idesc_bf16(Np),
                         (c > 0 || ks > 0) ? 1u : 0u);
            mma_commit(mb);
            if (loaded < nc) {                           // the chunk's buffers are free once its products are done
                mbar_wait(mb, mph, err, &s_abort);
                if (s_abort) { mbar_drain(mb, mph); break; }
                mph ^= 1;
                load(loaded++);
            } else {
                mbar_wait(mb, mph, err, &s_abort);
                if (s_abort) { mbar_drain(mb, mph); break; }
                mph ^= 1;
            }
        }
        for (int c = done; c < loaded; c++) mbar_drain(smem_addr(&bars[c & 1]), (c >> 1) & 1);     // after a give-up
    }
    __syncthreads();
    if (!s_abort) {
        tm_fence_after();
        const int row = m0 + 32 * (warp & 3) + lane;
        float* const P = t.c[l] + (int64_t)z * M * N;
        for (int c0 = 16 * (warp >> 2); c0 < N; c0 += 32) {
            float v[16];
            if (nc > 0) {
                tm_ld16(tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0, v);
                tm_wait_ld();
            } else {
#pragma unroll
                for (int j = 0; j < 16; j++) v[j] = 0.f;
            }
            if (row < M) {
#pragma unroll
                for (int j = 0; j < 16; j++)
                    if (c0 + j < N) P[(int64_t)(c0 + j) * M + row] = v[j];
            }
        }
    }
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    if (warp == 0) tm_dealloc(tbase, 256);
}

// The gradient sums and the Adam step after k_dw_tiles, as k_grad_adam takes them: a block per 32 x 32 tile of a
// weight matrix (the parts are read along the rows, as they were written, and the weights along the columns, by
// way of shared memory), then a block per layer for its bias (the last one also adds up the loss).
struct AdamArgs {
    float lr, b1, b2, eps, c1, c2;
    int update;
};
__device__ __forceinline__ float adam_step(const AdamArgs& a, float* w, float* m, float* v, int64_t i, float g) {
    // the moments with the new gradient's product fused, the old one's rounded (as the narrow networks' kernel is
    // compiled): a weight's last bit decides BF16 roundings of the next step
    const float mi = __fmaf_rn(1.f - a.b1, g, __fmul_rn(a.b1, m[i]));
    const float vi = __fmaf_rn(__fmul_rn(1.f - a.b2, g), g, __fmul_rn(a.b2, v[i]));
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
    w[i] = wi;
    return wi;
}
__global__ void __launch_bounds__(256) k_adam_tiles(float* __restrict__ w, float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                                                    const float* __restrict__ ws, const float* __restrict__ loss_part,
                                                    float* __restrict__ loss, const __grid_constant__ LayerTab tab,
                                                    const __grid_constant__ AdamArgs a, __nv_bfloat16* __restrict__ wk,
                                                    __nv_bfloat16* __restrict__ wkt) {
    __shared__ float s[32][33];
    int l = 0, r = blockIdx.x;
    for (; l < tab.L; l++) {
        const int n = ((tab.fo[l] + 31) / 32) * ((tab.fi[l] + 31) / 32);
        if (r < n) break;
        r -= n;
    }
    if (l < tab.L) {
        const int fo = tab.fo[l], fi = tab.fi[l], tr = (fo + 31) / 32, r0 = (r % tr) * 32, c0 = (r / tr) * 32;
        const int x = threadIdx.x & 31, y = threadIdx.x >> 5, split = tab.split[l];
        const int64_t nw = (int64_t)fo * fi;
        const float* P = ws + tab.ws_w[l];
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int c = c0 + y + 8 * e;
            if (r0 + x < fo && c < fi) {
                const float* p = P + (int64_t)c * fo + r0 + x;
                float sum = 0.f;
                int z = 0;
                for (; z + 16 <= split; z += 16) {        // sixteen loads in flight, added in order
                    float q[16];
#pragma unroll
                    for (int i = 0; i < 16; i++) q[i] = __ldcs(p + (z + i) * nw);
#pragma unroll
                    for (int i = 0; i < 16; i++) sum += q[i];
                }
                for (; z < split; z++) sum += p[z * nw];
                s[y + 8 * e][x] = sum;
            }
        }
        __syncthreads();
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int rr = r0 + y + 8 * e, c = c0 + x;
            if (rr >= fo || c >= fi) continue;
            const int64_t i = tab.w_off[l] + (int64_t)rr * fi + c;
            const float gi = s[x][y + 8 * e];
            if (!a.update) {
                g[i] = gi;
                continue;
            }
            const __nv_bfloat16 q = __float2bfloat16(adam_step(a, w, m, v, i, gi));
            wk[tab.wk_off[l] + chain_at(rr, c, tab.rows[l])] = q;
            if (l > 0 && l + 1 < tab.L) wkt[tab.wk_off[l] + chain_at(c, rr, tab.rows[l])] = q;
        }
        return;
    }
    // p[0] + p[stride] + ... over the 64-row blocks, in pairs (the row blocks of the launch-per-product form)
    auto block_sum = [&](const float* p, int64_t stride) {
        float sum = 0.f;
        int y = 0;
        for (; y + 16 <= tab.nrc; y += 16) {
            float q[16];
#pragma unroll
            for (int i = 0; i < 16; i++) q[i] = p[(y + i) * stride];
#pragma unroll
            for (int i = 0; i < 16; i += 2) sum += q[i] + q[i + 1];
        }
        for (; y < tab.nrc; y += 2) sum += p[y * stride] + (y + 1 < tab.nrc ? p[(y + 1) * stride] : 0.f);
        return sum;
    };
    l = r;                                                // bias blocks
    const int fo = tab.fo[l], f = threadIdx.x;
    if (f < fo) {
        const int64_t i = tab.w_off[l] + (int64_t)fo * tab.fi[l] + f;
        const float gi = block_sum(ws + tab.ws_b[l] + f, fo);
        if (a.update) adam_step(a, w, m, v, i, gi);
        else g[i] = gi;
    }
    if (l == tab.L - 1 && f == 32) *loss = block_sum(loss_part, 1);
}

// BF16 copies of the weights, zero-padded to [fout_pad][fin_pad] and [fin_pad][fout_pad]
// (at creation and on new parameters)
__global__ void k_refresh(const float* __restrict__ w, int fout, int fin, int fout_p, int fin_p, __nv_bfloat16* __restrict__ wb,
                          __nv_bfloat16* __restrict__ wt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= fout_p * fin_p) return;
    const int r = i / fin_p, c = i % fin_p;
    const __nv_bfloat16 q = __float2bfloat16((r < fout && c < fin) ? w[r * fin + c] : 0.f);
    wb[i] = q;
    wt[c * fout_p + r] = q;
}

static int pad16(int v) { return (v + 15) & ~15; }

static int layer_in(const hyb_mlp* m, int l) { return l == 0 ? m->n_in : m->width; }
static int layer_out(const hyb_mlp* m, int l) { return l == m->L - 1 ? 1 : m->width; }

// the same in k_mlp_chain's order; the padding is zero
__global__ void k_refresh_chain(const float* __restrict__ w, int fout, int fin, int rows, int kpad, __nv_bfloat16* __restrict__ wk,
                                __nv_bfloat16* __restrict__ wkt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows * kpad) return;
    const int r = i / kpad, c = i % kpad;
    wk[chain_at(r, c, rows)] = __float2bfloat16((r < fout && c < fin) ? w[(int64_t)r * fin + c] : 0.f);
    if (wkt) wkt[chain_at(r, c, rows)] = __float2bfloat16((r < fin && c < fout) ? w[(int64_t)c * fin + r] : 0.f);
}

// rows of a layer's operand in k_mlp_chain: hidden layers in whole 128-row tiles of the product; the output
// layer (an N = 16 operand) 16
static int chain_rows(const hyb_mlp* m, int l) { return l == m->L - 1 ? 16 : (m->width + 127) / 128 * 128; }

static hyb_status refresh(hyb_mlp* m, cudaStream_t s) {
    if (m->chain) {
        for (int l = 0; l < m->L; l++) {
            const int fo = layer_out(m, l), fi = layer_in(m, l), rows = m->tab.rows[l], kp = pad16(fi);
            k_refresh_chain<<<(rows * kp + 255) / 256, 256, 0, s>>>(m->master + m->w_off[l], fo, fi, rows, kp, m->wk + m->tab.wk_off[l],
                                                                   l > 0 && l + 1 < m->L ? m->wkt + m->tab.wk_off[l] : nullptr);
            m->launches++;
        }
        HYB_CUDA_TRY(cudaGetLastError());
        return HYB_OK;
    }
    for (int l = 0; l < m->L; l++) {
        const int fo = layer_out(m, l), fi = layer_in(m, l), fop = pad16(fo), fip = pad16(fi);
        k_refresh<<<(fop * fip + 255) / 256, 256, 0, s>>>(m->master + m->w_off[l], fo, fi, fop, fip, m->wbf + m->wb_off[l],
                                                          m->wbt + m->wb_off[l]);
        m->launches++;
    }
    HYB_CUDA_TRY(cudaGetLastError());
    return HYB_OK;
}

static hyb_status ensure_cap(hyb_mlp* m, int64_t B) {
    if (B <= m->cap) return HYB_OK;
    if (m->actT) { cudaFree(m->act); cudaFree(m->actT); cudaFree(m->pre); cudaFree(m->dhb); cudaFree(m->dhT); cudaFree(m->ws); }
    m->act = m->actT = m->dhb = m->dhT = nullptr;
    m->pre = m->ws = nullptr;
    m->cap = 0;
    const int64_t cap = ((B + 127) / 128) * 128;
    const size_t na = (size_t)std::max(1, m->L - 1) * cap * 256;
    const size_t nrb = (size_t)(cap / (m->chain ? CB : 128));
    size_t nb = 0;
    for (int l = 0; l < m->L; l++) nb += nrb * layer_out(m, l);
    HYB_CUDA_TRY(cudaMalloc(&m->pre, sizeof(float) * na));
    if (m->chain) {          // input and dH of every layer, in the order of the weight gradients' operands
        HYB_CUDA_TRY(cudaMalloc(&m->actT, sizeof(__nv_bfloat16) * (size_t)m->L * cap * 256));
        HYB_CUDA_TRY(cudaMalloc(&m->dhT, sizeof(__nv_bfloat16) * (size_t)m->L * cap * 256));
    } else {
        HYB_CUDA_TRY(cudaMalloc(&m->act, sizeof(__nv_bfloat16) * na));
        HYB_CUDA_TRY(cudaMalloc(&m->actT, sizeof(__nv_bfloat16) * na));
        HYB_CUDA_TRY(cudaMalloc(&m->dhb, sizeof(__nv_bfloat16) * 2 * (size_t)cap * 256));
        HYB_CUDA_TRY(cudaMalloc(&m->dhT, sizeof(__nv_bfloat16) * 2 * (size_t)cap * 256));
    }
    HYB_CUDA_TRY(cudaMalloc(&m->ws, sizeof(float) * (m->ws_w_size + nb + nrb)));
    // bias parts start after the weight parts, the loss parts after the bias parts
    size_t off = m->ws_w_size;
    for (int l = 0; l < m->L; l++) { m->tab.ws_b[l] = (int64_t)off; off += nrb * layer_out(m, l); }
    m->cap = cap;
    return HYB_OK;
}

static float* loss_parts(const hyb_mlp* m) {
    return m->ws + m->tab.ws_b[m->L - 1] + (size_t)(m->cap / (m->chain ? CB : 128)) * layer_out(m, m->L - 1);
}

// input of layer l >= 1 (BF16 activations of layer l - 1): row-major [cap][256] and feature-major [256][cap]
static __nv_bfloat16* act_in(const hyb_mlp* m, int l) { return m->act + (size_t)(l - 1) * m->cap * 256; }
static __nv_bfloat16* actT_in(const hyb_mlp* m, int l) { return m->actT + (size_t)(l - 1) * m->cap * 256; }
// dH of layer l (BF16): two buffers of each layout, so that the dX product of layer l reads one
// while its epilogue writes dH of layer l - 1 into the other
static int dh_buf(const hyb_mlp* m, int l) { return (m->L - 1 - l) & 1; }
static __nv_bfloat16* dh_of(const hyb_mlp* m, int l) { return m->dhb + (size_t)dh_buf(m, l) * m->cap * 256; }
static __nv_bfloat16* dhT_of(const hyb_mlp* m, int l) { return m->dhT + (size_t)dh_buf(m, l) * m->cap * 256; }

// forward pass: one GEMM per layer, bias and tanh in its epilogue; with a target the output
// layer's epilogue also forms dH of the output layer and the parts of the loss and its bias gradient
static hyb_status chain_pass(hyb_mlp* m, const float* x, int64_t B, float* y, const float* tgt, cudaStream_t s);
static hyb_status forward(hyb_mlp* m, const float* x, int64_t B, float* y, const float* tgt, cudaStream_t s) {
    if (m->chain) return chain_pass(m, x, B, y, tgt, s);
    hyb_status st = ensure_cap(m, B);
    if (st != HYB_OK) return st;
    const int64_t cap = m->cap;
    for (int l = 0; l < m->L; l++) {
        const int fi = pad16(layer_in(m, l)), fo = pad16(layer_out(m, l));
        const __nv_bfloat16* W = m->wbf + m->wb_off[l];
        Epi ep;
        ep.bias = m->master + m->b_off[l];
        ep.n = layer_out(m, l);
        ep.invB = 1.f / (float)B;
        ep.ldT = cap;
        // H[B][fo] = X[B][fi] W^T, W stored [fo][fi]
        if (l < m->L - 1) {
            ep.pre = m->pre + (size_t)l * cap * 256;
            ep.act = act_in(m, l + 1);
            ep.actT = actT_in(m, l + 1);
            if (l == 0) gemm<EP_HIDDEN>((int)B, fo, fi, x, m->n_in, 1, W, 1, fi, ep, s, m->launches, m->err);
            else gemm<EP_HIDDEN>((int)B, fo, fi, act_in(m, l), 256, 1, W, 1, fi, ep, s, m->launches, m->err);
        } else {
            ep.out = y;
            ep.tgt = tgt;
            ep.loss_part = loss_parts(m);
            ep.db_part = m->ws + m->tab.ws_b[l];
            ep.act = dh_of(m, l);
            ep.actT = dhT_of(m, l);
            if (l == 0) gemm<EP_OUTPUT>((int)B, fo, fi, x, m->n_in, 1, W, 1, fi, ep, s, m->launches, m->err);
            else gemm<EP_OUTPUT>((int)B, fo, fi, act_in(m, l), 256, 1, W, 1, fi, ep, s, m->launches, m->err);
        }
    }
    HYB_CUDA_TRY(cudaGetLastError());
    return HYB_OK;
}

// backward pass after forward(.., tgt): per layer the parts of the weight gradient dW = dH^T X
// (split K) and, below the first layer, dX = dH W with tanh' and the parts of the bias
// gradient of the layer below in the epilogue
static hyb_status backward(hyb_mlp* m, const float* x, int64_t B, cudaStream_t s) {
    if (m->chain) return HYB_OK;                        // done with the forward pass
    const int64_t cap = m->cap;
    m->tab.nrb = (int)((B + TM - 1) / TM);
    for (int l = m->L - 1; l >= 0; l--) {
        const int fi = pad16(layer_in(m, l)), fo = pad16(layer_out(m, l));
        const int ni = layer_in(m, l), no = layer_out(m, l);
        Epi ep;
        ep.c = m->ws + m->tab.ws_w[l];
        m->tab.split[l] = split_of(no, ni, (int)B);
        // dW[no][ni] = dH^T X: M = no, N = ni, K = B, both operands read batch-contiguous
        if (l == 0) gemm<EP_PART>(no, ni, (int)B, dhT_of(m, l), cap, 1, x, m->n_in, 1, ep, s, m->launches, m->err);
        else gemm<EP_PART>(no, ni, (int)B, dhT_of(m, l), cap, 1, actT_in(m, l), 1, cap, ep, s, m->launches, m->err);
        if (l > 0) {
            // dX[B][fi] = dH[B][fo] W[fo][fi] (W read transposed, K = fo contiguous), then dH of layer l - 1
            Epi ed;
            ed.pre = m->pre + (size_t)(l - 1) * cap * 256;
            ed.act = dh_of(m, l - 1);
            ed.actT = dhT_of(m, l - 1);
            ed.ldT = cap;
            ed.db_part = m->ws + m->tab.ws_b[l - 1];
            ed.n = ni;
            gemm<EP_DX>((int)B, fi, fo, dh_of(m, l), 256, 1, m->wbt + m->wb_off[l], 1, fo, ed, s, m->launches, m->err);
        }
    }
    HYB_CUDA_TRY(cudaGetLastError());
    return HYB_OK;
}

// the chain of a whole batch; with a target also the backward products, and then every layer's
// weight-gradient parts: two launches
static hyb_status chain_pass(hyb_mlp* m, const float* x, int64_t B, float* y, const float* tgt, cudaStream_t s) {
    if (tgt) {
        hyb_status st = ensure_cap(m, B);
        if (st != HYB_OK) return st;
    }
    const int64_t cap = m->cap;
    ChainArgs c{};
    c.n_in = m->n_in;
    c.width = m->width;
    c.depth = m->depth;
    c.B = B;
    c.cap = cap;
    c.x = x;
    c.tgt = tgt;
    c.y = y;
    c.invB = 1.f / (float)B;
    c.err = m->err;
    for (int l = 0; l < m->L; l++) {
        c.wk[l] = m->wk + m->tab.wk_off[l];
        c.wkt[l] = m->wkt + m->tab.wk_off[l];
        c.bias[l] = m->master + m->b_off[l];
        c.db_part[l] = m->ws + m->tab.ws_b[l];
    }
    if (tgt) {
        c.act = m->actT;
        c.dh = m->dhT;
        c.th = m->pre;
        c.loss_part = loss_parts(m);
    }
    const size_t smem = chain_smem(m->n_in, m->width);
    const cudaError_t attr = func_attr_once((const void*)k_mlp_chain, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)chain_smem(256, 256));
    if (attr != cudaSuccess) return cuda_fail(attr, "k_mlp_chain");
    k_mlp_chain<<<(unsigned)((B + CB - 1) / CB), CT, smem, s>>>(c);
    m->launches++;
    if (tgt) {
        m->tab.nrb = (int)((B + TM - 1) / TM);
        m->tab.nrc = (int)((B + CB - 1) / CB);
        const int Kp = (int)((B + 15) & ~(int64_t)15);
        DwTab t{};
        t.L = m->L;
        int nblk = 0;
        for (int l = 0; l < m->L; l++) {
            const int no = layer_out(m, l), ni = layer_in(m, l), split = split_of(no, ni, (int)B);
            m->tab.split[l] = split;
            t.first[l] = nblk;
            t.M[l] = no;
            t.N[l] = ni;
            t.ra[l] = m->tab.rows[l];
            t.rb[l] = l == 0 ? pad16(ni) : m->tab.rows[l - 1];
            t.kchunk[l] = ((Kp + split - 1) / split + 15) & ~15;
            t.a[l] = m->dhT + (size_t)l * cap * 256;
            t.b[l] = m->actT + (size_t)l * cap * 256;
            t.c[l] = m->ws + m->tab.ws_w[l];
            nblk += ((no + 127) / 128) * split;
        }
        t.first[m->L] = nblk;
        const cudaError_t room = func_attr_once((const void*)k_dw_tiles, cudaFuncAttributeMaxDynamicSharedMemorySize, kDwSmem);
        if (room != cudaSuccess) return cuda_fail(room, "k_dw_tiles");
        k_dw_tiles<<<nblk, DT, kDwSmem, s>>>(t, Kp, m->err);
        m->launches++;
    }
    HYB_CUDA_TRY(cudaGetLastError());
    return HYB_OK;
}

// the gradient sums (and with update the Adam step) over all parameters: one launch
static hyb_status reduce_update(hyb_mlp* m, int update, float lr, cudaStream_t s) {
    const float b1 = 0.9f, b2 = 0.999f;
    float c1 = 1.f, c2 = 1.f;
    if (update) {
        m->step++;
        c1 = 1.f - powf(b1, (float)m->step);
        c2 = 1.f - powf(b2, (float)m->step);
    }
    if (m->chain) {
        const AdamArgs a{lr, b1, b2, 1e-8f, c1, c2, update};
        int blocks = m->L;
        for (int l = 0; l < m->L; l++) blocks += ((layer_out(m, l) + 31) / 32) * ((layer_in(m, l) + 31) / 32);
        k_adam_tiles<<<blocks, 256, 0, s>>>(m->master, m->grad, m->adam_m, m->adam_v, m->ws, loss_parts(m), m->loss, m->tab, a, m->wk, m->wkt);
        m->launches++;
        HYB_CUDA_TRY(cudaGetLastError());
        return HYB_OK;
    }
    k_grad_adam<<<(unsigned)((m->n_params + 255) / 256), 256, 0, s>>>(m->master, m->grad, m->adam_m, m->adam_v, m->ws, loss_parts(m),
                                                                     m->loss, (int64_t)m->n_params, update, lr, b1, b2, 1e-8f, c1,
                                                                     c2, m->tab, m->wbf, m->wbt);
    m->launches++;
    HYB_CUDA_TRY(cudaGetLastError());
    return HYB_OK;
}

}  // namespace hyb

using namespace hyb;

extern "C" {

hyb_status hyb_mlp_create(int n_in, int width, int depth, const float* init_params, hyb_mlp** out) {
    if (!out || n_in < 1 || n_in > 256 || width < 1 || width > 256 || depth < 1 || depth > kMaxLayers - 1) {
        set_error("hyb_mlp_create: bad sizes");
        return HYB_EINVAL;
    }
    *out = nullptr;
    hyb_mlp* m = new hyb_mlp();
    m->n_in = n_in; m->width = width; m->depth = depth; m->L = depth + 1;
    m->chain = width > kNarrow;
    size_t off = 0, woff = 0, wsw = 0, wkoff = 0;
    m->tab.L = m->L;
    for (int l = 0; l < m->L; l++) {
        const int fi = layer_in(m, l), fo = layer_out(m, l);
        m->w_off.push_back(off); off += (size_t)fo * fi;
        m->b_off.push_back(off); off += fo;
        m->wb_off.push_back(woff); woff += (size_t)pad16(fo) * pad16(fi);
        m->tab.w_off[l] = (int64_t)m->w_off[l];
        m->tab.wb_off[l] = (int64_t)m->wb_off[l];
        m->tab.ws_w[l] = (int64_t)wsw; wsw += (size_t)kMaxSplit * fo * fi;
        m->tab.fo[l] = fo;
        m->tab.fi[l] = fi;
        m->tab.fop[l] = pad16(fo);
        m->tab.fip[l] = pad16(fi);
        m->tab.rows[l] = chain_rows(m, l);
        m->tab.wk_off[l] = (int64_t)wkoff; wkoff += (size_t)m->tab.rows[l] * pad16(fi);
    }
    m->n_params = off;
    m->ws_w_size = wsw;
    cudaError_t e = cudaMalloc(&m->master, sizeof(float) * off);
    if (e == cudaSuccess) e = cudaMalloc(&m->adam_m, sizeof(float) * off);
    if (e == cudaSuccess) e = cudaMalloc(&m->adam_v, sizeof(float) * off);
    if (e == cudaSuccess) e = cudaMalloc(&m->grad, sizeof(float) * off);
    if (m->chain) {
        if (e == cudaSuccess) e = cudaMalloc(&m->wk, sizeof(__nv_bfloat16) * wkoff);
        if (e == cudaSuccess) e = cudaMalloc(&m->wkt, sizeof(__nv_bfloat16) * wkoff);
    } else {
        if (e == cudaSuccess) e = cudaMalloc(&m->wbf, sizeof(__nv_bfloat16) * woff);
        if (e == cudaSuccess) e = cudaMalloc(&m->wbt, sizeof(__nv_bfloat16) * woff);
    }
    if (e == cudaSuccess) e = cudaMalloc(&m->loss, sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&m->err, sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(m->err, 0, sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(m->adam_m, 0, sizeof(float) * off);
    if (e == cudaSuccess) e = cudaMemset(m->adam_v, 0, sizeof(float) * off);
    if (e == cudaSuccess && init_params) e = cudaMemcpy(m->master, init_params, sizeof(float) * off, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) { hyb_status st = cuda_fail(e, "hyb_mlp_create"); hyb_mlp_destroy(m); return st; }
    if (!init_params) cudaMemset(m->master, 0, sizeof(float) * off);
    hyb_status st = refresh(m, nullptr);
    if (st != HYB_OK) { hyb_mlp_destroy(m); return st; }
    cudaDeviceSynchronize();
    *out = m;
    return HYB_OK;
}

int64_t hyb_mlp_num_params(const hyb_mlp* m) { return m ? (int64_t)m->n_params : 0; }

hyb_status hyb_mlp_set_params(hyb_mlp* m, const float* params_host) {
    if (!m || !params_host) { set_error("null argument"); return HYB_EINVAL; }
    HYB_CUDA_TRY(cudaMemcpy(m->master, params_host, sizeof(float) * m->n_params, cudaMemcpyHostToDevice));
    return refresh(m, nullptr);
}

hyb_status hyb_mlp_get_params(hyb_mlp* m, float* params_host) {
    if (!m || !params_host) { set_error("null argument"); return HYB_EINVAL; }
    HYB_CUDA_TRY(cudaDeviceSynchronize());
    HYB_CUDA_TRY(cudaMemcpy(params_host, m->master, sizeof(float) * m->n_params, cudaMemcpyDeviceToHost));
    int h = 0;
    HYB_CUDA_TRY(cudaMemcpy(&h, m->err, sizeof(int), cudaMemcpyDeviceToHost));
    if (h) {
        cudaMemset(m->err, 0, sizeof(int));
        set_error("a bounded device-side wait in the surrogate's GEMMs gave up");
        return HYB_ETIMEOUT;
    }
    return HYB_OK;
}

hyb_status hyb_mlp_forward(hyb_mlp* m, const float* x, int64_t B, float* y, void* stream) {
    if (!m || !x || !y || B < 1) { set_error("hyb_mlp_forward: bad arguments"); return HYB_EINVAL; }
    return forward(m, x, B, y, nullptr, (cudaStream_t)stream);
}

hyb_status hyb_mlp_gradients(hyb_mlp* m, const float* x, const float* target, int64_t B, float* grad_host, float* loss_host,
                             void* stream) {
    if (!m || !x || !target || B < 1) { set_error("hyb_mlp_gradients: bad arguments"); return HYB_EINVAL; }
    cudaStream_t s = (cudaStream_t)stream;
    hyb_status st = forward(m, x, B, nullptr, target, s);
    if (st == HYB_OK) st = backward(m, x, B, s);
    if (st == HYB_OK) st = reduce_update(m, 0, 0.f, s);
    if (st != HYB_OK) return st;
    HYB_CUDA_TRY(cudaStreamSynchronize(s));
    if (grad_host) HYB_CUDA_TRY(cudaMemcpy(grad_host, m->grad, sizeof(float) * m->n_params, cudaMemcpyDeviceToHost));
    if (loss_host) HYB_CUDA_TRY(cudaMemcpy(loss_host, m->loss, sizeof(float), cudaMemcpyDeviceToHost));
    return HYB_OK;
}

hyb_status hyb_mlp_train_step(hyb_mlp* m, const float* x, const float* target, int64_t B, float lr, float* loss_dev,
                              void* stream) {
    if (!m || !x || !target || B < 1) { set_error("hyb_mlp_train_step: bad arguments"); return HYB_EINVAL; }
    cudaStream_t s = (cudaStream_t)stream;
    hyb_status st = forward(m, x, B, nullptr, target, s);
    if (st == HYB_OK) st = backward(m, x, B, s);
    if (st == HYB_OK) st = reduce_update(m, 1, lr, s);
    if (st != HYB_OK) return st;
    if (loss_dev) HYB_CUDA_TRY(cudaMemcpyAsync(loss_dev, m->loss, sizeof(float), cudaMemcpyDeviceToDevice, s));
    return HYB_OK;
}

int64_t hyb_mlp_launch_count(const hyb_mlp* m) { return m ? m->launches : 0; }

hyb_status hyb_mlp_destroy(hyb_mlp* m) {
    if (!m) return HYB_OK;
    cudaDeviceSynchronize();
    cudaFree(m->master); cudaFree(m->adam_m); cudaFree(m->adam_v); cudaFree(m->grad); cudaFree(m->wbf); cudaFree(m->wbt);
    cudaFree(m->loss);
    cudaFree(m->err);
    cudaFree(m->act); cudaFree(m->actT); cudaFree(m->pre); cudaFree(m->dhb); cudaFree(m->dhT); cudaFree(m->ws);
    cudaFree(m->wk); cudaFree(m->wkt);
    delete m;
    return HYB_OK;
}

}  // extern "C"
