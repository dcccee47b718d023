// order.cu -- cell order of scattered particles.  The particle kernels are fast when consecutive
// particles share cells (fields staged once per block, currents summed in registers); after some
// hundred steps of a run they no longer do, since nothing moves the caller's particles in memory.  A PIC step
// therefore lists them cell by cell and visits them through that list: counts per cell, a range of the
// list for each cell, the list (each particle takes its cell's next place).  FP32 only: in FP64 the push and the
// deposit are bound by their arithmetic and atomics in any order (1 M shuffled particles, 512 x 256, order 2: a step of
// 1319 us as stored, 1394 listed).
//
// Whether that pays is decided on the device: every block of k_count looks at the same 512 pairs of consecutive
// particles; when at most half of them leave the cell and its right neighbour, the particles are in order, and it
// and the other two kernels return at once.  All of it runs on a stream of its own beside the formation of B^n, which does
// not touch the particles; the push waits for it.  Particles in order pay 8 us of a replayed step for the decision and 10 to
// 13 of a step of plain launches (18 to 22 with five launches on the grid's stream, one of them to clear the counts).
#include <algorithm>

#include "hyb_internal.cuh"

namespace hyb {

constexpr int kOrderThreads = 512;
// Particles from which the list is made, by shape order.  k1-resident steps, 256 x 256, us, as stored and listed:
//   order 1: shuffled 270 K 68 and 77, 600 K 124 and 120, 1 M 191 and 168; in order 600 K 65 and 74;
//   order 2: shuffled 132 K 74 and 64, 270 K 134 and 91, 1 M 361 and 195; in order 132 K 44 and 51;
//   order 3: shuffled 100 K 86 and 64, 270 K 189 and 102, 1 M 584 and 226; in order 100 K 43 and 52.
// (At orders 2 and 3 shuffled sets of 60 K gain a little already, those in order lose a fifth.)
static int64_t order_min(int shape) { return shape == 1 ? 1 << 19 : shape == 2 ? 1 << 17 : 3 << 15; }
// and up to which.  Sets beyond the L2 (some 3 M particles) come from memory a sector at a time when listed, 0.3 ns a
// particle and step whatever the order; as stored they take 0.16, 0.32 and 0.5 ns at orders 1, 2 and 3.  Shuffled, 256 x 256, us as
// stored and listed: order 1 2 M 350 and 337, 4 M 671 and 896, 8 M 1303 and 2430; order 2 6 M 2065 and 1792, 16 M 5126 and 5790;
// order 3 16 M 8800 and 5944.  At order 1 fewer than three particles per cell do not pay either (1024 x 1000: 1 M 290 and 301, 2 M
// 449 and 480).
static int64_t order_max(int shape) { return shape == 1 ? 1 << 21 : shape == 2 ? 6 << 20 : INT32_MAX; }
static bool order_pays(const hyb_grid* g, int64_t np, int shape) {
    return np >= order_min(shape) && np <= order_max(shape) && (shape > 1 || np >= 3 * g->cells);
}
constexpr int kSamplePairs = kOrderThreads;         // a pair per thread
constexpr int kScanCells = 4;                       // cells per thread of k_ranges

// the cell that holds a particle (its offsets may lie in [-1, 2)); 0 for one the push will reject
__device__ __forceinline__ int particle_key(const int32_t* __restrict__ cell, const float* __restrict__ off, int64_t p, int n1, int n2) {
    int cx = cell[2 * p], cy = cell[2 * p + 1];
    float ox = off[2 * p], oy = off[2 * p + 1];
    if (cx < 0 || cx >= n1 || cy < 0 || cy >= n2 || !renormalise(cx, ox, n1) || !renormalise(cy, oy, n2)) return 0;
    return cy * n1 + cx;
}

// The decision (the same in every block) and, for scattered particles, their number per cell; count is zero on entry.
// ctl: jumps among the sampled pairs, the list's cursor.
__global__ void __launch_bounds__(kOrderThreads) k_count(const int32_t* __restrict__ cell, const float* __restrict__ off, int64_t np, int n1,
                                                         int n2, int* __restrict__ count, unsigned* __restrict__ ctl, unsigned limit) {
    const int64_t s = (np - 1) * (int64_t)threadIdx.x / kSamplePairs;
    const int a = particle_key(cell, off, s, n1, n2), b = particle_key(cell, off, s + 1, n1, n2);
    const unsigned jumps = (unsigned)__syncthreads_count(b != a && b != a + 1);
    if (blockIdx.x == 0 && threadIdx.x == 0) { ctl[0] = jumps; ctl[1] = 0u; }
    if (jumps <= limit) return;
    for (int64_t p = blockIdx.x * (int64_t)kOrderThreads + threadIdx.x; p < np; p += (int64_t)gridDim.x * kOrderThreads)
        atomicAdd(count + particle_key(cell, off, p, n1, n2), 1);
}

// count -> next: first place of the cell in the list; count back to zero.  A block's cells share a range taken from
// the cursor, so the order of the ranges is that in which the blocks get there (no block waits for another).
__global__ void __launch_bounds__(kOrderThreads) k_ranges(int* __restrict__ count, int* __restrict__ next, int64_t cells,
                                                          unsigned* __restrict__ ctl, Visit v) {
    __shared__ int wsum[kOrderThreads / 32];
    __shared__ int base;
    if (!visit_perm(v)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t c0 = (blockIdx.x * (int64_t)kOrderThreads + threadIdx.x) * kScanCells;
    int n[kScanCells], sum = 0;
#pragma unroll
    for (int e = 0; e < kScanCells; e++) {
        n[e] = c0 + e < cells ? count[c0 + e] : 0;
        sum += n[e];
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < kOrderThreads / 32; w++) { const int x = wsum[w]; wsum[w] = t; t += x; }
        base = t ? (int)atomicAdd(ctl + 1, (unsigned)t) : 0;
    }
    __syncthreads();
    int at = base + wsum[warp] + incl - sum;
#pragma unroll
    for (int e = 0; e < kScanCells; e++) {
        if (c0 + e < cells) { next[c0 + e] = at; count[c0 + e] = 0; }
        at += n[e];
    }
}

__global__ void __launch_bounds__(kOrderThreads) k_list(const int32_t* __restrict__ cell, const float* __restrict__ off, int64_t np, int n1,
                                                        int n2, int* __restrict__ next, int* __restrict__ perm, Visit v) {
    if (!visit_perm(v)) return;
    for (int64_t p = blockIdx.x * (int64_t)kOrderThreads + threadIdx.x; p < np; p += (int64_t)gridDim.x * kOrderThreads)
        perm[atomicAdd(next + particle_key(cell, off, p, n1, n2), 1)] = (int)p;
}

void order_free(Order& o) {
    if (o.side) cudaStreamSynchronize(o.side);
    for (void* p : o.blocks) cudaFree(p);
    if (o.fork) cudaEventDestroy(o.fork);
    if (o.join) cudaEventDestroy(o.join);
    if (o.side) cudaStreamDestroy(o.side);
    o = Order();
}

// ints of a list of n particles: control words, counts and next places per cell, the list
static size_t order_ints(const hyb_grid* g, int64_t n) { return (size_t)(4 + 2 * g->cells + n); }
static void order_at(Order& o, const hyb_grid* g, int* p, int64_t n) {
    o.ctl = reinterpret_cast<unsigned*>(p);
    o.count = p + 4;
    o.next = o.count + g->cells;
    o.perm = o.next + g->cells;
    o.cap = n;
    o.cells = g->cells;
}
// the side stream; count starts at zero, whatever the grid's stream is doing or capturing
static bool order_clear(Order& o) {
    if ((o.side || cudaStreamCreateWithFlags(&o.side, cudaStreamNonBlocking) == cudaSuccess) &&
        (o.fork || cudaEventCreateWithFlags(&o.fork, cudaEventDisableTiming) == cudaSuccess) &&
        (o.join || cudaEventCreateWithFlags(&o.join, cudaEventDisableTiming) == cudaSuccess) &&
        cudaMemsetAsync(o.count, 0, sizeof(int) * (size_t)o.cells, cudaStreamPerThread) == cudaSuccess &&
        cudaStreamSynchronize(cudaStreamPerThread) == cudaSuccess)
        return true;
    cudaGetLastError();
    return false;
}
// A first list beside the step's scratch: 32 particles per cell, at most 16 MB (an allocation inside the first step
// cost it 50 us, half its time on a grid of this size); none where such sets stay as stored at every
// shape order
static int64_t order_first(const hyb_grid* g) {
    const int64_t n = std::min<int64_t>(32 * (int64_t)g->cells, 1 << 22);
    return g->d.dims == 2 && g->d.precision == 32 && g->cells <= 1 << 20 && n >= order_min(3) ? n : 0;
}
size_t order_bytes(const hyb_grid* g) {
    const int64_t n = order_first(g);
    return n ? sizeof(int) * order_ints(g, n) : 0;
}
void order_place(Order& o, const hyb_grid* g, void* at) {
    order_at(o, g, reinterpret_cast<int*>(at), order_first(g));
    o.off = !order_clear(o);
}

bool order_reserve(Order& o, const hyb_grid* g, int64_t np, int shape) {
    // 2D, FP32; small sets stay as stored (their kernels are bound by launches and latency); places are ints
    if (o.off || g->d.dims != 2 || g->d.precision != 32 || !order_pays(g, np, shape) || g->cells > INT32_MAX) return false;
    if (np <= o.cap && g->cells == o.cells) return true;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(g->stream, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) { cudaGetLastError(); return false; }
    // one allocation.  Earlier ones stay until order_free (a graph the caller
    // captured may refer to them); each is at least twice the one before, so all together hold at most twice the last.
    const int64_t n = std::max(np, 2 * o.cap);
    int* p = nullptr;
    if (cudaMalloc(&p, sizeof(int) * order_ints(g, n)) != cudaSuccess) { cudaGetLastError(); return false; }
    o.blocks.push_back(p);
    order_at(o, g, p, n);
    o.off = !order_clear(o);
    return !o.off;
}

hyb_status order_particles(Order& o, hyb_grid* g, const int32_t* cell, const float* off, int64_t np, Visit* v) {
    const int n1 = g->d.n1, n2 = g->d.n2;
    v->perm = o.perm;
    v->jumps = o.ctl;
    v->limit = (unsigned)kSamplePairs / 2;
    int sms = 0;
    HYB_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g->device));
    const int64_t all = (np + kOrderThreads - 1) / kOrderThreads, per = (int64_t)kOrderThreads * kScanCells;
    o.off = true;                                       // should a launch fail, the counts may be left half done
    const cudaStream_t s = o.side;
    HYB_CUDA_TRY(cudaEventRecord(o.fork, g->stream));
    HYB_CUDA_TRY(cudaStreamWaitEvent(s, o.fork, 0));
    k_count<<<(unsigned)std::min<int64_t>(all, 2 * sms), kOrderThreads, 0, s>>>(cell, off, np, n1, n2, o.count, o.ctl, v->limit);
    k_ranges<<<(unsigned)((g->cells + per - 1) / per), kOrderThreads, 0, s>>>(o.count, o.next, g->cells, o.ctl, *v);
    k_list<<<(unsigned)std::min<int64_t>(all, 4 * sms), kOrderThreads, 0, s>>>(cell, off, np, n1, n2, o.next, o.perm, *v);
    const cudaError_t e = cudaGetLastError();
    HYB_CUDA_TRY(cudaEventRecord(o.join, s));          // also of launches that failed: what was started is joined
    HYB_CUDA_TRY(e);
    o.off = false;
    return HYB_OK;
}

hyb_status order_listed(const Order& o, const hyb_grid* g, int* listed) {
    unsigned jumps = 0;
    HYB_CUDA_TRY(cudaMemcpyAsync(&jumps, o.ctl, sizeof(jumps), cudaMemcpyDeviceToHost, g->stream));
    HYB_CUDA_TRY(cudaStreamSynchronize(g->stream));
    *listed = jumps > (unsigned)kSamplePairs / 2;
    return HYB_OK;
}

hyb_status order_wait(const Order& o, hyb_grid* g, const Visit& v) {
    if (v.perm) HYB_CUDA_TRY(cudaStreamWaitEvent(g->stream, o.join, 0));
    return HYB_OK;
}

}  // namespace hyb
