// order.cu -- cell order of scattered particles.  The particle kernels are fast when consecutive
// particles share cells (fields staged once per block, currents summed in registers); after some
// hundred steps of a run they no longer do, since nothing moves the caller's particles in memory.  A PIC step
// therefore lists them cell by cell and visits them through that list: counts per cell, a range of the
// list for each cell, the list (each particle takes its cell's next place).  FP32 only: in FP64 the push and the
// deposit are bound by their arithmetic and atomics in any order (1 M shuffled particles, 512 x 256, order 2: a step of
// 1319 us as stored, 1394 listed).
//
// Whether that pays is decided on the device: k_jumps looks at 16384 pairs of consecutive
// particles; when at most half of them leave the cell and its right neighbour, the particles are in order and
// the other kernels return at once.  1 M particles of the 256 x 256 box after 1500 steps: push 113 -> 79
// and deposit 203 -> 76 us (a listed particle's loads and stores are scattered) for 37 us of listing; in order the four
// launches cost 15 us.
#include <algorithm>

#include "hyb_internal.cuh"

namespace hyb {

constexpr int kOrderThreads = 256;
// particles from which the list is made: it takes about 20 us whatever their number, and saves 160 us of the push and deposit of
// 1 M particles at shape order 2 (67584 of them lost: 79 -> 96 us per step; 118784 at order 3 gained: 161 -> 99)
constexpr int kOrderMin = 1 << 17;
static int64_t order_min(int shape) { return shape == 1 ? 2 * kOrderMin : shape == 2 ? kOrderMin : kOrderMin / 4 * 3; }
constexpr int kSamplePairs = 1 << 14;
constexpr int kScanCells = 4;                       // cells per thread of k_ranges

// the cell that holds a particle (its offsets may lie in [-1, 2)); 0 for one the push will reject
__device__ __forceinline__ int particle_key(const int32_t* __restrict__ cell, const float* __restrict__ off, int64_t p, int n1, int n2) {
    int cx = cell[2 * p], cy = cell[2 * p + 1];
    float ox = off[2 * p], oy = off[2 * p + 1];
    if (cx < 0 || cx >= n1 || cy < 0 || cy >= n2 || !renormalise(cx, ox, n1) || !renormalise(cy, oy, n2)) return 0;
    return cy * n1 + cx;
}

__global__ void __launch_bounds__(kOrderThreads) k_jumps(const int32_t* __restrict__ cell, const float* __restrict__ off, int64_t np, int n1,
                                                         int n2, int pairs, unsigned* __restrict__ ctl) {
    const int i = blockIdx.x * kOrderThreads + threadIdx.x;
    bool jump = false;
    if (i < pairs) {
        const int64_t p = (np - 1) * (int64_t)i / pairs;
        const int a = particle_key(cell, off, p, n1, n2), b = particle_key(cell, off, p + 1, n1, n2);
        jump = b != a && b != a + 1;
    }
    const int n = __syncthreads_count(jump);
    if (threadIdx.x == 0 && n) atomicAdd(ctl, (unsigned)n);
}

__global__ void __launch_bounds__(kOrderThreads) k_count(const int32_t* __restrict__ cell, const float* __restrict__ off, int64_t np, int n1,
                                                         int n2, int* __restrict__ count, Visit v) {
    if (!visit_perm(v)) return;
    for (int64_t p = blockIdx.x * (int64_t)kOrderThreads + threadIdx.x; p < np; p += (int64_t)gridDim.x * kOrderThreads)
        atomicAdd(count + particle_key(cell, off, p, n1, n2), 1);
}

// count -> first place of the cell in the list.  A block's cells share a range taken from the cursor, so the
// order of the ranges is that in which the blocks get there (no block waits for another).
__global__ void __launch_bounds__(kOrderThreads) k_ranges(int* __restrict__ count, int64_t cells, unsigned* __restrict__ ctl, Visit v) {
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
        if (c0 + e < cells) count[c0 + e] = at;
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
    for (void* p : o.blocks) cudaFree(p);
    o = Order();
}

static void order_at(Order& o, const hyb_grid* g, int* p, int64_t n) {
    o.ctl = reinterpret_cast<unsigned*>(p);
    o.count = p + 4;
    o.perm = o.count + g->cells;
    o.cap = n;
    o.cells = g->cells;
}
// A first list beside the step's scratch: 32 particles per cell, at most 16 MB (an allocation inside the first step
// cost it 50 us, half its time on a grid of this size); none for sets that stay as stored
static int64_t order_first(const hyb_grid* g) {
    const int64_t n = std::min<int64_t>(32 * (int64_t)g->cells, 1 << 22);
    return g->d.dims == 2 && g->d.precision == 32 && g->cells <= 1 << 20 && n >= kOrderMin ? n : 0;
}
size_t order_bytes(const hyb_grid* g) {
    const int64_t n = order_first(g);
    return n ? sizeof(int) * (size_t)(4 + g->cells + n) : 0;
}
void order_place(Order& o, const hyb_grid* g, void* at) { order_at(o, g, reinterpret_cast<int*>(at), order_first(g)); }

bool order_reserve(Order& o, const hyb_grid* g, int64_t np, int shape) {
    // 2D, FP32; small sets stay as stored (their kernels are bound by launches and latency); places are ints
    if (g->d.dims != 2 || g->d.precision != 32 || np < order_min(shape) || np > INT32_MAX || g->cells > INT32_MAX) return false;
    if (np <= o.cap && g->cells == o.cells) return true;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(g->stream, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) { cudaGetLastError(); return false; }
    // one allocation: control words, counts, list.  Earlier ones stay until order_free (a graph the caller
    // captured may refer to them); each is at least twice the one before, so all together hold at most twice the last.
    const int64_t n = std::max(np, 2 * o.cap);
    int* p = nullptr;
    if (cudaMalloc(&p, sizeof(int) * (size_t)(4 + g->cells + n)) != cudaSuccess) { cudaGetLastError(); return false; }
    o.blocks.push_back(p);
    order_at(o, g, p, n);
    return true;
}

hyb_status order_particles(Order& o, hyb_grid* g, const int32_t* cell, const float* off, int64_t np, Visit* v) {
    const int n1 = g->d.n1, n2 = g->d.n2, pairs = kSamplePairs;
    v->perm = o.perm;
    v->jumps = o.ctl;
    v->limit = (unsigned)pairs / 2;
    int sms = 0;
    HYB_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g->device));
    const unsigned blocks = (unsigned)std::min<int64_t>((np + kOrderThreads - 1) / kOrderThreads, (int64_t)sms * 16);
    const int64_t per = (int64_t)kOrderThreads * kScanCells;
    HYB_CUDA_TRY(cudaMemsetAsync(o.ctl, 0, sizeof(int) * (size_t)(4 + g->cells), g->stream));      // and the counts after it
    k_jumps<<<(pairs + kOrderThreads - 1) / kOrderThreads, kOrderThreads, 0, g->stream>>>(cell, off, np, n1, n2, pairs, o.ctl);
    k_count<<<blocks, kOrderThreads, 0, g->stream>>>(cell, off, np, n1, n2, o.count, *v);
    k_ranges<<<(unsigned)((g->cells + per - 1) / per), kOrderThreads, 0, g->stream>>>(o.count, g->cells, o.ctl, *v);
    k_list<<<blocks, kOrderThreads, 0, g->stream>>>(cell, off, np, n1, n2, o.count, o.perm, *v);
    HYB_CUDA_TRY(cudaGetLastError());
    return HYB_OK;
}

}  // namespace hyb
