// deposit.cu -- charge-conserving current deposit (Sec. 2.3) of particles that
// move from x^n to x^{n+1} within one step, in Esirkepov's density-
// decomposition form, which satisfies the finite-difference continuity
// equation (Eq. continuity) exactly:
//   2D: W1 = dS1 (S2^0 + S2^1)/2,  W2 = dS2 (S1^0 + S1^1)/2,
//       j1(i+1/2,j) = -q/(dt dx2) sum_{i'<=i} W1(i',j),
//       j2(i,j+1/2) = -q/(dt dx1) sum_{j'<=j} W2(i,j'),
//       j3(i,j) = q v3 [S1^0 S2^0/3 + S1^1 S2^0/6 + S1^0 S2^1/6 + S1^1 S2^1/3] / dV;
//   3D: W1 = dS1 (S2^0 S3^0 + dS2 S3^0/2 + S2^0 dS3/2 + dS2 dS3/3), cyclic for W2, W3,
//       j_a = -q/(dt dV/dx_a) cumulative sum of W_a along axis a.
// S are B-spline shape factors of order 1, 2 or 3 (grid points at integers).
// FP32 2D: a lane adds up a run of particles of one cell in registers (k_deposit2d_runs);
// otherwise one thread per particle adds its contributions with atomics.
#include <algorithm>
#include <type_traits>

#include "hyb_internal.cuh"

namespace hyb {

template <int ORDER, typename T>
__device__ __forceinline__ T bspline(T d) {
    T a = d < (T)0 ? -d : d;
    if (ORDER == 1) return a < (T)1 ? (T)1 - a : (T)0;
    if (ORDER == 2) {
        if (a <= (T)0.5) return (T)0.75 - a * a;
        if (a < (T)1.5) { T t = (T)1.5 - a; return (T)0.5 * t * t; }
        return (T)0;
    }
    if (a <= (T)1) return ((T)4 - (T)6 * a * a + (T)3 * a * a * a) * ((T)1 / (T)6);
    if (a < (T)2) { T t = (T)2 - a; return t * t * t * ((T)1 / (T)6); }
    return (T)0;
}

template <int ORDER> struct Win { static constexpr int lo = (ORDER == 1) ? -1 : -2; static constexpr int n = (ORDER == 1) ? 4 : 6; };

__device__ __forceinline__ int wrapi(int i, int n) { i %= n; return i < 0 ? i + n : i; }

constexpr int kDepThreads = 256;

// One particle's moves and 1D shapes: WN = ORDER + 2 consecutive points per axis from gx, gy (relative to
// the cell), outside which the shapes at x^n and at x^{n+1} (|x^{n+1} - x^n| < 1 cell) are zero and the
// cumulative sums are back to 0; the start is clamped into the full window LO .. LO + W - 1, which
// at a rounding edge only drops a point of weight 0.
template <typename T, int ORDER>
struct Move2d {
    static constexpr int WN = ORDER + 2;
    int gx, gy;
    T Sx0[WN], Sx1[WN], Sy0[WN], Sy1[WN];
    __device__ __forceinline__ void set(T x0, T x1, T y0, T y1) {
        constexpr int W = Win<ORDER>::n, LO = Win<ORDER>::lo;
        gx = min(max((int)floor((x0 < x1 ? x0 : x1) - (T)0.5 * (T)(ORDER + 1)) + 1, LO), LO + W - WN);
        gy = min(max((int)floor((y0 < y1 ? y0 : y1) - (T)0.5 * (T)(ORDER + 1)) + 1, LO), LO + W - WN);
#pragma unroll
        for (int w = 0; w < WN; w++) {
            const T px = (T)(gx + w), py = (T)(gy + w);
            Sx0[w] = bspline<ORDER>(x0 - px); Sx1[w] = bspline<ORDER>(x1 - px);
            Sy0[w] = bspline<ORDER>(y0 - py); Sy1[w] = bspline<ORDER>(y1 - py);
        }
    }
};
// the conditions on a particle (NaN offsets fail them); a particle that breaks them is skipped and flagged
template <typename T>
__device__ __forceinline__ bool move_ok(int cx, int cy, T x0, T x1, T y0, T y1, int n1, int n2) {
    const T dx = x1 - x0, dy = y1 - y0;
    return x0 >= (T)0 && x0 < (T)1 && y0 >= (T)0 && y0 < (T)1 && dx > (T)-1 && dx < (T)1 && dy > (T)-1 && dy < (T)1 &&
           cx >= 0 && cx < n1 && cy >= 0 && cy < n2;
}

// one particle, each contribution added with its own atomic
template <typename T, int ORDER>
__device__ __forceinline__ void deposit_one(T* J1, T* J2, T* J3, int n1, int n2, int cx, int cy, const Move2d<T, ORDER>& m, T c1, T c2,
                                            T c3) {
    constexpr int WN = ORDER + 2;
    T* const Jc[3] = {J1, J2, J3};
    int col[WN];
    int64_t row[WN];
#pragma unroll
    for (int w = 0; w < WN; w++) { col[w] = wrapi(cx + m.gx + w, n1); row[w] = (int64_t)wrapi(cy + m.gy + w, n2) * n1; }
    auto add = [&](int c, int i, int j, T v) { atomicAdd(Jc[c] + row[j] + col[i], v); };
#pragma unroll
    for (int j = 0; j < WN; j++) {
        const T sy = (T)0.5 * (m.Sy0[j] + m.Sy1[j]);
        if (sy == (T)0) continue;
        T acc = (T)0;
#pragma unroll
        for (int i = 0; i < WN; i++) {
            acc += (m.Sx1[i] - m.Sx0[i]) * sy;
            if (acc != (T)0) add(0, i, j, c1 * acc);
        }
    }
#pragma unroll
    for (int i = 0; i < WN; i++) {
        const T sx = (T)0.5 * (m.Sx0[i] + m.Sx1[i]);
        if (sx == (T)0) continue;
        T acc = (T)0;
#pragma unroll
        for (int j = 0; j < WN; j++) {
            acc += (m.Sy1[j] - m.Sy0[j]) * sx;
            if (acc != (T)0) add(1, i, j, c2 * acc);
        }
    }
    if (c3 != (T)0) {
        // S1^0 S2^0/3 + S1^1 S2^0/6 + S1^0 S2^1/6 + S1^1 S2^1/3 = S1^0 a_j + S1^1 b_j
#pragma unroll
        for (int j = 0; j < WN; j++) {
            const T aj = (m.Sy0[j] + m.Sy0[j] + m.Sy1[j]) * ((T)1 / (T)6), bj = (m.Sy0[j] + m.Sy1[j] + m.Sy1[j]) * ((T)1 / (T)6);
#pragma unroll
            for (int i = 0; i < WN; i++) {
                const T w3 = m.Sx0[i] * aj + m.Sx1[i] * bj;
                if (w3 != (T)0) add(2, i, j, c3 * w3);
            }
        }
    }
}

// 2D, one thread per particle (FP64): lanes take particles BS / 32 apart within each chunk of BS, so
// that for a sorted chunk the lanes of a warp sit in different (mostly consecutive) cells and their
// atomic adds at the same window offset go to different, neighbouring addresses.
template <typename T, int ORDER, bool VISIT>
__global__ void __launch_bounds__(kDepThreads) k_deposit2d(T* __restrict__ J1, T* __restrict__ J2, T* __restrict__ J3,
                                                          int n1, int n2, const int32_t* __restrict__ cell,
                                                          const T* __restrict__ off0, const T* __restrict__ off1,
                                                          const T* __restrict__ v3, const T* __restrict__ q, int64_t np,
                                                          T c1s, T c2s, T c3s, int* __restrict__ flag, Visit visit) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int* const perm = VISIT ? visit_perm(visit) : nullptr;
    for (int64_t base = blockIdx.x * (int64_t)blockDim.x; base < np; base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = base + lane * (int)(blockDim.x >> 5) + warp;
        if (i >= np) continue;
        const int64_t p = visit_at(perm, i);
        const int cx = cell[2 * p], cy = cell[2 * p + 1];
        const T x0 = off0[2 * p], y0 = off0[2 * p + 1], x1 = off1[2 * p], y1 = off1[2 * p + 1];
        if (!move_ok(cx, cy, x0, x1, y0, y1, n1, n2)) {
            atomicOr(flag, 1);
            continue;
        }
        Move2d<T, ORDER> m;
        m.set(x0, x1, y0, y1);
        const T qp = q[p];
        deposit_one<T, ORDER>(J1, J2, J3, n1, n2, cx, cy, m, c1s * qp, c2s * qp, v3 ? c3s * qp * v3[p] : (T)0);
    }
}

// FP32 2D.  Bound before: one atomic per particle, point and component, 48 at order 2, at the L2's rate of
// about 155 G sectors/s when they scatter and 110 G when a warp's are consecutive (measured): 5.1 ms for
// the 67 M particles of the drifting plasma, 1.5 ms now.  Every current is a sum of products of a function of x1 and one of x2,
//   j1 = c1 P1(i) sy(j), j2 = sx(i) c2 P2(j), j3 = S1^0(i) c3 a(j) + S1^1(i) c3 b(j)
// (P the cumulative sum of dS, s = (S^0 + S^1)/2), and particles stored in cell order come in runs of one
// cell, whose functions all fit the same N x N window, N = ORDER + 3 points.  A warp therefore cuts
// its particles into runs and gives each lane one: the lane adds its run's particles in registers and
// only then touches memory.  When the 32 cells are consecutive, each row of the window is first
// summed across the lanes (shuffles), so that a row of 32 + N - 1 points takes two atomics of the warp;
// otherwise each lane adds its window, one atomic per point, neighbouring lanes to neighbouring addresses.
// Where that would touch more sectors than the particles one by one (runs too short and
// scattered), each lane adds one particle's points on its own.
// (Also tried: the particles' functions in shared memory and a lane per window point, for any order of
// particles: 3.7 ms, bound by the shared-memory reads, 10 wavefronts per particle; scattered
// particles' rows as aligned quads with red.v4: 0.24 against 0.20 ms for 1 M particles.)
// The shapes S^0 (x0 in [0, 1)) and S^1 (x1) at the N points of a window from B0, for a particle whose own
// points lie in it: bspline()'s values, bit for bit (the last product of a piece is rounded on its own: the
// differences dS of a cold plasma's moves are a few units of it), with only the pieces that each point can need.
template <int ORDER>
__device__ __forceinline__ float spline_in(float a) {       // |d| = a below the first knot
    if (ORDER == 1) return 1.f - a;
    if (ORDER == 2) return 0.75f - a * a;
    return __fmul_rn(4.f - 6.f * a * a + 3.f * a * a * a, 1.f / 6.f);
}
template <int ORDER>
__device__ __forceinline__ float spline_out(float a) {      // above it
    if (ORDER == 1) return 0.f;
    if (ORDER == 2) { const float t = fmaxf(1.5f - a, 0.f); return __fmul_rn(0.5f * t, t); }
    const float t = fmaxf(2.f - a, 0.f);
    return __fmul_rn(t * t * t, 1.f / 6.f);
}
template <int ORDER>
__device__ __forceinline__ float spline_any(float d) {
    const float a = fabsf(d);
    if (ORDER == 1) return fmaxf(1.f - a, 0.f);
    return a <= (ORDER == 2 ? 0.5f : 1.f) ? spline_in<ORDER>(a) : spline_out<ORDER>(a);
}
template <int ORDER>
__device__ __forceinline__ void window_shapes(float x0, float x1, float (&S0)[ORDER + 3], float (&S1)[ORDER + 3]) {
    if constexpr (ORDER == 1) {                              // points -1 .. 2, x1 in (-1, 2)
        S0[0] = 0.f; S0[1] = spline_in<1>(x0); S0[2] = spline_in<1>(fabsf(x0 - 1.f)); S0[3] = 0.f;
#pragma unroll
        for (int e = 0; e < 4; e++) S1[e] = spline_any<1>(x1 - (float)(e - 1));
    } else if constexpr (ORDER == 2) {                       // points -1 .. 3, x1 in [-1/2, 2)
        S0[0] = spline_out<2>(x0 + 1.f); S0[1] = spline_any<2>(x0); S0[2] = spline_any<2>(x0 - 1.f); S0[3] = spline_out<2>(2.f - x0); S0[4] = 0.f;
        S1[0] = spline_out<2>(x1 + 1.f);
#pragma unroll
        for (int e = 1; e < 4; e++) S1[e] = spline_any<2>(x1 - (float)(e - 1));
        S1[4] = spline_out<2>(3.f - x1);
    } else {                                                 // points -2 .. 3, x1 in (-1, 2)
        S0[0] = 0.f; S0[1] = spline_out<3>(x0 + 1.f); S0[2] = spline_in<3>(x0); S0[3] = spline_in<3>(fabsf(x0 - 1.f));
        S0[4] = spline_out<3>(2.f - x0); S0[5] = 0.f;
        S1[0] = spline_out<3>(x1 + 2.f);
#pragma unroll
        for (int e = 1; e < 5; e++) S1[e] = spline_any<3>(x1 - (float)(e - 2));
        S1[5] = spline_out<3>(3.f - x1);
    }
}

// one particle on its own (kept out of line: rare in the run kernel)
template <int ORDER>
__device__ __noinline__ void deposit_alone(float* J1, float* J2, float* J3, int n1, int n2, int2 cc, float2 o0, float2 o1, float c1,
                                           float c2, float c3) {
    Move2d<float, ORDER> m;
    m.set(o0.x, o1.x, o0.y, o1.y);
    deposit_one<float, ORDER>(J1, J2, J3, n1, n2, cc.x, cc.y, m, c1, c2, c3);
}

constexpr int kRunWarps = 4, kRunScan = 512;      // warps per block; particles looked at for 32 runs
constexpr int kRunMax = 32;                       // a longer run is cut (at multiples of this many particles)
// Particles taken one by one where there are no runs.  32 at a time, with 64 cells looked at before each, 2 M shuffled particles
// (1024 x 512, order 2) took 388 us; 361 now, 335 with a thread per particle and no runs looked for.
constexpr int kAlone = 256;

// warps below `full` take `per` particles each, the others `fine`
struct RunSplit { int64_t per, full, fine; };

template <int ORDER, bool VISIT>
__global__ void __launch_bounds__(32 * kRunWarps, ORDER == 3 ? 3 : 4)
k_deposit2d_runs(float* __restrict__ J1, float* __restrict__ J2, float* __restrict__ J3, int n1, int n2,
                 const int2* __restrict__ cell, const float2* __restrict__ off0, const float2* __restrict__ off1,
                 const float* __restrict__ v3, const float* __restrict__ q, int64_t np, const __grid_constant__ RunSplit split, float c1s, float c2s,
                 float c3s, int* __restrict__ flag, Visit visit) {
    constexpr int WN = ORDER + 2, N = ORDER + 3, B0 = ORDER == 3 ? -2 : -1;
    __shared__ int s_start[kRunWarps][64];       // at most 32 + 32 heads
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int* const start = s_start[warp];
    const int* const perm = VISIT ? visit_perm(visit) : nullptr;
    const int64_t w = (int64_t)blockIdx.x * kRunWarps + warp, mine = w < split.full ? split.per : split.fine;
    const int64_t first = w < split.full ? w * split.per : split.full * split.per + (w - split.full) * split.fine;
    const int64_t last = first + mine < np ? first + mine : np;
    int64_t base = first;
    while (base < last) {
        // ---- the next runs: places (from base) where the cell changes or a multiple of kRunMax begins
        int nr = 0, seen = 0;
        const int avail = (int)(last - base < kRunScan ? last - base : kRunScan);
        int2 carry = make_int2(0, 0);
        while (seen < avail && nr <= 32) {
            const int i = seen + lane;
            const int2 c = i < avail ? cell[visit_at(perm, base + i)] : make_int2(0, 0);
            {   // the rest of these particles into L2: two 128-byte lines of either offset array, one of q and v3
                const int64_t g = base + seen + (lane & 1) * 16;
                const void* line = lane < 2 ? (const void*)(off0 + g) : lane < 4 ? (const void*)(off1 + g)
                                   : lane == 4 ? (const void*)(q + g) : (const void*)(v3 + g);
                if (!perm && g < last && lane < (v3 ? 7 : 5) && lane != 5) asm volatile("prefetch.global.L2 [%0];" :: "l"(line));
            }
            int2 pc = make_int2(__shfl_up_sync(0xffffffffu, c.x, 1), __shfl_up_sync(0xffffffffu, c.y, 1));
            if (lane == 0) pc = carry;
            const bool head = i < avail && (i == 0 || c.x != pc.x || c.y != pc.y || ((base + i) & (kRunMax - 1)) == 0);
            const unsigned h = __ballot_sync(0xffffffffu, head);
            if (head) start[nr + __popc(h & ((1u << lane) - 1u))] = i;
            nr += __popc(h);
            carry = make_int2(__shfl_sync(0xffffffffu, c.x, 31), __shfl_sync(0xffffffffu, c.y, 31));
            seen += 32;
        }
        __syncwarp();
        const int runs = min(nr, 32);
        int end = nr > 32 ? start[32] : min(seen, avail);                   // particles of these runs
        const int s0 = lane < runs ? start[lane] : end, s1 = lane + 1 < runs ? start[lane + 1] : end;
        const int2 cc = lane < runs ? cell[visit_at(perm, base + s0)] : make_int2(-1, -1);
        const bool inside = cc.x >= 0 && cc.x < n1 && cc.y >= 0 && cc.y < n2;
        __syncwarp();
        // ---- which way: consecutive cells of a row; else by the sectors touched
        const int2 c0 = make_int2(__shfl_sync(0xffffffffu, cc.x, 0), __shfl_sync(0xffffffffu, cc.y, 0));
        const bool row = __all_sync(0xffffffffu, inside && cc.y == c0.y && cc.x == c0.x + lane);
        const int2 left = make_int2(__shfl_up_sync(0xffffffffu, cc.x, 1), __shfl_up_sync(0xffffffffu, cc.y, 1));
        const int sectors = __popc(__ballot_sync(0xffffffffu, lane < runs && (lane == 0 || left.y != cc.y || (left.x >> 3) != (cc.x >> 3))));
        if (row || N * N * sectors <= WN * WN * end) {
            float a1[N][N], a2[N][N], a3[N][N];
#pragma unroll
            for (int j = 0; j < N; j++)
#pragma unroll
                for (int i = 0; i < N; i++) a1[j][i] = a2[j][i] = a3[j][i] = 0.f;
            float2 n0 = make_float2(0.f, 0.f), nw = n0;
            float nq = 0.f, nv = 0.f;
            int nat = VISIT && perm && s0 < s1 ? perm[base + s0] : 0;      // a listed particle's place, one fetch ahead
            auto fetch = [&](int i) {
                if (i < s1) {
                    const int64_t p = VISIT && perm ? (int64_t)nat : base + i;
                    if (VISIT && perm && i + 1 < s1) nat = perm[base + i + 1];
                    n0 = off0[p];
                    nw = off1[p];
                    nq = q[p];
                    nv = v3 ? v3[p] : 0.f;
                }
            };
            fetch(s0);
            const int longest = __reduce_max_sync(0xffffffffu, s1 - s0);
            for (int t = 0; t < longest; t++) {
                const bool here = s0 + t < s1;
                const float2 o0 = n0, o1 = nw;
                const float qp = nq, vp = nv;
                fetch(s0 + t + 1);
                if (!here) continue;
                if (!move_ok(cc.x, cc.y, o0.x, o1.x, o0.y, o1.y, n1, n2)) {
                    atomicOr(flag, 1);
                    continue;
                }
                const float c1 = c1s * qp, c2 = c2s * qp, c3 = c3s * qp * vp;
                const float lx = o0.x < o1.x ? o0.x : o1.x, ly = o0.y < o1.y ? o0.y : o1.y;
                // the first of the particle's own WN points, from the window's first
                const int ox = (int)floorf(lx - 0.5f * (float)(ORDER + 1)) + 1 - B0, oy = (int)floorf(ly - 0.5f * (float)(ORDER + 1)) + 1 - B0;
                // an order-2 particle that moves back by more than half a cell leaves the window, and 0 times a
                // non-finite charge would spread over it: such a particle on its own (without v3 it has no j3, infinite or not)
                if (ox < 0 || oy < 0 || !(isfinite(c1) && isfinite(c2) && isfinite(c3))) {
                    deposit_alone<ORDER>(J1, J2, J3, n1, n2, cc, o0, o1, c1, c2, v3 ? c3 : 0.f);
                    continue;
                }
                float Sx0[N], Sx1[N], Sy0[N], Sy1[N], p1[N], sx[N];
                window_shapes<ORDER>(o0.x, o1.x, Sx0, Sx1);
                window_shapes<ORDER>(o0.y, o1.y, Sy0, Sy1);
                float p = 0.f;
#pragma unroll
                for (int e = 0; e < N; e++) {
                    p += Sx1[e] - Sx0[e];
                    p1[e] = c1 * p;
                    sx[e] = 0.5f * (Sx0[e] + Sx1[e]);
                }
                if (ox == 0) p1[N - 1] = 0.f;            // past the particle's own points the sum is back to 0
                p = 0.f;
#pragma unroll
                for (int e = 0; e < N; e++) {
                    const float y0 = Sy0[e], y1 = Sy1[e];
                    p += y1 - y0;
                    const float sy = 0.5f * (y0 + y1), p2 = e == N - 1 && oy == 0 ? 0.f : c2 * p;
                    const float a = c3 * ((y0 + y0 + y1) * (1.f / 6.f)), b = c3 * ((y0 + y1 + y1) * (1.f / 6.f));
#pragma unroll
                    for (int i = 0; i < N; i++) {
                        a1[e][i] = fmaf(p1[i], sy, a1[e][i]);
                        a2[e][i] = fmaf(sx[i], p2, a2[e][i]);
                        a3[e][i] = fmaf(Sx0[i], a, fmaf(Sx1[i], b, a3[e][i]));
                    }
                }
            }
            if (row) {
                // column c0.x + B0 + lane gets point i of lane - i; the last lanes' points beyond lane 31
                // come round to the first lanes (tail)
                const int col = (c0.x + B0 + lane) & (n1 - 1), tcol = (c0.x + B0 + 32 + lane) & (n1 - 1);
                auto rowsum = [&](const float (&v)[N], float* J) {
                    float s = v[0], tail = 0.f;
#pragma unroll
                    for (int i = 1; i < N; i++) {
                        const float o = __shfl_sync(0xffffffffu, v[i], (lane - i) & 31);
                        s += lane >= i ? o : 0.f;
                        tail += lane >= i ? 0.f : o;
                    }
                    if (s != 0.f) atomicAdd(J + col, s);
                    if (lane < N - 1 && tail != 0.f) atomicAdd(J + tcol, tail);
                };
#pragma unroll
                for (int j = 0; j < N; j++) {
                    const int64_t at = (int64_t)wrapi(c0.y + B0 + j, n2) * n1;
                    rowsum(a1[j], J1 + at);
                    rowsum(a2[j], J2 + at);
                    rowsum(a3[j], J3 + at);
                }
            } else if (inside) {
                int col[N];
#pragma unroll
                for (int i = 0; i < N; i++) col[i] = (cc.x + B0 + i) & (n1 - 1);
#pragma unroll
                for (int j = 0; j < N; j++) {
                    const int64_t at = (int64_t)wrapi(cc.y + B0 + j, n2) * n1;
#pragma unroll
                    for (int i = 0; i < N; i++) {
                        if (a1[j][i] != 0.f) atomicAdd(J1 + at + col[i], a1[j][i]);
                        if (a2[j][i] != 0.f) atomicAdd(J2 + at + col[i], a2[j][i]);
                        if (a3[j][i] != 0.f) atomicAdd(J3 + at + col[i], a3[j][i]);
                    }
                }
            }
        } else {
            // ---- scattered: a particle per lane, kAlone of them before looking for runs again (asking for the next particle's
            // data ahead was worth 2 % of this, and its registers cost the runs as much)
            if (end > 32) end &= ~31;                                // whole warps; the rest in the next round
            end = max(end, (int)min((int64_t)kAlone, last - base));
            for (int i = lane; i < end; i += 32) {
                const int64_t p = visit_at(perm, base + i);
                const int2 pc = cell[p];
                const float2 o0 = off0[p], o1 = off1[p];
                if (!move_ok(pc.x, pc.y, o0.x, o1.x, o0.y, o1.y, n1, n2)) {
                    atomicOr(flag, 1);
                    continue;
                }
                const float qp = q[p];
                deposit_alone<ORDER>(J1, J2, J3, n1, n2, pc, o0, o1, c1s * qp, c2s * qp, v3 ? c3s * qp * v3[p] : 0.f);
            }
        }
        base += end;
    }
}

template <typename T, int ORDER>
__global__ void k_deposit3d(T* __restrict__ J1, T* __restrict__ J2, T* __restrict__ J3, int n1, int n2, int n3,
                            const int32_t* __restrict__ cell, const T* __restrict__ off0, const T* __restrict__ off1,
                            const T* __restrict__ q, int64_t np, T c1s, T c2s, T c3s, int* __restrict__ flag) {
    constexpr int W = Win<ORDER>::n, LO = Win<ORDER>::lo;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < np; p += (int64_t)gridDim.x * blockDim.x) {
        int c[3];
        T a0[3], a1[3];
        bool ok = true;
        const int ext[3] = {n1, n2, n3};
#pragma unroll
        for (int a = 0; a < 3; a++) {
            c[a] = cell[3 * p + a];
            a0[a] = off0[3 * p + a];
            a1[a] = off1[3 * p + a];
            const T d = a1[a] - a0[a];
            ok = ok && a0[a] >= (T)0 && a0[a] < (T)1 && d > (T)-1 && d < (T)1 && c[a] >= 0 && c[a] < ext[a];
        }
        if (!ok) { atomicOr(flag, 1); continue; }
        T S0[3][W], dS[3][W];
        int idx[3][W];
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int w = 0; w < W; w++) {
                const T gp = (T)(w + LO);
                S0[a][w] = bspline<ORDER>(a0[a] - gp);
                dS[a][w] = bspline<ORDER>(a1[a] - gp) - S0[a][w];
                idx[a][w] = wrapi(c[a] + LO + w, ext[a]);
            }
        const T qp = q[p];
        const T cc[3] = {c1s * qp, c2s * qp, c3s * qp};
        T* Jd[3] = {J1, J2, J3};
        // component a accumulates along axis a; (b, c) are the two transverse axes
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const int b = (a + 1) % 3, e = (a + 2) % 3;
            for (int u = 0; u < W; u++)
                for (int v = 0; v < W; v++) {
                    const T tw = S0[b][u] * S0[e][v] + (T)0.5 * dS[b][u] * S0[e][v] + (T)0.5 * S0[b][u] * dS[e][v]
                               + dS[b][u] * dS[e][v] * ((T)1 / (T)3);
                    if (tw == (T)0) continue;
                    T acc = (T)0;
                    for (int i = 0; i < W; i++) {
                        acc += dS[a][i] * tw;
                        if (acc == (T)0) continue;
                        int ii[3];
                        ii[a] = idx[a][i]; ii[b] = idx[b][u]; ii[e] = idx[e][v];
                        atomicAdd(Jd[a] + ((int64_t)ii[2] * n2 + ii[1]) * n1 + ii[0], cc[a] * acc);
                    }
                }
        }
    }
}

__global__ void k_zero3(uint4* __restrict__ a, uint4* __restrict__ b, uint4* __restrict__ c, int64_t n) {
    uint4* const p = blockIdx.y == 0 ? a : blockIdx.y == 1 ? b : c;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) p[i] = make_uint4(0u, 0u, 0u, 0u);
}

template <int ORDER>
static cudaError_t launch_runs(hyb_grid* g, float* J1, float* J2, float* J3, const int32_t* cell, const float* off_old,
                               const float* off_new, const float* v3, const float* q, int64_t np, float c1, float c2, float c3, const Visit& visit) {
    const auto kern = visit.perm ? k_deposit2d_runs<ORDER, true> : k_deposit2d_runs<ORDER, false>;
    // A contiguous range of particles per warp: 256 or a multiple of it, four waves of resident blocks.  A call that would leave
    // resident warps idle that way (up to 160 particles for each of them) spreads over all of them, down to 32 particles a
    // warp; over a quarter of them where that leaves a warp some 16 cells' worth, which still makes runs.  8192 particles of a
    // 256 x 256 grid, order 1, 2, 3: 12, 12, 12 us; 256 to a warp, one after another, 27, 41, 51 us; one thread per particle 19,
    // 23, 25.  With 192 to a warp already (400000 particles) ranges of 256 are faster again, 35 against 37 us.
    const int64_t warps = (int64_t)resident_grid((const void*)kern, 32 * kRunWarps, 0) * kRunWarps;
    const int64_t even = (np + warps - 1) / warps;
    int64_t per = ((np + 4 * warps - 1) / (4 * warps) + 255) / 256 * 256;
    if (even <= 160) per = std::min<int64_t>(256, (std::max(even, std::min<int64_t>(16 * np / g->cells, 4 * even)) + 31) / 32 * 32);
    // Up to 1.4 waves of 256: one wave of longer ranges (the second would be nearly empty; order 3, 614400 particles of a 1024 x
    // 300 grid, in cell order 74 -> 58 us, shuffled 222 -> 184).  Ranges longer than 256: half a wave's worth at the end in
    // halves, so that the last wave ends evenly (2 M, 1024 x 512, order 3, in cell order 193 -> 172 us, shuffled 696 -> 555; 4 M,
    // order 2, 216 -> 208 and 691 -> 685), as long as those hold 16 cells' worth: ranges of 256 in halves make too few runs of 16
    // particles per cell (31 -> 39 us), ranges of 512 of 38 (256 x 256, order 2, 2.5 M, 101 -> 111).  Beyond 4096 the last wave
    // is short against the rest (67 M: 1543 us whole, 1550 with halves).
    else if (even > 256 && 10 * np <= 14 * 256 * warps) per = (even + 31) / 32 * 32;
    RunSplit split{per, (np + per - 1) / per, per};
    int64_t all = split.full;
    if (per > 256 && per <= 4096 && 10 * np > 14 * 256 * warps) {
        split.fine = std::min(per, std::max<int64_t>({256, per / 2, 16 * np / g->cells}));
        split.full = (np - std::min(np / 2, warps * per / 2)) / per;
        all = split.full + (np - split.full * per + split.fine - 1) / split.fine;
    }
    const unsigned blocks = (unsigned)((all + kRunWarps - 1) / kRunWarps);
    kern<<<blocks, 32 * kRunWarps, 0, g->stream>>>(J1, J2, J3, g->d.n1, g->d.n2, reinterpret_cast<const int2*>(cell),
                                                   reinterpret_cast<const float2*>(off_old),
                                                   reinterpret_cast<const float2*>(off_new), v3, q, np, split, c1, c2, c3, g->dflag, visit);
    return cudaGetLastError();
}

template <typename T>
hyb_status deposit(hyb_grid* g, const int32_t* cell, const T* off_old, const T* off_new, const T* v3, const T* q,
                   int64_t np, int order, Visit visit) {
    const hyb_grid_desc& d = g->d;
    int dev_sms = 0;
    cudaDeviceGetAttribute(&dev_sms, cudaDevAttrMultiProcessorCount, g->device);
    {   // one launch for the three arrays (16-byte aligned, a whole number of 16-byte words: n1 >= 8)
        const int64_t n = g->cells * (int64_t)sizeof(T) / 16;
        const unsigned blocks = (unsigned)std::min<int64_t>((n + 255) / 256, (int64_t)dev_sms * 8);
        k_zero3<<<dim3(blocks, 3), 256, 0, g->stream>>>((uint4*)g->J[0], (uint4*)g->J[1], (uint4*)g->J[2], n);
        HYB_CUDA_TRY(cudaGetLastError());
    }
    if (np == 0) return HYB_OK;
    T* J1 = (T*)g->J[0]; T* J2 = (T*)g->J[1]; T* J3 = (T*)g->J[2];
    if (d.dims == 2) {
        const T c1 = (T)(-1.0 / (d.dt * d.dx2)), c2 = (T)(-1.0 / (d.dt * d.dx1)), c3 = (T)(1.0 / (d.dx1 * d.dx2));
        // the run kernel reads a particle's pairs at once
        const bool pairs = ((((uintptr_t)cell | (uintptr_t)off_old | (uintptr_t)off_new) & 7) == 0);
        if constexpr (std::is_same<T, float>::value) {
            if (pairs) {
#define HYB_DEPR(O) HYB_CUDA_TRY((launch_runs<O>(g, J1, J2, J3, cell, off_old, off_new, v3, q, np, c1, c2, c3, visit)))
                if (order == 1) HYB_DEPR(1); else if (order == 2) HYB_DEPR(2); else HYB_DEPR(3);
#undef HYB_DEPR
                return HYB_OK;
            }
        }
        // small calls: smaller blocks, so that the particles spread over the SMs
        int threads = kDepThreads;
        while (threads > 32 && np < (int64_t)threads * dev_sms) threads >>= 1;
        const unsigned blocks = (unsigned)std::min<int64_t>((np + threads - 1) / threads, (int64_t)dev_sms * 32);
#define HYB_DEP2(O) (visit.perm ? k_deposit2d<T, O, sizeof(T) == 4> : k_deposit2d<T, O, false>)<<<blocks, threads, 0, g->stream>>>(J1, J2, J3, d.n1, d.n2, cell, off_old, off_new, v3, q, np, c1, c2, c3, g->dflag, visit)
        if (order == 1) HYB_DEP2(1); else if (order == 2) HYB_DEP2(2); else HYB_DEP2(3);
#undef HYB_DEP2
    } else {
        const int threads = kDepThreads;
        const unsigned blocks = (unsigned)std::min<int64_t>((np + threads - 1) / threads, (int64_t)dev_sms * 32);
        const T c1 = (T)(-1.0 / (d.dt * d.dx2 * d.dx3)), c2 = (T)(-1.0 / (d.dt * d.dx1 * d.dx3)), c3 = (T)(-1.0 / (d.dt * d.dx1 * d.dx2));
#define HYB_DEP3(O) k_deposit3d<T, O><<<blocks, threads, 0, g->stream>>>(J1, J2, J3, d.n1, d.n2, d.n3, cell, off_old, off_new, q, np, c1, c2, c3, g->dflag)
        if (order == 1) HYB_DEP3(1); else if (order == 2) HYB_DEP3(2); else HYB_DEP3(3);
#undef HYB_DEP3
    }
    HYB_CUDA_TRY(cudaGetLastError());
    return HYB_OK;
}

template hyb_status deposit<float>(hyb_grid*, const int32_t*, const float*, const float*, const float*, const float*, int64_t, int, Visit);
template hyb_status deposit<double>(hyb_grid*, const int32_t*, const double*, const double*, const double*, const double*, int64_t, int, Visit);

}  // namespace hyb
