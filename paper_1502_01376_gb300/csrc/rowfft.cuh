// rowfft.cuh -- register-resident real row transforms: the complex FFT of M = n1/2 points, z[j] = x[2j] + i
// x[2j+1], by a team of TT = M/P threads that hold P points each (8 or 4), and the split to the n1/2 + 1
// coefficients.
//
// Stockham passes of radix P (and a last one of the radix that is left): in every pass thread t takes the points
// t + TT i, i = 0..P-1, the points it holds already before the first pass and after the last, so a transform of M
// points costs one exchange through shared memory less than it has passes, and one for the split: the coefficients
// k and M - k come from the points k = t + TT i (i < P/2) of thread t and M - k = (TT - t) + TT (P - 1 - i) of thread TT - t
// (thread 0 with itself).
// An exchange is a write, one barrier of the team and a read; two buffers take turns, which also separates one row's
// last exchange from the next row's first.  Point i lies at rswz(i): 16 consecutive points and the scatters of the
// first passes reach 16 different bank pairs per half-warp.  The twiddles of a pass are read from a table in the
// order of the passes (8 points; W_M^j read at strides took 16 us more of the 8192 x 512 step).
//
// FP32 P = 8 (16 points for rows of 4096, three passes instead of four, measured the same: 94 and 93 against 88 and
// 95 us for 8192 x 512, twiddles from L1); FP64 P = 4: an FP64 instruction occupies a quarter of an SM for about 50 cycles however many
// lanes it has, so the few rows of a small grid want few instructions per warp (128 x 64: forward 10.7 -> 7, Ampere and
// inverse 15.3 -> 9.5 us).
#pragma once
#include "hyb_internal.cuh"
#include "packed_dev.cuh"
#include "tm_dev.cuh"
#include "tm_sched.cuh"

namespace hyb {

// products and small DFTs by precision: packed pairs in FP32
__device__ __forceinline__ float2 rmul(float2 a, float2 b) { return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x)); }
__device__ __forceinline__ float2 rmulc(float2 a, float2 b) { return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y)); }
__device__ __forceinline__ double2 rmul(double2 a, double2 b) { return cmul(a, b); }
__device__ __forceinline__ double2 rmulc(double2 a, double2 b) { return cmulc(a, b); }
template <bool INV> __device__ __forceinline__ void rdft8(float2 (&v)[8]) { dft8x<INV>(v); }
template <bool INV> __device__ __forceinline__ void rdft8(double2 (&v)[8]) { sdft8<double2, INV>(v); }
template <bool INV> __device__ __forceinline__ void rdft4(float2& a, float2& b, float2& c, float2& d) { dft4x<INV>(a, b, c, d); }
template <bool INV> __device__ __forceinline__ void rdft4(double2& a, double2& b, double2& c, double2& d) { sdft4<double2, INV>(a, b, c, d); }

// bits 0..2 flipped by bits 4..6 and bit 3 by bits 6 and 7
__device__ __forceinline__ int rswz(int i) { return i ^ ((i >> 4) & 7) ^ (((i >> 3) ^ (i >> 4)) & 8); }

// DFT of P points in place, natural order
template <bool INV, typename C> __device__ __forceinline__ void rdft(C (&v)[4]) { rdft4<INV>(v[0], v[1], v[2], v[3]); }
template <bool INV, typename C> __device__ __forceinline__ void rdft(C (&v)[8]) { rdft8<INV>(v); }

template <typename T, int LG> constexpr int pts() { return sizeof(T) == 8 ? 4 : 8; }

template <typename T, int LG, bool TM = false>
struct RowFft {
    using C = cplx<T>;
    static constexpr int P = pts<T, LG>(), LGP = P == 8 ? 3 : 2;
    static constexpr int M = 1 << LG, TT = M / P, H = P / 2;
    C* a;                                               // the buffer of the next exchange, and the other one
    C* b;
    int t, bar;                                         // thread of the team, its barrier
    const C* tw;                                        // table(): twiddles
    // 8 points: stockham_twiddles(M), the pass of span NS and radix R holds W_{R NS}^{r k} at NS - 1 + (r - 1) NS + k;
    // 4 points: W_M^j, j < M
    static __host__ __device__ __forceinline__ const C* table(const ModeTables<T>& t) { return P == 8 ? t.twS : t.twM; }
    template <int R, int NS> __device__ __forceinline__ C twiddle(int r, int k) const {
        return P == 8 ? tw[NS - 1 + (r - 1) * NS + k] : tw[(M / (R * NS)) * r * k];
    }

    // TM: a thread's twiddles in tensor memory, words from ta on: 16 per radix-8 pass after the first (7 twiddles), 16
    // (radix 4) or 8 (radix 2) of the last, then H of the split.  The threads of a lane quarter with the same t share them.
    static constexpr int FULL = LG / LGP - 1, REST = LG % LGP, OFF_N = 16 * FULL + (REST == 2 ? 16 : REST == 1 ? 8 : 0);
    static constexpr int SETS = TT > 128 ? TT / 128 : 1, COLS = 64 * SETS;
    static_assert(!TM || (sizeof(T) == 4 && OFF_N + 2 * H <= 64), "tensor-memory twiddles");
    uint32_t ta;
    __device__ __forceinline__ void tm_fill(const C* __restrict__ twN) const {
        if constexpr (TM) fill_pass<LGP>(twN);
    }
    template <int LGNS>
    __device__ __forceinline__ void fill_pass(const C* __restrict__ twN) const {
        constexpr int NS = 1 << LGNS, LEFT = LG - LGNS, OFF = 16 * (LGNS / LGP - 1);
        float r[16];
#pragma unroll
        for (int i = 0; i < 16; i++) r[i] = 0.f;
        if constexpr (LEFT >= LGP) {
#pragma unroll
            for (int k = 1; k < P; k++) { const C w = twiddle<P, NS>(k, t & (NS - 1)); r[2 * k - 2] = w.x; r[2 * k - 1] = w.y; }
            tm_st16(ta + OFF, r);
            fill_pass<LGNS + LGP>(twN);
        } else {
            if constexpr (LEFT > 0) {
                constexpr int RR = 1 << LEFT, Q = P / RR;
#pragma unroll
                for (int m = 0; m < Q; m++)
#pragma unroll
                    for (int k = 1; k < RR; k++) {
                        const C w = twiddle<RR, NS>(k, t + TT * m);
                        r[2 * (m * (RR - 1) + k - 1)] = w.x;
                        r[2 * (m * (RR - 1) + k - 1) + 1] = w.y;
                    }
                if constexpr (RR == 4) tm_st16(ta + OFF, r);
                else { float q[8]; for (int i = 0; i < 8; i++) q[i] = r[i]; tm_st8(ta + OFF, q); }
            }
            float q[8];
#pragma unroll
            for (int i = 0; i < H; i++) { const C w = twN[t + TT * i]; q[2 * i] = w.x; q[2 * i + 1] = w.y; }
            tm_st8(ta + OFF_N, q);
        }
    }
    // the split's twiddles W_N^{t + TT i}
    __device__ __forceinline__ void split_tw(const C* __restrict__ twN, C (&w)[H]) const {
        if constexpr (TM) {
            float q[8];
            tm_ld8(ta + OFF_N, q);
            tm_wait_ld();
#pragma unroll
            for (int i = 0; i < H; i++) w[i] = mkc<C>(q[2 * i], q[2 * i + 1]);
        } else {
#pragma unroll
            for (int i = 0; i < H; i++) w[i] = twN[t + TT * i];
        }
    }

    __device__ __forceinline__ void sync() const {
        if (TT <= 32) __syncwarp();
        else asm volatile("bar.sync %0, %1;" :: "r"(bar), "r"(TT) : "memory");
    }
    __device__ __forceinline__ void swap() { C* c = a; a = b; b = c; }
    template <bool INV> static __device__ __forceinline__ C turn(C x, C w) { return INV ? rmulc(x, w) : rmul(x, w); }

    template <bool INV, int LGNS>
    __device__ __forceinline__ void pass(C (&v)[P]) {
        constexpr int NS = 1 << LGNS, LEFT = LG - LGNS;
        if constexpr (LEFT >= LGP) {
            const int k = t & (NS - 1);
            if constexpr (LGNS > 0 && TM) {
                C w[8];
                tw_tmem(ta + 16 * (LGNS / LGP - 1), w);
#pragma unroll
                for (int r = 1; r < P; r++) v[r] = turn<INV>(v[r], w[r]);
            } else if constexpr (LGNS > 0) {
#pragma unroll
                for (int r = 1; r < P; r++) v[r] = turn<INV>(v[r], twiddle<P, NS>(r, k));
            }
            rdft<INV>(v);
            if constexpr (LEFT > LGP) {
                const int o = (t - k) * P + k;
#pragma unroll
                for (int r = 0; r < P; r++) a[rswz(o + r * NS)] = v[r];
                sync();
#pragma unroll
                for (int i = 0; i < P; i++) v[i] = a[rswz(t + i * TT)];
                swap();
                pass<INV, LGNS + LGP>(v);
            }
        } else if constexpr (LEFT > 0) {                // P/R butterflies of the radix R = 4 or 2 that is left: span M/R
            constexpr int R = 1 << LEFT, Q = P / R;
            float q[16];
            if constexpr (TM && R == 4) { tm_ld16(ta + 16 * (LGNS / LGP - 1), q); tm_wait_ld(); }
            if constexpr (TM && R == 2) {
                float q8[8];
                tm_ld8(ta + 16 * (LGNS / LGP - 1), q8);
                tm_wait_ld();
#pragma unroll
                for (int i = 0; i < 8; i++) q[i] = q8[i];
            }
#pragma unroll
            for (int m = 0; m < Q; m++) {
                C x[R];
                x[0] = v[m];
#pragma unroll
                for (int r = 1; r < R; r++) {
                    const int e = 2 * (m * (R - 1) + r - 1);
                    x[r] = turn<INV>(v[m + Q * r], TM ? mkc<C>((T)q[e], (T)q[e + 1]) : twiddle<R, NS>(r, t + TT * m));
                }
                if constexpr (R == 2) { const C y = x[0]; x[0] = cadd(y, x[1]); x[1] = csub(y, x[1]); }
                else rdft<INV>(x);
#pragma unroll
                for (int r = 0; r < R; r++) v[m + Q * r] = x[r];
            }
        }
    }

    // A thread's coefficients: slot i < H holds k = t + TT i, slot H + i holds M - k, slot P (thread 0 only) M/2;
    // forward() leaves them where inverse() wants them.
    // v[i] = z[t + TT i] -> coefficients: put(slot, k, X[k]) for k = 0..M
    template <class Put>
    __device__ __forceinline__ void forward(C (&v)[P], const C* __restrict__ twN, Put put) {
        pass<false, 0>(v);
#pragma unroll
        for (int i = 0; i < H; i++) a[i * TT + t] = v[H + i];
        sync();
        // X[k] = e - u, X[M-k] = conj(e + u), e = (Z[k] + Z*[M-k])/2, u = (i/2) W_N^k (Z[k] - Z*[M-k])
        C w[H];
        split_tw(twN, w);
        auto pair = [&](int slot, int k, C zk, C zm, C wk, bool both) {
            const C e = mkc<C>((T)0.5 * (zk.x + zm.x), (T)0.5 * (zk.y - zm.y));
            const C wd = rmul(wk, mkc<C>(zk.x - zm.x, zk.y + zm.y));
            put(slot, k, mkc<C>(e.x + (T)0.5 * wd.y, e.y - (T)0.5 * wd.x));
            if (both) put(H + slot, M - k, mkc<C>(e.x - (T)0.5 * wd.y, -(e.y + (T)0.5 * wd.x)));
        };
#pragma unroll
        for (int i = 0; i < H; i++) pair(i, t + TT * i, v[i], i == 0 && t == 0 ? v[0] : a[(H - i) * TT - t], w[i], true);
        if (t == 0) pair(P, M / 2, v[H], v[H], twN[M / 2], false);
        swap();
    }

    // each(slot, k) for this thread's coefficients
    template <class Each>
    __device__ __forceinline__ void modes(Each each) const {
#pragma unroll
        for (int i = 0; i < H; i++) {
            each(i, t + TT * i);
            each(H + i, M - t - TT * i);
        }
        if (t == 0) each(P, M / 2);
    }

    // X[k] = ld(slot, k), k = 0..M (each once) -> v[i] = z[t + TT i] M (unscaled); imaginary parts of X[0], X[M] dropped
    template <class Ld>
    __device__ __forceinline__ void inverse(C (&v)[P], const C* __restrict__ twN, Ld ld) {
        // Z[k] = E + iO, Z[M-k] = conj(E - iO), E = (X[k] + X*[M-k])/2, O = conj(W_N^k)(X[k] - X*[M-k])/2
        C w[H];
        split_tw(twN, w);
        auto pair = [&](C xk, C xm, C wk, C& zm) {
            const C e = mkc<C>((T)0.5 * (xk.x + xm.x), (T)0.5 * (xk.y - xm.y));
            const C o = rmulc(mkc<C>((T)0.5 * (xk.x - xm.x), (T)0.5 * (xk.y + xm.y)), wk);
            zm = mkc<C>(e.x + o.y, o.x - e.y);
            return mkc<C>(e.x - o.y, e.y + o.x);
        };
#pragma unroll
        for (int i = 0; i < H; i++) {
            const int k = t + TT * i;
            C xk = ld(i, k), xm = ld(H + i, M - k), zm;
            if (i == 0 && t == 0) { xk.y = (T)0; xm.y = (T)0; }
            v[i] = pair(xk, xm, w[i], zm);
            if (i > 0 || t > 0) a[(H - i) * TT - t] = zm;
        }
        if (t == 0) {
            const C x = ld(P, M / 2);
            C zm;
            a[0] = pair(x, x, twN[M / 2], zm);
        }
        sync();
#pragma unroll
        for (int i = 0; i < H; i++) v[H + i] = a[i * TT + t];
        swap();
        pass<true, 0>(v);
    }
};

}  // namespace hyb
