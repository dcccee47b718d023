// rowfft.cuh -- register-resident real row transforms: the complex FFT of M = n1/2 points, z[j] = x[2j] + i
// x[2j+1], by a team of TT = M/8 threads that hold 8 points each, and the split to the n1/2 + 1 coefficients.
//
// Stockham passes of radix 8 (and a last one of radix 4 or 2): in every pass thread t takes the points t + TT i,
// i = 0..7, the points it holds already before the first pass and after the last, so a transform of M points costs
// one exchange through shared memory less than it has passes, and one for the split: the coefficients k and M - k
// come from the points k = t + TT i (i < 4) of thread t and M - k = (TT - t) + TT (7 - i) of thread TT - t (thread 0 with itself).
// An exchange is a write, one barrier of the team and a read; two buffers take turns, which also separates one row's
// last exchange from the next row's first.  Point i lies at rswz(i): 16 consecutive points and the scatters of the
// passes of span 1, 8 and 64 all reach 16 different bank pairs per half-warp.  Of a pass's seven twiddles W, .., W^7
// three (W, W^2, W^4) are loaded and four formed by one product each: the load and store pipe bounds these
// kernels (4096 points: 60 % busy with all seven loaded and one pass's scatter in conflict, 88 us for nine fields of
// 512 rows).
#pragma once
#include "hyb_internal.cuh"
#include "packed_dev.cuh"

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

// bits 0..2 flipped by bits 4..6 and bit 3 by bit 6
__device__ __forceinline__ int rswz(int i) { return i ^ ((i >> 4) & 7) ^ ((i >> 3) & 8); }

template <typename T, int LG>
struct RowFft {
    using C = cplx<T>;
    static constexpr int M = 1 << LG, TT = M / 8;
    C* a;                                               // the buffer of the next exchange, and the other one
    C* b;
    int t, bar;                                         // thread of the team, its barrier
    const C* tw;                                        // stockham_twiddles(M)

    __device__ __forceinline__ void sync() const {
        if (TT <= 32) __syncwarp();
        else asm volatile("bar.sync %0, %1;" :: "r"(bar), "r"(TT) : "memory");
    }
    __device__ __forceinline__ void swap() { C* c = a; a = b; b = c; }

    template <bool INV, int LGNS>
    __device__ __forceinline__ void pass(C (&v)[8]) {
        constexpr int NS = 1 << LGNS, REST = LG - LGNS;
        if constexpr (REST >= 3) {
            const int k = t & (NS - 1);
            if constexpr (LGNS > 0) {
                const C w1 = tw[NS - 1 + k], w2 = tw[2 * NS - 1 + k], w4 = tw[4 * NS - 1 + k], w3 = rmul(w1, w2);
                const C w[8] = {w1, w1, w2, w3, w4, rmul(w1, w4), rmul(w2, w4), rmul(w3, w4)};
#pragma unroll
                for (int r = 1; r < 8; r++) v[r] = INV ? rmulc(v[r], w[r]) : rmul(v[r], w[r]);
            }
            rdft8<INV>(v);
            if constexpr (REST > 3) {
                const int o = (t - k) * 8 + k;
#pragma unroll
                for (int r = 0; r < 8; r++) a[rswz(o + r * NS)] = v[r];
                sync();
#pragma unroll
                for (int i = 0; i < 8; i++) v[i] = a[rswz(t + i * TT)];
                swap();
                pass<INV, LGNS + 3>(v);
            }
        } else if constexpr (REST == 2) {               // two butterflies of radix 4
#pragma unroll
            for (int m = 0; m < 2; m++) {
#pragma unroll
                for (int r = 1; r < 4; r++) {
                    const C w = tw[NS - 1 + (r - 1) * NS + t + TT * m];
                    v[m + 2 * r] = INV ? rmulc(v[m + 2 * r], w) : rmul(v[m + 2 * r], w);
                }
                rdft4<INV>(v[m], v[m + 2], v[m + 4], v[m + 6]);
            }
        } else if constexpr (REST == 1) {               // four of radix 2
#pragma unroll
            for (int m = 0; m < 4; m++) {
                const C w = tw[NS - 1 + t + TT * m];
                const C x = INV ? rmulc(v[m + 4], w) : rmul(v[m + 4], w);
                v[m + 4] = csub(v[m], x);
                v[m] = cadd(v[m], x);
            }
        }
    }

    // v[i] = z[t + TT i] -> coefficients: put(k, X[k]) for k = 0..M
    template <class Put>
    __device__ __forceinline__ void forward(C (&v)[8], const C* __restrict__ twN, Put put) {
        pass<false, 0>(v);
#pragma unroll
        for (int i = 0; i < 4; i++) a[i * TT + t] = v[4 + i];
        sync();
        // X[k] = e - u, X[M-k] = conj(e + u), e = (Z[k] + Z*[M-k])/2, u = (i/2) W_N^k (Z[k] - Z*[M-k])
        auto pair = [&](int k, C zk, C zm, bool both) {
            const C e = mkc<C>((T)0.5 * (zk.x + zm.x), (T)0.5 * (zk.y - zm.y));
            const C wd = rmul(twN[k], mkc<C>(zk.x - zm.x, zk.y + zm.y));
            put(k, mkc<C>(e.x + (T)0.5 * wd.y, e.y - (T)0.5 * wd.x));
            if (both) put(M - k, mkc<C>(e.x - (T)0.5 * wd.y, -(e.y + (T)0.5 * wd.x)));
        };
#pragma unroll
        for (int i = 0; i < 4; i++) pair(t + TT * i, v[i], i == 0 && t == 0 ? v[0] : a[(4 - i) * TT - t], true);
        if (t == 0) pair(M / 2, v[4], v[4], false);
        swap();
    }

    // X[k] = ld(k), k = 0..M (each once) -> v[i] = z[t + TT i] M (unscaled); imaginary parts of X[0], X[M] dropped
    template <class Ld>
    __device__ __forceinline__ void inverse(C (&v)[8], const C* __restrict__ twN, Ld ld) {
        // Z[k] = E + iO, Z[M-k] = conj(E - iO), E = (X[k] + X*[M-k])/2, O = conj(W_N^k)(X[k] - X*[M-k])/2
        auto pair = [&](int k, C xk, C xm, C& zm) {
            const C e = mkc<C>((T)0.5 * (xk.x + xm.x), (T)0.5 * (xk.y - xm.y));
            const C o = rmulc(mkc<C>((T)0.5 * (xk.x - xm.x), (T)0.5 * (xk.y + xm.y)), twN[k]);
            zm = mkc<C>(e.x + o.y, o.x - e.y);
            return mkc<C>(e.x - o.y, e.y + o.x);
        };
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int k = t + TT * i;
            C xk = ld(k), xm = ld(M - k), zm;
            if (i == 0 && t == 0) { xk.y = (T)0; xm.y = (T)0; }
            v[i] = pair(k, xk, xm, zm);
            if (i > 0 || t > 0) a[(4 - i) * TT - t] = zm;
        }
        if (t == 0) {
            const C x = ld(M / 2);
            C zm;
            a[0] = pair(M / 2, x, x, zm);
        }
        sync();
#pragma unroll
        for (int i = 0; i < 4; i++) v[4 + i] = a[i * TT + t];
        swap();
        pass<true, 0>(v);
    }
};

}  // namespace hyb
