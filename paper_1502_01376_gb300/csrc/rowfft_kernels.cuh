// rowfft_kernels.cuh -- the kernels of the register-resident row transforms (rowfft.cuh) and their launches, one
// precision per translation unit (rowfft.cu, rowfft64.cu): the forward transform, the inverse, and the inverse
// with the Ampere update of the E fields formed as their spectra are loaded, and (FP32) the updates with the forward and
// the inverse transform around them.
#pragma once
#include <algorithm>

#include "rowfft.cuh"
#include "rowfft_api.cuh"

namespace hyb {

// the largest block, whole teams, and the blocks per SM its registers are held to: 64 registers a thread, FP64 128
template <typename T, int LG> constexpr int row_threads() { return RowFft<T, LG>::TT > 256 ? RowFft<T, LG>::TT : 256; }
template <typename T, int LG> constexpr int row_blocks() { return (sizeof(T) == 4 ? 1024 : 512) / row_threads<T, LG>(); }
// of the update kernels: 128 registers hold a row's points and its coefficients (64 and 80 spill: 1024 x 256 x 256 step 2400 and
// 2000 us against 1870)
template <typename T, int LG> constexpr int upd_blocks() { return 512 / row_threads<T, LG>(); }

template <typename T, int LG, bool TM = false>
__device__ __forceinline__ RowFft<T, LG, TM> row_team(unsigned char* smem, const cplx<T>* tw, int* team) {
    using F = RowFft<T, LG, TM>;
    F f;
    *team = threadIdx.x / F::TT;
    f.t = threadIdx.x % F::TT;
    f.bar = 1 + *team;
    f.a = reinterpret_cast<cplx<T>*>(smem) + (size_t)*team * 2 * F::M;
    f.b = f.a + F::M;
    f.tw = tw;
    return f;
}

__device__ __forceinline__ void l2_prefetch(const void* p) { asm volatile("prefetch.global.L2 [%0];" :: "l"(p)); }

// TM blocks (whole groups of four warps): tensor memory for the twiddles, its first SETS groups of four warps fill it
template <typename T, int LG>
__device__ __forceinline__ void tm_open(RowFft<T, LG, true>& f, const cplx<T>* __restrict__ twN) {
    using F = RowFft<T, LG, true>;
    __shared__ uint32_t s_base;
    const int warp = threadIdx.x >> 5;
    if (warp == 0) {
        tm_alloc(smem_addr(&s_base), F::COLS);
        tm_relinquish();
    }
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    f.ta = s_base + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(64 * ((warp >> 2) % F::SETS));
    if (warp < 4 * F::SETS) {
        f.tm_fill(twN);
        tm_wait_st();
    }
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
}
template <typename T, int LG>
__device__ __forceinline__ void tm_close(const RowFft<T, LG, true>& f) {
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    if (threadIdx.x < 32) tm_dealloc(f.ta, RowFft<T, LG, true>::COLS);
}

// Persistent: a block takes groups of blockDim / TT rows (row j of the nf fields' rows: field j / rows) and holds the next
// group's samples in registers while it transforms the current one.
template <typename T, int LG, bool TM>
__global__ void __launch_bounds__((row_threads<T, LG>()), (row_blocks<T, LG>())) k_rfft_reg(const __grid_constant__ RowPtrs in, cplx<T>* __restrict__ out, unsigned rows,
                                                                                     unsigned total, const cplx<T>* __restrict__ tw,
                                                                                     const cplx<T>* __restrict__ twN) {
    using F = RowFft<T, LG, TM>;
    using C = cplx<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int team;
    F f = row_team<T, LG, TM>(smem_raw, tw, &team);
    const unsigned R = blockDim.x / F::TT, step = gridDim.x * R;
    C nx[F::P];
    auto fetch = [&](unsigned j) {
        if (j < total) {
            const unsigned fl = j / rows;
            const C* z = reinterpret_cast<const C*>(in.p[fl]) + (size_t)(j - fl * rows) * F::M;
#pragma unroll
            for (int i = 0; i < F::P; i++) nx[i] = __ldcs(z + f.t + F::TT * i);
        }
    };
    unsigned j = blockIdx.x * R + team;
    fetch(j);
    if constexpr (TM) tm_open(f, twN);
    for (unsigned g = blockIdx.x * R; g < total; g += step, j += step) {
        C v[F::P];
#pragma unroll
        for (int i = 0; i < F::P; i++) v[i] = nx[i];
        const bool live = j < total;
        if (total - j > step) fetch(j + step);                 // (unsigned: also when j is past the end)
        C* const X = out + (size_t)(live ? j : 0) * (F::M + 1);
        f.forward(v, twN, [&](int, int k, C x) { if (live) X[k] = x; });
    }
    if constexpr (TM) tm_close(f);
}

template <typename T, int LG>
__global__ void __launch_bounds__((row_threads<T, LG>()), (row_blocks<T, LG>())) k_irfft_reg(const cplx<T>* __restrict__ in, const __grid_constant__ RowPtrsW out,
                                                                                      unsigned rows, const cplx<T>* __restrict__ tw,
                                                                                      const cplx<T>* __restrict__ twN) {
    using F = RowFft<T, LG>;
    using C = cplx<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int team;
    F f = row_team<T, LG>(smem_raw, tw, &team);
    const unsigned R = blockDim.x / F::TT, row = blockIdx.x * R + team;
    const int fl = blockIdx.y;
    const bool live = row < rows;
    const C* X = in + ((size_t)fl * rows + (live ? row : 0)) * (F::M + 1);
    C v[F::P];
    f.inverse(v, twN, [&](int, int k) { return X[k]; });
    if (live) {
        C* z = reinterpret_cast<C*>(out.p[fl]) + (size_t)row * F::M;
        const T inv = (T)1 / (T)F::M;
#pragma unroll
        for (int i = 0; i < F::P; i++) z[f.t + F::TT * i] = cscale(v[i], inv);
    }
}

// Ampere (Eqs. hybrid2de1-hybrid2de3; the x3 differences of Sec. 2.4) formed mode by mode as the inverse transform
// loads E_f (fields 0-2; Sm = -conj(S)); fields 3-5 invert B.  The six fields of a row group are consecutive
// blocks, so that the B rows three of them read come from L2.  WB (k1-resident state): the updated E spectrum is
// also stored back (each mode of a row is loaded once, by the block of that row and field).
template <typename T, int LG, bool D3, bool WB>
__global__ void __launch_bounds__((row_threads<T, LG>()), (row_blocks<T, LG>())) k_ampere_irfft_reg(cplx<T>* __restrict__ spec, const __grid_constant__ RowPtrsW out,
                                                                                             unsigned rows, int n2, int n3,
                                                                                             const cplx<T>* __restrict__ tw,
                                                                                             const cplx<T>* __restrict__ twN,
                                                                                             const cplx<T>* __restrict__ S,
                                                                                             const T* __restrict__ cj1,
                                                                                             const T* __restrict__ cj, T a2, T a3) {
    using F = RowFft<T, LG>;
    using C = cplx<T>;
    constexpr int NK = F::M + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int team;
    F f = row_team<T, LG>(smem_raw, tw, &team);
    const unsigned R = blockDim.x / F::TT, row = blockIdx.x / 6u * R + team;
    const int fl = blockIdx.x % 6u;
    const bool live = row < rows;
    const unsigned r = live ? row : 0u;
    const int i3 = (int)(r / (unsigned)n2), i2 = (int)(r - (unsigned)i3 * (unsigned)n2);
    const size_t fs = (size_t)rows * NK;
    C* Xr = spec + (size_t)r * NK;                                                               // field 0 of row r
    const C* Xm2 = spec + ((size_t)i3 * n2 + (i2 == 0 ? n2 - 1 : i2 - 1)) * NK;                  // row i2 - 1
    const C* Xm3 = spec + ((size_t)(D3 ? (i3 == 0 ? n3 - 1 : i3 - 1) : i3) * n2 + i2) * NK;      // row i3 - 1
    C v[F::P];
    auto axpy = [](C y, T s, C x) { return mkc<C>(fma(s, x.x, y.x), fma(s, x.y, y.y)); };
    auto keep = [&](C* at, C e) {
        if (WB && live) *at = e;
        return e;
    };
    if (fl == 0) {
        f.inverse(v, twN, [&](int, int k) {
            C e = axpy(Xr[k], a2, csub(Xr[5 * fs + k], Xm2[5 * fs + k]));
            if (D3) e = axpy(e, -a3, csub(Xr[4 * fs + k], Xm3[4 * fs + k]));
            return keep(Xr + k, axpy(e, -cj1[k], Xr[6 * fs + k]));
        });
    } else if (fl == 1) {
        f.inverse(v, twN, [&](int, int k) {
            const C s = S[k], b3 = Xr[5 * fs + k];
            C e = Xr[fs + k];
            e = mkc<C>(e.x + (s.x * b3.x + s.y * b3.y), e.y + (s.x * b3.y - s.y * b3.x));        // - Sm B3 = conj(S) B3
            if (D3) e = axpy(e, a3, csub(Xr[3 * fs + k], Xm3[3 * fs + k]));
            return keep(Xr + fs + k, axpy(e, -cj[k], Xr[7 * fs + k]));
        });
    } else if (fl == 2) {
        f.inverse(v, twN, [&](int, int k) {
            const C s = S[k], b2 = Xr[4 * fs + k];
            C e = Xr[2 * fs + k];
            e = mkc<C>(e.x - (s.x * b2.x + s.y * b2.y), e.y - (s.x * b2.y - s.y * b2.x));        // + Sm B2
            e = axpy(e, -a2, csub(Xr[3 * fs + k], Xm2[3 * fs + k]));
            return keep(Xr + 2 * fs + k, axpy(e, -cj[k], Xr[8 * fs + k]));
        });
    } else {
        const C* X = Xr + fl * fs;
        f.inverse(v, twN, [&](int, int k) { return X[k]; });
    }
    if (live) {
        C* z = reinterpret_cast<C*>(out.p[fl]) + (size_t)row * F::M;
        const T inv = (T)1 / (T)F::M;
#pragma unroll
        for (int i = 0; i < F::P; i++) z[f.t + F::TT * i] = cscale(v[i], inv);
    }
}

// The updates with transforms on both sides, for FP32 grids whose rows fill the chip: a coefficient stays with its thread
// from the forward transform to the inverse, so that j's spectra (k_ampere_reg), and B's before the update
// (k_faraday_reg), are neither stored nor read: 39 and 30 passes over a field per step instead of 45.
// Bound by the shared-memory pipe (half of its cycles) and by what latency is left; so the twiddles of a
// persistent block lie in tensor memory (TM; from L1 they were a quarter of the wavefronts: 8192 x 512 step 204 -> 184 us,
// 4096 x 1024 177 -> 156), every team asks for the lines of its next row while it works on this one (1024 x 256 x 256 step
// 2250 -> 1990, 8192 x 512 189 -> 170), and the sums over the spectra, all loads, come before the row's transform (after
// it: 2285 -> 2425).  Blocks nfl q .. nfl q + nfl - 1 take the nfl components of the row groups q, q + grid/nfl, ..., a
// block another component each time: two of three components read the same spectra, at the same time, from L2, and the
// work evens out.  One block taking all components of a group in turn, its spectra from L1, lost (1880 -> 2270).
//
// Faraday on the rows of B, stored as spectra (Ampere's differences read them) and as rows:
//   B1 += a3 d3+E2 - a2 d2+E3;  B2 += S E3 - a3 d3+E1;  B3 += a2 d2+E1 - S E2
template <typename T, int LG, bool D3, bool TM>
__global__ void __launch_bounds__((row_threads<T, LG>()), (upd_blocks<T, LG>())) k_faraday_reg(cplx<T>* __restrict__ spec, const __grid_constant__ RowPtrsW B,
                                                                                        unsigned rows, int n2, int n3,
                                                                                        const cplx<T>* __restrict__ tw,
                                                                                        const cplx<T>* __restrict__ twN,
                                                                                        const cplx<T>* __restrict__ S, T a2, T a3) {
    using F = RowFft<T, LG, TM>;
    using C = cplx<T>;
    constexpr int NK = F::M + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int team;
    F f = row_team<T, LG, TM>(smem_raw, tw, &team);
    if constexpr (TM) tm_open(f, twN);
    const unsigned R = blockDim.x / F::TT, step = gridDim.x / 3u * R;
    const size_t fs = (size_t)rows * NK;
    struct Rows { const C *e, *p2, *p3; };            // E1's spectrum of row r, of rows i2 + 1, i3 + 1
    auto rows_at = [&](unsigned r) {
        const int i3 = (int)(r / (unsigned)n2), i2 = (int)(r - (unsigned)i3 * (unsigned)n2);
        return Rows{spec + (size_t)r * NK, spec + ((size_t)i3 * n2 + (i2 + 1 == n2 ? 0 : i2 + 1)) * NK,
                    spec + ((size_t)(D3 ? (i3 + 1 == n3 ? 0 : i3 + 1) : i3) * n2 + i2) * NK};
    };
    unsigned n = blockIdx.x % 3u;
    for (unsigned base = blockIdx.x / 3u * R; base < rows; base += step, n++) {
    const unsigned row = base + team;
    const int fl = (int)(n % 3u);
    const bool live = row < rows;
    const unsigned r = live ? row : 0u;
    const Rows q = rows_at(r);
    const C *E = q.e, *Ep2 = q.p2, *Ep3 = q.p3;
    C* X = spec + (size_t)(3 + fl) * fs + (size_t)r * NK;
    C* z = reinterpret_cast<C*>(B.p[fl]) + (size_t)r * F::M;
    if (TM && rows - base > step && row + step < rows && f.t <= F::TT / 2) {
        const unsigned nf = (n + 1) % 3u;
        const Rows p = rows_at(row + step);
        const int k = 16 * f.t;
        if (f.t < F::TT / 2) l2_prefetch(reinterpret_cast<const C*>(B.p[nf]) + (size_t)(row + step) * F::M + k);
        if (nf == 0) { l2_prefetch(p.e + 2 * fs + k); l2_prefetch(p.p2 + 2 * fs + k); if (D3) { l2_prefetch(p.e + fs + k); l2_prefetch(p.p3 + fs + k); } }
        if (nf == 1) { l2_prefetch(p.e + 2 * fs + k); if (D3) { l2_prefetch(p.e + k); l2_prefetch(p.p3 + k); } }
        if (nf == 2) { l2_prefetch(p.e + fs + k); l2_prefetch(p.e + k); l2_prefetch(p.p2 + k); }
    }
    auto axpy = [](C y, T s, C x) { return mkc<C>(fma(s, x.x, y.x), fma(s, x.y, y.y)); };
    C v[F::P], x[F::P + 1];
#pragma unroll
    for (int i = 0; i < F::P; i++) v[i] = __ldcs(z + f.t + F::TT * i);
    if (fl == 0) {
        f.modes([&](int m, int k) {
            x[m] = cscale(csub(E[2 * fs + k], Ep2[2 * fs + k]), a2);
            if (D3) x[m] = axpy(x[m], a3, csub(Ep3[fs + k], E[fs + k]));
        });
    } else if (fl == 1) {
        f.modes([&](int m, int k) {
            x[m] = cmul(S[k], E[2 * fs + k]);
            if (D3) x[m] = axpy(x[m], a3, csub(E[k], Ep3[k]));
        });
    } else {
        f.modes([&](int m, int k) { x[m] = csub(cscale(csub(Ep2[k], E[k]), a2), cmul(S[k], E[fs + k])); });
    }
    f.forward(v, twN, [&](int m, int k, C b) {
        x[m] = cadd(b, x[m]);
        if (live) X[k] = x[m];
    });
    f.inverse(v, twN, [&](int m, int) { return x[m]; });
    if (live) {
        const T inv = (T)1 / (T)F::M;
#pragma unroll
        for (int i = 0; i < F::P; i++) z[f.t + F::TT * i] = cscale(v[i], inv);
    }
    }
    if constexpr (TM) tm_close(f);
}

// Ampere and E's inverse, the row of j_c transformed on the way (the sums of k_ampere_irfft_reg); of nfl = 6 components, E
// and B in turn, the last three are B's inverse.
template <typename T, int LG, bool D3, bool WB, bool TM>
__global__ void __launch_bounds__((row_threads<T, LG>()), (upd_blocks<T, LG>())) k_ampere_reg(cplx<T>* __restrict__ spec, const __grid_constant__ RowPtrs J,
                                                                                       const __grid_constant__ RowPtrsW out, unsigned rows,
                                                                                       int n2, int n3, const cplx<T>* __restrict__ tw,
                                                                                       const cplx<T>* __restrict__ twN,
                                                                                       const cplx<T>* __restrict__ S,
                                                                                       const T* __restrict__ cj1, const T* __restrict__ cj, T a2,
                                                                                       T a3, unsigned nfl) {
    using F = RowFft<T, LG, TM>;
    using C = cplx<T>;
    constexpr int NK = F::M + 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int team;
    F f = row_team<T, LG, TM>(smem_raw, tw, &team);
    if constexpr (TM) tm_open(f, twN);
    const unsigned R = blockDim.x / F::TT;
    const size_t fs = (size_t)rows * NK;
    struct Rows { C *x; const C *b, *m2, *m3; };      // field fl's spectrum of row r; B1's of row r, of rows i2 - 1, i3 - 1
    auto rows_at = [&](unsigned r, int fl) {
        const int i3 = (int)(r / (unsigned)n2), i2 = (int)(r - (unsigned)i3 * (unsigned)n2);
        const C* b1 = spec + 3 * fs;
        return Rows{spec + (size_t)fl * fs + (size_t)r * NK, b1 + (size_t)r * NK,
                    b1 + ((size_t)i3 * n2 + (i2 == 0 ? n2 - 1 : i2 - 1)) * NK,
                    b1 + ((size_t)(D3 ? (i3 == 0 ? n3 - 1 : i3 - 1) : i3) * n2 + i2) * NK};
    };
    unsigned n = blockIdx.x % nfl;
    const unsigned step = gridDim.x / nfl * R;
    auto field = [&](unsigned n) { return (int)(nfl == 6 ? (n & 1u) * 3u + n / 2u % 3u : n % 3u); };
    for (unsigned base = blockIdx.x / nfl * R; base < rows; base += step, n++) {
    const unsigned row = base + team;
    const int fl = field(n);
    const bool live = row < rows;
    const unsigned r = live ? row : 0u;
    const Rows q = rows_at(r, fl);
    C* X = q.x;
    const C *B = q.b, *Bm2 = q.m2, *Bm3 = q.m3;
    if (TM && rows - base > step && row + step < rows && f.t <= F::TT / 2) {
        const int nf = field(n + 1);
        const Rows p = rows_at(row + step, nf);
        const int k = 16 * f.t;
        l2_prefetch(p.x + k);
        if (nf < 3) {
            if (f.t < F::TT / 2) l2_prefetch(reinterpret_cast<const C*>(J.p[nf]) + (size_t)(row + step) * F::M + k);
            if (nf == 0) { l2_prefetch(p.b + 2 * fs + k); l2_prefetch(p.m2 + 2 * fs + k); if (D3) { l2_prefetch(p.b + fs + k); l2_prefetch(p.m3 + fs + k); } }
            if (nf == 1) { l2_prefetch(p.b + 2 * fs + k); if (D3) { l2_prefetch(p.b + k); l2_prefetch(p.m3 + k); } }
            if (nf == 2) { l2_prefetch(p.b + fs + k); l2_prefetch(p.b + k); l2_prefetch(p.m2 + k); }
        }
    }
    auto axpy = [](C y, T s, C x) { return mkc<C>(fma(s, x.x, y.x), fma(s, x.y, y.y)); };
    C v[F::P];
    if (fl < 3) {
        C x[F::P + 1];
        const C* j = reinterpret_cast<const C*>(J.p[fl]) + (size_t)r * F::M;
#pragma unroll
        for (int i = 0; i < F::P; i++) v[i] = __ldcs(j + f.t + F::TT * i);
        const T* c = fl == 0 ? cj1 : cj;
        if (fl == 0) {
            f.modes([&](int m, int k) {
                C e = axpy(X[k], a2, csub(B[2 * fs + k], Bm2[2 * fs + k]));
                if (D3) e = axpy(e, -a3, csub(B[fs + k], Bm3[fs + k]));
                x[m] = e;
            });
        } else if (fl == 1) {
            f.modes([&](int m, int k) {
                const C s = S[k], b3 = B[2 * fs + k];
                C e = X[k];
                e = mkc<C>(e.x + (s.x * b3.x + s.y * b3.y), e.y + (s.x * b3.y - s.y * b3.x));             // - Sm B3 = conj(S) B3
                if (D3) e = axpy(e, a3, csub(B[k], Bm3[k]));
                x[m] = e;
            });
        } else {
            f.modes([&](int m, int k) {
                const C s = S[k], b2 = B[fs + k];
                C e = X[k];
                e = axpy(mkc<C>(e.x - (s.x * b2.x + s.y * b2.y), e.y - (s.x * b2.y - s.y * b2.x)), -a2, csub(B[k], Bm2[k]));   // + Sm B2
                x[m] = e;
            });
        }
        f.forward(v, twN, [&](int m, int k, C a) { x[m] = axpy(x[m], -c[k], a); });
        if (WB && live) f.modes([&](int m, int k) { X[k] = x[m]; });
        f.inverse(v, twN, [&](int m, int) { return x[m]; });
    } else {
        f.inverse(v, twN, [&](int, int k) { return X[k]; });
    }
    if (live) {
        C* z = reinterpret_cast<C*>(out.p[fl]) + (size_t)row * F::M;
        const T inv = (T)1 / (T)F::M;
#pragma unroll
        for (int i = 0; i < F::P; i++) z[f.t + F::TT * i] = cscale(v[i], inv);
    }
    }
    if constexpr (TM) tm_close(f);
}

// ---------------------------------------------------------------- launches
// rounds of a persistent launch from which the twiddles go to tensor memory (k_rfft_reg, k_faraday_reg, k_ampere_reg): from
// two on it is not slower (step of 8192 x 32 22.7 and 22.6 us, 128 x 4000 26.7 and 26.4, 256 x 4000 40 and 37, 128 x
// 30000 163 and 137); a single round would fill it for one row
constexpr int kTmRounds = 2;
// threads of a block: the largest, fewer while that leaves under `blocks` of them: about four per SM
constexpr int kRowBlocks = 600;
template <typename T, int LG>
static int threads_for(int64_t total_rows, int blocks = kRowBlocks) {
    constexpr int TT = RowFft<T, LG>::TT;
    int th = row_threads<T, LG>();
    while (th > std::max(TT, 32) && total_rows < (int64_t)(th / TT) * blocks) th >>= 1;
    return th;
}
// of a step's forward transforms and Ampere with E's inverse (rows of all their fields): two per SM for FP32 rows of 1024
// points (steps of 1024 x 128 12.3 us instead of 14.4, 1024 x 260 14.4 instead of 16.4), four for others (two: 512 x 1100 22.5 us
// instead of 20.6, FP64 128 x 400 26.7 instead of 24.8)
template <typename T, int LG> constexpr int row_step_blocks() { return sizeof(T) == 4 && LG == 9 ? kRowBlocks / 2 : kRowBlocks; }
template <typename T, int LG>
static size_t smem_for(int threads) { return sizeof(cplx<T>) * 2 * RowFft<T, LG>::M * (size_t)(threads / RowFft<T, LG>::TT); }
// shared memory for the kernel's largest block, and a carveout that holds `blocks` of them and leaves the rest to L1: rows
// of spectra and the mode tables are read from it (with all of it as shared memory the 1024 x 256 x 256 step took 1896 us
// instead of 1666, 8192 x 512 170 instead of 160)
static cudaError_t room(const void* kern, size_t smem_max, int blocks) {
    const int percent = std::min<int>(100, (int)(100 * blocks * (smem_max + 1024) / (228 * 1024)) + 1);
    cudaError_t e = func_attr_once(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
    return e == cudaSuccess ? func_attr_once(kern, cudaFuncAttributePreferredSharedMemoryCarveout, percent) : e;
}

template <typename T, int LG>
static cudaError_t rfft_lg(const RowPtrs& p, int nf, cplx<T>* out, int64_t rows, const ModeTables<T>& t, cudaStream_t s) {
    if (!RowFft<T, LG>::table(t) || !t.twN) return cudaErrorInvalidValue;
    const int64_t total = rows * nf;
    cudaError_t e = room((const void*)k_rfft_reg<T, LG, false>, smem_for<T, LG>((row_threads<T, LG>())), row_blocks<T, LG>());
    if (e != cudaSuccess) return e;
    if constexpr (sizeof(T) == 4) {
        constexpr int th = row_threads<T, LG>(), R = th / RowFft<T, LG>::TT;
        const size_t smem = smem_for<T, LG>(th);
        const int resident = resident_grid((const void*)k_rfft_reg<T, LG, false>, th, smem);     // of the same launch bounds
        if (total >= (int64_t)kTmRounds * R * resident) {
            const auto kern = k_rfft_reg<T, LG, true>;
            e = room((const void*)kern, smem, row_blocks<T, LG>());
            if (e != cudaSuccess) return e;
            kern<<<resident, th, smem, s>>>(p, out, (unsigned)rows, (unsigned)total, RowFft<T, LG>::table(t), t.twN);
            return cudaGetLastError();
        }
    }
    const auto kern = k_rfft_reg<T, LG, false>;
    const int th = threads_for<T, LG>(total, row_step_blocks<T, LG>()), R = th / RowFft<T, LG>::TT;
    const size_t smem = smem_for<T, LG>(th);
    const int64_t blocks = std::min<int64_t>((total + R - 1) / R, resident_grid((const void*)kern, th, smem));
    kern<<<(unsigned)blocks, th, smem, s>>>(p, out, (unsigned)rows, (unsigned)total, RowFft<T, LG>::table(t), t.twN);
    return cudaGetLastError();
}
template <typename T, int LG>
static cudaError_t irfft_lg(const cplx<T>* in, const RowPtrsW& p, int nf, int64_t rows, const ModeTables<T>& t, cudaStream_t s) {
    if (!RowFft<T, LG>::table(t) || !t.twN) return cudaErrorInvalidValue;
    const auto kern = k_irfft_reg<T, LG>;
    cudaError_t e = room((const void*)kern, smem_for<T, LG>((row_threads<T, LG>())), row_blocks<T, LG>());
    if (e != cudaSuccess) return e;
    const int th = threads_for<T, LG>(rows * nf), R = th / RowFft<T, LG>::TT;
    kern<<<dim3((unsigned)((rows + R - 1) / R), nf), th, smem_for<T, LG>(th), s>>>(in, p, (unsigned)rows, RowFft<T, LG>::table(t), t.twN);
    return cudaGetLastError();
}
template <typename T, int LG>
static cudaError_t ampere_lg(cplx<T>* spec, const RowPtrsW& p, int64_t rows, int n2, int n3, bool d3, bool wb, const ModeTables<T>& t, T a2,
                             T a3, cudaStream_t s) {
    if (!RowFft<T, LG>::table(t) || !t.twN || !t.S || !t.cj1 || !t.cj) return cudaErrorInvalidValue;
    const auto kern = d3 ? (wb ? k_ampere_irfft_reg<T, LG, true, true> : k_ampere_irfft_reg<T, LG, true, false>)
                         : (wb ? k_ampere_irfft_reg<T, LG, false, true> : k_ampere_irfft_reg<T, LG, false, false>);
    cudaError_t e = room((const void*)kern, smem_for<T, LG>((row_threads<T, LG>())), row_blocks<T, LG>());
    if (e != cudaSuccess) return e;
    const int th = threads_for<T, LG>(rows * 6, row_step_blocks<T, LG>()), R = th / RowFft<T, LG>::TT;
    kern<<<(unsigned)((rows + R - 1) / R * 6), th, smem_for<T, LG>(th), s>>>(spec, p, (unsigned)rows, n2, n3, RowFft<T, LG>::table(t), t.twN, t.S, t.cj1, t.cj,
                                                                            a2, a3);
    return cudaGetLastError();
}

// Faraday and Ampere with the transforms they need (rowfft_api.cuh)
template <typename T, int LG>
static cudaError_t update_lg(cplx<T>* spec, const RowPtrsW& EB, const RowPtrs& J, int64_t rows, int n2, int n3, bool d3, bool faraday, bool wb,
                             const ModeTables<T>& t, T a2, T a3, cudaStream_t s) {
    if (!RowFft<T, LG>::table(t) || !t.twN || !t.S || !t.cj1 || !t.cj) return cudaErrorInvalidValue;
    constexpr int TT = RowFft<T, LG>::TT, most = row_threads<T, LG>();
    const unsigned nfl = faraday ? 3u : 6u;
    const size_t full = smem_for<T, LG>(most);
    const auto any = (const void*)k_ampere_reg<T, LG, true, true, false>;                        // the launch bounds of all
    cudaError_t e = room(any, full, upd_blocks<T, LG>());
    if (e != cudaSuccess) return e;
    const unsigned resident = (unsigned)resident_grid(any, most, full) / 6u * 6u;
    const bool tm = resident && (rows * TT + most - 1) / most * nfl >= (int64_t)kTmRounds * resident;
    const int th = tm ? most : threads_for<T, LG>(rows * nfl);
    const unsigned blocks = tm ? resident : (unsigned)((rows + th / TT - 1) / (th / TT) * nfl);
    const size_t smem = smem_for<T, LG>(th);
    const cplx<T>* tw = RowFft<T, LG>::table(t);
    if (faraday) {
        RowPtrsW B{};
        for (int c = 0; c < 3; c++) B.p[c] = EB.p[3 + c];
        const auto kern = d3 ? (tm ? k_faraday_reg<T, LG, true, true> : k_faraday_reg<T, LG, true, false>)
                             : (tm ? k_faraday_reg<T, LG, false, true> : k_faraday_reg<T, LG, false, false>);
        e = room((const void*)kern, full, upd_blocks<T, LG>());
        if (e != cudaSuccess) return e;
        kern<<<blocks, th, smem, s>>>(spec, B, (unsigned)rows, n2, n3, tw, t.twN, t.S, a2, a3);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const auto kern = d3 ? (wb ? (tm ? k_ampere_reg<T, LG, true, true, true> : k_ampere_reg<T, LG, true, true, false>)
                               : (tm ? k_ampere_reg<T, LG, true, false, true> : k_ampere_reg<T, LG, true, false, false>))
                         : (wb ? (tm ? k_ampere_reg<T, LG, false, true, true> : k_ampere_reg<T, LG, false, true, false>)
                               : (tm ? k_ampere_reg<T, LG, false, false, true> : k_ampere_reg<T, LG, false, false, false>));
    e = room((const void*)kern, full, upd_blocks<T, LG>());
    if (e != cudaSuccess) return e;
    kern<<<blocks, th, smem, s>>>(spec, J, EB, (unsigned)rows, n2, n3, tw, t.twN, t.S, t.cj1, t.cj, a2, a3, nfl);
    return cudaGetLastError();
}

}  // namespace hyb
