// rowfft_kernels.cuh -- the kernels of the register-resident row transforms (rowfft.cuh) and their launches, one
// precision per translation unit (rowfft.cu, rowfft64.cu): the forward transform, the inverse, and the inverse
// with the Ampere update of the E fields formed as their spectra are loaded.
#pragma once
#include <algorithm>

#include "rowfft.cuh"
#include "rowfft_api.cuh"

namespace hyb {

// the largest block, whole teams, and the blocks per SM its registers are held to: 64 registers a thread, FP64 128
template <typename T, int LG> constexpr int row_threads() { return RowFft<T, LG>::TT > 256 ? RowFft<T, LG>::TT : 256; }
template <typename T, int LG> constexpr int row_blocks() { return (sizeof(T) == 4 ? 1024 : 512) / row_threads<T, LG>(); }

template <typename T, int LG>
__device__ __forceinline__ RowFft<T, LG> row_team(unsigned char* smem, const cplx<T>* tw, int* team) {
    using F = RowFft<T, LG>;
    F f;
    *team = threadIdx.x / F::TT;
    f.t = threadIdx.x % F::TT;
    f.bar = 1 + *team;
    f.a = reinterpret_cast<cplx<T>*>(smem) + (size_t)*team * 2 * F::M;
    f.b = f.a + F::M;
    f.tw = tw;
    return f;
}

// Persistent: a block takes groups of blockDim / TT rows (row j of the nf fields' rows: field j / rows) and holds the next
// group's samples in registers while it transforms the current one.
template <typename T, int LG>
__global__ void __launch_bounds__((row_threads<T, LG>()), (row_blocks<T, LG>())) k_rfft_reg(const __grid_constant__ RowPtrs in, cplx<T>* __restrict__ out, unsigned rows,
                                                                                     unsigned total, const cplx<T>* __restrict__ tw,
                                                                                     const cplx<T>* __restrict__ twN) {
    using F = RowFft<T, LG>;
    using C = cplx<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int team;
    F f = row_team<T, LG>(smem_raw, tw, &team);
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
    for (unsigned g = blockIdx.x * R; g < total; g += step, j += step) {
        C v[F::P];
#pragma unroll
        for (int i = 0; i < F::P; i++) v[i] = nx[i];
        const bool live = j < total;
        if (total - j > step) fetch(j + step);                 // (unsigned: also when j is past the end)
        C* const X = out + (size_t)(live ? j : 0) * (F::M + 1);
        f.forward(v, twN, [&](int k, C x) { if (live) X[k] = x; });
    }
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
    f.inverse(v, twN, [&](int k) { return X[k]; });
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
        f.inverse(v, twN, [&](int k) {
            C e = axpy(Xr[k], a2, csub(Xr[5 * fs + k], Xm2[5 * fs + k]));
            if (D3) e = axpy(e, -a3, csub(Xr[4 * fs + k], Xm3[4 * fs + k]));
            return keep(Xr + k, axpy(e, -cj1[k], Xr[6 * fs + k]));
        });
    } else if (fl == 1) {
        f.inverse(v, twN, [&](int k) {
            const C s = S[k], b3 = Xr[5 * fs + k];
            C e = Xr[fs + k];
            e = mkc<C>(e.x + (s.x * b3.x + s.y * b3.y), e.y + (s.x * b3.y - s.y * b3.x));        // - Sm B3 = conj(S) B3
            if (D3) e = axpy(e, a3, csub(Xr[3 * fs + k], Xm3[3 * fs + k]));
            return keep(Xr + fs + k, axpy(e, -cj[k], Xr[7 * fs + k]));
        });
    } else if (fl == 2) {
        f.inverse(v, twN, [&](int k) {
            const C s = S[k], b2 = Xr[4 * fs + k];
            C e = Xr[2 * fs + k];
            e = mkc<C>(e.x - (s.x * b2.x + s.y * b2.y), e.y - (s.x * b2.y - s.y * b2.x));        // + Sm B2
            e = axpy(e, -a2, csub(Xr[3 * fs + k], Xm2[3 * fs + k]));
            return keep(Xr + 2 * fs + k, axpy(e, -cj[k], Xr[8 * fs + k]));
        });
    } else {
        const C* X = Xr + fl * fs;
        f.inverse(v, twN, [&](int k) { return X[k]; });
    }
    if (live) {
        C* z = reinterpret_cast<C*>(out.p[fl]) + (size_t)row * F::M;
        const T inv = (T)1 / (T)F::M;
#pragma unroll
        for (int i = 0; i < F::P; i++) z[f.t + F::TT * i] = cscale(v[i], inv);
    }
}

// ---------------------------------------------------------------- launches
// threads of a block: the largest, fewer while that leaves under about four blocks per SM
template <typename T, int LG>
static int threads_for(int64_t total_rows) {
    constexpr int TT = RowFft<T, LG>::TT;
    int th = row_threads<T, LG>();
    while (th > std::max(TT, 32) && total_rows < (int64_t)(th / TT) * 600) th >>= 1;
    return th;
}
template <typename T, int LG>
static size_t smem_for(int threads) { return sizeof(cplx<T>) * 2 * RowFft<T, LG>::M * (size_t)(threads / RowFft<T, LG>::TT); }
static cudaError_t room(const void* kern, size_t smem_max) {
    cudaError_t e = func_attr_once(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
    return e == cudaSuccess ? func_attr_once(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100) : e;
}

template <typename T, int LG>
static cudaError_t rfft_lg(const RowPtrs& p, int nf, cplx<T>* out, int64_t rows, const ModeTables<T>& t, cudaStream_t s) {
    if (!RowFft<T, LG>::table(t) || !t.twN) return cudaErrorInvalidValue;
    const auto kern = k_rfft_reg<T, LG>;
    cudaError_t e = room((const void*)kern, smem_for<T, LG>((row_threads<T, LG>())));
    if (e != cudaSuccess) return e;
    const int64_t total = rows * nf;
    const int th = threads_for<T, LG>(total), R = th / RowFft<T, LG>::TT;
    const size_t smem = smem_for<T, LG>(th);
    const int64_t blocks = std::min<int64_t>((total + R - 1) / R, resident_grid((const void*)kern, th, smem));
    kern<<<(unsigned)blocks, th, smem, s>>>(p, out, (unsigned)rows, (unsigned)total, RowFft<T, LG>::table(t), t.twN);
    return cudaGetLastError();
}
template <typename T, int LG>
static cudaError_t irfft_lg(const cplx<T>* in, const RowPtrsW& p, int nf, int64_t rows, const ModeTables<T>& t, cudaStream_t s) {
    if (!RowFft<T, LG>::table(t) || !t.twN) return cudaErrorInvalidValue;
    const auto kern = k_irfft_reg<T, LG>;
    cudaError_t e = room((const void*)kern, smem_for<T, LG>((row_threads<T, LG>())));
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
    cudaError_t e = room((const void*)kern, smem_for<T, LG>((row_threads<T, LG>())));
    if (e != cudaSuccess) return e;
    const int th = threads_for<T, LG>(rows * 6), R = th / RowFft<T, LG>::TT;
    kern<<<(unsigned)((rows + R - 1) / R * 6), th, smem_for<T, LG>(th), s>>>(spec, p, (unsigned)rows, n2, n3, RowFft<T, LG>::table(t), t.twN, t.S, t.cj1, t.cj,
                                                                            a2, a3);
    return cudaGetLastError();
}

}  // namespace hyb
