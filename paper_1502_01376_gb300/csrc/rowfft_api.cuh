// rowfft_api.cuh -- the register-resident row transforms (rowfft.cu) as the three-pass path calls them.
#pragma once
#include "hyb_internal.cuh"

namespace hyb {

struct RowPtrs { const void* p[9]; };
struct RowPtrsW { void* p[9]; };

// Whether they take `rows` rows of n1 points.  FP32: n1 = 128 .. 8192 (rows of up to nine fields are counted in 32
// bits).  FP64: n1 = 64 .. 256 and at most 65536 cells; beyond that the FP64 units are busy and the four-point passes, which
// take more operations than the shared-memory transform's radix 8, lose (a step of 128 x 64: 18.5 against 26.7 us, 256 x 200
// 36 against 41, 128 x 500 41 against 51, 256 x 500 83 against 82, 256 x 1000 154 against 141).
constexpr int64_t kReg64Cells = 1 << 16;
template <typename T> bool row_reg_supported(int n1, int64_t rows);
template <> bool row_reg_supported<float>(int n1, int64_t rows);
template <> bool row_reg_supported<double>(int n1, int64_t rows);
cudaError_t row_reg_rfft(const RowPtrs& p, int nf, float2* out, int n1, int64_t rows, const ModeTables<float>& t, cudaStream_t s);
cudaError_t row_reg_irfft(const float2* in, const RowPtrsW& p, int nf, int n1, int64_t rows, const ModeTables<float>& t, cudaStream_t s);
cudaError_t row_reg_ampere(float2* spec, const RowPtrsW& p, int n1, int64_t rows, int n2, int n3, bool d3, bool wb, const ModeTables<float>& t,
                           float a2, float a3, cudaStream_t s);
cudaError_t row_reg_rfft(const RowPtrs& p, int nf, double2* out, int n1, int64_t rows, const ModeTables<double>& t, cudaStream_t s);
cudaError_t row_reg_irfft(const double2* in, const RowPtrsW& p, int nf, int n1, int64_t rows, const ModeTables<double>& t, cudaStream_t s);
cudaError_t row_reg_ampere(double2* spec, const RowPtrsW& p, int n1, int64_t rows, int n2, int n3, bool d3, bool wb, const ModeTables<double>& t,
                           double a2, double a3, cudaStream_t s);

}  // namespace hyb
