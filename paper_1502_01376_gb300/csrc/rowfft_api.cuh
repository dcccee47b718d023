// rowfft_api.cuh -- the register-resident row transforms (rowfft.cu) as the three-pass path calls them.
#pragma once
#include "hyb_internal.cuh"

namespace hyb {

struct RowPtrs { const void* p[9]; };
struct RowPtrsW { void* p[9]; };

// FP32 rows of n1 = 128 .. 8192 points; rows of up to nine fields are counted in 32 bits
bool row_reg_supported(int n1, int64_t rows);
cudaError_t row_reg_rfft(const RowPtrs& p, int nf, float2* out, int n1, int64_t rows, const ModeTables<float>& t, cudaStream_t s);
cudaError_t row_reg_irfft(const float2* in, const RowPtrsW& p, int nf, int n1, int64_t rows, const ModeTables<float>& t, cudaStream_t s);
cudaError_t row_reg_ampere(float2* spec, const RowPtrsW& p, int n1, int64_t rows, int n2, int n3, bool d3, bool wb, const ModeTables<float>& t,
                           float a2, float a3, cudaStream_t s);

}  // namespace hyb
