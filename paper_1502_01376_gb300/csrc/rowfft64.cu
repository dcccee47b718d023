// rowfft64.cu -- the batched row transforms of the three-pass path for small FP64 grids with short rows.
#include "rowfft_kernels.cuh"

namespace hyb {

#define HYB_ROW_LG(CALL)                    \
    switch (31 - __builtin_clz(n1 / 2)) {   \
        case 5: return CALL(5);             \
        case 6: return CALL(6);             \
        case 7: return CALL(7);             \
        default: return cudaErrorInvalidValue; \
    }

template <> bool row_reg_supported<double>(int n1, int64_t rows) { return n1 >= 64 && n1 <= 256 && rows * n1 <= kReg64Cells; }

cudaError_t row_reg_rfft(const RowPtrs& p, int nf, double2* out, int n1, int64_t rows, const ModeTables<double>& t, cudaStream_t s) {
#define HYB_CALL(LG) rfft_lg<double, LG>(p, nf, out, rows, t, s)
    HYB_ROW_LG(HYB_CALL)
#undef HYB_CALL
}
cudaError_t row_reg_irfft(const double2* in, const RowPtrsW& p, int nf, int n1, int64_t rows, const ModeTables<double>& t, cudaStream_t s) {
#define HYB_CALL(LG) irfft_lg<double, LG>(in, p, nf, rows, t, s)
    HYB_ROW_LG(HYB_CALL)
#undef HYB_CALL
}
cudaError_t row_reg_ampere(double2* spec, const RowPtrsW& p, int n1, int64_t rows, int n2, int n3, bool d3, bool wb, const ModeTables<double>& t,
                           double a2, double a3, cudaStream_t s) {
#define HYB_CALL(LG) ampere_lg<double, LG>(spec, p, rows, n2, n3, d3, wb, t, a2, a3, s)
    HYB_ROW_LG(HYB_CALL)
#undef HYB_CALL
}

}  // namespace hyb
