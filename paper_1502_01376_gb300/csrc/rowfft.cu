// rowfft.cu -- the batched row transforms of the three-pass path for FP32 rows of 128 .. 8192 points.
#include "rowfft_kernels.cuh"

namespace hyb {

#define HYB_ROW_LG(CALL)                    \
    switch (31 - __builtin_clz(n1 / 2)) {   \
        case 6: return CALL(6);             \
        case 7: return CALL(7);             \
        case 8: return CALL(8);             \
        case 9: return CALL(9);             \
        case 10: return CALL(10);           \
        case 11: return CALL(11);           \
        case 12: return CALL(12);           \
        default: return cudaErrorInvalidValue; \
    }

template <> bool row_reg_supported<float>(int n1, int64_t rows) { return n1 >= 128 && n1 <= 8192 && rows <= (int64_t)1 << 27; }

cudaError_t row_reg_rfft(const RowPtrs& p, int nf, float2* out, int n1, int64_t rows, const ModeTables<float>& t, cudaStream_t s) {
#define HYB_CALL(LG) rfft_lg<float, LG>(p, nf, out, rows, t, s)
    HYB_ROW_LG(HYB_CALL)
#undef HYB_CALL
}
cudaError_t row_reg_irfft(const float2* in, const RowPtrsW& p, int nf, int n1, int64_t rows, const ModeTables<float>& t, cudaStream_t s) {
#define HYB_CALL(LG) irfft_lg<float, LG>(in, p, nf, rows, t, s)
    HYB_ROW_LG(HYB_CALL)
#undef HYB_CALL
}
cudaError_t row_reg_ampere(float2* spec, const RowPtrsW& p, int n1, int64_t rows, int n2, int n3, bool d3, bool wb, const ModeTables<float>& t,
                           float a2, float a3, cudaStream_t s) {
#define HYB_CALL(LG) ampere_lg<float, LG>(spec, p, rows, n2, n3, d3, wb, t, a2, a3, s)
    HYB_ROW_LG(HYB_CALL)
#undef HYB_CALL
}
cudaError_t row_reg_update(float2* spec, const RowPtrsW& EB, const RowPtrs& J, int n1, int64_t rows, int n2, int n3, bool d3, bool faraday, bool wb,
                           const ModeTables<float>& t, float a2, float a3, cudaStream_t s) {
#define HYB_CALL(LG) update_lg<float, LG>(spec, EB, J, rows, n2, n3, d3, faraday, wb, t, a2, a3, s)
    HYB_ROW_LG(HYB_CALL)
#undef HYB_CALL
}

}  // namespace hyb
