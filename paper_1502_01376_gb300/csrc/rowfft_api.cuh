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
// A step in FP32, by the cells of the grid (us per step; the fields whose rows are transformed before the updates):
//   all nine, then Faraday, then row_reg_ampere: small grids, where the three launches' own time counts and a second
//     transform in the last one shows (8192 x 64 29 against 31, 8192 x 128 45 against 47, 1024 x 300 17 against 18.5);
//   E and B, j inside the update (row_reg_update): 4096 x 1024 140 -> 130, 8192 x 512 157 -> 152, 4096 x 64 x 16 149 -> 141;
//   E only, B and j inside the updates (row_reg_update, faraday): rows of up to 1024 points, whose transforms are short
//     against the passes they save (1024 x 777 29 -> 25, 512 x 4000 58 -> 51, 1024 x 128 x 32 117 -> 113), and any rows of
//     grids many times the L2 (1024 x 256 x 256 1832 -> 1625, 2048 x 64 x 64 259 -> 240, 8192 x 64 x 64 1218 -> 1193;
//     but 8192 x 512 152 and 162, 2048 x 64 x 16 72 and 75).
enum class RowForm { kAll, kEB, kE };
inline RowForm row_form(int n1, int64_t cells) {
    if (n1 <= 1024) return cells < (int64_t)1 << 19 ? RowForm::kAll : RowForm::kE;
    if (cells <= (int64_t)1 << 20) return RowForm::kAll;
    return cells >= (int64_t)1 << 23 ? RowForm::kE : RowForm::kEB;
}
// The updates of a step with the transforms that run inside them (spec: E's spectra).  faraday: B's rows are transformed,
// updated, stored as spectra and as rows; without it B's updated spectra are in spec and their rows are written.  Then Ampere
// with j's transforms, and E's rows; wb: E's updated spectra are stored too.
cudaError_t row_reg_update(float2* spec, const RowPtrsW& EB, const RowPtrs& J, int n1, int64_t rows, int n2, int n3, bool d3, bool faraday, bool wb,
                           const ModeTables<float>& t, float a2, float a3, cudaStream_t s);
cudaError_t row_reg_rfft(const RowPtrs& p, int nf, double2* out, int n1, int64_t rows, const ModeTables<double>& t, cudaStream_t s);
cudaError_t row_reg_irfft(const double2* in, const RowPtrsW& p, int nf, int n1, int64_t rows, const ModeTables<double>& t, cudaStream_t s);
cudaError_t row_reg_ampere(double2* spec, const RowPtrsW& p, int n1, int64_t rows, int n2, int n3, bool d3, bool wb, const ModeTables<double>& t,
                           double a2, double a3, cudaStream_t s);

}  // namespace hyb
