// Launch interface of the smoothing and resampling kernels (internal to libmamute).
#pragma once

#include <cuda_runtime.h>

namespace mamute {

// Coefficients of one tridiagonal solve (s - mu D) u = f along a row of n
// cells (see postproc.cu): the ratio r + rlo, K, r^len for a lane's length,
// r^(n mod len) for the last lane's, r^n and 1 / (1 - r^{2n}).
struct alignas(16) RowCoef {
  float r, rlo, K, rl, rt, rn, w, pad;
};

// A ratio r in (0, 1) with d = 1 - r as hi + lo, to the accuracy of d: FP32
// alone would round d, and with it the length of the filter, by 6e-8 / d.
__host__ __device__ inline void split_ratio(double r, double d, float* hi, float* lo) {
  *hi = (float)r;
  *lo = (float)(*hi >= 0.5f ? (1.0 - (double)*hi) - d : r - (double)*hi);
}

RowCoef row_coef_host(double s, double mu, int n);
// Row (ky, kz) of DCT modes: s = 1 + my lambda_ky + mz lambda_kz, lambda_k =
// 4 sin^2(pi k / (2 n)); out [nz][ny].
cudaError_t launch_row_coef(RowCoef* out, int ny, int nz, double my, double mz, double mx, int nx,
                            cudaStream_t s);
// Solves every row of [rows][n] (coef: one set per row, or NULL: `one` for
// all); in may be out.  scratch: an array like out (not in or out) where
// rows_need_scratch(n), else unused.
bool rows_need_scratch(int n);
cudaError_t launch_rows(const float* in, float* out, float* scratch, int n, long long rows,
                        const RowCoef* coef, const RowCoef& one, cudaStream_t s);
// The lines of one axis of a volume below: element (L, j) of line L is at
// (L / inner) * outer + (L % inner) + j * st.
//
// Solves every line with the factors of its matrix, g[0 .. n] (as hi and lo,
// g_0 = g_n = 0) and inv[0 .. n - 1]: z_j = f_j + g_j z_{j-1}, u_j = inv_j z_j +
// g_{j+1} u_{j+1}; in may be out.  carry: with the sums' rounding errors, for
// filters of more than kCarryCells cells.
constexpr double kCarryCells = 64.0;
cudaError_t launch_sweep(const float* in, float* out, const float2* g, const float* inv, bool carry, int n,
                         long long lines, long long inner, long long outer, long long st,
                         cudaStream_t s);
// Orthonormal DCT-II of every line (inverse: its transpose) from the half
// matrices E and O (see dct_kernel); in and out differ.
cudaError_t launch_dct(const float* in, float* out, const float* E, const float* O, bool inverse,
                       int n, long long lines, long long inner, long long outer, long long st,
                       cudaStream_t s);
// y[r][m] = sum_{j < len[m]} w[j][m] x[r][c0[m] + j] for every trace r: a
// banded matrix whose row m covers the contiguous columns c0[m] ..
// c0[m] + len[m] - 1, weights stored tap-major (w[j][m] at j n_out + m);
// taps is the largest len[m].
cudaError_t launch_band_rows(const float* x, int n_in, const int* c0, const int* len,
                             const float* w, int taps, int n_out, int n_traces, float* y,
                             cudaStream_t s);

// out = a - b elementwise.
cudaError_t launch_sub(const float* a, const float* b, long long n, float* out, cudaStream_t s);

}  // namespace mamute
