// Launch interface of the smoothing and resampling kernels (internal to libmamute).
#pragma once

#include <cuda_runtime.h>

namespace mamute {

// Coefficients of one tridiagonal solve (s - mu D) u = f along a row of n
// cells (see postproc.cu): r, K, r^len for the per-lane length, r^n and
// 1 / (1 - r^{2n}).
struct RowCoef {
  float r, K, rl, rn, w;
};

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
// Solves every line with the factors fac[j] = (inv_j, g_j) of its matrix:
// y_j = inv_j f_j + g_j y_{j-1}, u_j = y_j + g_j u_{j+1}; in may be out.
cudaError_t launch_sweep(const float* in, float* out, const float2* fac, int n, long long lines,
                         long long inner, long long outer, long long st, cudaStream_t s);
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
