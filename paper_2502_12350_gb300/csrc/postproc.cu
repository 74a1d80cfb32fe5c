// Gradient smoothing filters and seismic-data time resampling.
//
// Smoothing (Sec. 2, FWI gradient preconditioning: Bessel or Laplace filter
// with lengths lx, ly, lz; Algorithm 3: GradientPreconditioning).  Both
// filters are inverses of operators built from the 3-point second difference
// D with reflecting ends, and both are applied exactly.
//   Laplace, prod_a (I - l_a^2 D_aa)^-1: one tridiagonal solve per axis, along
// x by row_kernel, along y and z by sweep_kernel.
//   Bessel, (I - sum_a l_a^2 D_aa)^-1: the orthonormal DCT-II diagonalises D
// along y and z, with eigenvalues -4 sin^2(pi k / (2 n)), so after the
// transforms along y and z (dct_kernel) every row is one tridiagonal system
// along x with its own diagonal (row_kernel), and the transposed transforms
// along z and y follow.
// The 600x600x200 Bessel filter takes 2.92 ms, 2.7 of them the transforms; six
// dense transforms and a spectral multiplier took 15.9.
//
// Resampling (Sec. 2: time interpolation by nearest neighbour or sinc;
// Table 1 Interpolate).  The resampling of every trace is the same sparse
// matrix, built on the host in FP64 (see api.cu); each of its rows covers a
// contiguous run of input samples, so it is stored as a band (first column,
// length, tap-major weights) and applied to every trace by band_rows_kernel;
// its transpose is another banded matrix.
#include "postproc.h"

#include <cmath>
#include <cstdint>
#include <type_traits>

namespace mamute {

namespace {

// ---- tridiagonal solves (s - mu D) u = f with reflecting ends ----
//
// The inverse on the line is u_i = K (p_i + r q_{i+1}) with the recursions
// p_i = f_i + r p_{i-1} and q_i = f_i + r q_{i+1}, r in (0, 1) the root of
// mu r^2 - (s + 2 mu) r + mu = 0 and K = (1 - r) / (s (1 + r)); the
// reflecting ends are the even images of f, which enter only through
// p_{-1} = (q0 + r^n p0) / (1 - r^{2n}) (q0, p0: q_0 and p_{n-1} of the line
// alone) and q_n = p_{n-1}.  All terms have the sign of f: no cancellation.

// Formed in FP64 from x = 1 / r - 1 = a + sqrt(a (a + 2)), a = s / (2 mu), which
// gives 1 - r without a cancellation however long the filter.
__host__ __device__ inline RowCoef row_coef(double s, double mu, int n, int len) {
  const double a = s / (2.0 * mu), x = a + sqrt(a) * sqrt(a + 2.0);
  const double r = 1.0 / (1.0 + x), d = x / (1.0 + x);
  const double lr = r < 0.5 ? log(r) : log1p(-d);
  RowCoef c{};
  split_ratio(r, d, &c.r, &c.rlo);
  c.K = (float)(d / (s * (1.0 + r)));
  c.rl = (float)exp(len * lr);
  c.rt = (float)exp(n % len * lr);
  c.rn = (float)exp(n * lr);
  c.w = (float)(-1.0 / expm1(2.0 * n * lr));
  return c;
}

// One coefficient set per row (y, z) of DCT modes along y and z.
__global__ void row_coef_kernel(RowCoef* out, int ny, int nz, double my, double mz, double mu, int n,
                                int len) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= ny * nz) return;
  const double sy = sinpi(0.5 * (double)(q % ny) / ny), sz = sinpi(0.5 * (double)(q / ny) / nz);
  out[q] = row_coef(1.0 + 4.0 * (my * sy * sy + mz * sz * sz), mu, n, len);
}

// Solves along x, one row per warp.  Lane l owns the `len` cells from l len
// (len odd: no bank conflicts), runs both recursions on them from zero, takes
// the others' part from a warp scan, and runs them again from the true start.
// The row is staged in shared memory (row and p, 8 bytes a cell) so that
// DRAM sees one read and one write, or, for rows beyond kRowSmem bytes, left
// in global memory with p in `scratch`.  Bound by HBM and the shared-memory
// accesses (about 9 a cell), so that the second multiply-add of a step, for the
// low part of r, costs 10 us of the 2.92 ms of the 600x600x200 Bessel filter.
// Without it the length that was applied was off by 6e-8 of itself per cell of
// it (relative L2 errors on zero-mean rows of 700 cells 1.9e-6 at 200 cells, now
// 2.4e-7; no result above 3e7, where r rounds to 1).  What is left are the roundings of
// the lanes' sums and of the scan: below 1e-6 however long the filter.
__global__ void row_kernel(const float* in, float* out, float* scratch, int n, int len,
                           long long rows, const RowCoef* __restrict__ coef, RowCoef one, bool staged) {
  extern __shared__ float row_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  for (long long row = (long long)blockIdx.x * warps + warp; row < rows;
       row += (long long)gridDim.x * warps) {
    const RowCoef c = coef ? coef[row] : one;
    const float* f = in + row * n;
    float* p = scratch + row * n;
    float* o = out + row * n;
    if (staged) {
      float* sf = row_smem + (size_t)warp * 2 * n;
      __syncwarp();
      for (int j = lane; j < n; j += 32) sf[j] = f[j];
      __syncwarp();
      f = sf;
      p = sf + n;
    }
    const int b = min(lane * len, n), e = min(b + len, n);
    auto times_r = [&](float v, float add) { return fmaf(c.r, v, fmaf(c.rlo, v, add)); };
    float cp = 0.0f, cq = 0.0f;  // p of the last and q of the first owned cell, from zero
    for (int j = b; j < e; ++j) cp = times_r(cp, f[j]);
    for (int j = e - 1; j >= b; --j) cq = times_r(cq, f[j]);
    float ap = e - b == len ? c.rl : (e > b ? c.rt : 1.0f), aq = ap;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const float pc = __shfl_up_sync(0xffffffffu, cp, d), pa = __shfl_up_sync(0xffffffffu, ap, d);
      const float qc = __shfl_down_sync(0xffffffffu, cq, d), qa = __shfl_down_sync(0xffffffffu, aq, d);
      if (lane >= d) {
        cp = fmaf(ap, pc, cp);
        ap *= pa;
      }
      if (lane + d < 32) {
        cq = fmaf(aq, qc, cq);
        aq *= qa;
      }
    }
    const float pend = __shfl_sync(0xffffffffu, cp, 31), q0 = __shfl_sync(0xffffffffu, cq, 0);
    const float pm1 = c.w * fmaf(c.rn, pend, q0), qn = fmaf(c.rn, pm1, pend);
    // the neighbouring lanes' inclusive values, and the ends
    const float pc = __shfl_up_sync(0xffffffffu, cp, 1), pa = __shfl_up_sync(0xffffffffu, ap, 1);
    const float qc = __shfl_down_sync(0xffffffffu, cq, 1), qa = __shfl_down_sync(0xffffffffu, aq, 1);
    float pv = lane == 0 ? pm1 : fmaf(pa, pm1, pc);
    float qv = lane == 31 ? qn : fmaf(qa, qn, qc);
    for (int j = b; j < e; ++j) {
      pv = times_r(pv, f[j]);
      p[j] = pv;
    }
    float* res = staged ? p : o;
    for (int j = e - 1; j >= b; --j) {
      const float fj = f[j];
      res[j] = c.K * times_r(qv, p[j]);
      qv = times_r(qv, fj);
    }
    if (staged) {
      __syncwarp();
      for (int j = lane; j < n; j += 32) o[j] = p[j];
    }
  }
}

constexpr int kRowSmem = 200 * 1024;

// v <- g v + f, g as hi + lo.  CARRY: v as hi + lo too, lo taking what the
// rounding of hi drops (the product's and the sum's errors); one multiply-add
// lies on the chain of hi and one on that of lo.
template <bool CARRY>
__device__ __forceinline__ void recur(float& hi, float& lo, float g, float glo, float f) {
  if (!CARRY) {
    hi = fmaf(g, hi, fmaf(glo, hi, f));
    return;
  }
  const float s = fmaf(g, hi, f);
  const float p = __fmul_rn(g, hi), pe = fmaf(glo, hi, fmaf(g, hi, -p));
  // s - p = b + be exactly
  const float b = __fsub_rn(s, p), q = __fsub_rn(s, b);
  const float be = __fadd_rn(__fsub_rn(s, __fadd_rn(b, q)), __fsub_rn(q, p));
  lo = fmaf(g, lo, __fadd_rn(__fsub_rn(__fsub_rn(f, b), be), pe));
  hi = s;
}

// Solves along y or z in place, one column per thread (consecutive threads on
// consecutive x): z_i = f_i + g_i z_{i-1} upwards and u_i = inv_i z_i + g_{i+1}
// u_{i+1} downwards, with the factors of the one matrix all columns share
// (formed on the host in FP64; every g is below 1, g_0 = g_n = 0).  Two reads and
// two writes of the volume; the loads of 8 cells are issued together.
//
// CARRY for filters beyond kCarryCells: the roundings of v add up over a filter's
// length (relative L2 errors of 1.3e-7 at 30 cells, 2.2e-7 at 100 and 1.7e-6 at
// 30,000 on lines of 700, where dense transforms have 3.3e-7, 4.0e-7 and 1.0e-6);
// carried they stay below 1e-7.  The Laplace filter of 600x600x200 takes 622 us
// without and 672 with it (4 blocks per SM without: with 3 it takes 700).
template <bool CARRY>
__global__ void __launch_bounds__(256, CARRY ? 3 : 4) sweep_kernel(const float* in, float* out,
                                                    const float2* __restrict__ g,
                                                    const float* __restrict__ inv, int n,
                                                    long long lines, long long inner,
                                                    long long outer, long long st) {
  const long long L = blockIdx.x * 256LL + threadIdx.x;
  if (L >= lines) return;
  const long long base = (L / inner) * outer + L % inner;
  const float* f = in + base;
  float* u = out + base;
  float hi = 0.0f, lo = 0.0f;
  for (int i0 = 0; i0 < n; i0 += 8) {
    float t[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) t[k] = i0 + k < n ? f[(i0 + k) * st] : 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (i0 + k < n) {
        const float2 c = __ldg(g + i0 + k);
        recur<CARRY>(hi, lo, c.x, c.y, t[k]);
        u[(i0 + k) * st] = CARRY ? hi + lo : hi;
      }
  }
  hi = lo = 0.0f;
  for (int i0 = (n - 1) / 8 * 8; i0 >= 0; i0 -= 8) {
    float t[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) t[k] = i0 + k < n ? u[(i0 + k) * st] : 0.0f;
#pragma unroll
    for (int k = 7; k >= 0; --k)
      if (i0 + k < n) {
        const float2 c = __ldg(g + i0 + k + 1);
        recur<CARRY>(hi, lo, c.x, c.y, __ldg(inv + i0 + k) * t[k]);
        u[(i0 + k) * st] = CARRY ? hi + lo : hi;
      }
  }
}

// ---- DCT-II along y or z ----
//
// The even modes are symmetric about the middle of the line and the odd ones
// antisymmetric, so the n x n product splits into two of half the size on the
// sums and differences of the mirrored cells (half the operations, shorter
// sums).  A block makes 64 even and 64 odd modes (inverse: 64 mirrored pairs
// of cells) of 128 lines: half of its 256 threads the product with E, half that
// with O, 8 lines x 8 outputs each, fed by float4 shared-memory reads, with the
// next chunk's global loads in registers while a chunk is multiplied; the two
// products of an output meet in shared memory at the end.  Bound by issue and
// the shared-memory reads, 4 for 32 packed multiply-adds: 680 us a launch at
// 600x600x200, 0.49 of the FP32 peak (8 lines x 4 outputs of both products per
// thread, 3 reads for 16 packed multiply-adds: 3.37 ms for the filter).
constexpr int kTL = 128, kTI = 64, kTK = 8;
constexpr int kAP = kTL + 4;  // A row pitch

// forward (INV = false): out[2 i] = sum_j E[j][i] (f_j + f_{n-1-j}),
//   out[2 i + 1] = sum_j O[j][i] (f_j - f_{n-1-j}) over j < h = ceil(n / 2)
//   (the middle cell of an odd n counts once);
// inverse: e_i = sum_j E[j][i] F_{2j}, o_i = sum_j O[j][i] F_{2j+1},
//   out[i] = e_i + o_i, out[n-1-i] = e_i - o_i.
// E and O are [h][h], zero-padded.
template <bool INV>
__global__ void __launch_bounds__(256, 2)
    dct_kernel(const float* __restrict__ in, float* __restrict__ out, const float* __restrict__ E,
               const float* __restrict__ O, int n, long long lines, long long inner,
               long long outer, long long st) {
  __shared__ union {
    struct {
      __align__(16) float a[2][2][kTK][kAP], b[2][2][kTK][kTI];
    } s;
    float x[32][256];  // the other product's half of a tile, at the end
  } sm;
  auto& As = sm.s.a;
  auto& Bs = sm.s.b;
  const int h = (n + 1) / 2;
  // warps 0 to 3 make the product with E (v = 0), 4 to 7 that with O; a warp
  // holds 4 x 8 of the product's 8 x 16 threads
  const int tid = threadIdx.x, v = tid >> 7;
  const int tx = (tid & 3) + (tid >> 5 & 1) * 4, ty = (tid >> 2 & 7) + (tid >> 6 & 1) * 8;
  const long long L0 = (long long)blockIdx.x * kTL;
  const int i0 = blockIdx.y * kTI;
  // loads: 128 lines x 8 cells x 2 = 4 pairs per thread (one line each), and
  // 8 x 64 of each matrix = 2 per thread
  const int al = tid & (kTL - 1), aj = tid / kTL;
  const long long LA = L0 + al;
  const bool lok = LA < lines;
  const float* src = in + (lok ? (LA / inner) * outer + LA % inner : 0);
  const int bi = tid & (kTI - 1), bj = tid / kTI;
  float ra[2][4], rb[2][2];
  // cells p and q of the thread's next pair, and from one pair to its next
  const float* fp = src + (INV ? 2 * aj : aj) * st;
  const float* fq = src + (INV ? 2 * aj + 1 : n - 1 - aj) * st;
  const long long dp = (INV ? 4 : 2) * st, dq = INV ? dp : -dp;
  const float* ep = E + (long long)bj * h + i0 + bi;
  const float* op = O + (long long)bj * h + i0 + bi;
  const bool iok = i0 + bi < h;
  auto load = [&](int j0) {
    int j = j0 + aj;
#pragma unroll
    for (int k = 0; k < 4; ++k, j += 2) {
      const bool ok = lok && j < h;
      ra[0][k] = ok ? *fp : 0.0f;
      ra[1][k] = ok && (INV ? 2 * j + 1 < n : 2 * j + 1 != n) ? *fq : 0.0f;
      fp += dp;
      fq += dq;
    }
    j = j0 + bj;
#pragma unroll
    for (int k = 0; k < 2; ++k, j += 4) {
      rb[0][k] = iok && j < h ? __ldg(ep) : 0.0f;
      rb[1][k] = iok && j < h ? __ldg(op) : 0.0f;
      ep += 4 * h;
      op += 4 * h;
    }
  };
  auto stage = [&](int s) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      As[s][0][aj + 2 * k][al] = INV ? ra[0][k] : ra[0][k] + ra[1][k];
      As[s][1][aj + 2 * k][al] = INV ? ra[1][k] : ra[0][k] - ra[1][k];
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      Bs[s][0][bj + 4 * k][bi] = rb[0][k];
      Bs[s][1][bj + 4 * k][bi] = rb[1][k];
    }
  };
  float2 acc[4][8] = {};  // [two lines][output]
  load(0);
  stage(0);
  __syncthreads();
  int s = 0;
  for (int j0 = 0; j0 < h; j0 += kTK, s ^= 1) {
    const bool more = j0 + kTK < h;
    if (more) load(j0 + kTK);
#pragma unroll 2
    for (int k = 0; k < kTK; ++k) {
      // lines 4 ty .. and 64 + 4 ty .., outputs 4 tx .. and 32 + 4 tx ..: the
      // threads of a warp read consecutive float4s
      const float4 a0 = *reinterpret_cast<const float4*>(&As[s][v][k][ty * 4]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[s][v][k][64 + ty * 4]);
      const float4 b0 = *reinterpret_cast<const float4*>(&Bs[s][v][k][tx * 4]);
      const float4 b1 = *reinterpret_cast<const float4*>(&Bs[s][v][k][32 + tx * 4]);
      const float2 a[4] = {{a0.x, a0.y}, {a0.z, a0.w}, {a1.x, a1.y}, {a1.z, a1.w}};
      const float bb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int c = 0; c < 8; ++c)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[r][c] = __ffma2_rn(a[r], make_float2(bb[c], bb[c]), acc[r][c]);
    }
    if (more) stage(s ^ 1);
    __syncthreads();
  }
  // The two products of an output meet: a thread gives the other product's
  // thread the lines that that one writes (v = 0 lines 4 ty .., v = 1 the 64th
  // on), and writes its own lines' outputs p and q.
#pragma unroll
  for (int c = 0; c < 8; ++c)
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const float2 t = v == 0 ? acc[2 + r][c] : acc[r][c];
      sm.x[4 * c + 2 * r][tid] = t.x;
      sm.x[4 * c + 2 * r + 1][tid] = t.y;
    }
  __syncthreads();
  const long long L = L0 + 64 * v + ty * 4;
  if (L >= lines) return;
  // four consecutive lines share a 16-byte store where the layout allows it
  const long long b0 = (L / inner) * outer + L % inner;
  const bool vec = L % inner + 4 <= inner && ((b0 | st) & 3) == 0 && L + 4 <= lines &&
                   ((unsigned long long)out & 15) == 0;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int i = i0 + (c / 4) * 32 + tx * 4 + c % 4;
    if (i >= h) continue;
    const int p = INV ? i : 2 * i, q = INV ? n - 1 - i : 2 * i + 1;
    float e[4], o[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float2 m = v == 0 ? acc[r / 2][c] : acc[2 + r / 2][c];
      const float mine = r & 1 ? m.y : m.x, other = sm.x[4 * c + r][tid ^ 128];
      const float x = v == 0 ? mine : other, y = v == 0 ? other : mine;
      e[r] = INV ? x + y : x;
      o[r] = INV ? x - y : y;
    }
    if (vec) {
      *reinterpret_cast<float4*>(out + b0 + p * st) = make_float4(e[0], e[1], e[2], e[3]);
      if (q < n && q != p)
        *reinterpret_cast<float4*>(out + b0 + q * st) = make_float4(o[0], o[1], o[2], o[3]);
    } else {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (L + r >= lines) continue;
        const long long b = ((L + r) / inner) * outer + (L + r) % inner;
        out[b + p * st] = e[r];
        if (q < n && q != p) out[b + q * st] = o[r];
      }
    }
  }
}

// Banded product over traces, short bands or few traces: one output and 8
// traces per thread, straight from global memory (each weight loaded once for
// them).  Bound by the loads in flight; not compiled for blocks of 128 threads
// alone, whose larger register budget left fewer resident (65,536 traces of 4000
// samples, 16 taps: 829 us, 952 with it).
constexpr int kFT = 8;

__global__ void band_few_kernel(const float* __restrict__ x, int n_in, const int* __restrict__ c0,
                                const int* __restrict__ len, const float* __restrict__ w, int n_out,
                                int n_traces, float* __restrict__ y) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= n_out) return;
  const int c = c0[m], L = len[m];
  const int groups = (n_traces + kFT - 1) / kFT;
  for (int tg = blockIdx.y; tg < groups; tg += gridDim.y) {
    const int t0 = tg * kFT;
    const float* row[kFT];
    float acc[kFT] = {};
#pragma unroll
    for (int t = 0; t < kFT; ++t) row[t] = x + (long long)min(t0 + t, n_traces - 1) * n_in + c;
    for (int j = 0; j < L; ++j) {
      const float wj = __ldg(w + (long long)j * n_out + m);
#pragma unroll
      for (int t = 0; t < kFT; ++t) acc[t] = fmaf(wj, __ldg(row[t] + j), acc[t]);
    }
#pragma unroll
    for (int t = 0; t < kFT; ++t)
      if (t0 + t < n_traces) y[(long long)(t0 + t) * n_out + m] = acc[t];
  }
}

// Banded product over traces, long bands.  A block makes 32 outputs of 128 traces: warp g
// the outputs 8 g .. 8 g + 7, lane l the traces 4 l .. 4 l + 3, 32 sums in
// registers.  The input window of the block's outputs passes through shared
// memory in chunks of kBK samples, [sample][trace], beside the weights of
// each (sample, output), zero outside the output's band; per sample a thread
// reads 4 trace values and 8 weights for 32 multiply-adds, two outputs per
// instruction.  Zero weights add nothing to a finite sum of finite samples, so
// the outputs' bands need no branches; a thread also sums zero times every
// sample, which is not zero if a sample is not finite, and then the block
// takes its chunks again with a mask of the outputs whose band holds the
// sample (such a sample reaches only those).  65,536 traces of 4000 samples to
// 1000 take 0.84 ms; one output and 8 traces per thread, straight from global
// memory, 33 L1 wavefronts per 8 multiply-adds with bands dt_out / dt_in samples
// apart, took 1.76.  Bound by issue and the barriers of the chunks: a warp's 8
// outputs take about half of the block's window.  Every output is the same sum
// in the same order.
constexpr int kBM = 32, kBT = 128, kBK = 32;
constexpr int kBP = kBT + 4;  // sample pitch: 8 samples x 4 traces of a load fall on 32 banks

struct BandStage {
  float x[kBK][kBP];
  float w[kBK][kBM];
  unsigned mask[kBK];
};

__device__ __forceinline__ void cp_async4(void* dst, const float* src, bool ok) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(ok ? 4 : 0)
               : "memory");
}

__global__ void __launch_bounds__(kBT)
    band_rows_kernel(const float* __restrict__ x, int n_in, const int* __restrict__ c0,
                     const int* __restrict__ len, const float* __restrict__ w, int n_out,
                     int n_traces, float* __restrict__ y) {
  extern __shared__ __align__(16) unsigned char band_smem[];
  BandStage* st = reinterpret_cast<BandStage*>(band_smem);
  const int tid = threadIdx.x, lane = tid & 31, g = tid >> 5;
  const int m0 = blockIdx.x * kBM;
  // this lane's output of the block, and the windows of the block and of each
  // warp's 8 outputs
  const int mc = m0 + lane < n_out ? c0[m0 + lane] : 0;
  const int ml = m0 + lane < n_out ? len[m0 + lane] : 0;
  int lo = ml > 0 ? mc : 0x7fffffff, hi = ml > 0 ? mc + ml : 0;
#pragma unroll
  for (int d = 1; d < 8; d <<= 1) {
    lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, d));
    hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, d));
  }
  const int glo = __shfl_sync(0xffffffffu, lo, 8 * g), ghi = __shfl_sync(0xffffffffu, hi, 8 * g);
#pragma unroll
  for (int d = 8; d < 32; d <<= 1) {
    lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, d));
    hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, d));
  }
  lo = lo < hi ? lo & ~7 : hi;
  const int groups = (n_traces + kBT - 1) / kBT;
  for (int tg = blockIdx.y; tg < groups; tg += gridDim.y) {
    const int t0 = tg * kBT;
    auto issue = [&](int kc, BandStage& s) {
      const int n = min(kBK, hi - kc);
      // 8 consecutive samples of 4 traces per warp and load
      const int kk = lane & 7, tt = lane >> 3;
      for (int t = 4 * g + tt; t < kBT; t += 16) {
        const float* row = x + (long long)min(t0 + t, n_traces - 1) * n_in + kc;
        for (int k = kk; k < n; k += 8)
          cp_async4(&s.x[k][t], row + k, t0 + t < n_traces);
      }
      for (int k = g; k < n; k += kBT / 32) {
        const int j = kc + k - mc;
        const bool in = j >= 0 && j < ml;
        cp_async4(&s.w[k][lane], in ? w + (long long)j * n_out + m0 + lane : w, in);
        const unsigned b = __ballot_sync(0xffffffffu, in);
        if (lane == 0) s.mask[k] = b;
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float2 acc[4][4];  // [two outputs][trace]
    // All chunks into acc; true if a sample the thread has met is not finite.
    auto chunks = [&](auto masked) {
      constexpr bool kMasked = decltype(masked)::value;
      float2 met = {0.0f, 0.0f};  // zero times every sample
#pragma unroll
      for (int o = 0; o < 4; ++o)
#pragma unroll
        for (int t = 0; t < 4; ++t) acc[o][t] = make_float2(0.0f, 0.0f);
      __syncthreads();  // the previous traces' last chunk is read
      if (lo < hi) issue(lo, st[0]);
      int b = 0;
      for (int kc = lo; kc < hi; kc += kBK, b ^= 1) {
        if (kc + kBK < hi) {
          issue(kc + kBK, st[b ^ 1]);
          asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
          asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const BandStage& s = st[b];
        const int k0 = max(glo, kc) - kc, k1 = min(ghi, kc + kBK) - kc;
#pragma unroll 4
        for (int k = k0; k < k1; ++k) {
          const float4 xv = *reinterpret_cast<const float4*>(&s.x[k][4 * lane]);
          const float4 w0 = *reinterpret_cast<const float4*>(&s.w[k][8 * g]);
          const float4 w1 = *reinterpret_cast<const float4*>(&s.w[k][8 * g + 4]);
          const float2 ww[4] = {{w0.x, w0.y}, {w0.z, w0.w}, {w1.x, w1.y}, {w1.z, w1.w}};
          const float xx[4] = {xv.x, xv.y, xv.z, xv.w};
          const unsigned mk = kMasked ? s.mask[k] >> (8 * g) : 0u;
          if (!kMasked) {
            met = __ffma2_rn(make_float2(xv.x, xv.y), make_float2(0.0f, 0.0f), met);
            met = __ffma2_rn(make_float2(xv.z, xv.w), make_float2(0.0f, 0.0f), met);
          }
#pragma unroll
          for (int o = 0; o < 4; ++o)
#pragma unroll
            for (int t = 0; t < 4; ++t) {
              const float2 v = __ffma2_rn(ww[o], make_float2(xx[t], xx[t]), acc[o][t]);
              if (!kMasked || (mk >> (2 * o) & 1)) acc[o][t].x = v.x;
              if (!kMasked || (mk >> (2 * o + 1) & 1)) acc[o][t].y = v.y;
            }
        }
        __syncthreads();
      }
      return !(met.x + met.y == 0.0f);
    };
    if (__syncthreads_or(chunks(std::false_type{}))) chunks(std::true_type{});
    const int m = m0 + 8 * g;
    const bool vec = (n_out & 3) == 0 && ((unsigned long long)y & 15) == 0 && m + 8 <= n_out;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      if (t0 + 4 * lane + t >= n_traces) break;
      float* yr = y + (long long)(t0 + 4 * lane + t) * n_out + m;
      if (vec) {
        reinterpret_cast<float4*>(yr)[0] = make_float4(acc[0][t].x, acc[0][t].y, acc[1][t].x, acc[1][t].y);
        reinterpret_cast<float4*>(yr)[1] = make_float4(acc[2][t].x, acc[2][t].y, acc[3][t].x, acc[3][t].y);
      } else {
#pragma unroll
        for (int o = 0; o < 8; ++o)
          if (m + o < n_out) yr[o] = o & 1 ? acc[o / 2][t].y : acc[o / 2][t].x;
      }
    }
  }
}

__global__ void sub_kernel(const float* __restrict__ a, const float* __restrict__ b, long long n,
                           float* __restrict__ out) {
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n;
       p += (long long)gridDim.x * blockDim.x)
    out[p] = a[p] - b[p];
}

}  // namespace

cudaError_t launch_sub(const float* a, const float* b, long long n, float* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  long long blk = (n + 255) / 256;
  if (blk > 152 * 16) blk = 152 * 16;
  sub_kernel<<<(unsigned)blk, 256, 0, s>>>(a, b, n, out);
  return cudaGetLastError();
}

int row_len(int n) { return ((n + 31) / 32) | 1; }

RowCoef row_coef_host(double s, double mu, int n) { return row_coef(s, mu, n, row_len(n)); }

cudaError_t launch_row_coef(RowCoef* out, int ny, int nz, double my, double mz, double mx, int nx,
                            cudaStream_t s) {
  row_coef_kernel<<<(ny * nz + 127) / 128, 128, 0, s>>>(out, ny, nz, my, mz, mx, nx, row_len(nx));
  return cudaGetLastError();
}

bool rows_need_scratch(int n) { return 8LL * n > kRowSmem; }

cudaError_t launch_rows(const float* in, float* out, float* scratch, int n, long long rows,
                        const RowCoef* coef, const RowCoef& one, cudaStream_t s) {
  if (rows <= 0 || n <= 0) return cudaSuccess;
  const bool staged = !rows_need_scratch(n);
  // 8 rows a block, fewer where they would leave less than two blocks per SM
  int warps = 8;
  while (staged && warps > 1 && 8LL * n * warps > 100 * 1024) warps /= 2;
  const size_t smem = staged ? (size_t)8 * n * warps : 0;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(row_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kRowSmem);
    if (e != cudaSuccess) return e;
  }
  const long long blocks = (rows + warps - 1) / warps;
  row_kernel<<<(unsigned)(blocks < 152 * 64 ? blocks : 152 * 64), 32 * warps, smem, s>>>(
      in, out, scratch, n, row_len(n), rows, coef, one, staged);
  return cudaGetLastError();
}

cudaError_t launch_sweep(const float* in, float* out, const float2* g, const float* inv, bool carry, int n,
                         long long lines, long long inner, long long outer, long long st, cudaStream_t s) {
  if (lines <= 0 || n <= 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((lines + 255) / 256);
  if (carry)
    sweep_kernel<true><<<blocks, 256, 0, s>>>(in, out, g, inv, n, lines, inner, outer, st);
  else
    sweep_kernel<false><<<blocks, 256, 0, s>>>(in, out, g, inv, n, lines, inner, outer, st);
  return cudaGetLastError();
}

cudaError_t launch_dct(const float* in, float* out, const float* E, const float* O, bool inverse,
                       int n, long long lines, long long inner, long long outer, long long st,
                       cudaStream_t s) {
  if (lines <= 0 || n <= 0) return cudaSuccess;
  const int h = (n + 1) / 2;
  const dim3 g((unsigned)((lines + kTL - 1) / kTL), (unsigned)((h + kTI - 1) / kTI));
  if (inverse)
    dct_kernel<true><<<g, 256, 0, s>>>(in, out, E, O, n, lines, inner, outer, st);
  else
    dct_kernel<false><<<g, 256, 0, s>>>(in, out, E, O, n, lines, inner, outer, st);
  return cudaGetLastError();
}

cudaError_t launch_band_rows(const float* x, int n_in, const int* c0, const int* len,
                             const float* w, int taps, int n_out, int n_traces, float* y,
                             cudaStream_t s) {
  if (n_traces <= 0 || n_out <= 0) return cudaSuccess;
  const int groups = (n_traces + kBT - 1) / kBT, tiles = (n_out + kBM - 1) / kBM;
  // A thread per output below 48 taps (its loads of neighbouring outputs fall
  // into the same lines: 65,536 traces of 4000 samples, nearest, 185 us against
  // 511; sinc of equal steps, 16 taps, 829 against 1062; sinc to 1818 samples, 36
  // taps, 1018 against 1150, but 79 taps 1336 against 842) and where the tiles
  // leave SMs idle (79 taps: 84 tiles 27 us against 36, 104 30 against 37, 280
  // 50 against 41).
  if (taps < 48 || (long long)groups * tiles < 200) {
    const int few = (n_traces + kFT - 1) / kFT;
    const dim3 g((unsigned)((n_out + 127) / 128), (unsigned)(few < 65535 ? few : 65535));
    band_few_kernel<<<g, 128, 0, s>>>(x, n_in, c0, len, w, n_out, n_traces, y);
    return cudaGetLastError();
  }
  cudaError_t e = cudaFuncSetAttribute(band_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       2 * (int)sizeof(BandStage));
  if (e != cudaSuccess) return e;
  const dim3 g((unsigned)tiles, (unsigned)(groups < 65535 ? groups : 65535));
  band_rows_kernel<<<g, kBT, 2 * sizeof(BandStage), s>>>(x, n_in, c0, len, w, n_out, n_traces, y);
  return cudaGetLastError();
}

}  // namespace mamute
