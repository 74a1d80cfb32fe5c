// Convolutional PML (Sec. 2: the second absorbing boundary, after Roden and
// Gedney) for modelling and for the gradient.
//
// In the layer each derivative d/dx_a is (1/s_a) d/dx_a, s_a = 1 + d_a /
// (alpha_a + i w), and the second derivative is carried by two memory
// variables per axis, updated by recursive convolution.  With the unscaled
// eighth-order stencils D2_a (weights c0..c4) and D1_a (4/5, -1/5, 4/105,
// -1/280) and the memory variables scaled by h and h^2 (so that the update
// uses A = c^2 dt^2 / h^2 like the damping kernels):
//   Psi_a'  = b_a Psi_a  + c_a D1_a u
//   Zeta_a' = b_a Zeta_a + c_a (D2_a u + D1_a Psi_a')
//   u'      = (2 - M) u - v + A (lap u + E) + source,  E = sum_a (D1_a Psi_a' + Zeta_a')
// with b_a = exp(-(d_a + alpha_a) dt), c_a = d_a (b_a - 1) / (d_a + alpha_a)
// (profiles built on the host; b = 1, c = 0 outside the layer).
//
// The gradient is the exact transpose of this recursion.  In the adjoint
// level psi (the multiplier of u scaled by A, which the main kernel
// propagates with the forward operator itself), one reverse step is
//   per axis, in the layer:  y_a = c_a (Zb_a + psi),  Zb_a' = b_a (Zb_a + psi)
//                            p_a = Pb_a - D1_a (psi + y_a),  Pb_a' = b_a p_a
//   psi' = (2 - M) psi - psi_prev + A (lap psi + E) + injection,
//   E = sum_a (D2_a y_a - D1_a (c_a p_a))
// (Zb, Pb the multipliers of Zeta and Psi; D2 is symmetric, D1 antisymmetric,
// the fields are zero outside the padded window).
//
// Work split.  E depends on the old state alone, so one launch per axis makes
// the whole memory-variable part before the main step, which reads E as one
// more centre tile: per layer point and axis the field, the two memory
// variables (read and written) and E, 28 bytes written or read once by the
// slab kernel and the main step together.  A cell needs the new Psi (p) of its
// 4 neighbours on each side; they are made again from the old values instead
// of being exchanged, so Psi, and in the reverse both multipliers, are kept
// twice (read one copy, write the other) and a slab may be cut anywhere.
// 448x448x256 with density takes 326 us a step, 59, 37 and 50 of them the z, y
// and x slabs and 179 the main step, which is bound by HBM; updating Psi before
// the main step, Zeta after it and correcting u', the imaging term and the
// accumulator in place (40 bytes forward and 60 in reverse, 6 and 7 launches)
// took 577.
#include "cpml.h"

#include <algorithm>

namespace mamute {

namespace {

constexpr int kThreads = 128;
constexpr int kDepth = 4;  // cells in flight per marching thread

// First and second difference at the centre of 9 consecutive values.
__device__ __forceinline__ float d1(float m4, float m3, float m2, float m1, float p1, float p2,
                                    float p3, float p4) {
  float s = 4.0f / 5.0f * (p1 - m1);
  s = fmaf(-1.0f / 5.0f, p2 - m2, s);
  s = fmaf(4.0f / 105.0f, p3 - m3, s);
  return fmaf(-1.0f / 280.0f, p4 - m4, s);
}

__device__ __forceinline__ float d2(float m4, float m3, float m2, float m1, float v, float p1,
                                    float p2, float p3, float p4) {
  float s = MAMUTE_C0 * v;
  s = fmaf(MAMUTE_C1, p1 + m1, s);
  s = fmaf(MAMUTE_C2, p2 + m2, s);
  s = fmaf(MAMUTE_C3, p3 + m3, s);
  return fmaf(MAMUTE_C4, p4 + m4, s);
}

#define D1Q(q, k, e) \
  d1(q[(k) - 4][e], q[(k) - 3][e], q[(k) - 2][e], q[(k) - 1][e], q[(k) + 1][e], q[(k) + 2][e], \
     q[(k) + 3][e], q[(k) + 4][e])
#define D2Q(q, k, e) \
  d2(q[(k) - 4][e], q[(k) - 3][e], q[(k) - 2][e], q[(k) - 1][e], q[k][e], q[(k) + 1][e], \
     q[(k) + 2][e], q[(k) + 3][e], q[(k) + 4][e])
#define D1R(q, k) \
  d1(q[(k) - 4], q[(k) - 3], q[(k) - 2], q[(k) - 1], q[(k) + 1], q[(k) + 2], q[(k) + 3], q[(k) + 4])
#define D2R(q, k) \
  d2(q[(k) - 4], q[(k) - 3], q[(k) - 2], q[(k) - 1], q[k], q[(k) + 1], q[(k) + 2], q[(k) + 3], \
     q[(k) + 4])

template <int V>
struct VecT;
template <>
struct VecT<2> {
  using T = float2;
};
template <>
struct VecT<4> {
  using T = float4;
};

template <int V>
__device__ __forceinline__ void unpack(const typename VecT<V>::T& t, float (&v)[V]) {
  v[0] = t.x;
  v[1] = t.y;
  if constexpr (V == 4) {
    v[2] = t.z;
    v[3] = t.w;
  }
}

template <int V>
__device__ __forceinline__ typename VecT<V>::T pack(const float (&v)[V]) {
  if constexpr (V == 4)
    return make_float4(v[0], v[1], v[2], v[3]);
  else
    return make_float2(v[0], v[1]);
}

// Asynchronous copy of V floats into the thread's own shared-memory slot;
// zeros where ok is false (the source address is then not read).
template <int V>
__device__ __forceinline__ void cp_async(void* dst, const float* src, bool ok) {
  const int n = ok ? V * 4 : 0;
  if constexpr (V == 4)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src),
                 "r"(n)
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(smem_u32(dst)), "l"(src),
                 "r"(n)
                 : "memory");
}

__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// One thread's march along axis A (1: y, 2: z): V consecutive x cells of one
// column, the cells [s0, s1) of the slab region [r0, r1), in element strides
// st (fields) and sc (slab arrays).
template <int A, int V>
struct March {
  int s0, s1, r0, r1, N;
  bool add;  // E already holds another axis's part here
  long long st, sc;
  const float* u;
  long long m;  // slab-array element of cell r0
  float* E;
  int prof;
  __device__ __forceinline__ bool init(const CpmlArgs& c, int chunk, int first) {
    const VolDesc& D = c.vols[blockIdx.y];
    const CpmlVol& W = c.cv[blockIdx.y];
    N = A == 2 ? D.Nz : D.Ny;
    const int lo = W.lo[A], hi = W.hi[A];
    const bool merged = lo == hi;  // one range [0, N)
    const int nlo = merged ? 0 : (lo + chunk - 1) / chunk;
    int k = first + blockIdx.z;
    if (k < nlo) {
      r0 = 0;
      r1 = lo;
    } else {
      k -= nlo;
      r0 = merged ? 0 : hi;
      r1 = N;
    }
    s0 = r0 + k * chunk;
    s1 = min(s0 + chunk, r1);
    if (s0 >= r1) return false;
    const unsigned nxv = (unsigned)(D.Nx + V - 1) / V;
    const unsigned q = blockIdx.x * kThreads + threadIdx.x;
    const unsigned o = q / nxv;
    if (o >= (unsigned)(A == 2 ? D.Ny : D.Nz)) return false;
    const int x = (int)(q - o * nxv) * V;
    const long long plane = (long long)D.Ny * D.pitch;
    const int slot = merged || r0 == 0 ? 0 : lo;  // slot of cell r0
    st = A == 2 ? plane : D.pitch;
    sc = st;
    const long long f = D.off + (A == 2 ? (long long)o * D.pitch : (long long)o * plane) + x;
    u = c.u + f;
    E = c.E + f;
    m = W.off[A] + x + (A == 2 ? ((long long)slot * D.Ny + o) * D.pitch
                              : ((long long)o * W.n[A] + slot) * D.pitch);
    prof = W.prof[A] + kCpmlPad;
    add = A == 1 && ((int)o < W.lo[2] || (int)o >= W.hi[2]);
    return true;
  }
};

// Forward, axes z and y: the thread marches along the axis with the field in a
// 13-deep register queue and the new Psi in a 9-deep one, at step p making
// Psi'(p) and finishing cell s = p - 4.  Bound by HBM; the loads of the next
// kDepth - 1 cells are in flight as asynchronous copies into the thread's own
// shared-memory slots (no barrier), which costs no registers.
template <int A>
__global__ void __launch_bounds__(kThreads, 3) fwd_march_kernel(CpmlArgs c, int chunk, int first) {
  constexpr int V = 4;
  using T = VecT<V>::T;
  __shared__ T ring[kDepth][4][kThreads];  // u, Psi, Zeta, E
  March<A, V> w;
  if (!w.init(c, chunk, first)) return;
  const int tid = threadIdx.x;
  const int p0 = w.s0 - 4, p1 = w.s1 + 4;
  auto issue = [&](int p) {
    if (p < p1) {
      T* r = &ring[(p - p0) % kDepth][0][tid];
      const int e = p + 4, s = p - 4;
      cp_async<V>(r, w.u + (e >= 0 && e < w.N ? e : 0) * w.st, e >= 0 && e < w.N);
      const bool in = p >= w.r0 && p < w.r1;
      cp_async<V>(r + kThreads, c.m1 + w.m + (in ? p - w.r0 : 0) * w.sc, in);
      if (s >= w.s0) {
        cp_async<V>(r + 2 * kThreads, c.m2 + w.m + (s - w.r0) * w.sc, true);
        if (w.add) cp_async<V>(r + 3 * kThreads, w.E + s * w.st, true);
      }
    }
    cp_commit();
  };
  for (int k = 0; k < kDepth - 1; ++k) issue(p0 + k);
  float uq[13][V], pq[9][V];  // u(p - 8 .. p + 4), Psi'(p - 8 .. p)
#pragma unroll
  for (int k = 1; k < 13; ++k) {
    const int e = p0 - 9 + k;
    T t{};
    if (k > 4 && e >= 0 && e < w.N) t = *reinterpret_cast<const T*>(w.u + e * w.st);
    unpack<V>(t, uq[k]);
  }
#pragma unroll
  for (int k = 0; k < 9; ++k)
#pragma unroll
    for (int e = 0; e < V; ++e) pq[k][e] = 0.0f;
  for (int p = p0; p < p1; ++p) {
    const float bp = __ldg(c.b + w.prof + p), cp = __ldg(c.c + w.prof + p);
    const int s = p - 4;
    const float bs = __ldg(c.b + w.prof + s), cs = __ldg(c.c + w.prof + s);
    cp_wait<kDepth - 2>();
    const T* r = &ring[(p - p0) % kDepth][0][tid];
#pragma unroll
    for (int k = 0; k < 12; ++k)
#pragma unroll
      for (int e = 0; e < V; ++e) uq[k][e] = uq[k + 1][e];
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
      for (int e = 0; e < V; ++e) pq[k][e] = pq[k + 1][e];
    unpack<V>(r[0], uq[12]);
    unpack<V>(r[kThreads], pq[8]);
    issue(p + kDepth - 1);  // into the slot whose values the last step has used
    if (cp != 0.0f || bp != 1.0f) {
#pragma unroll
      for (int e = 0; e < V; ++e) pq[8][e] = fmaf(bp, pq[8][e], cp * D1Q(uq, 8, e));
    }
    if (p >= w.s0 && p < w.s1)
      *reinterpret_cast<T*>(c.m1n + w.m + (p - w.r0) * w.sc) = pack<V>(pq[8]);
    if (s >= w.s0) {
      float z[V], ev[V];
      unpack<V>(r[2 * kThreads], z);
#pragma unroll
      for (int e = 0; e < V; ++e) ev[e] = D1Q(pq, 4, e);
      if (cs != 0.0f || bs != 1.0f) {
#pragma unroll
        for (int e = 0; e < V; ++e) {
          z[e] = fmaf(bs, z[e], cs * (D2Q(uq, 4, e) + ev[e]));
          ev[e] += z[e];
        }
        *reinterpret_cast<T*>(c.m2n + w.m + (s - w.r0) * w.sc) = pack<V>(z);
      }
      if (w.add) {
        float o[V];
        unpack<V>(r[3 * kThreads], o);
#pragma unroll
        for (int e = 0; e < V; ++e) ev[e] += o[e];
      }
      *reinterpret_cast<T*>(w.E + s * w.st) = pack<V>(ev);
    }
  }
}

// Reverse, axes z and y: at step e cell e enters (y, psi + y and its Zeta
// multiplier), p = e - 4 gets its Psi multiplier and z, and s = e - 8 is
// finished.  Two x cells per thread: the three queues hold 31 values a cell.
template <int A>
__global__ void __launch_bounds__(kThreads, 4) rev_march_kernel(CpmlArgs c, int chunk, int first) {
  constexpr int V = 2;
  using T = VecT<V>::T;
  __shared__ T ring[kDepth][4][kThreads];  // psi, Zb, Pb, E
  March<A, V> w;
  if (!w.init(c, chunk, first)) return;
  const int tid = threadIdx.x;
  const int e0 = w.s0 - 8, e1 = w.s1 + 8;
  auto issue = [&](int e) {
    if (e < e1) {
      T* r = &ring[(e - e0) % kDepth][0][tid];
      const bool inw = e >= 0 && e < w.N, in = e >= w.r0 && e < w.r1;
      cp_async<V>(r, w.u + (inw ? e : 0) * w.st, inw);
      cp_async<V>(r + kThreads, c.m2 + w.m + (in ? e - w.r0 : 0) * w.sc, in);
      const int p = e - 4, s = e - 8;
      const bool inp = p >= w.r0 && p < w.r1;
      cp_async<V>(r + 2 * kThreads, c.m1 + w.m + (inp ? p - w.r0 : 0) * w.sc, inp);
      if (w.add && s >= w.s0) cp_async<V>(r + 3 * kThreads, w.E + s * w.st, true);
    }
    cp_commit();
  };
  for (int k = 0; k < kDepth - 1; ++k) issue(e0 + k);
  float yq[13][V], vq[9][V], zq[9][V];  // y(e - 12 .. e), (psi + y)(e - 8 .. e), z(e - 12 .. e - 4)
#pragma unroll
  for (int v = 0; v < V; ++v) {
#pragma unroll
    for (int k = 0; k < 13; ++k) yq[k][v] = 0.0f;
#pragma unroll
    for (int k = 0; k < 9; ++k) vq[k][v] = zq[k][v] = 0.0f;
  }
  for (int e = e0; e < e1; ++e) {
    const int p = e - 4, s = e - 8;
    const float be = __ldg(c.b + w.prof + e), ce = __ldg(c.c + w.prof + e);
    const float bp = __ldg(c.b + w.prof + p), cp = __ldg(c.c + w.prof + p);
    cp_wait<kDepth - 2>();
    const T* r = &ring[(e - e0) % kDepth][0][tid];
#pragma unroll
    for (int v = 0; v < V; ++v) {
#pragma unroll
      for (int k = 0; k < 12; ++k) yq[k][v] = yq[k + 1][v];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        vq[k][v] = vq[k + 1][v];
        zq[k][v] = zq[k + 1][v];
      }
      yq[12][v] = zq[8][v] = 0.0f;
    }
    unpack<V>(r[0], vq[8]);
    issue(e + kDepth - 1);  // into the slot whose values the last step has used
    if (ce != 0.0f || be != 1.0f) {
      float zb[V];
      unpack<V>(r[kThreads], zb);
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const float zt = zb[v] + vq[8][v];
        yq[12][v] = ce * zt;
        vq[8][v] += yq[12][v];
        zb[v] = be * zt;
      }
      if (e >= w.s0 && e < w.s1)
        *reinterpret_cast<T*>(c.m2n + w.m + (e - w.r0) * w.sc) = pack<V>(zb);
    }
    if (cp != 0.0f || bp != 1.0f) {
      float pb[V];
      unpack<V>(r[2 * kThreads], pb);
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const float pt = pb[v] - D1Q(vq, 4, v);
        zq[8][v] = cp * pt;
        pb[v] = bp * pt;
      }
      if (p >= w.s0 && p < w.s1)
        *reinterpret_cast<T*>(c.m1n + w.m + (p - w.r0) * w.sc) = pack<V>(pb);
    }
    if (s >= w.s0) {
      float ev[V];
#pragma unroll
      for (int v = 0; v < V; ++v) ev[v] = D2Q(yq, 4, v) - D1Q(zq, 4, v);
      if (w.add) {
        float o[V];
        unpack<V>(r[3 * kThreads], o);
#pragma unroll
        for (int v = 0; v < V; ++v) ev[v] += o[v];
      }
      *reinterpret_cast<T*>(w.E + s * w.st) = pack<V>(ev);
    }
  }
}

// One thread's 4 cells of the x slabs: x0 (a multiple of 4) of row (y, z).
struct XCell {
  int x0, r0, r1, n4;  // slab region [r0, r1) of the cells; row length rounded up to 4
  bool add;
  long long f, m;  // field element of the row's start; slab-array element of cell r0
  int prof;
  __device__ __forceinline__ bool init(const CpmlArgs& c) {
    const VolDesc& D = c.vols[blockIdx.y];
    const CpmlVol& W = c.cv[blockIdx.y];
    const unsigned G = (unsigned)W.n[0] / 4;
    if (G == 0) return false;
    const unsigned q = blockIdx.x * kThreads + threadIdx.x;
    const unsigned row = q / G;
    const unsigned z = row / (unsigned)D.Ny;
    if (z >= (unsigned)D.Nz) return false;
    const int y = (int)(row - z * (unsigned)D.Ny), sl = (int)(q - row * G) * 4;
    const int lo = W.lo[0], hi = W.hi[0];
    n4 = (D.Nx + 3) & ~3;
    const bool low = sl < lo;
    r0 = low ? 0 : hi;
    r1 = low && lo != hi ? lo : n4;
    if (lo == hi) r0 = 0;
    x0 = low || lo == hi ? sl : sl - lo + hi;
    f = D.off + (long long)row * D.pitch;
    m = W.off[0] + (long long)row * W.n[0] + (r0 == 0 ? 0 : lo);
    prof = W.prof[0] + kCpmlPad + x0;
    add = y < W.lo[1] || y >= W.hi[1] || (int)z < W.lo[2] || (int)z >= W.hi[2];
    return true;
  }
  // 4 values at x0 + 4 k: of a field (zero outside the row) or a slab array
  // (zero outside the region).
  __device__ __forceinline__ float4 field(const float* a, int k) const {
    const int x = x0 + 4 * k;
    return (x >= 0 && x < n4) ? __ldg(reinterpret_cast<const float4*>(a + f + x))
                              : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __device__ __forceinline__ float4 slab(const float* a, int k) const {
    const int x = x0 + 4 * k;
    return (x >= r0 && x < r1) ? __ldg(reinterpret_cast<const float4*>(a + m + (x - r0)))
                               : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __device__ __forceinline__ void store(float* a, const float (&v)[4]) const {
    *reinterpret_cast<float4*>(a + m + (x0 - r0)) = make_float4(v[0], v[1], v[2], v[3]);
  }
};

__device__ __forceinline__ void put(float* d, const float4& t) {
  d[0] = t.x;
  d[1] = t.y;
  d[2] = t.z;
  d[3] = t.w;
}

__device__ __forceinline__ void profile4(const float* p, float* d) {
  put(d, __ldg(reinterpret_cast<const float4*>(p)));
}

// x slabs: 4 cells per thread, the neighbours in 16-byte loads that mostly hit
// the lines of the neighbouring threads (5 of the field, 3 of Psi for the 12
// Psi' of the cell's own D1), no exchange between threads.
__global__ void __launch_bounds__(kThreads) fwd_x_kernel(CpmlArgs c) {
  XCell w;
  if (!w.init(c)) return;
  float u[20], ps[12], b[12], cc[12], z[4], ev[4];
#pragma unroll
  for (int k = 0; k < 5; ++k) put(u + 4 * k, w.field(c.u, k - 2));
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    put(ps + 4 * k, w.slab(c.m1, k - 1));
    profile4(c.b + w.prof + 4 * (k - 1), b + 4 * k);
    profile4(c.c + w.prof + 4 * (k - 1), cc + 4 * k);
  }
  // Zeta is updated in place by its own thread alone: a plain load
  put(z, *reinterpret_cast<const float4*>(c.m2 + w.m + (w.x0 - w.r0)));
  float4 old = make_float4(0.f, 0.f, 0.f, 0.f);
  float4* Ep = reinterpret_cast<float4*>(c.E + w.f + w.x0);
  if (w.add) old = *Ep;
#pragma unroll
  for (int k = 0; k < 12; ++k) ps[k] = fmaf(b[k], ps[k], cc[k] * D1R(u, k + 4));
  const float pn[4] = {ps[4], ps[5], ps[6], ps[7]};
  w.store(c.m1n, pn);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float d1p = D1R(ps, e + 4);
    z[e] = fmaf(b[e + 4], z[e], cc[e + 4] * (D2R(u, e + 8) + d1p));
    ev[e] = d1p + z[e];
  }
  w.store(c.m2n, z);
  *Ep = make_float4(old.x + ev[0], old.y + ev[1], old.z + ev[2], old.w + ev[3]);
}

__global__ void __launch_bounds__(kThreads) rev_x_kernel(CpmlArgs c) {
  XCell w;
  if (!w.init(c)) return;
  float v[20], y[20], cc[20], z[12], b[4];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    put(v + 4 * k, w.field(c.u, k - 2));
    put(y + 4 * k, w.slab(c.m2, k - 2));
    profile4(c.c + w.prof + 4 * (k - 2), cc + 4 * k);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) put(z + 4 * k, w.slab(c.m1, k - 1));
  profile4(c.b + w.prof, b);
  float4 old = make_float4(0.f, 0.f, 0.f, 0.f);
  float4* Ep = reinterpret_cast<float4*>(c.E + w.f + w.x0);
  if (w.add) old = *Ep;
  float nz[4], np[4];
#pragma unroll
  for (int k = 0; k < 20; ++k) {
    const float zt = y[k] + v[k];
    if (k >= 8 && k < 12) nz[k - 8] = cc[k] != 0.0f || b[k - 8] != 1.0f ? b[k - 8] * zt : 0.0f;
    y[k] = cc[k] * zt;
    v[k] += y[k];
  }
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const float pt = z[k] - D1R(v, k + 4);
    if (k >= 4 && k < 8) np[k - 4] = cc[k + 4] != 0.0f || b[k - 4] != 1.0f ? b[k - 4] * pt : 0.0f;
    z[k] = cc[k + 4] * pt;
  }
  w.store(c.m2n, nz);
  w.store(c.m1n, np);
  float ev[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) ev[e] = D2R(y, e + 8) - D1R(z, e + 4);
  *Ep = make_float4(old.x + ev[0], old.y + ev[1], old.z + ev[2], old.w + ev[3]);
}

// Threads that a marching launch should have: enough columns leave the slabs
// whole (a cut makes 8 or 16 cells of the neighbouring piece again); with
// fewer, the slabs are cut into pieces of at least 3 cells.  250 gradient steps
// of 256^3 take 92.1, 92.3, 94.4, 100.7 and 119.5 ms with 128, 256, 512, 1024
// and 2048 threads per SM asked for, 300 steps of 448x448x256 107.5 to 108.2
// up to 1024 and 111.8 at 2048.
constexpr long long kMarchThreads = 152LL * 256;

int piece(const CpmlExtent& e, int a) {
  long long cuts = std::max(1LL, kMarchThreads / std::max(1LL, e.threads[a]));
  cuts = std::min<long long>(cuts, std::max(1, e.len[a] / 3));
  return std::max(1, (int)((e.len[a] + cuts - 1) / cuts));
}

// Grid of a marching launch: columns of V cells, windows, pieces of both slabs.
dim3 march_grid(const CpmlExtent& e, int a, int V, int chunk) {
  const long long threads = e.cols[a] * (4 / V);
  return dim3((unsigned)((threads + kThreads - 1) / kThreads), (unsigned)e.nvol,
              (unsigned)(2 * ((e.len[a] + chunk - 1) / chunk)));
}

// Launches that the pieces of an axis's slabs are spread over (see CpmlExtent::apart).
int parts(const CpmlExtent& e, int a) {
  const int k = piece(e, a), pieces = 2 * ((e.len[a] + k - 1) / k);
  return e.apart ? std::min(pieces, a == 2 ? 4 : 2) : 1;
}

template <int A>
void forward_axis(const CpmlArgs& c, const CpmlExtent& e, cudaStream_t s) {
  if (e.len[A] <= 0) return;
  const int k = piece(e, A), n = parts(e, A);
  dim3 g = march_grid(e, A, 4, k);
  const int pieces = (int)g.z;
  for (int i = 0; i < n; ++i) {
    const int first = pieces * i / n;
    g.z = (unsigned)(pieces * (i + 1) / n - first);
    fwd_march_kernel<A><<<g, kThreads, 0, s>>>(c, k, first);
  }
}

template <int A>
void reverse_axis(const CpmlArgs& c, const CpmlExtent& e, cudaStream_t s) {
  if (e.len[A] <= 0) return;
  const int k = piece(e, A);
  rev_march_kernel<A><<<march_grid(e, A, 2, k), kThreads, 0, s>>>(c, k, 0);
}

dim3 x_grid(const CpmlExtent& e) {
  return dim3((unsigned)((e.cols[0] + kThreads - 1) / kThreads), (unsigned)e.nvol);
}

}  // namespace

int cpml_launches(const CpmlExtent& e) {
  int n = e.cols[0] > 0 ? 1 : 0;
  for (int a = 1; a < 3; ++a)
    if (e.len[a] > 0) n += parts(e, a);
  return n;
}

cudaError_t launch_cpml_forward(const CpmlArgs& c, const CpmlExtent& e, cudaStream_t s) {
  forward_axis<2>(c, e, s);
  forward_axis<1>(c, e, s);
  if (e.cols[0] > 0) fwd_x_kernel<<<x_grid(e), kThreads, 0, s>>>(c);
  return cudaGetLastError();
}

cudaError_t launch_cpml_reverse(const CpmlArgs& c, const CpmlExtent& e, cudaStream_t s) {
  reverse_axis<2>(c, e, s);
  reverse_axis<1>(c, e, s);
  if (e.cols[0] > 0) rev_x_kernel<<<x_grid(e), kThreads, 0, s>>>(c);
  return cudaGetLastError();
}

}  // namespace mamute
