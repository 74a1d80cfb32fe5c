// Forward and adjoint time steps of the eighth-order acoustic scheme
// (Eq. 1; Sec. 2.1; Table 1 ModelingStep + ReadReceiver; Algorithm 3
// backward loop with the cross-correlation imaging condition).
//
// One CTA owns a TX x TY tile of one shot's padded grid and marches through
// its planes in z (2.5-D blocking).  A producer warp streams, with TMA,
//   * the propagated field plane by plane with its 4-cell xy halo into a ring
//     of shared-memory stages (zero fill outside the grid = the Dirichlet
//     exterior), and
//   * the centre tiles of the other per-point arrays (previous level, A,
//     A m2, accumulator) into a second ring,
// both guarded by mbarriers.  Each compute thread owns 4 consecutive x points
// of one row and keeps the 9-plane z column of its points in a register
// queue, so only the xy neighbours are read from shared memory.
//
// Update (forward and adjoint alike; the adjoint runs the same operator on
// psi = A g lambda, which makes it the exact transpose of the forward):
//   out = g (2 u - M u - g prev + A lap u),   M = A m2 (0 without density)
// with A = c^2 dt^2 / h^2 and lap the unscaled 25-point sum.  With the
// convolutional PML (PML), lap + E takes the place of lap, E the memory
// variables' part (see cpml.cu), read as one more centre tile on the planes
// and tiles that meet a layer slab.
#pragma once

#include "common.cuh"
#include "stencil.h"

namespace mamute {

namespace {

struct F4 {
  float v[4];
};

__device__ __forceinline__ F4 ld4s(const float* p) {
  float4 t = *reinterpret_cast<const float4*>(p);
  return F4{{t.x, t.y, t.z, t.w}};
}

__device__ __forceinline__ void st4g(float* p, const F4& a) {
  *reinterpret_cast<float4*>(p) = make_float4(a.v[0], a.v[1], a.v[2], a.v[3]);
}

__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }

// lap for the 4 points of a thread: halo stage `st` (row pitch TX + 8), row
// ly, columns lx..lx+3; the z column comes from the register queue q.
template <int TX>
__device__ __forceinline__ void lap4(const float* st, int lx, int ly, const F4 (&q)[9],
                                     float (&out)[4]) {
  constexpr int RP = TX + 2 * kHalo;
  const float* row = st + (ly + kHalo) * RP + lx;
  F4 L = ld4s(row), R = ld4s(row + 8);
  float xs[12];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    xs[e] = L.v[e];
    xs[4 + e] = q[4].v[e];
    xs[8 + e] = R.v[e];
  }
  F4 ym[4], yp[4];
#pragma unroll
  for (int m = 1; m <= 4; ++m) {
    ym[m - 1] = ld4s(row + kHalo - m * RP);
    yp[m - 1] = ld4s(row + kHalo + m * RP);
  }
  // The 25-point sums of two points at a time, in a fixed order of IEEE
  // operations (no contraction freedom), so that every kernel that forms them
  // for the same field gets bitwise the same values.  Packed instructions,
  // because on windows of a few tiles per SM a step is bound by issue as much
  // as by HBM.  Against one point per instruction, all else equal: 500 steps of
  // 96^3 3.43 ms instead of 3.67, a step of four 243x191x137 windows 95 us
  // instead of 101, a whole label of 20 windows of 136x120x104 and 500 steps
  // 96 ms instead of 101.
  const float cw[4] = {MAMUTE_C1, MAMUTE_C2, MAMUTE_C3, MAMUTE_C4};
#pragma unroll
  for (int e = 0; e < 4; e += 2) {
    auto at = [&](const F4& f) { return make_float2(f.v[e], f.v[e + 1]); };
    float2 acc = __fmul2_rn(both(3.0f * MAMUTE_C0), at(q[4]));
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const float2 xm = make_float2(xs[3 + e - m], xs[4 + e - m]);
      const float2 xp = make_float2(xs[5 + e + m], xs[6 + e + m]);
      const float2 s = __fadd2_rn(__fadd2_rn(__fadd2_rn(xm, xp), __fadd2_rn(at(ym[m]), at(yp[m]))),
                                  __fadd2_rn(at(q[3 - m]), at(q[5 + m])));
      acc = __ffma2_rn(both(cw[m]), s, acc);
    }
    out[e] = acc.x;
    out[e + 1] = acc.y;
  }
}

// ev: the memory variables' part E with the CPML, taken as a term of its own
// (lap + E, rounded first, would lose the bits that lap carries beyond E).
template <bool PML>
__device__ __forceinline__ float2 update(float2 u, float2 prev, float2 A, float2 M, float2 g,
                                         float2 lap, float2 ev, bool dens) {
  const float2 ng = make_float2(-g.x, -g.y);
  float2 s = __ffma2_rn(both(2.0f), u, __fmul2_rn(ng, prev));
  if (dens) s = __ffma2_rn(make_float2(-M.x, -M.y), u, s);
  s = __ffma2_rn(A, lap, s);
  if (PML) s = __ffma2_rn(A, ev, s);
  return __fmul2_rn(g, s);
}

// Imaging term A (lap + E - m2) u in the scheme's units: A lap u + A E - M u.
template <bool PML>
__device__ __forceinline__ float img_term(float u, float A, float M, float lap, float ev, bool dens) {
  float t = __fmul_rn(A, lap);
  if (PML) t = __fmaf_rn(A, ev, t);
  if (dens) t = __fmaf_rn(-M, u, t);
  return t;
}

// Shared-memory layout and mode traits of one kernel variant.
template <int TX, int TY, bool DENS, int MODE, bool PML>
struct Layout {
  static constexpr bool ADJ = MODE == MODE_ADJ || MODE == MODE_ADJ_STORED ||
                              MODE == MODE_ADJ_STEP || MODE == MODE_ADJ_TERM;
  static constexpr bool RECOMP = MODE == MODE_ADJ;  // a second halo'd field (u for the imaging)
  static constexpr bool ACC = MODE == MODE_FWD_PH || MODE == MODE_FWD_STORE_PH ||
                              MODE == MODE_ADJ || MODE == MODE_ADJ_STORED;
  static constexpr int NT = MODE == MODE_ADJ_STORED ? kImgSteps : 0;  // stored-term tiles
  static constexpr int NCT = (TX / 4) * TY;  // compute threads
  static constexpr int HS = (TX + 2 * kHalo) * (TY + 2 * kHalo);  // halo stage floats
  static constexpr int CS = TX * TY;  // centre tile floats
  static constexpr int NC = 2 + (DENS ? 1 : 0) + (ACC ? 1 : 0) + NT + (PML ? 1 : 0);  // centre arrays
  // Halo ring depth: 5 planes in use plus 3 ahead (2 ahead where two halo'd
  // fields share each stage or the centre ring is at its widest, to keep two
  // CTAs per SM).
  static constexpr int NSU = (RECOMP || (NT && (DENS || PML))) ? 7 : 8;
  // Centre ring depth: a stage of the imaging launch holds up to 7 tiles, so
  // two of them are as many bytes in flight as four of a plain step.
  static constexpr int NSC = NT ? 2 : (ADJ ? 4 : 3);
  static constexpr int NHALO = RECOMP ? 2 : 1;  // halo'd fields per stage
};

// Per-plane metadata staged in shared memory: sponge factor gz and the
// receiver-entry range of the plane.
struct PlaneInfo {
  float gz;
  int rb, re;
  int ext;  // PML: the tile has a non-zero E on this plane
};

}  // namespace

// Kernel modes.
//   MODE_FWD        forward step
//   MODE_FWD_PH     forward step + pseudo-Hessian accumulation (acc += (g t)^2)
//   MODE_FWD_STORE  forward step + store of the imaging term t on the interior
//   MODE_FWD_STORE_PH  both of the above (all-terms gradient with pseudo-Hessian)
//   MODE_ADJ        adjoint step + imaging against a recomputed forward field
//   MODE_ADJ_STEP   adjoint step alone
//   MODE_ADJ_STORED adjoint step + imaging of the last 1 to kImgSteps levels
//                   against their stored terms
//   MODE_ADJ_TERM   adjoint step + store of the new level on the interior
//
// The accumulator is read and written once per kImgSteps = 3 adjoint steps:
// an adjoint step reads the levels k + 2 (centre tile) and k + 1 (halo'd
// planes) and makes level k, so the launch that images has the three levels
// at hand and takes their three terms T_{k+1}, T_k, T_{k-1} in the same order
// of fused multiply-adds as one term per step would (the same bits).  Per
// three steps and point that is 48 + 8 + 12 bytes (the terms on the model
// interior only) instead of 48 + 24 + 12, and the two launches that do not
// image need less than half of the centre ring.  Bound by HBM: on a 320^3
// window with a 256^3 model a plain step takes 80 us and one with the imaging of
// three levels 147; every step that images its own took 159.
// Resident CTAs per SM the register budget is sized for: the adjoint with a
// recomputed forward field on large tiles needs more than 200 KB of shared
// memory per pair, so it runs one CTA per SM with the full register file;
// small tiles run as many as their shared memory lets in.
template <int TX, int TY, int MODE>
struct MinBlocks {
  static constexpr int kThreads = (TX / 4) * TY + 32;
  static constexpr int value = MODE == MODE_ADJ ? (TX * TY >= 1024 ? 1 : 2)
                                                : (kThreads <= 96 ? 5 : (kThreads <= 160 ? 3 : 2));
};

template <int TX, int TY, bool DENS, int MODE, bool PML>
__global__ void __launch_bounds__((TX / 4) * TY + 32, (MinBlocks<TX, TY, MODE>::value))
    step_kernel(const StepArgs a) {
  using LY = Layout<TX, TY, DENS, MODE, PML>;
  constexpr bool ADJ = LY::ADJ, RECOMP = LY::RECOMP, ACC = LY::ACC;
  constexpr bool TERM = LY::NT > 0;  // stored imaging terms as centre arrays
  constexpr int NCT = LY::NCT, HS = LY::HS, CS = LY::CS, NSU = LY::NSU, NSC = LY::NSC;
  constexpr int NHALO = LY::NHALO, NC = LY::NC;
  constexpr int CI_PREV = 0, CI_A = 1, CI_M = 2, CI_ACC = DENS ? 3 : 2, CI_T = CI_ACC + 1;
  constexpr int CI_E = NC - 1;

  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* ring = reinterpret_cast<float*>(smem_raw);           // NSU * NHALO * HS
  float* cring = ring + NSU * NHALO * HS;                       // NSC * NC * CS
  float* otile = cring + NSC * NC * CS;                         // CS
  uint64_t* bars = reinterpret_cast<uint64_t*>(otile + CS);     // 2*NSU + 2*NSC
  uint64_t* fullF = bars;
  uint64_t* emptyF = bars + NSU;
  uint64_t* fullC = bars + 2 * NSU;
  uint64_t* emptyC = bars + 2 * NSU + NSC;
  PlaneInfo* pinfo = reinterpret_cast<PlaneInfo*>(bars + 2 * NSU + 2 * NSC);  // npl entries

  const WorkItem it = a.items[blockIdx.x];
  const VolDesc V = a.vols[it.vol];
  const ShotMaps* sm = a.maps + it.vol;
  const int x0 = it.x0, y0 = it.y0, zb = it.zb, ze = it.ze;
  const int npl = ze - zb;
  const int tid = threadIdx.x;

  for (int j = tid; j < npl; j += blockDim.x) {
    PlaneInfo pi;
    pi.gz = a.gz[zb + j];
    pi.rb = pi.re = 0;
    if (it.rec_tab >= 0) {
      pi.rb = a.rec_ptr[it.rec_tab + j];
      pi.re = a.rec_ptr[it.rec_tab + j + 1];
    }
    // E is zero but on the layer slabs: its tile is loaded only where the item
    // meets one.
    pi.ext = PML && (x0 < V.ex0 || x0 + it.w > V.ex1 || y0 < V.ey0 || y0 + it.h > V.ey1 ||
                     zb + j < V.ez0 || zb + j >= V.ez1);
    pinfo[j] = pi;
  }
  if (tid == 0) {
    for (int s = 0; s < NSU; ++s) {
      mbar_init(&fullF[s], 1);
      mbar_init(&emptyF[s], NCT / 32);
    }
    for (int s = 0; s < NSC; ++s) {
      mbar_init(&fullC[s], 1);
      mbar_init(&emptyC[s], NCT / 32);
    }
    fence_barrier_init();
  }
  __syncthreads();
  // A chained launch (StepArgs::chained) may start while the previous step
  // ends: everything above reads tables that no step writes.  The producer
  // waits for the previous step before its first load; the other threads act
  // on its loads alone, so the wait covers their stores too.  All else equal, 500
  // steps of 96^3 took 4.98 ms chained and 5.58 not, 800 launches of a 320^3
  // gradient 85.7 and 88.5.

  // Maps of the buffers this launch reads (chosen by the host per step).
  const CUtensorMap* mapF = a.mF + (long long)it.vol * a.sF;
  const CUtensorMap* mapP = a.mP + (long long)it.vol * a.sP;
  const CUtensorMap* mapU = a.mU + (long long)it.vol * a.sU;  // forward field for imaging
  const CUtensorMap* mapAcc = &sm->m[ADJ ? 11 : 8];
  const CUtensorMap* mapT = &sm->m[12];
  const CUtensorMap* mapE = &sm->m[ADJ ? 14 : 13];
  const CUtensorMap* mapA = &a.cmaps->m[0];
  const CUtensorMap* mapM = &a.cmaps->m[1];

  if (tid >= NCT) {
    // ------------------------------------------------------------ producer
    if (tid == NCT) {
      tmap_acquire(mapF);
      tmap_acquire(mapP);
      tmap_acquire(mapA);
      if (DENS) tmap_acquire(mapM);
      if (RECOMP) tmap_acquire(mapU);
      if (ACC) tmap_acquire(mapAcc);
      if (TERM) tmap_acquire(mapT);
      if (PML) tmap_acquire(mapE);
      dependency_wait();
      const int nu = npl + 2 * kHalo;
      const int cx = V.cx0 + x0, cy = V.cy0 + y0;
      int nF = 0, nC = 0;  // loads issued into the halo and centre rings
      // After a wait runs out: let every load already issued land before the
      // CTA exits (bulk copies must not target the shared memory of a CTA
      // that has finished).  Stage s of a ring holds loads s, s + depth, ...;
      // the last one issued into it completes phase (count - 1).
      auto drain = [&]() {
        for (int s = 0; s < NSU && s < nF; ++s)
          mbar_wait(&fullF[s], (uint32_t)(((nF - 1 - s) / NSU) & 1), a.status);
        for (int c = 0; c < NSC && c < nC; ++c)
          mbar_wait(&fullC[c], (uint32_t)(((nC - 1 - c) / NSC) & 1), a.status);
      };
      for (int i = 0; i < nu; ++i) {
        const int s = i % NSU, r = i / NSU;
        if (r > 0 && !mbar_wait(&emptyF[s], (r & 1) ^ 1, a.status)) {
          drain();
          return;
        }
        // Above a free surface at plane zs the plane is the image of plane
        // 2 zs - p (the consumers negate it).
        const int p0 = zb - kHalo + i;
        const int p = (a.zs >= 0 && p0 < a.zs) ? 2 * a.zs - p0 : p0;
        mbar_arrive_expect_tx(&fullF[s], NHALO * HS * 4);
        float* dst = ring + s * NHALO * HS;
        tma_load_3d(dst, mapF, x0 - kHalo, y0 - kHalo, p, &fullF[s]);
        if (RECOMP) tma_load_3d(dst + HS, mapU, x0 - kHalo, y0 - kHalo, p, &fullF[s]);
        ++nF;
        if (i >= 2 * kHalo) {
          const int j = i - 2 * kHalo, q = zb + j;
          const int c = j % NSC, rc = j / NSC;
          if (rc > 0 && !mbar_wait(&emptyC[c], (rc & 1) ^ 1, a.status)) {
            drain();
            return;
          }
          const bool ext = PML && pinfo[j].ext;
          const int absent = (TERM ? kImgSteps - a.nimg : 0) + (PML && !ext ? 1 : 0);
          mbar_arrive_expect_tx(&fullC[c], (NC - absent) * CS * 4);
          float* cd = cring + c * NC * CS;
          tma_load_3d(cd + CI_PREV * CS, mapP, x0, y0, q, &fullC[c]);
          tma_load_3d(cd + CI_A * CS, mapA, cx, cy, q, &fullC[c]);
          if (DENS) tma_load_3d(cd + CI_M * CS, mapM, cx, cy, q, &fullC[c]);
          if (ACC) tma_load_3d(cd + CI_ACC * CS, mapAcc, x0, y0, q, &fullC[c]);
          if (TERM)
            for (int m = 0; m < a.nimg; ++m)
              tma_load_4d(cd + (CI_T + m) * CS, mapT, x0 - V.txoff, y0 - V.iy0, q - V.border,
                          a.tstep + m, &fullC[c]);
          if (PML && ext) tma_load_3d(cd + CI_E * CS, mapE, x0, y0, q, &fullC[c]);
          ++nC;
        }
      }
      launch_dependents();  // every load is issued: the last planes remain
    }
    return;
  }

  // -------------------------------------------------------------- consumers
  constexpr int RP = TX + 2 * kHalo;
  const int lx = (tid % (TX / 4)) * 4, ly = tid / (TX / 4);
  const int gxl = x0 + lx, gyl = y0 + ly;  // local padded coordinates of point 0
  const int lane = tid & 31;
  const bool row_ok = ly < it.h && gyl < V.Ny;
  const bool col_ok = lx < it.w && gxl < V.Nx;  // tile widths are multiples of 4
  float gxv[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) gxv[e] = (gxl + e < V.Nx) ? a.gx[V.gx_off + gxl + e] : 0.0f;
  const float gyv = row_ok ? a.gy[V.gy_off + gyl] : 0.0f;
  const int my_off = (ly + kHalo) * RP + lx + kHalo;  // centre of my row in a halo stage

  // A wait that runs out marks the CTA dead: it records the timeout and then
  // runs to completion without waiting, so every named barrier is reached.
  bool dead = false;
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (!dead && !mbar_wait(bar, parity, a.status)) dead = true;
  };
  F4 q[9], qu[9];
  // z column entry of plane p from its ring stage (negated above a free
  // surface, where the stage holds the image plane).
  auto zload = [&](const float* st, int p) {
    F4 v = ld4s(st);
    if (a.zs >= 0 && p < a.zs) {
#pragma unroll
      for (int e = 0; e < 4; ++e) v.v[e] = -v.v[e];
    }
    return v;
  };
  // Four points of an interior array (imaging term or adjoint level) on the
  // imaging region.
  auto store_term = [&](int z, const F4& v) {
    const int zi = z - V.border, yi = gyl - V.iy0;
    if (row_ok && col_ok && yi >= 0 && yi < V.nyi && zi >= 0 && zi < V.nzi) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int xi = gxl + e - V.ix0;
        if (xi >= 0 && xi < V.nxi)
          a.tstore[V.toff + ((long long)zi * V.nyi + yi) * V.tpitch + (gxl + e - V.txoff)] = v.v[e];
      }
    }
  };
  // Priming: planes zb-4 .. zb+3 fill queue slots 0..7.
  for (int i = 0; i < 2 * kHalo; ++i) {
    const int s = i % NSU;
    wait(&fullF[s], (i / NSU) & 1);
    q[i] = zload(ring + s * NHALO * HS + my_off, zb - kHalo + i);
    if (RECOMP) qu[i] = zload(ring + s * NHALO * HS + HS + my_off, zb - kHalo + i);
    if (i < kHalo || zb - kHalo + i >= ze) {
      __syncwarp();
      if (lane == 0) mbar_arrive(&emptyF[s]);
    }
  }

  // Planes per pass of the loop: the register queue moves on by 32 registers a
  // plane, which unrolling folds into the names; as many as the 96 registers of
  // the tiles with two CTAs of 288 and 320 threads take without spilling.
  // 400 steps of 576x576x320 with density (72x16): one 139.6 ms, two 135.4, three
  // 144.3 (they spill); four 243x191x137 windows (64x16): one 29.0, two 29.6 (spills),
  // three 28.2; a 256^3 gradient (64x16, the adjoint): one 84.1, two 82.4, three 84.9
  // (spills); 96^3 (48x16, few planes a block) is best with one.
  constexpr int kUnroll = TX == 72 && TY == 16 ? 2 : (TX == 64 && TY == 16 ? (ADJ ? 2 : 3) : 1);
#pragma unroll kUnroll
  for (int j = 0; j < npl; ++j) {
    const int z = zb + j;
    {  // queue slot 8 <- plane z + 4
      const int i = j + 2 * kHalo, s = i % NSU;
      wait(&fullF[s], (i / NSU) & 1);
      q[8] = zload(ring + s * NHALO * HS + my_off, z + kHalo);
      if (RECOMP) qu[8] = zload(ring + s * NHALO * HS + HS + my_off, z + kHalo);
      if (z + kHalo >= ze) {
        __syncwarp();
        if (lane == 0) mbar_arrive(&emptyF[s]);
      }
    }
    const int c = j % NSC;
    wait(&fullC[c], (j / NSC) & 1);
    const int su = (j + kHalo) % NSU;
    const float* st = ring + su * NHALO * HS;
    const float* cs = cring + c * NC * CS + ly * TX + lx;

    float lap[4];
    lap4<TX>(st, lx, ly, q, lap);
    const F4 prev = ld4s(cs + CI_PREV * CS);
    const F4 Av = ld4s(cs + CI_A * CS);
    F4 Mv = {{0.f, 0.f, 0.f, 0.f}};
    if (DENS) Mv = ld4s(cs + CI_M * CS);
    const PlaneInfo pi = pinfo[j];
    F4 ev = {{0.f, 0.f, 0.f, 0.f}};
    if (PML && pi.ext) ev = ld4s(cs + CI_E * CS);  // the memory variables' part of the Laplacian
    const float gyz = __fmul_rn(gyv, pi.gz);
    F4 out;
#pragma unroll
    for (int e = 0; e < 4; e += 2) {
      auto at = [&](const F4& f) { return make_float2(f.v[e], f.v[e + 1]); };
      const float2 g = __fmul2_rn(make_float2(gxv[e], gxv[e + 1]), both(gyz));
      const float2 o = update<PML>(at(q[4]), at(prev), at(Av), at(Mv), g, make_float2(lap[e], lap[e + 1]),
                                   at(ev), DENS);
      out.v[e] = o.x;
      out.v[e + 1] = o.y;
    }
    // Source injection (forward only): u^{n+1} += w_e dt^2 w[n] / (h^3 sqrt rho_e)
    // at the corners e of the source cell (one corner for the nearest node).
    if (!ADJ) {
      const int dz = z - V.src_z, dy = gyl - V.src_y;
      if ((unsigned)dz < 2u && (unsigned)dy < 2u) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int dx = gxl + e - V.src_x;
          if ((unsigned)dx < 2u) {
            const float sc = a.vols[it.vol].src_sc[dx + 2 * dy + 4 * dz];  // global: dynamic index
            if (sc != 0.0f) out.v[e] = __fmaf_rn(sc, a.wn, out.v[e]);
          }
        }
      }
    }
    // Receivers of this tile on this plane.
    {
      const int rb = pi.rb, re = pi.re;
      if (rb < re) {
        *reinterpret_cast<float4*>(otile + ly * TX + lx) =
            make_float4(out.v[0], out.v[1], out.v[2], out.v[3]);
        compute_sync(NCT);
        if (!ADJ) {
          if (a.dout)
            for (int e = rb + tid; e < re; e += NCT) {
              const RecEntry r = a.rec[e];
              a.dout[r.col] = r.fscale * otile[r.lxy];
            }
        } else {
          for (int e = rb + tid; e < re; e += NCT) {
            const RecEntry r = a.rec[e];
            if (r.group > 0) {
              float add = 0.0f;
              for (int k = 0; k < r.group; ++k) {
                const RecEntry rk = a.rec[e + k];
                add = __fmaf_rn(rk.ascale, a.rin[rk.col], add);
              }
              otile[r.lxy] += add;
            }
          }
        }
        compute_sync(NCT);
        if (ADJ) out = ld4s(otile + ly * TX + lx);
      }
    }
    // Interior store of the new adjoint level.
    if (MODE == MODE_ADJ_TERM) store_term(z, out);
    // Imaging / accumulation.
    if (MODE == MODE_FWD_PH || MODE == MODE_FWD_STORE || MODE == MODE_FWD_STORE_PH ||
        MODE == MODE_ADJ || MODE == MODE_ADJ_STORED) {
      F4 t;
      if (MODE == MODE_ADJ) {
        float lu[4];
        lap4<TX>(st + HS, lx, ly, qu, lu);
#pragma unroll
        for (int e = 0; e < 4; ++e) t.v[e] = img_term<false>(qu[4].v[e], Av.v[e], Mv.v[e], lu[e], 0.f, DENS);
      } else if (MODE != MODE_ADJ_STORED) {
#pragma unroll
        for (int e = 0; e < 4; ++e) t.v[e] = img_term<PML>(q[4].v[e], Av.v[e], Mv.v[e], lap[e], ev.v[e], DENS);
      }
      if (MODE == MODE_FWD_STORE || MODE == MODE_FWD_STORE_PH) store_term(z, t);
      if (ACC) {
        F4 nacc = ld4s(cs + CI_ACC * CS);
        if (TERM) {  // the older levels first: k + 2, k + 1, k
          if (a.nimg > 2) {
            t = ld4s(cs + (CI_T + 2) * CS);
#pragma unroll
            for (int e = 0; e < 4; ++e) nacc.v[e] = __fmaf_rn(prev.v[e], t.v[e], nacc.v[e]);
          }
          if (a.nimg > 1) {
            t = ld4s(cs + (CI_T + 1) * CS);
#pragma unroll
            for (int e = 0; e < 4; ++e) nacc.v[e] = __fmaf_rn(q[4].v[e], t.v[e], nacc.v[e]);
          }
          t = ld4s(cs + CI_T * CS);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (ADJ) {
            nacc.v[e] = __fmaf_rn(out.v[e], t.v[e], nacc.v[e]);
          } else {
            const float g = __fmul_rn(gxv[e], gyz);
            const float gt = __fmul_rn(g, t.v[e]);
            nacc.v[e] = __fmaf_rn(gt, gt, nacc.v[e]);
          }
        }
        // (whole window; the gradient and pseudo-Hessian read its imaging region)
        if (row_ok && col_ok) {
          float* ap = a.acc + V.off + ((long long)z * V.Ny + gyl) * V.pitch + gxl;
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (gxl + e >= V.Nx) nacc.v[e] = 0.0f;
          st4g(ap, nacc);
        }
      }
    }
    // Store the new level over the previous one.
    if (row_ok && col_ok) {
      float* op = a.fout + V.off + ((long long)z * V.Ny + gyl) * V.pitch + gxl;
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (gxl + e >= V.Nx) out.v[e] = 0.0f;
      st4g(op, out);
    }
    // Release this plane's stages.
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(&emptyF[su]);
      mbar_arrive(&emptyC[c]);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      q[k] = q[k + 1];
      if (RECOMP) qu[k] = qu[k + 1];
    }
  }
}

template <int TX, int TY, bool DENS, int MODE, bool PML>
static size_t smem_bytes_base() {
  using LY = Layout<TX, TY, DENS, MODE, PML>;
  return sizeof(float) * (size_t)(LY::NSU * LY::NHALO * LY::HS + LY::NSC * LY::NC * LY::CS + LY::CS) +
         sizeof(uint64_t) * (2 * LY::NSU + 2 * LY::NSC);
}

// Dynamic shared memory of one launch: rings, output tile, barriers and the
// per-plane table for up to max_planes planes per item.
template <int TX, int TY, bool DENS, int MODE, bool PML>
static size_t smem_bytes(int max_planes) {
  return smem_bytes_base<TX, TY, DENS, MODE, PML>() + sizeof(PlaneInfo) * (size_t)max_planes;
}

template <int TX, int TY, bool DENS, int MODE, bool PML>
static cudaError_t launch_one(const StepArgs& a, int n_items, int max_planes, cudaStream_t s,
                              int* occupancy) {
  const size_t sm = smem_bytes<TX, TY, DENS, MODE, PML>(max_planes);
  static SmemLimit limit;
  const cudaError_t e = allow_smem(limit, step_kernel<TX, TY, DENS, MODE, PML>, sm);
  if (e != cudaSuccess) return e;
  if (occupancy) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occupancy, step_kernel<TX, TY, DENS, MODE, PML>,
                                                         (TX / 4) * TY + 32, sm);
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)n_items);
  cfg.blockDim = dim3((TX / 4) * TY + 32);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = a.chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, step_kernel<TX, TY, DENS, MODE, PML>, a);
}

template <int TX, int TY, int MODE, bool PML = false>
static cudaError_t launch_mode(const StepArgs& a, int n_items, int max_planes, bool dens,
                               cudaStream_t s, int* occ) {
  return dens ? launch_one<TX, TY, true, MODE, PML>(a, n_items, max_planes, s, occ)
              : launch_one<TX, TY, false, MODE, PML>(a, n_items, max_planes, s, occ);
}

// Compiled tile shapes (TX, TY).
#define MAMUTE_TILES(X) X(64, 16) X(64, 8) X(32, 16) X(32, 8) X(128, 8) X(72, 16) X(96, 8) X(48, 16)

cudaError_t dispatch_forward(const StepArgs& a, int n_items, int max_planes, int tx, int ty,
                             bool dens, int mode, cudaStream_t s, int* occ);
cudaError_t dispatch_adjoint(const StepArgs& a, int n_items, int max_planes, int tx, int ty,
                             bool dens, int mode, cudaStream_t s, int* occ);
// The same with the CPML's E added to the 25-point sum.
cudaError_t dispatch_pml_forward(const StepArgs& a, int n_items, int max_planes, int tx, int ty,
                                 bool dens, int mode, cudaStream_t s, int* occ);
cudaError_t dispatch_pml_adjoint(const StepArgs& a, int n_items, int max_planes, int tx, int ty,
                                 bool dens, int mode, cudaStream_t s, int* occ);

}  // namespace mamute
