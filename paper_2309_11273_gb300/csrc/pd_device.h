// Device helpers shared by the step kernels (pd_step.cu) and the resident step kernel (pd_resident.cu).
#pragma once

#include <type_traits>

#include "pd_internal.h"
#include "pd_order.h"

namespace pd {
namespace {

constexpr unsigned kFull = 0xffffffffu;

struct SliceIdx {
  int64_t i;
  int64_t base;
  int W;
  int lane;
  int sub;
  bool active;
};

template <int SPLIT>
__device__ __forceinline__ SliceIdx slice_index(int64_t n_pad, const int64_t* __restrict__ slice_ptr) {
  SliceIdx r;
  const int64_t gwarp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  r.lane = threadIdx.x & 31;
  r.sub = (int)(gwarp % SPLIT);
  const int64_t s = gwarp / SPLIT;
  r.i = s * 32 + r.lane;
  r.active = r.i < n_pad;  // n_pad is a multiple of 32: uniform over the warp
  r.base = 0;
  r.W = 0;
  if (r.active) {
    r.base = slice_ptr[s];
    r.W = (int)((slice_ptr[s + 1] - r.base) >> 5);
  }
  return r;
}

// Partial sums of the SPLIT warps sharing a slice, combined by the first warp (fixed order).
template <int SPLIT, int NC, class T>
__device__ __forceinline__ void split_reduce(T (&v)[NC]) {
  if (SPLIT == 1) return;
  extern __shared__ unsigned char smem_raw[];
  T* red = reinterpret_cast<T*>(smem_raw);
#pragma unroll
  for (int c = 0; c < NC; ++c) red[c * blockDim.x + threadIdx.x] = v[c];
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w % SPLIT == 0) {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      T s = red[c * blockDim.x + w * 32 + lane];
#pragma unroll
      for (int q = 1; q < SPLIT; ++q) s += red[c * blockDim.x + (w + q) * 32 + lane];
      v[c] = s;
    }
  }
}

// The sums of the tabled FP64 kernels run in four parts, slot k in part k mod 4, combined as (0 + 2) +
// (1 + 3) whatever the number of warps that share a slice: a warp holds 4 / SPLIT of them, so the result
// is bitwise the same for every split (and four independent chains of FP64 additions are shorter).
// P = 1: each warp's plain sum in slot order, which the relaxation solver keeps (block_tree).
template <int SPLIT, int NC, int P = 4 / SPLIT>
__device__ __forceinline__ void parts_sum(const double (&p)[NC][P], double (&v)[NC]) {
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    if constexpr (P == 1) v[c] = p[c][0];  // (split 4: one part per warp)
    else if constexpr (SPLIT == 1) v[c] = (p[c][0] + p[c][2]) + (p[c][1] + p[c][3]);
    else v[c] = p[c][0] + p[c][1];
  }
}
// ... and across the warps of the slice (their parts combined by the first warp; SERIAL, the relaxation solver:
// the warps' sums added one after the other).
template <int SPLIT, int NC, bool SERIAL = false>
__device__ __forceinline__ void parts_across(double (&v)[NC]) {
  if (SPLIT == 1) return;
  if constexpr (SERIAL) {
    split_reduce<SPLIT, NC>(v);
    return;
  }
  extern __shared__ unsigned char smem_raw[];
  double* red = reinterpret_cast<double*>(smem_raw);
#pragma unroll
  for (int c = 0; c < NC; ++c) red[c * blockDim.x + threadIdx.x] = v[c];
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w % SPLIT == 0) {
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const double* r = red + c * blockDim.x + w * 32 + lane;
      v[c] = SPLIT == 2 ? r[0] + r[32] : (r[0] + r[64]) + (r[32] + r[96]);
    }
  }
}

// Eq 2.11 for a free particle with the force density f and the body force b (nullptr: none): v += (dt / rho)
// (f + b), u += dt v, two FMAs per component and an addition for b (an FP64 instruction occupies its pipe for 64
// cycles per warp); f + b is formed first, so that a particle in balance gets no rounding of dt f / rho.  The z
// components stay as they are in 2D.
template <int DIM>
__device__ __forceinline__ void explicit_move(const BodyDev& bp, const double f[3], const double4* b, double4& u,
                                              double4& v) {
  double g[3] = {f[0], f[1], f[2]};
  if (b) {
    g[0] += b->x;
    g[1] += b->y;
    if (DIM == 3) g[2] += b->z;
  }
  v.x = fma(bp.dt_rho, g[0], v.x);
  v.y = fma(bp.dt_rho, g[1], v.y);
  if (DIM == 3) v.z = fma(bp.dt_rho, g[2], v.z);
  u.x = fma(bp.dt, v.x, u.x);
  u.y = fma(bp.dt, v.y, u.y);
  if (DIM == 3) u.z = fma(bp.dt, v.z, u.z);
}

// Row e of a per-slot table of the linearized FP64 kernels.  In 2D the table holds no z: all pairs (x, y),
// then all fourth words, 24 bytes per slot instead of 32 (a 400 x 160 plate's tables, index and extension
// streams then stay in L2).
template <int DIM>
__device__ __forceinline__ double4 slot_row(const double4* __restrict__ table, int64_t ne, int64_t e) {
  if (DIM == 3) return table[e];
  const double2 xy = reinterpret_cast<const double2*>(table)[e];
  return make_double4(xy.x, xy.y, 0.0, reinterpret_cast<const double*>(table)[2 * ne + e]);
}
template <int DIM>
__device__ __forceinline__ void set_slot_row(double4* table, int64_t ne, int64_t e, const double4& v) {
  if (DIM == 3) {
    table[e] = v;
  } else {
    reinterpret_cast<double2*>(table)[e] = make_double2(v.x, v.y);
    reinterpret_cast<double*>(table)[2 * ne + e] = v.w;
  }
}

// bS_i from the status bits and bB, in slot order (so bS is a function of the bits alone).  The
// words are read through L2: other warps of the block may have just written them.
template <int DIM>
__device__ __forceinline__ void bond_sum_row(const StepArgs& a, const SliceIdx& t) {
  const uint32_t* bw = a.bits + (t.base >> 5);
  double sx = 0.0, sy = 0.0, sz = 0.0;
  for (int k = 0; k < t.W; ++k) {
    if ((__ldcg(bw + k) >> t.lane) & 1u) {
      const double4 g = slot_row<DIM>(a.bB, a.ne, t.base + t.lane + ((int64_t)k << 5));
      sx += g.x;
      sy += g.y;
      sz += g.z;
    }
  }
  a.bS[t.i] = make_double4(sx, sy, sz, 0.0);
}

// xi = x_j - x_i, du = u_j - u_i, d = xi . du, q = xi . xi in FP64.  Shared by the FP64 path and by
// the FP64 re-decision of the mixed path, so both decide a bond with identical arithmetic.
template <int DIM>
__device__ __forceinline__ void bond_f64(const double4& pi, const double4& pj, const double4& ui,
                                         const double4& uj, double& ex, double& ey, double& ez,
                                         double& d, double& q) {
  ex = pj.x - pi.x;
  ey = pj.y - pi.y;
  const double dx = uj.x - ui.x, dy = uj.y - ui.y;
  d = ex * dx + ey * dy;
  q = ex * ex + ey * ey;
  if (DIM == 3) {
    ez = pj.z - pi.z;
    const double dz = uj.z - ui.z;
    d = fma(ez, dz, d);
    q = fma(ez, ez, q);
  } else {
    ez = 0.0;
  }
}

// FP64 decision of one bond.  Out of line for the general mixed kernels, which call it only for the
// few bonds inside their rounding band; inlined into the lattice kernel's slow path (fewer registers
// held across a call in its hot loop).
template <int DIM>
__device__ __forceinline__ bool fp64_breaks_inl(const StepArgs& a, int64_t i, int32_t j,
                                                const double4* __restrict__ disp, double s0) {
  double ex, ey, ez, d, q;
  bond_f64<DIM>(a.pos[i], a.pos[j], disp[i], disp[j], ex, ey, ez, d, q);
  return d >= s0 * q;
}
// Explicit update (Eq 2.11) with the diagonal mass rho V_i (Eqs 2.1, 2.12) and the boundary
// conditions at t_{n+1}; f = F_i / V_i.
template <int DIM>
__device__ __forceinline__ void update(const StepArgs& a, int64_t i, int b, const double f[3],
                                       const double4* __restrict__ disp, double4* __restrict__ disp_out,
                                       double4& u) {
  const BodyDev& bp = a.bp[b];
  if (a.adr) {  // adaptive dynamic relaxation: k_adr_update moves the particles after the reduction
    const double4 bb = a.bacc ? a.bacc[i] : make_double4(0.0, 0.0, 0.0, 0.0);
    a.gnew[i] = make_double4(f[0] + bb.x, f[1] + bb.y, f[2] + bb.z, 0.0);
    u = disp[i];
    return;
  }
  const uint8_t fl = a.flag ? a.flag[i] : (uint8_t)0;
  u = disp[i];
  double4 v = a.vel[i];
  if (fl == 0) {
    explicit_move<DIM>(bp, f, a.bacc ? a.bacc + i : nullptr, u, v);
  } else if (fl == 1) {
    u = make_double4(0.0, 0.0, 0.0, u.w);
    v = make_double4(0.0, 0.0, 0.0, 0.0);
  } else {
    const double t1 = (double)(*a.d_step + 1) * bp.dt;
    const double4 g = a.gvec[i];
    const double rt = bp.rate * t1;
    u = make_double4(rt * g.x, rt * g.y, rt * g.z, u.w);
    v = make_double4(bp.rate * g.x, bp.rate * g.y, bp.rate * g.z, 0.0);
  }
  disp_out[i] = u;  // .w carries V_i unchanged
  a.vel[i] = v;
}

// A bond of the geometrically nonlinear model in FP64 (the comment above k_pass1_nl), and the FP64
// re-decision of the mixed kernels with the same arithmetic.
template <int DIM>
struct BondNL {
  double yx, yy, yz;  // Y
  double p;           // |Y|^2 - |xi|^2
  double q;           // |xi|^2
};

template <int DIM>
__device__ __forceinline__ BondNL<DIM> bond_nl(const double4& pi, const double4& pj, const double4& ui,
                                              const double4& uj) {
  BondNL<DIM> r;
  const double ex = pj.x - pi.x, ey = pj.y - pi.y, ez = DIM == 3 ? pj.z - pi.z : 0.0;
  const double hx = uj.x - ui.x, hy = uj.y - ui.y, hz = DIM == 3 ? uj.z - ui.z : 0.0;
  r.yx = ex + hx;
  r.yy = ey + hy;
  r.yz = ez + hz;
  r.p = hx * (ex + r.yx) + hy * (ey + r.yy);
  r.q = ex * ex + ey * ey;
  if (DIM == 3) {
    r.p = fma(hz, ez + r.yz, r.p);
    r.q = fma(ez, ez, r.q);
  }
  return r;
}

template <int DIM>
__device__ __noinline__ bool fp64_breaks_nl(const StepArgs& a, int64_t i, int32_t j,
                                            const double4* __restrict__ disp) {
  const int b = a.body ? a.body[i] : 0;
  const BondNL<DIM> r = bond_nl<DIM>(a.pos[i], a.pos[j], disp[i], disp[j]);
  return r.p >= a.bp[b].s0nl * r.q;
}

// The hardware approximations of 1 / sqrt(x) and 1 / x with a subnormal x read as zero (PTX
// rsqrt.approx.ftz.f32, rcp.approx.ftz.f32), for the FP32 nonlinear kernels: without .ftz each call
// carries a test and rescaling for subnormal inputs.  Their arguments are squared bond lengths and
// sums of bond lengths: |Y|^2 and |Y| + |xi| in units of the coordinate quantum (|xi| >= 1), and
// |Y'|^2 = |n|^2 + p and |Y'| + |n| >= 1 in lattice units, normal numbers for every bond not
// compressed to within 2^-63 of its length, where the results equal those of rsqrtf and __fdividef
// bit for bit.
__device__ __forceinline__ float rsqrt_ftz(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rcp_ftz(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

}  // namespace
}  // namespace pd
