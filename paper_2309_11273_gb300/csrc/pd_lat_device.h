// Device side of the lattice layout, for the mixed step kernels (pd_step.cu) and their resident form
// (pd_resident_lat.cu): direction tables in constant memory (one copy per translation unit), update and shadow.
#pragma once

#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "pd_device.h"
#include "pd_lattice.h"

namespace pd {
namespace {

// Sized to a multiple of 4: slice widths are rounded up to 4 slots, and the slots past the table
// (unused, status 0) still index it.
constexpr int kLatPad3 = (kLatDirs3 + 3) & ~3, kLatPad2 = (kLatDirs2 + 3) & ~3;
__constant__ float4 c_lat3[kLatPad3];   // (n_x, n_y, n_z, |n|^2)
__constant__ float2 c_latr3[kLatPad3];  // 1 / |n|^2 as hi + lo
__constant__ float4 c_lat2[kLatPad2];
__constant__ float2 c_latr2[kLatPad2];
// w' = 1 / |n| as hi + lo: the per-direction factor of the influence function w = delta / |xi|
// (w = (delta / h) w', and delta / h cancels between w and m_i)
__constant__ float2 c_latw3[kLatPad3];
__constant__ float2 c_latw2[kLatPad2];
// |n| rounded to FP32 (nonlinear bonds: e' = (|Y'|^2 - |n|^2) / (|Y'| + |n|) and the dilatation term |n| e')
__constant__ float c_latn3[kLatPad3];
__constant__ float c_latn2[kLatPad2];

template <int DIM>
__device__ __forceinline__ float4 lat_dir(int k) {
  return DIM == 3 ? c_lat3[k] : c_lat2[k];
}
template <int DIM>
__device__ __forceinline__ float2 lat_rcp(int k) {
  return DIM == 3 ? c_latr3[k] : c_latr2[k];
}
template <int DIM>
__device__ __forceinline__ float2 lat_wgt(int k) {
  return DIM == 3 ? c_latw3[k] : c_latw2[k];
}
template <int DIM>
__device__ __forceinline__ float lat_len(int k) {
  return DIM == 3 ? c_latn3[k] : c_latn2[k];
}
// Entry k ^ 1 of the table is -entry k exactly (integer components), with the same |n|^2, 1 / |n|^2
// and w', and a batch starts at a multiple of 4 slots: its four directions are two loaded entries
// and their negations, the sign folded into the arithmetic that uses them (bitwise the same values
// as loading all four).
__device__ __forceinline__ float4 lat_twin(const float4& d, bool odd) {
  return odd ? make_float4(-d.x, -d.y, -d.z, d.w) : d;
}

// The update of the lattice kernels (Eq 2.11 as update() computes it) with F_i / V_i = lat_C x the
// FP32 force sum f and the constants folded: v += lat_K f (+ lat_Kb b), u += dt v, so that a free
// particle costs two FP64 FMAs per component; the z components stay zero in 2D.  Particles under a
// boundary condition and the relaxation solver take update().
template <int DIM>
__device__ __forceinline__ void update_lat(const StepArgs& a, int64_t i, int b, const float f[3],
                                           const double4* __restrict__ disp, double4* __restrict__ disp_out,
                                           double4& u) {
  const BodyDev& bp = a.bp[b];
  const uint8_t fl = a.flag ? a.flag[i] : (uint8_t)0;
  if (a.adr || fl != 0) {
    const double C = bp.lat_C;
    const double fd[3] = {C * (double)f[0], C * (double)f[1], C * (double)f[2]};
    update<DIM>(a, i, b, fd, disp, disp_out, u);
    return;
  }
  u = disp[i];
  double4 v = a.vel[i];
  const double K = bp.lat_K;
  v.x = fma(K, (double)f[0], v.x);
  v.y = fma(K, (double)f[1], v.y);
  if (DIM == 3) v.z = fma(K, (double)f[2], v.z);
  if (a.bacc) {
    const double4 bb = a.bacc[i];
    const double kb = bp.lat_Kb;
    v.x = fma(kb, bb.x, v.x);
    v.y = fma(kb, bb.y, v.y);
    if (DIM == 3) v.z = fma(kb, bb.z, v.z);
  }
  const double dt = bp.dt;
  u.x = fma(dt, v.x, u.x);
  u.y = fma(dt, v.y, u.y);
  if (DIM == 3) u.z = fma(dt, v.z, u.z);
  disp_out[i] = u;  // .w carries V_i unchanged
  a.vel[i] = v;
}

// The FP32 shadow of a displacement in lattice units, (u / h, |u / h|_inf).
template <int DIM>
__device__ __forceinline__ float4 shadow_lat(double inv_h, const double4& u) {
  const float x = (float)(u.x * inv_h), y = (float)(u.y * inv_h), z = DIM == 3 ? (float)(u.z * inv_h) : 0.0f;
  return make_float4(x, y, z, fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z))));
}

// lat_dprime with the x and y differences as one packed FP32 pair addition (the same roundings).
template <int DIM>
__device__ __forceinline__ float lat_dprime_pair(const float4& dn, const float4& uj, const float4& nui) {
  const float2 dxy = __fadd2_rn(make_float2(uj.x, uj.y), make_float2(nui.x, nui.y));
  return lat_dprime_d<DIM>(dn.x, dn.y, dn.z, dxy.x, dxy.y, uj.z + nui.z);
}

// The two-word shadow: hi as shadow_lat, lo = u / h - hi rounded to FP32 (the subtraction is exact in
// FP64), so that hi + lo carries u / h to about 2^-48 of its size.
template <int DIM>
__device__ __forceinline__ void shadow_lat_lo(double inv_h, const double4& u, float4& hi, float4& lo) {
  const double x = u.x * inv_h, y = u.y * inv_h, z = DIM == 3 ? u.z * inv_h : 0.0;
  const float hx = (float)x, hy = (float)y, hz = (float)z;
  hi = make_float4(hx, hy, hz, fmaxf(fabsf(hx), fmaxf(fabsf(hy), fabsf(hz))));
  lo = make_float4((float)(x - (double)hx), (float)(y - (double)hy), (float)(z - (double)hz), 0.0f);
}

// The FP32 shadow of a displacement in the context's format.
__device__ __forceinline__ float4 shadow_of(const StepArgs& a, int b, const double4& u) {
  if (a.lattice) {
    const double s = a.bp[b].lat_inv_h;
    const float x = (float)(u.x * s), y = (float)(u.y * s), z = (float)(u.z * s);
    return make_float4(x, y, z, fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z))));
  }
  const double sc = a.uscale;
  return make_float4((float)(u.x * sc), (float)(u.y * sc), (float)(u.z * sc), 0.0f);
}

// Raises the body's bound umax[b] to at least U (|u'|_inf of a shadow just written; non-negative
// floats order as their bits): one atomic per warp when its particles share a body, else one per
// lane.  All 32 lanes call it.  A NaN U raises the bound to NaN, which settles nothing.
__device__ __forceinline__ void lat_raise_umax(unsigned* umax, int b, float U) {
  const unsigned bits = __float_as_uint(U);
  const int b0 = __shfl_sync(kFull, b, 0);
  if (__all_sync(kFull, b == b0)) {
    const unsigned m = __reduce_max_sync(kFull, bits);
    if ((threadIdx.x & 31) == 0) atomicMax(umax + b0, m);
  } else {
    atomicMax(umax + b, bits);
  }
}

// The direction tables of the lattice kernels, once per device (every context uses the same
// tables, so later uploads would write the same values).
inline pd_status upload_lattice_constants(int device) {
  static std::mutex mu;
  static std::vector<int> done;
  std::lock_guard<std::mutex> lock(mu);
  if (std::find(done.begin(), done.end(), device) != done.end()) return PD_OK;
  for (int dim = 2; dim <= 3; ++dim) {
    const std::vector<LatDir> t = lattice_directions(dim);
    const size_t pad = dim == 3 ? kLatPad3 : kLatPad2;
    std::vector<float4> dn(pad, make_float4(0.0f, 0.0f, 0.0f, 1.0f));
    std::vector<float2> rc(pad, make_float2(0.0f, 0.0f));
    for (size_t k = 0; k < t.size(); ++k) {
      dn[k] = make_float4((float)t[k].n[0], (float)t[k].n[1], (float)t[k].n[2], (float)t[k].q);
      const double r = 1.0 / t[k].q;
      const float hi = (float)r;
      rc[k] = make_float2(hi, (float)(r - (double)hi));
    }
    std::vector<float> ln(pad, 1.0f);
    for (size_t k = 0; k < t.size(); ++k) ln[k] = (float)std::sqrt((double)t[k].q);
    std::vector<float2> wt(pad, make_float2(0.0f, 0.0f));
    for (size_t k = 0; k < t.size(); ++k) {
      const double r = 1.0 / std::sqrt((double)t[k].q);
      const float hi = (float)r;
      wt[k] = make_float2(hi, (float)(r - (double)hi));
    }
    if (dim == 3) {
      PD_CUDA(cudaMemcpyToSymbol(c_lat3, dn.data(), sizeof(float4) * dn.size()));
      PD_CUDA(cudaMemcpyToSymbol(c_latr3, rc.data(), sizeof(float2) * rc.size()));
      PD_CUDA(cudaMemcpyToSymbol(c_latw3, wt.data(), sizeof(float2) * wt.size()));
      PD_CUDA(cudaMemcpyToSymbol(c_latn3, ln.data(), sizeof(float) * ln.size()));
    } else {
      PD_CUDA(cudaMemcpyToSymbol(c_lat2, dn.data(), sizeof(float4) * dn.size()));
      PD_CUDA(cudaMemcpyToSymbol(c_latr2, rc.data(), sizeof(float2) * rc.size()));
      PD_CUDA(cudaMemcpyToSymbol(c_latw2, wt.data(), sizeof(float2) * wt.size()));
      PD_CUDA(cudaMemcpyToSymbol(c_latn2, ln.data(), sizeof(float) * ln.size()));
    }
  }
  done.push_back(device);
  return PD_OK;
}

}  // namespace
}  // namespace pd
