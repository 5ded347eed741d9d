// The resident step kernel of the mixed form on the lattice layout: bodies that fit the chip in one wave
// take all the steps of a pd_step call in one cooperative launch (see pd_resident.cu).
//
// One warp holds one 32-particle slice: its neighbour indices stay in shared memory for the whole call
// (they are most of what a pass reads; rows too long for it are read through L2), its particles' FP64 state
// in registers, and the two passes of a step are separated by a grid barrier.  The arithmetic and the order
// of every sum are those of k_pass1_lat / k_pass2_lat (nonlinear bonds: k_pass1_latnl / k_pass2_latnl), so the
// results are bitwise theirs.  What bounds a step is the barrier (about 1.3 us, twice) and per pass the round trips of a row's gathers: a 402 x 201 plate
// 21.1 -> 14.3 us per step (100 steps and a read), where instruction issue counts too (27 %).
#include <algorithm>
#include <type_traits>

#include "pd_internal.h"
#include "pd_grid.h"
#include "pd_lat_device.h"

namespace pd {
namespace {

struct LatRun {
  double4* disp[2];  // u^n, and the other displacement buffer
  float4* u32[2];    // their FP32 shadows
  float4* lo32[2];   // the shadows' lo words (two-word shadow)
  unsigned* umax[2];  // per body, the bounds of |u'|_inf of the two shadows
  int nsteps;
  int check0;      // the failure check at the head of the first step
  int64_t step0;   // index of the first step
  GridBar grid;
  int row_bytes;   // shared memory of a warp's indices, 0: read through L2
};

constexpr int kLatRowSmem = 200 * 1024;  // shared memory for the rows of a block

// MAXT: the largest block.  A warp keeps the gathers of NB batches of four slots in flight: four up to 256
// threads (255 registers), else two (one with the two-word shadow); the FP64 state stays in registers up to
// 512 threads and is read again at the update beyond.
template <int DIM, bool WI, bool LO, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_resident_lat(StepArgs a, LatRun r) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr bool kKeep = MAXT <= 512;  // the FP64 state in registers
  constexpr int NB = MAXT <= 256 ? 4 : (LO ? 1 : 2);
  constexpr int U = 4;
  // an earlier launch gave up and its error is not yet reported (one answer for the whole block)
  if (__syncthreads_or(ld_relaxed(r.grid.bar + 1) != 0u)) return;
  unsigned target = r.grid.base;
  const SliceIdx t = slice_index<1>(a.n_pad, a.slice_ptr);
  const int lane = t.lane;
  const int64_t i = t.active ? t.i : 0;
  const int W = t.W;
  const int b = t.active && a.body ? a.body[i] : 0;
  const BodyDev& bp = a.bp[b];
  const double s0 = bp.s0;
  const float s0f = bp.lat_s0;
  const bool can_break = bp.breaks != 0;
  const uint32_t lmask = 1u << lane;
  uint32_t* bw = a.bits + (t.base >> 5);
  const int32_t* cs = a.col + t.base + lane;
  if (r.row_bytes) {
    int4* row = reinterpret_cast<int4*>(smem + (threadIdx.x >> 5) * r.row_bytes);
    const int4* src = reinterpret_cast<const int4*>(a.col + t.base);  // slices start on 128-byte boundaries
    for (int k = lane; k < W * 8; k += 32) row[k] = src[k];
    __syncwarp();
    cs = reinterpret_cast<const int32_t*>(row) + lane;
  }
  const uint8_t fl = t.active && a.flag ? a.flag[i] : (uint8_t)0;
  const float2 lf = t.active ? a.lat_f[i] : make_float2(0.0f, 0.0f);  // (N_ref / N_i, A / N_i)
  const bool interior = t.active && a.lat_int[i >> 5] != 0;           // uniform over the warp
  double4 u = make_double4(0.0, 0.0, 0.0, 0.0), v = u;
  if (kKeep && t.active) {
    u = r.disp[0][i];
    v = a.vel[i];
  }
  for (int step = 0; step < r.nsteps; ++step) {
    const int cur = step & 1;
    // (selects, not indices: an indexed kernel argument is copied to local memory)
    const double4* disp = cur ? r.disp[1] : r.disp[0];
    const float4* u32 = cur ? r.u32[1] : r.u32[0];
    const float4* lo32 = cur ? r.lo32[1] : r.lo32[0];
    const unsigned* umax = cur ? r.umax[1] : r.umax[0];
    unsigned* umax_next = cur ? r.umax[0] : r.umax[1];
    const bool checking = step > 0 || r.check0;
    const bool last = step + 1 == r.nsteps;
    // ---- pass 1 (k_pass1_lat)
    if (blockIdx.x == 0)  // the bound of the shadow that pass 2 writes next starts from zero
      for (int k = threadIdx.x; k < a.nbody; k += blockDim.x) umax_next[k] = 0u;
    float4 Ui = make_float4(0.0f, 0.0f, 0.0f, 0.0f), Li = Ui;
    float P = 0.0f;
    if (t.active) {
      Ui = u32[i];
      if (LO) Li = lo32[i];
      const float4 nUi = make_float4(-Ui.x, -Ui.y, -Ui.z, 0.0f);
      const float umax_b = lat_umax_bound(__uint_as_float(__ldcg(umax + b)));
      const float scr_i = (can_break && checking) ? lat_screen_part(bp.lat_Kfast, Ui.w, umax_b, bp.lat_Kcfast) : -INFINITY;
      float acc = 0.0f;
      for (int k0 = 0; k0 < W; k0 += NB * U) {
        uint4 w4[NB];
        float4 Uj[NB][U], Lj[NB][U];
#pragma unroll
        for (int h = 0; h < NB; ++h) {
          const int k = k0 + h * U;
          w4[h] = k < W ? *reinterpret_cast<const uint4*>(bw + k) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
          for (int q = 0; q < U; ++q) {
            const int32_t j = cs[min(k + q, W - 1) * 32];
            Uj[h][q] = u32[j];
            if (LO) Lj[h][q] = lo32[j];
          }
        }
#pragma unroll
        for (int h = 0; h < NB; ++h) {
          const int k = k0 + h * U;
          if ((w4[h].x | w4[h].y | w4[h].z | w4[h].w) == 0u) continue;  // the same words in every lane
          const uint32_t wd[U] = {w4[h].x, w4[h].y, w4[h].z, w4[h].w};
          float dm[U];
          float gmax = -INFINITY;
          const float4 dA = lat_dir<DIM>(k), dB = lat_dir<DIM>(k + 2);
#pragma unroll
          for (int q = 0; q < U; ++q) {
            const float4 dn = lat_twin(q < 2 ? dA : dB, q & 1);
            const float d = LO ? lat_dprime_d<DIM>(dn.x, dn.y, dn.z, lat_delta_lo(Uj[h][q].x, Lj[h][q].x, Ui.x, Li.x),
                                                   lat_delta_lo(Uj[h][q].y, Lj[h][q].y, Ui.y, Li.y),
                                                   lat_delta_lo(Uj[h][q].z, Lj[h][q].z, Ui.z, Li.z))
                               : lat_dprime_pair<DIM>(dn, Uj[h][q], nUi);
            dm[q] = (wd[q] & lmask) ? d : 0.0f;
          }
          gmax = lat_max3_nan(gmax, lat_g(lat_max_nan(dm[0], dm[1]), s0f, dA.w), lat_g(lat_max_nan(dm[2], dm[3]), s0f, dB.w));
          if (__any_sync(kFull, !(gmax + scr_i < 0.0f))) {
            // full band for the bonds the screen did not settle, FP64 inside it
            unsigned brk = 0u;
#pragma unroll 1
            for (int q = 0; q < U; ++q) {
              int code = 0;
              const uint32_t w = q == 0 ? w4[h].x : (q == 1 ? w4[h].y : (q == 2 ? w4[h].z : w4[h].w));
              if (checking && can_break && (w & lmask) != 0u) {
                const int32_t jj = cs[(k + q) * 32];
                const float qn = lat_dir<DIM>(k + q).w;
                const float du = q == 0 ? dm[0] : (q == 1 ? dm[1] : (q == 2 ? dm[2] : dm[3]));
                code = lat_code(lat_g(du, s0f, qn), Ui.w, u32[jj].w, s0f, qn, bp.lat_Kf, bp.lat_sq, bp.lat_eps_c, bp.lat_s0n1);
                if (code == 2) {
                  code = fp64_breaks_inl<DIM>(a, i, jj, disp, s0) ? 1 : 0;
                  atomicAdd(&a.counters[0], 1ull);
                }
              }
              const unsigned m = __ballot_sync(kFull, code == 1);
              if (m) {
                if (lane == 0) bw[k + q] = w & ~m;
                if (code == 1) brk |= 1u << q;
              }
            }
#pragma unroll
            for (int q = 0; q < U; ++q) dm[q] = ((brk >> q) & 1u) ? 0.0f : dm[q];
          }
          float2 wA = make_float2(1.0f, 0.0f), wB = wA;
          if (WI) {
            wA = lat_wgt<DIM>(k);
            wB = lat_wgt<DIM>(k + 2);
          }
#pragma unroll
          for (int q = 0; q < U; ++q) {
            if (WI) {
              const float2 wk = q < 2 ? wA : wB;
              acc = fmaf(wk.x, dm[q], fmaf(wk.y, dm[q], acc));
            } else {
              acc += dm[q];
            }
          }
        }
      }
      if (last) a.theta32[i] = lf.y * acc;
      const float x = acc * (lf.x * lf.x);
      P = fmaf(bp.lat_lam_hi, x, bp.lat_lam_lo * x);
      a.lat_up[i] = make_float4(Ui.x, Ui.y, Ui.z, P);
    }
    if (!grid_barrier(a, r.grid, target)) return;
    // ---- pass 2 (k_pass2_lat)
    if (t.active) {
      float f[3] = {0.0f, 0.0f, 0.0f};
      auto row = [&](auto intr) {
        constexpr bool INTR = decltype(intr)::value;
        for (int k0 = 0; k0 < W; k0 += NB * U) {
          uint4 w4[NB];
          float4 Uj[NB][U], Lj[NB][U];
          float rr[NB][U];
#pragma unroll
          for (int h = 0; h < NB; ++h) {
            const int k = k0 + h * U;
            w4[h] = k < W ? *reinterpret_cast<const uint4*>(bw + k) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int q = 0; q < U; ++q) {
              const int32_t j = cs[min(k + q, W - 1) * 32];
              Uj[h][q] = a.lat_up[j];
              if (LO) Lj[h][q] = lo32[j];
              rr[h][q] = INTR ? 2.0f : lf.x + a.lat_rho[j];
            }
          }
#pragma unroll
          for (int h = 0; h < NB; ++h) {
            const int k = k0 + h * U;
            if ((w4[h].x | w4[h].y | w4[h].z | w4[h].w) == 0u) continue;
            const uint32_t wd[U] = {w4[h].x, w4[h].y, w4[h].z, w4[h].w};
            const float4 dA = lat_dir<DIM>(k), dB = lat_dir<DIM>(k + 2);
            const float2 rA = lat_rcp<DIM>(k), rB = lat_rcp<DIM>(k + 2);
            float2 wA = make_float2(1.0f, 0.0f), wB = wA;
            if (WI) {
              wA = lat_wgt<DIM>(k);
              wB = lat_wgt<DIM>(k + 2);
            }
            float cfm[U];
#pragma unroll
            for (int q = 0; q < U; ++q) {
              const float4 dn = lat_twin(q < 2 ? dA : dB, q & 1);
              const float2 rc = q < 2 ? rA : rB;
              const float d = LO ? lat_dprime_d<DIM>(dn.x, dn.y, dn.z, lat_delta_lo(Uj[h][q].x, Lj[h][q].x, Ui.x, Li.x),
                                                     lat_delta_lo(Uj[h][q].y, Lj[h][q].y, Ui.y, Li.y),
                                                     lat_delta_lo(Uj[h][q].z, Lj[h][q].z, Ui.z, Li.z))
                                 : lat_dprime<DIM>(dn.x, dn.y, dn.z, Uj[h][q].x, Uj[h][q].y, Uj[h][q].z, Ui.x, Ui.y, Ui.z);
              const float dr = fmaf(d, rc.x, d * rc.y);
              float cf = fmaf(rr[h][q], dr, P + Uj[h][q].w);
              if (WI) {
                const float2 wk = q < 2 ? wA : wB;
                cf = fmaf(cf, wk.x, cf * wk.y);
              }
              cfm[q] = (wd[q] & lmask) ? cf : 0.0f;
            }
#pragma unroll
            for (int p = 0; p < U / 2; ++p) {
              const float dd = cfm[2 * p] - cfm[2 * p + 1];
              const float4& dn = p == 0 ? dA : dB;
              f[0] = fmaf(dd, dn.x, f[0]);
              f[1] = fmaf(dd, dn.y, f[1]);
              if (DIM == 3) f[2] = fmaf(dd, dn.z, f[2]);
            }
          }
        }
      };
      if (interior) row(std::true_type{});
      else row(std::false_type{});
      // update (update_lat, update)
      if (!kKeep) {
        u = disp[i];
        v = a.vel[i];
      }
      if (fl == 0) {
        const double K = bp.lat_K, dt = bp.dt;
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
        u.x = fma(dt, v.x, u.x);
        u.y = fma(dt, v.y, u.y);
        if (DIM == 3) u.z = fma(dt, v.z, u.z);
      } else if (fl == 1) {
        u = make_double4(0.0, 0.0, 0.0, u.w);
        v = make_double4(0.0, 0.0, 0.0, 0.0);
      } else {
        const double t1 = (double)(r.step0 + step + 1) * bp.dt;
        const double4 g = a.gvec[i];
        const double rt = bp.rate * t1;
        u = make_double4(rt * g.x, rt * g.y, rt * g.z, u.w);
        v = make_double4(bp.rate * g.x, bp.rate * g.y, bp.rate * g.z, 0.0);
      }
      (cur ? r.disp[0] : r.disp[1])[i] = u;
      float4 hi;
      if (LO) {
        float4 lo;
        shadow_lat_lo<DIM>(bp.lat_inv_h, u, hi, lo);
        (cur ? r.lo32[0] : r.lo32[1])[i] = lo;
      } else {
        hi = shadow_lat<DIM>(bp.lat_inv_h, u);
      }
      (cur ? r.u32[0] : r.u32[1])[i] = hi;
      lat_raise_umax(umax_next, b, hi.w);
      if (!kKeep || last) a.vel[i] = v;
    }
    if (!last && !grid_barrier(a, r.grid, target)) return;
  }
  if (t.active && (!isfinite(u.x) || !isfinite(u.y) || !isfinite(u.z))) atomicExch(&a.counters[5], 1ull);
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.d_step = r.step0 + r.nsteps - 1;
}

// The same with geometrically nonlinear bonds (k_pass1_latnl / k_pass2_latnl).
template <int DIM, bool LO, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_resident_latnl(StepArgs a, LatRun r) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr bool kKeep = MAXT <= 512;  // the FP64 state in registers
  constexpr int NB = MAXT <= 256 ? 4 : (LO ? 1 : 2);
  constexpr int U = 4;
  // an earlier launch gave up and its error is not yet reported (one answer for the whole block)
  if (__syncthreads_or(ld_relaxed(r.grid.bar + 1) != 0u)) return;
  unsigned target = r.grid.base;
  const SliceIdx t = slice_index<1>(a.n_pad, a.slice_ptr);
  const int lane = t.lane;
  const int64_t i = t.active ? t.i : 0;
  const int W = t.W;
  const int b = t.active && a.body ? a.body[i] : 0;
  const BodyDev& bp = a.bp[b];
  const float c32 = bp.s0nl32;
  const bool can_break = bp.breaks != 0;
  const uint32_t lmask = 1u << lane;
  uint32_t* bw = a.bits + (t.base >> 5);
  const int32_t* cs = a.col + t.base + lane;
  if (r.row_bytes) {
    int4* row = reinterpret_cast<int4*>(smem + (threadIdx.x >> 5) * r.row_bytes);
    const int4* src = reinterpret_cast<const int4*>(a.col + t.base);  // slices start on 128-byte boundaries
    for (int k = lane; k < W * 8; k += 32) row[k] = src[k];
    __syncwarp();
    cs = reinterpret_cast<const int32_t*>(row) + lane;
  }
  const uint8_t fl = t.active && a.flag ? a.flag[i] : (uint8_t)0;
  const float2 lf = t.active ? a.lat_f[i] : make_float2(0.0f, 0.0f);  // (N_ref / N_i, A / N_i)
  const bool interior = t.active && a.lat_int[i >> 5] != 0;           // uniform over the warp
  double4 u = make_double4(0.0, 0.0, 0.0, 0.0), v = u;
  if (kKeep && t.active) {
    u = r.disp[0][i];
    v = a.vel[i];
  }
  for (int step = 0; step < r.nsteps; ++step) {
    const int cur = step & 1;
    // (selects, not indices: an indexed kernel argument is copied to local memory)
    const double4* disp = cur ? r.disp[1] : r.disp[0];
    const float4* u32 = cur ? r.u32[1] : r.u32[0];
    const float4* lo32 = cur ? r.lo32[1] : r.lo32[0];
    const unsigned* umax = cur ? r.umax[1] : r.umax[0];
    unsigned* umax_next = cur ? r.umax[0] : r.umax[1];
    const bool checking = step > 0 || r.check0;
    const bool last = step + 1 == r.nsteps;
    // ---- pass 1 (k_pass1_latnl)
    if (blockIdx.x == 0)  // the bound of the shadow that pass 2 writes next starts from zero
      for (int k = threadIdx.x; k < a.nbody; k += blockDim.x) umax_next[k] = 0u;
    float4 Ui = make_float4(0.0f, 0.0f, 0.0f, 0.0f), Li = Ui;
    float P = 0.0f;
    if (t.active) {
      Ui = u32[i];
      if (LO) Li = lo32[i];
      const float4 nUi = make_float4(-Ui.x, -Ui.y, -Ui.z, 0.0f);
      const bool screening = can_break && checking;
      const float Smax = Ui.w + lat_umax_bound(__uint_as_float(__ldcg(umax + b)));
      const float f0 = fmaf(bp.nl_F0s, Smax, bp.nl_F0), f1 = fmaf(bp.nl_F1s, Smax, bp.nl_F1), F2 = bp.nl_F2;
      float acc = 0.0f;
      for (int k0 = 0; k0 < W; k0 += NB * U) {
        uint4 w4[NB];
        float4 Uj[NB][U], Lj[NB][U];
#pragma unroll
        for (int h = 0; h < NB; ++h) {
          const int k = k0 + h * U;
          w4[h] = k < W ? *reinterpret_cast<const uint4*>(bw + k) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
          for (int q = 0; q < U; ++q) {
            const int32_t j = cs[min(k + q, W - 1) * 32];
            Uj[h][q] = u32[j];
            if (LO) Lj[h][q] = lo32[j];
          }
        }
#pragma unroll
        for (int h = 0; h < NB; ++h) {
          const int k = k0 + h * U;
          if ((w4[h].x | w4[h].y | w4[h].z | w4[h].w) == 0u) continue;  // the same words in every lane
          const uint32_t wd[U] = {w4[h].x, w4[h].y, w4[h].z, w4[h].w};
          float ev[U];  // e' of the intact bonds (0 for the others)
          float smax = -INFINITY;
          const float4 dA = lat_dir<DIM>(k), dB = lat_dir<DIM>(k + 2);
          const float lA = lat_len<DIM>(k), lB = lat_len<DIM>(k + 2);
#pragma unroll
          for (int q = 0; q < U; ++q) {
            const float4 dn = lat_twin(q < 2 ? dA : dB, q & 1);
            const float nl = q < 2 ? lA : lB;
            const float2 exy = LO ? make_float2(lat_delta_lo(Uj[h][q].x, Lj[h][q].x, Ui.x, Li.x),
                                                lat_delta_lo(Uj[h][q].y, Lj[h][q].y, Ui.y, Li.y))
                                  : __fadd2_rn(make_float2(Uj[h][q].x, Uj[h][q].y), make_float2(nUi.x, nUi.y));
            const float ez = DIM == 3 ? (LO ? lat_delta_lo(Uj[h][q].z, Lj[h][q].z, Ui.z, Li.z) : Uj[h][q].z + nUi.z) : 0.0f;
            const bool in = (wd[q] & lmask) != 0u;
            const float pp = lat_p_nl<DIM>(dn.x, dn.y, dn.z, exy.x, exy.y, ez);
            const float q2 = dn.w + pp;  // |Y'|^2 = |n|^2 + p
            const float pm = in ? pp : 0.0f;
            ev[q] = in ? pp * rcp_ftz(fmaf(q2, rsqrt_ftz(q2), nl)) : 0.0f;
            if (screening) {
              const float Dn = in ? fabsf(exy.x) + fabsf(exy.y) + fabsf(ez) : 0.0f;
              smax = lat_max_nan(smax, lat_g_nl(pm, c32, dn.w) + lat_screen_nl(Dn, f0, f1, F2));
            }
          }
          unsigned brk = 0u;
          if (__any_sync(kFull, screening && !(smax < 0.0f))) {
            // full band for every intact bond of the batch, FP64 inside it
#pragma unroll 1
            for (int q = 0; q < U; ++q) {
              int code = 0;
              const uint32_t w = q == 0 ? w4[h].x : (q == 1 ? w4[h].y : (q == 2 ? w4[h].z : w4[h].w));
              if (checking && can_break && (w & lmask) != 0u) {
                const int32_t jj = cs[(k + q) * 32];
                const float4 uj = u32[jj];
                const float4 lj = LO ? lo32[jj] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                const float4 dn = lat_dir<DIM>(k + q);
                const float ex = LO ? lat_delta_lo(uj.x, lj.x, Ui.x, Li.x) : uj.x - Ui.x;
                const float ey = LO ? lat_delta_lo(uj.y, lj.y, Ui.y, Li.y) : uj.y - Ui.y;
                const float ez = DIM == 3 ? (LO ? lat_delta_lo(uj.z, lj.z, Ui.z, Li.z) : uj.z - Ui.z) : 0.0f;
                const float g = lat_g_nl(lat_p_nl<DIM>(dn.x, dn.y, dn.z, ex, ey, ez), c32, dn.w);
                LatBandNL band;
                band.A0 = bp.nl_A0;
                band.A0s = bp.nl_A0s;
                band.A1 = bp.nl_A1;
                band.A1s = bp.nl_A1s;
                band.A2 = bp.nl_A2;
                band.Ag = bp.nl_Ag;
                code = lat_code_nl(g, fabsf(ex) + fabsf(ey) + fabsf(ez), Ui.w + uj.w, band);
                if (code == 2) {
                  code = fp64_breaks_nl<DIM>(a, i, jj, disp) ? 1 : 0;
                  atomicAdd(&a.counters[0], 1ull);
                }
              }
              const unsigned m = __ballot_sync(kFull, code == 1);
              if (m) {
                if (lane == 0) bw[k + q] = w & ~m;
                if (code == 1) brk |= 1u << q;
              }
            }
          }
#pragma unroll
          for (int q = 0; q < U; ++q) acc = fmaf(q < 2 ? lA : lB, ((brk >> q) & 1u) ? 0.0f : ev[q], acc);
        }
      }
      if (last) a.theta32[i] = lf.y * acc;
      const float x = acc * (lf.x * lf.x);
      P = fmaf(bp.lat_lam_hi, x, bp.lat_lam_lo * x);
      a.lat_up[i] = make_float4(Ui.x, Ui.y, Ui.z, P);
    }
    if (!grid_barrier(a, r.grid, target)) return;
    // ---- pass 2 (k_pass2_latnl)
    if (t.active) {
      float f[3] = {0.0f, 0.0f, 0.0f};
      const float4 nUi = make_float4(-Ui.x, -Ui.y, -Ui.z, 0.0f);
      auto row = [&](auto intr) {
        constexpr bool INTR = decltype(intr)::value;
        for (int k0 = 0; k0 < W; k0 += NB * U) {
          uint4 w4[NB];
          float4 Uj[NB][U], Lj[NB][U];
          float rr[NB][U];
#pragma unroll
          for (int h = 0; h < NB; ++h) {
            const int k = k0 + h * U;
            w4[h] = k < W ? *reinterpret_cast<const uint4*>(bw + k) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int q = 0; q < U; ++q) {
              const int32_t j = cs[min(k + q, W - 1) * 32];
              Uj[h][q] = a.lat_up[j];
              if (LO) Lj[h][q] = lo32[j];
              rr[h][q] = INTR ? 2.0f : lf.x + a.lat_rho[j];
            }
          }
#pragma unroll
          for (int h = 0; h < NB; ++h) {
            const int k = k0 + h * U;
            if ((w4[h].x | w4[h].y | w4[h].z | w4[h].w) == 0u) continue;
            const uint32_t wd[U] = {w4[h].x, w4[h].y, w4[h].z, w4[h].w};
            const float4 dA = lat_dir<DIM>(k), dB = lat_dir<DIM>(k + 2);
            const float lA = lat_len<DIM>(k), lB = lat_len<DIM>(k + 2);
#pragma unroll
            for (int q = 0; q < U; ++q) {
              const float4 dn = lat_twin(q < 2 ? dA : dB, q & 1);
              const float nl = q < 2 ? lA : lB;
              const float2 exy = LO ? make_float2(lat_delta_lo(Uj[h][q].x, Lj[h][q].x, Ui.x, Li.x),
                                                  lat_delta_lo(Uj[h][q].y, Lj[h][q].y, Ui.y, Li.y))
                                    : __fadd2_rn(make_float2(Uj[h][q].x, Uj[h][q].y), make_float2(nUi.x, nUi.y));
              const float ez = DIM == 3 ? (LO ? lat_delta_lo(Uj[h][q].z, Lj[h][q].z, Ui.z, Li.z) : Uj[h][q].z + nUi.z) : 0.0f;
              const float pp = lat_p_nl<DIM>(dn.x, dn.y, dn.z, exy.x, exy.y, ez);
              const float yx = dn.x + exy.x, yy = dn.y + exy.y, yz = dn.z + ez;
              const float q2 = dn.w + pp;
              const float ry = rsqrt_ftz(q2);
              const float e = pp * rcp_ftz(fmaf(q2, ry, nl));
              float cf = fmaf(rr[h][q], e, (P + Uj[h][q].w) * nl) * ry;
              cf = (wd[q] & lmask) ? cf : 0.0f;
              f[0] = fmaf(cf, yx, f[0]);
              f[1] = fmaf(cf, yy, f[1]);
              if (DIM == 3) f[2] = fmaf(cf, yz, f[2]);
            }
          }
        }
      };
      if (interior) row(std::true_type{});
      else row(std::false_type{});
      // update (update_lat, update)
      if (!kKeep) {
        u = disp[i];
        v = a.vel[i];
      }
      if (fl == 0) {
        const double K = bp.lat_K, dt = bp.dt;
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
        u.x = fma(dt, v.x, u.x);
        u.y = fma(dt, v.y, u.y);
        if (DIM == 3) u.z = fma(dt, v.z, u.z);
      } else if (fl == 1) {
        u = make_double4(0.0, 0.0, 0.0, u.w);
        v = make_double4(0.0, 0.0, 0.0, 0.0);
      } else {
        const double t1 = (double)(r.step0 + step + 1) * bp.dt;
        const double4 g = a.gvec[i];
        const double rt = bp.rate * t1;
        u = make_double4(rt * g.x, rt * g.y, rt * g.z, u.w);
        v = make_double4(bp.rate * g.x, bp.rate * g.y, bp.rate * g.z, 0.0);
      }
      (cur ? r.disp[0] : r.disp[1])[i] = u;
      float4 hi;
      if (LO) {
        float4 lo;
        shadow_lat_lo<DIM>(bp.lat_inv_h, u, hi, lo);
        (cur ? r.lo32[0] : r.lo32[1])[i] = lo;
      } else {
        hi = shadow_lat<DIM>(bp.lat_inv_h, u);
      }
      (cur ? r.u32[0] : r.u32[1])[i] = hi;
      lat_raise_umax(umax_next, b, hi.w);
      if (!kKeep || last) a.vel[i] = v;
    }
    if (!last && !grid_barrier(a, r.grid, target)) return;
  }
  if (t.active && (!isfinite(u.x) || !isfinite(u.y) || !isfinite(u.z))) atomicExch(&a.counters[5], 1ull);
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.d_step = r.step0 + r.nsteps - 1;
}

cudaError_t launch(pd_ctx* c, const void* kernel, StepArgs a, LatRun r, unsigned grid, int block) {
  const size_t sm = (size_t)(block / 32) * r.row_bytes;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kLatRowSmem);
  if (e != cudaSuccess) return e;
  void* args[] = {&a, &r};
  return cudaLaunchCooperativeKernel(kernel, dim3(grid), dim3((unsigned)block), args, sm, c->stream);
}

template <int DIM, bool LO, int MAXT>
const void* kernel_of(const pd_ctx* c) {
  if (c->kin == PD_NONLINEAR) return (const void*)k_resident_latnl<DIM, LO, MAXT>;
  return c->prm[0].influence == PD_W_INV ? (const void*)k_resident_lat<DIM, true, LO, MAXT>
                                         : (const void*)k_resident_lat<DIM, false, LO, MAXT>;
}

template <int DIM, bool LO>
const void* kernel_for(const pd_ctx* c, int block) {
  return block > 512 ? kernel_of<DIM, LO, 768>(c) : (block > 256 ? kernel_of<DIM, LO, 512>(c) : kernel_of<DIM, LO, 256>(c));
}

}  // namespace

pd_status upload_resident_tables(int device) { return upload_lattice_constants(device); }

ResidentPlan resident_lat_plan(const pd_ctx* c) {
  ResidentPlan p;
  if (!c->resident || !c->auto_map || c->precision != PD_MIXED || !c->lattice || c->validate || c->profile ||
      c->solver != PD_SOLVER_EXPLICIT || c->sms <= 0)
    return p;
  const int64_t warps = (c->nslices + c->sms - 1) / c->sms;  // per block, one block per SM
  if (warps > 24) return p;                                 // 768 threads of 80 registers
  p.split = 1;
  p.block = (int)warps * 32;
  p.grid = (unsigned)((c->nslices + warps - 1) / warps);
  return p;
}

pd_status run_resident_lat(pd_ctx* c, const StepArgs& a, const ResidentPlan& p, int64_t nsteps, bool check0, bool* done) {
  *done = false;
  if (const pd_status st = ensure_grid_bar(c); st != PD_OK) {
    if (st != PD_ERR_OOM) return st;
    clear_error();
    return PD_OK;  // no room for the barrier's words: the pass kernels take the steps
  }
  LatRun r{};
  for (int k = 0; k < 2; ++k) {
    const int s = c->cur ^ k;
    r.disp[k] = c->disp[s];
    r.u32[k] = c->u32[s];
    r.lo32[k] = c->shadow_lo ? c->u32lo[s] : nullptr;
    r.umax[k] = c->lat_umax + (size_t)s * c->nbodies;
  }
  r.nsteps = (int)nsteps;
  r.check0 = check0 ? 1 : 0;
  r.step0 = c->steps;
  r.grid = GridBar{c->bar, c->bar_base};
  const int row = c->lat_wmax * 128;
  r.row_bytes = row * (p.block / 32) <= kLatRowSmem ? row : 0;
  const void* kernel = c->dim == 3 ? (c->shadow_lo ? kernel_for<3, true>(c, p.block) : kernel_for<3, false>(c, p.block))
                                   : (c->shadow_lo ? kernel_for<2, true>(c, p.block) : kernel_for<2, false>(c, p.block));
  const cudaError_t e = launch(c, kernel, a, r, p.grid, p.block);
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
    cudaGetLastError();
    c->sms = 0;  // this device (or this share of it) cannot hold the grid: the pass kernels take the steps
    return PD_OK;
  }
  if (e != cudaSuccess) return cuda_fail(e, "cudaLaunchCooperativeKernel");
  c->bar_base += p.grid * (2u * (unsigned)nsteps - 1u);
  if (nsteps & 1) c->cur ^= 1;
  *done = true;
  return PD_OK;
}

}  // namespace pd
