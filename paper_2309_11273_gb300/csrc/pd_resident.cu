// The resident step kernel: bodies that fit the chip in one wave take all the steps of a pd_step call in
// one cooperative launch.
//
// On a body of up to about a hundred thousand particles a step of the pass kernels is shorter than what
// surrounds it: three launches, each with its ramp up and its last warps, and per launch the chain index ->
// gather -> sum of a slice's row.  Here one block per SM holds its slices for the whole call; the
// displacements and velocities of its particles stay in registers, and the passes are separated by a grid
// barrier (about 1.3 us) instead of a launch: a 40 x 40 plate 33.7 -> 8.6 us per step (100 steps and a read), a
// 400 x 160 plate 63 -> 34 us, bound there by the FP64 pipe (60 %) and the passes' ramps.  The arithmetic is that of
// k_pass1a_f64p / k_pass1b_f64p / k_pass2_f64t (pair form) or k_pass1_f64t / k_pass2_f64t, with the same
// order of every sum (parts_sum), so the results are bitwise those of the pass kernels.
#include <algorithm>

#include "pd_internal.h"
#include "pd_device.h"
#include "pd_grid.h"

namespace pd {
namespace {

struct ResidentArgs {
  double4* disp;       // u^n
  double4* disp_out;   // the other displacement buffer
  int nsteps;
  int check0;          // the failure check at the head of the first step
  int64_t step0;       // index of the first step
  GridBar grid;
  int uv;              // every body has one particle volume
};

// A line of a static stream to L2, some batches before its load.
__device__ __forceinline__ void to_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
template <int DIM>
__device__ __forceinline__ void row_to_l2(const double4* table, int64_t ne, int64_t e) {
  if (DIM == 3) {
    to_l2(table + e);
  } else {
    to_l2(reinterpret_cast<const double2*>(table) + e);
    to_l2(reinterpret_cast<const double*>(table) + 2 * ne + e);
  }
}

// PAIR: pass 1 in its pair form (fewer FP64 instructions, one barrier more).  MAXT: the largest block.  Up to
// 512 threads (128 registers) four slots are in flight per warp (eight up to 256 threads without the pair
// form) and the state stays in registers; up to
// 768 (80 registers) two, and the state is read again at the update.  Without the pair form, on the
// smallest bodies, the neighbour indices are loaded a batch ahead, and a pass's first ones before the
// barrier in front of it, so that a batch waits for one round trip to L2 instead of two (40 x 40 plate 9.7
// -> 9.1 us per step); the pair form spills with it (400 x 160 plate 39.8 -> 41.3 us).
template <int DIM, int SPLIT, bool PAIR, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_resident(StepArgs a, ResidentArgs r) {
  constexpr int P = 4 / SPLIT;
  constexpr bool kKeep = MAXT <= 512;  // the particles' state in registers
  constexpr int U = MAXT <= 256 && !PAIR ? 8 : (kKeep ? 4 : 2);
  constexpr int H = P > U ? P / U : 1;
  // Batches of the static streams fetched to L2 ahead: the tables of a larger 3D body do not stay there from step to
  // step, and each batch waited for its indices and then its rows from memory.  With four warps per slice the body
  // (up to 19,456 particles) is small enough to stay.  us per step with 0 / 2 / 4 batches: two warps per slice, 28^3
  // 74 / 70 / 73, 32^3 90 / 87 / 92, 36^3 120 / 107 / 114; four, 20^3 32.4 / 36.0 / 36.1, 24^3 43.9 / 46.9 / 47.4.
  constexpr int kAhead = PAIR && DIM == 3 && SPLIT < 4 ? 2 : 0;
  // an earlier launch gave up and its error is not yet reported (one answer for the whole block)
  if (__syncthreads_or(ld_relaxed(r.grid.bar + 1) != 0u)) return;
  unsigned target = r.grid.base;
  const SliceIdx t = slice_index<SPLIT>(a.n_pad, a.slice_ptr);
  const bool lead = t.active && t.sub == 0;
  const int64_t i = t.active ? t.i : 0, s = i >> 5;
  const int b = t.active && a.body ? a.body[i] : 0;
  const BodyDev& bp = a.bp[b];
  const bool can_break = bp.breaks != 0;
  const int own = t.active ? a.own0[i] : 0, cnt = t.active ? a.cnt[i] : 0;
  const int nown = __reduce_max_sync(kFull, (unsigned)(cnt - own));
  uint32_t* bw = a.bits + (t.base >> 5);
  const int32_t* cl = a.col + t.base + t.lane;
  const int32_t* tw = a.twin + t.base + t.lane;
  const int64_t e0 = t.base + t.lane;
  double* td = a.bd + t.base + t.lane;
  const uint8_t fl = lead && a.flag ? a.flag[i] : (uint8_t)0;
  double4 u = make_double4(0.0, 0.0, 0.0, 0.0), v = u, bb = u;
  auto load_state = [&](const double4* disp) {  // of the slice's first warp
    if (!lead) return;
    u = disp[i];
    v = a.vel[i];
    if (a.bacc) bb = a.bacc[i];
  };
  if (kKeep) load_state(r.disp);
  const double vi = t.active ? a.pos[i].w : 0.0;
  // the neighbours of a batch of slots (past the row: its last one), loaded in place or ahead
  int32_t jn[U];
  auto slots = [&](int k0, bool ahead) {
    if (ahead == PAIR || !t.active || k0 >= t.W) return;
#pragma unroll
    for (int q = 0; q < U; ++q) jn[q] = cl[(int64_t)min(k0 + q * SPLIT, t.W - 1) << 5];
  };
  slots(t.sub, true);
  for (int step = 0; step < r.nsteps; ++step) {
    const double4* disp = (step & 1) ? r.disp_out : r.disp;
    double4* disp_out = (step & 1) ? r.disp : r.disp_out;
    const bool check = (step > 0 || r.check0) && can_break;
    double sum[2] = {0.0, 0.0}, part1[1][P] = {};
    // ---- pass 1
    if (PAIR) {
      if (t.active) {
        const double4 ui = disp[i];
        for (int m0 = t.sub; m0 < nown; m0 += U * SPLIT) {
          int32_t j[U], te[U];
          double4 g[U], uj[U];
#pragma unroll
          for (int q = 0; q < U; ++q) {
            const int64_t k = (int64_t)min(own + m0 + q * SPLIT, max(cnt - 1, 0)) << 5;
            j[q] = cl[k];
            te[q] = tw[k];
            g[q] = slot_row<DIM>(a.bA, a.ne, e0 + k);
            uj[q] = disp[j[q]];
          }
          if (kAhead > 0)
#pragma unroll
            for (int q = 0; q < U; ++q) {
              const int64_t k = (int64_t)min(own + m0 + (q + kAhead * U) * SPLIT, max(cnt - 1, 0)) << 5;
              to_l2(cl + k);
              to_l2(tw + k);
              row_to_l2<DIM>(a.bA, a.ne, e0 + k);
            }
#pragma unroll
          for (int q = 0; q < U; ++q) {
            const int k = own + m0 + q * SPLIT;
            if (k >= cnt) continue;
            double d = g[q].x * (uj[q].x - ui.x) + g[q].y * (uj[q].y - ui.y);
            if (DIM == 3) d = fma(g[q].z, uj[q].z - ui.z, d);
            td[(int64_t)k << 5] = d;
            a.bd[te[q]] = d;
            if (check && ((bw[k] >> t.lane) & 1u) && pd_ge_threshold(d, g[q].w)) {  // d >= s0 |xi|^2
              atomicAnd(&bw[k], ~(1u << t.lane));
              atomicAnd(a.bits + (te[q] >> 5), ~(1u << (te[q] & 31)));
              a.dirty[s] = 1;
              a.dirty[j[q] >> 5] = 1;
            }
          }
        }
      }
      if (!grid_barrier(a, r.grid, target)) return;
      if (t.active) {
        for (int k0 = t.sub; k0 < t.W; k0 += 4) {  // slots k0, k0 + SPLIT, ...: the sum's parts
#pragma unroll
          for (int q = 0; q < P; ++q) {
            const int k = k0 + q * SPLIT;
            const double vj = r.uv ? vi : disp[cl[(int64_t)k << 5]].w;
            if ((bw[k] >> t.lane) & 1u) part1[0][q] = fma(vj, td[(int64_t)k << 5], part1[0][q]);
          }
        }
      }
    } else {
      if (t.active) {
        const double4 ui = disp[i];
        for (int kb = t.sub; kb < t.W; kb += H * U * SPLIT) {
#pragma unroll
          for (int h = 0; h < H; ++h) {
            const int k0 = kb + h * U * SPLIT;
            uint32_t wd[U];
            double4 g[U], uj[U];
#pragma unroll
            for (int q = 0; q < U; ++q) {
              const int k = min(k0 + q * SPLIT, t.W - 1);
              wd[q] = k0 + q * SPLIT < t.W ? bw[k] : 0u;
              g[q] = slot_row<DIM>(a.bA, a.ne, e0 + ((int64_t)k << 5));
              uj[q] = disp[jn[q]];
            }
            slots(k0 + U * SPLIT, true);
#pragma unroll
            for (int q = 0; q < U; ++q) {
              double d = g[q].x * (uj[q].x - ui.x) + g[q].y * (uj[q].y - ui.y);
              if (DIM == 3) d = fma(g[q].z, uj[q].z - ui.z, d);
              const int k = k0 + q * SPLIT;
              if (k < t.W) td[(int64_t)k << 5] = d;
              bool intact = (wd[q] >> t.lane) & 1u;
              const unsigned m = __ballot_sync(kFull, check && intact && pd_ge_threshold(d, g[q].w));
              if (m) {
                if ((m >> t.lane) & 1u) intact = false;
                if (t.lane == 0) bw[k] = wd[q] & ~m;
                sum[1] = 1.0;
              }
              part1[0][(h * U + q) % P] = fma(intact ? uj[q].w : 0.0, d, part1[0][(h * U + q) % P]);
            }
          }
        }
      }
      slots(t.sub, true);
      __syncwarp();
    }
    double th1[1];
    parts_sum<SPLIT, 1>(part1, th1);
    sum[0] = th1[0];
    parts_across<SPLIT, 2>(sum);
    double ti = 0.0;
    if (lead) {
      const double th = a.aA[i] * sum[0], mu = a.mu[i];
      ti = bp.Kp * (th * mu);
      a.thm[i].x = ti;
      if (step + 1 == r.nsteps) a.theta[i] = th;
      // The marks are consumed here alone: in the pair form every store to them and to the bits they stand for
      // lies before the barrier above, and without it only a check between calls sets them, before the launch.
      const bool marked = (PAIR || step == 0) && a.dirty[s] != 0;  // uniform over the warp
      if (marked || sum[1] != 0.0) {
        bond_sum_row<DIM>(a, t);
        __syncwarp();
        if (marked && t.lane == 0) a.dirty[s] = 0;
      }
    }
    if (!grid_barrier(a, r.grid, target)) return;
    // ---- pass 2
    double f[3], part[3][P] = {};
    if (t.active) {
      for (int kb = t.sub; kb < t.W; kb += H * U * SPLIT) {
#pragma unroll
        for (int h = 0; h < H; ++h) {
          const int k0 = kb + h * U * SPLIT;
          uint32_t wd[U];
          double4 g[U];
          double d[U], tj[U];
          slots(k0, false);
#pragma unroll
          for (int q = 0; q < U; ++q) {
            const int k = min(k0 + q * SPLIT, t.W - 1);
            wd[q] = k0 + q * SPLIT < t.W ? bw[k] : 0u;
            g[q] = slot_row<DIM>(a.bB, a.ne, e0 + ((int64_t)k << 5));
            d[q] = td[(int64_t)k << 5];
            tj[q] = a.thm[jn[q]].x;
          }
          if (kAhead > 0)
#pragma unroll
            for (int q = 0; q < U; ++q) {
              const int64_t k = (int64_t)min(k0 + (q + kAhead * U) * SPLIT, t.W - 1) << 5;
              to_l2(cl + k);
              to_l2(td + k);
              row_to_l2<DIM>(a.bB, a.ne, e0 + k);
            }
          slots(k0 + U * SPLIT, true);
#pragma unroll
          for (int q = 0; q < U; ++q) {
            double c = fma(g[q].w, d[q], tj[q]);
            c = ((wd[q] >> t.lane) & 1u) ? c : 0.0;
            const int n = (h * U + q) % P;
            part[0][n] = fma(c, g[q].x, part[0][n]);
            part[1][n] = fma(c, g[q].y, part[1][n]);
            if (DIM == 3) part[2][n] = fma(c, g[q].z, part[2][n]);
          }
        }
      }
    }
    if (!kKeep) load_state(disp);
    parts_sum<SPLIT, 3>(part, f);
    parts_across<SPLIT, 3>(f);
    if (lead) {
      const double4 S = a.bS[i];
      f[0] = fma(ti, S.x, f[0]);
      f[1] = fma(ti, S.y, f[1]);
      if (DIM == 3) f[2] = fma(ti, S.z, f[2]);
    }
    // ---- update (as update())
    if (lead) {
      if (fl == 0) {
        explicit_move<DIM>(bp, f, a.bacc ? &bb : nullptr, u, v);
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
      disp_out[i] = u;  // .w carries V_i unchanged
    }
    const bool last = step + 1 == r.nsteps;
    if (lead && (!kKeep || last)) a.vel[i] = v;
    if (last) break;
    slots(t.sub, true);
    if (!grid_barrier(a, r.grid, target)) return;
  }
  if (lead && (!isfinite(u.x) || !isfinite(u.y) || !isfinite(u.z))) atomicExch(&a.counters[5], 1ull);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *a.d_step = r.step0 + r.nsteps - 1;
  }
}

template <int DIM, int SPLIT, bool PAIR, int MAXT>
cudaError_t launch(pd_ctx* c, StepArgs a, ResidentArgs r, unsigned grid, int block) {
  void* args[] = {&a, &r};
  const size_t sm = SPLIT > 1 ? (size_t)block * 3 * sizeof(double) : 0;
  const void* k = (const void*)k_resident<DIM, SPLIT, PAIR, MAXT>;
  return cudaLaunchCooperativeKernel(k, dim3(grid), dim3((unsigned)block), args, sm, c->stream);
}

// (Only the forms that resident_plan names: four warps per slice up to 512 threads, two and one from 288 on, one in
// 2D only.)
template <int DIM, int SPLIT>
cudaError_t launch_form(pd_ctx* c, const StepArgs& a, const ResidentArgs& r, unsigned grid, int block, bool pair) {
  if (block > 512) {
    if constexpr (SPLIT < 4) return launch<DIM, SPLIT, true, 768>(c, a, r, grid, block);
    return cudaErrorInvalidConfiguration;
  }
  if (pair) return launch<DIM, SPLIT, true, 512>(c, a, r, grid, block);
  if constexpr (SPLIT == 4)
    if (block <= 256) return launch<DIM, SPLIT, false, 256>(c, a, r, grid, block);
  return launch<DIM, SPLIT, false, 512>(c, a, r, grid, block);
}

template <int DIM>
cudaError_t launch_split(pd_ctx* c, const StepArgs& a, const ResidentArgs& r, unsigned grid, int block, int split,
                         bool pair) {
  if (split == 4) return launch_form<DIM, 4>(c, a, r, grid, block, pair);
  if (split == 2) return launch_form<DIM, 2>(c, a, r, grid, block, pair);
  if constexpr (DIM == 2) return launch_form<DIM, 1>(c, a, r, grid, block, pair);
  return cudaErrorInvalidConfiguration;
}

}  // namespace

ResidentPlan resident_plan(const pd_ctx* c) {
  ResidentPlan p;
  if (!c->resident || !c->auto_map || c->precision != PD_FP64 || c->kin != PD_LINEARIZED || !c->bond_cache || !c->pairs || !c->pairs_ok ||
      c->solver != PD_SOLVER_EXPLICIT || c->profile || c->sms <= 0)
    return p;
  // Warps per slice: four while that leaves an SM at most 16 warps (128 registers each), two up to 20, in 2D
  // one up to 24 (80 registers beyond 16), but not where two warps per slice of the pass kernels fill just one wave
  // (tight_wave).  Elsewhere the pass kernels are the faster ones.  us per step, resident against pass kernels: plates
  // of 262^2 33.8 / 37.1, 278^2 (2,416 slices) 37.1 / 40.8, 279^2 (2,433) 50.0 / 40.2, 295^2 (2,720) 52.5 / 43.9, 297^2
  // 52.8 / 53.2, 340^2 59 / 65; blocks of 34^3 97 / 115, with one warp per slice 40^3 163 / 155.
  const int64_t ns = c->nslices, sms = c->sms;
  int split = 0;
  if (ns * 4 <= sms * 16) split = 4;
  else if (ns * 2 <= sms * 20) split = 2;
  else if (ns <= sms * 24 && c->dim == 2 && !tight_wave(c, 2)) split = 1;
  if (!split) return p;
  // One block per SM; a slice's warps share a block (parts_across).
  int64_t warps = (ns * split + sms - 1) / sms;
  warps = (warps + split - 1) / split * split;
  p.split = split;
  p.block = (int)warps * 32;
  p.grid = (unsigned)((ns * split + warps - 1) / warps);
  // The pair form has fewer FP64 instructions and one barrier more (us per step without / with it: plates of 140^2,
  // 536,000 bonds, 16.8 / 17.0, 160^2, 702,000, 19.2 / 18.7; blocks of 16^3, 394,000, 23.6 / 26.9, 18^3, 576,000,
  // 33.5 / 31.8, 24^3, 1.44M, 48.3 / 42.6).
  p.pair = c->nbonds > 600000;
  return p;
}

pd_status run_resident(pd_ctx* c, const StepArgs& a, const ResidentPlan& p, int64_t nsteps, bool check0, bool* done) {
  *done = false;
  if (const pd_status st = ensure_grid_bar(c); st != PD_OK) {
    if (st != PD_ERR_OOM) return st;
    clear_error();
    return PD_OK;  // no room for the barrier's words: the pass kernels take the steps
  }
  ResidentArgs r{};
  r.disp = c->disp[c->cur];
  r.disp_out = c->disp[c->cur ^ 1];
  r.nsteps = (int)nsteps;
  r.check0 = check0 ? 1 : 0;
  r.step0 = c->steps;
  r.grid = GridBar{c->bar, c->bar_base};
  r.uv = c->vol_uniform ? 1 : 0;
  const cudaError_t e = c->dim == 3 ? launch_split<3>(c, a, r, p.grid, p.block, p.split, p.pair)
                                    : launch_split<2>(c, a, r, p.grid, p.block, p.split, p.pair);
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
    cudaGetLastError();
    c->sms = 0;  // this device (or this share of it) cannot hold the grid: the pass kernels take the steps
    return PD_OK;
  }
  if (e != cudaSuccess) return cuda_fail(e, "cudaLaunchCooperativeKernel");
  const bool pair = p.pair || p.block > 512;
  const unsigned per_step = pair ? 3u : 2u;
  c->bar_base += p.grid * (per_step * (unsigned)nsteps - 1u);
  if (nsteps & 1) c->cur ^= 1;
  *done = true;
  return PD_OK;
}

}  // namespace pd
