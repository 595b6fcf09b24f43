// Per-env step loop shared by the step kernels (mg_step.cu) and the fused task step
// (mg_task.cu): commands from the action cursor, k RK4 sub-steps in registers, optional
// trajectory record, and the launch-completion count that advances the device-side cursor.
#pragma once

#include "mg_device.cuh"

namespace mg {

// Register caps: the narrow diagonal-mass step keeps 128 registers (16 resident warps per SM, for
// the per-step form and large per-step grids; no spills with the mirrored allocation, 70-440 bytes
// with the others); the general step keeps 168.
constexpr int kRegsDiag = 128;
constexpr int kRegsGeneral = 168;
// The wide diagonal-mass variants (mg_set_schedule's wide): the work-queue kernel runs at 8
// warps/SM, where 256 registers per thread would fit; with the mirrored allocation ptxas uses
// 164-168 (65,536 envs x 1,000 sub-steps: 1.29 ms; the static grid at 128 registers 1.38 ms).  The
// static grid takes it where that pays (wide_kernel in mg_step.cu).
constexpr int kRegsWide = 200;
// With the off-diagonal hydrodynamics the 45 extra coefficients stay in registers too (no
// spills up to 255; 8 resident warps per SM).
constexpr int kRegsXH = 255;

// Action cursor at the start of the launch's mg_step call (read through L2: the previous call's
// last block wrote it).
__device__ __forceinline__ int64_t launch_cursor(const FleetView &fv) {
  return (int64_t)__ldcg(reinterpret_cast<const unsigned long long *>(fv.cursor));
}

// Called by every thread of every block once it is done: the last block to finish advances the
// cursor by k and re-arms the counter.  Every block read the cursor before it counted itself
// finished, so all of them saw the launch's starting value.
__device__ __forceinline__ void finish_launch(const FleetView &fv, int32_t k) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned prev = atomicAdd(fv.done_blocks, 1u);
    if (prev == gridDim.x - 1) {
      atomicAdd(reinterpret_cast<unsigned long long *>(fv.cursor), (unsigned long long)k);
      atomicExch(fv.done_blocks, 0u);
      __threadfence();
    }
  }
}

// f(std::integral_constant<int, L>()) for the allocation `layout`: those the diagonal-mass kernels
// are compiled for, or the general ones (dense, mirrored).
template <bool DIAG, typename F>
auto with_layout(int layout, F f) {
  if (layout == MG_LAYOUT_MIRRORED) return f(std::integral_constant<int, MG_LAYOUT_MIRRORED>());
  if constexpr (DIAG) {
    if (layout == MG_LAYOUT_MIRRORED_G)
      return f(std::integral_constant<int, MG_LAYOUT_MIRRORED_G>());
    if (layout == MG_LAYOUT_VECTORED) return f(std::integral_constant<int, MG_LAYOUT_VECTORED>());
  }
  return f(std::integral_constant<int, MG_LAYOUT_DENSE>());
}

// The cursor a static-grid step launch starts at: 0 when the launch carries a rewind that the
// device has not seen (rewinding is then true), else the device's word.
__device__ __forceinline__ int64_t start_cursor(const FleetView &fv, bool &rewinding) {
  rewinding = fv.rewind && __ldcg(fv.rewind_gen) != fv.rewind;
  return rewinding ? 0 : launch_cursor(fv);
}

// Static-grid form of finish_launch, for kernels whose idle threads have already returned (no
// block barrier possible): each warp adds its live lanes to the block's shared counter s_done
// (zeroed before the block's first barrier); the warp that completes the block's count of live
// envs adds one finished block to the grid's counter, and the block that completes the grid
// advances the cursor by k and re-arms the counter.  Every thread read the cursor before its
// warp counted itself, so every block saw the launch's starting value.
__device__ __forceinline__ void finish_envs(const FleetView &fv, unsigned *s_done, int count,
                                            int32_t k, bool rewinding = false) {
  const unsigned mask = __activemask();
  __syncwarp(mask);
  if ((threadIdx.x & 31) == (unsigned)(__ffs(mask) - 1)) {
    const unsigned add = __popc(mask);
    if (atomicAdd(s_done, add) + add == (unsigned)count &&
        atomicAdd(fv.done_blocks, 1u) == gridDim.x - 1) {
      unsigned long long *cursor = reinterpret_cast<unsigned long long *>(fv.cursor);
      if (rewinding) {
        atomicExch(cursor, (unsigned long long)k);
        atomicExch(fv.rewind_gen, fv.rewind);
      } else {
        atomicAdd(cursor, (unsigned long long)k);
      }
      atomicExch(fv.done_blocks, 0u);
    }
  }
}

// The task kernel's form, called by one thread of every block after its dependency wait: the cursor
// the launch starts at, which that thread alone reads for its block.  The block is counted at once,
// by an increment that depends on the value read, so the last block to begin knows that all have
// read the cursor and advances it (the next launch looks after this one's end).  In a kernel of a
// few sub-steps the count's round trip at the end stands between the last sub-step and the next
// launch: 1,000-env environment steps 5.60 us with it there, 5.39 here, 65,536-env mixed ones 22.2
// and 21.9.  The step kernels keep theirs at the end: their loops come out slower with this one
// (1,048,576 envs x 50 on the static grid 937 against 957 us).
// use_cursor = false: the launch only counts (it has its own command).
__device__ __forceinline__ int64_t begin_launch(const FleetView &fv, bool use_cursor) {
  const int64_t at = use_cursor ? launch_cursor(fv) : 0;
  if (fv.cursor_adv) {
    const unsigned one = at < 0 ? 2u : 1u;  // 1: the cursor is never negative
    if (atomicAdd(fv.done_blocks, one) == gridDim.x - 1) {
      atomicAdd(reinterpret_cast<unsigned long long *>(fv.cursor),
                (unsigned long long)fv.cursor_adv);
      atomicExch(fv.done_blocks, 0u);
    }
  }
  return at;
}

// Stage a block's off-diagonal hydrodynamic coefficients in shared memory: row t of sx (stride
// MG_NXPARAM, coprime with the 32 banks) receives env env0 + t's coefficients from the
// component-major planes xh [MG_NXPARAM][n] (each component read coalesced).
__device__ __forceinline__ void stage_xh(const float *__restrict__ xh, int64_t n, int64_t env0,
                                         int count, float *sx) {
  for (int c = 0; c < MG_NXPARAM; ++c)
    for (int t = threadIdx.x; t < count; t += blockDim.x)
      sx[t * MG_NXPARAM + c] = __ldg(xh + (int64_t)c * n + env0 + t);
}

template <int MT>
__device__ __forceinline__ void load_commands(const FleetView &fv, int64_t e, int64_t seg,
                                              int nt, float (&c)[MT]) {
  if (fv.proc) {
    procedural_commands<MT>(fv.cmd_seed, (uint64_t)(fv.gid0 + e), seg, c);
  } else if (fv.n_seg > 0) {
    const int64_t sg = seg < fv.n_seg - 1 ? seg : fv.n_seg - 1;
    if (MT == 6 && fv.act_w == 6) {
      // 24-byte rows (no padding): three 8-byte loads; a warp's rows are 768 contiguous bytes
      const float2 *a = reinterpret_cast<const float2 *>(fv.act + (sg * fv.n + e) * 6);
      const float2 x = __ldg(a), y = __ldg(a + 1), z = __ldg(a + 2);
      c[0] = x.x; c[1] = x.y; c[2] = y.x; c[3] = y.y; c[4] = z.x; c[5] = z.y;
    } else {
      const float4 *a = reinterpret_cast<const float4 *>(fv.act + (sg * fv.n + e) * MG_MAX_THR);
      const float4 lo = __ldg(a), hi = __ldg(a + 1);
      c[0] = lo.x; c[1] = lo.y; c[2] = lo.z; c[3] = lo.w; c[4] = hi.x; c[5] = hi.y;
      if constexpr (MT > 6) {
        c[6] = hi.z;
        c[7] = hi.w;
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < MT; ++i) c[i] = 0.f;
  }
  // Entries past the vehicle's thruster count are ignored (the lag state there stays zero).
#pragma unroll
  for (int i = 0; i < MT; ++i) c[i] = (i < nt) ? c[i] : 0.f;
}

// Lag entries past a six-thruster vehicle's thrusters in a mixed fleet's eight-entry loop, as zero:
// the mirrored sums add the forces of all eight (the other allocations multiply each by its own
// direction, which is zero there), and a caller's state may hold anything in them.
template <int MT, bool MIXED, int NH>
__device__ __forceinline__ void drop_unused_lag(St<MT> &s, int nt) {
  if constexpr (MIXED && MT > 6 && mirrored_sums(NH)) {
#pragma unroll
    for (int i = 6; i < MT; ++i) s.n[i] = i < nt ? s.n[i] : 0.f;
  }
}

__device__ __forceinline__ void prefetch_l1(const void *p) {
  asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}

// Start moving the env's row of the command segment after seg into the L1, for kernels that record
// a trajectory: their stores keep the memory pipe busy and a segment's first load waits behind
// them (30,000 recorded 8-thruster envs x 200 sub-steps 264 -> 253 us).  Without recording the load
// is already hidden (1,024 envs x 500: 225 us either way) or the instruction costs more than it
// saves (65,536 on the work queue 1,333 -> 1,350 us).
__device__ __forceinline__ void prefetch_commands(const FleetView &fv, int64_t e, int64_t seg) {
  if (seg + 1 < fv.n_seg) prefetch_l1(fv.act + ((seg + 1) * fv.n + e) * fv.act_w);
}

template <int MT>
__device__ __forceinline__ void record(float *__restrict__ traj, int64_t n, int64_t e,
                                       const St<MT> &s) {
  float *t = traj + e;
  t[0 * n] = s.p[0]; t[1 * n] = s.p[1]; t[2 * n] = s.p[2];
  t[3 * n] = s.q[0]; t[4 * n] = s.q[1]; t[5 * n] = s.q[2]; t[6 * n] = s.q[3];
  t[7 * n] = s.v[0]; t[8 * n] = s.v[1]; t[9 * n] = s.v[2];
  t[10 * n] = s.w[0]; t[11 * n] = s.w[1]; t[12 * n] = s.w[2];
}

template <int MT>
__device__ __forceinline__ bool all_finite(const St<MT> &s) {
  // x * 0 is 0 for finite x and NaN for +-Inf or NaN, so the sum is 0 exactly when all are
  // finite.
  float z = 0.f;
#pragma unroll
  for (int i = 0; i < 3; ++i) z += s.p[i] * 0.f + s.v[i] * 0.f + s.w[i] * 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) z += s.q[i] * 0.f;
#pragma unroll
  for (int i = 0; i < MT; ++i) z += s.n[i] * 0.f;
  return z == 0.f;
}

// The command of the sub-step at action-cursor position step0: sub-step j uses segment j / hold
// (clamped to the last buffered segment).
template <int MT>
__device__ __forceinline__ void scheduled_start(const FleetView &fv, int64_t e, int nt,
                                                int64_t step0, float (&c)[MT], int64_t &seg,
                                                int32_t &left) {
  seg = step0 / fv.hold;
  left = fv.hold - (int32_t)(step0 - seg * fv.hold);
  load_commands<MT>(fv, e, seg, nt, c);
}

// Advance env e by k sub-steps, leaving the result in
// s (the caller stores it: store_and_flag, or a fused epilogue).  L2: state loads bypass L1
// (work-queue schedule, where another SM may have written them).
// XH: xh is the env's row of staged off-diagonal hydrodynamic coefficients.
// start(c, seg, left) sets the first sub-step's command c, its segment and the sub-steps left in it
// (scheduled_start, or a fused kernel's own source).
// loaded: the parameters, where the caller has loaded them and the state s already (the task
// kernel, before its block barrier; the step kernels' loops come out 2 % slower that way). PACK:
// packed stage updates (see axpy).
template <int MT, bool DIAG, bool MIXED, bool REC, bool L2, int NH, bool XH, bool PACK,
          bool LOADED = false, typename Start = void>
__device__ __forceinline__ void advance_env(const FleetView &fv, int64_t e, int nt,
                                            const float4 *gdir, const float4 *garm, Start start,
                                            int32_t k, float *traj, St<MT> &s, const float *xh,
                                            const Par<DIAG> *loaded = nullptr) {
  const bool current_accel = !(fv.model_flags & MG_MODEL_NO_CURRENT_ACCEL);

  if constexpr (!LOADED) load_state<MT, L2>(fv.st, e, s);
  drop_unused_lag<MT, MIXED, NH>(s, nt);
  float c[MT];
  int64_t seg;
  int32_t left;
  // The command's address depends on the action cursor and starts its load before the parameters'
  // 34 floats arrive; the work queue, whose warps overlap one another's loads, runs faster the
  // other way round (registers: 65,536 envs x 1,000 sub-steps 1.29 against 1.35 ms; the static grid
  // 1.39 against 1.44 ms in this order), and so do mixed fleets on the static grid (262,144 x 500
  // 2.65 against 2.67 ms).
  if constexpr (!L2 && !MIXED) start(c, seg, left);
  Coef<DIAG, NH> P;
  {
    Par<DIAG> raw;
    if constexpr (LOADED) raw = *loaded;
    else load_par<DIAG>(fv.pa, e, raw);
    P = make_coef<DIAG, NH>(raw, gdir, garm);
  }
  const LagEnv L = lag_env(P.itau, fv.dt);
  if constexpr (L2 || MIXED) start(c, seg, left);
  if constexpr (REC)
    if (left < k) prefetch_commands(fv, e, seg);

  for (int32_t it = 0; it < k; ++it) {
    if (left == 0) {
      ++seg;
      left = fv.hold;
      load_commands<MT>(fv, e, seg, nt, c);
      if constexpr (REC)
        if (left < k - it) prefetch_commands(fv, e, seg);
    }
    if constexpr (PACK)
      rk4_step<MT, DIAG, MIXED, NH, XH>(s, c, L, P, gdir, garm, nt, current_accel, fv.rk2, xh);
    else
      rk4_step<MT, DIAG, MIXED, NH, XH>(s, c, L, P, gdir, garm, nt, current_accel, fv.rk, xh);
    --left;
    if constexpr (REC) record<MT>(traj + (int64_t)it * MG_NTRAJ * fv.n, fv.n, e, s);
  }
}

// Mark env e non-finite (flag bit 0, counted once) unless already marked.  L2: the flag is read
// through L2 (work-queue schedule).
template <bool L2>
__device__ __forceinline__ void flag_nonfinite(const FleetView &fv, int64_t e) {
  const uint32_t old = L2 ? __ldcg(fv.flags + e) : fv.flags[e];
  if (!(old & 1u)) {
    fv.flags[e] = old | 1u;
    atomicAdd(fv.counters, 1ull);
  }
}

template <int MT, bool L2>
__device__ __forceinline__ void store_and_flag(const FleetView &fv, int64_t e, const St<MT> &s) {
  store_state<MT>(fv.st, e, s);
  if (!all_finite<MT>(s)) flag_nonfinite<L2>(fv, e);
}

}  // namespace mg
