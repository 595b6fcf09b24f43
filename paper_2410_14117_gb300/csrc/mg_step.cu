// Fleet step kernels: one thread per vehicle advancing Eq. 1 (§METHOD) by RK4 sub-steps with
// the state and parameters held in registers.
//
// Two schedules share the per-vehicle loop (advance_env):
//   k_fleet        static grid, one block per BlockDesc, k sub-steps per launch.  k = 1 is the
//                  plain per-step form (state and parameters through HBM every sub-step); k > 1
//                  is the persistent form (read once, stepped k times, written once).
//   k_fleet_queue  one launch for all k sub-steps: each warp repeatedly claims a unit (one
//                  32-env slice, one chunk of sub-steps) from an atomic counter in chunk-major
//                  order, waits until that slice's previous chunk is done, and runs it.  Warps
//                  that run faster claim more units, so the work spreads evenly over the 608
//                  schedulers whatever the fleet size (a static grid of 65,536 envs gives 3 or 4
//                  warps to each scheduler and idles the 3-warp ones for a quarter of the time).
//
// Blocks / slices cover envs of a single vehicle type, so the thruster geometry is a broadcast
// from shared memory and no warp diverges on the type.  Fleets whose types have different
// thruster counts run the 8-thruster loop for every env ("padded"): absent thrusters have zero
// direction and arm and zero command, so they add exact zeros.
#include <algorithm>
#include <type_traits>

#include "mg_advance.cuh"

namespace mg {

namespace {

constexpr int kMaxThreads = 256;

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_release(uint32_t *p, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// XH: off-diagonal hydrodynamics (general path), the block's coefficients staged in dynamic
// shared memory [blockDim.x][MG_NXPARAM].  WIDE (diagonal mass, no recording): 200 registers.
template <int NTV, bool DIAG, bool REC, int NH, bool XH = false, bool WIDE = false>
__global__ void __maxnreg__(XH ? kRegsXH : !DIAG ? kRegsGeneral : WIDE ? kRegsWide : kRegsDiag)
    k_fleet(const FleetView fv, const BlockDesc *__restrict__ blocks, const int32_t k,
            float *__restrict__ traj) {
  constexpr int MT = (NTV == NT_6) ? 6 : 8;
  constexpr bool MIXED = (NTV == NT_MIXED);
  __shared__ float4 sdir[MG_MAX_THR], sarm[MG_MAX_THR];
  __shared__ unsigned s_done;
  __shared__ int64_t s_cursor;
  __shared__ bool s_rewinding;
  extern __shared__ float sxh[];

  const BlockDesc bd = blocks[blockIdx.x];
  if (threadIdx.x < MG_MAX_THR) {
    sdir[threadIdx.x] = fv.geo[bd.type].dir[threadIdx.x];
    sarm[threadIdx.x] = fv.geo[bd.type].arm[threadIdx.x];
  }
  // Programmatic dependent launch: everything above reads only buffers written before any step
  // launch, and everything below waits for the previous launch in the stream to complete.
  cudaGridDependencySynchronize();
  if (threadIdx.x == 0) {
    s_done = 0u;
    bool rewinding;
    s_cursor = start_cursor(fv, rewinding);
    s_rewinding = rewinding;
  }
  if constexpr (XH) stage_xh(fv.xh, fv.n, bd.env0, bd.count, sxh);
  __syncthreads();
  if ((int)threadIdx.x >= bd.count) return;
  const int64_t e = (int64_t)bd.env0 + threadIdx.x;
  St<MT> st;
  const int nt = MIXED ? bd.n_thr : MT;
  const int64_t step0 = s_cursor + fv.cursor_off;
  advance_env<MT, DIAG, MIXED, REC, false, NH, XH, XH || (REC && MT > 6)>(
      fv, e, nt, sdir, sarm,
      [&](float (&c)[MT], int64_t &seg, int32_t &left) {
        scheduled_start<MT>(fv, e, nt, step0, c, seg, left);
      },
      k, traj, st, XH ? sxh + threadIdx.x * MG_NXPARAM : nullptr);
  // The next launch's blocks may be placed once every block of this one has come here (k = 1) or
  // ended.  Placed earlier they take the slots that happen to be free, two on one SM and none on
  // another, and the launch runs as long as its fullest SM: with the trigger before the sub-steps,
  // launches of 10 took 16.2 us for 30,000 envs instead of 10.6, and 9.5 instead of 7.4 for 15,000.
  // After them it is still too early where the last blocks run on (19,456 envs x 10: 9.8 instead
  // of 7.5), and only pays for one sub-step (65,536 envs in a graph: 3.8 us, without it 4.0).
  if (k == 1) cudaTriggerProgrammaticLaunchCompletion();
  store_and_flag<MT, false>(fv, e, st);
  if (fv.cursor_adv) finish_envs(fv, &s_done, bd.count, fv.cursor_adv, s_rewinding);
}

// XH (general path): each warp stages the off-diagonal hydrodynamic coefficients of the slice it
// claimed into its own rows of dynamic shared memory [kQueueWarps * 32][MG_NXPARAM] (every lane
// writes and reads only its own row, so program order suffices).
template <int NTV, bool DIAG, bool WIDE, int NH, bool XH = false>
__global__ void __maxnreg__(XH ? kRegsXH : !DIAG ? kRegsGeneral : WIDE ? kRegsWide : kRegsDiag)
    k_fleet_queue(const FleetView fv, const BlockDesc *__restrict__ slices, const int32_t n_slices,
                  const int32_t k_total, const int32_t chunk, uint32_t *__restrict__ sched) {
  static_assert(!(XH && DIAG), "the off-diagonal hydrodynamics use the general path");
  extern __shared__ float sxh[];
  constexpr int MT = (NTV == NT_6) ? 6 : 8;
  constexpr bool MIXED = (NTV == NT_MIXED);
  // Thruster geometry of every vehicle type at fixed shared addresses (a per-warp copy at a
  // run-time address costs the sub-step loop dozens of registers).
  __shared__ float4 sgeo[MG_MAX_TYPES][2 * MG_MAX_THR];
  for (int i = threadIdx.x; i < fv.n_types * 2 * MG_MAX_THR; i += blockDim.x) {
    const int t = i / (2 * MG_MAX_THR), j = i % (2 * MG_MAX_THR);
    sgeo[t][j] = j < MG_MAX_THR ? fv.geo[t].dir[j] : fv.geo[t].arm[j - MG_MAX_THR];
  }
  const int64_t step0 = launch_cursor(fv) + fv.cursor_off;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const uint32_t n_chunks = (uint32_t)((k_total + chunk - 1) / chunk);
  const uint32_t n_units = (uint32_t)n_slices * n_chunks;  // < 2^31, checked by the launcher

  for (;;) {
    uint32_t u = 0;
    if (lane == 0) u = atomicAdd(sched, 1u);
    u = __shfl_sync(0xffffffffu, u, 0);
    if (u >= n_units) break;
    const int32_t c = (int32_t)(u / (uint32_t)n_slices);
    const int32_t d = (int32_t)(u % (uint32_t)n_slices);
    if (c > 0 && lane == 0) {
      // The slice's previous chunk was claimed earlier by a running warp, so it completes.  The
      // wait is bounded (fv.spin_limit polls of ~128 ns, MG_WAIT_POLLS_DEFAULT unless set by
      // mg_set_wait_limit): on expiry it is counted as a time-out and the unit proceeds.
      uint32_t polls = 0;
      while (ld_acquire(sched + 4 + d) < (uint32_t)c) {
        if (++polls > fv.spin_limit) {
          atomicAdd(fv.counters + 2, 1ull);
          break;
        }
        __nanosleep(128);
      }
    }
    __syncwarp();
    const BlockDesc bd = slices[d];
    const float4 *gdir = sgeo[bd.type & (MG_MAX_TYPES - 1)], *garm = gdir + MG_MAX_THR;
    if (lane < bd.count) {
      const int64_t e = (int64_t)bd.env0 + lane;
      float *row = sxh + threadIdx.x * MG_NXPARAM;
      if constexpr (XH)
        for (int j = 0; j < MG_NXPARAM; ++j) row[j] = __ldg(fv.xh + (int64_t)j * fv.n + e);
      St<MT> st;
      const int nt = MIXED ? bd.n_thr : MT;
      advance_env<MT, DIAG, MIXED, false, true, NH, XH, XH>(
          fv, e, nt, gdir, garm,
          [&](float (&cmd)[MT], int64_t &seg, int32_t &left) {
            scheduled_start<MT>(fv, e, nt, step0 + (int64_t)c * chunk, cmd, seg, left);
          },
          min(chunk, k_total - c * chunk), nullptr, st, XH ? row : nullptr);
      store_and_flag<MT, true>(fv, e, st);
    }
    __syncwarp();
    if (lane == 0) {
      __threadfence();
      st_release(sched + 4 + d, (uint32_t)(c + 1));
    }
  }
  if (fv.cursor_adv) finish_launch(fv, fv.cursor_adv);
}

// Launch a static-grid step kernel with programmatic stream serialisation: it may begin while
// the previous kernel in the stream finishes (see the wait in k_fleet).
template <typename Kernel>
cudaError_t launch_pdl(Kernel kernel, int n_blocks, int threads, size_t smem, cudaStream_t stream,
                       const FleetView &fv, const BlockDesc *blocks, int32_t k, float *traj) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)n_blocks);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, fv, blocks, k, traj);
}

// The vectored allocation is only instantiated for the diagonal-mass step, the off-diagonal
// hydrodynamics (XH) only for the general one, the wide register budget only for the diagonal-mass
// step without recording.
template <int NTV, bool DIAG, bool REC, bool WIDE>
cudaError_t launch_t(const FleetView &fv, const BlockDesc *blocks, int n_blocks, int threads,
                     int layout, int32_t k, float *traj, cudaStream_t stream) {
  return with_layout<DIAG>(layout, [&](auto l) {
    constexpr int L = decltype(l)::value;
    if constexpr (!DIAG)
      if (fv.xh)
        return launch_pdl(k_fleet<NTV, false, REC, L, true>, n_blocks, threads,
                          sizeof(float) * MG_NXPARAM * threads, stream, fv, blocks, k, traj);
    constexpr bool W = WIDE && !(mirrored_sums(L) && NTV == NT_6);  // wide_kernel
    return launch_pdl(k_fleet<NTV, DIAG, REC, L, false, W>, n_blocks, threads, 0, stream, fv,
                      blocks, k, traj);
  });
}

// Whether the static grid takes the 200-register kernel.  The mirrored allocation fits 128
// registers without spilling, which puts four 128-thread blocks on an SM against three: 65,536 envs
// x 200 in 288 us against 373, 1,048,576 x 50 in 937 against 966; six thrusters gain nothing by
// more registers at any size (1,000 envs x 200: 90 us both, 50,000: 223 against 233).  Eight, and
// mixed fleets, do while all blocks are resident at once (1,000 envs: 95 against 102 us; 50,000:
// 241 against 246).  The other allocations spill at 128.
template <int NTV>
bool wide_kernel(bool wide, int layout, int n_blocks, int threads) {
  if (!wide || !mirrored_sums(layout)) return wide;
  int dev = 0, n_sm = 0;
  return NTV != NT_6 && cudaGetDevice(&dev) == cudaSuccess &&
         cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
         n_blocks <= n_sm * (12 / (threads / 32));
}

template <int NTV, bool DIAG>
cudaError_t launch_r(const FleetView &fv, const BlockDesc *blocks, int n_blocks, int threads,
                     int layout, bool wide, int32_t k, float *traj, cudaStream_t stream) {
  if (traj)
    return launch_t<NTV, DIAG, true, false>(fv, blocks, n_blocks, threads, layout, k, traj,
                                            stream);
  if constexpr (DIAG)
    if (wide_kernel<NTV>(wide, layout, n_blocks, threads))
      return launch_t<NTV, true, false, true>(fv, blocks, n_blocks, threads, layout, k,
                                              traj, stream);
  return launch_t<NTV, DIAG, false, false>(fv, blocks, n_blocks, threads, layout, k, traj,
                                           stream);
}

template <int NTV>
cudaError_t launch_d(const FleetView &fv, const BlockDesc *blocks, int n_blocks, int threads,
                     bool diag, int layout, bool wide, int32_t k, float *traj,
                     cudaStream_t stream) {
  return diag ? launch_r<NTV, true>(fv, blocks, n_blocks, threads, layout, wide, k, traj,
                                    stream)
              : launch_r<NTV, false>(fv, blocks, n_blocks, threads, layout, wide, k, traj,
                                     stream);
}

template <int NTV, bool DIAG, bool REC, bool WIDE = false>
const void *kernel_ptr(int layout) {
  return with_layout<DIAG>(layout, [](auto l) {
    constexpr int L = decltype(l)::value;
    return reinterpret_cast<const void *>(
        &k_fleet<NTV, DIAG, REC, L, false, WIDE && !(mirrored_sums(L) && NTV == NT_6)>);
  });
}

template <int NTV, bool DIAG>
const void *queue_ptr(bool wide, int layout, bool xh) {
  return with_layout<DIAG>(layout, [&](auto l) {
    constexpr int L = decltype(l)::value;
    if constexpr (!DIAG)
      if (xh) return reinterpret_cast<const void *>(&k_fleet_queue<NTV, false, false, L, true>);
    return wide ? reinterpret_cast<const void *>(&k_fleet_queue<NTV, DIAG, true, L>)
                : reinterpret_cast<const void *>(&k_fleet_queue<NTV, DIAG, false, L>);
  });
}

const void *queue_kernel(NtVariant ntv, bool diag, bool wide, int layout, bool xh) {
  switch (ntv) {
    case NT_6:
      return diag ? queue_ptr<NT_6, true>(wide, layout, false)
                  : queue_ptr<NT_6, false>(wide, layout, xh);
    case NT_8:
      return diag ? queue_ptr<NT_8, true>(wide, layout, false)
                  : queue_ptr<NT_8, false>(wide, layout, xh);
    default:
      return diag ? queue_ptr<NT_MIXED, true>(wide, layout, false)
                  : queue_ptr<NT_MIXED, false>(wide, layout, xh);
  }
}

// Dynamic shared memory of the XH work-queue kernel (one coefficient row per thread).
constexpr size_t kQueueXhBytes = sizeof(float) * kQueueWarps * 32 * MG_NXPARAM;

template <int NTV, bool DIAG, int NH>
void queue_launch_w(bool wide, int grid, size_t smem, const FleetView &fv, const BlockDesc *slices,
                    int32_t n_slices, int32_t k, int32_t chunk, uint32_t *sched,
                    cudaStream_t stream) {
  if constexpr (!DIAG)
    if (fv.xh) {
      k_fleet_queue<NTV, false, false, NH, true><<<grid, kQueueWarps * 32, smem, stream>>>(
          fv, slices, n_slices, k, chunk, sched);
      return;
    }
  if (wide)
    k_fleet_queue<NTV, DIAG, true, NH><<<grid, kQueueWarps * 32, smem, stream>>>(
        fv, slices, n_slices, k, chunk, sched);
  else
    k_fleet_queue<NTV, DIAG, false, NH><<<grid, kQueueWarps * 32, smem, stream>>>(
        fv, slices, n_slices, k, chunk, sched);
}

// Dynamic shared memory (at least `need`) that lets per_sm blocks of kernel f onto an SM and no
// more: the warps_per_sm cap would otherwise only size the grid, and where more blocks fit, a
// kernel on another stream (the background draw of mg_randomize_prefetch) makes the hardware
// place three of them on some SMs and one on others.  65,536 six-thruster envs x 1,000 sub-steps
// with the next episode's draw beside them, 8 warps per SM: 1,840 us without, 1,510 with
// (1,400 for the steps alone).
cudaError_t queue_even_smem(const void *f, const cudaFuncAttributes &attr, int per_sm,
                            size_t need, size_t *smem) {
  *smem = need;
  int dev = 0, per_sm_bytes = 0, per_block = 0, reserved = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&per_sm_bytes, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&per_block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
  if (e != cudaSuccess) return e;
  const size_t fixed = attr.sharedSizeBytes + (size_t)reserved;
  // a block's share when per_sm + 1 of them would just not fit
  const size_t share = (size_t)per_sm_bytes / (per_sm + 1) + 1024;
  if (share < fixed + need || share * per_sm > (size_t)per_sm_bytes ||
      share - reserved > (size_t)per_block)
    return cudaSuccess;
  *smem = share - fixed;
  // the same limit whatever the cap: it belongs to the function, which other sims launch too
  return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              per_block - (int)attr.sharedSizeBytes);
}

template <int NTV>
void queue_launch(bool diag, bool wide, int layout, int grid, size_t smem, const FleetView &fv,
                  const BlockDesc *slices, int32_t n_slices, int32_t k, int32_t chunk,
                  uint32_t *sched, cudaStream_t stream) {
  if (diag)
    with_layout<true>(layout, [&](auto l) {
      queue_launch_w<NTV, true, decltype(l)::value>(wide, grid, smem, fv, slices, n_slices, k,
                                                    chunk, sched, stream);
    });
  else
    with_layout<false>(layout, [&](auto l) {
      queue_launch_w<NTV, false, decltype(l)::value>(wide, grid, smem, fv, slices, n_slices, k,
                                                     chunk, sched, stream);
    });
}

}  // namespace

cudaError_t launch_fleet(const FleetView &fv, const BlockDesc *blocks, int n_blocks, int threads,
                         NtVariant ntv, bool diag, int layout, bool wide, int32_t k,
                         float *traj, cudaStream_t stream) {
  if (threads < 32 || threads > kMaxThreads || threads % 32 || n_blocks < 1 || k < 1 ||
      (fv.xh && diag))
    return cudaErrorInvalidValue;
  switch (ntv) {
    case NT_6:
      return launch_d<NT_6>(fv, blocks, n_blocks, threads, diag, layout, wide, k, traj,
                            stream);
    case NT_8:
      return launch_d<NT_8>(fv, blocks, n_blocks, threads, diag, layout, wide, k, traj,
                            stream);
    default:
      return launch_d<NT_MIXED>(fv, blocks, n_blocks, threads, diag, layout, wide, k, traj,
                                stream);
  }
}

cudaError_t fleet_kernel_attributes(NtVariant ntv, bool diag, int layout, bool rec, bool wide,
                                    int n_blocks, int threads, cudaFuncAttributes *attr) {
  const void *f = nullptr;
#define MG_PICK(N)                                                                      \
  f = diag ? (rec ? kernel_ptr<N, true, true>(layout)                               \
                  : wide_kernel<N>(wide, layout, n_blocks, threads)                     \
                      ? kernel_ptr<N, true, false, true>(layout)                        \
                      : kernel_ptr<N, true, false>(layout))                             \
           : (rec ? kernel_ptr<N, false, true>(layout) : kernel_ptr<N, false, false>(layout));
  switch (ntv) {
    case NT_6: MG_PICK(NT_6) break;
    case NT_8: MG_PICK(NT_8) break;
    default: MG_PICK(NT_MIXED) break;
  }
#undef MG_PICK
  return cudaFuncGetAttributes(attr, f);
}

size_t queue_sched_bytes(int n_slices) { return 16 + 4 * (size_t)n_slices; }

cudaError_t queue_kernel_attributes(NtVariant ntv, bool diag, bool wide, int layout,
                                    bool xh, cudaFuncAttributes *attr, int *blocks_per_sm) {
  xh = xh && !diag;
  const void *f = queue_kernel(ntv, diag, wide, layout, xh);
  cudaError_t e = cudaFuncGetAttributes(attr, f);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, f, kQueueWarps * 32,
                                                       xh ? kQueueXhBytes : 0);
}

cudaError_t launch_fleet_queue(const FleetView &fv, const BlockDesc *slices, int n_slices,
                               NtVariant ntv, bool diag, int layout, bool wide,
                               int warps_per_sm, int32_t k, int32_t chunk, uint32_t *sched,
                               int n_sm, cudaStream_t stream) {
  if (n_slices < 1 || k < 1 || chunk < 1 || n_sm < 1 || (fv.xh && diag))
    return cudaErrorInvalidValue;
  cudaFuncAttributes attr;
  int per_sm = 0;
  cudaError_t e = queue_kernel_attributes(ntv, diag, wide, layout, fv.xh != nullptr, &attr,
                                          &per_sm);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  // Resident warps: at most what fits (and at most warps_per_sm per SM when that is > 0), and no
  // more than there are slices in a chunk.
  size_t smem = fv.xh ? kQueueXhBytes : 0;
  const int cap = std::max(1, warps_per_sm / kQueueWarps);
  if (warps_per_sm > 0 && cap < per_sm) {
    per_sm = cap;
    e = queue_even_smem(queue_kernel(ntv, diag, wide, layout, fv.xh != nullptr), attr, per_sm, smem,
                        &smem);
    if (e != cudaSuccess) return e;
  }
  int grid = per_sm * n_sm;
  const int need = (n_slices + kQueueWarps - 1) / kQueueWarps;
  if (grid > need) grid = need;
  // One launch per piece of the horizon whose unit count fits the 31-bit counter.
  const int64_t max_chunks = ((int64_t)1 << 31) / n_slices;
  if (max_chunks < 1) return cudaErrorInvalidValue;
  for (int64_t done = 0; done < k;) {
    const int64_t left = k - done;
    const int32_t kk = (int32_t)std::min<int64_t>(left, max_chunks * (int64_t)chunk);
    e = cudaMemsetAsync(sched, 0, queue_sched_bytes(n_slices), stream);
    if (e != cudaSuccess) return e;
    FleetView piece = fv;  // this piece's offset in the call; only the last piece advances
    piece.cursor_off = fv.cursor_off + (int32_t)done;
    piece.cursor_adv = (done + kk == k) ? fv.cursor_adv : 0;
    switch (ntv) {
      case NT_6:
        queue_launch<NT_6>(diag, wide, layout, grid, smem, piece, slices, n_slices, kk, chunk,
                           sched, stream);
        break;
      case NT_8:
        queue_launch<NT_8>(diag, wide, layout, grid, smem, piece, slices, n_slices, kk, chunk,
                           sched, stream);
        break;
      default:
        queue_launch<NT_MIXED>(diag, wide, layout, grid, smem, piece, slices, n_slices, kk, chunk,
                               sched, stream);
        break;
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    done += kk;
  }
  return cudaSuccess;
}

}  // namespace mg
