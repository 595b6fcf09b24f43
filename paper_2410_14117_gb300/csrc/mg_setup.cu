// Set-up kernels, run when parameters or episodes change (not per sub-step):
//   - domain randomisation (§METHOD) from Philox4x32-10 draws, the values FP64 arithmetic stores,
//     formed in two-float arithmetic (mg_df32.cuh) where that decides their rounding to FP32;
//   - derivation of what the step reads, including M^-1 of the 6x6 mass matrix M_RB + M_A of
//     Eq. 1: its reciprocals where it is diagonal, else by an FP64 Cholesky factorisation (M is
//     symmetric positive definite for any physical vehicle; a non-positive pivot is counted and
//     reported);
//   - episode reset, and conversions between the SoA planes and the record layouts of mg.h.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "mg_device.cuh"
#include "mg_df32.cuh"

namespace mg {

namespace {

constexpr int kThreads = 256;

inline int blocks_for(int64_t n) { return (int)((n + kThreads - 1) / kThreads); }

// Index of the j-th of the 27 randomised scalars in the parameter record, in draw order: m,
// I_g (3), M_A (6), D_l (6), D_q (6), W, B (record entries 0..23 in order), then r_b,z, k_T,
// tau_m.  A compile-time function, so that the unrolled draw loop addresses the record in
// registers.
static_assert(MG_P_M == 0 && MG_P_IG == 1 && MG_P_MA == 4 && MG_P_DL == 10 && MG_P_DQ == 16 &&
                  MG_P_W == 22 && MG_P_B == 23 && MG_P_TAU == MG_P_KT + 1,
              "randomised-scalar order assumes the record layout of mg.h");
__host__ __device__ constexpr int rand_idx(int j) {
  return j < 24 ? j : j == 24 ? MG_P_RB + 2 : j == 25 ? MG_P_KT : MG_P_TAU;
}
// Block size of the randomisation kernel and of the record copies.
constexpr int kRandThreads = 128;
// Background form: 64-thread blocks (two warps, 4.6 K registers) striding over the fleet, which fit
// beside the work queue's resident blocks on every SM.
constexpr int kRandBgThreads = 64;

__device__ __forceinline__ bool aligned16(const void *p) {
  return (reinterpret_cast<uintptr_t>(p) & 15u) == 0;
}

// Copy count floats, all threads of the block taking part; 16-byte vectors when both ends allow.
__device__ __forceinline__ void block_copy(float *dst, const float *src, int count) {
  int done = 0;
  if (aligned16(dst) && aligned16(src)) {
    done = count & ~3;
    for (int i = threadIdx.x; i < done / 4; i += blockDim.x)
      reinterpret_cast<float4 *>(dst)[i] = reinterpret_cast<const float4 *>(src)[i];
  }
  for (int i = done + threadIdx.x; i < count; i += blockDim.x) dst[i] = src[i];
}

// Tell the host of an r_b off the body's z axis (the mirrored thruster allocation needs it on it).
__device__ __forceinline__ void note_off_axis(const SetupView &v, const float *p) {
  if (p[MG_P_RB] != 0.f || p[MG_P_RB + 1] != 0.f) atomicOr(v.any_offdiag, 2u);
}

// M^-1 of a diagonal mass matrix in FP64, for the few envs with a reciprocal whose rounding df_rcp
// leaves open.
__device__ __noinline__ void invert_diag_fp64(const ParamPlanes &pa, int64_t e, float m, float Ix,
                                              float Iy, float Iz, float a0, float a1, float a2,
                                              float a3, float a4, float a5) {
  auto inv = [](float a, float b) {
    const double M = (double)a + (double)b;
    return M > 0.0 ? (float)(1.0 / M) : 0.f;
  };
  pa.d7[e] = make_float4(inv(m, a0), inv(m, a1), inv(m, a2), inv(Ix, a3));
  pa.d8[e] = make_float2(inv(Iy, a4), inv(Iz, a5));
}

// The step's parameter planes of an env whose mass matrix is diagonal (r_g = 0, no off-diagonal
// added mass) from its record p[MG_NPARAM]: I_o = I_g exactly, M^-1 = diag(1 / M_jj) and every
// off-diagonal entry is +0.  Each stored value is the FP64 expression's, rounded once: a sum,
// difference or product of two FP32 numbers is one FP32 operation, and 1 / (a + b) is formed in two
// floats, or in FP64 where those leave its rounding open.
__device__ __forceinline__ void derive_diag(const SetupView &v, int64_t e, const float *p) {
  const float m = p[MG_P_M];
  const float *ma = p + MG_P_MA, *rg = p + MG_P_RG, *rb = p + MG_P_RB;
  float J[3], mi[6];
  bool spd = true, open = false;
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    const df32 M = two_sum(j < 3 ? m : p[MG_P_IG + j - 3], ma[j]);
    if (j >= 3) J[j - 3] = M.h;
    if (!(M.h > 0.f)) spd = false;
    bool o;
    const float r = df_rcp(M, o);
    mi[j] = M.h > 0.f ? r : 0.f;
    open = open || o;
  }
  if (!spd) atomicAdd(v.n_not_spd, 1ull);
  note_off_axis(v, p);
  const float W = p[MG_P_W], B = p[MG_P_B];
  float G[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) G[i] = __fsub_rn(__fmul_rn(W, rg[i]), __fmul_rn(B, rb[i]));
  const ParamPlanes &pa = v.pa;
  pa.d0[e] = make_float4(m, ma[0], ma[1], ma[2]);
  pa.d1[e] = make_float4(J[0], J[1], J[2], __fsub_rn(W, B));
  pa.d2[e] = make_float4(p[MG_P_DL], p[MG_P_DL + 1], p[MG_P_DL + 2], p[MG_P_DL + 3]);
  pa.d3[e] = make_float4(p[MG_P_DL + 4], p[MG_P_DL + 5], p[MG_P_DQ], p[MG_P_DQ + 1]);
  pa.d4[e] = make_float4(p[MG_P_DQ + 2], p[MG_P_DQ + 3], p[MG_P_DQ + 4], p[MG_P_DQ + 5]);
  pa.d5[e] = make_float4(G[0], G[1], G[2], p[MG_P_KT]);
  pa.d6[e] = make_float4(p[MG_P_VC], p[MG_P_VC + 1], p[MG_P_VC + 2], __frcp_rn(p[MG_P_TAU]));
  pa.d7[e] = make_float4(mi[0], mi[1], mi[2], mi[3]);
  pa.d8[e] = make_float2(mi[4], mi[5]);
  if (open)
    invert_diag_fp64(pa, e, m, p[MG_P_IG], p[MG_P_IG + 1], p[MG_P_IG + 2], ma[0], ma[1], ma[2],
                     ma[3], ma[4], ma[5]);
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  pa.g0[e] = make_float4(__fmul_rn(m, rg[0]), __fmul_rn(m, rg[1]), __fmul_rn(m, rg[2]), 0.f);
  pa.g1[e] = z;
  pa.g2[e] = z;
  pa.g3[e] = z;
  pa.g4[e] = z;
  pa.g5[e] = 0.f;
}

// Derive the step's parameter planes for env e from its record f[MG_NPARAM]; a full mass matrix
// is inverted in FP64.
__device__ void derive(const SetupView &v, int64_t e, const float *f32) {
  const int64_t xs = v.xh_stride ? v.xh_stride : v.n;
  if (f32[MG_P_RG] == 0.f && f32[MG_P_RG + 1] == 0.f && f32[MG_P_RG + 2] == 0.f) {
    bool xh_zero = true;
    if (v.xh)
      for (int t = 0; t < 15; ++t) xh_zero = xh_zero && v.xh[(int64_t)t * xs + e] == 0.f;
    if (xh_zero) {
      derive_diag(v, e, f32);
      return;
    }
  }
  double p[MG_NPARAM];
  for (int j = 0; j < MG_NPARAM; ++j) p[j] = (double)f32[j];
  const double m = p[MG_P_M];
  const double rg[3] = {p[MG_P_RG], p[MG_P_RG + 1], p[MG_P_RG + 2]};
  const double *ma = p + MG_P_MA;
  const double r2 = rg[0] * rg[0] + rg[1] * rg[1] + rg[2] * rg[2];
  // I_o = I_g - m S(r_g)^2 = I_g + m (|r_g|^2 I - r_g r_g^T)  (inertia about the body origin)
  double Io[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j)
      Io[i][j] = (i == j ? p[MG_P_IG + i] + m * r2 : 0.0) - m * rg[i] * rg[j];

  // M = M_RB + M_A = [[m I + Ma_lin, -m S(r_g)], [m S(r_g), I_o + Ma_rot]], plus M_A's
  // off-diagonal entries from the extension (FP32 values, as the step reads them).
  double M[6][6];
  const double S[3][3] = {{0.0, -rg[2], rg[1]}, {rg[2], 0.0, -rg[0]}, {-rg[1], rg[0], 0.0}};
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      M[i][j] = (i == j) ? m + ma[i] : 0.0;
      M[i][3 + j] = -m * S[i][j];
      M[3 + i][j] = m * S[i][j];
      M[3 + i][3 + j] = Io[i][j] + ((i == j) ? ma[3 + i] : 0.0);
    }
  if (v.xh) {
    int t = 0;
    for (int i = 0; i < 6; ++i)
      for (int j = i + 1; j < 6; ++j, ++t) {
        const double a = (double)v.xh[(int64_t)t * xs + e];
        M[i][j] += a;
        M[j][i] += a;
      }
  }

  // Cholesky M = L L^T; L^-1 by forward substitution; M^-1 = L^-T L^-1.
  double L[6][6] = {}, Li[6][6] = {}, Mi[6][6] = {};
  bool spd = true;
  for (int j = 0; j < 6; ++j) {
    double d = M[j][j];
    for (int k = 0; k < j; ++k) d -= L[j][k] * L[j][k];
    if (!(d > 0.0)) {
      spd = false;
      d = 1.0;
    }
    L[j][j] = sqrt(d);
    for (int i = j + 1; i < 6; ++i) {
      double s = M[i][j];
      for (int k = 0; k < j; ++k) s -= L[i][k] * L[j][k];
      L[i][j] = s / L[j][j];
    }
  }
  for (int j = 0; j < 6; ++j) {
    Li[j][j] = 1.0 / L[j][j];
    for (int i = j + 1; i < 6; ++i) {
      double s = 0.0;
      for (int k = j; k < i; ++k) s += L[i][k] * Li[k][j];
      Li[i][j] = -s / L[i][i];
    }
  }
  for (int i = 0; i < 6; ++i)
    for (int j = 0; j < 6; ++j) {
      double s = 0.0;
      for (int k = (i > j ? i : j); k < 6; ++k) s += Li[k][i] * Li[k][j];
      Mi[i][j] = s;
    }
  if (!spd) atomicAdd(v.n_not_spd, 1ull);
  atomicOr(v.any_offdiag, 1u);
  note_off_axis(v, f32);

  const double W = p[MG_P_W], B = p[MG_P_B];
  const double G[3] = {W * rg[0] - B * p[MG_P_RB], W * rg[1] - B * p[MG_P_RB + 1],
                       W * rg[2] - B * p[MG_P_RB + 2]};
  const ParamPlanes &pa = v.pa;
  auto f = [](double x) { return (float)x; };
  pa.d0[e] = make_float4(f(m), f(ma[0]), f(ma[1]), f(ma[2]));
  pa.d1[e] = make_float4(f(Io[0][0] + ma[3]), f(Io[1][1] + ma[4]), f(Io[2][2] + ma[5]),
                         f(W - B));
  pa.d2[e] = make_float4(f(p[MG_P_DL]), f(p[MG_P_DL + 1]), f(p[MG_P_DL + 2]),
                         f(p[MG_P_DL + 3]));
  pa.d3[e] = make_float4(f(p[MG_P_DL + 4]), f(p[MG_P_DL + 5]), f(p[MG_P_DQ]),
                         f(p[MG_P_DQ + 1]));
  pa.d4[e] = make_float4(f(p[MG_P_DQ + 2]), f(p[MG_P_DQ + 3]), f(p[MG_P_DQ + 4]),
                         f(p[MG_P_DQ + 5]));
  pa.d5[e] = make_float4(f(G[0]), f(G[1]), f(G[2]), f(p[MG_P_KT]));
  pa.d6[e] = make_float4(f(p[MG_P_VC]), f(p[MG_P_VC + 1]), f(p[MG_P_VC + 2]),
                         f(1.0 / p[MG_P_TAU]));
  pa.d7[e] = make_float4(f(Mi[0][0]), f(Mi[1][1]), f(Mi[2][2]), f(Mi[3][3]));
  pa.d8[e] = make_float2(f(Mi[4][4]), f(Mi[5][5]));
  pa.g0[e] = make_float4(f(m * rg[0]), f(m * rg[1]), f(m * rg[2]), f(Io[0][1]));
  pa.g1[e] = make_float4(f(Io[0][2]), f(Io[1][2]), f(Mi[0][1]), f(Mi[0][2]));
  pa.g2[e] = make_float4(f(Mi[0][3]), f(Mi[0][4]), f(Mi[0][5]), f(Mi[1][2]));
  pa.g3[e] = make_float4(f(Mi[1][3]), f(Mi[1][4]), f(Mi[1][5]), f(Mi[2][3]));
  pa.g4[e] = make_float4(f(Mi[2][4]), f(Mi[2][5]), f(Mi[3][4]), f(Mi[3][5]));
  pa.g5[e] = f(Mi[4][5]);
}

// What a randomisation draws: each of the 27 scalars times lo + (hi - lo) u with hi - lo in two
// floats, the current's sigma and the half-width of r_g.
struct Draw {
  uint64_t seed;
  float lo, hi;
  df32 width;
  float sigma;
  uint32_t open;  // draws that FP64 alone does: none, or all where magnitudes are extreme
  double rg_halfwidth;
};
constexpr int kDraws = 30;  // 27 scalars, three of the current

// nominal x (lo + (hi - lo) u), rounded once; open: two floats (error 2^-45) leave the rounding
// undecided.
__device__ __forceinline__ float scaled(const Draw &d, float nominal, float u, bool &open) {
  df32 p = two_prod(d.width.h, u);
  p.l = __fmaf_rn(d.width.l, u, p.l);
  df32 s = fast_two_sum(fmaxf(d.lo, p.h), fminf(d.lo, p.h));
  s.l = __fadd_rn(s.l, p.l);
  const float q = __fmul_rn(s.h, nominal);
  const float r = __fmaf_rn(s.l, nominal, __fmaf_rn(s.h, nominal, -q));
  return round_df(q, r, q, 0x1p-43f, open);
}

// c + sigma r x, rounded once; open as above (error of the normal 2^-40.6).
__device__ __forceinline__ float current(const Draw &d, float c, df32 r, df32 x, bool &open) {
  const df32 z = df_mul(r, x);
  df32 p = two_prod(d.sigma, z.h);
  p.l = __fmaf_rn(d.sigma, z.l, p.l);
  const df32 s = two_sum(c, p.h);
  return round_df(s.h, __fadd_rn(s.l, p.l), __fadd_rn(fabsf(c), fabsf(p.h)), 0x1p-39f, open);
}

// Word j of an env's parameter draws from its block x of four.
__device__ __forceinline__ uint32_t draw_word(const uint4 &x, int j) {
  return (j % 4 == 0) ? x.x : (j % 4 == 1) ? x.y : (j % 4 == 2) ? x.z : x.w;
}

// The draws whose bits are set in `open` again, in FP64, into the record `row`: the 27 scalars,
// then the current.  One env in 3,000 comes here, mostly for one value.
__device__ __noinline__ void redraw_fp64(uint32_t open, const float *__restrict__ nom,
                                         const Draw &d, uint64_t gid, float *row) {
  for (; open; open &= open - 1u) {
    const int j = __ffs(open) - 1;
    if (j < 27) {
      const uint4 x = draw4(d.seed, gid, STREAM_PARAMS, (uint32_t)(j / 4));
      const double lo = (double)d.lo, u = u01d(draw_word(x, j));
      row[rand_idx(j)] = (float)((double)nom[rand_idx(j)] * (lo + ((double)d.hi - lo) * u));
    } else {
      const uint4 x = draw4(d.seed, gid, STREAM_CURRENT, 0u);
      const double r = sqrt(-2.0 * log(u01d(j < 29 ? x.x : x.z)));
      const double a = 2.0 * u01d(j < 29 ? x.y : x.w);
      const int i = MG_P_VC + j - 27;
      row[i] = (float)((double)nom[i] + (double)d.sigma * (r * (j == 28 ? sinpi(a) : cospi(a))));
    }
  }
}

// Draw one tile of blockDim.x envs from e0 on (of the given vehicle type, or of v.types): each
// thread draws and derives its env, the records are staged in rows [blockDim.x][MG_NPARAM] and
// leave as one contiguous run (a thread's own row is 140 bytes, so direct stores would touch 32
// sectors each). FP32 pairs but where they leave a rounding open: the FP64 form of the same draws
// took 840 us for 1,048,576 envs, FP64-pipe bound, against 55 us for the 360 bytes per env it
// stores; this takes 71 us (63 without the test of each rounding, which left 7 of 3.5 million
// values off by an ulp). DIAG: every mass matrix is diagonal (no r_g, no extension), so the FP64
// Cholesky is not compiled in (it doubles the registers).
template <bool DIAG>
__device__ __forceinline__ void randomize_tile(const SetupView &v,
                                               const float *__restrict__ nominal, const Draw &d,
                                               int64_t e0, float *rows, int32_t type = -1) {
  const int64_t e = e0 + threadIdx.x;
  if (e < v.n) {
    const uint64_t gid = (uint64_t)(v.gid0 + e);
    const float *nom = nominal + (int64_t)(type < 0 ? v.types[e] : type) * MG_NPARAM;
    float p[MG_NPARAM];
    uint32_t open = d.open;  // draws left to FP64
    bool o;
#pragma unroll
    for (int j = 0; j < MG_NPARAM; ++j) p[j] = nom[j];
    uint4 x = make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int j = 0; j < 27; ++j) {
      if (j % 4 == 0) x = draw4(d.seed, gid, STREAM_PARAMS, (uint32_t)(j / 4));
      p[rand_idx(j)] = scaled(d, p[rand_idx(j)], u01f(draw_word(x, j)), o);
      if (o) open |= 1u << j;
    }
    // Box-Muller normals of the current: two of the first pair, the cosine of the second
    const uint4 c = draw4(d.seed, gid, STREAM_CURRENT, 0u);
    df32 cs, sn;
    df32 r = df_normal_radius(u01f(c.x));
    df_cos_sin_turn(u01f(c.y), cs, sn);
    p[MG_P_VC] = current(d, p[MG_P_VC], r, cs, o);
    if (o) open |= 1u << 27;
    p[MG_P_VC + 1] = current(d, p[MG_P_VC + 1], r, sn, o);
    if (o) open |= 1u << 28;
    r = df_normal_radius(u01f(c.z));
    df_cos_sin_turn(u01f(c.w), cs, sn);
    p[MG_P_VC + 2] = current(d, p[MG_P_VC + 2], r, cs, o);
    if (o) open |= 1u << 29;
    if constexpr (!DIAG) {
      if (d.rg_halfwidth > 0.0) {  // off-centre gravity: nominal + U[-w, w] per axis
        const uint4 g = draw4(d.seed, gid, STREAM_PARAMS, 7u);
        const uint32_t w[3] = {g.x, g.y, g.z};
#pragma unroll
        for (int i = 0; i < 3; ++i)
          p[MG_P_RG + i] =
              (float)((double)p[MG_P_RG + i] + d.rg_halfwidth * (2.0 * u01d(w[i]) - 1.0));
      }
    }
    // Everything the step reads is derived from the stored FP32 values, so that it is consistent
    // with what mg_get_params reports.
    float *row = rows + threadIdx.x * MG_NPARAM;
#pragma unroll
    for (int j = 0; j < MG_NPARAM; ++j) row[j] = p[j];
    if (open) {
      redraw_fp64(open, nom, d, gid, row);
#pragma unroll
      for (int j = 0; j < MG_NPARAM; ++j) p[j] = row[j];
    }
    if constexpr (DIAG) derive_diag(v, e, p);
    else derive(v, e, p);
  }
  __syncthreads();
  const int64_t left = v.n - e0;
  block_copy(v.raw + e0 * MG_NPARAM, rows,
             (int)(left < blockDim.x ? left : blockDim.x) * MG_NPARAM);
}

// One env per thread.
template <bool DIAG>
__global__ void __launch_bounds__(kRandThreads)
    k_randomize(const SetupView v, const float *__restrict__ nominal, const Draw d) {
  __shared__ __align__(16) float rows[kRandThreads * MG_NPARAM];
  randomize_tile<DIAG>(v, nominal, d, (int64_t)blockIdx.x * kRandThreads, rows);
}

// Background form: up to 16 small blocks per SM stride over the fleet beside a step kernel on
// another stream.  Beside the work queue four of them fit an SM at a time; a static grid lets them
// in at its tail, which they then fill (one block per SM ran on alone after it: whole episodes of
// 1,048,576 envs x 50 sub-steps 1,225 us against 1,054, of 65,536 x 10 55.6 against 42.7).  Same
// per-env arithmetic.
__global__ void __launch_bounds__(kRandBgThreads)
    k_randomize_bg(const SetupView v, const float *__restrict__ nominal, const Draw d) {
  __shared__ __align__(16) float rows[kRandBgThreads * MG_NPARAM];
  const int64_t stride = (int64_t)gridDim.x * kRandBgThreads;
  for (int64_t e0 = (int64_t)blockIdx.x * kRandBgThreads; e0 < v.n; e0 += stride) {
    randomize_tile<true>(v, nominal, d, e0, rows);
    __syncthreads();
  }
}

// Admission of a serving job in one launch: its envs' type, parameters and start state (episode 0
// of the job's own seed).  As four operations (fill, draw, clear, reset), each bound by its own
// latency and launch, it took 9 us longer a job: 12 jobs of 64 to 32,768 envs served in 1,015 us,
// 909 so.
template <bool DIAG>
__global__ void __launch_bounds__(kRandThreads)
    k_admit(const SetupView v, const float *__restrict__ nominal, const Draw d, int32_t type,
            int32_t *types, const StatePlanes st, double nu0_sigma, uint32_t *episode,
            uint32_t *flags, unsigned long long *nonfinite_count) {
  __shared__ __align__(16) float rows[kRandThreads * MG_NPARAM];
  const int64_t e0 = (int64_t)blockIdx.x * kRandThreads, e = e0 + threadIdx.x;
  if (e < v.n) {
    types[e] = type;
    episode[e] = 0u;
    reset_env(st, e, (uint64_t)(v.gid0 + e), d.seed, nu0_sigma, episode, flags, nonfinite_count);
  }
  randomize_tile<DIAG>(v, nominal, d, e0, rows, type);
}

// in may be the stored records themselves (re-derived in place).
__global__ void __launch_bounds__(kRandThreads)
    k_import_params(const SetupView v, const float *in) {
  __shared__ __align__(16) float rows[kRandThreads * MG_NPARAM];
  const int64_t e0 = (int64_t)blockIdx.x * kRandThreads;
  const int64_t left = v.n - e0;
  const int total = (int)(left < kRandThreads ? left : kRandThreads) * MG_NPARAM;
  block_copy(rows, in + e0 * MG_NPARAM, total);
  __syncthreads();
  if (in != v.raw) block_copy(v.raw + e0 * MG_NPARAM, rows, total);
  if ((int64_t)threadIdx.x >= left) return;
  float p[MG_NPARAM];
#pragma unroll
  for (int j = 0; j < MG_NPARAM; ++j) p[j] = rows[threadIdx.x * MG_NPARAM + j];
  derive(v, e0 + threadIdx.x, p);
}

// Off-diagonal hydrodynamics between the record layout [n][MG_NXPARAM] and the planes
// [MG_NXPARAM][n] the step reads (to_planes), or back.
__global__ void k_xh_transpose(const float *__restrict__ in, float *__restrict__ out, int64_t n,
                               bool to_planes, int64_t stride) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  for (int c = 0; c < MG_NXPARAM; ++c) {
    if (to_planes)
      out[(int64_t)c * stride + e] = in[e * MG_NXPARAM + c];
    else
      out[e * MG_NXPARAM + c] = in[(int64_t)c * stride + e];
  }
}

// The records as they are, a contiguous run per block.
__global__ void __launch_bounds__(kThreads)
    k_export_params(const SetupView v, float *__restrict__ out) {
  constexpr int kRun = kThreads * 16;
  const int64_t i0 = (int64_t)blockIdx.x * kRun, left = v.n * MG_NPARAM - i0;
  block_copy(out + i0, v.raw + i0, (int)(left < kRun ? left : kRun));
}

__global__ void k_reset(const StatePlanes st, int64_t n, int64_t gid0,
                        const uint8_t *__restrict__ mask, uint64_t seed, double sigma,
                        uint32_t *__restrict__ episode, uint32_t *__restrict__ flags,
                        unsigned long long *nonfinite_count) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n || (mask && !mask[e])) return;
  reset_env(st, e, (uint64_t)(gid0 + e), seed, sigma, episode, flags, nonfinite_count);
}

// State rows ([n][MG_NSTATE], 84 B each) <-> planes, staged through shared memory so that a
// block's rows move as one contiguous span (16-byte vectors when the row buffer is 16-byte
// aligned: a block's span starts at a multiple of kRowThreads x 84 B = 10,752 B).
constexpr int kRowThreads = 128;

__global__ void __launch_bounds__(kRowThreads)
    k_export_state(const StatePlanes st, int64_t n, float *__restrict__ out) {
  __shared__ __align__(16) float rows[kRowThreads * MG_NSTATE];
  const int64_t e0 = (int64_t)blockIdx.x * kRowThreads;
  const int t = (int)threadIdx.x;
  const int64_t e = e0 + t;
  // Programmatic dependent launch, both ways: this kernel's launch overlaps the step that writes
  // the state, and the next step's launch overlaps this kernel (each waits here for the one before
  // it).
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
  if (e < n) {
    const float4 a = st.s0[e], b = st.s1[e], c = st.s2[e], d = st.s3[e], f = st.s4[e];
    const float r[MG_NSTATE] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z,
                                c.w, d.x, d.y, d.z, d.w, f.x, f.y, f.z, f.w, st.s5[e]};
#pragma unroll
    for (int j = 0; j < MG_NSTATE; ++j) rows[t * MG_NSTATE + j] = r[j];
  }
  __syncthreads();
  const int total = (int)(n - e0 < kRowThreads ? n - e0 : kRowThreads) * MG_NSTATE;
  float *o = out + e0 * MG_NSTATE;
  int done = 0;
  if (aligned16(out)) {
    done = total & ~3;
    float4 *o4 = reinterpret_cast<float4 *>(o);
    const float4 *r4 = reinterpret_cast<const float4 *>(rows);
    for (int i = t; i < done / 4; i += kRowThreads) o4[i] = r4[i];
  }
  for (int i = done + t; i < total; i += kRowThreads) o[i] = rows[i];
}

__global__ void __launch_bounds__(kRowThreads)
    k_import_state(const StatePlanes st, int64_t n, const float *__restrict__ in) {
  __shared__ __align__(16) float rows[kRowThreads * MG_NSTATE];
  const int64_t e0 = (int64_t)blockIdx.x * kRowThreads;
  const int t = (int)threadIdx.x;
  const int total = (int)(n - e0 < kRowThreads ? n - e0 : kRowThreads) * MG_NSTATE;
  const float *src = in + e0 * MG_NSTATE;
  int done = 0;
  if (aligned16(in)) {
    done = total & ~3;
    const float4 *i4 = reinterpret_cast<const float4 *>(src);
    float4 *r4 = reinterpret_cast<float4 *>(rows);
    for (int i = t; i < done / 4; i += kRowThreads) r4[i] = i4[i];
  }
  for (int i = done + t; i < total; i += kRowThreads) rows[i] = src[i];
  __syncthreads();
  const int64_t e = e0 + t;
  if (e >= n) return;
  const float *r = rows + t * MG_NSTATE;
  st.s0[e] = make_float4(r[0], r[1], r[2], r[3]);
  st.s1[e] = make_float4(r[4], r[5], r[6], r[7]);
  st.s2[e] = make_float4(r[8], r[9], r[10], r[11]);
  st.s3[e] = make_float4(r[12], r[13], r[14], r[15]);
  st.s4[e] = make_float4(r[16], r[17], r[18], r[19]);
  st.s5[e] = r[20];
}

__global__ void k_rewind(unsigned long long *cursor, uint32_t *gen_word, uint32_t gen,
                         bool always) {
  if (always || *gen_word != gen) {
    *cursor = 0;
    *gen_word = gen;
  }
}

__global__ void k_flags_to_bytes(const uint32_t *__restrict__ flags, int64_t n,
                                 uint8_t *__restrict__ out) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n) out[e] = (uint8_t)(flags[e] & 1u);
}

__global__ void k_philox(const uint32_t *__restrict__ ctr, const uint32_t *__restrict__ key,
                         uint32_t *__restrict__ out, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint4 r = philox4x32_10(make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2],
                                           ctr[4 * i + 3]),
                                make_uint2(key[2 * i], key[2 * i + 1]));
  out[4 * i] = r.x;
  out[4 * i + 1] = r.y;
  out[4 * i + 2] = r.z;
  out[4 * i + 3] = r.w;
}

}  // namespace

namespace {

Draw make_draw(const SetupView &v, uint64_t seed, double lo, double hi, double current_sigma,
               double rg_halfwidth) {
  Draw d{};
  d.seed = seed;
  d.lo = (float)lo;  // the bounds are FP32 numbers
  d.hi = (float)hi;
  const double width = hi - lo;
  d.width.h = (float)width;
  d.width.l = (float)(width - (double)d.width.h);
  d.sigma = (float)current_sigma;
  // Two floats hold 48 bits only while the lower one is a normal number.
  const bool plain = v.plain && lo >= 1e-6 && hi <= 1e6 &&
                     (current_sigma == 0.0 || (current_sigma >= 1e-25 && current_sigma <= 1e25));
  d.open = plain ? 0u : (1u << kDraws) - 1u;
  d.rg_halfwidth = rg_halfwidth;
  return d;
}

}  // namespace

cudaError_t launch_admit(const SetupView &v, const float *nominal, const mg_job_spec &job,
                         int32_t *types, const StatePlanes &st, uint32_t *episode, uint32_t *flags,
                         unsigned long long *nonfinite_count, cudaStream_t stream) {
  const mg_ranges &r = job.ranges;
  const Draw d = make_draw(v, job.param_seed, (double)r.lo, (double)r.hi, (double)r.current_sigma,
                           (double)r.rg_halfwidth);
  const int blocks = (int)((v.n + kRandThreads - 1) / kRandThreads);
  const auto kernel = v.diag_only && r.rg_halfwidth == 0.f ? k_admit<true> : k_admit<false>;
  kernel<<<blocks, kRandThreads, 0, stream>>>(v, nominal, d, job.vehicle_type, types, st,
                                              (double)r.nu0_sigma, episode, flags,
                                              nonfinite_count);
  return cudaGetLastError();
}

cudaError_t launch_randomize(const SetupView &v, const float *nominal, uint64_t seed, double lo,
                             double hi, double current_sigma, double rg_halfwidth,
                             cudaStream_t stream, int background_blocks) {
  const Draw d = make_draw(v, seed, lo, hi, current_sigma, rg_halfwidth);
  if (background_blocks > 0) {
    if (!v.diag_only || rg_halfwidth != 0.0) return cudaErrorInvalidValue;
    const int64_t full = (v.n + kRandBgThreads - 1) / kRandBgThreads;
    const int blocks = (int)std::min<int64_t>(full, background_blocks);
    k_randomize_bg<<<blocks, kRandBgThreads, 0, stream>>>(v, nominal, d);
    return cudaGetLastError();
  }
  const int blocks = (int)((v.n + kRandThreads - 1) / kRandThreads);
  if (v.diag_only && rg_halfwidth == 0.0)
    k_randomize<true><<<blocks, kRandThreads, 0, stream>>>(v, nominal, d);
  else
    k_randomize<false><<<blocks, kRandThreads, 0, stream>>>(v, nominal, d);
  return cudaGetLastError();
}

cudaError_t launch_xh_transpose(const float *in, float *out, int64_t n, bool to_planes,
                                cudaStream_t stream, int64_t stride) {
  if (stride < n) stride = n;
  k_xh_transpose<<<blocks_for(n), kThreads, 0, stream>>>(in, out, n, to_planes, stride);
  return cudaGetLastError();
}

cudaError_t launch_import_params(const SetupView &v, const float *in, cudaStream_t stream) {
  k_import_params<<<(int)((v.n + kRandThreads - 1) / kRandThreads), kRandThreads, 0, stream>>>(v,
                                                                                            in);
  return cudaGetLastError();
}

cudaError_t launch_export_params(const SetupView &v, float *out, cudaStream_t stream) {
  constexpr int64_t kRun = (int64_t)kThreads * 16;
  k_export_params<<<(int)((v.n * MG_NPARAM + kRun - 1) / kRun), kThreads, 0, stream>>>(v, out);
  return cudaGetLastError();
}

cudaError_t launch_reset(const StatePlanes &st, int64_t n, int64_t gid0, const uint8_t *mask,
                         uint64_t seed, double nu0_sigma, uint32_t *episode, uint32_t *flags,
                         unsigned long long *nonfinite_count, cudaStream_t stream) {
  k_reset<<<blocks_for(n), kThreads, 0, stream>>>(st, n, gid0, mask, seed, nu0_sigma, episode,
                                                  flags, nonfinite_count);
  return cudaGetLastError();
}

cudaError_t launch_rewind(unsigned long long *cursor, uint32_t *gen_word, uint32_t gen, bool always,
                          cudaStream_t stream) {
  k_rewind<<<1, 1, 0, stream>>>(cursor, gen_word, gen, always);
  return cudaGetLastError();
}

cudaError_t launch_export_state(const StatePlanes &st, int64_t n, float *out,
                                cudaStream_t stream) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)((n + kRowThreads - 1) / kRowThreads));
  cfg.blockDim = dim3(kRowThreads);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_export_state, st, n, out);
}

cudaError_t launch_import_state(const StatePlanes &st, int64_t n, const float *in,
                                cudaStream_t stream) {
  k_import_state<<<(int)((n + kRowThreads - 1) / kRowThreads), kRowThreads, 0, stream>>>(st, n,
                                                                                      in);
  return cudaGetLastError();
}

cudaError_t launch_flags_to_bytes(const uint32_t *flags, int64_t n, uint8_t *out,
                                  cudaStream_t stream) {
  k_flags_to_bytes<<<blocks_for(n), kThreads, 0, stream>>>(flags, n, out);
  return cudaGetLastError();
}

cudaError_t launch_philox(const uint32_t *ctr, const uint32_t *key, uint32_t *out, int64_t n,
                          cudaStream_t stream) {
  k_philox<<<blocks_for(n), kThreads, 0, stream>>>(ctr, key, out, n);
  return cudaGetLastError();
}

}  // namespace mg
