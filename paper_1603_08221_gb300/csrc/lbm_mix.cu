// lbm_mix.cu — sm_103a implementation of the C ABI in include/lbm_mix.h.
//
// One time step of the two-species D2Q9 MRT lattice Boltzmann model of
// Wang, Xu & Guo (arXiv:1603.08221, Sec. 3) is ONE fused kernel launch
// (lbm_step_kernel; on grids of several waves and with 16-bit storage,
// lbm_walls_kernel computes the wall parameters r and tau_q of every column
// ahead of it), and small FP32 channels take several steps per launch
// (lbm_tile_kernel, lbm_tile.cuh): pull-streaming from the previous post-collision buffer
// with the diffuse-bounce-back walls (Eqs. bot, bot2, R) and the
// extrapolation-correction ends (Eqs. rho1, rho2) folded into the loads,
// moments (Eq. rhou), effective relaxation times (Eqs. EQFrb, EQFrsp, psi,
// taos, taoq, A12), the MRT collision (Eqs. MR, m, S, feq) for both species,
// the store of the new post-collision buffer, and per-column reductions (pairs
// of floats, 2^-44 of the sum and better, FP64 over the columns) that feed the
// next step's density correction and the separation diagnostics (Eqs. C, CL,
// Clline).
//
// Data layout in HBM (per buffer): the channel is cut into strips of 32
// columns; strip s holds, row after row, the nine populations of its 32
// columns, each as one segment of 32 species pairs (a, b):
//   offset(sp, i, j, x) = (x / 32) * SS + j * RS + i * 64 + 2 * (x % 32) + sp
// with RS = 576 elements per strip row and SS = N * RS per strip.  A node's
// two species of population i are adjacent, so one 8-byte (FP32) or 4-byte
// (BF16/FP16) access per lane fetches both and a warp access is one aligned
// contiguous segment; all offsets inside a strip are compile-time
// immediates.  Two buffers A/B alternate.  The CTAs of one strip (one per
// row block) sweep their rows in steps of TY; the per-column quantities (the
// tau_q of the two walls, the column sums) are produced by the CTAs of that
// strip alone, without floating-point atomics and in a fixed order.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdarg.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <time.h>
#include <string.h>

#include <mutex>
#include <algorithm>
#include <new>
#include <type_traits>

#include "../../include/lbm_mix.h"

namespace {

#include "lbm_psi_table.cuh"

// ---------------------------------------------------------------- errors
thread_local char g_err[512] = "";

int set_err(int code, const char* fmt, ...) __attribute__((format(printf, 2, 3)));
int set_err(int code, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof g_err, fmt, ap);
  va_end(ap);
  return code;
}

#define CK(call)                                                                      \
  do {                                                                                \
    cudaError_t e_ = (call);                                                          \
    if (e_ != cudaSuccess)                                                            \
      return set_err(LBM_ECUDA, "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), \
                     __FILE__, __LINE__);                                             \
  } while (0)

// ------------------------------------------------------- lattice constants
constexpr int TX = 32;          // columns per CTA = strip width (one warp per row segment)
constexpr int RS = 18 * TX;     // elements per row of a strip (9 populations x 32 pairs)
constexpr int PS = 2 * TX;      // elements per population segment (32 columns x 2 species)
constexpr int TY = 8;           // rows per sweep iteration
constexpr int NPART = 8;        // doubles per CTA partial
constexpr int NREC = 8;         // doubles per diagnostic record
constexpr int DIAG_CAP = 4096;  // diagnostic records kept
constexpr float kPi = 3.14159265358979323846f;

// What the FP32 node arithmetic and the tile kernel need; small, so that a
// launch can carry one for each channel of a sweep.
struct LatCore {
  int N, Nx;
  unsigned SS;           // floats per strip: N * RS
  int x_periodic;
  int wall_mode;         // LBM_WALL_DBB or LBM_WALL_BSR
  int r_form;            // LBM_R_FIRST, LBM_R_SPECIES or LBM_R_SECOND (Eq. R)
  int lam_mix;           // lambda_s with the mixture (1) or partial (0) pressure
  float rsqrt_mh[2];     // 1 / sqrt(m_s / m_min)
  float s[2];            // s_sigma = m_min / m_sigma
  // per-species constants as (species a, species b) pairs for the packed
  // FP32x2 arithmetic; ce2, cp2: coefficients of the non-equilibrium energy
  // moments on the deviations (rest, axis, diagonal: e: -2s, 3 - 2s, 6 - 2s;
  // eps: 3s, 3s - 6, 3s - 3) times om_e / 36 and om_eps / 36, cu2: of rho u^2
  // (-3, 3) likewise
  float2 s2, cw1_2, cw5_2, c_xl2, inv_c_xl2, ce2[3], cp2[3], cu2[2];
  float inv_c_lam;       // 1 / (3 mu sqrt(pi/6))
  float c_lam;           // 3 mu sqrt(pi/6): lambda = c_lam / (n sqrt(m_x))
  float c_ts;            // sqrt(6/pi)
  float c_td;            // (3/2) sqrt(3 m0 m_a m_b / m_min)
  float c_m0;
  float H;               // channel height = N
  float2 end_mass[2][2]; // N rho_s at the inlet, outlet ([end][species]) as a
                         // sum of two floats
};

struct Lat : LatCore {
  int pitch;
  int light;             // index of the light species
  float cw0[2];          // rest-equilibrium weights w_i alpha_si: rest (9 - 5s)/9,
  float cw1[2], cw5[2];  // axis s/9, diagonal s/36
  float2 ke2[3], kp2[3]; // the coefficients behind ce2, cp2, unscaled
  float om_e, om_eps;    // 1/tau_e, 1/tau_eps
  double mh[2];          // m_sigma / m_min
  double rho_in[2], rho_out[2];
  double C_in, C_out;    // light-species mole fraction at the ends
};

// ------------------------------------------------------ special functions
// E_1(x) for 0 < x <= 1 from its convergent series (Abramowitz & Stegun
// 5.1.11) truncated after ten terms (remainder < 2.3e-9 at x = 1):
// E_1(x) = -gamma - ln x + sum_{k=1}^{10} (-1)^{k+1} x^k / (k k!).
__device__ __forceinline__ float e1_series(float x) {
  float p = -1.0f / 36288000.0f;
  p = fmaf(p, x, 1.0f / 3265920.0f);
  p = fmaf(p, x, -1.0f / 322560.0f);
  p = fmaf(p, x, 1.0f / 35280.0f);
  p = fmaf(p, x, -1.0f / 4320.0f);
  p = fmaf(p, x, 1.0f / 600.0f);
  p = fmaf(p, x, -1.0f / 96.0f);
  p = fmaf(p, x, 1.0f / 18.0f);
  p = fmaf(p, x, -0.25f);
  p = fmaf(p, x, 1.0f);
  return fmaf(p, x, -0.5772156649f) - logf(x);
}

// x e^x E_1(x) for x >= 1: Hastings' rational approximation as tabulated in
// Abramowitz & Stegun 5.1.56 (absolute error < 2e-8).
__device__ __forceinline__ float xexe1_rational(float x) {
  float num = x + 8.5733287401f, den = x + 9.5733223454f;
  num = fmaf(num, x, 18.0590169730f);
  num = fmaf(num, x, 8.6347608925f);
  num = fmaf(num, x, 0.2677737343f);
  den = fmaf(den, x, 25.6329561486f);
  den = fmaf(den, x, 21.0996530827f);
  den = fmaf(den, x, 3.9584969228f);
  return num / den;
}

__device__ __forceinline__ float e1_dev(float x) {
  return x <= 1.0f ? e1_series(x) : expf(-x) * xexe1_rational(x) / x;
}

// psi(a) = 1 + (a - 1) e^{-a} - a^2 E_1(a)  (Eq. psi) and psi'(a), a >= 0,
// from the cubics of lbm_psi_table.cuh: 12 instructions and one 16-byte load
// that the lanes of a row share, against the 25 of a series for a <= 1 and a
// rational form beyond, both evaluated.  At 57 % issue the FMA pipe was as
// busy as the issue slots, and half of its work was psi.  Relative error below
// 1.6e-7 (series and rational form: 1.9e-7).  T: the table, in shared memory
// wherever a thread evaluates more than one value.
__device__ __forceinline__ float psi_cubic(const float4* T, float am) {
  const unsigned edge = __float_as_uint(fmaxf(am, 0x1p-22f)) & 0xfff80000u;
  const float4 q = *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(T) +
                                                    ((edge >> 15) - (105u << 8)));
  const float u = am - __uint_as_float(edge);
  return fmaf(fmaf(fmaf(q.w, u, q.z), u, q.y), u, q.x);
}
__device__ __forceinline__ float psi_dev(const float4* T, float a) {
  return __fmul_rn(psi_cubic(T, fminf(a, 16.0f)), fminf(a, 1.0f));
}
__device__ __forceinline__ float dpsi_dev(const float4* T, float a) {
  return psi_cubic(T, fminf(a, 16.0f));
}

// Copies psi's table to shared memory (the caller synchronises).
__device__ __forceinline__ void load_psi_table(float4* dst, int tid, int threads) {
  for (int k = tid; k < PSI_SEGMENTS; k += threads) dst[k] = kPsiTab[k];
}

// Reciprocal and reciprocal square root of the special-function unit (1 and
// 2 ulp), without the scaling steps for subnormal arguments: densities,
// masses and mean free paths are nowhere near them.
__device__ __forceinline__ float rcp_fast(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rsqrt_fast(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ------------------------------------------------- packed FP32x2 helpers
// The two species run the same arithmetic on different data; Blackwell's
// packed FP32x2 instructions do both in one issue slot.  Each component is
// rounded exactly as the scalar operation would be.
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  return __ffma2_rn(b, f2(-1.0f), a);  // exact: a - b with one rounding
}

// ------------------------------------------------------------- storage
// Populations are stored as deviations d_i = f_i - w_i alpha_si rhobar_s(x)
// from the rest equilibrium (Eq. feq with u = 0) of a fixed per-column
// reference density rhobar_s(x) (the initial profile).  The heavy species'
// rest population carries ~90% of its mass, so storing f_i itself would put
// FP32 rounding of that large number into every moment; the deviations are
// small and keep their full relative precision.  All arithmetic below works
// on deviations relative to the node's own column reference.
template <typename ST>
struct Stor;
// ld/st move one species' value; ld2/st2 move the (a, b) pair of a node's
// population at p (p points at species a, aligned to the pair).
template <>
struct Stor<float> {
  static __device__ __forceinline__ float ld(const float* p) { return __ldg(p); }
  static __device__ __forceinline__ void st(float* p, float v) { *p = v; }
  static __device__ __forceinline__ float2 ld2(const float* p) {
    return __ldg(reinterpret_cast<const float2*>(p));
  }
  static __device__ __forceinline__ void st2(float* p, float2 v) {
    *reinterpret_cast<float2*>(p) = v;
  }
  static __device__ __forceinline__ void st2_sr(float* p, float2 v, unsigned) { st2(p, v); }
};
// Reduced-precision storage of the same deviations: loads widen to FP32, all
// arithmetic is FP32, stores round to nearest.
// Stochastic rounding of an FP32 pair to 16 bits (Blackwell's cvt.rs): each
// value rounds up with probability equal to the fraction of the spacing it
// lies above the lower neighbour, decided by the random bits rbits.  The
// pair is packed with species a (the lower address) in the low half.
__device__ __forceinline__ unsigned cvt_rs_bf16x2(float a, float b, unsigned rbits) {
  unsigned d;
  asm("cvt.rs.satfinite.bf16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(b), "f"(a), "r"(rbits));
  return d;
}
__device__ __forceinline__ unsigned cvt_rs_f16x2(float a, float b, unsigned rbits) {
  unsigned d;
  asm("cvt.rs.satfinite.f16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(b), "f"(a), "r"(rbits));
  return d;
}

template <>
struct Stor<__nv_bfloat16> {
  static __device__ __forceinline__ float ld(const __nv_bfloat16* p) {
    return __bfloat162float(__ldg(p));
  }
  static __device__ __forceinline__ void st(__nv_bfloat16* p, float v) {
    *p = __float2bfloat16_rn(v);
  }
  static __device__ __forceinline__ float2 ld2(const __nv_bfloat16* p) {
    return __bfloat1622float2(__ldg(reinterpret_cast<const __nv_bfloat162*>(p)));
  }
  static __device__ __forceinline__ void st2(__nv_bfloat16* p, float2 v) {
    *reinterpret_cast<__nv_bfloat162*>(p) = __float22bfloat162_rn(v);
  }
  static __device__ __forceinline__ void st2_sr(__nv_bfloat16* p, float2 v, unsigned rbits) {
    *reinterpret_cast<unsigned*>(p) = cvt_rs_bf16x2(v.x, v.y, rbits);
  }
};
template <>
struct Stor<__half> {
  static __device__ __forceinline__ float ld(const __half* p) { return __half2float(__ldg(p)); }
  static __device__ __forceinline__ void st(__half* p, float v) { *p = __float2half_rn(v); }
  static __device__ __forceinline__ float2 ld2(const __half* p) {
    return __half22float2(__ldg(reinterpret_cast<const __half2*>(p)));
  }
  static __device__ __forceinline__ void st2(__half* p, float2 v) {
    *reinterpret_cast<__half2*>(p) = __float22half2_rn(v);
  }
  static __device__ __forceinline__ void st2_sr(__half* p, float2 v, unsigned rbits) {
    *reinterpret_cast<unsigned*>(p) = cvt_rs_f16x2(v.x, v.y, rbits);
  }
};

struct Ends {
  float kin[2], kout[2];  // Eq. rho2 density-correction factors
  float gin[2], gout[2];  // ghost reference offsets kappa(2 rb(1) - rb(2)) - rb(0), per species
};

__device__ __forceinline__ unsigned idx(const Lat& L, int sp, int i, int j, int x) {
  return (unsigned)(x >> 5) * L.SS + (unsigned)(j * RS + i * PS + 2 * (x & 31) + sp);
}

// Programmatic dependent launch: a kernel launched with the programmatic
// stream-serialisation attribute may start while the kernel before it in the
// stream is still running.  The kernels of the step sequence wait for their
// predecessor's completion and memory (wait) before their first global
// memory access.  The wall kernel and the tile kernel let their successor
// launch as soon as all of their own CTAs run (launch_dependents); the step
// kernel lets it launch when it completes (the next kernel's CTAs are then
// spread evenly over the SMs the step frees: 0.2197 against 0.2235 s for 5000
// steps of a 1280 x 64 channel).  Launched without the attribute, both
// instructions return at once.
__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Bulk prefetch of one strip row (all 18 populations of 32 columns, one
// contiguous RS-element run) into L2.  Issued by one lane per warp for the
// row that warp sweeps next, so the DRAM reads of row j + TY are in flight
// while row j is computed, with no registers or shared memory held for them.
template <typename ST>
__device__ __forceinline__ void prefetch_row_l2(const ST* row) {
  static_assert((RS * sizeof(ST)) % 16 == 0, "bulk prefetch size must be a multiple of 16 B");
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(row),
               "r"((int)(RS * sizeof(ST)))
               : "memory");
}

template <typename ST>
__device__ __forceinline__ float ld(const ST* __restrict__ f, const Lat& L, int sp, int i, int j,
                                    int x) {
  return Stor<ST>::ld(f + idx(L, sp, i, j, x));
}

// Deviation (relative to the SOURCE column's reference) that population i
// carries from column xs at row js; the inlet/outlet ghost columns (Eq. rho1,
// all nine populations extrapolated and scaled by Eq. rho2) are virtual.
template <typename ST>
__device__ __forceinline__ float src(const ST* __restrict__ f, const Lat& L, const Ends& E,
                                     float cwi, int sp, int i, int js, int xs) {
  if (!L.x_periodic) {
    if (xs == 0)
      return fmaf(E.kin[sp], 2.0f * ld(f, L, sp, i, js, 1) - ld(f, L, sp, i, js, 2),
                  cwi * E.gin[sp]);
    if (xs == L.Nx - 1)
      return fmaf(E.kout[sp],
                  2.0f * ld(f, L, sp, i, js, L.Nx - 2) - ld(f, L, sp, i, js, L.Nx - 3),
                  cwi * E.gout[sp]);
  }
  return ld(f, L, sp, i, js, xs);
}

// Per-thread column data: own reference density and the reference
// differences to the left and right neighbour columns.
struct ColRef {
  float rb[2], dl[2], dr[2];
};

__device__ __forceinline__ ColRef col_ref(const Lat& L, const float* __restrict__ refrho, int x) {
  ColRef c;
  int xm = x - 1, xp = x + 1;
  if (xm < 0) xm += L.Nx;
  if (xp >= L.Nx) xp -= L.Nx;
  const bool ok = x < L.Nx;
#pragma unroll
  for (int sp = 0; sp < 2; ++sp) {
    const float* r = refrho + sp * L.Nx;
    float r0 = ok ? __ldg(r + x) : 0.0f;
    c.rb[sp] = r0;
    c.dl[sp] = ok ? __ldg(r + xm) - r0 : 0.0f;  // exact: adjacent columns differ < 2x
    c.dr[sp] = ok ? __ldg(r + xp) - r0 : 0.0f;
  }
  return c;
}

// Pre-collision deviations of node (x, j): f_i(x) = f'_i(x - c_i) (Eq. MRT)
// re-referenced to column x, with the unknown populations of the wall rows
// from diffuse bounce-back (Eqs. bot, bot2) on the post-collision state of
// the same node.  The wall equilibrium f^eq_i(rho_w, u_w = 0) = w_i s rho_w
// with rho_w from zero normal species flux equals 6 w_i (sum of the outgoing
// f'); its rest part cancels against the reference, leaving
// d_i = (1 - r) d'_opp(i) + r (w_i/(1/6)) sum_outgoing d'.
template <typename ST>
__device__ __forceinline__ void pull_node(const ST* __restrict__ f, const Lat& L, const Ends& E,
                                          const ColRef& C, int x, int j, float2 r_bot2,
                                          float2 r_top2, float fs[2][9]) {
  int xm = x - 1, xp = x + 1;
  if (L.x_periodic) {
    if (xm < 0) xm += L.Nx;
    if (xp >= L.Nx) xp -= L.Nx;
  }
  const bool bot = (j == 0), top = (j == L.N - 1);
#pragma unroll
  for (int sp = 0; sp < 2; ++sp) {
    float* g = fs[sp];
    const float c1 = L.cw1[sp], c5 = L.cw5[sp];
    const float dl = C.dl[sp], dr = C.dr[sp];
    const float r_bot = sp ? r_bot2.y : r_bot2.x, r_top = sp ? r_top2.y : r_top2.x;
    g[0] = ld(f, L, sp, 0, j, x);
    g[1] = fmaf(c1, dl, src(f, L, E, c1, sp, 1, j, xm));
    g[3] = fmaf(c1, dr, src(f, L, E, c1, sp, 3, j, xp));
    if (bot && L.wall_mode == LBM_WALL_BSR) {
      // bounce-back (fraction r) and specular reflection (1 - r): the
      // mirror image of c_5 = (1,1) leaves column x - 1 as c_8, that of c_6
      // leaves column x + 1 as c_7
      const float q = 1.0f - r_bot;
      g[2] = ld(f, L, sp, 4, j, x);
      g[5] = fmaf(r_bot, ld(f, L, sp, 7, j, x),
                  __fmul_rn(q, fmaf(c5, dl, src(f, L, E, c5, sp, 8, j, xm))));
      g[6] = fmaf(r_bot, ld(f, L, sp, 8, j, x),
                  __fmul_rn(q, fmaf(c5, dr, src(f, L, E, c5, sp, 7, j, xp))));
    } else if (bot) {
      float o4 = ld(f, L, sp, 4, j, x), o7 = ld(f, L, sp, 7, j, x), o8 = ld(f, L, sp, 8, j, x);
      // the equilibrium parts t/6, t/6 and t - 2 t/6 sum to t exactly up
      // to one rounding, so the wall conserves mass without an FP32 bias
      float t = __fmul_rn(r_bot, o4 + o7 + o8), q = 1.0f - r_bot, t6 = __fmul_rn(t, 1.0f / 6.0f);
      g[2] = fmaf(q, o4, fmaf(-2.0f, t6, t));
      g[5] = fmaf(q, o7, t6);
      g[6] = fmaf(q, o8, t6);
    } else {
      g[2] = ld(f, L, sp, 2, j - 1, x);
      g[5] = fmaf(c5, dl, src(f, L, E, c5, sp, 5, j - 1, xm));
      g[6] = fmaf(c5, dr, src(f, L, E, c5, sp, 6, j - 1, xp));
    }
    if (top && L.wall_mode == LBM_WALL_BSR) {
      // mirror images: c_7 = (-1,-1) of c_6 from column x + 1, c_8 = (1,-1)
      // of c_5 from column x - 1
      const float q = 1.0f - r_top;
      g[4] = ld(f, L, sp, 2, j, x);
      g[7] = fmaf(r_top, ld(f, L, sp, 5, j, x),
                  __fmul_rn(q, fmaf(c5, dr, src(f, L, E, c5, sp, 6, j, xp))));
      g[8] = fmaf(r_top, ld(f, L, sp, 6, j, x),
                  __fmul_rn(q, fmaf(c5, dl, src(f, L, E, c5, sp, 5, j, xm))));
    } else if (top) {
      float o2 = ld(f, L, sp, 2, j, x), o5 = ld(f, L, sp, 5, j, x), o6 = ld(f, L, sp, 6, j, x);
      float t = __fmul_rn(r_top, o2 + o5 + o6), q = 1.0f - r_top, t6 = __fmul_rn(t, 1.0f / 6.0f);
      g[4] = fmaf(q, o2, fmaf(-2.0f, t6, t));
      g[7] = fmaf(q, o5, t6);
      g[8] = fmaf(q, o6, t6);
    } else {
      g[4] = ld(f, L, sp, 4, j + 1, x);
      g[7] = fmaf(c5, dr, src(f, L, E, c5, sp, 7, j + 1, xp));
      g[8] = fmaf(c5, dl, src(f, L, E, c5, sp, 8, j + 1, xm));
    }
  }
}

// The same pull for a node whose row is not a wall row and whose strip does
// not contain an end column: nine pair loads (both species) at immediate
// offsets from the row pointers of columns x (p), x - 1 (pl) and x + 1 (pr),
// re-referenced to column x in FP32x2.
template <typename ST>
__device__ __forceinline__ void pull_fast(const ST* __restrict__ p, const ST* __restrict__ pl,
                                          const ST* __restrict__ pr, const Lat& L,
                                          const ColRef& C, float2 g[9]) {
  const float2 dl = make_float2(C.dl[0], C.dl[1]), dr = make_float2(C.dr[0], C.dr[1]);
  g[0] = Stor<ST>::ld2(p);
  g[1] = fma2(L.cw1_2, dl, Stor<ST>::ld2(pl + 1 * PS));
  g[3] = fma2(L.cw1_2, dr, Stor<ST>::ld2(pr + 3 * PS));
  g[2] = Stor<ST>::ld2(p + 2 * PS - RS);
  g[5] = fma2(L.cw5_2, dl, Stor<ST>::ld2(pl + 5 * PS - RS));
  g[6] = fma2(L.cw5_2, dr, Stor<ST>::ld2(pr + 6 * PS - RS));
  g[4] = Stor<ST>::ld2(p + 4 * PS + RS);
  g[7] = fma2(L.cw5_2, dr, Stor<ST>::ld2(pr + 7 * PS + RS));
  g[8] = fma2(L.cw5_2, dl, Stor<ST>::ld2(pl + 8 * PS + RS));
}

// pull_fast for a strip that holds column 1 or N_x - 2: their neighbours
// outside are the virtual ghost columns (src), everything else is as above.
template <typename ST>
__device__ __forceinline__ void pull_edge(const ST* __restrict__ f, const ST* __restrict__ p,
                                          const ST* __restrict__ pl, const ST* __restrict__ pr,
                                          const Lat& L, const Ends& E, const ColRef& C, int x,
                                          int j, float2 g[9]) {
  pull_fast(p, pl, pr, L, C, g);
  if (x == 1) {
    auto ghost = [&](int sp, int i, int js, float cw) {
      return fmaf(cw, C.dl[sp], src(f, L, E, cw, sp, i, js, 0));
    };
    g[1] = make_float2(ghost(0, 1, j, L.cw1[0]), ghost(1, 1, j, L.cw1[1]));
    g[5] = make_float2(ghost(0, 5, j - 1, L.cw5[0]), ghost(1, 5, j - 1, L.cw5[1]));
    g[8] = make_float2(ghost(0, 8, j + 1, L.cw5[0]), ghost(1, 8, j + 1, L.cw5[1]));
  }
  if (x == L.Nx - 2) {
    auto ghost = [&](int sp, int i, int js, float cw) {
      return fmaf(cw, C.dr[sp], src(f, L, E, cw, sp, i, js, L.Nx - 1));
    };
    g[3] = make_float2(ghost(0, 3, j, L.cw1[0]), ghost(1, 3, j, L.cw1[1]));
    g[6] = make_float2(ghost(0, 6, j - 1, L.cw5[0]), ghost(1, 6, j - 1, L.cw5[1]));
    g[7] = make_float2(ghost(0, 7, j + 1, L.cw5[0]), ghost(1, 7, j + 1, L.cw5[1]));
  }
}

// ---------------------------------------------------------------- moments
// The node arithmetic is written with explicit fma, mul and add wherever a
// product feeds a sum, so that every kernel that inlines it rounds alike:
// the step kernel, the wall kernel and the tile kernel give the same bits.
struct Macro {
  float sd[2];           // sum of deviations: rho_s - rhobar_s
  float rho[2];
  float n, inv_n, mx;
};

__device__ __forceinline__ float number_density(const LatCore& L, float rho_a, float rho_b) {
  return fmaf(rho_a, L.s[0], __fmul_rn(rho_b, L.s[1]));  // Eq. P
}

// m_x = rho / n.  NaN where n < 0: with both species negative the ratio is that
// of a gas, and psi's table, which takes no note of its argument's sign, would
// go on from there with finite rates.
__device__ __forceinline__ float mixture_mass(float rho, float n, float inv_n) {
  return n < 0.0f ? NAN : __fmul_rn(rho, inv_n);
}

__device__ __forceinline__ void macro(const Lat& L, const ColRef& C, const float fs[2][9],
                                      Macro& m) {
#pragma unroll
  for (int sp = 0; sp < 2; ++sp) {
    const float* g = fs[sp];
    // the order of density_sum, so that every wall task gives the same bits
    m.sd[sp] = g[0] + (((g[1] + g[3]) + (g[2] + g[4])) + ((g[5] + g[7]) + (g[6] + g[8])));
    m.rho[sp] = C.rb[sp] + m.sd[sp];
  }
  m.n = number_density(L, m.rho[0], m.rho[1]);
  m.inv_n = rcp_fast(m.n);
  m.mx = mixture_mass(__fadd_rn(m.rho[0], m.rho[1]), m.n, m.inv_n);
}

// ------------------------------------------- packed per-node arithmetic
// The node update of the step and moments kernels works on g[i] =
// (species a, species b) pairs of the pre-collision deviations.
struct Macro2 {
  float2 sd;   // sum of deviations: rho_s - rhobar_s
  float2 rho;  // species densities
  float n, inv_n, inv_rho, mx;
};

// Density deviations of both species from the pulled populations.
__device__ __forceinline__ float2 density_sum(const float2 g[9]) {
  const float2 a14 = add2(add2(g[1], g[3]), add2(g[2], g[4]));
  const float2 a58 = add2(add2(g[5], g[7]), add2(g[6], g[8]));
  return add2(g[0], add2(a14, a58));
}

__device__ __forceinline__ void macro2(const LatCore& L, float2 rb, const float2 g[9], Macro2& m) {
  m.sd = density_sum(g);
  m.rho = add2(rb, m.sd);
  const float rho = __fadd_rn(m.rho.x, m.rho.y);
  m.inv_rho = rcp_fast(rho);
  m.n = number_density(L, m.rho.x, m.rho.y);
  m.inv_n = rcp_fast(m.n);
  m.mx = mixture_mass(rho, m.n, m.inv_n);
}

// Sums and differences of opposite populations, from which the momenta, the
// other moments and the collision are formed, and the mixture velocity.
// Formed after the relaxation rates: carried across their evaluation they
// would not fit the registers.
struct Flow2 {
  float2 s13, s24, s57, s68, d13, d24, d57, d68, dx, dy, jx, jy;
  float ux, uy;
};
__device__ __forceinline__ void flow2(const float2 g[9], float inv_rho, Flow2& w) {
  w.s13 = add2(g[1], g[3]);
  w.s24 = add2(g[2], g[4]);
  w.s57 = add2(g[5], g[7]);
  w.s68 = add2(g[6], g[8]);
  w.d13 = sub2(g[1], g[3]);
  w.d24 = sub2(g[2], g[4]);
  w.d57 = sub2(g[5], g[7]);
  w.d68 = sub2(g[6], g[8]);
  w.dx = sub2(w.d57, w.d68);  // diagonal momenta
  w.dy = add2(w.d57, w.d68);
  w.jx = add2(w.d13, w.dx);
  w.jy = add2(w.d24, w.dy);
  w.ux = __fmul_rn(__fadd_rn(w.jx.x, w.jx.y), inv_rho);
  w.uy = __fmul_rn(__fadd_rn(w.jy.x, w.jy.y), inv_rho);
}

// 1/tau_s (Eq. taos) and 1/tau_d (Eq. EQFrsp with lambda_se = lambda_s
// Psi(y; lambda_s), lambda_s = (mu_s/p_s) sqrt(pi k_B T/(2 m_s)), p_s = x_s p),
// with the wall-confinement factor Psi(y) = (psi(y/lambda) + psi((H-y)/lambda))/2
// of the effective mean free path.  T: psi's table in shared memory.
__device__ __forceinline__ void rates2(const LatCore& L, const float4* T, const Macro2& m, float y,
                                       float& om_s, float& om_d) {
  const float rs_mx = rsqrt_fast(m.mx);
  const float lam = __fmul_rn(__fmul_rn(L.c_lam, m.inv_n), rs_mx);  // mixture mean free path
  const float inv_lam = __fmul_rn(__fmul_rn(L.inv_c_lam, m.n), __fmul_rn(m.mx, rs_mx));
  const float y2 = __fsub_rn(L.H, y);
  // 1 / lambda_s: n_s / c_xl with the partial pressure, n / c_xl with the
  // mixture pressure
  const float2 ns = mul2(m.rho, L.s2);
  const float2 inv_ls = mul2(L.lam_mix ? f2(m.n) : ns, L.inv_c_xl2);
  auto confined = [&](float il) {  // 2 Psi
    return __fadd_rn(psi_dev(T, __fmul_rn(y, il)), psi_dev(T, __fmul_rn(y2, il)));
  };
  const float pm = confined(inv_lam);
  const float2 ps = make_float2(confined(inv_ls.x), confined(inv_ls.y));
  // tau_s - 1/2 = lambda Psi c_ts / sqrt(m_x)
  const float tsm = __fmul_rn(__fmul_rn(lam, __fmul_rn(0.5f, pm)), L.c_ts);
  om_s = rcp_fast(fmaf(tsm, rs_mx, 0.5f));
  // x_s lambda_se = c_xl / n * Psi(y; lambda_s) (partial pressure), times
  // x_s = n_s / n with the mixture pressure
  const float2 xs = L.lam_mix ? mul2(ns, f2(m.inv_n)) : f2(1.0f);
  const float2 xle = mul2(mul2(mul2(L.c_xl2, f2(__fmul_rn(0.5f, m.inv_n))), xs), ps);
  const float br = __fadd_rn(rsqrt_fast(xle.x), rsqrt_fast(xle.y));
  // tau_d = 1/2 + c_td / (m_x br^2)  =>  1/tau_d = d / (d/2 + c_td), d = m_x br^2
  const float d = __fmul_rn(__fmul_rn(m.mx, br), br);
  om_d = __fmul_rn(d, rcp_fast(fmaf(0.5f, d, L.c_td)));
}

// MRT collision of both species at once (Eqs. MR, S, feq) on the deviations g from
// the rest equilibrium of the column reference, in moment space:
// f' = f - M^{-1} S (m - m^eq), M^{-1} = M^T diag(1/9, 1/36, 1/36, 1/6, 1/12,
// 1/6, 1/12, 1/4, 1/4), m^eq = rho_s (1, -4 + 2s + 3u^2, 4 - 3s - 3u^2, u_x,
// -u_x, u_y, -u_y, u_x^2 - u_y^2, u_x u_y).  The reference has m = m^eq(u=0),
// so e - e^eq = sum_i (e_i + 4 - 2s) g_i - 3 rho u^2 and
// eps - eps^eq = sum_i (eps_i - 4 + 3s) g_i + 3 rho u^2 need no large terms
// (ce2, cp2 hold those coefficients for the rest, axis and diagonal classes,
// times om_e / 36 and om_eps / 36, the classes' common factor in M^{-1}).
// Returns the x components of the species momenta of Eq. rhou,
// j_x - (j_x - rho_s u_x)/(2 tau_d).
__device__ __forceinline__ float2 collide2(float2 g[9], const LatCore& L, const Macro2& m, float om_d,
                                           float om_q, float om_s) {
  Flow2 w;
  flow2(g, m.inv_rho, w);
  const float ux = w.ux, uy = w.uy, uy2 = __fmul_rn(uy, uy);
  const float2 rho = m.rho;
  const float2 ru2 = mul2(f2(fmaf(ux, ux, uy2)), rho);
  const float2 a14 = add2(w.s13, w.s24), a58 = add2(w.s57, w.s68);
  const float2 de = fma2(L.ce2[0], g[0],
                         fma2(L.ce2[1], a14, fma2(L.ce2[2], a58, mul2(L.cu2[0], ru2))));
  const float2 dp = fma2(L.cp2[0], g[0],
                         fma2(L.cp2[1], a14, fma2(L.cp2[2], a58, mul2(L.cu2[1], ru2))));
  const float2 qx = fma2(f2(-2.0f), w.d13, w.dx);
  const float2 qy = fma2(f2(-2.0f), w.d24, w.dy);
  const float2 pxx = sub2(w.s13, w.s24), pxy = sub2(w.s57, w.s68);
  // relaxed moments over |M_k|^2: momenta om_d / 6, heat fluxes om_q / 12,
  // stresses om_s / 4
  const float2 od = f2(__fmul_rn(om_d, 1.0f / 6.0f)), oq = f2(__fmul_rn(om_q, 1.0f / 12.0f)),
               os = f2(__fmul_rn(om_s, 0.25f));
  const float2 Jx = mul2(od, fma2(rho, f2(-ux), w.jx));
  const float2 Jy = mul2(od, fma2(rho, f2(-uy), w.jy));
  const float2 Qx = mul2(oq, fma2(rho, f2(ux), qx));
  const float2 Qy = mul2(oq, fma2(rho, f2(uy), qy));
  const float2 pp = mul2(os, fma2(rho, f2(fmaf(-ux, ux, uy2)), pxx));
  const float2 pq = mul2(os, fma2(rho, f2(__fmul_rn(-ux, uy)), pxy));
  const float2 c14 = fma2(f2(2.0f), dp, de);  // axis class
  const float2 c58 = fma2(f2(2.0f), de, dp);  // minus the diagonal class
  const float2 ax = fma2(f2(-2.0f), Qx, Jx), ay = fma2(f2(-2.0f), Qy, Jy);
  const float2 bx = add2(Jx, Qx), by = add2(Jy, Qy);
  const float2 u1 = sub2(c14, pp), u2 = add2(c14, pp);  // shared by opposite axis pairs
  const float2 v5 = add2(c58, pq), v6 = sub2(c58, pq);  // and by opposite diagonal pairs
  const float2 w5 = add2(bx, by), w6 = sub2(bx, by);
  g[0] = fma2(f2(4.0f), sub2(de, dp), g[0]);
  g[1] = add2(g[1], sub2(u1, ax));
  g[3] = add2(g[3], add2(u1, ax));
  g[2] = add2(g[2], sub2(u2, ay));
  g[4] = add2(g[4], add2(u2, ay));
  g[5] = sub2(g[5], add2(v5, w5));
  g[7] = sub2(g[7], sub2(v5, w5));
  g[6] = sub2(g[6], sub2(v6, w6));
  g[8] = sub2(g[8], add2(v6, w6));
  return fma2(f2(-3.0f), Jx, w.jx);
}

// (A1, A2) of Eq. A12 from a wall node's accommodation coefficient.
__device__ __forceinline__ float2 slip_coefficients(float alpha) {
  const float A1 = __fmul_rn((2.0f - alpha) / alpha, fmaf(-0.1817f, alpha, 1.0f));
  return make_float2(A1, fmaf(__fmul_rn(0.5f, A1), A1, 1.0f / kPi));
}

// 1/tau_q of Eq. taoq from the wall node's n, 1/n and m_x (tau'_s(0) in its
// last term, dx = 1) and A = (A1, A2) of its accommodation coefficient.  P,
// D: the tables of psi and psi'.
__device__ __forceinline__ float inv_tau_q(const LatCore& L, const float4* P, const float4* D,
                                           float n, float inv_n, float mx, float2 A) {
  const float vs = 0.72360125455f;  // varsigma = sqrt(pi/6)
  const float rs_mx = rsqrt_fast(mx);
  const float lam = __fmul_rn(__fmul_rn(L.c_lam, inv_n), rs_mx);
  const float a = __fmul_rn(L.H, __fmul_rn(__fmul_rn(L.inv_c_lam, n), __fmul_rn(mx, rs_mx)));
  const float g = __fmul_rn(L.c_ts, rs_mx);  // sqrt(6/(pi m_x))
  const float tt = __fmul_rn(__fmul_rn(__fmul_rn(lam, 0.5f), psi_dev(P, a)), g);
  const float dtt = __fmul_rn(__fmul_rn(0.5f, g), __fsub_rn(2.0f, dpsi_dev(D, a)));
  const float tt2 = __fmul_rn(tt, tt);
  // tau_q = 1/2 + p / (16 tt) + dtt q / (16 tt^2) over one denominator
  const float p = fmaf(__fmul_rn(24.0f * vs * vs, tt2), A.y, 3.0f);
  const float q = fmaf(__fmul_rn(30.0f * vs, tt), A.x, 12.0f);
  const float num = fmaf(dtt, q, __fmul_rn(tt, p));
  const float den = __fmul_rn(16.0f, tt2);
  return den / fmaf(0.5f, den, num);
}

// r of Eq. R, r = 2 - 2/(1 + X), from the mixture molecular mass of the
// reflected post-collision state at the wall node, c_m = c_m0
// (2-alpha)/alpha, for both species: X = c_m sqrt(pi m_x/6) (first printed
// form, the same for both species; masses in units of m_min), c_m sqrt(pi
// m_x/(6 m_s)) (m_min replaced by the species mass) or c_m sqrt(pi m_x^2/(6
// m_s)) (second printed form, m_r = m_s/m_x).  With the BSR wall the
// bounce-back fraction 1/(1 + X) of the same slip factor X.
__device__ __forceinline__ float slip_cm(const LatCore& L, float alpha) {
  return __fmul_rn(L.c_m0, __fsub_rn(2.0f, alpha)) / alpha;
}
__device__ __forceinline__ float2 slip_r(const LatCore& L, float rho_a, float rho_b, float cm) {
  const float mx = __fadd_rn(rho_a, rho_b) / number_density(L, rho_a, rho_b);
  const float q = sqrtf(__fmul_rn(kPi / 6.0f, mx));
  float X0 = __fmul_rn(cm, q);
  if (L.r_form == LBM_R_SECOND) X0 = __fmul_rn(X0, sqrtf(mx));
  float r[2];
#pragma unroll
  for (int sp = 0; sp < 2; ++sp) {
    // 1 + X with one rounding
    const float den =
        L.r_form == LBM_R_FIRST ? fmaf(cm, q, 1.0f) : fmaf(X0, L.rsqrt_mh[sp], 1.0f);
    r[sp] = L.wall_mode == LBM_WALL_BSR ? 1.0f / den : __fsub_rn(2.0f, 2.0f / den);
  }
  return make_float2(r[0], r[1]);
}
template <typename ST>
__device__ __forceinline__ float2 dbb_r(const Lat& L, const ColRef& C, const ST* __restrict__ f,
                                        int x, int j, float alpha) {
  float rho[2];
#pragma unroll
  for (int sp = 0; sp < 2; ++sp) {
    float acc = 0.0f;
#pragma unroll
    for (int i = 0; i < 9; ++i) acc += ld(f, L, sp, i, j, x);
    rho[sp] = C.rb[sp] + acc;
  }
  return slip_r(L, rho[0], rho[1], slip_cm(L, alpha));
}

// A sum of two floats, hi + lo with |lo| <= ulp(hi) / 2: 48 bits of the
// slow FP64 pipe's work in a few FP32 operations.
__device__ __forceinline__ float2 split_double(double v) {
  const float hi = (float)v;
  return make_float2(hi, (float)(v - (double)hi));
}
// a + b with its rounding error (Knuth's two-sum).
__device__ __forceinline__ float2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}
// The same for |a| >= |b| (Dekker).
__device__ __forceinline__ float2 quick_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return make_float2(s, __fsub_rn(b, __fsub_rn(s, a)));
}

// kappa = mass / (2 c1 - c2) of one species at one end (Eq. rho2; mass = N
// rho_end) from the column sums c1, c2 of the two columns next to it, and the
// ghost reference offset kappa (2 r1 - r2) - r0.  In float pairs: sixteen
// dependent FP64 operations took 2400 cycles, this takes under 200, and its
// error (2^-44) vanishes in the rounding of the results to FP32.
__device__ __forceinline__ void end_factors(float2 mass, float2 c1, float2 c2, float r0, float r1,
                                            float r2, float& kappa, float& offset) {
  float2 D = two_sum(__fmul_rn(2.0f, c1.x), -c2.x);
  D = quick_two_sum(D.x, __fadd_rn(D.y, fmaf(2.0f, c1.y, -c2.y)));
  const float inv = rcp_fast(D.x);
  const float q = __fmul_rn(mass.x, inv);
  const float rest = __fadd_rn(fmaf(-q, D.x, mass.x), fmaf(-q, D.y, mass.y));
  const float2 k = quick_two_sum(q, __fmul_rn(rest, inv));
  const float2 R = two_sum(__fmul_rn(2.0f, r1), -r2);
  const float p = __fmul_rn(k.x, R.x);
  const float pl = __fadd_rn(fmaf(k.x, R.x, -p), fmaf(k.x, R.y, __fmul_rn(k.y, R.x)));
  const float2 o = two_sum(p, -r0);
  kappa = k.x;
  offset = __fadd_rn(o.x, __fadd_rn(o.y, pl));
}

// Density-correction factors of Eq. rho2 for the ghost columns, from the
// column sums of the state being streamed, and the ghost reference offsets;
// only a block whose columns [x0, x0 + width) hold column 1 or column
// N_x - 2 reads them (the others keep kappa = 1, which they never use).
__device__ __forceinline__ Ends load_ends(const Lat& L, const double* __restrict__ cs,
                                          const float* __restrict__ refrho, int x0, int width) {
  Ends E;
#pragma unroll
  for (int sp = 0; sp < 2; ++sp) {
    E.kin[sp] = E.kout[sp] = 1.0f;
    E.gin[sp] = E.gout[sp] = 0.0f;
  }
  if (L.x_periodic) return E;
  const int Nx = L.Nx;
#pragma unroll
  for (int sp = 0; sp < 2; ++sp) {
    const double* c = cs + (size_t)sp * Nx;
    const float* r = refrho + sp * Nx;
    if (x0 <= 1 && 1 < x0 + width)
      end_factors(L.end_mass[0][sp], split_double(c[1]), split_double(c[2]), r[0], r[1], r[2],
                  E.kin[sp], E.gin[sp]);
    if (x0 <= Nx - 2 && Nx - 2 < x0 + width)
      end_factors(L.end_mass[1][sp], split_double(c[Nx - 2]), split_double(c[Nx - 3]), r[Nx - 1],
                  r[Nx - 2], r[Nx - 3], E.kout[sp], E.gout[sp]);
  }
  return E;
}

__device__ __forceinline__ bool interior(const LatCore& L, int x) {
  return L.x_periodic ? (x < L.Nx) : (x >= 1 && x <= L.Nx - 2);
}

#include "lbm_node16.cuh"

// The density-correction factors in the storage form's arithmetic.
template <typename ST>
__device__ __forceinline__ Ends ends_of(const Lat& L, const double* __restrict__ cs,
                                        const float* __restrict__ refrho, int x0, int width) {
  if constexpr (sizeof(ST) < 4) return n16::load_ends(L, cs, refrho, x0, width);
  else return load_ends(L, cs, refrho, x0, width);
}

// Per-CTA wall data for the strip: r (both walls), 1/tau_q (both walls).
struct WallSmem {
  float2 r[2][TX];  // (species a, species b) per wall and column
  float om_q[2][TX];
};

// Prologue of the step and moments kernels for the CTA's rows
// [j_begin, j_end): r of a wall is needed only by the CTA that holds that
// wall's row, 1/tau_q of a wall only by CTAs with rows in that wall's half.
// The four tasks run on four warps at once (ty = 0, 1: r of the bottom and
// top wall; ty = 2, 3: their tau_q).  tau_q depends on the wall node's
// pre-collision species densities only (through lambda and m_x), and the
// DBB rule conserves each species' mass at the node whatever r is, so the
// tau_q warps pull the wall node with r = 0 and need not wait for r (the
// BSR rule moves mass between columns: there they evaluate r themselves).
// One wall task of column x: r of wall `wall` (tq false) or 1/tau_q of
// its half (tq true), from the post-collision state fin of the step about
// to run.  Columns outside the interior get r = 1 and 1/tau_q = 1 (unused).
template <typename ST>
__device__ __forceinline__ void wall_task(const Lat& L, const ST* __restrict__ fin,
                                          const float* __restrict__ alpha, const Ends& E,
                                          const ColRef& C, int x, int wall, bool tq, float2& rv,
                                          float& v) {
  v = 1.0f;
  rv = make_float2(1.0f, 1.0f);
  if (!interior(L, x)) return;
  const int jw = wall == 0 ? 0 : L.N - 1;
  const float al = alpha[wall * L.Nx + x];
  auto r_of = [&]() -> float2 {
    if constexpr (sizeof(ST) < 4) return n16::dbb_r(L, C, fin, x, jw, al);
    else return dbb_r(L, C, fin, x, jw, al);
  };
  if (!tq) {
    rv = r_of();
  } else {
    float fs[2][9];
    const float2 rr = L.wall_mode == LBM_WALL_BSR ? r_of() : make_float2(0.0f, 0.0f);
    pull_node(fin, L, E, C, x, jw, rr, rr, fs);
    if constexpr (sizeof(ST) < 4) {
      n16::Macro m;
      n16::macro(L, C, fs, m);
      v = 1.0f / n16::tau_q_wall(L, m, al);
    } else {
      Macro m;
      macro(L, C, fs, m);
      v = inv_tau_q(L, kPsiTab, kDpsiTab, m.n, m.inv_n, m.mx, slip_coefficients(al));
    }
  }
}

template <bool WITH_TQ, typename ST>
__device__ __forceinline__ void wall_prologue(const Lat& L, const ST* __restrict__ fin,
                                              const float* __restrict__ alpha, const Ends& E,
                                              const ColRef& C, int x, int j_begin, int j_end,
                                              WallSmem& sm) {
  const int tx = threadIdx.x, ty = threadIdx.y;
  if (ty < (WITH_TQ ? 4 : 2)) {
    const int wall = ty & 1;
    const bool tq = ty >= 2;
    const int half = (L.N + 1) / 2;  // rows j < half use the bottom tau_q
    const bool needed = tq ? (wall == 0 ? j_begin < half : j_end > half)
                           : (wall == 0 ? j_begin == 0 : j_end == L.N);
    float v = 1.0f;
    float2 rv = make_float2(1.0f, 1.0f);
    if (needed) wall_task(L, fin, alpha, E, C, x, wall, tq, rv, v);
    if (tq)
      sm.om_q[wall][tx] = v;
    else
      sm.r[wall][tx] = rv;
  }
  __syncthreads();
}

// The wall tasks of every column as a kernel of their own, ahead of the step
// kernel (16-bit storage, and FP32 grids of several waves): the prologue's
// barrier held the CTA's other warps up while the tau_q warps waited on
// their loads (8 % of the 16-bit step, 4 % of the FP32 step).
// One thread per column and task (blockIdx.y: 0, 1 = r of the bottom, top
// wall; 2, 3 = 1/tau_q of the bottom, top half): r_out [2][Nx] (species
// pair), omq_out [2][Nx].
constexpr int WALL_COLS = 128;  // columns of a block
template <typename ST>
__device__ __forceinline__ void walls_cta(const Lat& L, int block, int task,
                                          const ST* __restrict__ fin,
                                          const float* __restrict__ refrho,
                                          const double* __restrict__ cs_in,
                                          const float* __restrict__ alpha,
                                          float2* __restrict__ r_out,
                                          float* __restrict__ omq_out) {
  pdl_launch_dependents();
  pdl_wait();
  const int x = block * WALL_COLS + threadIdx.x;
  if (x >= L.Nx) return;
  const int wall = task & 1;
  const bool tq = task >= 2;
  const ColRef C = col_ref(L, refrho, x);
  const Ends E = ends_of<ST>(L, cs_in, refrho, block * WALL_COLS, WALL_COLS);
  float2 rv;
  float v;
  wall_task(L, fin, alpha, E, C, x, wall, tq, rv, v);
  if (tq)
    omq_out[wall * L.Nx + x] = v;
  else
    r_out[wall * L.Nx + x] = rv;
}
template <typename ST>
__global__ void __launch_bounds__(WALL_COLS)
    lbm_walls_kernel(Lat L, const ST* __restrict__ fin, const float* __restrict__ refrho,
                     const double* __restrict__ cs_in, const float* __restrict__ alpha,
                     float2* __restrict__ r_out, float* __restrict__ omq_out) {
  walls_cta(L, blockIdx.x, blockIdx.y, fin, refrho, cs_in, alpha, r_out, omq_out);
}

// Running sum with the rounding error of every addition kept (Knuth's two-sum).
// (Kahan's form, one operation less, loses the bits of the running sum below a
// larger term's last: 1e-8 of a column's deviations.  Its four operations are
// also one chain, of these six only the sum's own is.)
struct Sum1 {
  float s = 0.0f, e = 0.0f;
  __device__ __forceinline__ void add(float v) {
    const float2 t = two_sum(s, v);
    e = __fadd_rn(e, t.y);
    s = t.x;
  }
};

// Two of them, packed, in seven instructions: a thread's partials over its rows
// of one column, handed to column_epilogue.
struct Sum2 {
  float2 s = {0.0f, 0.0f}, e = {0.0f, 0.0f};
  __device__ __forceinline__ void add(float2 v) {
    const float2 t = add2(s, v), b = sub2(t, s);
    e = add2(e, add2(sub2(s, sub2(t, b)), sub2(v, b)));
    s = t;
  }
};

// Sum of two (sum, error) pairs of floats, to about 2^-46 of its larger terms.
__device__ __forceinline__ float2 pair_add(float2 a, float2 b) {
  const float2 s = two_sum(a.x, b.x);
  return quick_two_sum(s.x, __fadd_rn(s.y, __fadd_rn(a.y, b.y)));
}

// Sum of v(0) .. v(N - 1), the rows of a column, by eight neighbouring lanes
// (sub = lane & 7, every lane of the warp here): each takes every eighth row in
// order, then three additions, all error-free but for the errors' own sum.
// Every lane of the eight gets the same (sum, error) pair.
template <typename V>
__device__ __forceinline__ float2 column_sum8(int N, int sub, V&& v) {
  Sum1 a;
  for (int j = sub; j < N; j += 8) a.add(v(j));
  float hi = a.s, lo = a.e;
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
    const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
    const float2 s = two_sum(hi, h2);
    lo = __fadd_rn(__fadd_rn(lo, l2), s.y);
    hi = s.x;
  }
  return make_float2(hi, lo);
}
__device__ __forceinline__ double pair_value(float2 v) { return (double)v.x + (double)v.y; }

// N ref + (sum of deviations) as a float pair whose low part is cut at 2^-48
// of the high one, so that its FP64 value splits into the same pair again: a
// launch that starts from the stored FP64 sums continues bit for bit.
__device__ __forceinline__ float2 column_total(int N, float ref, float2 dev) {
  const float n = (float)N, p = __fmul_rn(n, ref), pl = fmaf(n, ref, -p);
  float2 s = two_sum(p, dev.x);
  s = quick_two_sum(s.x, __fadd_rn(s.y, __fadd_rn(pl, dev.y)));
  const float grid = __fmul_rn(s.x, 0x1p-24f);
  return make_float2(s.x, __fsub_rn(__fadd_rn(s.y, grid), grid));
}

// ------------------------------------------------------------ step kernel
// Random bits of the stochastic rounding: a 32-bit integer hash (the
// "lowbias32" xorshift-multiply hash of C. Wellons) seeds one linear
// congruential generator per thread and launch (multiplier 1664525 and
// increment 1013904223, the quick generator of Numerical Recipes), whose
// state is folded (high half into the low half) so that both 16-bit halves
// of each word are usable.
__device__ __forceinline__ unsigned hash32(unsigned x) {
  x ^= x >> 16;
  x *= 0x7feb352du;
  x ^= x >> 15;
  x *= 0x846ca68bu;
  x ^= x >> 16;
  return x;
}
__device__ __forceinline__ unsigned lcg_next(unsigned& s) {
  s = s * 1664525u + 1013904223u;
  return s ^ (s >> 16);
}

// Rows of one sequence of the stochastic rounding: a thread's generator is
// seeded anew every RNG_ROWS rows and takes nine numbers per row it visits
// (every TY-th), so a node's random bits depend on its place and the step
// alone, not on the rows per CTA.
constexpr int RNG_ROWS = 96;
static_assert(RNG_ROWS % TY == 0, "a thread's rows meet a seeding row");
// Nine steps of lcg_next's congruence at once: s -> A9 s + C9.
struct Lcg9 {
  unsigned a = 1u, c = 0u;
  constexpr Lcg9() {
    for (int k = 0; k < 9; ++k) {
      a *= 1664525u;
      c = c * 1664525u + 1013904223u;
    }
  }
};

template <typename ST>
struct StepArgs {
  const ST* __restrict__ fin;     // post-collision deviations of step t-1
  ST* __restrict__ fout;          // post-collision deviations of step t
  const float* __restrict__ refrho;  // [2][Nx] reference densities
  const double* __restrict__ cs_in;  // [4][Nx] column sums of the state in fin
  double* __restrict__ cs_out;       // [4][Nx] column sums of the state of step t
  const float* __restrict__ alpha;   // [2][Nx]
  double* __restrict__ partials;     // [NPART][strips]
  unsigned* __restrict__ counter;
  double* __restrict__ diag;         // [DIAG_CAP][NREC]
  unsigned long long* __restrict__ diag_count;
  double* __restrict__ clprof;       // [Nx]
  float2* __restrict__ colpart;      // [R][4][Nx] per-row-block column sums (R > 1)
  unsigned* __restrict__ strip_cnt;  // [strips] row blocks finished this step
  int rows_per_block;                // rows of one row block (multiple of TY)
  unsigned seed;                     // 16-bit storage: per-step seed of the
                                     // stochastic rounding; 0 = round to nearest
  // r and 1/tau_q of every column from lbm_walls_kernel ([2][Nx] each,
  // bottom then top), in place of the wall prologue (WK kernels only)
  const float2* __restrict__ wall_r;
  const float* __restrict__ wall_omq;
  // [4][N] density deviations of columns 1, 2, Nx - 2, Nx - 3 (FP32 storage
  // with pressure ends; null: their sums come from the row blocks like all
  // others)
  float2* __restrict__ end_sd;
};

struct RedSmem {
  float2 col[4][TY][TX];
  double total[4][TX];
  double sum[NPART];
  int last;
  int last_strip;
};

// Warp-level FP64 sum and (min, argmin) with ties to the smaller column.
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ void warp_min(double& v, int& idx) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    double ov = __shfl_xor_sync(0xffffffffu, v, o);
    int oi = __shfl_xor_sync(0xffffffffu, idx, o);
    if (ov < v || (ov == v && oi < idx)) {
      v = ov;
      idx = oi;
    }
  }
}

// g: the CTA's place in its channel's grid.
struct GridPos {
  int strip, block;     // strip and row block of this CTA
  int strips, blocks;   // of the channel
};
// The place of CTA b of a channel: the row blocks of the two end strips first,
// then the other strips, row block by row block (the shorter last ones fill
// the tail of the launch).  The end strips also reduce their column sums at
// every step, a chain of some microseconds; last in the grid, it and their
// rows were a tail of 14 us of a 107 us step (BF16 16384 x 256) and of 9 us of
// 27 us (FP16 5001 x 130).
__device__ __forceinline__ GridPos grid_pos(const LatCore& L, int b, int strips, int blocks) {
  if (L.x_periodic || strips < 3) return GridPos{b % strips, b / strips, strips, blocks};
  const int inner = strips - 2, r = b - 2 * blocks;
  if (r < 0) return GridPos{(b & 1) ? strips - 1 : 0, b >> 1, strips, blocks};
  return GridPos{1 + r % inner, r / inner, strips, blocks};
}
// Most rows whose end columns column_sum8 adds up, eight lanes a column, as in
// lbm_tile_kernel (whose tiles hold at most 424 rows); beyond, all threads of
// the CTA take a column after the other, 256 rows at a time.
constexpr int END_ROWS = 512;
// Column sums -> next step's density correction, C_l(x), per-strip partials;
// the last CTA to finish reduces the partials in strip order into one record.
// DIAG = false (end strips only): the sums that the next step's Eq. rho2 needs,
// with FP32 storage those of the four end columns alone; DIAG = true: those of
// every column, C_l(x), the per-strip partials and the record.
// Every CTA of a DIAG step comes here, and an FP64 instruction holds its SM
// sub-partition for some 64 cycles; the sums of a CTA are therefore pairs of
// floats, by one warp per quantity, and FP64 begins at the strip's totals.
// Sums in FP64 throughout, most of them in one warp, cost a DIAG step of
// 32768 x 512 80 us beyond the others (45 now, mostly the fence and the ticket
// of each CTA), one of 5001 x 130 29 us (14).
// A channel of many rows has long chains here, in one CTA a strip: the row
// blocks' sums (a hundred cycles a block) and the end columns' rows.  All rows
// by eight lanes a column and the row blocks at every step took 188 us per step
// of 64 x 16384, 606 of 64 x 65536 (one row block of 512: 17.2); whole CTAs for
// the end columns and row blocks at DIAG steps alone 60, 188 (13.5).
template <bool DIAG, typename ST>
__device__ __forceinline__ void column_epilogue(const Lat& L, const StepArgs<ST>& a,
                                                const GridPos& gp, int x, const Sum2 acc[2],
                                                RedSmem& rs) {
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int tid = ty * TX + tx;
  const int R = gp.blocks;  // row blocks per strip
  const bool in = interior(L, x);
  // sums of all of the strip's columns; otherwise of the end columns alone,
  // whose rows are in end_sd (FP32 storage: the strips are then end strips)
  constexpr bool SUMS = DIAG || sizeof(ST) < 4;
  float2 c = make_float2(0.0f, 0.0f);  // quantity ty of column x, in warps 0 .. 3
  if constexpr (SUMS) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      rs.col[2 * k][ty][tx] = make_float2(acc[k].s.x, acc[k].e.x);
      rs.col[2 * k + 1][ty][tx] = make_float2(acc[k].s.y, acc[k].e.y);
    }
    __syncthreads();
    if (ty < 4) {
      c = rs.col[ty][0][tx];
#pragma unroll
      for (int t = 1; t < TY; ++t) c = pair_add(c, rs.col[ty][t][tx]);
    }
  }
  if (R > 1) {
    // Row-block partials of this strip; the last of its R CTAs to finish
    // adds them in row-block order (independent of arrival order).  A fence
    // after a barrier, by the thread that takes the ticket too, publishes what
    // the CTA's threads wrote before that barrier (the rows of end_sd).
    if (SUMS && ty < 4) {
      if (x < L.Nx) a.colpart[((size_t)gp.block * 4 + ty) * L.Nx + x] = c;
      __threadfence();
    }
    __syncthreads();
    if (tid == 0) {
      if (!SUMS) __threadfence();
      unsigned ticket = atomicAdd(a.strip_cnt + gp.strip, 1u);
      rs.last_strip = (ticket == (unsigned)R - 1u);
    }
    __syncthreads();
    if (!rs.last_strip) return;
    __threadfence();
    if (SUMS && ty < 4 && x < L.Nx) {
      const float2* cp = a.colpart + (size_t)ty * L.Nx + x;
      c = __ldcg(cp);
#pragma unroll 4
      for (int r = 1; r < R; ++r) c = pair_add(c, __ldcg(cp + (size_t)r * 4 * L.Nx));
    }
    if (tid == 0) a.strip_cnt[gp.strip] = 0u;
  }
  if (SUMS && ty < 4) {
    // column sum of rho_s = N rhobar_s + sum of deviations
    double v = pair_value(c);
    if (ty < 2 && in) v += (double)L.N * (double)a.refrho[ty * L.Nx + x];
    rs.total[ty][tx] = v;
  }
  if (sizeof(ST) == 4 && a.end_sd) {
    // The columns behind the next step's density correction, in an order that
    // depends on N alone: the populations of a run are then the same bits under
    // every schedule, this kernel's and lbm_tile_kernel's.  e: which column.
    auto end_column = [&](int e) {
      return e == 0 ? 1 : e == 1 ? 2 : e == 2 ? L.Nx - 2 : L.Nx - 3;
    };
    const int x0 = x - tx;
    // the sum over end column x of species sp, from that of its deviations
    auto put = [&](int sp, float2 v) {
      const double t = pair_value(column_total(L.N, a.refrho[sp * L.Nx + x], v));
      if constexpr (SUMS)
        rs.total[sp][tx] = t;
      else
        a.cs_out[(size_t)sp * L.Nx + x] = t;
    };
    __syncthreads();
    if (L.N <= END_ROWS) {
      // as lbm_tile_kernel does; one warp for each column and species
      const int e = ty >> 1, sp = ty & 1, xe = end_column(e);
      if (xe >= x0 && xe < x0 + TX) {  // warp-uniform
        const float2 v = column_sum8(L.N, tx & 7, [&](int r) {
          const float2 d = __ldcg(a.end_sd + (size_t)e * L.N + r);
          return sp ? d.y : d.x;
        });
        if (x == xe) put(sp, v);
      }
    } else {
      // the whole CTA, one column after another
      for (int e = 0; e < 4; ++e) {
        const int xe = end_column(e);
        if (xe < x0 || xe >= x0 + TX) continue;  // CTA-uniform
        const float2* d = a.end_sd + (size_t)e * L.N;
        Sum2 v;
#pragma unroll 8
        for (int r = tid; r < L.N; r += TX * TY) v.add(__ldcg(d + r));
        float2 pa = make_float2(v.s.x, v.e.x), pb = make_float2(v.s.y, v.e.y);
#pragma unroll
        for (int o = 1; o < TX; o <<= 1) {
          pa = pair_add(pa, make_float2(__shfl_xor_sync(0xffffffffu, pa.x, o),
                                        __shfl_xor_sync(0xffffffffu, pa.y, o)));
          pb = pair_add(pb, make_float2(__shfl_xor_sync(0xffffffffu, pb.x, o),
                                        __shfl_xor_sync(0xffffffffu, pb.y, o)));
        }
        if (tx == 0) {
          rs.col[0][ty][0] = pa;
          rs.col[1][ty][0] = pb;
        }
        __syncthreads();
        if (ty < 2 && x == xe) {
          float2 t = rs.col[ty][0][0];
          for (int w = 1; w < TY; ++w) t = pair_add(t, rs.col[ty][w][0]);
          put(ty, t);
        }
        __syncthreads();
      }
    }
    __syncthreads();
  }
  // (a warp writes back the totals that it formed itself, or all have met)
  if (SUMS && ty < 4 && x < L.Nx) a.cs_out[(size_t)ty * L.Nx + x] = rs.total[ty][tx];
  if (!DIAG) return;
  __syncthreads();
  // The strip's partials: a quantity's sum over the columns in each of four
  // warps, C_l in a fifth.
  double* p = a.partials + gp.strip;
  if (ty < 4) {
    const double v = warp_sum(in ? rs.total[ty][tx] : 0.0);
    if (tx == 0) p[(size_t)(ty < 2 ? 5 + ty : 1 + ty) * gp.strips] = v;
  } else if (ty == 4) {
    double Cl = 0.0;
    if (in) {
      double na = rs.total[0][tx] * L.s[0], nb = rs.total[1][tx] * L.s[1];
      Cl = (L.light == 0 ? na : nb) / (na + nb);
      a.clprof[x] = Cl;
    } else if (x < L.Nx) {
      a.clprof[x] = (x == 0) ? L.C_in : L.C_out;
    }
    double vmin = in ? Cl : INFINITY;
    int imin = in ? x : 0x7fffffff;
    warp_min(vmin, imin);
    const double dev = warp_sum(in ? Cl - L.C_in : 0.0);
    const int cols = __popc(__ballot_sync(0xffffffffu, in));
    if (tx == 0) {
      p[0] = vmin;
      p[(size_t)1 * gp.strips] = (double)imin;
      p[(size_t)2 * gp.strips] = dev;
      p[(size_t)7 * gp.strips] = (double)cols;
    }
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    unsigned ticket = atomicAdd(a.counter, 1u);
    rs.last = (ticket == (unsigned)gp.strips - 1u);
  }
  __syncthreads();
  if (!rs.last) return;
  __threadfence();
  // Last CTA: each warp folds one partial over the strips, every lane a fixed
  // subset in strip order, then a fixed shuffle tree, so the result does not
  // depend on which CTA finished last.
  static_assert(TY == NPART, "a warp per partial");
  if (ty == 0) {
    double vmin = INFINITY;
    int imin = 0x7fffffff;
    for (int b = tx; b < gp.strips; b += TX) {
      const double v = __ldcg(a.partials + b);
      const int i = (int)__ldcg(a.partials + gp.strips + b);
      if (v < vmin || (v == vmin && i < imin)) {
        vmin = v;
        imin = i;
      }
    }
    warp_min(vmin, imin);
    if (tx == 0) {
      rs.sum[0] = vmin;
      rs.sum[1] = (double)imin;
    }
  } else if (ty != 1) {
    double v = 0.0;
    for (int b = tx; b < gp.strips; b += TX) v += __ldcg(a.partials + (size_t)ty * gp.strips + b);
    v = warp_sum(v);
    if (tx == 0) rs.sum[ty] = v;
  }
  __syncthreads();
  if (tid < NREC) {
    const unsigned long long cnt = *a.diag_count + 1ull;
    double dev = rs.sum[2];
    if (!L.x_periodic) dev += (L.C_out - L.C_in);  // the outlet boundary column
    const double ncol = rs.sum[7];
    // one division for all eight entries
    double num = 0.0, den = 1.0;
    switch (tid) {
      case 0: num = (double)cnt; break;
      case 1: num = L.C_in - rs.sum[0], den = L.C_in; break;
      case 2: num = dev, den = (double)L.Nx * L.C_in; break;
      case 3: num = rs.sum[3], den = ncol; break;
      case 4: num = rs.sum[4], den = ncol; break;
      case 5: num = rs.sum[1]; break;
      case 6: num = rs.sum[5]; break;
      case 7: num = rs.sum[6]; break;
    }
    a.diag[(size_t)((cnt - 1ull) % DIAG_CAP) * NREC + tid] = num / den;
    __syncwarp((1u << NREC) - 1u);
    if (tid == 0) {
      *a.diag_count = cnt;
      *a.counter = 0u;
    }
    __threadfence();
  }
}

// DIAG: reduce the separation diagnostics of the new state (every
// diag_every-th step); otherwise only the strips holding the end columns
// reduce the column sums the next step's density correction needs.
// WK: r and 1/tau_q of the columns come from lbm_walls_kernel, launched
// ahead of the step (always with 16-bit storage), instead of the CTA's wall
// prologue.
template <typename ST, bool WK>
__device__ __forceinline__ void step_cta(const Lat& L, const StepArgs<ST>& a, const GridPos& gp,
                                         bool diag) {
  __shared__ WallSmem wsm;
  __shared__ RedSmem rsm;
  constexpr bool FP32 = sizeof(ST) == 4;
  __shared__ float4 psi_tab[FP32 ? PSI_SEGMENTS : 1];
  const int tx = threadIdx.x, ty = threadIdx.y;
  if (FP32) load_psi_table(psi_tab, ty * TX + tx, TX * TY);  // overlaps the kernel before
  pdl_wait();
  const int x0 = gp.strip * TX, x = x0 + tx;
  const ColRef C = col_ref(L, a.refrho, x);
  const Ends E = ends_of<ST>(L, a.cs_in, a.refrho, gp.strip * TX, TX);
  const int j_begin = gp.block * a.rows_per_block;
  const int j_end = min(L.N, j_begin + a.rows_per_block);
  // the first row of each warp is on its way into L2 while the wall prologue
  // (if any) runs
  if (tx == 0 && j_begin + ty < j_end)
    prefetch_row_l2(a.fin + (size_t)gp.strip * L.SS + (size_t)(j_begin + ty) * RS);
  // r and 1/tau_q of this column: from lbm_walls_kernel (WK, read where they
  // are used) or from the CTA's wall prologue
  const int xc = x < L.Nx ? x : L.Nx - 1;
  if constexpr (!WK)
    wall_prologue<true>(L, a.fin, a.alpha, E, C, x, j_begin, j_end, wsm);
  else if (FP32)
    __syncthreads();  // psi's table
  auto wall_r = [&](int w) -> float2 {
    if constexpr (WK) return a.wall_r[w * L.Nx + xc];
    else return wsm.r[w][tx];
  };
  auto wall_omq = [&](int h) -> float {
    if constexpr (WK) return a.wall_omq[h * L.Nx + xc];
    else return wsm.om_q[h][tx];
  };
  const bool in = interior(L, x);
  // strips holding one of the columns 1, 2, N_x - 3, N_x - 2 take the general
  // pull (ghost columns) and reduce their column sums at every step
  const bool edge_strip = !L.x_periodic && (x0 <= 2 || x0 + TX > L.Nx - 3);
  const int end_l = x == 1 ? 0 : x == 2 ? 1 : -1;
  const int end_r = x == L.Nx - 2 ? 2 : x == L.Nx - 3 ? 3 : -1;
  int xm = x - 1, xp = x + 1;
  if (xm < 0) xm += L.Nx;
  if (xp >= L.Nx) xp -= L.Nx;
  const unsigned base = gp.strip * L.SS + 2 * tx;  // row 0, i = 0, species a of column x
  const int offl = (int)(idx(L, 0, 0, 0, xm) - base), offr = (int)(idx(L, 0, 0, 0, xp) - base);
  const int half = (L.N + 1) / 2;  // rows j < half (1-based 2J <= N+1) use the bottom tau_q
  Sum2 acc[2];  // species densities, species x momenta
  const bool reduce = diag || edge_strip;
  unsigned rng = 0u;  // generator of the stochastic rounding
  // one run over the rows, with 16-bit storage one per sequence of random bits
  for (int js = j_begin, je; in && js < j_end; js = je) {
    je = j_end;
    if (!FP32 && a.seed != 0u) {
      constexpr Lcg9 jump;
      const int block = js / RNG_ROWS;
      je = min(j_end, (block + 1) * RNG_ROWS);
      rng = hash32(a.seed ^ hash32((block * gp.strips + gp.strip) * (TX * TY) + ty * TX + tx));
      for (int r = (js - block * RNG_ROWS) / TY; r > 0; --r) rng = rng * jump.a + jump.c;
    }
    for (int j = js + ty; j < je; j += TY) {
      float2 g[9];
      const ST* p = a.fin + base + j * RS;
      // row start is 16-byte aligned (RS * sizeof(ST) is a multiple of 16);
      // the prefetched row lies inside this strip (j + TY < j_end <= N)
      if (tx == 0 && j + TY < j_end) prefetch_row_l2(p + TY * RS);
      if (!edge_strip && j != 0 && j != L.N - 1) {
        pull_fast(p, p + offl, p + offr, L, C, g);
      } else if (j != 0 && j != L.N - 1) {
        pull_edge(a.fin, p, p + offl, p + offr, L, E, C, x, j, g);
      } else {
        float fs[2][9];
        pull_node(a.fin, L, E, C, x, j, wall_r(0), wall_r(1), fs);
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = make_float2(fs[0][i], fs[1][i]);
      }
      float2 sd, mxs;
      float om_s, om_d;
      if constexpr (FP32) {
        Macro2 m;
        macro2(L, make_float2(C.rb[0], C.rb[1]), g, m);
        rates2(L, psi_tab, m, (float)j + 0.5f, om_s, om_d);
        const float om_q = wall_omq(j < half ? 0 : 1);
        mxs = collide2(g, L, m, om_d, om_q, om_s);
        sd = m.sd;
      } else {
        n16::Macro2 m;
        n16::macro2(L, C, g, m);
        n16::rates2(L, m, (float)j + 0.5f, om_s, om_d);
        const float om_q = wall_omq(j < half ? 0 : 1);
        mxs = n16::collide2(g, L, m.rho, m.ux, m.uy, L.om_e, L.om_eps, om_d, om_q, om_s);
        sd = m.sd;
      }
      if (FP32 && edge_strip && a.end_sd) {
        if (end_l >= 0) a.end_sd[end_l * L.N + j] = sd;
        if (end_r >= 0) a.end_sd[end_r * L.N + j] = sd;
      }
      if (FP32 ? diag : reduce) {
        acc[0].add(sd);
        acc[1].add(mxs);
      }
      ST* o = a.fout + base + j * RS;
      if (sizeof(ST) < 4 && a.seed != 0u) {
#pragma unroll
        for (int i = 0; i < 9; ++i) Stor<ST>::st2_sr(o + i * PS, g[i], lcg_next(rng));
      } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) Stor<ST>::st2(o + i * PS, g[i]);
      }
    }
  }
  if (!reduce) return;  // CTA-uniform
  if (diag)
    column_epilogue<true>(L, a, gp, x, acc, rsm);
  else
    column_epilogue<false>(L, a, gp, x, acc, rsm);
}

template <typename ST, bool DIAG, bool WK = (sizeof(ST) < 4)>
__global__ void __launch_bounds__(TX* TY, 3) lbm_step_kernel(Lat L, StepArgs<ST> a) {
  const GridPos gp =
      grid_pos(L, blockIdx.y * gridDim.x + blockIdx.x, (int)gridDim.x, (int)gridDim.y);
  step_cta<ST, WK>(L, a, gp, DIAG);
}

// The channel whose CTAs [block0[q], block0[q + 1]) hold b, by bisection.
template <int NI>
__device__ __forceinline__ int channel_of(const int* block0, int b) {
  int lo = 0, hi = NI;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (b >= block0[mid])
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

// One step of several channels (FP32 storage) as one launch: the CTAs of
// channel q are [block0[q], block0[q + 1]), strips fastest, as in the channel's
// own grid.  A sweep of 52 channels of 700 x 20 spent 147 us per step on 52
// launches from as many graphs, 2.8 us each.  WK: r and 1/tau_q come from
// lbm_walls_batch_kernel ahead of it, blocks of it first channel first too.
struct StepInst {
  Lat L;
  StepArgs<float> a;
  float2* wall_r;
  float* wall_omq;
  int strips, blocks, diag;
};
template <int NI>
struct StepBatch {
  int block0[NI + 1], wall0[NI + 1];
  StepInst inst[NI];
};
template <int NI, bool WK>
__global__ void __launch_bounds__(TX* TY, 3)
    lbm_step_batch_kernel(const __grid_constant__ StepBatch<NI> B) {
  const int q = channel_of<NI>(B.block0, blockIdx.x);
  const StepInst& I = B.inst[q];
  const int b = (int)blockIdx.x - B.block0[q];
  const GridPos gp = grid_pos(I.L, b, I.strips, I.blocks);
  step_cta<float, WK>(I.L, I.a, gp, I.diag != 0);
}
template <int NI>
__global__ void __launch_bounds__(WALL_COLS)
    lbm_walls_batch_kernel(const __grid_constant__ StepBatch<NI> B) {
  const int q = channel_of<NI>(B.wall0, blockIdx.x);
  const StepInst& I = B.inst[q];
  walls_cta(I.L, (int)blockIdx.x - B.wall0[q], blockIdx.y, I.a.fin, I.a.refrho, I.a.cs_in,
            I.a.alpha, I.wall_r, I.wall_omq);
}

#include "lbm_tile.cuh"

// ---------------------------------------------------------- moments kernel
// Fields of the state obtained by streaming fin (direct = 0), or of fin
// itself (direct = 1), FP64 [6][N][Nx]: rho_a, rho_b, u_a (x, y), u_b (x, y)
// with the species momentum of Eq. rhou.
template <typename ST>
__global__ void __launch_bounds__(TX* TY)
    lbm_moments_kernel(Lat L, const ST* __restrict__ fin, const float* __restrict__ refrho,
                       const double* __restrict__ cs_in, const float* __restrict__ alpha,
                       int direct, double* __restrict__ out) {
  __shared__ WallSmem wsm;
  __shared__ float4 psi_tab[PSI_SEGMENTS];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int x = blockIdx.x * TX + tx;
  load_psi_table(psi_tab, ty * TX + tx, TX * TY);
  const ColRef C = col_ref(L, refrho, x);
  const Ends E = load_ends(L, cs_in, refrho, blockIdx.x * TX, TX);
  if (!direct)
    wall_prologue<false>(L, fin, alpha, E, C, x, 0, L.N, wsm);
  else
    __syncthreads();
  if (!interior(L, x)) return;
  const size_t plane = (size_t)L.N * L.Nx;
  for (int j = ty; j < L.N; j += TY) {
    float fs[2][9];
    if (direct) {
#pragma unroll
      for (int sp = 0; sp < 2; ++sp)
#pragma unroll
        for (int i = 0; i < 9; ++i) fs[sp][i] = ld(fin, L, sp, i, j, x);
    } else {
      pull_node(fin, L, E, C, x, j, wsm.r[0][tx], wsm.r[1][tx], fs);
    }
    float2 g[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = make_float2(fs[0][i], fs[1][i]);
    Macro2 m;
    macro2(L, make_float2(C.rb[0], C.rb[1]), g, m);
    float om_s, om_d;
    rates2(L, psi_tab, m, (float)j + 0.5f, om_s, om_d);
    Flow2 w;
    flow2(g, m.inv_rho, w);
    // Eq. rhou: (2 tau_d - 1)/(2 tau_d) = 1 - om_d/2, 1/(2 tau_d) = om_d/2
    const float w1 = 1.0f - 0.5f * om_d, w2 = 0.5f * om_d;
    const size_t o = (size_t)j * L.Nx + x;
    const float rho_s[2] = {m.rho.x, m.rho.y}, sd[2] = {m.sd.x, m.sd.y};
    const float jxs[2] = {w.jx.x, w.jx.y}, jys[2] = {w.jy.x, w.jy.y};
#pragma unroll
    for (int sp = 0; sp < 2; ++sp) {
      float mx = fmaf(w1, jxs[sp], w2 * rho_s[sp] * w.ux);
      float my = fmaf(w1, jys[sp], w2 * rho_s[sp] * w.uy);
      out[sp * plane + o] = (double)C.rb[sp] + (double)sd[sp];
      out[(2 + 2 * sp) * plane + o] = (double)(mx / rho_s[sp]);
      out[(3 + 2 * sp) * plane + o] = (double)(my / rho_s[sp]);
    }
  }
}

// Boundary columns of the moment fields (pressure ends): rho_s =
// kappa_s (2 rho_s(1) - rho_s(2)) with kappa_s of Eq. rho2, u_s linearly
// extrapolated.  Block 0: inlet, block 1: outlet.
__global__ void lbm_moments_ends_kernel(Lat L, double* __restrict__ out) {
  __shared__ double red[2][256];
  const int end = blockIdx.x, tid = threadIdx.x;
  const int xb = end == 0 ? 0 : L.Nx - 1, x1 = end == 0 ? 1 : L.Nx - 2,
            x2 = end == 0 ? 2 : L.Nx - 3;
  const size_t plane = (size_t)L.N * L.Nx;
  double sa = 0.0, sb = 0.0;
  for (int j = tid; j < L.N; j += blockDim.x) {
    size_t o = (size_t)j * L.Nx;
    sa += 2.0 * out[o + x1] - out[o + x2];
    sb += 2.0 * out[plane + o + x1] - out[plane + o + x2];
  }
  red[0][tid] = sa;
  red[1][tid] = sb;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (tid < w) {
      red[0][tid] += red[0][tid + w];
      red[1][tid] += red[1][tid + w];
    }
    __syncthreads();
  }
  const double* tgt = end == 0 ? L.rho_in : L.rho_out;
  const double ka = L.N * tgt[0] / red[0][0], kb = L.N * tgt[1] / red[1][0];
  for (int j = tid; j < L.N; j += blockDim.x) {
    size_t o = (size_t)j * L.Nx;
    out[o + xb] = ka * (2.0 * out[o + x1] - out[o + x2]);
    out[plane + o + xb] = kb * (2.0 * out[plane + o + x1] - out[plane + o + x2]);
    for (int k = 2; k < 6; ++k)
      out[k * plane + o + xb] = 2.0 * out[k * plane + o + x1] - out[k * plane + o + x2];
  }
}

// ------------------------------------------------------------ init kernels
// Column sums of a state: sum_j rho_s = N rhobar_s + sum_j sum_i d_i and the
// raw x momenta, used as the density-correction input of the first step
// after init or a state upload.
template <typename ST>
__global__ void lbm_colsum_kernel(Lat L, const ST* __restrict__ f,
                                  const float* __restrict__ refrho, double* __restrict__ cs) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= L.Nx) return;
  for (int sp = 0; sp < 2; ++sp) {
    double r = 0.0, m = 0.0;
    for (int j = 0; j < L.N; ++j) {
      float v[9];
      for (int i = 0; i < 9; ++i) v[i] = ld(f, L, sp, i, j, x);
      r += (double)(((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7])) + v[8]);
      m += (double)((v[1] - v[3]) + (v[5] - v[6]) + (v[8] - v[7]));
    }
    cs[(size_t)sp * L.Nx + x] = (double)L.N * (double)refrho[sp * L.Nx + x] + r;
    cs[(size_t)(2 + sp) * L.Nx + x] = m;
  }
}

// Re-referencing: new reference rhobar'_s(x) = cs[s][x] / N (the column
// mean of the current state) for the updated columns, unchanged elsewhere;
// d_i <- d_i + w_i alpha_si (rhobar_s - rhobar'_s) in place, in both
// buffers (the moments of the current step are formed by streaming the
// previous one).  One thread per (x, j), both species of a population as
// one pair.
template <typename ST>
__global__ void lbm_reref_kernel(Lat L, ST* __restrict__ f, ST* __restrict__ f_prev,
                                 const float* __restrict__ ref_old,
                                 const double* __restrict__ cs, float* __restrict__ ref_new) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y;
  if (x >= L.Nx) return;
  float2 ro = make_float2(ref_old[x], ref_old[L.Nx + x]), rn = ro;
  if (interior(L, x))
    rn = make_float2((float)(cs[x] / L.N), (float)(cs[L.Nx + x] / L.N));
  if (j == 0) {
    ref_new[x] = rn.x;
    ref_new[L.Nx + x] = rn.y;
  }
  const float2 dr = sub2(ro, rn);
  ST* p = f + idx(L, 0, 0, j, x);
  ST* q = f_prev + idx(L, 0, 0, j, x);
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const float2 cw = i == 0 ? make_float2(L.cw0[0], L.cw0[1])
                             : (i < 5 ? L.cw1_2 : L.cw5_2);
    Stor<ST>::st2(p + i * PS, fma2(cw, dr, Stor<ST>::ld2(p + i * PS)));
    Stor<ST>::st2(q + i * PS, fma2(cw, dr, Stor<ST>::ld2(q + i * PS)));
  }
}

// Full populations <-> stored deviations.  to_dev = 1: reads f from `in`
// (FP32, unpadded [2][9][N][Nx]) and stores d = f - ref in the strip layout;
// to_dev = 0: writes f = d + ref to `out` (T = float or double, unpadded).
template <typename ST, typename T>
__global__ void lbm_convert_kernel(Lat L, ST* __restrict__ f, const float* __restrict__ refrho,
                                   int to_dev, const float* __restrict__ in, T* __restrict__ out) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y, sp = blockIdx.z;
  if (x >= L.Nx) return;
  const float rb = refrho[sp * L.Nx + x];
  for (int i = 0; i < 9; ++i) {
    const float cw = i == 0 ? L.cw0[sp] : (i < 5 ? L.cw1[sp] : L.cw5[sp]);
    const float ref = cw * rb;
    ST* p = f + idx(L, sp, i, j, x);
    const size_t h = (((size_t)sp * 9 + i) * L.N + j) * L.Nx + x;
    if (to_dev)
      Stor<ST>::st(p, in[h] - ref);
    else
      out[h] = (T)Stor<ST>::ld(p) + (T)ref;
  }
}

// Volume flow through column x: sum over the rows of the mixture velocity u_x
// = (j_a,x + j_b,x) / (rho_a + rho_b), to which the species velocities of Eq.
// rhou add up, of the state obtained by streaming fin (direct = 0) or of fin
// itself (direct = 1); one block, fixed order, straight to host memory.
template <typename ST>
__global__ void __launch_bounds__(256)
    lbm_volume_flow_kernel(Lat L, const ST* __restrict__ fin, const float* __restrict__ refrho,
                           const double* __restrict__ cs_in, const float* __restrict__ alpha,
                           int direct, int x, double* __restrict__ out) {
  __shared__ double red[8];
  const ColRef C = col_ref(L, refrho, x);
  const Ends E = load_ends(L, cs_in, refrho, x, 1);
  double v = 0.0;
  for (int j = threadIdx.x; j < L.N; j += 256) {
    float fs[2][9];
    if (direct) {
#pragma unroll
      for (int sp = 0; sp < 2; ++sp)
#pragma unroll
        for (int i = 0; i < 9; ++i) fs[sp][i] = ld(fin, L, sp, i, j, x);
    } else {
      float2 r = make_float2(0.0f, 0.0f);
      if (j == 0 || j == L.N - 1)
        r = dbb_r(L, C, fin, x, j, alpha[(j == 0 ? 0 : L.Nx) + x]);
      pull_node(fin, L, E, C, x, j, r, r, fs);
    }
    float2 g[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = make_float2(fs[0][i], fs[1][i]);
    Flow2 w;
    flow2(g, 0.0f, w);
    const float2 sd = density_sum(g);
    const double ra = (double)C.rb[0] + sd.x, rb = (double)C.rb[1] + sd.y;
    // without a positive density of both species Eq. rhou has no velocities
    v += ra > 0.0 && rb > 0.0 ? ((double)w.jx.x + (double)w.jx.y) / (ra + rb) : (double)NAN;
  }
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int k = 0; k < 8; ++k) s += red[k];
    *out = s;
  }
}

// The number of records, the latest one and (profile != 0) C_l(x), straight to
// host memory: out[0], out[1 .. NREC], out[16 ...].  One launch and one wait
// where the count, the record and the profile took a copy and a wait each.  One
// block writes the profile, and the host copies it on: up to PINNED_COLUMNS no
// slower than a copy and a wait of its own (5000 columns 21 us, 32768 38, 40000 43
// against 31; 200 000 152 against 37, 10^6 691 against 71).
constexpr int PINNED_COLUMNS = 32768;
__global__ void __launch_bounds__(256)
    lbm_latest_kernel(const double* __restrict__ diag,
                      const unsigned long long* __restrict__ diag_count,
                      const double* __restrict__ clprof, int Nx, int profile,
                      double* __restrict__ out) {
  const unsigned long long cnt = *diag_count;
  const int t = threadIdx.x;
  if (t == 0) out[0] = (double)cnt;
  if (t < NREC) out[1 + t] = cnt == 0 ? 0.0 : diag[(size_t)((cnt - 1) % DIAG_CAP) * NREC + t];
  if (profile)
    for (int x = t; x < Nx; x += 256) out[16 + x] = clprof[x];
}

// Steady-state residual over the column sums: R = |c - c_old| / (K |c|),
// then c_old = c.  One CTA per channel.
struct ResidInst {
  const double* c;
  double* c_old;
  long n;
  int have_old;
};
template <int NI>
struct ResidBatch {
  ResidInst inst[NI];
};
template <int NI>
__global__ void lbm_residual_kernel(const __grid_constant__ ResidBatch<NI> B, double K,
                                    double* __restrict__ R) {
  __shared__ double s1[32], s2[32];
  const double* __restrict__ c = B.inst[blockIdx.x].c;
  double* __restrict__ c_old = B.inst[blockIdx.x].c_old;
  const long n = B.inst[blockIdx.x].n;
  const int have_old = B.inst[blockIdx.x].have_old;
  double d2 = 0.0, c2 = 0.0;
  for (long k = threadIdx.x; k < n; k += blockDim.x) {
    double v = c[k];
    double d = v - c_old[k];
    d2 += d * d;
    c2 += v * v;
    c_old[k] = v;
  }
  d2 = warp_sum(d2);
  c2 = warp_sum(c2);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    s1[wid] = d2;
    s2[wid] = c2;
  }
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x >> 5;
    d2 = lane < nw ? s1[lane] : 0.0;
    c2 = lane < nw ? s2[lane] : 0.0;
    d2 = warp_sum(d2);
    c2 = warp_sum(c2);
    if (lane == 0) R[blockIdx.x] = have_old ? sqrt(d2) / (K * sqrt(c2)) : INFINITY;
  }
}

__global__ void lbm_special_kernel(const double* __restrict__ x, double* __restrict__ e1,
                                   double* __restrict__ ps, long n) {
  long k = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  float v = (float)x[k];
  e1[k] = (double)e1_dev(v);
  ps[k] = (double)psi_dev(kPsiTab, v);
}

}  // namespace

// ================================================================ host API
struct lbm_mix {
  lbm_mix_params p;
  Lat L;
  int device;
  int nsm;            // streaming multiprocessors of the device
  cudaStream_t stream;
  bool own_stream;
  long launches;     // kernels launched by its own steps so far
  bool pending;      // a call may have left work on the stream (see join_handles)
  int nblocks;
  void* buf[2];       // post-collision deviations, A/B (element type per storage)
  size_t elem;        // bytes per stored population
  float* refrho;      // [2][Nx] reference densities rhobar_s(x)
  float* refrho_alt;  // the next reference table of lbm_mix_rereference
  double* cs_tmp;     // [4][Nx] column sums of lbm_mix_rereference
  float* scratch;     // full-population staging for get_post_state (lazy)
  double* cs[2];
  double* cs_snap;
  float* alpha;
  double* partials;
  unsigned* counter;
  double* diag;
  unsigned long long* diag_count;
  double* clprof;
  float2* wall_r;      // [2][Nx] r per wall and column (lbm_walls_kernel)
  float* wall_omq;     // [2][Nx] 1/tau_q per half and column (lbm_walls_kernel)
  float2* end_sd;      // [4][N] (FP32 storage with pressure ends, else null)
  float2* colpart;     // [R][4][Nx]
  float2* colpart0;    // its place in the arena
  void* arena;         // holds the arrays above and below but scratch and mom
  unsigned* strip_cnt; // [nblocks]
  int R, rows_per_block;
  int R_alloc;        // row blocks colpart has room for
  double* mom;
  double* h_pinned;  // [16 + min(Nx, PINNED_COLUMNS)] pinned: what the getters' kernels write
  // Several steps per launch (lbm_tile_kernel): own columns per tile and
  // most steps of a launch; tile_W = 0: the channel does not qualify.  A
  // schedule the caller set (rows_set) takes the step kernel instead.
  int tile_W, tile_k;
  bool rows_set;
  float2* hist;      // [hist_rows][4][Nx] column sums awaiting lbm_records_kernel
  int hist_rows;
  double* rec_part;  // [hist_rows][NPART][record_blocks]: see lbm_records_kernel
  unsigned* rec_cnt; // [hist_rows]
  int cur;           // buffer holding the latest post-collision state
  long steps;
  bool have_snap;
};

namespace {

int validate(const lbm_mix_params* p, int* Nx_out) {
  if (!p) return set_err(LBM_EINVAL, "params is NULL");
  if (!(p->m_a > 0 && p->m_b > 0 && isfinite(p->m_a) && isfinite(p->m_b)))
    return set_err(LBM_EINVAL, "masses must be positive and finite");
  if (!(p->C_l > 0 && p->C_l < 1)) return set_err(LBM_EINVAL, "C_l must be in (0,1)");
  if (p->C_l_out >= 0 && !(p->C_l_out > 0 && p->C_l_out < 1))
    return set_err(LBM_EINVAL, "C_l_out must be in (0,1) or negative");
  if (!(p->theta >= 1.0 && isfinite(p->theta))) return set_err(LBM_EINVAL, "theta must be >= 1");
  if (!(p->Kn_out > 0 && isfinite(p->Kn_out))) return set_err(LBM_EINVAL, "Kn_out must be > 0");
  if (p->N < 2) return set_err(LBM_EINVAL, "N must be >= 2");
  long Nx = p->N_x;
  if (Nx <= 0) {
    if (!(p->L_over_H > 0 && isfinite(p->L_over_H)))
      return set_err(LBM_EINVAL, "L_over_H must be > 0 when N_x <= 0");
    Nx = lround(p->N * p->L_over_H);
  }
  if (Nx < 4) return set_err(LBM_EINVAL, "need N_x >= 4 columns (got %ld)", Nx);
  if (!(p->accommodation > 0 && p->accommodation <= 1))
    return set_err(LBM_EINVAL, "accommodation must be in (0,1]");
  if (!(p->c_m0 >= 0 && isfinite(p->c_m0))) return set_err(LBM_EINVAL, "c_m0 must be >= 0");
  if (!(p->tau_rho > 0.5 && p->tau_e > 0.5 && p->tau_eps > 0.5))
    return set_err(LBM_EINVAL, "tau_rho, tau_e, tau_eps must exceed 1/2");
  if (!(p->mu_ratio_a > 0 && p->mu_ratio_b > 0))
    return set_err(LBM_EINVAL, "viscosity ratios must be > 0");
  if (p->storage != LBM_FP32 && p->storage != LBM_BF16 && p->storage != LBM_FP16)
    return set_err(LBM_EINVAL, "storage must be LBM_FP32, LBM_BF16 or LBM_FP16");
  if (p->x_periodic != 0 && p->x_periodic != 1) return set_err(LBM_EINVAL, "x_periodic is 0 or 1");
  if (p->diag_every < 1) return set_err(LBM_EINVAL, "diag_every must be >= 1");
  if (p->reref_every < -1) return set_err(LBM_EINVAL, "reref_every must be >= -1");
  if (p->r_form != LBM_R_FIRST && p->r_form != LBM_R_SPECIES && p->r_form != LBM_R_SECOND)
    return set_err(LBM_EINVAL, "r_form must be LBM_R_FIRST, LBM_R_SPECIES or LBM_R_SECOND");
  if (p->lambda_pressure != 0 && p->lambda_pressure != 1)
    return set_err(LBM_EINVAL, "lambda_pressure must be 0 (partial) or 1 (mixture)");
  if (p->wall != LBM_WALL_DBB && p->wall != LBM_WALL_BSR)
    return set_err(LBM_EINVAL, "wall must be LBM_WALL_DBB or LBM_WALL_BSR");
  if (p->rounding != LBM_ROUND_STOCHASTIC && p->rounding != LBM_ROUND_NEAREST)
    return set_err(LBM_EINVAL, "rounding must be LBM_ROUND_STOCHASTIC or LBM_ROUND_NEAREST");
  long pitch = (Nx + 31) / 32 * 32;
  double elems = 18.0 * (double)p->N * (double)pitch;
  if (elems >= 2147483648.0)
    return set_err(LBM_EINVAL, "lattice too large: 18*N*pitch must stay below 2^31");
  *Nx_out = (int)Nx;
  return LBM_OK;
}

// Lattice constants in the units of the header (k_B T = 1/3, m_min = 1,
// outlet number density 1), derived in FP64.
Lat derive(const lbm_mix_params* p, int Nx) {
  Lat L;
  memset(&L, 0, sizeof L);
  const double PI = 3.14159265358979323846;
  L.N = p->N;
  L.Nx = Nx;
  L.pitch = (Nx + 31) / 32 * 32;
  L.SS = (unsigned)((long)L.N * RS);
  L.x_periodic = p->x_periodic;
  L.wall_mode = p->wall;
  L.r_form = p->r_form;
  L.lam_mix = p->lambda_pressure;
  double m_min = fmin(p->m_a, p->m_b);
  double mh[2] = {p->m_a / m_min, p->m_b / m_min};
  L.light = (p->m_a <= p->m_b) ? 0 : 1;
  double Cin = p->C_l, Cout = p->C_l_out < 0 ? p->C_l : p->C_l_out;
  double Ci[2], Co[2];
  Ci[L.light] = Cin;
  Ci[1 - L.light] = 1.0 - Cin;
  Co[L.light] = Cout;
  Co[1 - L.light] = 1.0 - Cout;
  L.C_in = Cin;
  L.C_out = Cout;
  double mx_out = Co[0] * mh[0] + Co[1] * mh[1];
  double lam_out = p->Kn_out * p->N;
  // lambda = (mu / p) sqrt(pi k_B T / (2 m_x)) with p_out = 1/3 at the outlet
  double mu = lam_out * (1.0 / 3.0) / sqrt(PI / (6.0 * mx_out));
  double mu_s[2] = {p->mu_ratio_a * mu, p->mu_ratio_b * mu};
  for (int sp = 0; sp < 2; ++sp) {
    L.s[sp] = (float)(1.0 / mh[sp]);
    L.cw0[sp] = (float)((9.0 - 5.0 * (double)L.s[sp]) / 9.0);
    L.cw1[sp] = (float)((double)L.s[sp] / 9.0);
    L.cw5[sp] = (float)((double)L.s[sp] / 36.0);
  }
  for (int sp = 0; sp < 2; ++sp) {
    float* s2 = &L.s2.x;
    s2[sp] = L.s[sp];
    (&L.cw1_2.x)[sp] = L.cw1[sp];
    (&L.cw5_2.x)[sp] = L.cw5[sp];
    const double we = 1.0 / (36.0 * p->tau_e), wp = 1.0 / (36.0 * p->tau_eps);
    const double sd = (double)L.s[sp];
    const float sf = L.s[sp];
    const float ke[3] = {-2.0f * sf, 3.0f - 2.0f * sf, 6.0f - 2.0f * sf};
    const float kp[3] = {3.0f * sf, 3.0f * sf - 6.0f, 3.0f * sf - 3.0f};
    for (int k = 0; k < 3; ++k) {
      (&L.ke2[k].x)[sp] = ke[k];
      (&L.kp2[k].x)[sp] = kp[k];
      (&L.ce2[k].x)[sp] = (float)(we * (3.0 * k - 2.0 * sd));
      (&L.cp2[k].x)[sp] = (float)(wp * (3.0 * sd - (k == 0 ? 0.0 : k == 1 ? 6.0 : 3.0)));
    }
    (&L.cu2[0].x)[sp] = (float)(-3.0 * we);
    (&L.cu2[1].x)[sp] = (float)(3.0 * wp);
    L.mh[sp] = mh[sp];
    L.rsqrt_mh[sp] = (float)(1.0 / sqrt(mh[sp]));
    double cxl = 3.0 * mu_s[sp] * sqrt(PI / (6.0 * mh[sp]));
    (&L.c_xl2.x)[sp] = (float)cxl;
    (&L.inv_c_xl2.x)[sp] = (float)(1.0 / cxl);
    L.rho_in[sp] = p->theta * Ci[sp] * mh[sp];
    L.rho_out[sp] = Co[sp] * mh[sp];
    for (int end = 0; end < 2; ++end) {
      const double m = L.N * (end == 0 ? L.rho_in[sp] : L.rho_out[sp]);
      L.end_mass[end][sp] = make_float2((float)m, (float)(m - (double)(float)m));
    }
  }
  double clam = 3.0 * mu * sqrt(PI / 6.0);
  L.c_lam = (float)clam;
  L.inv_c_lam = (float)(1.0 / clam);
  L.c_ts = (float)sqrt(6.0 / PI);
  L.c_td = (float)(1.5 * sqrt(3.0 * (mh[0] + mh[1]) * mh[0] * mh[1] / 1.0));
  L.om_e = (float)(1.0 / p->tau_e);
  L.om_eps = (float)(1.0 / p->tau_eps);
  L.c_m0 = (float)p->c_m0;
  L.H = (float)p->N;
  return L;
}

// Host copy of the step kernel's seed hash (lowbias32).
unsigned host_hash32(unsigned x) {
  x ^= x >> 16;
  x *= 0x7feb352du;
  x ^= x >> 15;
  x *= 0x846ca68bu;
  x ^= x >> 16;
  return x;
}

// Rows of one strip per CTA of the step kernel unless the caller sets a
// schedule: as many as leave `waves` waves of resident CTAs (3 per SM), a
// multiple of TY within [16, 56] (FP32) or [16, 96] (16-bit).  A warp takes
// its CTA's rows one after another, every TY-th, so on a channel of few strips
// fewer rows per CTA shorten the step until the CTAs' own start-up counts.
// Measured on GB300, us per step at 96 rows and at this rule's count: FP32
// 5001 x 130 37.8 -> 26.0 (16 rows), 8000 x 128 42.8 -> 32.6 (24), 20000 x 64
// 39.5 (32), 16384 x 256 104 -> 102 (56), 32768 x 512 367 -> 367 (56); BF16
// 39.9 -> 27.9 (16), 42.2 -> 34.4 (24), 16384 x 256 102 (96), 32768 x 512 345
// (96).
constexpr int WAVES = 3;
int default_rows(int N, int strips, int nsm, bool fp32) {
  const int n8 = (N + TY - 1) / TY * TY, most = fp32 ? 56 : 96;
  const long ctas = (long)WAVES * 3 * (nsm > 0 ? nsm : 1);
  long rows = ((long)N * strips / ctas + TY - 1) / TY * TY;
  rows = rows < 16 ? 16 : rows < most ? rows : most;
  const long fit = (N + 65534L) / 65535;  // a grid has 65535 row blocks at most
  if (rows < fit) rows = (fit + TY - 1) / TY * TY;
  return (int)(rows < n8 ? rows : n8);
}
int default_rows(const lbm_mix* h) {
  return default_rows(h->L.N, h->nblocks, h->nsm, h->p.storage == LBM_FP32);
}

// Rows of one strip per CTA of a recorded step under the default schedule.
// Every CTA of such a step ends in column_epilogue (a fence, a ticket), so
// twice the rows pay there: at least 56, at most 96 (FP32) or 128 (16-bit).
// us per recorded step at the rows of the others and at these: FP32 5001 x 130
// 38.4 -> 30.9 (16, 56 rows), 12000 x 200 82.4 -> 73.5 (56, 96), 15000 x 300
// 128.2 -> 126.0, 32768 x 512 407.9 -> 392.3; BF16 40.3 -> 38.4 (16, 56), 32768
// x 512 389.4 -> 381.5 (96, 128).
int recorded_rows(const lbm_mix* h) {
  const int rows = h->rows_per_block, n8 = (h->L.N + TY - 1) / TY * TY;
  const int most = h->p.storage == LBM_FP32 ? 96 : 128;
  int r = 2 * rows < 56 ? 56 : 2 * rows < most ? 2 * rows : most;
  if (r > n8) r = n8;
  return h->rows_set || r < rows ? rows : r;
}

// Calls f(type tag) with the storage element type of the handle.
template <typename F>
int with_storage(const lbm_mix* h, F&& f) {
  switch (h->p.storage) {
    case LBM_FP32: return f(float());
    case LBM_BF16: return f(__nv_bfloat16());
    case LBM_FP16: return f(__half());
    default: return set_err(LBM_EINVAL, "unknown storage %d", h->p.storage);
  }
}

int launch_colsum(lbm_mix* h, int b) {
  return with_storage(h, [&](auto tag) -> int {
    using ST = decltype(tag);
    dim3 blk(128), grd((h->L.Nx + 127) / 128);
    lbm_colsum_kernel<ST><<<grd, blk, 0, h->stream>>>(h->L, (const ST*)h->buf[b], h->refrho,
                                                      h->cs[b]);
    CK(cudaGetLastError());
    return LBM_OK;
  });
}

// Column sums of the current state into cs_tmp, then the in-place rewrite
// of the deviations against the new column means; the reference tables swap.
int rereference(lbm_mix* h) {
  const int b = h->cur;
  int st = with_storage(h, [&](auto tag) -> int {
    using ST = decltype(tag);
    dim3 blk(128), grd((h->L.Nx + 127) / 128);
    lbm_colsum_kernel<ST><<<grd, blk, 0, h->stream>>>(h->L, (const ST*)h->buf[b], h->refrho,
                                                      h->cs_tmp);
    CK(cudaGetLastError());
    dim3 grd2((h->L.Nx + 127) / 128, h->L.N);
    lbm_reref_kernel<ST><<<grd2, blk, 0, h->stream>>>(h->L, (ST*)h->buf[b], (ST*)h->buf[1 - b],
                                                      h->refrho, h->cs_tmp, h->refrho_alt);
    CK(cudaGetLastError());
    return LBM_OK;
  });
  if (st) return st;
  h->launches += 2;
  float* t = h->refrho;
  h->refrho = h->refrho_alt;
  h->refrho_alt = t;
  return LBM_OK;
}

// Steady-state residual of the last k steps (Sec. 4 convergence check, over
// the column sums of the latest DIAG step) into h->h_pinned[0], async, by the
// kernel itself.
int launch_residual(lbm_mix* h, long k) {
  ResidBatch<1> B;
  B.inst[0] = ResidInst{h->cs[h->cur], h->cs_snap, 4L * h->L.Nx, h->have_snap ? 1 : 0};
  lbm_residual_kernel<1><<<1, 1024, 0, h->stream>>>(B, (double)k, h->h_pinned);
  CK(cudaGetLastError());
  h->have_snap = true;
  return LBM_OK;
}

// Waits for the handle's stream.
cudaError_t wait_stream(lbm_mix* h) {
  const cudaError_t e = cudaStreamSynchronize(h->stream);
  if (e == cudaSuccess) h->pending = false;
  return e;
}

// Node-to-CTA schedule: rows per CTA (a multiple of TY); the per-row-block
// partials grow when a schedule needs more row blocks than allocated.
int set_rows_per_block(lbm_mix* h, int rows) {
  const int nmax = (h->L.N + TY - 1) / TY * TY;
  if (rows <= 0) rows = default_rows(h);
  if (rows % TY != 0) return set_err(LBM_EINVAL, "rows per block must be a multiple of %d", TY);
  if (rows > nmax) rows = nmax;
  const int R = (h->L.N + rows - 1) / rows;
  if (R > h->R_alloc) {
    float2* cp = nullptr;
    CK(wait_stream(h));
    CK(cudaMalloc((void**)&cp, sizeof(double) * 4 * (size_t)h->L.Nx * (size_t)R));
    if (h->colpart != h->colpart0) cudaFree(h->colpart);
    h->colpart = cp;
    h->R_alloc = R;
  }
  h->rows_per_block = rows;
  h->R = R;
  return LBM_OK;
}

int reset_diag(lbm_mix* h) {
  CK(cudaMemsetAsync(h->diag_count, 0, sizeof(unsigned long long), h->stream));
  CK(cudaMemsetAsync(h->diag, 0, sizeof(double) * DIAG_CAP * NREC, h->stream));
  h->have_snap = false;
  return LBM_OK;
}

// FP32 storage takes r and tau_q from lbm_walls_kernel when the step's grid
// holds at least WALL_KERNEL_WAVES waves of resident CTAs (3 per SM): there
// the prologue's barrier in every CTA costs more than a launch and its 7 us
// (32768 x 512, 22 waves: 369.5 against 367 us; 15000 x 300, 6.2 waves: 109.0
// against 108.2; the other way 5001 x 130, 3.1 waves: 25.9 against 31.8, and
// 20000 x 64, 4.1 waves: 37.6 against 42.5).  A schedule that the caller
// set, often of few rows per CTA, and the launches of a sweep take it from two
// waves on (64 x 6000 at 8 rows: 23.5 against 20.5 us; 24 mixed channels 98.6
// against 101.4).  16-bit storage always uses the wall kernel.
constexpr long WALL_KERNEL_WAVES = 5, WALL_KERNEL_WAVES_SET = 2;
bool uses_wall_kernel(const lbm_mix* h) {
  const long ctas = (long)h->nblocks * (long)h->R;
  const long waves = h->rows_set ? WALL_KERNEL_WAVES_SET : WALL_KERNEL_WAVES;
  return ctas >= waves * 3L * (long)(h->nsm > 0 ? h->nsm : 1);
}

// Arguments of h's next step.
template <typename ST>
StepArgs<ST> step_args(const lbm_mix* h) {
  const int b = h->cur;
  StepArgs<ST> a;
  a.fin = (const ST*)h->buf[b];
  a.fout = (ST*)h->buf[1 - b];
  a.refrho = h->refrho;
  a.cs_in = h->cs[b];
  a.cs_out = h->cs[1 - b];
  a.alpha = h->alpha;
  a.partials = h->partials;
  a.counter = h->counter;
  a.diag = h->diag;
  a.diag_count = h->diag_count;
  a.clprof = h->clprof;
  a.colpart = h->colpart;
  a.strip_cnt = h->strip_cnt;
  a.rows_per_block = h->rows_per_block;
  // stochastic rounding of 16-bit stores: a fresh seed every step (never 0)
  a.seed = (sizeof(ST) < 4 && h->p.rounding == LBM_ROUND_STOCHASTIC)
               ? (host_hash32((unsigned)(h->steps + 1)) | 1u)
               : 0u;
  a.wall_r = h->wall_r;
  a.wall_omq = h->wall_omq;
  a.end_sd = h->end_sd;
  return a;
}

int launch_step(lbm_mix* h, bool diag) {
  int st = with_storage(h, [&](auto tag) -> int {
    using ST = decltype(tag);
    StepArgs<ST> a = step_args<ST>(h);
    if (diag) a.rows_per_block = recorded_rows(h);  // no fewer than R was sized for
    // Both kernels are launched with programmatic stream serialisation, so
    // that each one's launch and CTA ramp overlap the end of the kernel
    // before it (see pdl_wait).
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = h->stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const bool wk = sizeof(ST) < 4 || uses_wall_kernel(h);
    if (wk) {
      cfg.gridDim = dim3((h->L.Nx + WALL_COLS - 1) / WALL_COLS, 4);
      cfg.blockDim = dim3(WALL_COLS);
      CK(cudaLaunchKernelEx(&cfg, lbm_walls_kernel<ST>, h->L, a.fin, (const float*)h->refrho,
                            (const double*)a.cs_in, (const float*)h->alpha, h->wall_r,
                            h->wall_omq));
      h->launches++;
    }
    cfg.gridDim = dim3(h->nblocks, (h->L.N + a.rows_per_block - 1) / a.rows_per_block);
    cfg.blockDim = dim3(TX, TY);
    if (sizeof(ST) < 4 || !wk) {
      if (diag)
        CK(cudaLaunchKernelEx(&cfg, lbm_step_kernel<ST, true>, h->L, a));
      else
        CK(cudaLaunchKernelEx(&cfg, lbm_step_kernel<ST, false>, h->L, a));
    } else {
      if (diag)
        CK(cudaLaunchKernelEx(&cfg, lbm_step_kernel<ST, true, true>, h->L, a));
      else
        CK(cudaLaunchKernelEx(&cfg, lbm_step_kernel<ST, false, true>, h->L, a));
    }
    return LBM_OK;
  });
  if (st) return st;
  h->launches++;
  h->cur = 1 - h->cur;
  h->steps++;
  return LBM_OK;
}

// ------------------------------------------------- several steps per launch
// Estimated time of one step (us) of a channel cut into tiles of W columns
// that take k steps per launch on `sms` SMs: a launch costs TILE_LAUNCH_US,
// each wave of tiles TILE_LOAD_US to load and store, and each of its steps
// TILE_STEP_US plus TILE_NODE_US per node of the tile.  Fitted to channels of
// 16 to 128 rows and 5 000 to 600 000 nodes, k = 1 ... 15 (within 20 %; the
// minimum over k is flat).
constexpr double TILE_LAUNCH_US = 0.6, TILE_LOAD_US = 4.0, TILE_STEP_US = 1.0,
                 TILE_NODE_US = 0.0025;
double tile_cost(int N, int nup, int W, int k, int sms) {
  const int tiles = (nup + W - 1) / W;
  const double waves = (tiles + sms - 1) / sms;
  // sum over t = 1 ... k of the W + 2 (k - t) columns of step t
  const double nodes = (double)k * (W + k - 1) * tile_stride(N);
  return (TILE_LAUNCH_US + waves * (TILE_LOAD_US + k * TILE_STEP_US + TILE_NODE_US * nodes)) / k;
}
// The same for the step kernel under its default schedule as the tiles were
// fitted against it (64 x 3000 18.3 us, 128 x 8000 32.6).  With the end strips first
// it has since become faster, 10 us up to some 100 000 nodes and 14 at 250 000, so
// near the line tiles are no longer the better choice: columns x rows 4000 x 64
// 12.8 us by tiles and 13.4, 14000 x 32 18.9 and 14.1, 2000 x 128 21.1 and 13.2.
double step_kernel_cost(int N, int Nx) { return 15.0 + 1.75e-5 * (double)N * Nx; }

// Tile width and steps per launch (odd, so that launches alternate the two
// buffers as single steps do) of least estimated cost on `sms` SMs; W = 0
// where no tile fits shared memory.
void plan_tiles(const Lat& L, int sms, int* W_out, int* k_out, double* us_out) {
  const int nup = L.x_periodic ? L.Nx : L.Nx - 2;
  *W_out = 0;
  *k_out = 0;
  *us_out = INFINITY;
  for (int k = 1; k <= TILE_KMAX; k += 2) {
    if (tile_smem(L.N, 1 + 2 * k) > (size_t)TILE_SMEM_MAX) break;
    for (int W = 1; W <= nup; ++W) {
      if (tile_smem(L.N, W + 2 * k) > (size_t)TILE_SMEM_MAX) break;
      const double us = tile_cost(L.N, nup, W, k, sms);
      if (us < *us_out) {
        *us_out = us;
        *W_out = W;
        *k_out = k;
      }
      if ((nup + W - 1) / W == 1) break;
    }
  }
}

// Size of a handle's record rows.
constexpr long HIST_BYTES = 2 << 20;

bool uses_tiles(const lbm_mix* h) { return h->tile_W > 0 && !h->rows_set; }

// Launches kernel<NI> for n channels with programmatic stream serialisation.
template <typename B>
int launch_batch(void (*kern)(B), const B& batch, dim3 grid, dim3 block, size_t smem,
                 cudaStream_t st) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  CK(cudaLaunchKernelEx(&cfg, kern, batch));
  return LBM_OK;
}

// One launch of k steps for the n <= NI channels hs in tiles of W[] columns,
// whose record rows used so far are rows[]; last: step k ends the call.
template <int NI>
int launch_tiles(lbm_mix* const* hs, const int* W, int n, int k, bool last, int* rows,
                 cudaStream_t st) {
  TileBatch<NI> B;
  B.k = k;
  int blocks = 0, nodes = 0;
  size_t smem = 0;
  for (int q = 0; q < NI; ++q) {
    B.block0[q] = blocks;
    if (q >= n) continue;
    lbm_mix* h = hs[q];
    const Lat& L = h->L;
    TileInst& I = B.inst[q];
    const int b = h->cur, de = h->p.diag_every;
    I.L = L;
    I.fin = (const float*)h->buf[b];
    I.fout = (float*)h->buf[1 - b];
    I.refrho = h->refrho;
    I.alpha = h->alpha;
    I.cs_in = h->cs[b];
    I.cs_out = h->cs[1 - b];
    I.hist = h->hist + (size_t)rows[q] * 4 * L.Nx;
    I.W = W[q];
    I.diag_every = de;
    I.diag_phase = (int)(h->steps % de);
    I.last = last ? 1 : 0;
    rows[q] += (int)((h->steps + k) / de - h->steps / de);
    if (last && (h->steps + k) % de != 0) rows[q]++;
    const int nup = L.x_periodic ? L.Nx : L.Nx - 2;
    blocks += (nup + I.W - 1) / I.W;
    const int own = I.W < nup ? I.W : nup, busy = (own + 2 * k - 2) * (L.N - 2);
    nodes = busy > nodes ? busy : nodes;
    const size_t sm = tile_smem(L.N, own + 2 * k);
    smem = sm > smem ? sm : smem;
  }
  B.block0[NI] = blocks;
  int threads = (nodes + 31) / 32 * 32;
  threads = threads < 32 ? 32 : threads < TILE_INNER ? threads : TILE_INNER;
  int s = launch_batch(lbm_tile_kernel<NI>, B, dim3(blocks),
                       dim3(threads + TILE_WALL + TILE_TAUQ), smem, st);
  if (s) return s;
  if (NI == 1) hs[0]->launches++;
  for (int q = 0; q < n; ++q) {
    hs[q]->cur = 1 - hs[q]->cur;
    hs[q]->steps += k;
  }
  return LBM_OK;
}

// The records of rows[] column-sum rows of every channel; rows[] to zero.
template <int NI>
int launch_records(lbm_mix* const* hs, int n, int* rows, cudaStream_t st) {
  RecBatch<NI> B;
  int most = 0, blocks = 1;
  for (int q = 0; q < n; ++q) {
    lbm_mix* h = hs[q];
    const Lat& L = h->L;
    B.inst[q] = RecInst{L.N,     L.Nx,    L.x_periodic, L.light, {L.s[0], L.s[1]}, L.C_in,
                        L.C_out, h->hist, h->refrho,    h->diag, h->diag_count,    h->counter,
                        h->clprof, h->rec_part, h->rec_cnt, rows[q], record_blocks(L.Nx)};
    most = rows[q] > most ? rows[q] : most;
    blocks = B.inst[q].blocks > blocks ? B.inst[q].blocks : blocks;
    rows[q] = 0;
  }
  if (most == 0) return LBM_OK;
  if (NI == 1) hs[0]->launches++;
  return launch_batch(lbm_records_kernel<NI>, B, dim3(blocks, most, n), dim3(256), 0, st);
}

// Columns beyond which a lone channel takes single steps by lbm_step_kernel: a
// launch of lbm_tile_kernel for one step fills, sums and empties its tiles for
// it, and its record is a launch of its own.  us per call of one step, by tiles
// and record and by the step kernel: 700 x 20 17.7 and 15, 2000 x 16 19 and 15,
// 4000 x 16 32 and 17, 8000 x 16 41 and 18, 40000 x 8 78 and 39 (as many calls
// in a row as the host issues; up to 2000 it bounds either).
constexpr int SINGLE_STEP_COLUMNS = 2048;

// nsteps steps of the n <= NI channels hs on stream st: launches of kmax
// steps or fewer, the last one of a single step, so that the two buffers end
// up holding the states of the last two steps.  end: the last step ends the
// call and is recorded.
template <int NI>
int tile_steps(lbm_mix* const* hs, const int* W, int n, int kmax, long nsteps, bool end,
               cudaStream_t st) {
  int rows[NI] = {};
  int s = LBM_OK;
  for (long left = nsteps; left > 0;) {
    int k = left - 1 < kmax ? (int)(left - 1) : kmax;
    k -= 1 - (k & 1);  // odd
    if (k < 1) k = 1;
    if (NI == 1 && k == 1 && hs[0]->L.Nx > SINGLE_STEP_COLUMNS) {
      const bool diag = (end && left == 1) || (hs[0]->steps + 1) % hs[0]->p.diag_every == 0;
      if ((s = launch_records<NI>(hs, n, rows, st)) || (s = launch_step(hs[0], diag))) return s;
      --left;
      continue;
    }
    bool full = false;
    for (int q = 0; q < n; ++q) full |= rows[q] + k + 1 > hs[q]->hist_rows;
    if (full && (s = launch_records<NI>(hs, n, rows, st))) return s;
    if ((s = launch_tiles<NI>(hs, W, n, k, end && left == k, rows, st))) return s;
    left -= k;
  }
  return launch_records<NI>(hs, n, rows, st);
}

int launch_moments(lbm_mix* h, double* d_out) {
  // The state of step n is the stream of buffer P_{n-1}; right after init or
  // an upload only the buffer itself exists.
  const bool direct = (h->steps == 0);
  const int b = direct ? h->cur : 1 - h->cur;
  dim3 blk(TX, TY), grd(h->nblocks);
  int st = with_storage(h, [&](auto tag) -> int {
    using ST = decltype(tag);
    lbm_moments_kernel<ST><<<grd, blk, 0, h->stream>>>(h->L, (const ST*)h->buf[b], h->refrho,
                                                       h->cs[b], h->alpha, direct ? 1 : 0, d_out);
    CK(cudaGetLastError());
    return LBM_OK;
  });
  if (st) return st;
  if (!h->L.x_periodic) {
    lbm_moments_ends_kernel<<<2, 256, 0, h->stream>>>(h->L, d_out);
    CK(cudaGetLastError());
  }
  return LBM_OK;
}

// On entry to a call; one that may enqueue work has a handle that is not const.
int check_handle(const lbm_mix* h) {
  if (!h) return set_err(LBM_EINVAL, "handle is NULL");
  return LBM_OK;
}
int check_handle(lbm_mix* h) {
  if (!h) return set_err(LBM_EINVAL, "handle is NULL");
  h->pending = true;
  return LBM_OK;
}

// Latest diagnostic record (host copy) and, where wanted, C_l(x). Returns
// LBM_ENONFINITE on NaN/Inf.  A profile of more than PINNED_COLUMNS columns is
// copied to the caller's array by itself.
int latest_record(lbm_mix* h, double rec[NREC], double* profile) {
  const bool wide = h->L.Nx > PINNED_COLUMNS;
  lbm_latest_kernel<<<1, 256, 0, h->stream>>>(h->diag, h->diag_count, h->clprof, h->L.Nx,
                                              profile && !wide ? 1 : 0, h->h_pinned);
  CK(cudaGetLastError());
  CK(wait_stream(h));
  const unsigned long long cnt = (unsigned long long)h->h_pinned[0];
  if (cnt == 0) return set_err(LBM_EINVAL, "no step taken yet");
  memcpy(rec, h->h_pinned + 1, sizeof(double) * NREC);
  for (int k = 1; k < NREC; ++k)
    if (!isfinite(rec[k])) return set_err(LBM_ENONFINITE, "non-finite diagnostic at step %llu", cnt);
  if (profile && wide) {
    CK(cudaMemcpyAsync(profile, h->clprof, sizeof(double) * (size_t)h->L.Nx,
                       cudaMemcpyDeviceToHost, h->stream));
    CK(wait_stream(h));
  } else if (profile) {
    memcpy(profile, h->h_pinned + 16, sizeof(double) * (size_t)h->L.Nx);
  }
  return LBM_OK;
}

}  // namespace

// ---------------------------------------------- allocation-free stepping
// Scratch of lbm_mix_step_noalloc: the per-strip partial sums, the per-strip
// and grid arrival tickets and the record counter of lbm_step_kernel, in one
// static device array so that a caller who cannot allocate device memory can
// still run a step.  Every GPU that loads the library holds it until exit:
//   partials  NOALLOC_MAX_STRIPS * NPART doubles   (64 KiB)
//   counters  NOALLOC_MAX_STRIPS + 4 words          (4 KiB + 16 B)
constexpr int NOALLOC_MAX_STRIPS = 1024;  // N_x <= 32 * 1024 = 32768 columns
constexpr size_t NOALLOC_PART_DOUBLES = (size_t)NOALLOC_MAX_STRIPS * NPART;
constexpr size_t NOALLOC_CNT_WORDS = NOALLOC_MAX_STRIPS + 4;
constexpr size_t NOALLOC_DOUBLES = NOALLOC_PART_DOUBLES + (NOALLOC_CNT_WORDS + 1) / 2;
static __device__ __align__(256) double g_noalloc_scratch[NOALLOC_DOUBLES];

// The calling thread's current CUDA context (the driver's cuCtxGetCurrent,
// reached through the runtime so that the library needs no link against
// the driver library); nullptr if none is current or the query fails.
void* current_context() {
  typedef int (*CtxGetCurrent)(void**);
  static CtxGetCurrent fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return (CtxGetCurrent)f;
  }();
  void* ctx = nullptr;
  if (!fn || fn(&ctx) != 0) return nullptr;
  return ctx;
}

// Device address of g_noalloc_scratch in the current device's context.  In
// host code the symbol's name only stands for the device array; kernels
// must be given this address.  It is looked up on the first call on a
// device and again whenever the current context is not the one it was
// looked up in (a device reset or another primary context loads the module
// anew, at another address).
int noalloc_scratch_address(double** out) {
  static std::mutex mu;
  static double* addr[64] = {};
  static void* ctx_of[64] = {};
  int dev = 0;
  CK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return set_err(LBM_EINVAL, "device ordinal %d out of range", dev);
  std::lock_guard<std::mutex> lock(mu);
  void* ctx = current_context();
  if (!addr[dev] || !ctx || ctx != ctx_of[dev]) {
    void* ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    if (e != cudaSuccess || !ptr)
      return set_err(LBM_ECUDA, "cudaGetSymbolAddress(scratch) failed on device %d: %s", dev,
                     cudaGetErrorString(e));
    addr[dev] = (double*)ptr;
    ctx_of[dev] = current_context();  // the lookup made the primary context current
  }
  *out = addr[dev];
  return LBM_OK;
}

template <typename T>
int get_post_state_t(lbm_mix* h, T* f, long n) {
  int st = check_handle(h);
  if (st) return st;
  const long need = 18L * h->L.N * h->L.Nx;
  if (!f || n != need) return set_err(LBM_EINVAL, "need %ld populations", need);
  const size_t bytes = sizeof(T) * (size_t)need;
  // staging area sized for the FP64 variant, shared by both getters
  if (!h->scratch) CK(cudaMalloc((void**)&h->scratch, sizeof(double) * (size_t)need));
  dim3 blk(128), grd((h->L.Nx + 127) / 128, h->L.N, 2);
  if ((st = with_storage(h, [&](auto tag) -> int {
         using ST = decltype(tag);
         lbm_convert_kernel<ST, T><<<grd, blk, 0, h->stream>>>(h->L, (ST*)h->buf[h->cur],
                                                               h->refrho, 0, nullptr,
                                                               (T*)h->scratch);
         CK(cudaGetLastError());
         return LBM_OK;
       })))
    return st;
  CK(cudaMemcpyAsync(f, h->scratch, bytes, cudaMemcpyDeviceToHost, h->stream));
  CK(wait_stream(h));
  return LBM_OK;
}

extern "C" {

void lbm_mix_default_params(lbm_mix_params* p) {
  if (!p) return;
  memset(p, 0, sizeof *p);
  p->m_a = 4.003;
  p->m_b = 39.948;
  p->C_l = 0.5;
  p->C_l_out = -1.0;
  p->theta = 2.0;
  p->Kn_out = 0.1;
  p->N = 16;
  p->N_x = 0;
  p->L_over_H = 20.0;
  p->accommodation = 1.0;
  p->c_m0 = 1.016;
  p->tau_rho = 1.0;
  p->tau_e = 1.1;
  p->tau_eps = 1.2;
  p->mu_ratio_a = 1.0;
  p->mu_ratio_b = 1.0;
  p->storage = LBM_FP32;
  p->x_periodic = 0;
  p->diag_every = 1;
  p->reref_every = -1;
  p->rounding = LBM_ROUND_STOCHASTIC;
  p->wall = LBM_WALL_DBB;
}

const char* lbm_mix_strerror(int s) {
  switch (s) {
    case LBM_OK: return "success";
    case LBM_EINVAL: return "invalid argument";
    case LBM_ENOMEM: return "out of memory";
    case LBM_ECUDA: return "CUDA error";
    case LBM_ENONFINITE: return "non-finite value in the state";
    case LBM_ENOTCONVERGED: return "not converged within max_steps";
    case LBM_ETIMEOUT: return "device wait timed out";
    default: return "unknown status";
  }
}

const char* lbm_mix_last_error(void) { return g_err; }

void lbm_mix_destroy(lbm_mix* h) {
  if (!h) return;
  int prev = 0;
  cudaGetDevice(&prev);
  cudaSetDevice(h->device);
  if (h->stream) cudaStreamSynchronize(h->stream);
  cudaFree(h->arena);
  if (h->colpart != h->colpart0) cudaFree(h->colpart);
  cudaFree(h->scratch);
  cudaFree(h->mom);
  if (h->h_pinned) cudaFreeHost(h->h_pinned);
  if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
  cudaSetDevice(prev);
  delete h;
}

int lbm_mix_create(const lbm_mix_params* p, void* stream, lbm_mix** out) {
  if (!out) return set_err(LBM_EINVAL, "out is NULL");
  *out = nullptr;
  int Nx = 0;
  int st = validate(p, &Nx);
  if (st != LBM_OK) return st;
  lbm_mix* h = new (std::nothrow) lbm_mix;
  if (!h) return set_err(LBM_ENOMEM, "host allocation failed");
  memset(h, 0, sizeof *h);
  h->p = *p;
  h->L = derive(p, Nx);
  if (cudaGetDevice(&h->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&h->nsm, cudaDevAttrMultiProcessorCount, h->device) != cudaSuccess) {
    delete h;
    return set_err(LBM_ECUDA, "no CUDA device");
  }
  h->nblocks = (Nx + TX - 1) / TX;
  if (stream) {
    h->stream = (cudaStream_t)stream;
  } else {
    if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess) {
      delete h;
      return set_err(LBM_ECUDA, "cudaStreamCreate failed");
    }
    h->own_stream = true;
  }
  h->elem = (p->storage == LBM_FP32) ? sizeof(float) : 2;
  const size_t fbytes = h->elem * 18 * (size_t)h->L.N * h->L.pitch;
  const size_t cbytes = sizeof(double) * 4 * (size_t)Nx;
  cudaError_t e = cudaSuccess;
  // Row blocks: each strip's rows are split over R CTAs (default_rows).
  h->rows_per_block = default_rows(h);
  h->R = (h->L.N + h->rows_per_block - 1) / h->rows_per_block;
  h->R_alloc = h->R;
  if (p->storage == LBM_FP32) {
    double us = 0.0;
    plan_tiles(h->L, h->nsm, &h->tile_W, &h->tile_k, &us);
    if (us > step_kernel_cost(h->L.N, Nx)) h->tile_W = 0;
    if (h->tile_W > 0) {
      const long fit = HIST_BYTES / (long)(sizeof(float2) * 4 * (size_t)Nx);
      h->hist_rows = (int)(fit < TILE_KMAX + 1 ? TILE_KMAX + 1 : fit < 256 ? fit : 256);
      e = cudaFuncSetAttribute(lbm_tile_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               TILE_SMEM_MAX);
    }
  }
  // One allocation holds every array of the handle (twenty calls took most of
  // lbm_mix_create); the row-block partials can grow and may move out of it.
  // Arrays that start at zero come first.
  size_t zeroed = 0, total = 0;
  auto carve = [&](char* base, size_t bytes, auto** ptr) {
    if (base) *ptr = (std::remove_reference_t<decltype(*ptr)>)(base + total);
    total += (bytes + 255) / 256 * 256;
  };
  auto layout = [&](char* base) {
    total = 0;
    carve(base, fbytes, &h->buf[0]);
    carve(base, fbytes, &h->buf[1]);
    carve(base, sizeof(unsigned), &h->counter);
    carve(base, sizeof(unsigned) * (size_t)h->nblocks, &h->strip_cnt);
    carve(base, cbytes, &h->cs[0]);
    carve(base, cbytes, &h->cs[1]);
    carve(base, sizeof(unsigned long long), &h->diag_count);
    carve(base, sizeof(double) * DIAG_CAP * NREC, &h->diag);
    if (h->tile_W > 0) carve(base, sizeof(unsigned) * h->hist_rows, &h->rec_cnt);
    zeroed = total;
    carve(base, sizeof(float) * 2 * (size_t)Nx, &h->refrho);
    carve(base, sizeof(float) * 2 * (size_t)Nx, &h->refrho_alt);
    carve(base, sizeof(float) * 2 * (size_t)Nx, &h->alpha);
    carve(base, cbytes, &h->cs_tmp);
    carve(base, cbytes, &h->cs_snap);
    carve(base, sizeof(double) * NPART * (size_t)h->nblocks, &h->partials);
    carve(base, sizeof(double) * (size_t)Nx, &h->clprof);
    carve(base, sizeof(float2) * 2 * (size_t)Nx, &h->wall_r);
    carve(base, sizeof(float) * 2 * (size_t)Nx, &h->wall_omq);
    if (p->storage == LBM_FP32 && !p->x_periodic)
      carve(base, sizeof(float2) * 4 * (size_t)h->L.N, &h->end_sd);
    carve(base, sizeof(float2) * 4 * (size_t)Nx * (size_t)h->R, &h->colpart0);
    if (h->tile_W > 0) {
      carve(base, sizeof(float2) * 4 * (size_t)Nx * h->hist_rows, &h->hist);
      carve(base, sizeof(double) * NPART * record_blocks(Nx) * (size_t)h->hist_rows, &h->rec_part);
    }
  };
  layout(nullptr);
  if (e == cudaSuccess) e = cudaMalloc((void**)&h->arena, total);
  if (e == cudaSuccess) {
    layout((char*)h->arena);
    h->colpart = h->colpart0;
  }
  if (e == cudaSuccess) e = cudaMallocHost((void**)&h->h_pinned,
                                            sizeof(double) * (16 + std::min(Nx, PINNED_COLUMNS)));
  if (e != cudaSuccess) {
    int code = (e == cudaErrorMemoryAllocation) ? LBM_ENOMEM : LBM_ECUDA;
    set_err(code, "allocation failed: %s", cudaGetErrorString(e));
    cudaGetLastError();
    lbm_mix_destroy(h);
    return code;
  }
  // zero, so that padding and ghost columns hold defined values
  e = cudaMemsetAsync(h->arena, 0, zeroed, h->stream);
  if (e == cudaSuccess) {
    float* a = (float*)malloc(sizeof(float) * 4 * Nx);
    if (!a) e = cudaErrorMemoryAllocation;
    else {
      for (int k = 0; k < 2 * Nx; ++k) a[k] = (float)p->accommodation;
      // reference densities: the initial profile of lbm_mix_init
      float* rb = a + 2 * Nx;
      for (int x = 0; x < Nx; ++x) {
        double t = h->L.x_periodic ? 1.0 : (double)x / (Nx - 1);
        double n = h->L.x_periodic ? 1.0 : p->theta + (1.0 - p->theta) * t;
        double Cl = h->L.C_in + (h->L.C_out - h->L.C_in) * t;
        for (int sp = 0; sp < 2; ++sp) {
          double C = (sp == h->L.light) ? Cl : 1.0 - Cl;
          rb[sp * Nx + x] = (float)(n * C * h->L.mh[sp]);
        }
      }
      e = cudaMemcpyAsync(h->alpha, a, sizeof(float) * 2 * Nx, cudaMemcpyHostToDevice, h->stream);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(h->refrho, rb, sizeof(float) * 2 * Nx, cudaMemcpyHostToDevice,
                            h->stream);
      if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
      free(a);
    }
  }
  if (e != cudaSuccess) {
    set_err(LBM_ECUDA, "initialisation failed: %s", cudaGetErrorString(e));
    lbm_mix_destroy(h);
    return LBM_ECUDA;
  }
  *out = h;
  return LBM_OK;
}

int lbm_mix_init(lbm_mix* h) {
  int st = check_handle(h);
  if (st) return st;
  h->cur = 0;
  h->steps = 0;
  // the initial state is the rest equilibrium of the reference densities:
  // all stored deviations are zero
  CK(cudaMemsetAsync(h->buf[0], 0, h->elem * 18 * (size_t)h->L.N * h->L.pitch,
                     h->stream));
  if ((st = launch_colsum(h, 0))) return st;
  return reset_diag(h);
}

int lbm_mix_step(lbm_mix* h, long nsteps) {
  int st = check_handle(h);
  if (st) return st;
  if (nsteps < 0) return set_err(LBM_EINVAL, "nsteps < 0");
  const long reref = h->p.reref_every >= 0 ? h->p.reref_every
                                           : (h->p.storage == LBM_FP32 ? 0 : 256);
  if (uses_tiles(h)) {
    for (long left = nsteps; left > 0;) {
      long n = left;
      if (reref > 0 && n > reref - h->steps % reref) n = reref - h->steps % reref;
      if ((st = tile_steps<1>(&h, &h->tile_W, 1, h->tile_k, n, n == left, h->stream))) return st;
      if (reref > 0 && h->steps % reref == 0 && (st = rereference(h))) return st;
      left -= n;
    }
    return LBM_OK;
  }
  // diagnostics on every diag_every-th step and on the last step of the call
  for (long t = 0; t < nsteps; ++t) {
    const bool diag = (t == nsteps - 1) || ((h->steps + 1) % h->p.diag_every == 0);
    if ((st = launch_step(h, diag))) return st;
    if (reref > 0 && h->steps % reref == 0 && (st = rereference(h))) return st;
  }
  return LBM_OK;
}

int lbm_mix_rereference(lbm_mix* h) {
  int st = check_handle(h);
  if (st) return st;
  return rereference(h);
}

int lbm_mix_run_to_steady(lbm_mix* h, double tol, long max_steps, long check_every,
                          long* steps_out, double* residual_out) {
  int st = check_handle(h);
  if (st) return st;
  if (!(tol > 0) || max_steps < 0 || check_every < 1)
    return set_err(LBM_EINVAL, "need tol > 0, max_steps >= 0, check_every >= 1");
  long taken = 0;
  double R = INFINITY;
  int result = LBM_ENOTCONVERGED;
  while (taken < max_steps) {
    long k = check_every < max_steps - taken ? check_every : max_steps - taken;
    if ((st = lbm_mix_step(h, k))) return st;
    taken += k;
    if ((st = launch_residual(h, k))) return st;
    CK(wait_stream(h));
    R = h->h_pinned[0];
    if (isnan(R)) {
      result = set_err(LBM_ENONFINITE, "non-finite residual after %ld steps", taken);
      break;
    }
    if (R <= tol) {
      result = LBM_OK;
      break;
    }
  }
  if (steps_out) *steps_out = taken;
  if (residual_out) *residual_out = R;
  if (result == LBM_ENOTCONVERGED)
    set_err(LBM_ENOTCONVERGED, "residual %.3e above %.3e after %ld steps", R, tol, taken);
  return result;
}

int lbm_mix_set_rows_per_block(lbm_mix* h, int rows) {
  int st = check_handle(h);
  if (st) return st;
  if ((st = set_rows_per_block(h, rows))) return st;
  h->rows_set = rows > 0;
  return LBM_OK;
}

int lbm_mix_tune_rows(lbm_mix* h, const int* candidates, int n, long steps, int* best_rows) {
  int st = check_handle(h);
  if (st) return st;
  static const int kDefault[] = {64, 72, 80, 88, 96, 112, 128};
  const bool own_list = !candidates;
  if (own_list) {
    candidates = kDefault;
    n = (int)(sizeof kDefault / sizeof kDefault[0]);
  }
  if (n < 1 || steps < 1) return set_err(LBM_EINVAL, "need n >= 1 candidates and steps >= 1");
  for (int k = 0; k < n; ++k)
    if (candidates[k] <= 0 || candidates[k] % TY != 0)
      return set_err(LBM_EINVAL, "candidate %d: rows must be a positive multiple of %d", k, TY);
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    if (e0) cudaEventDestroy(e0);
    return set_err(LBM_ECUDA, "cudaEventCreate failed");
  }
  int best = h->rows_set ? h->rows_per_block : 0;  // 0: the default schedule
  float best_ms = INFINITY;
  // the library's own list is of counts beyond its default's, which it tries first
  for (int k = own_list ? -1 : 0; k < n && st == LBM_OK; ++k) {
    const int rows = k < 0 ? 0 : candidates[k];
    if ((st = lbm_mix_set_rows_per_block(h, rows))) break;
    // two untimed steps settle the new schedule (first-touch of its buffers)
    if ((st = lbm_mix_step(h, 2))) break;
    if (cudaEventRecord(e0, h->stream) != cudaSuccess ||
        (st = lbm_mix_step(h, steps)) != LBM_OK || cudaEventRecord(e1, h->stream) != cudaSuccess ||
        cudaEventSynchronize(e1) != cudaSuccess) {
      if (st == LBM_OK) st = set_err(LBM_ECUDA, "timing a candidate schedule failed");
      break;
    }
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (ms < best_ms) {
      best_ms = ms;
      best = rows == 0 ? 0 : h->rows_per_block;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st) return st;
  if ((st = lbm_mix_set_rows_per_block(h, best))) return st;
  if (best_rows) *best_rows = best;
  return LBM_OK;
}

int lbm_mix_moments_device(lbm_mix* h, double* d_out) {
  int st = check_handle(h);
  if (st) return st;
  if (!d_out) return set_err(LBM_EINVAL, "d_out is NULL");
  return launch_moments(h, d_out);
}

int lbm_mix_moments(lbm_mix* h, double* rho_a, double* rho_b, double* ua_x, double* ua_y,
                    double* ub_x, double* ub_y) {
  int st = check_handle(h);
  if (st) return st;
  const size_t plane = (size_t)h->L.N * h->L.Nx;
  if (!h->mom) CK(cudaMalloc((void**)&h->mom, sizeof(double) * 6 * plane));
  if ((st = launch_moments(h, h->mom))) return st;
  double* outs[6] = {rho_a, rho_b, ua_x, ua_y, ub_x, ub_y};
  for (int k = 0; k < 6; ++k)
    if (outs[k])
      CK(cudaMemcpyAsync(outs[k], h->mom + k * plane, sizeof(double) * plane,
                         cudaMemcpyDeviceToHost, h->stream));
  CK(wait_stream(h));
  return LBM_OK;
}

int lbm_mix_device_ptrs(lbm_mix* h, void** populations, long* n_populations, void** refrho,
                        void** alpha, void** colsum) {
  int st = check_handle(h);
  if (st) return st;
  if (populations) *populations = h->buf[h->cur];
  if (n_populations) *n_populations = 18L * h->L.N * h->L.pitch;
  if (refrho) *refrho = h->refrho;
  if (alpha) *alpha = h->alpha;
  if (colsum) *colsum = h->cs[h->cur];
  return LBM_OK;
}

int lbm_mix_volume_flow(lbm_mix* h, int x, double* Qv) {
  int st = check_handle(h);
  if (st) return st;
  if (!Qv) return set_err(LBM_EINVAL, "Qv is NULL");
  if (x < 0) x = h->L.x_periodic ? 0 : h->L.Nx - 2;
  if (x >= h->L.Nx || (!h->L.x_periodic && (x < 1 || x > h->L.Nx - 2)))
    return set_err(LBM_EINVAL, "column %d is not an updated column", x);
  // the state of step n is the stream of buffer P_{n-1} (launch_moments)
  const int direct = h->steps == 0 ? 1 : 0, b = direct ? h->cur : 1 - h->cur;
  st = with_storage(h, [&](auto tag) -> int {
    using ST = decltype(tag);
    lbm_volume_flow_kernel<ST><<<1, 256, 0, h->stream>>>(h->L, (const ST*)h->buf[b], h->refrho,
                                                         h->cs[b], h->alpha, direct, x,
                                                         h->h_pinned);
    CK(cudaGetLastError());
    return LBM_OK;
  });
  if (st) return st;
  CK(wait_stream(h));
  *Qv = h->h_pinned[0];
  if (!isfinite(*Qv)) return set_err(LBM_ENONFINITE, "non-finite volume flow");
  return LBM_OK;
}

int lbm_mix_separation(lbm_mix* h, double* CL, double* Cl_tilde, double* mdot_a, double* mdot_b,
                       double* Cl_profile, int* x_min) {
  int st = check_handle(h);
  if (st) return st;
  double rec[NREC];
  if ((st = latest_record(h, rec, Cl_profile))) return st;
  if (CL) *CL = rec[1];
  if (Cl_tilde) *Cl_tilde = rec[2];
  if (mdot_a) *mdot_a = rec[3];
  if (mdot_b) *mdot_b = rec[4];
  if (x_min) *x_min = (int)rec[5];
  return LBM_OK;
}

int lbm_mix_history(lbm_mix* h, double* rec, long max_records, long* count) {
  int st = check_handle(h);
  if (st) return st;
  if (!rec || max_records < 0 || !count) return set_err(LBM_EINVAL, "bad history arguments");
  unsigned long long cnt = 0;
  CK(cudaMemcpyAsync(&cnt, h->diag_count, sizeof cnt, cudaMemcpyDeviceToHost, h->stream));
  CK(wait_stream(h));
  long have = (long)(cnt < (unsigned long long)DIAG_CAP ? cnt : DIAG_CAP);
  long take = have < max_records ? have : max_records;
  for (long k = 0; k < take; ++k) {
    unsigned long long idx = (cnt - take + k) % DIAG_CAP;
    CK(cudaMemcpyAsync(rec + k * NREC, h->diag + idx * NREC, sizeof(double) * NREC,
                       cudaMemcpyDeviceToHost, h->stream));
  }
  CK(wait_stream(h));
  *count = take;
  return LBM_OK;
}

int lbm_mix_set_accommodation_field(lbm_mix* h, const double* alpha, long n) {
  int st = check_handle(h);
  if (st) return st;
  if (!alpha || n != 2L * h->L.Nx) return set_err(LBM_EINVAL, "need 2*N_x accommodation values");
  float* a = (float*)malloc(sizeof(float) * n);
  if (!a) return set_err(LBM_ENOMEM, "host allocation failed");
  for (long k = 0; k < n; ++k) {
    if (!(alpha[k] > 0 && alpha[k] <= 1)) {
      free(a);
      return set_err(LBM_EINVAL, "accommodation[%ld] = %g outside (0,1]", k, alpha[k]);
    }
    a[k] = (float)alpha[k];
  }
  cudaError_t e = cudaMemcpyAsync(h->alpha, a, sizeof(float) * n, cudaMemcpyHostToDevice, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  free(a);
  if (e != cudaSuccess) return set_err(LBM_ECUDA, "upload failed: %s", cudaGetErrorString(e));
  return LBM_OK;
}

int lbm_mix_set_post_state(lbm_mix* h, const float* f, long n) {
  int st = check_handle(h);
  if (st) return st;
  const long need = 18L * h->L.N * h->L.Nx;
  if (!f || n != need) return set_err(LBM_EINVAL, "need %ld populations", need);
  h->cur = 0;
  h->steps = 0;
  if (!h->scratch) CK(cudaMalloc((void**)&h->scratch, sizeof(double) * (size_t)need));
  CK(cudaMemcpyAsync(h->scratch, f, sizeof(float) * (size_t)need, cudaMemcpyHostToDevice,
                     h->stream));
  {
    dim3 blk(128), grd((h->L.Nx + 127) / 128, h->L.N, 2);
    if ((st = with_storage(h, [&](auto tag) -> int {
           using ST = decltype(tag);
           lbm_convert_kernel<ST, float><<<grd, blk, 0, h->stream>>>(
               h->L, (ST*)h->buf[0], h->refrho, 1, (const float*)h->scratch, (float*)nullptr);
           CK(cudaGetLastError());
           return LBM_OK;
         })))
      return st;
  }
  if ((st = launch_colsum(h, 0))) return st;
  if ((st = reset_diag(h))) return st;
  CK(wait_stream(h));
  return LBM_OK;
}

int lbm_mix_get_post_state(lbm_mix* h, float* f, long n) { return get_post_state_t(h, f, n); }

int lbm_mix_get_post_state_f64(lbm_mix* h, double* f, long n) {
  return get_post_state_t(h, f, n);
}

int lbm_mix_dims(const lbm_mix* h, int* N, int* N_x, long* steps) {
  int st = check_handle(h);
  if (st) return st;
  if (N) *N = h->L.N;
  if (N_x) *N_x = h->L.Nx;
  if (steps) *steps = h->steps;
  return LBM_OK;
}

int lbm_mix_launches_per_step(const lbm_mix* h) {
  int st = check_handle(h);
  if (st) return st;
  const bool tiles = uses_tiles(h) && h->L.Nx <= SINGLE_STEP_COLUMNS;
  return (h->elem < 4 || tiles || uses_wall_kernel(h)) ? 2 : 1;
}

long lbm_mix_launches(const lbm_mix* h) {
  int st = check_handle(h);
  return st ? st : h->launches;
}

int lbm_mix_sync(lbm_mix* h) {
  int st = check_handle(h);
  if (st) return st;
  CK(wait_stream(h));
  return LBM_OK;
}

int lbm_mix_eval_special(const double* x, double* e1, double* psi, long n) {
  if (!x || n < 0) return set_err(LBM_EINVAL, "bad arguments");
  if (n == 0) return LBM_OK;
  for (long k = 0; k < n; ++k)
    if (!(x[k] > 0)) return set_err(LBM_EINVAL, "x[%ld] must be > 0", k);
  double *dx = nullptr, *de = nullptr, *dp = nullptr;
  const size_t b = sizeof(double) * n;
  cudaError_t e = cudaMalloc((void**)&dx, b);
  if (e == cudaSuccess) e = cudaMalloc((void**)&de, b);
  if (e == cudaSuccess) e = cudaMalloc((void**)&dp, b);
  if (e == cudaSuccess) e = cudaMemcpy(dx, x, b, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    lbm_special_kernel<<<(unsigned)((n + 255) / 256), 256>>>(dx, de, dp, n);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && e1) e = cudaMemcpy(e1, de, b, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && psi) e = cudaMemcpy(psi, dp, b, cudaMemcpyDeviceToHost);
  cudaFree(dx);
  cudaFree(de);
  cudaFree(dp);
  if (e != cudaSuccess) return set_err(LBM_ECUDA, "eval_special: %s", cudaGetErrorString(e));
  return LBM_OK;
}

int lbm_mix_step_noalloc(const lbm_mix_params* p, const float* d_in, float* d_out,
                         const float* d_refrho, const float* d_alpha, const double* d_colsum_in,
                         double* d_colsum_out, double* d_record, double* d_cl_profile,
                         void* stream) {
  int Nx = 0;
  int st = validate(p, &Nx);
  if (st != LBM_OK) return st;
  if (!d_in || !d_out || !d_refrho || !d_alpha || !d_colsum_in || !d_colsum_out || !d_record ||
      !d_cl_profile)
    return set_err(LBM_EINVAL, "lbm_mix_step_noalloc: every buffer must be a device pointer");
  if (d_in == d_out) return set_err(LBM_EINVAL, "lbm_mix_step_noalloc: d_in and d_out alias");
  if (p->storage != LBM_FP32)
    return set_err(LBM_EINVAL, "lbm_mix_step_noalloc: FP32 storage only");
  const int nstrips = (Nx + TX - 1) / TX;
  if (nstrips > NOALLOC_MAX_STRIPS)
    return set_err(LBM_EINVAL,
                   "lbm_mix_step_noalloc: N_x = %d exceeds the %d columns its static scratch "
                   "covers",
                   Nx, NOALLOC_MAX_STRIPS * TX);
  double* scratch = nullptr;
  if ((st = noalloc_scratch_address(&scratch))) return st;
  const Lat L = derive(p, Nx);
  cudaStream_t s = (cudaStream_t)stream;
  unsigned* cnt = (unsigned*)(scratch + NOALLOC_PART_DOUBLES);
  // tickets and the record counter must start at zero; the partials are
  // overwritten before they are read
  CK(cudaMemsetAsync(cnt, 0, sizeof(unsigned) * NOALLOC_CNT_WORDS, s));
  StepArgs<float> a;
  a.fin = d_in;
  a.fout = d_out;
  a.refrho = d_refrho;
  a.cs_in = d_colsum_in;
  a.cs_out = d_colsum_out;
  a.alpha = d_alpha;
  a.partials = scratch;
  a.strip_cnt = cnt;
  a.counter = cnt + NOALLOC_MAX_STRIPS;
  a.diag_count = (unsigned long long*)(cnt + NOALLOC_MAX_STRIPS + 2);
  a.diag = d_record;  // the zeroed counter puts the record at index 0
  a.clprof = d_cl_profile;
  a.colpart = nullptr;  // one row block per strip: no row-block partials
  a.rows_per_block = (L.N + TY - 1) / TY * TY;
  a.seed = 0u;  // FP32 storage: no rounding to 16 bits
  a.wall_r = nullptr;  // FP32 storage: the wall prologue computes r and tau_q
  a.wall_omq = nullptr;
  a.end_sd = nullptr;  // no room in the scratch: sums by row blocks
  dim3 blk(TX, TY), grd(nstrips, 1);
  lbm_step_kernel<float, true><<<grd, blk, 0, s>>>(L, a);
  CK(cudaGetLastError());
  return LBM_OK;
}

}  // extern "C"

// ---------------------------------------------------------------- sweeps
// A parametric study (Table 1) runs many independent channels, each too small
// to fill the GPU.  A sweep advances all of them by common launches on a
// stream of its own, its handles keep theirs for calls of their own: the channels that fit tiles by lbm_tile_kernel, k steps a launch,
// in tiles wide enough that the redundant halo work stays small; the others
// by lbm_step_batch_kernel, one step a launch; then one launch each for the
// records and for the residuals of a convergence check.  The launches carry
// every channel's constants and pointers as kernel parameters, so each call
// starts from the handles' state as it is.  The first blocks of
// lbm_sweep_run_to_steady can serve as an autotuner of the node-to-CTA
// schedule: each candidate runs one real block of steps, the fastest is kept.
// Schedules change only the order of the column sums, not the time
// integration.
struct lbm_sweep {
  int n = 0;
  lbm_mix** h = nullptr;
  cudaStream_t stream = nullptr;
  cudaEvent_t joined = nullptr;  // see join_handles
  double* h_resid = nullptr;  // [n] residuals of a check, pinned
  int policy = -1;            // schedule in use (-1: the library default)
  double round_ms[LBM_SWEEP_NPOLICY] = {};
};

namespace {

// Channels of one launch (the parameters of a launch end at 32 764 bytes).
constexpr int TILE_BATCH = 96, STEP_BATCH = 32;
static_assert(sizeof(TileBatch<TILE_BATCH>) <= 32764 && sizeof(StepBatch<STEP_BATCH>) <= 32764 &&
                  sizeof(RecBatch<TILE_BATCH>) <= 32764,
              "kernel parameters");

// Rows per CTA of instance h under schedule policy p.
int policy_rows(const lbm_mix* h, int p) {
  const int N = h->L.N;
  switch (p) {
    case 0: return 0;  // library default
    case 1: return 64;
    case 2: return 32;
    case 3: return 16;
    default: {  // fill: about two CTAs per SM for this instance alone
      const long want = 2L * (h->nsm > 0 ? h->nsm : 1);
      long rows = ((long)N * h->nblocks + want - 1) / want;
      rows = (rows + TY - 1) / TY * TY;
      if (rows < 16) rows = 16;
      if (rows > 128) rows = 128;
      return (int)rows;
    }
  }
}

int apply_policy(lbm_sweep* s, int p) {
  for (int i = 0; i < s->n; ++i) {
    int st = set_rows_per_block(s->h[i], policy_rows(s->h[i], p));
    if (st) return st;
    s->h[i]->rows_set = p > 0;
  }
  s->policy = p;
  return LBM_OK;
}

// Estimated time (us) of one step of channels with that many nodes in all by
// lbm_step_batch_kernel: 8 us of launch, start-up and tail, then 38 G nodes/s.
double batch_step_cost(double nodes) { return 8.0 + nodes * 2.6e-5; }

// Tile widths W[] and steps per launch of n channels of equal N advanced
// together: for each k and each bound on a tile's nodes the estimate of
// tile_cost with the channels' tiles sharing the waves, the least one kept.
// Returns that estimate (us per step).
double plan_batch(lbm_mix* const* hs, int n, int* W, int* k_out) {
  const int sms = hs[0]->nsm > 0 ? hs[0]->nsm : 1, N = hs[0]->L.N, S = tile_stride(N);
  int most = 0;  // columns of the largest tile
  while (tile_smem(N, most + 1) <= (size_t)TILE_SMEM_MAX) ++most;
  auto updated = [](const Lat& L) { return L.x_periodic ? L.Nx : L.Nx - 2; };
  double best = INFINITY;
  int best_w = 1;
  *k_out = 1;
  for (int k = 1; k <= TILE_KMAX && 2 * k < most; k += 2)
    for (int w = most - 2 * k; w >= 1; w -= w > 8 ? w / 8 : 1) {
      long tiles = 0;
      for (int q = 0; q < n; ++q) tiles += (updated(hs[q]->L) + w - 1) / w;
      const double us = (TILE_LAUNCH_US +
                         (double)((tiles + sms - 1) / sms) *
                             (TILE_LOAD_US + k * TILE_STEP_US +
                              TILE_NODE_US * k * (w + k - 1) * (double)S)) / k;
      if (us < best) {
        best = us;
        best_w = w;
        *k_out = k;
      }
    }
  for (int q = 0; q < n; ++q) {  // tiles of even width
    const int nup = updated(hs[q]->L), tiles = (nup + best_w - 1) / best_w;
    W[q] = (nup + tiles - 1) / tiles;
  }
  return best;
}

// One step of the n <= STEP_BATCH channels hs; end: it ends the call.
int launch_step_batch(lbm_mix* const* hs, int n, bool end, cudaStream_t st) {
  StepBatch<STEP_BATCH> B;
  // rows per CTA for some eight waves of the whole launch's CTAs, but no fewer
  // than a channel's own schedule has: with 2 to 8 waves 24 mixed channels, 33 of
  // 500 x 256, 12 of 3000 x 600 and 96 of 1000 x 64 are within 2 % of each other,
  // with 16 3 to 6 % slower (two of 5001 x 130: 39.7 us at 3, 42.5 at 8)
  long strip_rows = 0;
  for (int q = 0; q < n; ++q) strip_rows += (long)hs[q]->L.N * hs[q]->nblocks;
  const long most = (strip_rows / (8 * 3L * (hs[0]->nsm > 0 ? hs[0]->nsm : 1)) + TY - 1) / TY * TY;
  int blocks = 0, walls = 0;
  for (int q = 0; q < STEP_BATCH; ++q) {
    B.block0[q] = blocks;
    B.wall0[q] = walls;
    if (q >= n) continue;
    lbm_mix* h = hs[q];
    StepInst& I = B.inst[q];
    I.L = h->L;
    I.a = step_args<float>(h);
    if (!h->rows_set) {
      const long n8 = (h->L.N + TY - 1) / TY * TY, rows = most < 56 ? most : 56;
      if (rows > I.a.rows_per_block) I.a.rows_per_block = (int)(rows < n8 ? rows : n8);
    }
    I.strips = h->nblocks;
    I.blocks = (h->L.N + I.a.rows_per_block - 1) / I.a.rows_per_block;
    I.diag = end || (h->steps + 1) % h->p.diag_every == 0;
    blocks += I.strips * I.blocks;
    walls += (h->L.Nx + WALL_COLS - 1) / WALL_COLS;
    I.wall_r = h->wall_r;
    I.wall_omq = h->wall_omq;
  }
  B.block0[STEP_BATCH] = blocks;
  B.wall0[STEP_BATCH] = walls;
  int s = LBM_OK;
  if (blocks < WALL_KERNEL_WAVES_SET * 3L * (hs[0]->nsm > 0 ? hs[0]->nsm : 1)) {
    s = launch_batch(lbm_step_batch_kernel<STEP_BATCH, false>, B, dim3(blocks), dim3(TX, TY), 0,
                     st);
  } else {
    s = launch_batch(lbm_walls_batch_kernel<STEP_BATCH>, B, dim3(walls, 4), dim3(WALL_COLS), 0, st);
    if (!s)
      s = launch_batch(lbm_step_batch_kernel<STEP_BATCH, true>, B, dim3(blocks), dim3(TX, TY), 0,
                       st);
  }
  if (s) return s;
  for (int q = 0; q < n; ++q) {
    hs[q]->cur = 1 - hs[q]->cur;
    hs[q]->steps++;
  }
  return LBM_OK;
}

// Lets the sweep's stream wait for what calls on its handles left on theirs.
// (The other way round every call of a sweep ends with a wait of the host.)
int join_handles(lbm_sweep* s) {
  for (int i = 0; i < s->n; ++i) {
    lbm_mix* h = s->h[i];
    if (!h->pending) continue;
    CK(cudaEventRecord(s->joined, h->stream));
    CK(cudaStreamWaitEvent(s->stream, s->joined, 0));
    h->pending = false;
  }
  return LBM_OK;
}

// nsteps steps of the n channels hs of a sweep, on its stream.  Channels that
// qualify for tiles take them, grouped by N, unless one step kernel over all
// channels is estimated to be faster (many nodes in all, or tall channels) or
// the call has one or two steps of more than SINGLE_STEP_COLUMNS columns, each of
// which would be a launch of tiles (us per step of calls of two: 8 channels of
// 400 x 32 30.8 by tiles, 18.2 by the step kernel, 3 of 700 x 20 22.0 and 20.6;
// one of 320 x 16 17.1 and 19.5); the populations are the same bits either way.
int batch_steps(lbm_sweep* s, lbm_mix* const* hs, int n, long nsteps) {
  if (nsteps < 1) return LBM_OK;
  lbm_mix** order = (lbm_mix**)malloc(2 * sizeof(lbm_mix*) * (size_t)n);
  int* W = (int*)malloc(sizeof(int) * (size_t)n);
  if (!order || !W) {
    free(order), free(W);
    return set_err(LBM_ENOMEM, "host allocation failed");
  }
  lbm_mix** rest = order + n;  // channels of the step kernel
  int nt = 0, nr = 0, st = LBM_OK;
  double nodes_t = 0.0, nodes_r = 0.0, us = 0.0;
  long columns = 0;
  for (int q = 0; q < n; ++q) {
    columns += hs[q]->L.Nx;
    const double nodes = (double)hs[q]->L.N * hs[q]->L.Nx;
    (uses_tiles(hs[q]) ? nodes_t : nodes_r) += nodes;
    if (uses_tiles(hs[q])) order[nt++] = hs[q];
  }
  std::sort(order, order + nt, [](const lbm_mix* a, const lbm_mix* b) { return a->L.N < b->L.N; });
  auto group_end = [&](int q0) {
    int q = q0;
    while (q < nt && q - q0 < TILE_BATCH && order[q]->L.N == order[q0]->L.N) ++q;
    return q;
  };
  int k = 1;
  for (int q0 = 0, q1; q0 < nt; q0 = q1) us += plan_batch(order + q0, (q1 = group_end(q0)) - q0, W, &k);
  const bool tiles = (nsteps > 2 || columns <= SINGLE_STEP_COLUMNS) &&
                     us + (nodes_r > 0 ? batch_step_cost(nodes_r) : 0.0) <=
                         batch_step_cost(nodes_t + nodes_r);
  for (int q0 = 0, q1; tiles && q0 < nt && !st; q0 = q1) {
    const int m = (q1 = group_end(q0)) - q0;
    plan_batch(order + q0, m, W, &k);
    st = m <= 8 ? tile_steps<8>(order + q0, W, m, k, nsteps, true, s->stream)
                : tile_steps<TILE_BATCH>(order + q0, W, m, k, nsteps, true, s->stream);
  }
  for (int q = 0; q < n; ++q)
    if (!tiles || !uses_tiles(hs[q])) rest[nr++] = hs[q];
  for (int q0 = 0; q0 < nr && !st; q0 += STEP_BATCH)
    for (long t = 1; t <= nsteps && !st; ++t)
      st = launch_step_batch(rest + q0, nr - q0 < STEP_BATCH ? nr - q0 : STEP_BATCH, t == nsteps,
                             s->stream);
  free(order), free(W);
  return st;
}

// Residuals of the n channels hs of a sweep after k steps into s->h_resid, in
// order; waits for them.
int batch_residuals(lbm_sweep* s, lbm_mix* const* hs, int n, long k) {
  for (int q0 = 0; q0 < n; q0 += TILE_BATCH) {
    ResidBatch<TILE_BATCH> B;
    const int m = n - q0 < TILE_BATCH ? n - q0 : TILE_BATCH;
    for (int q = 0; q < m; ++q) {
      lbm_mix* h = hs[q0 + q];
      B.inst[q] = ResidInst{h->cs[h->cur], h->cs_snap, 4L * h->L.Nx, h->have_snap ? 1 : 0};
      h->have_snap = true;
    }
    lbm_residual_kernel<TILE_BATCH><<<m, 1024, 0, s->stream>>>(B, (double)k, s->h_resid + q0);
    CK(cudaGetLastError());
  }
  CK(cudaStreamSynchronize(s->stream));
  return LBM_OK;
}

double now_ms() {
  struct timespec ts;
  clock_gettime(CLOCK_MONOTONIC, &ts);
  return ts.tv_sec * 1e3 + ts.tv_nsec * 1e-6;
}

}  // namespace

extern "C" {

int lbm_sweep_create(const lbm_mix_params* params, int n, lbm_sweep** out) {
  if (!out) return set_err(LBM_EINVAL, "out is NULL");
  *out = nullptr;
  if (!params || n < 1) return set_err(LBM_EINVAL, "need n >= 1 parameter sets");
  for (int i = 0; i < n; ++i) {
    int Nx = 0;
    int st = validate(&params[i], &Nx);
    if (st) {
      char why[sizeof g_err];
      memcpy(why, g_err, sizeof why);
      return set_err(st, "instance %d: %s", i, why);
    }
    if (params[i].storage != LBM_FP32)
      return set_err(LBM_EINVAL, "instance %d: sweeps run FP32 storage only", i);
  }
  lbm_sweep* s = new (std::nothrow) lbm_sweep;
  if (!s) return set_err(LBM_ENOMEM, "host allocation failed");
  s->h = (lbm_mix**)calloc(n, sizeof(lbm_mix*));
  if (!s->h) {
    lbm_sweep_destroy(s);
    return set_err(LBM_ENOMEM, "host allocation failed");
  }
  s->n = n;
  cudaError_t e = cudaStreamCreateWithFlags(&s->stream, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&s->joined, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaMallocHost((void**)&s->h_resid, sizeof(double) * n);
  for (auto kern : {(const void*)lbm_tile_kernel<8>, (const void*)lbm_tile_kernel<TILE_BATCH>})
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, TILE_SMEM_MAX);
  if (e != cudaSuccess) {
    const int code = e == cudaErrorMemoryAllocation ? LBM_ENOMEM : LBM_ECUDA;
    set_err(code, "sweep: %s", cudaGetErrorString(e));
    cudaGetLastError();
    lbm_sweep_destroy(s);
    return code;
  }
  for (int i = 0; i < n; ++i) {
    lbm_mix_params p = params[i];
    p.reref_every = 0;
    int st = lbm_mix_create(&p, nullptr, &s->h[i]);  // a stream of its own
    if (st) {
      lbm_sweep_destroy(s);
      return st;
    }
  }
  *out = s;
  return LBM_OK;
}

void lbm_sweep_destroy(lbm_sweep* s) {
  if (!s) return;
  if (s->stream) cudaStreamSynchronize(s->stream);
  for (int i = 0; i < s->n; ++i)
    if (s->h) lbm_mix_destroy(s->h[i]);
  free(s->h);
  if (s->h_resid) cudaFreeHost(s->h_resid);
  if (s->joined) cudaEventDestroy(s->joined);
  if (s->stream) cudaStreamDestroy(s->stream);
  delete s;
}

int lbm_sweep_init(lbm_sweep* s) {
  if (!s) return set_err(LBM_EINVAL, "sweep is NULL");
  for (int i = 0; i < s->n; ++i) {
    int st = lbm_mix_init(s->h[i]);
    if (st) return st;
  }
  return LBM_OK;
}

int lbm_sweep_step(lbm_sweep* s, long nsteps) {
  if (!s) return set_err(LBM_EINVAL, "sweep is NULL");
  if (nsteps < 0) return set_err(LBM_EINVAL, "nsteps < 0");
  int st = join_handles(s);
  if (!st) st = batch_steps(s, s->h, s->n, nsteps);
  const cudaError_t e = cudaStreamSynchronize(s->stream);  // also after an error
  if (st) return st;
  CK(e);
  return LBM_OK;
}

int lbm_sweep_run_to_steady(lbm_sweep* s, double tol, long max_steps, long check_every,
                            int autotune, long* steps_out, double* residual_out,
                            int* status_out) {
  if (!s) return set_err(LBM_EINVAL, "sweep is NULL");
  if (!(tol > 0) || max_steps < 0 || check_every < 2 || check_every % 2 != 0)
    return set_err(LBM_EINVAL, "need tol > 0, max_steps >= 0, even check_every >= 2");
  const int n = s->n;
  long* taken = (long*)calloc(n, sizeof(long));
  double* R = (double*)malloc(n * sizeof(double));
  int* status = (int*)malloc(n * sizeof(int));
  int* act = (int*)malloc(n * sizeof(int));
  lbm_mix** hs = (lbm_mix**)malloc(n * sizeof(lbm_mix*));
  if (!taken || !R || !status || !act || !hs) {
    free(taken), free(R), free(status), free(act), free(hs);
    return set_err(LBM_ENOMEM, "host allocation failed");
  }
  int na = 0;
  for (int i = 0; i < n; ++i) {
    R[i] = INFINITY;
    status[i] = LBM_ENOTCONVERGED;
    // one diagnostic record per check block
    s->h[i]->p.diag_every = (int)check_every;
    if (max_steps > 0) act[na++] = i;
  }
  int st = join_handles(s);
  int trial = autotune ? 0 : -1;  // next schedule to try
  if (st == LBM_OK && !autotune && s->policy < 0) st = apply_policy(s, 0);
  while (na > 0 && st == LBM_OK) {
    if (trial >= 0 && (st = apply_policy(s, trial))) break;
    // every active instance advances k steps
    const long left = max_steps - taken[act[0]];
    const long k = check_every < left ? check_every : left;
    for (int a = 0; a < na; ++a) hs[a] = s->h[act[a]];
    const double t0 = now_ms();
    if ((st = batch_steps(s, hs, na, k)) || (st = batch_residuals(s, hs, na, k))) break;
    int nb = 0;
    for (int a = 0; a < na; ++a) {
      const int i = act[a];
      taken[i] += k;
      R[i] = s->h_resid[a];
      if (isnan(R[i])) status[i] = LBM_ENONFINITE;
      else if (R[i] <= tol) status[i] = LBM_OK;
      else if (taken[i] < max_steps) act[nb++] = i;
    }
    if (trial >= 0) {
      s->round_ms[trial] = now_ms() - t0;
      if (++trial == LBM_SWEEP_NPOLICY) {
        int best = 0;
        for (int p = 1; p < LBM_SWEEP_NPOLICY; ++p)
          if (s->round_ms[p] < s->round_ms[best]) best = p;
        trial = -1;
        st = apply_policy(s, best);
      }
    }
    na = nb;
  }
  if (st) cudaStreamSynchronize(s->stream);
  for (int i = 0; i < n; ++i) {
    if (steps_out) steps_out[i] = taken[i];
    if (residual_out) residual_out[i] = R[i];
    if (status_out) status_out[i] = status[i];
  }
  free(taken), free(R), free(status), free(act), free(hs);
  return st;
}

int lbm_sweep_instance(lbm_sweep* s, int k, lbm_mix** out) {
  if (!s || !out || k < 0 || k >= s->n) return set_err(LBM_EINVAL, "bad sweep, index or out");
  *out = s->h[k];
  return LBM_OK;
}

int lbm_sweep_schedule(lbm_sweep* s, int* policy, int* rows_per_block, double* round_ms) {
  if (!s) return set_err(LBM_EINVAL, "sweep is NULL");
  if (policy) *policy = s->policy;
  if (rows_per_block)
    for (int i = 0; i < s->n; ++i) rows_per_block[i] = s->h[i]->rows_per_block;
  if (round_ms)
    for (int p = 0; p < LBM_SWEEP_NPOLICY; ++p) round_ms[p] = s->round_ms[p];
  return LBM_OK;
}

}  // extern "C"

// ------------------------------------------- helpers for other translation units
#include "lbm_internal.h"

int lbm_internal_error(int code, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof g_err, fmt, ap);
  va_end(ap);
  return code;
}

int lbm_internal_validate(const lbm_mix_params* p, int* Nx_out) { return validate(p, Nx_out); }
