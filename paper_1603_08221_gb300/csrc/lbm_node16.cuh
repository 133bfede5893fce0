// lbm_node16.cuh - node arithmetic of the 16-bit storage forms.  Included by
// lbm_mix.cu inside its anonymous namespace.
//
// Stochastic rounding turns a difference in the last bit of an FP32 result
// into a different rounding decision about once in 2^16 stores, and after some
// tens of steps single BF16 populations then differ by a large part of their
// size.  So that a seeded 16-bit run reproduces across builds, its arithmetic
// is kept as it was first released, operation for operation: psi from a
// series and a rational form in packed FP32x2, and the moments, rates and
// collision formed population by population.  FP32 storage uses the shorter
// forms of lbm_mix.cu (psi from a table, sums shared by moments and
// collision); here they would save a fifth of the instructions (445 against 566 a
// node) and, when last measured, 12 % of the step (BF16 16384 x 256 at 40 rows per
// CTA: 113 against 127 us).  What does not change a bit is
// taken: the reciprocals and reciprocal square roots of the special-function
// unit without the scaling for subnormal arguments (5 %).

namespace n16 {

// a / b as the PTX ISA defines div.approx.f32, a times the approximate reciprocal
// of b, for arguments far from the ends of the FP32 range.
__device__ __forceinline__ float quotient(float a, float b) { return __fmul_rn(a, rcp_fast(b)); }

// psi(a) = 1 + (a - 1) e^{-a} - a^2 E_1(a)  (Eq. psi).
//  a <= 1: with the series of E_1, psi(a) = Q(a) + a^2 ln a where
//          Q(a) = 1 + (a - 1) e^{-a} + gamma a^2 - a^2 sum_k (-1)^{k+1} a^k/(k k!)
//          is entire; its Taylor coefficients are 2, gamma - 3/2 and
//          (-1)^m 2 / ((m - 2) m!) for m >= 3 (worked out from the two
//          series); eleven terms leave < 4e-10 on [0, 1].
//  1 < a < 15: psi = 1 + e^{-a} [(a - 1) - a (x e^x E_1)(a)] with the
//          rational approximation above (no cancellation).
//  a >= 15: 1 - psi < 2e^{-a}/a < 3e-8, below half an FP32 ulp of 1.
__device__ __forceinline__ float psi_dev(float a) {
  if (a <= 1.0f) {
    if (!(a > 0.0f)) return 0.0f;
    float q = -1.0f / 179625600.0f;
    q = fmaf(q, a, 1.0f / 14515200.0f);
    q = fmaf(q, a, -1.0f / 1270080.0f);
    q = fmaf(q, a, 1.0f / 120960.0f);
    q = fmaf(q, a, -1.0f / 12600.0f);
    q = fmaf(q, a, 1.0f / 1440.0f);
    q = fmaf(q, a, -1.0f / 180.0f);
    q = fmaf(q, a, 1.0f / 24.0f);
    q = fmaf(q, a, -1.0f / 3.0f);
    q = fmaf(q, a, 0.5772156649f - 1.5f);
    q = fmaf(q, a, 2.0f);
    // __logf: absolute error ~2^-21 on ln a near a = 1, i.e. < 2e-7 in a^2 ln a
    return fmaf(a * a, __logf(a), q * a);
  }
  if (a >= 16.0f) return 1.0f;  // 1 - psi(a) < 2 e^{-a}/a < 2^{-25}
  float num = (((a + 8.5733287401f) * a + 18.0590169730f) * a + 8.6347608925f) * a +
              0.2677737343f;
  float den = (((a + 9.5733223454f) * a + 25.6329561486f) * a + 21.0996530827f) * a +
              3.9584969228f;
  return fmaf(__expf(-a), (a - 1.0f) - a * __fdividef(num, den), 1.0f);
}

// psi'(a) = 2 e^{-a} - 2 a E_1(a).
__device__ __forceinline__ float dpsi_dev(float a) {
  if (a <= 1.0f) {
    if (!(a > 0.0f)) return 2.0f;
    return 2.0f * expf(-a) - 2.0f * a * e1_series(a);
  }
  return 2.0f * expf(-a) * (1.0f - xexe1_rational(a));
}

// psi at two positive arguments at once.  The lanes of a warp sweep one row
// (the same y) of 32 neighbouring columns, whose mean free paths differ
// little, so the two formulas of psi_dev are warp-uniform branches: the
// entire-part series when some lane has an argument <= 1, the rational form when
// some lane has one in (1, 16) (the kernel is bound by instruction issue).  At a
// >= 16, 1 - psi(a) < 2 e^{-a}/a < 2^{-25} rounds away and psi = 1.
__device__ __forceinline__ float2 psi2(float2 a) {
  const bool small = (a.x <= 1.0f) || (a.y <= 1.0f);
  const bool mid = (a.x > 1.0f && a.x < 16.0f) || (a.y > 1.0f && a.y < 16.0f);
  const unsigned lanes = __activemask();
  const bool do_small = __any_sync(lanes, small), do_mid = __any_sync(lanes, mid);
  float2 ps = f2(0.0f), pl = f2(1.0f);
  if (do_small) {
    const float2 as = make_float2(fminf(a.x, 1.0f), fminf(a.y, 1.0f));
    float2 q = f2(-1.0f / 179625600.0f);
    q = fma2(q, as, f2(1.0f / 14515200.0f));
    q = fma2(q, as, f2(-1.0f / 1270080.0f));
    q = fma2(q, as, f2(1.0f / 120960.0f));
    q = fma2(q, as, f2(-1.0f / 12600.0f));
    q = fma2(q, as, f2(1.0f / 1440.0f));
    q = fma2(q, as, f2(-1.0f / 180.0f));
    q = fma2(q, as, f2(1.0f / 24.0f));
    q = fma2(q, as, f2(-1.0f / 3.0f));
    q = fma2(q, as, f2(0.5772156649f - 1.5f));
    q = fma2(q, as, f2(2.0f));
    const float2 lg = make_float2(__logf(as.x), __logf(as.y));
    ps = fma2(mul2(as, as), lg, mul2(q, as));
  }
  if (do_mid) {
    // the argument is clamped to [1, 16]: at 16 the formula gives 1 in FP32
    // (1 - psi(16) < 2^-25), and larger arguments cannot overflow it
    const float2 al = make_float2(fminf(fmaxf(a.x, 1.0f), 16.0f), fminf(fmaxf(a.y, 1.0f), 16.0f));
    float2 num = add2(al, f2(8.5733287401f));
    num = fma2(num, al, f2(18.0590169730f));
    num = fma2(num, al, f2(8.6347608925f));
    num = fma2(num, al, f2(0.2677737343f));
    float2 den = add2(al, f2(9.5733223454f));
    den = fma2(den, al, f2(25.6329561486f));
    den = fma2(den, al, f2(21.0996530827f));
    den = fma2(den, al, f2(3.9584969228f));
    const float2 R = make_float2(quotient(num.x, den.x), quotient(num.y, den.y));
    const float2 e = make_float2(__expf(-al.x), __expf(-al.y));
    // 1 + e^{-a} [(a - 1) - a R]
    pl = fma2(e, fma2(make_float2(-al.x, -al.y), R, add2(al, f2(-1.0f))), f2(1.0f));
  }
  // arguments are y / lambda > 0 (y >= 1/2)
  return make_float2(a.x <= 1.0f ? ps.x : pl.x, a.y <= 1.0f ? ps.y : pl.y);
}

struct Macro {
  float sd[2];  // sum of deviations: rho_s - rhobar_s
  float rho[2];
  float n, inv_n, mx;
};

__device__ __forceinline__ void macro(const Lat& L, const ColRef& C, const float fs[2][9],
                                      Macro& m) {
#pragma unroll
  for (int sp = 0; sp < 2; ++sp) {
    const float* g = fs[sp];
    m.sd[sp] = ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7])) + g[8];
    m.rho[sp] = C.rb[sp] + m.sd[sp];
  }
  m.n = fmaf(m.rho[0], L.s[0], m.rho[1] * L.s[1]);  // number density (Eq. P)
  m.inv_n = __fdividef(1.0f, m.n);
  m.mx = (m.rho[0] + m.rho[1]) * m.inv_n;  // m_x = rho / n
}

// ------------------------------------------- packed per-node arithmetic
// The node update of the step kernel works on g[i] = (species a, species b)
// pairs of the pre-collision deviations.  (The moment fields of 16-bit states
// are read with the FP32 forms.)
struct Macro2 {
  float2 sd;   // sum of deviations: rho_s - rhobar_s
  float2 rho;  // species densities
  float2 jx, jy;
  float ux, uy;
  float n, inv_n, mx;
};

__device__ __forceinline__ void macro2(const Lat& L, const ColRef& C, const float2 g[9],
                                       Macro2& m) {
  m.sd = add2(add2(add2(add2(g[0], g[1]), add2(g[2], g[3])), add2(add2(g[4], g[5]), add2(g[6], g[7]))),
              g[8]);
  m.rho = add2(make_float2(C.rb[0], C.rb[1]), m.sd);
  m.jx = add2(add2(sub2(g[1], g[3]), sub2(g[5], g[6])), sub2(g[8], g[7]));
  m.jy = add2(add2(sub2(g[2], g[4]), sub2(g[5], g[7])), sub2(g[6], g[8]));
  const float rho = m.rho.x + m.rho.y;
  const float inv_rho = rcp_fast(rho);
  m.ux = (m.jx.x + m.jx.y) * inv_rho;
  m.uy = (m.jy.x + m.jy.y) * inv_rho;
  m.n = fmaf(m.rho.x, L.s[0], m.rho.y * L.s[1]);  // number density (Eq. P)
  m.inv_n = rcp_fast(m.n);
  m.mx = rho * m.inv_n;  // m_x = rho / n
}

// 1/tau_s (Eq. taos) and 1/tau_d (Eq. EQFrsp with lambda_se = lambda_s
// Psi(y; lambda_s), lambda_s = (mu_s/p_s) sqrt(pi k_B T/(2 m_s)), p_s = x_s p),
// with the wall-confinement factor Psi(y) = (psi(y/lambda) + psi((H-y)/lambda))/2
// of the effective mean free path; the six psi values come from three packed
// evaluations.
__device__ __forceinline__ void rates2(const Lat& L, const Macro2& m, float y, float& om_s,
                                       float& om_d) {
  const float rs_mx = rsqrt_fast(m.mx);
  const float lam = L.c_lam * m.inv_n * rs_mx;                // mixture mean free path
  const float inv_lam = L.inv_c_lam * m.n * (m.mx * rs_mx);  // 1 / lambda
  const float2 yy = make_float2(y, L.H - y);
  // 1 / lambda_s: n_s / c_xl with the partial pressure, n / c_xl with the
  // mixture pressure
  const float2 ns = mul2(m.rho, L.s2);
  const float2 inv_ls = mul2(L.lam_mix ? f2(m.n) : ns, L.inv_c_xl2);
  const float2 pm = psi2(mul2(yy, f2(inv_lam)));
  const float2 pa = psi2(mul2(yy, f2(inv_ls.x)));
  const float2 pb = psi2(mul2(yy, f2(inv_ls.y)));
  const float ts = lam * (0.5f * (pm.x + pm.y)) * L.c_ts * rs_mx;  // tau_s - 1/2
  om_s = rcp_fast(0.5f + ts);
  // x_s lambda_se = c_xl / n * Psi(y; lambda_s) (partial pressure), times
  // x_s = n_s / n with the mixture pressure
  const float2 xs = L.lam_mix ? mul2(ns, f2(m.inv_n)) : f2(1.0f);
  const float2 xle = mul2(mul2(mul2(L.c_xl2, f2(0.5f * m.inv_n)), xs),
                          make_float2(pa.x + pa.y, pb.x + pb.y));
  const float br = rsqrt_fast(xle.x) + rsqrt_fast(xle.y);
  // tau_d = 1/2 + c_td / (m_x br^2)  =>  1/tau_d = d / (d/2 + c_td), d = m_x br^2
  const float d = m.mx * br * br;
  om_d = quotient(d, fmaf(0.5f, d, L.c_td));
}

// MRT collision of both species at once (Eqs. MR, S, feq) on the deviations g from
// the rest equilibrium of the column reference, in moment space:
// f' = f - M^{-1} S (m - m^eq), M^{-1} = M^T diag(1/9, 1/36, 1/36, 1/6, 1/12,
// 1/6, 1/12, 1/4, 1/4), m^eq = rho_s (1, -4 + 2s + 3u^2, 4 - 3s - 3u^2, u_x,
// -u_x, u_y, -u_y, u_x^2 - u_y^2, u_x u_y).  The reference has m = m^eq(u=0),
// so e - e^eq = sum_i (e_i + 4 - 2s) g_i - 3 rho u^2 and
// eps - eps^eq = sum_i (eps_i - 4 + 3s) g_i + 3 rho u^2 need no large terms
// (ke, kp hold those coefficients for the rest, axis and diagonal classes).
// Returns the x components of the species momenta of Eq. rhou,
// j_x - (j_x - rho_s u_x)/(2 tau_d).
__device__ __forceinline__ float2 collide2(float2 g[9], const Lat& L, float2 rho, float ux,
                                           float uy, float om_e, float om_eps, float om_d,
                                           float om_q, float om_s) {
  const float2 ru2 = mul2(f2(3.0f * (ux * ux + uy * uy)), rho);
  const float2 a14 = add2(add2(g[1], g[2]), add2(g[3], g[4]));
  const float2 a58 = add2(add2(g[5], g[6]), add2(g[7], g[8]));
  const float2 ne =
      fma2(L.ke2[0], g[0], fma2(L.ke2[1], a14, fma2(L.ke2[2], a58, make_float2(-ru2.x, -ru2.y))));
  const float2 neps = fma2(L.kp2[0], g[0], fma2(L.kp2[1], a14, fma2(L.kp2[2], a58, ru2)));
  const float2 d13 = sub2(g[1], g[3]), d24 = sub2(g[2], g[4]);
  const float2 dx56 = add2(sub2(g[5], g[6]), sub2(g[8], g[7]));
  const float2 dy56 = add2(sub2(g[5], g[7]), sub2(g[6], g[8]));
  const float2 jx = add2(d13, dx56);
  const float2 jy = add2(d24, dy56);
  const float2 qx = fma2(f2(-2.0f), d13, dx56);
  const float2 qy = fma2(f2(-2.0f), d24, dy56);
  const float2 pxx = sub2(add2(g[1], g[3]), add2(g[2], g[4]));
  const float2 pxy = sub2(add2(g[5], g[7]), add2(g[6], g[8]));
  const float2 de = mul2(f2(om_e), ne);
  const float2 deps = mul2(f2(om_eps), neps);
  const float2 djx = mul2(f2(om_d), fma2(rho, f2(-ux), jx));
  const float2 djy = mul2(f2(om_d), fma2(rho, f2(-uy), jy));
  const float2 dqx = mul2(f2(om_q), fma2(rho, f2(ux), qx));
  const float2 dqy = mul2(f2(om_q), fma2(rho, f2(uy), qy));
  const float2 dpxx = mul2(f2(om_s), fma2(rho, f2(-(ux * ux - uy * uy)), pxx));
  const float2 dpxy = mul2(f2(om_s), fma2(rho, f2(-(ux * uy)), pxy));
  const float2 c0 = mul2(sub2(de, deps), f2(1.0f / 9.0f));
  const float2 c14 = fma2(de, f2(1.0f / 36.0f), mul2(deps, f2(1.0f / 18.0f)));
  const float2 c58 = fma2(de, f2(-1.0f / 18.0f), mul2(deps, f2(-1.0f / 36.0f)));
  const float2 ax = mul2(sub2(dqx, djx), f2(1.0f / 6.0f));
  const float2 ay = mul2(sub2(dqy, djy), f2(1.0f / 6.0f));
  const float2 bx = fma2(djx, f2(-1.0f / 6.0f), mul2(dqx, f2(-1.0f / 12.0f)));
  const float2 by = fma2(djy, f2(-1.0f / 6.0f), mul2(dqy, f2(-1.0f / 12.0f)));
  const float2 pp = mul2(dpxx, f2(0.25f)), pq = mul2(dpxy, f2(0.25f));
  const float2 u1 = sub2(c14, pp), u2 = add2(c14, pp);  // shared by opposite axis pairs
  const float2 v5 = sub2(c58, pq), v6 = add2(c58, pq);  // and by opposite diagonal pairs
  const float2 w5 = add2(bx, by), w6 = sub2(by, bx);
  g[0] = add2(g[0], c0);
  g[1] = add2(g[1], add2(u1, ax));
  g[3] = add2(g[3], sub2(u1, ax));
  g[2] = add2(g[2], add2(u2, ay));
  g[4] = add2(g[4], sub2(u2, ay));
  g[5] = add2(g[5], add2(v5, w5));
  g[7] = add2(g[7], sub2(v5, w5));
  g[6] = add2(g[6], add2(v6, w6));
  g[8] = add2(g[8], sub2(v6, w6));
  return fma2(f2(-0.5f), djx, jx);
}

// tau_q of Eq. taoq from the wall node's lambda and m_x (tau'_s(0) in its
// last term, dx = 1) and the node's accommodation coefficient (Eq. A12).
__device__ __forceinline__ float tau_q_wall(const Lat& L, const Macro& m, float alpha) {
  const float vs = 0.72360125455f;  // varsigma = sqrt(pi/6)
  float rs_mx = rsqrtf(m.mx);
  float lam = L.c_lam * m.inv_n * rs_mx;
  float g = L.c_ts * rs_mx;  // sqrt(6/(pi m_x))
  float a = L.H / lam;
  float tt = lam * 0.5f * psi_dev(a) * g;
  float dtt = 0.5f * g * (2.0f - dpsi_dev(a));
  float A1 = (2.0f - alpha) / alpha * (1.0f - 0.1817f * alpha);
  float A2 = 1.0f / kPi + 0.5f * A1 * A1;
  return 0.5f + (3.0f + 24.0f * vs * vs * tt * tt * A2) / (16.0f * tt) +
         dtt * (12.0f + 30.0f * tt * vs * A1) / (16.0f * tt * tt);
}

// r of Eq. R, r = 2 - 2/(1 + X), from the mixture molecular mass of the
// reflected post-collision state at the wall node, c_m = c_m0
// (2-alpha)/alpha, for both species: X = c_m sqrt(pi m_x/6) (first printed
// form, the same for both species; masses in units of m_min), c_m sqrt(pi
// m_x/(6 m_s)) (m_min replaced by the species mass) or c_m sqrt(pi m_x^2/(6
// m_s)) (second printed form, m_r = m_s/m_x).  With the BSR wall the
// bounce-back fraction 1/(1 + X) of the same slip factor X.
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
  float mx = (rho[0] + rho[1]) / fmaf(rho[0], L.s[0], rho[1] * L.s[1]);
  float cm = L.c_m0 * (2.0f - alpha) / alpha;
  const float X0 = cm * sqrtf(kPi * mx / 6.0f) * (L.r_form == LBM_R_SECOND ? sqrtf(mx) : 1.0f);
  float r[2];
#pragma unroll
  for (int sp = 0; sp < 2; ++sp) {
    const float X = L.r_form == LBM_R_FIRST ? X0 : X0 * L.rsqrt_mh[sp];
    r[sp] = L.wall_mode == LBM_WALL_BSR ? 1.0f / (1.0f + X) : 2.0f - 2.0f / (1.0f + X);
  }
  return make_float2(r[0], r[1]);
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
    if (x0 <= 1 && 1 < x0 + width) {
      double k = L.N * L.rho_in[sp] / (2.0 * c[1] - c[2]);
      E.kin[sp] = (float)k;
      E.gin[sp] = (float)(k * (2.0 * (double)r[1] - (double)r[2]) - (double)r[0]);
    }
    if (x0 <= Nx - 2 && Nx - 2 < x0 + width) {
      double k = L.N * L.rho_out[sp] / (2.0 * c[Nx - 2] - c[Nx - 3]);
      E.kout[sp] = (float)k;
      E.gout[sp] = (float)(k * (2.0 * (double)r[Nx - 2] - (double)r[Nx - 3]) - (double)r[Nx - 1]);
    }
  }
  return E;
}

}  // namespace n16
