// ap_adjoint.cu -- discrete adjoint of the gather + Boris push (row a13).
//
// Objective per set s: J_s = (1/N_s) sum_{i in s} gamma_i(T).  Gradients with
// respect to the pulse parameters theta = (a0, w0, z_f, beta_f) of every set
// (beta_f only for the closed-form flying focus; zero otherwise), by the
// exact reverse of the discrete forward map (the same float-float or double
// arithmetic as ap_gather_push):
//
//   forward:  x^{n+1} = x^n + dt u^{n+1}/gamma^{n+1},  u^{n+1} = Boris(u^n, E(x^n), B(x^n))
//   reverse:  lu'  = lu^{n+1} + dt/gamma' (lx - v' (v'.lx))         (position update)
//             (lu^n, lE, lB) = Boris^T(lu')                          (hand-written VJP)
//             lx^n = lx^{n+1} + (dF/dx)^T (lE, lB),  g += (dF/dtheta)^T (lE, lB)
//
// with seed lu^N = u^N / (gamma^N N_s), lx^N = 0.  dF/dx and dF/dtheta are
// the derivatives in (x, y, z - z_f, w0, beta_f): in closed form for the
// Gaussian beam and the closed-form flying focus (beam_reverse), and from
// the field functions instantiated with forward-mode dual numbers for the
// other kinds; a0 enters linearly (dF/da0 = F / a0) and z_f only through
// z - z_f (dF/dz_f = -dF/dz for the analytic part).
//
// Memory: one persistent launch; every resident thread slot pushes its
// particle forward storing a checkpoint every K steps, then sweeps the
// segments backwards, recomputing each from its checkpoint into a per-slot
// tape.  Checkpoints and tapes live in the caller's workspace, sized by the
// number of resident thread slots, not by the number of particles.
#include <cuda_runtime.h>

#include <cstring>

#include "ap_dual.cuh"
#include "ap_kernels.cuh"

namespace apt {

constexpr int kAdjBlock = 128;
constexpr int kAdjBlocksPerSm = 4;
constexpr int kAdjMaxK = 256;
constexpr int kAdjSlotsPerSm = 768;    // particle slots of the workspace
constexpr int kAdjStateBytes = 48;  // one saved state: 6 doubles or 9 floats
// tangents: x, y, z - z_f, w0 and, for the closed-form flying focus only,
// beta_f (the other kinds do not depend on it: a fifth tangent would be
// dead arithmetic in every dual operation)
template <int KIND>
__host__ __device__ constexpr int tangents() { return KIND == AP_FLYING_CF ? 5 : 4; }
constexpr int kNp = 4;   // parameters: a0, w0, z_f, beta_f

// Pulse view with the w0-dependent constants as duals (tangent slot 3) and,
// for the closed-form flying focus, the beta_f-dependent ones (slot 4).
template <typename R, int NT>
struct PulseAD {
  static constexpr bool kHasPlasma = true;
  int32_t kind, pol, env, lon, lg_p, lg_al, lg_sgn, sg_order, plasma;
  R amp, bratio, lonE, lonB, env_a, env_b, sg_max, px_re, px_im, py_re, py_im;
  R fdc, inv_w, lg_c1, lg_c2;  // plane wave in a plasma (Sec. 4, Eq. b_corr_t)
  R lg_alf;                    // |l| as a number
  R lg_r[6][kLgMaxP];
  Dual<R, NT> inv_w0sq, inv_zR, lg_pref, beta_f;
};

template <int NT, typename R>
__device__ __forceinline__ PulseAD<R, NT> make_ad(const Pulse<R> &P) {
  using D = Dual<R, NT>;
  PulseAD<R, NT> A;
  A.kind = P.kind; A.pol = P.pol; A.env = P.env; A.lon = P.lon;
  A.lg_p = P.lg_p; A.lg_al = P.lg_al; A.lg_sgn = P.lg_sgn; A.sg_order = P.sg_order;
  A.plasma = P.plasma; A.fdc = P.fdc; A.inv_w = P.inv_w; A.lg_c1 = P.lg_c1; A.lg_c2 = P.lg_c2;
  A.lg_alf = P.lg_alf;
  A.amp = P.amp_unit;  // unit a0: the physical field is a0 times this one
  A.bratio = P.bratio; A.lonE = P.lonE; A.lonB = P.lonB;
  A.env_a = P.env_a; A.env_b = P.env_b; A.sg_max = P.sg_max;
  A.px_re = P.px_re; A.px_im = P.px_im; A.py_re = P.py_re; A.py_im = P.py_im;
  for (int r = 0; r < 6; ++r)
    for (int k = 0; k < kLgMaxP; ++k) A.lg_r[r][k] = P.lg_r[r][k];
  const R iw = P.inv_w0;
  // d(1/w0^2)/dw0 = -2/w0^3; z_R ~ w0^2; (sqrt2/w0)^|l| ~ w0^-|l|
  A.inv_w0sq = D::seed(P.inv_w0sq, 3, R(-2) * P.inv_w0sq * iw);
  A.inv_zR = D::seed(P.inv_zR, 3, R(-2) * P.inv_zR * iw);
  A.lg_pref = D::seed(P.lg_pref, 3, -R(P.lg_al) * P.lg_pref * iw);
  A.beta_f = D(P.beta_f);
  if constexpr (NT == 5) {
    // closed-form flying focus: zeta = ((z - z_f) - beta_f (t - t_f)) / z_R',
    // 1/z_R' = 1 / ((1 - beta_f) z_R) -> d/dbeta_f = (1/z_R') / (1 - beta_f)
    A.beta_f.d[4] = R(1);
    A.inv_zR.d[4] = P.inv_zR * P.inv_1mb;
  }
  return A;
}

// Saved particle state (checkpoints and tape), strided by thread slot.
template <int PREC>
struct StateIO;

template <>
struct StateIO<AP_FP32_PHASEFF> {
  static constexpr int W = 9;
  __device__ static void put(float *base, size_t stride, const Pos<AP_FP32_PHASEFF> &p,
                             const float u[3]) {
    base[0 * stride] = p.x.hi; base[1 * stride] = p.x.lo;
    base[2 * stride] = p.y.hi; base[3 * stride] = p.y.lo;
    base[4 * stride] = p.z.hi; base[5 * stride] = p.z.lo;
    base[6 * stride] = u[0]; base[7 * stride] = u[1]; base[8 * stride] = u[2];
  }
  __device__ static void get(const float *base, size_t stride, Pos<AP_FP32_PHASEFF> &p, float u[3]) {
    p.x.hi = base[0 * stride]; p.x.lo = base[1 * stride];
    p.y.hi = base[2 * stride]; p.y.lo = base[3 * stride];
    p.z.hi = base[4 * stride]; p.z.lo = base[5 * stride];
    u[0] = base[6 * stride]; u[1] = base[7 * stride]; u[2] = base[8 * stride];
  }
  using T = float;
};

template <>
struct StateIO<AP_FP64> {
  static constexpr int W = 6;
  __device__ static void put(double *base, size_t stride, const Pos<AP_FP64> &p, const double u[3]) {
    base[0 * stride] = p.x; base[1 * stride] = p.y; base[2 * stride] = p.z;
    base[3 * stride] = u[0]; base[4 * stride] = u[1]; base[5 * stride] = u[2];
  }
  __device__ static void get(const double *base, size_t stride, Pos<AP_FP64> &p, double u[3]) {
    p.x = base[0 * stride]; p.y = base[1 * stride]; p.z = base[2 * stride];
    u[0] = base[3 * stride]; u[1] = base[4 * stride]; u[2] = base[5 * stride];
  }
  using T = double;
};

struct AdjArgs {
  PushArgs base;              // particles (read only), grid, t0, dt, n_steps, status
  const long long *set_offsets;  // nullptr: one set [0, n)
  int n_sets;
  int K;                      // steps per segment
  int n_seg;
  unsigned int *tile_counter;
  void *ckpt;                 // [n_seg][W][nslots]
  void *tape;                 // [K][W][nslots]
  long long nslots;
  double *dJ;                 // [n_sets][AP_NPARAM]
  double *J;                  // [n_sets] or null
};

template <typename R>
struct GridGrad {
  R v[6];
  R g[6][3];
};

// Trilinear value and gradient from the cached cell (zero gradient along an
// axis on which the position is clamped to the box).
template <typename R>
__device__ __forceinline__ void grid_value_grad(const GridView &g, GridCache<R> &gc, R x, R y, R z,
                                                GridGrad<R> &out) {
  R E[3] = {R(0), R(0), R(0)}, B[3] = {R(0), R(0), R(0)};
  grid_gather<R>(g, gc, x, y, z, E, B);  // refreshes the cache and the weights
  R idd[3], off[3];
  if constexpr (std::is_same<R, double>::value) {
    for (int a = 0; a < 3; ++a) { idd[a] = g.inv_d_d[a]; off[a] = g.off_d[a]; }
  } else {
    for (int a = 0; a < 3; ++a) { idd[a] = g.inv_d[a]; off[a] = g.off[a]; }
  }
  // unclamped grid coordinates: the gradient vanishes along clamped axes
  const R fxr = fma(x, idd[0], off[0]), fyr = fma(y, idd[1], off[1]), fzr = fma(z, idd[2], off[2]);
  const R wx = gc.wx, wy = gc.wy, wz = gc.wz;
  const R ux = R(1) - wx, uy = R(1) - wy, uz = R(1) - wz;
  const R sx = (fxr >= R(0) && fxr <= R(g.nx - 1)) ? idd[0] : R(0);
  const R sy = (fyr >= R(0) && fyr <= R(g.ny - 1)) ? idd[1] : R(0);
  const R sz = (fzr >= R(0) && fzr <= R(g.nz - 1)) ? idd[2] : R(0);
  out.v[0] = E[0]; out.v[1] = E[1]; out.v[2] = E[2];
  out.v[3] = B[0]; out.v[4] = B[1]; out.v[5] = B[2];
  for (int c = 0; c < 6; ++c) {
    // raw corners k[cx + 2 cy + 4 cz]; derivative of the trilinear weights
    const R *k = gc.c[c];
    R dfx = (k[1] - k[0]) * uy * uz + (k[3] - k[2]) * wy * uz + (k[5] - k[4]) * uy * wz +
            (k[7] - k[6]) * wy * wz;
    R dfy = (k[2] - k[0]) * ux * uz + (k[3] - k[1]) * wx * uz + (k[6] - k[4]) * ux * wz +
            (k[7] - k[5]) * wx * wz;
    R dfz = (k[4] - k[0]) * ux * uy + (k[5] - k[1]) * wx * uy + (k[6] - k[2]) * ux * wy +
            (k[7] - k[3]) * wx * wy;
    out.g[c][0] = dfx * sx;
    out.g[c][1] = dfy * sy;
    out.g[c][2] = dfz * sz;
  }
}

template <int KIND, typename R, int NT>
__device__ __forceinline__ void fields_ad(const PulseAD<R, NT> &A, const Local<Dual<R, NT>> &L,
                                          Dual<R, NT> E[3], Dual<R, NT> B[3]) {
  if constexpr (KIND == AP_PLANE) fields_plane(A, L, E, B);
  else if constexpr (KIND == AP_GAUSS) fields_gauss(A, L, E, B);
  else if constexpr (KIND == AP_FLYING_CF) fields_gauss<true>(A, L, E, B);
  else fields_lg(A, L, E, B);
}

// Logarithmic derivative Gamma'/Gamma of the envelope at eta, given the
// factor `mul` that `envelope` returned (zero outside the sin^2 window and
// for a continuous wave).  SIN2: Gamma = cos^2(env_a eta), so -2 env_a
// tan(env_a eta); GAUSS: Gamma = 2^(-env_a eta^2); SGAUSS: Gamma =
// 2^(-env_b u^(2g)), u = env_a eta.
template <typename R>
__device__ __forceinline__ R unless_zero(R v, R m) { return m == R(0) ? R(0) : v; }
__device__ __forceinline__ F2 unless_zero(F2 v, F2 m) {
  return F2(m.x == 0.0f ? 0.0f : v.x, m.y == 0.0f ? 0.0f : v.y);
}

template <class PT, typename R>
__device__ __forceinline__ R envelope_dlog(const PT &P, R eta, R mul) {
  constexpr double kLn2 = 0.69314718055994531;
  switch (P.env) {
    case AP_ENV_SIN2: {
      // evaluated in both halves of a pair, each cleared where its factor is 0
      R s, c;
      sincos_r(eta * P.env_a, &s, &c);
      return unless_zero(R(-2) * P.env_a * s * rcp_r(c), mul);
    }
    case AP_ENV_GAUSS:
      return R(-2 * kLn2) * P.env_a * eta;
    case AP_ENV_SGAUSS: {
      const R u = sg_bound(eta * P.env_a, P.sg_max);
      const R s = u * u;
      R p = R(1);  // s^(g-1)
      for (int i = 1; i < P.sg_order; ++i) p *= s;
      return R(-2 * kLn2) * P.env_b * R(P.sg_order) * P.env_a * u * p;
    }
    default:
      return R(0);
  }
}

// The reverse of one Boris step and position update, given the fields F at
// the step's position: from the adjoints lx, lu of the state after the step,
// the cotangent Fb of the fields (E, B), with lu updated to the momentum
// adjoint before the step (lx changes only through the fields:
// lx += (dF/dx)^T Fb).  Generic over the arithmetic type (float, double, or
// the packed pair of the two-particle kernel); adv_xy = 0 holds the
// transverse position (1D-3V).
template <typename R>
__device__ __forceinline__ void boris_cotangent(const R F[6], const R u[3], R dt, R adv_xy,
                                                const R lx[3], R lu[3], R Fb[6]) {
  const R h = R(-0.5) * dt;
  const R E[3] = {F[0], F[1], F[2]}, B[3] = {F[3], F[4], F[5]};
  // Boris forward intermediates
  R am[3] = {fma(h, E[0], u[0]), fma(h, E[1], u[1]), fma(h, E[2], u[2])};
  R ig = rsqrt_r(R(1) + am[0] * am[0] + am[1] * am[1] + am[2] * am[2]);
  R tau[3] = {h * ig * B[0], h * ig * B[1], h * ig * B[2]};
  R tt = tau[0] * tau[0] + tau[1] * tau[1] + tau[2] * tau[2];
  R f = R(2) * rcp_r(R(1) + tt);
  R s[3] = {f * tau[0], f * tau[1], f * tau[2]};
  R p[3] = {am[0] + (am[1] * tau[2] - am[2] * tau[1]), am[1] + (am[2] * tau[0] - am[0] * tau[2]),
            am[2] + (am[0] * tau[1] - am[1] * tau[0])};
  R bq[3] = {am[0] + (p[1] * s[2] - p[2] * s[1]), am[1] + (p[2] * s[0] - p[0] * s[2]),
             am[2] + (p[0] * s[1] - p[1] * s[0])};
  R un[3] = {fma(h, E[0], bq[0]), fma(h, E[1], bq[1]), fma(h, E[2], bq[2])};
  R ign = rsqrt_r(R(1) + un[0] * un[0] + un[1] * un[1] + un[2] * un[2]);
  R v[3] = {un[0] * ign, un[1] * ign, un[2] * ign};
  // position update: x'_k = x_k + dt_k u'_k / gamma', dt_k = (dt_xy, dt_xy, dt)
  // (dt_xy = 0 for a 1D-3V set): d x'_k / d u'_j = dt_k ign (delta_kj - v_k v_j)
  const R dtk[3] = {dt * adv_xy, dt * adv_xy, dt};
  R vl = dtk[0] * v[0] * lx[0] + dtk[1] * v[1] * lx[1] + dtk[2] * v[2] * lx[2];
  R ub[3];
  for (int k = 0; k < 3; ++k) ub[k] = lu[k] + ign * (dtk[k] * lx[k] - v[k] * vl);
  // Boris reverse
  R Eb[3], Bb[3], ab[3], pb[3], sbar[3], tb[3];
  for (int k = 0; k < 3; ++k) Eb[k] = h * ub[k];
  // b = a + p x s
  pb[0] = s[1] * ub[2] - s[2] * ub[1];
  pb[1] = s[2] * ub[0] - s[0] * ub[2];
  pb[2] = s[0] * ub[1] - s[1] * ub[0];
  sbar[0] = ub[1] * p[2] - ub[2] * p[1];
  sbar[1] = ub[2] * p[0] - ub[0] * p[2];
  sbar[2] = ub[0] * p[1] - ub[1] * p[0];
  // p = a + a x tau
  ab[0] = ub[0] + pb[0] + (tau[1] * pb[2] - tau[2] * pb[1]);
  ab[1] = ub[1] + pb[1] + (tau[2] * pb[0] - tau[0] * pb[2]);
  ab[2] = ub[2] + pb[2] + (tau[0] * pb[1] - tau[1] * pb[0]);
  tb[0] = pb[1] * am[2] - pb[2] * am[1];
  tb[1] = pb[2] * am[0] - pb[0] * am[2];
  tb[2] = pb[0] * am[1] - pb[1] * am[0];
  // s = f tau, f = 2 / (1 + tau^2)
  R ts = tau[0] * sbar[0] + tau[1] * sbar[1] + tau[2] * sbar[2];
  for (int k = 0; k < 3; ++k) tb[k] += f * sbar[k] - f * f * tau[k] * ts;
  // tau = h ig B
  R igb = h * (B[0] * tb[0] + B[1] * tb[1] + B[2] * tb[2]);
  for (int k = 0; k < 3; ++k) Bb[k] = h * ig * tb[k];
  // ig = (1 + a^2)^(-1/2)
  R c3 = -ig * ig * ig * igb;
  for (int k = 0; k < 3; ++k) ab[k] += c3 * am[k];
  for (int k = 0; k < 3; ++k) {
    Eb[k] += h * ab[k];
    lu[k] = ab[k];
  }
  for (int k = 0; k < 3; ++k) {
    Fb[k] = Eb[k];
    Fb[k + 3] = Bb[k];
  }
}

// The grid's share of a reverse step: its interpolated fields join the
// analytic ones before the Boris reverse, and its gradient joins the
// position adjoint after it.
struct NoGridPart {
  template <typename R>
  __device__ __forceinline__ void add(R *) const {}
  template <typename R>
  __device__ __forceinline__ void contract(const R *, R *) const {}
};
template <typename R>
struct GridPart {
  GridGrad<R> gg;
  __device__ __forceinline__ void add(R F[6]) const {
    for (int c = 0; c < 6; ++c) F[c] += gg.v[c];
  }
  __device__ __forceinline__ void contract(const R Fb[6], R lx[3]) const {
    for (int c = 0; c < 6; ++c)
      for (int k = 0; k < 3; ++k) lx[k] += Fb[c] * gg.g[c][k];
  }
};

// One reverse step of the Gaussian beam (MOVING: the closed-form flying
// focus), with the field derivatives in the directions j = (x, y, z - z_f,
// w0[, beta_f]) in closed form rather than by dual numbers, each contracted
// with the field cotangent Fb as soon as it is formed (no Jacobian is kept).
// The value part is the arithmetic of gauss_z and gauss_xy.  With G the
// amplitude times the envelope and a = r^2/w0^2, the profile is
// U0 = G e^{i psi} exp(-a q), U = q U0 and W = q U (the longitudinal terms'
// factor), and dq/dzeta = i q^2; so every derivative is a complex factor
// times U or W:
//   dU/dj = U alpha_j,  alpha_j = i q (1 - a q) zeta_j - a_j q + L1 eta_j + i psi_j,
//   dW/dj = W beta_j,   beta_j = alpha_j + i q zeta_j,
// L1 = Gamma'/Gamma, where zeta_j, a_j, eta_j, psi_j are the derivatives of
// zeta, a, eta = T - (z - z_f)/v_g and psi = C - k (z - z_f).  The fields
// are linear in U and W (finish_beam), with the longitudinal terms also
// linear in x, y and g = -2/w0^2, whose derivatives add those terms at unit
// x, at unit y, and times g'/g = -2/w0.  Order: the value and the factors
// the derivatives share, the Boris reverse for Fb, then Fb . dF/dj per
// direction.  F = a0 f with f the unit-a0 fields: dF/da0 = f, d/dz_f =
// -d/d(z - z_f).
template <int POL, bool LON, bool MOVING, class PT, typename R, class GP>
__device__ __forceinline__ void beam_reverse_t(const PT &P, const Local<R> &L, R a0, const R u[3],
                                               R dt, R adv_xy, R lx[3], R lu[3], R gr[kNp],
                                               const GP &grid) {
  constexpr int NT = MOVING ? 5 : 4;
  R mul, l2;
  envelope(P, L.eta, mul, l2);
  R zeta;
  if constexpr (MOVING) zeta = fma(-P.beta_f, L.T, L.dz) * P.inv_zR;
  else zeta = L.dz * P.inv_zR;
  const R inv = rcp_r(fma(zeta, zeta, R(1)));
  const Cx<R> q{inv, zeta * inv};
  const R x = L.x, y = L.y;
  const R a = (x * x + y * y) * P.inv_w0sq;
  const R mag = (P.amp_unit * mul) * exp2_r(fma(a * q.re, R(-kLog2e), l2));
  const R ang = reduce_angle<R>(L.psi - a * q.im);
  R sn, cs;
  sincos_r(ang, &sn, &cs);
  const Cx<R> U = cmul(q, Cx<R>{mag * cs, mag * sn});
  const Cx<R> W = cmul(q, U);
  const R g = R(-2) * P.inv_w0sq;
  R f[6], F[6], Fb[6];
  {
    R E[3], B[3];
    finish_beam_pol<POL>(P, x, y, U, W, g, LON, E, B);
    for (int c = 0; c < 3; ++c) {
      f[c] = E[c];
      f[c + 3] = B[c];
    }
  }
  for (int c = 0; c < 6; ++c) F[c] = a0 * f[c];
  grid.add(F);
  boris_cotangent<R>(F, u, dt, adv_xy, lx, lu, Fb);
  grid.contract(Fb, lx);
  R sa0 = Fb[0] * f[0];
  for (int c = 1; c < 6; ++c) sa0 = fma(Fb[c], f[c], sa0);
  // shared factors: i q and i q (1 - a q)
  const Cx<R> iq{-q.im, q.re};
  const Cx<R> Q1 = cmul(iq, Cx<R>{R(1) - a * q.re, -a * q.im});
  const R L1 = envelope_dlog(P, L.eta, mul);
  const R w2 = R(2) * P.inv_w0sq, m2w = R(-2) * P.inv_w0;
  R zj[NT], aj[NT], ej[NT], pj[NT], sj[NT];
  zj[0] = R(0); aj[0] = w2 * x; ej[0] = R(0); pj[0] = R(0);
  zj[1] = R(0); aj[1] = w2 * y; ej[1] = R(0); pj[1] = R(0);
  zj[2] = P.inv_zR; aj[2] = R(0); ej[2] = -P.inv_vg * L1; pj[2] = -R(P.k);
  zj[3] = m2w * zeta; aj[3] = m2w * a; ej[3] = R(0); pj[3] = R(0);
  if constexpr (NT == 5) {
    zj[4] = fma(-L.T, P.inv_zR, zeta * P.inv_1mb);
    aj[4] = R(0); ej[4] = R(0); pj[4] = R(0);
  }
#pragma unroll
  for (int j = 0; j < NT; ++j) {
    const Cx<R> al{zj[j] * Q1.re - aj[j] * q.re + ej[j], zj[j] * Q1.im - aj[j] * q.im + pj[j]};
    const Cx<R> be{al.re + zj[j] * iq.re, al.im + zj[j] * iq.im};
    R Ej[3], Bj[3];
    finish_beam_pol<POL>(P, x, y, cmul(U, al), cmul(W, be), g, LON, Ej, Bj);
    R t = Fb[0] * Ej[0];
    t = fma(Fb[1], Ej[1], t);
    t = fma(Fb[2], Ej[2], t);
    t = fma(Fb[3], Bj[0], t);
    t = fma(Fb[4], Bj[1], t);
    sj[j] = fma(Fb[5], Bj[2], t);
  }
  if constexpr (LON) {
    // the longitudinal terms' own x, y and g factors (components E_z, B_z)
    const Cx<R> zero{R(0), R(0)};
    R Ex[3], Bx[3], Ey[3], By[3], Eg[3], Bg[3];
    finish_beam_pol<POL>(P, R(1), R(0), zero, W, g, true, Ex, Bx);
    finish_beam_pol<POL>(P, R(0), R(1), zero, W, g, true, Ey, By);
    finish_beam_pol<POL>(P, x, y, zero, W, g, true, Eg, Bg);
    sj[0] = fma(Fb[2], Ex[2], fma(Fb[5], Bx[2], sj[0]));
    sj[1] = fma(Fb[2], Ey[2], fma(Fb[5], By[2], sj[1]));
    sj[3] = fma(m2w, fma(Fb[2], Eg[2], Fb[5] * Bg[2]), sj[3]);
  }
  lx[0] = fma(a0, sj[0], lx[0]);
  lx[1] = fma(a0, sj[1], lx[1]);
  lx[2] = fma(a0, sj[2], lx[2]);
  gr[0] += sa0;
  gr[1] = fma(a0, sj[3], gr[1]);
  gr[2] = fma(-a0, sj[2], gr[2]);
  if constexpr (NT == 5) gr[3] = fma(a0, sj[4], gr[3]);
}

// beam_reverse_t with the polarisation and the longitudinal switch (uniform
// over a set) selected once rather than in each of its field assemblies.
template <bool MOVING, class PT, typename R, class GP>
__device__ __forceinline__ void beam_reverse(const PT &P, const Local<R> &L, R a0, const R u[3], R dt,
                                             R adv_xy, R lx[3], R lu[3], R gr[kNp], const GP &grid) {
  const bool lon = P.lon != 0;
#define APT_BEAM_REV(POLV)                                                                    \
  if (lon) beam_reverse_t<POLV, true, MOVING>(P, L, a0, u, dt, adv_xy, lx, lu, gr, grid);   \
  else beam_reverse_t<POLV, false, MOVING>(P, L, a0, u, dt, adv_xy, lx, lu, gr, grid)
  switch (P.pol) {
    case AP_LIN_X: APT_BEAM_REV(AP_LIN_X); break;
    case AP_LIN_Y: APT_BEAM_REV(AP_LIN_Y); break;
    case AP_CIRC_P: APT_BEAM_REV(AP_CIRC_P); break;
    default: APT_BEAM_REV(AP_CIRC_M); break;
  }
#undef APT_BEAM_REV
}

// One reverse step.  State before the step (pos, u), step value st, adjoints
// lx, lu of the state after the step (updated in place to the state before),
// gradient accumulators g[0..3] = d/d(a0, w0, z_f, beta_f).
template <int KIND, int PREC, bool GRID>
__device__ __forceinline__ void reverse_step(const Pulse<Real<PREC>> &P,
                                             const PulseAD<Real<PREC>, tangents<KIND>()> &A,
                                             const AdjArgs &aa, const typename TimeBase<PREC>::Step &st,
                                             const Pos<PREC> &pos, const Real<PREC> u[3],
                                             Real<PREC> lx[3], Real<PREC> lu[3], Real<PREC> g[kNp],
                                             GridCache<Real<PREC>> &gc) {
  using R = Real<PREC>;
  constexpr int NT = tangents<KIND>();
  using DR = Dual<R, NT>;
  const R dt = (R)aa.base.dt;
  const R a0 = P.a0;
  const R adv = P.adv_xy;
  // fields with derivatives in (x, y, z - z_f, w0, beta_f)
  const Local<R> L = local_coords<PREC>(P, st, pos);
  auto run = [&](const auto &grid) {
    if constexpr (KIND == AP_GAUSS || KIND == AP_FLYING_CF) {
      beam_reverse<KIND == AP_FLYING_CF>(P, L, a0, u, dt, adv, lx, lu, g, grid);
    } else {
      // the other kinds: dual numbers through the generic field functions
      R F[6], dFx[6][3], dFth[6][kNp];  // field, d/dx, d/d(a0, w0, z_f, beta_f)
      Local<DR> LD;
      LD.x = DR::seed(L.x, 0);
      LD.y = DR::seed(L.y, 1);
      LD.dz = DR::seed(L.dz, 2);
      LD.psi = DR(L.psi);
      LD.psi.d[2] = -R(P.k);  // psi = C - k (z - z_f)
      LD.eta = DR(L.eta);
      LD.eta.d[2] = -P.inv_vg;  // eta = T - (z - z_f) / v_g
      LD.T = DR(L.T);
      LD.phi_hi = DR(R(0));
      LD.phi_lo = DR(R(0));
      DR Ed[3], Bd[3];
      fields_ad<KIND, R, NT>(A, LD, Ed, Bd);
      const DR *Fd[6] = {&Ed[0], &Ed[1], &Ed[2], &Bd[0], &Bd[1], &Bd[2]};
      for (int c = 0; c < 6; ++c) {
        const DR &f = *Fd[c];
        F[c] = a0 * f.v;
        dFx[c][0] = a0 * f.d[0];
        dFx[c][1] = a0 * f.d[1];
        dFx[c][2] = a0 * f.d[2];
        dFth[c][0] = f.v;
        dFth[c][1] = a0 * f.d[3];
        dFth[c][2] = -a0 * f.d[2];
        if constexpr (NT == 5) dFth[c][3] = a0 * f.d[4];
        else dFth[c][3] = R(0);
      }
      grid.add(F);
      R Fb[6];
      boris_cotangent<R>(F, u, dt, adv, lx, lu, Fb);
      grid.contract(Fb, lx);
      for (int c = 0; c < 6; ++c) {
        for (int k = 0; k < 3; ++k) lx[k] += Fb[c] * dFx[c][k];
        for (int k = 0; k < kNp; ++k) g[k] += Fb[c] * dFth[c][k];
      }
    }
  };
  if constexpr (GRID) {
    GridPart<R> gp;
    grid_value_grad<R>(aa.base.grid, gc, L.x, L.y, pos.zr(), gp.gg);
    run(gp);
  } else {
    run(NoGridPart{});
  }
}

template <int KIND, int PREC, bool GRID>
// residency target: kAdjBlocksPerSm blocks for the float kernels without a
// grid, two for the larger FP64 and grid ones (without a minimum the FP64
// kernel was held at 128 registers and spilled)
__global__ void __launch_bounds__(kAdjBlock, (PREC == AP_FP64 || GRID) ? 2 : kAdjBlocksPerSm)
    adjoint_kernel(const Pulse<Real<PREC>> *__restrict__ sets,
                                                            const __grid_constant__ AdjArgs aa) {
  using R = Real<PREC>;
  using IO = StateIO<PREC>;
  using T = typename IO::T;
  __shared__ long long s_tile;
  __shared__ int s_set;
  __shared__ double s_red[32];
  __shared__ StepFF s_steps[kAdjMaxK];
  __shared__ __align__(16) unsigned char s_pulse_raw[sizeof(Pulse<R>)];
  __shared__ long long s_prefix[AP_MAX_SETS + 1];
  // dynamic: the tape state of the next reverse step, copied in while the
  // current one is computed (double buffer [2][W][kAdjBlock], this thread's
  // column only)
  extern __shared__ __align__(16) unsigned char s_adj_dyn[];
  T *s_next = reinterpret_cast<T *>(s_adj_dyn);
  Pulse<R> &P = *reinterpret_cast<Pulse<R> *>(s_pulse_raw);
  const PushArgs &a = aa.base;
  const int Tt = blockDim.x;
  tile_prefix(s_prefix, aa.n_sets, Tt,
              [&](int s) { return aa.set_offsets ? aa.set_offsets[s + 1] - aa.set_offsets[s] : a.n; });
  if (threadIdx.x == 0) s_set = -1;
  __syncthreads();
  const long long total = s_prefix[aa.n_sets];
  const size_t slot = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t stride = (size_t)aa.nslots;
  T *ck = static_cast<T *>(aa.ckpt) + slot;
  T *tp = static_cast<T *>(aa.tape) + slot;
  for (;;) {
    if (threadIdx.x == 0) s_tile = (long long)atomicAdd(aa.tile_counter, 1u);
    __syncthreads();
    const long long tile = s_tile;
    if (tile >= total) break;
    int lo = 0, hi = aa.n_sets;
    while (hi - lo > 1) {
      int mid = (lo + hi) >> 1;
      if (s_prefix[mid] <= tile) lo = mid; else hi = mid;
    }
    const int set = lo;
    if (set != s_set) {
      const int words = (int)(sizeof(Pulse<R>) / 4);
      const uint32_t *src = reinterpret_cast<const uint32_t *>(sets + set);
      uint32_t *dst = reinterpret_cast<uint32_t *>(s_pulse_raw);
      for (int w = threadIdx.x; w < words; w += blockDim.x) dst[w] = src[w];
      __syncthreads();
      if (threadIdx.x == 0) s_set = set;
    }
    __syncthreads();
    const long long off0 = aa.set_offsets ? aa.set_offsets[set] : 0;
    const long long off1 = aa.set_offsets ? aa.set_offsets[set + 1] : a.n;
    const long long i = off0 + (tile - s_prefix[set]) * Tt + threadIdx.x;
    const bool valid = i >= 0 && i < off1 && i < a.n;
    const double Ns = (double)(off1 - off0);
    // ---- forward pass with checkpoints
    Pos<PREC> pos;
    R u[3] = {R(0), R(0), R(0)};
    pos.load(valid ? a.x[i] : 0.0, valid ? a.y[i] : 0.0, valid ? a.z[i] : 0.0);
    if (valid) {
      u[0] = static_cast<const R *>(a.ux)[i];
      u[1] = static_cast<const R *>(a.uy)[i];
      u[2] = static_cast<const R *>(a.uz)[i];
    }
    TimeBase<PREC> tb;
    tb.init(P, a.t0, a.dt);
    const R dtR = (R)a.dt;
    const R dtxy = dtR * P.adv_xy;
    GridCache<R> gc;
    grid_cache_reset(gc);
    for (int seg = 0; seg < aa.n_seg; ++seg) {
      const long long s0 = (long long)seg * aa.K;
      const int cnt = (int)(a.n_steps - s0 < aa.K ? a.n_steps - s0 : aa.K);
      IO::put(ck + (size_t)seg * IO::W * stride, stride, pos, u);
      if constexpr (PREC == AP_FP32_PHASEFF) {
        __syncthreads();
        for (int k = threadIdx.x; k < cnt; k += blockDim.x) s_steps[k] = tb.at(s0 + k);
        __syncthreads();
      }
      for (int k = 0; k < cnt; ++k) {
        typename TimeBase<PREC>::Step st;
        if constexpr (PREC == AP_FP32_PHASEFF) st = s_steps[k];
        else st = tb.at(s0 + k);
        Local<R> L = local_coords<PREC>(P, st, pos);
        R E[3], B[3];
        analytic_fields<KIND, PREC>(P, L, E, B);
        if constexpr (GRID) grid_gather<R>(a.grid, gc, L.x, L.y, pos.zr(), E, B);
        R ig = boris(u, E, B, dtR);
        pos.advance(u[0] * ig, u[1] * ig, u[2] * ig, dtxy, dtR);
      }
    }
    // ---- objective and seed
    const double gN = sqrt(1.0 + (double)u[0] * u[0] + (double)u[1] * u[1] + (double)u[2] * u[2]);
    R lx[3] = {R(0), R(0), R(0)}, lu[3];
    for (int k = 0; k < 3; ++k) lu[k] = valid ? (R)((double)u[k] / (gN * Ns)) : R(0);
    double Jv = valid ? gN / Ns : 0.0;
    double gacc[kNp] = {0.0, 0.0, 0.0, 0.0};
    const PulseAD<R, tangents<KIND>()> A = make_ad<tangents<KIND>()>(P);
    // ---- reverse sweep over segments
    for (int seg = aa.n_seg - 1; seg >= 0; --seg) {
      const long long s0 = (long long)seg * aa.K;
      const int cnt = (int)(a.n_steps - s0 < aa.K ? a.n_steps - s0 : aa.K);
      IO::get(ck + (size_t)seg * IO::W * stride, stride, pos, u);
      if constexpr (PREC == AP_FP32_PHASEFF) {
        __syncthreads();
        for (int k = threadIdx.x; k < cnt; k += blockDim.x) s_steps[k] = tb.at(s0 + k);
        __syncthreads();
      }
      for (int k = 0; k < cnt; ++k) {
        IO::put(tp + (size_t)k * IO::W * stride, stride, pos, u);
        typename TimeBase<PREC>::Step st;
        if constexpr (PREC == AP_FP32_PHASEFF) st = s_steps[k];
        else st = tb.at(s0 + k);
        Local<R> L = local_coords<PREC>(P, st, pos);
        R E[3], B[3];
        analytic_fields<KIND, PREC>(P, L, E, B);
        if constexpr (GRID) grid_gather<R>(a.grid, gc, L.x, L.y, pos.zr(), E, B);
        R ig = boris(u, E, B, dtR);
        pos.advance(u[0] * ig, u[1] * ig, u[2] * ig, dtxy, dtR);
      }
      // the tape entries this thread just stored are read back by its own
      // asynchronous copies
      __threadfence_block();
      auto stage = [&](int k) {
        const T *src = tp + (size_t)k * IO::W * stride;
#pragma unroll
        for (int w = 0; w < IO::W; ++w) {
          const unsigned dst = (unsigned)__cvta_generic_to_shared(
              s_next + ((k & 1) * IO::W + w) * kAdjBlock + threadIdx.x);
          if constexpr (sizeof(T) == 8) cp_async8(dst, src + (size_t)w * stride);
          else cp_async4(dst, src + (size_t)w * stride);
        }
      };
      R gs[kNp] = {R(0), R(0), R(0), R(0)};
      stage(cnt - 1);
      for (int k = cnt - 1; k >= 0; --k) {
        cp_async_wait_all();
        IO::get(s_next + (k & 1) * IO::W * kAdjBlock + threadIdx.x, kAdjBlock, pos, u);
        if (k > 0) stage(k - 1);
        typename TimeBase<PREC>::Step st;
        if constexpr (PREC == AP_FP32_PHASEFF) st = s_steps[k];
        else st = tb.at(s0 + k);
        reverse_step<KIND, PREC, GRID>(P, A, aa, st, pos, u, lx, lu, gs, gc);
      }
      for (int k = 0; k < kNp; ++k) gacc[k] += (double)gs[k];
    }
    if (!valid) {
      gacc[0] = gacc[1] = gacc[2] = gacc[3] = 0.0;
      Jv = 0.0;
    } else if (!(isfinite(gacc[0]) && isfinite(gacc[1]) && isfinite(gacc[2]) && isfinite(gacc[3]))) {
      atomicOr(a.status, kStatusNonfinite);
    }
    // per-set reduction (every particle of the tile belongs to `set`)
    for (int k = 0; k < kNp; ++k) {
      double t = block_sum(gacc[k], s_red);
      if (threadIdx.x == 0) atomicAdd(aa.dJ + (size_t)set * AP_NPARAM + k, t);
    }
    if (aa.J) {
      double t = block_sum(Jv, s_red);
      if (threadIdx.x == 0) atomicAdd(aa.J + set, t);
    }
    __syncthreads();
  }
}

// ------------------------------------------------- two particles per thread
// The float-float adjoint of the Gaussian kinds without a grid, with each
// thread carrying two particles in the two halves of packed (f32x2) values.
// The forward sweep and the recomputation are the steps of the push
// (ap_step.cuh), in the pulse's frame; the reverse step is written for them.
// Tiles hold 2 kAdjBlock particles of one set (thread t: t and t + kAdjBlock).
//
// Bound by the FP32 pipe and its dependency chains: 155 operations per
// particle-step in the two forward passes and about 155 in the reverse step,
// where differentiating the field in each direction and the generic Boris
// reverse took 307 (and the two forward passes 250).  Measured, 64 sets, 1e6
// particles, 200 steps: 3.9 -> 2.47 ms with 3 blocks per SM (144 registers,
// FMA pipe 58 %, 12 warps) -> 2.30 ms with 4 (128 registers, 16 B spilled).
constexpr int kAdjPairBlocksPerSm = 4;

// A checkpoint holds the whole state; a tape entry what the reverse step
// reads (x and y to float, Z and the momentum).
struct PairIO {
  static constexpr int kCkpt = 9, kTape = 7;
  template <bool FULL>
  __device__ __forceinline__ static void put(float2 *b, size_t s, const FF2 &x, const FF2 &y, const FF2 &z, const F2 u[3]) {
    b[0 * s] = f2v(x.hi); b[1 * s] = f2v(y.hi); b[2 * s] = f2v(z.hi); b[3 * s] = f2v(z.lo);
    b[4 * s] = f2v(u[0]); b[5 * s] = f2v(u[1]); b[6 * s] = f2v(u[2]);
    if constexpr (FULL) { b[7 * s] = f2v(x.lo); b[8 * s] = f2v(y.lo); }
  }
  template <bool FULL>
  __device__ __forceinline__ static void get(const float2 *b, size_t s, FF2 &x, FF2 &y, FF2 &z, F2 u[3]) {
    x.hi = pair::f2of(b[0 * s]); y.hi = pair::f2of(b[1 * s]); z.hi = pair::f2of(b[2 * s]); z.lo = pair::f2of(b[3 * s]);
    u[0] = pair::f2of(b[4 * s]); u[1] = pair::f2of(b[5 * s]); u[2] = pair::f2of(b[6 * s]);
    if constexpr (FULL) { x.lo = pair::f2of(b[7 * s]); y.lo = pair::f2of(b[8 * s]); }
  }
};

// The reverse step's own constants: the factors of StepBase for a unit
// amplitude, and those of the field's derivatives with the amplitude in.
struct RevConst {
  float hbr, hce, hcb;    // h times B0/E0, the E_z and the B_z factor
  float dxy, dt;          // position increments per unit velocity
  float w2, a0;           // 2 a0/w0^2, a0
  float zr, k, eta, vg;   // 1/z_R, k, 2 ln2 s_env / v_g (Gaussian envelope), 1/v_g
  float omb;              // 1/(1 - beta_f)
};

// Gamma'/Gamma of the envelope at eta s_env (see envelope_dlog), times 1: the
// general form, for envelopes other than the Gaussian
template <class PT>
__device__ __forceinline__ F2 dlog_scaled(const PT &P, F2 e, F2 mul) {
  switch (P.env) {
    case AP_ENV_SIN2: {
      F2 s, c;
      sincos_r(e, &s, &c);
      return unless_zero(F2(-2.0f * P.fast.s_env) * s * rcp_r(c), mul);
    }
    case AP_ENV_GAUSS:
      return F2(-1.38629436f * P.fast.s_env) * e;
    case AP_ENV_SGAUSS: {
      const F2 u = sg_bound(e, P.sg_max), s = u * u;
      F2 p = F2(1.0f);
      for (int i = 1; i < P.sg_order; ++i) p *= s;
      return F2(-1.38629436f * P.env_b * (float)P.sg_order * P.fast.s_env) * u * p;
    }
    default:
      return F2(0.0f);
  }
}

// One reverse step for a thread's two particles: state (x, y, Z, u) before the
// step, adjoints lx (of x, y, z - z_f), lu after it, updated to before it.
//
// With q = 1/(1 - i zeta), a = r^2/w0^2, M the unit-amplitude envelope and
// carrier times e^{-a q}: U = q M, W = q U, and the unit fields are Re U, Im U,
// and x, y times Re W, Im W.  Let c be the cotangent of the fields (from the
// Boris reverse) in complex form, so that F . dF = Re(cU dU) + Re(cW dW) +
// (terms of x and y themselves).  Every derivative of U and W is a factor
// times U and W,
//   dU = U alpha, dW = W (alpha + i q dzeta),
//   alpha = i q (1 - a q) dzeta - q da + (Gamma'/Gamma) deta + i dpsi,
// so with Y = cU U + cW W the derivatives in da, dzeta, deta, dpsi are the
// four real numbers
//   S_a = -Re(q Y), S_zeta = Re(i q (1 - a q) Y) + Re(i q cW W),
//   (Gamma'/Gamma) Re Y, -Im Y,
// formed once, and each direction (x, y, z - z_f, w0, beta_f) is a short real
// combination of them.  Re Y is also F . f, the derivative in a0.
// gr: d/da0, (w0/2) d/dw0 / a0, d/dz_f / a0, d/dbeta_f / a0.
template <int KIND, int POL, int ENV, class PT>
__device__ __forceinline__ void reverse_step_pair(const PT &P, const StepBase &sb, const RevConst &rc, const float4 st,
                                                  F2 x, F2 y, F2 zhi, F2 zlo, const F2 u[3], F2 lx[3], F2 lu[3],
                                                  F2 gr[kNp]) {
  using R = F2;
  const FastPulse &F = P.fast;
  // unit fields, as in unit_fields_beam
  R eta = rfma(zhi, R(F.c_eta), R(st.y));
  if constexpr (ENV != kEnvGauss) eta = rfma(zhi, R(F.c_eta_lo), eta);
  R mul, g;
  envelope_fast<ENV>(P, eta, mul, g);
  const R zn = KIND == AP_FLYING_CF ? rfma(zhi, R(F.c_zn), R(st.z)) : rmul(zhi, R(F.c_zn));
  const R inv = rcp_r(rfma(zn, zn, R(1.0f)));
  const R nq = rmul(zn, inv), qi = rneg(nq);
  const R b = rmul(rfma(x, x, rmul(y, y)), R(F.c_a));
  const R ang = phase_angle(rfma(b, rmul(nq, R(kTurnsPerExp)), R(st.x)), zhi, zlo);
  R sn, cs;
  sincos_r(ang, &sn, &cs);
  R mag = exp2_neg(rfma(b, inv, g));
  if constexpr (ENV == kEnvAny) mag = rmul(mag, mul);
  const R mc = rmul(mag, cs), ms = rmul(mag, sn);
  const R Ur = rfma(inv, mc, rmul(nq, ms)), Ui = rfma(inv, ms, rmul(qi, mc));
  const R Wr = rfma(inv, Ur, rmul(nq, Ui)), Wi = rfma(inv, Ui, rmul(qi, Ur));
  const R ny = rneg(y);
  const R ez = POL == kLin ? rmul(x, Wi) : rfma(x, Wi, rmul(ny, Wr));
  const R bz = POL == kLin ? rmul(y, Wi) : rfma(x, Wr, rmul(y, Wi));
  // Boris forward intermediates (boris_unit)
  const R a0 = rfma(R(sb.hA), Ur, u[0]), a1 = POL == kCirc ? rfma(R(sb.hA), Ui, u[1]) : u[1];
  const R a2 = rfma(R(sb.hAce), ez, u[2]);
  const R am[3] = {a0, a1, a2};
  const R ig = inv_gamma(am);
  const R hb = rmul(R(sb.hAbr), ig);
  const R t1 = rmul(hb, Ur), nt1 = rneg(t1);
  const R t2 = rmul(rmul(R(sb.hAcb), ig), bz), nt2 = rneg(t2);
  R t0 = R(0.0f), nt0 = R(0.0f);
  R tt = rfma(t1, t1, rfma(t2, t2, R(1.0f)));
  R p0 = rfma(a1, t2, rfma(a2, nt1, a0)), p1 = rfma(a0, nt2, a1), p2 = rfma(a0, t1, a2);
  if constexpr (POL == kCirc) {
    nt0 = rmul(hb, Ui);
    t0 = rneg(nt0);
    tt = rfma(t0, t0, tt);
    p1 = rfma(a2, t0, p1);
    p2 = rfma(a1, nt0, p2);
  }
  const R ii = rcp_r(tt);
  const R f = radd(ii, ii);
  const R s1 = rmul(f, t1), s2 = rmul(f, t2), ns1 = rneg(s1), ns2 = rneg(s2);
  const R s0 = POL == kCirc ? rmul(f, t0) : R(0.0f), ns0 = POL == kCirc ? rneg(s0) : R(0.0f);
  R un[3] = {rfma(R(sb.hA), Ur, rfma(p1, s2, rfma(p2, ns1, a0))), rfma(p0, ns2, a1), rfma(p0, s1, a2)};
  if constexpr (POL == kCirc) {
    un[1] = rfma(R(sb.hA), Ui, rfma(p2, s0, un[1]));
    un[2] = rfma(p1, ns0, un[2]);
  }
  un[2] = rfma(R(sb.hAce), ez, un[2]);
  const R ign = inv_gamma(un);
  // position update: ub = lu + (d - v (v . d)) / gamma', d = dt lx
  const R v[3] = {rmul(un[0], ign), rmul(un[1], ign), rmul(un[2], ign)};
  const R d[3] = {rmul(R(rc.dxy), lx[0]), rmul(R(rc.dxy), lx[1]), rmul(R(rc.dt), lx[2])};
  const R nvl = rneg(rfma(v[0], d[0], rfma(v[1], d[1], rmul(v[2], d[2]))));
  const R b0 = rfma(ign, rfma(v[0], nvl, d[0]), lu[0]), b1 = rfma(ign, rfma(v[1], nvl, d[1]), lu[1]);
  const R b2 = rfma(ign, rfma(v[2], nvl, d[2]), lu[2]);
  // rotation: pb = s x ub, sbar = ub x p, ab = ub + pb + t x pb, tb = pb x a + ds/dt sbar
  R pb0 = rfma(s1, b2, rmul(ns2, b1)), pb1 = rmul(s2, b0), pb2 = rmul(ns1, b0);
  if constexpr (POL == kCirc) {
    pb1 = rfma(ns0, b2, pb1);
    pb2 = rfma(s0, b1, pb2);
  }
  const R nb0 = rneg(b0), npb0 = rneg(pb0);
  const R sb1 = rfma(b2, p0, rmul(nb0, p2)), sb2 = rfma(b0, p1, rmul(rneg(b1), p0));
  R ab0 = rfma(t1, pb2, rfma(nt2, pb1, radd(b0, pb0)));
  R ab1 = rfma(t2, pb0, radd(b1, pb1));
  R ab2 = rfma(t1, npb0, radd(b2, pb2));
  R tb1 = rfma(pb2, a0, rmul(npb0, a2)), tb2 = rfma(pb0, a1, rmul(rneg(pb1), a0));
  R ts = rfma(t1, sb1, rmul(t2, sb2));
  R tb0 = R(0.0f);
  R sb0 = R(0.0f);
  if constexpr (POL == kCirc) {
    ab1 = rfma(nt0, pb2, ab1);
    ab2 = rfma(t0, pb1, ab2);
    sb0 = rfma(b1, p2, rmul(rneg(b2), p1));
    tb0 = rfma(pb1, a2, rmul(rneg(pb2), a1));
    ts = rfma(t0, sb0, ts);
  }
  // s = f t, f = 2/(1 + t^2): tb += f (sbar - f (t . sbar) t)
  const R nfts = rneg(rmul(f, ts));
  tb1 = rfma(f, rfma(nfts, t1, sb1), tb1);
  tb2 = rfma(f, rfma(nfts, t2, sb2), tb2);
  if constexpr (POL == kCirc) tb0 = rfma(f, rfma(nfts, t0, sb0), tb0);
  // t = h B / gamma: the cotangent of 1/gamma is (t . tb) gamma
  R tt2 = rfma(t1, tb1, rmul(t2, tb2));
  if constexpr (POL == kCirc) tt2 = rfma(t0, tb0, tt2);
  const R c3 = rneg(rmul(rmul(ig, ig), tt2));
  ab0 = rfma(c3, a0, ab0);
  ab1 = rfma(c3, a1, ab1);
  ab2 = rfma(c3, a2, ab2);
  lu[0] = ab0;
  lu[1] = ab1;
  lu[2] = ab2;
  // cotangents of the unit fields' parts
  const R hb1 = rmul(R(rc.hbr), ig);
  const R cR = rfma(R(sb.h), radd(b0, ab0), rmul(hb1, tb1));
  const R cE = rmul(R(rc.hce), radd(b2, ab2)), cB = rmul(rmul(R(rc.hcb), ig), tb2);
  const R cWi = rfma(cE, x, rmul(cB, y));
  R Zr = rmul(cWi, Wi), Zi = rmul(rneg(cWi), Wr);  // cW W
  R Yr = rmul(cR, Ur), Yi = rmul(cR, Ui);
  if constexpr (POL == kCirc) {
    const R cWr = rfma(cB, x, rmul(cE, ny));
    Zr = rfma(cWr, Wr, Zr);
    Zi = rfma(cWr, Wi, Zi);
    const R cI = rfma(R(sb.h), radd(b1, ab1), rmul(rneg(hb1), tb0));
    Yr = rfma(cI, Ui, Yr);
    Yi = rfma(rneg(cI), Ur, Yi);
  }
  Yr = radd(Yr, Zr);
  Yi = radd(Yi, Zi);
  const R Pr = rfma(inv, Yr, rmul(nq, Yi)), Pi = rfma(inv, Yi, rmul(qi, Yr));
  const R qPi = rfma(inv, Pi, rmul(qi, Pr));
  const R a = rmul(b, R(0.693147181f));
  // S_zeta = a Im(q^2 Y) - Im(q Y) - Im(q cW W)
  const R Sz = rsub(rfma(a, qPi, rmul(nq, Zr)), rfma(inv, Zi, Pi));
  // direct terms of x and y, and the directions
  const R wE = rmul(R(rc.a0), cE), wB = rmul(R(rc.a0), cB);
  const R sa = rmul(R(-rc.w2), Pr);
  lx[0] = rfma(sa, x, rfma(wE, Wi, lx[0]));
  lx[1] = rfma(sa, y, rfma(wB, Wi, lx[1]));
  if constexpr (POL == kCirc) {
    lx[0] = rfma(wB, Wr, lx[0]);
    lx[1] = rfma(rneg(wE), Wr, lx[1]);
  }
  R dz = rfma(R(rc.k), Yi, rmul(R(rc.zr), Sz));
  if constexpr (ENV == kEnvGauss) dz = rfma(rmul(R(rc.eta), eta), Yr, dz);
  else dz = rfma(rmul(R(-rc.vg), dlog_scaled(P, eta, mul)), Yr, dz);
  // per unit amplitude: k = 1 stays exact (a rounded k a0 would shift the whole
  // carrier part of d/dz_f, which cancels to a small rest over the particles)
  lx[2] = rfma(R(rc.a0), dz, lx[2]);
  gr[0] = radd(gr[0], Yr);
  gr[1] = rfma(Pr, a, rfma(Sz, zn, rsub(gr[1], Zr)));
  gr[2] = rsub(gr[2], dz);
  if constexpr (KIND == AP_FLYING_CF)
    gr[3] = rfma(Sz, rfma(zn, R(-rc.omb), R(-rc.zr * st.w)), gr[3]);
}

template <int KIND>
__global__ void __launch_bounds__(kAdjBlock, kAdjPairBlocksPerSm)
    adjoint_kernel_pair(const Pulse<float> *__restrict__ sets, const __grid_constant__ AdjArgs aa) {
  static_assert(KIND == AP_GAUSS || KIND == AP_FLYING_CF, "kinds with closed-form field derivatives");
  __shared__ long long s_tile;
  __shared__ int s_set;
  __shared__ double s_red[32];
  __shared__ float4 s_steps[kAdjMaxK];
  __shared__ StepBase s_base;
  __shared__ RevConst s_rev;
  __shared__ __align__(16) unsigned char s_pulse_raw[sizeof(PulseHead<float>)];
  // dynamic: the next reverse step's tape entry, [2][kTape][kAdjBlock] float2,
  // then the [n_sets + 1] tile prefix
  extern __shared__ __align__(16) unsigned char s_adj_dyn[];
  float2 *s_next = reinterpret_cast<float2 *>(s_adj_dyn);
  long long *s_prefix = reinterpret_cast<long long *>(s_adj_dyn + 2 * PairIO::kTape * kAdjBlock * sizeof(float2));
  PulseHead<float> &P = *reinterpret_cast<PulseHead<float> *>(s_pulse_raw);
  const PushArgs &a = aa.base;
  constexpr int kPer = 2 * kAdjBlock;  // particles per tile
  tile_prefix(s_prefix, aa.n_sets, kPer,
              [&](int s) { return aa.set_offsets ? aa.set_offsets[s + 1] - aa.set_offsets[s] : a.n; });
  if (threadIdx.x == 0) s_set = -1;
  __syncthreads();
  const long long total = s_prefix[aa.n_sets];
  const size_t slot = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t stride = (size_t)gridDim.x * kAdjBlock;  // thread slots
  float2 *ck = static_cast<float2 *>(aa.ckpt) + slot;
  float2 *tp = static_cast<float2 *>(aa.tape) + slot;
  const float *uxs = static_cast<const float *>(a.ux);
  const float *uys = static_cast<const float *>(a.uy);
  const float *uzs = static_cast<const float *>(a.uz);
  for (;;) {
    if (threadIdx.x == 0) s_tile = (long long)atomicAdd(aa.tile_counter, 1u);
    __syncthreads();
    const long long tile = s_tile;
    if (tile >= total) break;
    int lo = 0, hi = aa.n_sets;
    while (hi - lo > 1) {
      int mid = (lo + hi) >> 1;
      if (s_prefix[mid] <= tile) lo = mid; else hi = mid;
    }
    const int set = lo;
    if (set != s_set) {
      const int words = (int)(sizeof(PulseHead<float>) / 4);
      const uint32_t *src = reinterpret_cast<const uint32_t *>(sets + set);
      uint32_t *dst = reinterpret_cast<uint32_t *>(s_pulse_raw);
      for (int w = threadIdx.x; w < words; w += blockDim.x) dst[w] = src[w];
      __syncthreads();
      if (threadIdx.x == 0) {
        s_set = set;
        s_base = make_step_base(P, a.t0, a.dt, a.grid);
        const FastPulse &F = P.fast;
        const float g = P.lon ? -2.0f * P.inv_w0sq : 0.0f, a0 = P.a0, h = s_base.h;
        // the derivatives' constants from the rounded ones of the step itself, so
        // that the reverse differentiates the map that ran (the terms of d/dz_f
        // cancel to a small rest)
        const double eta_z = (double)F.c_eta * F.z_scale;  // d(eta s_env)/dz
        s_rev = RevConst{h * P.bratio, h * P.lonE * g, h * P.bratio * P.lonB * g,
                         (float)a.dt * P.adv_xy, (float)((double)s_base.cz * F.z_len),
                         (float)(2.0 * 0.69314718055994531 * (double)F.c_a) * a0, a0,
                         (float)(-(double)F.c_zn * F.z_scale), (float)P.k,
                         (float)(-2.0 * 0.69314718055994531 * eta_z), (float)(-eta_z / (double)F.s_env), P.inv_1mb};
      }
    }
    __syncthreads();
    const long long off0 = aa.set_offsets ? aa.set_offsets[set] : 0;
    const long long off1 = aa.set_offsets ? aa.set_offsets[set + 1] : a.n;
    const long long i0 = off0 + (tile - s_prefix[set]) * kPer + threadIdx.x;
    const long long i1 = i0 + kAdjBlock;
    const bool v0 = i0 >= 0 && i0 < off1 && i0 < a.n;
    const bool v1 = i1 >= 0 && i1 < off1 && i1 < a.n;
    const double Ns = (double)(off1 - off0);
    // ---- load, in the pulse's frame
    FF px[2], py[2], pz[2];
    float uu[2][3];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      px[h] = py[h] = pz[h] = FF{0.0f, 0.0f};
      uu[h][0] = uu[h][1] = uu[h][2] = 0.0f;
      if (h ? v1 : v0) {
        const long long i = h ? i1 : i0;
        px[h] = split_double(a.x[i]);
        py[h] = split_double(a.y[i]);
        pz[h] = split_double(__dmul_rn(__dsub_rn(a.z[i], P.z_f), P.fast.z_scale));
        uu[h][0] = uxs[i];
        uu[h][1] = uys[i];
        uu[h][2] = uzs[i];
        to_frame(P.fast.frame, px[h], py[h], uu[h]);
      }
    }
    FF2 x{F2(px[0].hi, px[1].hi), F2(px[0].lo, px[1].lo)};
    FF2 y{F2(py[0].hi, py[1].hi), F2(py[0].lo, py[1].lo)};
    FF2 z{F2(pz[0].hi, pz[1].hi), F2(pz[0].lo, pz[1].lo)};
    F2 u[3] = {F2(uu[0][0], uu[1][0]), F2(uu[0][1], uu[1][1]), F2(uu[0][2], uu[1][2])};
    double Jv = 0.0, gacc[kNp] = {0.0, 0.0, 0.0, 0.0};

    auto sweep = [&](auto pol_c, auto env_c) {
      constexpr int POL = decltype(pol_c)::value, ENV = decltype(env_c)::value;
      auto table = [&](long long s0, int cnt) {
        __syncthreads();
        for (int k = threadIdx.x; k < cnt; k += blockDim.x)
          s_steps[k] = step_entry<KIND>(P.fast, s_base, (float)(int)(s0 + k));
        __syncthreads();
      };
      auto step = [&](int k) {
        const UnitFields<F2> f = unit_fields<KIND, POL, ENV>(P, nullptr, s_steps[k], x.hi, y.hi, z.hi, z.lo);
        const F2 ig = boris_unit<POL, true>(u, f, s_base);
        const F2 kxy = rmul(F2(s_base.cxy), ig);
        advance(x, u[0], kxy);
        advance(y, u[1], kxy);
        advance(z, u[2], rmul(F2(s_base.cz), ig));
      };
      // ---- forward pass with checkpoints
      for (int seg = 0; seg < aa.n_seg; ++seg) {
        const long long s0 = (long long)seg * aa.K;
        const int cnt = (int)(a.n_steps - s0 < aa.K ? a.n_steps - s0 : aa.K);
        PairIO::put<true>(ck + (size_t)seg * PairIO::kCkpt * stride, stride, x, y, z, u);
        table(s0, cnt);
        for (int k = 0; k < cnt; ++k) step(k);
      }
      // ---- objective and seed, per particle
      float sd[2][3];
      for (int h = 0; h < 2; ++h) {
        const bool vh = h ? v1 : v0;
        const double d0 = lane_of(u[0], h), d1 = lane_of(u[1], h), d2 = lane_of(u[2], h);
        const double gN = sqrt(1.0 + d0 * d0 + d1 * d1 + d2 * d2);
        const double w = vh ? 1.0 / (gN * Ns) : 0.0;
        sd[h][0] = (float)(d0 * w);
        sd[h][1] = (float)(d1 * w);
        sd[h][2] = (float)(d2 * w);
        if (vh) Jv += gN / Ns;
      }
      F2 lx[3] = {F2(0.0f), F2(0.0f), F2(0.0f)};
      F2 lu[3] = {F2(sd[0][0], sd[1][0]), F2(sd[0][1], sd[1][1]), F2(sd[0][2], sd[1][2])};
      // ---- reverse sweep over segments
      for (int seg = aa.n_seg - 1; seg >= 0; --seg) {
        const long long s0 = (long long)seg * aa.K;
        const int cnt = (int)(a.n_steps - s0 < aa.K ? a.n_steps - s0 : aa.K);
        PairIO::get<true>(ck + (size_t)seg * PairIO::kCkpt * stride, stride, x, y, z, u);
        table(s0, cnt);
        for (int k = 0; k < cnt; ++k) {
          PairIO::put<false>(tp + (size_t)k * PairIO::kTape * stride, stride, x, y, z, u);
          step(k);
        }
        // the tape entries this thread just stored are read back by its own
        // asynchronous copies
        __threadfence_block();
        auto stage = [&](int k) {
          const float2 *src = tp + (size_t)k * PairIO::kTape * stride;
#pragma unroll
          for (int w = 0; w < PairIO::kTape; ++w)
            cp_async8((unsigned)__cvta_generic_to_shared(s_next + ((k & 1) * PairIO::kTape + w) * kAdjBlock +
                                                         threadIdx.x),
                      src + (size_t)w * stride);
        };
        F2 gs[kNp] = {F2(0.0f), F2(0.0f), F2(0.0f), F2(0.0f)};
        stage(cnt - 1);
        for (int k = cnt - 1; k >= 0; --k) {
          cp_async_wait_all();
          PairIO::get<false>(s_next + (k & 1) * PairIO::kTape * kAdjBlock + threadIdx.x, kAdjBlock, x, y, z, u);
          if (k > 0) stage(k - 1);
          reverse_step_pair<KIND, POL, ENV>(P, s_base, s_rev, s_steps[k], x.hi, y.hi, z.hi, z.lo, u, lx, lu, gs);
        }
        for (int k = 0; k < kNp; ++k)
          gacc[k] += (v0 ? (double)gs[k].x : 0.0) + (v1 ? (double)gs[k].y : 0.0);
      }
    };
    using Lin = std::integral_constant<int, kLin>;
    using Circ = std::integral_constant<int, kCirc>;
    using EnvG = std::integral_constant<int, kEnvGauss>;
    using EnvA = std::integral_constant<int, kEnvAny>;
    if (P.fast.circ) sweep(Circ{}, EnvA{});
    else if (P.env == AP_ENV_GAUSS) sweep(Lin{}, EnvG{});
    else sweep(Lin{}, EnvA{});
    gacc[1] *= 2.0 * (double)P.inv_w0 * (double)P.a0;
    gacc[2] *= (double)P.a0;
    gacc[3] *= (double)P.a0;

    if ((v0 || v1) && !(isfinite(gacc[0]) && isfinite(gacc[1]) && isfinite(gacc[2]) && isfinite(gacc[3])))
      atomicOr(a.status, kStatusNonfinite);
    // per-set reduction (every particle of the tile belongs to `set`)
    for (int k = 0; k < kNp; ++k) {
      double t = block_sum(gacc[k], s_red);
      if (threadIdx.x == 0) atomicAdd(aa.dJ + (size_t)set * AP_NPARAM + k, t);
    }
    if (aa.J) {
      double t = block_sum(Jv, s_red);
      if (threadIdx.x == 0) atomicAdd(aa.J + set, t);
    }
    __syncthreads();
  }
}

// The two-particle kernel's segment length: any split of the steps whose
// checkpoints (9 floats) and tape (7 floats per step) fit the caller's
// workspace (n_seg + K states of 12 floats for aa.nslots particles, shared out
// over `slots` here) retraces the same states (the gradient's last bits depend on
// it: each segment is summed in float), and the shorter the segment the
// smaller the tape.  From 16 steps up it stays in the L2 cache (70 MB of 129 at
// 16 steps; at 100 steps 436 MB would go through HBM, 56 bytes per
// particle-step), below 16 the checkpoints' own traffic grows.
inline void pair_segments(AdjArgs &aa, long long slots) {
  const long long n = aa.base.n_steps, budget = 12LL * (aa.n_seg + aa.K) * aa.nslots / slots;
  for (int K = 16; K < aa.K; K += 4) {
    const long long seg = (n + K - 1) / K;
    if (PairIO::kCkpt * seg + PairIO::kTape * K <= budget) {
      aa.K = K;
      aa.n_seg = (int)seg;
      return;
    }
  }
}

template <int KIND>
int launch_adjoint_pair(const Pulse<float> *sets, const AdjArgs &a0, void *stream) {
  auto kern = adjoint_kernel_pair<KIND>;
  AdjArgs aa = a0;
  const int grid = aa.base.sm_count * kAdjPairBlocksPerSm;
  const long long slots = (long long)grid * 2 * kAdjBlock;
  static_assert(kAdjPairBlocksPerSm * 2 * kAdjBlock * 3 <= kAdjSlotsPerSm * 4,
                "9 n_seg + 7 K floats fit the workspace for every K");
  pair_segments(aa, slots);
  aa.tape = static_cast<char *>(aa.ckpt) + sizeof(float) * PairIO::kCkpt * (size_t)aa.n_seg * (size_t)slots;
  const size_t dyn = 2 * (size_t)PairIO::kTape * kAdjBlock * sizeof(float2) + (size_t)(aa.n_sets + 1) * sizeof(long long);
  constexpr size_t most =
      2 * (size_t)PairIO::kTape * kAdjBlock * sizeof(float2) + (size_t)(AP_MAX_SETS + 1) * sizeof(long long);
  if (allow_smem(reinterpret_cast<const void *>(kern), most) != AP_OK) return AP_ERR_CUDA;
  kern<<<grid, kAdjBlock, dyn, static_cast<cudaStream_t>(stream)>>>(sets, aa);
  return cudaGetLastError() == cudaSuccess ? AP_OK : AP_ERR_CUDA;
}

template <int KIND, int PREC, bool GRID>
int launch_adjoint_t(const Pulse<Real<PREC>> *sets, const AdjArgs &aa, int grid, void *stream) {
  auto kern = adjoint_kernel<KIND, PREC, GRID>;
  const size_t dyn = 2 * (size_t)StateIO<PREC>::W * kAdjBlock * sizeof(typename StateIO<PREC>::T);
  // static (about 40 KB) plus dynamic shared memory passes 48 KB: opt in
  if (allow_smem(reinterpret_cast<const void *>(kern), dyn) != AP_OK) return AP_ERR_CUDA;
  kern<<<grid, kAdjBlock, dyn, static_cast<cudaStream_t>(stream)>>>(sets, aa);
  return cudaGetLastError() == cudaSuccess ? AP_OK : AP_ERR_CUDA;
}

template <int KIND>
int launch_adjoint_k(int precision, const Pulse<double> *dpd, const Pulse<float> *dpf,
                     const AdjArgs &aa, int grid, void *stream) {
  const bool gr = aa.base.grid_on != 0;
  if (precision == AP_FP64)
    return gr ? launch_adjoint_t<KIND, AP_FP64, true>(dpd, aa, grid, stream)
              : launch_adjoint_t<KIND, AP_FP64, false>(dpd, aa, grid, stream);
  if (precision == AP_FP32_PHASEFF) {
    if (gr) return launch_adjoint_t<KIND, AP_FP32_PHASEFF, true>(dpf, aa, grid, stream);
    if constexpr (KIND == AP_GAUSS || KIND == AP_FLYING_CF) return launch_adjoint_pair<KIND>(dpf, aa, stream);
    else return launch_adjoint_t<KIND, AP_FP32_PHASEFF, false>(dpf, aa, grid, stream);
  }
  return AP_ERR_UNSUPPORTED;
}

}  // namespace apt

// Host side: the handle internals live in ap_api.cu; these accessors expose
// what the adjoint launch needs.
namespace apt {
int handle_info(ap_handle h, int *device, int *sm_count, int *n_sets, int *uniform_kind,
                const Pulse<double> **dpd, const Pulse<float> **dpf, int **status);
int handle_push_args(ap_handle h, const ap_particles *p, const ap_grid *g, double t0, double dt,
                     int64_t n_steps, int32_t precision, PushArgs *a, void *stream);
}  // namespace apt

namespace {
// particle slots of the workspace (the one-particle kernel uses kAdjBlocksPerSm
// blocks of kAdjBlock per SM of them; the two-particle kernel shares the same
// bytes out over its own slots)
long long adj_slots(int sm_count) { return (long long)sm_count * apt::kAdjSlotsPerSm; }
}  // namespace

extern "C" {

size_t ap_adjoint_workspace_bytes(ap_handle h, int64_t n, int64_t n_steps, int32_t ckpt_every) {
  int dev, sm, ns, uk, *st;
  const apt::Pulse<double> *pd;
  const apt::Pulse<float> *pf;
  if (!h || n < 0 || n_steps < 1 || ckpt_every < 1 || ckpt_every > apt::kAdjMaxK) return 0;
  if (apt::handle_info(h, &dev, &sm, &ns, &uk, &pd, &pf, &st) != AP_OK) return 0;
  const long long slots = adj_slots(sm);
  const long long n_seg = (n_steps + ckpt_every - 1) / ckpt_every;
  return 256 + (size_t)(n_seg + ckpt_every) * apt::kAdjStateBytes * (size_t)slots;
}

int ap_push_adjoint(ap_handle h, const ap_particles *p0, const ap_grid *g, double t0, double dt,
                    int64_t n_steps, int32_t ckpt_every, int32_t objective, int32_t precision,
                    double *dJ_dparams, double *J_out, void *workspace, size_t ws_bytes,
                    void *stream) {
  int dev, sm, ns, uk, *status;
  const apt::Pulse<double> *dpd;
  const apt::Pulse<float> *dpf;
  if (!h || !p0 || !dJ_dparams) return AP_ERR_ARG;
  int rc = apt::handle_info(h, &dev, &sm, &ns, &uk, &dpd, &dpf, &status);
  if (rc != AP_OK) return rc;
  if (objective != AP_OBJ_MEAN_GAMMA) return AP_ERR_ARG;
  if (precision != AP_FP64 && precision != AP_FP32_PHASEFF) return AP_ERR_UNSUPPORTED;
  if (uk < 0 || uk == AP_FLYING_SUM) return AP_ERR_UNSUPPORTED;
  if (n_steps < 1 || ckpt_every < 1 || ckpt_every > apt::kAdjMaxK) return AP_ERR_ARG;
  if (p0->set_offsets ? p0->n_sets != ns : ns != 1) return AP_ERR_ARG;
  const size_t need = ap_adjoint_workspace_bytes(h, p0->n, n_steps, ckpt_every);
  if (!workspace || ws_bytes < need) return AP_ERR_WORKSPACE;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return AP_ERR_ALIGN;
  apt::AdjArgs aa;
  std::memset(&aa, 0, sizeof(aa));
  rc = apt::handle_push_args(h, p0, g, t0, dt, n_steps, precision, &aa.base, stream);
  if (rc != AP_OK) return rc;
  if (aa.base.grid.cells) {
    rc = apt::drop_cell_layout(aa.base.grid);
    if (rc != AP_OK) return rc;
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (cudaMemsetAsync(dJ_dparams, 0, sizeof(double) * AP_NPARAM * ns, s) != cudaSuccess ||
      (J_out && cudaMemsetAsync(J_out, 0, sizeof(double) * ns, s) != cudaSuccess) ||
      cudaMemsetAsync(workspace, 0, 256, s) != cudaSuccess)
    return AP_ERR_CUDA;
  if (p0->n == 0) return AP_OK;
  const long long slots = adj_slots(sm);
  const long long n_seg = (n_steps + ckpt_every - 1) / ckpt_every;
  char *ws = static_cast<char *>(workspace);
  const size_t w = (precision == AP_FP64) ? sizeof(double) * 6 : sizeof(float) * 9;
  aa.set_offsets = reinterpret_cast<const long long *>(p0->set_offsets);
  aa.n_sets = ns;
  aa.K = ckpt_every;
  aa.n_seg = (int)n_seg;
  aa.tile_counter = reinterpret_cast<unsigned int *>(ws);
  aa.ckpt = ws + 256;
  aa.tape = ws + 256 + (size_t)n_seg * w * slots;
  aa.nslots = slots;
  aa.dJ = dJ_dparams;
  aa.J = J_out;
  const int grid = sm * apt::kAdjBlocksPerSm;  // the one-particle kernel's launch
  switch (uk) {
    case AP_PLANE: return apt::launch_adjoint_k<AP_PLANE>(precision, dpd, dpf, aa, grid, stream);
    case AP_GAUSS: return apt::launch_adjoint_k<AP_GAUSS>(precision, dpd, dpf, aa, grid, stream);
    case AP_LG: return apt::launch_adjoint_k<AP_LG>(precision, dpd, dpf, aa, grid, stream);
    case AP_FLYING_CF:
      return apt::launch_adjoint_k<AP_FLYING_CF>(precision, dpd, dpf, aa, grid, stream);
    default: return AP_ERR_UNSUPPORTED;
  }
}

}  // extern "C"
