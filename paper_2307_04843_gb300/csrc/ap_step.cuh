// ap_step.cuh -- one float-float step (AP_FP32_PHASEFF) of the push with as
// few FP32 operations as the method needs, for one particle (R = float) or
// two (R = F2, ap_pair.cuh) per thread.
//
// The push without a grid is bound by the FP32 pipe, so what counts is how
// many lane operations a step takes.  Against the generic field code of
// ap_device.cuh (which the FP64 and PHASE64 pushes, the node kernels and the
// field hook use) four things are done differently:
//
//   - the longitudinal position is carried in turns of the carrier,
//     Z = k (z - z_f) / 2 pi, as a float-float sum: the carrier phase modulo
//     one turn is then Z minus its nearest integer, which is exact in float,
//     instead of a float-float product by k and a two-constant reduction by
//     2 pi.  The profile's own phase (curvature and Gouy) joins before the one
//     reduction.  26 -> 9 operations per particle-step;
//   - every product that feeds a sum is one fused operation (the packed type
//     is not contracted by the compiler): the cross products of the Boris
//     rotation, the complex products, the position update;
//   - the polarisation is a compile-time parameter (linear or circular; y and
//     the other handedness run in a rotated or mirrored frame), so identically
//     zero components cost nothing, and amplitude, B0/E0, the longitudinal
//     factors and the half step are folded into the kick's constants;
//   - the high part of a compensated sum is already its rounded value: x, y
//     and Z are read without adding the low part.
//
// For a linearly polarised Gaussian beam this is 77 packed operations per
// step against 131.  Every operation is written with a single rounding
// (rmul, radd, rsub, rfma), and no product has sums alone for its uses (the
// assembler would fuse a packed one with them, see ap_pair.cuh), so the one- and
// two-particle kernels give the same bits.
//
// Measured on a GB300, before and after (two particles per thread; ncu of the
// batched Gaussian: 112 instructions per pair-step, FMA pipe 71 %, special
// functions 51 %; of the flying focus: 22 FP32 and 7 special-function
// instructions per component and pair, pipes 60 and 71 %):
//   256 Gaussian sets, 4e6 particles x 500 steps     7.43 -> 4.88 ms
//   CP LG_{1,2}, 3.2e6 x 300                         6.56 -> 4.80 ms
//   64-component flying focus, 1e6 x 200            15.40 -> 11.52 ms
//   Gaussian + 256^3 grid, 4e6 x 400                11.62 -> 10.13 ms
// The error against 64 bits fell too, to about half (the largest relative error,
// norm over norm, of an output, on one set of inputs each: 1.7e-6 -> 7.6e-7, 1.6e-6
// -> 8.9e-7, 7.5e-6 -> 3.3e-7, 1.3e-6 -> 5.9e-7).
#pragma once

#include "ap_pair.cuh"

namespace apt {

// ----------------------------------------------- operations of one rounding
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float rsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float rneg(float a) { return -a; }
__device__ __forceinline__ float exp2_neg(float a) { return mufu_ex2(-a); }
__device__ __forceinline__ float sin2_window(float m, float eta, float b) { return fabsf(eta) > b ? 0.0f : m; }
__device__ __forceinline__ FF two_diff(float a, float b) { return two_sum(a, -b); }
__device__ __forceinline__ float clamp_abs(float a, float b) { return fminf(fmaxf(a, -b), b); }

// double: the FP64 push's Boris step (push_d); sums of products contract by
// themselves
__device__ __forceinline__ double rmul(double a, double b) { return a * b; }
__device__ __forceinline__ double radd(double a, double b) { return a + b; }
__device__ __forceinline__ double rfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double rneg(double a) { return -a; }

namespace pair {
__device__ __forceinline__ F2 rmul(F2 a, F2 b) { return a * b; }
__device__ __forceinline__ F2 radd(F2 a, F2 b) { return a + b; }
__device__ __forceinline__ F2 rsub(F2 a, F2 b) { return a - b; }
__device__ __forceinline__ F2 rfma(F2 a, F2 b, F2 c) { return fma(a, b, c); }
// sign flip of both halves on the integer pipe, which the step leaves idle
// (a packed negation would be a packed multiplication on the FP32 pipe)
__device__ __forceinline__ F2 rneg(F2 a) {
  F2 d;
  asm("xor.b32 %0, %2, 0x80000000;\n\txor.b32 %1, %3, 0x80000000;"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y));
  return d;
}
__device__ __forceinline__ F2 exp2_neg(F2 a) { return F2(mufu_ex2(-a.x), mufu_ex2(-a.y)); }
__device__ __forceinline__ F2 clamp_abs(F2 a, float b) {
  return F2(fminf(fmaxf(a.x, -b), b), fminf(fmaxf(a.y, -b), b));
}
}  // namespace pair

template <typename R>
struct FFOf {
  using type = FF;
};
template <>
struct FFOf<F2> {
  using type = FF2;
};

template <typename R>
__device__ __forceinline__ R round_magic(R x) {
  return rsub(radd(x, R(kRoundMagic)), R(kRoundMagic));
}

// ------------------------------------------------------- per-call constants
// What a step needs of (t0, dt), the pulse and the grid, in the arithmetic of
// the step.  Made once per launch on the host for a single set and once per
// set of a tile on the device for the batched launch, by the same double
// operations (each rounded by itself), so both give the same bits.
__host__ __device__ inline double d_mul(double a, double b) {
#ifdef __CUDA_ARCH__
  return __dmul_rn(a, b);
#else
  return a * b;
#endif
}
__host__ __device__ inline double d_add(double a, double b) {
#ifdef __CUDA_ARCH__
  return __dadd_rn(a, b);
#else
  return a + b;
#endif
}

__host__ __device__ inline double d_div(double a, double b) {
#ifdef __CUDA_ARCH__
  return __ddiv_rn(a, b);
#else
  return a / b;
#endif
}

struct StepBase {
  FF om0, del;  // carrier phase of step n, in turns: om0 + n del
  FF T0, DT;    // T_n = T0 + n DT: t_n - t_f, for the flying focus in turns of omega
  float cxy, cz;               // position increments per unit velocity: dt, and dt k / 2 pi
  float h, k;                  // the half and the whole electric kick: -dt/2, -dt
  float hA, hAbr, hAce, hAcb;  // h times the field factors of FastPulse
  float kA, kAce;              // k times them
  float gz_s;                  // grid units along z: Z gz_s + gz_o
  FF gz_o;
};

__host__ __device__ inline FF d_split(double v) {
  FF r;
  r.hi = (float)v;
  r.lo = (float)d_add(v, -(double)r.hi);
  return r;
}

__host__ __device__ inline StepBase make_step_base(const PulseHead<float> &P, double t0, double dt, const GridView &g) {
  const FastPulse &F = P.fast;
  const double inv2pi = 0.15915494309189535;
  StepBase s;
  const double T = d_add(t0, -P.t_f);
  double c0 = d_add(d_mul(d_add(d_mul(P.omega, T), P.phase0), inv2pi), F.turn0);
  c0 = d_add(c0, -rint(c0));
  double d = d_mul(d_mul(P.omega, dt), inv2pi);
  d = d_add(d, -rint(d));
  s.om0 = d_split(c0);
  s.del = d_split(d);
  const double ts = P.kind == AP_FLYING_SUM ? d_mul(P.omega, inv2pi) : 1.0;
  s.T0 = d_split(d_mul(T, ts));
  s.DT = d_split(d_mul(dt, ts));
  s.cxy = (float)d_mul(dt, (double)P.adv_xy);
  s.cz = (float)d_mul(dt, F.z_scale);
  s.h = (float)d_mul(dt, -0.5);
  s.hA = (float)d_mul((double)s.h, (double)F.A);
  s.hAbr = (float)d_mul((double)s.h, (double)F.Abr);
  s.hAce = (float)d_mul((double)s.h, (double)F.Ace);
  s.hAcb = (float)d_mul((double)s.h, (double)F.Acb);
  s.k = 2.0f * s.h;
  s.kA = 2.0f * s.hA;
  s.kAce = 2.0f * s.hAce;
  // the offset that belongs to the rounded factor: right in the grid's middle, so
  // within 2^-25 of its half-length at its ends, wherever the focus is
  const double gs = d_mul(g.inv_d_d[2], F.z_len), mid = d_mul(0.5, (double)(g.nz - 1));
  s.gz_s = (float)gs;
  const double o = d_add(d_mul(P.z_f, g.inv_d_d[2]), g.off_d[2]);
  s.gz_o = d_split(gs != 0.0 ? d_add(mid, -d_mul(d_add(mid, -o), d_div((double)s.gz_s, gs))) : 0.0);
  return s;
}

// The grid unit of Z = hi + lo.  Z is measured from the focus, so Z s and the
// offset o cancel when the focus lies away from the grid: their high parts meet
// in one fused operation, exact up to the rounding of the (small) result, and
// the low parts join as one correction.  The error is then that of the unit
// itself (2^-24 of it), wherever the focus is; with the high parts alone it
// grows with the distance (workload 2's grid: 1.5e-5 of a cell with the focus at
// 0, 3e-3 at 1e4 wavelengths).
template <typename R>
__device__ __forceinline__ R grid_unit_z(R zhi, R zlo, R s, R o_hi, R o_lo) {
  return radd(rfma(zhi, s, o_hi), rfma(zlo, s, o_lo));
}

// The step table's entry for step n (an integer below 2^23, in float):
// {C_n in turns, |C_n| <= 1/2; T_n scaled for the envelope, for the moving
// focus, and itself}; for the flying-focus sum {-, -, T_n in turns as hi, lo}.
template <int KIND>
__device__ __forceinline__ float4 step_entry(const FastPulse &F, const StepBase &s, float nf) {
  const FF nt = two_prod(nf, s.DT.hi);
  FF T = two_sum(s.T0.hi, nt.hi);
  T.lo = __fadd_rn(T.lo, __fadd_rn(nt.lo, __fmaf_rn(nf, s.DT.lo, s.T0.lo)));
  if constexpr (KIND == AP_FLYING_SUM) {
    return make_float4(0.0f, 0.0f, T.hi, T.lo);
  } else {
    const FF nd = two_prod(nf, s.del.hi);
    const FF c = two_sum(s.om0.hi, nd.hi);
    const float clo = __fadd_rn(__fadd_rn(c.lo, nd.lo), __fmaf_rn(nf, s.del.lo, s.om0.lo));
    const float C = __fadd_rn(__fsub_rn(c.hi, round_magic(c.hi)), clo);
    auto scaled = [&](float hi, float lo) {  // (hi + lo) T
      return __fmaf_rn(T.hi, hi, __fmaf_rn(T.hi, lo, __fmul_rn(T.lo, hi)));
    };
    return make_float4(C, scaled(F.s_env, F.s_env_lo), scaled(F.c_tz, F.c_tz_lo), __fadd_rn(T.hi, T.lo));
  }
}

// ------------------------------------------------------------- unit fields
// The fields of a unit-amplitude pulse: E_perp = p U, B_perp = (z x p) V, and
// the longitudinal parts up to their constants.  Linear: p = (1, 0), only the
// real parts are used; circular: p = (1, -i).
template <typename R>
struct UnitFields {
  R Ur, Ui, Vr, Vi, ez, bz;
};

constexpr int kLin = 0, kCirc = 1;
constexpr int kEnvGauss = 0, kEnvAny = 1;

// 2 pi times (y - Z) less its nearest integer, Z = hi + lo in turns: the
// integer m of the rounded difference is added to hi exactly (the sum is a
// multiple of hi's last place of magnitude at most |y| + 1/2), and only then
// does the low part join.
template <typename R>
__device__ __forceinline__ R phase_angle(R y, R zhi, R zlo) {
  const R m = round_magic(rsub(y, zhi));
  const R g = radd(radd(zhi, m), zlo);
  return rmul(rsub(y, g), R(kTwoPiHi));
}

// g: the envelope's share of the exponent of 2, negated; mul: its factor
template <int ENV, class PT, typename R>
__device__ __forceinline__ void envelope_fast(const PT &P, R eta, R &mul, R &g) {
  if constexpr (ENV == kEnvGauss) {
    g = rmul(eta, eta);
  } else {
    mul = R(1.0f);
    g = R(0.0f);
    switch (P.env) {
      case AP_ENV_SIN2: {
        const R c = cos_r(eta);
        mul = sin2_window(rmul(c, c), eta, P.fast.env_w);
        break;
      }
      case AP_ENV_GAUSS:
        g = rmul(eta, eta);
        break;
      case AP_ENV_SGAUSS: {
        const R s = rmul(eta, eta);
        R p = s;
        for (int i = 1; i < P.sg_order; ++i) p = rmul(p, s);
        g = rmul(R(P.env_b), p);
        break;
      }
      default:
        break;
    }
  }
}

template <typename R>
__device__ __forceinline__ Cx<R> rcmul(Cx<R> a, Cx<R> b, R nb_im) {
  return {rfma(a.re, b.re, rmul(a.im, nb_im)), rfma(a.re, b.im, rmul(a.im, b.re))};
}
template <typename R>
__device__ __forceinline__ Cx<R> rcmul(Cx<R> a, Cx<R> b) {
  return rcmul(a, b, rneg(b.im));
}

// 1 / (2 pi log2(e)): from r^2 log2(e) / w0^2 to turns
constexpr float kTurnsPerExp = 0.110317801f;

template <int KIND, int POL, int ENV, class PT, typename R>
__device__ __forceinline__ UnitFields<R> unit_fields_beam(const PT &P, const float4 st, R x, R y, R zhi, R zlo) {
  const FastPulse &F = P.fast;
  UnitFields<R> o;
  R eta = rfma(zhi, R(F.c_eta), R(st.y));
  if constexpr (ENV != kEnvGauss) eta = rfma(zhi, R(F.c_eta_lo), eta);
  R mul, g;
  envelope_fast<ENV>(P, eta, mul, g);
  if constexpr (KIND == AP_PLANE) {
    R s, c;
    sincos_r(phase_angle(R(st.x), zhi, zlo), &s, &c);
    R mag = exp2_neg(g);
    if constexpr (ENV == kEnvAny) mag = rmul(mag, mul);
    o.Ur = rmul(mag, c);
    o.Ui = rmul(mag, s);
    o.Vr = o.Ur;
    o.Vi = o.Ui;
    if (P.plasma) {
      // B from the finite-duration terms (envelope_logd and finite_duration, in
      // operations of one rounding)
      const R e = rmul(eta, R(F.env_len));  // back to the envelope's own argument
      R L1 = R(0.0f), L2 = R(0.0f);
      if (P.env == AP_ENV_GAUSS) {
        L1 = rmul(R(-P.lg_c1), e);
        L2 = rfma(L1, L1, R(-P.lg_c2));
      } else if (P.env == AP_ENV_SGAUSS) {
        const R u = sg_bound(rmul(e, R(P.env_a)), P.sg_max), s2 = rmul(u, u);
        R q = R(1.0f);
        for (int i = 1; i < P.sg_order; ++i) q = rmul(q, s2);
        L1 = rmul(rmul(R(-P.lg_c1), u), q);
        L2 = rfma(L1, L1, rmul(R(-P.lg_c2), q));
      }
      const R th = rmul(rmul(R(P.fdc), L1), R(P.inv_w));
      const R A = rfma(rmul(R(0.5f), th), th, rfma(rmul(rmul(R(-P.fdc), L2), R(P.inv_w)), R(P.inv_w), R(1.0f)));
      R sn_t, cs_t;
      sincos_r(th, &sn_t, &cs_t);
      o.Vr = rmul(A, rfma(o.Ur, cs_t, rmul(rneg(o.Ui), sn_t)));
      o.Vi = rmul(A, rfma(o.Ur, sn_t, rmul(o.Ui, cs_t)));
    }
    o.ez = R(0.0f);
    o.bz = R(0.0f);
    return o;
  } else {
    // q = 1 / (1 - i zeta) = inv (1 + i zeta); zn = -zeta
    const R zn = KIND == AP_FLYING_CF ? rfma(zhi, R(F.c_zn), R(st.z)) : rmul(zhi, R(F.c_zn));
    const R inv = rcp_r(rfma(zn, zn, R(1.0f)));
    const R nq = rmul(zn, inv), qi = rneg(nq);
    const R b = rmul(rfma(x, x, rmul(y, y)), R(F.c_a));  // r^2 log2(e) / w0^2
    const R ang = phase_angle(rfma(b, rmul(nq, R(kTurnsPerExp)), R(st.x)), zhi, zlo);
    R sn, cs;
    sincos_r(ang, &sn, &cs);
    if constexpr (KIND != AP_LG) {
      R mag = exp2_neg(rfma(b, inv, g));
      if constexpr (ENV == kEnvAny) mag = rmul(mag, mul);
      const R mc = rmul(mag, cs), ms = rmul(mag, sn);
      // U = q m e^{i ang}, W = q U
      o.Ur = rfma(inv, mc, rmul(nq, ms));
      o.Ui = rfma(inv, ms, rmul(qi, mc));
      const R Wi = rfma(inv, o.Ui, rmul(qi, o.Ur));
      if constexpr (POL == kLin) {
        o.ez = rmul(x, Wi);
        o.bz = rmul(y, Wi);
      } else {
        const R Wr = rfma(inv, o.Ur, rmul(nq, o.Ui));
        o.ez = rfma(x, Wi, rmul(rneg(y), Wr));
        o.bz = rfma(x, Wr, rmul(y, Wi));
      }
    } else {
      // u = (x + i sgn y)^l L_p^l(s) q^{l+1} (q/q*)^p e^{-r^2 q / w0^2}, l = |l|,
      // s = 2 r^2 |q|^2 / w0^2, (sqrt2 / w0)^l inside the amplitude factor
      const R bi = rmul(b, inv);
      R mag = exp2_neg(rfma(b, inv, g));
      if constexpr (ENV == kEnvAny) mag = rmul(mag, mul);
      const R s = rmul(bi, R(1.38629436f));  // 2 / log2(e)
      const Cx<R> q{inv, qi};
      // L_p^l and dL/ds = -L_{p-1}^{l+1} by the three-term recurrence (row 3 r
      // + 1 and 3 r + 2 of lg_n hold the negated coefficients), (q/q*)^p and
      // q^{l+1}; the loops start at their first iteration that multiplies
      R Lp = R(1.0f), nD = R(0.0f);  // nD = -dL/ds
      Cx<R> K = q;
      for (int i = 0; i < P.lg_al; ++i) K = rcmul(K, q, nq);
      if (P.lg_p > 0) {
        const Cx<R> gg{rfma(R(2.0f), inv, R(-1.0f)), radd(qi, qi)};
        const R ngi = rmul(R(2.0f), nq);
        K = rcmul(K, gg, ngi);
        Lp = rfma(R(F.lg_n[1][0]), s, R(F.lg_n[0][0]));
        nD = R(1.0f);
        R Lm = R(1.0f), Dm = R(0.0f);
        for (int k = 1; k < P.lg_p; ++k) {
          K = rcmul(K, gg, ngi);
          const R Dn = rfma(rfma(R(F.lg_n[4][k - 1]), s, R(F.lg_n[3][k - 1])), nD, rmul(R(F.lg_n[5][k - 1]), Dm));
          Dm = nD;
          nD = Dn;
          const R Ln = rfma(rfma(R(F.lg_n[1][k]), s, R(F.lg_n[0][k])), Lp, rmul(R(F.lg_n[2][k]), Lm));
          Lm = Lp;
          Lp = Ln;
        }
      }
      const Cx<R> base = rcmul(K, Cx<R>{rmul(mag, cs), rmul(mag, sn)});
      // Tb = base xi^{l-1} (l > 0) and Bp = base xi^l
      Cx<R> Tb = base, Bp = base;
      if (P.lg_al > 0) {
        const Cx<R> xi{x, rmul(R(F.lg_sg), y)};
        const R nxi = rneg(xi.im);
        for (int i = 1; i < P.lg_al; ++i) Tb = rcmul(Tb, xi, nxi);
        Bp = rcmul(Tb, xi, nxi);
      }
      o.Ur = rmul(Bp.re, Lp);
      o.Ui = rmul(Bp.im, Lp);
      // dU/dx = T + x V, dU/dy = i sgn T + y V with T = l L base xi^{l-1} and
      // V = base xi^l D, D = (4 |q|^2 dL/ds - 2 L q) / w0^2
      const R m2L = rmul(R(F.lg_m2w), Lp);
      const Cx<R> D{rmul(inv, rfma(R(F.lg_m4w), nD, m2L)), rmul(m2L, qi)};
      const Cx<R> V = rcmul(Bp, D);
      const R aL = rmul(R(P.lg_alf), Lp);
      if constexpr (POL == kLin) {
        o.ez = rfma(aL, Tb.im, rmul(x, V.im));
        o.bz = rfma(rmul(R(F.lg_sg), aL), Tb.re, rmul(y, V.im));
      } else {
        // DE = dU/dx - i dU/dy = (1 + sgn) T + (x - i y) V and DB = i DE
        const R a2 = rmul(R(F.lg_sp), aL);  // (1 + sgn) l L
        o.ez = rfma(a2, Tb.im, rfma(x, V.im, rmul(rneg(y), V.re)));
        o.bz = rfma(a2, Tb.re, rfma(x, V.re, rmul(y, V.im)));
      }
    }
    o.Vr = o.Ur;
    o.Vi = o.Ui;
    return o;
  }
}

// One component's constants {-2 pi / (k z_R,j), zoff_j, theta_j, 1/k_j}, theta_j
// as a 32-bit fraction of a turn; for two particles each twice (operand
// pairs, no per-step broadcast).
template <typename R>
struct CompConst {
  R cz, zoff, ik;
  unsigned th;
};
__device__ __forceinline__ CompConst<float> comp_const(const float4 *t, int j, float) {
  const float4 v = t[j];
  return {v.x, v.y, v.w, __float_as_uint(v.z)};
}
__device__ __forceinline__ CompConst<F2> comp_const(const float4 *t, int j, F2) {
  const float4 a = t[2 * j], b = t[2 * j + 1];
  return {F2(a.x, a.y), F2(a.z, a.w), F2(b.x, b.y), __float_as_uint(b.z)};
}
template <typename R>
__device__ __forceinline__ void comp_table(const Pulse<float> &P, float4 *t) {
  for (int j = threadIdx.x; j < P.n_comp; j += blockDim.x) {
    const float4 v = P.fcomp[j];
    if constexpr (IsPair<R>::value) {
      t[2 * j] = make_float4(v.x, v.x, v.y, v.y);
      t[2 * j + 1] = make_float4(v.w, v.w, v.z, 0.0f);
    } else {
      t[j] = v;
    }
  }
}

// Phases as 32-bit fractions of a turn (sums wrap modulo one turn by
// themselves, on the integer pipe).  A fraction becomes the float 1 + frac by
// one funnel shift of its upper 23 bits under the exponent of one.
__device__ __forceinline__ unsigned turn_bits(float hi, float lo) {
  return (unsigned)__float2int_rn(__fmul_rn(hi, 4294967296.0f)) + (unsigned)__float2int_rn(__fmul_rn(lo, 4294967296.0f));
}
__device__ __forceinline__ float turn_float(unsigned q) { return __uint_as_float(__funnelshift_r(q, 0x7fu, 9)); }
template <typename R>
struct Turn {
  unsigned a;
  __device__ __forceinline__ Turn(R hi, R lo) : a(turn_bits(hi, lo)) {}
  __device__ __forceinline__ void operator+=(const Turn &o) { a += o.a; }
  __device__ __forceinline__ R plus(unsigned th) const { return turn_float(a + th); }
};
template <>
struct Turn<F2> {
  unsigned a, b;
  __device__ __forceinline__ Turn(F2 hi, F2 lo) : a(turn_bits(hi.x, lo.x)), b(turn_bits(hi.y, lo.y)) {}
  __device__ __forceinline__ void operator+=(const Turn &o) {
    a += o.a;
    b += o.b;
  }
  __device__ __forceinline__ F2 plus(unsigned th) const { return F2(turn_float(a + th), turn_float(b + th)); }
};

// Flying focus (sum of Gaussian components).  The phase of component j is
// r_0 phi + j r_d phi + theta_j turns, phi = T - Z in turns of omega, r_0 =
// w_first / omega, r_d = dw / omega: reduced in float-float once per step,
// then stepped from component to component as 32-bit fractions of a turn, so
// each component gets its own sine and cosine.  That replaces the complex
// rotation of the phase factor and the product with the component's constant
// (35 -> 19.5 FP32 operations per component), and its error: the rotation
// multiplied the rounding of its step by up to n_comp.  Two components share
// one reciprocal, 1/(d1 d2): 3.5 special-function operations per component.
// d stays below 2^60 because Z is clamped where the largest |zeta| reaches 1e9 (the
// others follow within the bandwidth's factor; the field there is 1e-9 of the
// focus).
template <int POL, typename R>
__device__ __forceinline__ UnitFields<R> unit_fields_flying(const Pulse<float> &P, const float4 *comps, const float4 st,
                                                            R x, R y, R zhi, R zlo) {
  const FastPulse &F = P.fast;
  const auto ph = two_diff(R(st.z), zhi);
  const R plo = radd(ph.lo, rsub(R(st.w), zlo));
  auto turns = [&](float rh, float rl) {  // r phi less its nearest integer
    const R p = rmul(R(rh), ph.hi);
    const R ne = rfma(ph.hi, R(-rh), p);  // minus the product's rounding error
    const R lo = rsub(rfma(R(rh), plo, rmul(R(rl), ph.hi)), ne);
    return Turn<R>(rsub(p, round_magic(p)), lo);
  };
  Turn<R> turn = turns(F.r0_hi, F.r0_lo);
  const Turn<R> step = turns(F.rd_hi, F.rd_lo);
  const R b = rmul(rfma(x, x, rmul(y, y)), R(F.c_a));
  const R a = rmul(b, R(0.693147181f));  // r^2 / w0^2
  const R zc = clamp_abs(zhi, F.z_max);
  R S0r = R(0.0f), S0i = R(0.0f), S1r = R(0.0f), S1i = R(0.0f);
  auto add = [&](const CompConst<R> &c, R zn, R inv) {
    const R nq = rmul(zn, inv), qi = rneg(nq);
    const R mag = exp2_neg(rmul(b, inv));
    const R ang = rfma(radd(turn.plus(c.th), R(-1.5f)), R(kTwoPiHi), rmul(a, nq));
    turn += step;
    R sn, cs;
    sincos_r(ang, &sn, &cs);
    const R mc = rmul(mag, cs), ms = rmul(mag, sn);
    const R Ur = rfma(inv, mc, rmul(nq, ms));
    const R Ui = rfma(inv, ms, rmul(qi, mc));
    S0r = radd(S0r, Ur);
    S1i = rfma(c.ik, rfma(inv, Ui, rmul(qi, Ur)), S1i);
    if constexpr (POL == kCirc) {
      S0i = radd(S0i, Ui);
      S1r = rfma(c.ik, rfma(inv, Ur, rmul(nq, Ui)), S1r);
    }
  };
  const int nc = P.n_comp;
  auto two = [&](int j) {
    const CompConst<R> c0 = comp_const(comps, j, R(0.0f)), c1 = comp_const(comps, j + 1, R(0.0f));
    const R z0 = rfma(zc, c0.cz, c0.zoff), z1 = rfma(zc, c1.cz, c1.zoff);
    const R d0 = rfma(z0, z0, R(1.0f)), d1 = rfma(z1, z1, R(1.0f));
    const R r = rcp_r(rmul(d0, d1));
    add(c0, z0, rmul(r, d1));
    add(c1, z1, rmul(r, d0));
  };
  int j = 0;
#pragma unroll 2
  for (; j + 1 < nc; j += 2) two(j);
  if (j < nc) {
    const CompConst<R> c0 = comp_const(comps, j, R(0.0f));
    const R z0 = rfma(zc, c0.cz, c0.zoff);
    add(c0, z0, rcp_r(rfma(z0, z0, R(1.0f))));
  }
  UnitFields<R> o;
  o.Ur = S0r;
  o.Ui = S0i;
  o.Vr = S0r;
  o.Vi = S0i;
  if constexpr (POL == kLin) {
    o.ez = rmul(x, S1i);
    o.bz = rmul(y, S1i);
  } else {
    o.ez = rfma(x, S1i, rmul(rneg(y), S1r));
    o.bz = rfma(x, S1r, rmul(y, S1i));
  }
  return o;
}

template <int KIND, int POL, int ENV, class PT, typename R>
__device__ __forceinline__ UnitFields<R> unit_fields(const PT &P, const float4 *comps, const float4 st, R x, R y, R zhi,
                                                     R zlo) {
  if constexpr (KIND == AP_FLYING_SUM) return unit_fields_flying<POL>(P, comps, st, x, y, zhi, zlo);
  else return unit_fields_beam<KIND, POL, ENV>(P, st, x, y, zhi, zlo);
}

// -------------------------------------------------------------- Boris step
template <typename R>
__device__ __forceinline__ R inv_gamma(const R u[3]) {
  return rsqrt_r(rfma(u[0], u[0], rfma(u[1], u[1], rfma(u[2], u[2], R(1.0f)))));
}

// The Boris step, u' = u + (k E + p x s) with um = u + (k/2) E, p = um + um x t
// and s = 2 t / (1 + t^2): the kick and the rotation are summed first and
// join the momentum with one rounding (the textbook order um, um + p x s, + kick
// rounds at the momentum's magnitude three times, which for a relativistic
// electron is most of the step's error).  Each cross product is written out
// for the components that can differ from zero.

// the analytic field alone, from its unit fields and the kick's constants
// (LON: the kind has longitudinal fields); returns 1/gamma of the new momentum
template <int POL, bool LON, typename R, class S>
__device__ __forceinline__ R boris_unit(R u[3], const UnitFields<R> &f, const S &s) {
  R um[3] = {rfma(R(s.hA), f.Ur, u[0]), u[1], u[2]};
  if constexpr (POL == kCirc) um[1] = rfma(R(s.hA), f.Ui, u[1]);
  if constexpr (LON) um[2] = rfma(R(s.hAce), f.ez, u[2]);
  const R ig = inv_gamma(um);
  // t = (h/gamma) B, nt = -t
  const R hb = rmul(R(s.hAbr), ig);
  const R t1 = rmul(hb, f.Vr), nt1 = rneg(t1);
  R t0 = R(0.0f), nt0 = t0, t2 = t0, nt2 = t0;
  R tt = rfma(t1, t1, R(1.0f));
  R p0 = rfma(um[2], nt1, um[0]), p1 = um[1], p2 = rfma(um[0], t1, um[2]);
  if constexpr (LON) {
    t2 = rmul(rmul(R(s.hAcb), ig), f.bz);
    nt2 = rneg(t2);
    tt = rfma(t2, t2, tt);
    p0 = rfma(um[1], t2, p0);
    p1 = rfma(um[0], nt2, p1);
  }
  if constexpr (POL == kCirc) {
    nt0 = rmul(hb, f.Vi);
    t0 = rneg(nt0);
    tt = rfma(t0, t0, tt);
    p1 = rfma(um[2], t0, p1);
    p2 = rfma(um[1], nt0, p2);
  }
  const R i = rcp_r(tt);
  const R sc = radd(i, i);
  const R s1 = rmul(sc, t1);
  R d0 = rfma(p2, rneg(s1), rmul(R(s.kA), f.Ur));  // -p2 s1 + kick
  // a product that is added to nothing but the momentum joins it fused
  R d2 = POL == kLin && !LON ? R(0.0f) : rmul(p0, s1);
  if constexpr (LON) {
    const R s2 = rmul(sc, t2);
    d0 = rfma(p1, s2, d0);
    d2 = rfma(R(s.kAce), f.ez, d2);
    if constexpr (POL == kCirc) u[1] = radd(u[1], rfma(p0, rneg(s2), rfma(p2, rmul(sc, t0), rmul(R(s.kA), f.Ui))));
    else u[1] = rfma(p0, rneg(s2), u[1]);
  } else if constexpr (POL == kCirc) {
    u[1] = radd(u[1], rfma(p2, rmul(sc, t0), rmul(R(s.kA), f.Ui)));
  }
  if constexpr (POL == kCirc) d2 = rfma(p1, rmul(sc, nt0), d2);
  u[0] = radd(u[0], d0);
  u[2] = POL == kLin && !LON ? rfma(p0, s1, u[2]) : radd(u[2], d2);
  return inv_gamma(u);
}

// any E, B (the analytic field plus the grid's)
template <typename R>
__device__ __forceinline__ R boris_full(R u[3], const R E[3], const R B[3], float hs, float ks) {
  const R h = R(hs), k = R(ks);
  const R um[3] = {rfma(h, E[0], u[0]), rfma(h, E[1], u[1]), rfma(h, E[2], u[2])};
  const R hg = rmul(h, inv_gamma(um));
  const R t[3] = {rmul(hg, B[0]), rmul(hg, B[1]), rmul(hg, B[2])};
  const R nt[3] = {rneg(t[0]), rneg(t[1]), rneg(t[2])};
  const R i = rcp_r(rfma(t[0], t[0], rfma(t[1], t[1], rfma(t[2], t[2], R(1.0f)))));
  const R sc = radd(i, i);
  const R p[3] = {rfma(um[1], t[2], rfma(um[2], nt[1], um[0])), rfma(um[2], t[0], rfma(um[0], nt[2], um[1])),
                  rfma(um[0], t[1], rfma(um[1], nt[0], um[2]))};
  const R sv[3] = {rmul(sc, t[0]), rmul(sc, t[1]), rmul(sc, t[2])};
  const R ns[3] = {rneg(sv[0]), rneg(sv[1]), rneg(sv[2])};
  const R d0 = rfma(p[1], sv[2], rfma(p[2], ns[1], rmul(k, E[0])));
  const R d1 = rfma(p[2], sv[0], rfma(p[0], ns[2], rmul(k, E[1])));
  const R d2 = rfma(p[0], sv[1], rfma(p[1], ns[0], rmul(k, E[2])));
  u[0] = radd(u[0], d0);
  u[1] = radd(u[1], d1);
  u[2] = radd(u[2], d2);
  return inv_gamma(u);
}

// Compensated position update p += u k: the product joins the low part in one
// fused operation, and the sum's own rounding error becomes the new low part
// (exact whenever |hi| >= |increment|, the normal case), so hi is the rounded
// value of hi + lo.
template <typename R, typename FFR>
__device__ __forceinline__ void advance(FFR &p, R u, R k) {
  const R d = rfma(u, k, p.lo);
  const R t = radd(p.hi, d);
  p.lo = rsub(d, rsub(t, p.hi));
  p.hi = t;
}

}  // namespace apt
