// ap_line.cu -- 1-D lines with a linear cold-plasma current (Sec. 4, the
// analytic pulse technique with an analytic current J1).
//
// Two updates of one line carrying E_x on the whole nodes z_k, B_y on the
// half nodes and the current J_x on the whole nodes at half time levels:
//   traditional: the Yee scheme of Sec. 2.1 with the current advanced by the
//     leapfrog dJ/dt = omega_p^2 E (the simulation Sec. 4 compares with);
//   split (APT): E, B hold the internally advanced E2, B2; the physical
//     current J is driven by E1 + E2, and E2 is sourced by J - J1, with the
//     analytic E1 (at t_n) and J1 (at t_n + dt/2) of a plane-wave pulse
//     evaluated in the kernel every step (Eqs. E_1_j, E_2_j, j1).
//
// One block per line; the line (E, B, J and a_k = dt omega_p^2(z_k)) stays
// on chip for all n_steps and is written back once: in registers for float
// lines of up to 8192 nodes (plasma_line_pair_kernel in ap_yee.cu, split_line_kernel), in
// shared memory otherwise (line_kernel).  Per step of line_kernel: the
// B half step; a barrier; the current and E update of each node (one pass:
// both read only the node's own E and J and the neighbouring B); a barrier;
// the second B half step.  The second B half step and the next step's first
// one write only their own node and read only E, so no barrier separates
// them.  Each product, sum and difference is rounded separately in the
// stated order, so the double traditional line reproduces a plain double
// loop of the same expressions bit for bit.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>

#include "ap_kernels.cuh"
#include "ap_lines.cuh"

namespace apt {
namespace {

constexpr int kLineBlock = 1024;

__device__ __forceinline__ double l_sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double l_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double l_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float l_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float l_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float l_mul(float a, float b) { return __fmul_rn(a, b); }

// Local coordinates of node k (x = y = 0) at one time level (double).
__device__ __forceinline__ Local<double> node_local(const Pulse<double> &P, const LineArgs &a, double st, int k) {
  Pos<AP_FP64> pos;
  pos.load(0.0, 0.0, __dadd_rn(a.z0, __dmul_rn((double)k, a.dz)));
  return local_coords<AP_FP64>(P, st, pos);
}

// The line in shared memory: double lines, split (APT) or traditional, and
// traditional float lines of more than 8192 nodes.
template <typename T, bool APT>
__global__ void __launch_bounds__(kLineBlock) line_kernel(const __grid_constant__ Pulse<double> P,
                                                          const __grid_constant__ LineArgs a) {
  static_assert(!APT || sizeof(T) == 8, "the float split line runs in registers");
  extern __shared__ __align__(16) unsigned char line_smem[];
  const int nz = a.nz;
  T *e = reinterpret_cast<T *>(line_smem);
  T *b = e + nz;
  T *j = b + nz;
  T *q = j + nz;  // a_k = dt omega_p^2(z_k)
  const size_t off = (size_t)blockIdx.x * (size_t)nz;
  T *Eg = static_cast<T *>(a.E) + off;
  T *Bg = static_cast<T *>(a.B) + off;
  T *Jg = static_cast<T *>(a.J) + off;
  const T *W = a.wp2 ? static_cast<const T *>(a.wp2) + off : nullptr;
  const T dt = (T)a.dt;
  const T r = (T)(a.dt / a.dz);
  const T hr = (T)(0.5 * (a.dt / a.dz));
  const T wpu = (T)a.omega_p2;
  const int t = threadIdx.x, bd = blockDim.x;
  for (int k = t; k < nz; k += bd) {
    e[k] = Eg[k];
    b[k] = Bg[k];
    j[k] = Jg[k];
    q[k] = l_mul(dt, W ? W[k] : wpu);
  }
  TimeBase<AP_FP64> tb;
  if constexpr (APT) tb.init(P, a.t0, 0.5 * a.dt);  // level 2n: t_n, 2n + 1: t_n + dt/2
  __syncthreads();
  for (long long n = 0; n < a.n_steps; ++n) {
    // B^{n+1/2} = B^n - (r/2)(E_{k+1}^n - E_k^n)
    for (int k = t; k < nz - 1; k += bd) b[k] = l_sub(b[k], l_mul(hr, l_sub(e[k + 1], e[k])));
    __syncthreads();
    double st_e = 0.0, st_j = 0.0;
    if constexpr (APT) {
      st_e = tb.at(2 * n);
      st_j = tb.at(2 * n + 1);
    }
    // J^{n+1/2} = J^{n-1/2} + a_k (E1 + E2)^n;  E^{n+1} = (E^n - r dB) - dt (J - J1)^{n+1/2}
    for (int k = t; k < nz; k += bd) {
      const T ek = e[k];
      T drive = ek;
      if constexpr (APT) {
        double E1[3], B1[3];
        analytic_fields<AP_PLANE, AP_FP64>(P, node_local(P, a, st_e, k), E1, B1);
        drive = l_add(E1[0], ek);
      }
      const T jk = l_add(j[k], l_mul(q[k], drive));
      j[k] = jk;
      if (k >= 1) {
        T src = jk;
        if constexpr (APT) {
          double J1[3];
          current_plane(P, node_local(P, a, st_j, k), J1);
          src = l_sub(jk, J1[0]);
        }
        e[k] = l_sub(l_sub(ek, l_mul(r, l_sub(b[k], b[k - 1]))), l_mul(dt, src));
      }
    }
    __syncthreads();
    // B^{n+1} = B^{n+1/2} - (r/2)(E_{k+1}^{n+1} - E_k^{n+1})
    for (int k = t; k < nz - 1; k += bd) b[k] = l_sub(b[k], l_mul(hr, l_sub(e[k + 1], e[k])));
  }
  // every node is written back by the thread that last wrote it
  for (int k = t; k < nz; k += bd) {
    Eg[k] = e[k];
    Bg[k] = b[k];
    Jg[k] = j[k];
  }
}

// ------------------------------------------------------------- split line
// Constants of the split float line, made on the host: the pulse along the
// line in turns and in the envelope's own scale.
struct SplitArgs {
  LineArgs line;
  StepBase base;            // carrier phase and time of step n (make_step_base)
  FastPulse fast;           // s_env (here of the scaled argument below), turn0
  int env, g;               // envelope kind; order of the super-Gaussian (Gaussian: 1)
  float zs_hi, zs_lo;       // k / 2 pi
  float zf_hi, zf_lo;
  float su_vg, su_vg_lo;    // scale of the envelope argument over v_g
  float hu;                 // dt/2 in the scaled argument
  bool finite;              // th and A stay finite over all nodes and steps of the call
  float s_max;              // square of the scaled argument from which the super-Gaussian is zero
  float env_w;              // half-width of the sin^2 window, scaled
  float amp, jamp;          // a0, and the amplitude of J1
  float delta;              // omega dt/2
  float k1, k2;             // th = k1 u q, A = 1 - th^2/2 + k2 q
};

// Envelope form of a split-line kernel: the order g of the super-Gaussian where
// it is compiled in (1: Gaussian and continuous wave), any order, or the sin^2
// window.  The envelope is 2^-(u^{2g}) of the scaled argument u.
constexpr int kOrderAny = 0, kSin2 = -1;

// s^n by squaring; N = 0: 0 <= n <= 15 at run time (the bits of n are the same
// for all threads), N > 0: n = N
template <int N>
__device__ __forceinline__ F2 upow(F2 s, int n) {
  if constexpr (N == 0) {
    F2 q = n & 1 ? s : F2(1.0f);
    s = rmul(s, s);
    if (n & 2) q = rmul(q, s);
    s = rmul(s, s);
    if (n & 4) q = rmul(q, s);
    if (n & 8) q = rmul(q, rmul(s, s));
    return q;
  } else if constexpr (N == 1) {
    return s;
  } else if constexpr (N % 2 == 0) {
    return upow<N / 2>(rmul(s, s), 0);
  } else {
    return rmul(upow<N - 1>(s, 0), s);
  }
}
__device__ __forceinline__ F2 window2(F2 u, float w) {
  const F2 c = cos_r(u);
  return sin2_window(rmul(c, c), u, w);
}

// The split line of Sec. 4 in registers: E2, B2 and J of two runs of C nodes
// per thread (ap_lines.cuh), each node's phase and envelope constants and a_k in
// shared memory.  Per step and node the analytic E1 at t_n and J1 at t_n + dt/2:
//   E1 = a0 G(eta) cos(psi),
//   J1 = J0 G(eta') A sin(psi + omega dt/2 + th),  th = L1/omega,
// where psi + omega dt/2 is J1's carrier and th the finite-duration phase
// (Eq. j1), so one sine takes the place of a rotation, a sine, a cosine and a
// complex product: four special-function operations per node instead of six.
// The carrier phase is kept in turns, a node's share reduced once per launch.
// The two B half steps that meet between E updates are one whole step.  34
// packed operations per pair of nodes against about 75 (149 instructions per
// node-step with the line in shared memory).
// 304 lines of 4096 nodes, 500 steps: 3.10 -> 0.83 ms.
template <int C, int MAXT, int G>
__global__ void __launch_bounds__(MAXT) split_line_kernel(const __grid_constant__ SplitArgs sa) {
  __shared__ float s_b[2 * MAXT + 1], s_e[2 * MAXT + 1];
  extern __shared__ __align__(16) unsigned char s_split[];
  F2 *s_turn = reinterpret_cast<F2 *>(s_split);  // [C][block] each
  const LineArgs &a = sa.line;
  const int nz = a.nz, t = threadIdx.x, bd = blockDim.x, H = C * bd;
  F2 *s_eta = s_turn + C * bd, *s_q = s_eta + C * bd;
  const size_t off = (size_t)blockIdx.x * (size_t)nz;
  float *Eg = static_cast<float *>(a.E) + off;
  float *Bg = static_cast<float *>(a.B) + off;
  float *Jg = static_cast<float *>(a.J) + off;
  const float *W = a.wp2 ? static_cast<const float *>(a.wp2) + off : nullptr;
  const float dtf = (float)a.dt, rf = (float)(a.dt / a.dz);
  const LineEdge eb{s_b}, ee{s_e};
  F2 e[C], b[C], j[C];
  line_load<C>(e, Eg, nz);
  line_load<C>(b, Bg, nz);
  line_load<C>(j, Jg, nz);
  LineEnds ends;
  ends.init<C>(nz, b);
  const float e0 = e[0].x;
#pragma unroll 1
  for (int i = 0; i < C; ++i) {
    F2 q, tn, en2;
    for (int h = 0; h < 2; ++h) {
      const int k = t * C + i + (h ? H : 0);
      // z_k - z_f and its turns, float-float
      const FF zk = node_coord_ff((float)k, a.z0_hi, a.z0_lo, a.dz_hi, a.dz_lo);
      FF dz = two_sum(zk.hi, -sa.zf_hi);
      dz.lo = __fadd_rn(dz.lo, __fsub_rn(zk.lo, sa.zf_lo));
      FF tr = two_prod(sa.zs_hi, dz.hi);
      tr.lo = __fadd_rn(tr.lo, __fmaf_rn(sa.zs_hi, dz.lo, __fmul_rn(sa.zs_lo, dz.hi)));
      const float turn = __fadd_rn(__fsub_rn(tr.hi, round_magic(tr.hi)), tr.lo);
      const float ek =
          __fmaf_rn(sa.su_vg, dz.hi, __fmaf_rn(sa.su_vg, dz.lo, __fmul_rn(sa.su_vg_lo, dz.hi)));
      const float qk = __fmul_rn(dtf, k < nz ? (W ? W[k] : (float)a.omega_p2) : 0.0f);
      if (h) { tn.y = turn; en2.y = ek; q.y = qk; } else { tn.x = turn; en2.x = ek; q.x = qk; }
    }
    s_turn[i * bd + t] = tn;
    s_eta[i * bd + t] = en2;
    s_q[i * bd + t] = q;
  }
  const F2 nr = F2(-rf), ndt = F2(-dtf);
  auto b_step = [&](F2 en, F2 nh) {
#pragma unroll
    for (int i = 0; i < C; ++i) b[i] = rfma(nh, rsub(i + 1 < C ? e[i + 1 < C ? i + 1 : i] : en, e[i]), b[i]);
    ends.restore<C>(b);
  };
  ee.put(e[0]);
  __syncthreads();
  b_step(ee.next(), F2(-0.5f * rf));
  float nf = 0.0f;  // the step in float (exact: fewer than 2^23 steps)
  for (long long n = 0; n < a.n_steps; ++n, nf += 1.0f) {
    eb.put(b[C - 1]);
    __syncthreads();
    const F2 bp = eb.prev();
    const float4 st = step_entry<AP_PLANE>(sa.fast, sa.base, nf);
    F2 bq = bp;  // B before node i
#pragma unroll
    for (int i = 0; i < C; ++i) {
      // psi = C - the node's turns, reduced
      F2 turn = rsub(F2(st.x), s_turn[i * bd + t]);
      turn = rsub(turn, round_magic(turn));
      const F2 u0 = rsub(F2(st.y), s_eta[i * bd + t]), u1 = radd(u0, F2(sa.hu));
      F2 m0, m1, th = F2(0.0f), A = F2(1.0f);
      if constexpr (G == kSin2) {
        m0 = window2(u0, sa.env_w);
        m1 = window2(u1, sa.env_w);
      } else {
        const F2 s0 = rmul(u0, u0);
        m0 = exp2_neg(G == kOrderAny ? rmul(upow<0>(s0, sa.g - 1), s0) : upow<G>(s0, 0));
        if constexpr (G == 1) {
          m1 = exp2_neg(rmul(u1, u1));
          th = rmul(F2(sa.k1), u1);
          A = rfma(rmul(F2(-0.5f), th), th, F2(1.0f + sa.k2));
        } else {
          F2 s = rmul(u1, u1);
          // held where the envelope is zero, as th and A would overflow (see
          // sg_bound; the compiled orders are for lines on which they do not)
          if constexpr (G == kOrderAny) s = F2(fminf(s.x, sa.s_max), fminf(s.y, sa.s_max));
          const F2 q = upow<(G > 1 ? G - 1 : 0)>(s, sa.g - 1);
          m1 = exp2_neg(rmul(q, s));
          th = rmul(F2(sa.k1), rmul(u1, q));
          A = rfma(F2(sa.k2), q, rfma(rmul(F2(-0.5f), th), th, F2(1.0f)));
        }
      }
      const F2 c0 = cos_r(rmul(turn, F2(kTwoPiHi)));
      const F2 aj = rfma(turn, F2(kTwoPiHi), radd(th, F2(sa.delta)));
      const F2 sj = F2(mufu_sin(aj.x), mufu_sin(aj.y));
      // J^{n+1/2} = J^{n-1/2} + a_k (E1 + E2)^n;  E^{n+1} = (E^n - r dB) - dt (J - J1)^{n+1/2}
      j[i] = rfma(s_q[i * bd + t], rfma(F2(sa.amp), rmul(m0, c0), e[i]), j[i]);
      const F2 src = rfma(rmul(F2(-sa.jamp), m1), rmul(A, sj), j[i]);
      e[i] = rfma(ndt, src, rfma(nr, rsub(b[i], bq), e[i]));
      bq = b[i];
    }
    if (t == 0) e[0].x = e0;
    ee.put(e[0]);
    __syncthreads();
    b_step(ee.next(), n + 1 < a.n_steps ? nr : F2(-0.5f * rf));
  }
  line_store<C>(e, Eg, nz);
  line_store<C>(b, Bg, nz);
  line_store<C>(j, Jg, nz);
}

template <int C, int MAXT, int G>
int launch_split_g(const SplitArgs &sa, void *stream) {
  auto kern = split_line_kernel<C, MAXT, G>;
  const int block = line_block<C>(sa.line.nz);
  const size_t smem = 3 * sizeof(F2) * (size_t)C * block;
  if (smem > 32 * 1024 && allow_smem(reinterpret_cast<const void *>(kern), 3 * sizeof(F2) * (size_t)C * MAXT) != AP_OK)
    return AP_ERR_CUDA;
  kern<<<(unsigned)sa.line.n_lines, block, smem, static_cast<cudaStream_t>(stream)>>>(sa);
  return cudaGetLastError() == cudaSuccess ? AP_OK : AP_ERR_CUDA;
}

template <int C, int MAXT>
int launch_split(const SplitArgs &sa, void *stream) {
  if (sa.env == AP_ENV_SIN2) return launch_split_g<C, MAXT, kSin2>(sa, stream);
  if (sa.g == 1) return launch_split_g<C, MAXT, 1>(sa, stream);
  // low orders (2 to 4) have their powers compiled in; above, and where the
  // powers need holding, the order is a run-time number (304 lines of 4096 nodes,
  // 500 steps: orders 2, 3, 4 777, 816, 820 us, 5 and 8 1014, 1027 us; with a loop
  // over the order 930, 1037, -, 1139, 1305)
  if (sa.finite && sa.g == 2) return launch_split_g<C, MAXT, 2>(sa, stream);
  if (sa.finite && sa.g == 3) return launch_split_g<C, MAXT, 3>(sa, stream);
  if (sa.finite && sa.g == 4) return launch_split_g<C, MAXT, 4>(sa, stream);
  return launch_split_g<C, MAXT, kOrderAny>(sa, stream);
}

SplitArgs split_args(const Pulse<double> &pd, const Pulse<float> &pf, const LineArgs &a) {
  SplitArgs s;
  auto split = [](double v, float &hi, float &lo) {
    hi = (float)v;
    lo = (float)(v - (double)hi);
  };
  s.line = a;
  s.fast = pf.fast;
  s.env = pd.env;
  // 2^-(u^{2g}) with u = su eta; the logarithmic derivatives are given in
  // eta (Gaussian) or eta/tau (super-Gaussian), ratio: that argument over u
  const double log2e = 1.4426950408889634;
  double su = 0.0, ratio = 0.0;
  s.g = 1;
  if (pd.env == AP_ENV_GAUSS) {
    su = std::sqrt(pd.env_a);
    ratio = 1.0 / su;
  } else if (pd.env == AP_ENV_SGAUSS) {
    s.g = pd.sg_order;
    const double sc = std::pow(log2e, 0.5 / s.g);  // env_a = 1/tau, env_b = log2e
    su = pd.env_a * sc;
    ratio = 1.0 / sc;
  } else if (pd.env == AP_ENV_SIN2) {
    su = pd.env_a;
  }
  // both scales in two floats: a step's and a node's terms are made once each
  split(su, s.fast.s_env, s.fast.s_env_lo);
  split(su * pd.inv_vg, s.su_vg, s.su_vg_lo);
  s.fast.c_tz = s.fast.c_tz_lo = 0.0f;
  GridView none;
  std::memset(&none, 0, sizeof(none));
  s.base = make_step_base(pf, a.t0, a.dt, none);
  split(pf.fast.z_scale, s.zs_hi, s.zs_lo);
  s.zf_hi = pf.zf_hi;
  s.zf_lo = pf.zf_lo;
  s.hu = (float)(0.5 * a.dt * su);
  s.s_max = (float)std::pow(158.0, 1.0 / s.g);  // 2^-158 is zero in float
  s.env_w = (float)(pd.env_a * pd.env_b);
  s.amp = (float)pd.amp;
  s.jamp = (float)(pd.jamp * pd.amp);
  s.delta = (float)(0.5 * pd.omega * a.dt);
  s.k1 = (float)(-pd.lg_c1 * pd.inv_w * std::pow(ratio, 2.0 * s.g - 1.0));
  s.k2 = (float)(pd.lg_c2 * pd.inv_w * pd.inv_w * std::pow(ratio, 2.0 * s.g - 2.0));
  if (pd.env != AP_ENV_GAUSS && pd.env != AP_ENV_SGAUSS) s.k1 = s.k2 = 0.0f;
  // largest |u| of the call: either end of the line at either end of the time
  const double T = std::max(std::fabs(a.t0 - pd.t_f), std::fabs(a.t0 + ((double)a.n_steps + 1.0) * a.dt - pd.t_f));
  const double Z = std::max(std::fabs(a.z0 - pd.z_f), std::fabs(a.z0 + (double)a.nz * a.dz - pd.z_f));
  const double u = std::max(1.0, su * (T + Z * pd.inv_vg)), q = std::pow(u, 2.0 * s.g - 2.0);
  s.finite = std::fabs(s.k1) * u * q < 1e18 && std::fabs(s.k2) * q < 1e36;  // A takes in th^2
  return s;
}

template <typename T, bool APT>
int launch_line_t(const Pulse<double> &P, const LineArgs &a, void *stream) {
  auto kern = line_kernel<T, APT>;
  const size_t smem = 4u * sizeof(T) * (size_t)a.nz;
  constexpr size_t most = 4u * sizeof(T) * (sizeof(T) == 8 ? AP_LINE1D_MAX_NODES_F64 : AP_LINE1D_MAX_NODES_F32);
  if (allow_smem(reinterpret_cast<const void *>(kern), most) != AP_OK) return AP_ERR_CUDA;
  int block = (a.nz + 31) / 32 * 32;
  if (block > kLineBlock) block = kLineBlock;
  kern<<<(unsigned)a.n_lines, block, smem, static_cast<cudaStream_t>(stream)>>>(P, a);
  return cudaGetLastError() == cudaSuccess ? AP_OK : AP_ERR_CUDA;
}

}  // namespace

int launch_line(bool apt_mode, int precision, const Pulse<double> &pd, const Pulse<float> &pf,
                const LineArgs &a, void *stream) {
  if (precision != AP_FP64) {
    // the line in registers, two runs of C nodes per thread
    if (apt_mode) {
      const SplitArgs s = split_args(pd, pf, a);
      // measured at 1 to 304 lines: shorter runs (more threads) while the
      // barriers weigh most, longer ones as the line grows (304 lines, 60
      // steps, C = 1/2/4/8: 700 nodes 68/65/73/75 us, 2000 nodes
      // 116/107/95/97, 4096 nodes -/-/148/150)
      if (a.nz <= 512) return launch_split<1, 256>(s, stream);
      if (a.nz <= 1536) return launch_split<2, 384>(s, stream);
      if (a.nz <= 4096) return launch_split<4, 512>(s, stream);
      return launch_split<8, 512>(s, stream);
    }
    if (a.nz <= kPlasmaPairNodes) return launch_plasma_float(a, stream);
    return launch_line_t<float, false>(pd, a, stream);
  }
  return apt_mode ? launch_line_t<double, true>(pd, a, stream) : launch_line_t<double, false>(pd, a, stream);
}

}  // namespace apt
