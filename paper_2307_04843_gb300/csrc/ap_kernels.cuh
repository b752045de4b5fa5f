// ap_kernels.cuh -- kernels of the gather + push (rows a2-a12 of the hot
// path) and their launchers, instantiated once per pulse kind by
// ap_push_<kind>.cu (AP_KIND_ID / AP_KIND_NAME set before inclusion).
#pragma once

#include <type_traits>

#include "ap_step.cuh"

namespace apt {

// Steps per chunk of the per-warp step table (float-float variant): one
// entry per lane.
constexpr int kStepChunk = 32;

// Dynamic shared memory of the push kernels, per block of T threads: the
// per-warp step tables (16 B per thread), then for the float grid kernels the
// cell-cache slots (16 slots x 16 B per thread).
__host__ __device__ constexpr size_t step_table_bytes(int threads) { return 16u * (size_t)threads; }
__host__ __device__ constexpr size_t grid_slot_bytes(int threads) { return 256u * (size_t)threads; }

// Grid modes of the push kernels: no grid, corner values (component arrays
// or the node-interleaved copy), per-cell coefficients (float kernels only).
constexpr int kGridNone = 0;
constexpr int kGridNodes = 1;
constexpr int kGridCells = 2;
constexpr int kGridCellsReg = 3;  // per-cell coefficients cached in registers
constexpr int kGridCellsMix = 4;  // two particles per thread: the first's cell in registers,
                                  // the second's in shared memory

// Grid cell cache of a variant: registers for double, shared memory for float.
template <int PREC, int GRID>
struct CacheOf {
  using type = GridCache<Real<PREC>>;
};
template <>
struct CacheOf<AP_FP32_PHASE64, kGridNodes> {
  using type = GridSlots;
};
template <>
struct CacheOf<AP_FP32_PHASEFF, kGridNodes> {
  using type = GridSlots;
};
template <>
struct CacheOf<AP_FP32_PHASE64, kGridCells> {
  using type = CellSlots;
};
template <>
struct CacheOf<AP_FP32_PHASEFF, kGridCells> {
  using type = CellSlots;
};
template <>
struct CacheOf<AP_FP32_PHASE64, kGridCellsReg> {
  using type = CellRegs;
};
template <>
struct CacheOf<AP_FP32_PHASEFF, kGridCellsReg> {
  using type = CellRegs;
};

// shared-memory bytes of the cell cache per block of T threads carrying NP
// particles each
template <int PREC, int GRID, int NP = 1>
__host__ __device__ constexpr size_t grid_cache_bytes(int threads) {
  return PREC == AP_FP64 || GRID == kGridNone || GRID == kGridCellsReg ? 0
         : GRID == kGridCells                                         ? 12u * kCellSlotStride * NP
         : GRID == kGridCellsMix                                      ? 12u * kCellSlotStride
                                                                      : grid_slot_bytes(threads);
}

// One particle through n_steps fused steps in double or with native double
// phase and position: load (a2), per step the local coordinates and phase
// (a3), envelope and profile (a4-a7), grid gather (a8), Boris and position
// (a9), light-front diagnostic (a10); then store (a11).  Every lane of a warp
// calls this together; `valid` is false for padding threads, which run the
// loop on a dummy particle so that warp operations see every lane.  Returns
// the final gamma (double) of a valid particle, 0 otherwise.
template <int KIND, int PREC, int GRID>
__device__ __forceinline__ double push_one(const Pulse<Real<PREC>> &P, const PushArgs &a, long long i, bool valid,
                                           void *slots) {
  static_assert(PREC != AP_FP32_PHASEFF, "push_ff");
  using R = Real<PREC>;
  double X = 0.0, Y = 0.0, Z = 0.0;
  R u[3] = {R(0), R(0), R(0)};
  if (valid) {
    X = a.x[i];
    Y = a.y[i];
    Z = a.z[i];
    const R *ux = static_cast<const R *>(a.ux);
    const R *uy = static_cast<const R *>(a.uy);
    const R *uz = static_cast<const R *>(a.uz);
    u[0] = ux[i];
    u[1] = uy[i];
    u[2] = uz[i];
  }
  Pos<PREC> pos;
  pos.load(X, Y, Z);
  TimeBase<PREC> tb;
  tb.init(P, a.t0, a.dt);
  const R dtR = (R)a.dt;
  const R dtxy = dtR * P.adv_xy;
  const R h0 = R(1) / rsqrt_r(fma(u[0], u[0], fma(u[1], u[1], fma(u[2], u[2], R(1))))) - u[2];
  typename CacheOf<PREC, GRID>::type gc;
  if constexpr (GRID && !std::is_same<R, double>::value) grid_slots_init(gc, slots);
  else grid_cache_reset(gc);
  double *lf = a.diag.lf;
  // the step loop, compiled twice: with the per-step light-front diagnostic
  // and without it (its test would otherwise cost every step an issue slot)
  auto steps = [&](auto with_lf) {
    constexpr bool LF = decltype(with_lf)::value;
    // in chunks: an int counter in the loop itself costs the step fewer
    // instructions than a long long one (PHASE64, Gaussian and per-cell grid: 1304
    // against 1268 us)
    for (long long s0 = 0; s0 < a.n_steps; s0 += kStepChunk) {
      const int cnt = (int)(a.n_steps - s0 < kStepChunk ? a.n_steps - s0 : kStepChunk);
      for (int k = 0; k < cnt; ++k) {
        const typename TimeBase<PREC>::Step st = tb.at(s0 + k);
        Local<R> L = local_coords<PREC>(P, st, pos);
        if constexpr (GRID && std::is_same<R, double>::value) grid_fetch(a.grid, gc, L.x, L.y, pos.zr());
        else if constexpr (GRID) grid_fetch_at(a.grid, gc, L.x, L.y, pos.zr());
        R E[3], B[3];
        analytic_fields<KIND, PREC>(P, L, E, B);
        if constexpr (GRID) grid_eval(gc, E, B);
        R ig = boris(u, E, B, dtR);
        pos.advance(u[0] * ig, u[1] * ig, u[2] * ig, dtxy, dtR);
        if constexpr (LF) {
          R dev = valid ? fabs((R(1) / ig - u[2]) - h0) : R(0);
          warp_max_to(lf + s0 + k, dev, 0xffffffffu);
        }
      }
    }
  };
  if (lf) steps(std::true_type{});
  else steps(std::false_type{});
  if (!valid) return 0.0;
  pos.store(a.x + i, a.y + i, a.z + i);
  R *ux = static_cast<R *>(a.ux);
  R *uy = static_cast<R *>(a.uy);
  R *uz = static_cast<R *>(a.uz);
  ux[i] = u[0];
  uy[i] = u[1];
  uz[i] = u[2];
  const double dx = (double)u[0], dy = (double)u[1], dz = (double)u[2];
  if (!all_finite(a.x[i], a.y[i], a.z[i], dx, dy, dz)) atomicOr(a.status, kStatusNonfinite);
  // gamma in double from the stored momentum, fixed operation order
  return __dsqrt_rn(__dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)),
                                        __dmul_rn(dz, dz)),
                              1.0));
}

// The FP64 push without a grid of plane waves and Gaussian beams.  A double
// instruction holds a scheduler's unit for 64 cycles, so a step costs its
// instructions: the polarisation is a compile-time parameter (in the pulse's
// frame, as in push_ff), so that zero components and the unused half of a sine
// and cosine are not evaluated, and the Boris step is boris_unit (kick and
// rotation summed before they join the momentum).  Arguments and result as for
// push_one.  1e4 electrons in a plane wave, 2000 steps with the light-front
// diagnostic: 9.96 -> 6.62 ms.
template <int KIND>
constexpr bool kPushD = KIND == AP_PLANE || KIND == AP_GAUSS || KIND == AP_FLYING_CF;

struct KickD {
  double hA, hAbr, hAce, hAcb, kA, kAce;
};

template <int KIND, int POL>
__device__ __forceinline__ UnitFields<double> unit_fields_d(const Pulse<double> &P, const Local<double> &L) {
  UnitFields<double> f;
  double mul, l2;
  envelope(P, L.eta, mul, l2);
  if constexpr (KIND == AP_PLANE) {
    double mag = mul;
    if (l2 != 0.0) mag *= exp2(l2);
    if (POL == kLin && !P.plasma) {
      f.Ur = mag * cos(L.psi);
      f.Ui = 0.0;
    } else {
      double s, c;
      sincos(L.psi, &s, &c);
      f.Ur = mag * c;
      f.Ui = mag * s;
    }
    f.Vr = f.Ur;
    f.Vi = f.Ui;
    if (P.plasma) {
      double L1, L2;
      envelope_logd(P, L.eta, L1, L2);
      const Cx<double> V = finite_duration(Cx<double>{f.Ur, f.Ui}, P.fdc, L1, L2, P.inv_w);
      f.Vr = V.re;
      f.Vi = V.im;
    }
    f.ez = f.bz = 0.0;
  } else {
    const BeamZ<double> Z = gauss_z<KIND == AP_FLYING_CF>(P, L);
    const double a = (L.x * L.x + L.y * L.y) * P.inv_w0sq;
    const double mag = mul * exp2(fma(a * Z.q.re, -kLog2e, l2));
    double s, c;
    sincos(L.psi - a * Z.q.im, &s, &c);
    const Cx<double> U = cmul(Z.q, Cx<double>{mag * c, mag * s});
    f.Ur = f.Vr = U.re;
    f.Ui = f.Vi = U.im;
    f.ez = f.bz = 0.0;
    if (P.lon) {
      const Cx<double> W = cmul(Z.q, U);
      f.ez = POL == kLin ? L.x * W.im : fma(L.x, W.im, -(L.y * W.re));
      f.bz = POL == kLin ? L.y * W.im : fma(L.x, W.re, L.y * W.im);
    }
  }
  return f;
}

template <int KIND>
__device__ __forceinline__ double push_d(const Pulse<double> &P, const PushArgs &a, long long i, bool valid) {
  double *uxs = static_cast<double *>(a.ux), *uys = static_cast<double *>(a.uy), *uzs = static_cast<double *>(a.uz);
  const int frame = P.fast.frame;
  Pos<AP_FP64> pos;
  double u[3] = {0.0, 0.0, 0.0};
  pos.load(0.0, 0.0, 0.0);
  if (valid) {
    pos.load(a.x[i], a.y[i], a.z[i]);
    u[0] = uxs[i];
    u[1] = uys[i];
    u[2] = uzs[i];
    if (frame == 1) {
      const double t = pos.x, tu = u[0];
      pos.x = pos.y;
      pos.y = -t;
      u[0] = u[1];
      u[1] = -tu;
    } else if (frame == 2) {
      pos.y = -pos.y;
      u[1] = -u[1];
    }
  }
  const double dt = a.dt, dtxy = dt * P.adv_xy, h = -0.5 * dt, g = P.lon ? -2.0 * P.inv_w0sq : 0.0;
  KickD k;
  k.hA = h * P.amp;
  k.hAbr = k.hA * P.bratio;
  k.hAce = k.hA * P.lonE * g;
  k.hAcb = k.hAbr * P.lonB * g;
  k.kA = 2.0 * k.hA;
  k.kAce = 2.0 * k.hAce;
  // gamma from 1 + u^2 and its inverse root (no division)
  auto gamma_of = [&](double ig) { return fma(u[0], u[0], fma(u[1], u[1], fma(u[2], u[2], 1.0))) * ig; };
  const double h0 = gamma_of(inv_gamma(u)) - u[2];
  double *lf = a.diag.lf;
  auto steps = [&](auto pol_c, auto lf_c) {
    constexpr int POL = decltype(pol_c)::value;
    constexpr bool LF = decltype(lf_c)::value;
    double nd = 0.0;
    for (long long n = 0; n < a.n_steps; ++n, nd += 1.0) {
      const Local<double> L = local_coords<AP_FP64>(P, fma(nd, dt, a.t0), pos);
      const UnitFields<double> f = unit_fields_d<KIND, POL>(P, L);
      const double ig = boris_unit<POL, KIND != AP_PLANE>(u, f, k);
      pos.advance(u[0] * ig, u[1] * ig, u[2] * ig, dtxy, dt);
      if constexpr (LF) warp_max_to(lf + n, valid ? fabs((gamma_of(ig) - u[2]) - h0) : 0.0, 0xffffffffu);
    }
  };
  using Lin = std::integral_constant<int, kLin>;
  using Circ = std::integral_constant<int, kCirc>;
  if (P.fast.circ) {
    if (lf) steps(Circ{}, std::true_type{});
    else steps(Circ{}, std::false_type{});
  } else {
    if (lf) steps(Lin{}, std::true_type{});
    else steps(Lin{}, std::false_type{});
  }
  if (!valid) return 0.0;
  if (frame == 1) {
    const double t = pos.x, tu = u[0];
    pos.x = -pos.y;
    pos.y = t;
    u[0] = -u[1];
    u[1] = tu;
  } else if (frame == 2) {
    pos.y = -pos.y;
    u[1] = -u[1];
  }
  pos.store(a.x + i, a.y + i, a.z + i);
  uxs[i] = u[0];
  uys[i] = u[1];
  uzs[i] = u[2];
  if (!all_finite(pos.x, pos.y, pos.z, u[0], u[1], u[2])) atomicOr(a.status, kStatusNonfinite);
  return __dsqrt_rn(__dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(u[0], u[0]), __dmul_rn(u[1], u[1])), __dmul_rn(u[2], u[2])),
                              1.0));
}

// One or two particles of a thread (R = float or F2) through n_steps fused
// float-float steps (ap_step.cuh): load (a2), per step the phase and unit
// fields (a3-a7), grid gather (a8), Boris and position (a9), light-front
// diagnostic (a10); then store (a11).  With two, particle i0 rides in the low
// half and i1 in the high half of every packed value, so each FP32
// instruction serves both; each keeps its own grid cell (its refetch is its
// own warp-uniform branch).  Every lane of a warp calls this together: the
// step table (phase C_n and time T_n) is made for the warp in shared memory
// 32 steps at a time, one entry per lane, __syncwarp only, so warps never
// wait for each other.  `v0`, `v1` are false for padding particles, which run
// the loop on a dummy state.  g receives the final gammas.
//
// Without a grid the pulse's frame is applied on load and store (y-polarised:
// x' = y, y' = -x; left-handed: y' = -y), so the loop knows two polarisations.
// With a grid the particles stay in the grid's frame and the analytic field
// is turned into it.  The loop is compiled for the common combinations (linear
// with a Gaussian envelope; linear; circular) and with and without the
// light-front test, which would otherwise cost every step its branches.

// grid units of the coordinates, and the thread's constants of grid_fetch2:
// written by the first four threads; the caller synchronises the block before
// use
__device__ __forceinline__ void grid_pair_consts(const GridView &g, const StepBase &s, float4 *gk) {
  if (threadIdx.x < 3) {
    const int ax = threadIdx.x;
    const float f = ax == 2 ? s.gz_s : g.inv_d[ax], o = ax == 2 ? s.gz_o.hi : g.off[ax];
    gk[ax] = make_float4(f, f, o, o);
  } else if (threadIdx.x == 3) {
    gk[3] = make_float4(0.5f, 0.5f, s.gz_o.lo, s.gz_o.lo);
  }
}

// the cell caches of a thread's one or two particles
template <int GRID, typename R>
struct Caches {
  using A = typename CacheOf<AP_FP32_PHASEFF, GRID>::type;
  A a;
  __device__ __forceinline__ void init(void *slots) {
    if constexpr (GRID != kGridNone) grid_slots_init(a, slots);
  }
  __device__ __forceinline__ void fetch(const GridView &g, const StepBase &s, const float4 *, R x, R y, R zhi, R zlo) {
    const float fz = grid_unit_z(zhi, zlo, s.gz_s, s.gz_o.hi, s.gz_o.lo);
    grid_fetch_units(g, a, grid_unit<float>(x, g.inv_d[0], g.off[0], g.top[0]),
                     grid_unit<float>(y, g.inv_d[1], g.off[1], g.top[1]), fminf(fmaxf(fz, 0.0f), g.top[2]));
  }
  __device__ __forceinline__ void values(R G[6]) {
    if constexpr (GRID != kGridCellsReg) cp_async_wait_all();  // this thread's copies landed
    grid_values(a, G);
  }
};
template <int GRID>
struct Caches<GRID, F2> {
  using A = typename std::conditional<GRID == kGridCells, CellSlots, CellRegs>::type;
  using B = typename std::conditional<GRID == kGridCellsReg, CellRegs, CellSlots>::type;
  A a;
  B b;
  __device__ __forceinline__ void init(void *slots) {
    if constexpr (GRID == kGridCellsMix) {
      grid_slots_init(a, nullptr);
      grid_slots_init(b, slots);
    } else if constexpr (GRID != kGridNone) {
      grid_slots_init(a, slots);
      grid_slots_init(b, static_cast<unsigned char *>(slots) + 12u * kCellSlotStride);
    }
  }
  __device__ __forceinline__ void fetch(const GridView &g, const StepBase &, const float4 *gk, F2 x, F2 y, F2 zhi,
                                        F2 zlo) {
    const float4 kz = gk[2], kl = gk[3];
    grid_fetch2(g, a, b, x, y, grid_unit_z(zhi, zlo, F2(kz.x, kz.y), F2(kz.z, kz.w), F2(kl.z, kl.w)), gk);
  }
  __device__ __forceinline__ void values(F2 G[6]) {
    if constexpr (GRID != kGridCellsReg) cp_async_wait_all();
    float oa[6], ob[6];
    grid_values(a, oa);
    grid_values(b, ob);
#pragma unroll
    for (int c = 0; c < 6; ++c) G[c] = F2(oa[c], ob[c]);
  }
};

// grid value plus factor times unit field, by scalar operations (the two
// particles' grid values come from different register pairs)
__device__ __forceinline__ float grid_plus(float f, float u, float g) { return rfma(f, u, g); }
__device__ __forceinline__ F2 grid_plus(float f, F2 u, F2 g) { return F2(rfma(f, u.x, g.x), rfma(f, u.y, g.y)); }

template <typename R>
__device__ __forceinline__ R pack_lanes(float a, float b) {
  if constexpr (IsPair<R>::value) return R(a, b);
  else return a;
}
__device__ __forceinline__ float lane_of(float v, int) { return v; }
__device__ __forceinline__ float lane_of(F2 v, int h) { return h ? v.y : v.x; }

// a state into the pulse's frame
__device__ __forceinline__ void to_frame(int frame, FF &x, FF &y, float u[3]) {
  if (frame == 1) {
    const FF t = x;
    x = y;
    y = FF{-t.hi, -t.lo};
    const float tu = u[0];
    u[0] = u[1];
    u[1] = -tu;
  } else if (frame == 2) {
    y = FF{-y.hi, -y.lo};
    u[1] = -u[1];
  }
}

template <int KIND, int GRID, typename R, class PT>
__device__ __forceinline__ void push_ff(const PT &P, const StepBase &sb, const PushArgs &a, long long i0, long long i1,
                                        bool v0, bool v1, float4 *s_steps, const float4 *comps, void *slots,
                                        const float4 *gk, double g[2]) {
  using FFR = typename FFOf<R>::type;
  constexpr int NP = IsPair<R>::value ? 2 : 1;
  const FastPulse &F = P.fast;
  const long long idx[2] = {i0, i1};
  const bool val[2] = {v0, v1};
  const int frame = GRID == kGridNone ? F.frame : 0;
  FF px[2], py[2], pz[2];
  float uu[2][3], h0[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    px[h] = py[h] = pz[h] = FF{0.0f, 0.0f};
    uu[h][0] = uu[h][1] = uu[h][2] = 0.0f;
    if (h < NP && val[h]) {
      const long long i = idx[h];
      px[h] = split_double(a.x[i]);
      py[h] = split_double(a.y[i]);
      pz[h] = split_double(__dmul_rn(__dsub_rn(a.z[i], P.z_f), F.z_scale));
      uu[h][0] = static_cast<const float *>(a.ux)[i];
      uu[h][1] = static_cast<const float *>(a.uy)[i];
      uu[h][2] = static_cast<const float *>(a.uz)[i];
      to_frame(frame, px[h], py[h], uu[h]);
    }
    // light-front reference h0 = gamma - u_z on entry
    h0[h] = 1.0f / rsqrt_r(fmaf(uu[h][0], uu[h][0], fmaf(uu[h][1], uu[h][1], fmaf(uu[h][2], uu[h][2], 1.0f)))) -
            uu[h][2];
  }
  FFR x{pack_lanes<R>(px[0].hi, px[1].hi), pack_lanes<R>(px[0].lo, px[1].lo)};
  FFR y{pack_lanes<R>(py[0].hi, py[1].hi), pack_lanes<R>(py[0].lo, py[1].lo)};
  FFR z{pack_lanes<R>(pz[0].hi, pz[1].hi), pack_lanes<R>(pz[0].lo, pz[1].lo)};
  R u[3] = {pack_lanes<R>(uu[0][0], uu[1][0]), pack_lanes<R>(uu[0][1], uu[1][1]), pack_lanes<R>(uu[0][2], uu[1][2])};
  Caches<GRID, R> gc;
  gc.init(slots);
  double *lf = a.diag.lf;
  float4 *wsteps = s_steps + (threadIdx.x >> 5) * kStepChunk;
  const int lane = threadIdx.x & 31;

  auto steps = [&](auto pol_c, auto env_c, auto lf_c) {
    constexpr int POL = decltype(pol_c)::value, ENV = decltype(env_c)::value;
    constexpr bool LF = decltype(lf_c)::value;
    for (long long s0 = 0; s0 < a.n_steps; s0 += kStepChunk) {
      const int cnt = (int)(a.n_steps - s0 < kStepChunk ? a.n_steps - s0 : kStepChunk);
      __syncwarp();  // no lane still reads the previous chunk
      if (lane < cnt) wsteps[lane] = step_entry<KIND>(F, sb, (float)(int)(s0 + lane));
      __syncwarp();
#pragma unroll 2
      for (int k = 0; k < cnt; ++k) {
        const float4 st = wsteps[k];
        R ig;
        if constexpr (GRID == kGridNone) {
          const UnitFields<R> f = unit_fields<KIND, POL, ENV>(P, comps, st, x.hi, y.hi, z.hi, z.lo);
          ig = boris_unit<POL, KIND != AP_PLANE>(u, f, sb);
        } else {
          gc.fetch(a.grid, sb, gk, x.hi, y.hi, z.hi, z.lo);
          R xe = x.hi, ye = y.hi;
          if constexpr (ENV == kEnvAny) {  // the common case has no frame
            if (F.frame == 1) {
              xe = y.hi;
              ye = rneg(x.hi);
            } else if (F.frame == 2) {
              ye = rneg(y.hi);
            }
          }
          const UnitFields<R> f = unit_fields<KIND, POL, ENV>(P, comps, st, xe, ye, z.hi, z.lo);
          R G[6];
          gc.values(G);
          if (POL == kLin) {
            if (ENV == kEnvGauss || F.frame == 0) {
              G[0] = grid_plus(F.A, f.Ur, G[0]);
              G[4] = grid_plus(F.Abr, f.Vr, G[4]);
            } else {
              G[1] = grid_plus(F.A, f.Ur, G[1]);
              G[3] = grid_plus(-F.Abr, f.Vr, G[3]);
            }
            G[2] = grid_plus(F.Ace, f.ez, G[2]);
            G[5] = grid_plus(F.Acb, f.bz, G[5]);
          } else {
            const float sg = F.frame == 2 ? -1.0f : 1.0f;  // exact signs
            G[0] = grid_plus(F.A, f.Ur, G[0]);
            G[1] = grid_plus(sg * F.A, f.Ui, G[1]);
            G[2] = grid_plus(F.Ace, f.ez, G[2]);
            G[3] = grid_plus(-sg * F.Abr, f.Vi, G[3]);
            G[4] = grid_plus(F.Abr, f.Vr, G[4]);
            G[5] = grid_plus(sg * F.Acb, f.bz, G[5]);
          }
          ig = boris_full(u, G, G + 3, sb.h, sb.k);
        }
        const R kxy = rmul(R(sb.cxy), ig);
        advance(x, u[0], kxy);
        advance(y, u[1], kxy);
        advance(z, u[2], rmul(R(sb.cz), ig));
        if constexpr (LF) {
          float dev = 0.0f;
#pragma unroll
          for (int h = 0; h < NP; ++h)
            if (val[h]) dev = fmaxf(dev, fabsf((1.0f / lane_of(ig, h) - lane_of(u[2], h)) - h0[h]));
          warp_max_to(lf + s0 + k, dev, 0xffffffffu);
        }
      }
    }
  };
  using Lin = std::integral_constant<int, kLin>;
  using Circ = std::integral_constant<int, kCirc>;
  using EnvG = std::integral_constant<int, kEnvGauss>;
  using EnvA = std::integral_constant<int, kEnvAny>;
  // kinds without an envelope switch or with no Gaussian default take the
  // general loop
  constexpr bool kGaussLoop = KIND == AP_GAUSS || KIND == AP_FLYING_CF;
  if (lf) {
    if (F.circ) steps(Circ{}, EnvA{}, std::true_type{});
    else steps(Lin{}, EnvA{}, std::true_type{});
  } else if (F.circ) {
    steps(Circ{}, EnvA{}, std::false_type{});
  } else if (kGaussLoop && P.env == AP_ENV_GAUSS && (GRID == kGridNone || F.frame == 0)) {
    if constexpr (kGaussLoop) steps(Lin{}, EnvG{}, std::false_type{});
  } else {
    steps(Lin{}, EnvA{}, std::false_type{});
  }

#pragma unroll
  for (int h = 0; h < NP; ++h) {
    g[h] = 0.0;
    if (!val[h]) continue;
    const long long i = idx[h];
    double X = (double)lane_of(x.hi, h) + (double)lane_of(x.lo, h);
    double Y = (double)lane_of(y.hi, h) + (double)lane_of(y.lo, h);
    const double Z = __dadd_rn(__dmul_rn((double)lane_of(z.hi, h) + (double)lane_of(z.lo, h), F.z_len), P.z_f);
    float fu[3] = {lane_of(u[0], h), lane_of(u[1], h), lane_of(u[2], h)};
    if (frame == 1) {
      const double t = X;
      X = -Y;
      Y = t;
      const float tu = fu[0];
      fu[0] = -fu[1];
      fu[1] = tu;
    } else if (frame == 2) {
      Y = -Y;
      fu[1] = -fu[1];
    }
    a.x[i] = X;
    a.y[i] = Y;
    a.z[i] = Z;
    static_cast<float *>(a.ux)[i] = fu[0];
    static_cast<float *>(a.uy)[i] = fu[1];
    static_cast<float *>(a.uz)[i] = fu[2];
    const double dx = (double)fu[0], dy = (double)fu[1], dz = (double)fu[2];
    if (!all_finite(X, Y, Z, dx, dy, dz)) atomicOr(a.status, kStatusNonfinite);
    // gamma in double from the stored momentum, fixed operation order
    g[h] = __dsqrt_rn(__dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)), 1.0));
  }
}

__device__ __forceinline__ void hist_add(uint32_t *s_hist, const DiagView &d, double g) {
  if (!isfinite(g)) return;
  double f = floor(__dmul_rn(__dsub_rn(g, d.hist_lo), d.hist_scale));
  int b = f < 0.0 ? 0 : (f > (double)(d.bins - 1) ? d.bins - 1 : (int)f);
  atomicAdd(&s_hist[b], 1u);
}

// block sum of a double; result valid in thread 0
__device__ __forceinline__ double block_sum(double v, double *s_red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s_red[w] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int k = 0; k < nw; ++k) r += s_red[k];
  return r;
}

// The pulse a float-float kernel is given: the component tables only where
// the kind has them.
template <int KIND>
using FFPulse = typename std::conditional<KIND == AP_FLYING_SUM, Pulse<float>, PulseHead<float>>::type;

// float4 of a block's component table (one particle per thread reads 16 bytes
// per component, two 32)
template <int KIND, int NP>
__host__ __device__ constexpr int comp_slots() { return KIND == AP_FLYING_SUM ? kMaxComp * NP : 1; }

// Plain launch: a grid-stride loop over block-sized chunks of particles (the
// trip count is uniform across the block), every step fused.  Dynamic shared
// memory: step tables, grid slots (float grid kernels), then the histogram
// (hist_off bytes in).  `push` advances the particles at base + threadIdx.x
// (and, with two per thread, one block further) and returns their gammas.
template <int NP, class Push>
__device__ __forceinline__ void push_chunks(const PushArgs &a, unsigned char *s_dyn, unsigned hist_off, const Push &push) {
  __shared__ double s_red[32];
  uint32_t *s_hist = reinterpret_cast<uint32_t *>(s_dyn + hist_off);
  const bool hist = a.diag.hist != nullptr;
  if (hist) {
    for (int b = threadIdx.x; b < a.diag.bins; b += blockDim.x) s_hist[b] = 0u;
    __syncthreads();
  }
  double acc = 0.0;
  // NP particles per thread: a block covers NP * blockDim.x consecutive
  // particles, thread t the ones at t and t + blockDim.x (coalesced)
  const long long stride = (long long)NP * gridDim.x * blockDim.x;
  for (long long base = (long long)NP * blockIdx.x * blockDim.x; base < a.n; base += stride) {
    const long long i = base + threadIdx.x;
    double g[2] = {0.0, 0.0};
    push(i, g);
#pragma unroll
    for (int h = 0; h < NP; ++h) {
      if (i + h * (long long)blockDim.x < a.n) {
        acc += g[h];
        if (hist) hist_add(s_hist, a.diag, g[h]);
      }
    }
  }
  if (a.diag.set_sum) {
    double t = block_sum(acc, s_red);
    if (threadIdx.x == 0) atomicAdd(a.diag.set_sum, t);
  }
  if (hist) {
    __syncthreads();
    for (int b = threadIdx.x; b < a.diag.bins; b += blockDim.x)
      if (s_hist[b]) atomicAdd(&a.diag.hist[b], s_hist[b]);
  }
}

// double, or native double phase: one particle per thread
template <int KIND, int PREC, int GRID>
__device__ __forceinline__ void push_body(const Pulse<Real<PREC>> &P, const PushArgs &a, unsigned hist_off) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  push_chunks<1>(a, s_dyn, hist_off, [&](long long i, double g[2]) {
    if constexpr (PREC == AP_FP64 && GRID == kGridNone && kPushD<KIND>) g[0] = push_d<KIND>(P, a, i, i < a.n);
    else g[0] = push_one<KIND, PREC, GRID>(P, a, i, i < a.n, s_dyn + step_table_bytes(blockDim.x));
  });
}

// float-float: NP particles per thread
template <int KIND, int GRID, int NP>
__device__ __forceinline__ void push_ff_body(const FFPulse<KIND> &P, const StepBase &sb, const PushArgs &a,
                                             unsigned hist_off) {
  using R = typename std::conditional<NP == 2, F2, float>::type;
  extern __shared__ __align__(16) unsigned char s_dyn[];
  __shared__ float4 s_gridk[4];
  __shared__ float4 s_comp[comp_slots<KIND, NP>()];
  if constexpr (KIND == AP_FLYING_SUM) comp_table<R>(P, s_comp);
  if constexpr (NP == 2 && GRID != kGridNone) grid_pair_consts(a.grid, sb, s_gridk);
  if constexpr (KIND == AP_FLYING_SUM || (NP == 2 && GRID != kGridNone)) __syncthreads();
  push_chunks<NP>(a, s_dyn, hist_off, [&](long long i, double g[2]) {
    const long long i1 = i + blockDim.x;
    push_ff<KIND, GRID, R>(P, sb, a, i, i1, i < a.n, NP == 2 && i1 < a.n, reinterpret_cast<float4 *>(s_dyn), s_comp,
                           s_dyn + step_table_bytes(blockDim.x), s_gridk, g);
  });
}

// Two entries for the same body.  The per-cell coefficient variants name a
// residency target (3 blocks of 256 with the cell in shared memory, 2 with
// it in registers); the others keep the compiler's own register choice (an
// explicit minimum of one block lets it spend registers freely, which cost
// the flying-focus kernel 7 % through lost occupancy).
template <int KIND, int PREC, int GRID>
__global__ void __launch_bounds__(256)
    push_kernel(const __grid_constant__ Pulse<Real<PREC>> P, const __grid_constant__ PushArgs a,
                unsigned hist_off) {
  push_body<KIND, PREC, GRID>(P, a, hist_off);
}

template <int KIND, int PREC, int GRID>
__global__ void __launch_bounds__(256, GRID == kGridCells ? 3 : 2)
    push_kernel_cells(const __grid_constant__ Pulse<Real<PREC>> P, const __grid_constant__ PushArgs a,
                      unsigned hist_off) {
  push_body<KIND, PREC, GRID>(P, a, hist_off);
}

template <int KIND, int PREC, int GRID>
constexpr auto push_entry() {
  if constexpr (GRID == kGridCells || GRID == kGridCellsReg) return push_kernel_cells<KIND, PREC, GRID>;
  else return push_kernel<KIND, PREC, GRID>;
}

// float-float: without a residency target, and with one (blocks of 256 per
// SM: 3 for one particle per thread with its cell in shared memory, 2 with it
// in registers or with two particles per thread and a cell in shared memory)
template <int KIND, int GRID, int NP>
__global__ void __launch_bounds__(256)
    push_ff_kernel(const __grid_constant__ FFPulse<KIND> P, const __grid_constant__ StepBase sb,
                   const __grid_constant__ PushArgs a, unsigned hist_off) {
  push_ff_body<KIND, GRID, NP>(P, sb, a, hist_off);
}
template <int KIND, int GRID, int NP>
__global__ void __launch_bounds__(256, NP == 1 && GRID == kGridCells ? 3 : 2)
    push_ff_kernel_cells(const __grid_constant__ FFPulse<KIND> P, const __grid_constant__ StepBase sb,
                         const __grid_constant__ PushArgs a, unsigned hist_off) {
  push_ff_body<KIND, GRID, NP>(P, sb, a, hist_off);
}

template <int KIND, int GRID, int NP>
constexpr auto push_ff_entry() {
  if constexpr (GRID == kGridCells || GRID == kGridCellsMix || (GRID == kGridCellsReg && NP == 1))
    return push_ff_kernel_cells<KIND, GRID, NP>;
  else return push_ff_kernel<KIND, GRID, NP>;
}

// Batched persistent launch (row a12): blocks pop fixed-size tiles of
// (set, particles) from a global counter until the tile count is reached;
// each set's pulse is copied to shared memory; the loop is bounded by the
// tile count and no block waits on another.
// Dynamic shared memory: step tables, grid slots (float grid kernels), then
// the [n_sets + 1] tile prefix (prefix_off bytes in).

// Exclusive prefix of the sets' tile counts (tiles of set s = ceil(N_s / per))
// into prefix[0 .. n_sets] by the block's first warp; the caller synchronises
// the block.  `count(s)` is the set's particle count.
template <class Count>
__device__ __forceinline__ void tile_prefix(long long *prefix, int n_sets, int per, const Count &count) {
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x;
  long long acc = 0;
  for (int s0 = 0; s0 < n_sets; s0 += 32) {
    const int s = s0 + lane;
    const long long ns = s < n_sets ? count(s) : 0;
    // malformed offsets (ns < 0): no tiles (particles are bounds-checked by the caller)
    const long long t = ns > 0 ? (ns + per - 1) / per : 0;
    long long v = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long w = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += w;
    }
    if (s < n_sets) prefix[s] = acc + v - t;
    acc += __shfl_sync(0xffffffffu, v, 31);
  }
  if (lane == 0) prefix[n_sets] = acc;
}

template <int KIND, int PREC, int GRID, int NP>
__device__ __forceinline__ void batch_body(const Pulse<Real<PREC>> *__restrict__ sets,
                                           const BatchArgs &ba, unsigned prefix_off) {
  using R = Real<PREC>;
  constexpr bool kFF = PREC == AP_FP32_PHASEFF;
  // the part of the pulse the kind reads (a multiple of 4 bytes)
  using PT = typename std::conditional<KIND == AP_FLYING_SUM || !kFF, Pulse<R>, PulseHead<R>>::type;
  extern __shared__ __align__(16) unsigned char s_dyn[];
  __shared__ double s_red[32];
  __shared__ long long s_tile;
  __shared__ int s_set;
  void *slots = s_dyn + step_table_bytes(blockDim.x);
  long long *s_prefix = reinterpret_cast<long long *>(s_dyn + prefix_off);
  __shared__ __align__(16) unsigned char s_pulse_raw[sizeof(PT)];
  PT &sp = *reinterpret_cast<PT *>(s_pulse_raw);
  const PushArgs &a = ba.base;
  const int T = ba.tile;
  __shared__ float4 s_gridk[4];
  __shared__ StepBase s_base;
  __shared__ float4 s_comp[kFF ? comp_slots<KIND, NP>() : 1];
  tile_prefix(s_prefix, ba.n_sets, T,
              [&](int s) { return ba.set_offsets[s + 1] - ba.set_offsets[s]; });
  if (threadIdx.x == 0) s_set = -1;
  __syncthreads();
  const long long total = s_prefix[ba.n_sets];
  for (;;) {
    if (threadIdx.x == 0) s_tile = (long long)atomicAdd(ba.tile_counter, 1u);
    __syncthreads();
    const long long tile = s_tile;
    if (tile >= total) break;
    // set of this tile: last s with prefix[s] <= tile (binary search)
    int lo = 0, hi = ba.n_sets;
    while (hi - lo > 1) {
      int mid = (lo + hi) >> 1;
      if (s_prefix[mid] <= tile) lo = mid; else hi = mid;
    }
    const int set = lo;
    if (set != s_set) {
      const int words = (int)(sizeof(PT) / 4);
      const uint32_t *src = reinterpret_cast<const uint32_t *>(sets + set);
      uint32_t *dst = reinterpret_cast<uint32_t *>(s_pulse_raw);
      for (int w = threadIdx.x; w < words; w += blockDim.x) dst[w] = src[w];
      __syncthreads();
      if (threadIdx.x == 0) s_set = set;
      if constexpr (kFF) {
        using RR = typename std::conditional<NP == 2, F2, float>::type;
        if (threadIdx.x == 0) s_base = make_step_base(sp, a.t0, a.dt, a.grid);
        if constexpr (KIND == AP_FLYING_SUM) comp_table<RR>(sp, s_comp);
        if constexpr (NP == 2 && GRID != kGridNone) {
          __syncthreads();
          grid_pair_consts(a.grid, s_base, s_gridk);
        }
      }
    }
    __syncthreads();
    const long long first = ba.set_offsets[set] + (tile - s_prefix[set]) * T;
    const long long end_set = ba.set_offsets[set + 1];
    double acc = 0.0;
    // T is a multiple of NP * blockDim.x: every thread runs the same trip count
    for (int k = threadIdx.x; k < T; k += NP * blockDim.x) {
      const long long i = first + k;
      const bool valid = i >= 0 && i < end_set && i < a.n;
      if constexpr (kFF) {
        using RR = typename std::conditional<NP == 2, F2, float>::type;
        const long long i1 = i + blockDim.x;
        const bool valid1 = NP == 2 && i1 >= 0 && i1 < end_set && i1 < a.n;
        double g[2];
        push_ff<KIND, GRID, RR>(sp, s_base, a, i, i1, valid, valid1, reinterpret_cast<float4 *>(s_dyn), s_comp, slots,
                                s_gridk, g);
        if (valid) acc += g[0];
        if (valid1) acc += g[1];
      } else {
        double g;
        if constexpr (PREC == AP_FP64 && GRID == kGridNone && kPushD<KIND>) g = push_d<KIND>(sp, a, i, valid);
        else g = push_one<KIND, PREC, GRID>(sp, a, i, valid, slots);
        if (valid) acc += g;
      }
    }
    if (a.diag.set_sum) {
      double t = block_sum(acc, s_red);
      if (threadIdx.x == 0) atomicAdd(a.diag.set_sum + set, t);
    }
    __syncthreads();
  }
}

template <int KIND, int PREC, int GRID, int NP = 1>
__global__ void __launch_bounds__(256) batch_kernel(const Pulse<Real<PREC>> *__restrict__ sets,
                                                    const __grid_constant__ BatchArgs ba,
                                                    unsigned prefix_off) {
  batch_body<KIND, PREC, GRID, NP>(sets, ba, prefix_off);
}
// two particles per thread: 2 blocks of 256 with one or both cells in shared
// memory; 4 for the beams without a grid that fit 64 registers (batched_256:
// 256 sets, 4e6 particles, 500 steps: 5.05 -> 4.88 ms against the compiler's own 80)
template <int KIND, int GRID>
__global__ void __launch_bounds__(256, GRID == kGridNone ? 4 : 2)
    batch_kernel_pair_minb(const Pulse<float> *__restrict__ sets, const __grid_constant__ BatchArgs ba,
                         unsigned prefix_off) {
  batch_body<KIND, AP_FP32_PHASEFF, GRID, 2>(sets, ba, prefix_off);
}

// Field evaluation hook: one point per thread, the push's own code path at
// step 0 of a time base starting at the point's t.
template <int KIND, int PREC>
__global__ void __launch_bounds__(256) eval_kernel(const __grid_constant__ Pulse<Real<PREC>> P,
                                                   const __grid_constant__ EvalArgs a) {
  using R = Real<PREC>;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.n) return;
  const double x = a.xyzt[i], y = a.xyzt[a.n + i], z = a.xyzt[2 * a.n + i],
               t = a.xyzt[3 * a.n + i];
  Pos<PREC> pos;
  pos.load(x, y, z);
  TimeBase<PREC> tb;
  tb.init(P, t, 0.0);
  Local<R> L = local_coords<PREC>(P, tb.at(0), pos);
  R E[3], B[3];
  analytic_fields<KIND, PREC>(P, L, E, B);
  for (int c = 0; c < 3; ++c) {
    a.EB[(long long)c * a.n + i] = (double)E[c];
    a.EB[(long long)(c + 3) * a.n + i] = (double)B[c];
  }
}

// Analytic fields on the staggered nodes of a Yee grid (ap_eval_nodes).
// blockIdx.y picks one present component c; threads stride over the nodes,
// x fastest, so every store is coalesced.  Component c is sampled at
// lo + (idx + off_c) d with the Yee offsets off = Ex (1/2,0,0), Ey (0,1/2,0),
// Ez (0,0,1/2), Bx (0,1/2,1/2), By (1/2,0,1/2), Bz (1/2,1/2,0); E and B both
// at time t.  The node index advances by the fixed grid stride with carries
// (one division per thread), and in the float-float variant the node
// position is formed in float-float arithmetic, so the loop issues no
// double-precision instruction.
__device__ __forceinline__ FF node_coord_ff(float f, float lo_hi, float lo_lo, float d_hi, float d_lo) {
  FF p = two_prod(f, d_hi);
  p.lo = __fmaf_rn(f, d_lo, p.lo);
  FF s = two_sum(lo_hi, p.hi);
  s.lo = __fadd_rn(s.lo, __fadd_rn(lo_lo, p.lo));
  const float hi = __fadd_rn(s.hi, s.lo);
  return {hi, __fsub_rn(s.lo, __fsub_rn(hi, s.hi))};
}

// What a node receives: the analytic E1, B1, or (plane waves, `current`)
// the analytic current J1 in place of E with B zero.
template <int KIND, int PREC>
__device__ __forceinline__ void node_values(const Pulse<Real<PREC>> &P, const Local<Real<PREC>> &L,
                                            int current, Real<PREC> E[3], Real<PREC> B[3]) {
  if constexpr (KIND == AP_PLANE) {
    if (current) {
      current_plane(P, L, E);
      B[0] = B[1] = B[2] = Real<PREC>(0);
      return;
    }
  }
  analytic_fields<KIND, PREC>(P, L, E, B);
}

template <int KIND, int PREC, typename T>
__global__ void __launch_bounds__(256) nodes_kernel(const __grid_constant__ Pulse<Real<PREC>> P,
                                                    const __grid_constant__ NodeArgs a) {
  using R = Real<PREC>;
  using W = typename std::conditional<(sizeof(T) > sizeof(R)), T, R>::type;
  const int c = a.comp[blockIdx.y];
  T *__restrict__ f = static_cast<T *>(a.f[c]);
  const float ox = (c == 0 || c == 4 || c == 5) ? 0.5f : 0.0f;
  const float oy = (c == 1 || c == 3 || c == 5) ? 0.5f : 0.0f;
  const float oz = (c == 2 || c == 3 || c == 4) ? 0.5f : 0.0f;
  const long long nxy = (long long)a.nx * a.ny;
  const long long total = nxy * a.nz;
  long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= total) return;
  const long long stride = (long long)gridDim.x * blockDim.x;
  // node (i, j, k) of n and the stride split the same way; every index is
  // below 2^23 (checked on the host), so index + stride stays exact in float
  int k = (int)(n / nxy);
  int j = (int)((n - (long long)k * nxy) / a.nx);
  int i = (int)(n - (long long)k * nxy - (long long)j * a.nx);
  const long long sk64 = stride / nxy;
  const int sj = (int)((stride - sk64 * nxy) / a.nx);
  const int si = (int)(stride - sk64 * nxy - (long long)sj * a.nx);
  const int sk = (int)(sk64 < (1 << 30) ? sk64 : (1 << 30));
  // float copies of the indices, advanced alongside (int -> float
  // conversions run on the double-precision pipe)
  float fi = (float)i, fj = (float)j, fk = (float)k;
  const float fsi = (float)si, fsj = (float)sj, fsk = (float)sk;
  const float fnx = (float)a.nx, fny = (float)a.ny;
  TimeBase<PREC> tb;
  tb.init(P, a.t, 0.0);
  const typename TimeBase<PREC>::Step st = tb.at(0);
  for (; n < total; n += stride) {
    Pos<PREC> pos;
    if constexpr (PREC == AP_FP32_PHASEFF) {
      // the transverse coordinates enter the fields in float; only z feeds
      // the carrier phase and needs the float-float sum
      pos.x = FF{fmaf(fi + ox, a.d_hi[0], a.lo_hi[0]), 0.0f};
      pos.y = FF{fmaf(fj + oy, a.d_hi[1], a.lo_hi[1]), 0.0f};
      pos.z = node_coord_ff(fk + oz, a.lo_hi[2], a.lo_lo[2], a.d_hi[2], a.d_lo[2]);
    } else {
      pos.load(fma((double)i + ox, a.d[0], a.lo[0]), fma((double)j + oy, a.d[1], a.lo[1]),
               fma((double)k + oz, a.d[2], a.lo[2]));
    }
    Local<R> L = local_coords<PREC>(P, st, pos);
    R E[3], B[3];
    node_values<KIND, PREC>(P, L, a.current, E, B);
    const R v = c == 0 ? E[0] : c == 1 ? E[1] : c == 2 ? E[2] : c == 3 ? B[0] : c == 4 ? B[1] : B[2];
    f[n] = a.accumulate ? (T)((W)f[n] + (W)v) : (T)v;
    // advance (i, j, k) by the stride (k only grows until the loop ends)
    i += si;
    fi += fsi;
    int cj = 0;
    if (i >= a.nx) { i -= a.nx; fi -= fnx; cj = 1; }
    j += sj + cj;
    fj += fsj + (cj ? 1.0f : 0.0f);
    int ck = 0;
    if (j >= a.ny) { j -= a.ny; fj -= fny; ck = 1; }
    k = min(k + sk + ck, 1 << 30);
    fk += fsk + (ck ? 1.0f : 0.0f);
  }
}

// ------------------------------------------------------------ launchers

template <typename K>
inline int occupancy_blocks(K kernel, int block, size_t smem) {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, block, smem) != cudaSuccess)
    return 1;
  return nb > 0 ? nb : 1;
}

// dynamic shared memory before the kernel-specific tail (histogram / prefix)
template <int PREC, int GRID, int NP = 1>
inline size_t push_smem_head(int block) {
  return step_table_bytes(block) + grid_cache_bytes<PREC, GRID, NP>(block);
}

// opt in above what every kernel gets without asking: 48 KB less its static
// shared memory (up to 14 KB here: a pulse, a component table).  The most that a
// push asks for: a block of 256, with a histogram of 8192 bins or the prefix of
// AP_MAX_SETS sets.
template <int PREC, int GRID, int NP, typename K>
inline int set_smem(K kern, size_t smem) {
  constexpr size_t tail = (AP_MAX_SETS + 1) * sizeof(long long);
  static_assert(tail >= 8192 * sizeof(uint32_t), "the longer tail");
  return smem <= 32 * 1024
             ? AP_OK
             : allow_smem(reinterpret_cast<const void *>(kern), push_smem_head<PREC, GRID, NP>(256) + tail);
}

template <int KIND, int PREC, int GRID>
int launch_push_t(const Pulse<Real<PREC>> &P, const PushArgs &a, void *stream) {
  auto kern = push_entry<KIND, PREC, GRID>();
  const int block = a.shape.block;
  const size_t head = push_smem_head<PREC, GRID>(block);
  const size_t smem = head + (a.diag.hist ? (size_t)a.diag.bins * sizeof(uint32_t) : 0);
  if (set_smem<PREC, GRID, 1>(kern, smem) != AP_OK) return AP_ERR_CUDA;
  const long long npad = (a.n + 31) & ~31LL;
  long long want = (npad + block - 1) / block;
  int per_sm = a.shape.blocks_per_sm > 0 ? a.shape.blocks_per_sm : occupancy_blocks(kern, block, smem);
  long long cap = (long long)a.sm_count * per_sm;
  int grid = (int)(want < cap ? want : cap);
  if (grid < 1) grid = 1;
  kern<<<grid, block, smem, static_cast<cudaStream_t>(stream)>>>(P, a, (unsigned)head);
  return cudaGetLastError() == cudaSuccess ? AP_OK : AP_ERR_CUDA;
}

// float-float: NP particles per thread, the call's constants made here
template <int KIND, int GRID, int NP>
int launch_push_ff_t(const Pulse<float> &P, const PushArgs &a, void *stream) {
  auto kern = push_ff_entry<KIND, GRID, NP>();
  const int block = a.shape.block;
  const size_t head = push_smem_head<AP_FP32_PHASEFF, GRID, NP>(block);
  const size_t smem = head + (a.diag.hist ? (size_t)a.diag.bins * sizeof(uint32_t) : 0);
  if (set_smem<AP_FP32_PHASEFF, GRID, NP>(kern, smem) != AP_OK) return AP_ERR_CUDA;
  // Node corners: four blocks of 128 per SM and the rest of the 256 KB to the L1
  // cache.  At 80 registers six fit, whose slots would leave it 30 KB, and the
  // gather from plain component arrays (48 loads of 4 bytes per cell, sectors
  // shared by neighbouring corners) lives from it (256^3 grid, 2e6 particles, 50
  // steps: plain arrays 2519 us with the driver's choice, 1305 so; packed nodes
  // 965 / 870).
  if (GRID == kGridNodes &&
      cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 60) != cudaSuccess)
    return AP_ERR_CUDA;
  const long long per_block = (long long)NP * block;
  const long long want = (a.n + per_block - 1) / per_block;
  int per_sm = a.shape.blocks_per_sm > 0 ? a.shape.blocks_per_sm : occupancy_blocks(kern, block, smem);
  long long cap = (long long)a.sm_count * per_sm;
  int grid = (int)(want < cap ? want : cap);
  if (grid < 1) grid = 1;
  const StepBase sb = make_step_base(P, a.t0, a.dt, a.grid);
  kern<<<grid, block, smem, static_cast<cudaStream_t>(stream)>>>(P, sb, a, (unsigned)head);
  return cudaGetLastError() == cudaSuccess ? AP_OK : AP_ERR_CUDA;
}

template <int KIND, int PREC>
int launch_eval_t(const Pulse<Real<PREC>> &P, const EvalArgs &a, void *stream) {
  const int block = 128;
  const long long grid = (a.n + block - 1) / block;
  eval_kernel<KIND, PREC><<<(unsigned)grid, block, 0, static_cast<cudaStream_t>(stream)>>>(P, a);
  return cudaGetLastError() == cudaSuccess ? AP_OK : AP_ERR_CUDA;
}

// All requested components of every node in one thread.  The six staggered
// positions of a node share two z levels -- the whole node (Ex, Ey, Bz) and
// the half node (Ez, Bx, By) -- so the z- and t-only part of the evaluation
// (local coordinates and carrier phase, envelope, and for beams the complex
// q = 1/(1 - i zeta)) is computed once per level: the six evaluations are
// straight-line code with identical z-only inputs, which the compiler
// computes once.  Used when three or more components are requested.
template <int KIND, int PREC, typename T>
__global__ void __launch_bounds__(256) nodes_all_kernel(const __grid_constant__ Pulse<Real<PREC>> P,
                                                        const __grid_constant__ NodeArgs a) {
  using R = Real<PREC>;
  using W = typename std::conditional<(sizeof(T) > sizeof(R)), T, R>::type;
  unsigned want = 0u;  // bit c: component c requested (a register, not an indexed array)
  for (int q = 0; q < a.n_comp; ++q) want |= 1u << a.comp[q];
  const long long nxy = (long long)a.nx * a.ny;
  const long long total = nxy * a.nz;
  long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= total) return;
  const long long stride = (long long)gridDim.x * blockDim.x;
  // node (i, j, k) of n and of the stride, advanced as in nodes_kernel (float
  // copies of the indices: no int-to-float conversion per node)
  int k = (int)(n / nxy);
  int j = (int)((n - (long long)k * nxy) / a.nx);
  int i = (int)(n - (long long)k * nxy - (long long)j * a.nx);
  const long long sk64 = stride / nxy;
  const int sj = (int)((stride - sk64 * nxy) / a.nx);
  const int si = (int)(stride - sk64 * nxy - (long long)sj * a.nx);
  const int sk = (int)(sk64 < (1 << 30) ? sk64 : (1 << 30));
  float fi = (float)i, fj = (float)j, fk = (float)k;
  const float fsi = (float)si, fsj = (float)sj, fsk = (float)sk;
  const float fnx = (float)a.nx, fny = (float)a.ny;
  TimeBase<PREC> tb;
  tb.init(P, a.t, 0.0);
  const typename TimeBase<PREC>::Step st = tb.at(0);
  for (; n < total; n += stride) {
    Local<R> Lz[2];
    R xs[2], ys[2];  // transverse coordinates at the whole and the half node
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float o = h ? 0.5f : 0.0f;
      Pos<PREC> pos;
      if constexpr (PREC == AP_FP32_PHASEFF) {
        pos.x = FF{0.0f, 0.0f};
        pos.y = FF{0.0f, 0.0f};
        pos.z = node_coord_ff(fk + o, a.lo_hi[2], a.lo_lo[2], a.d_hi[2], a.d_lo[2]);
        xs[h] = fmaf(fi + o, a.d_hi[0], a.lo_hi[0]);
        ys[h] = fmaf(fj + o, a.d_hi[1], a.lo_hi[1]);
      } else {
        pos.load(0.0, 0.0, fma((double)k + o, a.d[2], a.lo[2]));
        xs[h] = (R)fma((double)i + o, a.d[0], a.lo[0]);
        ys[h] = (R)fma((double)j + o, a.d[1], a.lo[1]);
      }
      Lz[h] = local_coords<PREC>(P, st, pos);
    }
    // component c at (x, y, z) offsets (Ex (1/2,0,0), Ey (0,1/2,0), Ez (0,0,1/2),
    // Bx (0,1/2,1/2), By (1/2,0,1/2), Bz (1/2,1/2,0))
    constexpr int kOx[6] = {1, 0, 0, 0, 1, 1}, kOy[6] = {0, 1, 0, 1, 0, 1}, kOz[6] = {0, 0, 1, 1, 1, 0};
    R v[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      Local<R> L = Lz[kOz[c]];
      L.x = xs[kOx[c]];
      L.y = ys[kOy[c]];
      R E[3], B[3];
      node_values<KIND, PREC>(P, L, a.current, E, B);
      v[c] = c < 3 ? E[c] : B[c - 3];
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      if (!((want >> c) & 1u)) continue;
      T *f = static_cast<T *>(a.f[c]);
      f[n] = a.accumulate ? (T)((W)f[n] + (W)v[c]) : (T)v[c];
    }
    i += si;
    fi += fsi;
    int cj = 0;
    if (i >= a.nx) { i -= a.nx; fi -= fnx; cj = 1; }
    j += sj + cj;
    fj += fsj + (cj ? 1.0f : 0.0f);
    int ck = 0;
    if (j >= a.ny) { j -= a.ny; fj -= fny; ck = 1; }
    k = min(k + sk + ck, 1 << 30);
    fk += fsk + (ck ? 1.0f : 0.0f);
  }
}

// Rows of nx >= 32 nodes, three or more components: one warp per (y, z)
// row, lane l taking the nodes x = l, l + 32, ... (coalesced stores).  The
// z/t part of the six staggered evaluations (local coordinates and carrier
// phase, envelope, q) depends only on the row's two z levels: each lane
// computes it once per row and reuses it for all its nodes, so per node only
// the position part of the six evaluations remains (straight-line code, as
// in nodes_all_kernel).
template <int KIND, int PREC, typename T>
__global__ void __launch_bounds__(256) nodes_row_kernel(const __grid_constant__ Pulse<Real<PREC>> P,
                                                        const __grid_constant__ NodeArgs a) {
  using R = Real<PREC>;
  using W = typename std::conditional<(sizeof(T) > sizeof(R)), T, R>::type;
  unsigned want = 0u;
  for (int q = 0; q < a.n_comp; ++q) want |= 1u << a.comp[q];
  const long long rows = (long long)a.ny * a.nz;
  const int lane = threadIdx.x & 31;
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  const float flane = (float)lane;
  TimeBase<PREC> tb;
  tb.init(P, a.t, 0.0);
  const typename TimeBase<PREC>::Step st = tb.at(0);
  constexpr int kOx[6] = {1, 0, 0, 0, 1, 1}, kOy[6] = {0, 1, 0, 1, 0, 1}, kOz[6] = {0, 0, 1, 1, 1, 0};
  for (long long r = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < rows; r += warps) {
    const int k = (int)(r / a.ny);
    const int j = (int)(r - (long long)k * a.ny);
    Local<R> Lz[2];
    R ys[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float o = h ? 0.5f : 0.0f;
      Pos<PREC> pos;
      if constexpr (PREC == AP_FP32_PHASEFF) {
        pos.x = FF{0.0f, 0.0f};
        pos.y = FF{0.0f, 0.0f};
        pos.z = node_coord_ff((float)k + o, a.lo_hi[2], a.lo_lo[2], a.d_hi[2], a.d_lo[2]);
        ys[h] = fmaf((float)j + o, a.d_hi[1], a.lo_hi[1]);
      } else {
        pos.load(0.0, 0.0, fma((double)k + o, a.d[2], a.lo[2]));
        ys[h] = (R)fma((double)j + o, a.d[1], a.lo[1]);
      }
      Lz[h] = local_coords<PREC>(P, st, pos);
    }
    const long long base = r * a.nx;
    float fi = flane;
    for (int i = lane; i < a.nx; i += 32, fi += 32.0f) {
      R xs[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float o = h ? 0.5f : 0.0f;
        if constexpr (PREC == AP_FP32_PHASEFF) xs[h] = fmaf(fi + o, a.d_hi[0], a.lo_hi[0]);
        else xs[h] = (R)fma((double)i + o, a.d[0], a.lo[0]);
      }
      R v[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        Local<R> L = Lz[kOz[c]];
        L.x = xs[kOx[c]];
        L.y = ys[kOy[c]];
        R E[3], B[3];
        node_values<KIND, PREC>(P, L, a.current, E, B);
        v[c] = c < 3 ? E[c] : B[c - 3];
      }
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        if (!((want >> c) & 1u)) continue;
        T *f = static_cast<T *>(a.f[c]) + base;
        f[i] = a.accumulate ? (T)((W)f[i] + (W)v[c]) : (T)v[c];
      }
    }
  }
}

// The row kernel with two nodes per lane and iteration (float-float, beams):
// lane l takes x = l + 64 m and l + 64 m + 32, the two halves of every packed
// value (ap_pair.cuh), so the position part of the six evaluations -- the
// only per-node work -- issues once for both nodes.  Each warp takes a
// contiguous run of rows, so the z/t part of its rows (carrier phase and
// envelope argument; for Gaussian beams also the envelope and q) is computed
// only when the z index changes, once per run of up to ny rows, instead of once
// per row.  Stores stay coalesced: the warp writes 32 consecutive elements for
// each half.
template <int KIND, typename T>
__global__ void __launch_bounds__(256) nodes_row_pair_kernel(const __grid_constant__ Pulse<float> P,
                                                             const __grid_constant__ NodeArgs a) {
  using W = typename std::conditional<(sizeof(T) > sizeof(float)), T, float>::type;
  constexpr bool kGaussZ = KIND == AP_GAUSS || KIND == AP_FLYING_CF;
  unsigned want = 0u;
  for (int q = 0; q < a.n_comp; ++q) want |= 1u << a.comp[q];
  const long long rows = (long long)a.ny * a.nz;
  const int lane = threadIdx.x & 31;
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  const long long wid = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long long per = (rows + warps - 1) / warps;
  const long long r0 = wid * per, r1 = r0 + per < rows ? r0 + per : rows;
  const float flane = (float)lane;
  TimeBase<AP_FP32_PHASEFF> tb;
  tb.init(P, a.t, 0.0);
  const StepFF st = tb.at(0);
  constexpr int kOx[6] = {1, 0, 0, 0, 1, 1}, kOy[6] = {0, 1, 0, 1, 0, 1}, kOz[6] = {0, 0, 1, 1, 1, 0};
  int kcur = -1;
  Local<F2> Lz[2];
  BeamZ<F2> Bz[2];
  // (j, k) of the run's first row by one division, then stepped row by row
  int k = (int)(r0 / a.ny);
  int j = (int)(r0 - (long long)k * a.ny);
  for (long long r = r0; r < r1; ++r, ++j) {
    if (j == a.ny) {
      j = 0;
      ++k;
    }
    if (k != kcur) {  // uniform across the warp
      kcur = k;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        Pos<AP_FP32_PHASEFF> pos;
        pos.x = FF{0.0f, 0.0f};
        pos.y = FF{0.0f, 0.0f};
        pos.z = node_coord_ff((float)k + (h ? 0.5f : 0.0f), a.lo_hi[2], a.lo_lo[2], a.d_hi[2], a.d_lo[2]);
        const Local<float> l = local_coords<AP_FP32_PHASEFF>(P, st, pos);
        if constexpr (kGaussZ) {
          const BeamZ<float> b = gauss_z<KIND == AP_FLYING_CF>(P, l);
          Bz[h] = BeamZ<F2>{Cx<F2>{F2(b.q.re), F2(b.q.im)}, F2(b.amp_mul), F2(b.l2), F2(b.psi)};
        } else {
          Lz[h] = Local<F2>{F2(l.x), F2(l.y), F2(l.dz), F2(l.psi), F2(l.eta), F2(l.T), F2(l.phi_hi), F2(l.phi_lo)};
        }
      }
    }
    const float ys[2] = {fmaf((float)j, a.d_hi[1], a.lo_hi[1]), fmaf((float)j + 0.5f, a.d_hi[1], a.lo_hi[1])};
    const long long base = r * a.nx;
    float fi = flane;
    for (int i = lane; i < a.nx; i += 64, fi += 64.0f) {
      const bool second = i + 32 < a.nx;
      F2 xs[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float o = h ? 0.5f : 0.0f;
        xs[h] = fma(F2(fi + o, fi + (32.0f + o)), F2(a.d_hi[0]), F2(a.lo_hi[0]));
      }
      F2 v[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        F2 E[3], B[3];
        if constexpr (kGaussZ) {
          gauss_xy(P, Bz[kOz[c]], xs[kOx[c]], F2(ys[kOy[c]]), E, B);
        } else {
          Local<F2> L = Lz[kOz[c]];
          L.x = xs[kOx[c]];
          L.y = F2(ys[kOy[c]]);
          analytic_fields<KIND, AP_FP32_PHASEFF, F2>(P, L, E, B);
        }
        v[c] = c < 3 ? E[c] : B[c - 3];
      }
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        if (!((want >> c) & 1u)) continue;
        T *f = static_cast<T *>(a.f[c]) + base;
        f[i] = a.accumulate ? (T)((W)f[i] + (W)v[c].x) : (T)v[c].x;
        if (second) f[i + 32] = a.accumulate ? (T)((W)f[i + 32] + (W)v[c].y) : (T)v[c].y;
      }
    }
  }
}

// Gaussian beams (AP_GAUSS, AP_FLYING_CF) in float-float arithmetic, three or
// more components: exp(-(x^2 + y^2) q / w0^2) is a product of an x and a y
// factor, so with z fixed every node value is
//   v = Re(X P) + x Re(X Q),
// X the complex x factor of the node's column and P, Q complex numbers of its
// row (Q only for the longitudinal components).  A warp takes slabs of one z
// index, 128 columns and up to 32 rows: each lane keeps the x factors of its
// four columns (whole and half node, both z levels) in registers, lane l makes
// the 16 coefficients of row l, and the rows then cost 18 FP32 operations per
// node and no special functions.  The rows of all column blocks are divided
// evenly over one resident wave of warps (a warp's share may span slabs).  Per-node evaluation took 122 instructions
// and 18 special-function operations and was bound by latency at half the
// store bandwidth; this is bound by the stores (256^3, 402 MB: 88.5 -> 72.6 us, 5.5 TB/s).  The
// factors are made with the accurate library functions (each is used by tens of nodes), so that their
// product is as good as one approximate exponential was.
// VEC: four consecutive columns per lane and 16-byte accesses (float rows aligned
// to 16 bytes); otherwise columns 32 apart, stores only.  slab_wins says which
// shapes come here.
constexpr int kSlabCols = 128;
constexpr int kSlabRows = 32;  // at most; one lane makes one row's coefficients

// e^{-a q} with a >= 0 a real number times 1/w0^2: 2^-(a log2e Re q), angle -a Im q
__device__ __forceinline__ Cx<float> beam_factor(float a, Cx<float> q, float turn) {
  const float mag = exp2f(-(a * q.re) * (float)kLog2e);
  float s, c;
  // the angle in half turns, reduced by sincospif
  sincospif(2.0f * fmaf(-a * q.im, kInvTwoPi, turn), &s, &c);
  return {mag * c, mag * s};
}

template <int KIND, typename T, bool VEC>
__global__ void __launch_bounds__(256) nodes_slab_kernel(const __grid_constant__ PulseHead<float> P,
                                                         const __grid_constant__ NodeArgs a) {
  __shared__ float4 s_row[8][kSlabRows][4];
  unsigned want = 0u;
  for (int q = 0; q < a.n_comp; ++q) want |= 1u << a.comp[q];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nxc = (a.nx + kSlabCols - 1) / kSlabCols;
  const long long total = (long long)nxc * a.nz * a.ny;  // rows of column blocks, (k, block, j) in order
  const long long n_warps = (long long)gridDim.x * 8, wid = (long long)blockIdx.x * 8 + warp;
  const long long per = total / n_warps, more = total - per * n_warps;
  long long row = wid * per + (wid < more ? wid : more);
  const long long row_end = row + per + (wid < more ? 1 : 0);
  TimeBase<AP_FP32_PHASEFF> tb;
  tb.init(P, a.t, 0.0);
  const StepFF st = tb.at(0);
  constexpr int kStep = VEC ? 1 : 32;
  long long kb_cur = -1;
  int k = 0, i0 = 0;
  Cx<float> q[2];            // of the two z levels
  float amp[2], turn[2];     // envelope and carrier
  float xw[4];
  Cx<float> X[2][2][4];      // x factors of the lane's columns: [z level][whole, half]
  while (row < row_end) {
    const long long kb = row / a.ny;
    const int j0 = (int)(row - kb * a.ny);
    int nj = a.ny - j0 < kSlabRows ? a.ny - j0 : kSlabRows;
    if (nj > row_end - row) nj = (int)(row_end - row);
    row += nj;
    if (kb != kb_cur) {
      kb_cur = kb;
      k = (int)(kb / nxc);
      i0 = (int)(kb - (long long)k * nxc) * kSlabCols + (VEC ? 4 * lane : lane);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        Pos<AP_FP32_PHASEFF> pos;
        pos.x = FF{0.0f, 0.0f};
        pos.y = FF{0.0f, 0.0f};
        pos.z = node_coord_ff((float)k + (h ? 0.5f : 0.0f), a.lo_hi[2], a.lo_lo[2], a.d_hi[2], a.d_lo[2]);
        const BeamZ<float> b = gauss_z<KIND == AP_FLYING_CF>(P, local_coords<AP_FP32_PHASEFF>(P, st, pos));
        q[h] = b.q;
        amp[h] = b.amp_mul * exp2f(b.l2);
        turn[h] = b.psi * kInvTwoPi;
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const float fi = (float)(i0 + m * kStep);
        xw[m] = fmaf(fi, a.d_hi[0], a.lo_hi[0]);
        const float xh = fmaf(fi + 0.5f, a.d_hi[0], a.lo_hi[0]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          X[h][0][m] = beam_factor(xw[m] * xw[m] * P.inv_w0sq, q[h], 0.0f);
          X[h][1][m] = beam_factor(xh * xh * P.inv_w0sq, q[h], 0.0f);
        }
      }
    }
    // row coefficients of row j0 + lane
    if (lane < nj) {
      const float fj = (float)(j0 + lane);
      const float y[2] = {fmaf(fj, a.d_hi[1], a.lo_hi[1]), fmaf(fj + 0.5f, a.d_hi[1], a.lo_hi[1])};
      auto row = [&](int h, int o) {  // U less its x factor
        const Cx<float> f = beam_factor(y[o] * y[o] * P.inv_w0sq, q[h], turn[h]);
        return cscale(cmul(q[h], f), amp[h]);
      };
      const float g = -2.0f * P.inv_w0sq, ce = P.lon ? P.lonE * g : 0.0f, cb = P.lon ? P.bratio * P.lonB * g : 0.0f;
      const float br = P.bratio;
      const Cx<float> u00 = row(0, 0), u01 = row(0, 1), u10 = row(1, 0), u11 = row(1, 1);
      const Cx<float> wz = cmul(q[1], u10), wb = cmul(q[0], u01);  // W of Ez and of Bz
      // E = Re[p U], B_perp = br Re[(z x p) U]; E_z = ce Im[(p_x x + p_y y) W],
      // B_z = cb Im[(p_x y - p_y x) W]; Im w = Re(-i w)
      const Cx<float> px{P.px_re, P.px_im}, py{P.py_re, P.py_im};
      auto mi = [](Cx<float> w, float s) { return Cx<float>{s * w.im, -s * w.re}; };
      const Cx<float> p0 = cmul(px, u00), p1 = cmul(py, u01), p3 = cscale(cmul(py, u11), -br), p4 = cscale(cmul(px, u10), br);
      const Cx<float> q2 = mi(cmul(px, wz), ce), p2 = mi(cmul(py, wz), ce * y[0]);
      const Cx<float> q5 = mi(cmul(py, wb), -cb), p5 = mi(cmul(px, wb), cb * y[1]);
      float4 *r = s_row[warp][lane];
      r[0] = make_float4(p0.re, p0.im, p1.re, p1.im);
      r[1] = make_float4(p2.re, p2.im, q2.re, q2.im);
      r[2] = make_float4(p3.re, p3.im, p4.re, p4.im);
      r[3] = make_float4(p5.re, p5.im, q5.re, q5.im);
    }
    __syncwarp();
    long long at = ((long long)k * a.ny + j0) * a.nx + i0;
    for (int r = 0; r < nj; ++r, at += a.nx) {
      const float4 c0 = s_row[warp][r][0], c1 = s_row[warp][r][1], c2 = s_row[warp][r][2], c3 = s_row[warp][r][3];
      float v[6][4];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        auto re = [](Cx<float> x, float cr, float ci) { return fmaf(x.re, cr, -(x.im * ci)); };
        const Cx<float> w0 = X[0][0][m], h0 = X[0][1][m], w1 = X[1][0][m], h1 = X[1][1][m];
        const float xh = fmaf((float)(i0 + m * kStep) + 0.5f, a.d_hi[0], a.lo_hi[0]);
        v[0][m] = re(h0, c0.x, c0.y);
        v[1][m] = re(w0, c0.z, c0.w);
        v[2][m] = fmaf(xw[m], re(w1, c1.z, c1.w), re(w1, c1.x, c1.y));
        v[3][m] = re(w1, c2.x, c2.y);
        v[4][m] = re(h1, c2.z, c2.w);
        v[5][m] = fmaf(xh, re(h0, c3.z, c3.w), re(h0, c3.x, c3.y));
      }
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        if (!((want >> c) & 1u)) continue;
        T *f = static_cast<T *>(a.f[c]) + at;
        if constexpr (VEC) {
          if (i0 < a.nx) {
            float4 *f4 = reinterpret_cast<float4 *>(f);
            float4 o = make_float4(v[c][0], v[c][1], v[c][2], v[c][3]);
            if (a.accumulate) {
              const float4 p = *f4;
              o = make_float4(p.x + o.x, p.y + o.y, p.z + o.z, p.w + o.w);
            }
            *f4 = o;
          }
        } else {
#pragma unroll
          for (int m = 0; m < 4; ++m)
            if (i0 + 32 * m < a.nx) f[32 * m] = (T)v[c][m];
        }
      }
    }
    __syncwarp();
  }
}

// One warp writes the value v along a row of n elements (store, or add to
// what the row holds, rounding once to T): a scalar head up to the first
// 16-byte boundary, then 16-byte vector stores, then a scalar tail.  The row
// is aligned to sizeof(T) (checked on the host), so the head is at most
// 16 / sizeof(T) - 1 elements.
template <typename T, typename W>
__device__ __forceinline__ void row_put(T *__restrict__ row, int n, W v, bool acc, int lane) {
  using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
  constexpr int kVe = 16 / (int)sizeof(T);
  int head = (int)(((16u - ((unsigned)reinterpret_cast<uintptr_t>(row) & 15u)) & 15u) / sizeof(T));
  if (head > n) head = n;
  const int nv = (n - head) / kVe;
  const int tail = head + nv * kVe;
  V *rv = reinterpret_cast<V *>(row + head);
  // two separate loops: the store path must not read the row
  if (acc) {
    if (lane < head) row[lane] = (T)((W)row[lane] + v);
    for (int i = lane; i < nv; i += 32) {
      V x = rv[i];
      if constexpr (sizeof(T) == 4) {
        x.x = (T)((W)x.x + v); x.y = (T)((W)x.y + v); x.z = (T)((W)x.z + v); x.w = (T)((W)x.w + v);
      } else {
        x.x = (T)((W)x.x + v); x.y = (T)((W)x.y + v);
      }
      rv[i] = x;
    }
    for (int i = tail + lane; i < n; i += 32) row[i] = (T)((W)row[i] + v);
  } else {
    const T vt = (T)v;
    V x;
    if constexpr (sizeof(T) == 4) x = make_float4(vt, vt, vt, vt);
    else x = make_double2(vt, vt);
    if (lane < head) row[lane] = vt;
#pragma unroll 4
    for (int i = lane; i < nv; i += 32) rv[i] = x;
    for (int i = tail + lane; i < n; i += 32) row[i] = vt;
  }
}

// Whether a Gaussian beam's nodes go in slabs (nodes_slab_kernel) or row by row
// (nodes_row_pair_kernel, two columns of 32 per pass).  A slab pays its set-up, 16
// exponentials and sines per lane, for each z index and 128 columns, and does the
// work of 128 columns also where fewer are left; without 16-byte accesses
// (double nodes, unaligned rows) it stores and sums by single elements, where
// the row kernel is as wide; and where rows end inside a 32-byte sector, the
// sectors at the slabs' edges are written in two parts far apart in time, which
// tells once the arrays pass the L2 cache (4e6 nodes are 96 of 129 MB).
// Measured, slabs / rows, us (1.7e7 nodes where ny allows):
//   float nodes, stored: nx 256 78 / 93, with ny = 1, 2, 3 97 / 59, 107 / 97, 84 / 96;
//     nx 64 with ny = 3, 5, 8 67 / 53, 65 / 61, 55 / 61; nx 160 with ny = 3, 4 69 / 65, 61 /
//     63; unaligned, nx 33 with ny = 6, 12 99 / 84, 100 / 100; rows that end inside a
//     sector: nx 300 129 / 100, nx 180 138 / 100, nx 250 123 / 108, with ny = 3 99 / 110,
//     in L2: 132 x 95 x 171 23 / 31, 164 x 45 x 97 16.5 / 19.4;
//   float nodes, summed: nx 256 229 / 397, nx 64 360 / 388, with ny = 1 61 / 44, nx 32
//     656 / 427; unaligned, nx 250 679 / 400;
//   double nodes, stored: nx 64 188 / 102, nx 160 156 / 122, nx 250 207 / 191, nx 256
//     180 / 182, nx 1000 182 / 201; summed: nx 256 717 / 534.
inline bool slab_wins(const NodeArgs &a, bool vec) {
  const int slabs = (a.nx + kSlabCols - 1) / kSlabCols, pairs = (a.nx + 63) / 64;
  const bool full = pairs == 2 * slabs;
  if (a.f64) return !a.accumulate && full && a.nx % 4 == 0 && a.ny >= 4;
  if (a.accumulate) return vec && (pairs > slabs || (a.nx == 64 && a.ny > 2));
  if (slabs > 1 && a.nx % 8 != 0 && (double)a.nx * a.ny * a.nz >= 4e6) return full && a.ny >= 3 && a.ny < 6;
  if (!vec && pairs == slabs) return a.ny >= 12;
  return (long long)a.ny * pairs >= 6LL * slabs;
}

// Plane waves (Eqs. plane_func, plane_b) depend on z and t only.  A row of
// nx nodes (fixed y, z) holds two z positions: the whole node z_k (Ex, Ey,
// Bz) and the half node z_k + dz/2 (Ez, Bx, By).  A warp evaluates the field
// (every lane computes the same value) and streams each requested component
// along its rows with 16-byte stores, so for nx >= 32 the kernel is bound by the
// stores, not the arithmetic.
// RUNS: each warp takes a contiguous run of rows and evaluates once per z index; otherwise rows are dealt out in turn, one
// evaluation per row.  plane_runs says which, with the times of both.
template <int PREC, typename T, bool RUNS>
__global__ void __launch_bounds__(256) nodes_plane_kernel(const __grid_constant__ Pulse<Real<PREC>> P,
                                                          const __grid_constant__ NodeArgs a) {
  using R = Real<PREC>;
  using W = typename std::conditional<(sizeof(T) > sizeof(R)), T, R>::type;
  bool need[2] = {false, false};  // whole, half
  for (int i = 0; i < a.n_comp; ++i) {
    const int c = a.comp[i];
    if (c == 2 || c == 3 || c == 4) need[1] = true;
    else need[0] = true;
  }
  const long long rows = (long long)a.ny * a.nz;
  const int lane = threadIdx.x & 31;
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  const long long wid = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  TimeBase<PREC> tb;
  tb.init(P, a.t, 0.0);
  const typename TimeBase<PREC>::Step st = tb.at(0);
  auto eval = [&](int k, R v[6]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (!need[h]) continue;
      const float oz = h ? 0.5f : 0.0f;
      Pos<PREC> pos;
      if constexpr (PREC == AP_FP32_PHASEFF) {
        pos.x = FF{0.0f, 0.0f};
        pos.y = FF{0.0f, 0.0f};
        pos.z = node_coord_ff((float)k + oz, a.lo_hi[2], a.lo_lo[2], a.d_hi[2], a.d_lo[2]);
      } else {
        pos.load(0.0, 0.0, fma((double)k + oz, a.d[2], a.lo[2]));
      }
      Local<R> L = local_coords<PREC>(P, st, pos);
      R E[3], B[3];
      node_values<AP_PLANE, PREC>(P, L, a.current, E, B);
      if (h == 0) {
        v[0] = E[0];
        v[1] = E[1];
        v[5] = B[2];
      } else {
        v[2] = E[2];
        v[3] = B[0];
        v[4] = B[1];
      }
    }
  };
  auto put = [&](long long r, const R v[6]) {
    for (int i = 0; i < a.n_comp; ++i) {
      const int c = a.comp[i];
      const R val = c == 0 ? v[0] : c == 1 ? v[1] : c == 2 ? v[2] : c == 3 ? v[3] : c == 4 ? v[4] : v[5];
      row_put<T, W>(static_cast<T *>(a.f[c]) + r * a.nx, a.nx, (W)val, a.accumulate != 0, lane);
    }
  };
  if constexpr (RUNS) {
    const long long per = (rows + warps - 1) / warps;
    const long long r0 = wid * per, r1 = r0 + per < rows ? r0 + per : rows;
    int kcur = -1;
    R v[6] = {R(0), R(0), R(0), R(0), R(0), R(0)};
    for (long long r = r0; r < r1; ++r) {
      const int k = (int)(r / a.ny);
      if (k != kcur) eval(k, v);
      kcur = k;
      put(r, v);
    }
  } else {
    for (long long r = wid; r < rows; r += warps) {
      R v[6] = {R(0), R(0), R(0), R(0), R(0), R(0)};
      eval((int)(r / a.ny), v);
      put(r, v);
    }
  }
}

// Whether plane-wave rows go in runs (see nodes_plane_kernel).  Runs save
// evaluations, which counts where one is in double or the rows are short, and
// fill the warps where there are about as many rows as warps; dealt out in turn,
// neighbouring rows are written at the same time, which counts for many wide
// rows, above all where they end inside a 128-byte line.  Measured, rows in turn /
// in runs, all components, us:
//   float nodes, stored: 250 x 133 x 251 48.8 / 53.4, 1000 x 140 x 140 83.5 / 91.3,
//     300 x 250 x 200 69.1 / 76.7, but 256 x 136 x 87 (1.2 rows per warp) 33.5 / 32.0,
//     400 x 136 x 87 37.8 / 33.7, 700 x 136 x 87 again 42.9 / 47.9, 64 x 512 x 300 139 / 96;
//   float nodes, summed: 400 x 250 x 200 89.2 / 95.8, 288 x 250 x 200 75.1 / 78.5, 250 x 250 x
//     200 68.8 / 60.2, 700 x 136 x 87 40.1 / 36.4;
//   double nodes: 256^3 136 / 130, summed 159 / 139, 1000 x 140 x 140 156 / 166, summed
//     160 / 146; evaluated in double 256^3 475 / 138.
inline bool plane_runs(int precision, const NodeArgs &a) {
  if (precision != AP_FP32_PHASEFF || a.nx < 192) return true;
  const long long rows = (long long)a.ny * a.nz, warps = 64LL * a.sm_count;
  if (a.f64) return a.accumulate || (a.nx * sizeof(double)) % 128 == 0;
  if (a.accumulate) return a.nx < 288 || rows < 4 * warps;
  return a.nx < 640 && rows < 2 * warps;
}

template <int KIND, int PREC>
int launch_nodes_t(const Pulse<Real<PREC>> &P, const NodeArgs &a, void *stream) {
  const long long total = (long long)a.nx * a.ny * a.nz;
  const int block = 256;
  if constexpr (KIND == AP_PLANE) {
    if (a.nx >= 32) {
      const long long rows = (long long)a.ny * a.nz;
      long long gx = (rows + 7) / 8;  // 8 warps (rows) per block, every component of a row
      const long long cap = (long long)a.sm_count * 8;
      if (gx > cap) gx = cap;
      if (gx < 1) gx = 1;
      const dim3 grid((unsigned)gx, 1u);
      cudaStream_t s = static_cast<cudaStream_t>(stream);
      const bool runs = plane_runs(PREC, a);
      auto kern = a.f64 ? (runs ? nodes_plane_kernel<PREC, double, true> : nodes_plane_kernel<PREC, double, false>)
                        : (runs ? nodes_plane_kernel<PREC, float, true> : nodes_plane_kernel<PREC, float, false>);
      kern<<<grid, block, 0, s>>>(P, a);
      return cudaGetLastError() == cudaSuccess ? AP_OK : AP_ERR_CUDA;
    }
  }
  if (a.n_comp >= 3 && a.nx >= 32) {
    const long long rows = (long long)a.ny * a.nz;
    long long gx = (rows + 7) / 8;  // 8 warps (rows) per block
    const long long cap = (long long)a.sm_count * 8;
    if (gx > cap) gx = cap;
    if (gx < 1) gx = 1;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if constexpr (PREC == AP_FP32_PHASEFF && KIND != AP_PLANE) {
      if constexpr (KIND == AP_GAUSS || KIND == AP_FLYING_CF) {
        bool vec = !a.f64 && a.nx % 4 == 0;
        for (int i = 0; i < a.n_comp; ++i) vec = vec && (reinterpret_cast<uintptr_t>(a.f[a.comp[i]]) & 15u) == 0;
        if (slab_wins(a, vec)) {
          auto kern = a.f64 ? nodes_slab_kernel<KIND, double, false>
                      : vec ? nodes_slab_kernel<KIND, float, true> : nodes_slab_kernel<KIND, float, false>;
          // one resident wave, and at least four rows for each warp's set-up
          const long long units = (long long)((a.nx + kSlabCols - 1) / kSlabCols) * rows;
          long long gp = (long long)a.sm_count * occupancy_blocks(kern, block, 0);
          if (gp > (units + 31) / 32) gp = (units + 31) / 32;
          kern<<<(unsigned)gp, block, 0, s>>>(P, a);
          return cudaGetLastError() == cudaSuccess ? AP_OK : AP_ERR_CUDA;
        }
      }
      {  // two nodes per lane, packed; one resident wave of blocks, each warp a contiguous run of rows
        auto kern = a.f64 ? nodes_row_pair_kernel<KIND, double> : nodes_row_pair_kernel<KIND, float>;
        long long gp = (long long)a.sm_count * occupancy_blocks(kern, block, 0);
        if (gp > (rows + 7) / 8) gp = (rows + 7) / 8;
        if (gp < 1) gp = 1;
        kern<<<(unsigned)gp, block, 0, s>>>(P, a);
        return cudaGetLastError() == cudaSuccess ? AP_OK : AP_ERR_CUDA;
      }
    }
    if (a.f64) nodes_row_kernel<KIND, PREC, double><<<(unsigned)gx, block, 0, s>>>(P, a);
    else nodes_row_kernel<KIND, PREC, float><<<(unsigned)gx, block, 0, s>>>(P, a);
    return cudaGetLastError() == cudaSuccess ? AP_OK : AP_ERR_CUDA;
  }
  if (a.n_comp >= 3) {
    long long gx = (total + block - 1) / block;
    const long long cap = (long long)a.sm_count * 8;
    if (gx > cap) gx = cap;
    if (gx < 1) gx = 1;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (a.f64) nodes_all_kernel<KIND, PREC, double><<<(unsigned)gx, block, 0, s>>>(P, a);
    else nodes_all_kernel<KIND, PREC, float><<<(unsigned)gx, block, 0, s>>>(P, a);
    return cudaGetLastError() == cudaSuccess ? AP_OK : AP_ERR_CUDA;
  }
  long long gx = (total + block - 1) / block;
  // enough resident threads per component to fill the GPU, then grid-stride
  long long cap = ((long long)a.sm_count * 8 + a.n_comp - 1) / a.n_comp;
  if (gx > cap) gx = cap;
  if (gx < 1) gx = 1;
  const dim3 grid((unsigned)gx, (unsigned)a.n_comp);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (a.f64) nodes_kernel<KIND, PREC, double><<<grid, block, 0, s>>>(P, a);
  else nodes_kernel<KIND, PREC, float><<<grid, block, 0, s>>>(P, a);
  return cudaGetLastError() == cudaSuccess ? AP_OK : AP_ERR_CUDA;
}

template <int KIND, int PREC, int GRID, int NP = 1>
int launch_batch_t(const Pulse<Real<PREC>> *sets, const BatchArgs &ba, void *stream) {
  auto kern = batch_kernel<KIND, PREC, GRID, NP>;
  constexpr bool kBeam = KIND == AP_PLANE || KIND == AP_GAUSS || KIND == AP_FLYING_CF;
  if constexpr (PREC == AP_FP32_PHASEFF && NP == 2 &&
                (GRID == kGridCells || GRID == kGridCellsMix || (GRID == kGridNone && kBeam)))
    kern = batch_kernel_pair_minb<KIND, GRID>;
  const int block = ba.base.shape.block;
  const size_t head = push_smem_head<PREC, GRID, NP>(block);
  const size_t smem = head + (size_t)(ba.n_sets + 1) * sizeof(long long);
  if (set_smem<PREC, GRID, NP>(kern, smem) != AP_OK) return AP_ERR_CUDA;
  int per_sm = ba.base.shape.blocks_per_sm > 0 ? ba.base.shape.blocks_per_sm
                                                : occupancy_blocks(kern, block, smem);
  const int grid = ba.base.sm_count * per_sm;
  kern<<<grid, block, smem, static_cast<cudaStream_t>(stream)>>>(sets, ba, (unsigned)head);
  return cudaGetLastError() == cudaSuccess ? AP_OK : AP_ERR_CUDA;
}

// grid mode of a call: none, corners, or (float kernels) per-cell coefficients
// Whether a float-float call runs two particles per thread: requested in the
// launch shape, and a grid mode the two-particle kernels have.
inline bool pair_mode(const PushArgs &a) {
  return a.shape.pairs && (!a.grid_on || a.grid.cells);
}

template <int KIND, int PREC>
int launch_push_mode(const Pulse<Real<PREC>> &P, const PushArgs &a, void *stream) {
  if constexpr (PREC == AP_FP32_PHASEFF) {
    if (pair_mode(a))
      return !a.grid_on                 ? launch_push_ff_t<KIND, kGridNone, 2>(P, a, stream)
             : a.shape.grid_cache == 2 ? launch_push_ff_t<KIND, kGridCellsMix, 2>(P, a, stream)
             : a.shape.grid_cache      ? launch_push_ff_t<KIND, kGridCellsReg, 2>(P, a, stream)
                                       : launch_push_ff_t<KIND, kGridCells, 2>(P, a, stream);
    if (!a.grid_on) return launch_push_ff_t<KIND, kGridNone, 1>(P, a, stream);
    if (!a.grid.cells) return launch_push_ff_t<KIND, kGridNodes, 1>(P, a, stream);
    return a.shape.grid_cache ? launch_push_ff_t<KIND, kGridCellsReg, 1>(P, a, stream)
                              : launch_push_ff_t<KIND, kGridCells, 1>(P, a, stream);
  } else {
    if (!a.grid_on) return launch_push_t<KIND, PREC, kGridNone>(P, a, stream);
    if constexpr (PREC != AP_FP64) {
      if (a.grid.cells)
        return a.shape.grid_cache ? launch_push_t<KIND, PREC, kGridCellsReg>(P, a, stream)
                                  : launch_push_t<KIND, PREC, kGridCells>(P, a, stream);
    }
    return launch_push_t<KIND, PREC, kGridNodes>(P, a, stream);
  }
}

template <int KIND, int PREC>
int launch_batch_mode(const Pulse<Real<PREC>> *sets, const BatchArgs &ba, void *stream) {
  if constexpr (PREC == AP_FP32_PHASEFF) {
    if (pair_mode(ba.base))
      return !ba.base.grid_on ? launch_batch_t<KIND, PREC, kGridNone, 2>(sets, ba, stream)
             : ba.base.shape.grid_cache == 2 ? launch_batch_t<KIND, PREC, kGridCellsMix, 2>(sets, ba, stream)
             : ba.base.shape.grid_cache      ? launch_batch_t<KIND, PREC, kGridCellsReg, 2>(sets, ba, stream)
                                             : launch_batch_t<KIND, PREC, kGridCells, 2>(sets, ba, stream);
  }
  if (!ba.base.grid_on) return launch_batch_t<KIND, PREC, kGridNone>(sets, ba, stream);
  if constexpr (PREC != AP_FP64) {
    if (ba.base.grid.cells)
      return ba.base.shape.grid_cache ? launch_batch_t<KIND, PREC, kGridCellsReg>(sets, ba, stream)
                                      : launch_batch_t<KIND, PREC, kGridCells>(sets, ba, stream);
  }
  return launch_batch_t<KIND, PREC, kGridNodes>(sets, ba, stream);
}

}  // namespace apt

// Per-kind launchers: dispatch on precision and grid.
#define APT_DEFINE_KIND(K, KID)                                                                   \
  namespace apt {                                                                                 \
  int launch_push_##K(int precision, const Pulse<double> &pd, const Pulse<float> &pf,             \
                      const PushArgs &a, void *stream) {                                          \
    switch (precision) {                                                                          \
      case AP_FP64:                                                                               \
        return launch_push_mode<KID, AP_FP64>(pd, a, stream);                                     \
      case AP_FP32_PHASE64:                                                                       \
        return launch_push_mode<KID, AP_FP32_PHASE64>(pf, a, stream);                             \
      case AP_FP32_PHASEFF:                                                                       \
        return launch_push_mode<KID, AP_FP32_PHASEFF>(pf, a, stream);                             \
      default:                                                                                    \
        return AP_ERR_ARG;                                                                        \
    }                                                                                             \
  }                                                                                               \
  int launch_eval_##K(int precision, const Pulse<double> &pd, const Pulse<float> &pf,             \
                      const EvalArgs &a, void *stream) {                                          \
    switch (precision) {                                                                          \
      case AP_FP64: return launch_eval_t<KID, AP_FP64>(pd, a, stream);                            \
      case AP_FP32_PHASE64: return launch_eval_t<KID, AP_FP32_PHASE64>(pf, a, stream);            \
      case AP_FP32_PHASEFF: return launch_eval_t<KID, AP_FP32_PHASEFF>(pf, a, stream);            \
      default: return AP_ERR_ARG;                                                                 \
    }                                                                                             \
  }                                                                                               \
  int launch_nodes_##K(int precision, const Pulse<double> &pd, const Pulse<float> &pf,            \
                       const NodeArgs &a, void *stream) {                                         \
    switch (precision) {                                                                          \
      case AP_FP64: return launch_nodes_t<KID, AP_FP64>(pd, a, stream);                           \
      case AP_FP32_PHASE64: return launch_nodes_t<KID, AP_FP32_PHASE64>(pf, a, stream);           \
      case AP_FP32_PHASEFF: return launch_nodes_t<KID, AP_FP32_PHASEFF>(pf, a, stream);           \
      default: return AP_ERR_ARG;                                                                 \
    }                                                                                             \
  }                                                                                               \
  int launch_batch_##K(int precision, const Pulse<double> *dpd, const Pulse<float> *dpf,          \
                       const BatchArgs &a, void *stream) {                                        \
    switch (precision) {                                                                          \
      case AP_FP64:                                                                               \
        return launch_batch_mode<KID, AP_FP64>(dpd, a, stream);                                   \
      case AP_FP32_PHASE64:                                                                       \
        return launch_batch_mode<KID, AP_FP32_PHASE64>(dpf, a, stream);                           \
      case AP_FP32_PHASEFF:                                                                       \
        return launch_batch_mode<KID, AP_FP32_PHASEFF>(dpf, a, stream);                           \
      default:                                                                                    \
        return AP_ERR_ARG;                                                                        \
    }                                                                                             \
  }                                                                                               \
  }
