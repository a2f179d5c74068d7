// pair_f64.cuh -- per (track, antenna) arithmetic of the FP64 path: the plain
// formulas of the two formalisms (§1) and the straight-line propagator (§2) in
// FP64, in the order of their definitions (one exception: the ZHS factor
// K_A/(R |D_m| dt) is formed once per interval rather than once per bin), and for
// the one-bin deposit in the plain media with fewer and fused operations
// (OpsF64Plain, which the adjoint's geometry and bins are taken from).  This
// translation unit is compiled without FMA contraction so that every operation
// rounds as written.
#pragma once

#include "kernels.cuh"

namespace c8r {

#define TF(f) T[(f) * kTileT + l]

struct EndpointEvalD {
  GeoD g0, g1, gm;
  double V0[3], V1[3], Vm[3];
  double D0, D1, Dm;
  double E0, E1, Em;
  int branch;
  double ua, ub;
  bool valid;
};

__device__ __forceinline__ void field_vec_f64(const double b[3], const GeoD& g, double V[3], double& D) {
  const double c = b[0] * g.rh[0] + b[1] * g.rh[1] + b[2] * g.rh[2];
  V[0] = c * g.rh[0] - b[0];
  V[1] = c * g.rh[1] - b[1];
  V[2] = c * g.rh[2] - b[2];
  D = 1.0 - g.n_src * c;
}

// stop_near: a near-Cherenkov pair stops after the branch decision (branch 1,
// valid false), for a caller that evaluates those pairs in a later pass
__device__ __forceinline__ void endpoint_eval_f64(const double* T, int l, const AntRec& A, const MedParams& M,
                                                  EndpointEvalD& e, bool stop_near = false) {
  e.valid = false;
  e.branch = 0;
  const double b[3] = {TF(fd::BX), TF(fd::BY), TF(fd::BZ)};
  const double x0 = TF(fd::X0), y0 = TF(fd::Y0), z0 = TF(fd::Z0);
  const double x1 = TF(fd::X1), y1 = TF(fd::Y1), z1 = TF(fd::Z1);
  const double t0 = TF(fd::T0), t1 = TF(fd::T1);
  e.E0 = TF(fd::E0);
  e.E1 = TF(fd::E1);
  e.Em = TF(fd::EM);
  geo_f64(M, A, x0, y0, z0, e.E0, e.g0);
  geo_f64(M, A, x1, y1, z1, e.E1, e.g1);
  if (e.g0.R == 0.0 || e.g1.R == 0.0) return;
  field_vec_f64(b, e.g0, e.V0, e.D0);
  field_vec_f64(b, e.g1, e.V1, e.D1);
  if (fmin(fabs(e.D0), fabs(e.D1)) >= M.eps_Cd) {
    e.branch = 0;
    e.ua = arrival_f64(M, e.g0, t0, A.t_ref);
    e.ub = arrival_f64(M, e.g1, t1, A.t_ref);
    e.valid = true;
    return;
  }
  e.branch = 1;
  if (stop_near) return;
  geo_f64(M, A, 0.5 * (x0 + x1), 0.5 * (y0 + y1), 0.5 * (z0 + z1), e.Em, e.gm);
  if (e.gm.R == 0.0) return;
  field_vec_f64(b, e.gm, e.Vm, e.Dm);
  const double dte = t1 - t0;
  const double tm = 0.5 * (t0 + t1);
  const double tarr_rel = (tm - A.t_ref) + e.gm.n_avg * e.gm.R * M.inv_c_ns;
  e.ua = (tarr_rel - e.Dm * dte / 2.0) / M.dt_ns;
  e.ub = (tarr_rel + e.Dm * dte / 2.0) / M.dt_ns;
  e.valid = true;
}

// Linear (two-bin) deposit (reading LD), in FP64: a deposit arriving at u
// covers [u - 1/2, u + 1/2]; bin k0 = floor(u - 1/2) receives
// (k0 + 1) - (u - 1/2) of it and bin k0 + 1 receives (u + 1/2) - (k0 + 1).
template <class Sink>
__device__ __forceinline__ void dep_lin_f64(Sink& out, int N, double u, double x, double y, double z) {
  const double k0 = floor(u - 0.5);
  const double w0 = (k0 + 1.0) - (u - 0.5), w1 = (u + 0.5) - (k0 + 1.0);
  if (k0 >= 0.0 && k0 < (double)N && w0 > 0.0) out.dep((int)k0, x * w0, y * w0, z * w0);
  if (k0 + 1.0 >= 0.0 && k0 + 1.0 < (double)N && w1 > 0.0) out.dep((int)k0 + 1, x * w1, y * w1, z * w1);
}

// the share of bin k of a deposit arriving at u (the tent max(0, 1 - |u - k - 1/2|))
__device__ __forceinline__ double lin_share_f64(double u, double k) {
  const double lo = fmax(u - 0.5, k), hi = fmin(u + 0.5, k + 1.0);
  return hi > lo ? hi - lo : 0.0;
}

// integral of that share over u in [a, b]: the tent is linear between its knots
// k - 1/2, k + 1/2, k + 3/2, so each piece is its length times the tent at its
// middle
__device__ __forceinline__ double lin_share_integral_f64(double a, double b, double k) {
  double sum = 0.0;
  for (int p = 0; p < 2; ++p) {
    const double lo = fmax(a, k - 0.5 + p), hi = fmin(b, k + 0.5 + p);
    if (hi > lo) sum += (hi - lo) * lin_share_f64(0.5 * (lo + hi), k);
  }
  return sum;
}

// dL/dtrace seen by a unit deposit at u, and its rate of change with u
__device__ __forceinline__ void gather_lin_f64(const Acc4D* G, int N, double u, double g[3], double slope[3]) {
  const double k0 = floor(u - 0.5);
  const double w0 = (k0 + 1.0) - (u - 0.5), w1 = (u + 0.5) - (k0 + 1.0);
  const Acc4D zero{0.0, 0.0, 0.0, 0.0};
  const Acc4D g0 = (k0 >= 0.0 && k0 < (double)N) ? G[(int)k0] : zero;
  const Acc4D g1 = (k0 + 1.0 >= 0.0 && k0 + 1.0 < (double)N) ? G[(int)k0 + 1] : zero;
  g[0] = w0 * g0.x + w1 * g1.x;
  g[1] = w0 * g0.y + w1 * g1.y;
  g[2] = w0 * g0.z + w1 * g1.z;
  slope[0] = g1.x - g0.x;
  slope[1] = g1.y - g0.y;
  slope[2] = g1.z - g0.z;
}

// a track of a staged tile: the FP64 path reads its fields where it needs them
struct TrackD {
  const double* T;
  int l;
  double q;
};

template <int FORM>
struct OpsF64Plain;

template <int FORM, bool LIN = false>
struct OpsF64 {
  using acc_t = double;
  using Track = TrackD;
  static constexpr int kPrec = C8R_FP64;
  static constexpr int kTileBytes = kTileBytesF64;
  static constexpr int kMinBlocks = 4;
  // Endpoint (one-bin deposit): the near-Cherenkov pairs (about one in ten on a
  // shower, in most warps) are set aside by the main pass and evaluated
  // together afterwards, so that the midpoint form's FP64 arithmetic runs in
  // full warps instead of holding the other lanes of nearly every warp.  The
  // arithmetic of each pair is the same either way.  (The adjoint, adj_main,
  // evaluates every pair in its main pass; its set-aside lists stay empty.)
  static constexpr bool kDefers = FORM == C8R_ENDPOINT && !LIN;
  static constexpr bool kFastBins = false;
  static constexpr int kBwdMinBlocks = 2;
  static constexpr int kBwdGridBlocks = 2;
  static constexpr int kAccRows = 1;      // no box deposits

  using Ant = AntRec;
  static __device__ __forceinline__ void stage_ant(AntRec* p, const AntRec& A, const MedParams&) { *p = A; }
  static __device__ __forceinline__ AntRec load_ant(const AntRec* p) { return *p; }

  static __device__ __forceinline__ void load(const void* Tv, int l, const MedParams&, TrackD& t) {
    t.T = static_cast<const double*>(Tv);
    t.l = l;
    t.q = t.T[fd::Q * kTileT + l];
  }
  static __device__ __forceinline__ bool live(const TrackD& t) { return t.q != 0.0; }
  // the adjoint's main pass: with the one-bin deposit (plain media only) the track
  // as the forward pass holds it
  using Plain = OpsF64Plain<FORM>;
  using MainTrack = std::conditional_t<LIN, TrackD, typename Plain::AdjTrack>;
  using FwdTrack = TrackD;
  using FwdAnt = AntRec;
  static constexpr int kFwdThreads = kTileT;
  static __device__ __forceinline__ void load_fwd(const void* Tv, int l, const MedParams& M, TrackD& t) {
    load(Tv, l, M, t);
  }
  struct MainGrad {
    double g[11];
  };
  static __device__ __forceinline__ void zero(MainGrad& m) {
#pragma unroll
    for (int k = 0; k < 11; ++k) m.g[k] = 0.0;
  }
  static __device__ __forceinline__ void collect(const MainGrad& m, double tg[11]) {
#pragma unroll
    for (int k = 0; k < 11; ++k) tg[k] = m.g[k];
  }
  static __device__ __forceinline__ void load_main(const void* Tv, int l, const MedParams& M, MainTrack& t) {
    if constexpr (LIN) {
      load(Tv, l, M, t);
    } else {
      t.T = Tv;
      t.l = l;
      Plain::load_fwd(Tv, l, M, t.t);
    }
  }
  template <class T, class = decltype(T::t)>
  static __device__ __forceinline__ bool live(const T& t) { return Plain::live(t.t); }
  template <class Sink>
  static __device__ __forceinline__ void pair(const TrackD& t, const AntRec& A, const MedParams& M, Sink& out) {
    if constexpr (FORM == C8R_ENDPOINT)
      endpoint(t.T, t.l, A, M, out);
    else
      zhs(t.T, t.l, A, M, out);
  }
  // main pass: every pair but (kDefers) the near-Cherenkov ones, returned as
  // kDeferPair with nothing deposited; pair_deferred evaluates those in full
  template <class Sink>
  static __device__ __forceinline__ int pair_main(const TrackD& t, const AntRec* p, const void*, int, const MedParams& M,
                                                  Sink& out) {
    const AntRec A = *p;
    if constexpr (kDefers) return endpoint(t.T, t.l, A, M, out, true);
    pair(t, A, M, out);
    return kDeferNone;
  }
  template <class Sink>
  static __device__ __forceinline__ void pair_deferred(const TrackD& t, const AntRec& A, const MedParams& M,
                                                       Sink& out) {
    if constexpr (kDefers) pair(t, A, M, out);
  }
  template <class Sink>
  static __device__ __forceinline__ void end_deferred(const void*, int, const AntRec&, const MedParams&, Sink&, int) {}
  template <bool ADJ = false>
  static __device__ __forceinline__ bool near_zero_fast(const void*, int, const AntRec&, const MedParams&) {
    return false;
  }

  // returns kDeferPair (nothing deposited) for a near-Cherenkov pair when
  // defer_near is set, kDeferNone otherwise
  template <class Sink>
  static __device__ __forceinline__ int endpoint(const double* T, int l, const AntRec& A, const MedParams& M,
                                                 Sink& out, bool defer_near = false) {
    const double q = TF(fd::Q);
    if (q == 0.0) return kDeferNone;
    const int N = M.n_bins;
    EndpointEvalD e;
    endpoint_eval_f64(T, l, A, M, e, defer_near);
    if (defer_near && e.branch == 1) return kDeferPair;
    if (!e.valid) return kDeferNone;
    out.rec(e.branch, e.ua, e.ub);
    const double K = q * kKendpoint;
    const double dt_s = M.dt_ns * 1e-9;
    if constexpr (LIN) {
      // reading LD
      if (e.branch == 0) {
        const double s0 = +K / (e.D0 * e.g0.R * dt_s);
        const double s1 = -K / (e.D1 * e.g1.R * dt_s);
        dep_lin_f64(out, N, e.ua, s0 * e.V0[0], s0 * e.V0[1], s0 * e.V0[2]);
        dep_lin_f64(out, N, e.ub, s1 * e.V1[0], s1 * e.V1[1], s1 * e.V1[2]);
        return kDeferNone;
      }
      const double Ja = floor(e.ua + 0.5), Jb = floor(e.ub + 0.5);
      if (Ja == Jb) {
        // both arrivals in one cell: the exact limit K (dt_e/dt) V/(R dt) into
        // bin J - 1 and its negative into bin J
        const double B = K * ((TF(fd::T1) - TF(fd::T0)) / M.dt_ns) / (e.gm.R * dt_s);
        if (Ja - 1.0 >= 0.0 && Ja - 1.0 < (double)N) out.dep((int)Ja - 1, B * e.Vm[0], B * e.Vm[1], B * e.Vm[2]);
        if (Ja >= 0.0 && Ja < (double)N) out.dep((int)Ja, -B * e.Vm[0], -B * e.Vm[1], -B * e.Vm[2]);
        return kDeferNone;
      }
      const double s = K / (e.Dm * e.gm.R * dt_s);
      dep_lin_f64(out, N, e.ua, s * e.Vm[0], s * e.Vm[1], s * e.Vm[2]);
      dep_lin_f64(out, N, e.ub, -s * e.Vm[0], -s * e.Vm[1], -s * e.Vm[2]);
      return kDeferNone;
    }
    const double ka = floor(e.ua), kb = floor(e.ub);
    const bool ina = ka >= 0.0 && ka < (double)N, inb = kb >= 0.0 && kb < (double)N;
    if (e.branch == 0) {
      const double s0 = +K / (e.D0 * e.g0.R * dt_s);
      const double s1 = -K / (e.D1 * e.g1.R * dt_s);
      if (ina) out.dep((int)ka, s0 * e.V0[0], s0 * e.V0[1], s0 * e.V0[2]);
      if (inb) out.dep((int)kb, s1 * e.V1[0], s1 * e.V1[1], s1 * e.V1[2]);
      return kDeferNone;
    }
    if (ka == kb) return kDeferNone;  // both linearised arrivals in one bin: zero
    const double s = K / (e.Dm * e.gm.R * dt_s);
    if (ina) out.dep((int)ka, s * e.Vm[0], s * e.Vm[1], s * e.Vm[2]);
    if (inb) out.dep((int)kb, -s * e.Vm[0], -s * e.Vm[1], -s * e.Vm[2]);
    return kDeferNone;
  }

  template <class Sink>
  static __device__ __forceinline__ void zhs(const double* T, int l, const AntRec& A, const MedParams& M, Sink& out) {
    const double q = TF(fd::Q);
    if (q == 0.0) return;
    const int N = M.n_bins;
    const double b[3] = {TF(fd::BX), TF(fd::BY), TF(fd::BZ)};
    const double x0 = TF(fd::X0), y0 = TF(fd::Y0), z0 = TF(fd::Z0);
    const double x1 = TF(fd::X1), y1 = TF(fd::Y1), z1 = TF(fd::Z1);
    const double t0 = TF(fd::T0), t1 = TF(fd::T1);
    const double KA = q * kKzhs;
    GeoD gm;
    geo_f64(M, A, 0.5 * (x0 + x1), 0.5 * (y0 + y1), 0.5 * (z0 + z1), TF(fd::EM), gm);
    if (gm.R == 0.0) return;
    const double c = b[0] * gm.rh[0] + b[1] * gm.rh[1] + b[2] * gm.rh[2];
    const double Dm = 1.0 - gm.n_src * c;
    const double bp[3] = {b[0] - c * gm.rh[0], b[1] - c * gm.rh[1], b[2] - c * gm.rh[2]};
    const double dte = t1 - t0;
    const double tm = 0.5 * (t0 + t1);
    const double tarr_rel = (tm - A.t_ref) + gm.n_avg * gm.R * M.inv_c_ns;
    const double half = fabs(Dm) * dte / 2.0;
    const double t_lo = tarr_rel - half, t_hi = tarr_rel + half;
    const double dt = M.dt_ns;
    const double u_lo = t_lo / dt, u_hi = t_hi / dt;
    const double k_lo = floor(u_lo), k_hi = floor(u_hi);
    out.rec(k_lo == k_hi ? 2 : 3, u_lo, u_hi);
    if (!(u_lo < (double)N + 1.0 && u_hi > -1.0)) return;
    if constexpr (LIN) {
      // reading LD: the tent weights averaged over [u_lo, u_hi]
      const double A1 = KA * dte / (gm.R * dt);
      if (floor(u_lo + 0.5) == floor(u_hi + 0.5)) {
        dep_lin_f64(out, N, 0.5 * (u_lo + u_hi), A1 * bp[0], A1 * bp[1], A1 * bp[2]);
        return;
      }
      const double W = u_hi - u_lo;
      const double kb = fmax(floor(u_lo - 0.5), 0.0), ke = fmin(floor(u_hi + 0.5), (double)(N - 1));
      for (double kd = kb; kd <= ke; kd += 1.0) {
        const double w = lin_share_integral_f64(u_lo, u_hi, kd) / W;
        if (w > 0.0) out.dep((int)kd, A1 * w * bp[0], A1 * w * bp[1], A1 * w * bp[2]);
      }
      return;
    }
    if (k_lo == k_hi) {
      const double s = KA * dte / (gm.R * dt);
      if (k_lo >= 0.0 && k_lo < (double)N) out.dep((int)k_lo, s * bp[0], s * bp[1], s * bp[2]);
      return;
    }
    const double kb = fmax(k_lo, 0.0), ke = fmin(k_hi, (double)(N - 1));
    // K_A beta_perp/(R |D_m|) times the overlap o of the interval with the bin,
    // over dt; the factor is formed once for the interval's bins
    const double sc = KA / (gm.R * fabs(Dm) * dt);
    for (double kd = kb; kd <= ke; kd += 1.0) {
      const double e_lo = kd * dt, e_hi = (kd + 1.0) * dt;
      const double o = fmin(t_hi, e_hi) - fmax(t_lo, e_lo);
      if (o <= 0.0) continue;
      const double s = sc * o;
      out.dep((int)kd, s * bp[0], s * bp[1], s * bp[2]);
    }
  }

  template <class Sink>
  static __device__ __forceinline__ void fwd(const void* Tv, int l, const AntRec& A, const MedParams& M, Sink& out) {
    const double* T = static_cast<const double*>(Tv);
    if constexpr (FORM == C8R_ENDPOINT)
      endpoint(T, l, A, M, out);
    else
      zhs(T, l, A, M, out);
  }

  static __device__ __forceinline__ int adj_main(const MainTrack& tr, const AntRec* p, const MedParams& M,
                                                 const Acc4D* G, const PrefixFF* Gp, MainGrad& m, double ga[3],
                                                 double& dn) {
    const AntRec A = *p;
    if constexpr (FORM == C8R_ZHS)
      adj_zhs(tr, A, M, G, Gp, m.g, ga, dn);
    else
      adj(tr, A, M, G, m.g, ga, dn);
    return kDeferNone;
  }
  static __device__ __forceinline__ int lone_end(const void*, int, const AntRec&, const MedParams&) { return 0; }
  static __device__ __forceinline__ void adj_deferred(const TrackD&, const AntRec&, const MedParams&, const Acc4D*,
                                                      const PrefixFF*, double*, double*, double&) {}
  static __device__ __forceinline__ void adj_end_deferred(const void*, int, const AntRec&, const MedParams&,
                                                          const Acc4D*, const c8r_track_grads&, int64_t, double*,
                                                          double&, int) {}

  // ZHS adjoint (bins of the interval ends held fixed; see the mixed path for
  // the formulas): in FP64, times in ns, positions in m.  The geometry and the
  // interval are the forward pass's own: with the one-bin deposit OpsF64Plain's, so
  // that an arrival within rounding of an edge is in one bin for both
  static __device__ __forceinline__ void adj_zhs(const MainTrack& tr, const AntRec& A, const MedParams& M,
                                                 const Acc4D* G, const PrefixFF*, double tg[11], double ga[3],
                                                 double& dn) {
    const double* T = static_cast<const double*>(tr.T);
    const int l = tr.l;
    const double q = TF(fd::Q);
    if (q == 0.0) return;
    const int N = M.n_bins;
    const double b[3] = {TF(fd::BX), TF(fd::BY), TF(fd::BZ)};
    const double t0 = TF(fd::T0), t1 = TF(fd::T1);
    const double Em = TF(fd::EM);
    const double dte = t1 - t0;
    const double dt = M.dt_ns;
    GeoD gm;
    double c, Dm, u_lo, u_hi, k_lo, k_hi;
    if constexpr (LIN) {
      geo_f64(M, A, 0.5 * (TF(fd::X0) + TF(fd::X1)), 0.5 * (TF(fd::Y0) + TF(fd::Y1)),
              0.5 * (TF(fd::Z0) + TF(fd::Z1)), Em, gm);
      if (gm.R == 0.0) return;
      c = b[0] * gm.rh[0] + b[1] * gm.rh[1] + b[2] * gm.rh[2];
      Dm = 1.0 - gm.n_src * c;
      const double tm = 0.5 * (t0 + t1);
      const double tarr_rel = (tm - A.t_ref) + gm.n_avg * gm.R * M.inv_c_ns;
      const double half = fabs(Dm) * dte / 2.0;
      u_lo = (tarr_rel - half) / dt;
      u_hi = (tarr_rel + half) / dt;
      k_lo = floor(u_lo);
      k_hi = floor(u_hi);
    } else {
      typename Plain::Eval e;
      if (!Plain::eval(tr.t, tr.t.p[0], A, M, e)) return;
      typename Plain::Interval v;
      Plain::interval(tr.t, e, N, v);
      if (v.one && v.lo.bin < 0) return;  // (also NaN: out of FP64's range)
      Plain::geometry(tr.t.p[0], A, e, gm);
      c = e.c;
      Dm = e.D;
      u_lo = v.u_lo;
      u_hi = v.u_hi;
      k_lo = v.lo.k;
      k_hi = v.one ? v.lo.k : v.hi.k;
    }
    const double KA = q * kKzhs;
    double Av[3];
    for (int k = 0; k < 3; ++k) Av[k] = KA * (b[k] - c * gm.rh[k]) * dte / (gm.R * dt);
    double S[3] = {0.0, 0.0, 0.0};
    double dLdu = 0.0, dLdh = 0.0;  // per bin of u, per bin of h = half/dt
    if constexpr (LIN) {
      // reading LD: S = sum_k w_k G_k with the tent weights averaged over the
      // interval; the interval-end values p = A.(G seen by a deposit at the end)
      double sl[3];
      if (floor(u_lo + 0.5) == floor(u_hi + 0.5)) {
        gather_lin_f64(G, N, 0.5 * (u_lo + u_hi), S, sl);
        dLdu = Av[0] * sl[0] + Av[1] * sl[1] + Av[2] * sl[2];
      } else {
        const double W = u_hi - u_lo;
        const double kb = fmax(floor(u_lo - 0.5), 0.0), ke = fmin(floor(u_hi + 0.5), (double)(N - 1));
        for (double kd = kb; kd <= ke; kd += 1.0) {
          const double w = lin_share_integral_f64(u_lo, u_hi, kd) / W;
          const Acc4D g = G[(int)kd];
          S[0] += w * g.x;
          S[1] += w * g.y;
          S[2] += w * g.z;
        }
        double glo[3], ghi[3];
        gather_lin_f64(G, N, u_lo, glo, sl);
        gather_lin_f64(G, N, u_hi, ghi, sl);
        const double p_lo = Av[0] * glo[0] + Av[1] * glo[1] + Av[2] * glo[2];
        const double p_hi = Av[0] * ghi[0] + Av[1] * ghi[1] + Av[2] * ghi[2];
        const double AS = Av[0] * S[0] + Av[1] * S[1] + Av[2] * S[2];
        dLdu = (p_hi - p_lo) / W;
        dLdh = (p_hi + p_lo - 2.0 * AS) / W;
      }
    } else if (k_lo == k_hi) {
      if (!(k_lo >= 0.0 && k_lo < (double)N)) return;
      const Acc4D g = G[(int)k_lo];
      S[0] = g.x; S[1] = g.y; S[2] = g.z;
    } else {
      // S = sum of (overlap / width) G over the bins of the interval inside the
      // window, bin by bin (the FP64 path does not use the running sums)
      const double W = u_hi - u_lo;
      const bool inlo = k_lo >= 0.0 && k_lo < (double)N, inhi = k_hi >= 0.0 && k_hi < (double)N;
      const Acc4D zero{0.0, 0.0, 0.0, 0.0};
      const Acc4D glo = inlo ? G[(int)k_lo] : zero, ghi = inhi ? G[(int)k_hi] : zero;
      const double kb = fmax(k_lo, 0.0), ke = fmin(k_hi, (double)(N - 1));
      for (double kd = kb; kd <= ke; kd += 1.0) {
        const double o = fmin(u_hi, kd + 1.0) - fmax(u_lo, kd);
        if (o <= 0.0) continue;
        const Acc4D g = G[(int)kd];
        S[0] += (o / W) * g.x;
        S[1] += (o / W) * g.y;
        S[2] += (o / W) * g.z;
      }
      const double g_lo = Av[0] * glo.x + Av[1] * glo.y + Av[2] * glo.z;
      const double g_hi = Av[0] * ghi.x + Av[1] * ghi.y + Av[2] * ghi.z;
      const double AS = Av[0] * S[0] + Av[1] * S[1] + Av[2] * S[2];
      dLdu = (g_hi - g_lo) / W;
      dLdh = (g_hi + g_lo - 2.0 * AS) / W;
    }
    const double AS = Av[0] * S[0] + Av[1] * S[1] + Av[2] * S[2];
    const double ka = KA * dte / (gm.R * dt);
    double sb[3], dLdb[3], dLdr[3];
    for (int k = 0; k < 3; ++k) sb[k] = ka * S[k];
    const double sbr = sb[0] * gm.rh[0] + sb[1] * gm.rh[1] + sb[2] * gm.rh[2];
    for (int k = 0; k < 3; ++k) {
      dLdb[k] = sb[k] - sbr * gm.rh[k];
      dLdr[k] = -c * sb[k] - sbr * b[k];
    }
    // dte enters A and h = |D| dte / (2 dt); u_m = tau_m - tau_a + n_avg R / (c dt)
    double dLd_dte = AS / dte + dLdh * fabs(Dm) / (2.0 * dt);
    double dLdR = -AS / gm.R;
    const double dLdD = dLdh * (Dm < 0.0 ? -1.0 : 1.0) * dte / (2.0 * dt);
    const double dLdn = -c * dLdD;
    for (int k = 0; k < 3; ++k) {
      dLdb[k] -= gm.n_src * gm.rh[k] * dLdD;
      dLdr[k] -= gm.n_src * b[k] * dLdD;
    }
    const RefrGrad<double> rg =
        refraction_grad<double>(M.kind, gm.R, gm.d[2] * M.invH, Em, M.N0, M.invH, M.n - 1.0);
    const double dLdopt = dLdu * M.inv_c_ns / dt;
    dLdR += dLdopt * (1.0 + rg.dF_dR);
    const double dLdzm = dLdopt * rg.dF_dzm + dLdn * rg.dn_dzm;
    const double dLdza = dLdopt * rg.dF_dza;
    dn += dLdopt * rg.dF_dN0 + dLdn * rg.dn_dN0;
    const double rdr = dLdr[0] * gm.rh[0] + dLdr[1] * gm.rh[1] + dLdr[2] * gm.rh[2];
    for (int k = 0; k < 3; ++k) {
      const double dd = (dLdr[k] - rdr * gm.rh[k]) / gm.R + dLdR * gm.rh[k];
      const double dm = -dd + (k == 2 ? dLdzm : 0.0);
      tg[k] += 0.5 * dm;
      tg[3 + k] += 0.5 * dm;
      tg[8 + k] += dLdb[k];
      ga[k] += dd + (k == 2 ? dLdza : 0.0);
    }
    tg[6] += 0.5 * dLdu / dt - dLd_dte;
    tg[7] += 0.5 * dLdu / dt + dLd_dte;
  }

  // chain rule through an arrival position u = (t_e - t_a)/dt + n_avg R/(c dt)
  // of the emission point at d = x_a - x_e (refractivity factor E): adds dL/dx_e
  // x w_e to pos0 (and pos1), dL/dx_a and dL/dN0 (the caller adds dL/dt_e)
  static __device__ __forceinline__ void arrival_grad(const GeoD& g, double E, const MedParams& M, double dLdu,
                                                      double* pos0, double* pos1, double w_e, double ga[3],
                                                      double& dn) {
    const RefrGrad<double> rg = refraction_grad<double>(M.kind, g.R, g.d[2] * M.invH, E, M.N0, M.invH, M.n - 1.0);
    const double dLdopt = dLdu * M.inv_c_ns / M.dt_ns;
    const double dLdR = dLdopt * (1.0 + rg.dF_dR);
    for (int k = 0; k < 3; ++k) {
      const double v = dLdR * g.rh[k];
      ga[k] += v;
      pos0[k] -= w_e * v;
      if (pos1) pos1[k] -= w_e * v;
    }
    pos0[2] += w_e * dLdopt * rg.dF_dzm;
    if (pos1) pos1[2] += w_e * dLdopt * rg.dF_dzm;
    ga[2] += dLdopt * rg.dF_dza;
    dn += dLdopt * rg.dF_dN0;
  }

  // Endpoint adjoint with the linear deposit (reading LD): the amplitude against
  // the spread of dL/dtrace each deposit sees, plus the slide of the deposits with
  // their arrivals (dL/du = l(G_{k0+1} - G_{k0})), through the arrival times and,
  // near Cherenkov, through u_a, u_b = u_m -/+ D dt_e/(2 dt).  Times in ns.
  static __device__ __forceinline__ void adj_lin(const double* T, int l, const EndpointEvalD& e, const double b[3],
                                                 double K, double dt_s, const MedParams& M, const Acc4D* G,
                                                 double tg[11], double ga[3], double& dn) {
    const int N = M.n_bins;
    const double dt = M.dt_ns;
    double dd[3], db[3], dns, gv[3], sl[3];
    if (e.branch == 0) {
      for (int j = 0; j < 2; ++j) {
        const GeoD& g = j == 0 ? e.g0 : e.g1;
        const double* V = j == 0 ? e.V0 : e.V1;
        const double D = j == 0 ? e.D0 : e.D1;
        const double E = j == 0 ? e.E0 : e.E1;
        const double kap = (j == 0 ? K : -K) / dt_s;
        gather_lin_f64(G, N, j == 0 ? e.ua : e.ub, gv, sl);
        const double c = b[0] * g.rh[0] + b[1] * g.rh[1] + b[2] * g.rh[2];
        deposit_adjoint<double>(g.rh, V, c, D, g.R, g.n_src, gv, kap, dd, db, dns);
        const RefrGrad<double> rg =
            refraction_grad<double>(M.kind, g.R, g.d[2] * M.invH, E, M.N0, M.invH, M.n - 1.0);
        for (int cc = 0; cc < 3; ++cc) {
          tg[3 * j + cc] -= dd[cc];
          ga[cc] += dd[cc];
          tg[8 + cc] += db[cc];
        }
        tg[3 * j + 2] += dns * rg.dn_dzm;
        dn += dns * rg.dn_dN0;
        const double dLdu = kap * (V[0] * sl[0] + V[1] * sl[1] + V[2] * sl[2]) / (D * g.R);
        arrival_grad(g, E, M, dLdu, tg + 3 * j, nullptr, 1.0, ga, dn);
        tg[6 + j] += dLdu / dt;
      }
      return;
    }
    const GeoD& g = e.gm;
    const double c = b[0] * g.rh[0] + b[1] * g.rh[1] + b[2] * g.rh[2];
    const double dte = TF(fd::T1) - TF(fd::T0);
    const double Ja = floor(e.ua + 0.5), Jb = floor(e.ub + 0.5);
    if (Ja == Jb) {
      // l = kap (g.V)/R, kap = K (dt_e/dt)/dt_s, g = G_{J-1} - G_J: the deposit
      // adjoint with D = 1 and n = 0, and dl/d dt_e = l/dt_e
      const Acc4D zero{0.0, 0.0, 0.0, 0.0};
      const Acc4D g0 = (Ja - 1.0 >= 0.0 && Ja - 1.0 < (double)N) ? G[(int)Ja - 1] : zero;
      const Acc4D g1 = (Ja >= 0.0 && Ja < (double)N) ? G[(int)Ja] : zero;
      gv[0] = g0.x - g1.x;
      gv[1] = g0.y - g1.y;
      gv[2] = g0.z - g1.z;
      const double kap = K * (dte / dt) / dt_s;
      deposit_adjoint<double>(g.rh, e.Vm, c, 1.0, g.R, 0.0, gv, kap, dd, db, dns);
      for (int cc = 0; cc < 3; ++cc) {
        tg[cc] -= 0.5 * dd[cc];
        tg[3 + cc] -= 0.5 * dd[cc];
        ga[cc] += dd[cc];
        tg[8 + cc] += db[cc];
      }
      const double lv = kap * (gv[0] * e.Vm[0] + gv[1] * e.Vm[1] + gv[2] * e.Vm[2]) / g.R;
      tg[6] -= lv / dte;
      tg[7] += lv / dte;
      return;
    }
    double gav[3], gbv[3], sla[3], slb[3];
    gather_lin_f64(G, N, e.ua, gav, sla);
    gather_lin_f64(G, N, e.ub, gbv, slb);
    for (int cc = 0; cc < 3; ++cc) gv[cc] = gav[cc] - gbv[cc];
    deposit_adjoint<double>(g.rh, e.Vm, c, e.Dm, g.R, g.n_src, gv, K / dt_s, dd, db, dns);
    const RefrGrad<double> rg = refraction_grad<double>(M.kind, g.R, g.d[2] * M.invH, e.Em, M.N0, M.invH, M.n - 1.0);
    for (int cc = 0; cc < 3; ++cc) {
      tg[cc] -= 0.5 * dd[cc];
      tg[3 + cc] -= 0.5 * dd[cc];
      ga[cc] += dd[cc];
      tg[8 + cc] += db[cc];
    }
    tg[2] += 0.5 * dns * rg.dn_dzm;
    tg[5] += 0.5 * dns * rg.dn_dzm;
    dn += dns * rg.dn_dN0;
    // the slide of the two spread deposits +/- s V, s = K/(D R dt_s)
    const double sm = K / (e.Dm * g.R * dt_s);
    const double dLdua = sm * (e.Vm[0] * sla[0] + e.Vm[1] * sla[1] + e.Vm[2] * sla[2]);
    const double dLdub = -sm * (e.Vm[0] * slb[0] + e.Vm[1] * slb[1] + e.Vm[2] * slb[2]);
    const double dLdum = dLdua + dLdub;
    const double dtau = dte / dt;
    const double dLdD = (dLdub - dLdua) * dtau / 2.0;
    const double dLd_dtau = (dLdub - dLdua) * e.Dm / 2.0;
    // D = 1 - n_src (beta.rhat), rhat = d/R, d = x_a - x_m
    double dLdr[3];
    for (int k = 0; k < 3; ++k) {
      tg[8 + k] -= g.n_src * g.rh[k] * dLdD;
      dLdr[k] = -g.n_src * b[k] * dLdD;
    }
    const double rdr = dLdr[0] * g.rh[0] + dLdr[1] * g.rh[1] + dLdr[2] * g.rh[2];
    for (int k = 0; k < 3; ++k) {
      const double v = (dLdr[k] - rdr * g.rh[k]) / g.R;
      tg[k] -= 0.5 * v;
      tg[3 + k] -= 0.5 * v;
      ga[k] += v;
    }
    const double dLdn = -c * dLdD;
    tg[2] += 0.5 * dLdn * rg.dn_dzm;
    tg[5] += 0.5 * dLdn * rg.dn_dzm;
    dn += dLdn * rg.dn_dN0;
    arrival_grad(g, e.Em, M, dLdum, tg, tg + 3, 0.5, ga, dn);
    tg[6] += (0.5 * dLdum - dLd_dtau) / dt;
    tg[7] += (0.5 * dLdum + dLd_dtau) / dt;
  }

  static __device__ __forceinline__ void adj(const MainTrack& tr, const AntRec& A, const MedParams& M,
                                             const Acc4D* G, double tg[11], double ga[3], double& dn) {
    static_assert(FORM == C8R_ENDPOINT, "adjoint is defined for the Endpoint formalism");
    const double* T = static_cast<const double*>(tr.T);
    const int l = tr.l;
    const double q = TF(fd::Q);
    if (q == 0.0) return;
    const int N = M.n_bins;
    const double b[3] = {TF(fd::BX), TF(fd::BY), TF(fd::BZ)};
    const double K = q * kKendpoint;
    const double dt_s = M.dt_ns * 1e-9;
    if constexpr (LIN) {
      EndpointEvalD e;
      endpoint_eval_f64(T, l, A, M, e);
      if (e.valid) adj_lin(T, l, e, b, K, dt_s, M, G, tg, ga, dn);
    } else {
      // the forward pass's own evaluation, as in adj_zhs
      const bool expo = M.kind == C8R_EXPONENTIAL;
      double dd[3], db[3], dns;
      typename Plain::Eval e[2];
      if (!Plain::eval(tr.t, tr.t.p[0], A, M, e[0]) || !Plain::eval(tr.t, tr.t.p[1], A, M, e[1])) return;
      if (fmin(fabs(e[0].D), fabs(e[1].D)) >= M.eps_Cd) {
        for (int j = 0; j < 2; ++j) {
          const int k = Plain::bin(e[j].u, N);
          if (k < 0) continue;
          const double gv[3] = {G[k].x, G[k].y, G[k].z};
          const typename Plain::Point& p = tr.t.p[j];
          GeoD g;
          Plain::geometry(p, A, e[j], g);
          deposit_adjoint<double>(g.rh, e[j].V, e[j].c, e[j].D, g.R, p.n, gv, (j == 0 ? K : -K) / dt_s, dd, db, dns);
          for (int cc = 0; cc < 3; ++cc) {
            tg[3 * j + cc] -= dd[cc];
            ga[cc] += dd[cc];
            tg[8 + cc] += db[cc];
          }
          if (expo) {
            tg[3 * j + 2] += dns * (-M.N0 * p.E / M.H);
            dn += dns * p.E;
          } else {
            dn += dns;
          }
        }
        return;
      }
      typename Plain::Point pm;
      typename Plain::Eval em;
      typename Plain::Near v;
      if (!Plain::near_arrivals(tr.t, T, l, A, M, pm, em, v)) return;
      if (v.a.k == v.b.k || (v.a.bin < 0 && v.b.bin < 0)) return;  // (also NaN, as in adj_zhs)
      double gv[3];
      for (int cc = 0; cc < 3; ++cc)
        gv[cc] = (v.a.bin >= 0 ? (&G[v.a.bin].x)[cc] : 0.0) - (v.b.bin >= 0 ? (&G[v.b.bin].x)[cc] : 0.0);
      GeoD g;
      Plain::geometry(pm, A, em, g);
      deposit_adjoint<double>(g.rh, em.V, em.c, em.D, g.R, pm.n, gv, K / dt_s, dd, db, dns);
      for (int cc = 0; cc < 3; ++cc) {
        tg[cc] -= 0.5 * dd[cc];
        tg[3 + cc] -= 0.5 * dd[cc];
        ga[cc] += dd[cc];
        tg[8 + cc] += db[cc];
      }
      if (expo) {
        tg[2] += 0.5 * dns * (-M.N0 * pm.E / M.H);
        tg[5] += 0.5 * dns * (-M.N0 * pm.E / M.H);
        dn += dns * pm.E;
      } else {
        dn += dns;
      }
    }
  }
};

// ---------------------------------------------------------------------------
// The forward pass, the arrival listing and the adjoint's geometry and bins in the
// plain media (uniform, exponential) with the one-bin deposit.  Bound by the FP64 pipe, which on this
// part runs at 1/64 of the FP32 rate, so the arithmetic is arranged for few FP64
// operations: one reciprocal square root and two reciprocals per emission point
// in place of a square root and five quotients, fused multiply-adds, what
// depends on the track alone formed once per track and held in registers, bins
// from the low word of a rounded-down sum.  About 90 -> 42 FP64 operations per
// emission point; and a ZHS interval's whole bins go in as a box (two edges)
// rather than bin by bin.  Measured, ms: 1e5 tracks x 16 antennas Endpoint in the
// uniform medium 0.92 -> 0.49 (0.32 with push_a_tile's tiles), 1e5 x 160 ZHS in the
// exponential one 6.2 -> 2.3.  Error of an Endpoint deposit against long double
// (rms over a shower, emulated, test_f64_plain_rounding): 2.0e-14 to 3.8e-14 -> 1.5e-14
// to 3.3e-14 relative, since a fused operation rounds once.
// ---------------------------------------------------------------------------
// 1/sqrt(x) and 1/x for normal x: the hardware's approximation (20 bits or more)
// and one third-order step (Householder's iteration: the residual e = 1 - x y^2
// or 1 - x r is of order 2^-20, and what is left is of order e^3)
__device__ __forceinline__ double rsqrt_f64(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = __fma_rn(-__dmul_rn(x, y), y, 1.0);
  return __fma_rn(__fma_rn(e, 0.375, 0.5), __dmul_rn(y, e), y);
}
__device__ __forceinline__ double rcp_f64(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = __fma_rn(-x, r, 1.0);
  return __fma_rn(r, __fma_rn(e, e, e), r);
}

// floor of an arrival position and its bin: k inside the window, or -1.  1.5 x
// 2^52 added with rounding down leaves floor(u) in the low word for |u| < 2^31;
// the high word tells whether it is one of 0 .. 2^32 - 1
struct FloorD {
  double k;
  int bin;
};
__device__ __forceinline__ FloorD floor_bin(double u, int n_bins) {
  const double magic = 6755399441055744.0;
  const double t = __dadd_rd(u, magic);
  const int lo = __double2loint(t);
  return FloorD{__dsub_rn(t, magic),
                __double2hiint(t) == 0x43380000 && (unsigned)lo < (unsigned)n_bins ? lo : -1};
}

template <int FORM>
struct OpsF64Plain {
  using acc_t = double;
  static constexpr int kPrec = C8R_FP64;
  static constexpr int kTileBytes = kTileBytesF64;
  static constexpr int kMinBlocks = 4;
  static constexpr int kFwdThreads = kTileT;
  static constexpr bool kDefers = FORM == C8R_ENDPOINT;  // near-Cherenkov pairs, as OpsF64
  static constexpr bool kFastBins = false;
  static constexpr int kAccRows = 1;  // (ZHS: the box edges lie apart, FwdShape::edge_off)

  // an emission point of the track
  struct Point {
    double x, y, z, t;
    double n;  // refractive index
    double E;  // exp(-z/H)
    double r;  // n_avg - 1 where every antenna has the same (uniform medium, flat array)
  };
  struct FwdTrack {
    Point p[FORM == C8R_ENDPOINT ? 2 : 1];  // start and end, or the midpoint
    double bx, by, bz;
    double amp;  // q K/dt, or q K_A (t1 - t0)/dt
    double hw;   // ZHS: (t1 - t0)/(2 dt)
  };
  using FwdAnt = AntRec;
  using Ant = AntRec;
  static __device__ __forceinline__ void stage_ant(AntRec* p, const AntRec& A, const MedParams&) { *p = A; }
  static __device__ __forceinline__ AntRec load_ant(const AntRec* p) { return *p; }

  // n_avg - 1 of the path from altitude z_e to z_a, dz = z_a - z_e, in the
  // exponential medium (the series within 1e-3 H)
  static __device__ __forceinline__ double refr(const MedParams& M, double Ea, double Ee, double dz) {
    const double x = __dmul_rn(dz, M.invH);
    double ratio;
    if (fabs(x) > 1e-3)
      ratio = __dmul_rn(__dsub_rn(Ee, Ea), rcp_f64(x));
    else
      ratio = Ee * (1.0 + x * (-0.5 + x * (1.0 / 6.0 + x * (-1.0 / 24.0 + x * (1.0 / 120.0)))));
    return __dmul_rn(M.N0, ratio);
  }
  static __device__ __forceinline__ void point(const MedParams& M, double x, double y, double z, double t, double E,
                                               Point& p) {
    p.x = x;
    p.y = y;
    p.z = z;
    p.t = t;
    p.E = E;
    p.r = M.n - 1.0;
    p.n = M.n;
    if (M.kind != C8R_UNIFORM) p.n = __fma_rn(M.N0, E, 1.0);
    if (M.flat) p.r = refr(M, M.flat_E, E, __dsub_rn(M.flat_z, z));
  }
  static __device__ __forceinline__ void load_fwd(const void* Tv, int l, const MedParams& M, FwdTrack& t) {
    const double* T = static_cast<const double*>(Tv);
    const double q = TF(fd::Q);
    t.amp = q;
    if (q == 0.0) return;
    t.bx = TF(fd::BX);
    t.by = TF(fd::BY);
    t.bz = TF(fd::BZ);
    if constexpr (FORM == C8R_ENDPOINT) {
      t.amp = q * (kKendpoint / (M.dt_ns * 1e-9));
      point(M, TF(fd::X0), TF(fd::Y0), TF(fd::Z0), TF(fd::T0), TF(fd::E0), t.p[0]);
      point(M, TF(fd::X1), TF(fd::Y1), TF(fd::Z1), TF(fd::T1), TF(fd::E1), t.p[1]);
    } else {
      const double dte = TF(fd::T1) - TF(fd::T0);
      t.hw = 0.5 * dte * M.inv_dt;
      t.amp = q * kKzhs * dte * M.inv_dt;
      midpoint(Tv, l, M, t.p[0]);
    }
  }
  static __device__ __forceinline__ void midpoint(const void* Tv, int l, const MedParams& M, Point& p) {
    const double* T = static_cast<const double*>(Tv);
    point(M, 0.5 * (TF(fd::X0) + TF(fd::X1)), 0.5 * (TF(fd::Y0) + TF(fd::Y1)), 0.5 * (TF(fd::Z0) + TF(fd::Z1)),
          0.5 * (TF(fd::T0) + TF(fd::T1)), TF(fd::EM), p);
  }
  static __device__ __forceinline__ bool live(const FwdTrack& t) { return t.amp != 0.0; }

  // propagator and field: rhat, V = rhat (rhat.beta) - beta, D, 1/R and the
  // arrival position u; false when the emission point sits on the antenna
  struct Eval {
    double V[3], D, iR, u;
    double rh[3], c, R;  // (the adjoint's)
  };
  // a track for the adjoint's main pass, with its place in the staged tile
  struct AdjTrack {
    FwdTrack t;
    const void* T;
    int l;
  };
  static __device__ __forceinline__ bool eval(const FwdTrack& t, const Point& p, const AntRec& A, const MedParams& M,
                                              Eval& e) {
    const double dx = __dsub_rn(A.x, p.x), dy = __dsub_rn(A.y, p.y), dz = __dsub_rn(A.z, p.z);
    const double S = __fma_rn(dz, dz, __fma_rn(dy, dy, __dmul_rn(dx, dx)));
    if (!(S >= 2.2250738585072014e-308)) return false;
    e.iR = rsqrt_f64(S);
    double R = __dmul_rn(S, e.iR);
    R = __fma_rn(__fma_rn(-R, R, S), __dmul_rn(0.5, e.iR), R);
    const double rx = __dmul_rn(dx, e.iR), ry = __dmul_rn(dy, e.iR), rz = __dmul_rn(dz, e.iR);
    const double c = __fma_rn(t.bz, rz, __fma_rn(t.by, ry, __dmul_rn(t.bx, rx)));
    e.rh[0] = rx;
    e.rh[1] = ry;
    e.rh[2] = rz;
    e.c = c;
    e.R = R;
    e.V[0] = __fma_rn(c, rx, -t.bx);
    e.V[1] = __fma_rn(c, ry, -t.by);
    e.V[2] = __fma_rn(c, rz, -t.bz);
    e.D = __fma_rn(-p.n, c, 1.0);
    double r = p.r;
    if (M.kind != C8R_UNIFORM && !M.flat) r = refr(M, A.Ea, p.E, dz);
    e.u = __dmul_rn(__fma_rn(__fma_rn(r, R, R), M.inv_c_ns, __dsub_rn(p.t, A.t_ref)), M.inv_dt);
    return true;
  }

  // the geometry of an evaluated point as the adjoint's chain rule takes it
  static __device__ __forceinline__ void geometry(const Point& p, const AntRec& A, const Eval& e, GeoD& g) {
    g.d[0] = __dsub_rn(A.x, p.x);
    g.d[1] = __dsub_rn(A.y, p.y);
    g.d[2] = __dsub_rn(A.z, p.z);
    g.R = e.R;
    for (int k = 0; k < 3; ++k) g.rh[k] = e.rh[k];
    g.n_src = p.n;
  }
  static __device__ __forceinline__ int bin(double u, int N) { return floor_bin(u, N).bin; }
  // ZHS: the ends of the arrival interval and their bins; `one`: in one bin
  struct Interval {
    double u_lo, u_hi, h;
    FloorD lo, hi;
    bool one;
  };
  static __device__ __forceinline__ void interval(const FwdTrack& t, const Eval& e, int N, Interval& v) {
    v.h = __dmul_rn(fabs(e.D), t.hw);
    v.u_lo = __dsub_rn(e.u, v.h);
    v.u_hi = __dadd_rn(e.u, v.h);
    v.lo = floor_bin(v.u_lo, N);
    v.hi = floor_bin(v.u_hi, N);
    // (also when |d|^2 overflows: u is NaN then, in no bin, and an interval of it
    // must not go in as a box)
    v.one = !(v.lo.k < v.hi.k);
  }
  // the adjoint of a near-Cherenkov pair: the midpoint and the bins of its linearised
  // arrivals by near_pair's operations (near_pair itself, built on this, took 0.7 %
  // longer per push); false when the midpoint sits on the antenna
  struct Near {
    FloorD a, b;
  };
  static __device__ __forceinline__ bool near_arrivals(const FwdTrack& t, const void* Tv, int l, const AntRec& A,
                                                       const MedParams& M, Point& p, Eval& e, Near& v) {
    const double* T = static_cast<const double*>(Tv);
    midpoint(Tv, l, M, p);
    if (!eval(t, p, A, M, e)) return false;
    const double h = e.D * (0.5 * (TF(fd::T1) - TF(fd::T0)) * M.inv_dt);
    v.a = floor_bin(e.u - h, M.n_bins);
    v.b = floor_bin(e.u + h, M.n_bins);
    return true;
  }

  template <class Sink>
  static __device__ __forceinline__ int pair_main(const FwdTrack& t, const AntRec* pa, const void*, int,
                                                  const MedParams& M, Sink& out) {
    const AntRec& A = *pa;
    const int N = M.n_bins;
    if constexpr (FORM == C8R_ENDPOINT) {
      Eval e0, e1;
      if (!eval(t, t.p[0], A, M, e0) || !eval(t, t.p[1], A, M, e1)) return kDeferNone;
      if (!(fmin(fabs(e0.D), fabs(e1.D)) >= M.eps_Cd)) return kDeferPair;
      out.rec(0, e0.u, e1.u);
      const int ka = floor_bin(e0.u, N).bin, kb = floor_bin(e1.u, N).bin;
      const double s0 = __dmul_rn(__dmul_rn(t.amp, e0.iR), rcp_f64(e0.D));
      const double s1 = -__dmul_rn(__dmul_rn(t.amp, e1.iR), rcp_f64(e1.D));
      // both in one bin: added in registers
      const bool same = ka >= 0 && ka == kb;
      if (same) {
        out.dep(ka, __fma_rn(s1, e1.V[0], s0 * e0.V[0]), __fma_rn(s1, e1.V[1], s0 * e0.V[1]),
                __fma_rn(s1, e1.V[2], s0 * e0.V[2]));
      } else {
        if (ka >= 0) out.dep(ka, s0 * e0.V[0], s0 * e0.V[1], s0 * e0.V[2]);
        if (kb >= 0) out.dep(kb, s1 * e1.V[0], s1 * e1.V[1], s1 * e1.V[2]);
      }
    } else {
      Eval e;
      if (!eval(t, t.p[0], A, M, e)) return kDeferNone;
      Interval v;
      interval(t, e, N, v);
      const double u_lo = v.u_lo, u_hi = v.u_hi, h = v.h;
      const FloorD lo = v.lo, hi = v.hi;
      const bool one = v.one;
      out.rec(one ? 2 : 3, u_lo, u_hi);
      const double s = -__dmul_rn(t.amp, e.iR);  // beta_perp = -V
      const double invW = one ? 1.0 : rcp_f64(__dadd_rn(h, h));
      // the share of the interval in its first bin (all of it when it has one),
      // in its last, and 1/W in each whole bin between
      if (lo.bin >= 0) {
        const double w = one ? s : s * (__dsub_rn(lo.k + 1.0, u_lo) * invW);
        out.dep(lo.bin, w * e.V[0], w * e.V[1], w * e.V[2]);
      }
      if (one) return kDeferNone;
      if (hi.bin >= 0) {
        const double w = s * (__dsub_rn(u_hi, hi.k) * invW);
        out.dep(hi.bin, w * e.V[0], w * e.V[1], w * e.V[2]);
      }
      const double kb = fmax(lo.k + 1.0, 0.0), ke = fmin(hi.k - 1.0, (double)(N - 1));
      if (kb <= ke) {
        const double w = s * invW;
        out.dep_box((int)kb, (int)ke, w * e.V[0], w * e.V[1], w * e.V[2]);
      }
    }
    return kDeferNone;
  }

  // a near-Cherenkov Endpoint pair (reading C): the midpoint and its linearised
  // arrivals
  template <class Sink>
  static __device__ __forceinline__ void near_pair(const void* Tv, int l, const AntRec& A, const MedParams& M,
                                                   Sink& out) {
    const double* T = static_cast<const double*>(Tv);
    FwdTrack t;
    t.bx = TF(fd::BX);
    t.by = TF(fd::BY);
    t.bz = TF(fd::BZ);
    const int N = M.n_bins;
    midpoint(Tv, l, M, t.p[0]);
    Eval e;
    if (!eval(t, t.p[0], A, M, e)) return;
    const double h = e.D * (0.5 * (TF(fd::T1) - TF(fd::T0)) * M.inv_dt);
    const double ua = e.u - h, ub = e.u + h;
    out.rec(1, ua, ub);
    const FloorD a = floor_bin(ua, N), b = floor_bin(ub, N);
    if (a.k == b.k) return;  // both linearised arrivals in one bin: zero
    const double s = TF(fd::Q) * (kKendpoint / (M.dt_ns * 1e-9)) * e.iR * rcp_f64(e.D);
    if (a.bin >= 0) out.dep(a.bin, s * e.V[0], s * e.V[1], s * e.V[2]);
    if (b.bin >= 0) out.dep(b.bin, -s * e.V[0], -s * e.V[1], -s * e.V[2]);
  }
  // set-aside pairs come with the staged tile and the lane
  struct Track {
    const void* T;
    int l;
  };
  static __device__ __forceinline__ void load(const void* Tv, int l, const MedParams&, Track& t) {
    t.T = Tv;
    t.l = l;
  }
  template <class Sink>
  static __device__ __forceinline__ void pair_deferred(const Track& t, const AntRec& A, const MedParams& M,
                                                       Sink& out) {
    if constexpr (kDefers) near_pair(t.T, t.l, A, M, out);
  }
  template <class Sink>
  static __device__ __forceinline__ void end_deferred(const void*, int, const AntRec&, const MedParams&, Sink&, int) {}
  static __device__ __forceinline__ bool near_zero_fast(const void*, int, const AntRec&, const MedParams&) {
    return false;
  }
  // one pair from a tile (the arrival listing)
  template <class Sink>
  static __device__ __forceinline__ void fwd(const void* Tv, int l, const AntRec& A, const MedParams& M, Sink& out) {
    FwdTrack t;
    load_fwd(Tv, l, M, t);
    if (live(t) && pair_main(t, &A, Tv, l, M, out) == kDeferPair) near_pair(Tv, l, A, M, out);
  }
};

#undef TF

// uniform or flat exponential: the medium of OpsF64Plain
inline bool plain_medium(const MedParams& M) { return M.kind == C8R_UNIFORM || M.kind == C8R_EXPONENTIAL; }

// forward and adjoint launches for one deposit shape
template <bool LIN>
cudaError_t forward_f64(int formalism, const void* tiles, int64_t n_tiles, const AntRec* ants, int n_ant,
                        const MedParams& M, void* acc, const FwdShape& shape, int sm_count, int* err,
                        cudaStream_t st) {
  FwdArgs a{tiles, n_tiles, ants, n_ant, shape.a_tile, acc, err, FwdGrid{}, M};
  auto go = [&](auto ops) {
    using O = decltype(ops);
    a.replicas = shape.replicas > 1 ? shape.replicas : 1;
    a.replica_stride = (int64_t)n_ant * M.n_bins * O::kAccRows;
    a.edge_off = shape.edge_off;
    const int64_t ctas = forward_grid(a, shape, sm_count * forward_blocks_per_sm<O>(shape.a_tile),
                                      sizeof(Acc4D) * (shape.edge_off ? 2 : 1));
    return launch_forward_ops<O>(a, ctas, st);
  };
  if constexpr (!LIN) {
    if (plain_medium(M)) return formalism == C8R_ENDPOINT ? go(OpsF64Plain<C8R_ENDPOINT>{}) : go(OpsF64Plain<C8R_ZHS>{});
  }
  return formalism == C8R_ENDPOINT ? go(OpsF64<C8R_ENDPOINT, LIN>{}) : go(OpsF64<C8R_ZHS, LIN>{});
}

template <bool LIN>
cudaError_t backward_f64(int formalism, BwdArgs& a, const FwdShape& shape, int sm_count, cudaStream_t st) {
  if (formalism == C8R_ZHS) return launch_backward_ops<OpsF64<C8R_ZHS, LIN>>(a, shape, sm_count, st);
  return launch_backward_ops<OpsF64<C8R_ENDPOINT, LIN>>(a, shape, sm_count, st);
}

}  // namespace c8r
