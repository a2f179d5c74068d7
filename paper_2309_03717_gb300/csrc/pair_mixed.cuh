// pair_mixed.cuh -- per (track, antenna) arithmetic of the mixed-precision path.
//
// FP32 field arithmetic; the arrival time, the bin index and the ends of the
// arrival interval are float-float (about 48 significant bits), which keeps the
// bin of every deposit identical to an FP64 evaluation except within ~1e-7 bin
// of an edge.  The Doppler factor D = 1 - n beta.rhat is formed without the
// cancellation of the direct form (see field_mixed), from 1 - |beta| computed
// per track in FP64 by the ingest kernel.
//
// A thread loads one track of a staged tile into registers (TrackM) once and
// then evaluates it against every antenna of the CTA's antenna tile.
#pragma once

#include "kernels.cuh"

namespace c8r {

// track fields of lane l in a field-major tile
#define TF(f) T[(f) * kTileT + l]

// one track, held in registers while it is evaluated against the antennas
struct TrackM {
  float x0, y0, z0, x1, y1, z1;  // FP32-exact endpoints
  float bx, by, bz, bmag;
  float amp;                     // q K/dt (Endpoint) or q K_A (t1-t0)/dt (ZHS); 0 = dropped
  float tau0h, tau0l, tau1h, tau1l, dtauh, dtaul;
  // a flat antenna array (MedParams::flat, exponential medium): the quotient of
  // the refractivity term at the midpoint, the same for every antenna
  float qmh, qml;
  ZPart zm;                      // ZHS, flat array: the z part of the midpoint's d
  float E0h, E0l, E1h, E1l, Emh, Eml;
  float nm1_0, nm1_1, nm1_m;     // n - 1 at start, end, midpoint
  float om0, om1, om_m;          // 1 - n|beta| at start, end, midpoint
  // midpoint position and time, float-float
  float mx, mxl, my, myl, mz, mzl, tmh, tml;
};

template <int FORM, int KIND, bool FLAT = false>
__device__ __forceinline__ void load_track_mixed(const float* T, int l, const MedParams& M, TrackM& t) {
  t.amp = FORM == C8R_ENDPOINT ? TF(fm::AMPE) : (TF(fm::AMPE) == 0.0f ? 0.0f : TF(fm::AMPZ));
  if (t.amp == 0.0f) return;  // filtered track or padding
  t.x0 = TF(fm::X0); t.y0 = TF(fm::Y0); t.z0 = TF(fm::Z0);
  t.x1 = TF(fm::X1); t.y1 = TF(fm::Y1); t.z1 = TF(fm::Z1);
  t.bx = TF(fm::BX); t.by = TF(fm::BY); t.bz = TF(fm::BZ);
  t.bmag = TF(fm::BMAG);
  const float omb = TF(fm::OMB);
  t.tau0h = TF(fm::TAU0H); t.tau0l = TF(fm::TAU0L);
  t.tau1h = TF(fm::TAU1H); t.tau1l = TF(fm::TAU1L);
  t.dtauh = TF(fm::DTAUH); t.dtaul = TF(fm::DTAUL);
  // n - 1 is formed directly (N0 E, or the uniform n - 1 rounded from FP64): as
  // (1 + x) - 1 in FP32 it would lose ~6e-8, comparable to D near Cherenkov
  t.E0h = t.E1h = t.Emh = 1.0f;
  t.E0l = t.E1l = t.Eml = 0.0f;
  t.nm1_0 = t.nm1_1 = t.nm1_m = M.nm1f;
  if (KIND != C8R_UNIFORM) {
    t.E0h = TF(fm::E0H); t.E0l = TF(fm::E0L);
    t.E1h = TF(fm::E1H); t.E1l = TF(fm::E1L);
    t.Emh = TF(fm::EMH); t.Eml = TF(fm::EML);
    t.nm1_0 = __fmul_rn(M.N0f, t.E0h);
    t.nm1_1 = __fmul_rn(M.N0f, t.E1h);
    t.nm1_m = __fmul_rn(M.N0f, t.Emh);
  }
  if (KIND == C8R_EXPONENTIAL_SPHERICAL) {
    // n - 1 at the points over the sphere: the flat N0 exp(-z/H) times exp(-delta/H)
    t.nm1_0 = __fmul_rn(t.nm1_0, expf(-sphere_excess(t.x0, t.y0, t.z0, M.RE_f) * M.invH_h));
    t.nm1_1 = __fmul_rn(t.nm1_1, expf(-sphere_excess(t.x1, t.y1, t.z1, M.RE_f) * M.invH_h));
    t.nm1_m = __fmul_rn(t.nm1_m, expf(-sphere_excess(0.5f * (t.x0 + t.x1), 0.5f * (t.y0 + t.y1),
                                                     0.5f * (t.z0 + t.z1), M.RE_f) * M.invH_h));
  }
  // 1 - n|beta| = (1 - |beta|) - (n - 1)|beta|
  t.om0 = __fsub_rn(omb, __fmul_rn(t.nm1_0, t.bmag));
  t.om1 = __fsub_rn(omb, __fmul_rn(t.nm1_1, t.bmag));
  t.om_m = __fsub_rn(omb, __fmul_rn(t.nm1_m, t.bmag));
  // midpoint time (t0 + t1)/(2 dt), float-float
  two_sum(t.tau0h, t.tau1h, t.tmh, t.tml);
  t.tml = __fadd_rn(t.tml, __fadd_rn(t.tau0l, t.tau1l));
  t.tmh *= 0.5f;
  t.tml *= 0.5f;
  if (FORM == C8R_ZHS) {
    // midpoint position (x0 + x1)/2, exact in float-float
    two_sum(t.x0, t.x1, t.mx, t.mxl);
    two_sum(t.y0, t.y1, t.my, t.myl);
    two_sum(t.z0, t.z1, t.mz, t.mzl);
    t.mx *= 0.5f; t.mxl *= 0.5f; t.my *= 0.5f; t.myl *= 0.5f; t.mz *= 0.5f; t.mzl *= 0.5f;
  }
  if constexpr (FLAT && KIND != C8R_UNIFORM && FORM == C8R_ZHS) {
    // the refractivity quotient against the array's altitude, formed as the
    // per-pair arithmetic forms it (the altitude difference as geo_lite forms
    // it), so the values are the same
    float dzh, dzl;
    two_sum(M.flat_zh, -t.mz, dzh, dzl);
    dzl = __fadd_rn(dzl, __fsub_rn(M.flat_zl, t.mzl));
    refr_quotient(M, M.flat_Eh, M.flat_El, dzh, dzl, t.Emh, t.Eml, t.qmh, t.qml);
    t.zm = z_part(dzh, dzl, t.bz);
  }
}

// a track for the main pass of the one-bin Endpoint kernels: its two endpoints
// as pairs
struct TrackE {
  float2 x, y, z;        // FP32-exact endpoints
  float2 Th, Tl;         // shifted times tau + k z (arrival_fast)
  float2 Eh, El;         // exp(-z/H)
  float2 q;              // flat antenna array: the refractivity quotient (MedParams::flat)
  float2 om, n;          // 1 - n|beta|, n
  float bx, by, bz, bmag;
  float amp;             // q K/dt; 0 = dropped
};

template <int KIND, int AF, bool FLAT>
__device__ __forceinline__ void load_track_endpoints(const float* T, int l, const MedParams& M, TrackE& t) {
  t.amp = TF(fm::AMPE);
  if (t.amp == 0.0f) return;  // filtered track or padding
  t.x = make_float2(TF(fm::X0), TF(fm::X1));
  t.y = make_float2(TF(fm::Y0), TF(fm::Y1));
  t.z = make_float2(TF(fm::Z0), TF(fm::Z1));
  t.bx = TF(fm::BX); t.by = TF(fm::BY); t.bz = TF(fm::BZ);
  t.bmag = TF(fm::BMAG);
  const float kh = KIND == C8R_UNIFORM ? M.s_h : M.kc_h, kl = KIND == C8R_UNIFORM ? M.s_l : M.kc_l;
  if constexpr (AF == kFormAxis) {
    const float p0[3] = {t.x.x, t.y.x, t.z.x}, p1[3] = {t.x.y, t.y.y, t.z.y}, low[3] = {0.0f, 0.0f, 0.0f};
    axis_time(M, TF(fm::TAU0H), TF(fm::TAU0L), p0, low, t.Th.x, t.Tl.x);
    axis_time(M, TF(fm::TAU1H), TF(fm::TAU1L), p1, low, t.Th.y, t.Tl.y);
  } else {
    shifted_time(TF(fm::TAU0H), TF(fm::TAU0L), t.z.x, 0.0f, kh, kl, t.Th.x, t.Tl.x);
    shifted_time(TF(fm::TAU1H), TF(fm::TAU1L), t.z.y, 0.0f, kh, kl, t.Th.y, t.Tl.y);
  }
  float2 nm1 = bc<float2>(M.nm1f);
  t.Eh = bc<float2>(1.0f);
  if constexpr (KIND == C8R_EXPONENTIAL) {
    t.Eh = make_float2(TF(fm::E0H), TF(fm::E1H));
    t.El = make_float2(TF(fm::E0L), TF(fm::E1L));
    nm1 = mul_rn(bc<float2>(M.N0f), t.Eh);
  }
  // 1 - n|beta| = (1 - |beta|) - (n - 1)|beta|
  t.om = sub_rn(bc<float2>(TF(fm::OMB)), mul_rn(nm1, bc<float2>(t.bmag)));
  t.n = add_rn(bc<float2>(1.0f), nm1);
  // the quotient against the array's altitude, as the per-pair arithmetic forms
  // it (the altitude difference as geo_fast forms it), so the same values
  if constexpr (FLAT) {
    t.q.x = fast_quotient(M, M.flat_Eh, M.flat_El, __fsub_rn(M.flat_zh, t.z.x), t.Eh.x, t.El.x);
    t.q.y = fast_quotient(M, M.flat_Eh, M.flat_El, __fsub_rn(M.flat_zh, t.z.y), t.Eh.y, t.El.y);
  }
}

// an antenna in shared memory for those kernels: what the main pass takes is
// stored twice, as operands for pairs (four 16-byte loads), the rest follows
struct alignas(16) AntE {
  float2 x, y, z, Th, Tl, Eh, El;
  float fb_abs, fb_rel_v;
  float xl, yl, zl, tauh, taul, pad[3];
};
static_assert(sizeof(AntE) == sizeof(AntRec), "fwd_layout reckons with one antenna record size");

// What the spherical-Earth and curved-ray propagators need of a track for a flat
// antenna array, where the path's heights and the refractivity along it are the
// same for every antenna (two tracks, halves x and y).  Per pair and node the
// quadratures took an exponential, a root and a quotient (sphere) or six roots
// and quotients (rays) on the XU pipe; these take none.  ZHS, ms: 2.5e5 tracks x
// 1024 antennas over a sphere 4.43 -> 3.21, x 256 antennas along rays 1.69 -> 0.82
// (6 CTAs of 64 threads per SM; 7 and 8, with 128 registers: 3.45, 3.50 and 0.82,
// 0.84).
template <int KIND>
struct PathZ {};

// Spherical Earth: the curvature part of the optical path (sphere_path_correction),
//   N0 R sum_j w_j E_j (exp(-d_j/H) - 1),  E_j = exp(-z_j/H), d_j the altitude
//   excess of node j at the distance y_j^(1/2) from the vertical through the
//   origin.  With x_j = y_j h_j, h_j = 1/(2 (z_j + R_E) H), and k = H/(2 R_E), d_j/H =
//   x_j (1 - k x_j + ...) and the bracket is -x_j [1 - x_j (k + 1/2) + x_j^2 (k + 1/6)]
//   up to x^3/24 of it: 4e-8 for x_j < 0.01, which holds within 32 km of the origin
//   (antennas: checked by the host, tracks: `small`).  Per track: w_j E_j h_j, and
//   h as a linear function along the path for the bracket.  k is taken at the sphere's
//   radius and 2 k^2 x^2 dropped: the host asks for H < R_E/250 (the Earth: R_E/800)
//   and `small` for altitude differences below 3 % of the radius, which keep both
//   and the linear h below 6e-7 of the correction.
template <>
struct PathZ<C8R_EXPONENTIAL_SPHERICAL> {
  float2 weh[kSphNodes];
  float2 h0, h1;
  bool small;
  __device__ __forceinline__ void set(const MedParams& M, float2 mx, float2 my, float2 mz, float2 dz) {
    const float inv2H = 0.5f * M.invH_h;
    h0 = make_float2(div_ap(inv2H, M.RE_f + M.flat_zh), div_ap(inv2H, M.RE_f + M.flat_zh));
    h1 = make_float2(div_ap(inv2H, M.RE_f + mz.x) - h0.x, div_ap(inv2H, M.RE_f + mz.y) - h0.y);
    const float2 y = fma_rn(mx, mx, mul_rn(my, my));
    small = fmaxf(y.x * h0.x, y.y * h0.y) < 0.01f &&
            fmaxf(fabsf(dz.x), fabsf(dz.y)) < 0.03f * (M.RE_f + M.flat_zh);
#pragma unroll
    for (int j = 0; j < kSphNodes; ++j) {
      const float f = 1.0f - (float)kSphSigma[j];
      const float2 z = fma_rn(bc<float2>(-f), dz, bc<float2>(M.flat_zh));
      const float w = (float)kSphWeight[j] * inv2H;
      weh[j] = make_float2(div_ap(w * exp_ap(-z.x * M.invH_h), M.RE_f + z.x),
                           div_ap(w * exp_ap(-z.y * M.invH_h), M.RE_f + z.y));
    }
  }
  // the change of the optical path to the antenna at (ax, ay), m
  __device__ __forceinline__ float2 path(const MedParams& M, float2 ax, float2 ay, const GeoT<float2>& g) const {
    const float k = 0.5f * M.RE_k;
    float2 sum = bc<float2>(0.0f);
#pragma unroll
    for (int j = 0; j < kSphNodes; ++j) {
      const float f = 1.0f - (float)kSphSigma[j];
      const float2 x = fma_rn(bc<float2>(-f), g.s[0], ax), y = fma_rn(bc<float2>(-f), g.s[1], ay);
      const float2 r2 = fma_rn(x, x, mul_rn(y, y));
      const float2 xj = mul_rn(r2, fma_rn(bc<float2>(f), h1, h0));
      const float2 p = fma_rn(xj, fma_rn(xj, bc<float2>(k + 1.0f / 6.0f), bc<float2>(-k - 0.5f)), bc<float2>(1.0f));
      sum = fma_rn(mul_rn(weh[j], r2), p, sum);
    }
    return mul_rn(mul_rn(bc<float2>(-M.N0f), g.R0), sum);
  }
};

// Curved rays (ray_fix): with a_j = 1/n_j at the Gauss-Legendre nodes, abar their
// weighted mean, b_j = a_j/abar - 1 (~1e-4), B_k = sum_j w_j b_j^k and T = tan of the
// straight line's angle from the vertical, the ray's constant is p = S (1 + t)/abar,
// and expanding the end-point condition and Fermat's time saved in b (a series in
// T^2 b, carried to b^4) gives
//   t = -(3/2) T^2 B2 - (1/2) T^2 (1 + 5 T^2) B3,
//   path change = -(R T^2/abar) [B2/2 + (T^2 - 1) B3/2 + (4 - 3 T^2 + 5 T^4) B4/8 -
//                 (9/8) T^4 B2^2],
//   C Q at x_e = e (1 + T^2 e/2 + T^4 e^2/2),  e = t + (1 + t) b_e.
// The rest is of order (T^2 b)^3 and of b^3 of these: below 3e-7 (path) and 2e-7
// (turn) for T^2 b < 4e-3 and b < 1e-2, the pairs taken here (zenith angles to ~78
// degrees in air, where b is 3e-4; at b = 0.02 the path is off by 3e-6, at 0.2 by
// 1e-3).  Everything but T^2 is a property of the track; b is formed from r_j =
// nu_j/n_j without cancellation.
template <>
struct PathZ<C8R_EXPONENTIAL_RAY> {
  float2 inv_abar, B2, B3, B4, be, bmax, inv_dz2;
  __device__ __forceinline__ void set(const MedParams& M, float2 nu_e, float2 dz) {
    float2 r[kSphNodes], mean = bc<float2>(0.0f);
#pragma unroll
    for (int j = 0; j < kSphNodes; ++j) {
      const float c = -(float)kSphSigma[j] * M.invH_h;
      const float2 nu = mul_rn(nu_e, make_float2(exp_ap(c * dz.x), exp_ap(c * dz.y)));
      r[j] = mul_rn(nu, rcp_ap(add_rn(bc<float2>(1.0f), nu)));
      mean = fma_rn(bc<float2>((float)kSphWeight[j]), r[j], mean);
    }
    inv_abar = rcp_ap(sub_rn(bc<float2>(1.0f), mean));
    B2 = B3 = B4 = bc<float2>(0.0f);
#pragma unroll
    for (int j = 0; j < kSphNodes; ++j) {
      const float2 b = mul_rn(sub_rn(mean, r[j]), inv_abar), b2 = mul_rn(b, b);
      const float2 w = bc<float2>((float)kSphWeight[j]);
      B2 = fma_rn(w, b2, B2);
      B3 = fma_rn(w, mul_rn(b2, b), B3);
      B4 = fma_rn(w, mul_rn(b2, b2), B4);
    }
    be = mul_rn(sub_rn(mean, mul_rn(nu_e, rcp_ap(add_rn(bc<float2>(1.0f), nu_e)))), inv_abar);
    // b at the antenna's end
    const float2 nu_a = mul_rn(nu_e, make_float2(exp_ap(-M.invH_h * dz.x), exp_ap(-M.invH_h * dz.y)));
    const float2 ba = mul_rn(sub_rn(mean, mul_rn(nu_a, rcp_ap(add_rn(bc<float2>(1.0f), nu_a)))), inv_abar);
    bmax = make_float2(fmaxf(fabsf(be.x), fabsf(ba.x)), fmaxf(fabsf(be.y), fabsf(ba.y)));
    // beyond the range of b: no T^2 is in range
    if (!(bmax.x < 1e-2f)) bmax.x = 1e30f;
    if (!(bmax.y < 1e-2f)) bmax.y = 1e30f;
    inv_dz2 = rcp_ap(mul_rn(dz, dz));
  }
  // the change of the optical path (m) and the turn of the direction at x_e (the
  // change of R rhat); false for pairs outside the series' range
  __device__ __forceinline__ bool path(const GeoT<float2>& g, float2& dop, float2 turn[3]) const {
    const float2 T2 = mul_rn(fma_rn(g.s[0], g.s[0], mul_rn(g.s[1], g.s[1])), inv_dz2);
    const float2 q = mul_rn(T2, bmax);
    if (!(fmaxf(q.x, q.y) < 4e-3f) || !(fmaxf(T2.x, T2.y) < 1e5f)) return false;
    const float2 half = bc<float2>(0.5f);
    const float2 hT = mul_rn(half, T2);
    const float2 t = neg(mul_rn(hT, fma_rn(bc<float2>(3.0f), B2, mul_rn(B3, fma_rn(bc<float2>(5.0f), T2, bc<float2>(1.0f))))));
    const float2 c4 = fma_rn(T2, fma_rn(T2, bc<float2>(0.625f), bc<float2>(-0.375f)), half);
    float2 v = fma_rn(half, B2, mul_rn(B3, fma_rn(half, T2, bc<float2>(-0.5f))));
    v = fma_rn(c4, B4, v);
    const float2 TB = mul_rn(T2, B2);
    v = fma_rn(mul_rn(bc<float2>(-1.125f), TB), TB, v);
    dop = neg(mul_rn(mul_rn(mul_rn(g.R0, T2), inv_abar), v));
    const float2 e = fma_rn(t, be, add_rn(t, be));
    // sin(turn) = T cq, cos(turn) - 1 = -(T cq)^2/2 to a relative 1e-8
    const float2 cq = mul_rn(e, fma_rn(mul_rn(hT, e), fma_rn(T2, e, bc<float2>(1.0f)), bc<float2>(1.0f)));
    const float2 cm = neg(mul_rn(mul_rn(hT, cq), cq));
    const float2 f = add_rn(cm, cq);
    turn[0] = mul_rn(f, g.s[0]);
    turn[1] = mul_rn(f, g.s[1]);
    turn[2] = mul_rn(fma_rn(neg(T2), cq, cm), g.s[2]);
    return true;
  }
};

// two tracks for the forward pass of the ZHS kernels, halves x and y; the
// midpoint of each
template <int KIND>
struct TrackZ : PathZ<KIND> {
  float2 mx, mxl, my, myl, mz, mzl;   // position, float-float
  float2 bx, by, bz, nm1;
  float2 tmh, tml, dtauh, dtaul;      // (t0 + t1)/(2 dt), (t1 - t0)/dt
  float2 Eh, El;                      // exp(-z/H); a flat antenna array: the refractivity quotient instead
  ZPartT<float2> zm;                  // flat antenna array: the z part of d
  float2 amp;                         // -q K_A (t1 - t0)/dt
  bool live;
};

template <int KIND, bool FLAT>
__device__ __forceinline__ void load_track_pair(const float* T, int l, const MedParams& M, TrackZ<KIND>& t) {
  auto ld = [&](int f) { return *reinterpret_cast<const float2*>(T + f * kTileT + 2 * l); };
  const float2 keep = ld(fm::AMPE);
  t.live = keep.x != 0.0f || keep.y != 0.0f;
  if (!t.live) return;
  t.amp = neg(ld(fm::AMPZ));
  const float2 half = bc<float2>(0.5f);
  two_sum(ld(fm::X0), ld(fm::X1), t.mx, t.mxl);
  two_sum(ld(fm::Y0), ld(fm::Y1), t.my, t.myl);
  two_sum(ld(fm::Z0), ld(fm::Z1), t.mz, t.mzl);
  t.mx = mul_rn(t.mx, half); t.mxl = mul_rn(t.mxl, half);
  t.my = mul_rn(t.my, half); t.myl = mul_rn(t.myl, half);
  t.mz = mul_rn(t.mz, half); t.mzl = mul_rn(t.mzl, half);
  t.bx = ld(fm::BX); t.by = ld(fm::BY); t.bz = ld(fm::BZ);
  two_sum(ld(fm::TAU0H), ld(fm::TAU1H), t.tmh, t.tml);
  t.tml = add_rn(t.tml, add_rn(ld(fm::TAU0L), ld(fm::TAU1L)));
  t.tmh = mul_rn(t.tmh, half);
  t.tml = mul_rn(t.tml, half);
  // a filtered track or padding next to a live one: an arrival far before every
  // window, so that it deposits nothing
  if (keep.x == 0.0f) t.tmh.x = -1e30f;
  if (keep.y == 0.0f) t.tmh.y = -1e30f;
  t.dtauh = ld(fm::DTAUH); t.dtaul = ld(fm::DTAUL);
  t.nm1 = bc<float2>(M.nm1f);
  if constexpr (KIND != C8R_UNIFORM) {
    t.Eh = ld(fm::EMH); t.El = ld(fm::EML);
    t.nm1 = mul_rn(bc<float2>(M.N0f), t.Eh);
  }
  if constexpr (KIND == C8R_EXPONENTIAL_SPHERICAL) {
    // n - 1 at the midpoint over the sphere, as load_track_mixed has it
    t.nm1.x *= expf(-sphere_excess(t.mx.x, t.my.x, t.mz.x, M.RE_f) * M.invH_h);
    t.nm1.y *= expf(-sphere_excess(t.mx.y, t.my.y, t.mz.y, M.RE_f) * M.invH_h);
  }
  if constexpr (FLAT) {
    // per track as the per-pair arithmetic forms it, so the same values
    float2 dzh, dzl, q0, q1;
    two_sum(bc<float2>(M.flat_zh), neg(t.mz), dzh, dzl);
    dzl = add_rn(dzl, sub_rn(bc<float2>(M.flat_zl), t.mzl));
    refr_quotient(M, M.flat_Eh, M.flat_El, dzh.x, dzl.x, t.Eh.x, t.El.x, q0.x, q1.x);
    refr_quotient(M, M.flat_Eh, M.flat_El, dzh.y, dzl.y, t.Eh.y, t.El.y, q0.y, q1.y);
    t.zm = z_part(dzh, dzl, t.bz);
    t.Eh = q0;
    t.El = q1;
    if constexpr (KIND == C8R_EXPONENTIAL_SPHERICAL) t.set(M, t.mx, t.my, t.mz, dzh);
    if constexpr (KIND == C8R_EXPONENTIAL_RAY) t.set(M, t.nm1, dzh);
  }
}

// an antenna in shared memory for those kernels, each value twice
struct alignas(16) AntZ {
  float2 x, y, xl, yl, tauh, taul, z, zl, Eh, El;
  float pad[4];
};
static_assert(sizeof(AntZ) == sizeof(AntRec), "fwd_layout reckons with one antenna record size");

// geometry shared by the forward and the adjoint Endpoint evaluation
struct EndpointEvalM {
  GeoM g0, g1, gm;
  FieldM f0, f1, fm;
  int branch;     // 0 two endpoints, 1 midpoint
  ff ua, ub;      // arrivals (start/end, or the two linearised midpoint arrivals)
  bool valid;
  float dop0, dop1;  // curved rays: optical-path change of the start and end paths (m)
};

// curved rays (C8R_EXPONENTIAL_RAY): turn the direction of g (a copy used for
// the field arithmetic; the straight geometry stays with the arrival time and
// the amplitude's R) and return the ray's optical-path change and the change of
// D = 1 - n beta.rhat that the turn makes
__device__ __forceinline__ float ray_turn(const GeoM& g, float nu_e, const MedParams& M, float t[3]) {
  const float dx = g.s[0], dy = g.s[1], dz = g.s[2], R = g.R0;
  const RayFix<float> r = ray_fix<float, 1>(dx * dx + dy * dy, dz, R, nu_e, M.invH_h);
  ray_turn_vector<float>(dx, dy, dz, R, r.Q, t);
  return r.dop;
}
__device__ __forceinline__ void ray_turn_mixed(GeoM& g, float nu_e, float bx, float by, float bz, const MedParams& M,
                                               float& dop, float& dD) {
  float t[3];
  dop = ray_turn(g, nu_e, M, t);
  g.s[0] = __fadd_rn(g.s[0], t[0]);
  g.s[1] = __fadd_rn(g.s[1], t[1]);
  g.s[2] = __fadd_rn(g.s[2], t[2]);
  dD = -(1.0f + nu_e) * (bx * t[0] + by * t[1] + bz * t[2]) * g.y;
}

// D in float-float plus a small FP32 change, renormalised
template <typename T>
__device__ __forceinline__ ffT<T> ff_add_small(ffT<T> D, T d) {
  T h, l;
  two_sum(D.h, d, h, l);
  l = add_rn(l, D.l);
  ffT<T> r;
  r.h = add_rn(h, l);
  r.l = sub_rn(l, sub_rn(r.h, h));
  return r;
}

// Endpoint evaluation in three steps, shared by the forward pass (which runs
// the near-Cherenkov pairs apart from the others) and the adjoint.
// (1) propagator and field at both endpoints; false when an emission point
// sits on the antenna (outside the domain of the formula)
template <int KIND>
__device__ __forceinline__ bool endpoint_fields(const TrackM& t, const AntRec& A, const MedParams& M,
                                                EndpointEvalM& e) {
  geo_lite(A, t.x0, t.y0, t.z0, e.g0);
  geo_lite(A, t.x1, t.y1, t.z1, e.g1);
  if (e.g0.R0 == 0.0f || e.g1.R0 == 0.0f) return false;
  if constexpr (KIND == C8R_EXPONENTIAL_RAY) {
    // the field along the ray's direction at each endpoint
    GeoM r0 = e.g0, r1 = e.g1;
    float dD;
    ray_turn_mixed(r0, t.nm1_0, t.bx, t.by, t.bz, M, e.dop0, dD);
    ray_turn_mixed(r1, t.nm1_1, t.bx, t.by, t.bz, M, e.dop1, dD);
    field_mixed(r0, t.bx, t.by, t.bz, t.bmag, t.om0, __fadd_rn(1.0f, t.nm1_0), e.f0);
    field_mixed(r1, t.bx, t.by, t.bz, t.bmag, t.om1, __fadd_rn(1.0f, t.nm1_1), e.f1);
  } else {
    e.dop0 = e.dop1 = 0.0f;
    field_mixed(e.g0, t.bx, t.by, t.bz, t.bmag, t.om0, __fadd_rn(1.0f, t.nm1_0), e.f0);
    field_mixed(e.g1, t.bx, t.by, t.bz, t.bmag, t.om1, __fadd_rn(1.0f, t.nm1_1), e.f1);
  }
  return true;
}

// the near-Cherenkov test: min(|D_start|, |D_end|) < eps_C
__device__ __forceinline__ bool endpoint_near_cherenkov(const EndpointEvalM& e, const MedParams& M) {
  return !(fminf(fabsf(e.f0.D), fabsf(e.f1.D)) >= M.eps_C);
}

// (2a) arrival positions of the two endpoints
template <int KIND>
__device__ __forceinline__ void endpoint_arrivals(const TrackM& t, const AntRec& A, const MedParams& M,
                                                  EndpointEvalM& e) {
  GeoM g0 = e.g0, g1 = e.g1;
  geo_refine(g0);
  geo_refine(g1);
  e.ua = arrival_mixed<KIND>(M, A, g0, t.tau0h, t.tau0l, t.E0h, t.E0l, e.dop0);
  e.ub = arrival_mixed<KIND>(M, A, g1, t.tau1h, t.tau1l, t.E1h, t.E1l, e.dop1);
  e.branch = 0;
}

// (2b) near-Cherenkov: midpoint geometry and the linearised arrivals
// t_m -/+ D_m (t1 - t0)/2; false when the midpoint sits on the antenna
template <int KIND>
__device__ __forceinline__ bool endpoint_midpoint(const TrackM& t, const AntRec& A, const MedParams& M,
                                                  EndpointEvalM& e) {
  float dopm = 0.0f, dDm = 0.0f;
  if constexpr (KIND == C8R_EXPONENTIAL_RAY) {
    // the midpoint's own ray (its direction is not the mean of the endpoints')
    float mx, mxl, my, myl, mz, mzl;
    two_sum(t.x0, t.x1, mx, mxl);
    two_sum(t.y0, t.y1, my, myl);
    two_sum(t.z0, t.z1, mz, mzl);
    geo_lite(A, 0.5f * mx, 0.5f * my, 0.5f * mz, 0.5f * mxl, 0.5f * myl, 0.5f * mzl, e.gm);
    if (e.gm.R0 == 0.0f) return false;
    GeoM r = e.gm;
    ray_turn_mixed(r, t.nm1_m, t.bx, t.by, t.bz, M, dopm, dDm);
    field_mixed(r, t.bx, t.by, t.bz, t.bmag, t.om_m, __fadd_rn(1.0f, t.nm1_m), e.fm);
  } else {
    midpoint_from_endpoints(e.g0, e.g1, e.f0, e.f1, t.bmag, t.om_m, __fadd_rn(1.0f, t.nm1_m), e.gm, e.fm);
    if (e.gm.R0 == 0.0f) return false;
  }
  GeoM g = e.gm;
  geo_refine(g);
  const ff u0 = arrival_mixed<KIND>(M, A, g, t.tmh, t.tml, t.Emh, t.Eml, dopm);
  ff Dm = doppler_ff(g, t.bx, t.by, t.bz, t.nm1_m);
  if constexpr (KIND == C8R_EXPONENTIAL_RAY) Dm = ff_add_small(Dm, dDm);
  // the amplitude's 1/D_m, too, from the float-float D: here |D_m| can be far
  // below the FP32 form's absolute accuracy
  e.fm.D = __fadd_rn(Dm.h, Dm.l);
  float hh, hl;  // D_m (t1 - t0)/(2 dt), float-float
  two_prod(Dm.h, t.dtauh, hh, hl);
  hl = __fmaf_rn(Dm.h, t.dtaul, __fmaf_rn(Dm.l, t.dtauh, hl));
  hh *= 0.5f;
  hl *= 0.5f;
  two_sum(u0.h, -hh, e.ua.h, e.ua.l);
  e.ua.l = __fadd_rn(e.ua.l, __fsub_rn(u0.l, hl));
  two_sum(u0.h, hh, e.ub.h, e.ub.l);
  e.ub.l = __fadd_rn(e.ub.l, __fadd_rn(u0.l, hl));
  e.branch = 1;
  return true;
}

template <int KIND>
__device__ __forceinline__ void endpoint_eval_mixed(const TrackM& t, const AntRec& A, const MedParams& M,
                                                    EndpointEvalM& e) {
  e.valid = false;
  if (!endpoint_fields<KIND>(t, A, M, e)) return;
  if (endpoint_near_cherenkov(e, M)) {
    if (!endpoint_midpoint<KIND>(t, A, M, e)) return;
  } else {
    endpoint_arrivals<KIND>(t, A, M, e);
  }
  e.valid = true;
}

// Linear (two-bin) deposit (reading LD): a deposit arriving at u is spread over
// [u - 1/2, u + 1/2].  With J = floor(u + 1/2) (the "cell" between the bin
// centres J - 1/2 and J + 1/2) and s = u + 1/2 - J, bins J - 1 and J receive
// 1 - s and s of it.  Cells outside [0, N] touch no bin of the window; bin_raw
// clamps them to -1 or N + 1.
__device__ __forceinline__ int lin_cell(ff u, int N, float& s) {
  ff v;
  two_sum(u.h, 0.5f, v.h, v.l);
  v.l = __fadd_rn(v.l, u.l);
  return bin_raw(v, N + 1, s);
}

// ZHS with the linear deposit, an interval [u_lo, u_hi] over more than one cell:
// the tent weights averaged over it, for the bins around its two ends (per unit
// of the whole interval's deposit); every bin strictly between them receives
// 1/W.  First cell: bins J_lo - 1 and J_lo get (1 - s_lo)^2/2 and
// (1 - s_lo^2)/2; last cell: J_hi - 1 and J_hi get s_hi (1 - s_hi/2) and
// s_hi^2/2; every whole cell in between gives 1/2 to each of its two bins.
struct LinEnds {
  int k[4];
  float w[4];
  int n;
};
__device__ __forceinline__ LinEnds lin_ends(int Jlo, float slo, int Jhi, float shi, float invW) {
  const float a = 1.0f - slo;
  const float lo0 = 0.5f * a * a, lo1 = 0.5f * (1.0f - slo * slo);
  const float hi0 = shi * (1.0f - 0.5f * shi), hi1 = 0.5f * shi * shi;
  LinEnds z;
  z.k[0] = Jlo - 1;
  z.w[0] = lo0 * invW;
  z.k[1] = Jlo;
  if (Jhi == Jlo + 1) {
    z.w[1] = (lo1 + hi0) * invW;
    z.k[2] = Jhi;
    z.w[2] = hi1 * invW;
    z.k[3] = -1;
    z.w[3] = 0.0f;
    z.n = 3;
  } else {
    z.w[1] = (lo1 + 0.5f) * invW;
    z.k[2] = Jhi - 1;
    z.w[2] = (hi0 + 0.5f) * invW;
    z.k[3] = Jhi;
    z.w[3] = hi1 * invW;
    z.n = 4;
  }
  return z;
}

template <int FORM, int KIND, bool LIN = false, int AF = kFormDirect, bool FLAT = false>
struct OpsMixed {
  using acc_t = float;
  using Track = TrackM;
  static constexpr int kPrec = C8R_MIXED;
  static constexpr int kTileBytes = kTileBytesMixed;
  // CTAs of 128 threads per SM the register budget is set for (curved rays
  // carry the ray solve as well, and the spherical Endpoint kernel its
  // curvature quadrature: fewer CTAs, more registers each; the spherical one at
  // 5 CTAs has no spills and is 1.6 % faster than at 6)
  static constexpr int kMinBlocks =
      FORM == C8R_ENDPOINT ? (KIND == C8R_EXPONENTIAL_RAY ? 4 : (KIND == C8R_EXPONENTIAL_SPHERICAL ? 5 : 6))
                           : (KIND == C8R_EXPONENTIAL_RAY || (KIND == C8R_EXPONENTIAL_SPHERICAL && FLAT) ? 6 : 8);
  // Endpoint: the near-Cherenkov pairs (a minority, spread over most warps)
  // are set aside by the main pass and evaluated together afterwards
  static constexpr bool kDefers = FORM == C8R_ENDPOINT;
  // Endpoint with the one-bin deposit in the plain straight-line media: the
  // main pass takes each bin from the FP32 arrival with its error bound
  // (arrival_fast, decide_bins) and sets aside only the endpoints it cannot decide,
  // for the float-float arrival after the main pass
  static constexpr bool kFastBins =
      FORM == C8R_ENDPOINT && !LIN && (KIND == C8R_UNIFORM || KIND == C8R_EXPONENTIAL);
  // ZHS in those media, and in the others for a flat array: the forward kernel
  // evaluates two tracks at a time
  static constexpr bool kTwoTracks = FORM == C8R_ZHS && (KIND == C8R_UNIFORM || KIND == C8R_EXPONENTIAL || FLAT);
  static constexpr int kFwdThreads = kTwoTracks ? kTileT / 2 : kTileT;
  // the form of x = R - w in the FP32 arrival (arrival_fast): the split one
  // for lines of sight near the vertical, the direct one otherwise.  Either is
  // exact to its own bound; the host picks the kernel per launch from the
  // share of tracks that see the antenna array from above within 45 degrees
  // (counted by the ingest of earlier launches)
  static constexpr int kAF = kFastBins ? AF : kFormDirect;
  // a flat antenna array: the refractivity quotient per track, in the one-bin
  // Endpoint kernels and in the ZHS forward and adjoint kernels, which also take
  // the z part of the midpoint's d once per track (ZPart; the host picks the
  // kernel, MedParams::flat).  Both the per-pair quotient and its operands leave
  // the pair's registers.  Endpoint, per-pair quotient -> per track: 4e6-track
  // vertical shower x 160 antennas (split form) 4.71 -> 4.58 ms; adjoint on 1e6
  // tracks x 64 antennas 963 -> 942 us (split), 1039 -> 988 (axis); 64 uneven
  // showers in a batch 2.99 -> 2.96 ms.  ZHS, one track per thread, 2e7-track
  // vertical shower: 31.96 -> 29.56 ms, and 28.50 with the z part as well
  static constexpr bool kFlat = FLAT && KIND != C8R_UNIFORM && (kFastBins || FORM == C8R_ZHS);
  // the main pass's Doppler factor with its last product and sum fused: in the
  // direct and axis kernels without a per-pair quotient, where the assembler had made
  // them one operation; apart in the others, as in the plain arithmetic.  Either is
  // within a rounding, but the near-Cherenkov decision is taken from it, so each
  // kernel states which it has: its forward pass, adjoint and listing agree
  static constexpr bool kFusedD = kFastBins && AF != kFormSplit && (KIND == C8R_UNIFORM || FLAT);
  // adjoint CTAs (128 threads) per SM the registers are set for (the linear
  // Endpoint adjoint carries the slide of each deposit as well)
  static constexpr int kBwdMinBlocks = (LIN && FORM == C8R_ENDPOINT) ? 4 : (kFastBins ? 5 : 6);
  // resident CTAs per SM that the adjoint's track ranges are cut for
  static constexpr int kBwdGridBlocks = (LIN && FORM == C8R_ENDPOINT) ? 4 : 6;
  // ZHS: a second accumulator row holds the edges of box deposits
  static constexpr int kAccRows = FORM == C8R_ZHS ? 2 : 1;

  // the antenna record that the forward and adjoint kernels hold in shared memory
  using FwdAnt = std::conditional_t<kTwoTracks, AntZ, std::conditional_t<kFastBins, AntE, AntRec>>;
  using Ant = std::conditional_t<kFastBins, AntE, AntRec>;
  static __device__ __forceinline__ void stage_ant(AntZ* p, const AntRec& A, const MedParams&) {
    AntZ z;
    z.x = bc<float2>(A.xh); z.y = bc<float2>(A.yh); z.z = bc<float2>(A.zh);
    z.xl = bc<float2>(A.xl); z.yl = bc<float2>(A.yl); z.zl = bc<float2>(A.zl);
    z.tauh = bc<float2>(A.tauh); z.taul = bc<float2>(A.taul);
    z.Eh = bc<float2>(A.Eah); z.El = bc<float2>(A.Eal);
    z.pad[0] = z.pad[1] = z.pad[2] = z.pad[3] = 0.0f;
    *p = z;
  }
  static __device__ __forceinline__ AntRec load_ant(const AntZ* p) {
    AntRec r;
    r.xh = p->x.x; r.yh = p->y.x; r.zh = p->z.x;
    r.xl = p->xl.x; r.yl = p->yl.x; r.zl = p->zl.x;
    r.tauh = p->tauh.x; r.taul = p->taul.x;
    r.Eah = p->Eh.x; r.Eal = p->El.x;
    return r;
  }
  static __device__ __forceinline__ void stage_ant(Ant* p, const AntRec& A, const MedParams& M) {
    if constexpr (kFastBins) {
      AntE e;
      e.x = bc<float2>(A.xh); e.y = bc<float2>(A.yh); e.z = bc<float2>(A.zh);
      e.Th = bc<float2>(A.Tah); e.Tl = bc<float2>(A.Tal);
      e.Eh = bc<float2>(A.Eah); e.El = bc<float2>(A.Eal);
      e.fb_abs = A.fb_abs; e.fb_rel_v = A.fb_rel_v;
      e.xl = A.xl; e.yl = A.yl; e.zl = A.zl; e.tauh = A.tauh; e.taul = A.taul;
      e.pad[0] = e.pad[1] = e.pad[2] = 0.0f;
      if constexpr (kAF == kFormAxis) {
        // the antenna's shifted time along the axis, and 16 u^2 of it for the bound
        const float ph[3] = {A.xh, A.yh, A.zh}, pl[3] = {A.xl, A.yl, A.zl};
        float Th, Tl;
        axis_time(M, A.tauh, A.taul, ph, pl, Th, Tl);
        e.Th = bc<float2>(Th);
        e.Tl = bc<float2>(Tl);
        e.fb_abs = __fmaf_rn(5.7e-14f, fabsf(Th), e.fb_abs);
      }
      *p = e;
    } else {
      *p = A;
    }
  }
  // the float-float part of an antenna record (loads whose fields a pass does
  // not use are dropped by the compiler)
  static __device__ __forceinline__ AntRec load_ant(const Ant* p) {
    AntRec r;
    if constexpr (kFastBins) {
      r.xh = p->x.x; r.yh = p->y.x; r.zh = p->z.x;
      r.xl = p->xl; r.yl = p->yl; r.zl = p->zl;
      r.tauh = p->tauh; r.taul = p->taul;
      r.Eah = p->Eh.x; r.Eal = p->El.x;
      r.Tah = p->Th.x; r.Tal = p->Tl.x;
      r.fb_abs = p->fb_abs; r.fb_rel_v = p->fb_rel_v;
    } else {
      // three 16-byte loads
      const float4* f = reinterpret_cast<const float4*>(&p->xh);
      const float4 a = f[0], b = f[1], c = f[2];
      r.xh = a.x; r.yh = a.y; r.zh = a.z; r.xl = a.w;
      r.yl = b.x; r.zl = b.y; r.tauh = b.z; r.taul = b.w;
      r.Eah = c.x; r.Eal = c.y;
    }
    return r;
  }

  static __device__ __forceinline__ void load(const void* Tv, int l, const MedParams& M, TrackM& t) {
    load_track_mixed<FORM, KIND, kFlat>(static_cast<const float*>(Tv), l, M, t);
  }
  // the track as the main passes hold it
  using MainTrack = std::conditional_t<kFastBins, TrackE, TrackM>;
  static __device__ __forceinline__ void load_main(const void* Tv, int l, const MedParams& M, MainTrack& t) {
    if constexpr (kFastBins)
      load_track_endpoints<KIND, kAF, kFlat>(static_cast<const float*>(Tv), l, M, t);
    else
      load(Tv, l, M, t);
  }
  static __device__ __forceinline__ bool live(const TrackE& t) { return t.amp != 0.0f; }
  static __device__ __forceinline__ bool live(const TrackZ<KIND>& t) { return t.live; }
  // what a thread of the forward main pass holds: a track, or two of them
  using FwdTrack = std::conditional_t<kTwoTracks, TrackZ<KIND>, MainTrack>;
  static __device__ __forceinline__ void load_fwd(const void* Tv, int l, const MedParams& M, FwdTrack& t) {
    if constexpr (kTwoTracks)
      load_track_pair<KIND, kFlat>(static_cast<const float*>(Tv), l, M, t);
    else
      load_main(Tv, l, M, t);
  }
  static __device__ __forceinline__ bool live(const TrackM& t) { return t.amp != 0.0f; }

  // -------------------------------------------------------------------------
  // Endpoint (§1; James et al.): +amp V/(D R) at the start's arrival bin and
  // -amp V/(D R) at the end's, amp = q K / dt; midpoint form near Cherenkov.
  // -------------------------------------------------------------------------
  // The deposits of an evaluated pair; the evaluation is split between
  // pair_main and pair_deferred below.
  // a deposit (x, y, z) arriving in cell J at s, spread over bins J - 1 and J
  template <class Sink>
  static __device__ __forceinline__ void dep_lin(Sink& out, int N, int J, float s, float x, float y, float z) {
    const float r = 1.0f - s;
    if (J >= 1 && J - 1 < N) out.dep(J - 1, x * r, y * r, z * r);
    if (J >= 0 && J < N) out.dep(J, x * s, y * s, z * s);
  }

  // Endpoint deposits spread over two bins each (reading LD).  Near Cherenkov,
  // when both linearised arrivals lie in one cell J, the two spread deposits
  // +/- amp V/(D R) combine to the exact amp (dt_e/dt) V/R into bin J - 1 and
  // its negative into bin J, with no division by D.
  template <class Sink>
  static __device__ __forceinline__ void endpoint_deposit_lin(const TrackM& t, const EndpointEvalM& e,
                                                              const MedParams& M, Sink& out) {
    const int N = M.n_bins;
    out.rec(e.branch, e.ua, e.ub);
    float sa, sb;
    const int Ja = lin_cell(e.ua, N, sa);
    const int Jb = lin_cell(e.ub, N, sb);
    const float amp = t.amp;
    if (e.branch == 0) {
      const float c0 = div_ap(amp, e.f0.D * e.g0.R0) * (e.f0.invR * e.f0.invR);
      const float c1 = div_ap(-amp, e.f1.D * e.g1.R0) * (e.f1.invR * e.f1.invR);
      if (Ja == Jb) {
        // both in one cell: add them in registers, two reductions
        const float a0 = c0 * (1.0f - sa), b0 = c1 * (1.0f - sb), a1 = c0 * sa, b1 = c1 * sb;
        if (Ja >= 1 && Ja - 1 < N)
          out.dep(Ja - 1, a0 * e.f0.V[0] + b0 * e.f1.V[0], a0 * e.f0.V[1] + b0 * e.f1.V[1],
                  a0 * e.f0.V[2] + b0 * e.f1.V[2]);
        if (Ja >= 0 && Ja < N)
          out.dep(Ja, a1 * e.f0.V[0] + b1 * e.f1.V[0], a1 * e.f0.V[1] + b1 * e.f1.V[1],
                  a1 * e.f0.V[2] + b1 * e.f1.V[2]);
      } else {
        dep_lin(out, N, Ja, sa, c0 * e.f0.V[0], c0 * e.f0.V[1], c0 * e.f0.V[2]);
        dep_lin(out, N, Jb, sb, c1 * e.f1.V[0], c1 * e.f1.V[1], c1 * e.f1.V[2]);
      }
      return;
    }
    const float i2 = e.fm.invR * e.fm.invR;
    if (Ja == Jb) {
      const float c = amp * t.dtauh * (i2 * e.fm.invR);
      if (Ja >= 1 && Ja - 1 < N) out.dep(Ja - 1, c * e.fm.V[0], c * e.fm.V[1], c * e.fm.V[2]);
      if (Ja >= 0 && Ja < N) out.dep(Ja, -c * e.fm.V[0], -c * e.fm.V[1], -c * e.fm.V[2]);
      return;
    }
    const float c = div_ap(amp, e.fm.D * e.gm.R0) * i2;
    dep_lin(out, N, Ja, sa, c * e.fm.V[0], c * e.fm.V[1], c * e.fm.V[2]);
    dep_lin(out, N, Jb, sb, -c * e.fm.V[0], -c * e.fm.V[1], -c * e.fm.V[2]);
  }

  template <class Sink>
  static __device__ __forceinline__ void endpoint_deposit(const TrackM& t, const EndpointEvalM& e,
                                                          const MedParams& M, Sink& out) {
    if constexpr (LIN) {
      endpoint_deposit_lin(t, e, M, out);
      return;
    }
    const int N = M.n_bins;
    out.rec(e.branch, e.ua, e.ub);
    float fa, fb;
    const int ka = bin_raw(e.ua, N, fa);
    const int kb = bin_raw(e.ub, N, fb);
    const bool ina = ka >= 0 && ka < N, inb = kb >= 0 && kb < N;
    const float amp = t.amp;
    if (e.branch == 0) {
      const float c0 = div_ap(amp, e.f0.D * e.g0.R0) * (e.f0.invR * e.f0.invR);
      const float c1 = div_ap(-amp, e.f1.D * e.g1.R0) * (e.f1.invR * e.f1.invR);
      if (ina && inb && ka == kb) {
        // both deposits in one bin: add them in registers, one reduction
        out.dep(ka, c0 * e.f0.V[0] + c1 * e.f1.V[0], c0 * e.f0.V[1] + c1 * e.f1.V[1],
                c0 * e.f0.V[2] + c1 * e.f1.V[2]);
      } else {
        if (ina) out.dep(ka, c0 * e.f0.V[0], c0 * e.f0.V[1], c0 * e.f0.V[2]);
        if (inb) out.dep(kb, c1 * e.f1.V[0], c1 * e.f1.V[1], c1 * e.f1.V[2]);
      }
      return;
    }
    if (ka == kb) return;  // one bin (or both outside on one side): the bin average of E vanishes
    const float c = div_ap(amp, e.fm.D * e.gm.R0) * (e.fm.invR * e.fm.invR);
    if (ina) out.dep(ka, c * e.fm.V[0], c * e.fm.V[1], c * e.fm.V[2]);
    if (inb) out.dep(kb, -c * e.fm.V[0], -c * e.fm.V[1], -c * e.fm.V[2]);
  }

  // -------------------------------------------------------------------------
  // ZHS (§1; Zas, Halzen & Stanev): bin averages of the midpoint step
  // potential K_A beta_perp/(R |D|) over [t_m - |D| dt_e/2, t_m + |D| dt_e/2];
  // written as (K_A beta_perp dt_e/(R dt)) x (fraction of the interval in the
  // bin), which needs no division by D and is exact for a one-bin interval.
  // -------------------------------------------------------------------------
  template <class Sink>
  static __device__ __forceinline__ void zhs(const TrackM& t, const AntRec& A, const MedParams& M, Sink& out) {
    const int N = M.n_bins;
    GeoM gm;
    if constexpr (kFlat)
      geo_lite(A.xh, A.yh, A.xl, A.yl, t.mx, t.my, t.mxl, t.myl, t.zm, gm);
    else
      geo_lite(A, t.mx, t.my, t.mz, t.mxl, t.myl, t.mzl, gm);
    if (gm.R0 == 0.0f) return;
    FieldM f;
    float dop = 0.0f, dD = 0.0f;
    if constexpr (KIND == C8R_EXPONENTIAL_RAY) {
      GeoM r = gm;
      ray_turn_mixed(r, t.nm1_m, t.bx, t.by, t.bz, M, dop, dD);
      field_mixed(r, t.bx, t.by, t.bz, t.bmag, t.om_m, __fadd_rn(1.0f, t.nm1_m), f);
    } else {
      field_mixed(gm, t.bx, t.by, t.bz, t.bmag, t.om_m, __fadd_rn(1.0f, t.nm1_m), f);
    }
    ff um, aD;
    if constexpr (kFlat) {
      geo_refine(gm, t.zm);
      if constexpr (KIND == C8R_EXPONENTIAL_SPHERICAL)
        dop = sphere_path_correction<float>(A.xh, A.yh, A.zh, gm.s[0], gm.s[1], gm.s[2], gm.R0, M.N0f, M.invH_h, M.RE_f);
      um = arrival_mixed_q<KIND>(M, A.tauh, A.taul, gm, t.tmh, t.tml, t.qmh, t.qml, dop);
      aD = doppler_ff(gm, t.bx, t.by, t.zm, t.nm1_m);
    } else {
      geo_refine(gm);
      um = arrival_mixed<KIND>(M, A, gm, t.tmh, t.tml, t.Emh, t.Eml, dop);
      aD = doppler_ff(gm, t.bx, t.by, t.bz, t.nm1_m);
    }
    if constexpr (KIND == C8R_EXPONENTIAL_RAY) aD = ff_add_small(aD, dD);
    if (aD.h < 0.0f) {
      aD.h = -aD.h;
      aD.l = -aD.l;
    }
    float hh, hl;  // |D| (t1 - t0)/(2 dt), float-float
    two_prod(aD.h, t.dtauh, hh, hl);
    hl = __fmaf_rn(aD.h, t.dtaul, __fmaf_rn(aD.l, t.dtauh, hl));
    hh *= 0.5f;
    hl *= 0.5f;
    ff ulo, uhi;
    two_sum(um.h, -hh, ulo.h, ulo.l);
    ulo.l = __fadd_rn(ulo.l, __fsub_rn(um.l, hl));
    two_sum(um.h, hh, uhi.h, uhi.l);
    uhi.l = __fadd_rn(uhi.l, __fadd_rn(um.l, hl));
    const float s = -t.amp * (f.invR * f.invR) * f.invR;  // beta_perp = -V
    const float Mx = s * f.V[0], My = s * f.V[1], Mz = s * f.V[2];
    float flo, fhi;
    const int klo = bin_raw(ulo, N, flo);
    const int khi = bin_raw(uhi, N, fhi);
    out.rec(klo == khi ? 2 : 3, ulo, uhi);
    if constexpr (LIN) {
      zhs_deposit_lin(ulo, uhi, hh, Mx, My, Mz, N, out);
    } else {
      const float invW = div_ap(1.0f, 2.0f * hh);  // 1 / interval length in bins (unused when in one bin)
      zhs_deposit(klo, khi, klo == khi ? 1.0f : gap_to_next_edge(ulo, klo) * invW, fhi * invW, invW, Mx, My, Mz, N, out);
    }
  }

  // the deposits of an evaluated ZHS interval [ulo, uhi] (bins klo, khi; M the
  // whole deposit, invW = 1/W): the first bin takes it all (an interval inside
  // one bin: weight 1, M x 1 = M exactly) or the share it covers, in one
  // reduction either way, so that lanes of both kinds take one path; the partly
  // covered last bin; and the whole bins in between, which all receive M / W
  template <class Sink>
  static __device__ __forceinline__ void zhs_deposit(int klo, int khi, float wlo, float whi, float invW, float Mx,
                                                     float My, float Mz, int N, Sink& out) {
    if ((unsigned)klo < (unsigned)N && wlo > 0.0f) out.dep(klo, Mx * wlo, My * wlo, Mz * wlo);
    if (klo == khi) return;
    if ((unsigned)khi < (unsigned)N && whi > 0.0f) out.dep(khi, Mx * whi, My * whi, Mz * whi);
    const int kb = klo + 1 < 0 ? 0 : klo + 1;
    const int ke = khi - 1 > N - 1 ? N - 1 : khi - 1;
    if (kb <= ke) out.dep_box(kb, ke, Mx * invW, My * invW, Mz * invW);
  }
  // the same for the linear deposit (reading LD): the tent weights averaged over
  // the interval
  template <class Sink>
  static __device__ __forceinline__ void zhs_deposit_lin(ff ulo, ff uhi, float hh, float Mx, float My, float Mz, int N,
                                                         Sink& out) {
    float slo, shi;
    const int Jlo = lin_cell(ulo, N, slo);
    const int Jhi = lin_cell(uhi, N, shi);
    if (Jlo == Jhi) {
      // inside one cell the tents are linear: the tent at the middle
      dep_lin(out, N, Jlo, 0.5f * (slo + shi), Mx, My, Mz);
      return;
    }
    const float invW = div_ap(1.0f, 2.0f * hh);
    const LinEnds z = lin_ends(Jlo, slo, Jhi, shi, invW);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i < z.n && z.k[i] >= 0 && z.k[i] < N) out.dep(z.k[i], Mx * z.w[i], My * z.w[i], Mz * z.w[i]);
    const int kb = Jlo + 1 < 0 ? 0 : Jlo + 1;
    const int ke = Jhi - 2 > N - 1 ? N - 1 : Jhi - 2;
    if (kb <= ke) out.dep_box(kb, ke, Mx * invW, My * invW, Mz * invW);
  }

  // ZHS of two tracks against one antenna, the arithmetic of `zhs` in both halves
  // (float2), with a sink for each: 302 -> 170 warp instructions per 32 pairs.
  // Bound by the FP32 pipe (63 % of its cycles, the float-float sums) and, for a
  // vertical shower on few antennas, by its reductions.  Measured with the
  // accumulator copies, ms: 2e7 tracks x 160 antennas 29.4 -> 25.6; 3e5 tracks x 512
  // antennas 1.61 -> 1.47.  What has a rarer form takes it half by half, and only
  // that part of the arithmetic does: the quotient's series (the altitude
  // difference within 1e-3 H) and the propagator's quadrature where the series of
  // PathZ does not hold.
  template <class Sink>
  static __device__ __forceinline__ void zhs_two(const TrackZ<KIND>& t, const AntZ& A, const MedParams& M, Sink& outx,
                                                 Sink& outy) {
    const int N = M.n_bins;
    GeoT<float2> g;
    ffT<float2> um, aD;
    if constexpr (kFlat) {
      geo_lite(A.x, A.y, A.xl, A.yl, t.mx, t.my, t.mxl, t.myl, t.zm, g);
      float2 corr = bc<float2>(0.0f), turn[3];
      if constexpr (KIND == C8R_EXPONENTIAL_SPHERICAL) {
        if (t.small) {
          corr = t.path(M, A.x, A.y, g);
        } else {
          corr.x = sphere_half<0>(A, M, g);
          corr.y = sphere_half<1>(A, M, g);
        }
      }
      if constexpr (KIND == C8R_EXPONENTIAL_RAY) {
        if (!t.path(g, corr, turn)) {
          float tx[3], ty[3];
          corr.x = ray_turn(half_of<0>(g), t.nm1.x, M, tx);
          corr.y = ray_turn(half_of<1>(g), t.nm1.y, M, ty);
#pragma unroll
          for (int c = 0; c < 3; ++c) turn[c] = make_float2(tx[c], ty[c]);
        }
      }
      geo_refine(g, t.zm);
      um = arrival_mixed_q<KIND>(M, A.tauh, A.taul, g, t.tmh, t.tml, t.Eh, t.El, corr);
      aD = doppler_ff(g, t.bx, t.by, t.zm, t.nm1);
      if constexpr (KIND == C8R_EXPONENTIAL_RAY) {
        // the field along the ray, and the change of D that the turn makes
        const float2 bt = fma_rn(t.bx, turn[0], fma_rn(t.by, turn[1], mul_rn(t.bz, turn[2])));
        aD = ff_add_small(aD, neg(mul_rn(mul_rn(add_rn(bc<float2>(1.0f), t.nm1), bt), g.y)));
#pragma unroll
        for (int c = 0; c < 3; ++c) g.s[c] = add_rn(g.s[c], turn[c]);
      }
    } else {
      float2 dzh, dzl, q0 = bc<float2>(0.0f), q1 = q0;
      two_sum(A.z, neg(t.mz), dzh, dzl);
      dzl = add_rn(dzl, sub_rn(A.zl, t.mzl));
      if constexpr (KIND == C8R_EXPONENTIAL) {
        if (fminf(fabsf(dzh.x), fabsf(dzh.y)) > -M.dz_series) {
          refr_quotient(M, A.Eh, A.El, dzh, dzl, t.Eh, t.El, q0, q1);
        } else {
          refr_quotient(M, A.Eh.x, A.El.x, dzh.x, dzl.x, t.Eh.x, t.El.x, q0.x, q1.x);
          refr_quotient(M, A.Eh.y, A.El.y, dzh.y, dzl.y, t.Eh.y, t.El.y, q0.y, q1.y);
        }
      }
      const ZPartT<float2> z = z_part(dzh, dzl, t.bz);
      geo_lite(A.x, A.y, A.xl, A.yl, t.mx, t.my, t.mxl, t.myl, z, g);
      geo_refine(g, z);
      um = arrival_mixed_q<KIND>(M, A.tauh, A.taul, g, t.tmh, t.tml, q0, q1);
      aD = doppler_ff(g, t.bx, t.by, z, t.nm1);
    }
    // |D|: D renormalised, so its sign is that of the high part
    if (aD.h.x < 0.0f) aD.l.x = -aD.l.x;
    if (aD.h.y < 0.0f) aD.l.y = -aD.l.y;
    aD.h = abs_of(aD.h);
    float2 hh, hl;  // |D| (t1 - t0)/(2 dt), float-float
    two_prod(aD.h, t.dtauh, hh, hl);
    hl = fma_rn(aD.h, t.dtaul, fma_rn(aD.l, t.dtauh, hl));
    const float2 half = bc<float2>(0.5f);
    hh = mul_rn(hh, half);
    hl = mul_rn(hl, half);
    ffT<float2> ulo, uhi;
    two_sum(um.h, neg(hh), ulo.h, ulo.l);
    ulo.l = add_rn(ulo.l, sub_rn(um.l, hl));
    two_sum(um.h, hh, uhi.h, uhi.l);
    uhi.l = add_rn(uhi.l, add_rn(um.l, hl));
    // the deposit A beta_perp/R = -A V, V R^2 = d x (d x beta)
    const float2 wx = fma_rn(g.s[1], t.bz, neg(mul_rn(g.s[2], t.by)));
    const float2 wy = fma_rn(g.s[2], t.bx, neg(mul_rn(g.s[0], t.bz)));
    const float2 wz = fma_rn(g.s[0], t.by, neg(mul_rn(g.s[1], t.bx)));
    const float2 s = mul_rn(mul_rn(t.amp, mul_rn(g.y, g.y)), g.y);
    const float2 Mx = mul_rn(s, fma_rn(g.s[1], wz, neg(mul_rn(g.s[2], wy))));
    const float2 My = mul_rn(s, fma_rn(g.s[2], wx, neg(mul_rn(g.s[0], wz))));
    const float2 Mz = mul_rn(s, fma_rn(g.s[0], wy, neg(mul_rn(g.s[1], wx))));
    const ff lox{ulo.h.x, ulo.l.x}, loy{ulo.h.y, ulo.l.y}, hix{uhi.h.x, uhi.l.x}, hiy{uhi.h.y, uhi.l.y};
    if constexpr (Sink::kRecords) {
      float f;
      outx.rec(bin_raw(lox, N, f) == bin_raw(hix, N, f) ? 2 : 3, lox, hix);
      outy.rec(bin_raw(loy, N, f) == bin_raw(hiy, N, f) ? 2 : 3, loy, hiy);
      return;
    }
    if constexpr (LIN) {
      zhs_deposit_lin(lox, hix, hh.x, Mx.x, My.x, Mz.x, N, outx);
      zhs_deposit_lin(loy, hiy, hh.y, Mx.y, My.y, Mz.y, N, outy);
    } else {
      const float2 invW = rcp_ap(mul_rn(bc<float2>(2.0f), hh));  // 1 / interval length in bins
      int klox, kloy, khix, khiy;
      float2 klo, khi, flo, fhi;
      bins_of(ulo, N, klox, kloy, klo, flo);
      bins_of(uhi, N, khix, khiy, khi, fhi);
      // gap_to_next_edge
      const float2 gap = sub_rn(sub_rn(add_rn(klo, bc<float2>(1.0f)), ulo.h), ulo.l);
      const float2 wlo = mul_rn(gap, invW), whi = mul_rn(fhi, invW);
      zhs_deposit(klox, khix, klox == khix ? 1.0f : wlo.x, whi.x, invW.x, Mx.x, My.x, Mz.x, N, outx);
      zhs_deposit(kloy, khiy, kloy == khiy ? 1.0f : wlo.y, whi.y, invW.y, Mx.y, My.y, Mz.y, N, outy);
    }
  }
  // the curvature quadrature of one half
  template <int J>
  static __device__ __forceinline__ float sphere_half(const AntZ& A, const MedParams& M, const GeoT<float2>& g) {
    return sphere_path_correction<float>(A.x.x, A.y.x, A.z.x, half_of<J>(g.s[0]), half_of<J>(g.s[1]),
                                         half_of<J>(g.s[2]), half_of<J>(g.R0), M.N0f, M.invH_h, M.RE_f);
  }

  // one endpoint of a pair in which some condition of the usual forms fails: its
  // arrival, bound and Doppler factor with each form chosen
  template <int J>
  static __device__ __forceinline__ void endpoint_rare(const TrackE& t, const AntE& A, const MedParams& M,
                                                       const GeoT<float2>& g2, float2 S, float2 P, float& uf,
                                                       float& eps, float& D) {
    const GeoM g = half_of<J>(g2);
    float q = 0.0f;
    if constexpr (kFlat)
      q = half_of<J>(t.q);
    else if constexpr (KIND == C8R_EXPONENTIAL)
      q = fast_quotient(M, A.Eh.x, A.El.x, g.s[2], half_of<J>(t.Eh), half_of<J>(t.El));
    eps = arrival_fast<KIND, kAF>(M, g, half_of<J>(S), half_of<J>(P), half_of<J>(t.Th), half_of<J>(t.Tl), A.Th.x,
                                     A.Tl.x, A.fb_abs, A.fb_rel_v, q, 0.0f, uf);
    FieldM f;
    field_mixed(g, t.bx, t.by, t.bz, t.bmag, half_of<J>(t.om), half_of<J>(t.n), f);
    D = f.D;
  }

  // the geometry, the field and the bins (arrival_fast in the form this kernel
  // is compiled for) of a pair's two endpoints; true for a near-Cherenkov pair.
  // An endpoint without a geometry (on the antenna, |d| = 0, or out of FP32's range)
  // has D = NaN and no bin.  The forward pass leaves it at that; the adjoint (ADJ)
  // sets the pair aside with the near ones (lone_end), to keep 0 x NaN out of its sums.
  // Both endpoints at once (float2): 291 -> 187 thread instructions per pair with
  // the set-aside bits (Aside).  Measured, ms: 4e6 tracks x 1024 antennas at 60
  // degrees 40.3 -> 36.9, 64 uneven showers 3.30 -> 3.03, the adjoint on 1e6
  // tracks x 64 antennas 1.23 -> 0.96 (5 CTAs per SM; 1.20 with 6, 1.11 with 4);
  // a vertical shower x 160 antennas, 5.65 -> 5.3 to 5.5, is bound by its
  // reductions (3.8 without them and the set-aside work)
  template <bool ADJ = false>
  static __device__ __forceinline__ bool endpoints_main(const TrackE& t, const AntE& A, const MedParams& M,
                                                        GeoT<float2>& g, FieldT<float2>& f, int& ka, int& kb) {
    float2 S, P, uf, q = bc<float2>(0.0f);
    geo_fast(A.x, A.y, A.z, t.x, t.y, t.z, g, S, P);
    if constexpr (kFlat)
      q = t.q;
    else if constexpr (KIND == C8R_EXPONENTIAL)
      q = fast_quotient(M, A.Eh, A.El, g.s[2], t.Eh, t.El);
    float2 eps = arrival_fast<KIND, kAF>(M, g, S, P, t.Th, t.Tl, A.Th, A.Tl, A.fb_abs, A.fb_rel_v, q, 0.0f, uf);
    field_mixed<float2, kFusedD>(g, bc<float2>(t.bx), bc<float2>(t.by), bc<float2>(t.bz), bc<float2>(t.bmag), t.om,
                                 t.n, f);
    // the usual forms: bd >= 0 (the Doppler factor); an altitude difference
    // beyond 1e-3 H, tested at 1.001e-3 H so that no rounding lets one through
    // (the refractivity quotient); an emission point above the antenna (the
    // split form); an antenna ahead of it along the axis (the axis form)
    bool usual = fminf(f.bd.x, f.bd.y) >= 0.0f;
    if constexpr (kAF == kFormAxis) {
      const float2 w = axis_w(M, g);
      usual = usual && fminf(w.x, w.y) >= 0.0f;
    }
    if constexpr (kAF == kFormSplit)
      usual = usual && fmaxf(g.s[2].x, g.s[2].y) < (KIND == C8R_EXPONENTIAL ? M.dz_series : 0.0f);
    else if constexpr (KIND == C8R_EXPONENTIAL && !kFlat)
      usual = usual && fminf(fabsf(g.s[2].x), fabsf(g.s[2].y)) > -M.dz_series;
    if (!usual) {
      endpoint_rare<0>(t, A, M, g, S, P, uf.x, eps.x, f.D.x);
      endpoint_rare<1>(t, A, M, g, S, P, uf.y, eps.y, f.D.y);
    }
    decide_bins(uf, eps, M.n_bins, ka, kb);
    const float d0 = fabsf(f.D.x), d1 = fabsf(f.D.y);
    return !((ADJ ? min_nan(d0, d1) : fminf(d0, d1)) >= M.eps_C);
  }

  // main pass: every pair except (Endpoint) the near-Cherenkov ones, for which
  // it deposits nothing and returns kDeferPair, and (kFastBins) the endpoints
  // whose bin the FP32 arrival leaves open, returned as kDeferEnd0/kDeferEnd1
  // bits after the other endpoint's deposit
  template <class Sink>
  static __device__ __forceinline__ int pair_main(const FwdTrack& t, const FwdAnt* p, const void* Tv, int l,
                                                  const MedParams& M, Sink& out) {
    if constexpr (kTwoTracks) {
      zhs_two(t, *p, M, out, out);
      return kDeferNone;
    } else if constexpr (kFastBins) {
      GeoT<float2> g;
      FieldT<float2> f;
      int ka, kb;
      const bool near = endpoints_main(t, *p, M, g, f, ka, kb);
      // decided and inside the window; no branch for near pairs, which almost
      // every warp holds one of
      const bool ina = ka >= 0 && !near, inb = kb >= 0 && !near;
      const float2 c = mul_rn(div_ap(make_float2(t.amp, -t.amp), mul_rn(f.D, g.R0)), mul_rn(f.invR, f.invR));
      // both deposits in one bin add in registers (one reduction); otherwise
      // one each.  One code path for both kinds of lane: the start's deposit
      // carries the end's when they share the bin (the end's weight 0 else)
      const bool same = ina && ka == kb;
      const float c1s = same ? c.y : 0.0f;
      const float2 dx = mul_rn(c, f.V[0]), dy = mul_rn(c, f.V[1]), dz = mul_rn(c, f.V[2]);
      if (ina)
        out.dep(ka, __fmaf_rn(c1s, f.V[0].y, dx.x), __fmaf_rn(c1s, f.V[1].y, dy.x), __fmaf_rn(c1s, f.V[2].y, dz.x));
      if (inb && !same) out.dep(kb, dx.y, dy.y, dz.y);
      const int ends = (ka == kFastUndecided ? kDeferEnd0 : 0) | (kb == kFastUndecided ? kDeferEnd1 : 0);
      return near ? kDeferPair : ends;
    } else if constexpr (FORM == C8R_ENDPOINT) {
      const AntRec A = load_ant(p);
      EndpointEvalM e;
      if (!endpoint_fields<KIND>(t, A, M, e)) return kDeferNone;
      if (endpoint_near_cherenkov(e, M)) return kDeferPair;
      endpoint_arrivals<KIND>(t, A, M, e);
      endpoint_deposit(t, e, M, out);
      return kDeferNone;
    } else {
      zhs(t, load_ant(p), M, out);
      return kDeferNone;
    }
  }

  // A near-Cherenkov pair (kFastBins) whose two linearised arrivals
  // u_m -/+ D_m (t1 - t0)/(2 dt) lie in one bin, or both before or both after
  // the window, contributes exactly 0 (reading C), and so does its adjoint.
  // Decided here from FP32 midpoint geometry, as decide_bins decides a
  // bin: the midpoint d_m = (s0 + s1)/2 from the endpoints' FP32 d (the
  // float-float path's high part; its roundings move each component by at most
  // 2u |s_i| + u L_i / 2, which moves x = R - w by at most 6u x + u L1 / 2, so
  // the arrival bound takes 3 more u k x and 2 u k L1, L1 >= L), the FP32
  // Doppler factor D_m (field_mixed: off the float-float D_m by at most
  // 8 u n + 16 u |D_m|, from the direction's rounding and its own), and two
  // more roundings on the interval ends.  True when the pair is decided to be
  // zero, false when the float-float evaluation must run (about 4 % of the
  // near-Cherenkov pairs of a shower).
  template <bool ADJ = false>
  static __device__ __forceinline__ bool near_zero_fast(const void* Tv, int l, const AntRec& A, const MedParams& M) {
    if constexpr (kFastBins) {
      constexpr float u = 5.9604644775390625e-8f;  // 2^-24
      const float* T = static_cast<const float*>(Tv);
      const float x0 = TF(fm::X0), y0 = TF(fm::Y0), z0 = TF(fm::Z0);
      const float x1 = TF(fm::X1), y1 = TF(fm::Y1), z1 = TF(fm::Z1);
      const float a0x = __fadd_rn(A.xh, -x0), a0y = __fadd_rn(A.yh, -y0), a0z = __fadd_rn(A.zh, -z0);
      const float a1x = __fadd_rn(A.xh, -x1), a1y = __fadd_rn(A.yh, -y1), a1z = __fadd_rn(A.zh, -z1);
      GeoM g;
      g.s[0] = 0.5f * __fadd_rn(a0x, a1x);
      g.s[1] = 0.5f * __fadd_rn(a0y, a1y);
      g.s[2] = 0.5f * __fadd_rn(a0z, a1z);
      const float rho2 = __fmaf_rn(g.s[0], g.s[0], __fmul_rn(g.s[1], g.s[1]));
      const float S = __fmaf_rn(g.s[2], g.s[2], rho2);
      g.y = rsqrt_ap(S);
      g.R0 = __fmul_rn(S, g.y);
      g.R1 = 0.0f;
      if (g.R0 == 0.0f) return true;  // the midpoint on the antenna: no deposit
      const float L1 = fabsf(__fsub_rn(a0x, a1x)) + fabsf(__fsub_rn(a0y, a1y)) + fabsf(__fsub_rn(a0z, a1z));
      // (adjoint) an endpoint on the antenna, at half the track's length from the
      // midpoint: not this form
      if constexpr (ADJ)
        if (g.R0 <= L1) return false;
      const float bx = TF(fm::BX), by = TF(fm::BY), bz = TF(fm::BZ), bmag = TF(fm::BMAG);
      float Eh = 1.0f, El = 0.0f, nm1 = M.nm1f;
      if (KIND != C8R_UNIFORM) {
        Eh = TF(fm::EMH);
        El = TF(fm::EML);
        nm1 = __fmul_rn(M.N0f, Eh);
      }
      const float om = __fsub_rn(TF(fm::OMB), __fmul_rn(nm1, bmag));
      FieldM f;
      field_mixed<float>(g, bx, by, bz, bmag, om, __fadd_rn(1.0f, nm1), f);
      // midpoint time (t0 + t1)/(2 dt), float-float, as load_track_mixed forms
      // it, shifted by k z_m at the exact midpoint height z_m = (z0 + z1)/2
      float tmh, tml;
      two_sum(TF(fm::TAU0H), TF(fm::TAU1H), tmh, tml);
      tml = __fadd_rn(tml, __fadd_rn(TF(fm::TAU0L), TF(fm::TAU1L)));
      tmh *= 0.5f;
      tml *= 0.5f;
      float zmh, zml;
      two_sum(z0, z1, zmh, zml);
      const float kh = KIND == C8R_UNIFORM ? M.s_h : M.kc_h, kl = KIND == C8R_UNIFORM ? M.s_l : M.kc_l;
      float Tmh, Tml;
      if constexpr (kAF == kFormAxis) {
        float xmh, xml, ymh, yml;
        two_sum(x0, x1, xmh, xml);
        two_sum(y0, y1, ymh, yml);
        const float ph[3] = {0.5f * xmh, 0.5f * ymh, 0.5f * zmh}, pl[3] = {0.5f * xml, 0.5f * yml, 0.5f * zml};
        axis_time(M, tmh, tml, ph, pl, Tmh, Tml);
      } else {
        shifted_time(tmh, tml, 0.5f * zmh, 0.5f * zml, kh, kl, Tmh, Tml);
      }
      float uf;
      const float qv = KIND == C8R_EXPONENTIAL ? fast_quotient<float>(M, A.Eah, A.Eal, g.s[2], Eh, El) : 0.0f;
      // the kernel's arrival form (either is exact to its own bound; one form
      // for every lane keeps the warp on one path)
      const float eps_a =
          arrival_fast<KIND, kAF, float>(M, g, S, rho2, Tmh, Tml, A.Tah, A.Tal, A.fb_abs, A.fb_rel_v, qv, 3.0f, uf);
      const float eps_u = __fmaf_rn(2.0f * u * kh, L1, eps_a);
      const float dtau = TF(fm::DTAUH);
      const float aD = fabsf(f.D);
      const float h = 0.5f * __fmul_rn(aD, dtau);
      const float dh = __fmul_rn(__fmaf_rn(16.0f * u, aD, 8.0f * u * __fadd_rn(1.0f, nm1)), dtau);
      const float e = __fadd_rn(__fadd_rn(eps_u, dh), 2.0f * u * __fadd_rn(fabsf(uf), h));
      const float lo = __fsub_rn(__fsub_rn(uf, h), e), hi = __fadd_rn(__fadd_rn(uf, h), e);
      return hi < 0.0f || lo >= (float)M.n_bins || floorf(lo) == floorf(hi);
    } else {
      return false;
    }
  }

  // one endpoint set aside by the main pass (kFastBins; `end` is kDeferEnd0 or
  // kDeferEnd1), read from the staged tile (lane l): its float-float arrival
  // decides the bin.  The endpoint's fields are picked by index, so lanes with
  // different endpoints run one code path and only one endpoint's values are
  // live; they are formed as load_track_mixed forms them, and the deposit is
  // the one the main pass would have made (the same geometry and field
  // functions, so the same values)
  template <class Sink>
  static __device__ __forceinline__ void end_deferred(const void* Tv, int l, const AntRec& A, const MedParams& M,
                                                      Sink& out, int end) {
    if constexpr (kFastBins) {
      const float* T = static_cast<const float*>(Tv);
      const int N = M.n_bins;
      const int j = end == kDeferEnd1 ? 1 : 0;
      const float amp = TF(fm::AMPE);
      const float bx = TF(fm::BX), by = TF(fm::BY), bz = TF(fm::BZ), bmag = TF(fm::BMAG);
      float Eh = 1.0f, El = 0.0f, nm1 = M.nm1f;
      if (KIND != C8R_UNIFORM) {
        Eh = TF(fm::E0H + 2 * j);
        El = TF(fm::E0L + 2 * j);
        nm1 = __fmul_rn(M.N0f, Eh);
      }
      const float om = __fsub_rn(TF(fm::OMB), __fmul_rn(nm1, bmag));
      GeoM g;
      geo_lite(A, TF(fm::X0 + 3 * j), TF(fm::Y0 + 3 * j), TF(fm::Z0 + 3 * j), g);
      FieldM f;
      field_mixed(g, bx, by, bz, bmag, om, __fadd_rn(1.0f, nm1), f);
      geo_refine(g);
      const ff ua = arrival_mixed<KIND>(M, A, g, TF(fm::TAU0H + 2 * j), TF(fm::TAU0L + 2 * j), Eh, El);
      float fr;
      const int k = bin_raw(ua, N, fr);
      if (k < 0 || k >= N) return;
      const float c = div_ap(j ? -amp : amp, f.D * g.R0) * (f.invR * f.invR);
      out.dep(k, c * f.V[0], c * f.V[1], c * f.V[2]);
    }
  }

  // a pair set aside by the main pass (Endpoint near the Cherenkov angle)
  template <class Sink>
  static __device__ __forceinline__ void pair_deferred(const TrackM& t, const AntRec& A, const MedParams& M,
                                                       Sink& out) {
    if constexpr (FORM == C8R_ENDPOINT) {
      EndpointEvalM e;
      if (!endpoint_fields<KIND>(t, A, M, e)) return;
      if (!endpoint_midpoint<KIND>(t, A, M, e)) return;
      endpoint_deposit(t, e, M, out);
    }
  }

  // one pair, complete, with float-float arrivals throughout (the arrival
  // listing records them)
  template <class Sink>
  static __device__ __forceinline__ void pair(const TrackM& t, const AntRec& A, const MedParams& M, Sink& out) {
    if constexpr (FORM == C8R_ENDPOINT) {
      EndpointEvalM e;
      endpoint_eval_mixed<KIND>(t, A, M, e);
      if (e.valid) endpoint_deposit(t, e, M, out);
    } else {
      zhs(t, A, M, out);
    }
  }

  // one pair from a staged tile, for the arrival listing: as the forward kernel
  // has it, the track with its neighbour where that takes two at a time
  template <class Sink>
  static __device__ __forceinline__ void list(const void* Tv, int l, const AntRec& A, const MedParams& M, Sink& out) {
    if constexpr (kTwoTracks) {
      TrackZ<KIND> t;
      load_fwd(Tv, l / 2, M, t);
      if (static_cast<const float*>(Tv)[fm::AMPE * kTileT + l] == 0.0f) return;
      AntZ z;
      stage_ant(&z, A, M);
      Sink none = out;
      none.off = true;
      zhs_two(t, z, M, l & 1 ? none : out, l & 1 ? out : none);
    } else if constexpr (kFastBins) {
      // the main pass decides the near-Cherenkov pairs; which bin a pair's
      // endpoints have does not depend on the way it takes there
      TrackE te;
      load_main(Tv, l, M, te);
      if (!live(te)) return;
      AntE ae;
      stage_ant(&ae, A, M);
      GeoT<float2> g;
      FieldT<float2> f;
      int ka, kb;
      const bool near = endpoints_main(te, ae, M, g, f, ka, kb);
      TrackM t;
      load(Tv, l, M, t);
      EndpointEvalM e;
      if (!endpoint_fields<KIND>(t, A, M, e)) return;
      if (!near)
        endpoint_arrivals<KIND>(t, A, M, e);
      else if (!endpoint_midpoint<KIND>(t, A, M, e))
        return;
      out.rec(e.branch, e.ua, e.ub);
    } else {
      fwd(Tv, l, A, M, out);
    }
  }
  // one pair from a staged tile (the allocation-free pass uses this)
  template <class Sink>
  static __device__ __forceinline__ void fwd(const void* Tv, int l, const AntRec& A, const MedParams& M, Sink& out) {
    TrackM t;
    load(Tv, l, M, t);
    if (!live(t)) return;
    pair(t, A, M, out);
  }

  // -------------------------------------------------------------------------
  // adjoint of `endpoint` with bins and branch held fixed
  // -------------------------------------------------------------------------
  static __device__ __forceinline__ void deposit_grad(const GeoM& g, const FieldM& f, float D, float n,
                                                      const float gv[3], float kappa, float dd[3], float db[3],
                                                      float& dns) {
    const float invR = f.invR;
    const float rh[3] = {g.s[0] * invR, g.s[1] * invR, g.s[2] * invR};
    const float inv2 = invR * invR;
    const float V[3] = {f.V[0] * inv2, f.V[1] * inv2, f.V[2] * inv2};
    const float c = f.bd * invR;
    deposit_adjoint<float>(rh, V, c, D, g.R0, n, gv, kappa, dd, db, dns);
  }
  static __device__ __forceinline__ void deposit_grad(const GeoM& g, const FieldM& f, float n, const float gv[3],
                                                      float kappa, float dd[3], float db[3], float& dns) {
    deposit_grad(g, f, f.D, n, gv, kappa, dd, db, dns);
  }

  // dL/dtrace seen by a unit deposit in cell J at s (reading LD), and its rate of
  // change with the arrival (bins outside the window read 0)
  static __device__ __forceinline__ void gather_lin(const float4* G, int N, int J, float s, float gv[3],
                                                    float slope[3]) {
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 g0 = (J >= 1 && J - 1 < N) ? G[J - 1] : z4;
    const float4 g1 = (J >= 0 && J < N) ? G[J] : z4;
    const float r = 1.0f - s;
    gv[0] = r * g0.x + s * g1.x;
    gv[1] = r * g0.y + s * g1.y;
    gv[2] = r * g0.z + s * g1.z;
    slope[0] = g1.x - g0.x;
    slope[1] = g1.y - g0.y;
    slope[2] = g1.z - g0.z;
  }

  // chain rule through an arrival position u = (t_e - t_a)/dt + (R + F)/(c dt)
  // of the emission point at d = x_a - x_e (refractivity factor E): adds
  // dL/dx_e x w_e (w_e = 1, or 1/2 to each endpoint for the midpoint), dL/dx_a,
  // dL/dN0; the caller adds dL/dt_e
  static __device__ __forceinline__ void arrival_grad(const GeoM& g, float invR, float E, const MedParams& M,
                                                      float dLdu, float* tg_pos0, float* tg_pos1, float w_e,
                                                      float ga[3], float& dn) {
    const RefrGrad<float> rg = refraction_grad<float>(KIND, g.R0, g.s[2] * M.invH_h, E, M.N0f, M.invH_h, M.nm1f);
    const float dLdopt = dLdu * M.kc_h;
    const float dLdR = dLdopt * (1.0f + rg.dF_dR);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float v = dLdR * g.s[k] * invR;
      ga[k] += v;
      tg_pos0[k] -= w_e * v;
      if (tg_pos1) tg_pos1[k] -= w_e * v;
    }
    tg_pos0[2] += w_e * dLdopt * rg.dF_dzm;
    if (tg_pos1) tg_pos1[2] += w_e * dLdopt * rg.dF_dzm;
    ga[2] += dLdopt * rg.dF_dza;
    dn += dLdopt * rg.dF_dN0;
  }

  // a track's gradients while its main pass runs: for the one-bin Endpoint
  // kernels the positions of both endpoints as pairs, and beta with a sum per
  // endpoint (the deposits do not depend on the times); otherwise the eleven
  // gradients themselves
  struct GradE {
    float2 pos[3], beta[3];
  };
  struct GradPlain {
    float g[11];
  };
  using MainGrad = std::conditional_t<kFastBins, GradE, GradPlain>;
  static __device__ __forceinline__ void zero(MainGrad& m) {
    if constexpr (kFastBins) {
#pragma unroll
      for (int c = 0; c < 3; ++c) m.pos[c] = m.beta[c] = bc<float2>(0.0f);
    } else {
#pragma unroll
      for (int k = 0; k < 11; ++k) m.g[k] = 0.0f;
    }
  }
  static __device__ __forceinline__ void collect(const MainGrad& m, float tg[11]) {
    if constexpr (kFastBins) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        tg[c] = m.pos[c].x;
        tg[3 + c] = m.pos[c].y;
        tg[8 + c] = m.beta[c].x + m.beta[c].y;
      }
      tg[6] = tg[7] = 0.0f;
    } else {
#pragma unroll
      for (int k = 0; k < 11; ++k) tg[k] = m.g[k];
    }
  }

  // chain rule of a pair's two one-bin Endpoint deposits +/- amp V/(D R) (bins
  // held fixed, dL/dtrace ga and gb at them, zero for an endpoint without one):
  // deposit_adjoint on both endpoints at once
  static __device__ __forceinline__ void adj_ends(const GeoT<float2>& g, const FieldT<float2>& f, const TrackE& t,
                                                  const float4 ga4, const float4 gb4, const MedParams& M, GradE& m,
                                                  float ga[3], float& dn) {
    const float2 G[3] = {make_float2(ga4.x, gb4.x), make_float2(ga4.y, gb4.y), make_float2(ga4.z, gb4.z)};
    const float2 iR = f.invR, i2 = mul_rn(iR, iR), one = bc<float2>(1.0f);
    // 1/D and 1/R with a Newton step, as good as rounded once: the approximate
    // ones are off to one side by up to a bit, which the sums over all pairs
    // would keep
    float2 iD = rcp_ap(f.D), nR = iR;
    iD = fma_rn(fma_rn(neg(f.D), iD, one), iD, iD);
    nR = fma_rn(fma_rn(neg(g.R0), nR, one), nR, nR);
    float2 rh[3], V[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      rh[k] = mul_rn(g.s[k], iR);
      V[k] = mul_rn(f.V[k], i2);
    }
    const float2 c = mul_rn(f.bd, iR);
    const float2 gV = fma_rn(G[2], V[2], fma_rn(G[0], V[0], mul_rn(G[1], V[1])));
    const float2 rg = fma_rn(rh[2], G[2], fma_rn(rh[0], G[0], mul_rn(rh[1], G[1])));
    const float2 f2 = mul_rn(mul_rn(make_float2(t.amp, -t.amp), iD), nR), f1 = mul_rn(f2, nR);
    const float2 p = mul_rn(f2, fma_rn(mul_rn(gV, t.n), iD, rg)), q = neg(f2);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      // dl/dd = f1 x, x = c (g - rhat rg) - rg V - gV (n V/D + rhat); the order
      // of these roundings is deposit_adjoint's as compiled, so that the two
      // agree bit for bit (the set-aside pairs take that one)
      const float2 x = fma_rn(neg(gV), fma_rn(mul_rn(t.n, V[k]), iD, rh[k]),
                              fma_rn(c, fma_rn(neg(rh[k]), rg, G[k]), mul_rn(neg(rg), V[k])));
      m.pos[k] = fma_rn(neg(f1), x, m.pos[k]);
      ga[k] = __fmaf_rn(f1.y, x.y, __fmaf_rn(f1.x, x.x, ga[k]));
      // dl/dbeta = f2 [(rg + gV n/D) rhat - g]
      m.beta[k] = add_rn(m.beta[k], fma_rn(p, rh[k], mul_rn(q, G[k])));
    }
    const float2 dns = mul_rn(mul_rn(mul_rn(f2, gV), c), iD);  // dl/dn
    if constexpr (KIND == C8R_EXPONENTIAL)
      m.pos[2] = fma_rn(mul_rn(dns, bc<float2>(-M.N0f * M.invH_h)), t.Eh, m.pos[2]);
    dn = __fmaf_rn(dns.y, t.Eh.y, __fmaf_rn(dns.x, t.Eh.x, dn));
  }

  // of a pair that the adjoint's main pass set aside whole: the one endpoint with a
  // geometry where the other has none and that one is not near the Cherenkov angle
  // (kDeferEnd0 or kDeferEnd1), or 0
  static __device__ __forceinline__ int lone_end(const void* Tv, int l, const AntRec& A, const MedParams& M) {
    if constexpr (kFastBins) {
      const float* T = static_cast<const float*>(Tv);
      GeoM g0, g1;
      geo_lite(A, TF(fm::X0), TF(fm::Y0), TF(fm::Z0), g0);
      geo_lite(A, TF(fm::X1), TF(fm::Y1), TF(fm::Z1), g1);
      if (g0.R0 + g1.R0 > 0.0f) return 0;
      const int end = g0.R0 > 0.0f ? kDeferEnd0 : kDeferEnd1;
      const GeoM& g = end == kDeferEnd0 ? g0 : g1;
      const float bmag = TF(fm::BMAG);
      float nm1 = M.nm1f;
      if (KIND != C8R_UNIFORM) nm1 = __fmul_rn(M.N0f, end == kDeferEnd0 ? TF(fm::E0H) : TF(fm::E1H));
      FieldM f;
      field_mixed<float>(g, TF(fm::BX), TF(fm::BY), TF(fm::BZ), bmag, __fsub_rn(TF(fm::OMB), __fmul_rn(nm1, bmag)),
                         __fadd_rn(1.0f, nm1), f);
      return fabsf(f.D) >= M.eps_C ? end : 0;
    } else {
      return 0;
    }
  }

  // adjoint main pass: every pair except (Endpoint) the near-Cherenkov ones, for
  // which it adds nothing and returns kDeferPair, and (kFastBins) the endpoints
  // whose bin the FP32 arrival leaves open (kDeferEnd0/kDeferEnd1 bits), after
  // the other endpoint's part
  static __device__ __forceinline__ int adj_main(const MainTrack& t, const Ant* p, const MedParams& M,
                                                 const float4* G, const PrefixFF* Gp, MainGrad& m, float ga[3],
                                                 float& dn) {
    if constexpr (FORM == C8R_ZHS) {
      adj_zhs(t, load_ant(p), M, G, Gp, m.g, ga, dn);
      return kDeferNone;
    } else if constexpr (kFastBins) {
      GeoT<float2> g;
      FieldT<float2> f;
      int ka, kb;
      if (endpoints_main<true>(t, *p, M, g, f, ka, kb)) return kDeferPair;
      const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      const float4 g0 = ka >= 0 ? G[ka] : zero, g1 = kb >= 0 ? G[kb] : zero;
      if (ka >= 0 || kb >= 0) adj_ends(g, f, t, g0, g1, M, m, ga, dn);
      return (ka == kFastUndecided ? kDeferEnd0 : 0) | (kb == kFastUndecided ? kDeferEnd1 : 0);
    } else {
      const AntRec A = load_ant(p);
      EndpointEvalM e;
      if (!endpoint_fields<KIND>(t, A, M, e)) return kDeferNone;
      if (endpoint_near_cherenkov(e, M)) return kDeferPair;
      endpoint_arrivals<KIND>(t, A, M, e);
      adj_deposits(t, e, M, G, m.g, ga, dn);
      return kDeferNone;
    }
  }

  // the adjoint of one endpoint set aside by the main pass (kFastBins; `end` is
  // kDeferEnd0 or kDeferEnd1), read from the staged tile (lane l) as
  // end_deferred reads it: the float-float arrival gives the bin, the chain
  // rule is adj_end's, and the track gradients (positions of that endpoint,
  // beta) go to the output of track i with one reduction each; ga and dn
  // collect the antenna and N0 parts
  static __device__ __forceinline__ void adj_end_deferred(const void* Tv, int l, const AntRec& A, const MedParams& M,
                                                          const float4* G, const c8r_track_grads& out, int64_t i,
                                                          float ga[3], float& dn, int end) {
    if constexpr (kFastBins) {
      const float* T = static_cast<const float*>(Tv);
      const int N = M.n_bins;
      const int j = end == kDeferEnd1 ? 1 : 0;
      const float amp = TF(fm::AMPE);
      const float bx = TF(fm::BX), by = TF(fm::BY), bz = TF(fm::BZ), bmag = TF(fm::BMAG);
      float Eh = 1.0f, El = 0.0f, nm1 = M.nm1f;
      if (KIND != C8R_UNIFORM) {
        Eh = TF(fm::E0H + 2 * j);
        El = TF(fm::E0L + 2 * j);
        nm1 = __fmul_rn(M.N0f, Eh);
      }
      const float om = __fsub_rn(TF(fm::OMB), __fmul_rn(nm1, bmag));
      GeoM g;
      geo_lite(A, TF(fm::X0 + 3 * j), TF(fm::Y0 + 3 * j), TF(fm::Z0 + 3 * j), g);
      FieldM f;
      field_mixed(g, bx, by, bz, bmag, om, __fadd_rn(1.0f, nm1), f);
      GeoM gr = g;
      geo_refine(gr);
      const ff ua = arrival_mixed<KIND>(M, A, gr, TF(fm::TAU0H + 2 * j), TF(fm::TAU0L + 2 * j), Eh, El);
      float fr;
      const int k = bin_raw(ua, N, fr);
      if (k < 0 || k >= N) return;
      const float dNdz_fac = (KIND == C8R_EXPONENTIAL) ? -M.N0f * M.invH_h : 0.0f;
      const float4 g4 = G[k];
      const float gv[3] = {g4.x, g4.y, g4.z};
      float dd[3], db[3], dns;
      deposit_grad(g, f, 1.0f + nm1, gv, j ? -amp : amp, dd, db, dns);
      float* px = static_cast<float*>(j ? out.x1 : out.x0);
      float* py = static_cast<float*>(j ? out.y1 : out.y0);
      float* pz = static_cast<float*>(j ? out.z1 : out.z0);
      const float gz = -dd[2] + dns * dNdz_fac * Eh;
      if (dd[0] != 0.0f) atomicAdd(px + i, -dd[0]);
      if (dd[1] != 0.0f) atomicAdd(py + i, -dd[1]);
      if (gz != 0.0f) atomicAdd(pz + i, gz);
      if (db[0] != 0.0f) atomicAdd(static_cast<float*>(out.bx) + i, db[0]);
      if (db[1] != 0.0f) atomicAdd(static_cast<float*>(out.by) + i, db[1]);
      if (db[2] != 0.0f) atomicAdd(static_cast<float*>(out.bz) + i, db[2]);
#pragma unroll
      for (int c = 0; c < 3; ++c) ga[c] += dd[c];
      dn += dns * Eh;
    }
  }
  static __device__ __forceinline__ void adj_deferred(const TrackM& t, const AntRec& A, const MedParams& M,
                                                      const float4* G, const PrefixFF*, float tg[11], float ga[3],
                                                      float& dn) {
    if constexpr (FORM == C8R_ENDPOINT) {
      EndpointEvalM e;
      if (!endpoint_fields<KIND>(t, A, M, e)) return;
      if (!endpoint_midpoint<KIND>(t, A, M, e)) return;
      adj_deposits(t, e, M, G, tg, ga, dn);
    }
  }

  // G summed over bins kb..ke from the float-float running sums: the FP32
  // difference of the high parts is exact or rounded relative to the result,
  // and the low parts restore what the high parts dropped, so the sum comes out
  // rounded to FP32 plus the running sums' own error (~2k u^2 of the largest
  // partial sum after k bins), without the FP64 pipe
  static __device__ __forceinline__ void run_sum(const PrefixFF* Gp, int kb, int ke, float& ix, float& iy,
                                                 float& iz) {
    const PrefixFF p1 = Gp[ke + 1], p0 = Gp[kb];
    ix = __fadd_rn(__fsub_rn(p1.hx, p0.hx), __fsub_rn(p1.lx, p0.lx));
    iy = __fadd_rn(__fsub_rn(p1.hy, p0.hy), __fsub_rn(p1.ly, p0.ly));
    iz = __fadd_rn(__fsub_rn(p1.hz, p0.hz), __fsub_rn(p1.lz, p0.lz));
  }

  // ZHS adjoint (bins of the interval ends held fixed): the forward arithmetic
  // of `zhs`, then the chain rule through the one-bin deposit A = amp beta_perp/R
  // (amp = q K_A (t1 - t0)/dt) and the weights of [u_m - h, u_m + h] over its
  // bins: with S = sum_k w_k G_k, g_lo/g_hi = A.G at the first/last bin and W =
  // 2h, dL/du_m = (g_hi - g_lo)/W and dL/dh = (g_hi + g_lo - 2 A.S)/W (both 0
  // for a one-bin interval).  The sum of G over the whole bins in between comes
  // from the running sums Gp.  Times in ns, positions in m.
  static __device__ __forceinline__ void adj_zhs(const TrackM& t, const AntRec& A, const MedParams& M,
                                                 const float4* G, const PrefixFF* Gp, float tg[11], float ga[3],
                                                 float& dn) {
    const int N = M.n_bins;
    GeoM gm;
    if constexpr (kFlat)
      geo_lite(A.xh, A.yh, A.xl, A.yl, t.mx, t.my, t.mxl, t.myl, t.zm, gm);
    else
      geo_lite(A, t.mx, t.my, t.mz, t.mxl, t.myl, t.mzl, gm);
    if (gm.R0 == 0.0f) return;
    FieldM f;
    field_mixed(gm, t.bx, t.by, t.bz, t.bmag, t.om_m, __fadd_rn(1.0f, t.nm1_m), f);
    ff um, aD;
    if constexpr (kFlat) {
      geo_refine(gm, t.zm);
      um = arrival_mixed_q<KIND>(M, A.tauh, A.taul, gm, t.tmh, t.tml, t.qmh, t.qml);
      aD = doppler_ff(gm, t.bx, t.by, t.zm, t.nm1_m);
    } else {
      geo_refine(gm);
      um = arrival_mixed<KIND>(M, A, gm, t.tmh, t.tml, t.Emh, t.Eml);
      aD = doppler_ff(gm, t.bx, t.by, t.bz, t.nm1_m);
    }
    const float sgn = aD.h < 0.0f ? -1.0f : 1.0f;
    if (aD.h < 0.0f) {
      aD.h = -aD.h;
      aD.l = -aD.l;
    }
    float hh, hl;
    two_prod(aD.h, t.dtauh, hh, hl);
    hl = __fmaf_rn(aD.h, t.dtaul, __fmaf_rn(aD.l, t.dtauh, hl));
    hh *= 0.5f;
    hl *= 0.5f;
    ff ulo, uhi;
    two_sum(um.h, -hh, ulo.h, ulo.l);
    ulo.l = __fadd_rn(ulo.l, __fsub_rn(um.l, hl));
    two_sum(um.h, hh, uhi.h, uhi.l);
    uhi.l = __fadd_rn(uhi.l, __fadd_rn(um.l, hl));
    float flo, fhi;
    const int klo = bin_raw(ulo, N, flo);
    const int khi = bin_raw(uhi, N, fhi);
    const float invR = f.invR;
    const float rh[3] = {gm.s[0] * invR, gm.s[1] * invR, gm.s[2] * invR};
    const float b[3] = {t.bx, t.by, t.bz};
    const float c = f.bd * invR;
    const float Av[3] = {t.amp * (b[0] - c * rh[0]) * invR, t.amp * (b[1] - c * rh[1]) * invR,
                         t.amp * (b[2] - c * rh[2]) * invR};
    float S[3];
    float dLdu = 0.0f, dLdh = 0.0f;
    if constexpr (LIN) {
      float slo, shi;
      const int Jlo = lin_cell(ulo, N, slo);
      const int Jhi = lin_cell(uhi, N, shi);
      float sl[3];
      if (Jlo == Jhi) {
        if (Jlo < 0 || Jlo > N) return;
        gather_lin(G, N, Jlo, 0.5f * (slo + shi), S, sl);
        dLdu = Av[0] * sl[0] + Av[1] * sl[1] + Av[2] * sl[2];
      } else {
        const float invW = div_ap(1.0f, 2.0f * hh);
        const LinEnds z = lin_ends(Jlo, slo, Jhi, shi, invW);
        float ix = 0.0f, iy = 0.0f, iz = 0.0f;  // G summed over the bins strictly between the ends
        const int kb = Jlo + 1 < 0 ? 0 : Jlo + 1;
        const int ke = Jhi - 2 > N - 1 ? N - 1 : Jhi - 2;
        if (kb <= ke) run_sum(Gp, kb, ke, ix, iy, iz);
        S[0] = invW * ix;
        S[1] = invW * iy;
        S[2] = invW * iz;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (i < z.n && z.k[i] >= 0 && z.k[i] < N) {
            const float4 g = G[z.k[i]];
            S[0] += z.w[i] * g.x;
            S[1] += z.w[i] * g.y;
            S[2] += z.w[i] * g.z;
          }
        }
        float glo[3], ghi[3];
        gather_lin(G, N, Jlo, slo, glo, sl);
        gather_lin(G, N, Jhi, shi, ghi, sl);
        const float p_lo = Av[0] * glo[0] + Av[1] * glo[1] + Av[2] * glo[2];
        const float p_hi = Av[0] * ghi[0] + Av[1] * ghi[1] + Av[2] * ghi[2];
        const float AS = Av[0] * S[0] + Av[1] * S[1] + Av[2] * S[2];
        dLdu = (p_hi - p_lo) * invW;
        dLdh = (p_hi + p_lo - 2.0f * AS) * invW;
      }
    } else {
      // one path for intervals inside one bin (weight 1 on its bin, 1 G = G
      // exactly, and no dependence on the interval's ends: 1/W taken as 0) and
      // for intervals over several bins
      const bool one = klo == khi;
      const bool inlo = klo >= 0 && klo < N, inhi = !one && khi >= 0 && khi < N;
      if (one && !inlo) return;
      const float invW = one ? 0.0f : div_ap(1.0f, 2.0f * hh);
      const float4 glo = inlo ? G[klo] : make_float4(0.f, 0.f, 0.f, 0.f);
      const float4 ghi = inhi ? G[khi] : make_float4(0.f, 0.f, 0.f, 0.f);
      const float wlo = inlo ? (one ? 1.0f : gap_to_next_edge(ulo, klo) * invW) : 0.0f, whi = fhi * invW;
      float ix = 0.0f, iy = 0.0f, iz = 0.0f;  // G summed over the whole bins between
      const int kb = klo + 1 < 0 ? 0 : klo + 1;
      const int ke = khi - 1 > N - 1 ? N - 1 : khi - 1;
      if (kb <= ke) run_sum(Gp, kb, ke, ix, iy, iz);
      S[0] = wlo * glo.x + invW * ix + whi * ghi.x;
      S[1] = wlo * glo.y + invW * iy + whi * ghi.y;
      S[2] = wlo * glo.z + invW * iz + whi * ghi.z;
      const float g_lo = Av[0] * glo.x + Av[1] * glo.y + Av[2] * glo.z;
      const float g_hi = Av[0] * ghi.x + Av[1] * ghi.y + Av[2] * ghi.z;
      const float AS = Av[0] * S[0] + Av[1] * S[1] + Av[2] * S[2];
      dLdu = (g_hi - g_lo) * invW;
      dLdh = (g_hi + g_lo - 2.0f * AS) * invW;
    }
    const float AS = Av[0] * S[0] + Av[1] * S[1] + Av[2] * S[2];
    // through A
    const float ka = t.amp * invR;
    const float sb[3] = {ka * S[0], ka * S[1], ka * S[2]};
    const float sbr = sb[0] * rh[0] + sb[1] * rh[1] + sb[2] * rh[2];
    float dLdb[3], dLdr[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      dLdb[k] = sb[k] - sbr * rh[k];
      dLdr[k] = -c * sb[k] - sbr * b[k];
    }
    const float dtau = t.dtauh;  // (t1 - t0)/dt
    float dLd_dtau = div_ap(AS, dtau);
    float dLdR = -AS * invR;
    // through h = |D| dtau / 2
    const float absD = aD.h;
    const float dLdD = dLdh * sgn * 0.5f * dtau;
    dLd_dtau += dLdh * 0.5f * absD;
    // D = 1 - n c
    const float n = 1.0f + t.nm1_m;
    const float dLdn = -c * dLdD;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      dLdb[k] -= n * rh[k] * dLdD;
      dLdr[k] -= n * b[k] * dLdD;
    }
    // u_m = tau_m - tau_a + (R + F) / (c dt)
    const float R = gm.R0;
    const RefrGrad<float> rg = refraction_grad<float>(KIND, R, gm.s[2] * M.invH_h, t.Emh, M.N0f, M.invH_h, M.nm1f);
    const float dLdopt = dLdu * M.kc_h;
    dLdR += dLdopt * (1.0f + rg.dF_dR);
    const float dLdzm = dLdopt * rg.dF_dzm + dLdn * rg.dn_dzm;
    const float dLdza = dLdopt * rg.dF_dza;
    dn += dLdopt * rg.dF_dN0 + dLdn * rg.dn_dN0;
    // rhat = d/R, d = x_a - x_m
    const float rdr = dLdr[0] * rh[0] + dLdr[1] * rh[1] + dLdr[2] * rh[2];
    float dLdd[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) dLdd[k] = (dLdr[k] - rdr * rh[k]) * invR + dLdR * rh[k];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float dm = -dLdd[k] + (k == 2 ? dLdzm : 0.0f);
      tg[k] += 0.5f * dm;
      tg[3 + k] += 0.5f * dm;
      tg[8 + k] += dLdb[k];
      ga[k] += dLdd[k] + (k == 2 ? dLdza : 0.0f);
    }
    const float idt = M.idt_h;  // 1/dt (per ns)
    tg[6] += (0.5f * dLdu - dLd_dtau) * idt;
    tg[7] += (0.5f * dLdu + dLd_dtau) * idt;
  }

  // gradients of the linear (two-bin) Endpoint deposits of an evaluated pair:
  // the amplitude as for one bin, against the spread of dL/dtrace that the
  // deposit sees, plus its slide with the arrival, dL/du = l(G_J - G_{J-1}),
  // taken through the arrival time (and near Cherenkov through
  // u_a, u_b = u_m -/+ D (t1 - t0)/(2 dt)).  Times in ns, positions in m.
  static __device__ __forceinline__ void adj_deposits_lin(const TrackM& t, const EndpointEvalM& e,
                                                          const MedParams& M, const float4* G, float tg[11],
                                                          float ga[3], float& dn) {
    const int N = M.n_bins;
    float sa, sb;
    const int Ja = lin_cell(e.ua, N, sa);
    const int Jb = lin_cell(e.ub, N, sb);
    const float dNdz_fac = (KIND == C8R_EXPONENTIAL) ? -M.N0f * M.invH_h : 0.0f;
    const float idt = M.idt_h;
    const float amp = t.amp;
    float dd[3], db[3], dns, gv[3], sl[3];
    if (e.branch == 0) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int J = j == 0 ? Ja : Jb;
        if (J < 0 || J > N) continue;
        const GeoM& g = j == 0 ? e.g0 : e.g1;
        const FieldM& f = j == 0 ? e.f0 : e.f1;
        const float E = j == 0 ? t.E0h : t.E1h;
        const float kap = j == 0 ? amp : -amp;
        gather_lin(G, N, J, j == 0 ? sa : sb, gv, sl);
        deposit_grad(g, f, 1.0f + (j == 0 ? t.nm1_0 : t.nm1_1), gv, kap, dd, db, dns);
        for (int c = 0; c < 3; ++c) {
          tg[3 * j + c] -= dd[c];
          ga[c] += dd[c];
          tg[8 + c] += db[c];
        }
        tg[3 * j + 2] += dns * dNdz_fac * E;
        dn += dns * E;
        const float cj = div_ap(kap, f.D * g.R0) * (f.invR * f.invR);
        const float dLdu = cj * (f.V[0] * sl[0] + f.V[1] * sl[1] + f.V[2] * sl[2]);
        arrival_grad(g, f.invR, E, M, dLdu, tg + 3 * j, nullptr, 1.0f, ga, dn);
        tg[6 + j] += dLdu * idt;
      }
      return;
    }
    const float invR = e.fm.invR;
    if (Ja == Jb) {
      // l = amp (t1 - t0)/dt (g.V)/R with g = G_{J-1} - G_J: the deposit adjoint
      // with D = 1 and n = 0, and dl/d(t1 - t0) = l/(t1 - t0)
      if (Ja < 0 || Ja > N) return;
      const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
      const float4 g0 = (Ja >= 1 && Ja - 1 < N) ? G[Ja - 1] : z4;
      const float4 g1 = (Ja < N) ? G[Ja] : z4;
      gv[0] = g0.x - g1.x;
      gv[1] = g0.y - g1.y;
      gv[2] = g0.z - g1.z;
      const float kap = amp * t.dtauh;
      deposit_grad(e.gm, e.fm, 1.0f, 0.0f, gv, kap, dd, db, dns);
      for (int c = 0; c < 3; ++c) {
        tg[c] -= 0.5f * dd[c];
        tg[3 + c] -= 0.5f * dd[c];
        ga[c] += dd[c];
        tg[8 + c] += db[c];
      }
      const float l_dtau =
          amp * (gv[0] * e.fm.V[0] + gv[1] * e.fm.V[1] + gv[2] * e.fm.V[2]) * (invR * invR * invR);
      tg[6] -= l_dtau * idt;
      tg[7] += l_dtau * idt;
      return;
    }
    float ga_[3], gb_[3], sla[3], slb[3];
    gather_lin(G, N, Ja, sa, ga_, sla);
    gather_lin(G, N, Jb, sb, gb_, slb);
    gv[0] = ga_[0] - gb_[0];
    gv[1] = ga_[1] - gb_[1];
    gv[2] = ga_[2] - gb_[2];
    deposit_grad(e.gm, e.fm, 1.0f + t.nm1_m, gv, amp, dd, db, dns);
    for (int c = 0; c < 3; ++c) {
      tg[c] -= 0.5f * dd[c];
      tg[3 + c] -= 0.5f * dd[c];
      ga[c] += dd[c];
      tg[8 + c] += db[c];
    }
    tg[2] += 0.5f * dns * dNdz_fac * t.Emh;
    tg[5] += 0.5f * dns * dNdz_fac * t.Emh;
    dn += dns * t.Emh;
    // the slide of the two spread deposits +/- c V
    const float Dm = e.fm.D;
    const float cm = div_ap(amp, Dm * e.gm.R0) * (invR * invR);
    const float dLdua = cm * (e.fm.V[0] * sla[0] + e.fm.V[1] * sla[1] + e.fm.V[2] * sla[2]);
    const float dLdub = -cm * (e.fm.V[0] * slb[0] + e.fm.V[1] * slb[1] + e.fm.V[2] * slb[2]);
    const float dLdum = dLdua + dLdub;
    const float dLdD = (dLdub - dLdua) * 0.5f * t.dtauh;
    const float dLd_dtau = (dLdub - dLdua) * 0.5f * Dm;
    // D = 1 - n (beta.rhat), rhat = d/R, d = x_a - x_m
    const float n = 1.0f + t.nm1_m;
    const float rh[3] = {e.gm.s[0] * invR, e.gm.s[1] * invR, e.gm.s[2] * invR};
    const float b[3] = {t.bx, t.by, t.bz};
    const float cr = e.fm.bd * invR;
    float dLdr[3];
    for (int k = 0; k < 3; ++k) {
      tg[8 + k] -= n * rh[k] * dLdD;
      dLdr[k] = -n * b[k] * dLdD;
    }
    const float rdr = dLdr[0] * rh[0] + dLdr[1] * rh[1] + dLdr[2] * rh[2];
    for (int k = 0; k < 3; ++k) {
      const float v = (dLdr[k] - rdr * rh[k]) * invR;
      tg[k] -= 0.5f * v;
      tg[3 + k] -= 0.5f * v;
      ga[k] += v;
    }
    const float dLdn = -cr * dLdD;
    tg[2] += 0.5f * dLdn * dNdz_fac * t.Emh;
    tg[5] += 0.5f * dLdn * dNdz_fac * t.Emh;
    dn += dLdn * t.Emh;
    arrival_grad(e.gm, invR, t.Emh, M, dLdum, tg, tg + 3, 0.5f, ga, dn);
    tg[6] += (0.5f * dLdum - dLd_dtau) * idt;
    tg[7] += (0.5f * dLdum + dLd_dtau) * idt;
  }

  // gradients of the deposits of an evaluated pair
  static __device__ __forceinline__ void adj_deposits(const TrackM& t, const EndpointEvalM& e, const MedParams& M,
                                                      const float4* G, float tg[11], float ga[3], float& dn) {
    if constexpr (LIN) {
      adj_deposits_lin(t, e, M, G, tg, ga, dn);
      return;
    }
    const int N = M.n_bins;
    float fa, fb;
    const int ka = bin_raw(e.ua, N, fa);
    const int kb = bin_raw(e.ub, N, fb);
    const bool ina = ka >= 0 && ka < N, inb = kb >= 0 && kb < N;
    const float dNdz_fac = (KIND == C8R_EXPONENTIAL) ? -M.N0f * M.invH_h : 0.0f;
    const float amp = t.amp;
    float dd[3], db[3], dns;
    if (e.branch == 0) {
      for (int j = 0; j < 2; ++j) {
        const bool in = j == 0 ? ina : inb;
        if (!in) continue;
        const int k = j == 0 ? ka : kb;
        const float4 g4 = G[k];
        const float gv[3] = {g4.x, g4.y, g4.z};
        deposit_grad(j == 0 ? e.g0 : e.g1, j == 0 ? e.f0 : e.f1, 1.0f + (j == 0 ? t.nm1_0 : t.nm1_1), gv,
                     j == 0 ? amp : -amp, dd, db, dns);
        const float E = j == 0 ? t.E0h : t.E1h;
        for (int c = 0; c < 3; ++c) {
          tg[3 * j + c] -= dd[c];
          ga[c] += dd[c];
          tg[8 + c] += db[c];
        }
        tg[3 * j + 2] += dns * dNdz_fac * E;
        dn += dns * E;
      }
      return;
    }
    if (ka == kb) return;
    float gv[3];
    const float4 ga4 = ina ? G[ka] : make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 gb4 = inb ? G[kb] : make_float4(0.f, 0.f, 0.f, 0.f);
    gv[0] = ga4.x - gb4.x;
    gv[1] = ga4.y - gb4.y;
    gv[2] = ga4.z - gb4.z;
    deposit_grad(e.gm, e.fm, 1.0f + t.nm1_m, gv, amp, dd, db, dns);
    for (int c = 0; c < 3; ++c) {
      tg[c] -= 0.5f * dd[c];
      tg[3 + c] -= 0.5f * dd[c];
      ga[c] += dd[c];
      tg[8 + c] += db[c];
    }
    tg[2] += 0.5f * dns * dNdz_fac * t.Emh;
    tg[5] += 0.5f * dns * dNdz_fac * t.Emh;
    dn += dns * t.Emh;
  }
};

#undef TF

// The one-bin Endpoint kernels of the plain media come in the arrival forms (M.axis,
// M.split) and, in the exponential medium, for a flat antenna array (M.flat,
// OpsMixed::kFlat)
template <class F>
cudaError_t with_endpoint_ops(const MedParams& M, F go) {
  if (M.kind != C8R_EXPONENTIAL)
    return M.axis    ? go(OpsMixed<C8R_ENDPOINT, C8R_UNIFORM, false, kFormAxis>{})
           : M.split ? go(OpsMixed<C8R_ENDPOINT, C8R_UNIFORM, false, kFormSplit>{})
                     : go(OpsMixed<C8R_ENDPOINT, C8R_UNIFORM>{});
  if (M.flat)
    return M.axis    ? go(OpsMixed<C8R_ENDPOINT, C8R_EXPONENTIAL, false, kFormAxis, true>{})
           : M.split ? go(OpsMixed<C8R_ENDPOINT, C8R_EXPONENTIAL, false, kFormSplit, true>{})
                     : go(OpsMixed<C8R_ENDPOINT, C8R_EXPONENTIAL, false, kFormDirect, true>{});
  return M.axis    ? go(OpsMixed<C8R_ENDPOINT, C8R_EXPONENTIAL, false, kFormAxis>{})
         : M.split ? go(OpsMixed<C8R_ENDPOINT, C8R_EXPONENTIAL, false, kFormSplit>{})
                   : go(OpsMixed<C8R_ENDPOINT, C8R_EXPONENTIAL>{});
}

// forward and adjoint launches for one deposit shape (one-bin, or linear in a
// translation unit of its own so that the two compile in parallel)
template <bool LIN>
cudaError_t forward_mixed(int formalism, const void* tiles, int64_t n_tiles, const AntRec* ants, int n_ant,
                          const MedParams& M, void* acc, const FwdShape& shape, int sm_count, int* err,
                          cudaStream_t st) {
  FwdArgs a{tiles, n_tiles, ants, n_ant, shape.a_tile, acc, err, FwdGrid{}, M};
  auto go = [&](auto ops) {
    using O = decltype(ops);
    a.replicas = shape.replicas > 1 ? shape.replicas : 1;
    a.replica_stride = (int64_t)n_ant * M.n_bins * O::kAccRows;
    const int64_t ctas = forward_grid(a, shape, sm_count * forward_blocks_per_sm<O>(shape.a_tile),
                                      sizeof(float4) * O::kAccRows);
    return launch_forward_ops<O>(a, ctas, st);
  };
  const bool ex = M.kind == C8R_EXPONENTIAL;
  if (M.kind == C8R_EXPONENTIAL_SPHERICAL)
    return formalism == C8R_ENDPOINT ? go(OpsMixed<C8R_ENDPOINT, C8R_EXPONENTIAL_SPHERICAL, LIN>{})
           : M.flat                  ? go(OpsMixed<C8R_ZHS, C8R_EXPONENTIAL_SPHERICAL, LIN, kFormDirect, true>{})
                                     : go(OpsMixed<C8R_ZHS, C8R_EXPONENTIAL_SPHERICAL, LIN>{});
  if (M.kind == C8R_EXPONENTIAL_RAY)
    return formalism == C8R_ENDPOINT ? go(OpsMixed<C8R_ENDPOINT, C8R_EXPONENTIAL_RAY, LIN>{})
           : M.flat                  ? go(OpsMixed<C8R_ZHS, C8R_EXPONENTIAL_RAY, LIN, kFormDirect, true>{})
                                     : go(OpsMixed<C8R_ZHS, C8R_EXPONENTIAL_RAY, LIN>{});
  if constexpr (!LIN) {
    if (formalism == C8R_ENDPOINT) return with_endpoint_ops(M, go);
  }
  if (formalism == C8R_ENDPOINT)
    return ex ? go(OpsMixed<C8R_ENDPOINT, C8R_EXPONENTIAL, LIN>{}) : go(OpsMixed<C8R_ENDPOINT, C8R_UNIFORM, LIN>{});
  // ZHS in the exponential medium: for a flat array the kernel that forms the
  // midpoint's refractivity quotient and the z part of its d once per track
  // (OpsMixed::kFlat)
  if (ex && M.flat) return go(OpsMixed<C8R_ZHS, C8R_EXPONENTIAL, LIN, kFormDirect, true>{});
  return ex ? go(OpsMixed<C8R_ZHS, C8R_EXPONENTIAL, LIN>{}) : go(OpsMixed<C8R_ZHS, C8R_UNIFORM, LIN>{});
}

template <bool LIN>
cudaError_t backward_mixed(int formalism, BwdArgs& a, const FwdShape& shape, int sm_count, cudaStream_t st) {
  const bool ex = a.M.kind == C8R_EXPONENTIAL;
  if (formalism == C8R_ZHS) {
    if (ex && a.M.flat)
      return launch_backward_ops<OpsMixed<C8R_ZHS, C8R_EXPONENTIAL, LIN, kFormDirect, true>>(a, shape, sm_count, st);
    return ex ? launch_backward_ops<OpsMixed<C8R_ZHS, C8R_EXPONENTIAL, LIN>>(a, shape, sm_count, st)
              : launch_backward_ops<OpsMixed<C8R_ZHS, C8R_UNIFORM, LIN>>(a, shape, sm_count, st);
  }
  if constexpr (!LIN)
    return with_endpoint_ops(a.M, [&](auto ops) { return launch_backward_ops<decltype(ops)>(a, shape, sm_count, st); });
  return ex ? launch_backward_ops<OpsMixed<C8R_ENDPOINT, C8R_EXPONENTIAL, LIN>>(a, shape, sm_count, st)
            : launch_backward_ops<OpsMixed<C8R_ENDPOINT, C8R_UNIFORM, LIN>>(a, shape, sm_count, st);
}

}  // namespace c8r
