// c8r_device.cuh -- device-side building blocks of libc8r (sm_103a).
//
// The per-pair arithmetic follows the step the paper (§2) describes for every
// track and antenna: straight-line propagator -> formalism (Endpoint or ZHS,
// §1) -> deposit into the antenna's time-binned trace.  The formulas are those
// of the cited formalism papers (Endpoint: James et al., PRE 84 056602; ZHS:
// Zas, Halzen & Stanev, PRD 45 362), in SI units with times in ns at the
// interface.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>
#include <type_traits>

#include "../../include/c8r.h"

namespace c8r {

// ---------------------------------------------------------------------------
// physical constants (SI) and units
// ---------------------------------------------------------------------------
constexpr double kC = 299792458.0;              // m/s
constexpr double kCns = 0.299792458;            // m/ns
constexpr double kEps0 = 8.8541878128e-12;      // F/m
constexpr double kQe = 1.602176634e-19;         // C
constexpr double kPi = 3.14159265358979323846;
// Endpoint: K = e / (4 pi eps0 c)  [V s] per unit charge
constexpr double kKendpoint = kQe / (4.0 * kPi * kEps0 * kC);
// ZHS: K_A = mu0 e c / (4 pi), mu0 = 1/(eps0 c^2)  [V s] per unit charge
constexpr double kKzhs = (1.0 / (kEps0 * kC * kC)) * kQe * kC / (4.0 * kPi);

// tracks per derived tile (the unit of the TMA bulk copies)
constexpr int kTileT = 128;

// ---------------------------------------------------------------------------
// derived-track tiles written by the ingest kernel: per tile of kTileT tracks,
// field-major ([field][kTileT]) so one bulk copy moves a whole tile and lane i
// of a warp reads track i of a field without bank conflicts.
// ---------------------------------------------------------------------------
namespace fm {  // mixed precision (float fields)
enum : int {
  X0, Y0, Z0, X1, Y1, Z1,         // FP32 positions, m
  BX, BY, BZ,                     // beta
  AMPE,                           // q K / dt  [V]; 0 => track dropped by the filter
  AMPZ,                           // q K_A (t1 - t0)/dt  [V s]
  BMAG,                           // |beta|
  OMB,                            // 1 - |beta|
  TAU0H, TAU0L, TAU1H, TAU1L,     // t/dt, float-float
  DTAUH, DTAUL,                   // (t1 - t0)/dt, float-float
  E0H, E0L, E1H, E1L, EMH, EML,   // exp(-z/H) at start, end, midpoint (float-float)
  NFIELDS
};
}
namespace fd {  // FP64 path (double fields)
enum : int { X0, Y0, Z0, X1, Y1, Z1, BX, BY, BZ, Q, T0, T1, E0, E1, EM, NFIELDS };
}
constexpr int kTileBytesMixed = fm::NFIELDS * kTileT * 4;
constexpr int kTileBytesF64 = fd::NFIELDS * kTileT * 8;
static_assert(kTileBytesMixed % 16 == 0 && kTileBytesF64 % 16 == 0, "bulk copies move multiples of 16 bytes");

// ---------------------------------------------------------------------------
// antenna record (device table, built on the host in FP64)
// ---------------------------------------------------------------------------
struct AntRec {
  double x, y, z;        // m
  double t_ref;          // ns, first bin edge
  double Ea;             // exp(-z/H) (exponential medium), 1 otherwise
  // t_ref/dt + k z (k = n/(c dt) in the uniform medium, 1/(c dt) in the
  // exponential one) as float-float: the antenna's part of the shifted arrival
  // time of the FP32 arrival (arrival_fast)
  float Tah, Tal;
  float xh, yh, zh, xl, yl, zl;  // position as float-float
  float tauh, taul;              // t_ref / dt as float-float
  float Eah, Eal;                // Ea as float-float
  // constants of the error bound of the FP32 arrival (arrival_fast):
  // fb_abs = 2 x bins per metre x |low part of the position| + 16 u^2 |T_a| +
  // 1e-6 bin, and fb_rel_v = |z_l| / (1e-3 H), the relative error of the
  // refractivity term from the low part of the altitude (exponential medium;
  // 0 otherwise)
  float fb_abs, fb_rel_v;
};
static_assert(sizeof(AntRec) == 96, "antenna record layout");
static_assert(offsetof(AntRec, xh) % 16 == 0 && offsetof(AntRec, Tah) % 8 == 0,
              "the mixed path loads the float part as float4s and the shifted time as a float2");

// medium + binning parameters (kernel argument)
struct MedParams {
  int kind;              // C8R_UNIFORM / C8R_EXPONENTIAL
  int n_bins;
  double n;              // uniform index
  double N0, H, invH;    // exponential
  double R_E;            // spherical: Earth radius (m)
  double dt_ns, inv_dt;  // bin width and its reciprocal (per ns)
  double inv_c_ns;       // 1 / c in ns/m
  double eps_Cd;         // near-Cherenkov threshold (FP64 path)
  // float-float constants of the mixed path
  float kc_h, kc_l;      // 1/(c dt): bins per metre
  float s_h, s_l;        // uniform: n/(c dt)
  float cN_h, cN_l;      // exponential: N0 H /(c dt)
  float invH_h, invH_l;  // 1/H
  float N0f, nf;         // N0 and n as floats
  float idt_h, idt_l;    // 1/dt (per ns)
  float ampE;            // K/dt of the Endpoint amplitude (per unit charge), FP64 rounded once
  float kzhs;            // K_A of the ZHS amplitude
  float nm1f;            // uniform: n - 1 formed in FP64, then rounded (never (1 + x) - 1 in FP32)
  float RE_f;            // spherical: Earth radius (m)
  float RE_k;            // spherical: H / Earth radius
  float eps_C;           // near-Cherenkov threshold
  float dz_series;       // exponential: -1.001e-3 H, the altitude difference from where the quotient's series may apply
  uint32_t wait_limit;   // polls of a bounded wait on a staged track tile before it gives up
  // the form of the FP32 arrival (Endpoint, one-bin deposit, plain media): the
  // centroid of the antenna array, which the ingest's count of tracks seen
  // from above within 45 degrees refers to, and the host's choice from that
  // count (1: the split form of x = R - w)
  float cen_x, cen_y, cen_z;
  int split;
  // the axis form of the FP32 arrival, taken when axis != 0 (arrival_fast): the
  // axis, an FP32 vector of unit length up to rounding, and k/|ax| ax (k = n/(c dt)
  // or 1/(c dt)) as float-float
  int axis;
  float ax[3], kax_h[3], kax_l[3];
  // a flat antenna array (every antenna at one altitude z_a, exponential
  // media; spherical Earth: and within the range of its series, PathZ): z_a and exp(-z_a/H) as float-float, the same values the antenna
  // records hold, so that the quotient (E_e - E_a)/(z_a - z_e) of the
  // refractivity term, the same for every antenna, can be formed once per
  // track (OpsMixed::kFlat)
  int flat;
  float flat_zh, flat_zl, flat_Eh, flat_El;
  double flat_z, flat_E;  // the same for the FP64 path
};

// ---------------------------------------------------------------------------
// Reciprocal square root, quotient and exponential from the hardware's
// approximate operations (2 ulp), with denormal arguments taken as zero.  The
// plain rsqrtf, __fdividef and __expf cover denormals too and execute 4, 5 and
// about 4 instructions for it, against 1, 2 and 2 here (counted on this part);
// on normal arguments the values are the same, bit for bit (test_gpu_helpers).
// No argument here is denormal: distances are above 1e-19 m, and what divides
// is a distance, a product of distances or an altitude difference above
// 1e-3 H.  A pair has two such roots and eight quotients (Endpoint), so the
// counts per pair fall by about 30 of 290 instructions.  Measured, ms before ->
// after: Endpoint on 4e6 inclined tracks x 1024 antennas 43.3 -> 40.3; ZHS on
// 2.5e5 tracks over a spherical Earth x 1024 antennas 5.26 -> 4.46, with curved
// rays x 256 antennas 2.12 -> 1.70 (16 to 40 quotients, roots and exponentials
// per pair).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float rsqrt_ap(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rcp_ap(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float div_ap(float a, float b) { return __fmul_rn(a, rcp_ap(b)); }
// the smaller, or NaN if either is
__device__ __forceinline__ float min_nan(float a, float b) {
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float exp_ap(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__fmul_rn(x, 1.44269504088896341f)));
  return r;
}

// ---------------------------------------------------------------------------
// Two FP32 values at a time.  One add, multiply or fused multiply-add of a pair
// (add/mul/fma.rn.f32x2) takes one issue slot and rounds each half as the plain
// operation does; negations, absolute values and broadcast operands are free
// (counted on this part), while the FP32 pipe's rate per value stays the same.
// One exception, whatever -fmad says: the assembler makes one fused operation of
// a packed product that goes into packed sums only, which it never does with the
// plain ones.  Where such a sum decides a bin or a branch that other kernels form
// from plain values, the product is kept rounded: as two plain multiplications
// (mul_apart, an issue slot more), or with its sign turned (two_diff, none);
// test_gpu_bin_edges holds the outcome.
// The pair kernels are bound by issue, so the per-pair arithmetic is written
// once for T = float or float2 and the main passes run it on pairs: a pair's
// two endpoints (Endpoint).  Comparisons and the approximate reciprocals take
// each half apart.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float neg(float a) { return -a; }
__device__ __forceinline__ float abs_of(float a) { return fabsf(a); }
__device__ __forceinline__ float2 neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 abs_of(float2 a) { return make_float2(fabsf(a.x), fabsf(a.y)); }
__device__ __forceinline__ float2 add_rn(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub_rn(float2 a, float2 b) { return __fadd2_rn(a, neg(b)); }
__device__ __forceinline__ float2 mul_rn(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma_rn(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float mul_apart(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float2 mul_apart(float2 a, float2 b) {
  return make_float2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y));
}
__device__ __forceinline__ float2 rsqrt_ap(float2 x) { return make_float2(rsqrt_ap(x.x), rsqrt_ap(x.y)); }
__device__ __forceinline__ float2 rcp_ap(float2 x) { return make_float2(rcp_ap(x.x), rcp_ap(x.y)); }
__device__ __forceinline__ float2 div_ap(float2 a, float2 b) { return __fmul2_rn(a, rcp_ap(b)); }
// a value in every half
template <typename T>
__device__ __forceinline__ T bc(float a);
template <>
__device__ __forceinline__ float bc<float>(float a) { return a; }
template <>
__device__ __forceinline__ float2 bc<float2>(float a) { return make_float2(a, a); }
// Conditions that hold for nearly every pair (an emission point well above or
// below the antenna, an antenna ahead of the track) pick between two forms in
// the arithmetic below.  A plain value takes either; a float2 takes the usual
// form in both halves, and the caller, which tests all the conditions of a pair
// in one branch, redoes the rare pair half by half.
template <typename T>
constexpr bool kUsualForm = std::is_same<T, float2>::value;

// ---------------------------------------------------------------------------
// float-float ("double-float") arithmetic: error-free transformations after
// Knuth (TwoSum) and Dekker / the FMA form (TwoProd).  Intrinsics pin the
// rounding of every step; nothing here may be contracted or reassociated.
// ---------------------------------------------------------------------------
template <typename T>
struct ffT {
  T h, l;
};
using ff = ffT<float>;

template <typename T>
__device__ __forceinline__ void two_sum(T a, T b, T& s, T& e) {
  s = add_rn(a, b);
  const T bb = sub_rn(s, a);
  e = add_rn(sub_rn(a, sub_rn(s, bb)), sub_rn(b, bb));
}
// a - b exactly: the negated operand keeps a packed product b out of fused sums
template <typename T>
__device__ __forceinline__ void two_diff(T a, T b, T& s, T& e) {
  s = sub_rn(a, b);
  const T bb = sub_rn(s, a);
  e = sub_rn(sub_rn(a, sub_rn(s, bb)), add_rn(b, bb));
}
template <typename T>
__device__ __forceinline__ void two_prod(T a, T b, T& p, T& e) {
  p = mul_rn(a, b);
  e = fma_rn(a, b, neg(p));
}
// Dekker's Fast2Sum: exact when the exponent of a is at least that of b
template <typename T>
__device__ __forceinline__ void fast_two_sum(T a, T b, T& s, T& e) {
  s = add_rn(a, b);
  e = sub_rn(b, sub_rn(s, a));
}

// ---------------------------------------------------------------------------
// TMA bulk copies and mbarriers (inline PTX, sm_90+ forms valid on sm_103a)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
// global -> shared bulk copy; dst/src 16-byte aligned, bytes a multiple of 16
__device__ __forceinline__ void bulk_g2s(void* dst_smem, const void* src_gmem, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst_smem)),
      "l"(src_gmem), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: gives up after `limit` polls (each try_wait itself suspends for a
// while) and returns false.  Callers turn a give-up into an error status.
constexpr uint32_t kWaitLimit = 1u << 22;
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint32_t limit = kWaitLimit) {
  for (uint32_t i = 0; i < limit; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if (i > 64) __nanosleep(64);
  }
  return false;
}

// error word written by kernels that gave up a bounded wait
enum : int { kErrNone = 0, kErrWaitTimeout = 1, kErrCancelled = 2 };

// ---------------------------------------------------------------------------
// FP64 path: the plain formulas in FP64, in the order of their definition.
// ---------------------------------------------------------------------------
struct GeoD {
  double d[3], R, rh[3], n_src, n_avg;
};

// ---------------------------------------------------------------------------
// exponential atmosphere over a spherical Earth (centre (0, 0, -R_E)): the
// altitude excess of a point over the flat altitude z,
//   delta = h - z = |x - centre| - R_E - z = rho^2 / (|x - centre| + z + R_E),
// written without the cancellation of the first form.  The optical path is the
// flat closed form plus the integral along the straight path of
// N0 exp(-z/H) (exp(-delta/H) - 1), by 8-point Gauss-Legendre quadrature (nodes
// sigma_j on [0, 1] from the emission point, weights w_j summing to 1).
// ---------------------------------------------------------------------------
// Quotient, square root and exponential for the small corrections (the
// sphere's curvature part of the optical path, the curved ray's turn and time
// saved): their FP32 forms need ~1e-6 relative accuracy, so they use the
// approximate hardware operations; the FP64 forms round as written.
template <typename T>
__device__ __forceinline__ T approx_div(T a, T b) { return a / b; }
template <>
__device__ __forceinline__ float approx_div<float>(float a, float b) { return div_ap(a, b); }
template <typename T>
__device__ __forceinline__ T approx_sqrt(T x) { return sqrt(x); }  // x > 0
template <>
__device__ __forceinline__ float approx_sqrt<float>(float x) { return x * rsqrt_ap(x); }
template <typename T>
__device__ __forceinline__ T approx_exp(T x) { return exp(x); }
template <>
__device__ __forceinline__ float approx_exp<float>(float x) { return exp_ap(x); }

constexpr int kSphNodes = 8;
__device__ __constant__ const double kSphSigma[kSphNodes] = {
    0.019855071751231856, 0.10166676129318664, 0.2372337950418355, 0.4082826787521751,
    0.5917173212478249,   0.7627662049581645,  0.8983332387068134, 0.9801449282487681};
__device__ __constant__ const double kSphWeight[kSphNodes] = {
    0.05061426814518813, 0.11119051722668724, 0.15685332293894363, 0.18134189168918100,
    0.18134189168918100, 0.15685332293894363, 0.11119051722668724, 0.05061426814518813};

template <typename T>
__device__ __forceinline__ T sphere_excess(T x, T y, T z, T R_E) {
  const T rho2 = x * x + y * y;
  const T zr = z + R_E;
  return approx_div(rho2, approx_sqrt(rho2 + zr * zr) + zr);
}
// exp(-x) - 1 for x >= 0 without cancellation
template <typename T>
__device__ __forceinline__ T exp_m1_neg(T x) {
  if (x < T(0.1)) return -x * (T(1) + x * (T(-0.5) + x * (T(1) / T(6) + x * (T(-1) / T(24) + x * (T(1) / T(120))))));
  return approx_exp(-x) - T(1);
}
// the curvature part of the optical path from x_e to the antenna a, d = a - x_e
template <typename T>
__device__ __forceinline__ T sphere_path_correction(T ax, T ay, T az, T dx, T dy, T dz, T R, T N0, T invH, T R_E) {
  T sum = T(0);
#pragma unroll
  for (int j = 0; j < kSphNodes; ++j) {
    const T f = T(1) - T(kSphSigma[j]);  // the node at x_e + sigma d = a - (1 - sigma) d
    const T x = ax - f * dx, y = ay - f * dy, z = az - f * dz;
    const T ex = sphere_excess(x, y, z, R_E);
    sum += T(kSphWeight[j]) * approx_exp(-z * invH) * exp_m1_neg(ex * invH);
  }
  return N0 * R * sum;
}

// ---------------------------------------------------------------------------
// curved rays in the flat exponential atmosphere (C8R_EXPONENTIAL_RAY).  The ray
// from x_e to the antenna keeps n(z) sin(theta) = p.  Written p = S m, with S =
// rho/R and C = |dz|/R the straight line's sine and cosine from the vertical and
// mu = m - 1 an effective refractivity, the ray's turn away from the straight
// line at height z is
//   sin(theta - theta_s) = S Q,  Q = (mu - nu)(2 + mu + nu) / (n^2 (C m/n + cos theta)),
// nu = n - 1, free of the cancellation of the direct difference.  The end-point
// condition, integral over z of (tan theta - tan theta_s) = 0, reads
// sum_j w_j k_j (mu - nu_j) = 0 with k_j = (2 + mu + nu_j)/(n_j^2 (C m/n_j +
// cos theta_j) cos theta_j) > 0 at the Gauss-Legendre nodes, so mu is the
// k-weighted mean of nu: a fixed point whose contraction factor is ~1e-4 (each
// iteration gains about four digits; from the plain mean, one iteration leaves
// < 1e-12 of mu for paths up to 40 km, three leave < 1e-18).  The optical path then differs from the
// straight line's by exactly
//   - integral over z of 2 n sin^2((theta - theta_s)/2)/C
//   = - R S^2 sum_j w_j n_j Q_j^2 / (1 + cos(theta_j - theta_s))
// (Fermat: from n sin(theta) = p and the shared end points), a small negative
// quantity formed directly, which is added to the straight path's closed form.
// Paths within 1e-3 of the horizontal, and vertical ones, keep the straight line.
// ---------------------------------------------------------------------------
template <typename T>
struct RayFix {
  T Q;    // sin(turn at x_e) = S Q
  T dop;  // ray's optical path minus the straight line's (m, <= 0)
};
template <typename T, int ITERS>
__device__ __forceinline__ RayFix<T> ray_fix(T rho2, T dz, T R, T nu_e, T invH) {
  RayFix<T> r{T(0), T(0)};
  const T adz = fabs(dz);
  if (!(rho2 > T(0)) || !(adz >= T(1e-3) * R)) return r;
  const T invR = approx_div(T(1), R);
  const T S = approx_sqrt(rho2) * invR, C = adz * invR;
  T nu[kSphNodes];
  T mu = T(0);
#pragma unroll
  for (int j = 0; j < kSphNodes; ++j) {
    nu[j] = nu_e * approx_exp(-T(kSphSigma[j]) * dz * invH);  // z = z_e + sigma dz
    mu += T(kSphWeight[j]) * nu[j];
  }
#pragma unroll
  for (int it = 0; it < ITERS; ++it) {
    const T m = T(1) + mu;
    T num = T(0), den = T(0);
#pragma unroll
    for (int j = 0; j < kSphNodes; ++j) {
      const T in = approx_div(T(1), T(1) + nu[j]);
      const T a = S * m * in;
      const T c2 = T(1) - a * a;
      if (!(c2 > T(0))) return RayFix<T>{T(0), T(0)};
      const T c = approx_sqrt(c2);
      const T k = approx_div((T(2) + mu + nu[j]) * in * in, (C * m * in + c) * c);
      num += T(kSphWeight[j]) * k * nu[j];
      den += T(kSphWeight[j]) * k;
    }
    mu = approx_div(num, den);
  }
  const T m = T(1) + mu;
  T sum = T(0);
#pragma unroll
  for (int j = 0; j < kSphNodes; ++j) {
    const T n = T(1) + nu[j];
    const T in = approx_div(T(1), n);
    const T a = S * m * in;
    const T c2 = T(1) - a * a;
    if (!(c2 > T(0))) return RayFix<T>{T(0), T(0)};
    const T Q = approx_div((mu - nu[j]) * (T(2) + mu + nu[j]) * in * in, C * m * in + approx_sqrt(c2));
    const T sd = S * Q;
    sum += T(kSphWeight[j]) * approx_div(n * Q * Q, T(1) + approx_sqrt(T(1) - sd * sd));
  }
  r.dop = -R * S * S * sum;
  const T in = approx_div(T(1), T(1) + nu_e);
  const T a = S * m * in;
  const T c2 = T(1) - a * a;
  if (!(c2 > T(0))) return RayFix<T>{T(0), T(0)};
  r.Q = approx_div((mu - nu_e) * (T(2) + mu + nu_e) * in * in, C * m * in + approx_sqrt(c2));
  return r;
}

// the turn of the direction d = x_a - x_e (length R) at x_e in the vertical plane,
// as the change of R rhat: sin(delta) R t + (cos(delta) - 1) d, with t the unit
// vector away from the vertical, R t = (|dz| d_h/rho, -sgn(dz) rho) and
// sin(delta) = (rho/R) Q
template <typename T>
__device__ __forceinline__ void ray_turn_vector(T dx, T dy, T dz, T R, T Q, T out[3]) {
  const T rho2 = dx * dx + dy * dy;
  const T invR = approx_div(T(1), R);
  const T sd = approx_sqrt(rho2) * invR * Q;
  const T cdm1 = approx_div(-sd * sd, T(1) + approx_sqrt(T(1) - sd * sd));
  const T f = cdm1 + Q * fabs(dz) * invR;
  out[0] = f * dx;
  out[1] = f * dy;
  out[2] = cdm1 * dz - (dz < T(0) ? T(-1) : T(1)) * Q * rho2 * invR;
}

// straight emission path x_e -> antenna (propagator, §2): distance, direction,
// source index and path-averaged index of the medium
__device__ __forceinline__ void geo_f64(const MedParams& M, const AntRec& A, double xe, double ye, double ze,
                                        double Ee, GeoD& g) {
  g.d[0] = A.x - xe;
  g.d[1] = A.y - ye;
  g.d[2] = A.z - ze;
  g.R = sqrt(g.d[0] * g.d[0] + g.d[1] * g.d[1] + g.d[2] * g.d[2]);
  double invR = 1.0 / g.R;
  g.rh[0] = g.d[0] * invR;
  g.rh[1] = g.d[1] * invR;
  g.rh[2] = g.d[2] * invR;
  if (M.kind == C8R_UNIFORM) {
    g.n_src = M.n;
    g.n_avg = M.n;
  } else {
    g.n_src = 1.0 + M.N0 * Ee;
    // path average of N0 exp(-z/H) between z_e and z_a: N0 H (E_e - E_a) / dz,
    // or its series in x = dz/H when the two altitudes nearly coincide
    double dz = g.d[2];
    double x = dz * M.invH;
    double ratio;
    if (fabs(x) > 1e-3)
      ratio = (Ee - A.Ea) / x;
    else
      ratio = Ee * (1.0 + x * (-0.5 + x * (1.0 / 6.0 + x * (-1.0 / 24.0 + x * (1.0 / 120.0)))));
    g.n_avg = 1.0 + M.N0 * ratio;
    if (M.kind == C8R_EXPONENTIAL_SPHERICAL) {
      g.n_src = 1.0 + M.N0 * Ee * exp(-sphere_excess(xe, ye, ze, M.R_E) * M.invH);
      g.n_avg += sphere_path_correction<double>(A.x, A.y, A.z, g.d[0], g.d[1], g.d[2], g.R, M.N0, M.invH, M.R_E) /
                 g.R;
    } else if (M.kind == C8R_EXPONENTIAL_RAY) {
      // the refracted ray: its direction at x_e and its optical path
      const RayFix<double> r =
          ray_fix<double, 3>(g.d[0] * g.d[0] + g.d[1] * g.d[1], g.d[2], g.R, M.N0 * Ee, M.invH);
      double t[3];
      ray_turn_vector<double>(g.d[0], g.d[1], g.d[2], g.R, r.Q, t);
      for (int c = 0; c < 3; ++c) g.rh[c] = (g.d[c] + t[c]) * invR;
      g.n_avg += r.dop * invR;
    }
  }
}

// arrival position in bins relative to the antenna's first bin edge
__device__ __forceinline__ double arrival_f64(const MedParams& M, const GeoD& g, double t_e, double t_ref) {
  return ((t_e - t_ref) + g.n_avg * g.R * M.inv_c_ns) / M.dt_ns;
}

// ---------------------------------------------------------------------------
// mixed path: FP32 field arithmetic; arrival time in float-float
// ---------------------------------------------------------------------------
template <typename T>
struct GeoT {
  T s[3], e[3];  // d = x_a - x_e as float-float per component
  T R0, R1;      // |d| as float-float (R1 = 0 until geo_refine)
  T y;           // ~1/R0 (rsqrt estimate)
};
using GeoM = GeoT<float>;

// d = a - p (p given as float-float; p_l = 0 for the FP32-exact endpoints) and
// an FP32 estimate of R = |d| (enough for the Doppler factor and amplitudes)
__device__ __forceinline__ void geo_lite(const AntRec& A, float pxh, float pyh, float pzh, float pxl, float pyl,
                                         float pzl, GeoM& g) {
  two_sum(A.xh, -pxh, g.s[0], g.e[0]);
  two_sum(A.yh, -pyh, g.s[1], g.e[1]);
  two_sum(A.zh, -pzh, g.s[2], g.e[2]);
  g.e[0] = __fadd_rn(g.e[0], __fsub_rn(A.xl, pxl));
  g.e[1] = __fadd_rn(g.e[1], __fsub_rn(A.yl, pyl));
  g.e[2] = __fadd_rn(g.e[2], __fsub_rn(A.zl, pzl));
  const float S = __fmaf_rn(g.s[2], g.s[2], __fmaf_rn(g.s[0], g.s[0], __fmul_rn(g.s[1], g.s[1])));
  g.y = rsqrt_ap(S);
  g.R0 = __fmul_rn(S, g.y);
  g.R1 = 0.0f;
}

// R = |d| in float-float: the three exact squares are summed with TwoSum, then
// one Newton step corrects the FP32 estimate R0 (its square is formed exactly)
// the same for an FP32-exact point (no low part)
__device__ __forceinline__ void geo_lite(const AntRec& A, float px, float py, float pz, GeoM& g) {
  two_sum(A.xh, -px, g.s[0], g.e[0]);
  two_sum(A.yh, -py, g.s[1], g.e[1]);
  two_sum(A.zh, -pz, g.s[2], g.e[2]);
  g.e[0] = __fadd_rn(g.e[0], A.xl);
  g.e[1] = __fadd_rn(g.e[1], A.yl);
  g.e[2] = __fadd_rn(g.e[2], A.zl);
  const float S = __fmaf_rn(g.s[2], g.s[2], __fmaf_rn(g.s[0], g.s[0], __fmul_rn(g.s[1], g.s[1])));
  g.y = rsqrt_ap(S);
  g.R0 = __fmul_rn(S, g.y);
  g.R1 = 0.0f;
}

// the z part of d = a - p that every antenna of a flat array (one altitude)
// shares: d_z as float-float and the products of it that geo_refine and
// doppler_ff form, formed once per point as they form them (so the same values)
template <typename T>
struct ZPartT {
  T sh, sl;  // d_z = sh + sl (geo_lite's s[2], e[2])
  T qh, ql;  // sh^2, exact
  T se;      // fl(sh sl)
  T bh, bl;  // b_z sh, exact
  T be;      // fl(b_z sl)
};
using ZPart = ZPartT<float>;
template <typename T>
__device__ __forceinline__ ZPartT<T> z_part(T sh, T sl, T bz) {
  ZPartT<T> z;
  z.sh = sh;
  z.sl = sl;
  two_prod(sh, sh, z.qh, z.ql);
  z.se = mul_rn(sh, sl);
  two_prod(bz, sh, z.bh, z.bl);
  z.be = mul_rn(bz, sl);
  return z;
}

// geo_lite of a float-float point whose z part comes from ZPart; the antenna's
// x and y as float-float
template <typename T>
__device__ __forceinline__ void geo_lite(T axh, T ayh, T axl, T ayl, T pxh, T pyh, T pxl, T pyl, const ZPartT<T>& z,
                                         GeoT<T>& g) {
  two_sum(axh, neg(pxh), g.s[0], g.e[0]);
  two_sum(ayh, neg(pyh), g.s[1], g.e[1]);
  g.s[2] = z.sh;
  g.e[2] = z.sl;
  g.e[0] = add_rn(g.e[0], sub_rn(axl, pxl));
  g.e[1] = add_rn(g.e[1], sub_rn(ayl, pyl));
  const T S = fma_rn(g.s[2], g.s[2], fma_rn(g.s[0], g.s[0], mul_rn(g.s[1], g.s[1])));
  g.y = rsqrt_ap(S);
  g.R0 = mul_rn(S, g.y);
  g.R1 = bc<T>(0.0f);
}

// R from the exact squares of d's components (p2 + q2 = s_z^2 and se =
// fl(s_z e_z) given)
template <typename T>
__device__ __forceinline__ void geo_refine(GeoT<T>& g, T p2, T q2, T se) {
  T p0, q0, p1, q1;
  two_prod(g.s[0], g.s[0], p0, q0);
  two_prod(g.s[1], g.s[1], p1, q1);
  T S1, E1, S2, E2;
  two_sum(p0, p1, S1, E1);
  two_sum(S1, p2, S2, E2);
  const T cross = fma_rn(g.s[0], g.e[0], fma_rn(g.s[1], g.e[1], se));
  const T lo = add_rn(add_rn(add_rn(q0, q1), add_rn(q2, E1)), add_rn(E2, mul_rn(bc<T>(2.0f), cross)));
  T rq, rqe;
  two_prod(g.R0, g.R0, rq, rqe);
  const T rho = add_rn(sub_rn(sub_rn(S2, rq), rqe), lo);
  g.R1 = mul_rn(mul_rn(rho, bc<T>(0.5f)), g.y);
}
template <typename T>
__device__ __forceinline__ void geo_refine(GeoT<T>& g) {
  T p2, q2;
  two_prod(g.s[2], g.s[2], p2, q2);
  geo_refine(g, p2, q2, mul_rn(g.s[2], g.e[2]));
}
template <typename T>
__device__ __forceinline__ void geo_refine(GeoT<T>& g, const ZPartT<T>& z) {
  geo_refine(g, z.qh, z.ql, z.se);
}

// (E_e - E_a)/dz in float-float, the quotient of the refractivity term of the
// exponential medium, dz = dzh + dzl the altitude difference a - e: the FP32
// quotient corrected once from the exact residual, or for |dz/H| <= 1e-3 the
// series (E_e/H)(1 + f), f = -x/2 + x^2/6 - x^3/24, x = dz/H
template <typename T>
__device__ __forceinline__ void refr_quotient(const MedParams& M, T Eah, T Eal, T dzh, T dzl, T Eeh, T Eel, T& q0,
                                              T& q1) {
  if constexpr (!kUsualForm<T>) {
    const float x = __fmul_rn(dzh, M.invH_h);
    if (!(fabsf(x) > 1e-3f)) {
      const float f = __fmul_rn(x, __fmaf_rn(x, __fmaf_rn(x, -1.0f / 24.0f, 1.0f / 6.0f), -0.5f));
      float eh, el;
      two_prod(Eeh, M.invH_h, eh, el);
      el = __fmaf_rn(Eeh, M.invH_l, __fmaf_rn(Eel, M.invH_h, el));
      // (eh + el)(1 + f)
      float g0, g1;
      two_sum(eh, __fmul_rn(eh, f), g0, g1);
      q0 = g0;
      q1 = __fadd_rn(g1, __fmaf_rn(el, f, el));
      return;
    }
  }
  T Qh, Ql;
  two_sum(Eeh, neg(Eah), Qh, Ql);
  Ql = add_rn(Ql, sub_rn(Eel, Eal));
  const T r = rcp_ap(dzh);
  q0 = mul_rn(Qh, r);
  T ph, pl;
  two_prod(q0, dzh, ph, pl);
  q1 = mul_rn(sub_rn(add_rn(sub_rn(sub_rn(Qh, ph), pl), Ql), mul_rn(q0, dzl)), r);
}

// arrival position u = (t_e - t_ref)/dt + n_avg R / (c dt) in bins, float-float,
// with the refractivity quotient (q0, q1) given (exponential media; ignored in
// the uniform one).  tau_e = t_e/dt and the antenna's tau = t_ref/dt come in
// float-float.  KIND: the medium kind (a template argument, so each kernel
// carries only its own medium's arithmetic; it equals M.kind).  `corr` (curved
// rays, spherical Earth): the optical path minus the flat straight line's, m
template <int KIND, typename T>
__device__ __forceinline__ ffT<T> arrival_mixed_q(const MedParams& M, T atauh, T ataul, const GeoT<T>& g, T tauh, T taul,
                                                  T q0, T q1, T corr = bc<T>(0.0f)) {
  T ts, te;
  two_sum(tauh, neg(atauh), ts, te);
  te = add_rn(te, sub_rn(taul, ataul));
  const T sh = bc<T>((KIND == C8R_UNIFORM) ? M.s_h : M.kc_h);
  const T sl = bc<T>((KIND == C8R_UNIFORM) ? M.s_l : M.kc_l);
  T p, pe;
  two_prod(g.R0, sh, p, pe);
  pe = fma_rn(g.R0, sl, fma_rn(g.R1, sh, pe));
  if constexpr (KIND != C8R_UNIFORM) {
    // refractivity term (n_avg - 1) R/(c dt) = N0 H/(c dt) * (E_e - E_a)/dz * R
    T w, we;
    two_prod(q0, g.R0, w, we);
    we = fma_rn(q0, g.R1, fma_rn(q1, g.R0, we));
    T v, ve;
    two_prod(w, bc<T>(M.cN_h), v, ve);
    ve = fma_rn(w, bc<T>(M.cN_l), fma_rn(we, bc<T>(M.cN_h), ve));
    T p2, pe2;
    fast_two_sum(p, v, p2, pe2);  // |v| = (n_avg - 1)|p| < |p|
    p = p2;
    pe = add_rn(pe, add_rn(pe2, ve));
    if constexpr (KIND == C8R_EXPONENTIAL_SPHERICAL || KIND == C8R_EXPONENTIAL_RAY) {
      // the small change of the optical path in bins (the sphere's curvature,
      // ~1e-3 of the refractivity term; the ray's time saved, <~1 bin): FP32 is enough
      fast_two_sum(p, mul_apart(corr, bc<T>(M.kc_h)), p2, pe2);
      p = p2;
      pe = add_rn(pe, pe2);
    }
  }
  T uh, ue;
  two_sum(ts, p, uh, ue);
  ue = add_rn(ue, add_rn(te, pe));
  return ffT<T>{uh, ue};
}

// the same with the quotient formed here, from the emission point's E_e =
// exp(-z_e/H) and the altitude difference of g
template <int KIND>
__device__ __forceinline__ ff arrival_mixed(const MedParams& M, const AntRec& A, const GeoM& g, float tauh, float taul,
                                            float Eeh, float Eel, float dop = 0.0f) {
  float q0 = 0.0f, q1 = 0.0f;
  if constexpr (KIND != C8R_UNIFORM) refr_quotient(M, A.Eah, A.Eal, g.s[2], g.e[2], Eeh, Eel, q0, q1);
  if constexpr (KIND == C8R_EXPONENTIAL_SPHERICAL)
    dop = sphere_path_correction<float>(A.xh, A.yh, A.zh, g.s[0], g.s[1], g.s[2], g.R0, M.N0f, M.invH_h, M.RE_f);
  return arrival_mixed_q<KIND>(M, A.tauh, A.taul, g, tauh, taul, q0, q1, dop);
}

// bin index of a float-float arrival, clamped to [-1, n_bins]: -1 stands for
// "before the window" (or not a number), n_bins for "after it"; frac is the
// position inside the bin (meaningful only for an index inside the window)
__device__ __forceinline__ int bin_raw(ff u, int n_bins, float& frac) {
  frac = 0.0f;
  if (!(u.h > -1.0f)) return -1;
  // quick reject of arrivals well after the window (and of +inf).  The low part
  // is not renormalised: near 2^24 bins, where FP32 is spaced by 1 or 2, it can
  // reach a few units (u = 2^24 - 0.35, in the last bin of the largest window,
  // can come as u.h = 2^24 + 2, u.l = -2.35), so the bound leaves room for a low
  // part of up to 64 in magnitude (an arrival of ~1e9 bins)
  if (!(u.h < (float)n_bins + 64.0f)) return n_bins;
  float kf = floorf(u.h);
  float f = __fadd_rn(__fsub_rn(u.h, kf), u.l);
  // bring the fraction into [0, 1) by its own floor: the low part is not
  // renormalised, and for an arrival near 2^24 bins (FP32 spacing 1 or 2 there)
  // it can exceed 1 in magnitude, so a single step of +-1 would not do
  const float df = floorf(f);
  kf = __fadd_rn(kf, df);
  f = __fsub_rn(f, df);
  int k = (int)kf;
  frac = f;
  if (k < 0) return -1;
  if (k >= n_bins) return n_bins;
  return k;
}
// ---------------------------------------------------------------------------
// Bin of an arrival from plain FP32 arithmetic with a bound on its error, for
// the one-bin deposit (reading T: only the bin of an arrival matters there).
// The float-float arrival (arrival_mixed, ~1e-9 bin) costs about four times the
// FP32 one.  The FP32 arrival decides the bin whenever no bin edge (and neither
// end of the window) lies within its error bound; then it is the bin of the
// float-float arrival too, which is good to ~1e-7 bin at most, far inside the
// bound's 1e-6-bin floor.  Otherwise the caller evaluates the float-float
// arrival.
//
// Vertical split.  With w = z_e - z_a (the emission point's height above the
// antenna) and rho^2 = d_x^2 + d_y^2, the distance is R = w + x, where
// x = R - w = rho^2 / (R + w) since R^2 = w^2 + rho^2.  So
//   u = (tau_e - tau_a) + k R + v = (T_e - T_a) + k x + v,
//   T_e = tau_e + k z_e (per track endpoint), T_a = tau_a + k z_a (per antenna),
// with k = n/(c dt) in the uniform medium and 1/(c dt) in the exponential one
// (where v carries the refractivity).  T_e and T_a are formed once, in
// float-float, so no per-pair FP32 rounding acts on a term as large as k R
// (~1e5 bins): FP32 rounds T_e - T_a, about the arrival's own distance from
// the window start, and k x, which is small for emission points high above the
// antenna (x ~ R theta^2 / 2 at an angle theta off the vertical).  The split
// form x = rho^2 / (R + w) pays where x is small against R; elsewhere (an
// inclined line of sight, or a point below the antenna, w <= 0) the direct form
// x = R - w = fl(R + s_z) has the smaller error, and the caller picks the form
// (SPLIT below) for a whole warp: the split one when every lane's emission
// point lies within 45 degrees of the antenna's vertical (2 rho^2 < S, w > 0).
//
// The errors, with u = 2^-24 (the FP32 unit roundoff) and every step rounded
// once (intrinsics, no contraction):
//   s = fl(a_h - p): each component is off the exact d = a - p by at most
//     u |s_i| and the antenna's low part a_l.  x changes with s_z at the rate
//     x/R and with s_x, s_y at |s_{x,y}|/R, so the rounding moves x by at most
//     u (x + rho^2 / R) <= 3u x (also for w <= 0, where x >= R); a_l moves it by
//     at most 2 |a_l| (T_a holds the exact z_a);
//   rho^2 = fl(s_x^2 + s_y^2) (two roundings, 2u) and S = fl(s_z^2 + rho^2):
//     R' = S rsqrt(S) plus one Newton step with the residual fma(-R0, R0, S) is
//     sqrt(S) rounded once, within 2.5u R of |s|;
//   split form, w > 0: x = rho^2 / fl(R0 - s_z) with div_ap (2 ulp: 4u),
//     from the unrefined R0 = fl(S rsqrt_ap(S)) (rsqrtf 2 ulp: R0 within 6u R of
//     |s|, so the denominator R + |s_z| >= R carries 7u); with rho^2, 13u x.
//     (w <= 0: x = fl(R0 + s_z) >= R, 7u x.)  Direct form: x = fl(R' + s_z),
//     2.5u R + u x;
//   q = fl(x k_h): u, and u more for the dropped k_l;
//   Td = fl(fl(T_e,h - T_a,h) + fl(T_e,l - T_a,l)): 2u |Td|, plus terms of
//     u^2 |T_e| and u^2 |T_a| from the float-float forms of T_e and T_a;
//   v (exponential medium) = N0 H/(c dt) (E_e - E_a)/dz R' (R0 in the split
//     form): the quotient (2 ulp) or its series for |dz/H| <= 1e-3, four more
//     roundings and R' give at most 14u |v| (17.5u with R0), plus
//     |v| |z_l|/|dz| from the antenna altitude's low part, |dz| > 1e-3 H in
//     the quotient's branch;
//   uf = fl(fl(Td + q) + v): u |Td + q| <= u (|uf| + |v|) (Td + q is uf - v
//     before the last rounding, small against Td and q once the arrival is
//     near the window) and u |uf|, and one more u |uf| in the window test
//     uf - bound >= n_bins.
// The bound used is u (2.25 |Td| + c_q q + c_v |v| + 3.25 |uf|) + fb_rel_v |v| +
// fb_abs, with c_q = 19 and c_v = 22 in the split form (18 and 17.5 derived)
// and c_q = 6.25, c_v = 17 plus 2.5u k_h R in the direct one (6, 14 and 2.5),
// each coefficient above its derivation; fb_abs holds 2 k |a_l|,
// 16 u^2 |T_a| (the share of T_e, |T_e| <= |Td| + |T_a|, beyond what the |Td|
// term covers) and a floor of 1e-6 bin for the float-float arrival's own error
// and the rounding of uf - floor(uf).  A CPU emulation of these steps (2-ulp
// reciprocal square root and quotient) against the FP64 oracle's arrivals
// stays below 0.6 of the bound on the benchmark showers; on a vertical shower
// 1-10 km above 0.2-ns traces the bound is ~6e-4 bin and ~0.1 % of the
// endpoints are left to the float-float arrival (8 % with k R rounded in FP32
// per pair).  On a shower inclined by 60 degrees x is about R/2 and the direct
// form holds the bound near that of an arrival rounded in FP32 throughout.
// ---------------------------------------------------------------------------
// Along an axis (kFormAxis).  The vertical split carries over to any direction A:
// with w = -(d . A)/|A| and x = R - w = |d x A|^2/(|A| (|A| R - d . A)), T = tau + k
// (position . A)/|A|.  A shower's lines of sight all lie near its axis, so x and
// its error stay small for inclined showers too, where the direct form rounds
// terms of k R.  A is an FP32 vector taken exactly; its length, 1 within 3u, enters
// T through k/|A| and is dropped from x (9u x at most).  The errors, where w >= 0:
//   s: |delta| <= u R (2-norm), and x changes with d at |d/R + A| = sqrt(2x/R), so
//     u sqrt(2 x R); a_l: at most 2 |a_l|, as above;
//   c = fl(s x A): each component off by u |s_j A_k| + u |c_i|, u (R + rho) in 2-norm,
//     rho = |c|, rho^2 = x (2R - x) <= 2 x R; it moves x = rho^2/(R + w) by at most
//     2 rho u (R + rho)/R <= 4 u rho;
//   together at most 5.5 u sqrt(2 x R) <= 5.5 u (8 x + R/16), an arithmetic mean;
//   rho^2 3u, R0 6u R, w 3u R and the denominator's rounding u (R + w >= R), the
//     quotient 4u and |A| 9u: 26u x;
//   q, Td, v, uf as in the split form.
// The bound used is u (2.25 |Td| + 72 q + 22 |v| + 3.25 |uf| + 0.375 k R) + fb_rel_v |v|
// + fb_abs with 16 u^2 |T_a| of the axis' T_a (2 + 26 + 44 and 0.344 derived).  Where w <
// 0 (a line of sight beyond 90 degrees from the axis) x = fl(R0 - w), and 10 k R in
// place of 0.375 k R covers R0's and w's errors.  q_extra, for a geometry whose d is
// off by q_extra/1.5 times the above, adds u q_extra (8 q + k R/16).  On showers at 12 to
// 75 degrees 0.4 % of the in-window endpoints are left undecided at 0.2 ns per bin,
// against 0.3 to 12 % (split) and 2 to 7 % (direct); the worst error was 0.11 of the
// bound (test_fp32_axis_bound).
enum : int { kFormDirect = 0, kFormSplit = 1, kFormAxis = 2 };

constexpr int kFastOut = -1;        // the arrival lies outside the window: no deposit
constexpr int kFastUndecided = -2;  // an edge lies within the bound: the float-float arrival decides

// d = a_h - p in FP32 (no low parts), rho^2 = d_x^2 + d_y^2, S = |d|^2 and
// R0 = |d| as geo_lite forms them (the same s, y and R0 bit for bit)
template <typename T>
__device__ __forceinline__ void geo_fast(T ax, T ay, T az, T px, T py, T pz, GeoT<T>& g, T& S, T& rho2) {
  g.s[0] = sub_rn(ax, px);
  g.s[1] = sub_rn(ay, py);
  g.s[2] = sub_rn(az, pz);
  rho2 = fma_rn(g.s[0], g.s[0], mul_rn(g.s[1], g.s[1]));
  S = fma_rn(g.s[2], g.s[2], rho2);
  g.y = rsqrt_ap(S);
  g.R0 = mul_rn(S, g.y);
  g.R1 = bc<T>(0.0f);
}

// T = tau + k z as float-float, the shifted time of arrival_fast, for a height
// z = zh + zl (zl = 0 for an FP32-exact endpoint)
__device__ __forceinline__ void shifted_time(float tauh, float taul, float zh, float zl, float kh, float kl,
                                             float& Th, float& Tl) {
  float p, e;
  two_prod(zh, kh, p, e);
  e = __fmaf_rn(zh, kl, __fmaf_rn(zl, kh, e));
  float s, e2;
  two_sum(tauh, p, s, e2);
  e2 = __fadd_rn(e2, __fadd_rn(taul, e));
  fast_two_sum(s, e2, Th, Tl);
}

// T = tau + k (p . A)/|A| as float-float for a position p given as float-float
__device__ __forceinline__ void axis_time(const MedParams& M, float tauh, float taul, const float ph[3],
                                          const float pl[3], float& Th, float& Tl) {
  float h = tauh, l = taul;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float p, e, s, e2;
    two_prod(ph[c], M.kax_h[c], p, e);
    e = __fmaf_rn(ph[c], M.kax_l[c], __fmaf_rn(pl[c], M.kax_h[c], e));
    two_sum(h, p, s, e2);
    l = __fadd_rn(l, __fadd_rn(e, e2));
    h = s;
  }
  fast_two_sum(h, l, Th, Tl);
}

// w = -(d . A) of the axis form
template <typename T>
__device__ __forceinline__ T axis_w(const MedParams& M, const GeoT<T>& g) {
  return neg(fma_rn(g.s[0], bc<T>(M.ax[0]), fma_rn(g.s[1], bc<T>(M.ax[1]), mul_rn(g.s[2], bc<T>(M.ax[2])))));
}

// the FP32 quotient (E_e - E_a)/dz of the refractivity term for the FP32
// arrival (exponential medium); dz = s_z, the FP32 a_h - p of the emission
// point (the same for every antenna of a flat array); for |dz/H| <= 1e-3 its
// series (E_e/H)(1 + f)
template <typename T>
__device__ __forceinline__ T fast_quotient(const MedParams& M, T Eah, T Eal, T sz, T Eeh, T Eel) {
  if constexpr (!kUsualForm<T>) {
    const float x = __fmul_rn(sz, M.invH_h);
    if (!(fabsf(x) > 1e-3f)) {
      const float f = __fmul_rn(x, __fmaf_rn(x, __fmaf_rn(x, -1.0f / 24.0f, 1.0f / 6.0f), -0.5f));
      return __fmul_rn(__fmul_rn(Eeh, M.invH_h), __fadd_rn(1.0f, f));
    }
  }
  return div_ap(add_rn(sub_rn(Eeh, Eah), sub_rn(Eel, Eal)), sz);
}

// The FP32 arrival uf of the emission point of g (S = |d|^2, rho2 = d_x^2 +
// d_y^2, T_e = Teh + Tel, the antenna's T_a = Tah + Tal and bound constants, qv
// the refractivity quotient of fast_quotient) and its error bound, returned; AF picks the form of x; q_extra adds a term
// u * q_extra * k x for geometry whose d carries more than the one rounding of
// a_h - p (the midpoint)
template <int KIND, int AF, typename T>
__device__ __forceinline__ T arrival_fast(const MedParams& M, const GeoT<T>& g, T S, T rho2, T Teh, T Tel, T Tah, T Tal,
                                          float fb_abs, float fb_rel_v, T qv, float q_extra, T& uf_out) {
  static_assert(KIND == C8R_UNIFORM || KIND == C8R_EXPONENTIAL, "plain straight-line media only");
  constexpr float u = 5.9604644775390625e-8f;  // 2^-24
  // R' = sqrt(S) rounded once (the direct form), or the unrefined R0 (the
  // split form, whose x is small: R enters it only through its denominator)
  T R = g.R0;
  if constexpr (AF == kFormDirect) R = fma_rn(fma_rn(neg(g.R0), g.R0, S), mul_rn(bc<T>(0.5f), g.y), g.R0);
  // x = R - w, w = z_e - z_a = -s_z
  const T sz = g.s[2];
  T x;
  float kR = AF == kFormAxis ? 0.375f : 2.5f;
  if constexpr (AF == kFormAxis) {
    const T a0 = bc<T>(M.ax[0]), a1 = bc<T>(M.ax[1]), a2 = bc<T>(M.ax[2]);
    const T cx = fma_rn(g.s[1], a2, neg(mul_rn(sz, a1))), cy = fma_rn(sz, a0, neg(mul_rn(g.s[0], a2))),
            cz = fma_rn(g.s[0], a1, neg(mul_rn(g.s[1], a0)));
    const T w = axis_w(M, g);
    x = div_ap(fma_rn(cx, cx, fma_rn(cy, cy, mul_rn(cz, cz))), add_rn(R, w));
    kR = __fmaf_rn(q_extra, 0.0625f, kR);
    if constexpr (!kUsualForm<T>)
      if (!(w >= 0.0f)) {
        x = __fsub_rn(R, w);
        kR = 10.0f;
      }
  } else if constexpr (AF == kFormSplit) {
    x = div_ap(rho2, sub_rn(R, sz));
    if constexpr (!kUsualForm<T>) x = sz < 0.0f ? x : __fadd_rn(R, sz);
  } else {
    x = add_rn(R, sz);
  }
  const float kh = KIND == C8R_UNIFORM ? M.s_h : M.kc_h;
  const T q = mul_rn(x, bc<T>(kh));
  const T Td = add_rn(sub_rn(Teh, Tah), sub_rn(Tel, Tal));
  T v = bc<T>(0.0f);
  if constexpr (KIND == C8R_EXPONENTIAL) v = mul_rn(mul_rn(qv, R), bc<T>(M.cN_h));
  const T uf = add_rn(add_rn(Td, q), v);
  uf_out = uf;
  const T tail = fma_rn(bc<T>(2.25f * u), abs_of(Td),
                        fma_rn(bc<T>(__fmaf_rn(AF == kFormDirect ? 17.0f : 22.0f, u, fb_rel_v)), abs_of(v),
                               fma_rn(bc<T>(3.25f * u), abs_of(uf), bc<T>(fb_abs))));
  if constexpr (AF == kFormSplit) {
    return fma_rn(bc<T>(__fmaf_rn(q_extra, u, 19.0f * u)), q, tail);
  } else {
    const float cq = AF == kFormAxis ? __fmaf_rn(q_extra, 8.0f * u, 72.0f * u) : __fmaf_rn(q_extra, u, 6.25f * u);
    return fma_rn(bc<T>(cq), q, fma_rn(bc<T>(__fmul_rn(kR * u, kh)), R, tail));
  }
}

// The bin that an FP32 arrival uf, off by at most eps, decides: uf - eps and uf +
// eps (rounded; the one u |uf| that the bound keeps for it) must fall in one bin
// of the window, or both before or both after it.  Their floors come from a
// downward-rounded addition of 1.5 x 2^23, whose low bits then hold them: exact
// below 2^22, and above or below that range the sum still sorts after or before
// the window (as it does for an infinity; a NaN sorts after it, and deposits
// nothing in the float-float form either).  Windows of more than 2^22 bins take
// floorf (XU-pipe operations, as the conversion to an integer is).
constexpr int kMagicBinBits = 0x4B400000;  // 1.5 x 2^23
constexpr int kMagicBins = 1 << 22;
__device__ __forceinline__ int decide_bin(int lo, int hi, int n_bins) {
  const int k = lo == hi ? lo - kMagicBinBits : kFastUndecided;
  return (hi < kMagicBinBits || lo >= kMagicBinBits + n_bins) ? kFastOut : k;
}
__device__ __forceinline__ int decide_bin_wide(float uf, float eps, int n_bins) {
  if (uf < -eps || __fsub_rn(uf, eps) >= (float)n_bins) return kFastOut;
  const float k = floorf(uf);
  const float fr = __fsub_rn(uf, k);
  if (!(fr > eps && fr < __fsub_rn(1.0f, eps))) return kFastUndecided;  // also NaN
  return (int)k;
}
// the bins of a pair's two endpoints
__device__ __forceinline__ void decide_bins(float2 uf, float2 eps, int n_bins, int& ka, int& kb) {
  if (n_bins <= kMagicBins) {
    const float2 magic = make_float2(12582912.0f, 12582912.0f);
    const float2 lo = __fadd2_rd(sub_rn(uf, eps), magic), hi = __fadd2_rd(add_rn(uf, eps), magic);
    ka = decide_bin(__float_as_int(lo.x), __float_as_int(hi.x), n_bins);
    kb = decide_bin(__float_as_int(lo.y), __float_as_int(hi.y), n_bins);
  } else {
    ka = decide_bin_wide(uf.x, eps.x, n_bins);
    kb = decide_bin_wide(uf.y, eps.y, n_bins);
  }
}

// distance k + 1 - u from a float-float arrival u in bin k to the bin's upper
// edge, formed from the arrival rather than as 1 - frac: just below an edge the
// fraction is close to 1, where FP32 is spaced by 6e-8, while the distance is
// small and keeps its relative precision ((k + 1) - u_h is exact there).  The
// first bin of a narrow ZHS interval straddling an edge takes this share.
__device__ __forceinline__ float gap_to_next_edge(ff u, int k) {
  return __fsub_rn(__fsub_rn((float)(k + 1), u.h), u.l);
}

// The bins and fractions of two float-float arrivals as bin_raw has them: floors
// from rounded-down sums as in decide_bins, of the high part and then of the
// fraction with the low part.  Beyond 2^22 the first sum's spacing is 2, and the
// second floor takes what is left.  The index comes from the sums' low bits for
// windows of at most kMagicBins / 2 bins, by conversion for longer ones (XU pipe).
// Arrivals outside the window give any index outside it.
__device__ __forceinline__ void bins_of(ffT<float2> u, int n_bins, int& kx, int& ky, float2& kf, float2& frac) {
  const float2 magic = make_float2(12582912.0f, 12582912.0f);
  // a margin for the low part, as in bin_raw (fmaxf and fminf drop a NaN, to
  // outside); far outside, where the low part can be any size, it is dropped
  const float top = (float)n_bins + 128.0f;
  const float2 h = make_float2(fminf(fmaxf(u.h.x, -128.0f), top), fminf(fmaxf(u.h.y, -128.0f), top));
  const float2 l = make_float2(h.x == u.h.x ? u.l.x : 0.0f, h.y == u.h.y ? u.l.y : 0.0f);
  const float2 t = __fadd2_rd(h, magic);
  const float2 k0 = sub_rn(t, magic);
  const float2 f = add_rn(sub_rn(h, k0), l);
  const float2 t1 = __fadd2_rd(f, magic);
  const float2 df = sub_rn(t1, magic);
  kf = add_rn(k0, df);
  frac = sub_rn(f, df);
  if (n_bins <= kMagicBins / 2) {
    constexpr unsigned two = 2u * (unsigned)kMagicBinBits;
    kx = (int)(__float_as_uint(t.x) + __float_as_uint(t1.x) - two);
    ky = (int)(__float_as_uint(t.y) + __float_as_uint(t1.y) - two);
  } else {
    kx = __float2int_rn(kf.x);
    ky = __float2int_rn(kf.y);
  }
}

// field part at one emission point (FP32): w = d x beta, V = (d x w)/R^2 =
// rhat x (rhat x beta), D = 1 - n beta.rhat in a cancellation-free form:
//   D = (1 - n|beta|) + n |w|^2 / (R (|beta| R + beta.d))   when beta.d >= 0
// (the second term is n|beta|(1 - cos theta)); the direct form otherwise.
template <typename T>
struct FieldT {
  T V[3];  // rhat x (rhat x beta) times R^2  (i.e. d x w)
  T D;
  T invR;
  T bd;    // beta . d
  T w[3];  // d x beta
};
using FieldM = FieldT<float>;
// Every step uses explicit-rounding intrinsics so the forward and the adjoint
// kernels, which inline this in different contexts, take identical branch
// decisions.
// FUSED: D's last product and sum as one operation (pairs only), see mul_apart and
// OpsMixed::kFusedD.
template <typename T, bool FUSED = false>
__device__ __forceinline__ void field_mixed(const GeoT<T>& g, T bx, T by, T bz, T bmag, T om_nb, T n, FieldT<T>& f) {
  const T sx = g.s[0], sy = g.s[1], sz = g.s[2];
  // w = d x beta from the FP32 part of d (the low parts, ~2^-24 |d|, change D by
  // ~1e-7 relative even near the Cherenkov angle, below the FP32 field arithmetic)
  const T wx = fma_rn(sy, bz, neg(mul_rn(sz, by)));
  const T wy = fma_rn(sz, bx, neg(mul_rn(sx, bz)));
  const T wz = fma_rn(sx, by, neg(mul_rn(sy, bx)));
  const T bd = fma_rn(bx, sx, fma_rn(by, sy, mul_rn(bz, sz)));
  const T R = g.R0;
  const T invR = g.y;
  const T w2 = fma_rn(wx, wx, fma_rn(wy, wy, mul_rn(wz, wz)));
  const T den = mul_rn(R, fma_rn(bmag, R, bd));
  if constexpr (FUSED)
    f.D = fma_rn(mul_rn(n, w2), rcp_ap(den), om_nb);
  else
    f.D = add_rn(om_nb, mul_apart(mul_rn(n, w2), rcp_ap(den)));
  if constexpr (!kUsualForm<T>)
    if (!(bd >= 0.0f)) f.D = __fsub_rn(1.0f, __fmul_rn(__fmul_rn(n, bd), invR));
  // d x w = d (d.beta) - beta R^2  ->  V R^2
  f.V[0] = fma_rn(sy, wz, neg(mul_rn(sz, wy)));
  f.V[1] = fma_rn(sz, wx, neg(mul_rn(sx, wz)));
  f.V[2] = fma_rn(sx, wy, neg(mul_rn(sy, wx)));
  f.invR = invR;
  f.bd = bd;
  f.w[0] = wx;
  f.w[1] = wy;
  f.w[2] = wz;
}

// one half of a pair's geometry or field
template <int J>
__device__ __forceinline__ float half_of(float2 a) { return J == 0 ? a.x : a.y; }
template <int J>
__device__ __forceinline__ GeoM half_of(const GeoT<float2>& g) {
  GeoM r;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    r.s[c] = half_of<J>(g.s[c]);
    r.e[c] = half_of<J>(g.e[c]);
  }
  r.R0 = half_of<J>(g.R0);
  r.R1 = half_of<J>(g.R1);
  r.y = half_of<J>(g.y);
  return r;
}
template <int J>
__device__ __forceinline__ FieldM half_of(const FieldT<float2>& f) {
  FieldM r;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    r.V[c] = half_of<J>(f.V[c]);
    r.w[c] = half_of<J>(f.w[c]);
  }
  r.D = half_of<J>(f.D);
  r.invR = half_of<J>(f.invR);
  r.bd = half_of<J>(f.bd);
  return r;
}

// D = 1 - n (beta . d)/R in float-float, for a refined geometry (R = R0 + R1)
// and n - 1 given directly.  Its absolute error (~1e-10, set by n - 1 in FP32)
// is what the arrival interval ends u_m -/+ |D| (t1 - t0)/(2 dt) need: the
// half-width reaches ~10^2 bins, so D must be good to ~1e-9 absolute, which the
// FP32 form of field_mixed (good to ~1e-7 relative) is not for |D| of order 1.
// (p2 + q2 = b_z s_z exactly and bze = fl(b_z e_z) given)
template <typename T>
__device__ __forceinline__ ffT<T> doppler_ff(const GeoT<T>& g, T bx, T by, T p2, T q2, T bze, T nm1) {
  // beta . d with d = s + e exact: exact products of the high parts, summed
  // with TwoSum; the low parts and the rounding errors in FP32
  T p0, q0, p1, q1;
  two_prod(bx, g.s[0], p0, q0);
  two_prod(by, g.s[1], p1, q1);
  T S1, E1, S2, E2;
  two_sum(p0, p1, S1, E1);
  two_sum(S1, p2, S2, E2);
  const T be = fma_rn(bx, g.e[0], fma_rn(by, g.e[1], bze));
  const T lo = add_rn(add_rn(add_rn(q0, q1), add_rn(q2, E1)), add_rn(E2, be));
  // q = (beta . d)/R: FP32 quotient, then one correction from the exact residual
  const T qh = mul_rn(S2, g.y);
  T ph, pl;
  two_prod(qh, g.R0, ph, pl);
  const T r = sub_rn(add_rn(sub_rn(sub_rn(S2, ph), pl), lo), mul_rn(qh, g.R1));
  const T ql = mul_rn(r, g.y);
  // n q = q + (n - 1) q, then D = 1 - n q
  T nh, nl;
  two_diff(qh, mul_rn(neg(nm1), qh), nh, nl);
  nl = add_rn(nl, ql);
  T dh, dl;
  two_sum(bc<T>(1.0f), neg(nh), dh, dl);
  dl = sub_rn(dl, nl);
  // renormalise, so that the sign of D is the sign of D.h (near D = 0 the high
  // part alone can be 0 or of the other sign)
  ffT<T> D;
  D.h = add_rn(dh, dl);
  D.l = sub_rn(dl, sub_rn(D.h, dh));
  return D;
}
template <typename T>
__device__ __forceinline__ ffT<T> doppler_ff(const GeoT<T>& g, T bx, T by, T bz, T nm1) {
  T p2, q2;
  two_prod(bz, g.s[2], p2, q2);
  return doppler_ff(g, bx, by, p2, q2, mul_rn(bz, g.e[2]), nm1);
}
template <typename T>
__device__ __forceinline__ ffT<T> doppler_ff(const GeoT<T>& g, T bx, T by, const ZPartT<T>& z, T nm1) {
  return doppler_ff(g, bx, by, z.bh, z.bl, z.be, nm1);
}

// the same field quantities at the midpoint of a track, from those of its two
// endpoints: d_m = (d0 + d1)/2 exactly (float-float), and w = d x beta and
// beta.d are linear in d, so w_m = (w0 + w1)/2, (beta.d)_m = (bd0 + bd1)/2
__device__ __forceinline__ void midpoint_from_endpoints(const GeoM& g0, const GeoM& g1, const FieldM& f0,
                                                        const FieldM& f1, float bmag, float om_nb, float n, GeoM& gm,
                                                        FieldM& fmid) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float S, E;
    two_sum(g0.s[c], g1.s[c], S, E);
    gm.s[c] = 0.5f * S;
    gm.e[c] = 0.5f * __fadd_rn(E, __fadd_rn(g0.e[c], g1.e[c]));
    fmid.w[c] = 0.5f * __fadd_rn(f0.w[c], f1.w[c]);
  }
  const float S2 = __fmaf_rn(gm.s[0], gm.s[0], __fmaf_rn(gm.s[1], gm.s[1], __fmul_rn(gm.s[2], gm.s[2])));
  gm.y = rsqrt_ap(S2);
  gm.R0 = __fmul_rn(S2, gm.y);
  gm.R1 = 0.0f;
  const float bd = 0.5f * __fadd_rn(f0.bd, f1.bd);
  const float wx = fmid.w[0], wy = fmid.w[1], wz = fmid.w[2];
  const float sx = gm.s[0], sy = gm.s[1], sz = gm.s[2];
  if (bd >= 0.0f) {
    const float w2 = __fmaf_rn(wx, wx, __fmaf_rn(wy, wy, __fmul_rn(wz, wz)));
    const float den = __fmul_rn(gm.R0, __fmaf_rn(bmag, gm.R0, bd));
    fmid.D = __fadd_rn(om_nb, div_ap(__fmul_rn(n, w2), den));
  } else {
    fmid.D = __fsub_rn(1.0f, __fmul_rn(__fmul_rn(n, bd), gm.y));
  }
  fmid.V[0] = __fmaf_rn(sy, wz, -__fmul_rn(sz, wy));
  fmid.V[1] = __fmaf_rn(sz, wx, -__fmul_rn(sx, wz));
  fmid.V[2] = __fmaf_rn(sx, wy, -__fmul_rn(sy, wx));
  fmid.invR = gm.y;
  fmid.bd = bd;
}

}  // namespace c8r
