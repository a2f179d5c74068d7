// kernels_mixed.cu -- instantiation of the mixed-precision forward,
// arrival-listing and adjoint kernels (FP32 field arithmetic, float-float
// arrival times).
#include <cooperative_groups.h>

#include "pair_mixed.cuh"

namespace c8r {

cudaError_t launch_forward_mixed(int formalism, bool lin, const void* tiles, int64_t n_tiles, const AntRec* ants,
                                 int n_ant, const MedParams& M, void* acc, const FwdShape& shape, int sm_count,
                                 int* err, cudaStream_t st) {
  if (lin) return launch_forward_mixed_lin(formalism, tiles, n_tiles, ants, n_ant, M, acc, shape, sm_count, err, st);
  return forward_mixed<false>(formalism, tiles, n_tiles, ants, n_ant, M, acc, shape, sm_count, err, st);
}

// accumulator [n_ant][n_bins] float4 -> traces [n_ant][3][n_bins] (added or
// stored); `replicas` copies of the accumulator, `stride` elements apart, are
// summed, and zeroed if `clear`.  Bound by DRAM for large arrays and by the
// latency of its loads otherwise, so a thread has kFetchE bins (a block apart,
// coalesced) in flight.
constexpr int kFetchT = 256;
constexpr int kFetchE = 4;
__global__ void __launch_bounds__(kFetchT) k_acc_to_traces_f32(float4* acc, int64_t n_ant_bins, int n_bins, float* out,
                                                               bool add, bool clear, int replicas, int64_t stride) {
  const int64_t i0 = (int64_t)blockIdx.x * (kFetchT * kFetchE) + threadIdx.x;
  const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  float4 v[kFetchE];
#pragma unroll
  for (int e = 0; e < kFetchE; ++e) v[e] = zero;
#pragma unroll 2
  for (int r = 0; r < replicas; ++r) {
#pragma unroll
    for (int e = 0; e < kFetchE; ++e) {
      const int64_t i = i0 + e * kFetchT;
      if (i < n_ant_bins) {
        const float4 u = acc[i + r * stride];
        v[e].x += u.x;
        v[e].y += u.y;
        v[e].z += u.z;
      }
    }
  }
  if (clear)
    for (int r = 0; r < replicas; ++r)
#pragma unroll
      for (int e = 0; e < kFetchE; ++e)
        if (i0 + e * kFetchT < n_ant_bins) acc[i0 + e * kFetchT + r * stride] = zero;
  float* o[kFetchE];
  float4 w[kFetchE];
#pragma unroll
  for (int e = 0; e < kFetchE; ++e) {
    const int64_t i = i0 + e * kFetchT;
    const int64_t a = i / n_bins;
    o[e] = out + a * 3 * n_bins + (i - a * n_bins);
    w[e] = zero;
    if (add && i < n_ant_bins) w[e] = make_float4(o[e][0], o[e][n_bins], o[e][2 * (int64_t)n_bins], 0.0f);
  }
#pragma unroll
  for (int e = 0; e < kFetchE; ++e)
    if (i0 + e * kFetchT < n_ant_bins) {
      o[e][0] = w[e].x + v[e].x;
      o[e][n_bins] = w[e].y + v[e].y;
      o[e][2 * (int64_t)n_bins] = w[e].z + v[e].z;
    }
}

constexpr int kScanT = 256;         // threads of the float-float scans
constexpr int kScanE = 8;           // consecutive bins per thread and chunk

__device__ __forceinline__ ff ff_sum(ff a, ff b) {
  float s, e;
  two_sum(a.h, b.h, s, e);
  e = __fadd_rn(e, __fadd_rn(a.l, b.l));
  ff r;
  fast_two_sum(s, e, r.h, r.l);
  return r;
}
__device__ __forceinline__ ff ff_add_f(ff a, float b) {
  float s, e;
  two_sum(a.h, b, s, e);
  e = __fadd_rn(e, a.l);
  ff r;
  fast_two_sum(s, e, r.h, r.l);
  return r;
}

// exclusive prefix over the CTA (kScanT threads, all of them calling) of each
// thread's three float-float values v[], in excl[], and the CTA total, in
// tot[]: warp shuffles, then the totals of the warps before (warp_tot is
// written and read here; the caller synchronises before reusing it)
__device__ __forceinline__ void cta_exclusive_scan_ff3(const ff v[3], ff excl[3], ff tot[3],
                                                       ff (*warp_tot)[kScanT / 32]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  ff inc[3] = {v[0], v[1], v[2]};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const ff u{__shfl_up_sync(0xffffffffu, inc[c].h, d), __shfl_up_sync(0xffffffffu, inc[c].l, d)};
      if (lane >= d) inc[c] = ff_sum(inc[c], u);
    }
    if (lane == 31) warp_tot[c][wid] = inc[c];
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    ff before{0.0f, 0.0f};
    tot[c] = ff{0.0f, 0.0f};
#pragma unroll
    for (int w = 0; w < kScanT / 32; ++w) {
      const ff t = warp_tot[c][w];
      if (w < wid) before = ff_sum(before, t);
      tot[c] = ff_sum(tot[c], t);
    }
    ff lanes{__shfl_up_sync(0xffffffffu, inc[c].h, 1), __shfl_up_sync(0xffffffffu, inc[c].l, 1)};
    if (lane == 0) lanes = ff{0.0f, 0.0f};
    excl[c] = ff_sum(before, lanes);
  }
}

// accumulator and box edges, rows of n_bins elements `row` apart -> traces:
// out[k] = direct[k] + sum_{j <= k} edge[j], each summed over the `replicas`
// copies of the accumulator (`stride` elements apart; zeroed if `clear`).  A
// cluster of up to kFetchCluster CTAs has an antenna, each CTA kScanT x kFetchBins
// consecutive bins and each thread kFetchBins of them, read once: the thread's
// total of the edges, an exclusive scan over the CTA, the totals of the CTAs
// before through distributed shared memory, then the running sum over the
// thread's bins.  Longer windows take several rounds with a carry.  All sums in
// float-float on the FP32 pipe (~2^-44 relative after 2^24 bins, far below the
// FP32 output; FP64 runs at 1/64 of the FP32 rate on this part).  Bound by the
// latency of its loads on small arrays.  Against one CTA per antenna that read
// each bin twice: 4096 bins, 8 antennas with 8 copies 76 us, now 29 with 16;
// 160 antennas with 2 copies 45 us, now 30 with 4; 512 antennas 58 -> 43 us; 1024
// antennas x 8192 bins 200 -> 164 us.
constexpr int kFetchBins = 4;
constexpr int kFetchCluster = 8;
static_assert(kScanT / 32 == 8 && kFetchCluster == 8, "sum_before8 takes eight totals");

// the running sums of the fetch: float-float for the mixed path (on the FP32
// pipe; FP64 runs at 1/64 of its rate here), FP64 for the FP64 path
__device__ __forceinline__ double ff_sum(double a, double b) { return a + b; }
__device__ __forceinline__ double ff_add_f(double a, double b) { return a + b; }
__device__ __forceinline__ float rounded(ff a) { return __fadd_rn(a.h, a.l); }
__device__ __forceinline__ double rounded(double a) { return a; }
__device__ __forceinline__ ff from_lane(ff a, int l) {
  return ff{__shfl_sync(0xffffffffu, a.h, l), __shfl_sync(0xffffffffu, a.l, l)};
}
__device__ __forceinline__ double from_lane(double a, int l) { return __shfl_sync(0xffffffffu, a, l); }
template <typename T>
struct SumOf;
template <>
struct SumOf<float> {
  using type = ff;
};
template <>
struct SumOf<double> {
  using type = double;
};

// From eight totals of three components (t[c][q]), the sum of the first `n`
// (before) and of all (tot), in every lane of the warp: lane 8c + q takes one
// total and three shuffles add them
template <class S>
__device__ __forceinline__ void sum_before8(const S (*t)[8], int n, S before[3], S tot[3]) {
  const int lane = threadIdx.x & 31, q = lane & 7;
  S all = lane < 24 ? t[lane >> 3][q] : S{};
  S pre = q < n ? all : S{};
#pragma unroll
  for (int d = 1; d < 8; d <<= 1) {
    all = ff_sum(all, from_lane(all, lane ^ d));
    pre = ff_sum(pre, from_lane(pre, lane ^ d));
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    before[c] = from_lane(pre, 8 * c);
    tot[c] = from_lane(all, 8 * c);
  }
}

template <typename T>
__global__ void __launch_bounds__(kScanT) k_acc_scan_to_traces(typename AccOf<T>::type* acc,
                                                               typename AccOf<T>::type* edges, int64_t row, int n_bins,
                                                               T* out, bool add, bool clear, int replicas,
                                                               int64_t stride) {
  namespace cg = cooperative_groups;
  using S = typename SumOf<T>::type;
  using acc4 = typename AccOf<T>::type;
  const cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), n_cta = (int)cluster.num_blocks();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __shared__ S warp_tot[3][kScanT / 32];
  __shared__ S cta_tot[2][3][kFetchCluster];  // the cluster's totals, of this round and the next
  if (threadIdx.x < 6 * kFetchCluster) cta_tot[0][0][threadIdx.x] = S{};  // absent CTAs count as zero
  cluster.sync();
  const int a = blockIdx.x / n_cta;
  acc4* direct = acc + a * row;
  acc4* edge = edges + a * row;
  T* o = out + (size_t)a * 3 * n_bins;
  S carry[3] = {S{}, S{}, S{}};
  int buf = 0;
  for (int64_t base = 0; base < n_bins; base += (int64_t)n_cta * kScanT * kFetchBins, buf ^= 1) {
    const int64_t k0 = base + ((int64_t)rank * kScanT + threadIdx.x) * kFetchBins;
    S e[kFetchBins][3], d[kFetchBins][3];
#pragma unroll
    for (int b = 0; b < kFetchBins; ++b)
#pragma unroll
      for (int c = 0; c < 3; ++c) e[b][c] = d[b][c] = S{};
#pragma unroll 2
    for (int r = 0; r < replicas; ++r) {
#pragma unroll
      for (int b = 0; b < kFetchBins; ++b) {
        if (k0 + b >= n_bins) continue;
        const int64_t i = k0 + b + r * stride;
        const acc4 u = direct[i], w = edge[i];
        d[b][0] = ff_add_f(d[b][0], u.x);
        d[b][1] = ff_add_f(d[b][1], u.y);
        d[b][2] = ff_add_f(d[b][2], u.z);
        e[b][0] = ff_add_f(e[b][0], w.x);
        e[b][1] = ff_add_f(e[b][1], w.y);
        e[b][2] = ff_add_f(e[b][2], w.z);
      }
    }
    if (clear) {
      const acc4 zero{T(0), T(0), T(0), T(0)};
      for (int r = 0; r < replicas; ++r)
#pragma unroll
        for (int b = 0; b < kFetchBins; ++b)
          if (k0 + b < n_bins) direct[k0 + b + r * stride] = edge[k0 + b + r * stride] = zero;
    }
    // the edges before this thread's bins: of the lanes before it, of the warps
    // before its own, and of the CTAs before its own
    S lanes[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      S inc = e[0][c];
#pragma unroll
      for (int b = 1; b < kFetchBins; ++b) inc = ff_sum(inc, e[b][c]);
#pragma unroll
      for (int s = 1; s < 32; s <<= 1) {
        const S u = from_lane(inc, lane >= s ? lane - s : lane);
        if (lane >= s) inc = ff_sum(inc, u);
      }
      if (lane == 31) warp_tot[c][wid] = inc;
      lanes[c] = from_lane(inc, lane > 0 ? lane - 1 : 0);
      if (lane == 0) lanes[c] = S{};
    }
    __syncthreads();
    S run[3], tot[3];
    sum_before8(warp_tot, wid, run, tot);
#pragma unroll
    for (int c = 0; c < 3; ++c) run[c] = ff_sum(run[c], lanes[c]);
    if (n_cta > 1) {
      // every CTA's totals to every CTA; two buffers, so that a round's totals
      // are not overwritten before the slowest CTA has read them
      if (threadIdx.x < n_cta) {
        S(*peer)[3][kFetchCluster] = cluster.map_shared_rank(cta_tot, threadIdx.x);
#pragma unroll
        for (int c = 0; c < 3; ++c) peer[buf][c][rank] = tot[c];
      }
      cluster.sync();
      S before[3];
      sum_before8(cta_tot[buf], rank, before, tot);
#pragma unroll
      for (int c = 0; c < 3; ++c) run[c] = ff_sum(before[c], run[c]);
    } else {
      __syncthreads();  // warp_tot is rewritten by the next round
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      run[c] = ff_sum(carry[c], run[c]);
      carry[c] = ff_sum(carry[c], tot[c]);
    }
#pragma unroll
    for (int b = 0; b < kFetchBins; ++b) {
      if (k0 + b >= n_bins) continue;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        run[c] = ff_sum(run[c], e[b][c]);
        const T x = rounded(ff_sum(run[c], d[b][c]));
        T* q = o + (size_t)c * n_bins + k0 + b;
        *q = add ? *q + x : x;
      }
    }
  }
}

__global__ void k_acc_to_traces_f64(Acc4D* acc, int64_t n_ant_bins, int n_bins, double* out, bool clear,
                                    int replicas) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_ant_bins) return;
  const int64_t a = i / n_bins;
  const int k = (int)(i - a * n_bins);
  Acc4D v = acc[i];
  for (int r = 1; r < replicas; ++r) {
    const Acc4D w = acc[i + r * n_ant_bins];
    v.x += w.x;
    v.y += w.y;
    v.z += w.z;
  }
  if (clear)
    for (int r = 0; r < replicas; ++r) acc[i + r * n_ant_bins] = Acc4D{0.0, 0.0, 0.0, 0.0};
  double* o = out + a * 3 * n_bins + k;
  o[0] = v.x;
  o[n_bins] = v.y;
  o[2 * n_bins] = v.z;
}

cudaError_t launch_acc_to_traces(int precision, void* acc, int n_ant, int n_bins, int rows, void* out, bool add,
                                 bool clear, cudaStream_t st, int replicas, void* edges) {
  const int64_t n = (int64_t)n_ant * n_bins;
  if (n <= 0) return cudaSuccess;
  const int64_t stride = n * rows;  // accumulator elements per copy
  if (rows == 2 || edges) {
    // a cluster of CTAs per antenna, as many as one round over the window needs
    int n_cta = 1;
    while (n_cta < kFetchCluster && n_cta * kScanT * kFetchBins < n_bins) n_cta *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_ant * n_cta);
    cfg.blockDim = dim3(kScanT);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = n_cta;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const int64_t row = (int64_t)n_bins * rows;
    if (precision == C8R_FP64)
      return cudaLaunchKernelEx(&cfg, k_acc_scan_to_traces<double>, static_cast<Acc4D*>(acc),
                                static_cast<Acc4D*>(edges), row, n_bins, static_cast<double*>(out), add, clear,
                                replicas, stride);
    return cudaLaunchKernelEx(&cfg, k_acc_scan_to_traces<float>, static_cast<float4*>(acc),
                              static_cast<float4*>(acc) + n_bins, row, n_bins, static_cast<float*>(out), add, clear,
                              replicas, stride);
  }
  if (precision == C8R_FP64) {
    k_acc_to_traces_f64<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(static_cast<Acc4D*>(acc), n, n_bins,
                                                                    static_cast<double*>(out), clear, replicas);
  } else {
    constexpr int per = kFetchT * kFetchE;
    k_acc_to_traces_f32<<<(unsigned)((n + per - 1) / per), kFetchT, 0, st>>>(
        static_cast<float4*>(acc), n, n_bins, static_cast<float*>(out), add, clear, replicas, stride);
  }
  return cudaGetLastError();
}

// traces [n_ant][3][n_bins] (float or double) -> bin-major [n_ant][n_bins] of
// (x, y, z, 0), the layout the adjoint gathers one bin of from
template <typename T, typename T4>
__global__ void k_traces_to_bin_major(const T* g, int64_t n_ant_bins, int n_bins, T4* out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_ant_bins) return;
  const int64_t a = i / n_bins;
  const int k = (int)(i - a * n_bins);
  const T* s = g + a * 3 * n_bins + k;
  T4 v;
  v.x = s[0];
  v.y = s[n_bins];
  v.z = s[2 * (size_t)n_bins];
  v.w = T(0);
  out[i] = v;
}

cudaError_t launch_traces_to_bin_major(int precision, const void* g, int n_ant, int n_bins, void* out,
                                       cudaStream_t st) {
  const int64_t n = (int64_t)n_ant * n_bins;
  if (n <= 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((n + 255) / 256);
  if (precision == C8R_FP64)
    k_traces_to_bin_major<double, Acc4D><<<blocks, 256, 0, st>>>(static_cast<const double*>(g), n, n_bins,
                                                                 static_cast<Acc4D*>(out));
  else
    k_traces_to_bin_major<float, float4><<<blocks, 256, 0, st>>>(static_cast<const float*>(g), n, n_bins,
                                                                 static_cast<float4*>(out));
  return cudaGetLastError();
}

// running sums over the bins of a bin-major gradient, stored as float-float:
// out[a][k] = sum_{j < k} g[a][j], k = 0 .. n_bins (one CTA per antenna), laid
// out like the trace scan (kScanE consecutive bins per thread, a CTA-wide
// exclusive scan of the threads' totals, a carry over chunks), in float-float
// on the FP32 pipe: after k additions a sum is off by at most ~2k u^2 of the
// largest partial sum (u = 2^-24), ~1e-11 of it at 2048 bins, against the
// adjoint's need of ~1e-7 of the sums it forms from two of them
__device__ __forceinline__ PrefixFF prefix_ff(const ff s[3]) {
  PrefixFF p;
  p.hx = s[0].h;
  p.hy = s[1].h;
  p.hz = s[2].h;
  p.lx = s[0].l;
  p.ly = s[1].l;
  p.lz = s[2].l;
  p.hpad = p.lpad = 0.0f;
  return p;
}
__global__ void __launch_bounds__(kScanT) k_bin_running_sums(const float4* g, int n_bins, PrefixFF* out) {
  __shared__ ff warp_tot[3][kScanT / 32];
  const int a = blockIdx.x;
  const float4* row = g + (size_t)a * n_bins;
  PrefixFF* o = out + (size_t)a * (n_bins + 1);
  ff carry[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
  if (threadIdx.x == 0) o[0] = prefix_ff(carry);
  for (int base = 0; base < n_bins; base += kScanT * kScanE) {
    const int k0 = base + threadIdx.x * kScanE;
    const int k1 = min(k0 + kScanE, n_bins);
    ff v[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
    for (int k = k0; k < k1; ++k) {
      const float4 e = row[k];
      v[0] = ff_add_f(v[0], e.x);
      v[1] = ff_add_f(v[1], e.y);
      v[2] = ff_add_f(v[2], e.z);
    }
    ff excl[3], tot[3], run[3];
    cta_exclusive_scan_ff3(v, excl, tot, warp_tot);
#pragma unroll
    for (int c = 0; c < 3; ++c) run[c] = ff_sum(carry[c], excl[c]);
    for (int k = k0; k < k1; ++k) {
      const float4 e = row[k];
      run[0] = ff_add_f(run[0], e.x);
      run[1] = ff_add_f(run[1], e.y);
      run[2] = ff_add_f(run[2], e.z);
      o[k + 1] = prefix_ff(run);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) carry[c] = ff_sum(carry[c], tot[c]);
    __syncthreads();  // warp_tot is rewritten by the next chunk
  }
}

cudaError_t launch_bin_running_sums(const void* g, int n_ant, int n_bins, PrefixFF* out, cudaStream_t st) {
  if (n_ant <= 0 || n_bins <= 0) return cudaSuccess;
  k_bin_running_sums<<<(unsigned)n_ant, kScanT, 0, st>>>(static_cast<const float4*>(g), n_bins, out);
  return cudaGetLastError();
}

cudaError_t launch_arrivals_mixed(int formalism, const void* tiles, int64_t n, const AntRec* ants, int n_ant,
                                  const MedParams& M, int32_t* branch, int32_t* bin, float* frac, cudaStream_t st) {
  const unsigned blocks = (unsigned)((n * (int64_t)n_ant + 255) / 256);
  auto go = [&](auto ops) {
    k_arrivals<decltype(ops)><<<blocks, 256, 0, st>>>(tiles, n, ants, n_ant, M, branch, bin, frac);
    return cudaGetLastError();
  };
  // the kernels of forward_mixed
  if (formalism == C8R_ENDPOINT) {
    if (M.kind == C8R_EXPONENTIAL_RAY) return go(OpsMixed<C8R_ENDPOINT, C8R_EXPONENTIAL_RAY>{});
    if (M.kind == C8R_EXPONENTIAL_SPHERICAL) return go(OpsMixed<C8R_ENDPOINT, C8R_EXPONENTIAL_SPHERICAL>{});
    return with_endpoint_ops(M, go);
  }
  if (M.flat) {
    if (M.kind == C8R_EXPONENTIAL_RAY)
      return go(OpsMixed<C8R_ZHS, C8R_EXPONENTIAL_RAY, false, kFormDirect, true>{});
    if (M.kind == C8R_EXPONENTIAL_SPHERICAL)
      return go(OpsMixed<C8R_ZHS, C8R_EXPONENTIAL_SPHERICAL, false, kFormDirect, true>{});
    return go(OpsMixed<C8R_ZHS, C8R_EXPONENTIAL, false, kFormDirect, true>{});
  }
  if (M.kind == C8R_EXPONENTIAL_RAY) return go(OpsMixed<C8R_ZHS, C8R_EXPONENTIAL_RAY>{});
  if (M.kind == C8R_EXPONENTIAL_SPHERICAL) return go(OpsMixed<C8R_ZHS, C8R_EXPONENTIAL_SPHERICAL>{});
  return M.kind == C8R_EXPONENTIAL ? go(OpsMixed<C8R_ZHS, C8R_EXPONENTIAL>{})
                                   : go(OpsMixed<C8R_ZHS, C8R_UNIFORM>{});
}

cudaError_t launch_backward_mixed(int formalism, bool lin, BwdArgs& a, const FwdShape& shape, int sm_count,
                                  cudaStream_t st) {
  if (lin) return launch_backward_mixed_lin(formalism, a, shape, sm_count, st);
  return backward_mixed<false>(formalism, a, shape, sm_count, st);
}

}  // namespace c8r
