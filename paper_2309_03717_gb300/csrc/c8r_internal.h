// c8r_internal.h -- host-side declarations shared by the libc8r translation units.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/c8r.h"
#include "c8r_device.cuh"

namespace c8r {

// launch shape of the forward kernels
struct FwdShape {
  int a_tile;  // antennas per CTA: each thread holds one staged track and loops over them
  int waves;   // target number of waves (all CTAs resident at once) per launch
  int replicas = 1;  // copies of the accumulator (acc_replicas)
  int64_t edge_off = 0;  // FP64: accumulator elements from a row to its box edges, 0 without them
};

// SoA track pointers of the caller, already offset to a chunk
struct TrackPtrs {
  int dtype;
  const void* f[12];
};

size_t tile_bytes(int precision);
// bytes of one accumulator element (one bin of one antenna: x, y, z, pad)
inline size_t acc_elem_bytes(int precision) { return precision == C8R_FP64 ? 32 : 16; }
// accumulator rows per antenna, box edges included (ZHS)
inline int acc_rows(int formalism) { return formalism == C8R_ZHS ? 2 : 1; }
// and of the accumulator itself: the FP64 path keeps the edges apart, behind the
// accumulator or in memory of their own, where there is room for them (only the
// one-bin deposit of the plain media has boxes; without the edges they go in bin by
// bin)
inline int acc_rows(int precision, int formalism) { return precision == C8R_MIXED ? acc_rows(formalism) : 1; }
// copies of the accumulator the forward kernel spreads its reductions over (CTA
// range r adds into copy r % replicas; the fetch sums them).  Most reductions go
// into the few bins per antenna that the pulse arrives in, a few lines of L2
// each, and the slices that hold more of those lines become the bottleneck (the
// busiest ran at twice the mean with 4 copies).  4e6 tracks of a vertical shower x
// 160 antennas, Endpoint, ms with 1 / 2 / 4 / 8 / 16 copies: 7.8 / 5.7 / 5.15 /
// 4.71 / 4.74; ZHS, 2e7 tracks, 4 / 8 / 16: 26.5 / 24.7 / 24.8.  A copy costs its
// bytes once to zero and once to read per fetch, so few tracks take few copies.
// Us per push and fetch with 1 / 4 / 16 copies (4096 bins): Endpoint, 8 antennas,
// 1e6 tracks 646 / 224 / 152, 64 antennas 1123 / 752 / 625, 512 antennas x 3e5
// 1303 / 1310 / 1310; ZHS, 8 antennas 576 / 257 / 213; linear deposit, 64 antennas
// 2487 / 1612 / 1242.  With 3e4 tracks, Endpoint, 64 antennas 76 / 61 / 64.
//
// The FP64 path adds at a thirtieth of the mixed path's rate, but with three scalar
// reductions per deposit: hot bins bind it where the antennas are few (a trace's
// copies times its antennas: 64 for ZHS, 32 for Endpoint, where a pair has fewer
// deposits).  Us per push and fetch, 3.5e5 tracks, 1 copy / as chosen: ZHS 1 antenna 525
// / 204, 2 575 / 224, 8 872 / 488, 16 1220 / 871; Endpoint 2 473 / 230, 8 721 / 605, 16
// 1192 / 1138; linear deposit, 1e5 x 2 662 / 235.
//
// the batched launch: its many showers' antenna tiles spread the CTAs, so 2
// copies for ZHS and 1 for Endpoint
inline int acc_replicas(int formalism) { return acc_rows(formalism) == 2 ? 2 : 1; }
// bytes of the accumulator rows in use at a time (forward_grid groups the
// antenna tiles by it) and of all copies.  Above L2's 129 MB: the bins that the
// pulses reach, a small part of the rows, are what has to stay there
constexpr size_t kAccBudget = (size_t)192 << 20;
// the most copies a context uses (its accumulator is allocated for this many):
// one per 22 resident CTAs of an antenna tile (6 CTAs per SM), at most 16 and
// within the budget, as a power of two, and one below 64 CTAs.  That is where the
// measurements above part: 456 CTAs per tile (64 antennas) gain up to 16 copies,
// 182 (160 antennas) up to 8, 57 (512 antennas) none (linear deposit, 1e5 tracks:
// 906 us with 1, 920 with 2)
inline int acc_replicas(int precision, int formalism, int n_ant, int n_bins, int a_tile, int sm_count) {
  const int64_t ant_tiles = (n_ant + a_tile - 1) / a_tile;
  const int64_t per_tile = (int64_t)sm_count * 6 / (ant_tiles > 0 ? ant_tiles : 1);
  int64_t want = per_tile < 64 ? 1 : per_tile / 22;
  if (precision == C8R_FP64) want = (formalism == C8R_ZHS ? 64 : 32) / (n_ant > 0 ? n_ant : 1);
  const size_t one = (size_t)n_ant * n_bins * acc_elem_bytes(precision) * acc_rows(formalism);
  const int64_t fit = (int64_t)(kAccBudget / (one > 0 ? one : 1));
  int r = 1;
  while (r < 16 && r * 2 <= want && r * 2 <= fit) r *= 2;
  return r;
}
// the copies that a push of n tracks uses, of the `most` allocated: two tracks per
// bin, row and copy at least, where the cost of a copy (about 32 bytes per bin,
// row and antenna) falls below what it takes off the reductions of the tracks
// (FP64, whose copies are of few antennas: half a track)
inline int push_replicas(int precision, int most, int64_t n, int n_bins, int rows) {
  const int64_t per_copy = (int64_t)(precision == C8R_FP64 ? 1 : 4) * n_bins * rows;
  int r = 1;
  while (r * 2 <= most && r * per_copy <= n) r *= 2;
  return r;
}
// the copies that every mixed push uses, however few its tracks: the FP32 rounding
// of a bin's sum falls with the copies the sum is split over, most of all in the
// running sum of the ZHS box edges (error against 64 bits, ZHS, 4.4e4 tracks x 31
// antennas, 8192 bins: 1.2e-6 with one copy, 6.5e-7 with four).  One per 100
// CTAs of an antenna tile (Endpoint 200) or part of it, at most 8 and within 48 MB
inline int floor_replicas(int precision, int formalism, int n_ant, int n_bins, int a_tile, int sm_count) {
  if (precision != C8R_MIXED) return 1;
  const int64_t ant_tiles = (n_ant + a_tile - 1) / a_tile;
  const int64_t per_tile = (int64_t)sm_count * (acc_rows(formalism) == 2 ? 7 : 6) / (ant_tiles > 0 ? ant_tiles : 1);
  const int64_t per_copy = acc_rows(formalism) == 2 ? 100 : 200;
  const int64_t want = (per_tile + per_copy - 1) / per_copy;
  const size_t one = (size_t)n_ant * n_bins * acc_elem_bytes(precision) * acc_rows(formalism);
  const int64_t fit = (int64_t)(((size_t)48 << 20) / (one > 0 ? one : 1));
  int r = 1;
  while (r < 8 && r * 2 <= want && r * 2 <= fit) r *= 2;
  return r;
}
// antennas per CTA of a forward launch over n_tiles track tiles, `a_tile` at
// most.  A CTA walks its antennas one after the other, so few CTAs with many
// antennas leave the device waiting for the last of them, and each CTA costs its
// set-up and the per-track preparation once more: the tile is halved until the
// launch has enough CTAs per SM (14; 28 of the ZHS kernels' 64 threads), down to
// 4 antennas (FP64, where a pair takes longest: 2, or 1 below one CTA per SM).
// Measured, us per push with 32 / 16 / 8 / 4 / 2 antennas: Endpoint, 64 antennas x
// 3e4 tracks 55 / 46 / 40 / 40 / 50, 160 x 3e4 69 / 60 / 62 / 75 / 102, 160 x 3e3
// 28 / 24 / 23 / 23 / 24; ZHS, 160 x 3e4 99 / 78 / 75 / 74 / 72; FP64 Endpoint, 16
// antennas x 1e5 - / 530 / 362 / 342 / 367, 64 x 3e3 134 / 77 / 73 / 61 / 67; FP64
// ZHS, 8 antennas x 1e5 - / - / 416 / 261 / 193
inline int push_a_tile(int a_tile, int64_t n_tiles, int n_ant, int precision, int formalism, int sm_count) {
  const bool f64 = precision == C8R_FP64;
  const int64_t enough = (int64_t)sm_count * (!f64 && formalism == C8R_ZHS ? 28 : 14);
  const int least = f64 ? 2 : 4;
  auto ctas = [&](int a) { return n_tiles * ((n_ant + a - 1) / a); };
  int a = a_tile;
  while (a > least && ctas(a) < enough) a = (a + 1) / 2 > least ? (a + 1) / 2 : least;
  if (f64 && a == least && ctas(a) < sm_count) a = 1;
  return a;
}
// accumulator [replicas][n_ant][rows][n_bins] -> traces [n_ant][3][n_bins]: the
// copies are summed; box edges (the second row with rows == 2, or `edges`
// [replicas][n_ant][n_bins]) are integrated over the bins and added; add adds into
// out (FP32 only); clear zeroes the accumulator and the edges (the copies given) as
// they are read
cudaError_t launch_acc_to_traces(int precision, void* acc, int n_ant, int n_bins, int rows, void* out, bool add,
                                 bool clear, cudaStream_t st, int replicas = 1, void* edges = nullptr);

// dL/dtraces [n_ant][3][n_bins] -> bin-major [n_ant][n_bins] accumulator elements
cudaError_t launch_traces_to_bin_major(int precision, const void* g, int n_ant, int n_bins, void* out,
                                       cudaStream_t st);

// ingest: filter + derived per-track quantities into tiles; counts kept tracks
// into *kept unless kept is NULL, and (mixed precision, form not NULL) adds the
// kept tracks to form[0] and those whose start point sees the antenna array's
// centroid (M.cen_*) from above within 45 degrees to form[1]
cudaError_t launch_ingest(int precision, const TrackPtrs& t, int64_t n, void* tiles, const MedParams& M,
                          unsigned long long* kept, cudaStream_t st, unsigned long long* form = nullptr);

struct BwdArgs;

// per-precision launchers (kernels_f64.cu / kernels_mixed.cu); `lin` selects
// the linear (two-bin) deposit, whose kernels live in kernels_*_lin.cu
cudaError_t launch_forward_f64(int formalism, bool lin, const void* tiles, int64_t n_tiles, const AntRec* ants,
                               int n_ant, const MedParams& M, void* acc, const FwdShape& shape, int sm_count, int* err,
                               cudaStream_t st);
cudaError_t launch_forward_mixed(int formalism, bool lin, const void* tiles, int64_t n_tiles, const AntRec* ants,
                                 int n_ant, const MedParams& M, void* acc, const FwdShape& shape, int sm_count,
                                 int* err, cudaStream_t st);
cudaError_t launch_forward_f64_lin(int formalism, const void* tiles, int64_t n_tiles, const AntRec* ants, int n_ant,
                                   const MedParams& M, void* acc, const FwdShape& shape, int sm_count, int* err,
                                   cudaStream_t st);
cudaError_t launch_forward_mixed_lin(int formalism, const void* tiles, int64_t n_tiles, const AntRec* ants,
                                     int n_ant, const MedParams& M, void* acc, const FwdShape& shape, int sm_count,
                                     int* err, cudaStream_t st);
cudaError_t launch_arrivals_f64(int formalism, const void* tiles, int64_t n, const AntRec* ants, int n_ant,
                                const MedParams& M, int32_t* branch, int32_t* bin, float* frac, cudaStream_t st);
cudaError_t launch_arrivals_mixed(int formalism, const void* tiles, int64_t n, const AntRec* ants, int n_ant,
                                  const MedParams& M, int32_t* branch, int32_t* bin, float* frac, cudaStream_t st);
cudaError_t launch_backward_f64(int formalism, bool lin, BwdArgs& a, const FwdShape& shape, int sm_count,
                                cudaStream_t st);
cudaError_t launch_backward_mixed(int formalism, bool lin, BwdArgs& a, const FwdShape& shape, int sm_count,
                                  cudaStream_t st);
cudaError_t launch_backward_f64_lin(int formalism, BwdArgs& a, const FwdShape& shape, int sm_count, cudaStream_t st);
cudaError_t launch_backward_mixed_lin(int formalism, BwdArgs& a, const FwdShape& shape, int sm_count,
                                      cudaStream_t st);
// one running sum of the gradient over the bins, (x, y, z) as float-float
// (h + l): formed in FP64, stored as two FP32 parts so that the mixed adjoint
// takes the sum over a run of bins as (h1 - h0) + (l1 - l0) on the FP32 pipe
struct alignas(32) PrefixFF {
  float hx, hy, hz, hpad;
  float lx, ly, lz, lpad;
};
// running sums over the bins of a bin-major FP32 gradient [n_ant][n_bins]
// (mixed path): out [n_ant][n_bins + 1], entry k = the sum over bins < k
cudaError_t launch_bin_running_sums(const void* g, int n_ant, int n_bins, PrefixFF* out, cudaStream_t st);

// process-wide test knobs (c8r_set_wait_limit, c8r_inject_alloc_failures)
uint32_t current_wait_limit();
// cudaMalloc, unless an injected allocation failure is pending (then it
// returns cudaErrorMemoryAllocation without allocating)
cudaError_t dev_malloc(void** p, size_t bytes);
template <typename T>
inline cudaError_t dev_malloc(T** p, size_t bytes) {
  return dev_malloc(reinterpret_cast<void**>(p), bytes);
}

// helpers shared by the context and the batch runner
void fill_medium(MedParams& M, int kind, double n_or_N0, double H, int n_bins, double dt_ns, double eps_C,
                 double earth_radius = 0.0);
void fill_antenna(AntRec& r, double x, double y, double z, double t_ref_ns, const MedParams& M);
// the antenna array's centroid (MedParams::cen_*), which the ingest's votes for
// the arrival form of the one-bin Endpoint kernels refer to
void set_form_centroid(MedParams& M, const double* pos_xyz, int n_ant);
// MedParams::flat and its altitude terms: set when the medium is one of the
// exponential atmospheres and every antenna has the same z (exactly)
void set_flat_array(MedParams& M, const double* pos_xyz, int n_ant);
// the direction of the inclined front that the trace windows follow, if they
// do, and the axis form's constants for it (MedParams::ax, kax_*)
bool window_axis(const double* pos_xyz, const double* t_start_ns, int n_ant, double up[3]);
void set_axis(MedParams& M, const double up[3]);

}  // namespace c8r
