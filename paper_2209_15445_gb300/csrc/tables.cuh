// The raw rows of the physics tables (S2's tables; paper Sec. 2.2: initialisation apart from
// the run), shared by the arena build (kernels.cu) and the allocation-free one (noalloc.cu).
//
// Everything is FP64 on a pipe of two lanes an SM, so the work is spread: a lane per Simpson
// point of the range integrals and a thread per node and group of quantities, over as many
// blocks as that gives; only the running sums of the ranges are one thread's. One block per
// material and one thread per bin kept two SMs busy for 837 us (two materials; 0.50 ms in the
// arena build's kernels); now four launches, 84 us a call.
#pragma once
#include "layout.h"
#include "physics_init.cuh"

namespace adept {

enum { V_MUC, V_MUP, V_MUPH, V_SFULL, V_SE, V_IE, V_BE, V_SP, V_IP, V_BP, V_AP, V_RFULL, V_RE, V_RP, V_NROW };
enum { B_RFULL, B_RE, B_RP, B_NROW };

__device__ inline double s_full(const MatDev& M, double T) {
  return init::dedx_col(M, T, T, false) + init::dedx_rad(M, T, T);
}
__device__ inline double s_restr(const MatDev& M, double T, double Tc, double kc, bool pos) {
  return init::dedx_col(M, T, Tc, pos) + init::dedx_rad(M, T, kc);
}

constexpr int kRowWarps = 4;                                                    // warps a block
constexpr int kBinWarps = (kNNode - 1 + init::kBinsPerWarp - 1) / init::kBinsPerWarp;  // a row of bins
constexpr int kNodeWarps = (kNNode + 31) / 32;                                  // a row of nodes

// photon attenuations and the unrestricted stopping power: material blockIdx.y, set up from
// its record by every block and written down by the first
template <class Records>
static __global__ void __launch_bounds__(32 * kRowWarps) k_rows_full(Records in, MatDev* mats, TableRows r) {
  const int m = blockIdx.y;
  __shared__ MatDev M;
  if (threadIdx.x == 0) {
    init::setup_material(in.record(m), &M);
    if (blockIdx.x == 0) mats[m] = M;
  }
  __syncthreads();
  if (M.vacuum) return;
  double* v = r.v + m * r.v_stride;
  int w = blockIdx.x * kRowWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (w < kBinWarps) {
    const int first = w * init::kBinsPerWarp, k = lane / init::kSimpson;
    const double x = init::warp_bin_integral(first, [&](double T) { return s_full(M, T); });
    if (k < init::kBinsPerWarp && lane % init::kSimpson == 0 && first + k < kNNode - 1)
      r.b[m * r.b_stride + B_RFULL * kNNode + first + k] = x;
    return;
  }
  w -= kBinWarps;
  const int i = (w % kNodeWarps) * 32 + lane;
  if (i >= kNNode || w >= 2 * kNodeWarps) return;
  const double E = init::node_E(i);
  if (w < kNodeWarps) {
    v[V_MUC * kNNode + i] = init::mu_compton(M, E);
    v[V_MUP * kNNode + i] = init::mu_pair(M, E);
    v[V_MUPH * kNNode + i] = init::mu_photo(M, E);
  } else {
    v[V_SFULL * kNNode + i] = s_full(M, E);
  }
}
constexpr int kRowsFullBlocks = (kBinWarps + 2 * kNodeWarps + kRowWarps - 1) / kRowWarps;

// production thresholds of material blockIdx.x: e+- from the unrestricted range, gamma from
// five mean free paths
constexpr int kRowThreads = 320;  // a thread per node
static_assert(kRowThreads >= kNNode, "a thread per node");
static __global__ void __launch_bounds__(kRowThreads) k_rows_cuts(const MatDev* mats, double range_cut, TableRows r) {
  const int m = blockIdx.x, i = threadIdx.x;
  __shared__ double bins[kNNode], R[kNNode], mu[kNNode];
  __shared__ int first_r, first_mu;
  double *Tc = r.Tc + m * r.cut_stride, *kc = r.kc + m * r.cut_stride;
  if (mats[m].vacuum) {
    if (i == 0) { *Tc = 0.0; *kc = 0.0; }
    return;
  }
  double* v = r.v + m * r.v_stride;
  if (i == 0) { first_r = kNNode - 1; first_mu = kNNode - 1; }
  if (i < kNNode) {
    bins[i] = i < kNNode - 1 ? r.b[m * r.b_stride + B_RFULL * kNNode + i] : 0.0;
    mu[i] = v[V_MUC * kNNode + i] + v[V_MUP * kNNode + i] + v[V_MUPH * kNNode + i];
  }
  __syncthreads();
  const double target = 5.0 / range_cut;
  if (i == 0) init::prefix_range(v[V_SFULL * kNNode], bins, R);
  if (i < kNNode - 1 && mu[i + 1] <= target) atomicMin(&first_mu, i);
  __syncthreads();
  if (i < kNNode - 1 && R[i + 1] >= range_cut) atomicMin(&first_r, i);
  if (i < kNNode) v[V_RFULL * kNNode + i] = R[i];
  __syncthreads();
  if (i == 0) *Tc = init::clamp_cut(init::range_threshold(R, range_cut, first_r));
  if (i == 32) *kc = init::clamp_cut(init::gamma_threshold(mu, target, first_mu));
}

// the charged rows of material blockIdx.y
static __global__ void __launch_bounds__(32 * kRowWarps) k_rows_charged(const MatDev* mats, TableRows r) {
  const int m = blockIdx.y;
  const MatDev& M = mats[m];
  if (M.vacuum) return;
  const double tc = r.Tc[m * r.cut_stride], kk = r.kc[m * r.cut_stride];
  double* v = r.v + m * r.v_stride;
  int w = blockIdx.x * kRowWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (w < 2 * kBinWarps) {
    const bool pos = w >= kBinWarps;
    const int first = (w - (pos ? kBinWarps : 0)) * init::kBinsPerWarp, k = lane / init::kSimpson;
    const double x = init::warp_bin_integral(first, [&](double T) { return s_restr(M, T, tc, kk, pos); });
    if (k < init::kBinsPerWarp && lane % init::kSimpson == 0 && first + k < kNNode - 1)
      r.b[m * r.b_stride + (pos ? B_RP : B_RE) * kNNode + first + k] = x;
    return;
  }
  w -= 2 * kBinWarps;
  const int i = (w % kNodeWarps) * 32 + lane, group = w / kNodeWarps;
  if (i >= kNNode) return;
  const double T = init::node_E(i);
  if (group == 0) {
    v[V_SE * kNNode + i] = s_restr(M, T, tc, kk, false);
  } else if (group == 1) {
    v[V_SP * kNNode + i] = s_restr(M, T, tc, kk, true);
  } else if (group == 2) {
    v[V_IE * kNNode + i] = init::lambda_ioni(M, T, tc, false);
    v[V_AP * kNNode + i] = init::lambda_annih(M, T);
  } else if (group == 3) {
    v[V_IP * kNNode + i] = init::lambda_ioni(M, T, tc, true);
    const double b = init::lambda_brem(M, T, kk);
    v[V_BE * kNNode + i] = b;
    v[V_BP * kNNode + i] = b;
  }
}
constexpr int kRowsChargedBlocks = (2 * kBinWarps + 4 * kNodeWarps + kRowWarps - 1) / kRowWarps;

// the restricted range of e- (blockIdx.y = 0) or e+ (1) of material blockIdx.x, and the tables
// of that species (with e-, the photon's) to r.out
static __global__ void __launch_bounds__(kRowThreads) k_rows_ranges(const MatDev* mats, TableRows r) {
  const int m = blockIdx.x, pos = blockIdx.y, i = threadIdx.x;
  __shared__ double bins[kNNode], R[kNNode];
  double* v = r.v + m * r.v_stride;
  double* o = r.out ? r.out + (size_t)m * 12 * kNNode : nullptr;
  if (mats[m].vacuum) {
    if (o && i < kNNode)
      for (int t = pos ? 7 : 0; t < (pos ? 12 : 7); ++t) o[t * kNNode + i] = 0.0;
    return;
  }
  if (i < kNNode - 1) bins[i] = r.b[m * r.b_stride + (pos ? B_RP : B_RE) * kNNode + i];
  __syncthreads();
  if (i == 0) init::prefix_range(v[(pos ? V_SP : V_SE) * kNNode], bins, R);
  __syncthreads();
  if (i >= kNNode) return;
  v[(pos ? V_RP : V_RE) * kNNode + i] = R[i];
  if (!o) return;
  const int rows[12] = {V_MUC, V_MUP, V_MUPH, V_SE, V_RE, V_IE, V_BE, V_SP, V_RP, V_IP, V_BP, V_AP};
#pragma unroll
  for (int t = 0; t < 12; ++t)
    if ((t >= 7) == (pos != 0)) o[t * kNNode + i] = (t == 4 || t == 8) ? R[i] : v[rows[t] * kNNode + i];
}

template <class Records>
static cudaError_t launch_table_rows(const Records& in, int n_mat, double range_cut, MatDev* mats, const TableRows& r,
                              cudaStream_t st) {
  k_rows_full<<<dim3(kRowsFullBlocks, n_mat), 32 * kRowWarps, 0, st>>>(in, mats, r);
  k_rows_cuts<<<n_mat, kRowThreads, 0, st>>>(mats, range_cut, r);
  k_rows_charged<<<dim3(kRowsChargedBlocks, n_mat), 32 * kRowWarps, 0, st>>>(mats, r);
  k_rows_ranges<<<dim3(n_mat, 2), kRowThreads, 0, st>>>(mats, r);
  return cudaGetLastError();
}

}  // namespace adept
