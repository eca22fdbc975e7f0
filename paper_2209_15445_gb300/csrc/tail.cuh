// The tail kernel: the generations of a small population in one launch (S11, paper Sec. 5 on
// the idle GPU at the end of a batch).
//
// A generation of a few hundred tracks is bound by what stands between two generations: three
// launches with their fork and join, queue sizes read again, and tables loaded into an L1 that
// every launch finds cold. Here one thread-block cluster runs generation after generation, each
// block for one species, and the cluster's hardware barrier stands between them: its release
// and acquire order one generation's appends before the next one's loads (tracks and sizes are
// read from L2), nothing spins, and every block keeps its own copy of the tables and the
// geometry in shared memory. Every block reads the same queue sizes after the barrier, so all
// of them leave the loop at the same generation.
//
// It took the place of a conditional graph loop of the species kernels. Same box, two runs
// each: one 10 GeV shower 1.75 -> 1.28 ms (192 generations: 9.1 -> 6.7 us each), 10 showers
// 2.34 -> 2.13 ms, 100 showers 3.15 -> 2.84 ms, a round of 16 serving requests 5.15 -> 4.56 ms,
// 1500 barrel primaries with chords, which leave a few tracks looping for 10,000 generations,
// 345 -> 255 ms. What bounds it now: the dependent chain of one pass (a track's load, its step,
// its interaction, its append), about 4.5 us, and 0.3 us of barrier.
// Species by block: a block's loop then holds one species' step, and nothing spills.
#pragma once
#include <type_traits>

#define ADEPT_TABLES_IN_SHARED  // before device.cuh
#include "transport.cuh"

namespace adept {

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// What a block of species s reads of the tables and the geometry, in 16-byte units.
__host__ __device__ inline uint32_t units16(size_t bytes) { return (uint32_t)((bytes + 15) / 16); }
template <class R>
__host__ __device__ inline uint32_t tail_units(const Params& P, int s) {
  const size_t rec = 2 * sizeof(R) * (s == 0 ? kNTabG : (s == 1 ? kNTabE : kNTabP));
  uint32_t n = units16(rec * kNNode * P.n_mat) + units16(sizeof(double) * (P.geo.n_vol + (P.geo.kind == 0 ? 1 : 0))) +
               2 * units16(sizeof(int) * P.geo.n_vol) + 2 * units16(sizeof(double) * P.n_mat);
  if (s != 0) n += units16(sizeof(R) * kNNode * P.n_mat) + units16(sizeof(uint16_t) * kRangeKeys * P.n_mat);
  return n;
}

// Copy them into the block's shared memory and point Q's views there. The barrier between
// generations empties L1 (10 to 30 % of the load sectors hit), and a step's dozen dependent
// lookups then went to L2 each time. Same box, two runs each: one 10 GeV shower 1.29 -> 1.15 ms,
// 10 showers 2.06 -> 1.90 ms, 1500 barrel primaries with chords 235 -> 223 ms; FP64 unchanged.
// (Arrays of the arena start on 256 bytes, so the last unit of each may be read whole.)
extern __shared__ uint4 tail_shared_mem[];
template <class R, int S>
__device__ __forceinline__ void stage_tables(Params& Q) {
  uint4* at = tail_shared_mem;
  auto stage = [&](const auto*& p, size_t bytes) {
    const uint32_t n = units16(bytes);
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) at[i] = __ldg((const uint4*)p + i);
    p = (std::remove_reference_t<decltype(p)>)at;
    at += n;
  };
  TableView& T = Q.tab;
  const size_t nn = (size_t)kNNode * Q.n_mat, nx = sizeof(uint16_t) * kRangeKeys * Q.n_mat;
  if constexpr (sizeof(R) == 4) {
    if constexpr (S == 0) stage(T.g32, sizeof(float2) * kNTabG * nn);
    if constexpr (S == 1) { stage(T.e32, sizeof(float2) * kNTabE * nn); stage(T.re32, sizeof(float) * nn); stage(T.xe32, nx); }
    if constexpr (S == 2) { stage(T.p32, sizeof(float2) * kNTabP * nn); stage(T.rp32, sizeof(float) * nn); stage(T.xp32, nx); }
  } else {
    if constexpr (S == 0) stage(T.g64, sizeof(double2) * kNTabG * nn);
    if constexpr (S == 1) { stage(T.e64, sizeof(double2) * kNTabE * nn); stage(T.re64, sizeof(double) * nn); stage(T.xe64, nx); }
    if constexpr (S == 2) { stage(T.p64, sizeof(double2) * kNTabP * nn); stage(T.rp64, sizeof(double) * nn); stage(T.xp64, nx); }
  }
  stage(Q.geo.bnd, sizeof(double) * (Q.geo.n_vol + (Q.geo.kind == 0 ? 1 : 0)));
  stage(Q.geo.vol_mat, sizeof(int) * Q.geo.n_vol);
  stage(Q.geo.vol_bin, sizeof(int) * Q.geo.n_vol);
  stage(T.Tc, sizeof(double) * Q.n_mat);
  stage(T.kc, sizeof(double) * Q.n_mat);
  __syncthreads();
}

// The generations of species S on this block (index of count blocks with that species); V as in
// step_transport. Returns how many ran.
template <class R, int S, int V>
__device__ __forceinline__ uint32_t tail_species(Params P, uint32_t gen0, uint32_t max_gens, uint32_t index,
                                                 uint32_t count, WarpRing<R>& ring, uint32_t* nsteps, uint32_t* ncreated) {
  const uint32_t wpb = blockDim.x >> 5;
  if (P.tail_shared) stage_tables<R, S>(P);
  cluster_sync();  // the chunk is open
  for (uint32_t k = 0;; ++k) {
    const uint32_t gen = gen0 + k;
    const QCount* q = P.ctrl->count[gen % 3];
    const uint32_t n[3] = {min(__ldcg(&q[0].n), P.cap), min(__ldcg(&q[1].n), P.cap), min(__ldcg(&q[2].n), P.cap)};
    const uint32_t live = n[0] + n[1] + n[2];
    if (live == 0 || live >= P.tail_exit || k == max_gens) return k;
    if (blockIdx.x == 0 && threadIdx.x == 0) open_generation(P, gen, k);
    // as few tracks a warp as the warps allow: lanes on different paths of the step (the chord
    // and the bisection loops, the processes) run one after the other. Against full tiles, one
    // 10 GeV shower 1.06 -> 1.00 ms, 1500 barrel primaries with chords 184.5 -> 135 ms, 10 FP64
    // showers 6.57 -> 6.50 ms.
    const uint32_t warps = count * wpb;
    uint32_t shift = 0;
    while (shift < 5u && (n[S] >> shift) > warps) ++shift;
    run_tiles<R, S, V, true>(P, gen & 1, (gen + 1) % 3, (threadIdx.x >> 5) * count + index, (n[S] + (1u << shift) - 1u) >> shift,
                             count * wpb, n[S], ring, nsteps, ncreated, shift);
    cluster_sync();
  }
}

// Block b of the cluster steps species b mod 3. VG, VE: the variants of the photon and of the
// charged steps. The chunk's start (its single thread waits for host memory while the others
// copy their tables), its end and the marks of the live events are part of the kernel: against
// three launches more a chunk, one shower 1.12 -> 1.06 ms, 10 showers 1.82 -> 1.75 ms, a serving
// round 4.40 -> 4.30 ms.
template <class R, int VG, int VE>
__global__ void __launch_bounds__(256, 1) k_tail(Params P, uint32_t max_gens, int b) {
  __shared__ WarpRing<R> rings[8];
  __shared__ unsigned long long s_cnt[6];
  WarpRing<R>& ring = rings[threadIdx.x >> 5];
  if (threadIdx.x < 6) s_cnt[threadIdx.x] = 0;
  __syncthreads();
  if (blockIdx.x == 0 && threadIdx.x == 0) open_chunk(P, b);
  const uint32_t gen0 = __ldcg(&P.ctrl->gen);
  const uint32_t s = blockIdx.x % 3, index = blockIdx.x / 3, count = (gridDim.x + 2 - s) / 3;
  uint32_t nsteps[3] = {0, 0, 0}, ncreated[3] = {0, 0, 0}, k;
  if (s == 0) k = tail_species<R, 0, VG>(P, gen0, max_gens, index, count, ring, nsteps, ncreated);
  else if (s == 1) k = tail_species<R, 1, VE>(P, gen0, max_gens, index, count, ring, nsteps, ncreated);
  else k = tail_species<R, 2, VE>(P, gen0, max_gens, index, count, ring, nsteps, ncreated);
  if (k > 0) mark_events(P, gen0 + k, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
  for (int j = 0; j < 3; ++j) nsteps[j] = __reduce_add_sync(0xFFFFFFFFu, nsteps[j]);
  if ((threadIdx.x & 31) == 0)
    for (int j = 0; j < 3; ++j) {
      if (nsteps[j]) atomicAdd(&s_cnt[j], (unsigned long long)nsteps[j]);
      if (ncreated[j]) atomicAdd(&s_cnt[3 + j], (unsigned long long)ncreated[j]);
    }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int j = 0; j < 3; ++j) {
    if (s_cnt[j]) atomicAdd(&P.ctrl->steps[j], s_cnt[j]);
    if (s_cnt[3 + j]) atomicAdd(&P.ctrl->created[j], s_cnt[3 + j]);
  }
  if (blockIdx.x == 0) {
    P.ctrl->tail_k = k;
    close_chunk(P, gen0, k);
  }
}

}  // namespace adept
