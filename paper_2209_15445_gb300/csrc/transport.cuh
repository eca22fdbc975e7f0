// Device side of one transport step, shared by the per-species generation kernels
// (kernels.cu, variants.cu) and the one-kernel-per-generation form (fused.cu): track load
// and store, phase A (S1-S8), phase B (S9), scoring (S10), warp-aggregated appends and
// the per-warp ring of deferred interactions.
#pragma once
#include <cuda_runtime.h>

#include "device.cuh"
#include "layout.h"

namespace adept {

template <class R> struct Trk {
  double x, y, z;
  R u[3];
  double E;
  unsigned long long id;
  uint32_t ev, step, nav;
};

// the queue of species s in the buffers of parity p
__device__ __forceinline__ char* track_queue(const Params& P, int p, int s) {
  return P.queues + (size_t)(3 * p + s) * P.queue_bytes;
}
// event slot of track i of a queue (from L2: the tail kernel reads what other SMs wrote)
__device__ __forceinline__ uint32_t track_event(const Params& P, const char* q, uint32_t i) {
  const char* a = P.split ? q + (size_t)(i >> 5) * Tile<float>::kBytes + Tile<float>::kMeta + (i & 31u) * 16u + 8u
                          : q + (size_t)(i >> 5) * Tile<double>::kBytes + Tile<double>::kEv + (i & 31u) * 4u;
  return __ldcg((const uint32_t*)a);
}

// Queue loads are streaming (ld.global.cs): each slot is read once per generation. The tail
// kernel (L2 = true) reads in one generation what other SMs wrote in the one before, and goes
// to L2 (ld.global.cg; everywhere it took 33.1 instead of 32.7 ms on 10,000 10 GeV showers).
template <bool L2, class T> __device__ __forceinline__ T load_stream(const T* p) { return L2 ? __ldcg(p) : __ldcs(p); }
template <bool L2>
__device__ __forceinline__ void load_track(const char* q, uint32_t tile, uint32_t lane, Trk<double>& t) {
  using L = Tile<double>;  // lane: the track's place in its tile
  const char* a = q + (size_t)tile * L::kBytes;
  const double* d = (const double*)a + lane;
  const uint32_t* w = (const uint32_t*)(a + L::kEv) + lane;
  t.x = load_stream<L2>(d + L::kX / 8); t.y = load_stream<L2>(d + L::kY / 8); t.z = load_stream<L2>(d + L::kZ / 8);
  t.u[0] = load_stream<L2>(d + L::kUX / 8); t.u[1] = load_stream<L2>(d + L::kUY / 8);
  t.u[2] = load_stream<L2>(d + L::kUZ / 8);
  t.E = load_stream<L2>(d + L::kE / 8);
  t.id = load_stream<L2>((const unsigned long long*)d + L::kId / 8);
  t.ev = load_stream<L2>(w);
  t.step = load_stream<L2>(w + (L::kStep - L::kEv) / 4);
  t.nav = load_stream<L2>(w + (L::kNav - L::kEv) / 4);
}
template <bool L2>
__device__ __forceinline__ void load_track(const char* q, uint32_t tile, uint32_t lane, Trk<float>& t) {
  using L = Tile<float>;
  const char* r = q + (size_t)tile * L::kBytes + lane * 16u;
  const double2 a = load_stream<L2>((const double2*)(r + L::kXY)), b = load_stream<L2>((const double2*)(r + L::kZE));
  const float4 c = load_stream<L2>((const float4*)(r + L::kUN));
  const uint4 d = load_stream<L2>((const uint4*)(r + L::kMeta));
  t.x = a.x; t.y = a.y; t.z = b.x; t.E = b.y;
  t.u[0] = c.x; t.u[1] = c.y; t.u[2] = c.z;
  t.nav = __float_as_uint(c.w);
  t.id = (unsigned long long)d.x | ((unsigned long long)d.y << 32);
  t.ev = d.z;
  t.step = d.w;
}

template <class R>
__device__ __forceinline__ void store_track(char* q, uint32_t i, double x, double y, double z, R ux, R uy, R uz, double E,
                                            unsigned long long id, uint32_t ev, uint32_t step, uint32_t nav);
template <>
__device__ __forceinline__ void store_track<double>(char* q, uint32_t i, double x, double y, double z, double ux, double uy,
                                                    double uz, double E, unsigned long long id, uint32_t ev, uint32_t step,
                                                    uint32_t nav) {
  using L = Tile<double>;
  char* a = q + (size_t)(i >> 5) * L::kBytes;
  double* d = (double*)a + (i & 31u);
  uint32_t* w = (uint32_t*)(a + L::kEv) + (i & 31u);
  d[L::kX / 8] = x; d[L::kY / 8] = y; d[L::kZ / 8] = z;
  d[L::kUX / 8] = ux; d[L::kUY / 8] = uy; d[L::kUZ / 8] = uz;
  d[L::kE / 8] = E;
  ((unsigned long long*)d)[L::kId / 8] = id;
  w[0] = ev;
  w[(L::kStep - L::kEv) / 4] = step;
  w[(L::kNav - L::kEv) / 4] = nav;
}
template <>
__device__ __forceinline__ void store_track<float>(char* q, uint32_t i, double x, double y, double z, float ux, float uy,
                                                   float uz, double E, unsigned long long id, uint32_t ev, uint32_t step,
                                                   uint32_t nav) {
  using L = Tile<float>;
  char* r = q + (size_t)(i >> 5) * L::kBytes + (i & 31u) * 16u;
  *(double2*)(r + L::kXY) = make_double2(x, y);
  *(double2*)(r + L::kZE) = make_double2(z, E);
  *(float4*)(r + L::kUN) = make_float4(ux, uy, uz, __uint_as_float(nav));
  *(uint4*)(r + L::kMeta) = make_uint4((uint32_t)id, (uint32_t)(id >> 32), ev, step);
}

// an outgoing particle (paper Sec. 4: the GPU region hands back the particles that leave it)
__device__ __forceinline__ void record_leak(const Params& P, int pdg, uint32_t slot, double E, double x, double y,
                                            double z, double ux, double uy, double uz) {
  const unsigned long long i = atomicAdd(&P.ctrl->leak_count, 1ull);
  if (i - __ldcg(&P.ctrl->leak_floor) >= P.leak_cap) {
    atomicAdd(&P.ctrl->leak_dropped, 1ull);
    return;
  }
  LeakRec& r = P.leak[i % P.leak_cap];
  r.pdg = pdg; r.slot = slot; r.E = E;
  r.pos[0] = x; r.pos[1] = y; r.pos[2] = z;
  r.dir[0] = ux; r.dir[1] = uy; r.dir[2] = uz;
}

template <class R> __device__ __forceinline__ const typename Pair2<R>::T* tab_g(const TableView& T);
template <> __device__ __forceinline__ const double2* tab_g<double>(const TableView& T) { return T.g64; }
template <> __device__ __forceinline__ const float2* tab_g<float>(const TableView& T) { return T.g32; }
template <class R> __device__ __forceinline__ const typename Pair2<R>::T* tab_e(const TableView& T);
template <> __device__ __forceinline__ const double2* tab_e<double>(const TableView& T) { return T.e64; }
template <> __device__ __forceinline__ const float2* tab_e<float>(const TableView& T) { return T.e32; }
template <class R> __device__ __forceinline__ const typename Pair2<R>::T* tab_p(const TableView& T);
template <> __device__ __forceinline__ const double2* tab_p<double>(const TableView& T) { return T.p64; }
template <> __device__ __forceinline__ const float2* tab_p<float>(const TableView& T) { return T.p32; }
template <class R> __device__ __forceinline__ const R* range_nodes(const TableView& T, bool pos);
template <> __device__ __forceinline__ const double* range_nodes<double>(const TableView& T, bool pos) { return pos ? T.rp64 : T.re64; }
template <> __device__ __forceinline__ const float* range_nodes<float>(const TableView& T, bool pos) { return pos ? T.rp32 : T.re32; }

template <class R> __device__ __forceinline__ const uint16_t* range_index(const TableView& T, bool pos);
template <> __device__ __forceinline__ const uint16_t* range_index<double>(const TableView& T, bool pos) { return pos ? T.xp64 : T.xe64; }
template <> __device__ __forceinline__ const uint16_t* range_index<float>(const TableView& T, bool pos) { return pos ? T.xp32 : T.xe32; }

enum Outcome { kDead = 0, kAlive = 1, kInteract = 2 };

// Phase A of one step of one track of species S (0 gamma, 1 e-, 2 e+) -- paper Sec. 3:
// every live track advances by one step per generation. Cross sections and range at the
// pre-step energy (S2), sampled interaction length (S3), step limit (S4), boundary
// distance (S5/S6), move, continuous loss (S7) and boundary crossing (S8). A step that
// ends in a discrete interaction returns kInteract with the chosen process; the
// interaction itself (S9) runs later on a full warp. dep is the energy to score in
// dep_bin. A positron that stops also returns kInteract (process 3): its annihilation at
// rest runs with the interactions, from the same random stream, so that phase A emits no
// secondaries (its appends take the one-ballot path, and the e+ kernel needs fewer
// registers: 3 blocks per SM measured +2.4 % over 2). So does a track that leaves the world
// (process 4), recorded there with its exit state (+0.9 %). The variant V compiles
// in the optional parts, kept out of the kernels that do not use them: bit 0 the chord
// propagator of the field (P.chord_iter > 0), bit 1 multiple scattering and loss
// fluctuations (P.physics), bit 2 the validation histogram of step lengths (P.steplen;
// its never-taken branch cost the default kernels 1.6 %), bit 3 the helix of a charged
// track in the uniform field (P.field_T != 0; without it a track moves straight, and the
// kernels for the field-free calorimeters carry no helix code: +1.5 %), bit 4 the rounding of
// the one-kernel-per-generation form (see transverse2).
template <class R, int S, int V = 0>
__device__ __forceinline__ int step_transport(const Params& P, Trk<R>& t, Ixn<R>& sec, double& dep, int& dep_bin,
                                              uint32_t& pstep, int& proc) {
  constexpr int q = S == 1 ? -1 : (S == 2 ? 1 : 0);
  const double rest = S == 2 ? 2.0 * kMe : 0.0;
  const int vol = (int)(t.nav & 0xFFFFu);
  uint32_t vac = t.nav >> 16;
  const int m = ro(P.geo.vol_mat + vol);
  dep_bin = ro(P.geo.vol_bin + vol);
  sec.n = 0;
  dep = 0.0;
  const uint32_t step = t.step;
  pstep = step;
  if (step >= P.max_steps) { atomicAdd(P.evt.killed + t.ev, t.E + rest); return kDead; }
  if (m < 0) {
    if (vac >= P.max_vac) { atomicAdd(P.evt.killed + t.ev, t.E + rest); return kDead; }
    ++vac;
  } else {
    vac = 0;
  }
  const R tcut = (R)P.tcut;
  const R Er = to_r<R>(t.E);
  Stream<R> rs(P, __ldg(P.evt.key + t.ev), t.id, step);
  if (pos_lt(Er, tcut)) {
    dep = t.E;
    if (S == 2) { proc = 3; return kInteract; }  // annihilates at rest in phase B
    return kDead;
  }
  R u0, u1;
  rs.block0(&u0, &u1);

  // S2: cross sections and range at the pre-step energy
  R sg0 = 0, sg1 = 0, sg2 = 0, Rr = 0;
  int bin = 0;
  if (m >= 0) {
    R tt;
    grid_pos<R>(t.E, &bin, &tt);
    if (S == 0) {
      const auto* rec = tab_g<R>(P.tab) + ((size_t)m * kNNode + bin) * kNTabG;
      // a process switched off by the mask has a zero table (k_pack)
      sg0 = lerp_rec<R>(rec, 0, tt);
      sg1 = lerp_rec<R>(rec, 1, tt);
      sg2 = lerp_rec<R>(rec, 2, tt);
    } else if (S == 1) {
      const auto* rec = tab_e<R>(P.tab) + ((size_t)m * kNNode + bin) * kNTabE;
      Rr = lerp_rec<R>(rec, 1, tt);
      sg0 = lerp_rec<R>(rec, 2, tt);
      sg1 = lerp_rec<R>(rec, 3, tt);
    } else {
      const auto* rec = tab_p<R>(P.tab) + ((size_t)m * kNNode + bin) * kNTabP;
      Rr = lerp_rec<R>(rec, 1, tt);
      sg0 = lerp_rec<R>(rec, 2, tt);
      sg1 = lerp_rec<R>(rec, 3, tt);
      sg2 = lerp_rec<R>(rec, 4, tt);
    }
  }
  sg0 = not_negative(sg0);
  sg1 = not_negative(sg1);
  sg2 = not_negative(sg2);
  const R stot = sg0 + sg1 + sg2;
  // S3/S4: sampled interaction length and the range-based step limit
  R s_phys = is_positive(stot) ? M<R>::fdiv(-M<R>::flog(u0), stot) : M<R>::big();
  constexpr bool CH = (V & 1) != 0, PH = (V & 2) != 0 && S != 0;
  const bool msc = PH && (P.physics & 1u) != 0, fluct = PH && (P.physics & 2u) != 0;
  bool limited = false;  // the step limit, not the sampled interaction length, ends the step
  if (q != 0 && m >= 0) {
    const R part = (R)kAlphaR * Rr;
    R smax = pos_le(Rr, (R)kRhoF) ? Rr : (pos_lt((R)kRhoF, part) ? part : (R)kRhoF);
    if (PH && msc) {  // multiple-scattering step limit
      const R fR = (R)P.msc_f * Rr;
      const R sm = fR > (R)0.01 ? fR : (R)0.01;
      if (sm < smax) smax = sm;
    }
    if (pos_lt(smax, s_phys)) { s_phys = smax; limited = true; }
  }
  // S5/S6: distance to the boundary along the straight line or helix
  int next;
  const bool field = (V & 8) != 0 && (q != 0) && (P.field_T != 0.0);
  // the rounding of the navigation (see transverse2): written out but in the optional-physics
  // kernels, which have no tail kernel beside them (chords have their own)
  constexpr int F = (V & 2) != 0 ? 0 : (S != 0 && ((V & 16) != 0 || sizeof(R) == 8) ? 2 : 1);
  bool boundary;
  R s;
  if constexpr (CH) {
    // chord propagation (paper Sec. 2.3): a step whose integration does not finish within
    // the iteration cap kills its track, with the energy accounted
    R sd;
    const int rc = chord_step<R>(P.geo, P.field_T, t.E, q, s_phys, P.chord_iter, (R)P.delta_chord, (R)P.delta_int,
                                 &t.x, &t.y, &t.z, t.u, vol, &next, &sd);
    if (rc == 2) { atomicAdd(P.evt.killed + t.ev, t.E + rest); return kDead; }
    boundary = rc == 1;
    s = sd;
  } else {
    const R s_geom = field ? helix_distance<R, F>(P.geo, P.field_T, t.E, q, t.x, t.y, t.z, t.u, vol, &next)
                           : straight_distance<R, F>(P.geo, t.x, t.y, t.z, t.u, vol, &next);
    boundary = pos_le(s_geom, s_phys);
    s = boundary ? s_geom : s_phys;
    if (field) {
      helix_move<R, F>(P.field_T, t.E, q, s, &t.x, &t.y, &t.z, t.u);
    } else {
      t.x += to_d<R>(s * t.u[0]);
      t.y += to_d<R>(s * t.u[1]);
      t.z += to_d<R>(s * t.u[2]);
    }
  }
  if (boundary && P.geo.kind == 0 && next >= 0) t.z = ro(P.geo.bnd + (t.u[2] > (R)0 ? vol + 1 : vol));
  t.step = step + 1;
  if constexpr ((V & 4) != 0) {
    if (P.steplen && s > (R)0 && s < M<R>::big()) {
      // validation histogram of step lengths: bin = floor(log2 s[mm]) + 40
      int b = ilogb(s) + 40;
      b = b < 0 ? 0 : (b > 63 ? 63 : b);
      atomicAdd(P.steplen + 64 * S + b, 1ull);
    }
  }

  // S7: continuous loss by inverting the range table; optionally a Gaussian loss about
  // that mean for a track that survives the mean loss
  if (q != 0 && m >= 0) {
    R Epr = 0;
    if (pos_lt(s, Rr))
      Epr = inverse_range<R>(range_nodes<R>(P.tab, S == 2) + m * kNNode, range_index<R>(P.tab, S == 2) + m * kRangeKeys,
                             Rr - s);
    double Ep = pos_lt(Er, Epr) ? t.E : to_d<R>(Epr);
    if constexpr (PH) {
      if (fluct && s < Rr && Ep >= P.tcut) {
        const R xi = (R)(kTwoPiRe2Me * __ldg(&P.mat[m].n_el));
        const R sig = M<R>::sqrt(fluct_sigma2<R>(Er, xi, (R)ro(P.tab.Tc + m), s, S == 2));
        Ep = t.E - fluct_loss<R>(rs, t.E - Ep, sig);
        Epr = to_r<R>(Ep);
      }
    }
    dep += t.E - Ep;
    t.E = Ep;
    if (pos_lt(Epr, tcut)) {
      dep += t.E;
      t.E = 0.0;
      if (S == 2) { proc = 3; return kInteract; }  // annihilates at rest in phase B
      return kDead;
    }
    // optional multiple scattering: the direction at the end of the step
    if constexpr (PH) {
      if (msc && s > (R)0) msc_deflect<R>(rs, msc_theta0<R>(Er, (R)__ldg(&P.mat[m].inv_x0), s), t.u);
    }
  }
  // S8: boundary crossing
  if (boundary) {
    if (next < 0) { proc = 4; return kInteract; }  // recorded as it leaves, in phase B
    t.nav = (uint32_t)next | (vac << 16);
    return kAlive;
  }
  t.nav = (uint32_t)vol | (vac << 16);
  // a step cut short by the step limit ends with its continuous loss only
  if (limited) return kAlive;
  // S9 (deferred): the process is chosen with u1 over the fixed order
  const R xs = u1 * stot;
  proc = (S == 1) ? 1 : 2;
  if (xs < sg0) proc = 0;
  else if (xs < sg0 + sg1) proc = 1;
  return kInteract;
}

// Phase B: the discrete interaction (S9) of a track queued by phase A, the annihilation at
// rest of a positron that stopped (process 3), or the outgoing record of a track that left
// the world (process 4). Its random stream is rebuilt from (event,
// id, step): block 0 was consumed in phase A, the models draw from block 1 on. Returns
// whether the parent survives (with its new state in t).
template <class R, int S>
__device__ __forceinline__ bool step_interact(const Params& P, Trk<R>& t, uint32_t pstep, int proc, Ixn<R>& sec,
                                              double& dep) {
  Stream<R> rs(P, __ldg(P.evt.key + t.ev), t.id, pstep);
  if (proc == 4) {  // the track left the world: its energy and its outgoing record
    sec.happened = false;
    sec.n = 0;
    dep = 0.0;
    atomicAdd(P.evt.leaked + t.ev, t.E + (S == 2 ? 2.0 * kMe : 0.0));
    record_leak(P, S == 0 ? 22 : (S == 1 ? 11 : -11), t.ev, t.E, t.x, t.y, t.z, t.u[0], t.u[1], t.u[2]);
    return false;
  }
  if (S == 2 && proc == 3) {  // a positron that stopped: two photons, drawn from block 1 on
    sec.happened = false;
    dep = 0.0;
    annihilate_at_rest<R>(rs, sec);
    return false;
  }
  const int m = ro(P.geo.vol_mat + (int)(t.nav & 0xFFFFu));
  const double Tc = ro(P.tab.Tc + m), kc = ro(P.tab.kc + m);
  const R tcut = (R)P.tcut;
  sec.happened = false;
  sec.n = 0;
  dep = 0.0;
  if (S == 0) {
    if (proc == 0) compton<R>(rs, t.E, t.u, sec);
    else if (proc == 1) pair<R>(rs, t.E, t.u, sec);
    else photo<R>(t.E, t.u, sec);
  } else if (S == 1) {
    if (proc == 0) moller<R>(rs, t.E, Tc, t.u, sec);
    else brem<R>(rs, t.E, kc, t.u, sec);
  } else {
    if (proc == 0) bhabha<R>(rs, t.E, Tc, t.u, sec);
    else if (proc == 1) brem<R>(rs, t.E, kc, t.u, sec);
    else annihilate<R>(rs, t.E, t.u, sec);
  }
  if (!sec.happened) { sec.n = 0; return true; }
  // secondaries other than positrons below the tracking cut deposit locally
#pragma unroll
  for (int k = 0; k < 2; ++k)
    if (k < sec.n && sec.sp[k] != 2 && to_r<R>(sec.E[k]) < tcut) { dep += sec.E[k]; sec.sp[k] = -1; }
  if (!sec.parent_alive) return false;
  t.E = sec.parent_E;
  t.u[0] = sec.pd[0]; t.u[1] = sec.pd[1]; t.u[2] = sec.pd[2];
  if (S == 0 && to_r<R>(t.E) < tcut) { dep += t.E; return false; }
  return true;
}

__device__ __forceinline__ void score(const Params& P, uint32_t ev, int bin, double dep) {
  if (bin >= 0 && __double_as_longlong(dep) != 0) atomicAdd(P.evt.edep + (size_t)ev * P.geo.n_bins + bin, dep);
}

// Warp-aggregated appends (S9/S11): every lane of the warp calls this; a lane passes the
// surviving track (alive) and up to two secondaries, and gets consecutive slots of the
// next queues through one atomic per species per warp.
// Most passes append survivors of the kernel's own species only (every phase-A pass of a
// photon or an electron, and interactions whose secondaries all fell below the cuts): a
// warp-uniform test sends those through one ballot and one reservation instead of nine
// (measured +2.1 % on the 10 GeV showers).
template <class R, int S>
__device__ __forceinline__ void emit(const Params& P, int p, int cw, const Trk<R>& t, bool alive, const Ixn<R>& sec,
                                     uint32_t pstep, uint32_t* ncreated) {
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  if (!__any_sync(0xFFFFFFFFu, sec.n > 0 && (sec.sp[0] >= 0 || (sec.n > 1 && sec.sp[1] >= 0)))) {
    const uint32_t bs = __ballot_sync(0xFFFFFFFFu, alive);
    uint32_t bk = 0;
    if (lane == 0 && bs) bk = atomicAdd(&P.ctrl->count[cw][S].n, __popc(bs));
    bk = __shfl_sync(0xFFFFFFFFu, bk, 0);
    if (alive) {
      const uint32_t d = bk + __popc(bs & lt);
      if (d < P.cap) {
        store_track<R>(track_queue(P, p ^ 1, S), d, t.x, t.y, t.z, t.u[0], t.u[1], t.u[2], t.E, t.id, t.ev, t.step, t.nav);
      } else {
        atomicAdd(&P.ctrl->overflow, 1ull);
        atomicAdd(P.evt.killed + t.ev, t.E + (S == 2 ? 2.0 * kMe : 0.0));
      }
    }
    return;
  }
  const bool f1 = sec.n > 0 && sec.sp[0] >= 0;
  const bool f2 = sec.n > 1 && sec.sp[1] >= 0;
  const int s1 = f1 ? sec.sp[0] : -1, s2 = f2 ? sec.sp[1] : -1;
  uint32_t b0[3], b1[3], b2[3], wbase[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    b0[k] = __ballot_sync(0xFFFFFFFFu, alive && k == S);
    b1[k] = __ballot_sync(0xFFFFFFFFu, s1 == k);
    b2[k] = __ballot_sync(0xFFFFFFFFu, s2 == k);
    const uint32_t cnt = __popc(b0[k]) + __popc(b1[k]) + __popc(b2[k]);
    uint32_t bk = 0;
    if (lane == 0 && cnt) bk = atomicAdd(&P.ctrl->count[cw][k].n, cnt);
    wbase[k] = __shfl_sync(0xFFFFFFFFu, bk, 0);
    ncreated[k] += __popc(b1[k]) + __popc(b2[k]);
  }
  // pick entry k of a 3-array without dynamic indexing (which would place it in local memory)
  auto pick = [](const uint32_t* a, int k) { return k == 0 ? a[0] : (k == 1 ? a[1] : a[2]); };
  if (alive) {
    const uint32_t d = wbase[S] + __popc(b0[S] & lt);
    if (d < P.cap) {
      store_track<R>(track_queue(P, p ^ 1, S), d, t.x, t.y, t.z, t.u[0], t.u[1], t.u[2], t.E, t.id, t.ev, t.step, t.nav);
    } else {
      atomicAdd(&P.ctrl->overflow, 1ull);
      atomicAdd(P.evt.killed + t.ev, t.E + (S == 2 ? 2.0 * kMe : 0.0));
    }
  }
  const uint32_t vnav = t.nav & 0xFFFFu;  // secondaries start with no vacuum history
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int sk = k == 0 ? s1 : s2;
    if (sk < 0) continue;
    const uint32_t before = __popc(pick(b0, sk)) + (k == 1 ? __popc(pick(b1, sk)) : 0u);
    const uint32_t mine = __popc((k == 0 ? pick(b1, sk) : pick(b2, sk)) & lt);
    const uint32_t d = pick(wbase, sk) + before + mine;
    if (d < P.cap) {
      const unsigned long long cid = child_id(P, __ldg(P.evt.key + t.ev), t.id, pstep, (uint32_t)k);
      store_track<R>(track_queue(P, p ^ 1, sk), d, t.x, t.y, t.z, sec.d[k][0], sec.d[k][1], sec.d[k][2], sec.E[k], cid, t.ev, 0u,
                     vnav);
    } else {
      atomicAdd(&P.ctrl->overflow, 1ull);
      atomicAdd(P.evt.killed + t.ev, sec.E[k] + (sk == 2 ? 2.0 * kMe : 0.0));
    }
  }
}

// Per-warp ring of tracks waiting for their discrete interaction (64 entries: phase A of
// one tile adds at most 32 to fewer than 32 waiting, so nothing is overwritten before it
// is processed). Interactions then run 32 at a time on a full warp instead of on the few
// lanes of each tile that happened to interact.
// nav holds the volume in its low half and the process in its high half, in place of the
// vacuum-step count: a discrete interaction (processes 0-2) happens only in a material,
// where that count is 0, and the parent of processes 3 and 4 does not continue. The FP32
// form's entry is then 64 bytes, and three 256-thread blocks take 99 KiB of shared memory,
// which leaves the SM's L1 a larger share (see max_blocks_small_carveout).
constexpr int kRing = 64;
template <class R> struct WarpRing {
  double x[kRing], y[kRing], z[kRing], E[kRing];
  unsigned long long id[kRing];
  R ux[kRing], uy[kRing], uz[kRing];
  uint32_t ev[kRing], pstep[kRing], nav[kRing];
};

// Tiles go to a warp in a fixed stride, so its next tile is known while it steps this one:
// 16 lanes each ask L2 for one of the next tile's 16 lines, so that the tile's loads find
// them there instead of in DRAM (+0.9 % on the 10 GeV showers; two tiles ahead gained less).
// FP32 form: the FP64 form is bound by its FP64 pipe.
template <class R>
__device__ __forceinline__ void prefetch_tile(const char* q, uint32_t tile, uint32_t lane) {
  if constexpr (sizeof(R) == 4) {
    if (lane < 16u)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(q + (size_t)tile * Tile<R>::kBytes + lane * 128u));
  }
}

// All of one warp's tiles of species S (tile, tile + stride, ... below tiles). Each pass of
// the loop is either phase A of the next tile (load, step to the next boundary or
// interaction, queue the interactions in the ring) or, once 32 wait or no tile is left, a
// warp of up to 32 queued interactions. Both share the scoring and the appends, so every
// part of the step is inlined once per kernel (smaller code: fewer instruction-cache
// misses).
template <class R, int S, int V = 0, bool L2 = false>
__device__ __forceinline__ void run_tiles(const Params& P, int p, int cw, uint32_t tile, uint32_t tiles, uint32_t stride,
                                          uint32_t n, WarpRing<R>& ring, uint32_t* nsteps, uint32_t* ncreated,
                                          uint32_t shift = 5) {
  const uint32_t lane = threadIdx.x & 31;
  uint32_t head = 0, tail = 0;
  for (;;) {
    const uint32_t waiting = tail - head;
    const bool phase_a = waiting < 32u && tile < tiles;  // warp-uniform
    if (!phase_a && waiting == 0u) break;
    const uint32_t c = phase_a ? 0u : min(waiting, 32u);
    Trk<R> t;
    t.nav = 0; t.ev = 0; t.id = 0; t.E = 0.0; t.step = 0;
    Ixn<R> sec;
    sec.n = 0;
    uint32_t pstep = 0;
    int outcome = kDead, proc = 0, bin = -1;
    double dep = 0.0;
    if (phase_a) {
      // (only the tail kernel takes smaller tiles: 2^shift tracks)
      const uint32_t i = L2 ? (tile << shift) + lane : (tile << 5) + lane;
      const bool active = L2 ? (lane >> shift) == 0u && i < n : i < n;
      const char* q = track_queue(P, p, S);
      if (active) load_track<L2>(q, L2 ? i >> 5 : tile, L2 ? i & 31u : lane, t);
      if (!L2 && tile + stride < tiles) prefetch_tile<R>(q, tile + stride, lane);
      if (active) outcome = step_transport<R, S, V>(P, t, sec, dep, bin, pstep, proc);
      nsteps[S] += active ? 1u : 0u;  // per lane; reduced over the warp at the end
    } else if (lane < c) {
      const uint32_t j = (head + lane) & (kRing - 1);
      t.x = ring.x[j]; t.y = ring.y[j]; t.z = ring.z[j]; t.E = ring.E[j];
      t.u[0] = ring.ux[j]; t.u[1] = ring.uy[j]; t.u[2] = ring.uz[j];
      const uint32_t nv = ring.nav[j];
      t.id = ring.id[j]; t.ev = ring.ev[j]; t.nav = nv & 0xFFFFu;
      pstep = ring.pstep[j];
      t.step = pstep + 1;
      outcome = step_interact<R, S>(P, t, pstep, (int)(nv >> 16), sec, dep) ? kAlive : kDead;
      bin = ro(P.geo.vol_bin + (int)(t.nav & 0xFFFFu));
    }
    // S10: score the step's deposit in (event, layer, material)
    score(P, t.ev, bin, dep);
    emit<R, S>(P, p, cw, t, outcome == kAlive, sec, pstep, ncreated);
    if (phase_a) {
      const uint32_t need = __ballot_sync(0xFFFFFFFFu, outcome == kInteract);
      if (outcome == kInteract) {
        const uint32_t j = (tail + __popc(need & ((1u << lane) - 1u))) & (kRing - 1);
        ring.x[j] = t.x; ring.y[j] = t.y; ring.z[j] = t.z; ring.E[j] = t.E;
        ring.ux[j] = t.u[0]; ring.uy[j] = t.u[1]; ring.uz[j] = t.u[2];
        ring.id[j] = t.id; ring.ev[j] = t.ev; ring.nav[j] = (t.nav & 0xFFFFu) | ((uint32_t)proc << 16);
        ring.pstep[j] = pstep;
      }
      tail += __popc(need);
      tile += stride;
    } else {
      head += c;
    }
    // the next pass may write ring entries that lanes of this one read
    __syncwarp();
  }
}

// A warp's first tile in a grid that takes the tiles in a stride of all its warps. Few tiles
// fill one block after the other in the FP32 form, which shares each L1 that the tables are
// loaded into (spread over all SMs, 100 showers took 3.70 instead of 2.90 ms). The FP64 form
// and the chords give every block one tile before any gets a second: their warps queue for
// their SM's two-lane FP64 pipe (100 showers of 1 GeV 8.3 -> 5.4 ms, 300 of 10 GeV 25.7 ->
// 22.2 ms; 60 barrel primaries with chords 16.7 -> 15.6 ms).
template <class R, int V>
__device__ __forceinline__ uint32_t first_tile() {
  const uint32_t w = threadIdx.x >> 5;
  return sizeof(R) == 4 && (V & 1) == 0 ? blockIdx.x * (blockDim.x >> 5) + w : w * gridDim.x + blockIdx.x;
}

// Programmatic dependent launch between generations: a generation's kernels may be
// launched (and their blocks made resident) as soon as every block of the previous
// generation's kernels has started, so that they wait on the SMs instead of being launched
// after the previous generation ends. grid_dependency_wait() returns once the previous
// generation's grids have completed and their writes are visible; both are no-ops for a
// launch without programmatic dependencies.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void allow_dependent_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// The bookkeeping between generations, done by one thread of generation g while it runs:
// empty the size slot that generation g + 1 appends to (its last reader, generation g - 1,
// has ended), and log the sizes generation g - 1 left (final once it ended). gk = 0 (the
// first generation of a chunk) leaves the log to the end of the previous chunk.
__device__ __forceinline__ void open_generation(const Params& P, uint32_t gen, uint32_t gk) {
  volatile Ctrl* c = P.ctrl;
  const uint32_t cz = (gen + 2) % 3, cr = gen % 3;
  for (int k = 0; k < 3; ++k) c->count[cz][k].n = 0;
  if (gk == 0) return;
  const uint32_t ln = c->log_n;
  if (ln < P.max_log) {
    for (int k = 0; k < 3; ++k) P.gen_log[3 * ln + k] = min(c->count[cr][k].n, P.cap);
    c->log_n = ln + 1;
  }
}

// End of a chunk of gens generations that began at gen: log the sizes its last generation left,
// and advance the generation and its count. One thread.
__device__ __forceinline__ void close_chunk(const Params& P, uint32_t gen, uint32_t gens) {
  if (gens == 0) return;  // a tail chunk that found nothing to do
  volatile Ctrl* c = P.ctrl;
  const uint32_t ln = c->log_n;
  if (ln < P.max_log) {
    for (int k = 0; k < 3; ++k) P.gen_log[3 * ln + k] = min(c->count[(gen + gens) % 3][k].n, P.cap);
    c->log_n = ln + 1;
  }
  c->generations = c->generations + gens;
  c->gen = gen + gens;
}

// Start of a chunk in status buffer b: the outgoing-ring read position the host left in its
// pinned copy, and an empty done count for the chunk's finish pass. One thread.
__device__ __forceinline__ void open_chunk(const Params& P, int b) {
  P.ctrl->leak_floor = *reinterpret_cast<const volatile unsigned long long*>(P.h_floor[b]);
  P.ctrl->done_count[b] = 0;
}

// Mark the events that have tracks in the queues of generation gen, thread i of `threads`.
__device__ __forceinline__ void mark_events(const Params& P, uint32_t gen, uint32_t first, uint32_t threads) {
  const int p = gen & 1;
  const QCount* q = P.ctrl->count[gen % 3];
  const uint32_t n0 = min(__ldcg(&q[0].n), P.cap), n1 = min(__ldcg(&q[1].n), P.cap), n2 = min(__ldcg(&q[2].n), P.cap);
  const uint32_t total = n0 + n1 + n2;
  for (uint32_t i = first; i < total; i += threads) {
    const int sp = i < n0 ? 0 : (i < n0 + n1 ? 1 : 2);
    const uint32_t j = sp == 0 ? i : (sp == 1 ? i - n0 : i - n0 - n1);
    const uint32_t ev = track_event(P, track_queue(P, p, sp), j);
    if (P.evt.alive[ev] != gen) P.evt.alive[ev] = gen;
  }
}

// One generation of one species (paper Sec. 3: TransportElectrons, TransportPositrons and
// TransportGammas). Persistent launch: each warp takes 32-track tiles of the current queue.
// The three species kernels of a generation are independent (each reads its own current
// queue and appends to the next ones atomically), so they run concurrently on three
// streams, and the next generation's kernels start once all three have ended.
// gk: the generation's place in its chunk (gen, advanced only between chunks, plus gk).
// V: the variant of the step (see step_transport); variants.cu instantiates V = 1..3 for
// e- and e+.
template <class R, int S, int MINB, int V = 0>
__global__ void __launch_bounds__(256, MINB) k_transport(Params P, uint32_t gk) {
  __shared__ unsigned long long s_steps, s_created[3];
  __shared__ WarpRing<R> rings[8];
  grid_dependency_wait();
  allow_dependent_launch();
  const uint32_t gen = __ldcg(&P.ctrl->gen) + gk;
  const int p = gen & 1;
  if (threadIdx.x == 0) { s_steps = 0; s_created[0] = s_created[1] = s_created[2] = 0; }
  // one block of the e- kernel does the bookkeeping (any of the three could)
  if (S == 1 && blockIdx.x == 0 && threadIdx.x == 0) open_generation(P, gen, gk);
  __syncthreads();
  // injection may have counted past the capacity (those tracks were dropped)
  const uint32_t n = min(__ldcg(&P.ctrl->count[gen % 3][S].n), P.cap);
  const uint32_t tiles = (n + 31) >> 5;
  const uint32_t wpb = blockDim.x >> 5;
  WarpRing<R>& ring = rings[threadIdx.x >> 5];
  // counts of one generation (at most the queue capacity each: 32 bits suffice): steps per
  // lane, reduced over the warp at the end (a ballot per pass measured 1.2 % slower), and
  // secondaries per warp
  uint32_t nsteps[3] = {0, 0, 0}, ncreated[3] = {0, 0, 0};
  run_tiles<R, S, V>(P, p, (gen + 1) % 3, first_tile<R, V>(), tiles, gridDim.x * wpb, n, ring,
                     nsteps, ncreated);
  const uint32_t wsteps = __reduce_add_sync(0xFFFFFFFFu, nsteps[S]);
  if ((threadIdx.x & 31) == 0) {
    if (wsteps) atomicAdd(&s_steps, (unsigned long long)wsteps);
    for (int k = 0; k < 3; ++k)
      if (ncreated[k]) atomicAdd(&s_created[k], (unsigned long long)ncreated[k]);
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  if (s_steps) atomicAdd(&P.ctrl->steps[S], s_steps);
  for (int k = 0; k < 3; ++k)
    if (s_created[k]) atomicAdd(&P.ctrl->created[k], s_created[k]);
}

}  // namespace adept
