// Kernels of one step iteration (Sec. 2 of the paper): fill vacant slots from
// the track-initializer buffer, compute each track's step limit and next
// action, reorder slot indices by action (Sec. 3.1), propagate, and apply the
// discrete interactions, pushing secondaries back into the buffer.
//
// Every action kernel is persistent: a grid sized to the GPU (a multiple of
// the SM count) strides over its work range, which is either all slots with
// masking (policy NONE) or one contiguous range of the partition read from
// device memory (sorted policies), so that no host round trip is needed to
// size a launch.
#include "launch.h"
#include "physics.cuh"

namespace celer {

namespace {

// ------------------------------------------------------------------ helpers
// An event's tally row: its id modulo the rows. Ids below the row count (the
// usual case) skip the division, about 25 instructions at each of the many
// sites.
static __device__ __noinline__ uint32_t row_modulo(uint32_t ev, uint32_t rows) { return ev % rows; }
__device__ __forceinline__ uint32_t row_of(const Params& p, uint32_t ev) {
  return ev < p.max_events ? ev : row_modulo(ev, p.max_events);
}

static __device__ __noinline__ int z_bin(double z, double z0, double zscale, int n_bins) {
  int b = __double2int_rd((z - z0) * zscale);  // (int)floor, one conversion
  return b < 0 ? 0 : (b > n_bins - 1 ? n_bins - 1 : b);
}
__device__ __forceinline__ int tally_bin(const Params& p, int layer, double z) {
  return p.tally_mode == 1 ? layer : z_bin(z, p.z0, p.zscale, p.n_bins);
}

__device__ __forceinline__ void deposit(const Params& p, uint32_t ev, uint32_t prim, int layer, double z, double e) {
  if (((unsigned long long)__double_as_longlong(e) << 1) == 0ull) return;  // e == +-0 on the bits
  const int b = tally_bin(p, layer, z);
  atomicAdd(&p.tally[(size_t)row_of(p, ev) * p.n_bins + b], e);
  if (prim < p.hist_cap) atomicAdd(&p.hist_edep[(size_t)prim * p.n_bins + b], e);
}

__device__ __forceinline__ void escape(const Params& p, uint32_t ev, uint32_t prim, double e) {
  atomicAdd(&p.escaped[row_of(p, ev)], e);
  if (prim < p.hist_cap) atomicAdd(&p.hist_escaped[prim], e);
}

__device__ __forceinline__ void release(const Params& p, uint32_t slot, uint32_t ev) {
  p.trk.status[slot] = VACANT;
  p.trk.action[slot] = A_NONE;
  atomicSub(&p.event_live[row_of(p, ev)], 1u);
  atomicAdd(&p.vacant[slot >> 5], 1u);
  atomicAdd(&p.tile_vacant[slot >> 8], 1u);
}

// Warp-sum a per-thread counter and add it to a device counter (negated if
// asked). Called by whole warps at kernel end.
__device__ __forceinline__ void flush_counter(unsigned long long* dst, unsigned long long v, bool negate) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0 && v != 0) atomicAdd(dst, negate ? (0ull - v) : v);
}

// ---- the initializer buffer as a concurrent queue (asynchronous block loop)
//
// Entry i of the buffer (stored at i & ring_mask) carries a state word: with
// lap = i / capacity, 2 lap means free for the writer of i, 2 lap + 1 written
// and not yet read, 2 lap + 2 read (free for the writer of i + capacity).
// The count of free entries (ctl->room) goes with it. A reader claims written
// entries on an availability count (avail), takes their indices from the head,
// so that the head never passes the tail, and adds them to room after that. A
// writer takes its entries off room before it moves the tail (reserve_entries;
// what room is short of goes back). So the tail never passes head + capacity:
// the reader of i - capacity has claimed it before i is reserved.
// Waits: the reader of i waits for its writer, which has reserved it; the writer
// of i waits for the reader of i - capacity, which has claimed it. Neither side
// does anything else in between that could wait: a writer writes what it has
// reserved, a warp reads its fill, and a block pass reads all it has claimed
// before its first step (fill_block). A warp's lanes end their waits together, so
// a wait also lasts for the other entries of the same claim or reservation, some
// tens of indices away. Every chain of waits thus runs to lower indices, by about
// a capacity every second link, and ends.
__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* a) {
  unsigned v;
  asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* a) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.u64 %0, [%1];" : "=l"(v) : "l"(a) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u32(unsigned* a, unsigned v) {
  asm volatile("st.release.gpu.u32 [%0], %1;" ::"l"(a), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned ring_lap_code(const Params& p, unsigned long long index) {
  return (unsigned)(index >> __popcll(p.ring_mask)) * 2u;
}
// Bounded wait of one thread for entry `index` to reach state `code`. After
// `timeout` cycles (~1 s by default), or if another wait gave up first
// (ABORT_WAIT), it sets ABORT_WAIT and ERR_BARRIER_TIMEOUT and returns false. A
// run that ends early otherwise (ABORT_RUN) does not end the wait: a claimed
// entry that is not read, or a reserved one that is not written, is a track
// lost.
__device__ __noinline__ bool ring_wait_poll(const Params& p, const unsigned* st, unsigned code, long long timeout) {
  unsigned* abort_word = p.barrier + 2;
  const long long t0 = clock64();
  for (;;) {
    __nanosleep(32);
    if (ld_acquire_u32(st) == code) return true;
    if ((*reinterpret_cast<volatile unsigned*>(abort_word) & ABORT_WAIT) != 0u) return false;
    if (clock64() - t0 > timeout) {
      atomicOr(abort_word, ABORT_WAIT);
      atomicOr(&p.ctl->error, ERR_BARRIER_TIMEOUT);
      return false;
    }
  }
}
__device__ __forceinline__ bool ring_wait(const Params& p, unsigned long long index, unsigned code,
                                          long long timeout = kBarrierTimeoutCycles) {
  const unsigned* st = p.ring_state + (index & p.ring_mask);
  return ld_acquire_u32(st) == code || ring_wait_poll(p, st, code, timeout);
}

// An initializer record by its 16-byte parts.
__device__ __forceinline__ void put_record(InitRecord* r, double x, double y, double z, double ux, double uy, double uz,
                                           double E, unsigned long long tid, uint32_t ev, uint32_t prim, int32_t layer,
                                           uint8_t ptype) {
  double2* v = reinterpret_cast<double2*>(r);
  v[0] = make_double2(x, y);
  v[1] = make_double2(z, ux);
  v[2] = make_double2(uy, uz);
  v[3] = make_double2(E, __longlong_as_double((long long)tid));
  reinterpret_cast<uint4*>(r)[4] = make_uint4(ev, prim, (unsigned)layer, ptype);
}
struct InitParts {
  double2 xy, zu, uu, et;  // x, y; z, ux; uy, uz; E and the id's bits
  uint4 m;                 // event, primary, layer, particle type
};
// Read from L2: another block of the same launch may have written it.
__device__ __forceinline__ InitParts get_record(const InitRecord* r) {
  const double2* v = reinterpret_cast<const double2*>(r);
  return InitParts{__ldcg(v), __ldcg(v + 1), __ldcg(v + 2), __ldcg(v + 3), __ldcg(reinterpret_cast<const uint4*>(r) + 4)};
}
// A slot filled with a record, as a fresh track.
__device__ __forceinline__ void fill_slot(const Params& p, uint32_t slot, const InitParts& r) {
  const Tracks& t = p.trk;
  t.x[slot] = r.xy.x;
  t.y[slot] = r.xy.y;
  t.z[slot] = r.zu.x;
  t.ux[slot] = r.zu.y;
  t.uy[slot] = r.uu.x;
  t.uz[slot] = r.uu.y;
  t.E[slot] = r.et.x;
  t.tid[slot] = (unsigned long long)__double_as_longlong(r.et.y);
  t.event[slot] = r.m.x;
  t.primary[slot] = r.m.y;
  t.layer[slot] = (int32_t)r.m.z;
  t.ptype[slot] = (uint8_t)r.m.w;
  t.ctr[slot] = 0u;
  t.nmfp[slot] = -1.0;
  t.action[slot] = A_NONE;
  t.status[slot] = ALIVE;
}

__device__ __forceinline__ void write_initializer(const Params& p, unsigned long long index, double x, double y,
                                                  double z, double ux, double uy, double uz, double E,
                                                  unsigned long long tid, uint32_t ev, uint32_t prim, int32_t layer,
                                                  uint8_t ptype) {
  const unsigned long long i = index & p.ring_mask;
  unsigned code = 0;
  if (p.ring_state) {  // asynchronous loop: wait until the entry's last reader is done
    code = ring_lap_code(p, index);
    if (!ring_wait(p, index, code)) return;
  }
  put_record(p.ring.rec + i, x, y, z, ux, uy, uz, E, tid, ev, prim, layer, ptype);
  if (p.ring_state) {
    st_release_u32(p.ring_state + i, code + 1u);
    atomicAdd(&p.ctl->avail, 1ull);  // one more entry readers may claim
  }
}

struct Span {
  uint32_t lo, hi;
  const uint32_t* perm;
};

// Order in which the block-local policy deals its groups to the warps: the
// interactions (costliest first), then the charged along-steps, then the
// photon along-steps (unused keys last).
__constant__ uint8_t kPieceOrder[kMaxKeys] = {K_G_COMPTON, K_E_MOLLER, K_G_PAIR, K_E_BREMS, K_E_RANGE, K_E_GEOM,
                                              K_G_GEOM, K_G_PE, 8, 9, 10, 11, 12, 13, 14, 15};

__device__ __forceinline__ uint8_t key_of(int policy, uint8_t ptype, uint8_t act) {
  if (policy == POLICY_ACTION) return ptype == GAMMA ? KA_NEUTRAL : KA_CHARGED;
  if (ptype == GAMMA) {
    switch (act) {
      case A_COMPTON: return K_G_COMPTON;
      case A_PE: return K_G_PE;
      case A_PAIR: return K_G_PAIR;
      default: return K_G_GEOM;
    }
  }
  switch (act) {
    case A_RANGE: return K_E_RANGE;
    case A_MOLLER: return K_E_MOLLER;
    case A_BREMS: return K_E_BREMS;
    default: return K_E_GEOM;
  }
}

// Distance along a straight line to the first side plane within reach (kInf:
// none). Called, not inlined: most steps skip it.
static __device__ __noinline__ double straight_side(const Params& p, double x, double y, double ux, double uy,
                                                    double reach) {
  // the signs of ux, uy on their bits: nonzero (NaN included) and positive;
  // for a positive NaN the distance test fails either way
  double s_side = kInf;
  const long long bx = dbits(ux), by = dbits(uy);
  if (((unsigned long long)bx << 1) != 0ull) {
    const double d = bx > 0 ? p.hx - x : -p.hx - x;
    if ((bx > 0 ? d : -d) <= reach * fabs(ux)) s_side = quot(d, ux);
  }
  if (((unsigned long long)by << 1) != 0ull) {
    const double d = by > 0 ? p.hy - y : -p.hy - y;
    if ((by > 0 ? d : -d) <= reach * fabs(uy)) s_side = fmin(s_side, quot(d, uy));
  }
  return s_side;
}

// --------------------------------------------------------------- step limit
// Step limit of one live track: fresh number of mean free paths if unset,
// cross-sections from the shared-memory tables, range limit, distance to
// the layer's planes (straight line, or the exact helix for charged tracks in
// the field), the shortest of them with ties resolved boundary > range >
// interaction, and for an interaction the process, chosen now with the
// pre-step cross-sections. Writes the step length, the residual range after
// the step, n_mfp and the draw counter; returns the next action.
__device__ __forceinline__ uint8_t step_limit(const Params& p, uint32_t slot, const double2* tab, const double* zb,
                                              const int32_t* lmat) {
  const Tracks& t = p.trk;
  [[maybe_unused]] long long t_mark = CELER_LANE_CLOCK();  // diagnostic build only
  const double E = t.E[slot];
  CELER_LANES(LS_STEP_LIMIT);
  const uint8_t pt = t.ptype[slot];
  const int layer = t.layer[slot];
  double nmfp = t.nmfp[slot];
  TrackRng rng(p.seed, t.event[slot], t.tid[slot], t.ctr[slot]);
  // every field of the state in one round of loads, before the calls below
  // (the compiler keeps loads behind a call it cannot see into): +1-2 %
  const double x = t.x[slot], y = t.y[slot], z = t.z[slot];
  const double ux = t.ux[slot], uy = t.uy[slot], uz = t.uz[slot];
  const double gfrac = t.gfrac[slot];
  const int gbin = t.gbin[slot];
  // nmfp < 0 on the bits: -1 marks it unset; otherwise it is >= +0 (a
  // zero difference rounds to +0)
  const bool fresh = dbits(nmfp) < 0;
  if (fresh) nmfp = -fast_log(rng.uniform(), p.mtab);

  const double2* mt = tab + lmat[layer] * (kCols * kGrid);
  const bool charged = pt != GAMMA;
  if (!charged) CELER_LANE_MARK(LS_T_LIMIT, t_mark);
  // The grid position of E: computed at the step that samples n_mfp and kept
  // in the slot. A photon's energy changes only where n_mfp is reset
  // (creation, an interaction); a charged track's continuous loss forms its
  // new energy from its new grid position, which the along-step keeps. So
  // later steps reload it instead of taking the logarithm.
  GridPos g;
  if (fresh) {
    g = grid_pos(E, p.lnEmin, p.inv_dl, p.mtab);
    t.gbin[slot] = g.bin;
    t.gfrac[slot] = g.frac;
  } else {
    g = GridPos{gbin, gfrac};
  }
  if (!charged) CELER_LANE_MARK(LS_T_LIMIT + 1, t_mark);
  double mu0, mu1, mu2 = 0.0;
  if (!charged) {
    mu0 = interp(mt + COL_COMPTON * kGrid, g);
    mu1 = interp(mt + COL_PE * kGrid, g);
    // E > threshold on the bits (E >= +0; a NaN E makes mu NaN either way)
    mu2 = dbits(E) > dbits(kPairThreshold) ? interp(mt + COL_PAIR * kGrid, g) : 0.0;
  } else {
    mu0 = interp(mt + COL_MOLLER * kGrid, g);
    mu1 = interp(mt + COL_BREMS * kGrid, g);
  }
  const double mu = (mu0 + mu1) + mu2;
  const bool eloss = charged && (p.processes & PROC_ELOSS);
  const double R = eloss ? interp(mt + COL_RANGE * kGrid, g) : 0.0;
  if (!charged) CELER_LANE_MARK(LS_T_LIMIT + 2, t_mark);

  // The limits are compared in the order z-planes, side planes, range,
  // interaction, each candidate replacing the current one only if strictly
  // shorter. A candidate that is a quotient d / u (or bounded below by an
  // expression) is evaluated only if it can be shorter than the current
  // limit s, i.e. unless |d| > s |u| (1 + 2^-50): beyond that margin the
  // rounded quotient is >= s too, so skipping its division changes no choice
  // (the divisions dominate the FP64 cost of the step limit).
  double s_geo = kInf;
  uint8_t act = A_NONE;
  const long long uzb = __double_as_longlong(uz);
  const unsigned long long uza = (unsigned long long)uzb & 0x7FFFFFFFFFFFFFFFull;
  if (uza != 0ull && uza <= 0x7FF0000000000000ull) {  // uz nonzero, not NaN: one division whatever the sign
    const bool up = uzb >= 0;
    s_geo = quot(zb[up ? layer + 1 : layer] - z, uz);
    act = up ? A_ZUP : A_ZDOWN;
  }
  double s_side = kInf;
  const bool helix = charged && ((unsigned long long)dbits(p.Bz) << 1) != 0ull;  // Bz != 0 on the bits
  if (helix) {
    // Over a path s the transverse position moves by at most s, so a side
    // plane farther than s_geo + 1e-3 cm lies beyond the z-plane limit: its
    // helix distance (rounded within ~2e-5 cm even at grazing incidence)
    // cannot be the shorter one, and is not computed (+4 % on the 4 T
    // calorimeter, whose high-energy circles all cross the side planes).
    const double reach = s_geo + 1e-3;
    if (!(farther(p.hx - fabs(x), reach) && farther(p.hy - fabs(y), reach)))
      s_side = helix_side_distance(curvature(p, pt, E), x, y, ux, uy, p.hx, p.hy);
  } else {
    const double reach = s_geo * kLimitMargin;
    // both planes beyond reach along their axis (|u| <= 1 + 2^-52, hence
    // the second margin): both tests below would fail, and most steps skip
    // them (+4 % on the 4 T calorimeter, +8 % on the 1 GeV one)
    const double reach2 = reach * kLimitMargin;
    if (!(p.hx - fabs(x) > reach2 && p.hy - fabs(y) > reach2)) {
      s_side = straight_side(p, x, y, ux, uy, reach);
    }
  }
  // most steps reach no side plane (s_side = inf): those skip the FP64
  // comparison; s_geo < 0 on the bits (negative, not -0, which stays)
  if (dbits(s_side) != dbits(kInf) && s_side < s_geo) {
    s_geo = s_side;
    act = A_SIDE;
  }
  if (dbits(s_geo) < 0 && dbits(s_geo) != dbits(-0.0)) s_geo = 0.0;
  if (!charged) CELER_LANE_MARK(LS_T_LIMIT + 3, t_mark);

  double s = s_geo;
  if (eloss) {
    // s_rng = R (R <= f) or a R + f (1 - a)(2 - f / R) >= a R + f (1 - a)
    double s_rng = kInf;
    // R, s and the bound are >= +0 (a NaN fails both tests, as in FP64)
    if (dbits(R) <= dbits(kFinalR)) {
      s_rng = R;
    } else if (dbits(kAlphaR * R + kFinalR * (1.0 - kAlphaR)) <= dbits(s * kRangeMargin)) {
      s_rng = kAlphaR * R + kFinalR * (1.0 - kAlphaR) * (2.0 - quot(kFinalR, R));
    }
    if (dbits(s_rng) < dbits(s)) {  // s_rng >= +0; s >= +0 or -0 (then false either way)
      s = s_rng;
      act = A_RANGE;
    }
  }
  bool interact = false;
  // mu > 0 on the bits (mu >= +0: a sum of interpolated non-negative
  // tables); the quotient nmfp / mu can be below s only if nmfp is below
  // s mu (rounded) by the bits or within a few ulp of it (both >= +0; for a
  // NaN product the quotient is NaN and fails the test after)
  if (dbits(mu) > 0 && dbits(nmfp) <= dbits(s * mu) + kLimitUlps) {
    const double s_int = quot(nmfp, mu);
    if (dbits(s_int) < dbits(s)) {  // s_int >= +0; s >= +0 or -0 (then false either way)
      s = s_int;
      interact = true;
    }
  }
  if (dbits(s) == dbits(kInf)) {
    act = A_TRAPPED;
    s = 0.0;
  } else {
    // Runge-Kutta field propagation with a substep cap (Sec. 3.3): a step
    // needing more than `cap` substeps of 0.1 rad of turn is cut there and
    // ends without a crossing or an interaction, to go on next iteration
    if (helix && p.field_cap > 0) {
      const double kappa = curvature(p, pt, E).kappa;
      if (s * fabs(kappa) > kRkTurn * p.field_cap) {
        s = quot(kRkTurn * p.field_cap, fabs(kappa));
        act = A_FIELD;
        interact = false;
      }
    }
    nmfp -= s * mu;
  }
  if (interact) {
    // an interaction means a finite mu, so every operand below is finite
    // and >= +0: the comparisons on the bits are exact
    const double target = rng.uniform() * mu;
    int last = -1;
    if (dbits(mu0) > 0) last = 0;
    if (dbits(mu1) > 0) last = 1;
    if (dbits(mu2) > 0) last = 2;
    int sel;
    double acc = mu0;
    if (dbits(target) < dbits(acc)) {
      sel = 0;
    } else {
      acc += mu1;
      if (dbits(target) < dbits(acc)) {
        sel = 1;
      } else {
        acc += mu2;
        sel = (!charged && dbits(target) < dbits(acc)) ? 2 : last;
      }
    }
    act = charged ? (sel == 0 ? A_MOLLER : A_BREMS) : (uint8_t)(A_COMPTON + sel);
  }
  t.nmfp[slot] = nmfp;
  t.ctr[slot] = rng.ctr;
  t.step[slot] = s;
  if (eloss) t.rpost[slot] = R - s;
  t.action[slot] = act;
  if (!charged) CELER_LANE_MARK(LS_T_LIMIT + 4, t_mark);
  return act;
}

// ------------------------------------------------------------------ phases
// Each phase is executed by every thread of a block; bid / nb are the block's
// index and the number of blocks sharing the phase. The same functions run as
// stand-alone kernels (host loop or CUDA graph) and inside the persistent
// loop kernel. One iteration is three phases:
//   A  fill vacant slots from the initializer buffer and compute the step
//      limit (next action) of every live track, tile by tile; the last block
//      to finish does the bookkeeping (buffer head, vacancy counts, partition
//      offsets, whether secondaries are sure to fit);
//   B  scatter slot indices into the partition (sorted policies only);
//   C  along-step and, for tracks whose step ends in an interaction, the
//      interaction, in partition order; the last block to finish ends the
//      iteration (counters, trace, loop condition).

__device__ __forceinline__ bool static_arrived(unsigned bar) {
  unsigned done;
  asm volatile(
      "{\n .reg .pred q;\n mbarrier.try_wait.parity.shared::cta.b64 q, [%1], 0;\n selp.u32 %0, 1, 0, q;\n}"
      : "=r"(done)
      : "r"(bar)
      : "memory");
  return done != 0u;
}
// (each try suspends the thread for a while; the limit is far above any copy)
static __device__ __noinline__ void wait_static(const Params& p, unsigned bar) {
  for (int i = 0; i < (1 << 20); ++i)
    if (static_arrived(bar)) return;
  atomicOr(&p.ctl->error, ERR_BARRIER_TIMEOUT);
}

// Static data every step kernel needs in shared memory: cross-section and
// range tables, layer planes and layer materials (one contiguous run of
// static_bytes in device memory, laid out as here).
struct SharedStatic {
  double2* tab;
  double* zb;
  int32_t* lmat;
  unsigned bar;  // the copy's barrier (shared address)
  __device__ __forceinline__ void ready(const Params& p) const {
    if (!static_arrived(bar)) wait_static(p, bar);
  }
};

__device__ __forceinline__ SharedStatic carve_static(const Params& p, unsigned char* raw) {
  SharedStatic s;
  s.tab = reinterpret_cast<double2*>(raw);
  s.zb = reinterpret_cast<double*>(s.tab + p.n_materials * kCols * kGrid);
  s.lmat = reinterpret_cast<int32_t*>(s.zb + p.n_layers + 1);
  s.bar = 0u;
  return s;
}

// The copy of the static data into shared memory in the kernels launched every
// iteration, one bulk copy (TMA): one thread starts it, ready() waits for it
// (bounded) after the block's first loads (water cube in the graph loop 1.16 ->
// 1.12 ms). Waiting only where the data are first used, in the bodies shared
// with the persistent loops, cost those 3-4 %. Ends with a block barrier.
__device__ __forceinline__ void stage_static(const Params& p, SharedStatic& s, unsigned long long* bar) {
  s.bar = (unsigned)__cvta_generic_to_shared(bar);
  if (threadIdx.x == 0) {
    const unsigned dst = (unsigned)__cvta_generic_to_shared(s.tab);
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s.bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s.bar), "r"(p.static_bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(p.tables), "r"(p.static_bytes), "r"(s.bar)
                 : "memory");
  }
  __syncthreads();
}

// The same by every thread of the block, for the loops that do it once.
__device__ __forceinline__ void stage_static(const Params& p, const SharedStatic& s) {
  const uint4* src = reinterpret_cast<const uint4*>(p.tables);
  uint4* dst = reinterpret_cast<uint4*>(s.tab);
  for (uint32_t i = threadIdx.x; i < p.static_bytes / 16u; i += blockDim.x) dst[i] = src[i];
  __syncthreads();
}

// Clear the per-iteration counters (one thread).
__device__ __forceinline__ void clear_iteration_counters(Ctl* c) {
  for (int k = 0; k < kMaxKeys; ++k) {
    c->action_count[k] = 0;
    c->key_total[k] = 0;
  }
  c->steps_iter = 0;
  c->n_deferred = 0;
}

// True in exactly one block: the last one to reach this point in the current
// phase (the counter is reset for the next phase instance). The block that
// returns true sees every other block's writes of the phase.
__device__ __forceinline__ bool last_block_done(unsigned* counter, unsigned nb) {
  __shared__ unsigned s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned ticket = atomicAdd(counter, 1u);
    s_last = (ticket == nb - 1) ? 1u : 0u;
    if (s_last) *reinterpret_cast<volatile unsigned*>(counter) = 0u;
  }
  __syncthreads();
  const bool last = s_last != 0u;
  if (last) __threadfence();
  return last;
}

// Warp-interleaved walk over [lo, hi): chunk g of `width` elements (8, 16
// or 32; lanes at and above the width idle) goes to block g % nb, so
// consecutive chunks land on different SMs. With few live tracks this
// spreads the FP64 work over all SMs instead of stacking warps on the few
// SMs that own the first chunks (an FP64 warp instruction occupies its
// sub-partition's pipe for the same time whatever its active lanes).
struct ChunkWalk {
  uint32_t lo, hi, step, g, width;
  __device__ ChunkWalk(uint32_t lo_, uint32_t hi_, int bid, int nb, uint32_t width_ = 32u)
      : lo(lo_), hi(hi_), step((uint32_t)nb * (blockDim.x >> 5)), g((uint32_t)bid + (threadIdx.x >> 5) * (uint32_t)nb),
        width(width_) {}
  __device__ __forceinline__ bool more() const { return (unsigned long long)lo + (unsigned long long)width * g < hi; }
  __device__ __forceinline__ uint32_t index() const {
    const uint32_t lane = threadIdx.x & 31;
    return lane < width ? lo + width * g + lane : hi;
  }
  __device__ __forceinline__ void next() { g += step; }
};

// Width of the step-phase chunks for a partition range of n live tracks: as
// few tracks per warp as keep one warp per SM sub-partition (nb blocks of
// four), since a warp's time is set by its instruction count and the
// slowest of its lanes (rejection loops), not by how many lanes it runs.
__device__ __forceinline__ uint32_t spread_width(uint32_t n, int nb) {
  const uint32_t subs = (uint32_t)nb * 4u;
  return n <= subs * 8u ? 8u : (n <= subs * 16u ? 16u : 32u);
}

// ---- phase A: initializer fill + step limit, on 32-slot warp-tiles
// A warp owns a 32-slot chunk: it fills the chunk's vacant slots from the
// initializer buffer (the r-th vacant slot in ascending slot order over the
// whole store takes initializer head + r, for r < queued: deterministic
// filling; vprefix[g] = vacant slots before chunk g, scanned at the end of
// the previous iteration), then computes the step limit of every live slot
// of the chunk and adds the chunk's key counts to its 256-slot tile. Chunks
// are dealt to warps interleaved over the blocks, so a handful of live
// chunks is spread over as many SMs.
__device__ __forceinline__ void fill_and_limit_chunk(const Params& p, uint32_t g, const SharedStatic& ss, bool fill,
                                                     bool do_step, unsigned long long head,
                                                     unsigned long long queued, unsigned* s_acts,
                                                     unsigned* s_keys, unsigned long long& my_steps) {
  const int lane = threadIdx.x & 31;
  const uint32_t slot = g * 32u + lane;
  const bool real = slot < p.n_slots;
  unsigned nfill = 0;
  if (fill) {
    // vacant slots before this chunk: those before its tile, plus the ones in
    // the tile's earlier chunks (at most 7, read in parallel by the lanes)
    const uint32_t first = (g >> 3) << 3;
    unsigned part = (first + lane < g) ? __ldcg(&p.vacant[first + lane]) : 0u;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    const unsigned long long before = __ldcg(&p.tile_prefix[g >> 3]) + __shfl_sync(0xffffffffu, part, 0);
    if (before < queued) {
      const bool vac = real && p.trk.status[slot] == VACANT;
      const unsigned bal = __ballot_sync(0xffffffffu, vac);
      const unsigned long long r = before + __popc(bal & ((1u << lane) - 1u));
      if (vac && r < queued) {
        fill_slot(p, slot, get_record(p.ring.rec + ((head + r) & p.ring_mask)));
      }
      const unsigned long long left = queued - before;
      nfill = (unsigned)((unsigned long long)__popc(bal) < left ? __popc(bal) : left);
    }
    if (lane == 0) {
      p.filled[g] = nfill;
      if (nfill) atomicAdd(&p.ctl->filled_total, (unsigned long long)nfill);
    }
  } else if (do_step) {
    nfill = __ldcg(&p.filled[g]);  // set by a separate fill launch
  }
  if (!do_step) return;
  const bool sorted = global_partition(p.policy);
  const uint8_t vacant_key = p.policy == POLICY_ACTION ? KA_VACANT : K_VACANT_FULL;
  const unsigned csize = (p.n_slots - g * 32u) < 32u ? (p.n_slots - g * 32u) : 32u;
  const bool live = __ldcg(&p.vacant[g]) < csize || nfill > 0;  // warp-uniform
  uint8_t key = vacant_key;
  if (live) {
    if (real) {
      const uint8_t st = p.trk.status[slot];
      uint8_t act = A_NONE;
      if (st == ALIVE) {
        act = step_limit(p, slot, ss.tab, ss.zb, ss.lmat);
        ++my_steps;
      } else if (st == DEFERRED) {
        act = p.trk.action[slot];
      }
      if (st != VACANT) {
        atomicAdd(&s_acts[act], 1u);
        if (sorted) key = key_of(p.policy, p.trk.ptype[slot], act);
      }
    }
  }
  if (sorted) {
    if (real) p.trk.key[slot] = key;
    if (lane == 0) p.chunk_dirty[g] = live ? 1 : 0;
    // only live keys are counted (per block, for the scatter): the vacant
    // key is the last one, so its slots need no position
    const unsigned k = (real && key != vacant_key) ? (unsigned)key : 0xFFFFFFFFu;
    const unsigned peers = __match_any_sync(0xffffffffu, k);
    if (k != 0xFFFFFFFFu && lane == __ffs(peers) - 1) atomicAdd(&s_keys[k], (unsigned)__popc(peers));
  }
}

// Block-wide exclusive scan of n 32-bit counts: each thread takes a
// contiguous segment (a multiple of 32 entries), loads it eight 16-byte
// vectors at a time with all loads in flight, the segment sums are scanned
// across the block, and write(i, prefix) receives the exclusive prefix of
// entry i (written to a different array than `in`). Returns the total. One
// block; every thread must call it.
template <class Write>
__device__ unsigned long long block_scan_counts(const uint32_t* __restrict__ in, uint32_t n, Write write) {
  __shared__ unsigned long long s_warp[32];
  __shared__ unsigned long long s_total;
  const uint32_t per = ((n + blockDim.x - 1) / blockDim.x + 31u) & ~31u;
  const uint32_t beg = min(threadIdx.x * per, n);
  const uint32_t end = min(beg + per, n);
  const uint4* v = reinterpret_cast<const uint4*>(in);
  unsigned long long local = 0;
  uint32_t i = beg;
  // the first 32 values stay in registers for the second pass (all of them
  // when the segment is a single round, the common case)
  uint4 q0[8];
  const bool first = i + 32 <= end;
  if (first) {
#pragma unroll
    for (int k = 0; k < 8; ++k) q0[k] = __ldcg(v + (i >> 2) + k);
#pragma unroll
    for (int k = 0; k < 8; ++k) local += (unsigned long long)q0[k].x + q0[k].y + q0[k].z + q0[k].w;
    i += 32;
  }
  for (; i + 32 <= end; i += 32) {
    uint4 q[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) q[k] = __ldcg(v + (i >> 2) + k);
#pragma unroll
    for (int k = 0; k < 8; ++k) local += (unsigned long long)q[k].x + q[k].y + q[k].z + q[k].w;
  }
  for (; i < end; ++i) local += __ldcg(in + i);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  __syncthreads();
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const unsigned long long w = lane < (int)(blockDim.x >> 5) ? s_warp[lane] : 0ull;
    unsigned long long wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long t = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += t;
    }
    s_warp[lane] = wi - w;
    if (lane == 31) s_total = wi;
  }
  __syncthreads();
  unsigned long long run = s_warp[warp] + incl - local;
  i = beg;
  if (first) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      write(i + 4 * k, run);
      run += q0[k].x;
      write(i + 4 * k + 1, run);
      run += q0[k].y;
      write(i + 4 * k + 2, run);
      run += q0[k].z;
      write(i + 4 * k + 3, run);
      run += q0[k].w;
    }
    i += 32;
  }
  for (; i + 32 <= end; i += 32) {
    uint4 q[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) q[k] = __ldcg(v + (i >> 2) + k);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      write(i + 4 * k, run);
      run += q[k].x;
      write(i + 4 * k + 1, run);
      run += q[k].y;
      write(i + 4 * k + 2, run);
      run += q[k].z;
      write(i + 4 * k + 3, run);
      run += q[k].w;
    }
  }
  for (; i < end; ++i) {
    const unsigned t = __ldcg(in + i);
    write(i, run);
    run += t;
  }
  const unsigned long long total = s_total;
  __syncthreads();
  return total;
}

// Exclusive scan of the per-tile vacancy counts into tile_prefix and their
// total, by one block (end of an iteration, when every release is counted).
__device__ void scan_vacancy(const Params& p) {
  unsigned long long* out = p.tile_prefix;
  const unsigned long long total =
      block_scan_counts(p.tile_vacant, p.n_tiles, [out](uint32_t i, unsigned long long v) { out[i] = v; });
  if (threadIdx.x == 0) p.ctl->total_vacant = total;
}

// Bookkeeping at the end of phase A, by one block: commit the initializers
// taken and decide whether this iteration's secondaries are sure to fit.
__device__ void bookkeeping_after_fill_step(const Params& p, bool did_fill) {
  Ctl* c = p.ctl;
  if (did_fill && threadIdx.x == 0) {
    const unsigned long long queued = c->tail - c->head;
    const unsigned long long tv = c->total_vacant;
    const unsigned long long take = tv < queued ? tv : queued;
    if (take != c->filled_total) c->error |= ERR_VACANCY;
    c->filled_total = 0;
    c->head += take;
    c->alive += take;
    c->total_vacant = tv - take;
  }
  if (threadIdx.x == 0) {
    const unsigned long long queued = c->tail - c->head;
    const unsigned long long max_new =
        2ull * c->action_count[A_PAIR] + c->action_count[A_MOLLER] + c->action_count[A_BREMS];
    c->defer = (queued + max_new > p.ring_capacity) ? 1u : 0u;
  }
}

// Move the fills of this iteration into the vacancy counts (all blocks, any
// phase after the fill has finished everywhere).
__device__ __forceinline__ void apply_fills(const Params& p, int bid, int nb) {
  for (uint32_t g = bid * blockDim.x + threadIdx.x; g < p.n_chunks; g += nb * blockDim.x) {
    const unsigned f = __ldcg(&p.filled[g]);
    if (f) {
      atomicSub(&p.vacant[g], f);
      atomicSub(&p.tile_vacant[g >> 3], f);
      p.filled[g] = 0u;
    }
  }
}

// Phase A (or its two halves in the per-action launch mode).
__device__ void phase_fill_step(const Params& p, int bid, int nb, const SharedStatic& ss, bool do_fill, bool do_step,
                                bool bookkeeping) {
  __shared__ unsigned s_acts[A_COUNT];
  __shared__ unsigned s_keys[kMaxKeys];
  Ctl* c = p.ctl;
  const unsigned long long head = c->head;
  const unsigned long long queued = c->tail - head;
  const bool fill = do_fill && queued > 0;
  if (threadIdx.x < A_COUNT) s_acts[threadIdx.x] = 0;
  if (threadIdx.x < kMaxKeys) s_keys[threadIdx.x] = 0;
  __syncthreads();
  unsigned long long my_steps = 0;
  if (fill || do_step) {
    // This warp's chunks are g0, g0 + step, ...: 32 at a time, each lane reads
    // one chunk's vacancy (and its tile's prefix) so the warp visits only the
    // chunks that hold live tracks or may receive initializers.
    const int lane = threadIdx.x & 31;
    const uint32_t step = (uint32_t)nb * (blockDim.x >> 5);
    const uint32_t g0 = (uint32_t)bid + (threadIdx.x >> 5) * (uint32_t)nb;
    for (uint32_t base = g0; base < p.n_chunks; base += 32u * step) {
      const uint32_t g = base + lane * step;
      bool cand = false;
      if (g < p.n_chunks) {
        const unsigned csize = (p.n_slots - g * 32u) < 32u ? (p.n_slots - g * 32u) : 32u;
        const unsigned vac = __ldcg(&p.vacant[g]);
        cand = vac < csize;
        if (!cand && fill && vac > 0) cand = __ldcg(&p.tile_prefix[g >> 3]) < queued;
        if (!cand && !do_fill) cand = __ldcg(&p.filled[g]) > 0;  // filled by a separate fill launch
        if (!cand && do_step && global_partition(p.policy)) cand = p.chunk_dirty[g] != 0;  // keys to reset
      }
      unsigned mask = __ballot_sync(0xffffffffu, cand);
      while (mask) {
        const int j = __ffs(mask) - 1;
        mask &= mask - 1;
        fill_and_limit_chunk(p, base + (uint32_t)j * step, ss, fill, do_step, head, queued, s_acts, s_keys, my_steps);
      }
    }
  }
  __syncthreads();
  if (do_step) {
    if (threadIdx.x < A_COUNT && s_acts[threadIdx.x] != 0)
      atomicAdd(&c->action_count[threadIdx.x], s_acts[threadIdx.x]);
    if (global_partition(p.policy) && (int)threadIdx.x < p.n_keys - 1)
      p.block_counts[threadIdx.x * nb + bid] = s_keys[threadIdx.x];
    flush_counter(&c->steps_iter, my_steps, false);
  }
  if (bookkeeping && last_block_done(&c->done_a, nb)) {
    const long long t0 = clock64();
    bookkeeping_after_fill_step(p, true);
    if (threadIdx.x == 0) c->book_total[0] += (unsigned long long)(clock64() - t0);
  }
}

// Scatter slot indices into the partition. Every block sums the per-(key,
// block) counts of the live keys itself, one warp per key, into its first
// position per key (a scan by the last block of phase A held up all others,
// 2.4 us per iteration); block 0 notes the key offsets. Block b owns chunks b, b + nb,
// b + 2 nb, ... (the chunks it counted in phase A). It walks those that hold
// live keys in that order, one per warp, and places each live slot at: the
// block's first position for the key (from the scan) + the block's same-key
// slots placed so far (a running cursor) + same-key slots of earlier warps in
// this pass of the loop + same-key lanes below. The order within a key is thus by owning
// block, then chunk, then lane: deterministic, and no scan over all tiles.
__device__ void phase_scatter(const Params& p, int bid, int nb) {
  __shared__ unsigned s_cnt[kTile / 32][kMaxKeys];
  __shared__ unsigned s_cursor[kMaxKeys];
  __shared__ unsigned s_wlive[kTile / 32];
  __shared__ uint32_t s_live[kTile];
  const int live_keys = p.n_keys - 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = (int)(blockDim.x >> 5);
  const unsigned lt = (1u << lane) - 1u;
  __shared__ unsigned s_tot[kMaxKeys], s_before[kMaxKeys];
  for (int k = warp; k < live_keys; k += nwarps) {
    unsigned tot = 0, bef = 0;
    for (int i = lane; i < nb; i += 32) {
      const unsigned v = __ldcg(&p.block_counts[k * nb + i]);
      tot += v;
      bef += i < bid ? v : 0u;
    }
    tot = __reduce_add_sync(0xffffffffu, tot);
    bef = __reduce_add_sync(0xffffffffu, bef);
    if (lane == 0) {
      s_tot[k] = tot;
      s_before[k] = bef;
    }
  }
  __syncthreads();
  if ((int)threadIdx.x <= live_keys) {
    unsigned base = 0;
    for (int k = 0; k < (int)threadIdx.x; ++k) base += s_tot[k];
    if ((int)threadIdx.x < live_keys) s_cursor[threadIdx.x] = base + s_before[threadIdx.x];
    if (bid == 0) {
      p.ctl->offsets[threadIdx.x] = base;
      if ((int)threadIdx.x == live_keys) {
        p.ctl->offsets[p.n_keys] = p.n_slots;
        p.ctl->part_blocks = (unsigned)nb;
      }
    }
  }
  const uint32_t n_own = (uint32_t)bid < p.n_chunks ? (p.n_chunks - (uint32_t)bid + nb - 1) / nb : 0u;
  for (uint32_t m0 = 0; m0 < n_own; m0 += blockDim.x) {
    // this pass's live chunks of the block, compacted in order
    const uint32_t m = m0 + threadIdx.x;
    const uint32_t gm = (uint32_t)bid + (uint32_t)nb * m;
    const bool live = m < n_own && p.chunk_dirty[gm] != 0;
    const unsigned bal = __ballot_sync(0xffffffffu, live);
    __syncthreads();  // the previous round is done with s_wlive and s_live
    if (lane == 0) s_wlive[warp] = __popc(bal);
    __syncthreads();
    unsigned before = 0, nlive = 0;
    for (int w = 0; w < nwarps; ++w) {
      const unsigned cw = s_wlive[w];
      before += w < warp ? cw : 0u;
      nlive += cw;
    }
    if (live) s_live[before + __popc(bal & lt)] = gm;
    __syncthreads();
    for (unsigned j0 = 0; j0 < nlive; j0 += (unsigned)nwarps) {
      const unsigned j = j0 + (unsigned)warp;
      unsigned key = 0xFFFFFFFFu;
      uint32_t slot = 0;
      if (j < nlive) {
        slot = s_live[j] * 32u + lane;
        if (slot < p.n_slots && p.trk.status[slot] != VACANT) key = p.trk.key[slot];
        if (key >= (unsigned)live_keys) key = 0xFFFFFFFFu;
      }
      const unsigned peers = __match_any_sync(0xffffffffu, key);
      if (lane < live_keys) s_cnt[warp][lane] = 0u;
      __syncwarp();
      if (key != 0xFFFFFFFFu && lane == __ffs(peers) - 1) s_cnt[warp][key] = __popc(peers);
      __syncthreads();
      if (key != 0xFFFFFFFFu) {
        unsigned pos = s_cursor[key] + __popc(peers & lt);
        for (int w = 0; w < warp; ++w) pos += s_cnt[w][key];
        p.perm[pos] = slot;
      }
      __syncthreads();
      if ((int)threadIdx.x < live_keys) {
        unsigned add = 0;
        for (int w = 0; w < nwarps; ++w) add += s_cnt[w][threadIdx.x];
        s_cursor[threadIdx.x] += add;
      }
      __syncthreads();
    }
  }
}

// Along-step of one live track: move by the step length (straight line, or
// the exact helix for charged tracks in the field), continuous energy loss
// through the inverse range table, then the geometric post-step: next layer
// or escape through a z-plane, escape through a side plane, tracking cut.
// Returns true if the track ended.
__device__ __forceinline__ bool along_one(const Params& p, uint32_t slot, uint8_t pt, const SharedStatic& ss) {
  CELER_LANES(LS_ALONG);
  const Tracks& t = p.trk;
  const bool charged = pt != GAMMA;
  const uint8_t act = t.action[slot];
  const uint32_t ev = t.event[slot], prim = t.primary[slot];
  int layer = t.layer[slot];
  double E = t.E[slot];
  double z = t.z[slot];
  // the rest of the state in the same round of loads, ahead of the atomic
  const double s = t.step[slot];
  double x = t.x[slot], y = t.y[slot];
  double ux = t.ux[slot], uy = t.uy[slot];
  const double uz = t.uz[slot];
  if (prim < p.hist_cap) atomicAdd(&p.hist_steps[prim], 1ull);
  if (act == A_TRAPPED) {
    deposit(p, ev, prim, layer, z, E);
    release(p, slot, ev);
    return true;
  }
  const bool eloss = charged && (p.processes & PROC_ELOSS);
  const bool helix = charged && ((unsigned long long)dbits(p.Bz) << 1) != 0ull;  // Bz != 0 on the bits
  if (helix) {
    const Curvature cv = curvature(p, pt, E);
    if (p.field_cap > 0)
      rk_move(cv.kappa, s, act == A_FIELD ? p.field_cap : rk_substeps(cv.kappa, s), x, y, z, ux, uy, uz);
    else
      helix_move(cv, s, x, y, z, ux, uy, uz, p.mtab);
  } else {
    x += s * ux;
    y += s * uy;
    z += s * uz;
  }
  if (eloss) {
    const double2* R = ss.tab + (ss.lmat[layer] * kCols + COL_RANGE) * kGrid;
    GridPos g{0, 0.0};
    const double Ep = inverse_range(R, t.rpost[slot], p.lnEmin, p.dl, p.mtab, g);
    t.gbin[slot] = g.bin;
    t.gfrac[slot] = g.frac;
    deposit(p, ev, prim, layer, z, E - Ep);
    E = Ep;
  }
  bool out = false;
  if (act == A_ZUP) {
    layer += 1;
    if (layer >= p.n_layers) {
      out = true;
    } else {
      z = ss.zb[layer];
    }
  } else if (act == A_ZDOWN) {
    z = ss.zb[layer];
    layer -= 1;
    if (layer < 0) out = true;
  } else if (act == A_SIDE) {
    out = true;
  }
  if (out) {
    escape(p, ev, prim, E);
    release(p, slot, ev);
    return true;
  }
  // E < cut on the bits (E >= +0; a NaN E fails it, as in FP64)
  if (dbits(E) < dbits(p.cut_track)) {
    deposit(p, ev, prim, layer, z, E);
    release(p, slot, ev);
    return true;
  }
  t.x[slot] = x;
  t.y[slot] = y;
  t.z[slot] = z;
  if (helix) {
    t.ux[slot] = ux;
    t.uy[slot] = uy;
  }
  if (eloss) t.E[slot] = E;
  if (act == A_ZUP || act == A_ZDOWN) t.layer[slot] = layer;
  return false;
}

// ---- discrete interactions (one track each; return true if the track ended)

// Compton scattering: Klein-Nishina sampling, the recoil energy deposited
// locally, the photon rotated; below the tracking cut it is absorbed.
__device__ __forceinline__ bool compton_one(const Params& p, uint32_t slot) {
  CELER_LANES(LS_COMPTON);
  const Tracks& t = p.trk;
  const double E = t.E[slot];
  const uint32_t ev = t.event[slot], prim = t.primary[slot];
  const int layer = t.layer[slot];
  const double z = t.z[slot];
  TrackRng rng(p.seed, ev, t.tid[slot], t.ctr[slot]);
  double cost;
  bool ok;
  const double eps = sample_compton(E, rng, cost, ok, p.mtab);
  if (!ok) {  // non-finite input: end the track, flag the run
    atomicOr(&p.ctl->error, ERR_SAMPLING);
    deposit(p, ev, prim, layer, z, E);
    release(p, slot, ev);
    return true;
  }
  const double u_phi = rng.uniform();
  const double E1 = eps * E;
  deposit(p, ev, prim, layer, z, E - E1);
  if (dbits(E1) < dbits(p.cut_track)) {  // on the bits: a negative E1 passes, a positive NaN fails, as in FP64
    deposit(p, ev, prim, layer, z, E1);
    release(p, slot, ev);
    return true;
  }
  double ux = t.ux[slot], uy = t.uy[slot], uz = t.uz[slot];
  rotate_dir(ux, uy, uz, cost, u_phi, p.mtab);
  t.ux[slot] = ux;
  t.uy[slot] = uy;
  t.uz[slot] = uz;
  t.E[slot] = E1;
  t.nmfp[slot] = -1.0;
  t.ctr[slot] = rng.ctr;
  return false;
}

// Photoelectric absorption: all energy deposited locally.
__device__ __forceinline__ bool photoelectric_one(const Params& p, uint32_t slot) {
  CELER_LANES(LS_PE);
  const Tracks& t = p.trk;
  const uint32_t ev = t.event[slot];
  deposit(p, ev, t.primary[slot], t.layer[slot], t.z[slot], t.E[slot]);
  release(p, slot, ev);
  return true;
}

// Secondary-producing interactions reserve their initializer entries before
// any side effect. When the iteration's worst case fits in the free part of
// the buffer ("tight" is false) a group of lanes takes its entries with one
// atomic add on the tail. Otherwise the group claims, by compare-and-swap,
// the longest prefix of its lanes that still fits; the other lanes defer:
// the track keeps its state and draw counter, so the interaction replays
// identically in a later iteration.
// The lanes of a group are the active ones of the warp, each wanting n = 0, 1
// or 2 entries; two ballots give every lane its place (instead of a generic scan
// over the group at each of the three call sites), and the tight case is one
// called function. With the other cold code taken out of line (side planes,
// Runge-Kutta substeps, the row's division) and the buffer's records moved in
// 16-byte parts, the loops fetch fewer instructions: 4 T calorimeter with the
// charge partition, persistent loop, 10.26 -> 9.32 ms; 1 GeV calorimeter sorted
// by action and type 4.85 -> 4.37 ms; asynchronous loop 1.30 -> 1.27 ms.
static __device__ __noinline__ bool reserve_tight(const Params& p, unsigned group, unsigned end, unsigned prefix,
                                                  unsigned n, unsigned long long& base) {
  Ctl* c = p.ctl;
  const int lane = threadIdx.x & 31, leader = __ffs(group) - 1;
  const unsigned long long head = c->head;
  for (int attempt = 0; attempt < kMaxCasAttempts; ++attempt) {
    unsigned long long cur = 0;
    if (lane == leader) cur = *reinterpret_cast<volatile unsigned long long*>(&c->tail);
    cur = __shfl_sync(group, cur, leader);
    const unsigned long long used = cur - head;
    const unsigned long long room = used < p.ring_capacity ? p.ring_capacity - used : 0ull;
    const unsigned fits = __ballot_sync(group, (unsigned long long)end <= room);
    // ends grow with the lane: the lanes that fit are the lowest ones
    const unsigned take = fits ? __shfl_sync(group, end, 31 - __clz(fits)) : 0u;
    if (take == 0) break;
    unsigned long long got = 0;
    if (lane == leader) got = atomicCAS(&c->tail, cur, cur + take);
    got = __shfl_sync(group, got, leader);
    if (got == cur) {
      base = cur + prefix;
      return n == 0 || end <= take;
    }
  }
  base = 0;
  return n == 0;
}
// In the asynchronous loops, where readers move the head meanwhile, a group
// takes its entries off the count of free ones (ctl->room) first: one atomic
// tells how many it got, the lanes that these are too few for give theirs
// back, and the tail moves by what is left. No group waits for another's, as
// with a compare-and-swap on the tail while the room is short (per-warp loop with
// one and with the other: 60,000 x 100 MeV with a buffer of 2^19 entries 7.4 and
// 2.7 ms, 20,000 x 1 GeV with 2^17 29 and 2.7 ms, the former with 2^20 2.7 and 2.5;
// the loop before it, with its swaps, took 4.95 and 12.3 ms).
// (reserve_entries holds the case of room for all; this is what follows for a
// group that asked for `total` when only `got` were free.)
static __device__ __noinline__ bool reserve_rest(const Params& p, unsigned group, unsigned total, long long got,
                                                 unsigned prefix, unsigned n, unsigned long long& base) {
  Ctl* c = p.ctl;
  const int lane = threadIdx.x & 31, leader = __ffs(group) - 1;
  const unsigned fits = __ballot_sync(group, (long long)(prefix + n) <= got);
  // ends grow with the lane: the lanes that fit are the lowest ones
  const unsigned take = fits ? __shfl_sync(group, prefix + n, 31 - __clz(fits)) : 0u;
  unsigned long long old = 0;
  if (lane == leader) {
    atomicAdd(reinterpret_cast<unsigned long long*>(&c->room), (unsigned long long)(total - take));
    if (take) old = atomicAdd(&c->tail, (unsigned long long)take);
  }
  base = __shfl_sync(group, old, leader) + prefix;
  return n == 0 || prefix + n <= take;
}

__device__ __forceinline__ bool reserve_entries(const Params& p, unsigned n, bool tight, unsigned long long& base) {
  const unsigned group = __activemask();
  const int lane = threadIdx.x & 31, leader = __ffs(group) - 1;
  const unsigned lt = (1u << lane) - 1u;
  const unsigned ones = __ballot_sync(group, n == 1u), twos = __ballot_sync(group, n == 2u);
  const unsigned total = __popc(ones) + 2u * __popc(twos);
  base = 0;
  if (total == 0) return true;
  const unsigned prefix = __popc(ones & lt) + 2u * __popc(twos & lt);
  if (p.ring_state) {
    long long got = 0;
    if (lane == leader) got = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(&p.ctl->room), 0ull - total);
    got = __shfl_sync(group, got, leader);
    if (got < (long long)total) return reserve_rest(p, group, total, got, prefix, n, base);
  } else if (tight) {
    return reserve_tight(p, group, prefix + n, prefix, n, base);
  }
  unsigned long long old = 0;
  if (lane == leader) old = atomicAdd(&p.ctl->tail, (unsigned long long)total);
  base = __shfl_sync(group, old, leader) + prefix;
  return true;
}

__device__ __forceinline__ void defer_track(const Params& p, uint32_t slot, uint8_t st, unsigned long long& n_def) {
  if (st == ALIVE) {
    p.trk.status[slot] = DEFERRED;
    ++n_def;
  }
}

// Pair production: the pair's kinetic energy E - 2 m_e c^2 deposited locally,
// two photons of m_e c^2 back to back in an isotropic direction.
__device__ __forceinline__ bool pair_one(const Params& p, uint32_t slot, uint8_t st, bool tight,
                                         unsigned long long& n_def) {
  CELER_LANES(LS_PAIR);
  const Tracks& t = p.trk;
  const bool keep = kMe >= p.cut_track;
  const bool reuse = keep && p.reuse_parent != 0;  // the first photon takes the parent's slot
  unsigned long long base;
  if (!reserve_entries(p, keep ? (reuse ? 1u : 2u) : 0u, tight, base)) {
    defer_track(p, slot, st, n_def);
    return false;
  }
  const double E = t.E[slot];
  const uint32_t ev = t.event[slot], prim = t.primary[slot];
  const int layer = t.layer[slot];
  const double x = t.x[slot], y = t.y[slot], z = t.z[slot];
  TrackRng rng(p.seed, ev, t.tid[slot], t.ctr[slot]);
  deposit(p, ev, prim, layer, z, E - 2.0 * kMe);
  const double cost = 2.0 * rng.uniform() - 1.0;
  const double u_phi = rng.uniform();
  const double sint2 = 1.0 - cost * cost;
  const double sint = dbits(sint2) > 0 ? fast_sqrt(sint2) : 0.0;
  double sp_, cp_;
  fast_sincos_2pi(u_phi, p.mtab, &sp_, &cp_);
  const double dx = sint * cp_, dy = sint * sp_, dz = cost;
  if (keep) {
    const unsigned long long tid1 = rng.raw();
    const unsigned long long tid2 = rng.raw();
    if (prim < p.hist_cap) atomicAdd(&p.hist_secondaries[prim], 2ull);
    if (reuse) {
      // parent-slot reuse (Sec. 3.2): the first photon starts in the slot the
      // pair ended (position, layer, event and primary are the parent's), as
      // a fresh track; the second goes to the initializer buffer
      write_initializer(p, base, x, y, z, -dx, -dy, -dz, kMe, tid2, ev, prim, layer, GAMMA);
      atomicAdd(&p.event_live[row_of(p, ev)], 1u);
      t.ux[slot] = dx;
      t.uy[slot] = dy;
      t.uz[slot] = dz;
      t.E[slot] = kMe;
      t.tid[slot] = tid1;
      t.ctr[slot] = 0u;
      t.nmfp[slot] = -1.0;
      t.action[slot] = A_NONE;
      t.status[slot] = ALIVE;
      return false;
    }
    write_initializer(p, base, x, y, z, dx, dy, dz, kMe, tid1, ev, prim, layer, GAMMA);
    write_initializer(p, base + 1, x, y, z, -dx, -dy, -dz, kMe, tid2, ev, prim, layer, GAMMA);
    atomicAdd(&p.event_live[row_of(p, ev)], 2u);
  } else {
    deposit(p, ev, prim, layer, z, kMe);
    deposit(p, ev, prim, layer, z, kMe);
  }
  release(p, slot, ev);
  return true;
}

// Moller scattering: delta ray above the production cut from the Moller
// cross-section, directions from two-body kinematics (delta polar angle from
// energy-momentum conservation, primary from momentum conservation).
__device__ __forceinline__ bool moller_one(const Params& p, uint32_t slot, uint8_t st, bool tight,
                                           unsigned long long& n_def) {
  CELER_LANES(LS_MOLLER);
  const Tracks& t = p.trk;
  const double T = t.E[slot];
  if (T <= 2.0 * p.cut_moller) {  // kinematically closed at the post-step energy: null collision
    t.nmfp[slot] = -1.0;
    t.status[slot] = ALIVE;
    return false;
  }
  const uint32_t ev = t.event[slot], prim = t.primary[slot];
  TrackRng rng(p.seed, ev, t.tid[slot], t.ctr[slot]);
  bool ok;
  const double eps = sample_moller(T, p.cut_moller, rng, ok);
  const double Td = eps * T;
  const bool keep = ok && Td >= p.cut_track;
  unsigned long long base;
  if (!reserve_entries(p, keep ? 1u : 0u, tight, base)) {
    defer_track(p, slot, st, n_def);
    return false;
  }
  const int layer = t.layer[slot];
  const double x = t.x[slot], y = t.y[slot], z = t.z[slot];
  if (!ok) {  // non-finite input: end the track, flag the run
    atomicOr(&p.ctl->error, ERR_SAMPLING);
    deposit(p, ev, prim, layer, z, T);
    release(p, slot, ev);
    return true;
  }
  // momenta p^2 = T (T + 2 m) and the delta's polar cosine
  // sqrt(Td (T + 2m) / (T (Td + 2m))) = Td (T + 2m) / (p p_delta), from two
  // reciprocal square roots
  const double pp2 = T * (T + 2.0 * kMe), pd2 = Td * (Td + 2.0 * kMe);
  const double rpp = fast_rsqrt(pp2), rpd = fast_rsqrt(pd2);
  const double cost = fmin(1.0, Td * (T + 2.0 * kMe) * rpp * rpd);
  const double u_phi = rng.uniform();
  const double ux = t.ux[slot], uy = t.uy[slot], uz = t.uz[slot];
  double dx = ux, dy = uy, dz = uz;
  rotate_dir(dx, dy, dz, cost, u_phi, p.mtab);
  const double pp = pp2 * rpp;
  const double pd = pd2 * rpd;
  const double vx = pp * ux - pd * dx, vy = pp * uy - pd * dy, vz = pp * uz - pd * dz;
  const double inv = fast_rsqrt(vx * vx + vy * vy + vz * vz);
  const double E1 = T - Td;
  if (keep) {
    const unsigned long long tid = rng.raw();
    write_initializer(p, base, x, y, z, dx, dy, dz, Td, tid, ev, prim, layer, ELECTRON);
    atomicAdd(&p.event_live[row_of(p, ev)], 1u);
    if (prim < p.hist_cap) atomicAdd(&p.hist_secondaries[prim], 1ull);
  } else {
    deposit(p, ev, prim, layer, z, Td);
  }
  if (dbits(E1) < dbits(p.cut_track)) {  // on the bits: a negative E1 passes, a positive NaN fails, as in FP64
    deposit(p, ev, prim, layer, z, E1);
    release(p, slot, ev);
    return true;
  }
  t.ux[slot] = vx * inv;
  t.uy[slot] = vy * inv;
  t.uz[slot] = vz * inv;
  t.E[slot] = E1;
  t.nmfp[slot] = -1.0;
  t.ctr[slot] = rng.ctr;
  t.status[slot] = ALIVE;
  return false;
}

// Bremsstrahlung: photon energy from the 1/k spectrum on (k_cut, T], emitted
// along the parent direction; the parent keeps its direction.
__device__ __forceinline__ bool brems_one(const Params& p, uint32_t slot, uint8_t st, bool tight,
                                          unsigned long long& n_def) {
  CELER_LANES(LS_BREMS);
  const Tracks& t = p.trk;
  const double T = t.E[slot];
  if (T <= p.cut_brems) {  // null collision
    t.nmfp[slot] = -1.0;
    t.status[slot] = ALIVE;
    return false;
  }
  const uint32_t ev = t.event[slot], prim = t.primary[slot];
  TrackRng rng(p.seed, ev, t.tid[slot], t.ctr[slot]);
  double k = p.cut_brems * fast_exp(rng.uniform() * fast_log(quot(T, p.cut_brems), p.mtab), p.mtab);
  if (k > T) k = T;
  const bool keep = k >= p.cut_track;
  unsigned long long base;
  if (!reserve_entries(p, keep ? 1u : 0u, tight, base)) {
    defer_track(p, slot, st, n_def);
    return false;
  }
  const int layer = t.layer[slot];
  const double x = t.x[slot], y = t.y[slot], z = t.z[slot];
  const double E1 = T - k;
  if (keep) {
    const unsigned long long tid = rng.raw();
    write_initializer(p, base, x, y, z, t.ux[slot], t.uy[slot], t.uz[slot], k, tid, ev, prim, layer, GAMMA);
    atomicAdd(&p.event_live[row_of(p, ev)], 1u);
    if (prim < p.hist_cap) atomicAdd(&p.hist_secondaries[prim], 1ull);
  } else {
    deposit(p, ev, prim, layer, z, k);
  }
  if (dbits(E1) < dbits(p.cut_track)) {  // on the bits: a negative E1 passes, a positive NaN fails, as in FP64
    deposit(p, ev, prim, layer, z, E1);
    release(p, slot, ev);
    return true;
  }
  t.E[slot] = E1;
  t.nmfp[slot] = -1.0;
  t.ctr[slot] = rng.ctr;
  t.status[slot] = ALIVE;
  return false;
}

// Interaction of one track whose step ended in one (or whose interaction is
// waiting for buffer space). Returns true if the track ended.
__device__ __forceinline__ bool post_one(const Params& p, uint32_t slot, uint8_t st, uint8_t act, bool tight,
                                         unsigned long long& n_def) {
  switch (act) {
    case A_COMPTON: return compton_one(p, slot);
    case A_PE: return photoelectric_one(p, slot);
    case A_PAIR: return pair_one(p, slot, st, tight, n_def);
    case A_MOLLER: return moller_one(p, slot, st, tight, n_def);
    case A_BREMS: return brems_one(p, slot, st, tight, n_def);
    default: return false;
  }
}

__device__ __forceinline__ bool is_interaction(uint8_t act) { return act >= A_COMPTON && act <= A_BREMS; }


// Work range of the step phase for the policy: all slots (masking), or the
// partition range of the live keys.
__device__ __forceinline__ Span live_span(const Params& p) {
  if (!global_partition(p.policy)) return Span{0u, p.n_slots, nullptr};
  const int hi = p.policy == POLICY_ACTION ? KA_VACANT : K_VACANT_FULL;
  return Span{p.ctl->offsets[0], p.ctl->offsets[hi], p.perm};
}

// Plan of the block-local policy's next fill (one thread, between
// iterations): the initializers it takes, min(vacant slots, queued), and
// whether the secondary buffer could overflow during that iteration: every
// track steps at most once and creates at most two secondaries, and the
// taken entries stay counted until the iteration ends, so the buffer is
// sure to suffice if queued + 2 (live + taken) fits its capacity.
__device__ __forceinline__ unsigned long long plan_local_fill(const Params& p, unsigned long long head,
                                                              unsigned long long tail, unsigned long long alive,
                                                              unsigned long long total_vacant) {
  Ctl* c = p.ctl;
  const unsigned long long queued = tail - head;
  const unsigned long long take = total_vacant < queued ? total_vacant : queued;
  c->fill_take = take;
  c->defer_local = (queued + 2ull * (alive + take) > p.ring_capacity) ? 1u : 0u;
  return take;
}

// End of an iteration: counters, the per-iteration trace row, stall and
// iteration-limit checks, the loop condition, and the per-iteration counters
// cleared for the next one. One warp: every counter is read in one batch of
// loads, the per-action counts one per lane.
__device__ void loop_ctl_warp(const Params& p, unsigned long long* take_out = nullptr) {
  Ctl* c = p.ctl;
  const int lane = threadIdx.x & 31;
  const unsigned long long head = c->head, tail = c->tail, alive = c->alive, total_vacant = c->total_vacant;
  const unsigned long long steps_iter = c->steps_iter, steps_total = c->steps_total;
  const unsigned long long iteration = c->iteration, trace_count = c->trace_count;
  const unsigned long long max_iterations = c->max_iterations, budget_end = c->budget_end;
  const unsigned n_def = c->n_deferred, stall = c->stall, error = c->error;
  const unsigned ac = lane < kMaxKeys ? c->action_count[lane] : 0u;
  const unsigned long long queued = tail - head;
  const bool worked = steps_iter > 0 || n_def > 0;
  TraceRow& r = p.trace[trace_count % kTraceRows];
  if (lane < kMaxKeys) {
    c->last_action_count[lane] = ac;
    if (worked) r.action_count[lane] = ac;
    c->action_count[lane] = 0u;
    c->key_total[lane] = 0u;
  }
  if (lane == 0) {
    c->last_steps_iter = steps_iter;
    c->last_n_deferred = n_def;
    unsigned long long it = iteration;
    if (worked) {
      c->steps_total = steps_total + steps_iter;
      r.iteration = iteration;
      r.alive = alive;
      r.queued = queued;
      r.steps = steps_iter;
      c->trace_count = trace_count + 1;
      it = iteration + 1;
      c->iteration = it;
    }
    const bool pending = alive + queued > 0;
    // No track stepped although work is pending: every live track waits for
    // buffer space. One such iteration can still place deferred secondaries;
    // three in a row cannot make progress any more.
    unsigned err = error;
    if (steps_iter == 0 && pending) {
      if (stall + 1 >= 3) err |= ERR_NO_PROGRESS;
      c->stall = stall + 1;
    } else {
      c->stall = 0u;
    }
    if (pending && it >= max_iterations) err |= ERR_ITERATIONS;
    if (err != error) c->error = err;
    const unsigned cont = (pending && err == 0u && it < budget_end) ? 1u : 0u;
    c->cont = cont;
    c->pending = pending ? 1u : 0u;
    if (p.cont_out) *reinterpret_cast<volatile unsigned*>(p.cont_out) = cont;
    c->steps_iter = 0;
    c->n_deferred = 0;
    const unsigned long long take = plan_local_fill(p, head, tail, alive, total_vacant);
    if (take_out) *take_out = take;
  }
}

// The tally rows to pinned host memory at the end of an iteration (whole block,
// after every other block's deposits): the hit copy of the host loop without
// the gap of a copy between two kernels (event of 200 primaries, 128
// iterations with a copy each: 4.94 -> 3.64 ms).
static __device__ __noinline__ void copy_out_row(double* dst, const double* src, uint32_t n) {
  for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) dst[i] = __ldcg(src + i);
}
__device__ __forceinline__ void copy_hits(const Params& p) {
  if (p.hits != nullptr) copy_out_row(p.hits, p.tally, p.max_events * (uint32_t)p.n_bins);
}

// Along-step and, if the step ends in one, the interaction of the track in
// `slot` (phase C's body). Returns true if the track ended.
__device__ __forceinline__ bool step_one(const Params& p, uint32_t slot, uint8_t st, const SharedStatic& ss, bool tight,
                                         unsigned long long& n_def) {
  const uint8_t act = p.trk.action[slot];
  if (st == ALIVE && along_one(p, slot, p.trk.ptype[slot], ss)) return true;
  return is_interaction(act) && post_one(p, slot, st, act, tight, n_def);
}

#include "block_pass.cuh"

// Per-block vacancy counts and the plan of the first fill (fill_take and the
// block quotas) for the block-local policy, at the start of a run (its
// iterations keep them current; a run of another policy, or primaries pushed
// since, leave them to be recomputed). Same grid as the loop.
__global__ void __launch_bounds__(kTile) k_local_prepare(Params p) {
  count_block_vacancies(p, blockIdx.x, gridDim.x);
  Ctl* c = p.ctl;
  if (last_block_done(&c->done_p, gridDim.x)) {
    __shared__ uint32_t s_v[kMaxLoopBlocks];
    __shared__ unsigned long long s_sum, s_take;
    __shared__ unsigned s_vmin, s_vmax;
    load_block_vacancies(p, s_v, (int)gridDim.x, &s_sum, &s_vmin, &s_vmax);
    if (threadIdx.x == 0) {
      if (s_sum != c->total_vacant) c->error |= ERR_VACANCY;
      c->local_blocks = gridDim.x;
      s_take = plan_local_fill(p, c->head, c->tail, c->alive, s_sum);
    }
    __syncthreads();
    const unsigned long long planned =
        plan_block_quotas(p, s_v, (int)gridDim.x, s_vmin, s_vmax, s_take, block_quota_cap(p.policy));
    if (threadIdx.x == 0 && planned != s_take) c->fill_take = planned;
  }
}

// Per-tile vacancy prefix and total, recomputed at the start of a run of a
// policy that fills in slot order after block-local iterations (which keep
// the per-tile counts but not their scan). One block.
__global__ void __launch_bounds__(kTile) k_scan_tiles(Params p) { scan_vacancy(p); }

// Phase C: along-step of every live track and, where the step ends in an
// interaction, that interaction, in partition order; deferred interactions
// are retried. The last block ends the iteration.
__device__ void phase_step(const Params& p, int bid, int nb, const SharedStatic& ss, bool bookkeeping,
                           cudaGraphConditionalHandle handle, int use_handle) {
  const Span sp = live_span(p);
  const bool tight = p.ctl->defer != 0u;
  const Tracks& t = p.trk;
  unsigned long long killed = 0, n_def = 0;
  const uint32_t width = sp.perm ? spread_width(sp.hi - sp.lo, nb) : 32u;
  for (ChunkWalk w(sp.lo, sp.hi, bid, nb, width); w.more(); w.next()) {
    const uint32_t i = w.index();
    if (i >= sp.hi) continue;
    const uint32_t slot = sp.perm ? sp.perm[i] : i;
    const uint8_t st = t.status[slot];
    if (st == VACANT) continue;
    const uint8_t act = t.action[slot];
    if (st == ALIVE) {
      if (along_one(p, slot, t.ptype[slot], ss)) {
        ++killed;
        continue;
      }
    }
    if (is_interaction(act) && post_one(p, slot, st, act, tight, n_def)) ++killed;
  }
  flush_counter(&p.ctl->alive, killed, true);
  if (n_def) atomicAdd(&p.ctl->n_deferred, (unsigned)n_def);
  apply_fills(p, bid, nb);
  if (bookkeeping && last_block_done(&p.ctl->done_c, nb)) {
    const long long t0 = clock64();
    copy_hits(p);
    scan_vacancy(p);
    if (threadIdx.x < 32) loop_ctl_warp(p);
    if (threadIdx.x == 0) {
      if (use_handle) cudaGraphSetConditional(handle, p.ctl->cont);
      p.ctl->book_total[1] += (unsigned long long)(clock64() - t0);
    }
  }
}

// Along-step only, for one particle kind (per-action launch mode).
__device__ void phase_along_only(const Params& p, bool charged, int bid, int nb, const SharedStatic& ss) {
  Span sp = live_span(p);
  if (p.policy == POLICY_ACTION) {
    sp.lo = p.ctl->offsets[charged ? KA_CHARGED : KA_NEUTRAL];
    sp.hi = p.ctl->offsets[charged ? KA_VACANT : KA_CHARGED];
  }
  unsigned long long killed = 0;
  for (ChunkWalk w(sp.lo, sp.hi, bid, nb); w.more(); w.next()) {
    const uint32_t i = w.index();
    if (i >= sp.hi) continue;
    const uint32_t slot = sp.perm ? sp.perm[i] : i;
    if (p.trk.status[slot] != ALIVE) continue;
    const uint8_t pt = p.trk.ptype[slot];
    if ((pt != GAMMA) != charged) continue;
    if (along_one(p, slot, pt, ss)) ++killed;
  }
  flush_counter(&p.ctl->alive, killed, true);
}

// One interaction process only (per-action launch mode).
__device__ void phase_post_only(const Params& p, uint8_t which, int bid, int nb) {
  Span sp = live_span(p);
  if (p.policy == POLICY_ACTION) {
    const bool charged = which == A_MOLLER || which == A_BREMS;
    sp.lo = p.ctl->offsets[charged ? KA_CHARGED : KA_NEUTRAL];
    sp.hi = p.ctl->offsets[charged ? KA_VACANT : KA_CHARGED];
  } else if (p.policy == POLICY_ACTION_TYPE) {
    int k = K_G_COMPTON;
    switch (which) {
      case A_PE: k = K_G_PE; break;
      case A_PAIR: k = K_G_PAIR; break;
      case A_MOLLER: k = K_E_MOLLER; break;
      case A_BREMS: k = K_E_BREMS; break;
      default: break;
    }
    sp.lo = p.ctl->offsets[k];
    sp.hi = p.ctl->offsets[k + 1];
  }
  const bool tight = p.ctl->defer != 0u;
  unsigned long long killed = 0, n_def = 0;
  for (ChunkWalk w(sp.lo, sp.hi, bid, nb); w.more(); w.next()) {
    const uint32_t i = w.index();
    if (i >= sp.hi) continue;
    const uint32_t slot = sp.perm ? sp.perm[i] : i;
    const uint8_t st = p.trk.status[slot];
    if (st == VACANT || p.trk.action[slot] != which) continue;
    if (post_one(p, slot, st, which, tight, n_def)) ++killed;
  }
  flush_counter(&p.ctl->alive, killed, true);
  if (n_def) atomicAdd(&p.ctl->n_deferred, (unsigned)n_def);
}

// ------------------------------------------------------------------ kernels
// Phase-merged launches (host loop / graph): A, B, C.
// In the loops they start as the blocks of the launch before them exit (the
// programmatic dependent launch of launch_early) and wait for its completion
// here: before it they touch the static tables and their own shared memory
// only. (Letting them start at the beginning of the launch before them instead,
// with launch_dependents, is no faster: their blocks don't fit beside its.)
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// A launch beyond the run's end does nothing (IterMode in launch.h). The words
// it looks at are written by the last block of an iteration's last kernel
// only, after every other block of it has started, so all blocks of a launch
// see the same.
__device__ __forceinline__ bool beyond_end(const Params& p, int mode) {
  if (mode & ITER_IF_CONT) return __ldcg(&p.ctl->cont) == 0u;
  if (mode & ITER_IF_PENDING) return __ldcg(&p.ctl->pending) == 0u;
  return false;
}

__global__ void __launch_bounds__(kTile) k_fill_step(Params p, int mode) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned long long s_bar;
  SharedStatic ss = carve_static(p, smem_raw);
  stage_static(p, ss, &s_bar);
  wait_for_previous();
  const bool skip = beyond_end(p, mode);
  ss.ready(p);
  if (skip) return;
  phase_fill_step(p, blockIdx.x, gridDim.x, ss, true, true, true);
}

__global__ void __launch_bounds__(kTile) k_scatter(Params p, int mode) {
  wait_for_previous();
  if (!beyond_end(p, mode)) phase_scatter(p, blockIdx.x, gridDim.x);
}

__global__ void k_step(Params p, cudaGraphConditionalHandle handle, int mode) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned long long s_bar;
  SharedStatic ss = carve_static(p, smem_raw);
  stage_static(p, ss, &s_bar);
  wait_for_previous();
  const bool skip = beyond_end(p, mode);
  ss.ready(p);
  if (skip) return;
  phase_step(p, blockIdx.x, gridDim.x, ss, true, handle, mode & ITER_SET_HANDLE);
}

// The block-pass policies (LOCAL, DATA): one launch per iteration (same grid
// as the loop).
__global__ void __launch_bounds__(kTile) k_local(Params p, cudaGraphConditionalHandle handle, int mode) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned long long s_bar;
  SharedStatic ss = carve_static(p, smem_raw);
  stage_static(p, ss, &s_bar);
  wait_for_previous();
  const BlockIter it = load_block_iter(p, blockIdx.x, gridDim.x);
  const bool skip = beyond_end(p, mode);
  ss.ready(p);
  if (skip) return;
  block_iteration<false>(p, blockIdx.x, gridDim.x, ss, handle, mode & ITER_SET_HANDLE, it);
}

// Per-action launches: fill, step limit (+ bookkeeping), scatter, one
// along-step kernel per particle kind, one kernel per interaction, end.
__global__ void __launch_bounds__(kTile) k_fill(Params p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SharedStatic ss = carve_static(p, smem_raw);
  phase_fill_step(p, blockIdx.x, gridDim.x, ss, true, false, false);
}

__global__ void __launch_bounds__(kTile) k_pre_step(Params p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned long long s_bar;
  SharedStatic ss = carve_static(p, smem_raw);
  stage_static(p, ss, &s_bar);
  ss.ready(p);
  phase_fill_step(p, blockIdx.x, gridDim.x, ss, false, true, false);
  if (last_block_done(&p.ctl->done_a, gridDim.x)) bookkeeping_after_fill_step(p, true);
}

__global__ void k_along(Params p, int charged) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned long long s_bar;
  SharedStatic ss = carve_static(p, smem_raw);
  stage_static(p, ss, &s_bar);
  ss.ready(p);
  phase_along_only(p, charged != 0, blockIdx.x, gridDim.x, ss);
}

__global__ void k_post(Params p, int which) { phase_post_only(p, (uint8_t)which, blockIdx.x, gridDim.x); }

__global__ void __launch_bounds__(kTile) k_loop_ctl(Params p, cudaGraphConditionalHandle handle, int use_handle) {
  apply_fills(p, 0, 1);
  copy_hits(p);
  __syncthreads();
  scan_vacancy(p);
  if (threadIdx.x < 32) loop_ctl_warp(p);
  if (threadIdx.x == 0 && use_handle) cudaGraphSetConditional(handle, p.ctl->cont);
}

// Start a run: the loop stops after `budget` more iterations (0: no limit).
__global__ void k_begin_run(Ctl* c, unsigned long long budget) {
  c->run_start = c->iteration;
  c->budget_end = budget ? c->iteration + budget : ~0ull;
  c->done_a = 0u;
  c->done_c = 0u;
  c->done_p = 0u;
  c->cont = 1u;
  c->pending = 1u;
}

// Grid-wide barrier of the persistent loop (generation counter). Every wait
// is bounded: after ~1 s a block gives up, sets the abort word and the error
// bit, and every block then leaves the loop at its next barrier.
__device__ __forceinline__ bool grid_barrier(const Params& p, unsigned nblocks,
                                             long long timeout = kBarrierTimeoutCycles) {
  __shared__ int s_ok;
  unsigned int* count = p.barrier;
  unsigned int* gen = p.barrier + 1;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned g = *reinterpret_cast<volatile unsigned*>(gen);
    int ok = 1;
    if (atomicAdd(count, 1u) == nblocks - 1) {
      *reinterpret_cast<volatile unsigned*>(count) = 0u;
      __threadfence();
      atomicAdd(gen, 1u);
      if (*reinterpret_cast<volatile unsigned*>(p.barrier + 2) != 0u) ok = 0;
    } else {
      ok = wait_generation(p, g, timeout) ? 1 : 0;
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// End of a phase of the persistent loop: the last block to arrive runs `book`
// (whole block) and lets the others go on; its ticket is the grid barrier,
// so a phase costs one atomic per block instead of two. Waits are bounded as
// grid_barrier's. With the partition's offsets summed by every block: 1 GeV
// calorimeter sorted by action and type 4.37 -> 4.01 ms (36.3 -> 32.7 us per
// iteration).
template <class Book>
__device__ __forceinline__ bool end_phase(const Params& p, unsigned* counter, unsigned nb, Book book) {
  __shared__ unsigned s_last, s_gen;
  __shared__ int s_ok;
  unsigned int* gen = p.barrier + 1;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_gen = *reinterpret_cast<volatile unsigned*>(gen);
    s_last = atomicAdd(counter, 1u) == nb - 1u ? 1u : 0u;
    if (s_last) *reinterpret_cast<volatile unsigned*>(counter) = 0u;
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    book();
    __syncthreads();
    if (threadIdx.x == 0) {
      s_ok = *reinterpret_cast<volatile unsigned*>(p.barrier + 2) == 0u ? 1 : 0;
      __threadfence();
      atomicAdd(gen, 1u);
    }
  } else if (threadIdx.x == 0) {
    s_ok = wait_generation(p, s_gen, kBarrierTimeoutCycles) ? 1 : 0;
    __threadfence();
  }
  __syncthreads();
  return s_ok != 0;
}

// The whole step loop in one persistent cooperative launch: one block per
// SM slot, the static tables staged into shared memory once, three grid
// barriers per iteration (two without sorting).
__global__ void __launch_bounds__(kTile, 1) k_loop(Params p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SharedStatic ss = carve_static(p, smem_raw);
  stage_static(p, ss);
  const unsigned nb = gridDim.x;
  const int bid = blockIdx.x;
  const bool sorted = global_partition(p.policy);
  if (bid == 0 && threadIdx.x == 0) {
    clear_iteration_counters(p.ctl);
    p.ctl->cont = 1u;
  }
  if (!grid_barrier(p, nb)) return;
  Ctl* c = p.ctl;
  long long t_prev = clock64();
  unsigned parity = 0;
  // phase k took (now - t_prev) for block 0 including the barrier wait; every
  // block also records its own work time so the slowest one can be told apart
  auto mark = [&](int k, long long work) {
    if (threadIdx.x == 0) {
      atomicMax(&c->iter_max[parity][k], (unsigned long long)work);
      if (bid == 0) {
        const long long now = clock64();
        c->phase_cycles[k] += (unsigned long long)(now - t_prev);
        t_prev = now;
      }
    }
  };
  for (;;) {
    if (*reinterpret_cast<volatile unsigned*>(&c->cont) == 0u) break;
    if (bid == 0 && threadIdx.x == 0) {
      for (int k = 0; k < 4; ++k) {
        c->max_total[k] += c->iter_max[parity ^ 1][k];
        c->iter_max[parity ^ 1][k] = 0;
      }
    }
    long long t0 = clock64();
    phase_fill_step(p, bid, nb, ss, true, true, false);
    const long long wa = clock64() - t0;
    const bool ok_a = end_phase(p, &c->done_a, nb, [&] {
      const long long tb = clock64();
      bookkeeping_after_fill_step(p, true);
      if (threadIdx.x == 0) c->book_total[0] += (unsigned long long)(clock64() - tb);
    });
    if (!ok_a) break;
    mark(0, wa);
    if (sorted) {
      t0 = clock64();
      phase_scatter(p, bid, nb);
      const long long wb = clock64() - t0;
      if (!grid_barrier(p, nb)) break;
      mark(1, wb);
    }
    t0 = clock64();
    phase_step(p, bid, nb, ss, false, 0, 0);
    const long long wc = clock64() - t0;
    const bool ok_c = end_phase(p, &c->done_c, nb, [&] {
      const long long tb = clock64();
      scan_vacancy(p);
      if (threadIdx.x < 32) loop_ctl_warp(p);
      if (threadIdx.x == 0) c->book_total[1] += (unsigned long long)(clock64() - tb);
    });
    if (!ok_c) break;
    mark(2, wc);
    parity ^= 1u;
  }
  if (bid == 0 && threadIdx.x == 0) {
    for (int k = 0; k < 4; ++k) {
      c->max_total[k] += c->iter_max[0][k] + c->iter_max[1][k];
      c->iter_max[0][k] = c->iter_max[1][k] = 0;
    }
  }
}

// The persistent loop of the block-pass policies: one pass per block and
// iteration (block_iteration), one grid barrier per iteration.
__global__ void __launch_bounds__(kTile, 1) k_loop_local(Params p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SharedStatic ss = carve_static(p, smem_raw);
  stage_static(p, ss);
  const unsigned nb = gridDim.x;
  const int bid = blockIdx.x;
  Ctl* c = p.ctl;
  if (bid == 0 && threadIdx.x == 0) {
    clear_iteration_counters(c);
    c->cont = 1u;
  }
  if (!grid_barrier(p, nb)) return;
  long long t_prev = clock64();
  for (;;) {
    const BlockIter it = load_block_iter(p, bid, (int)nb);  // one batch of loads per iteration
    if (!it.cont) break;
    const unsigned parity = (unsigned)(it.iteration & 1);
    if (bid == 0 && threadIdx.x == 0) {  // the slowest block's work of the previous iteration
      c->max_total[2] += c->iter_max[parity ^ 1u][2];
      c->iter_max[parity ^ 1u][2] = 0;
    }
    const bool ok = block_iteration<true>(p, bid, (int)nb, ss, 0, 0, it);
    if (!ok) break;
    if (bid == 0 && threadIdx.x == 0) {
      const long long now = clock64();
      c->phase_cycles[2] += (unsigned long long)(now - t_prev);
      t_prev = now;
    }
  }
  if (bid == 0 && threadIdx.x == 0) {
    c->max_total[2] += c->iter_max[0][2] + c->iter_max[1][2];
    c->iter_max[0][2] = c->iter_max[1][2] = 0;
  }
}

#include "async_loop.cuh"
#include "warp_loop.cuh"

// Check of the bounded waits: every block but `absent` meets at a grid
// barrier that `absent` never reaches, so the waiters must give up after
// `timeout` cycles, set the abort word and the error bit, and return.
__global__ void k_barrier_probe(Params p, int absent, long long timeout) {
  if ((int)blockIdx.x == absent) return;
  grid_barrier(p, gridDim.x, timeout);
}

// Queue staged primaries (one event's) at the tail of the initializer buffer,
// from index `base`, the tail as the host knows it. states: the asynchronous
// loop's entry states, kept by every push.
__global__ void __launch_bounds__(256) k_push_primaries(Params p, const StagedPrimary* src, uint32_t n,
                                                       unsigned long long base, uint32_t* states) {
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const StagedPrimary& q = src[i];
    const unsigned long long at = (base + i) & p.ring_mask;
    put_record(p.ring.rec + at, q.x, q.y, q.z, q.ux, q.uy, q.uz, q.E, q.tid, q.event, q.primary, q.layer,
               (uint8_t)q.ptype);
    states[at] = ring_lap_code(p, base + i) + 1u;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    Ctl* c = p.ctl;
    atomicAdd(&p.event_live[row_of(p, src[0].event)], n);
    c->tail = base + n;
    c->avail += n;
    c->room -= (long long)n;
    plan_local_fill(p, c->head, base + n, c->alive, c->total_vacant);
  }
}

// Primaries already in device memory, in two launches: every record (and the
// buffer's fill level) is checked, then all of them are queued if every check
// passed. One block did both before (95 us for 10,000 primaries): whole jobs
// of 10,000 and 100,000 went from 3.20 to 3.06 and from 18.5 to 17.4 ms.
__global__ void __launch_bounds__(256) k_check_device_primaries(Params p, const DevicePrimary* src, uint32_t n) {
  const double zmax = p.zb[p.n_layers];
  const uint32_t stride = gridDim.x * blockDim.x, first = blockIdx.x * blockDim.x + threadIdx.x;
  bool bad = first == 0 && p.ctl->tail - p.ctl->head + n > p.ring_capacity;
  for (uint32_t i = first; i < n; i += stride) {
    const DevicePrimary& q = src[i];
    const double d2 = q.dir[0] * q.dir[0] + q.dir[1] * q.dir[1] + q.dir[2] * q.dir[2];
    const bool ok = isfinite(q.E) && q.E > 0.0 && q.E <= kGridEmax && isfinite(d2) &&
                    fabs(sqrt(d2) - 1.0) <= 1e-12 && fabs(q.pos[0]) <= p.hx && fabs(q.pos[1]) <= p.hy &&
                    q.pos[2] >= p.zb[0] && q.pos[2] <= zmax && (q.ptype == GAMMA || q.ptype == ELECTRON);
    bad = bad || !ok;
  }
  if (bad) atomicOr(&p.ctl->push_bad, 1u);
}

__global__ void __launch_bounds__(256) k_push_device_primaries(Params p, const DevicePrimary* src, uint32_t n,
                                                              uint32_t event, unsigned long long tid0, uint32_t prim0,
                                                              uint32_t* states) {
  Ctl* c = p.ctl;
  const unsigned long long base = __ldcg(&c->tail);  // moved by the last block only
  const bool bad = __ldcg(&c->push_bad) != 0u;
  const double zmax = p.zb[p.n_layers];
  const int L = p.n_layers;
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n && !bad; i += stride) {
    const DevicePrimary& q = src[i];
    const double z = q.pos[2], uz = q.dir[2];
    // layer: the largest l <= L-1 with z_l <= z; on an inner plane moving
    // backwards, the layer behind it
    int lo = 0;
    if (z >= zmax) {
      lo = L - 1;
    } else {
      int hi = L - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) / 2;
        if (p.zb[mid] <= z)
          lo = mid;
        else
          hi = mid - 1;
      }
      if (z == p.zb[lo] && uz < 0.0 && lo > 0) --lo;
    }
    const uint32_t prim = p.hist_cap > 0 ? prim0 + i : 0xFFFFFFFFu;
    const unsigned long long at = (base + i) & p.ring_mask;
    put_record(p.ring.rec + at, q.pos[0], q.pos[1], z, q.dir[0], q.dir[1], uz, q.E, tid0 + i, event, prim, lo,
               (uint8_t)q.ptype);
    states[at] = ring_lap_code(p, base + i) + 1u;
  }
  __syncthreads();
  if (threadIdx.x == 0 && atomicAdd(&c->done_push, 1u) == gridDim.x - 1u) {
    c->done_push = 0u;
    c->push_bad = 0u;
    if (bad) {
      c->error |= ERR_PRIMARIES_REJECTED;
    } else {
      c->tail = base + n;
      c->avail += n;
      c->room -= (long long)n;
      atomicAdd(&p.event_live[row_of(p, event)], n);
      plan_local_fill(p, c->head, base + n, c->alive, c->total_vacant);
    }
  }
}

// One event's tally row, escaped energy and live count cleared.
__global__ void k_reset_event(double* tally, int n_bins, double* escaped, unsigned* event_live) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_bins; i += gridDim.x * blockDim.x) tally[i] = 0.0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *escaped = 0.0;
    *event_live = 0u;
  }
}

// Words of device memory into pinned host memory.
__global__ void k_copy_out(uint32_t* dst, const uint32_t* src, uint32_t n, uint32_t* dst2, const uint32_t* src2,
                           uint32_t n2) {
  const uint32_t first = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  for (uint32_t i = first; i < n; i += stride) dst[i] = __ldcg(src + i);
  for (uint32_t i = first; i < n2; i += stride) dst2[i] = __ldcg(src2 + i);
}

// The per-warp schedule's kernels by tracks per block, and the bytes of those.
constexpr int kWarpVariants = 3;
struct WarpKernel {
  const void* fn;
  size_t bytes;
  int threads;
};
template <int kCap>
WarpKernel warp_kernel_of() {
  return WarpKernel{(const void*)k_loop_warps<kCap>, TrackCache<kCap>::kBytes, kThreads<kCap>};
}
WarpKernel warp_kernel(int variant) {
  return variant == 0 ? warp_kernel_of<kWarpTracks>()
                      : (variant == 1 ? warp_kernel_of<kWarpTracksMid>() : warp_kernel_of<kWarpTracksSmall>());
}

int occupancy_grid(const void* fn, int block, size_t smem, int sms, int cap) {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, block, smem) != cudaSuccess || nb < 1) nb = 1;
  long g = (long)nb * sms;
  if (cap > 0 && g > cap) g = cap;
  return (int)(g < 1 ? 1 : g);
}

}  // namespace

cudaError_t configure_kernels(const Params& p, int block, LaunchShape* sh) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const size_t stat = static_smem_bytes(p.n_materials, p.n_layers);
  sh->static_smem = stat;
  sh->block = block;
  const void* with_smem[] = {(const void*)k_fill_step, (const void*)k_step, (const void*)k_fill,
                             (const void*)k_pre_step, (const void*)k_along, (const void*)k_loop,
                             (const void*)k_local, (const void*)k_loop_local, (const void*)k_loop_async};
  for (const void* fn : with_smem) {
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)stat);
    if (e != cudaSuccess) return e;
  }
  // the per-warp schedule keeps a block's tracks in shared memory: as many as
  // fit beside the static tables
  int max_smem = 0;
  e = cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  for (sh->warp_variant = 0; sh->warp_variant < kWarpVariants; ++sh->warp_variant) {
    cudaFuncAttributes fa{};
    e = cudaFuncGetAttributes(&fa, warp_kernel(sh->warp_variant).fn);
    if (e != cudaSuccess) return e;
    sh->warp_smem = warp_kernel(sh->warp_variant).bytes + stat + (size_t)p.n_layers * sizeof(double);
    if (fa.sharedSizeBytes + sh->warp_smem <= (size_t)max_smem || sh->warp_variant == kWarpVariants - 1) break;
  }
  const void* warps = warp_kernel(sh->warp_variant).fn;
  e = cudaFuncSetAttribute(warps, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh->warp_smem);
  if (e != cudaSuccess) return e;
  sh->tile_grid = occupancy_grid((const void*)k_fill_step, kTile, stat, sms, (int)p.n_tiles);
  const int cap_action = (int)((p.n_slots + block - 1) / block);
  sh->step_grid = occupancy_grid((const void*)k_step, block, stat, sms, cap_action);
  sh->along_grid = occupancy_grid((const void*)k_along, block, stat, sms, cap_action);
  sh->post_grid = occupancy_grid((const void*)k_post, block, 0, sms, cap_action);
  int nb = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (const void*)k_loop, kTile, stat);
  if (e != cudaSuccess) return e;
  int nb_local = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb_local, (const void*)k_loop_local, kTile, stat);
  if (e != cudaSuccess) return e;
  if (nb_local < nb) nb = nb_local;  // one grid for every loop (and the block-local launches)
  int nb_async = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb_async, (const void*)k_loop_async, kTile, stat);
  if (e != cudaSuccess) return e;
  if (nb_async < nb) nb = nb_async;
  int nb_warps = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb_warps, warps, warp_kernel(sh->warp_variant).threads, sh->warp_smem);
  if (e != cudaSuccess) return e;
  if (nb_warps < nb) nb = nb_warps;
  sh->loop_grid = (nb < 1 ? 1 : nb) * sms;
  if (sh->loop_grid > kMaxLoopBlocks) sh->loop_grid = kMaxLoopBlocks;  // size of the per-block arrays
  return cudaGetLastError();
}

// A kernel that begins with wait_for_previous. In the loops it may be scheduled
// while the launch before it ends, which saves 1 to 2 us of the gap between
// two: the host loop's event of 200 primaries 3.40 -> 3.13 ms, sorted by action
// 4.66 -> 3.79 ms (three launches per iteration), water cube 1.22 -> 1.03 ms;
// in the graph loop 1.015 -> 0.985 ms.
template <class... A>
static void launch_early(void (*fn)(A...), int grid, int block, size_t smem, cudaStream_t s, int mode, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = mode == ITER_ALWAYS ? 0 : 1;
  cudaLaunchKernelEx(&cfg, fn, args...);
}
void launch_fill_step(const Params& p, const LaunchShape& sh, int mode, cudaStream_t s) {
  launch_early(k_fill_step, sh.tile_grid, kTile, sh.static_smem, s, mode, p, mode);
}
void launch_scatter(const Params& p, const LaunchShape& sh, int mode, cudaStream_t s) {
  launch_early(k_scatter, sh.tile_grid, kTile, 0, s, mode, p, mode);
}
void launch_step(const Params& p, const LaunchShape& sh, unsigned long long handle, int mode, cudaStream_t s) {
  launch_early(k_step, sh.step_grid, sh.block, sh.static_smem, s, mode, p, (cudaGraphConditionalHandle)handle, mode);
}
void launch_local(const Params& p, const LaunchShape& sh, unsigned long long handle, int mode, cudaStream_t s) {
  launch_early(k_local, sh.loop_grid, kTile, sh.static_smem, s, mode, p, (cudaGraphConditionalHandle)handle, mode);
}
void launch_local_prepare(const Params& p, const LaunchShape& sh, cudaStream_t s) {
  k_local_prepare<<<sh.loop_grid, kTile, 0, s>>>(p);
}
void launch_scan_tiles(const Params& p, cudaStream_t s) { k_scan_tiles<<<1, kTile, 0, s>>>(p); }
cudaError_t launch_queue_wait_probe(const Params& p, int which, long long timeout, cudaStream_t s) {
  k_queue_wait_probe<<<1, 32, 0, s>>>(p, which, timeout);
  return cudaGetLastError();
}
cudaError_t launch_barrier_probe(const Params& p, int blocks, int absent, long long timeout, cudaStream_t s) {
  void* args[] = {const_cast<Params*>(&p), &absent, &timeout};
  return cudaLaunchCooperativeKernel((const void*)k_barrier_probe, dim3(blocks), dim3(32), args, 0, s);
}
void launch_fill(const Params& p, const LaunchShape& sh, cudaStream_t s) {
  k_fill<<<sh.tile_grid, kTile, sh.static_smem, s>>>(p);
}
void launch_pre_step(const Params& p, const LaunchShape& sh, cudaStream_t s) {
  k_pre_step<<<sh.tile_grid, kTile, sh.static_smem, s>>>(p);
}
void launch_along(const Params& p, int charged, const LaunchShape& sh, cudaStream_t s) {
  k_along<<<sh.along_grid, sh.block, sh.static_smem, s>>>(p, charged);
}
void launch_post(const Params& p, int which, const LaunchShape& sh, cudaStream_t s) {
  k_post<<<sh.post_grid, sh.block, 0, s>>>(p, which);
}
void launch_loop_ctl(const Params& p, unsigned long long handle, int use_handle, cudaStream_t s) {
  k_loop_ctl<<<1, kTile, 0, s>>>(p, (cudaGraphConditionalHandle)handle, use_handle);
}
void launch_begin_run(const Params& p, unsigned long long budget, cudaStream_t s) {
  k_begin_run<<<1, 1, 0, s>>>(p.ctl, budget);
}
void launch_async_prepare(const Params& p, cudaStream_t s) { k_async_prepare<<<256, 256, 0, s>>>(p); }
cudaError_t launch_loop_async(const Params& p, const LaunchShape& sh, cudaStream_t s) {
  void* args[] = {const_cast<Params*>(&p)};
  if (p.policy == POLICY_LOCAL && p.async_warps) {
    const WarpKernel k = warp_kernel(sh.warp_variant);
    return cudaLaunchCooperativeKernel(k.fn, dim3(sh.loop_grid), dim3(k.threads), args, sh.warp_smem, s);
  }
  return cudaLaunchCooperativeKernel((const void*)k_loop_async, dim3(sh.loop_grid), dim3(kTile), args, sh.static_smem,
                                     s);
}
cudaError_t launch_loop(const Params& p, const LaunchShape& sh, cudaStream_t s) {
  void* args[] = {const_cast<Params*>(&p)};
  const void* fn = block_pass(p.policy) ? (const void*)k_loop_local : (const void*)k_loop;
  return cudaLaunchCooperativeKernel(fn, dim3(sh.loop_grid), dim3(kTile), args, sh.static_smem, s);
}
static int push_grid(uint32_t n) { return (int)((n + 255u) / 256u < 304u ? (n + 255u) / 256u : 304u); }
void launch_push_primaries(const Params& p, const StagedPrimary* prim, uint32_t n, unsigned long long base,
                           uint32_t* states, cudaStream_t s) {
  k_push_primaries<<<push_grid(n), 256, 0, s>>>(p, prim, n, base, states);
}
void launch_push_device_primaries(const Params& p, const DevicePrimary* src, uint32_t n, uint32_t event,
                                  unsigned long long tid0, uint32_t prim0, uint32_t* states, cudaStream_t s) {
  k_check_device_primaries<<<push_grid(n), 256, 0, s>>>(p, src, n);
  k_push_device_primaries<<<push_grid(n), 256, 0, s>>>(p, src, n, event, tid0, prim0, states);
}
void launch_reset_event(double* tally, int n_bins, double* escaped, unsigned* event_live, cudaStream_t s) {
  k_reset_event<<<push_grid((uint32_t)n_bins), 256, 0, s>>>(tally, n_bins, escaped, event_live);
}
void launch_copy_out(void* dst, const void* src, uint32_t words, void* dst2, const void* src2, uint32_t words2,
                     cudaStream_t s) {
  k_copy_out<<<push_grid(words > words2 ? words : words2), 256, 0, s>>>(
      static_cast<uint32_t*>(dst), static_cast<const uint32_t*>(src), words, static_cast<uint32_t*>(dst2),
      static_cast<const uint32_t*>(src2), words2);
}

const char* kernel_name(int id) {
  static const char* names[KID_COUNT] = {"fill_step", "scatter", "step", "fill", "pre_step", "along_neutral",
                                         "along_charged", "compton", "photoelectric", "pair", "moller", "brems",
                                         "loop_ctl", "loop", "local"};
  return (id >= 0 && id < KID_COUNT) ? names[id] : "?";
}

// Active-lane counters of the instrumented build: per site, visits and lanes
// summed over the copies, then cleared. Without the instrumentation there
// is nothing to read.
cudaError_t read_lane_counts(unsigned long long* host_out, int n_sites) {
#ifdef CELER_LANE_COUNTERS
  unsigned long long all[kLaneCopies][kLaneSites][kLaneValues];
  cudaError_t e = cudaMemcpyFromSymbol(all, g_lane_counts, sizeof(all));
  if (e != cudaSuccess) return e;
  for (int k = 0; k < n_sites && k < kLaneSites; ++k) {
    for (int j = 0; j < kLaneValues; ++j) {
      unsigned long long v = 0;
      for (int c = 0; c < kLaneCopies; ++c) v += all[c][k][j];
      host_out[kLaneValues * k + j] = v;
    }
  }
  static const unsigned long long zeros[kLaneCopies][kLaneSites][kLaneValues] = {};
  return cudaMemcpyToSymbol(g_lane_counts, zeros, sizeof(zeros));
#else
  (void)host_out;
  (void)n_sites;
  return cudaErrorNotSupported;
#endif
}

}  // namespace celer
