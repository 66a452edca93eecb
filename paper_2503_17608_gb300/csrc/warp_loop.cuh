// The per-warp schedule of the asynchronous loop (block-local policy):
// k_loop_warps, one cooperative launch of one block per SM in which every warp
// schedules itself. Included by step.cu inside its anonymous namespace, after
// the block passes and the buffer protocol (ring_wait) it uses.
//
// What bounds it is instruction fetch: the instruction cache of a GPC serves
// 0.48 requests per cycle to its SMs whatever the variant of the loop (ncu:
// requests x 2.1 cycles / 8 GPCs = the kernel's time), and a block alone on
// its GPC runs 1.5 times faster than a full grid's. Then the latency of a
// track's next step: a job lasts at least as long as its longest chain of
// dependent steps, and a GB300 sub-partition issues one FP64 warp instruction
// every 64 cycles. So:
//  * a block's live tracks sit in shared memory (TrackCache), not in the slot
//    store: a piece's 32 tracks are scattered, and a scattered 8-byte access
//    costs one L1 tag lookup per lane and field there, but a few bank
//    conflicts here; nothing is written through to L2 per step, and a whole
//    job never touches the slot store;
//  * a piece moves its tracks by as many steps as most of them take before an
//    interaction (fly_photons, step_electrons), in registers: a photon's
//    crossing then costs 6 FP64 instructions instead of ~20 and a queue round
//    trip;
//  * interactions wait in queues of their own kind, so their pieces are full,
//    and the warps that take full pieces follow one kind while it lasts, so
//    that they run the same code.
// Against one crossing per piece with the tracks in the slot store: one event
// of 12 particles 0.90 -> 0.68 ms, 1 GeV calorimeter 1.25 -> 1.05 ms, 4 T
// calorimeter 10,000 x 10 GeV 3.50 -> 3.10 ms, 100,000 x 10 GeV 25.4 -> 15.9 ms.
#pragma once

// ---- the shared-memory track store of a block
// One array per field; kCap entries (a power of two). meta: layer (bits
// 0-15), grid bin of its energy (16-23), particle type (24-25), pending
// interaction (26-29), kMetaStored: the track also holds a slot of the store
// (home), kMetaLive: the entry holds a track. Entry indices travel through
// the queues; the owner of a popped entry is the only one to touch it.
constexpr unsigned kMetaStored = 1u << 30, kMetaLive = 1u << 31;
constexpr unsigned kNoEntry = 0xFFFFFFFFu;

// Kinds of work a warp takes, each with a queue of entries (the free entries
// are the last queue).
enum WarpKind : int { W_PHOTON = 0, W_ELECTRON, W_COMPTON, W_PAIR, W_MOLLER, W_BREMS, kWarpKinds, W_FREE = kWarpKinds,
                      W_NONE = 15 };

template <int kCap>
struct TrackCache {
  unsigned char* base;
  static constexpr size_t kBytes = (size_t)kCap * (10 * 8 + 5 * 4 + 4 * (kWarpKinds + 1));
  template <class T, int kOff>
  __device__ __forceinline__ T& at(unsigned c) const {
    return reinterpret_cast<T*>(base + (size_t)kCap * kOff)[c];
  }
  __device__ __forceinline__ double& x(unsigned c) const { return at<double, 0>(c); }
  __device__ __forceinline__ double& y(unsigned c) const { return at<double, 8>(c); }
  __device__ __forceinline__ double& z(unsigned c) const { return at<double, 16>(c); }
  __device__ __forceinline__ double& ux(unsigned c) const { return at<double, 24>(c); }
  __device__ __forceinline__ double& uy(unsigned c) const { return at<double, 32>(c); }
  __device__ __forceinline__ double& uz(unsigned c) const { return at<double, 40>(c); }
  __device__ __forceinline__ double& E(unsigned c) const { return at<double, 48>(c); }
  __device__ __forceinline__ double& nmfp(unsigned c) const { return at<double, 56>(c); }
  __device__ __forceinline__ double& gfrac(unsigned c) const { return at<double, 64>(c); }
  __device__ __forceinline__ unsigned long long& tid(unsigned c) const { return at<unsigned long long, 72>(c); }
  __device__ __forceinline__ uint32_t& ctr(unsigned c) const { return at<uint32_t, 80>(c); }
  __device__ __forceinline__ uint32_t& event(unsigned c) const { return at<uint32_t, 84>(c); }
  __device__ __forceinline__ uint32_t& primary(unsigned c) const { return at<uint32_t, 88>(c); }
  __device__ __forceinline__ uint32_t& meta(unsigned c) const { return at<uint32_t, 92>(c); }
  __device__ __forceinline__ uint32_t& home(unsigned c) const { return at<uint32_t, 96>(c); }
  // queue k's entry at position t
  __device__ __forceinline__ volatile unsigned* queue(int k, unsigned t) const {
    return reinterpret_cast<unsigned*>(base + (size_t)kCap * 100) + (size_t)k * kCap + (t & (unsigned)(kCap - 1));
  }
};
__device__ __forceinline__ int meta_layer(unsigned m) { return (int)(m & 0xFFFFu); }
__device__ __forceinline__ int meta_gbin(unsigned m) { return (int)((m >> 16) & 0xFFu); }
__device__ __forceinline__ uint8_t meta_ptype(unsigned m) { return (uint8_t)((m >> 24) & 3u); }
__device__ __forceinline__ uint8_t meta_act(unsigned m) { return (uint8_t)((m >> 26) & 15u); }
__device__ __forceinline__ unsigned with_layer(unsigned m, int layer) { return (m & ~0xFFFFu) | (unsigned)layer; }
__device__ __forceinline__ unsigned with_act(unsigned m, unsigned act) { return (m & ~(15u << 26)) | (act << 26); }

// Queue entries: the high half holds a 16-bit state (2 lap: free for its
// writer; 2 lap + 1: written; lap = t / kCap modulo 2^15), the low half the
// entry index. Writers reserve on the tail counter and readers claim on the
// head counter; each side waits (bounded) only for the other side's access of
// the same queue entry, which follows that side's claim or reservation
// directly. The entry is written with a release store and read with an
// acquire load, so the pusher's writes of the track come before the reader's
// reads of it.
template <int kCap>
__device__ __forceinline__ unsigned lap_code(unsigned t) {
  return (2u * (t / (unsigned)kCap)) & 0xFFFFu;
}
// Append entry c of every lane in mask (not empty) to queue k, one counter
// update per warp; every lane of the warp calls it.
template <int kCap>
__device__ __forceinline__ void push_lanes(const Params& p, const TrackCache<kCap>& tc, unsigned* tail, int k,
                                           unsigned mask, unsigned c) {
  const unsigned lane = threadIdx.x & 31u;
  const int leader = __ffs(mask) - 1;
  unsigned t = 0;
  if ((int)lane == leader) t = atomicAdd(&tail[k], (unsigned)__popc(mask));
  t = __shfl_sync(0xffffffffu, t, leader) + (unsigned)__popc(mask & ((1u << lane) - 1u));
  if ((mask >> lane) & 1u) {
    volatile unsigned* e = tc.queue(k, t);
    const unsigned lap2 = lap_code<kCap>(t);
    if (wq_wait(p, e, lap2)) st_release_cta(e, (((lap2 + 1u) & 0xFFFFu) << 16) | c);
  }
}
// Read position t of queue k (one thread; t claimed by its warp) and free it
// for the next lap; kNoEntry if the wait gave up.
template <int kCap>
__device__ __forceinline__ unsigned pop_entry(const Params& p, const TrackCache<kCap>& tc, int k, unsigned t) {
  volatile unsigned* e = tc.queue(k, t);
  const unsigned lap2 = lap_code<kCap>(t);
  if (!wq_wait(p, e, (lap2 + 1u) & 0xFFFFu)) return kNoEntry;
  const unsigned v = ld_acquire_cta(e) & 0xFFFFu;
  *e = ((lap2 + 2u) & 0xFFFFu) << 16;
  return v;
}

// A piece stays in registers while at least kStay / 4 of the tracks it started
// with go on to another step, at most kMaxStay steps (a track that nothing
// limits, such as one circling in the field with its losses switched off, must
// return to the queue for the run's limits to end it).
// (Electrons stop with the first that ends or interacts: staying while half go
// on costs 10,000 x 10 GeV 3.85 -> 3.92 ms. Photons while half instead of a
// quarter fly on: 100,000 x 10 GeV 19.5 -> 20.0 ms.)
constexpr unsigned kStayPhotons = 1, kStayElectrons = 4;
constexpr int kMaxStay = 64;
// Rejection attempts of a Compton piece of at least kFewTracks tracks: 73 % of
// them are accepted, so the lanes still trying after two are few.
constexpr int kComptonAttempts = 2;
constexpr unsigned kFewTracks = 16;

// How a track leaves its piece's steps.
enum StepEnd : int { END_NONE = 0, END_DEPOSIT, END_ESCAPE, END_INTERACT };

// A track at the end of its piece's steps: the steps it took in its history,
// and what it leaves if it ended (deposit and escape in one form).
__device__ __forceinline__ void tally_end(const Params& p, int end, uint32_t ev, uint32_t prim, int layer, double z,
                                          double E, unsigned taken) {
  const bool ended = end == END_DEPOSIT || end == END_ESCAPE, out = end == END_ESCAPE;
  const uint32_t row = row_of(p, ev);
  int b = 0;
  if (ended) {
    b = out ? 0 : tally_bin(p, layer, z);
    atomicAdd(out ? p.escaped + row : p.tally + (size_t)row * p.n_bins + b, E);
  }
  if (prim < p.hist_cap) {
    atomicAdd(&p.hist_steps[prim], (unsigned long long)taken);
    if (ended) atomicAdd(out ? p.hist_escaped + prim : p.hist_edep + (size_t)prim * p.n_bins + b, E);
  }
}

// Steps of up to 32 photons, one per lane (c: its entry, kNoEntry for none):
// each crosses layers in straight flight until it interacts or ends, or until
// too few of the piece's photons fly on. A crossing is the step limit of
// step_limit and the move of along_one for a photon, with what a flight
// leaves unchanged computed once: 1/uz (the path over a layer is the rounded
// quotient d / uz by it), the cross section of the two materials met last, and
// whether the straight line leaves through the z planes before any side plane.
// What is left of a crossing is six FP64 instructions: three for the quotient,
// the mean free paths it takes, those left, and the path so far (the position
// is formed from it where it is needed). Returns the queue the photon goes to
// (W_FREE: it ended).
template <int kCap>
__device__ __forceinline__ int fly_photons(const Params& p, const TrackCache<kCap>& tc, const SharedStatic& ss,
                                           const double* thick, unsigned c, unsigned& steps) {
  const bool on = c != kNoEntry;
  const unsigned n0 = (unsigned)__popc(__ballot_sync(0xffffffffu, on));
  double x0 = 0, y0 = 0, z = 0, ux = 0, uy = 0, uz = 1, nmfp = 0, E = 0;
  GridPos g{0, 0.0};
  unsigned meta = 0;
  int layer = 0;
  if (on) {
    meta = tc.meta(c);
    x0 = tc.x(c);
    y0 = tc.y(c);
    z = tc.z(c);
    ux = tc.ux(c);
    uy = tc.uy(c);
    uz = tc.uz(c);
    E = tc.E(c);
    nmfp = tc.nmfp(c);
    layer = meta_layer(meta);
    g = GridPos{meta_gbin(meta), tc.gfrac(c)};
  }
  const double* zb = ss.zb;
  const bool up = dbits(uz) >= 0;
  // |uz| in [1e-100, 2) on the bits: 1/uz is finite; other values (0, NaN,
  // tiny) divide
  const unsigned long long uza = (unsigned long long)dbits(uz) & 0x7FFFFFFFFFFFFFFFull;
  const bool steep = uza >= (unsigned long long)dbits(1e-100) && uza < 0x4000000000000000ull;
  const double auz = fabs(uz), ainv = steep ? recip(auz) : 0.0;
  double d = up ? zb[layer + 1] - z : z - zb[layer];  // to the next plane, along uz
  // the line's displacement from here to the last z plane, with a margin far
  // above the roundings of the crossings on the way: less than the distance
  // to the side planes means that no crossing can reach one
  bool inside = false;
  if (steep) {
    const double path = fabs(zb[up ? p.n_layers : 0] - z) * ainv;
    inside = farther(p.hx - fabs(x0), fma(path, fabs(ux) * (1.0 + 1e-9), 1e-9)) &&
             farther(p.hy - fabs(y0), fma(path, fabs(uy) * (1.0 + 1e-9), 1e-9));
  }
  const bool low = dbits(E) < dbits(p.cut_track);  // E < cut on the bits (a NaN E fails it, as in FP64)
  // the two materials met last: their total cross section mu and the partial
  // sums muC (Compton) and muCP (and photoelectric)
  int mat = -1, mat2 = -1;
  double mu = 0.0, muC = 0.0, muCP = 0.0, mu2 = 0.0, muC2 = 0.0, muCP2 = 0.0;
  double path = 0.0, s = 0.0;
  int end = END_NONE;
  bool fly = on;
  unsigned taken = 0;
  for (int round = 0;;) {
    if (fly) {
      CELER_LANES(LS_ALONG);
      const int m = ss.lmat[layer];
      if (m != mat) {
        const double t = mu, tC = muC, tCP = muCP;
        const int tm = mat;
        mu = mu2;
        muC = muC2;
        muCP = muCP2;
        mat = mat2;
        mu2 = t;
        muC2 = tC;
        muCP2 = tCP;
        mat2 = tm;
        if (m != mat) {
          const double2* mt = ss.tab + m * (kCols * kGrid);
          muC = interp(mt + COL_COMPTON * kGrid, g);
          muCP = muC + interp(mt + COL_PE * kGrid, g);
          // E > threshold on the bits (E >= +0; a NaN E makes mu NaN either way)
          mu = muCP + (dbits(E) > dbits(kPairThreshold) ? interp(mt + COL_PAIR * kGrid, g) : 0.0);
          mat = m;
        }
      }
      // distance to the layer's planes (as in step_limit)
      bool side = false;
      if (steep) {
        s = quot_by(d, auz, ainv);
      } else {
        s = uza != 0ull && uza <= 0x7FF0000000000000ull ? quot_any(d, auz) : kInf;
      }
      if (!inside) {
        const double s_side = straight_side(p, fma(path, ux, x0), fma(path, uy, y0), ux, uy, s * kLimitMargin);
        if (dbits(s_side) != dbits(kInf) && s_side < s) {
          s = s_side;
          side = true;
        }
      }
      if (dbits(s) < 0 && dbits(s) != dbits(-0.0)) s = 0.0;
      // the interaction, if it can come first (as in step_limit; for mu = 0
      // the quotient is no less than s)
      const double t = s * mu;
      if (dbits(nmfp) <= dbits(t) + kLimitUlps) {
        const double s_int = quot(nmfp, mu);
        if (dbits(s_int) < dbits(s)) {
          s = s_int;
          end = END_INTERACT;
        }
      }
      ++taken;
      if (end == END_NONE) {
        if (dbits(s) == dbits(kInf)) {  // nothing limits the step: the track ends in place
          end = END_DEPOSIT;
          s = 0.0;
        } else {
          nmfp = fma(-s, mu, nmfp);
          path += s;
          layer += up ? 1 : -1;
          if (side || (unsigned)layer >= (unsigned)p.n_layers) {
            end = END_ESCAPE;
          } else {
            z = zb[up ? layer : layer + 1];
            d = thick[layer];
            if (low) end = END_DEPOSIT;
          }
        }
      }
      fly = end == END_NONE;
    }
    const unsigned left = (unsigned)__popc(__ballot_sync(0xffffffffu, fly));
    if (left * 4u < n0 * kStayPhotons || ++round >= kMaxStay || left == 0u) break;
  }
  if (!on) return W_NONE;
  steps += taken;
  const uint32_t ev = tc.event(c);
  int out = W_PHOTON;
  if (end == END_INTERACT) {
    path += s;
    z = fma(s, uz, z);
    if (low) {
      end = END_DEPOSIT;
    } else {
      // process selection with the cross sections of the interaction's layer
      // (finite operands >= +0: the comparisons on the bits are exact)
      TrackRng rng(p.seed, ev, tc.tid(c), tc.ctr(c));
      const double target = rng.uniform() * mu;
      // (if rounding leaves none: the last possible)
      int sel = dbits(muCP) < dbits(mu) ? 2 : (dbits(muC) < dbits(muCP) ? 1 : 0);
      if (dbits(target) < dbits(muC))
        sel = 0;
      else if (dbits(target) < dbits(muCP))
        sel = 1;
      if (sel == 1) end = END_DEPOSIT;  // photoelectric absorption: all energy deposited here
      tc.ctr(c) = rng.ctr;
      meta = with_act(meta, sel == 0 ? A_COMPTON : A_PAIR);
      out = sel == 0 ? W_COMPTON : W_PAIR;
    }
  }
  tally_end(p, end, ev, tc.primary(c), layer, z, E, taken);
  if (end == END_DEPOSIT || end == END_ESCAPE) return W_FREE;
  tc.nmfp(c) = nmfp;
  tc.x(c) = fma(path, ux, x0);
  tc.y(c) = fma(path, uy, y0);
  tc.z(c) = z;
  tc.meta(c) = with_layer(meta, layer);
  return out;
}

// Steps of up to 32 charged tracks: the step limit and the along-step of the
// synchronous loops (step_limit, along_one) in one pass in registers, again
// while most of the piece's tracks go on without an interaction.
template <int kCap>
__device__ __forceinline__ int step_electrons(const Params& p, const TrackCache<kCap>& tc, const SharedStatic& ss,
                                              unsigned c, unsigned& steps) {
  const bool on = c != kNoEntry;
  const unsigned n0 = (unsigned)__popc(__ballot_sync(0xffffffffu, on));
  double x = 0, y = 0, z = 0, ux = 0, uy = 0, uz = 1, nmfp = 0, E = 0;
  GridPos g{0, 0.0};
  unsigned meta = 0;
  int layer = 0;
  uint32_t ev = 0, prim = 0;
  if (on) {
    meta = tc.meta(c);
    ev = tc.event(c);
    prim = tc.primary(c);
    x = tc.x(c);
    y = tc.y(c);
    z = tc.z(c);
    ux = tc.ux(c);
    uy = tc.uy(c);
    uz = tc.uz(c);
    E = tc.E(c);
    nmfp = tc.nmfp(c);
    layer = meta_layer(meta);
    g = GridPos{meta_gbin(meta), tc.gfrac(c)};
  }
  const uint8_t pt = meta_ptype(meta);
  const double* zb = ss.zb;
  const bool eloss = (p.processes & PROC_ELOSS) != 0;
  const bool helix = ((unsigned long long)dbits(p.Bz) << 1) != 0ull;  // Bz != 0 on the bits
  double mu = 0.0, mu0 = 0.0, mu1 = 0.0;
  int end = END_NONE;
  bool go = on;
  unsigned taken = 0;
  for (int round = 0;;) {
    if (go) {
      CELER_LANES(LS_ALONG);
      const double2* mt = ss.tab + ss.lmat[layer] * (kCols * kGrid);
      mu0 = interp(mt + COL_MOLLER * kGrid, g);
      mu1 = interp(mt + COL_BREMS * kGrid, g);
      mu = mu0 + mu1;
      const double R = eloss ? interp(mt + COL_RANGE * kGrid, g) : 0.0;
      const Curvature cv = helix ? curvature(p, pt, E) : Curvature{0.0, 0.0};
      // step limit: z planes, side planes, range, interaction, in this order,
      // each replacing the current one only if shorter (step_limit has the
      // reasons of the margins and of the comparisons on the bits)
      double s = kInf;
      uint8_t act = A_NONE;
      const unsigned long long uza = (unsigned long long)dbits(uz) & 0x7FFFFFFFFFFFFFFFull;
      if (uza != 0ull && uza <= 0x7FF0000000000000ull) {
        const bool up = dbits(uz) >= 0;
        s = quot(zb[up ? layer + 1 : layer] - z, uz);
        act = up ? A_ZUP : A_ZDOWN;
      }
      double s_side = kInf;
      if (helix) {
        const double reach = s + 1e-3;
        if (!(farther(p.hx - fabs(x), reach) && farther(p.hy - fabs(y), reach)))
          s_side = helix_side_distance(cv, x, y, ux, uy, p.hx, p.hy);
      } else {
        const double reach = s * kLimitMargin;
        const double reach2 = reach * kLimitMargin;
        if (!(p.hx - fabs(x) > reach2 && p.hy - fabs(y) > reach2)) s_side = straight_side(p, x, y, ux, uy, reach);
      }
      if (dbits(s_side) != dbits(kInf) && s_side < s) {
        s = s_side;
        act = A_SIDE;
      }
      if (dbits(s) < 0 && dbits(s) != dbits(-0.0)) s = 0.0;
      if (eloss) {
        double s_rng = kInf;
        if (dbits(R) <= dbits(kFinalR)) {
          s_rng = R;
        } else {
          const double at_least = kAlphaR * R + kFinalR * (1.0 - kAlphaR);
          if (dbits(at_least) <= dbits(s * kRangeMargin))
            s_rng = kAlphaR * R + kFinalR * (1.0 - kAlphaR) * (2.0 - quot(kFinalR, R));
        }
        if (dbits(s_rng) < dbits(s)) {
          s = s_rng;
          act = A_RANGE;
        }
      }
      bool interact = false;
      if (dbits(mu) > 0 && dbits(nmfp) <= dbits(s * mu) + kLimitUlps) {
        const double s_int = quot(nmfp, mu);
        if (dbits(s_int) < dbits(s)) {
          s = s_int;
          interact = true;
        }
      }
      ++taken;
      if (dbits(s) == dbits(kInf)) {
        end = END_DEPOSIT;  // nothing limits the step: the track ends in place
      } else {
        if (helix && p.field_cap > 0 && s * fabs(cv.kappa) > kRkTurn * p.field_cap) {
          s = quot(kRkTurn * p.field_cap, fabs(cv.kappa));  // cut at the substep cap: no crossing, no interaction
          act = A_FIELD;
          interact = false;
        }
        nmfp = fma(-s, mu, nmfp);
        if (helix) {
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
          const double Ep = inverse_range(mt + COL_RANGE * kGrid, R - s, p.lnEmin, p.dl, p.mtab, g);
          deposit(p, ev, prim, layer, z, E - Ep);
          E = Ep;
        }
        if (interact) {
          end = END_INTERACT;
        } else if (act == A_ZUP || act == A_ZDOWN) {
          const bool up = act == A_ZUP;
          layer += up ? 1 : -1;
          if ((unsigned)layer >= (unsigned)p.n_layers)
            end = END_ESCAPE;
          else
            z = zb[up ? layer : layer + 1];
        } else if (act == A_SIDE) {
          end = END_ESCAPE;
        }
        if (end != END_ESCAPE && dbits(E) < dbits(p.cut_track)) end = END_DEPOSIT;
      }
      go = end == END_NONE;
    }
    const unsigned left = (unsigned)__popc(__ballot_sync(0xffffffffu, go));
    if (left * 4u < n0 * kStayElectrons || ++round >= kMaxStay || left == 0u) break;
  }
  if (!on) return W_NONE;
  steps += taken;
  tally_end(p, end, ev, prim, layer, z, E, taken);
  if (end == END_DEPOSIT || end == END_ESCAPE) return W_FREE;
  int out = W_ELECTRON;
  if (end == END_INTERACT) {
    // the process, with the cross sections before the last step (the last
    // possible one if rounding leaves none)
    TrackRng rng(p.seed, ev, tc.tid(c), tc.ctr(c));
    const double target = rng.uniform() * mu;
    tc.ctr(c) = rng.ctr;
    const bool moller = dbits(target) < dbits(mu0) || dbits(mu1) == 0ll;
    meta = with_act(meta, moller ? A_MOLLER : A_BREMS);
    out = moller ? W_MOLLER : W_BREMS;
  }
  tc.x(c) = x;
  tc.y(c) = y;
  tc.z(c) = z;
  if (helix) {
    tc.ux(c) = ux;
    tc.uy(c) = uy;
  }
  tc.E(c) = E;
  tc.nmfp(c) = nmfp;
  tc.gfrac(c) = g.frac;
  tc.meta(c) = (with_layer(meta, layer) & ~(0xFFu << 16)) | ((unsigned)g.bin << 16);
  return out;
}

// ---- discrete interactions of one track each. They return W_FREE if the
// track ended, W_NONE if it waits for buffer space, else the queue of its
// next step; the caller then samples its fresh number of mean free paths from
// rng, which follows the interaction's draws.

// Compton scattering (compton_one). At most `attempts` rejection attempts: a
// track that needs more goes back to its queue (W_COMPTON), its draw counter
// advanced, instead of holding the piece's other lanes.
template <int kCap>
__device__ __forceinline__ int compton_piece(const Params& p, const TrackCache<kCap>& tc, unsigned c, TrackRng& rng,
                                             int attempts) {
  CELER_LANES(LS_COMPTON);
  const double E = tc.E(c);
  const uint32_t ev = tc.event(c), prim = tc.primary(c);
  const int layer = meta_layer(tc.meta(c));
  const double z = tc.z(c);
  double cost;
  bool ok;
  const uint32_t ctr0 = rng.ctr;
  const double eps = sample_compton(E, rng, cost, ok, p.mtab, attempts);
  if (!ok && rng.ctr - ctr0 < 3u * kMaxAttempts) {
    tc.ctr(c) = rng.ctr;
    return W_COMPTON;
  }
  if (!ok) atomicOr(&p.ctl->error, ERR_SAMPLING);  // non-finite input: end the track, flag the run
  const double u_phi = rng.uniform();
  const double E1 = eps * E;
  // below the cut (on the bits: a negative E1 passes, a positive NaN fails, as
  // in FP64) the photon is absorbed: recoil and photon in one deposit
  const bool ends = !ok || dbits(E1) < dbits(p.cut_track);
  deposit(p, ev, prim, layer, z, ends ? E : E - E1);
  if (ends) return W_FREE;
  double ux = tc.ux(c), uy = tc.uy(c), uz = tc.uz(c);
  rotate_dir(ux, uy, uz, cost, u_phi, p.mtab);
  tc.ux(c) = ux;
  tc.uy(c) = uy;
  tc.uz(c) = uz;
  tc.E(c) = E1;
  return W_PHOTON;
}

// Pair production (pair_one).
template <int kCap>
__device__ __forceinline__ int pair_piece(const Params& p, const TrackCache<kCap>& tc, unsigned c, TrackRng& rng) {
  CELER_LANES(LS_PAIR);
  const bool keep = kMe >= p.cut_track;
  const bool reuse = keep && p.reuse_parent != 0;  // the first photon takes the parent's place
  unsigned long long base;
  if (!reserve_entries(p, keep ? (reuse ? 1u : 2u) : 0u, true, base)) return W_NONE;
  const uint32_t ev = tc.event(c), prim = tc.primary(c);
  const int layer = meta_layer(tc.meta(c));
  const double x = tc.x(c), y = tc.y(c), z = tc.z(c);
  deposit(p, ev, prim, layer, z, keep ? tc.E(c) - 2.0 * kMe : tc.E(c));
  if (!keep) return W_FREE;
  const double cost = 2.0 * rng.uniform() - 1.0;
  const double u_phi = rng.uniform();
  const double sint2 = 1.0 - cost * cost;
  const double sint = dbits(sint2) > 0 ? fast_sqrt(sint2) : 0.0;
  double sp_, cp_;
  fast_sincos_2pi(u_phi, p.mtab, &sp_, &cp_);
  const double dx = sint * cp_, dy = sint * sp_, dz = cost;
  const unsigned long long tid1 = rng.raw();
  const unsigned long long tid2 = rng.raw();
  if (prim < p.hist_cap) atomicAdd(&p.hist_secondaries[prim], 2ull);
  atomicAdd(&p.event_live[row_of(p, ev)], reuse ? 1u : 2u);
  if (!reuse) write_initializer(p, base, x, y, z, dx, dy, dz, kMe, tid1, ev, prim, layer, GAMMA);
  write_initializer(p, reuse ? base : base + 1, x, y, z, -dx, -dy, -dz, kMe, tid2, ev, prim, layer, GAMMA);
  if (!reuse) return W_FREE;
  tc.ux(c) = dx;
  tc.uy(c) = dy;
  tc.uz(c) = dz;
  tc.E(c) = kMe;
  tc.tid(c) = tid1;
  rng = TrackRng(p.seed, ev, tid1, 0u);
  return W_PHOTON;
}

// Moller scattering (moller_one).
template <int kCap>
__device__ __forceinline__ int moller_piece(const Params& p, const TrackCache<kCap>& tc, unsigned c, TrackRng& rng) {
  CELER_LANES(LS_MOLLER);
  const double T = tc.E(c);
  if (T <= 2.0 * p.cut_moller) return W_ELECTRON;  // closed at the post-step energy: null collision
  const uint32_t ev = tc.event(c), prim = tc.primary(c);
  bool ok;
  const double eps = sample_moller(T, p.cut_moller, rng, ok);
  const double Td = eps * T;
  const bool keep = ok && Td >= p.cut_track;
  unsigned long long base;
  if (!reserve_entries(p, keep ? 1u : 0u, true, base)) return W_NONE;
  const int layer = meta_layer(tc.meta(c));
  const double x = tc.x(c), y = tc.y(c), z = tc.z(c);
  if (!ok) {  // non-finite input: end the track, flag the run
    atomicOr(&p.ctl->error, ERR_SAMPLING);
    deposit(p, ev, prim, layer, z, T);
    return W_FREE;
  }
  const double pp2 = T * (T + 2.0 * kMe), pd2 = Td * (Td + 2.0 * kMe);
  const double rpp = fast_rsqrt(pp2), rpd = fast_rsqrt(pd2);
  const double cost = fmin(1.0, Td * (T + 2.0 * kMe) * rpp * rpd);
  const double u_phi = rng.uniform();
  const double ux = tc.ux(c), uy = tc.uy(c), uz = tc.uz(c);
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
  }
  const bool ends = dbits(E1) < dbits(p.cut_track);
  if (!keep || ends) deposit(p, ev, prim, layer, z, (keep ? 0.0 : Td) + (ends ? E1 : 0.0));
  if (ends) return W_FREE;
  tc.ux(c) = vx * inv;
  tc.uy(c) = vy * inv;
  tc.uz(c) = vz * inv;
  tc.E(c) = E1;
  return W_ELECTRON;
}

// Bremsstrahlung (brems_one).
template <int kCap>
__device__ __forceinline__ int brems_piece(const Params& p, const TrackCache<kCap>& tc, unsigned c, TrackRng& rng) {
  CELER_LANES(LS_BREMS);
  const double T = tc.E(c);
  if (T <= p.cut_brems) return W_ELECTRON;  // null collision
  const uint32_t ev = tc.event(c), prim = tc.primary(c);
  double k = p.cut_brems * fast_exp(rng.uniform() * fast_log(quot(T, p.cut_brems), p.mtab), p.mtab);
  if (k > T) k = T;
  const bool keep = k >= p.cut_track;
  unsigned long long base;
  if (!reserve_entries(p, keep ? 1u : 0u, true, base)) return W_NONE;
  const int layer = meta_layer(tc.meta(c));
  const double z = tc.z(c);
  const double E1 = T - k;
  const bool ends = dbits(E1) < dbits(p.cut_track);
  if (keep) {
    const unsigned long long tid = rng.raw();
    write_initializer(p, base, tc.x(c), tc.y(c), z, tc.ux(c), tc.uy(c), tc.uz(c), k, tid, ev, prim, layer, GAMMA);
    atomicAdd(&p.event_live[row_of(p, ev)], 1u);
    if (prim < p.hist_cap) atomicAdd(&p.hist_secondaries[prim], 1ull);
  }
  if (!keep || ends) deposit(p, ev, prim, layer, z, (keep ? 0.0 : k) + (ends ? E1 : 0.0));
  if (ends) return W_FREE;
  tc.E(c) = E1;
  return W_ELECTRON;
}

// ---- a block's tracks between the slot store and its shared memory

// The queue of a pending interaction.
__device__ __forceinline__ int queue_of(uint8_t act) {
  return act == A_COMPTON ? W_COMPTON : (act == A_PAIR ? W_PAIR : (act == A_MOLLER ? W_MOLLER : W_BREMS));
}

// Number of mean free paths to the next interaction and the grid position in
// ln E, for a track about to take its first step after its creation or an
// interaction.
template <int kCap>
__device__ __forceinline__ void renew(const Params& p, const TrackCache<kCap>& tc, unsigned c, unsigned meta,
                                      TrackRng& rng) {
  tc.nmfp(c) = -fast_log(rng.uniform(), p.mtab);
  tc.ctr(c) = rng.ctr;
  const GridPos g = grid_pos(tc.E(c), p.lnEmin, p.inv_dl, p.mtab);
  tc.gfrac(c) = g.frac;
  tc.meta(c) = (with_act(meta, 0u) & ~(0xFFu << 16)) | ((unsigned)g.bin << 16);
}

// The live track of `slot` into entry c; returns its queue. It keeps its slot
// (kMetaStored) until it ends or the run does.
template <int kCap>
__device__ __noinline__ int load_entry(const Params& p, const TrackCache<kCap>& tc, uint32_t slot, unsigned c) {
  const Tracks& t = p.trk;
  const uint8_t st = t.status[slot] & 3u, pt = t.ptype[slot];
  const double nmfp = t.nmfp[slot];
  tc.x(c) = t.x[slot];
  tc.y(c) = t.y[slot];
  tc.z(c) = t.z[slot];
  tc.ux(c) = t.ux[slot];
  tc.uy(c) = t.uy[slot];
  tc.uz(c) = t.uz[slot];
  tc.E(c) = t.E[slot];
  tc.nmfp(c) = nmfp;
  tc.gfrac(c) = t.gfrac[slot];
  tc.tid(c) = t.tid[slot];
  tc.ctr(c) = t.ctr[slot];
  tc.event(c) = t.event[slot];
  tc.primary(c) = t.primary[slot];
  tc.home(c) = slot;
  t.status[slot] = HELD;
  const bool pending = st == DEFERRED;
  const uint8_t act = pending ? t.action[slot] : (uint8_t)A_NONE;
  const unsigned meta = kMetaLive | kMetaStored | ((unsigned)act << 26) | ((unsigned)pt << 24) |
                        (((unsigned)t.gbin[slot] & 0xFFu) << 16) | ((unsigned)t.layer[slot] & 0xFFFFu);
  tc.meta(c) = meta;
  if (pending) return queue_of(act);
  if (dbits(nmfp) < 0) {  // unset (-1)
    TrackRng rng(p.seed, t.event[slot], t.tid[slot], t.ctr[slot]);
    renew(p, tc, c, meta, rng);
  }
  return pt == GAMMA ? W_PHOTON : W_ELECTRON;
}

// Entry c's track into `slot`, between two steps or with its interaction
// pending (deferred).
template <int kCap>
__device__ __forceinline__ void store_entry(const Params& p, const TrackCache<kCap>& tc, uint32_t slot, unsigned c) {
  const Tracks& t = p.trk;
  const unsigned meta = tc.meta(c);
  t.x[slot] = tc.x(c);
  t.y[slot] = tc.y(c);
  t.z[slot] = tc.z(c);
  t.ux[slot] = tc.ux(c);
  t.uy[slot] = tc.uy(c);
  t.uz[slot] = tc.uz(c);
  t.E[slot] = tc.E(c);
  t.nmfp[slot] = tc.nmfp(c);
  t.gfrac[slot] = tc.gfrac(c);
  t.gbin[slot] = meta_gbin(meta);
  t.tid[slot] = tc.tid(c);
  t.ctr[slot] = tc.ctr(c);
  t.event[slot] = tc.event(c);
  t.primary[slot] = tc.primary(c);
  t.layer[slot] = meta_layer(meta);
  t.ptype[slot] = meta_ptype(meta);
  t.action[slot] = meta_act(meta);
  t.status[slot] = meta_act(meta) != 0 ? DEFERRED : ALIVE;
}

// Slots of block bid.
__device__ __forceinline__ unsigned owned_slots(const Params& p, int bid, int nb, uint32_t n_own) {
  const bool owns_last = n_own > 0 && (uint32_t)bid + (uint32_t)nb * (n_own - 1u) == p.n_chunks - 1u;
  return n_own * 32u - (owns_last ? p.n_chunks * 32u - p.n_slots : 0u);
}

// A block's control words in shared memory that the functions below move too:
// one address for all of them, so that the loop keeps none of them in registers
// for the calls.
struct BlockWords {
  unsigned head[kWarpKinds + 1], tail[kWarpKinds + 1];  // of the queues
  unsigned live, parked, cursor, filling, exit, place;
};
__device__ __forceinline__ unsigned block_word(const unsigned& a) { return *reinterpret_cast<const volatile unsigned*>(&a); }

// The parked tracks of the next chunk that has any, if as many entries are free:
// each lane's slot (or ~0), their number in `take`, the first of the free entries
// claimed for them in f0. While the buffer is full (moving_only) the tracks whose
// interactions wait for room in it stay where they are. The tracks are marked,
// so that the warp can load them without the block's fill lock, which lane 0
// holds and this gives up; the lanes know theirs, since others of the chunk may
// be marked by another warp meanwhile. The whole warp calls it. (One lane looking
// at the chunk's slots in turn: a run that starts with 140,000 tracks, 0.9 -> 2.0
// ms.)
static __device__ __noinline__ uint32_t claim_parked_chunk(const Params& p, BlockWords& w, int bid, int nb, uint32_t n_own,
                                                           bool moving_only, unsigned& take, unsigned& f0) {
  const unsigned lane = threadIdx.x & 31u;
  unsigned m = 0, free_now = 0;
  if (lane == 0) {
    m = block_word(w.cursor);
    free_now = block_word(w.tail[W_FREE]) - block_word(w.head[W_FREE]);
  }
  m = __shfl_sync(0xffffffffu, m, 0);
  free_now = __shfl_sync(0xffffffffu, free_now, 0);
  uint32_t mine = 0xFFFFFFFFu;
  unsigned next = m;  // no parked track waits in a chunk before it
  take = 0;
  for (; m < n_own; ++m) {
    const uint32_t slot = ((uint32_t)bid + (uint32_t)nb * m) * 32u + lane;
    volatile uint8_t* status = p.trk.status + slot;
    const uint8_t st = slot < p.n_slots ? *status : (uint8_t)VACANT;
    const bool parked = st == ALIVE || (st == DEFERRED && !moving_only);
    const unsigned cnt = (unsigned)__popc(__ballot_sync(0xffffffffu, parked));
    const bool left = __any_sync(0xffffffffu, st == DEFERRED && moving_only);
    if (cnt > free_now) break;
    if (next == m && !left) next = m + 1u;
    if (cnt > 0) {
      if (parked) {
        *status = st | CLAIMED;
        mine = slot;
      }
      take = cnt;
      break;
    }
  }
  f0 = 0;
  if (lane == 0) {
    *reinterpret_cast<volatile unsigned*>(&w.cursor) = next;
    if (take) {
      f0 = atomicAdd(&w.head[W_FREE], take);  // only the holder of the lock claims free entries
      atomicAdd(&w.live, take);
      atomicSub(&w.parked, take);
    }
  }
  __threadfence_block();
  __syncwarp();
  if (lane == 0) atomicExch(&w.filling, 0u);
  return mine;
}

// The tracks still live at the end of a run back into the block's slots:
// those that hold one into it, the others into its vacant slots, in the order
// the warps find them. The whole block calls it; `list` holds kCap entries.
template <int kCap>
__device__ __noinline__ void store_tracks(const Params& p, const TrackCache<kCap>& tc, uint16_t* list, unsigned n_entries, int bid,
                             int nb) {
  __shared__ unsigned s_n, s_next;
  if (threadIdx.x == 0) s_n = s_next = 0u;
  __syncthreads();
  for (unsigned c = threadIdx.x; c < n_entries; c += blockDim.x) {
    const unsigned meta = tc.meta(c);
    if (!(meta & kMetaLive)) continue;
    if (meta & kMetaStored)
      store_entry(p, tc, tc.home(c), c);
    else
      list[atomicAdd(&s_n, 1u)] = (uint16_t)c;
  }
  __syncthreads();
  const unsigned n = s_n;
  const unsigned lane = threadIdx.x & 31u, nwarps = blockDim.x >> 5;
  for (uint32_t g = (uint32_t)bid + (uint32_t)nb * (threadIdx.x >> 5); g < p.n_chunks; g += (uint32_t)nb * nwarps) {
    // (read by lane 0: other warps move it, and the warp leaves as a whole or
    // not at all)
    unsigned next = 0;
    if (lane == 0) next = *reinterpret_cast<volatile unsigned*>(&s_next);
    if (__shfl_sync(0xffffffffu, next, 0) >= n) break;
    const uint32_t slot = g * 32u + lane;
    const bool vac = slot < p.n_slots && p.trk.status[slot] == VACANT;
    const unsigned bal = __ballot_sync(0xffffffffu, vac);
    if (bal == 0u) continue;
    unsigned r0 = 0;
    if (lane == 0) r0 = atomicAdd(&s_next, (unsigned)__popc(bal));
    r0 = __shfl_sync(0xffffffffu, r0, 0);
    const unsigned r = r0 + (unsigned)__popc(bal & ((1u << lane) - 1u));
    if (vac && r < n) store_entry(p, tc, slot, list[r]);
    const unsigned k = r0 < n ? (n - r0 < (unsigned)__popc(bal) ? n - r0 : (unsigned)__popc(bal)) : 0u;
    if (lane == 0 && k) {
      atomicSub(&p.vacant[g], k);
      atomicSub(&p.tile_vacant[g >> 3], k);
    }
    __syncwarp();
  }
}

// A block whose every entry holds a track that waits for buffer space moves up
// to 32 of them into its slots (their own, or vacant ones), their interactions
// pending, as the end of a run would store them; the entries take tracks out of
// the buffer then, which makes room in it, or parked tracks that can move.
// claim_parked_chunk brings them back once there is room. Not where nothing
// could take the entries: the block has no slot to spare and no track parked.
// (Without it a block could hold no more tracks than entries: 6 materials, 256
// entries, 20,000 x 1 GeV with a buffer of 2^17 ended with every entry of every
// block waiting.) The whole warp calls it.
template <int kCap>
__device__ __noinline__ void park_waiting(const Params& p, const TrackCache<kCap>& tc, BlockWords& w, int bid, int nb,
                                          uint32_t n_own) {
  const unsigned lane = threadIdx.x & 31u, lt = (1u << lane) - 1u;
  bool mine = false;
  uint32_t g = 0xFFFFFFFFu;  // a chunk with vacant slots
  unsigned h = 0, n = 0;
  int k = W_PAIR;
  if (lane == 0 && atomicCAS(&w.filling, 0u, 1u) == 0u) {
    mine = true;
    const unsigned parked = block_word(w.parked);
    if (block_word(w.tail[W_FREE]) == block_word(w.head[W_FREE]) &&
        (parked != 0u || block_word(w.live) < owned_slots(p, bid, nb, n_own))) {
      unsigned m = block_word(w.place);
      for (uint32_t i = 0; i < n_own && g == 0xFFFFFFFFu; ++i) {
        if (__ldcg(&p.vacant[(uint32_t)bid + (uint32_t)nb * m]) != 0u)
          g = (uint32_t)bid + (uint32_t)nb * m;
        else
          m = m + 1u < n_own ? m + 1u : 0u;
      }
      *reinterpret_cast<volatile unsigned*>(&w.place) = m;
      unsigned most = 0;
      for (int j = W_PAIR; j <= W_BREMS; ++j) {
        const unsigned hd = block_word(w.head[j]), q = block_word(w.tail[j]) - hd;  // the head before the tail
        if (q > most) {
          most = q;
          k = j;
          h = hd;
        }
      }
      n = min(most, 32u);
      if (n && atomicCAS(&w.head[k], h, h + n) != h) n = 0;  // another warp claimed: next time
    }
  }
  n = __shfl_sync(0xffffffffu, n, 0);
  if (n) {
    g = __shfl_sync(0xffffffffu, g, 0);
    h = __shfl_sync(0xffffffffu, h, 0);
    k = __shfl_sync(0xffffffffu, k, 0);
    const uint32_t slot0 = g * 32u + lane;
    const bool vac = g != 0xFFFFFFFFu && slot0 < p.n_slots &&
                     *reinterpret_cast<volatile uint8_t*>(p.trk.status + slot0) == VACANT;
    const unsigned bal = __ballot_sync(0xffffffffu, vac);
    const unsigned c = lane < n ? pop_entry(p, tc, k, h + lane) : kNoEntry;
    const bool stored = c != kNoEntry && (tc.meta(c) & kMetaStored) != 0u;
    const unsigned rank = (unsigned)__popc(__ballot_sync(0xffffffffu, c != kNoEntry && !stored) & lt);
    const bool placed = c != kNoEntry && !stored && rank < (unsigned)__popc(bal);
    const unsigned new_mask = __ballot_sync(0xffffffffu, placed), all = __ballot_sync(0xffffffffu, stored || placed);
    const unsigned rest = __ballot_sync(0xffffffffu, c != kNoEntry && !stored && !placed);
    if (stored || placed) {
      uint32_t slot = tc.home(c);
      if (placed) {  // the vacant slot of its rank
        unsigned left = bal;
        for (unsigned r = rank; r > 0; --r) left &= left - 1u;
        slot = g * 32u + (unsigned)(__ffs(left) - 1);
      }
      store_entry(p, tc, slot, c);
      tc.meta(c) = 0u;
      atomicMin(&w.cursor, ((slot >> 5) - (uint32_t)bid) / (uint32_t)nb);
    }
    if (lane == 0 && new_mask) {
      atomicSub(&p.vacant[g], (unsigned)__popc(new_mask));
      atomicSub(&p.tile_vacant[g >> 3], (unsigned)__popc(new_mask));
    }
    if (rest) push_lanes(p, tc, w.tail, k, rest, c);
    if (all) {
      push_lanes(p, tc, w.tail, W_FREE, all, c);
      if (lane == 0) {
        atomicAdd(&w.parked, (unsigned)__popc(all));
        atomicSub(&w.live, (unsigned)__popc(all));
      }
    }
    __syncwarp();
  }
  if (mine) {
    __threadfence_block();
    atomicExch(&w.filling, 0u);
  }
  __syncwarp();
}

// A fill's wait gives up only if the buffer's protocol is broken: what the lanes
// had claimed is lost to the run, which ends with its error status, and their
// entries, which never held a track, are free again. The whole warp calls it;
// returns how many lanes gave up.
template <int kCap>
__device__ __noinline__ unsigned give_back(const Params& p, const TrackCache<kCap>& tc, BlockWords& w, bool gave_up,
                                           unsigned c) {
  const unsigned lost = (unsigned)__popc(__ballot_sync(0xffffffffu, gave_up));
  const unsigned back = __ballot_sync(0xffffffffu, gave_up && c != kNoEntry);
  if (back) push_lanes(p, tc, w.tail, W_FREE, back, c);
  if ((threadIdx.x & 31u) == 0u) {
    atomicSub(&w.live, lost);
    atomicExch(&w.exit, 1u);
  }
  return lost;
}

// Warps of a block that take pieces of any size; the others take full pieces
// only: small pieces fetch the same instructions for fewer tracks. Measured
// with 1, 2 and 3: 1 GeV calorimeter 1.41, 1.17 and 1.18 ms, 4 T calorimeter
// 4.20, 3.49 and 3.53 ms. A block that holds kManyLive tracks always has a
// full piece waiting (six kinds hold 186 in part-filled ones), and its job ends
// later than its tracks' chains: there every warp takes full pieces only
// (100,000 x 10 GeV 17.6 -> 15.9 ms; 16.4 from 512 tracks on, 15.9 from 850),
// unless interactions wait for buffer space.
constexpr int kAnyPieceWarps = 2;
// Warps of a block that always look for work, and helpers beside them that
// take full pieces only while the block holds at least kManyLive tracks and a
// kind kHelpWaiting of them: they hide each other's fetches where work abounds
// (100,000 x 10 GeV 20.0 -> 18.6 ms), but slow down the chains of a smaller
// job that runs beside them (10,000 x 10 GeV without the first condition 3.3
// -> 4.0 ms).
constexpr int kBaseWarps = 8, kWarpThreads = 512;
constexpr unsigned kHelpWaiting = 64;
// kManyLive by the block's entries: 640 of 1,024 and 400 of 512, above the 186
// tracks that may sit in part-filled pieces (6 materials, 512 entries, 30,000 x
// 3 GeV: 4.85 ms without such a number, 4.71 with 400, 4.78 with 320; 10,000 x
// 10 GeV in 4 T: 3.11, 3.16 and 3.29 ms). Of 256 entries nothing is left
// between: there no block holds many tracks, and the helpers are not launched
// (8 materials, 800 layers, 30,000 x 3 GeV: 16.6 ms, and 20.0 with 205).
template <int kCap>
constexpr unsigned kManyLive = kCap == 1024 ? 640u : (kCap == 512 ? 400u : ~0u);
template <int kCap>
constexpr int kThreads = kCap >= 512 ? kWarpThreads : 32 * kBaseWarps;
// A block with tracks waiting looks at the buffer this often at most (~2 us).
constexpr unsigned kLookCycles = 4000;
// Live tracks a block fills itself up to from the buffer while no full piece
// waits: this part of its share of all tracks alive and queued, at least
// kFillLeast (a least of 32 put a small event's tracks on one block: 12
// particles 0.79 -> 0.69 ms with 2).
constexpr float kFillShare = 0.75f, kFillLeast = 2.0f;
// Entries of a block's track store: the most that fit beside the tables (1,024
// with up to five materials, 512 up to eight, 256 where the planes and materials
// of several hundred layers take the rest).
constexpr int kWarpTracks = 1024, kWarpTracksMid = 512, kWarpTracksSmall = 256;

// Warp sums of the per-lane counts since the last flush (32-bit sums), added
// to the device counters by lane 0. Ended tracks are counted after a fence,
// behind the tail reservations of their interactions (the run's end
// condition).
__device__ __forceinline__ void flush_warp_counts(const Params& p, unsigned& steps, unsigned& killed, unsigned& fill) {
  Ctl* c = p.ctl;
  const unsigned s = __reduce_add_sync(0xffffffffu, steps);  // killed and fill are warp-uniform
  if ((threadIdx.x & 31) == 0) {
    if (s) atomicAdd(&c->steps_total, (unsigned long long)s);
    const long long dalive = (long long)fill - (long long)killed;
    if (dalive != 0) atomicAdd(&c->alive, (unsigned long long)dalive);
    if (killed) {
      __threadfence();
      atomicAdd(&c->finished, (unsigned long long)killed);
    }
  }
  steps = killed = fill = 0;
}

// One thread of an idle warp: true if the block leaves (the run was aborted,
// every track of it has ended, or nothing has stepped for ~1 s, which aborts
// it).
static __device__ __noinline__ bool idle_poll(const Params& p, bool empty, unsigned long long& seen, long long& t_seen) {
  Ctl* ctl = p.ctl;
  if (*reinterpret_cast<volatile unsigned*>(p.barrier + 2) != 0u) return true;
  if (empty) {
    const unsigned long long f = ld_acquire_u64(&ctl->finished);
    if (f == *reinterpret_cast<volatile unsigned long long*>(&ctl->tail)) return true;
  }
  const unsigned long long now_steps = *reinterpret_cast<volatile unsigned long long*>(&ctl->steps_total);
  const long long now = clock64();
  if (now_steps != seen) {
    seen = now_steps;
    t_seen = now;
  } else if (now - t_seen > kBarrierTimeoutCycles) {
    atomicOr(&ctl->error, ERR_NO_PROGRESS);
    atomicOr(p.barrier + 2, ABORT_RUN);
    return true;
  }
  return false;
}

// The loop. Every warp takes up to 32 tracks waiting for the same kind of
// work from the block's queues, runs it and queues them again by what comes
// next; a warp with nothing waiting, or a block holding few tracks, takes
// initializers from the buffer (one warp at a time).
//
// A run with an iteration budget ends by draining: once a warp has run
// `budget` pieces the block stops filling and stepping, runs the pending
// interactions and leaves; its live tracks go back to the slot store between
// two steps, as a synchronous iteration leaves them. A pending interaction
// without buffer space is stored deferred. A run that is aborted (limits, no
// progress) does the same, without the interactions that need the buffer. A
// block that starts with more live tracks than it has entries steps them in
// turns: `parked` of them wait in their slots, and entries that come free take
// them, before any initializer unless the buffer is full. A block that runs out
// of entries while the buffer is full parks tracks too (park_waiting).
template <int kCap>
__global__ void __launch_bounds__(kThreads<kCap>, 1) k_loop_warps(Params p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const TrackCache<kCap> tc{smem_raw};
  const SharedStatic ss = carve_static(p, smem_raw + TrackCache<kCap>::kBytes);
  __shared__ BlockWords w;
  __shared__ unsigned s_drain, s_kind, s_looked, s_deferred;
  __shared__ unsigned s_vacant;
  __shared__ unsigned long long s_pieces;
  const int nb = (int)gridDim.x, bid = (int)blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  Ctl* ctl = p.ctl;
  unsigned* abort_word = p.barrier + 2;
  const uint32_t n_own = (uint32_t)bid < p.n_chunks ? (p.n_chunks - (uint32_t)bid + nb - 1) / nb : 0u;
  const unsigned owned = owned_slots(p, bid, nb, n_own);
  const unsigned n_entries = owned < (unsigned)kCap ? owned : (unsigned)kCap;
  const unsigned long long max_pieces = __ldcg(&ctl->max_iterations);  // per run
  const unsigned long long budget = p.run_budget;
  if (threadIdx.x == 0) s_vacant = 0u;
  __syncthreads();
  {  // the block's vacant slots
    unsigned v = 0;
    for (uint32_t m = threadIdx.x; m < n_own; m += blockDim.x) v += __ldcg(&p.vacant[(uint32_t)bid + (uint32_t)nb * m]);
    v = __reduce_add_sync(0xffffffffu, v);
    if (lane == 0 && v) atomicAdd(&s_vacant, v);
  }
  for (unsigned c = threadIdx.x; c < (unsigned)kCap; c += blockDim.x) {
    tc.meta(c) = 0u;
    for (int k = 0; k < kWarpKinds; ++k) *tc.queue(k, c) = 0u;
    *tc.queue(W_FREE, c) = c < n_entries ? ((1u << 16) | c) : 0u;  // every entry free, lap 0 written
  }
  if (threadIdx.x <= kWarpKinds) {
    w.head[threadIdx.x] = 0u;
    w.tail[threadIdx.x] = threadIdx.x == W_FREE ? n_entries : 0u;
  }
  if (threadIdx.x == 0) {
    w.live = 0u;
    w.filling = 0u;
    w.exit = 0u;
    s_drain = 0u;
    s_pieces = 0ull;
    w.cursor = 0u;
    w.parked = 0u;
    s_kind = (unsigned)W_PHOTON;
    s_deferred = 0u;
    w.place = 0u;
    s_looked = (unsigned)clock64() - 2u * kLookCycles;
  }
  double* thick = reinterpret_cast<double*>(smem_raw + TrackCache<kCap>::kBytes + p.static_bytes);  // layer thicknesses
  for (int l = threadIdx.x; l < p.n_layers; l += blockDim.x) thick[l] = p.zb[l + 1] - p.zb[l];
  stage_static(p, ss);  // ends with a block barrier
  const unsigned live0 = owned - s_vacant;
  if (threadIdx.x == 0) {
    atomicAdd(&ctl->vacant_seen, (unsigned long long)s_vacant);
    if (live0 > n_entries) w.parked = live0;  // they wait in their slots until entries take them
  }
  if (live0 > 0 && live0 <= n_entries) {
    // the live tracks of the block's chunks, one chunk per warp at a time,
    // take the first entries
    for (uint32_t m = (uint32_t)warp; m < n_own; m += blockDim.x >> 5) {
      const uint32_t slot = ((uint32_t)bid + (uint32_t)nb * m) * 32u + (uint32_t)lane;
      const bool live = slot < p.n_slots && p.trk.status[slot] != VACANT;
      const unsigned bal = __ballot_sync(0xffffffffu, live);
      if (bal == 0u) continue;
      unsigned f = 0;
      if (lane == 0) f = atomicAdd(&w.head[W_FREE], (unsigned)__popc(bal));
      f = __shfl_sync(0xffffffffu, f, 0) + (unsigned)__popc(bal & lt);
      unsigned c = kNoEntry;
      int k = W_NONE;
      if (live) {
        c = pop_entry(p, tc, W_FREE, f);
        if (c != kNoEntry) k = load_entry(p, tc, slot, c);
      }
      for (unsigned todo = __ballot_sync(0xffffffffu, k != W_NONE); todo;) {
        const int kk = __shfl_sync(0xffffffffu, k, __ffs(todo) - 1);
        const unsigned m2 = __ballot_sync(0xffffffffu, k == kk);
        push_lanes(p, tc, w.tail, kk, m2, c);
        todo &= ~m2;
      }
    }
    if (threadIdx.x == 0) w.live = live0;
  }
  __syncthreads();
  unsigned steps = 0, killed = 0, fill = 0, events = 0;
  unsigned long long pieces = 0, seen = ~0ull;
  long long t_seen = clock64();
  // Whole-job runs concentrate a block's work in full pieces (throughput);
  // budgeted runs (a serving loop's chunks, interactive stepping) let every
  // warp take any piece, so that no track waits for a free warp (latency).
  const int any_warps = budget == ~0ull ? kAnyPieceWarps : kBaseWarps;
  const bool helper = warp >= kBaseWarps;
  const float inv_nb = 1.0f / (float)nb;
  for (;;) {
    // the loop's flags, read by lane 0 and broadcast: every decision below
    // must be the same for the whole warp (its lanes may arrive here
    // diverged, and a lane leaving alone would strand the others' shuffles)
    unsigned flags = 0;
    if (lane == 0)
      flags = (*reinterpret_cast<volatile unsigned*>(&w.exit) != 0u ? 1u : 0u) |
              (*reinterpret_cast<volatile unsigned*>(&s_drain) != 0u ? 2u : 0u) |
              (*reinterpret_cast<volatile unsigned*>(&w.live) >= kManyLive<kCap> ? 4u : 0u) |
              (*reinterpret_cast<volatile unsigned*>(&s_deferred) != 0u ? 8u : 0u);
    flags = __shfl_sync(0xffffffffu, flags, 0);
    const bool drain = (flags & 3u) != 0u, many = (flags & 4u) != 0u, full_buffer = (flags & 8u) != 0u;
    if (helper && drain) break;
    // the kinds to choose from now: all; draining, the pending interactions;
    // aborted, only those that need no buffer space
    const unsigned allowed = (flags & 1u) ? (1u << W_COMPTON)
                                          : (drain ? (1u << W_COMPTON) | (1u << W_PAIR) | (1u << W_MOLLER) | (1u << W_BREMS)
                                                   : (1u << kWarpKinds) - 1u);
#ifdef CELER_LANE_COUNTERS
    const long long t_round = clock64();
    long long t_read = 0, t_done = 0;
#endif
    // Each of lanes 0..5 looks at one kind. Base warps below any_warps take
    // pieces of any size unless the block holds many tracks, the others full
    // ones only (while draining any warp takes any piece: a warp that leaves
    // the loop may have been the last one allowed to take a small piece): with
    // few tracks alive a block's work is concentrated in full warps instead of
    // spread over many part-filled ones.
    unsigned waiting = 0;
    if (lane < kWarpKinds && ((allowed >> lane) & 1u)) {
      const unsigned hd = *reinterpret_cast<volatile unsigned*>(&w.head[lane]);  // before the tail: hd <= tail
      waiting = *reinterpret_cast<volatile unsigned*>(&w.tail[lane]) - hd;
    }
    constexpr unsigned kMovingKinds = (1u << W_PHOTON) | (1u << W_ELECTRON) | (1u << W_COMPTON);  // make no tracks
    constexpr unsigned kChargedKinds = (1u << W_ELECTRON) | (1u << W_MOLLER) | (1u << W_BREMS);
    const bool any_size = drain || (warp < any_warps && (!many || full_buffer));
    const unsigned full = __ballot_sync(0xffffffffu, waiting >= 32u), some = __ballot_sync(0xffffffffu, waiting > 0u);
    // The kind to take: of those waiting enough, for a warp of any-size pieces
    // charged tracks first (their steps carry a shower's longest chains of
    // dependent steps, the primary crossing layer after layer and radiating,
    // so the job ends sooner when they wait least); for the others the kind
    // the block's last full piece was of, so that the warps run the same code
    // while it is in the instruction cache; then the most waiting. One
    // warp-wide maximum of preference, waiting tracks and 15 - kind.
    // After an interaction found no room in the buffer the kinds that make no
    // tracks come first, and the others only when none of those waits, in the
    // few any-size warps: tracks end and the buffer empties meanwhile. (Taking
    // them as ever, 60,000 x 100 MeV with a buffer of 2^17 entries ended with
    // every track of every block waiting for room; so 2.9 ms, and 2.7 ms with
    // room for all.)
    const unsigned kind_now = *reinterpret_cast<volatile unsigned*>(&s_kind);
    unsigned prefer = any_size ? kChargedKinds : 1u << kind_now, may = any_size ? some : full;
    if (full_buffer && !drain) {
      prefer = kMovingKinds;
      if ((some & kMovingKinds) != 0u || warp >= any_warps) may &= kMovingKinds;
    }
    const unsigned cand =
        (may >> lane) & 1u ? (((prefer >> lane) & 1u) << 24) | (waiting << 4) | (15u - (unsigned)lane) : 0u;
    const unsigned picked = __reduce_max_sync(0xffffffffu, cand);
    const unsigned pick_k = picked != 0u ? 15u - (picked & 15u) : 0xFFu;
    if (helper && (picked == 0u || ((picked >> 4) & 0xFFFFFu) < kHelpWaiting || !many)) {
      if (events != 0u) flush_warp_counts(p, steps, killed, fill);
      events = 0u;
      __nanosleep(10000);
      continue;
    }
    if (!any_size && lane == 0 && pick_k != 0xFFu && pick_k != kind_now)
      *reinterpret_cast<volatile unsigned*>(&s_kind) = pick_k;
    if (drain && pick_k == 0xFFu) break;  // nothing pending: the block's tracks sit between steps
    // no full piece waits (of the charged kinds, if charged tracks wait)
    const bool scarce = (some & kChargedKinds) ? (full & kChargedKinds) == 0u : full == 0u;
    // fill (one warp at a time) when nothing waits, or when no full piece
    // waits and the block holds fewer than its target: few tracks spread over
    // all SMs, many keep every block's pieces full
    unsigned take = 0, f0 = 0;
    unsigned long long first = 0;
    uint32_t load_slot = 0xFFFFFFFFu;  // the lane's parked track to load
    constexpr unsigned kParked = 0xFFFFFFFFu;
    // (interactions wait for buffer space: entries must be taken whatever the
    // target, or no block would make room for another)
    if (full_buffer && !drain && !helper && (some & kMovingKinds) == 0u)
      park_waiting(p, tc, w, bid, nb, n_own);
    bool look = !drain && !helper && (scarce || full_buffer);
    if (look && some != 0u)  // work waits here: look at the buffer every kLookCycles at most
      look = (unsigned)clock64() - *reinterpret_cast<volatile unsigned*>(&s_looked) > kLookCycles;
    if (__any_sync(0xffffffffu, look)) {
      if (lane == 0 && atomicCAS(&w.filling, 0u, 1u) == 0u) {
        const unsigned free_now = *reinterpret_cast<volatile unsigned*>(&w.tail[W_FREE]) -
                                  *reinterpret_cast<volatile unsigned*>(&w.head[W_FREE]);
        const long long a = (long long)*reinterpret_cast<volatile unsigned long long*>(&ctl->avail);
        const long long alive = (long long)*reinterpret_cast<volatile unsigned long long*>(&ctl->alive);
        const unsigned live = *reinterpret_cast<volatile unsigned*>(&w.live);
        const unsigned parked = *reinterpret_cast<volatile unsigned*>(&w.parked);
        if (full_buffer && a < (long long)(p.ring_capacity - p.ring_capacity / 8u))
          *reinterpret_cast<volatile unsigned*>(&s_deferred) = 0u;  // an eighth of it is free again
        // parked tracks come before initializers, unless the buffer is full:
        // then as many of those as the block has slots for
        unsigned spare = 0u;
        if (parked != 0u && full_buffer && a > 0) spare = owned_slots(p, bid, nb, n_own) - live - parked;
        if (parked != 0u && spare == 0u) {
          take = kParked;  // (the lock stays held)
        } else {
          *reinterpret_cast<volatile unsigned*>(&s_looked) = (unsigned)clock64();
          if (a > 0 && free_now > 0) {
            // at least this block's part of the buffer's entries, and up to
            // its target (single precision does for both)
            const float part = (float)a * inv_nb, fill_to = fmaxf(kFillShare * ((float)(alive + a) * inv_nb), kFillLeast);
            float more = fmaxf(ceilf(part), fill_to - (float)live);
            if (some != 0u && (float)live >= fill_to && !full_buffer) more = 0.0f;
            unsigned want = (unsigned)fminf(more, 32.0f);
            if (want > free_now) want = free_now;
            if ((long long)want > a) want = (unsigned)a;
            if (parked != 0u && want > spare) want = spare;
            if (want > 0u) {
              const long long old = (long long)atomicAdd(&ctl->avail, 0ull - (unsigned long long)want);
              if (old >= (long long)want) {
                take = want;
                CELER_LANES_N(LS_FILL, take);
                first = atomicAdd(&ctl->head, (unsigned long long)want);
                atomicAdd(reinterpret_cast<unsigned long long*>(&ctl->room), (unsigned long long)want);
              } else {
                atomicAdd(&ctl->avail, (unsigned long long)want);
              }
            }
          } else if (budget != ~0ull && live == 0u) {
            // a budgeted run, no track here and none to take (tracks enter
            // under this lock only): the rest is left to the next run
            if (a <= 0 || n_entries == 0u) atomicExch(&s_drain, 1u);
          }
        }
        if (take != kParked) {
          if (take > 0) {
            f0 = atomicAdd(&w.head[W_FREE], take);  // only the filler claims free entries
            atomicAdd(&w.live, take);
          }
          __threadfence_block();
          atomicExch(&w.filling, 0u);
        }
      }
      take = __shfl_sync(0xffffffffu, take, 0);
      if (take == kParked) load_slot = claim_parked_chunk(p, w, bid, nb, n_own, full_buffer, take, f0);
    }
    unsigned c = kNoEntry;
    int out = W_NONE;
    unsigned n = 0;
    bool fresh = false;  // the lane's track needs a number of mean free paths
    unsigned meta = 0;
    TrackRng rng(p.seed, 0u, 0ull, 0u);
    if (take > 0) {
      first = __shfl_sync(0xffffffffu, first, 0);
      f0 = __shfl_sync(0xffffffffu, f0, 0);
      const unsigned loads = __ballot_sync(0xffffffffu, load_slot != 0xFFFFFFFFu);
      if (loads) {
        __threadfence_block();
        if (load_slot != 0xFFFFFFFFu) {
          c = pop_entry(p, tc, W_FREE, f0 + (unsigned)__popc(loads & lt));
          if (c != kNoEntry) out = load_entry(p, tc, load_slot, c);
        }
        // (they were counted alive already)
      } else {
        fill += take;
        if ((unsigned)lane < take) {
          c = pop_entry(p, tc, W_FREE, f0 + (unsigned)lane);
          const unsigned long long index = first + (unsigned)lane, i = index & p.ring_mask;
          const unsigned code = ring_lap_code(p, index) + 1u;
          if (c != kNoEntry && ring_wait(p, index, code)) {
            const InitParts r = get_record(p.ring.rec + i);
            tc.x(c) = r.xy.x;
            tc.y(c) = r.xy.y;
            tc.z(c) = r.zu.x;
            tc.ux(c) = r.zu.y;
            tc.uy(c) = r.uu.x;
            tc.uz(c) = r.uu.y;
            tc.E(c) = r.et.x;
            const unsigned long long tid = (unsigned long long)__double_as_longlong(r.et.y);
            tc.tid(c) = tid;
            tc.event(c) = r.m.x;
            tc.primary(c) = r.m.y;
            meta = kMetaLive | (r.m.w << 24) | r.m.z;
            st_release_u32(p.ring_state + i, code + 1u);
            rng = TrackRng(p.seed, r.m.x, tid, 0u);
            fresh = true;
            out = r.m.w == GAMMA ? W_PHOTON : W_ELECTRON;
          }
        }
        if (__any_sync(0xffffffffu, (unsigned)lane < take && out == W_NONE)) {
          fill -= give_back(p, tc, w, (unsigned)lane < take && out == W_NONE, c);
          if (out == W_NONE) c = kNoEntry;
        }
      }
    } else if (pick_k != 0xFFu) {
      // claim up to 32 tracks of kind pick_k
      unsigned h = 0;
      if (lane == 0) {
        for (int a = 0; a < 8; ++a) {
          h = *reinterpret_cast<volatile unsigned*>(&w.head[pick_k]);
          const unsigned q = *reinterpret_cast<volatile unsigned*>(&w.tail[pick_k]) - h;
          if (q == 0) break;
          const unsigned want = q < 32u ? q : 32u;
          if (atomicCAS(&w.head[pick_k], h, h + want) == h) {
            n = want;
            break;
          }
        }
      }
      n = __shfl_sync(0xffffffffu, n, 0);
      if (n == 0) continue;
      h = __shfl_sync(0xffffffffu, h, 0);
      if ((unsigned)lane < n) c = pop_entry(p, tc, (int)pick_k, h + (unsigned)lane);
#ifdef CELER_LANE_COUNTERS
      __syncwarp();
      t_read = clock64();
#endif
      if (pick_k == W_PHOTON) {
        out = fly_photons(p, tc, ss, thick, c, steps);
      } else if (pick_k == W_ELECTRON) {
        out = step_electrons(p, tc, ss, c, steps);
      } else if (c != kNoEntry) {
        meta = tc.meta(c);
        rng = TrackRng(p.seed, tc.event(c), tc.tid(c), tc.ctr(c));
        if (pick_k == W_COMPTON)
          out = compton_piece(p, tc, c, rng, n >= kFewTracks ? kComptonAttempts : kMaxAttempts);
        else if (pick_k == W_PAIR)
          out = pair_piece(p, tc, c, rng);
        else if (pick_k == W_MOLLER)
          out = moller_piece(p, tc, c, rng);
        else
          out = brems_piece(p, tc, c, rng);
        fresh = out == W_PHOTON || out == W_ELECTRON;
      }
#ifdef CELER_LANE_COUNTERS
      __syncwarp();
      t_done = clock64();
#endif
    }
    if (take > 0 || n > 0) {
      if (fresh) renew(p, tc, c, meta, rng);
      __syncwarp();
      // a track whose interaction found no buffer space waits in its queue
      // (draining: in its entry, to be stored deferred)
      const bool waits = c != kNoEntry && out == W_NONE;
      const bool deferred = __any_sync(0xffffffffu, waits);
      if (deferred && lane == 0) *reinterpret_cast<volatile unsigned*>(&s_deferred) = 1u;
      if (waits && !drain) out = (int)pick_k;
      const unsigned ended = __ballot_sync(0xffffffffu, out == W_FREE);
      if (out == W_FREE) {
        const unsigned m = tc.meta(c);
        tc.meta(c) = 0u;
        const uint32_t ev = tc.event(c);
        atomicSub(&p.event_live[row_of(p, ev)], 1u);
        if (m & kMetaStored) {
          const uint32_t slot = tc.home(c);
          p.trk.action[slot] = A_NONE;
          __threadfence_block();  // park_waiting may take the slot as soon as it is vacant
          *reinterpret_cast<volatile uint8_t*>(p.trk.status + slot) = VACANT;
          atomicAdd(&p.vacant[slot >> 5], 1u);
          atomicAdd(&p.tile_vacant[slot >> 8], 1u);
        }
      }
      if (ended) {
        killed += (unsigned)__popc(ended);
        if (lane == 0) atomicSub(&w.live, (unsigned)__popc(ended));
      }
      for (unsigned todo = __ballot_sync(0xffffffffu, out != W_NONE); todo;) {
        const int kk = __shfl_sync(0xffffffffu, out, __ffs(todo) - 1);
        const unsigned m2 = __ballot_sync(0xffffffffu, out == kk);
        push_lanes(p, tc, w.tail, kk, m2, c);
        todo &= ~m2;
      }
#ifdef CELER_LANE_COUNTERS
      // pieces by kind, and those of photons, electrons and Compton
      // scatterings in three parts: choice and claim, the steps, the requeue
      __syncwarp();
      if (lane == 0) {
        const long long t_end = clock64();
        constexpr int key_of_kind[kWarpKinds] = {K_G_GEOM, K_E_GEOM, K_G_COMPTON, K_G_PAIR, K_E_MOLLER, K_E_BREMS};
        const int site = take > 0 ? (int)LS_FILL : LS_PIECE + key_of_kind[pick_k];
        if (take == 0) lane_site_n(site, n);
        lane_cycles(site, t_end - t_round);
        const int t3 = take > 0 ? -1
                                : (pick_k == W_PHOTON ? (int)LS_T_PHOTON
                                                      : (pick_k == W_ELECTRON ? (int)LS_T_ELECTRON
                                                                              : (pick_k == W_COMPTON ? (int)LS_T_COMPTON : -1)));
        if (t3 >= 0) {
          const long long part[3] = {t_read - t_round, t_done - t_read, t_end - t_done};
          for (int j = 0; j < 3; ++j) {
            lane_site_n(t3 + j, n);
            lane_cycles(t3 + j, part[j]);
          }
        }
      }
#endif
      if ((++events & 15u) == 0) {  // and whenever the warp idles
        flush_warp_counts(p, steps, killed, fill);
        // (a warp that never idles sees here that another block ended the run)
        if ((events & 63u) == 0 && lane == 0 && *reinterpret_cast<volatile unsigned*>(abort_word) != 0u)
          atomicExch(&w.exit, 1u);
      }
      if (take > 0) continue;
      ++pieces;
      if (pieces >= budget && lane == 0) atomicExch(&s_drain, 1u);
      if (pieces >= max_pieces && lane == 0) {
        atomicOr(&ctl->error, ERR_ITERATIONS);
        atomicOr(abort_word, ABORT_RUN);
        atomicExch(&w.exit, 1u);
      }
      // a piece without deferrals made progress; one with deferrals (the
      // buffer is full) goes on to the idle path: watchdog and a pause
      if (!deferred) continue;
    }
    // nothing done: leave if every track has ended, else poll (bounded)
    flush_warp_counts(p, steps, killed, fill);
    if (lane == 0) {
      const bool empty = *reinterpret_cast<volatile unsigned*>(&w.live) == 0u &&
                         *reinterpret_cast<volatile unsigned*>(&w.parked) == 0u;
      if (idle_poll(p, empty && budget == ~0ull, seen, t_seen)) atomicExch(&w.exit, 1u);
      __nanosleep(500);
#ifdef CELER_LANE_COUNTERS
      lane_site_n(LS_IDLE, 0u);
      lane_cycles(LS_IDLE, clock64() - t_round);
#endif
    }
    __syncwarp();
  }
  flush_warp_counts(p, steps, killed, fill);
  if (lane == 0) atomicMax(&s_pieces, pieces);
  __syncthreads();
  const unsigned live = w.live;
  if (live > 0)
    store_tracks(p, tc, reinterpret_cast<uint16_t*>(const_cast<unsigned*>(tc.queue(0, 0u))), n_entries, bid, nb);
  if (threadIdx.x == 0) end_async_block(p, nb, s_pieces);
}
