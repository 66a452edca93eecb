// The asynchronous step loop (CELER_LOOP_ASYNC) of the block-pass policies:
// the persistent kernel in which every block runs its own passes with no
// grid barrier (k_loop_async), the kernel that sets the buffer entries' states
// (k_async_prepare), and the waits and accesses of the per-warp schedule's
// queues (warp_loop.cuh) with their check (k_queue_wait_probe). Included by step.cu
// inside its anonymous namespace, after the block passes (local_pass,
// data_pass) and the buffer protocol (ring_wait, take_initializer) it uses.
#pragma once

// Block-wide sums of a pass's counts (every thread gets them).
__device__ PassCounts block_total(const PassCounts& n) {
  __shared__ unsigned long long s_n[4];
  if (threadIdx.x < 4) s_n[threadIdx.x] = 0;
  __syncthreads();
  unsigned long long v[4] = {n.killed, n.n_def, n.steps, n.fill};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    if ((threadIdx.x & 31) == 0 && v[k] != 0) atomicAdd(&s_n[k], v[k]);
  }
  __syncthreads();
  const PassCounts out{s_n[0], s_n[1], s_n[2], s_n[3]};
  __syncthreads();  // s_n is reused by the next call
  return out;
}

// The buffer entries' states from head and tail (entries in [head, tail)
// written and unread, the others free for their next writer) and the count of
// ended tracks, head - alive (every track came from a buffer entry; a pair
// photon that reuses its parent's slot continues the parent's count). An
// asynchronous run leaves all of it as the next one needs it, and so do the
// kernels that queue primaries; only after iterations of the synchronous
// loops, which keep neither, or an error is it made anew (32 MB of states at
// 2^20 slots, 10 us).
__global__ void k_async_prepare(Params p) {
  const unsigned long long head = p.ctl->head, tail = p.ctl->tail;
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long j = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; j < p.ring_capacity;
       j += stride) {
    const unsigned long long index = head + ((j - head) & p.ring_mask);  // the index in [head, head + capacity) at j
    p.ring_state[j] = ring_lap_code(p, index) + (index < tail ? 1u : 0u);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    p.ctl->finished = head - p.ctl->alive;
    p.ctl->avail = tail - head;
    p.ctl->room = (long long)(p.ring_capacity - (tail - head));
    p.ctl->async_passes = 0;
    p.ctl->vacant_seen = 0;
    p.ctl->done_x = 0u;
  }
}

// Live tracks a block of the asynchronous loop fills itself up to when
// entries are queued (it takes at least ceil(queued / blocks) in any case):
// a few per warp keeps every sub-partition busy without lengthening the pass.
constexpr unsigned kAsyncFill = 32;

// ---- waits and accesses of the per-warp schedule's shared-memory queues
// (warp_loop.cuh): an entry holds a 16-bit state in its high half.

// Bounded wait of one thread for a shared-memory queue entry to reach
// `state` (as ring_wait).
__device__ __noinline__ bool wq_wait_poll(const Params& p, volatile unsigned* e, unsigned state, long long timeout) {
  const long long t0 = clock64();
  for (;;) {
    __nanosleep(20);
    if ((*e >> 16) == state) return true;
    if (clock64() - t0 > timeout) {
      atomicOr(p.barrier + 2, ABORT_WAIT);
      atomicOr(&p.ctl->error, ERR_BARRIER_TIMEOUT);
      return false;
    }
  }
}
__device__ __forceinline__ bool wq_wait(const Params& p, volatile unsigned* e, unsigned state,
                                        long long timeout = kBarrierTimeoutCycles) {
  return (*e >> 16) == state || wq_wait_poll(p, e, state, timeout);
}

// Block-scope release store and acquire load of a shared-memory word.
__device__ __forceinline__ void st_release_cta(volatile unsigned* a, unsigned v) {
  const unsigned s = (unsigned)__cvta_generic_to_shared((const void*)a);
  asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(s), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned ld_acquire_cta(volatile unsigned* a) {
  const unsigned s = (unsigned)__cvta_generic_to_shared((const void*)a);
  unsigned v;
  asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(s) : "memory");
  return v;
}

// End of one block's part of an asynchronous run (one thread, after its last
// counter update): its passes, and in the last block to leave the run's
// totals.
__device__ __forceinline__ void end_async_block(const Params& p, int nb, unsigned long long passes) {
  Ctl* c = p.ctl;
  atomicMax(&c->async_passes, passes);
  __threadfence();
  if (atomicAdd(&c->done_x, 1u) == (unsigned)nb - 1u) {
    __threadfence();
    c->iteration = __ldcg(&c->iteration) + __ldcg(&c->async_passes);
    const unsigned long long queued = __ldcg(&c->tail) - __ldcg(&c->head), alive = __ldcg(&c->alive);
    // (the per-warp schedule's blocks count their vacant slots themselves)
    if (p.run_budget != 0ull && __ldcg(&c->vacant_seen) != c->total_vacant) atomicOr(&c->error, ERR_VACANCY);
    c->vacant_seen = 0;
    c->total_vacant = (unsigned long long)p.n_slots - alive;
    c->cont = (alive + queued > 0 && __ldcg(&c->error) == 0u) ? 1u : 0u;
    c->async_passes = 0;
    c->done_x = 0u;
  }
}

// The asynchronous block loop of the block-pass policies (LOCAL, DATA): one
// cooperative launch in which every block runs its own passes over its own
// chunks with no grid barrier. At the start of a pass a block claims
// written entries on an availability count (atomic, undone if short) and
// takes their indices from the head: ceil(queued / blocks) or enough to hold
// kAsyncFill live tracks, at most its vacant slots. Secondaries are reserved on
// the count of free entries (reserve_entries), and each entry's state word orders
// its writer and its reader. A track's steps and draws do not depend
// on where or when it runs (its random stream is keyed by its own id), so
// histories are those of the synchronous loops; only the tally summation
// order differs. The run ends when every track taken from the buffer has
// ended (finished reaches tail), or, with an iteration budget, when every
// block has run that many passes or holds no track. Every wait is bounded: a block with nothing to do polls, and if
// no track anywhere steps for ~1 s it sets ERR_NO_PROGRESS and the abort
// word; all blocks leave at their next pass. The last block to leave adds
// the most passes (pieces) any block ran to the iteration count.
__global__ void __launch_bounds__(kTile, 1) k_loop_async(Params p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const SharedStatic ss = carve_static(p, smem_raw);
  stage_static(p, ss);
  const int nb = (int)gridDim.x, bid = (int)blockIdx.x;
  Ctl* c = p.ctl;
  unsigned* abort_word = p.barrier + 2;
  __shared__ unsigned long long s_first;
  __shared__ unsigned s_take, s_vtot;
  __shared__ int s_go;  // 0 leave, 1 nothing to do yet, 2 run a pass
  const uint32_t n_own = (uint32_t)bid < p.n_chunks ? (p.n_chunks - (uint32_t)bid + nb - 1) / nb : 0u;
  const bool owns_last = n_own > 0 && (uint32_t)bid + (uint32_t)nb * (n_own - 1u) == p.n_chunks - 1u;
  const unsigned owned = n_own * 32u - (owns_last ? p.n_chunks * 32u - p.n_slots : 0u);
  const unsigned quota_cap = block_quota_cap(p.policy);
  unsigned long long passes = 0, seen = ~0ull;
  const unsigned long long max_passes = __ldcg(&c->max_iterations);  // per run
  const unsigned long long budget_end = __ldcg(&c->budget_end);
  const unsigned long long budget = budget_end == ~0ull ? ~0ull : budget_end - __ldcg(&c->iteration);
  long long t_seen = clock64();
  if (threadIdx.x == 0) {
    s_vtot = __ldcg(&p.block_vacant[bid]);
    if (__ldcg(&c->local_blocks) != (unsigned)nb) {  // vacancy counts made for another grid
      atomicOr(&c->error, ERR_VACANCY);
      atomicOr(abort_word, ABORT_RUN);
    }
  }
  __syncthreads();
  // thread 0: no track anywhere stepped for ~1 s
  auto watchdog = [&]() {
    const unsigned long long now_steps = *reinterpret_cast<volatile unsigned long long*>(&c->steps_total);
    const long long now = clock64();
    if (now_steps != seen) {
      seen = now_steps;
      t_seen = now;
    } else if (now - t_seen > kBarrierTimeoutCycles) {
      atomicOr(&c->error, ERR_NO_PROGRESS);
      atomicOr(abort_word, ABORT_RUN);
    }
  };
  for (;;) {
    __syncthreads();  // every thread has read the previous decision
    if (threadIdx.x == 0) {
      int go = 1;
      unsigned take = 0;
      unsigned long long first = 0;
      const unsigned vtot = s_vtot;
      if (*reinterpret_cast<volatile unsigned*>(abort_word) != 0u || passes >= budget) {
        go = 0;  // aborted, or the run's budget of passes is spent
      } else {
        // claim `want` written entries on the availability count (undone if
        // there were fewer), then their indices on the head: at least
        // ceil(avail / blocks), and up to kAsyncFill live tracks in the block
        const unsigned room = vtot < quota_cap ? vtot : quota_cap;
        const long long a = (long long)*reinterpret_cast<volatile unsigned long long*>(&c->avail);
        if (room > 0 && a > 0) {
          const unsigned live = owned - vtot;
          unsigned long long want = ((unsigned long long)a + (unsigned long long)nb - 1ull) / (unsigned long long)nb;
          const unsigned long long fill_up = live < kAsyncFill ? (unsigned long long)(kAsyncFill - live) : 0ull;
          if (want < fill_up) want = fill_up < (unsigned long long)a ? fill_up : (unsigned long long)a;
          if (want > room) want = room;
          const long long old = (long long)atomicAdd(&c->avail, 0ull - want);
          if (old >= (long long)want) {
            take = (unsigned)want;
            first = atomicAdd(&c->head, want);
            atomicAdd(reinterpret_cast<unsigned long long*>(&c->room), want);
          } else {
            atomicAdd(&c->avail, want);
          }
        }
        if (take > 0 || vtot < owned) {
          go = 2;
        } else if (budget != ~0ull) {
          go = 0;  // a budgeted run: nothing here now, the rest is left to the next run
        } else {
          const unsigned long long f = ld_acquire_u64(&c->finished);
          if (f == *reinterpret_cast<volatile unsigned long long*>(&c->tail)) go = 0;  // every track has ended
        }
      }
      s_go = go;
      s_take = take;
      s_first = first;
    }
    __syncthreads();
    const int go = s_go;
    if (go == 0) break;
    if (go == 1) {
      if (threadIdx.x == 0) {
        watchdog();
        __nanosleep(1000);  // about a microsecond between polls of the shared counters
      }
      continue;
    }
    const PassPlan pl{s_first, s_take, s_vtot, true, false, 0u};
    PassCounts n{0, 0, 0, 0};
    if (p.policy == POLICY_DATA)
      data_pass<true>(p, bid, nb, ss, pl, n);
    else
      local_pass<true>(p, bid, nb, ss, pl, n);
    const PassCounts tot = block_total(n);
    if (threadIdx.x == 0) {
      if (tot.fill != pl.quota) atomicOr(&c->error, ERR_VACANCY);
      s_vtot = (unsigned)((long long)pl.vtot + (long long)tot.killed - (long long)tot.fill);
      if (tot.steps) atomicAdd(&c->steps_total, tot.steps);
      const long long dalive = (long long)tot.fill - (long long)tot.killed;
      if (dalive != 0) atomicAdd(&c->alive, (unsigned long long)dalive);
      if (tot.killed) {
        __threadfence();  // the block's reservations on the tail precede its count of ended tracks
        atomicAdd(&c->finished, tot.killed);
      }
      ++passes;
      if (passes >= max_passes) {
        atomicOr(&c->error, ERR_ITERATIONS);
        atomicOr(abort_word, ABORT_RUN);
      }
      if (tot.steps == 0) watchdog();
    }
  }
  if (threadIdx.x == 0) {
    p.block_vacant[bid] = s_vtot;
    end_async_block(p, nb, passes);
  }
}

// Check of the queue waits of the asynchronous loop: one thread waits for
// an entry to be written, either buffer entry 0 (which = 0, 2) or an entry
// of a shared-memory queue (which = 1, 3). For which = 0, 1 nothing writes
// it, so the wait must give up after `timeout` cycles, set the abort word
// and ERR_BARRIER_TIMEOUT; for which = 2, 3 it was written first and the
// wait must pass.
__global__ void k_queue_wait_probe(Params p, int which, long long timeout) {
  __shared__ unsigned s_e;
  if (threadIdx.x == 0) {
    s_e = (which & 2) ? (1u << 16) : 0u;  // lap 0: 0 free, 1 written
    if (which & 2) p.ring_state[0] = 1u;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (which & 1)
      wq_wait(p, &s_e, 1u, timeout);
    else
      ring_wait(p, 0ull, 1u, timeout);
  }
}

