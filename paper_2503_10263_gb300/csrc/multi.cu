// multi.cu - persistent transport kernel over many requests (batched and
// served forms of the transport step).
//
// The event itself is the same as in the single-run kernel (event.cuh).  What
// differs is where work comes from and where it goes: every particle carries
// its request slot; idle lanes take their warp's products, then products from
// the shared ring, then primaries of any request whose current pass still has
// unclaimed primaries (a bitmap of slots); each request moves pass 1 ->
// target fields -> pass 2 -> final tallies inside the kernel, started by the
// lane whose atomic decrement emptied the request's pass.  A batch is a launch
// with every request published before it starts; a server keeps the launch
// running while the host publishes requests into free slots.
#include "event.cuh"
#include "multi.cuh"

namespace karl {

__device__ __forceinline__ int ld_acquire_i(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_i(int* p, int v) {
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// cross section from the channel-major table (target-field builder)
__device__ double sigma_cm(const double* sig, int n, double e_min, double log_ratio_h, double loss,
                           double e) {
  if (!(e > loss)) return 0.0;
  double x = log(e / e_min) / log_ratio_h;
  int i = (int)floor(x);
  double f;
  if (i < 0) { i = 0; f = 0.0; }
  else if (i > n - 2) { i = n - 2; f = 1.0; }
  else f = x - (double)i;
  return (1.0 - f) * sig[i] + f * sig[i + 1];
}

// Sums along z run one column a lane with ROWS rows of loads in flight (the
// sum is serial, the loads are not).
constexpr int ROWS = 8;

// out[row] = pt[row] + sum of rg up to row for the columns [32 u, 32 u + 32) of
// the time tally's (species, energy bin) pairs
__device__ void time_columns(const Params& P, unsigned long long* out, int u, int lane) {
  const int nz = P.nz, ntb = P.ntb, col = 32 * u + lane;
  if (col >= NSP * ntb) return;
  const size_t at = (size_t)(col / ntb) * (nz + 2) * ntb + col % ntb;
  const unsigned long long *pt = P.time_pt + at, *rg = P.time_rg + at;
  out += at;
  unsigned long long acc = 0;
  for (int row = 0; row < nz + 2; row += ROWS) {
    unsigned long long a[ROWS], b[ROWS];
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
      const size_t k = (size_t)min(row + i, nz + 1) * ntb;
      a[i] = rg[k];
      b[i] = pt[k];
    }
#pragma unroll
    for (int i = 0; i < ROWS; ++i)
      if (row + i < nz + 2) {
        acc += a[i];
        out[(size_t)(row + i) * ntb] = b[i] + acc;
      }
  }
}

// face crossings: one (direction, species) a lane
__device__ void cross_columns(const Params& P, const SlotDesc& d, int lane) {
  if (lane >= 2 * NSP) return;
  const int nz = P.nz, sp = lane % NSP;
  const unsigned long long* rg = (lane < NSP ? P.xpos_rg : P.xneg_rg) + (size_t)sp * (nz + 2);
  unsigned long long* out = (lane < NSP ? d.cpos_out : d.cneg_out) + (size_t)sp * (nz + 1);
  unsigned long long acc = 0;
  for (int k = 0; k <= nz; k += ROWS) {
    unsigned long long a[ROWS];
#pragma unroll
    for (int i = 0; i < ROWS; ++i) a[i] = rg[min(k + i, nz)];
#pragma unroll
    for (int i = 0; i < ROWS; ++i)
      if (k + i <= nz) out[k + i] = acc += a[i];
  }
}

// target fields of the recombination channels in segments [32 u, 32 u + 32)
// (Eq. target_field_density): the electron's partner density, or the sum over
// the electron field's energy bins of n sigma v for an ion; sigma and v of a
// bin are worked out by one lane for all
__device__ void field_rates(const Params& P, const SlotDesc& d, int u, int lane) {
  const int nz = P.nz, ntb = P.ntb, j = 32 * u + lane;
  const int jj = min(j, nz - 1);
  const double inv_qt = 1.0 / Q_T, tv = d.tsim * d.vol;
  for (int k = 0; k < P.nch; ++k) {
    const ChanDev& ch = P.ch[k];
    if (ch.kind != RECOMBINATION) continue;
    const unsigned long long* tj = d.time1 + ((size_t)ch.sout * (nz + 2) + (jj + 1)) * ntb;
    double acc = 0.0;
    for (int b0 = 0; b0 < ntb; b0 += 32) {
      double sg = 0.0, v = 0.0;
      if (ch.sin != SP_E && b0 + lane < ntb) {
        const int b = b0 + lane;
        const double eb = P.e_min * exp(P.log_ratio_h * (P.n_energy - 1) * (b + 0.5) / ntb);
        const double x = eb * P.inv_mass[SP_E];
        v = C_LIGHT * sqrt(x * (2.0 + x)) / (1.0 + x);
        sg = sigma_cm(d.sig_cm + (size_t)k * P.n_energy, P.n_energy, P.e_min, P.log_ratio_h,
                      ch.loss_ev, eb);
      }
      const int nb = min(32, ntb - b0);
      for (int i = 0; i < nb; ++i) {
        const unsigned long long tt = tj[b0 + i];
        const double n = tt ? div_call((double)tt * inv_qt, tv) : 0.0;
        const double sb = __shfl_sync(FULL, sg, i), vb = __shfl_sync(FULL, v, i);
        if (ch.sin == SP_E) acc = __dadd_rn(acc, n);
        else acc = __fma_rn(__dmul_rn(n, sb), vb, acc);
      }
    }
    if (j < nz) d.fpair[((size_t)k * (nz + 1) + j) * 2 + 1] = acc;
  }
}

// their columns, one channel a lane
__device__ void field_columns(const Params& P, const SlotDesc& d, int lane) {
  const int nz = P.nz;
  if (lane >= P.nch || P.ch[lane].kind != RECOMBINATION) return;
  double* f = d.fpair + (size_t)lane * (nz + 1) * 2;       // (column, rate) pairs
  double c = 0.0;
  f[0] = 0.0;
  for (int j = 0; j < nz; j += ROWS) {
    double a[ROWS];
#pragma unroll
    for (int i = 0; i < ROWS; ++i) a[i] = f[2 * min(j + i, nz - 1) + 1];
#pragma unroll
    for (int i = 0; i < ROWS; ++i)
      if (j + i < nz) f[2 * (j + i + 1)] = c = __fma_rn(a[i], P.dz, c);
  }
}

// densities, fields and currents (Eq. target_field_density, Sec. 2.3) of the
// 32 (species, segment) pairs and faces from 32 u
__device__ void normalise(const Params& P, const SlotDesc& d, int u, int lane) {
  const int nz = P.nz, ntb = P.ntb, t = 32 * u + lane;
  const double inv_qt = 1.0 / Q_T, tv = d.tsim * d.vol;
  if (t < NSP * nz) {
    const int sp = t / nz, j = t % nz;
    const size_t at = ((size_t)sp * (nz + 2) + (j + 1)) * ntb;
    const unsigned long long* to = d.time_out + at;
    const unsigned long long* t1 = (d.n_passes == 2 ? d.time1 : d.time_out) + at;
    double* field = d.field + ((size_t)sp * nz + j) * ntb;
    double tsum = 0.0;
    for (int b = 0; b < ntb; ++b) {
      tsum = __fma_rn((double)to[b], inv_qt, tsum);
      const unsigned long long tt = t1[b];
      field[b] = tt ? div_call((double)tt * inv_qt, tv) : 0.0;
    }
    d.density[(size_t)sp * nz + j] =
        tsum / tv - (double)P.recomb[(size_t)sp * nz + j] / d.vol;
  }
  if (t < NSP * (nz + 1))
    d.current[t] = ((double)d.cpos_out[t] - (double)d.cneg_out[t]) / (d.area * d.tsim);
}

__device__ __forceinline__ int task_units(const SlotDesc& d, int phase) {
  const int nz = d.P[0].nz, groups = (NSP * d.P[0].ntb + 31) / 32;
  switch (phase) {
    case TASK_TIME1: return groups;
    case TASK_FIELD: return (nz + 31) / 32;
    case TASK_COLUMN: return 1;
    case TASK_TIME2: return groups + 1;
    case TASK_NORM: return (NSP * (nz + 1) + 31) / 32;
  }
  return 0;
}

// The end of pass p of request s: publish the work that follows it.  One
// lane; the request is alive until that work completes, so its generation is
// current.  Called where the lane sees the pass empty and not kept for the end
// of its iteration: a lane can empty two passes in one, that of a primary born
// dead and that of the parked particle it takes next.
__device__ __noinline__ void end_pass(SlotDesc* D, SlotCtl* C, MultiCtl* M, int s, int p) {
  const int gen_bits = ld_acquire_i(&C[s].state) & ~0xff;
  const int from = gen_bits | (p == 1 ? SLOT_PASS1 : SLOT_PASS2);
  if (atomicCAS(&C[s].state, from, gen_bits | SLOT_TRANS) != from) return;
  C[s].task_done = 0;
  __threadfence();
  const int phase = p == 1 && D[s].n_passes == 2 ? TASK_TIME1 : TASK_TIME2;
  atomicExch(&C[s].task, (unsigned long long)phase << 32);
  atomicOr(&M->taskmap[s >> 5], 1u << (s & 31));
  atomicAdd(&M->tasks, 1);
}

// Take one unit of the work between the passes and do it, the whole warp;
// false if there was none.  A unit belongs to the phase that the claim itself
// returned, and a phase ends only when all of its units are done, so a late
// claim finds either units of the current phase or none.  (One warp did all of
// a request's work before: about 20 ms after pass 1 and 13 ms after pass 2 at
// 1000 segments and 64 energy bins, in which nothing of the request ran.)
__device__ __noinline__ bool do_task(SlotDesc* D, SlotCtl* C, MultiCtl* M, int lane) {
  int s = -1, phase = TASK_NONE, u = 0, units = 0;
  if (lane == 0) {
    for (int i = 0; i < MAX_SLOTS / 32 && phase == TASK_NONE; ++i) {
      unsigned bits = (unsigned)ld_relaxed_i((const int*)&M->taskmap[i]);
      while (bits && phase == TASK_NONE) {
        s = i * 32 + __ffs(bits) - 1;
        bits &= bits - 1;
        const unsigned long long w = ld_acquire(&C[s].task);
        if (!(w >> 32) || (int)(unsigned)w >= task_units(D[s], (int)(w >> 32))) continue;
        const unsigned long long old = atomicAdd(&C[s].task, 1ULL);
        __threadfence();                        // the descriptor of that phase's request
        const int n = task_units(D[s], (int)(old >> 32));
        if ((int)(unsigned)old < n) {
          phase = (int)(old >> 32);
          u = (int)(unsigned)old;
          units = n;
        }
      }
    }
  }
  phase = __shfl_sync(FULL, phase, 0);
  if (phase == TASK_NONE) return false;
  __threadfence();                              // what the units before it wrote
  s = __shfl_sync(FULL, s, 0);
  u = __shfl_sync(FULL, u, 0);
  const SlotDesc& d = D[s];
  const Params& P = d.P[phase == TASK_TIME1 || d.n_passes == 1 ? 0 : 1];
  switch (phase) {
    case TASK_TIME1: time_columns(P, d.time1, u, lane); break;
    case TASK_FIELD: field_rates(d.P[0], d, u, lane); break;
    case TASK_COLUMN: field_columns(d.P[0], d, lane); break;
    case TASK_TIME2:
      if (u + 1 < task_units(d, TASK_TIME2)) time_columns(P, d.time_out, u, lane);
      else cross_columns(P, d, lane);
      break;
    case TASK_NORM: normalise(P, d, u, lane); break;
  }
  __syncwarp();
  __threadfence_system();
  if (lane == 0 && (int)atomicAdd(&C[s].task_done, 1u) + 1 == units) {
    __threadfence();
    C[s].task_done = 0;
    __threadfence();
    if (phase == TASK_TIME1 || phase == TASK_FIELD || phase == TASK_TIME2) {
      atomicExch(&C[s].task, (unsigned long long)(phase + 1) << 32);
    } else {
      const int gen_bits = ld_acquire_i(&C[s].state) & ~0xff;
      atomicExch(&C[s].task, 0ULL);
      atomicAnd(&M->taskmap[s >> 5], ~(1u << (s & 31)));
      atomicAdd(&M->tasks, -1);
      if (phase == TASK_COLUMN) {
        *(volatile int*)&C[s].pass = 2;
        __threadfence();
        st_release_i(&C[s].state, gen_bits | SLOT_PASS2);
        atomicAdd(&M->c.prim_next, (unsigned long long)d.n_prim);
        atomicOr(&M->bitmap[s >> 5], 1u << (s & 31));
      } else {
        int* flag = d.done_flag;
        st_release_i(&C[s].state, gen_bits | SLOT_DONE);
        atomicAdd(&M->done_count, 1ULL);
        __threadfence_system();
        *(volatile int*)flag = 1;
        __threadfence_system();
      }
    }
  }
  __syncwarp();
  return true;
}

// A pass of request s empties when a decrement of its word leaves no live
// particle and every primary claimed.
__device__ __forceinline__ bool pass_emptied(unsigned long long old, unsigned long long dec,
                                             long long n_prim) {
  return word_live(old) == dec && word_next(old) >= n_prim;
}

// Claim up to k primaries of the current pass of the request in slot s, whose
// state the caller read as st (a pass state).  The claim is a compare-and-swap
// on the pass word that adds the same count to the next primary and to the
// live particles, only while the word carries the generation of st and
// primaries remain, so it never takes primaries past the end and never
// touches a later request in the slot.  Returns the count claimed (0 if
// none) and the first index; clears the slot's bit when it takes the last.
__device__ __forceinline__ int claim_primaries(SlotDesc* D, SlotCtl* C, MultiCtl* M, int s, int st,
                                               int k, unsigned long long* first) {
  const int p = state_kind(st) == SLOT_PASS2 ? 2 : 1;
  unsigned long long* word = &C[s].word[p - 1];
  // the descriptor of the generation read in st (admission writes the new
  // generation's pass words before its descriptor, so a newer descriptor
  // comes with a newer word, which the generation test below rejects)
  const long long n = (long long)ld_acquire((const unsigned long long*)&D[s].n_prim);
  const unsigned long long gen = (unsigned long long)(state_gen(st) & 31u);
  unsigned long long old = ld_acquire(word);
  for (int tries = 0; tries < 64; ++tries) {
    if (word_gen(old) != gen) return 0;               // the slot holds another request now
    const long long next = word_next(old);
    const long long left = n - next;
    if (left <= 0) return 0;                          // every primary of this pass claimed
    const int g = left < k ? (int)left : k;
    const unsigned long long nw =
        old + ((unsigned long long)g << WORD_NEXT_SHIFT) + (unsigned long long)g;
    const unsigned long long prev = atomicCAS(word, old, nw);
    if (prev == old) {
      if (next + g >= n) atomicAnd(&M->bitmap[s >> 5], ~(1u << (s & 31)));
      *first = (unsigned long long)next;
      return g;
    }
    old = prev;
  }
  return 0;                                           // contended: look elsewhere
}

// bps: blocks resident on an SM (gridDim.x is a multiple of it).  Measured with
// the schedule of transport.cu, the work between passes in units and the
// out-of-line rare path, one launch each, FP32 / FP64: one request of 1000
// decays 49 -> 14 / 57 -> 21 ms, 16 requests of 1e3 to 3e4 decays 345 -> 107 /
// 444 -> 147 ms, 32 of 1e3 to 1e5 606 -> 439 / 685 -> 616 ms.
template <bool F32>
__global__ void __launch_bounds__(256, 2) multi_kernel(SlotDesc* D, SlotCtl* C, MultiCtl* M, Ring R,
                                                    const volatile int* cancel,
                                                    unsigned long long timeout_ns, int bps) {
  const unsigned long long deadline = globaltimer_ns() + timeout_ns;
  __shared__ WarpQueue wq[WARPS];
  __shared__ RareBuf rbuf[WARPS];
  if (threadIdx.x < WARPS) {
    wq[threadIdx.x].top = 0;
    rbuf[threadIdx.x].n = 0;
    rbuf[threadIdx.x].r = 0;
  }
  __syncthreads();
  Control* ctl = &M->c;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  WarpQueue& Q = wq[threadIdx.x >> 5];
  RareBuf& Rb = rbuf[threadIdx.x >> 5];
  bool has = false;
  Lane L;
  L.slot = 0;
  const Params* Pl = &D[0].P[0];
  const RecordCols cols{};
  EventOut o;
  o.flights = o.colls = o.recoil = o.excit = 0;
  o.chan = -1;
  unsigned long long idle_iters = 0, busy_iters = 0, busy_lane_iters = 0, started = 0;
  unsigned idle_ns = 128;
  // a warp that holds particles but found nothing for its idle lanes skips
  // its next refill attempts (1, 3, 7, ... up to 63 iterations)
  int refill_skip = 0, refill_backoff = 0;
  RingPort port;
  port.R = &R;
  port.ctl = ctl;
  port.deadline = deadline;
  port.q = &Q;
  port.spilled = 0;
  port.slot_live = nullptr;

  // The schedule is the single-run kernel's (transport.cu): places this warp
  // holds in ctl->active without a particle (credit), warps taking part (those
  // of rank below T, in steps of one per scheduler over the SM's blocks),
  // particles handed to the ring by the others once no primary is left.
  const int nwarps = blockDim.x >> 5;
  const int step = max(1, 4 / bps);
  const int rank_w = ((threadIdx.x >> 5) + nwarps -
                      (step * (blockIdx.x / max(1, gridDim.x / bps))) % nwarps) % nwarps;
  const long long step_lanes = 32LL * step * gridDim.x;
  const long long all_lanes = (long long)gridDim.x * blockDim.x;
  int credit = 0, T = step, quota = 32;
  bool drained = false, share = false, eager = false, idle = false;

  // The lane's particle names its request and pass.  (The descriptor is the
  // one its claim or its parent was bound to: a particle taken from the ring
  // comes with an acquire of its cell.)
  auto second = [&]() { return (L.slot & SECOND) != 0; };
  auto slot_of = [&]() { return L.slot & (SECOND - 1); };
  auto bind = [&]() { Pl = &D[slot_of()].P[second()]; };
  // per-lane sums belong to the request of the lane's particle: they go to
  // its ledger whenever the lane lets the particle go (death, park, hand-back)
  auto flush_sums = [&]() {
    unsigned long long* led = Pl->ledger;
    if (o.flights) {
      atomicAdd(led + L_N_FLIGHT, o.flights);
      atomicAdd(led + L_N_FLIGHT_ALL, o.flights);
    }
    if (o.colls) {
      atomicAdd(led + L_N_COLL, o.colls);
      atomicAdd(led + L_N_COLL_ALL, o.colls);
    }
    if (o.recoil) atomicAdd(led + L_LOSS_RECOIL, o.recoil);
    if (o.excit) atomicAdd(led + L_LOSS_EXCIT, o.excit);
    o.flights = o.colls = o.recoil = o.excit = 0;
  };

  for (long long iter = 0;; ++iter) {
    if ((iter & 15) == 0 || idle) {
      int word = 0;
      if (lane == 0) {
        int stop = 0;
        if (ld_relaxed_i(&ctl->abort)) stop = 1;
        else if (cancel && ld_relaxed_i((const int*)cancel)) {
          atomicCAS(&ctl->error, 0, ERR_CANCELLED);
          atomicExch(&ctl->abort, 1);
          stop = 1;
        } else if (globaltimer_ns() > deadline) {
          atomicCAS(&ctl->error, 0, ERR_TIMEOUT);
          atomicExch(&ctl->abort, 1);
          stop = 1;
        }
        // adopt requests the host has published since the last look
        unsigned long long pub = ld_acquire(&M->published);
        unsigned long long ad = ld_relaxed(&M->adopted);
        while (ad < pub) {                       // (not once LEFT is set)
          const unsigned long long old = atomicCAS(&M->adopted, ad, ad + 1);
          if (old == ad) {
            const int s = (int)ld_acquire_i((const int*)&M->pubq[ad % MAX_SLOTS]);
            // (requests without primaries are finished by the host, never published)
            if (state_kind(ld_acquire_i(&C[s].state)) == SLOT_PASS1) {
              atomicAdd(&ctl->prim_next, ld_acquire((const unsigned long long*)&D[s].n_prim));
              atomicOr(&M->bitmap[s >> 5], 1u << (s & 31));
            }
            ++ad;
          } else {
            ad = old;
          }
        }
        const unsigned long long h = ld_relaxed(&ctl->head), t = ld_relaxed(&ctl->tail);
        const long long left = max(0LL, (long long)ld_relaxed(&ctl->prim_next));
        const long long act = ld_relaxed_s(&ctl->active);
        const long long alive = max(0LL, act - credit) + (t > h ? (long long)(t - h) : 0LL) + left;
        int n = T;
        while (n < nwarps && alive * 20 > step_lanes * (n / step) * 19) n += step;
        while (n > step && alive * 10 < step_lanes * (n / step - 1) * 7) n -= step;
        const long long places = (long long)gridDim.x * min(n, nwarps);
        const int qt = alive >= 32 * places ? 32 : (int)max(1LL, (alive + places - 1) / places);
        const int dr = left == 0;
        const int sh = dr && t - h < (unsigned long long)step_lanes &&
                       alive * 50 < all_lanes * 49;
        const int eg = alive < all_lanes;
        const int tk = ld_relaxed_i(&M->tasks) > 0;
        word = stop | (dr << 1) | (sh << 2) | (eg << 3) | (t > h ? 16 : 0) | (tk << 5) |
               (qt << 8) | (n << 16);
        if (credit > 0)
          atomicAdd((unsigned long long*)&ctl->active, (unsigned long long)(-(long long)credit));
      }
      credit = 0;
      word = __shfl_sync(FULL, word, 0);
      if (word & 1) break;
      drained = (word & 2) != 0;
      share = (word & 4) != 0;
      eager = (word & 8) != 0;
      if (word & 16) refill_skip = 0;             // the ring has work
      quota = (word >> 8) & 0xff;
      T = word >> 16;
      // work between the passes: units as long as there are any for an idle
      // warp, one for a warp with particles waiting
      if (word & 32)
        while (do_task(D, C, M, lane) && idle) {}
    }
    const bool serves = rank_w < T;

    // ---- warps from T on hand what they hold to the ring ----
    __syncwarp();
    if (!serves && drained) {
      const unsigned m = __ballot_sync(FULL, has);
      const int k = __popc(m), q = min(Q.top, WQ), r = Rb.r, tot = k + q + r;
      if (tot > 0) {
        unsigned long long pos = 0;
        if (lane == 0) pos = atomicAdd(&ctl->tail, (unsigned long long)tot);
        pos = __shfl_sync(FULL, pos, 0);
        if (has) {
          flush_sums();
          ring_put(R, ctl, pos + __popc(m & lt), L, deadline);
          started -= 1;                           // counted again when taken
          has = false;
        }
        if (lane < q) ring_put(R, ctl, pos + k + lane, Q.s[lane], deadline);
        if (lane < r) {
          ring_put(R, ctl, pos + k + q + lane, Rb.s[RB - r + lane], deadline);
          started -= 1;
        }
        __syncwarp();
        if (lane == 0) {
          Q.top = 0;
          Rb.r = 0;
          port.spilled += tot;
        }
        credit += tot;
        __syncwarp();
      }
    }

    // ---- idle lanes first resume particles handed back for a batch ----
    if (Rb.r > 0) {
      const unsigned needr = __ballot_sync(FULL, !has);
      const int r0 = Rb.r;
      const int tr = min(__popc(needr), r0);
      if (!has) {
        const int rank = __popc(needr & lt);
        if (rank < tr) {
          L = Rb.s[RB - r0 + rank];
          has = true;
          bind();
        }
      }
      __syncwarp();
      if (lane == 0) Rb.r = r0 - tr;
      __syncwarp();
    }

    // ---- idle lanes take the warp's own products first (newest first) ----
    int qleft;
    {
      const unsigned need0 = __ballot_sync(FULL, !has);
      const int top = Q.top;
      const int take = min(__popc(need0), top);
      if (!has) {
        const int rank = __popc(need0 & lt);
        if (rank < take) {
          L = Q.s[top - 1 - rank];
          has = true;
          started += 1;
          bind();
        }
      }
      qleft = top - take;
      if (share && qleft > 0) {
        unsigned long long pos = 0;
        if (lane == 0) pos = atomicAdd(&ctl->tail, (unsigned long long)qleft);
        pos = __shfl_sync(FULL, pos, 0);
        if (lane < qleft) ring_put(R, ctl, pos + lane, Q.s[lane], deadline);
        if (lane == 0) port.spilled += qleft;
        credit += qleft;
        qleft = 0;
      }
      __syncwarp();
      if (lane == 0) Q.top = qleft;
      __syncwarp();
    }

    // ---- other idle lanes: products from the ring, then primaries of a request ----
    unsigned need = serves ? __ballot_sync(FULL, !has) : 0u;
    if (need && need != FULL && refill_skip > 0) {
      --refill_skip;
      need = 0;
    }
    if (need) {
      const int k = __popc(need);
      const int spare = max(0, RING_BATCH - qleft);
      unsigned long long base = 0;
      int got = 0, src = 0, gslot = 0, gpass = 1, cr = credit;
      if (lane == 0) {
        unsigned long long h = ld_relaxed(&ctl->head), t = ld_relaxed(&ctl->tail);
        const unsigned long long ready = h < t ? t - h : 0ULL;
        const unsigned long long fair = ready / (2ULL * gridDim.x * nwarps);
        const int extra = fair <= (unsigned long long)k
                              ? 0
                              : (fair - k < (unsigned long long)spare ? (int)(fair - k) : spare);
        for (int tries = 0; tries < 16 && h < t; ++tries) {
          const unsigned long long want = (unsigned long long)(k + extra);
          unsigned long long take = t - h < want ? t - h : want;
          unsigned long long old = atomicCAS(&ctl->head, h, h + take);
          if (old == h) { base = h; got = (int)take; src = 1; break; }
          h = old;
          t = ld_relaxed(&ctl->tail);
        }
        const int room = max(0, min(k, quota - (32 - k)));
        if (got == 0 && !drained && room > 0) {
          // A request with unclaimed primaries.  The search starts at a slot
          // chosen by the block, so the warps of a block keep to one request
          // while it lasts and its parameters and column tables stay in L1.
          const unsigned long long pub = ld_relaxed(&M->published);
          const unsigned long long dn = ld_relaxed(&M->done_count);
          const unsigned long long act = pub > dn ? pub - dn : 1ULL;
          const int s0 = (int)((unsigned long long)blockIdx.x % (act < MAX_SLOTS ? act : MAX_SLOTS));
          for (int i = 0; i <= MAX_SLOTS / 32 && got == 0; ++i) {
            const int wi = ((s0 >> 5) + i) & (MAX_SLOTS / 32 - 1);
            unsigned bits = (unsigned)ld_relaxed_i((const int*)&M->bitmap[wi]);
            if (i == 0) bits &= ~0u << (s0 & 31);                       // from s0 on
            else if (i == MAX_SLOTS / 32) bits &= ~(~0u << (s0 & 31));  // wrapped: below s0
            while (bits && got == 0) {
              const int bit = __ffs(bits) - 1;
              bits &= bits - 1;
              const int s = wi * 32 + bit;
              const int st = ld_acquire_i(&C[s].state);
              if (state_kind(st) != SLOT_PASS1 && state_kind(st) != SLOT_PASS2) continue;
              // Only the claim that takes the last primaries clears the bit; a
              // claim on a pass that has ended takes nothing and leaves the bit
              // alone (the end of pass 1 sets it again for pass 2).  The taking
              // claim holds live particles, so the pass cannot end before its
              // clear.
              unsigned long long first = 0;
              const int g = claim_primaries(D, C, M, s, st, room, &first);
              if (g > 0) {
                got = g;
                base = first;
                src = 2;
                gslot = s;
                gpass = state_kind(st) == SLOT_PASS2 ? 2 : 1;
                atomicAdd(&ctl->prim_next, (unsigned long long)(-(long long)g));
              }
            }
          }
        }
        cr -= got;
        if (cr < 0) {
          atomicAdd((unsigned long long*)&ctl->active, (unsigned long long)(-(long long)cr));
          cr = 0;
        }
      }
      base = __shfl_sync(FULL, base, 0);
      got = __shfl_sync(FULL, got, 0);
      src = __shfl_sync(FULL, src, 0);
      gslot = __shfl_sync(FULL, gslot, 0);
      gpass = __shfl_sync(FULL, gpass, 0);
      credit = __shfl_sync(FULL, cr, 0);
      if (got == 0) {
        refill_backoff = refill_backoff * 2 + 1;
        if (refill_backoff > 63) refill_backoff = 63;
        refill_skip = refill_backoff;
      } else {
        refill_backoff = 0;
      }
      bool born_dead = false;
      if (!has && got > 0) {
        const int rank = __popc(need & lt);
        if (rank < got) {
          const unsigned long long idx = base + rank;
          if (src == 1) {
            has = ring_get(R, ctl, idx, L, deadline);
            if (has) bind();
          } else {
            Pl = &D[gslot].P[gpass - 1];
            const Params& P = *Pl;
            L.z = P.pz[idx];
            L.eq = quant_e(P.pe[idx]);
            L.mu = P.pmu[idx];
            L.sp = P.psp[idx];
            L.node = 0;
            L.tal = 0.0;
            L.ev = 0;
            L.pid = (unsigned long long)P.pid_offset + idx;
            L.j = segment_of(P, L.z);
            L.slot = gslot | (gpass == 2 ? SECOND : 0);
            sadd(P.ledger + L_E_IN_PRIMARY, L.eq);
            sadd(P.ledger + L_BIRTHS + L.sp, 1);
            if (L.sp == SP_E && L.eq < P.ecut_q) {
              die<F32>(P, P.ledger, L, R_CUTOFF, L_E_CUTOFF);
              born_dead = true;
              __threadfence();
              const unsigned long long o2 =
                  atomicAdd(&C[gslot].word[gpass - 1], (unsigned long long)0 - 1ULL);
              if (pass_emptied(o2, 1ULL, D[gslot].n_prim)) {
                __threadfence();
                end_pass(D, C, M, gslot, gpass);
              }
            } else {
              has = true;
            }
          }
          started += 1;
        }
      }
      credit += __popc(__ballot_sync(FULL, born_dead));
      if (got > k)                                  // more than the idle lanes: to the queue
        qleft = ring_to_queue(R, ctl, base + k, got - k, Q, qleft, deadline);
    }

    // ---- parked rare collisions: once enough have gathered, free lanes and
    // then busy ones -- whose particles wait in the slots the batch frees --
    // perform them together (fewer once no primary is left, one by one while
    // the particles do not fill the chip) ----
    __syncwarp();
    int rk = -1;
    const int nr = min(Rb.n, RB - Rb.r);
    const unsigned hm = __ballot_sync(FULL, has);
    const bool batch = nr >= (drained ? RB_TRIGGER_LATE : RB_TRIGGER) ||
                       (nr > 0 && (hm == 0 || eager));
    if (batch) {
      const int nfree = 32 - __popc(hm);
      const int rank = has ? nfree + __popc(hm & lt) : __popc(~hm & lt);
      const bool take = rank < nr;
      const bool give = take && has;
      Lane back;
      if (give) {
        flush_sums();                              // the lane changes particle
        back = L;
      }
      if (take) {
        L = Rb.s[nr - 1 - rank];
        rk = Rb.ch[nr - 1 - rank];
        has = true;
        bind();
      }
      __syncwarp();                                // every parked slot has been read
      const int r0 = Rb.r;
      if (give) Rb.s[RB - r0 - 1 - (rank - nfree)] = back;   // stays counted as live
      __syncwarp();
      if (lane == 0) {
        Rb.r = r0 + max(nr - nfree, 0);
        Rb.n = 0;
      }
      __syncwarp();
    }

    // ---- one event ----
    bool died = false;
    const unsigned busy = __ballot_sync(FULL, has);
    idle = !busy;
    if (busy) {
      idle_ns = 128;
      busy_lane_iters += __popc(busy);
      ++busy_iters;
      o.rare = -1;
      if (has && rk < 0) {
        event<F32>(*Pl, *Pl, cols, Pl->ledger, L, o);
        if (!o.alive) {
          has = false;
          died = true;
        } else if (o.rare >= 0) {
          const int i = atomicAdd(&Rb.n, 1);
          if (i < RB - Rb.r) {
            Rb.s[i] = L;
            Rb.ch[i] = (int8_t)o.rare;
            has = false;
            flush_sums();
          } else {
            rk = o.rare;
          }
        }
      }
      if (has && rk >= 0) {
        port.slot_live = &C[slot_of()].word[second()];
        Lane Mv = L;
        EventOut m;
        m.alive = true;
        m.recoil = 0;
        rare_kinematics<F32>(*Pl, Pl->ledger, Mv, m, port, rk);
        L = Mv;
        o.recoil += m.recoil;
        if (!m.alive) {
          has = false;
          died = true;
        }
      }
      __syncwarp();
      const int qtop = min(Q.top, WQ);
      __syncwarp();
      if (lane == 0) {
        Q.top = qtop;
        if (Rb.n > RB - Rb.r) Rb.n = RB - Rb.r;
      }
      // channel counts, one add per distinct (request, channel) per warp
      const unsigned mc = __ballot_sync(FULL, o.chan >= 0);
      if (o.chan >= 0) {
        const unsigned key = ((unsigned)L.slot << 5) | (unsigned)o.chan;
        const unsigned grp = __match_any_sync(mc, key);
        if (lane == __ffs(grp) - 1)
          atomicAdd(Pl->chan_count + o.chan, (unsigned long long)__popc(grp));
      }
      o.chan = -1;
      __syncwarp();                               // other lanes' counts before a lane's death
      if (died) {
        flush_sums();
        __threadfence();                          // its tallies before its death
        const unsigned long long o2 =
            atomicAdd(&C[slot_of()].word[second()], (unsigned long long)0 - 1ULL);
        if (pass_emptied(o2, 1ULL, D[slot_of()].n_prim)) {
          __threadfence();
          end_pass(D, C, M, slot_of(), second() ? 2 : 1);
        }
      }
      credit += __popc(__ballot_sync(FULL, died)) - (qtop - qleft);
      if (credit < 0) {
        if (lane == 0)
          atomicAdd((unsigned long long*)&ctl->active, (unsigned long long)(-(long long)credit));
        credit = 0;
      }
    }

    if (!busy) {
      // leave when the host has closed the session and every published
      // request is done (multi.cuh, LEFT)
      int done = 0;
      if (lane == 0) {
        if (credit > 0)
          atomicAdd((unsigned long long*)&ctl->active, (unsigned long long)(-(long long)credit));
        unsigned long long ad = ld_relaxed(&M->adopted);
        if (!(ad & LEFT) && ld_relaxed_i(&M->shutdown) && ad == ld_acquire(&M->published) &&
            ld_relaxed(&M->done_count) >= ad) {
          const unsigned long long old = atomicCAS(&M->adopted, ad, ad | LEFT);
          ad = old == ad ? ad | LEFT : old;
        }
        done = (ad & LEFT) != 0;
      }
      credit = 0;
      if (__shfl_sync(FULL, done, 0)) break;
      __nanosleep(idle_ns);
      if (idle_ns < 8192) idle_ns <<= 1;
      ++idle_iters;
    }
  }

  unsigned long long sp = port.spilled, st = started;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    sp += __shfl_down_sync(FULL, sp, off);
    st += __shfl_down_sync(FULL, st, off);
  }
  if (lane == 0) {
    atomicAdd(&ctl->idle_iters, idle_iters);
    atomicAdd(&ctl->busy_iters, busy_iters);
    atomicAdd(&ctl->busy_lane_iters, busy_lane_iters);
    atomicAdd(&ctl->spilled, sp);
    atomicAdd(&ctl->particles, st);
  }
}

cudaError_t launch_multi(bool f32, SlotDesc* D, SlotCtl* C, MultiCtl* M, const Ring& R,
                         const volatile int* cancel, unsigned long long timeout_ns, int grid,
                         int block, int bps, cudaStream_t st) {
  if (f32)
    multi_kernel<true><<<grid, block, 0, st>>>(D, C, M, R, cancel, timeout_ns, bps);
  else
    multi_kernel<false><<<grid, block, 0, st>>>(D, C, M, R, cancel, timeout_ns, bps);
  return cudaGetLastError();
}

cudaError_t multi_occupancy(bool f32, int block, int* blocks_per_sm) {
  if (f32)
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, multi_kernel<true>, block, 0);
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, multi_kernel<false>, block, 0);
}

}  // namespace karl
