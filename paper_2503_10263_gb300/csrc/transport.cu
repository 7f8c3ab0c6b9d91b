// transport.cu - persistent Monte Carlo transport kernel of the KARL hot path.
//
// One launch runs one pass over all primaries of a run (Sec. 2.1 main cycle,
// Fig. 1).  Every lane holds one particle in registers and performs one event
// per loop iteration: a free flight by optical depth (Eqs. mean_free_path and
// distance_from_mfp over the piecewise-constant column, equal in law to the
// segment-stop mover of Sec. 3.1), the time/density and current tallies of
// Secs. 2.2-2.3 as range adds, the terminator of Sec. 3.2, a channel chosen
// with probability sigma_i n_i / sum_j sigma_j n_j, and its kinematics
// (Sec. 3.3).  Products go to their warp's queue and, past its end or when
// lanes elsewhere are idle, to a device-wide ring; lanes whose particle ended
// take the next one from their queue, from the ring or from the primaries.
// All waits are bounded by iteration counts and a wall-clock deadline, after
// which the kernel records an error and returns.
#include <type_traits>

#include "event.cuh"

namespace karl {

// ---------------------------------------------------------------------------
// persistent kernel

// The column tables in the block's dynamic shared memory, one after the
// other: gas column and faces (nz + 1 each), density and its inverse (nz
// each), the inverse column, then column and rate of each field channel from
// the channel's offset.
struct StagedCols {
  const double* at;
  __device__ __forceinline__ double col(const Params&, int k) const { return at[k]; }
  __device__ __forceinline__ double face(const Params& P, int k) const { return at[P.nz + 1 + k]; }
  __device__ __forceinline__ double n(const Params& P, int j) const { return at[2 * P.nz + 2 + j]; }
  __device__ __forceinline__ double invn(const Params& P, int j) const { return at[3 * P.nz + 2 + j]; }
  __device__ __forceinline__ int ginv(const Params& P, int q) const {
    return ((const int*)(at + 4 * P.nz + 2))[q];
  }
  __device__ __forceinline__ double fcol(const Params& P, int c, int k) const {
    return at[P.foff[c] + k];
  }
  __device__ __forceinline__ double frate(const Params& P, int c, int j) const {
    return at[P.foff[c] + P.nz + 1 + j];
  }
};

__device__ __forceinline__ void stage_tables(const Params& P, double* at) {
  const int nz = P.nz;
  int* ginv = (int*)(at + 4 * nz + 2);
  for (int i = threadIdx.x; i <= nz; i += blockDim.x) {
    at[i] = P.colgas[i];
    at[nz + 1 + i] = P.faces[i];
  }
  for (int i = threadIdx.x; i < nz; i += blockDim.x) {
    at[2 * nz + 2 + i] = P.nseg[i];
    at[3 * nz + 2 + i] = P.invn[i];
  }
  if (P.ginv)
    for (int i = threadIdx.x; i <= P.nq; i += blockDim.x) ginv[i] = P.ginv[i];
  for (int c = 0; c < P.nch; ++c) {
    if (!P.fcol[c]) continue;
    double* f = at + P.foff[c];
    for (int i = threadIdx.x; i <= nz; i += blockDim.x) f[i] = P.fcol[c][i];
    for (int i = threadIdx.x; i < nz; i += blockDim.x) f[nz + 1 + i] = P.frate[c][i];
  }
}

// STAGED: the column tables fit the block's shared memory (dyn_doubles of it).
// The parameters are read from the constant bank and the staged columns at
// offsets of the block's shared memory, without a pointer; nothing takes the
// particle's address but copies on the rare paths, which are out of line.
// (With the parameters behind a shared-memory reference and the particle in
// local memory, the FP32 form's pass 1 took 28.2 ms at 1e5 decays, 26.1
// without, and 25.7 since the conversions are done on the bits; 3e5 decays at
// 3.1e21 m^-2 47, 42 and 40.5 ms.  The FP64 form, held by its FP64
// instructions, gained 1 %.)
template <bool F32, bool STAGED>
__global__ void __launch_bounds__(512, 1)
    transport_kernel(const __grid_constant__ Params P, const __grid_constant__ Ring R,
                     Control* ctl, const volatile int* cancel, unsigned long long timeout_ns,
                     int dyn_doubles) {
  const unsigned long long deadline = globaltimer_ns() + timeout_ns;
  if (threadIdx.x == 0 && ld_relaxed(&ctl->t_start) == 0)
    atomicCAS(&ctl->t_start, 0ULL, deadline - timeout_ns);
  // dynamic shared memory: the staged tables (dyn_doubles), then one product
  // queue and one batch of parked collisions per warp of the block
  extern __shared__ double dyn[];
  __shared__ Shared S;
  __shared__ Params SP;                           // for the functions out of line
  const int nwarps = blockDim.x >> 5;
  WarpQueue* wq = (WarpQueue*)(dyn + dyn_doubles);
  RareBuf* rbuf = (RareBuf*)(wq + nwarps);
  for (int i = threadIdx.x; i < LEDGER; i += blockDim.x) S.ledger[i] = 0;
  for (int i = threadIdx.x; i < MAXCH; i += blockDim.x) S.chan[i] = 0;
  if (threadIdx.x < nwarps) {
    wq[threadIdx.x].top = 0;
    rbuf[threadIdx.x].n = 0;
    rbuf[threadIdx.x].r = 0;
  }
  if (threadIdx.x == 0) SP = P;
  if (STAGED) stage_tables(P, dyn);
  __syncthreads();
  typename std::conditional<STAGED, StagedCols, GlobalCols>::type cols;
  if constexpr (STAGED) cols.at = dyn;

  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  WarpQueue& Q = wq[threadIdx.x >> 5];
  RareBuf& Rb = rbuf[threadIdx.x >> 5];
  const int wid = threadIdx.x >> 5;
  bool has = false;
  Lane L;
  EventOut o;
  o.flights = 0;
  o.colls = 0;
  o.recoil = 0;
  o.excit = 0;
  o.chan = -1;
  unsigned long long started = 0;
  unsigned long long idle_iters = 0, busy_iters = 0, busy_lane_iters = 0;
  unsigned idle_ns = 128;
  // A warp that still holds particles but found nothing for its idle lanes
  // skips its next refill attempts (1, 3, 7, ... up to 63 iterations): once
  // the primaries are used up, warps with a few long histories left would
  // otherwise contend for the ring head on every iteration.
  int refill_skip = 0, refill_backoff = 0;
  RingPort port;
  port.R = &R;
  port.ctl = ctl;
  port.deadline = deadline;
  port.q = &Q;
  port.spilled = 0;
  port.slot_live = nullptr;

  // ctl->active counts the particles the warps hold (lanes, queues, parked
  // collisions) plus each warp's `credit`: places counted there that hold
  // nothing now.  Deaths raise the credit, refills and products use it up
  // before they add to the counter, and what is left is returned at the next
  // look at the counters, so most deaths and refills take no global atomic.
  int credit = 0;
  // Warps of a block that take part, in steps of four (warp w of a block runs
  // on scheduler w mod 4).  A warp's FP64 instruction takes its scheduler's
  // pipe for 64 cycles whatever its active lanes, so particles that do not
  // fill the chip go to as few warps per scheduler as hold them: a run of few
  // primaries starts with an equal share (`quota`) on every participating
  // warp, and once the primaries are used up the warps from T on hand their
  // particles to the shared ring, where those below T take them.  T follows
  // the number of particles alive: up when 95 % of the places of the warps
  // below it are taken, down when the particles fill 70 % of the next fewer.
  // Measured with the claims of up to RING_BATCH below, pass 1 of the source
  // run: 1e5 decays FP64 144.8 -> 73 ms, FP32 108 -> 41 ms, 1e6 decays FP64
  // 524 -> 484 ms, 1e3 decays FP64 13.0 -> 8.5 ms.
  const long long step_lanes = 128LL * gridDim.x;
  int T = 4;
  while (T < nwarps && step_lanes * (T >> 2) < P.n_prim) T += 4;
  const long long first_warps = (long long)gridDim.x * min(T, nwarps);
  const int quota = (int)min(32LL, (P.n_prim + first_warps - 1) / first_warps);
  bool drained = false;       // every primary is claimed
  bool share = false;         // idle lanes elsewhere: surplus products go to the ring
  bool eager = false;         // parked collisions go at once
  bool idle = false;          // the last iteration found no particle

  for (long long iter = 0;; ++iter) {
    if ((iter & 15) == 0 || idle) {
      // lane 0 reads the counters and decides for the warp
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
        const unsigned long long h = ld_relaxed(&ctl->head), t = ld_relaxed(&ctl->tail);
        const long long pn = (long long)ld_relaxed(&ctl->prim_next);
        const long long act = ld_relaxed_s(&ctl->active);
        const long long left = max(0LL, P.n_prim - pn);
        const long long alive = max(0LL, act - credit) + (t > h ? (long long)(t - h) : 0LL) + left;
        int n = T;
        while (n < nwarps && alive * 20 > step_lanes * (n >> 2) * 19) n += 4;
        while (n > 4 && alive * 10 < step_lanes * ((n >> 2) - 1) * 7) n -= 4;
        const int dr = left == 0;
        const int sh = dr && t - h < (unsigned long long)step_lanes &&
                       alive * 50 < 32LL * gridDim.x * nwarps * 49;
        // The last histories set the end of the pass: once the particles no
        // longer fill the chip, parked collisions go at once so that those
        // histories are not held up.
        const int eg = alive < (long long)gridDim.x * blockDim.x;
        word = stop | (dr << 1) | (sh << 2) | (eg << 3) | (t > h ? 16 : 0) | (n << 8);
        if (credit > 0) {
          __threadfence();
          atomicAdd((unsigned long long*)&ctl->active, (unsigned long long)(-(long long)credit));
        }
      }
      credit = 0;
      word = __shfl_sync(FULL, word, 0);
      if (word & 1) break;
      drained = (word & 2) != 0;
      share = (word & 4) != 0;
      eager = (word & 8) != 0;
      if (word & 16) refill_skip = 0;             // the ring has work
      T = word >> 8;
    }
    const bool serves = wid < T;

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
        }
      }
      __syncwarp();
      if (lane == 0) Rb.r = r0 - tr;
      __syncwarp();
    }

    // ---- idle lanes take the warp's own products first (newest first) ----
    int qleft;                                    // products left in the queue
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
        }
      }
      qleft = top - take;
      // surplus products go to the shared ring while lanes elsewhere are idle
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

    // ---- other idle lanes take work: products from the ring, then primaries ----
    unsigned need = serves ? __ballot_sync(FULL, !has) : 0u;
    if (need && need != FULL && refill_skip > 0) {
      --refill_skip;
      need = 0;
    }
    if (need) {
      const int k = __popc(need);
      unsigned long long rbase = 0, pbase = 0;
      int rgot = 0, pgot = 0, cr = credit;
      // With a long ring a warp takes up to half its even share of it in one
      // claim: what its lanes have no room for waits in its queue.  (One
      // claim per few particles held the whole chip to about 11 particles a
      // microsecond, a fifth of what 75-event histories use up.)
      const int spare = max(0, RING_BATCH - qleft);
      if (lane == 0) {
        // Count the lanes as active only when work is visible, then claim it:
        // idle warps that find nothing leave the counter alone.  Lanes the
        // ring cannot fill take primaries in the same step -- also when a
        // contended claim on the ring fails -- unless the ring is three
        // quarters full (products first, so it cannot overflow).  Holding
        // lanes back for a ring only a quarter full left a quarter of the
        // FP32 form's lanes idle while every warp fought for the ring head.
        unsigned long long h = ld_relaxed(&ctl->head), t = ld_relaxed(&ctl->tail);
        const unsigned long long pn = drained ? (unsigned long long)P.n_prim
                                              : ld_relaxed(&ctl->prim_next);
        const int room = max(0, quota - (32 - k));          // primaries this warp may take
        const bool prim_work = pn < (unsigned long long)P.n_prim && room > 0 &&
                               (h >= t || t - h < R.cap / 4 * 3);
        const unsigned long long ready = h < t ? t - h : 0ULL;
        const unsigned long long fair = ready / (2ULL * gridDim.x * nwarps);
        const int extra = fair <= (unsigned long long)k
                              ? 0
                              : (fair - k < (unsigned long long)spare ? (int)(fair - k) : spare);
        const unsigned long long all = ready + (prim_work ? room : 0);
        const int want = all < (unsigned long long)(k + extra) ? (int)all : k + extra;
        if (want > 0) {
          if (cr < want) {
            atomicAdd((unsigned long long*)&ctl->active, (unsigned long long)(want - cr));
            __threadfence();
            cr = want;
          }
          for (int tries = 0; tries < 16 && h < t; ++tries) {
            unsigned long long take =
                t - h < (unsigned long long)want ? t - h : (unsigned long long)want;
            unsigned long long old = atomicCAS(&ctl->head, h, h + take);
            if (old == h) { rbase = h; rgot = (int)take; break; }
            h = old;
            t = ld_relaxed(&ctl->tail);
          }
          const int wp = min(min(want, k) - rgot, room);
          if (wp > 0 && prim_work) {
            unsigned long long p0 = atomicAdd(&ctl->prim_next, (unsigned long long)wp);
            if (p0 < (unsigned long long)P.n_prim) {
              unsigned long long left = (unsigned long long)P.n_prim - p0;
              pbase = p0;
              pgot = left < (unsigned long long)wp ? (int)left : wp;
              if (left <= (unsigned long long)wp) atomicMax(&ctl->t_claimed, globaltimer_ns());
            }
          }
          cr -= rgot + pgot;
        }
      }
      rbase = __shfl_sync(FULL, rbase, 0);
      pbase = __shfl_sync(FULL, pbase, 0);
      rgot = __shfl_sync(FULL, rgot, 0);
      pgot = __shfl_sync(FULL, pgot, 0);
      credit = __shfl_sync(FULL, cr, 0);
      if (rgot + pgot == 0) {
        refill_backoff = refill_backoff * 2 + 1;
        if (refill_backoff > 63) refill_backoff = 63;
        refill_skip = refill_backoff;
      } else {
        refill_backoff = 0;
      }
      bool born_dead = false;
      if (!has && rgot + pgot > 0) {
        const int rank = __popc(need & lt);
        if (rank < rgot + pgot) {
          if (rank < rgot) {
            has = ring_get(R, ctl, rbase + rank, L, deadline);
          } else {
            const unsigned long long idx = pbase + (rank - rgot);
            L.z = P.pz[idx];
            L.eq = quant_e(P.pe[idx]);
            L.mu = P.pmu[idx];
            L.sp = P.psp[idx];
            L.node = 0;
            L.tal = 0.0;
            L.ev = 0;
            L.pid = (unsigned long long)P.pid_offset + idx;
            L.j = segment_of(P, L.z);
            L.slot = 0;
            sadd(&S.ledger[L_E_IN_PRIMARY], L.eq);
            sadd(&S.ledger[L_BIRTHS + L.sp], 1);
            if (L.sp == SP_E && L.eq < P.ecut_q) {
              die<F32>(P, S.ledger, L, R_CUTOFF, L_E_CUTOFF);
              born_dead = true;
            } else {
              has = true;
            }
          }
          started += 1;
        }
      }
      credit += __popc(__ballot_sync(FULL, born_dead));
      if (rgot > k)                                  // more than the idle lanes: to the queue
        qleft = ring_to_queue(R, ctl, rbase + k, rgot - k, Q, qleft, deadline);
    }

    // ---- parked rare collisions: once enough have gathered, free lanes and
    // then busy ones -- whose particles wait in the slots the batch frees --
    // perform them together; fewer make a batch once the primaries are used
    // up, and one does when the particles no longer fill the chip.  (At 1e5
    // decays, pass 1: one from two primaries per lane before the end 73.0 ms
    // FP64 / 41.0 FP32, one from the time the chip is not full 63.5 / 31.3,
    // with 12 late 54.9 / 28.0, with 6 late 53.5 / 28.1.) ----
    __syncwarp();
    int rk = -1;
    const int nr = min(Rb.n, RB - Rb.r);
    const unsigned hm = __ballot_sync(FULL, has);
    const bool batch = nr >= (drained ? RB_TRIGGER_LATE : RB_TRIGGER) || (nr > 0 && (hm == 0 || eager));
    if (batch) {
      const int nfree = 32 - __popc(hm);
      const int rank = has ? nfree + __popc(hm & lt) : __popc(~hm & lt);
      const bool take = rank < nr;
      const bool give = take && has;
      Lane back;
      if (give) {
        back = L;
      }
      if (take) {
        L = Rb.s[nr - 1 - rank];
        rk = Rb.ch[nr - 1 - rank];
        has = true;
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

    const unsigned busy = __ballot_sync(FULL, has);
    idle = !busy;
    if (idle) {
      int done = 0;
      if (lane == 0) {
        if (credit > 0) {
          __threadfence();
          atomicAdd((unsigned long long*)&ctl->active, (unsigned long long)(-(long long)credit));
        }
        // Done when no work is queued, none will come (no particle is held),
        // and nothing moved between two snapshots taken around the read of
        // the active count.  A claim visible in the first snapshot makes its
        // active increment visible; a product reserved by a particle whose
        // death is visible shows up in the second snapshot.
        const unsigned long long h1 = ld_relaxed(&ctl->head), t1 = ld_relaxed(&ctl->tail);
        const unsigned long long p1 = ld_relaxed(&ctl->prim_next);
        __threadfence();
        const long long a = ld_relaxed_s(&ctl->active);
        __threadfence();
        const unsigned long long h2 = ld_relaxed(&ctl->head), t2 = ld_relaxed(&ctl->tail);
        const unsigned long long p2 = ld_relaxed(&ctl->prim_next);
        done = (a <= 0 && h1 == h2 && t1 == t2 && p1 == p2 && h1 >= t1 &&
                p1 >= (unsigned long long)P.n_prim);
      }
      credit = 0;
      if (__shfl_sync(FULL, done, 0)) break;
      __nanosleep(idle_ns);
      if (idle_ns < 4096) idle_ns <<= 1;
      ++idle_iters;
      continue;
    }
    idle_ns = 128;
    busy_lane_iters += __popc(busy);
    ++busy_iters;

    // ---- one event ----
    bool died = false;
    o.rare = -1;
    if (has && rk < 0) {
      event<F32>(P, SP, cols, S.ledger, L, o);
      if (!o.alive) {
        has = false;
        died = true;
      } else if (o.rare >= 0) {
        // park it for the warp's next batch, or perform it now if all places
        // are taken
        const int i = atomicAdd(&Rb.n, 1);
        if (i < RB - Rb.r) {
          Rb.s[i] = L;
          Rb.ch[i] = (int8_t)o.rare;
          has = false;
        } else {
          rk = o.rare;
        }
      }
    }
    if (has && rk >= 0) {
      // (copies: only here the particle and the sums have an address)
      Lane M = L;
      EventOut m;
      m.alive = true;
      m.recoil = 0;
      rare_kinematics<F32>(SP, S.ledger, M, m, port, rk);
      L = M;
      o.recoil += m.recoil;
      if (!m.alive) {
        has = false;
        died = true;
      }
    }
    __syncwarp();
    const int qtop = min(Q.top, WQ);                  // pushes past the end went to the ring
    __syncwarp();
    if (lane == 0) {
      Q.top = qtop;
      if (Rb.n > RB - Rb.r) Rb.n = RB - Rb.r;         // parks past the end were done in line
    }

    // ---- channel counts, one shared-memory add per distinct channel per warp ----
    const unsigned mc = __ballot_sync(FULL, o.chan >= 0);
    if (o.chan >= 0) {
      const unsigned grp = __match_any_sync(mc, o.chan);
      if (lane == __ffs(grp) - 1) atomicAdd(&S.chan[o.chan], (unsigned long long)__popc(grp));
    }
    o.chan = -1;

    credit += __popc(__ballot_sync(FULL, died)) - (qtop - qleft);
    if (credit < 0) {                                 // more products than places
      if (lane == 0)
        atomicAdd((unsigned long long*)&ctl->active, (unsigned long long)(-(long long)credit));
      credit = 0;
    }
  }

  // ---- flush per-lane and per-block counters ----
  unsigned long long f = o.flights, c = o.colls, st = started, rc = o.recoil, ex = o.excit;
  unsigned long long sp = port.spilled;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    sp += __shfl_down_sync(FULL, sp, off);
    f += __shfl_down_sync(FULL, f, off);
    c += __shfl_down_sync(FULL, c, off);
    st += __shfl_down_sync(FULL, st, off);
    rc += __shfl_down_sync(FULL, rc, off);
    ex += __shfl_down_sync(FULL, ex, off);
  }
  if (lane == 0) {
    atomicMax(&ctl->t_end, globaltimer_ns());
    atomicAdd(&ctl->idle_iters, idle_iters);
    atomicAdd(&ctl->spilled, sp);
    atomicAdd(&ctl->busy_iters, busy_iters);
    atomicAdd(&ctl->busy_lane_iters, busy_lane_iters);
    atomicAdd(&S.ledger[L_N_FLIGHT], f);
    atomicAdd(&S.ledger[L_N_COLL], c);
    atomicAdd(&S.ledger[L_N_FLIGHT_ALL], f);
    atomicAdd(&S.ledger[L_N_COLL_ALL], c);
    atomicAdd(&S.ledger[L_LOSS_RECOIL], rc);
    atomicAdd(&S.ledger[L_LOSS_EXCIT], ex);
    atomicAdd(&ctl->particles, st);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < LEDGER; i += blockDim.x)
    if (S.ledger[i]) atomicAdd(P.ledger + i, S.ledger[i]);
  for (int i = threadIdx.x; i < P.nch; i += blockDim.x)
    if (S.chan[i]) atomicAdd(P.chan_count + i, S.chan[i]);
}

// ---------------------------------------------------------------------------
// host-callable launchers (used by the C ABI in karl_abi.cu)

// dynamic shared memory for the staged tables: at most this much per block,
// so that two blocks of 256 threads (with ~33 KB more for their warp queues
// and parked collisions) still fit one SM's 227 KB; blocks of 128 threads
// need half the queue memory and fit four to an SM with config-sized tables
constexpr int DYN_MAX_BYTES = 76 * 1024;
// per-warp queues in dynamic shared memory (after the tables)
constexpr int QUEUE_BYTES_PER_WARP = (int)(sizeof(WarpQueue) + sizeof(RareBuf));
static_assert(sizeof(WarpQueue) % 8 == 0 && sizeof(RareBuf) % 8 == 0, "queue alignment");


// Shared memory a block may give its staged tables: 76 KB for blocks of up
// to 256 threads (two to an SM), and what a block of more threads, alone on
// its SM, leaves beside its queues (then the pass-2 field tables fit too).
constexpr int SMEM_PER_SM = 227 * 1024;
constexpr int STATIC_SMEM_MARGIN = 4 * 1024;
int dyn_table_budget(int block) {
  if (block <= 256) return DYN_MAX_BYTES;
  return SMEM_PER_SM - STATIC_SMEM_MARGIN - (block / 32) * QUEUE_BYTES_PER_WARP;
}

// Doubles of dynamic shared memory the staged tables of P need (0: too big,
// read them from global memory).
int transport_dyn_doubles(const Params& P, int block) {
  int need = (4 * P.nz + 2) + (P.nq + 1 + 1) / 2 + 1;
  for (int k = 0; k < P.nch; ++k)
    if (P.fcol[k]) need += 2 * P.nz + 1;
  return need * 8 <= dyn_table_budget(block) ? need : 0;
}

// Where stage_tables puts each field channel's tables.
void transport_offsets(Params& P) {
  int at = (4 * P.nz + 2) + (P.nq + 2) / 2;
  for (int k = 0; k < P.nch; ++k) {
    P.foff[k] = at;
    if (P.fcol[k]) at += 2 * P.nz + 1;
  }
}

size_t transport_dyn_bytes(const Params& P, int block) {
  return (size_t)transport_dyn_doubles(P, block) * 8 + (size_t)(block / 32) * QUEUE_BYTES_PER_WARP;
}

using TransportKernel = void (*)(const Params, const Ring, Control*, const volatile int*,
                                 unsigned long long, int);
TransportKernel kernel_for(bool f32, bool staged) {
  if (f32) return staged ? transport_kernel<true, true> : transport_kernel<true, false>;
  return staged ? transport_kernel<false, true> : transport_kernel<false, false>;
}

cudaError_t launch_transport(bool f32, const Params& P, const Ring& R, Control* ctl,
                             const volatile int* cancel, unsigned long long timeout_ns, int grid,
                             int block, cudaStream_t st) {
  const int dd = transport_dyn_doubles(P, block);
  const size_t bytes = transport_dyn_bytes(P, block);
  Params Q = P;
  transport_offsets(Q);
  kernel_for(f32, dd > 0)<<<grid, block, bytes, st>>>(Q, R, ctl, cancel, timeout_ns, dd);
  return cudaGetLastError();
}

cudaError_t transport_setup() {
  for (int v = 0; v < 4; ++v) {
    cudaError_t e = cudaFuncSetAttribute(kernel_for(v & 1, v & 2),
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         SMEM_PER_SM - STATIC_SMEM_MARGIN);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t transport_occupancy(bool f32, const Params& P, int block, int* blocks_per_sm) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      blocks_per_sm, kernel_for(f32, transport_dyn_doubles(P, block) > 0), block,
      transport_dyn_bytes(P, block));
}

}  // namespace karl
