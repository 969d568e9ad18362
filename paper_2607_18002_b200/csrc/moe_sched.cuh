// Scheduling pieces shared by the persistent kernels: bounded waits, the two-class tile queue
// (Sections 4.2 and 6.4), tile publication and the SwiGLU helper.
#pragma once
#include "moe_dev.cuh"
#include "moe_ptx.cuh"

namespace moe {

constexpr int kRing = 4;                               // tile-info ring depth
constexpr int kEnd = -1;

struct TileInfo {
  int kind, slot, tile, m, row0, rows, n, kblocks, expert, cls;
  unsigned long long t_claim;
};

__device__ __forceinline__ int expert_of(const TileInfo& ti) { return ti.expert & (kReadOnce - 1); }

// what a unit reads before it claims
struct ClaimWords {
  unsigned abort, budget, head[2];
};

// per-class queue tables of one launch (built once per CTA in shared memory)
struct QueueTables {
  unsigned run_off;                // of this launch
  int watched;                     // an op of the launch is: committed tiles are counted
  int two_classes;                 // (two tiles at a time) it has ops of both
  int n_cls[2];
  int cls_slot[2][kMaxOps];
  int cls_free[2][kMaxOps];        // 1: the op has no ready word and no predecessor
  unsigned twos[2][kMaxOps];       // an op's first tickets are two entries each: so many of them
  unsigned n_gemm[2][kMaxOps];     // tickets of the op's GEMM entries; those of the combine entries follow them
  int all_gemm[2][kMaxOps];        // gemm_done when its combine may run
  const int4* list[2][kMaxOps];
  unsigned cum[2][kMaxOps + 1];
  int carrier[2][kMaxOps];         // paired prefill op: the decode op (its place in that class) whose GEMM entries carry its rows, else -1
};

// ------------------------------------------------------------------ bounded waits
struct Ctx {
  const RunArgs* a;
  Status* st;
  unsigned run_off;              // 0 or run_bytes: the half of the run state this launch works on
};
__device__ __forceinline__ RunState* run_of(const Ctx& c, const OpDev* op) {
  return reinterpret_cast<RunState*>(reinterpret_cast<char*>(op->run) + c.run_off);
}
__device__ __forceinline__ int* g1_done_of(const Ctx& c, const OpDev* op) {
  return reinterpret_cast<int*>(reinterpret_cast<char*>(op->g1_done) + c.run_off);
}

__device__ __forceinline__ bool aborted(const Ctx& c) { return ld_volatile(&c.st->abort) != 0; }

// One look of a wait at the clock (t0: 0 at the wait's start), or at the abort word and the clock: false when it has to give up.
// where: a small code telling which wait gave up (reported in detail[0])
__device__ __noinline__ inline bool in_time(const Ctx& c, unsigned long long& t0, long long limit_ns, int where) {
  const unsigned long long now = gtime_ns();
  if (t0 == 0) t0 = now;
  else if ((long long)(now - t0) > limit_ns) {
    report(c.st, MOE_ETIMEOUT, where, (int)blockIdx.x, (int)threadIdx.x, 0);
    return false;
  }
  return true;
}
__device__ __forceinline__ bool still_waiting(const Ctx& c, unsigned long long& t0, int where) {
  return !aborted(c) && in_time(c, t0, c.a->wait_ns, where);
}
__device__ __noinline__ inline bool mbar_wait_slow(const Ctx& c, void* bar, unsigned parity, int where) {
  unsigned long long t0 = 0;
  for (unsigned it = 1;; ++it) {
    if (mbar_try(bar, parity)) return true;
    if ((it & 63u) == 0) {
      if (aborted(c)) return false;
      const unsigned long long now = gtime_ns();
      if (t0 == 0) t0 = now;
      else if ((long long)(now - t0) > c.a->wait_ns) {
        report(c.st, MOE_ETIMEOUT, where, (int)blockIdx.x, (int)threadIdx.x, (int)parity);
        return false;
      }
    }
  }
}
__device__ __forceinline__ bool mbar_wait(const Ctx& c, void* bar, unsigned parity, int where) {
  if (mbar_try(bar, parity)) return true;
  return mbar_wait_slow(c, bar, parity, where);
}

// the same wait without any function call: for code that keeps many registers live across it
__device__ __forceinline__ bool mbar_wait_inline(const Ctx& c, void* bar, unsigned parity, int where) {
  unsigned long long t0 = 0;
  for (unsigned it = 0;; ++it) {
    if (mbar_try(bar, parity)) return true;
    if ((it & 63u) == 63u) {
      if (aborted(c)) return false;
      const unsigned long long now = gtime_ns();
      if (t0 == 0) t0 = now;
      else if ((long long)(now - t0) > c.a->wait_ns) {
        if (atomicCAS(&c.st->code, 0, MOE_ETIMEOUT) == 0) {
          c.st->detail[0] = where; c.st->detail[1] = (int)blockIdx.x;
          c.st->detail[2] = (int)threadIdx.x; c.st->detail[3] = (int)parity;
        }
        __threadfence();
        atomicExch(&c.st->abort, 1);
        return false;
      }
    }
  }
}

// spin until *p >= target (acquire); one thread
__device__ __noinline__ inline bool wait_counter(const Ctx& c, const int* p, int target, int where) {
  unsigned long long t0 = 0;
  for (unsigned it = 0;; ++it) {
    if (ld_acquire(p) >= target) return true;
    if (it > 16) __nanosleep(64);
    if ((it & 63u) == 63u) {
      if (aborted(c)) return false;
      const unsigned long long now = gtime_ns();
      if (t0 == 0) t0 = now;
      else if ((long long)(now - t0) > c.a->wait_ns) {
        report(c.st, MOE_ETIMEOUT, where, (int)blockIdx.x, target, ld_acquire(p));
        return false;
      }
    }
  }
}

// ------------------------------------------------------------------ queues
// a slot whose plan was rejected (an expert id out of range) holds no tiles
__device__ __forceinline__ int op_total_tiles(const OpDev* op, int fuse) {
  if (op->plan->planned == 0) return 0;
  return op->plan->n_gemm_tiles + op->plan->n_extra_gemm + (fuse ? op->plan->n_comb_tiles : 0);
}
// Of `gemm` GEMM entries the down tiles.  They are what an op's combine waits for: none of them commits before its gate/up tiles.
__device__ __forceinline__ int down_tiles(const RunArgs* a, int gemm) {
  const int nt1 = a->I / kTileN1, nt2 = a->H / kTileN2;
  return gemm / (nt1 + nt2) * nt2;
}
__device__ __forceinline__ int op_down_tiles(const RunArgs* a, const OpDev* op) {
  return down_tiles(a, op->plan->n_gemm_tiles + op->plan->n_extra_gemm);
}

// An op without tiles (no tokens, or a plan that was rejected) never commits anything: it counts as
// finished as soon as its own predecessor has, and its ready word is not consulted.
__device__ inline bool op_finished(const Ctx& c, int slot) {
  const RunArgs* a = c.a;
  for (int hop = 0; slot >= 0 && hop <= kMaxOps; ++hop) {
    const OpDev* op = &a->ops[a->desc[slot]];
    if (op_total_tiles(op, a->fuse_combine) > 0) return ld_acquire(&run_of(c, op)->done) != 0;
    slot = op->after_op;
  }
  return true;
}

__device__ inline bool op_ready(const Ctx& c, const OpDev* op) {
  if (op->ready != nullptr && ld_acquire_sys(op->ready) == 0) return false;
  return op_finished(c, op->after_op);
}

// Marks as done every tile-less op of the run whose chain of predecessors ends at `finished`
// (-1: at no op at all) through tile-less ops only.  One thread; called at kernel start and when an
// op's last tile commits.
__device__ inline void finish_empty_ops(const Ctx& c, int finished) {
  const RunArgs* a = c.a;
  for (int i = 0; i < a->n_ops; ++i) {
    OpDev* op = &a->ops[a->slots[i]];
    if (op_total_tiles(op, a->fuse_combine) > 0) continue;
    int dep = op->after_op;
    for (int hop = 0; dep >= 0 && hop <= kMaxOps && op_total_tiles(&a->ops[a->desc[dep]], a->fuse_combine) == 0; ++hop)
      dep = a->ops[dep].after_op;
    if (dep != finished) continue;
    atomicExch(&run_of(c, op)->done, 1);
    if (op->done != nullptr) st_release_sys(op->done, 1u);
    if (op->notify != nullptr) st_release_sys(op->notify, 1u);
  }
}

// whether the decode queue's head has passed the GEMM entries of its op `j` (-1: there are none to pass)
__device__ __forceinline__ bool carriers_claimed(const QueueTables* sc, int j, unsigned decode_head) {
  return j < 0 || decode_head >= sc->cum[MOE_CLASS_DECODE][j] + sc->n_gemm[MOE_CLASS_DECODE][j];
}

__device__ __forceinline__ void fill_tile(const RunArgs* a, const int4& got, int slot, int at, int cls, TileInfo& ti) {
  ti.kind = entry_kind(got);
  ti.n = entry_n(got);
  ti.m = entry_m(got);
  ti.row0 = got.y;
  ti.rows = got.z;
  ti.expert = got.w;
  ti.slot = slot;
  ti.tile = at;
  ti.cls = cls;
  ti.kblocks = ti.kind == kCombine ? 0 : ti.kind == kDown ? a->kb_down : a->kb_gate_up;
}
// the (first) entry of an op's ticket
template <bool kTwos>
__device__ __forceinline__ unsigned first_entry(const QueueTables* sc, int cls, int i, unsigned ticket) {
  if constexpr (kTwos) return ticket + min(ticket, sc->twos[cls][i]);
  return ticket;
}

// Claim by the whole producer warp.  1: claimed (ti filled), 0: queue exhausted, -1: the op
// at the head of the queue is not ready.  The head is only peeked before the fetch-add, so no
// CTA can be starved by others (a compare-and-swap loop starves the SMs far from the counter);
// the price is that a ticket can land just past an op boundary, in an op that is not ready
// yet -- the caller then waits for it (bounded), holding only tickets whose predecessors in
// the queue are all claimed already.
// early_combine: also take a combine entry whose GEMM entries are still running -- all of them must have been claimed, or every unit
// could end up holding such an entry with none left for what they wait for.  The op's own are (the head stands behind them); those of
// the decode list that carry rows of a paired prefill op are once the head of the decode queue, other_head, has passed them.
// two (kTwos): the ticket holds the entry behind it too, the next n-block of the same work tile.
template <bool kTwos>
__device__ inline int try_claim(const Ctx& c, QueueTables* sc, RunHead* rh, int cls, unsigned h, unsigned other_head,
                                int lane, TileInfo& ti, bool& need_ready, bool& two, bool early_combine = false) {
  const RunArgs* a = c.a;
  const int n = sc->n_cls[cls];
  if (n == 0) return 0;
  const unsigned total = sc->cum[cls][n];
  h = __shfl_sync(0xffffffffu, h, 0);       // one peek for the whole warp: lanes index entries by it
  if (h >= total) return 0;
  int i = 0;
  while (h >= sc->cum[cls][i + 1]) ++i;
  int slot = sc->cls_slot[cls][i];
  const OpDev* op = &a->ops[slot];
  const unsigned base = h - sc->cum[cls][i];
  // Everything the warp branches on comes from ONE lane's loads: the lanes of this warp run apart after a
  // sleep, and words such as an op's done flag or the GEMM counter change between one lane's load and the next's.
  int takeable = 1;
  if (lane == 0) {
    if (!sc->cls_free[cls][i] && !op_ready(c, op)) takeable = 0;
    // The head stands at the op's combine entries while GEMM entries they depend on are still running
    // (other units hold them; for a paired prefill op, the decode list's carrier tiles): nothing to take here
    // yet -- the caller turns to the other class first.
    else if (base >= sc->n_gemm[cls][i] && !(early_combine && carriers_claimed(sc, sc->carrier[cls][i], other_head)) &&
             ld_acquire(&run_of(c, op)->gemm_done) < sc->all_gemm[cls][i])
      takeable = 0;
  }
  if (__shfl_sync(0xffffffffu, takeable, 0) == 0) return -1;
  // what the op's ready word announced is read by TMA too
  if (lane == 0 && !sc->cls_free[cls][i]) fence_async_proxy();
  // the 32 entries from the head on are fetched while the fetch-add is in flight
  const unsigned first = first_entry<kTwos>(sc, cls, i, base);
  const unsigned n_op = sc->cum[cls][i + 1] - sc->cum[cls][i] + (kTwos ? sc->twos[cls][i] : 0u);
  int4 e = make_int4(0, 0, 0, 0);
  unsigned t = 0;
  if (lane == 0) t = atomicAdd(&rh->heads[cls], 1u);
  if (first + lane < n_op) e = sc->list[cls][i][first + lane];
  t = __shfl_sync(0xffffffffu, t, 0);
  if (t >= total) return 0;
  need_ready = false;
  // the prefetched entries belong to the op at the peeked head: usable only while the ticket stays in it
  const bool same_op = t < sc->cum[cls][i + 1];
  if (!same_op) {                          // past the op boundary: a later op of the class
    while (t >= sc->cum[cls][i + 1]) ++i;
    slot = sc->cls_slot[cls][i];
    op = &a->ops[slot];
    need_ready = !sc->cls_free[cls][i];
  }
  const unsigned local = t - sc->cum[cls][i];
  // the op is instantiated by the claim of its first tile: its budget field takes effect now
  if (local == 0 && lane == 0 && op->op_budget > 0) atomicExch(&a->g->budget, op->op_budget);
  const unsigned at = first_entry<kTwos>(sc, cls, i, local);
  const unsigned d = at - first;
  const bool hit = same_op && d < 32u;
  int4 got;
  got.x = __shfl_sync(0xffffffffu, e.x, hit ? d : 0);
  got.y = __shfl_sync(0xffffffffu, e.y, hit ? d : 0);
  got.z = __shfl_sync(0xffffffffu, e.z, hit ? d : 0);
  got.w = __shfl_sync(0xffffffffu, e.w, hit ? d : 0);
  if (!hit) got = sc->list[cls][i][at];
  fill_tile(a, got, slot, (int)at, cls, ti);
  if constexpr (kTwos) two = local < sc->twos[cls][i];
  return 1;
}

// One pass of the decision at a tile boundary (whole producer warp): 1 = claimed, 0 = both
// queues exhausted, -1 = something exists but is not ready yet.  The abort word, the budget
// word and both queue heads are loaded together (one round trip), then at most one
// fetch-add per class.
// kEarlyCombine: a unit that finds nothing to run in either class takes a combine entry that has to wait for GEMM entries running
// elsewhere (see try_claim), so that the wait for the last of them starts with the entry in hand.  It claims nothing more meanwhile.
// seen: the words as the unit's start read them (its first claim); they only tell where to look, the fetch-add decides.
// kTwos: two: see try_claim.
template <bool kEarlyCombine, bool kTwos>
__device__ inline int claim_once(const Ctx& c, QueueTables* sc, RunHead* rh, int lane, TileInfo& ti,
                                 bool& need_ready, bool& two, const ClaimWords* seen = nullptr) {
  const RunArgs* a = c.a;
  ClaimWords w{};
  if (seen) {
    w = *seen;
  } else {
    // one lane reads the words and the warp takes ITS values: the budget word, the abort word and the heads
    // change while the kernel runs, and the lanes do not load them at the same instant
    if (lane == 0) {
      w.abort = (unsigned)ld_volatile(&c.st->abort);
      w.budget = (unsigned)ld_volatile(&a->g->budget);
      w.head[0] = *reinterpret_cast<volatile unsigned*>(&rh->heads[0]);
      w.head[1] = *reinterpret_cast<volatile unsigned*>(&rh->heads[1]);
    }
    w.abort = __shfl_sync(0xffffffffu, w.abort, 0);
    w.budget = __shfl_sync(0xffffffffu, w.budget, 0);
    w.head[0] = __shfl_sync(0xffffffffu, w.head[0], 0);
    w.head[1] = __shfl_sync(0xffffffffu, w.head[1], 0);
  }
  if (w.abort != 0) return 0;
  const unsigned h0 = w.head[0], h1 = w.head[1];
  const int first = ((int)blockIdx.x < (int)w.budget) ? MOE_CLASS_DECODE : MOE_CLASS_PREFILL;
  need_ready = false;
  int none[2] = {0, 0};                          // in the order tried: 0 nothing left, -1 not yet
  if constexpr (kEarlyCombine) {
    // one body for all attempts: a unit's first claim waits for these instructions to be fetched
#pragma unroll 1
    for (int p = 0; p < 4; ++p) {
      if (p >= 2 && none[p & 1] == 0) continue;
      const int cls = (p & 1) ? 1 - first : first;
      none[p & 1] = try_claim<kTwos>(c, sc, rh, cls, cls == 0 ? h0 : h1, cls == 0 ? h1 : h0, lane, ti, need_ready, two, p >= 2);
      if (none[p & 1] == 1) break;
    }
  } else {                                       // (in a loop this kernel's scheduler spills)
    none[0] = try_claim<kTwos>(c, sc, rh, first, first == 0 ? h0 : h1, 0u, lane, ti, need_ready, two);
    if (none[0] != 1) none[1] = try_claim<kTwos>(c, sc, rh, 1 - first, first == 0 ? h1 : h0, 0u, lane, ti, need_ready, two);
  }
  if (none[0] == 1 || none[1] == 1) {
    if (a->log_cap > 0) ti.t_claim = gtime_ns();
    return 1;
  }
  return (none[0] | none[1]) == 0 ? 0 : -1;
}

// A ticket that landed in an op that is not ready yet: wait for it (bounded).  Whole warp; lane 0 looks and
// decides, so that all lanes leave together.
__device__ inline bool wait_op_ready(const Ctx& c, int lane, const TileInfo& ti) {
  const RunArgs* a = c.a;
  const unsigned long long w0 = gtime_ns();
  while (true) {
    int r = 0;                                   // 1: ready, -1: give up
    if (lane == 0) {
      if (op_ready(c, &a->ops[ti.slot])) { r = 1; fence_async_proxy(); }
      else if (aborted(c)) r = -1;
      else if ((long long)(gtime_ns() - w0) > a->wait_ns) {
        report(c.st, MOE_ETIMEOUT, 11, (int)blockIdx.x, slot_of(a, ti.slot), ti.tile);
        r = -1;
      }
    }
    r = __shfl_sync(0xffffffffu, r, 0);
    if (r != 0) return r > 0;
    __nanosleep(256);
  }
}

// The plain (non-persistent) launch: unit `unit` of the grid takes queue entry `unit` of the run's only op
// and nothing else.  No queue head, no budget, no ready word.  A down tile still waits (bounded) for the
// gate/up tiles of its rows: they sit earlier in the list, i.e. in units with a lower index.
__device__ inline void claim_static(const RunArgs* a, int unit, TileInfo& ti) {
  const int slot = a->slots[0];
  const OpDev* op = &a->ops[slot];
  ti.kind = kEnd;
  if (unit >= op->plan->n_gemm_tiles) return;
  const int4 got = op->tile_list[unit];
  fill_tile(a, got, slot, unit, op->cls, ti);
  if (a->log_cap > 0) ti.t_claim = gtime_ns();
}

// Blocking form: waits (bounded) while an op exists that is not ready.  Returns with
// ti.kind == kEnd when nothing is left (or the run was aborted).
template <bool kEarlyCombine, bool kTwos>
__device__ inline void claim_next(const Ctx& c, QueueTables* sc, RunHead* rh, int lane, TileInfo& ti,
                                  bool& need_ready, bool& two, const ClaimWords* seen = nullptr) {
  unsigned long long t0 = 0;
  for (unsigned it = 0;; ++it) {
    const int r = claim_once<kEarlyCombine, kTwos>(c, sc, rh, lane, ti, need_ready, two, seen);
    seen = nullptr;
    if (r == 1) return;
    if (r == 0) break;
    __nanosleep(256);                         // an op exists but is not ready yet
    if ((it & 15u) == 15u) {                  // lane 0's clock decides for the warp
      int expired = 0;
      if (lane == 0) {
        const unsigned long long now = gtime_ns();
        if (t0 == 0) t0 = now;
        else if ((long long)(now - t0) > c.a->wait_ns) {
          report(c.st, MOE_ETIMEOUT, 1, (int)blockIdx.x, 0, 0);
          expired = 1;
        }
      }
      if (__shfl_sync(0xffffffffu, expired, 0)) break;
    }
  }
  ti.kind = kEnd;
}

// The words that wait for a tile of `op` (of a combine tile: not counted): a gate/up tile counts in g1_done of its work tile, where the
// down tiles of those rows look; a down tile in gemm_done, where the combine tiles look, and if the entry is one of a paired decode op's,
// which carry rows of the prefill op too, in that op's.  All units count at the end of a wave of tiles, and the words share an L2 slice:
// gate/up tiles in gemm_done too, and every warp of a tile of one row, made 2400 atomics of what are 600 (one token on 8 experts).
struct StoredWords {
  int* own;
  int* partner;
};
__device__ __forceinline__ StoredWords stored_words(const Ctx& c, const OpDev* op, const TileInfo& ti) {
  StoredWords w;
  const bool down = ti.kind == kDown;
  w.own = down ? &run_of(c, op)->gemm_done : &g1_done_of(c, op)[ti.m];
  w.partner = down && op->paired && ti.cls == MOE_CLASS_DECODE ? &run_of(c, &c.a->ops[op->partner])->gemm_done : nullptr;
  return w;
}
// By one lane of each warp that stores a tile, after a __syncwarp behind its last store, or by one thread for all of them.
__device__ __forceinline__ void count_stored(const StoredWords& w, int n) {
  fence_acq_rel_gpu();
  fence_async_proxy();
  atomicAdd(w.own, n);
  if (w.partner) atomicAdd(w.partner, n);
}

// one committed entry counted for `op` (descriptor `desc`): notify word, completion
__device__ inline void count_commit(const Ctx& c, OpDev* op, int desc) {
  const RunArgs* a = c.a;
  RunState* run = run_of(c, op);
  const int done = atomicAdd(&run->tiles_done, 1) + 1;
  if (op->notify != nullptr && done == op->notify_after) st_release_sys(op->notify, 1u);
  if (done == op_total_tiles(op, a->fuse_combine)) {
    __threadfence();
    atomicExch(&run->done, 1);
    if (op->done != nullptr) st_release_sys(op->done, 1u);
    finish_empty_ops(c, slot_of(a, desc));
  }
}

// Publishing a finished tile: log, op completion and done word where an op of the launch is watched, and unless the storing warps have
// done so (kCounts false) the words that other tiles wait for.  Called by one thread after all writers of the tile have fenced and
// synchronised.  (A launch that nobody watches saves a chain of three round trips behind its last tile.)
template <bool kCounts>
__device__ inline void commit_tile(const Ctx& c, RunHead* rh, const TileInfo& ti, bool watched) {
  const RunArgs* a = c.a;
  OpDev* op = &a->ops[ti.slot];
  const unsigned long long t_commit = a->log_cap > 0 ? gtime_ns() : 0ull;   // before it is published
  if (kCounts && ti.kind != kCombine) count_stored(stored_words(c, op, ti), 1);
  else if (watched) fence_acq_rel_gpu();
  if (watched) {
    count_commit(c, op, ti.slot);
    if (op->paired && op->cls == MOE_CLASS_DECODE && ti.kind != kCombine) count_commit(c, &a->ops[op->partner], op->partner);
  }
  if (a->log_cap > 0) {
    const unsigned idx = atomicAdd(&rh->log_count, 1u);
    if (idx < (unsigned)a->log_cap) {
      moe_tile_rec_t r;
      r.t_claim = ti.t_claim;
      r.t_commit = t_commit;
      r.slot = slot_of(a, ti.slot);
      r.tile = ti.tile;
      r.cls = (int16_t)ti.cls;
      r.kind = (int16_t)ti.kind;
      r.cta = (int16_t)blockIdx.x;
      unsigned smid;
      asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
      r.sm = (int16_t)smid;
      a->log[idx] = r;
    }
  }
}

// Start of a claiming unit, one warp: which half of the run state is this launch's, the per-class queue tables, and the words of the
// unit's first claim (heads: of both halves, the half is only known when they arrive).  All of it is one round trip: lane i reads
// the plan of op i, the last lanes a word each.  The unit asks for the half with a plain load; the fetch-add that counts it
// (take_turn) comes later, so that no claim waits behind those of all other units.
// per_tile: what a committed down tile adds to gemm_done.  max_rows: the tallest work tile this kernel has room for.
// kTwos: it runs two tiles at a time.  The last entries of a list, two a unit but a quarter of it at most, are handed out one by one all the same:
// the units end closer to one another (256 tokens on 64 experts: 314 us a pass without, 305).  (Two a unit of a short list is most of it: 128
// decode tokens on 8 experts next to 8192 of prefill, budget 16, done after 535 us, 443 with a quarter.)
// A decode op next to prefill ops is handed out one by one: latency is what its budget is bought for.  128 decode tokens on 8 experts next to
// 8192 of prefill, us from claim to commit of a tile at the 99th percentile and until the op is done, in twos / one by one: budget 16 80,
// 504 / 42, 452, budget 32 80, 276 / 43, 262, budget 64 82, 182 / 46, 190; 64 on 64 experts next to 4096, budget 64 69, 630 / 36, 598; launches as
// long as before (2320 / 2325, 1190 / 1187).  Not where its tiles carry prefill rows: those of more than 128 rows are slow one by one (16 384 + 256
// paired 3728 / 3862 us a launch, decode done 2483 / 2856).
template <bool kTwos>
__device__ inline ClaimWords begin_unit(const RunArgs* a, QueueTables* sc, const RunHead* first_half, int lane, int per_tile, int max_rows) {
  constexpr int kW = 25;
  static_assert(kMaxOps <= kW, "a lane per op, and one per word");
  const RunHead* second = reinterpret_cast<const RunHead*>(reinterpret_cast<const char*>(first_half) + a->run_bytes);
  unsigned word = 0;
  if (lane >= kW) {
    const void* p = lane == kW ? (const void*)&a->g->turn : lane == kW + 1 ? (const void*)&a->g->status.abort
                  : lane == kW + 2 ? (const void*)&a->g->budget
                  : (const void*)&(lane < kW + 5 ? first_half : second)->heads[(lane - kW - 3) & 1];
    word = *reinterpret_cast<const volatile unsigned*>(p);
  }
  PlanState ps{};
  int cls = -1;
  if (lane < a->n_ops) {
    ps = *a->plan[lane];
    cls = ps.cls;
    // The host picks the kernel by the plans it has issued.  A graph replayed in between can have left another plan in the slot.
    if (ps.planned != 0 && ps.work_rows > max_rows) {
      report(&a->g->status, MOE_EBOUNDS, slot_of(a, a->slots[lane]), ps.work_rows, max_rows, 5);
      ps.planned = 0;
    }
  }
  const unsigned decode_ops = __ballot_sync(0xffffffffu, cls == MOE_CLASS_DECODE);
  unsigned singly = 0;                             // decode ops next to prefill ops whose tiles carry no prefill rows
  if constexpr (kTwos) {
    const int carrier = lane < a->n_ops ? a->carrier[lane] : -1;
    const unsigned carriers = __reduce_or_sync(0xffffffffu, carrier < 0 ? 0u : 1u << carrier);
    const bool both = decode_ops != 0 && __popc(decode_ops) < a->n_ops;
    if (both) singly = decode_ops & ~carriers;
    if (lane == 0) sc->two_classes = both;
  }
  const int combines = ps.planned != 0 && a->fuse_combine ? ps.n_comb_tiles : 0, gemms = ps.planned != 0 ? ps.n_gemm_tiles : 0;
  const int all_gemm = down_tiles(a, ps.n_gemm_tiles + ps.n_extra_gemm) * per_tile;
  const unsigned watched = __ballot_sync(0xffffffffu, (ps.flags & kOpWatched) != 0);
  if (lane == 0) {
    sc->watched = watched != 0;
    sc->n_cls[0] = sc->n_cls[1] = 0;
    sc->cum[0][0] = sc->cum[1][0] = 0;
  }
  for (int i = 0; i < a->n_ops; ++i) {
    const int ei = __shfl_sync(0xffffffffu, combines, i), ci = __shfl_sync(0xffffffffu, cls, i);
    const int gi = __shfl_sync(0xffffffffu, gemms, i), ai = __shfl_sync(0xffffffffu, all_gemm, i);
    const int fi = __shfl_sync(0xffffffffu, ps.flags & kOpFree, i);
    if (lane == 0) {
      const int j = sc->n_cls[ci]++;
      sc->cls_slot[ci][j] = a->slots[i];
      sc->cls_free[ci][j] = fi;
      const int twos = kTwos && !((singly >> i) & 1u) ? (gi - min((int)gridDim.x, gi / 4)) / 2 : 0;
      if constexpr (kTwos) sc->twos[ci][j] = (unsigned)twos;
      sc->n_gemm[ci][j] = (unsigned)(gi - twos);
      sc->cum[ci][j + 1] = sc->cum[ci][j] + (unsigned)(gi - twos + ei);
      sc->all_gemm[ci][j] = ai;
      sc->list[ci][j] = a->tile_list[i];
      sc->carrier[ci][j] = a->carrier[i] < 0 ? -1 : __popc(decode_ops & ((1u << a->carrier[i]) - 1u));
    }
  }
  const unsigned turn = __shfl_sync(0xffffffffu, word, kW);
  const bool odd = (turn >> 31) != 0;
  if (lane == 0) sc->run_off = odd ? a->run_bytes : 0u;
  __syncwarp();
  ClaimWords w;
  w.abort = __shfl_sync(0xffffffffu, word, kW + 1);
  w.budget = __shfl_sync(0xffffffffu, word, kW + 2);
  w.head[0] = __shfl_sync(0xffffffffu, word, odd ? kW + 5 : kW + 3);
  w.head[1] = __shfl_sync(0xffffffffu, word, odd ? kW + 6 : kW + 4);
  return w;
}
// One lane, once a launch and after begin_unit: counts the unit.  The last of the grid's `units` units turns the halves over for the
// next launch (end_turn).
__device__ inline unsigned take_turn(const RunArgs* a) { return atomicAdd(&a->g->turn, 1u); }
__device__ inline void end_turn(const RunArgs* a, unsigned ticket, int units) {
  if ((ticket & 0x7fffffffu) == (unsigned)units - 1u) atomicExch(&a->g->turn, ~ticket & 0x80000000u);
}
// The launch parameters into the constant cache, while the kernel before still runs.
__device__ __forceinline__ void touch_params(const RunArgs& a) {
  const int* p = reinterpret_cast<const int*>(&a);
#pragma unroll
  for (int i = 0; i < (int)(sizeof(RunArgs) / 4); i += 16) asm volatile("" ::"r"(p[i]));
}
// One warp of the grid: zeroes the other half, which the launch before this one left behind.
__device__ inline void clear_next_run(const RunArgs* a, RunHead* first_half, unsigned run_off, int lane) {
  int4* p = reinterpret_cast<int4*>(reinterpret_cast<char*>(first_half) + (run_off ? 0u : a->run_bytes));
  for (unsigned i = lane; i < a->run_bytes / 16; i += 32) p[i] = make_int4(0, 0, 0, 0);
}

// silu(g) * u through the hardware tanh approximation (one special-function op per element;
// its error, |g| * 2.4e-4 at worst, stays below the bf16 rounding of the result)
__device__ __forceinline__ float silu_mul(float g, float u) {
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(0.5f * g));
  const float hg = 0.5f * g;
  return fmaf(hg, t, hg) * u;                     // g * sigmoid(g) = g/2 * (1 + tanh(g/2))
}

__device__ __forceinline__ unsigned pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const unsigned*>(&v);
}

// Stores 32 tokens x 32 features of bf16 through the warp's scratch: o[4 f + j] is the 8x8 matrix of feature group f and token group
// j; stored row i % 8 of group i / 8 is token `row` (of lane i).
__device__ __forceinline__ void store_features32(unsigned char* scratch, unsigned scratch_addr, const unsigned (&o)[16], int row,
                                                 unsigned char* dst, size_t pitch, int left, int lane) {
  __syncwarp();                                     // scratch free again
#pragma unroll
  for (int f = 0; f < 4; ++f)                       // XOR keeps the banks of eight rows apart
    st_matrix4_trans(scratch_addr + row * 64 + ((f ^ ((row >> 1) & 3)) << 4), o[4 * f], o[4 * f + 1], o[4 * f + 2], o[4 * f + 3]);
  __syncwarp();
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int r = 8 * j + (lane >> 2), f = lane & 3;
    const uint4 v4 = *reinterpret_cast<const uint4*>(scratch + r * 64 + ((f ^ ((r >> 1) & 3)) << 4));
    if (r < left) *reinterpret_cast<uint4*>(dst + (size_t)r * pitch + f * 16) = v4;
  }
}

}  // namespace moe
