// moe_run on CTA pairs: the bf16 persistent expert kernel with two SMs per tile.
//
// Same scheduling as the single-CTA kernel (two queues, budget word, claim at tile
// boundaries: Sections 4.2 and 6.4), but the unit that claims and runs a tile is a cluster of
// two CTAs on neighbouring SMs, and the MMAs are tcgen05.mma.cta_group::2:
//   - the WEIGHT rows are the M = 256 rows of the instruction (128 per CTA) and the tile's token rows its N columns,
//     N = rows rounded up to 16 (half of them in each CTA's shared memory).  A tile costs tensor time and energy for
//     the rows it has: with the tokens as M every tile of up to 128 rows paid for 128 of them, and the multipliers' power
//     alone held a 128-token decode launch at 1.15 GHz (1350 us a pass against 1160 us; a tile there has four rows);
//   - gate/up tiles take 64 features per CTA, the weight rows interleaved 8 gate / 8 up by one 5-D box, so that an
//     accumulator fragment holds both factors of a SwiGLU output in one thread; down tiles take 128 features per CTA;
//   - a stage is 16 KB of weights and room for this CTA's half of the tile's rows: six stages for tiles of up to 256 rows, eight
//     for 128, eleven for 32 (the launch's ops decide).  Where few units have work the rate of a unit is its bytes in
//     flight over the load latency (one token, 96 tiles on 74 units: 80 -> 73 us a pass with eleven stages for six), and where all
//     have, more bytes in flight keep HBM busier (128 tokens on 252 experts: 1085 -> 1040 us with eight);
//   - a tile uses up to 256 of the 512 TMEM columns, so the epilogue of one tile overlaps the MMAs of the next;
//   - one form of the kernel for tiles of up to 256 rows takes two neighbouring n-blocks of a work tile at a time where the list has them (kDual,
//     chosen in moe_run): a stage then holds 256 weight rows per CTA and the rows once, four stages of 48 KB, and both accumulators run side
//     by side.  Large launches run at the 1000 W limit, where time is energy, and a 256-row k-block came to 580 clocks of the SMs' intake from L2
//     for 513 of the tensor pipe (both measured without the other): two of them now take in 96 KB a pair instead of 128, and hand-overs,
//     TMA instructions and gather serve twice the weights.  Nothing overlaps the stores of two accumulators but the first MMAs of the next two
//     tiles.  us a pass, one by one / two at a time, in turn on one GPU: 8192 tokens 2458 / 2389, 12 288 3174 / 3065, 16 384 + 256 paired
//     4236 / 4113, 4096 + 64 on 64 experts 1254 / 1210, 777 1181 / 1159.  (What comes from DRAM does not shrink: 2048 tokens on 64 experts 2.01 GB /
//     2.03.)
// Roles per CTA (16 warps): leader only -- warp 0 scheduler (claims, waits for dependencies,
// publishes tile descriptors to both CTAs), warp 1 MMA issuer, warp 2 committer; both CTAs --
// warp 3 producer (TMA loads of its own half of the weights), warps 4-7 gather (a thread of warp 4 loads consecutive rows as boxes),
// warps 8-15 epilogue; second CTA only -- warp 1 relays the completion of its gather to the
// leader.  Tile descriptors reach the second CTA through distributed shared memory; its barrier
// arrivals that the leader waits for are remote mbarrier arrivals.  Its roles give a ring slot back to
// warp 2 (second CTA), which tells the leader.  Every wait is bounded, as in the single-CTA kernel.
#include "moe_combine.cuh"
#include "moe_ptx.cuh"
#include "moe_sched.cuh"

namespace moe {
namespace pairk {

constexpr int kThreads = 512;
constexpr int kGatherThreads = 128;
constexpr int kBBytes = 128 * kRowBytes;                 // this CTA's 128 weight rows of a tile's k-block
// the pipeline for work tiles of up to kTileRows rows
// kDual: two tiles at a time
template <int kTileRows, bool kDual>
struct Ring {
  static constexpr int kRows = kTileRows / 2;            // activation rows of this CTA
  static constexpr int kABytes = kRows * kRowBytes;
  static constexpr int kSB = kABytes + (kDual ? 2 : 1) * kBBytes;
  static constexpr int kNS = kDual ? 4 : kTileRows == 256 ? 6 : kTileRows == 128 ? 8 : 11;
};
// Two tiles at a time: of a tile that runs alone and has so few rows (a decode tile, the end of a list) a stage takes two k-blocks, the second's
// weights and rows in the second half of either part.  With one a stage, half of it was unused and four were in flight where six are
// in the other form: us from claim to commit of decode tiles next to 8192 prefill tokens, 128 tokens on 8 experts 43 that way, 31 now, 36 in the
// other form; 256 on all of 256 experts next to 16 384 37, 25, 31.
constexpr int kWideRows = 128;
constexpr int kWideBytes = kWideRows / 2 * kRowBytes;    // from the rows of the first k-block of a stage to those of the second
constexpr int kAccCols = 256;
// Warps that store a tile, in both CTAs.  Each counts the tile in the words that down and combine tiles wait for as soon as its own
// part is out: one token takes 63.9 us a pass where 65.9 with one thread that counts for all of them after they have met.  (In the
// e4m3 kernel the same costs registers that its epilogue needs, 4 % at 2000 tokens: there the committer counts.)
constexpr int kStoreWarps = 16;
constexpr long long kBeginLimitNs = 1000000000;         // for two round trips of the scheduler
constexpr int kFullCount = 2 + kGatherThreads + 1;
// instruction descriptor: D fp32, A/B bf16, K-major, M = 256 over the pair, N = the tile's columns
constexpr unsigned kIdescM256 = (1u << 4) | (1u << 7) | (1u << 10) | ((256u >> 4) << 24);
// accumulator columns of a tile (16 is the instruction's step), half of them from each CTA's shared memory
__device__ __forceinline__ int tile_cols(int rows) { return (rows + 15) & ~15; }
// k-blocks of a tile that share a stage.  (A launch that runs two tiles at a time has an even number of them in either GEMM: even numbers of n-blocks
// are multiples of 512 in H and of 256 in I.)
static_assert(2 * kTileN2 % (2 * kBlockK) == 0 && 2 * kTileN1 % (2 * kBlockK) == 0, "");
template <bool kDual>
__device__ __forceinline__ int kblocks_a_stage(int rows, bool dual) { return kDual && !dual && tile_cols(rows) <= kWideRows ? 2 : 1; }

template <int kTileRows, bool kDual>
struct SharedCtl {
  // One descriptor a ticket, of two tiles too: the second is the next n-block.  (With one a tile and eight of them a unit claimed up to eight single
  // tiles while its epilogue was at a combine tile: of 256 decode tokens that become ready in the middle of 16 384 of prefill, budget 16, the
  // slowest hundredth of the tiles took 157 us from claim to commit, with four 80.)
  alignas(16) TileInfo info[kRing];
  // leader's: everything the MMAs of a stage read is in place.  kFullCount arrivals: one expect_tx
  // per producer (TMA bytes of both CTAs), one per gather thread of the leader (completion of its
  // cp.async copies) and one from the other CTA's relay warp (that CTA's gathered rows are in
  // place); on tiles without a gather the leader's producer arrives in their place
  unsigned long long full[Ring<kTileRows, kDual>::kNS];
  unsigned long long fullA[Ring<kTileRows, kDual>::kNS];     // second CTA: completion of its own gather threads' copies
  unsigned long long goA[Ring<kTileRows, kDual>::kNS];       // producer -> gather warps: the stage may be overwritten (gathered rows)
  unsigned long long goR[Ring<kTileRows, kDual>::kNS];       // ... (consecutive rows: the thread that loads their boxes)
  unsigned long long empty[Ring<kTileRows, kDual>::kNS];     // both (multicast commit): the stage's MMAs retired
  unsigned long long tfull[2];       // both (multicast commit): accumulator complete
  unsigned long long tempty[2];      // leader's: accumulator drained by the 16 epilogue warps
  unsigned long long ifull[kRing];   // own: tile descriptor published
  unsigned long long iempty[kRing];  // leader's: ring slot released by its roles and, once for all of its own, by the other CTA
  unsigned long long iread[kRing];   // second CTA's: its roles have read the tile descriptor
  unsigned long long done[kRing];    // leader's: the 16 epilogue warps have stored the tile
  unsigned long long taken[kRing];   // leader's: its producer has started on the tile
  unsigned long long rows_in[kRing]; // own: the rows that the tile reads are in place (down tiles: its gate/up tiles are committed)
  // two tiles at a time: the rows of a gathered tile are in `list` (nullptr: none)
  unsigned long long listed[kRing];
  const unsigned char* list[kRing][kDual ? Ring<kTileRows, kDual>::kRows : 1];
  unsigned long long began;          // leader's: the queue tables and qt.run_off are in place
  unsigned combine_ready;            // own: combine tiles so far whose op's expert outputs were seen in place
  unsigned tmem_base;
  alignas(16) unsigned char epi_scratch[8][2048];
  QueueTables qt;
};
static_assert(sizeof(TileInfo) == 48, "descriptor is copied as three 16-byte words");

template <int kTileRows, bool kDual>
constexpr size_t kSmemBytes = 1024 + (size_t)Ring<kTileRows, kDual>::kNS * Ring<kTileRows, kDual>::kSB + sizeof(SharedCtl<kTileRows, kDual>);

// bounded wait on arrivals of the other CTA.  kTry: mbar_try_cluster, or mbar_try_relaxed where a fence of the caller's follows
template <bool (*kTry)(void*, unsigned)>
__device__ __noinline__ bool wait_slow(const Ctx& c, void* bar, unsigned parity, int where) {
  unsigned long long t0 = 0;
  for (unsigned it = 1;; ++it) {
    if (kTry(bar, parity)) return true;
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
template <bool (*kTry)(void*, unsigned)>
__device__ __forceinline__ bool bwait(const Ctx& c, void* bar, unsigned parity, int where) {
  if (kTry(bar, parity)) return true;
  return wait_slow<kTry>(c, bar, parity, where);
}
// whole-warp forms.  The cluster-scope wait is for the hand-offs where this thread then reads
// data the other CTA's threads wrote (the tile descriptor, stored outputs); pipeline barriers,
// whose data moves by TMA, tensor core or this CTA's own threads, take the plain wait.
__device__ __forceinline__ bool wwait_cluster(const Ctx& c, void* bar, unsigned parity, int where) {
  return __all_sync(0xffffffffu, bwait<mbar_try_cluster>(c, bar, parity, where));
}
// by the one thread that issues the MMAs
__device__ __forceinline__ bool wwait_relaxed(const Ctx& c, void* bar, unsigned parity, int where) {
  return bwait<mbar_try_relaxed>(c, bar, parity, where);
}
__device__ __forceinline__ bool wwait(const Ctx& c, void* bar, unsigned parity, int where) {
  return __all_sync(0xffffffffu, mbar_wait(c, bar, parity, where));
}

// A published tile descriptor: in the leader the scheduler's arrival is local, the other CTA reads
// words the leader stored remotely.  The only thing that can delay a descriptor is the scheduler,
// whose own waits are bounded and reported, so this wait gives up later than those (three times
// the limit): a never-ready op is then reported by the wait that met it.
__device__ __noinline__ bool info_wait_one(const Ctx& c, void* bar, unsigned parity, int where, bool leader) {
  unsigned long long t0 = 0;
  for (unsigned it = 1;; ++it) {
    if (leader ? mbar_try(bar, parity) : mbar_try_cluster(bar, parity)) return true;
    if ((it & 63u) == 0) {
      if (aborted(c)) return false;
      const unsigned long long now = gtime_ns();
      if (t0 == 0) t0 = now;
      else if ((long long)(now - t0) > 3 * c.a->wait_ns) {
        report(c.st, MOE_ETIMEOUT, where, (int)blockIdx.x, (int)threadIdx.x, (int)parity);
        return false;
      }
    }
  }
}
__device__ __forceinline__ bool wait_info(const Ctx& c, void* bar, unsigned parity, int where, bool leader) {
  return __all_sync(0xffffffffu, info_wait_one(c, bar, parity, where, leader));
}

// arrival on a barrier that lives in the leader's shared memory
__device__ __forceinline__ void arrive_at_leader(void* bar, bool leader) {
  if (leader) mbar_arrive(bar);
  else mbar_arrive_cluster(map_to_cta(bar, 0));
}

// A role has read what it needs of a ring slot.  In the second CTA it says so to warp 2 of its own CTA, which nothing waits for and which
// orders all of these reads before the leader's next descriptor with one release to the cluster.  A release by the role itself
// waits for its stores and copies: a round trip at the start of every tile, ahead of the gather (one token 57.8 us a pass in place
// of 55.4); arrivals without one, which left that order to the hardware, take as long as this (56.5, now 55.7).
template <int kTileRows, bool kDual>
__device__ __forceinline__ void release_slot(SharedCtl<kTileRows, kDual>* sc, int islot, bool leader) {
  mbar_arrive(leader ? &sc->iempty[islot] : &sc->iread[islot]);
}

// Arrival at the leader behind a fence that orders what it hands over: the fence.acq_rel.gpu of a warp that counts a stored tile (one that
// does not count has stored nothing), the tcgen05.fence of a warp that has drained an accumulator.  A release would wait for the
// stores again.
__device__ __forceinline__ void signal_leader(void* bar, bool leader) {
  if (leader) mbar_arrive(bar);
  else mbar_arrive_relaxed(map_to_cta(bar, 0));
}

// The consecutive rows that one CTA loads per k-block of a tile, as boxes: of the packed intermediate (down tile) or of x itself
// (masked-layout gate/up tile).  None where the rows are gathered.
struct RowPlan {
  const CUtensorMap* map;
  int y, boxes, box_rows;      // first row, number of boxes and their rows
  __device__ __forceinline__ unsigned bytes() const { return (unsigned)(boxes * box_rows * kRowBytes); }
};
__device__ __forceinline__ RowPlan row_plan(const OpDev* op, int kind, int row0, int rows, int rank) {
  const int rpc = tile_cols(rows) / 2;       // rows per CTA
  const int mine = kind == kGateUp ? 0 : min(rows - rank * rpc, rpc);
  const bool fromx = kind != kDown;
  RowPlan p{&op->tm_a8, row0 + rank * rpc, 0, 0};
  if (mine > 96) p = RowPlan{fromx ? &op->tm_x128 : &op->tm_a128, p.y, 1, 128};
  else if (mine > 16) p = RowPlan{fromx ? &op->tm_x32 : &op->tm_a32, p.y, (mine + 31) / 32, 32};
  else if (mine > 0) p = RowPlan{fromx ? &op->tm_x8 : &op->tm_a8, p.y, (mine + 7) / 8, 8};
  return p;
}

// The first feature that CTA `rank` computes of a tile.  Of two tiles that run together the first CTA takes the first half of the features of
// both, so that its weight rows are one box.
__device__ __forceinline__ int first_feature(const TileInfo& ti, int rank, bool dual) {
  const int w = ti.kind == kDown ? kTileN2 / 2 : kTileN1 / 2;             // of a CTA and tile
  return (2 * ti.n + (dual ? 2 * rank : rank)) * w;
}

// Two tiles at a time, in launches with ops of both classes: the k-block of two tiles at which the scheduler may claim what comes after them.  A
// claim at their start is held for twice their time, and that long a unit does not turn to the other class: 128 decode tokens on 8
// experts that arrive in the middle of 8192 of prefill were done after 512, 235 and 210 us at budgets 16, 64 and 128, tile by tile after 479, 183
// and 140, and so after 439, 174 and 134.  The claim and the list of rows need the time of some 16 k-blocks: us a launch with 16, 12, 8 and 4 to go
// (half the tile at most) 2048 + 128 tokens paired 1400, 1410, 1450, 1466, claimed at the start 1403; 1000 + 200 2211, 2221, 2285, 2313 /
// 2228; 2048 + 256 on 128 experts 1339, 1343, 1405, 1436 / 1318.  Launches of one class have nothing to turn to.
constexpr int kClaimBlocks = 16;
__device__ __forceinline__ int late_claim(int kblocks) { return max(0, min(kblocks / 2, kblocks - kClaimBlocks)); }

// The place of the weight rows of one CTA, and their L2 policy
struct WeightPlan {
  const CUtensorMap* map;
  int blk, expert;             // (see OpDev)
  unsigned long long policy;
};
__device__ __forceinline__ WeightPlan weight_plan(const OpDev* op, const TileInfo& ti, int rank, bool dual) {
  WeightPlan p;
  const bool w1 = ti.kind != kDown;          // gate/up weights
  p.map = dual ? (w1 ? &op->tm_w1 : &op->tm_w2) : (w1 ? &op->tm_p1 : &op->tm_p2);
  p.blk = first_feature(ti, rank, dual) / (w1 ? 8 : 16);
  p.expert = expert_of(ti);
  // Where one work tile reads an expert's weights, they are marked to leave L2 first and do not push out what is read again (one token: 72.7 ->
  // 68.8 us; 128 tokens on 8 experts: 88.1 -> 84.3, on 252: 1067 -> 1060).  A plan knows its own op only: of two unpaired ops of a launch
  // that share their weights both mark what the other reads too, at another time, and mostly gain.  Small ops (unmarked -> marked): 100 + 64
  // tokens on 64 experts 397 -> 383, on 8 active experts 91 -> 84, on 32 experts of 3 MB 84 -> 80, but 30 + 20 on 32 active experts 213 ->
  // 218.  Launches of 256-row tiles: 600 + 16 tokens on 64 experts 526 -> 505, 1000 + 32 1613 -> 1591, 300 + 200 1938 -> 1915, 1000 + 200
  // 2205 -> 2170, 8192 + 128 3140 -> 3067, 12288 + 64 3695 -> 3597, 4096 + 64 on 64 experts 1226 -> 1213 (within the spread), but 2048 + 256
  // on 128 experts 1255 -> 1274.  The weights of experts of several tiles are the data read again: marked, they cost (8192 tokens: 2390 ->
  // 2510).
  p.policy = kReadOnce & ti.expert ? l2_evict_first() : l2_evict_normal();
  return p;
}

// The epilogue warps' wait inside a combine tile: one lane of the CTA looks at the op's counter and counts the tile (its `turn`-th) in
// shared memory, where a lane of every warp looks.  Bounded like every wait: any of the warps may have left because the launch was
// aborted.  (With all lanes looking, or on an mbarrier, one token takes 65.4 us a pass where it takes 63.6 this way.)
struct CombineWhenDone {
  const Ctx* c;
  const OpDev* op;
  unsigned* ready;
  unsigned turn;
  bool look;
  __device__ __forceinline__ bool operator()() const {
    if (look && wait_counter(*c, &run_of(*c, op)->gemm_done, op_down_tiles(c->a, op) * kStoreWarps, 4)) st_release_cta(ready, turn);
    __syncwarp();
    const bool first = (threadIdx.x & 31) == 0;
    unsigned long long t0 = 0;
    for (unsigned it = 1;; ++it) {
      int state = 0;                                 // 1: in place, -1: give up
      if (first) {
        if (ld_acquire_cta(ready) >= turn) state = 1;
        else if ((it & 63u) == 0 && !still_waiting(*c, t0, 29)) state = -1;
      }
      state = __shfl_sync(0xffffffffu, state, 0);
      if (state != 0) return state > 0;
      __nanosleep(20);
    }
  }
};

// Two tiles at a time: one warp lists this CTA's rows for the gather warps while the tiles before are still being loaded.  By the gather warps
// themselves, four round trips behind one another at the start of a tile, the MMAs wait 4500 clocks for the first rows of 256.  Where the power
// limit has settled most of that comes back as clock: 8192 tokens 2472 -> 2458 us a pass, 12 288 3190 -> 3178, 4096 + 64 on 64 experts 1245 ->
// 1238; before it has, 2370 -> 2330 and 3030 -> 2940.  (Where tiles are short the scheduler, whose work this is in the leader, is what is
// waited for: 300 + 20 tokens on 32 experts of 3 MB 62.6 -> 64.1, the toy layer 30.5 -> 31.2.  There the gather warps do it.)
template <int kTileRows, bool kDual>
__device__ __forceinline__ void list_rows(const Ctx& c, SharedCtl<kTileRows, kDual>* sc, int islot, int slot, int row0, int rows, int rank,
                                          int lane) {
  const RunArgs& a = *c.a;
  const OpDev* op = &a.ops[slot];
  const bool paired = op->paired != 0;
  const OpDev* pop = paired ? &a.ops[op->partner] : op;
  const unsigned char* X = static_cast<const unsigned char*>(op->x);
  const unsigned char* Xp = static_cast<const unsigned char*>(pop->x);
  const int n_rows = op->n_rows, n_rows_p = pop->n_rows;
  const int own_tag = paired ? slot_of(&a, slot) : 0, partner_tag = paired ? slot_of(&a, op->partner) : 0;
  const int rpc = tile_cols(rows) / 2, first = rank * rpc;         // this CTA's first row of the tile
  const int* list = op->gather_list + row0 + first;
  bool bad = false;
#pragma unroll
  for (int i = 0; i < Ring<kTileRows, kDual>::kRows / 32; ++i) {
    const int r = lane + 32 * i;
    const bool mine = r < rpc && first + r < rows;
    const int v = mine ? list[r] : 0;
    const int tag = v >> kRowSlotShift, flat = v & kRowFlatMask;
    const bool theirs = tag != own_tag;
    const bool in_range = v >= 0 && (tag == own_tag || tag == partner_tag) && flat < (theirs ? n_rows_p : n_rows);   // as by the gather warps
    bad |= mine && !in_range;
    if (r < rpc) sc->list[islot][r] = mine && in_range ? (theirs ? Xp : X) + (size_t)(flat / a.k) * ((size_t)a.H * 2) : nullptr;
  }
  if (bad) report(c.st, MOE_EBOUNDS, slot_of(c.a, slot), row0, rows, 0);
  __syncwarp();
  if (lane == 0) mbar_arrive(&sc->listed[islot]);
}

// the scheduler hands a tile to the roles of both CTAs
template <int kTileRows, bool kDual>
__device__ __forceinline__ void publish(SharedCtl<kTileRows, kDual>* sc, int islot, const TileInfo& ti) {
  sc->info[islot] = ti;
  const unsigned ra = map_to_cta(&sc->info[islot], 1);      // same layout as TileInfo
  st_cluster_v4(ra, make_uint4((unsigned)ti.kind, (unsigned)ti.slot, (unsigned)ti.tile, (unsigned)ti.m));
  st_cluster_v4(ra + 16, make_uint4((unsigned)ti.row0, (unsigned)ti.rows, (unsigned)ti.n, (unsigned)ti.kblocks));
  st_cluster_v4(ra + 32, make_uint4((unsigned)ti.expert, (unsigned)ti.cls, (unsigned)(ti.t_claim & 0xffffffffull),
                                    (unsigned)(ti.t_claim >> 32)));
  mbar_arrive_cluster(map_to_cta(&sc->ifull[islot], 1));   // release: the stores above come first
  __threadfence_block();
  mbar_arrive(&sc->ifull[islot]);
}

template <int kTileRows, bool kDual>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
moe_apk_pair_kernel(const __grid_constant__ RunArgs args, RunHead* rh) {
  using R = Ring<kTileRows, kDual>;
  constexpr int kNS = R::kNS, kSB = R::kSB, kABytes = R::kABytes;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* stages = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  SharedCtl<kTileRows, kDual>* sc = reinterpret_cast<SharedCtl<kTileRows, kDual>*>(stages + (size_t)kNS * kSB);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const bool leader = rank == 0;
  Ctx c{&args, &args.g->status, 0u};

  if (threadIdx.x == 0) {
    for (int s = 0; s < kNS; ++s) {
      mbar_init(&sc->full[s], kFullCount);
      mbar_init(&sc->fullA[s], kGatherThreads);
      mbar_init(&sc->goA[s], 1);
      mbar_init(&sc->goR[s], 1);
      mbar_init(&sc->empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sc->tfull[s], 1);
      mbar_init(&sc->tempty[s], 16);
    }
    // a ring slot is released by: MMA warp, committer, producer, 4 gather warps (leader); warp 2 of the other CTA, where it is read by
    // producer, relay, 4 gather and 8 epilogue warps (the leader's are behind the committer), and the warp that lists rows
    for (int s = 0; s < kRing; ++s) {
      mbar_init(&sc->ifull[s], 1);
      mbar_init(&sc->iempty[s], 8);
      mbar_init(&sc->iread[s], kDual ? 15 : 14);
      mbar_init(&sc->done[s], 16);
      mbar_init(&sc->taken[s], 1);
      mbar_init(&sc->rows_in[s], 1);
      mbar_init(&sc->listed[s], 1);
    }
    mbar_init(&sc->began, 1);
    sc->combine_ready = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_proxy();
  }
  if (warp == 1) {   // TMEM of both CTAs (512 columns each); the same warp frees it
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&sc->tmem_base)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();          // the other CTA's barriers exist before anything arrives on them
  tc_fence_after();
  const unsigned tmem = sc->tmem_base;
  touch_params(args);
  grid_dep_wait();             // everything above overlaps the kernel before this one
  // From here to the first loads of a tile everything is latency: tables, first claim, hand-over.  So no barrier of the CTA stands in
  // between, only the scheduler's own two round trips (4300 + 3900 clocks to a claim before, 2750 + 3500 now).
  // The half of the run state is known to the scheduler first; the roles that need it read it behind a barrier.
  bool ended = true;           // false: this thread left its role because a wait gave up
  const auto set_run_off = [&] {
    c.run_off = sc->qt.run_off;
    rh = reinterpret_cast<RunHead*>(reinterpret_cast<char*>(rh) + c.run_off);
  };

  if (warp == 0 && leader) {
    // ============================================================ scheduler (leader)
    // Claims a tile, waits (bounded) for a free ring slot, the op's ready word and the tile's
    // dependencies, and publishes it to both CTAs.  The next claim starts when the producer has
    // taken the published tile (see late_claim), so the pair holds at most one claimed ticket, a tile or two that run
    // together, beyond the one whose loads are being issued.
    int islot = 0;
    unsigned iph = 0;
    bool lapped = false;                                  // every ring slot has been used
    TileInfo ti;
    bool need_ready = false, two = false;                 // two: the ticket's second tile is the next n-block and runs together with the first
    ti.kind = kEnd;
    ti.slot = ti.tile = ti.m = ti.row0 = ti.rows = ti.n = ti.kblocks = ti.expert = ti.cls = 0;
    ti.t_claim = 0;
    const ClaimWords seen = begin_unit<kDual>(&args, &sc->qt, rh, lane, kStoreWarps, kTileRows);
    set_run_off();
    if (lane == 0) mbar_arrive(&sc->began);
    const bool plain = args.static_kind >= 0;             // plain launch: this pair runs one given entry
    if (plain) claim_static(&args, (int)(blockIdx.x >> 1), ti);
    else claim_next<true, kDual>(c, &sc->qt, rh, lane, ti, need_ready, two, &seen);
    unsigned ticket = 0;
    bool asked = false;
    ended = false;
    while (true) {
      ti.kind = __shfl_sync(0xffffffffu, ti.kind, 0);
      const OpDev* op = &args.ops[ti.kind == kEnd ? args.slots[0] : ti.slot];
      const bool dual = kDual && two && ti.kind != kEnd;
      if (lapped && !wwait_cluster(c, &sc->iempty[islot], iph ^ 1u, 2)) break;
      if (dual) ti.expert |= kTwoTiles;
      if (ti.kind != kEnd && need_ready && !wait_op_ready(c, lane, ti)) ti.kind = kEnd;
      // A down tile is handed over at once: the producers fill the free stages with its weights and add the rows when its gate/up
      // tiles are committed (one token: 67.6 -> 67.0 us a pass, 128 tokens on 8 experts: 80.3 -> 79.1).
      int ok = 1;
      if (lane == 0) {
        publish(sc, islot, ti);
        if (ti.kind == kDown) {
          ok = wait_counter(c, &g1_done_of(c, op)[ti.m], args.I / kTileN1 * kStoreWarps, 3);
          fence_async_proxy();
        }
        if (ok) {
          mbar_arrive_cluster(map_to_cta(&sc->rows_in[islot], 1));
          mbar_arrive(&sc->rows_in[islot]);
        }
        // (asked before the first hand-over, that would wait for the answer: its arrivals release)
        if (!asked) ticket = take_turn(&args);
        asked = true;
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if constexpr (kDual) {
        if (ti.kind == kGateUp && ok) list_rows(c, sc, islot, ti.slot, ti.row0, ti.rows, 0, lane);
      } else {
        // The gather warps will read the tile's row list (4 bytes per row) first thing: pull it into L2
        // now, the weight stream has usually pushed it out since the plan wrote it.
        if (ti.kind == kGateUp && lane * 32 < ti.rows) prefetch_l2(op->gather_list + ti.row0 + lane * 32);
      }
      if (ti.kind == kEnd || !ok) { ended = ok; break; }
      // A combine tile is handed over at once: its epilogue warps read row indices and router weights and then wait for the op's
      // GEMM tiles themselves.  The next claim waits with them, so that a unit holds one such tile at most.
      if (ti.kind == kCombine) {
        if (lane == 0) ok = wait_counter(c, &run_of(c, op)->gemm_done, op_down_tiles(&args, op) * kStoreWarps, 4);
        if (__shfl_sync(0xffffffffu, ok, 0) == 0) break;
      }
      if (!wwait(c, &sc->taken[islot], iph, 26)) break;
      if (++islot == kRing) { islot = 0; iph ^= 1u; lapped = true; }
      two = false;
      if (plain) ti.kind = kEnd;
      else claim_next<true, kDual>(c, &sc->qt, rh, lane, ti, need_ready, two);
    }
    if (lane == 0) end_turn(&args, asked ? ticket : take_turn(&args), (int)(gridDim.x >> 1));
  } else if (kDual && warp == 0) {
    // ============================================================ lists of rows (second CTA; the leader's are its scheduler's)
    ended = false;
    int islot = 0;
    unsigned iph = 0;
    while (true) {
      if (!wait_info(c, &sc->ifull[islot], iph, 34, false)) break;
      const int kind = sc->info[islot].kind, slot = sc->info[islot].slot, row0 = sc->info[islot].row0, rows = sc->info[islot].rows;
      __syncwarp();
      if (kind == kEnd) { ended = true; break; }
      if (kind == kGateUp) list_rows(c, sc, islot, slot, row0, rows, 1, lane);
      if (lane == 0) release_slot(sc, islot, false);
      if (++islot == kRing) { islot = 0; iph ^= 1u; }
    }
  } else if (warp == 3) {
    // ============================================================ producer (both CTAs)
    // Reads tiles from the ring and loads this CTA's weights, one stage per k-block; the rows are loaded by the gather warps, because a TMA
    // instruction holds its thread for some 140 clocks.  One thread runs the whole role (see the MMA issuer).
    if (elect_one()) {
      ended = false;
      int islot = 0;
      unsigned iph = 0;
      unsigned stage = 0, par = 1;                           // parity of "stage is free"
      bool ready = false;                                    // the stage was seen free by the look-ahead test
      const unsigned w0 = smem_u32(stages) + (unsigned)kABytes, go_rows = smem_u32(&sc->goR[0]), go_gather = smem_u32(&sc->goA[0]);
      const unsigned full0 = leader ? smem_u32(&sc->full[0]) : map_to_cta(&sc->full[0], 0), empty0 = smem_u32(&sc->empty[0]);
      while (true) {
        if (!info_wait_one(c, &sc->ifull[islot], iph, 21, leader)) break;
        const TileInfo ti = sc->info[islot];
        if (ti.kind == kEnd) { ended = true; break; }
        const bool dual = kDual && (ti.expert & kTwoTiles) != 0;
        unsigned long long* const taken = &sc->taken[islot];
        const int claim_at = dual && leader && sc->qt.two_classes != 0 ? late_claim(ti.kblocks) : 0;
        if (leader && claim_at == 0) mbar_arrive(taken);
        release_slot(sc, islot, leader);
        if (++islot == kRing) { islot = 0; iph ^= 1u; }
        if (ti.kind == kCombine) continue;
        const OpDev* op = &args.ops[ti.slot];
        const WeightPlan wp = weight_plan(op, ti, rank, dual);
        const unsigned row_bytes = row_plan(op, ti.kind, ti.row0, ti.rows, rank).bytes();
        const unsigned w_bytes = (unsigned)(dual ? 2 * kBBytes : kBBytes);
        const bool g1 = ti.kind == kGateUp;
        const unsigned standin = leader && !g1 ? (unsigned)kGatherThreads + 1u : 0u;   // nobody gathers for this tile
        const unsigned go = g1 ? go_gather : go_rows, has_go = g1 || row_bytes ? 1u : 0u;
        const int step = kblocks_a_stage<kDual>(ti.rows, dual);
        bool fail = false;
        for (int kb = 0; kb < ti.kblocks; kb += step) {
          if (!ready && !mbar_wait(c, &sc->empty[stage], par, 5)) { fail = true; break; }
          if (claim_at > 0 && kb == claim_at) mbar_arrive(taken);
          const unsigned nstage = stage + 1 == kNS ? 0u : stage + 1, npar = stage + 1 == kNS ? par ^ 1u : par;
          ready = pair_issue_kblock(full0 + stage * 8u, (w_bytes + row_bytes) * (unsigned)step, smem_u32(&sc->full[stage]), standin,
                                    go + stage * 8u, has_go, w0 + stage * (unsigned)kSB, wp.map, kb * kBlockK, wp.blk, wp.expert, wp.policy,
                                    empty0 + nstage * 8u, npar);
          if (step == 2)
            pair_issue_weights(full0 + stage * 8u, w0 + stage * (unsigned)kSB + (unsigned)kBBytes, wp.map, (kb + 1) * kBlockK, wp.blk, wp.expert,
                               wp.policy);
          stage = nstage;
          par = npar;
        }
        if (fail) break;
      }
    }
    __syncwarp();
  } else if (warp == 1 && leader) {
    // ============================================================ MMA issuer (leader)
    // One thread runs the whole role.  Inside a branch on elect.sync the compiler knows that a single thread is there and feeds the
    // instructions from uniform registers as they are.  With the whole warp in the loop and an election around each group, the same four MMAs
    // and commit took 300 clocks to issue (350 with the fence of a gathered tile), whatever the tile's rows, now 240 (260); a probe without
    // loads issues them in 155, and in 315 that way.  A k-block of up to 64 gathered rows went from 445 to 390 clocks (4096 tokens on 16
    // experts), 16 384 + 256 paired from 4330 to 4300 us: the 1000 W cap takes most of it back as clock.  One token: 56.0 -> 54.9 us a pass.
    if (elect_one()) {
      ended = false;
      int islot = 0;
      unsigned iph = 0, gcount = 0;
      unsigned stage = 0, par = 0;
      bool ready = false;                             // the current stage was seen full by the look-ahead test
      const unsigned full0 = smem_u32(&sc->full[0]), empty0 = smem_u32(&sc->empty[0]);
      const unsigned long long desc0 = umma_desc(smem_u32(stages), kRowBytes);
      while (true) {
        if (!info_wait_one(c, &sc->ifull[islot], iph, 6, true)) break;
        const int kind = sc->info[islot].kind, kblocks = sc->info[islot].kblocks, rows = sc->info[islot].rows;
        const bool dual = kDual && (sc->info[islot].expert & kTwoTiles) != 0;
        if (kind == kEnd) { ended = true; break; }
        if (kind != kCombine) {
          const unsigned b = gcount & 1u;
          if (!wwait_relaxed(c, &sc->tempty[b], ((gcount >> 1) & 1u) ^ 1u, 7)) break;
          tc_fence_after();
          const unsigned d = tmem + b * (unsigned)kAccCols;
          const unsigned idesc = kIdescM256 | ((unsigned)tile_cols(rows) >> 3) << 17;
          const bool g1 = kind == kGateUp;
          bool fail = false;
          // Two tiles: while the other accumulator is still being stored, the first tile's MMAs of the k-blocks that are there are issued.  (With
          // this, and both tiles stored before either is counted: 8192 tokens 2365 -> 2290 us a pass, 12 288 3175 -> 2990.  Asked with
          // test_wait, which does not suspend the thread, the same or a little slower: 8192 2203 / 2205, 4096 + 64 on 64 experts 1126 / 1137.)
          int ahead = 0;
          if (dual) {
            unsigned st = stage, pa = par;
            unsigned long long* const other = sc->tempty + (b ^ 1u);
            for (; ahead < min(kNS, kblocks) && !mbar_try_relaxed(other, (((gcount + 1) >> 1) & 1u) ^ 1u); ++ahead) {
              if (!(ahead == 0 && ready) && !mbar_wait(c, &sc->full[st], pa, 8)) { fail = true; break; }
              if (g1) fence_async_proxy_smem();
              const unsigned long long xd = desc0 + st * (unsigned)(kSB / 16);
              pair_mma_half(d, xd + (unsigned)(kABytes / 16), xd, idesc, ahead ? 1u : 0u);
              if (++st == kNS) { st = 0; pa ^= 1u; }
            }
            if (fail) break;
            if (!wwait_relaxed(c, &sc->tempty[b ^ 1u], (((gcount + 1) >> 1) & 1u) ^ 1u, 7)) break;
            tc_fence_after();
          }
          // (one loop with a choice in it: 16 and 8 k-blocks a tile, 8000 tokens on 32 experts 185.2 us a pass in place of 183.6)
          const bool wide = kblocks_a_stage<kDual>(rows, dual) == 2;
          if (wide) {
            for (int kb = 0; kb < kblocks; kb += 2) {
              if (!ready && !mbar_wait(c, &sc->full[stage], par, 8)) { fail = true; break; }
              if (g1) fence_async_proxy_smem();
              const unsigned long long xd = desc0 + stage * (unsigned)(kSB / 16), wd = xd + (unsigned)(kABytes / 16);
              const unsigned nstage = stage + 1 == kNS ? 0u : stage + 1, npar = stage + 1 == kNS ? par ^ 1u : par;
              pair_mma_half(d, wd, xd, idesc, kb ? 1u : 0u);
              ready = pair_mma_kblock(d, wd + (unsigned)(kBBytes / 16), xd + (unsigned)(kWideBytes / 16), idesc, 1u, empty0 + stage * 8u,
                                      full0 + nstage * 8u, npar);
              stage = nstage;
              par = npar;
            }
          }
          for (int kb = 0; !wide && kb < kblocks; ++kb) {
            if (kb >= ahead) {
              if (!ready && !mbar_wait(c, &sc->full[stage], par, 8)) { fail = true; break; }
              if (g1) fence_async_proxy_smem();        // this CTA's cp.async-written rows -> tensor core reads
            }
            const unsigned long long xd = desc0 + stage * (unsigned)(kSB / 16), wd = xd + (unsigned)(kABytes / 16);
            const unsigned nstage = stage + 1 == kNS ? 0u : stage + 1, npar = stage + 1 == kNS ? par ^ 1u : par;
            // four MMAs (+32 bytes along K per step: the descriptor's address field counts 16 bytes), the
            // commit that frees the stage in both CTAs, and the test of the next stage's barrier (of the next tile's first one too)
            if (dual) {
              if (kb >= ahead) pair_mma_half(d, wd, xd, idesc, kb ? 1u : 0u);
              if (kb + 1 == kblocks) tc_commit_pair(&sc->tfull[b]);
              ready = pair_mma_kblock(d ^ (unsigned)kAccCols, wd + (unsigned)(kBBytes / 16), xd, idesc, kb ? 1u : 0u, empty0 + stage * 8u,
                                      full0 + nstage * 8u, npar);
            } else {
              ready = pair_mma_kblock(d, wd, xd, idesc, kb ? 1u : 0u, empty0 + stage * 8u, full0 + nstage * 8u, npar);
            }
            stage = nstage;
            par = npar;
          }
          if (fail) break;
          if (dual) ++gcount;
          tc_commit_pair(&sc->tfull[gcount & 1u]);      // accumulator complete, both CTAs
          ++gcount;
        }
        mbar_arrive(&sc->iempty[islot]);
        if (++islot == kRing) { islot = 0; iph ^= 1u; }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ============================================================ gather relay (second CTA)
    // When this CTA's gather threads' copies of a stage have landed it makes them visible to the
    // tensor core (proxy fence) and arrives on the leader's stage barrier.
    if (elect_one()) {
      ended = false;
      int islot = 0;
      unsigned iph = 0, kiter = 0, amask = 0;
      while (true) {
        if (!info_wait_one(c, &sc->ifull[islot], iph, 24, false)) break;
        const int kind = sc->info[islot].kind;
        const bool dual = kDual && (sc->info[islot].expert & kTwoTiles) != 0;
        const int n_stages = sc->info[islot].kblocks >> (kblocks_a_stage<kDual>(sc->info[islot].rows, dual) - 1);
        if (kind == kEnd) { ended = true; break; }
        release_slot(sc, islot, false);
        if (++islot == kRing) { islot = 0; iph ^= 1u; }
        if (kind == kCombine) continue;
        if (kind != kGateUp) { kiter += (unsigned)n_stages; continue; }
        bool fail = false;
        for (int i = 0; i < n_stages; ++i, ++kiter) {
          const int stage = (int)(kiter % kNS);
          if (!mbar_wait(c, &sc->fullA[stage], (amask >> stage) & 1u, 25)) { fail = true; break; }
          amask ^= 1u << stage;
          fence_async_proxy_smem();
          mbar_arrive_remote(map_to_cta(&sc->full[stage], 0));
        }
        if (fail) break;
      }
    }
    __syncwarp();
  } else if (warp >= 4 && warp < 4 + kGatherThreads / 32) {
    // ============================================================ gather warps (cp.async)
    // This CTA's rows of a gate/up tile: row r of the tile is token gather_list[row0 + r] / k.
    // Eight adjacent lanes copy one 128-byte row slice.  Completion is asynchronous: every
    // thread's copies arrive on a barrier when they land (the leader's stage barrier in the
    // leader, a local one that the relay warp forwards in the other CTA), so these warps never
    // wait for their own copies and run as far ahead of the MMAs as the producer does.
    const int gt = threadIdx.x - 128;
    constexpr int kCpr = kRowBytes / 16;                  // 16-byte chunks per row slice
    constexpr int kRowsPerPass = kGatherThreads / kCpr;   // 16 rows per cp.async round
    constexpr int kPasses = Ring<kTileRows, kDual>::kRows / kRowsPerPass;
    constexpr int kWidePasses = kWideRows / 2 / kRowsPerPass < kPasses ? kWideRows / 2 / kRowsPerPass : kPasses;
    const int chunk = gt % kCpr, rbase = gt / kCpr;
    // the swizzle XORs the chunk index with the row's place in its 8-row group, which is the same in every pass
    static_assert(kRowsPerPass % 8 == 0, "");
    const unsigned dst0 = smem_u32(stages) + rbase * kRowBytes + ((chunk ^ (rbase & 7)) << 4);
    ended = false;
    int islot = 0;
    unsigned iph = 0, kiter = 0, gmask = 0, rmask = 0, lmask = 0;
    const unsigned rows0 = smem_u32(stages), full0 = leader ? smem_u32(&sc->full[0]) : map_to_cta(&sc->full[0], 0);
    while (true) {
      if (!wait_info(c, &sc->ifull[islot], iph, 13, leader)) break;
      const int kind = sc->info[islot].kind;
      const int kblocks = sc->info[islot].kblocks;
      const int rows = sc->info[islot].rows, row0 = sc->info[islot].row0, slot = sc->info[islot].slot;
      const bool dual = kDual && (sc->info[islot].expert & kTwoTiles) != 0;
      const int step = kblocks_a_stage<kDual>(rows, dual);
      __syncwarp();
      if (kind == kEnd) { ended = true; break; }
      const int tslot = islot;
      const unsigned tph = iph;
      if (++islot == kRing) { islot = 0; iph ^= 1u; }
      const OpDev* op = &args.ops[slot];
      // Consecutive rows: one thread of one warp loads their boxes, once the scheduler has seen them in place (the weights of a down tile
      // are loaded meanwhile) and the producer has the stage.
      if (kind == kDown || kind == kGateUpDirect) {
        bool fail = false;
        if (warp == 4 && elect_one()) {
          if (kind == kDown) fail = !info_wait_one(c, &sc->rows_in[tslot], tph, 27, leader);
          release_slot(sc, tslot, leader);
          const RowPlan rp = row_plan(op, kind, row0, rows, rank);
          unsigned stage = kiter % (unsigned)kNS;
          if (rp.boxes > 0)
            for (int kb = 0; kb < kblocks && !fail; kb += step) {
              if (!mbar_wait(c, &sc->goR[stage], (rmask >> stage) & 1u, 32)) { fail = true; break; }
              rmask ^= 1u << stage;
              pair_issue_rows(full0 + stage * 8u, kb * kBlockK, rows0 + stage * (unsigned)kSB, rp.map, rp.y, (unsigned)rp.boxes,
                              (unsigned)rp.box_rows);
              if (step == 2)
                pair_issue_rows(full0 + stage * 8u, (kb + 1) * kBlockK, rows0 + stage * (unsigned)kSB + (unsigned)kWideBytes, rp.map, rp.y,
                                (unsigned)rp.boxes, (unsigned)rp.box_rows);
              if (++stage == kNS) stage = 0;
            }
        } else if (warp != 4 && lane == 0) {
          release_slot(sc, tslot, leader);
        }
        if (__any_sync(0xffffffffu, fail)) break;
        kiter += (unsigned)kblocks >> (step - 1);
        continue;
      }
      if (kind == kCombine) {
        if (lane == 0) release_slot(sc, tslot, leader);
        continue;
      }
      const int rpc = tile_cols(rows) / 2, first = rank * rpc;      // this CTA's first row of the tile
      const unsigned char* src[kPasses];                  // this thread's 16 bytes of the row's first k-block
      if constexpr (kDual) {
        if (!wwait(c, &sc->listed[tslot], (lmask >> tslot) & 1u, 35)) break;
        lmask ^= 1u << tslot;
#pragma unroll
        for (int j = 0; j < kPasses; ++j) {
          const int r = rbase + kRowsPerPass * j;
          const unsigned char* row = r < rpc ? sc->list[tslot][r] : nullptr;
          src[j] = row ? row + chunk * 16 : nullptr;
        }
        __syncwarp();
        if (lane == 0) release_slot(sc, tslot, leader);
      } else {
        if (lane == 0) release_slot(sc, tslot, leader);
        // a paired op's gather list also holds rows of its partner, tagged with their slot: those come from
        // the partner's activations
        const bool paired = op->paired != 0;
        const OpDev* pop = paired ? &args.ops[op->partner] : op;
        const unsigned char* X = static_cast<const unsigned char*>(op->x) + chunk * 16;
        const unsigned char* Xp = static_cast<const unsigned char*>(pop->x) + chunk * 16;
        const size_t pitch = (size_t)args.H * 2;
        const int n_rows = op->n_rows, n_rows_p = pop->n_rows;
        const int own_tag = paired ? slot_of(&args, slot) : 0, partner_tag = paired ? slot_of(&args, op->partner) : 0;
        bool bad = false;
#pragma unroll
        for (int j = 0; j < kPasses; ++j) {
          const int r = rbase + kRowsPerPass * j;
          const bool mine = r < rpc && first + r < rows;
          const int v = mine ? op->gather_list[row0 + first + r] : 0;
          const int tag = v >> kRowSlotShift, flat = v & kRowFlatMask;
          const bool theirs = tag != own_tag;
          // an index the plan never wrote is reported below and its row is skipped
          const bool in_range = v >= 0 && (tag == own_tag || tag == partner_tag) && flat < (theirs ? n_rows_p : n_rows);
          bad |= mine && !in_range;
          src[j] = mine && in_range ? (theirs ? Xp : X) + (size_t)(flat / args.k) * pitch : nullptr;
        }
        if (bad) report(c.st, MOE_EBOUNDS, slot_of(&args, slot), row0, rows, 0);
      }
      unsigned long long* landed = leader ? sc->full : sc->fullA;
      bool fail = false;
      for (int kb = 0; kb < kblocks; kb += step, ++kiter) {
        const int stage = (int)(kiter % kNS);
        if (!wwait(c, &sc->goA[stage], (gmask >> stage) & 1u, 14)) { fail = true; break; }
        gmask ^= 1u << stage;
        const unsigned sA = dst0 + stage * (unsigned)kSB;
#pragma unroll
        for (int j = 0; j < kPasses; ++j)
          if (src[j]) cp_async_16(sA + j * (kRowsPerPass * kRowBytes), src[j] + (size_t)kb * kRowBytes);
        if (step == 2) {
#pragma unroll
          for (int j = 0; j < kWidePasses; ++j)
            if (src[j]) cp_async_16(sA + kWideBytes + j * (kRowsPerPass * kRowBytes), src[j] + (size_t)(kb + 1) * kRowBytes);
        }
        cp_async_arrive_noinc(&landed[stage]);
      }
      if (fail) break;
    }
    cp_async_wait_all();
  } else if (warp == 2 && leader) {
    // ============================================================ committer (leader)
    int islot = 0;
    unsigned iph = 0;
    // The scheduler's arrival comes whatever the state of the launch, and the other half has to be cleared in any case (this launch turns
    // the halves over): neither the abort word, which may be set from before, nor a short wait limit ends this wait.
    unsigned long long t0 = 0;
    bool begun = true, watched = false;
    ended = false;
    for (unsigned it = 1; begun && !__all_sync(0xffffffffu, mbar_try(&sc->began, 0u)); ++it)
      if ((it & 63u) == 0) begun = __all_sync(0xffffffffu, in_time(c, t0, kBeginLimitNs, 28));
    if (begun) {
      if (blockIdx.x == 0) clear_next_run(&args, rh, sc->qt.run_off, lane);
      set_run_off();
      watched = sc->qt.watched != 0;
      if (blockIdx.x == 0 && lane == 0 && watched) finish_empty_ops(c, -1);
    }
    while (true) {
      if (!wait_info(c, &sc->ifull[islot], iph, 16, leader)) break;
      TileInfo ti;
      if (lane == 0) ti = sc->info[islot];
      const int kind = __shfl_sync(0xffffffffu, lane == 0 ? ti.kind : 0, 0);
      if (kind == kEnd) { ended = true; break; }
      if (!wwait_cluster(c, &sc->done[islot], iph, 17)) break;
      if (lane == 0) {
        commit_tile<false>(c, rh, ti, watched);
        if (kDual && (ti.expert & kTwoTiles) != 0) {
          ++ti.tile;
          commit_tile<false>(c, rh, ti, watched);
        }
        mbar_arrive(&sc->iempty[islot]);
      }
      __syncwarp();
      if (++islot == kRing) { islot = 0; iph ^= 1u; }
    }
  } else if (warp == 2) {
    // ============================================================ ring slots of the second CTA
    ended = false;
    int islot = 0;
    unsigned iph = 0;
    while (true) {
      if (!wait_info(c, &sc->ifull[islot], iph, 30, false)) break;
      const int kind = __shfl_sync(0xffffffffu, sc->info[islot].kind, 0);
      if (kind == kEnd) { ended = true; break; }
      if (!wait_info(c, &sc->iread[islot], iph, 31, true)) break;       // (an arrival of this CTA)
      if (lane == 0) mbar_arrive_cluster(map_to_cta(&sc->iempty[islot], 0));
      if (++islot == kRing) { islot = 0; iph ^= 1u; }
    }
  } else if (warp >= 8) {
    // ============================================================ epilogue (8 warps per CTA)
    // Warp w reads TMEM lanes 32 (w % 4) .. +31 (weight rows: 2 x (8 gate + 8 up), or 32 down features) and one half of the
    // tile's columns (token rows), 32 tokens per pass.  Fragment loads and transposed 8x8 stores turn a pass into
    // token-major rows of 32 (gate/up) or 64 bytes in the warp's scratch, which leave as 16-byte stores.
    const int q = warp & 3;
    const int half = (warp - 8) >> 2;             // the two warps of a quadrant split the tokens
    const int etid = threadIdx.x - 256;
    ended = false;
    int islot = 0;
    unsigned iph = 0, gcount = 0, combines = 0;
    bool first = true;
    unsigned char* scratch = sc->epi_scratch[warp - 8];
    const unsigned scratch_addr = smem_u32(scratch);
    while (true) {
      if (!wait_info(c, &sc->ifull[islot], iph, 9, leader)) break;
      const TileInfo ti = sc->info[islot];
      if (ti.kind == kEnd) { ended = true; break; }
      __syncwarp();
      if (!leader && lane == 0) release_slot(sc, islot, false);
      const bool dual = kDual && (ti.expert & kTwoTiles) != 0;
      OpDev* op = &args.ops[ti.slot];
      if (first) {
        first = false;
        if (leader) {
          c.run_off = sc->qt.run_off;
        } else {
          unsigned off;
          asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(off) : "r"(map_to_cta(&sc->qt.run_off, 0)) : "memory");
          c.run_off = off;
        }
      }
      bool ok = true;
      if (ti.kind == kCombine) {
        // The two CTAs share the tokens; of one, the columns: a thread then walks one slice of its row, a round trip, where it would walk two
        // and the other CTA none (one token: 56.5 -> 56.0 us a pass).  Two tokens are two slices a thread either way, and by columns both
        // CTAs read the rows and weights of both (82.1-83.1 us either way).
        const int vecs = args.H / 8, mid = ti.row0 + (ti.rows + 1) / 2;
        const bool by_columns = ti.rows == 1;
        const CombineWhenDone ready{&c, op, &sc->combine_ready, ++combines, warp == 8 && lane == 0};
        const int t0 = by_columns || leader ? ti.row0 : mid, t1 = by_columns || !leader ? ti.row0 + ti.rows : mid;
        ok = combine_tokens(op, t0, t1, by_columns && !leader ? vecs / 2 : 0, by_columns ? vecs / 2 : vecs, args.k, args.H, etid, 256, ready);
        if (!ok) break;
      } else {
        // read ahead of the accumulator: behind it these round trips, through a memory system full of weights, delay the tiles that wait
        // for this one (one token: 2.9 us from accumulator to store)
        const bool g1 = ti.kind != kDown;                     // gate/up tile: SwiGLU, output to A
        const StoredWords words = stored_words(c, op, ti);
        unsigned char* const out0 = reinterpret_cast<unsigned char*>(g1 ? (void*)op->A : (void*)op->D);
        const int cols = tile_cols(ti.rows) / 2;              // this warp's columns
        const int live = min(cols, ti.rows - half * cols);    // ... that hold token rows
        const int passes = (live + 31) / 32;
        // Of two tiles that run together both are stored before either is counted: the fence there waits for the stores, and the second
        // accumulator is to be handed back.
#pragma unroll 1
        for (int t = 0; t < (dual ? 2 : 1); ++t) {
          const int b = (int)(gcount & 1u);
          ok = wwait(c, &sc->tfull[b], (gcount >> 1) & 1u, 10);
          if (!ok) break;
          ++gcount;
          tc_fence_after();
          if (passes > 0) {
            const unsigned taddr = tmem + (unsigned)(b * kAccCols + half * cols) + ((unsigned)(q * 32) << 16);
            const size_t pitch = (size_t)(g1 ? args.I : args.H) * 2;
            unsigned char* out = out0 + (size_t)(ti.row0 + half * cols) * pitch +
                                 (size_t)(first_feature(ti, rank, dual) + t * (g1 ? kTileN1 / 2 : kTileN2 / 2) + q * (g1 ? 16 : 32)) * 2;
            unsigned lo[16], hi[16];                            // lanes 0..15 and 16..31 of the quadrant
            tc_ld_frag(taddr, lo);
            tc_ld_frag(taddr + (16u << 16), hi);
#pragma unroll 1
            for (int p = 0; p < passes; ++p) {
              tc_wait_ld();
              const bool last = p + 1 == passes;
              if (last) {                                       // all of it is in registers: the accumulator may be overwritten
                tc_fence_before();
                __syncwarp();
                if (lane == 0) signal_leader(&sc->tempty[b], leader);
              }
              unsigned o[16];
              if (g1) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  o[j] = pack_bf16(silu_mul(__uint_as_float(lo[4 * j]), __uint_as_float(lo[4 * j + 2])),
                                   silu_mul(__uint_as_float(lo[4 * j + 1]), __uint_as_float(lo[4 * j + 3])));
                  o[4 + j] = pack_bf16(silu_mul(__uint_as_float(hi[4 * j]), __uint_as_float(hi[4 * j + 2])),
                                       silu_mul(__uint_as_float(hi[4 * j + 1]), __uint_as_float(hi[4 * j + 3])));
                }
              } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
#pragma unroll
                  for (int r = 0; r < 2; ++r) {
                    o[4 * r + j] = pack_bf16(__uint_as_float(lo[4 * j + 2 * r]), __uint_as_float(lo[4 * j + 2 * r + 1]));
                    o[8 + 4 * r + j] = pack_bf16(__uint_as_float(hi[4 * j + 2 * r]), __uint_as_float(hi[4 * j + 2 * r + 1]));
                  }
                }
              }
              if (!last) {
                tc_ld_frag(taddr + (unsigned)((p + 1) * 32), lo);
                tc_ld_frag(taddr + (unsigned)((p + 1) * 32) + (16u << 16), hi);
              }
              unsigned char* dst = out + (size_t)(p * 32) * pitch;
              const int left = live - p * 32;
              if (g1) {
                __syncwarp();                                   // scratch free again
                // matrix i / 8 of a store is token group i / 8, its row i % 8 is token `lane` of the pass
#pragma unroll
                for (int f = 0; f < 2; ++f)
                  st_matrix4_trans(scratch_addr + lane * 32 + f * 16, o[4 * f], o[4 * f + 1], o[4 * f + 2], o[4 * f + 3]);
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                  const int r = 16 * j + (lane >> 1), f = lane & 1;
                  const uint4 v4 = *reinterpret_cast<const uint4*>(scratch + r * 32 + f * 16);
                  if (r < left) *reinterpret_cast<uint4*>(dst + (size_t)r * pitch + f * 16) = v4;
                }
              } else {
                store_features32(scratch, scratch_addr, o, lane, dst, pitch, left, lane);
              }
            }
          } else {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) signal_leader(&sc->tempty[b], leader);
          }
        }
        if (!ok) break;
        __syncwarp();
        const bool alone = ti.rows <= cols;                   // the columns of the quadrant's other warp hold no rows: one counts for both
        if (lane == 0 && (half == 0 || !alone)) count_stored(words, (alone ? 2 : 1) * (dual ? 2 : 1));
      }
      // The warp's stores, before the tile is published.  Those of a GEMM tile are behind the fence of count_stored (a warp that does not
      // count stores nothing); of a combine tile the arrival releases them (across the pair: at cluster scope).  The committer's
      // fence is cumulative over what it sees here.
      __syncwarp();
      if (lane == 0) {
        if (ti.kind == kCombine) arrive_at_leader(&sc->done[islot], leader);
        else signal_leader(&sc->done[islot], leader);
      }
      if (++islot == kRing) { islot = 0; iph ^= 1u; }
    }
  }

  // teardown: nothing is claimed any more.  Where a role gave up, asynchronous work may be under way: let it settle.  Then free TMEM
  tc_fence_before();
  if (__syncthreads_or(!ended)) __nanosleep(20000);
  cluster_sync_all();          // no CTA leaves while the other may still signal its barriers
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

}  // namespace pairk

template <int kTileRows, bool kDual>
static cudaError_t prepare_one() {
  return cudaFuncSetAttribute(pairk::moe_apk_pair_kernel<kTileRows, kDual>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)pairk::kSmemBytes<kTileRows, kDual>);
}
cudaError_t prepare_pair_kernel() {
  cudaError_t e = prepare_one<kWorkRowsBf16, true>();
  if (e == cudaSuccess) e = prepare_one<kWorkRowsBf16, false>();
  if (e == cudaSuccess) e = prepare_one<kWorkRowsMid, false>();
  return e == cudaSuccess ? prepare_one<kWorkRowsSmall, false>() : e;
}

// n_ctas: the persistent grid, or 2 x the number of queue entries for a plain launch
template <int kTileRows, bool kDual>
static cudaError_t launch_one(const RunArgs& args, RunHead* rh, int n_ctas, cudaStream_t stream) {
  return launch_after(pairk::moe_apk_pair_kernel<kTileRows, kDual>, n_ctas, pairk::kThreads, pairk::kSmemBytes<kTileRows, kDual>, stream, args, rh);
}
// dual: of a launch with work tiles of up to 256 rows
cudaError_t launch_pair(const RunArgs& args, RunHead* rh, int n_ctas, bool dual, cudaStream_t stream) {
  return args.work_rows <= kWorkRowsSmall ? launch_one<kWorkRowsSmall, false>(args, rh, n_ctas, stream)
         : args.work_rows <= kWorkRowsMid ? launch_one<kWorkRowsMid, false>(args, rh, n_ctas, stream)
         : dual                           ? launch_one<kWorkRowsBf16, true>(args, rh, n_ctas, stream)
                                          : launch_one<kWorkRowsBf16, false>(args, rh, n_ctas, stream);
}

}  // namespace moe
