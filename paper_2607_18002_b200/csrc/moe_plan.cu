// moe_plan: top-k expert ids -> per-expert counts, exclusive offsets (device prefix sum),
// the stable permutation of routed rows, the m-tile table (its length is the footprint
// x_moe of Section 6.2 of the paper) and the ordered tile list the persistent kernel's
// queues serve.
//
// The permutation is one stable counting-sort pass over the expert id.  Every block of the rank kernel owns a
// contiguous range of rows and knows, per expert, how many rows lie before its range; inside the block rows are
// ranked by warp and lane order.  Atomics only count, none decides an order, so the result is unique and reproducible.
//
// A plan is a chain of latencies, not of bytes (8192 tokens x 8: 0.26 MB of ids), so the work is cut for few
// launches and no serial part: the per-expert sums that every block needs are recomputed by every block instead of being
// handed on by one, and the list is written by all blocks, one warp per expert.
#include "moe_dev.cuh"

namespace moe {

constexpr int kPlanThreads = kPlanChunk;
constexpr int kPlanWarps = kPlanThreads / 32;
constexpr int kPlanDirectRows = 8192;   // up to here every block counts all rows itself: no histogram launch
// experts per block of a list, a warp each: the fewer, the more SMs share the stores (1024 rows over 252 experts: 0.7 us less a
// plan with 8 than with 32)
constexpr int kPlanListExperts = 8;
constexpr int kPlanMaxBlocks = 128;     // beyond kPlanMaxBlocks x kPlanChunk rows a block owns several chunks

// One warp: out[e] = f(rows[0]) + ... + f(rows[e - 1]) for e in [0, E], in shared memory.  Both arrays hold kScan entries, rows[e] is 0
// from E on and f(0) = 0: a lane's experts are neighbours and come four at a time.  The scans of a plan run side by side on different
// warps with one barrier behind them (8 rows over 256 experts: 5.2 us a plan with block-wide scans of three barriers each, one
// after the other; 4.1 us).
constexpr int kScan = kMaxExperts + 4;
template <class F>
__device__ __forceinline__ void warp_scan(int* out, const int* rows, int E, F f) {
  const int lane = threadIdx.x & 31, quads = ((E + 31) / 32 + 3) / 4;           // a lane has 4 * quads experts
  const int4* in = reinterpret_cast<const int4*>(rows) + lane * quads;
  int sum = 0;
#pragma unroll 2
  for (int i = 0; i < quads; ++i) {
    const int4 v = in[i];
    sum += f(v.x) + f(v.y) + f(v.z) + f(v.w);
  }
  int inc = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, inc, d);
    if (lane >= d) inc += v;
  }
  int pos = inc - sum;
#pragma unroll 2
  for (int i = 0; i < quads; ++i) {
    const int4 v = in[i];
    int4 o;
    o.x = pos;
    o.y = o.x + f(v.x);
    o.z = o.y + f(v.y);
    o.w = o.z + f(v.z);
    pos = o.w + f(v.w);
    reinterpret_cast<int4*>(out)[lane * quads + i] = o;
  }
  if (lane == 31) out[128 * quads] = inc;           // (E where E fills the lanes)
}

// tile: a power of two
__device__ __forceinline__ int tiles_of(int rows, int tile) { return (rows + tile - 1) >> (31 - __clz(tile)); }

// what a launch needs to know of the op before it looks at its descriptor
struct OpKind {
  int cls, flags;
};
static OpKind kind_of(const OpDev& h) {
  return OpKind{h.cls, (h.ready == nullptr && h.after_op < 0 ? kOpFree : 0) |
                           (h.done != nullptr || h.notify != nullptr || h.after_op >= 0 ? kOpWatched : 0)};
}

// The entries of the wx work tiles x nt n-blocks of one expert's GEMM, by one warp: put(i, n, j) for entry i, n-block n of work tile j.
// n-major over the work tiles, so that they share a weight tile in L2.  In
// lists that are handed out in twos (nt is even) two n-blocks of a work tile lie next to one another, and the sweeps over n go over kSweep work tiles
// at a time: the rows of a popular expert's tiles (1.6 MB each) are still in L2 for the next n-block, and its weights for the next tiles
// (16 384 + 256 tokens paired: 12.8 -> 12.3 GB read from DRAM, 4130 -> 4066 us a pass; 4 or 16 tiles 4073, 4089.  4096 + 512 tokens in e4m3, tiles
// of 0.8 MB: 13.0 -> 13.1 GB, 3289 -> 3307, so the lists of that kernel are swept whole).
constexpr int kSweep = 8;
template <class Put>
__device__ __forceinline__ void sweep(int wx, int nt, int twos, int lane, Put put) {
  if (!twos) {
    for (int i = lane; i < wx * nt; i += 32) {
      const int n = wx == 1 ? i : i / wx;
      put(i, n, i - n * wx);
    }
    return;
  }
  for (int j0 = 0; j0 < wx; j0 += kSweep) {
    const int w = min(kSweep, wx - j0);
    for (int i = lane; i < w * nt; i += 32) {
      int n = i, j = 0;
      if (w > 1) {
        const int p = w == kSweep ? i / (2 * kSweep) : i / (2 * w);           // (a division takes as long as the rest)
        n = 2 * p + (i & 1);
        j = (i - 2 * p * w) >> 1;
      }
      put(j0 * nt + i, n, j0 + j);
    }
  }
}

// ---------------------------------------------------------------- the ordered tile list of one op
// Writes this block's share of the queue list of an op whose expert e holds rows [off[e], off[e] + cnt[e]) of the
// packed row space (cnt / off / work in shared memory; work[e]: work tiles of the experts before e), and (block 0) its
// PlanState.  All blocks of the grid call it.  form.read_once: the mark of entries whose weights no other entry reads; other_work: the
// work tiles of the other list of a pair, like work.
// Work tiles (the unit the queues hand out): up to `work_rows` consecutive rows of one
// expert, i.e. one or two adjacent m-tiles that share each weight tile they read.
// Order: the gate/up entries in expert order, and the down entries of an expert in front of the first expert whose
// gate/up tiles start at least kLagWork work tiles behind its own, so by the time a down tile is claimed the tiles it
// depends on were claimed long before.  Every entry's place follows from the prefix sum of the work tiles.
__device__ __forceinline__ int build_tile_list(int4* tile_list, PlanState* plan, OpKind op, const int* cnt, const int* off, const int* work,
                                                int E, int NT1, int NT2, int T, int work_rows, int x_moe, int planned,
                                                int n_extra_gemm, ListForm form, const int* other_work = nullptr, int g1_kind = kGateUp) {
  const int n_work = work[E];
  // Inside an expert: n-major over its work tiles, so an expert's entries of one GEMM are one
  // contiguous run of the list.  One warp per expert writes them (a popular expert has hundreds).
  const int lane = threadIdx.x & 31;
  for (int x = (int)blockIdx.x + (int)gridDim.x * (int)(threadIdx.x >> 5); x < E; x += (int)gridDim.x * kPlanWarps) {
    const int mx = work[x], wx = work[x + 1] - mx;
    if (wx == 0) continue;
    const int cx = cnt[x], ox = off[x];
    const int ex = x | (wx == 1 && (!other_work || other_work[x + 1] == other_work[x]) ? form.read_once : 0);
    // Work tiles whose down entries come before expert x's gate/up entries (those of the experts that end kLagWork tiles
    // ahead of it), and whose gate/up entries come before its down entries (up to the first expert that starts kLagWork tiles
    // after its end): the largest work[i] <= mx - kLagWork, and the smallest work[i] >= mx + wx + kLagWork.
    int down_before = 0, up_before = n_work;
    for (int i = lane; i <= E; i += 32) {
      const int v = work[i];
      if (v <= mx - kLagWork) down_before = max(down_before, v);
      if (v >= mx + wx + kLagWork) up_before = min(up_before, v);
    }
    down_before = __reduce_max_sync(0xffffffffu, down_before);
    up_before = __reduce_min_sync(0xffffffffu, up_before);
    int4* g1 = tile_list + (size_t)mx * NT1 + (size_t)down_before * NT2;
    int4* g2 = tile_list + (size_t)up_before * NT1 + (size_t)mx * NT2;
    const auto entry = [&](int kind, int n, int j) {
      return make_entry(kind, n, mx + j, ox + j * work_rows, min(work_rows, cx - j * work_rows), ex);
    };
    sweep(wx, NT1, form.twos, lane, [&](int i, int n, int j) { g1[i] = entry(g1_kind, n, j); });
    sweep(wx, NT2, form.twos, lane, [&](int i, int n, int j) { g2[i] = entry(kDown, n, j); });
  }
  const int n_gemm = n_work * (NT1 + NT2);
  const int ct = combine_tile_tokens(T);
  const int n_comb = (T + ct - 1) / ct;
  for (int c = (int)(blockIdx.x * blockDim.x + threadIdx.x); c < n_comb; c += (int)(gridDim.x * blockDim.x))
    tile_list[n_gemm + c] = make_entry(kCombine, 0, c, c * ct, min(ct, T - c * ct), 0);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    PlanState ps;
    ps.n_mtiles = x_moe;
    ps.n_gemm_tiles = n_gemm;
    ps.n_comb_tiles = n_comb;
    ps.planned = planned;                   // a plan with a rejected id leaves the slot without tiles to run
    ps.n_extra_gemm = n_extra_gemm;
    ps.work_rows = work_rows;
    ps.cls = op.cls;
    ps.flags = op.flags;
    *plan = ps;
  }
  return n_gemm;
}

// ---------------------------------------------------------------- histogram and rank
// What the plan kernels read and write, by value: no descriptor has to be fetched first.
struct PlanArgs {
  const int* ids;       // [R]
  int* counts;          // [E]
  int* offsets;         // [E+1]
  int* s2f;             // [R]
  int* f2s;             // [R]
  int* hist;            // [blocks][E] rows per block and expert
  MTile* mtiles;
  int4* tile_list;
  PlanState* plan;
  Status* status;
  OpKind op;
  int slot, R, E, T, NT1, NT2, work_rows;
  ListForm form;
  int own;              // rows per block: block b owns rows [b * own, (b + 1) * own)
};

__global__ void __launch_bounds__(kPlanThreads) plan_hist_kernel(const __grid_constant__ PlanArgs a) {
  __shared__ int h[kMaxExperts];
  for (int e = threadIdx.x; e < a.E; e += kPlanThreads) h[e] = 0;
  grid_dep_wait();
  __syncthreads();
  const int i0 = (int)blockIdx.x * a.own, i1 = min(a.R, i0 + a.own);
  for (int i = i0 + (int)threadIdx.x; i < i1; i += kPlanThreads) {
    const int id = a.ids[i];
    if (id >= 0 && id < a.E) atomicAdd(&h[id], 1);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < a.E; e += kPlanThreads) a.hist[(size_t)blockIdx.x * a.E + e] = h[e];
}

// kDirect: no histogram was made, every block counts all rows itself (R <= kPlanDirectRows).  A warp's first 32 ids and their peers
// stay in registers from the count to the ranking (8 rows over 256 experts: 4.25 -> 3.70 us a plan, 1024 rows: 7.3 -> 5.8).
template <bool kDirect>
__global__ void __launch_bounds__(kPlanThreads) plan_rank_kernel(const __grid_constant__ PlanArgs a) {
  extern __shared__ int run[];              // [kPlanWarps][E]: next packed position of an expert's row per warp
  __shared__ alignas(16) int s_cnt[kScan], s_off[kScan], s_work[kScan], s_mtile[kScan];
  __shared__ int s_before[kMaxExperts];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int E = a.E, R = a.R;
  const int i0 = min(R, (int)blockIdx.x * a.own), i1 = min(R, i0 + a.own);

  const int share = a.own / kPlanWarps;
  const int w0 = min(i1, i0 + warp * share), w1 = min(i1, w0 + share);
  for (int e = tid; e < kMaxExperts; e += kPlanThreads) s_before[e] = s_cnt[e] = 0;
  for (int i = tid; i < kPlanWarps * E; i += kPlanThreads) run[i] = 0;
  grid_dep_wait();
  const int first_id = w0 + lane < w1 ? a.ids[w0 + lane] : -1;   // of this warp's share; read while the counts are
  __syncthreads();
  // rows per expert: all of them, and those before this block's range
  if (kDirect) {
#pragma unroll 4
    for (int i = tid; i < R; i += kPlanThreads) {
      const int id = a.ids[i];
      if (id >= 0 && id < E) {
        atomicAdd(&s_cnt[id], 1);
        if (i < i0) atomicAdd(&s_before[id], 1);
      }
    }
  } else {
    const int parts = max(1, kPlanThreads / E), part = tid / E, e = tid % E;
    const int nb = (int)gridDim.x, per = (nb + parts - 1) / parts;
    const int b0 = min(nb, part * per), b1 = min(nb, b0 + per);
    int before = 0, all = 0;
    if (part < parts) {
#pragma unroll 16
      for (int b = b0; b < b1; ++b) {
        const int v = a.hist[(size_t)b * E + e];
        if (b < (int)blockIdx.x) before += v;
        all += v;
      }
      if (before) atomicAdd(&s_before[e], before);
      if (all) atomicAdd(&s_cnt[e], all);
    }
  }
  // this block's rows: each warp counts a contiguous share of them per expert
  int* mine = run + warp * E;
  const unsigned lower = (1u << lane) - 1u;
  unsigned first_peers = 0;
  for (int base = w0; base < w1; base += 32) {
    const int i = base + lane;
    int id = base == w0 ? first_id : i < w1 ? a.ids[i] : -1;
    if (i < w1 && (id < 0 || id >= E)) {
      report(a.status, MOE_EBADID, a.slot, i, id, 0);
      id = -1;
    }
    const unsigned peers = __match_any_sync(0xffffffffu, id);
    if (base == w0) first_peers = peers;
    if (id >= 0 && (peers & lower) == 0) mine[id] += __popc(peers);
    __syncwarp();
  }
  __syncthreads();

  if (warp == 0) warp_scan(s_off, s_cnt, E, [](int rows) { return rows; });      // device prefix sum over experts
  if (warp == 1) warp_scan(s_work, s_cnt, E, [&](int rows) { return tiles_of(rows, a.work_rows); });
  if (warp == 2) warp_scan(s_mtile, s_cnt, E, [](int rows) { return tiles_of(rows, kTileM); });
  __syncthreads();
  const int cnt = tid < E ? s_cnt[tid] : 0, off = tid < E ? s_off[tid] : 0, total = s_off[E];
  if (tid < E) {
    int pos = off + s_before[tid];          // rows of the expert: earlier blocks, then the warps of this one
    const int warps = min(kPlanWarps, (i1 - i0 + share - 1) / share);
#pragma unroll 8
    for (int w = 0; w < warps; ++w) {
      const int v = run[w * E + tid];
      run[w * E + tid] = pos;
      pos += v;
    }
    if (blockIdx.x == 0) {
      a.counts[tid] = cnt;
      a.offsets[tid] = off;
      if (tid == 0) a.offsets[E] = total;
    }
  }
  __syncthreads();
  // stable positions
  for (int base = w0; base < w1; base += 32) {
    const int i = base + lane;
    int id = base == w0 ? first_id : i < w1 ? a.ids[i] : -1;
    if (id < 0 || id >= E) id = -1;         // reported above
    const unsigned peers = base == w0 ? first_peers : __match_any_sync(0xffffffffu, id);
    int p = -1;
    if (id >= 0) p = mine[id] + __popc(peers & lower);
    __syncwarp();
    if (id >= 0 && (peers & lower) == 0) mine[id] += __popc(peers);
    __syncwarp();
    if (i < w1) {
      a.f2s[i] = p;                         // -1: a rejected id, the row has no packed position
      if (p >= 0) a.s2f[p] = i;
    }
  }
  // rows with a rejected expert id take no packed position: the tail of the permutation that no row
  // will claim is marked, so that nothing downstream mistakes stale memory for an index
  for (int p = total + (int)(blockIdx.x * kPlanThreads) + tid; p < R; p += (int)gridDim.x * kPlanThreads) a.s2f[p] = -1;

  // m-tiles: ceil(m_e / M_t) per expert with rows (the footprint x_moe)
  if (blockIdx.x == 0 && tid < E)
    for (int j = 0, m0 = s_mtile[tid], me = s_mtile[tid + 1] - m0; j < me; ++j)
      a.mtiles[m0 + j] = MTile{tid, off + j * kTileM, min(kTileM, cnt - j * kTileM), 0};
  build_tile_list(a.tile_list, a.plan, a.op, s_cnt, s_off, s_work, E, a.NT1, a.NT2, a.T, a.work_rows, s_mtile[E], total == R ? 1 : 0, 0,
                  a.form);
}

// ---------------------------------------------------------------- masked layout
// The activations already sit in per-expert slabs of slab_rows rows; counts[e] (an input here) says how many
// rows of slab e are valid.  Nothing is permuted: the plan is the exclusive prefix sum for `offsets`, the
// m-tile table (first row of a tile = e * slab_rows + 128 j) and the queue list over the slabs' valid rows.
__global__ void __launch_bounds__(kPlanThreads) plan_masked_kernel(const __grid_constant__ PlanArgs a, int slab_rows) {
  __shared__ alignas(16) int s_cnt[kScan], s_pos[kScan], s_work[kScan], s_mtile[kScan];
  __shared__ int s_off[kMaxExperts];
  const int e = threadIdx.x, warp = e >> 5, E = a.E;
  int cnt = 0;
  grid_dep_wait();
  if (e < E) {
    cnt = a.counts[e];
    if (cnt < 0 || cnt > slab_rows) {        // a count the slab cannot hold: reported, the slab is left out
      if (blockIdx.x == 0) report(a.status, MOE_EBOUNDS, a.slot, e, cnt, 4);
      cnt = 0;
    }
    s_off[e] = e * slab_rows;
  }
  s_cnt[e] = cnt;                            // 0 from E on
  __syncthreads();
  if (warp == 0) warp_scan(s_pos, s_cnt, E, [](int rows) { return rows; });
  if (warp == 1) warp_scan(s_work, s_cnt, E, [&](int rows) { return tiles_of(rows, a.work_rows); });
  if (warp == 2) warp_scan(s_mtile, s_cnt, E, [](int rows) { return tiles_of(rows, kTileM); });
  __syncthreads();
  if (blockIdx.x == 0) {
    for (int i = e; i <= E; i += kPlanThreads) a.offsets[i] = s_pos[i];
    if (e < E)
      for (int j = 0, m0 = s_mtile[e], me = s_mtile[e + 1] - m0; j < me; ++j)
        a.mtiles[m0 + j] = MTile{e, e * slab_rows + j * kTileM, min(kTileM, cnt - j * kTileM), 0};
  }
  build_tile_list(a.tile_list, a.plan, a.op, s_cnt, s_off, s_work, E, a.NT1, a.NT2, 0, a.work_rows, s_mtile[E], 1, 0, a.form, nullptr,
                  kGateUpDirect);
}

// ---------------------------------------------------------------- the paired form of a decode + prefill op
// Two ops of one launch that share their expert weights can share weight tiles too.  The paired form puts
// the routed rows of both into ONE packed row space -- per expert the prefill rows (in their plan's order)
// followed by the decode rows (in theirs) -- and cuts it into two queue lists: per expert, the decode list
// takes the decode rows plus the ragged tail of the prefill rows just before them if it fits into the decode
// rows' last tile of `carrier_rows` rows ("carrier" tiles: claimed with decode priority, they stream a weight
// tile once for rows of both ops); the prefill list takes the rest.  Nothing about a row's arithmetic depends on the
// tile it sits in, so the outputs are those of the unpaired ops, bit for bit.
struct PairSide {
  const int* ids;             // the op's plain plan, as its moe_plan call left it earlier on the stream
  const int* counts;
  const int* offsets;
  const int* f2s;
  const PlanState* plain;
  int4* tile_list;            // the paired form's list and state, written here
  PlanState* plan;
  int* comb;                  // flat routed index -> row of the shared space
  int R, T, slot;
  OpKind op;
};
struct PairArgs {
  PairSide d, p;
  int* gather;                // row of the shared space -> flat routed index, tagged with its slot
  int E, NT1, NT2, work_rows, carrier_rows;
  ListForm form;
};

// One launch: every block scans the experts and writes its share of both lists, then moves its share of the rows
// into the shared row space.
__global__ void __launch_bounds__(kPlanThreads) plan_pair_kernel(const __grid_constant__ PairArgs a) {
  __shared__ alignas(16) int cnt_d[kScan], cnt_p[kScan], work_d[kScan], work_p[kScan];
  __shared__ int off_d[kMaxExperts], off_p[kMaxExperts];
  __shared__ int base_d[kMaxExperts], base_p[kMaxExperts];   // what a row's packed position is shifted by
  const int e = threadIdx.x, E = a.E;
  grid_dep_wait();
  if (e < E) {
    const int cd = a.d.counts[e], cp = a.p.counts[e];
    const int od = a.d.offsets[e], op = a.p.offsets[e];
    const int moff = od + op;
    // the carrier takes the ragged tail of the prefill rows (what is left over after the prefill op's full work
    // tiles) when that tail fits beside the decode rows: a prefill tile less to run.  A tail that does not fit
    // stays where it is -- moving part of it would make the carrier heavier and save nothing.
    const int room = cd > 0 ? (cd + a.carrier_rows - 1) / a.carrier_rows * a.carrier_rows - cd : 0;
    const int tail = cp % max(a.work_rows, a.carrier_rows);
    const int take = tail <= room ? tail : 0;
    cnt_p[e] = cp - take;
    off_p[e] = moff;
    cnt_d[e] = cd + take;
    off_d[e] = moff + cp - take;
    base_p[e] = od;                                          // the decode rows of the experts before
    base_d[e] = op + cp;                                     // ... and the expert's own prefill rows
  } else {
    cnt_p[e] = cnt_d[e] = 0;
  }
  __syncthreads();
  const int ok = (a.d.plain->planned && a.p.plain->planned) ? 1 : 0;
  // a carrier taller than the kernel's work tile (e4m3: 128 rows) is cut into work tiles that follow one another
  const int rows_d = min(a.carrier_rows, a.work_rows);
  if (e < 32) warp_scan(work_d, cnt_d, E, [&](int rows) { return tiles_of(rows, rows_d); });
  else if (e < 64) warp_scan(work_p, cnt_p, E, [&](int rows) { return tiles_of(rows, a.work_rows); });
  __syncthreads();
  const int n_dec = build_tile_list(a.d.tile_list, a.d.plan, a.d.op, cnt_d, off_d, work_d, E, a.NT1, a.NT2, a.d.T, rows_d,
                                    a.d.plain->n_mtiles, ok, 0, a.form, work_p);
  // every GEMM entry of the decode list may carry prefill rows: the prefill op is complete when they are too
  build_tile_list(a.p.tile_list, a.p.plan, a.p.op, cnt_p, off_p, work_p, E, a.NT1, a.NT2, a.p.T, a.work_rows, a.p.plain->n_mtiles, ok,
                  n_dec, a.form, work_d);
  // the shared row space's permutation
  for (int i = (int)(blockIdx.x * kPlanThreads + threadIdx.x); i < a.d.R + a.p.R; i += (int)gridDim.x * kPlanThreads) {
    const bool dec = i < a.d.R;
    const PairSide& s = dec ? a.d : a.p;
    const int j = dec ? i : i - a.d.R;
    const int x = s.ids[j], ps = s.f2s[j];
    int m = -1;
    if (x >= 0 && x < E && ps >= 0) {
      m = ps + (dec ? base_d[x] : base_p[x]);
      a.gather[m] = j | (s.slot << kRowSlotShift);
    }
    s.comb[j] = m;
  }
}

// ---------------------------------------------------------------- launches
// blocks that write a list
static int list_blocks(int E) { return (E + kPlanListExperts - 1) / kPlanListExperts; }

cudaError_t launch_plan_masked(const OpDev& h, int slot, int E, int NT1, int NT2, int slab_rows, int work_rows,
                               ListForm form, cudaStream_t stream) {
  PlanArgs a{};
  a.counts = h.counts; a.offsets = h.offsets; a.mtiles = h.mtiles; a.tile_list = h.tile_list; a.plan = h.plan;
  a.status = h.status;
  a.op = kind_of(h);
  a.slot = slot; a.E = E; a.NT1 = NT1; a.NT2 = NT2; a.work_rows = work_rows; a.form = form;
  return launch_after(plan_masked_kernel, list_blocks(E), kPlanThreads, 0, stream, a, slab_rows);
}

cudaError_t launch_plan_pair(const OpDev& hd, const OpDev& hp, const OpDev& d, const OpDev& p, int* gather, int* comb_d,
                             int* comb_p, int E, int NT1, int NT2, int work_rows, int carrier_rows, ListForm form,
                             int slot_d, int slot_p, cudaStream_t stream) {
  PairArgs a{};
  a.d = PairSide{d.topk_ids, d.counts, d.offsets, d.flat_to_sorted, d.plan, hd.tile_list, hd.plan, comb_d, d.n_rows, d.n_tokens, slot_d, kind_of(d)};
  a.p = PairSide{p.topk_ids, p.counts, p.offsets, p.flat_to_sorted, p.plan, hp.tile_list, hp.plan, comb_p, p.n_rows, p.n_tokens, slot_p, kind_of(p)};
  a.gather = gather;
  a.E = E; a.NT1 = NT1; a.NT2 = NT2; a.work_rows = work_rows; a.carrier_rows = carrier_rows; a.form = form;
  const int blocks = max(list_blocks(E), min(kPlanMaxBlocks, (d.n_rows + p.n_rows + kPlanThreads - 1) / kPlanThreads));
  return launch_after(plan_pair_kernel, blocks, kPlanThreads, 0, stream, a);
}

cudaError_t prepare_plan_kernels() {
  const int most = kPlanWarps * kMaxExperts * (int)sizeof(int);
  const cudaError_t e = cudaFuncSetAttribute(plan_rank_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(plan_rank_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

// h: the op's descriptor as the host holds it
cudaError_t launch_plan(const OpDev& h, int slot, int E, int NT1, int NT2, int work_rows, ListForm form, cudaStream_t stream) {
  PlanArgs a{};
  a.ids = h.topk_ids; a.counts = h.counts; a.offsets = h.offsets; a.s2f = h.sorted_to_flat; a.f2s = h.flat_to_sorted;
  a.hist = h.plan_hist; a.mtiles = h.mtiles; a.tile_list = h.tile_list; a.plan = h.plan; a.status = h.status;
  a.op = kind_of(h);
  a.slot = slot; a.R = h.n_rows; a.E = E; a.T = h.n_tokens; a.NT1 = NT1; a.NT2 = NT2; a.work_rows = work_rows;
  a.form = form;
  const size_t smem = (size_t)kPlanWarps * E * sizeof(int);
  if (a.R <= kPlanDirectRows) {
    const int blocks = list_blocks(E);
    a.own = max(1, ((a.R + blocks - 1) / blocks + kPlanThreads - 1) / kPlanThreads) * kPlanThreads;   // (an op without tokens too)
    return launch_after(plan_rank_kernel<true>, blocks, kPlanThreads, smem, stream, a);
  }
  a.own = kPlanThreads * (int)(((long long)a.R + kPlanThreads * kPlanMaxBlocks - 1) / (kPlanThreads * kPlanMaxBlocks));
  const int blocks = (a.R + a.own - 1) / a.own;
  const cudaError_t e = launch_after(plan_hist_kernel, blocks, kPlanThreads, 0, stream, a);
  return e != cudaSuccess ? e : launch_after(plan_rank_kernel<false>, blocks, kPlanThreads, smem, stream, a);
}

}  // namespace moe
