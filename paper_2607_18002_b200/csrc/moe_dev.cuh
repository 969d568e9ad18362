// Device-side data structures shared by the plan, run and combine kernels and the host
// code that lays them out inside the caller's workspace.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/moe_apk.h"

namespace moe {

constexpr int kTileM = MOE_TILE_M;   // token rows per tile (M_t)
constexpr int kTileN1 = 128;         // SwiGLU output columns per gate/up tile (256 weight rows)
constexpr int kTileN2 = 256;         // output columns per down-GEMM tile
constexpr int kBlockK = 64;          // K elements per pipeline stage (one 128-byte swizzle row of bf16)
constexpr int kRowBytes = kBlockK * 2;
constexpr int kCombineTokens = 16;   // tokens per combine tile ...
constexpr int kCombineTokensSmall = 4;     // ... of an op with at most kCombineSmallBatch tokens (a decode batch): its
constexpr int kCombineSmallBatch = 1024;   // combine is a latency chain per token, so it is spread over more units
constexpr int kPlanChunk = 1024;     // fewest routed rows a block of the plan kernels owns
constexpr int kLagWork = 16;         // gate/up work tiles listed between an expert's gate/up tiles and its down tiles
constexpr int kWorkRowsBf16 = 256;   // rows of a work tile: two m-tiles share each weight tile
constexpr int kWorkRowsMid = 128;    // bf16 on CTA pairs: ops whose experts get at most so many rows (unless a token names an expert
constexpr int kWorkRowsSmall = 32;   // twice) leave shared memory for a deeper pipeline, see moe_run_pair.cu
constexpr int kWorkRowsFp8 = 128;    // fp8: the accumulator and both partial buffers fill TMEM
constexpr int kWorkRowsFp8Small = 64;   // fp8 ops of up to so many tokens: see the small tiles in moe_run.cu
constexpr int kMaxOps = 16;
constexpr int kMaxExperts = 1024;

// kGateUpDirect: a gate/up tile whose activation rows are consecutive rows of x (masked layout): they are
// loaded by TMA like the rows of a down tile instead of being gathered through a permutation
__host__ __device__ inline int combine_tile_tokens(int T) { return T <= kCombineSmallBatch ? kCombineTokensSmall : kCombineTokens; }

enum TileKind : int { kGateUp = 0, kDown = 1, kCombine = 2, kGateUpDirect = 3 };

// Queue entry (16 bytes, one load per claim): x = kind | n-tile << 4 | m-tile << 12,
// y = first packed row (first token for a combine tile), z = valid rows, w = expert (| kReadOnce: no other work tile of the op, or of the
// pair, reads its weights; not in bf16 plans for the single-CTA kernel).
constexpr int kReadOnce = 1 << 16;
// ... in a tile descriptor only: the tile and the next n-block run together, see moe_run_pair.cu
constexpr int kTwoTiles = 1 << 17;
// what a plan's list is made for: kReadOnce or 0, and whether a launch may hand its GEMM entries out in twos: two n-blocks of a work tile, which run
// together
struct ListForm {
  int read_once, twos;
};
__host__ __device__ inline int4 make_entry(int kind, int n, int m, int row0, int rows, int expert) {
  return make_int4(kind | (n << 4) | (m << 12), row0, rows, expert);
}
__host__ __device__ inline int entry_kind(const int4& e) { return e.x & 15; }
__host__ __device__ inline int entry_n(const int4& e) { return (e.x >> 4) & 0xff; }
__host__ __device__ inline int entry_m(const int4& e) { return (e.x >> 12) & 0xfffff; }

struct MTile {   // one row block of one expert (the unit counted by x_moe)
  int expert, row0, rows, pad;
};

// Written by the plan kernel, read by the run kernel.
struct PlanState {
  int n_mtiles;       // x_moe
  int n_gemm_tiles;   // queue entries of kind gate/up or down
  int n_comb_tiles;   // queue entries of kind combine (follow the GEMM entries)
  int planned;        // 1 after a moe_plan that accepted every expert id, else 0
  int n_extra_gemm;   // paired prefill op: GEMM entries of the decode op's list that carry rows of this op
  int work_rows;      // most rows of a GEMM entry
  int cls;            // of the op that was planned
  int flags;          // kOpFree, kOpWatched
};
constexpr int kOpFree = 1;      // it has no ready word and no predecessor
constexpr int kOpWatched = 2;   // somebody looks at its progress: it has a done or a notify word, or it is chained behind another op of the run

// Part of the run state, see RunHead.
struct RunState {
  int gemm_done;      // committed down tiles (CTA pairs: times the warps that store one)
  int tiles_done;     // committed tiles of any kind
  int done;           // 1 when the op has fully finished
  int pad;
};

struct Status;

struct __align__(128) OpDev {
  CUtensorMap tm_a8;    // [Rmax, I]   box {64, 8}   packed intermediate, 8 consecutive rows
  CUtensorMap tm_a32;   // [Rmax, I]   box {64, 32}
  CUtensorMap tm_w1;    // gate/up weights as [1][E][gate, up][I][H], box of 128 gate rows and the 128 matching up rows x 128 bytes
  CUtensorMap tm_w2;    // down weights as [1][E][H/128][128][I], box of 256 consecutive rows x 128 bytes
                        // (CTA pairs: views of tm_p1 and tm_p2 with boxes of 256 rows, where two tiles may run together)
  CUtensorMap tm_a128;  // [Rmax, I]   box {64, 128}
  CUtensorMap tm_a256;  // [Rmax, I]   box {64, 256} (as tm_x256 not for CTA pairs)
  CUtensorMap tm_p1;    // weights as the M operand: gate/up rows x 128 bytes, a box holds 64 gate rows and the matching up rows in
                        // groups of eight (bf16: [E][I/8][gate, up][8][H]), or 128 of each (e4m3: [8][2 E I][gate, up][8 every other][H])
  CUtensorMap tm_p2;    // ... down, as [E][H/16][2][8][I], box of 128 (e4m3: 256) consecutive rows x 128 bytes
  CUtensorMap tm_x8;    // masked layout only: x as [E*slab_rows, H], boxes of 8 / 32 / 128 / 256 rows
  CUtensorMap tm_x32;
  CUtensorMap tm_x128;
  CUtensorMap tm_x256;
  int cls, n_tokens, n_rows, after_op;
  const void* x;
  const float* x_scale;
  const int* topk_ids;
  const float* topk_w;
  const void* w_gate_up;
  const void* w_down;
  const float* s_gate_up;
  const float* s_down;
  void* y;
  int* counts;
  int* offsets;
  int* sorted_to_flat;
  int* flat_to_sorted;
  const unsigned* ready;
  unsigned* done;
  unsigned* notify;      // set once notify_after tiles of the op have committed
  int notify_after;
  int op_budget;         // > 0: written to the budget word when the op's first tile is claimed
  // workspace-owned
  __nv_bfloat16* A;      // [Rmax, I]  SwiGLU output, packed order (e4m3 bytes in the fp8 path)
  float* a_scale;        // [Rmax, I/128] fp32 scales of A (fp8 path)
  __nv_bfloat16* D;      // [Rmax, H]  expert output, packed order
  MTile* mtiles;         // [max_mtiles]
  int4* tile_list;       // [max_tiles] queue entries in claim order
  int* plan_hist;        // [n_chunks, E] rows per plan block and expert
  PlanState* plan;
  RunState* run;         // in the first half of the run state
  int* g1_done;          // [max_mtiles] committed gate/up tiles per work tile, counted like gemm_done (first half)
  Status* status;        // the context's device status block
  // Which list of routed rows the run kernels walk.  A plain op: its own permutation (the plan's public
  // outputs).  The paired form of a decode + prefill op that share their weights (moe_plan_pair): one row
  // space for both, every entry of the gather list tagged with the slot whose row it is.
  const int* gather_list;   // packed row -> flat routed index (paired: | slot << kRowSlotShift)
  const int* comb_index;    // flat routed index -> packed row of D
  int space_rows;           // rows of the packed space that A, D and comb_index refer to
  int masked;               // 1: masked layout (x, A, y in per-expert slabs of slab_rows rows)
  int paired;               // 1: this is the paired form of the slot
  int partner;              // paired: descriptor index of the other op of the pair, else -1
  int pad_[2];
};
constexpr int kRowSlotShift = 27;                       // a flat routed index stays below 2^27 (moe_create checks)
constexpr int kRowFlatMask = (1 << kRowSlotShift) - 1;

struct Status {   // first error wins (atomicCAS on code)
  int code;
  int detail[4];
  int abort;      // set with code; every CTA stops claiming when it sees it
  int pad[2];
};

struct Global {
  Status status;
  int budget;             // decode SM budget q (Section 6.4)
  unsigned turn;          // bit 31: which half of the run state the next launch works on; below: claiming units of the
                          // current launch that have asked
  int pad[6];
};

// The run state exists twice.  A launch works on one half, which is zero when it starts, and zeroes the other for the
// next one; the unit that is last to ask turns the halves over.  That keeps a memset (with its gaps 6 us of a 70 us decode pass)
// off the stream.
// Start of a half; the per-slot RunState blocks and g1_done arrays follow it.
struct RunHead {
  unsigned heads[2];      // next ticket of the decode / prefill queue
  unsigned log_count;
  int pad[5];
};

// the half that the last launch worked on
__host__ __device__ inline unsigned last_run_off(unsigned turn, unsigned run_bytes) { return (turn >> 31) ? 0u : run_bytes; }

struct RunArgs {
  Global* g;
  OpDev* ops;             // indexed by slot
  moe_tile_rec_t* log;
  int log_cap;
  int n_ops;
  int fuse_combine;
  int E, k, H, I;
  int dtype;              // MOE_DTYPE_*
  int kb_gate_up, kb_down;   // k-blocks (pipeline stages: 64 elements of K in bf16, 128 in e4m3) of a gate/up and a down tile
  long long wait_ns;
  unsigned run_bytes;     // size of one half of the run state
  int n_slots;            // slots of the context; descriptor d >= n_slots is the paired form of slot d - n_slots
  signed char desc[kMaxOps];   // slot -> the descriptor that stands for it in this launch
  int work_rows;          // rows of the largest work tile of the launch's ops
  int static_kind;        // -1: persistent launch served from the queues.  >= 0: a plain launch, claiming unit u
                          // of the grid runs queue entry u of slots[0] and ends
  int slots[kMaxOps];     // descriptor indices of the launch's ops, in the order given
  const PlanState* plan[kMaxOps];   // of slots[i], as tile_list: where a slot keeps them.  What depends on the op that is bound to a slot
                                    // is read there and in its descriptor: a captured launch may be replayed on another op
  const int4* tile_list[kMaxOps];
  signed char carrier[kMaxOps];     // paired prefill op: its decode op's place in `slots` (that op's tiles carry rows of it), else -1
};

// ------------------------------------------------------------------ launches that overlap the tail of the one before
// All kernels of the library are launched so that their blocks may become resident while the previous kernel of the stream
// still runs.  Each calls grid_dep_wait before it touches global memory, which returns when that kernel is complete and its writes
// are visible, and then lets the next one in.
__device__ __forceinline__ void grid_dep_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <class... Params, class... Args>
inline cudaError_t launch_after(void (*kernel)(Params...), int blocks, int threads, size_t smem, cudaStream_t stream, Args&&... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
}

__device__ __forceinline__ int slot_of(const RunArgs* a, int desc) { return desc >= a->n_slots ? desc - a->n_slots : desc; }

__device__ __noinline__ inline void report(Status* st, int code, int d0, int d1, int d2, int d3) {
  if (atomicCAS(&st->code, 0, code) == 0) {
    st->detail[0] = d0; st->detail[1] = d1; st->detail[2] = d2; st->detail[3] = d3;
  }
  __threadfence();
  atomicExch(&st->abort, 1);
}

__device__ inline unsigned long long gtime_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

}  // namespace moe
