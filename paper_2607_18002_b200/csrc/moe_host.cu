// Host side of the C ABI: argument validation, the layout of the caller's workspace,
// TMA descriptors, and the launches.  No hidden host synchronisation except where the
// header says so.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>

#include "moe_dev.cuh"

namespace moe {
cudaError_t launch_plan(const OpDev& h, int slot, int E, int NT1, int NT2, int work_rows, ListForm form, cudaStream_t stream);
cudaError_t launch_plan_masked(const OpDev& h, int slot, int E, int NT1, int NT2, int slab_rows, int work_rows,
                               ListForm form, cudaStream_t stream);
cudaError_t launch_plan_pair(const OpDev& hd, const OpDev& hp, const OpDev& d, const OpDev& p, int* gather, int* comb_d,
                             int* comb_p, int E, int NT1, int NT2, int work_rows, int carrier_rows, ListForm form,
                             int slot_d, int slot_p, cudaStream_t stream);
cudaError_t launch_combine(const OpDev* d_op, int T, int k, int H, cudaStream_t stream);
cudaError_t prepare_run_kernel();
cudaError_t launch_run(const RunArgs& args, RunHead* rh, int n_ctas, cudaStream_t stream);
cudaError_t prepare_pair_kernel();
cudaError_t prepare_plan_kernels();
cudaError_t launch_pair(const RunArgs& args, RunHead* rh, int n_ctas, bool dual, cudaStream_t stream);
}  // namespace moe

using namespace moe;

namespace {

constexpr int kDualRounds = 10, kDualRoundsFew = 5, kDualFewRows = 64, kDualBlocks = 8;        // see moe_run

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

struct Layout {
  size_t global_off, ops_off, run_off, run_bytes, log_off, slots_off, slot_stride;
  // inside a slot
  size_t A_off, D_off, mtiles_off, tiles_off, hist_off, plan_off;
  size_t ptiles_off, pgather_off, pcomb_off, pplan_off;   // paired form: queue list, shared-space permutation, plan state
  // inside a half of the run state (after RunHead)
  size_t rs_stride;      // RunState + g1_done[max_mtiles], per slot
  size_t total;
  int max_rows, max_mtiles, max_tiles, NT1, NT2;
};

int check_config(const moe_config_t* c) {
  if (!c) return MOE_EINVAL;
  if (c->n_experts < 1 || c->n_experts > kMaxExperts) return MOE_EINVAL;
  if (c->top_k < 1 || c->top_k > 32 || c->top_k > c->n_experts) return MOE_EINVAL;
  if (c->hidden < kTileN2 || c->hidden % kTileN2) return MOE_EINVAL;
  if (c->inter < kTileN1 || c->inter % kTileN1) return MOE_EINVAL;
  // a queue entry keeps its n-tile index in eight bits
  if (c->inter / kTileN1 > 255 || c->hidden / kTileN2 > 255) return MOE_EINVAL;
  if (c->dtype != MOE_DTYPE_BF16 && c->dtype != MOE_DTYPE_FP8_E4M3) return MOE_EINVAL;
  if (c->max_tokens_per_op < 1 || c->max_ops < 1 || c->max_ops > kMaxOps) return MOE_EINVAL;
  // a flat routed index must fit below bit kRowSlotShift (the paired form tags it with a slot above that)
  if ((long long)c->max_tokens_per_op * c->top_k >= (1ll << kRowSlotShift)) return MOE_EINVAL;
  // the combine addresses the rows of the down-GEMM output by 32-bit offsets in 16-byte units
  if ((long long)c->max_tokens_per_op * c->top_k * (c->hidden / 8) >= (1ll << 32)) return MOE_EINVAL;
  if (c->wait_limit_us < 0 || c->tile_log_entries < 0 || c->n_ctas < 0) return MOE_EINVAL;
  return MOE_OK;
}

Layout make_layout(const moe_config_t* c) {
  Layout L{};
  const size_t E = c->n_experts, H = c->hidden, I = c->inter;
  L.max_rows = c->max_tokens_per_op * c->top_k;
  // Work tiles of an op: at most one partly filled tile per expert besides the full ones.  An op of few tokens is cut into lower tiles,
  // and where its tokens name an expert more than once it has more of them than m-tiles.
  const int low = c->dtype == MOE_DTYPE_FP8_E4M3 ? kWorkRowsFp8Small : kWorkRowsSmall;
  const int low_rows = (c->max_tokens_per_op < low ? c->max_tokens_per_op : low) * c->top_k;
  const int full_tiles = (L.max_rows + kTileM - 1) / kTileM, low_tiles = (low_rows + low - 1) / low;
  L.max_mtiles = (full_tiles > low_tiles ? full_tiles : low_tiles) + c->n_experts;
  L.NT1 = (int)(I / kTileN1);
  L.NT2 = (int)(H / kTileN2);
  // combine entries of the largest op: small batches use smaller combine tiles
  const int small_t = c->max_tokens_per_op < kCombineSmallBatch ? c->max_tokens_per_op : kCombineSmallBatch;
  const int comb_small = (small_t + kCombineTokensSmall - 1) / kCombineTokensSmall;
  const int comb_large = (c->max_tokens_per_op + kCombineTokens - 1) / kCombineTokens;
  const int max_comb = comb_small > comb_large ? comb_small : comb_large;
  L.max_tiles = L.max_mtiles * (L.NT1 + L.NT2) + max_comb;
  const size_t n_chunks = ((size_t)L.max_rows + kPlanChunk - 1) / kPlanChunk;   // at most one histogram per chunk

  size_t off = 0;
  L.A_off = off;       off = align_up(off + (size_t)L.max_rows * I * 2, 1024);
  L.D_off = off;       off = align_up(off + (size_t)L.max_rows * H * 2, 1024);
  L.mtiles_off = off;  off = align_up(off + (size_t)L.max_mtiles * sizeof(MTile), 1024);
  L.tiles_off = off;   off = align_up(off + (size_t)L.max_tiles * sizeof(int4), 1024);
  L.hist_off = off;    off = align_up(off + n_chunks * E * 4, 1024);
  L.plan_off = off;    off = align_up(off + sizeof(PlanState), 1024);
  L.ptiles_off = off;  off = align_up(off + (size_t)L.max_tiles * sizeof(int4), 1024);
  L.pgather_off = off; off = align_up(off + (size_t)L.max_rows * 4, 1024);
  L.pcomb_off = off;   off = align_up(off + (size_t)L.max_rows * 4, 1024);
  L.pplan_off = off;   off = align_up(off + sizeof(PlanState), 1024);
  L.slot_stride = off;

  size_t g = 0;
  L.global_off = g;    g = align_up(g + sizeof(Global), 1024);
  L.ops_off = g;       g = align_up(g + sizeof(OpDev) * 2 * c->max_ops, 1024);   // plain and paired descriptors
  L.run_off = g;
  L.rs_stride = align_up(sizeof(RunState) + (size_t)L.max_mtiles * 4, 16);
  L.run_bytes = align_up(sizeof(RunHead) + L.rs_stride * c->max_ops, 1024);
  g += 2 * L.run_bytes;
  L.log_off = g;       g = align_up(g + (size_t)c->tile_log_entries * sizeof(moe_tile_rec_t), 1024);
  L.slots_off = g;
  L.total = g + L.slot_stride * c->max_ops;
  return L;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// When the device has a descriptor, and when it has to be sent again.  A plan in a stream capture always brings its descriptor along,
// so that a replay runs the op that was captured, whatever the slot has been bound to since; and a slot that has been in a capture
// may have been rebound by a replay, which the host does not see.
struct Upload {
  bool sent;                    // the host's copy is what the last upload carries
  bool captured;                // one of the uploads was captured
  unsigned long long capture;   // where the last upload is: a capture, 0: none
  bool there(unsigned long long cap) const { return sent && (cap ? capture == cap : !captured); }
  void now(unsigned long long cap) { sent = true; captured |= cap != 0; capture = cap; }
};

// the capture that is under way on a stream, 0: none
unsigned long long capture_of(cudaStream_t stream) {
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;
  if (cudaStreamGetCaptureInfo(stream, &status, &id) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return status == cudaStreamCaptureStatusActive ? id | 1ull << 63 : 0;
}

}  // namespace

struct moe_ctx {
  moe_config_t cfg;
  Layout L;
  unsigned char* ws;
  int n_ctas, sm_count;
  bool pair_kernel;             // bf16 on an even grid: tiles run on CTA pairs (cta_group::2)
  bool poison;                  // debug: the scratch of every op of a launch is filled with NaN patterns first
  EncodeTiledFn encode;
  moe_op_t ops[kMaxOps];
  bool planned[kMaxOps];
  OpDev host_ops[kMaxOps];      // what the device copy of each slot holds (tensor maps included)
  OpDev host_pair[kMaxOps];     // what the device copy of each slot's paired descriptor holds
  Upload up[kMaxOps], pair_up[kMaxOps];
  int pair_of[kMaxOps];         // slot paired with this one by moe_plan_pair since both were last planned, or -1
  int work_rows[kMaxOps];       // rows of a work tile of the slot's plan
  unsigned long long plan_capture[kMaxOps];   // the stream capture that plan was issued in, 0: none
  bool ran_paired[kMaxOps];     // the slot's last moe_run used its paired form (moe_combine follows it)
  Global* g() const { return reinterpret_cast<Global*>(ws + L.global_off); }
  RunHead* rh() const { return reinterpret_cast<RunHead*>(ws + L.run_off); }
  unsigned char* slot_base(int s) const { return ws + L.slots_off + L.slot_stride * s; }
  OpDev* op_dev(int s) const { return reinterpret_cast<OpDev*>(ws + L.ops_off) + s; }
  unsigned char* rs_base(int s) const { return ws + L.run_off + sizeof(RunHead) + L.rs_stride * s; }
};

namespace {

// 2-D tensor map (bf16, or e4m3 bytes): `rows` x `cols` row-major, box = box_rows x kBlockK columns, swizzle
// as wide as a box row
int make_map(moe_ctx* ctx, CUtensorMap* out, const void* base, size_t rows, size_t cols,
             int box_rows) {
  const bool fp8 = ctx->cfg.dtype == MOE_DTYPE_FP8_E4M3;
  const size_t el = fp8 ? 1 : 2;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * el};
  cuuint32_t box[2] = {(cuuint32_t)(kRowBytes / el), (cuuint32_t)box_rows};   // 128 bytes per box row
  cuuint32_t estr[2] = {1, 1};
  CUresult r = ctx->encode(out, fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                           const_cast<void*>(base), dims,
                           strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           kRowBytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? MOE_OK : MOE_ECUDA;
}

// The weights of one GEMM: a 5-D view whose box is the 128 or 256 rows x 128 bytes of a stage in one copy.
// rows: what one step of dimensions 1..4 moves by, in weight rows.
int make_map_m(moe_ctx* ctx, CUtensorMap* out, const void* base, size_t cols, const size_t (&size)[4], const size_t (&rows)[4],
                  const cuuint32_t (&boxes)[4]) {
  const bool fp8 = ctx->cfg.dtype == MOE_DTYPE_FP8_E4M3;
  const size_t el = fp8 ? 1 : 2;
  cuuint64_t dims[5], strides[4];
  cuuint32_t box[5], estr[5] = {1, 1, 1, 1, 1};
  dims[0] = cols;
  box[0] = (cuuint32_t)(kRowBytes / el);
  for (int i = 0; i < 4; ++i) {
    dims[i + 1] = size[i];
    strides[i] = rows[i] * cols * el;
    box[i + 1] = boxes[i];
  }
  CUresult r = ctx->encode(out, fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base),
                           dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? MOE_OK : MOE_ECUDA;
}

// a stream-ordered 4-byte write: the value travels in the launch, not through host memory
__global__ void set_word_kernel(int* p, int v) {
  grid_dep_wait();
  *reinterpret_cast<volatile int*>(p) = v;
}

// the tile log of a run without tiles: no records (the ones of the run before are in the half that it worked on)
__global__ void empty_log_kernel(const Global* g, RunHead* first_half, unsigned run_bytes) {
  grid_dep_wait();
  reinterpret_cast<RunHead*>(reinterpret_cast<char*>(first_half) + last_run_off(g->turn, run_bytes))->log_count = 0;
}

// The op descriptor travels as a kernel parameter (no pageable-memory copy on the stream).
__global__ void write_op_kernel(const __grid_constant__ OpDev src, OpDev* dst) {
  grid_dep_wait();
  const int n = (int)(sizeof(OpDev) / sizeof(int));
  const int* s = reinterpret_cast<const int*>(&src);
  int* d = reinterpret_cast<int*>(dst);
  for (int i = threadIdx.x; i < n; i += blockDim.x) d[i] = s[i];
}

// Whether launches may run two neighbouring n-blocks at a time.  Only where both GEMMs have an even number of them: every expert's entries then
// start at an even place of the list and each ticket holds two that run together.  (In twos by place alone, most tickets of a layer
// with odd numbers held two that do not, which then ran singly in the stages made for two, the second without a look at the budget: us a
// pass, 4096 tokens on 64 experts: 13 and 13 n-blocks 1193 that way, 1176 tile by tile; 13 and 12 1092 / 1060, 12 and 13 1107 / 1068.)
bool may_run_twos(const moe_ctx* ctx) { return ctx->pair_kernel && ctx->L.NT1 % 2 == 0 && ctx->L.NT2 % 2 == 0; }
ListForm list_form(const moe_ctx* ctx) {
  return ListForm{ctx->pair_kernel || ctx->cfg.dtype == MOE_DTYPE_FP8_E4M3 ? kReadOnce : 0, may_run_twos(ctx) ? 1 : 0};
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

}  // namespace

extern "C" {

const char* moe_strerror(int code) {
  switch (code) {
    case MOE_OK: return "ok";
    case MOE_EINVAL: return "invalid argument";
    case MOE_ENOSPC: return "workspace or slot capacity too small";
    case MOE_ECUDA: return "CUDA call failed (is there a device?)";
    case MOE_ETIMEOUT: return "a device-side wait ran out";
    case MOE_EBADID: return "expert id out of range";
    case MOE_EBOUNDS: return "device-side index check failed";
    case MOE_ENOTPLANNED: return "slot has no plan";
    default: return "unknown error";
  }
}

int moe_workspace_bytes(const moe_config_t* cfg, size_t* out) {
  if (!out) return MOE_EINVAL;
  const int rc = check_config(cfg);
  if (rc) return rc;
  *out = make_layout(cfg).total;
  return MOE_OK;
}

int moe_create(const moe_config_t* cfg, void* dev_workspace, size_t bytes, moe_ctx_t** out) {
  if (!out || !dev_workspace) return MOE_EINVAL;
  int rc = check_config(cfg);
  if (rc) return rc;
  if (reinterpret_cast<uintptr_t>(dev_workspace) & 1023) return MOE_EINVAL;
  Layout L = make_layout(cfg);
  if (bytes < L.total) return MOE_ENOSPC;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return MOE_ECUDA;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return MOE_ECUDA;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess ||
      qres != cudaDriverEntryPointSuccess || !fn)
    return MOE_ECUDA;
  if (prepare_run_kernel() != cudaSuccess || prepare_pair_kernel() != cudaSuccess ||
      prepare_plan_kernels() != cudaSuccess)
    return MOE_ECUDA;
  moe_ctx* ctx = new (std::nothrow) moe_ctx();
  if (!ctx) return MOE_ENOSPC;
  ctx->cfg = *cfg;
  if (ctx->cfg.wait_limit_us == 0) ctx->cfg.wait_limit_us = 2000000;
  ctx->L = L;
  ctx->ws = static_cast<unsigned char*>(dev_workspace);
  ctx->sm_count = sms;
  ctx->n_ctas = cfg->n_ctas > 0 ? cfg->n_ctas : sms;
  // MOE_APK_SINGLE_CTA=1 in the environment keeps bf16 on the one-CTA-per-tile kernel (for comparisons)
  const char* single = getenv("MOE_APK_SINGLE_CTA");
  ctx->pair_kernel = cfg->dtype == MOE_DTYPE_BF16 && ctx->n_ctas >= 2 && ctx->n_ctas % 2 == 0 &&
                     !(single && single[0] == '1');
  // MOE_APK_POISON=1: a row of the intermediate or of the expert output that a launch fails to write then shows
  // as NaN in y instead of passing for whatever the previous launch left there
  const char* poison = getenv("MOE_APK_POISON");
  ctx->poison = poison && poison[0] == '1';
  ctx->encode = reinterpret_cast<EncodeTiledFn>(fn);
  memset(ctx->planned, 0, sizeof(ctx->planned));
  memset(ctx->up, 0, sizeof(ctx->up));
  memset(ctx->pair_up, 0, sizeof(ctx->pair_up));
  memset(ctx->plan_capture, 0, sizeof(ctx->plan_capture));
  memset(ctx->ran_paired, 0, sizeof(ctx->ran_paired));
  for (int s = 0; s < kMaxOps; ++s) ctx->pair_of[s] = -1;
  // zero the control blocks (status, budget, run state, plan states)
  cudaError_t e = cudaMemset(ctx->ws, 0, L.slots_off);
  for (int s = 0; s < cfg->max_ops && e == cudaSuccess; ++s) {
    e = cudaMemset(ctx->slot_base(s) + L.plan_off, 0, sizeof(PlanState));
    if (e == cudaSuccess) e = cudaMemset(ctx->slot_base(s) + L.pplan_off, 0, sizeof(PlanState));
  }
  // A plan that was captured and not replayed yet counts as issued: a launch on its slot has to find a descriptor, of an op without tiles.
  OpDev* first = e == cudaSuccess ? new (std::nothrow) OpDev[2 * cfg->max_ops]() : nullptr;
  for (int d = 0; d < 2 * cfg->max_ops && first; ++d) {
    const int s = d % cfg->max_ops;
    OpDev& h = first[d];
    h.after_op = h.partner = -1;
    h.plan = reinterpret_cast<PlanState*>(ctx->slot_base(s) + (d < cfg->max_ops ? L.plan_off : L.pplan_off));
    h.run = reinterpret_cast<RunState*>(ctx->rs_base(s));
    h.g1_done = reinterpret_cast<int*>(ctx->rs_base(s) + sizeof(RunState));
    h.status = &ctx->g()->status;
  }
  if (e == cudaSuccess && !first) { delete ctx; return MOE_ENOSPC; }
  if (e == cudaSuccess) e = cudaMemcpy(ctx->op_dev(0), first, sizeof(OpDev) * 2 * cfg->max_ops, cudaMemcpyHostToDevice);
  delete[] first;
  if (e != cudaSuccess) { delete ctx; return MOE_ECUDA; }
  *out = ctx;
  return MOE_OK;
}

void moe_destroy(moe_ctx_t* ctx) { delete ctx; }

int moe_sm_count(moe_ctx_t* ctx) { return ctx ? ctx->sm_count : MOE_EINVAL; }
int moe_ctas_per_tile(moe_ctx_t* ctx) { return ctx ? (ctx->pair_kernel ? 2 : 1) : MOE_EINVAL; }

int moe_plan(moe_ctx_t* ctx, int slot, const moe_op_t* op, void* stream) {
  if (!ctx || !op) return MOE_EINVAL;
  const moe_config_t& c = ctx->cfg;
  if (slot < 0 || slot >= c.max_ops) return MOE_EINVAL;
  if (op->cls != MOE_CLASS_DECODE && op->cls != MOE_CLASS_PREFILL) return MOE_EINVAL;
  const bool masked = op->layout == MOE_LAYOUT_MASKED;
  if (op->layout != MOE_LAYOUT_GATHERED && !masked) return MOE_EINVAL;
  if (op->n_tokens < 0) return MOE_EINVAL;
  if (!masked && op->n_tokens > c.max_tokens_per_op) return MOE_ENOSPC;
  if (op->after_op < -1 || op->after_op >= c.max_ops || op->after_op == slot) return MOE_EINVAL;
  if (op->notify && op->notify_after < 1) return MOE_EINVAL;
  if (op->decode_sms < 0) return MOE_EINVAL;
  if (!op->counts || !op->offsets) return MOE_EINVAL;
  if (!op->w_gate_up || !op->w_down || !aligned16(op->w_gate_up) || !aligned16(op->w_down)) return MOE_EINVAL;
  if (c.dtype == MOE_DTYPE_FP8_E4M3 && (!op->s_gate_up || !op->s_down || ((op->n_tokens > 0 || masked) && !op->x_scale)))
    return MOE_EINVAL;
  if (masked) {
    if (op->slab_rows < 1 || !op->x || !op->y || !aligned16(op->x) || !aligned16(op->y)) return MOE_EINVAL;
    // the slabs of the intermediate live in the slot's scratch, one row per slab row
    if ((long long)c.n_experts * op->slab_rows > (long long)c.max_tokens_per_op * c.top_k) return MOE_ENOSPC;
  } else if (op->n_tokens > 0) {
    if (!op->x || !op->topk_ids || !op->topk_w || !op->y || !op->sorted_to_flat || !op->flat_to_sorted)
      return MOE_EINVAL;
    if (!aligned16(op->x) || !aligned16(op->y)) return MOE_EINVAL;
  }
  const Layout& L = ctx->L;
  unsigned char* sb = ctx->slot_base(slot);
  OpDev h;
  memset(&h, 0, sizeof(h));
  h.cls = op->cls;
  h.n_tokens = masked ? 0 : op->n_tokens;                     // a masked op has no token-order output to combine
  h.n_rows = masked ? c.n_experts * op->slab_rows : op->n_tokens * c.top_k;
  h.after_op = op->after_op;
  h.x = op->x; h.x_scale = op->x_scale; h.topk_ids = op->topk_ids; h.topk_w = op->topk_w;
  h.w_gate_up = op->w_gate_up; h.w_down = op->w_down; h.s_gate_up = op->s_gate_up; h.s_down = op->s_down;
  h.y = op->y; h.counts = op->counts; h.offsets = op->offsets;
  h.sorted_to_flat = op->sorted_to_flat; h.flat_to_sorted = op->flat_to_sorted;
  h.ready = op->ready; h.done = op->done;
  h.notify = op->notify; h.notify_after = op->notify_after;
  h.op_budget = op->decode_sms;
  h.A = reinterpret_cast<__nv_bfloat16*>(sb + L.A_off);
  h.a_scale = reinterpret_cast<float*>(sb + L.A_off + align_up((size_t)L.max_rows * c.inter, 16));
  // masked layout: the expert outputs ARE the op's output, in the slab layout of x
  h.D = masked ? static_cast<__nv_bfloat16*>(op->y) : reinterpret_cast<__nv_bfloat16*>(sb + L.D_off);
  h.masked = masked ? 1 : 0;
  h.mtiles = reinterpret_cast<MTile*>(sb + L.mtiles_off);
  h.tile_list = reinterpret_cast<int4*>(sb + L.tiles_off);
  h.plan_hist = reinterpret_cast<int*>(sb + L.hist_off);
  h.plan = reinterpret_cast<PlanState*>(sb + L.plan_off);
  h.run = reinterpret_cast<RunState*>(ctx->rs_base(slot));
  h.g1_done = reinterpret_cast<int*>(ctx->rs_base(slot) + sizeof(RunState));
  h.status = &ctx->g()->status;
  h.gather_list = op->sorted_to_flat;
  h.comb_index = op->flat_to_sorted;
  h.space_rows = h.n_rows;
  h.paired = 0;
  h.partner = -1;
  // a new plan for the slot ends any pairing it was part of
  if (ctx->pair_of[slot] >= 0) ctx->pair_of[ctx->pair_of[slot]] = -1;
  ctx->pair_of[slot] = -1;
  ctx->ran_paired[slot] = false;
  // Re-planning a slot with the same buffers (the usual serving loop) reuses the descriptors
  // already on the device: encoding its tensor maps and uploading them is host time.
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const unsigned long long cap = capture_of(st);
  const bool same = ctx->up[slot].sent && memcmp(&ctx->ops[slot], op, sizeof(moe_op_t)) == 0;
  if (!same || !ctx->up[slot].there(cap)) {
    int rc = MOE_OK;
    if (same) {
      h = ctx->host_ops[slot];
    } else if (op->n_tokens > 0 || masked) {
      rc = make_map(ctx, &h.tm_a8, h.A, (size_t)L.max_rows, (size_t)c.inter, 8);
      if (!rc) rc = make_map(ctx, &h.tm_a32, h.A, (size_t)L.max_rows, (size_t)c.inter, 32);
      if (!rc) rc = make_map(ctx, &h.tm_a128, h.A, (size_t)L.max_rows, (size_t)c.inter, 128);
      if (!rc && !ctx->pair_kernel) rc = make_map(ctx, &h.tm_a256, h.A, (size_t)L.max_rows, (size_t)c.inter, 256);
      const size_t E = c.n_experts, H = c.hidden, I = c.inter;
      const bool fp8 = c.dtype == MOE_DTYPE_FP8_E4M3;
      if (!rc && ctx->pair_kernel)                 // 8 gate rows, the 8 matching up rows, the next 8 gate rows, ...
        rc = make_map_m(ctx, &h.tm_p1, op->w_gate_up, H, {8, 2, I / 8, E}, {1, I, 8, 2 * I}, {8, 2, 8, 1});
      if (!rc && may_run_twos(ctx))                // ... two n-blocks' rows at once
        rc = make_map_m(ctx, &h.tm_w1, op->w_gate_up, H, {8, 2, I / 8, E}, {1, I, 8, 2 * I}, {8, 2, 16, 1});
      if (!rc && may_run_twos(ctx))
        rc = make_map_m(ctx, &h.tm_w2, op->w_down, I, {8, 2, H / 16, E}, {1, 8, 16, H}, {8, 2, 16, 1});
      if (!rc && fp8)                              // ... of 16 rows: 8 even gate, 8 even up, 8 odd gate, 8 odd up rows
        rc = make_map_m(ctx, &h.tm_p1, op->w_gate_up, H, {8, 2, 2 * E * I, 8}, {2, I, 1, 16}, {8, 2, 2, 8});
      if (!rc && (ctx->pair_kernel || fp8))
        rc = make_map_m(ctx, &h.tm_p2, op->w_down, I, {8, 2, H / 16, E}, {1, 8, 16, H}, {8, 2, fp8 ? 16u : 8u, 1});
      if (!ctx->pair_kernel) {
        if (!rc) rc = make_map_m(ctx, &h.tm_w1, op->w_gate_up, H, {I, 2, E, 1}, {1, I, 2 * I, 2 * I}, {128, 2, 1, 1});
        if (!rc) rc = make_map_m(ctx, &h.tm_w2, op->w_down, I, {128, H / 128, E, 1}, {1, 128, H, H}, {128, 2, 1, 1});
      }
      if (masked) {
        const size_t xr = (size_t)c.n_experts * op->slab_rows;
        if (!rc) rc = make_map(ctx, &h.tm_x8, op->x, xr, (size_t)c.hidden, 8);
        if (!rc) rc = make_map(ctx, &h.tm_x32, op->x, xr, (size_t)c.hidden, 32);
        if (!rc) rc = make_map(ctx, &h.tm_x128, op->x, xr, (size_t)c.hidden, 128);
        if (!rc && !ctx->pair_kernel) rc = make_map(ctx, &h.tm_x256, op->x, xr, (size_t)c.hidden, 256);
      }
      if (rc) return rc;
    }
    ctx->planned[slot] = false;
    if (launch_after(write_op_kernel, 1, 128, 0, st, h, ctx->op_dev(slot)) != cudaSuccess) { ctx->up[slot].sent = false; return MOE_ECUDA; }
    ctx->host_ops[slot] = h;
    ctx->ops[slot] = *op;             // what the device copy of the slot now describes
    ctx->up[slot].now(cap);
  }
  int work_rows = c.dtype == MOE_DTYPE_FP8_E4M3 ? kWorkRowsFp8 : kWorkRowsBf16;
  const int most = masked ? op->slab_rows : op->n_tokens;       // rows an expert gets unless a token names it twice
  if (c.dtype == MOE_DTYPE_FP8_E4M3) {
    if (most <= kWorkRowsFp8Small) work_rows = kWorkRowsFp8Small;
  } else if (ctx->pair_kernel) {
    work_rows = most <= kWorkRowsSmall ? kWorkRowsSmall : most <= kWorkRowsMid ? kWorkRowsMid : kWorkRowsBf16;
  }
  ctx->work_rows[slot] = work_rows;
  ctx->plan_capture[slot] = cap;
  const ListForm form = list_form(ctx);
  const cudaError_t pe = masked ? launch_plan_masked(h, slot, c.n_experts, L.NT1, L.NT2, op->slab_rows, work_rows, form, st)
                                : launch_plan(h, slot, c.n_experts, L.NT1, L.NT2, work_rows, form, st);
  if (pe != cudaSuccess) {
    ctx->planned[slot] = false;
    return MOE_ECUDA;
  }
  ctx->planned[slot] = true;
  return MOE_OK;
}

int moe_run(moe_ctx_t* ctx, const int32_t* slots, int n_ops, int fuse_combine, void* stream) {
  if (!ctx || !slots || n_ops < 1 || n_ops > ctx->cfg.max_ops) return MOE_EINVAL;
  const moe_config_t& c = ctx->cfg;
  RunArgs a;
  memset(&a, 0, sizeof(a));
  for (int i = 0; i < n_ops; ++i) {
    const int s = slots[i];
    if (s < 0 || s >= c.max_ops) return MOE_EINVAL;
    if (!ctx->planned[s]) return MOE_ENOTPLANNED;
    for (int j = 0; j < i; ++j) if (slots[j] == s) return MOE_EINVAL;
    a.slots[i] = s;
  }
  // a slot whose pair partner is in the same launch runs in its paired form
  a.n_slots = c.max_ops;
  for (int s = 0; s < kMaxOps; ++s) a.desc[s] = (signed char)s;
  for (int i = 0; i < n_ops; ++i) {
    const int s = slots[i], q = ctx->pair_of[s];
    bool both = false;
    for (int j = 0; j < n_ops && q >= 0; ++j) both |= slots[j] == q;
    ctx->ran_paired[s] = both;
    if (both) {
      a.slots[i] = c.max_ops + s;
      a.desc[s] = (signed char)(c.max_ops + s);
    }
  }
  for (int i = 0; i < n_ops; ++i) {      // after_op must name an op of this run
    const int dep = ctx->ops[slots[i]].after_op;
    if (dep < 0) continue;
    bool found = false;
    for (int j = 0; j < n_ops; ++j) found |= slots[j] == dep;
    if (!found) return MOE_EINVAL;
  }
  a.g = ctx->g();
  a.ops = ctx->op_dev(0);
  a.log = reinterpret_cast<moe_tile_rec_t*>(ctx->ws + ctx->L.log_off);
  a.log_cap = c.tile_log_entries;
  a.n_ops = n_ops;
  a.fuse_combine = fuse_combine ? 1 : 0;
  a.E = c.n_experts; a.k = c.top_k; a.H = c.hidden; a.I = c.inter;
  a.dtype = c.dtype;
  const int kb_elems = c.dtype == MOE_DTYPE_FP8_E4M3 ? 128 : kBlockK;
  a.kb_gate_up = c.hidden / kb_elems;
  a.kb_down = c.inter / kb_elems;
  a.wait_ns = (long long)c.wait_limit_us * 1000;
  a.static_kind = -1;
  a.run_bytes = (unsigned)ctx->L.run_bytes;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const unsigned long long cap = capture_of(st);
  const int full = c.dtype == MOE_DTYPE_FP8_E4M3 ? kWorkRowsFp8 : kWorkRowsBf16;
  long long routed = 0;                  // rows of the launch's ops
  for (int i = 0; i < n_ops; ++i) {
    const OpDev& h = ctx->ran_paired[slots[i]] ? ctx->host_pair[slots[i]] : ctx->host_ops[slots[i]];
    a.plan[i] = h.plan;
    a.tile_list[i] = h.tile_list;
    a.carrier[i] = -1;
    if (ctx->ran_paired[slots[i]] && h.cls == MOE_CLASS_PREFILL)
      for (int j = 0; j < n_ops; ++j)
        if (slots[j] == ctx->pair_of[slots[i]]) a.carrier[i] = (signed char)j;
    // The kernels for small ops have room for small work tiles only.  Plan and launch captured together are replayed together; a launch
    // captured by itself runs whatever the slot has been planned for by then.
    const bool any_plan = ctx->ran_paired[slots[i]] || ctx->plan_capture[slots[i]] != cap;
    const int rows = any_plan ? full : ctx->work_rows[slots[i]];
    a.work_rows = rows > a.work_rows ? rows : a.work_rows;
    if (ctx->ops[slots[i]].layout != MOE_LAYOUT_MASKED) routed += (long long)ctx->ops[slots[i]].n_tokens * c.top_k;
  }
  if (ctx->poison) {
    for (int i = 0; i < n_ops; ++i) {
      unsigned char* sb = ctx->slot_base(slots[i]);
      const size_t a_bytes = ctx->L.D_off - ctx->L.A_off, d_bytes = ctx->L.mtiles_off - ctx->L.D_off;
      if (cudaMemsetAsync(sb + ctx->L.A_off, 0xff, a_bytes, st) != cudaSuccess) return MOE_ECUDA;
      if (cudaMemsetAsync(sb + ctx->L.D_off, 0xff, d_bytes, st) != cudaSuccess) return MOE_ECUDA;
    }
  }
  // Two tiles at a time (see moe_run_pair.cu) pay where there are enough of them for the units to share out and where their k-blocks outlast
  // the stores that nothing overlaps.  What is known here are the rows: a lower bound of the tiles, counted below in rounds of the units.
  // With few rounds the longer tickets leave units idle at the end.  us a pass, one by one / two at a time (rounds):
  //   48 and 24 k-blocks a tile, 8 experts: 500 tokens 130 / 141 (4.9), 800 214 / 219 (8.1), 1200 274 / 277 (12); 16 experts: 400 145 / 149 (3.9),
  //   700 203 / 213 (6.8); 32: 600 241 / 249 (5.8), 1000 309 / 310 (10); 256: 8192 2458 / 2389 (83);
  //   32 and 16, 32 experts: 700 137 / 146 (4.5), 1000 168 / 171 (6.7), 1500 214 / 212 (10); 64: 500 173 / 175 (3.2), 1000 220 / 222 (6.7);
  //   16 and 8, 32 experts: 2400 83 / 88 (4.0), 4000 112 / 117 (6.7), 6000 144 / 142 (10), 12 000 256 / 249 (20).
  // Where experts get few rows most tiles are short ones that the bound does not count, and two at a time pay earlier:
  //   48 and 24: 777 tokens on 256 experts 1181 / 1159 (7.8), 600 on 128 632 / 626 (5.8); 16 and 8: 1500 on 128 142 / 141 (5.0); but 32 and 16: 700
  //   on 128 315 / 320 (4.5).  Between three and five rounds it depends on how many experts the tokens choose, which is not known here: 400 tokens, 16
  //   of 256 experts 134 / 144, 32 of them 203 / 206, 96 472 / 473, 192 883 / 876, all 1112 / 1105.  8 or more k-blocks: 5000 tokens on 8 experts with 4 and 8 of them take 61 / 65.
  const long long rounds = routed <= (long long)kDualFewRows * c.n_experts ? kDualRoundsFew : kDualRounds;
  const bool dual = may_run_twos(ctx) && routed / kWorkRowsBf16 * (ctx->L.NT1 + ctx->L.NT2) >= rounds * (ctx->n_ctas / 2) &&
                    a.kb_gate_up >= kDualBlocks && a.kb_down >= kDualBlocks;
  const cudaError_t le = ctx->pair_kernel ? launch_pair(a, ctx->rh(), ctx->n_ctas, dual, st)
                                          : launch_run(a, ctx->rh(), ctx->n_ctas, st);
  if (le != cudaSuccess) return MOE_ECUDA;
  return MOE_OK;
}

int moe_run_plain(moe_ctx_t* ctx, int slot, void* stream) {
  if (!ctx || slot < 0 || slot >= ctx->cfg.max_ops) return MOE_EINVAL;
  if (!ctx->pair_kernel) return MOE_EINVAL;
  if (!ctx->planned[slot]) return MOE_ENOTPLANNED;
  if (ctx->ops[slot].after_op >= 0 || ctx->ops[slot].ready) return MOE_EINVAL;
  const moe_config_t& c = ctx->cfg;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // the grid is the op's entry count, which only the device knows: wait for the plan and read it
  PlanState ps;
  if (cudaStreamSynchronize(st) != cudaSuccess) return MOE_ECUDA;
  if (cudaMemcpy(&ps, ctx->slot_base(slot) + ctx->L.plan_off, sizeof(ps), cudaMemcpyDeviceToHost) != cudaSuccess)
    return MOE_ECUDA;
  if (!ps.planned) return MOE_ENOTPLANNED;
  RunArgs a;
  memset(&a, 0, sizeof(a));
  a.slots[0] = slot;
  a.g = ctx->g();
  a.ops = ctx->op_dev(0);
  a.log = reinterpret_cast<moe_tile_rec_t*>(ctx->ws + ctx->L.log_off);
  a.log_cap = c.tile_log_entries;
  a.n_ops = 1;
  a.fuse_combine = 0;
  a.E = c.n_experts; a.k = c.top_k; a.H = c.hidden; a.I = c.inter;
  a.dtype = c.dtype;
  a.kb_gate_up = c.hidden / kBlockK;
  a.kb_down = c.inter / kBlockK;
  a.wait_ns = (long long)c.wait_limit_us * 1000;
  a.n_slots = c.max_ops;
  for (int s = 0; s < kMaxOps; ++s) a.desc[s] = (signed char)s;
  ctx->ran_paired[slot] = false;
  a.static_kind = 0;
  a.run_bytes = (unsigned)ctx->L.run_bytes;
  a.plan[0] = ctx->host_ops[slot].plan;
  a.tile_list[0] = ctx->host_ops[slot].tile_list;
  a.carrier[0] = -1;
  a.work_rows = ps.work_rows;
  if (ps.n_gemm_tiles > 0) {
    if (launch_pair(a, ctx->rh(), 2 * ps.n_gemm_tiles, false, st) != cudaSuccess) return MOE_ECUDA;
  } else if (launch_after(empty_log_kernel, 1, 1, 0, st, ctx->g(), ctx->rh(), (unsigned)ctx->L.run_bytes) != cudaSuccess) {
    return MOE_ECUDA;
  }
  if (ctx->ops[slot].layout == MOE_LAYOUT_GATHERED &&
      launch_combine(ctx->op_dev(slot), ctx->ops[slot].n_tokens, c.top_k, c.hidden, st) != cudaSuccess)
    return MOE_ECUDA;
  return MOE_OK;
}

int moe_combine(moe_ctx_t* ctx, int slot, void* stream) {
  if (!ctx || slot < 0 || slot >= ctx->cfg.max_ops) return MOE_EINVAL;
  if (!ctx->planned[slot]) return MOE_ENOTPLANNED;
  if (ctx->ops[slot].layout != MOE_LAYOUT_GATHERED) return MOE_EINVAL;     // a masked op has nothing to combine
  // after a launch that ran the slot in its paired form, the expert outputs lie in the pair's shared row space
  const int desc = ctx->ran_paired[slot] ? ctx->cfg.max_ops + slot : slot;
  if (launch_combine(ctx->op_dev(desc), ctx->ops[slot].n_tokens, ctx->cfg.top_k, ctx->cfg.hidden,
                     static_cast<cudaStream_t>(stream)) != cudaSuccess)
    return MOE_ECUDA;
  return MOE_OK;
}

int moe_plan_pair(moe_ctx_t* ctx, int slot_prefill, int slot_decode, int carrier_rows, void* stream) {
  if (!ctx) return MOE_EINVAL;
  const moe_config_t& c = ctx->cfg;
  const int sp = slot_prefill, sd = slot_decode;
  if (sp < 0 || sp >= c.max_ops || sd < 0 || sd >= c.max_ops || sp == sd) return MOE_EINVAL;
  if (!ctx->planned[sp] || !ctx->planned[sd]) return MOE_ENOTPLANNED;
  const moe_op_t &op = ctx->ops[sp], &od = ctx->ops[sd];
  if (op.cls != MOE_CLASS_PREFILL || od.cls != MOE_CLASS_DECODE) return MOE_EINVAL;
  if (op.layout != MOE_LAYOUT_GATHERED || od.layout != MOE_LAYOUT_GATHERED) return MOE_EINVAL;
  // one weight tile can only serve rows of both ops if both ops read the same weights
  if (op.w_gate_up != od.w_gate_up || op.w_down != od.w_down || op.s_gate_up != od.s_gate_up || op.s_down != od.s_down)
    return MOE_EINVAL;
  const bool fp8 = c.dtype == MOE_DTYPE_FP8_E4M3;
  if (carrier_rows == 0) carrier_rows = fp8 ? kWorkRowsFp8 : kWorkRowsBf16;
  if (carrier_rows != 128 && carrier_rows != 256) return MOE_EINVAL;
  const Layout& L = ctx->L;
  const long long Rp = (long long)op.n_tokens * c.top_k, Rd = (long long)od.n_tokens * c.top_k;
  if (Rp + Rd > L.max_rows) return MOE_ENOSPC;      // the shared row space lives in one slot's scratch
  if (op.n_tokens == 0 || od.n_tokens == 0) return MOE_EINVAL;
  unsigned char *bp = ctx->slot_base(sp), *bd = ctx->slot_base(sd);
  int* gather_m = reinterpret_cast<int*>(bp + L.pgather_off);
  OpDev hp = ctx->host_ops[sp], hd = ctx->host_ops[sd];
  // both paired descriptors address the prefill slot's scratch (A, its scales, D) as the shared row space
  hd.A = hp.A; hd.a_scale = hp.a_scale; hd.D = hp.D;
  hd.tm_a8 = hp.tm_a8; hd.tm_a32 = hp.tm_a32; hd.tm_a128 = hp.tm_a128; hd.tm_a256 = hp.tm_a256;
  OpDev* both[2] = {&hp, &hd};
  for (int i = 0; i < 2; ++i) {
    OpDev* h = both[i];
    unsigned char* b = i == 0 ? bp : bd;
    h->tile_list = reinterpret_cast<int4*>(b + L.ptiles_off);
    h->plan = reinterpret_cast<PlanState*>(b + L.pplan_off);
    h->gather_list = gather_m;
    h->comb_index = reinterpret_cast<int*>(b + L.pcomb_off);
    h->space_rows = (int)(Rp + Rd);
    h->paired = 1;
    h->partner = c.max_ops + (i == 0 ? sd : sp);
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const unsigned long long cap = capture_of(st);
  // the usual loop pairs the same two ops on the same buffers again and again: upload only what changed
  const int which[2] = {sp, sd};
  for (int i = 0; i < 2; ++i) {
    const int s = which[i];
    if (ctx->pair_up[s].there(cap) && memcmp(&ctx->host_pair[s], both[i], sizeof(OpDev)) == 0) continue;
    if (launch_after(write_op_kernel, 1, 128, 0, st, *both[i], ctx->op_dev(c.max_ops + s)) != cudaSuccess) { ctx->pair_up[s].sent = false; return MOE_ECUDA; }
    ctx->host_pair[s] = *both[i];
    ctx->pair_up[s].now(cap);
  }
  if (launch_plan_pair(hd, hp, ctx->host_ops[sd], ctx->host_ops[sp], gather_m, reinterpret_cast<int*>(bd + L.pcomb_off),
                       reinterpret_cast<int*>(bp + L.pcomb_off), c.n_experts, L.NT1, L.NT2,
                       fp8 ? kWorkRowsFp8 : kWorkRowsBf16, carrier_rows, list_form(ctx), sd, sp, st) != cudaSuccess)
    return MOE_ECUDA;
  if (ctx->pair_of[sp] >= 0) ctx->pair_of[ctx->pair_of[sp]] = -1;
  if (ctx->pair_of[sd] >= 0) ctx->pair_of[ctx->pair_of[sd]] = -1;
  ctx->pair_of[sp] = sd;
  ctx->pair_of[sd] = sp;
  return MOE_OK;
}

int moe_set_budget(moe_ctx_t* ctx, int decode_sms, void* stream) {
  if (!ctx || decode_sms < 0) return MOE_EINVAL;
  return launch_after(set_word_kernel, 1, 1, 0, static_cast<cudaStream_t>(stream), &ctx->g()->budget, decode_sms) == cudaSuccess
             ? MOE_OK : MOE_ECUDA;
}

namespace {
// q' = min(q_max, ceil_c(q * x_moe / x_star)) from the slot's planned footprint (Section 6.4)
__global__ void scaled_budget_kernel(int* budget, const PlanState* plan, int q, double x_star, int q_max, int c) {
  grid_dep_wait();
  const double want = ceil((double)q * (double)plan->n_mtiles / x_star);
  long long v = want > 2147483000.0 ? 2147483000ll : (long long)want;
  v = (v + c - 1) / c * c;
  *budget = (int)(v < (long long)q_max ? v : (long long)q_max);
}
}  // namespace

int moe_set_budget_scaled(moe_ctx_t* ctx, int slot, int q, double x_moe_star, int q_max, void* stream) {
  if (!ctx || slot < 0 || slot >= ctx->cfg.max_ops || q < 0 || q_max < 0 || !(x_moe_star > 0.0)) return MOE_EINVAL;
  if (!ctx->planned[slot]) return MOE_ENOTPLANNED;
  const PlanState* ps = reinterpret_cast<const PlanState*>(ctx->slot_base(slot) + ctx->L.plan_off);
  return launch_after(scaled_budget_kernel, 1, 1, 0, static_cast<cudaStream_t>(stream), &ctx->g()->budget, ps, q, x_moe_star, q_max,
                      ctx->pair_kernel ? 2 : 1) == cudaSuccess ? MOE_OK : MOE_ECUDA;
}

int moe_get_budget(moe_ctx_t* ctx, int32_t* out) {
  if (!ctx || !out) return MOE_EINVAL;
  return cudaMemcpy(out, &ctx->g()->budget, sizeof(int32_t), cudaMemcpyDeviceToHost) == cudaSuccess ? MOE_OK : MOE_ECUDA;
}

int moe_status(moe_ctx_t* ctx, int32_t* code, int32_t detail[4]) {
  if (!ctx || !code) return MOE_EINVAL;
  Status s;
  if (cudaMemcpy(&s, &ctx->g()->status, sizeof(s), cudaMemcpyDeviceToHost) != cudaSuccess) return MOE_ECUDA;
  *code = s.code;
  if (detail) for (int i = 0; i < 4; ++i) detail[i] = s.detail[i];
  // a plan that met an expert id out of range left its slot without a usable permutation
  if (s.code == MOE_EBADID && s.detail[0] >= 0 && s.detail[0] < ctx->cfg.max_ops) {
    const int bad = s.detail[0];
    ctx->planned[bad] = false;
    if (ctx->pair_of[bad] >= 0) ctx->pair_of[ctx->pair_of[bad]] = -1;
    ctx->pair_of[bad] = -1;
  }
  if (s.code != 0 || s.abort != 0)
    if (cudaMemset(&ctx->g()->status, 0, sizeof(Status)) != cudaSuccess) return MOE_ECUDA;
  return MOE_OK;
}

int moe_footprint(moe_ctx_t* ctx, int slot, int32_t* x_moe, int32_t* n_tiles) {
  if (!ctx || slot < 0 || slot >= ctx->cfg.max_ops) return MOE_EINVAL;
  if (!ctx->planned[slot]) return MOE_ENOTPLANNED;
  PlanState ps;
  if (cudaMemcpy(&ps, ctx->slot_base(slot) + ctx->L.plan_off, sizeof(ps), cudaMemcpyDeviceToHost) != cudaSuccess)
    return MOE_ECUDA;
  if (x_moe) *x_moe = ps.n_mtiles;
  if (n_tiles) *n_tiles = ps.n_gemm_tiles + ps.n_comb_tiles;
  return MOE_OK;
}

int moe_read_tile_table(moe_ctx_t* ctx, int slot, int32_t* host_out, int max_tiles) {
  if (!ctx || !host_out || slot < 0 || slot >= ctx->cfg.max_ops || max_tiles < 0) return MOE_EINVAL;
  if (!ctx->planned[slot]) return MOE_ENOTPLANNED;
  int n = max_tiles < ctx->L.max_mtiles ? max_tiles : ctx->L.max_mtiles;
  if (n > 0 && cudaMemcpy(host_out, ctx->slot_base(slot) + ctx->L.mtiles_off, (size_t)n * sizeof(MTile),
                          cudaMemcpyDeviceToHost) != cudaSuccess)
    return MOE_ECUDA;
  return MOE_OK;
}

int moe_read_tile_log(moe_ctx_t* ctx, moe_tile_rec_t* host_out, int max_records, int* n) {
  if (!ctx || !host_out || !n || max_records < 0) return MOE_EINVAL;
  Global g;
  RunHead rh;
  if (cudaMemcpy(&g, ctx->g(), sizeof(g), cudaMemcpyDeviceToHost) != cudaSuccess) return MOE_ECUDA;
  const size_t half = last_run_off(g.turn, (unsigned)ctx->L.run_bytes);
  if (cudaMemcpy(&rh, reinterpret_cast<unsigned char*>(ctx->rh()) + half, sizeof(rh), cudaMemcpyDeviceToHost) != cudaSuccess)
    return MOE_ECUDA;
  int cnt = (int)rh.log_count;
  if (cnt > ctx->cfg.tile_log_entries) cnt = ctx->cfg.tile_log_entries;
  if (cnt > max_records) cnt = max_records;
  if (cnt > 0 && cudaMemcpy(host_out, ctx->ws + ctx->L.log_off, (size_t)cnt * sizeof(moe_tile_rec_t),
                            cudaMemcpyDeviceToHost) != cudaSuccess)
    return MOE_ECUDA;
  *n = cnt;
  return MOE_OK;
}

}  // extern "C"
