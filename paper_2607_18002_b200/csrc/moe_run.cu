// moe_run: the persistent expert kernel (the adaptive persistent kernel of Section 4 of the
// paper, rebuilt for sm_100a), one CTA per tile.  This kernel runs the FP8 e4m3 path, and bf16 on
// grids with an odd number of CTAs; bf16 on an even grid runs on CTA pairs (moe_run_pair.cu).
//
// One CTA per SM, 16 warps with fixed roles:
//   warp 0      scheduler.  At every tile boundary it reads the decode budget
//               word and the two queue heads, claims the next tile (decode first for CTAs
//               below the budget, prefill first for the others, each falling back to the
//               other class: Sections 4.2 and 6.4), waits for the tile's dependencies and hands the tile to the other warps
//               through a shared-memory ring guarded by mbarriers (the hand-off of
//               Section 4.3: the first pipeline warp decides, later warps follow).  The next claim starts when the producer
//               has started on the published tile, so a CTA holds one claimed tile beyond the one being loaded.
//   warp 1      one thread issues tcgen05.mma (128 x 256 x 16, bf16 -> fp32) into the TMEM accumulators;
//               tcgen05.commit releases pipeline stages and publishes the accumulators.  A
//               tile of up to 256 rows runs as two 128-row MMAs per k-step against the SAME
//               weight tile in shared memory, which halves the weight bytes moved per flop.
//   warp 2      committer: when the epilogue threads have stored a tile it fences and bumps the
//               dependency counters, the op's done word and the tile log.
//   warp 3      one thread loads the weights, one stage per k-block, by tiled TMA.
//   warps 4-7   gather: the activation rows of a gate/up tile are scattered tokens; they are
//               copied through the permutation with 16-byte cp.async into the swizzled
//               layout the tensor core reads.  Consecutive rows (down tiles, masked layout) one thread of warp 4 loads as boxes.
//   warps 8-15  epilogue: tcgen05.ld, SwiGLU (gate/up tiles), bf16 stores transposed through
//               shared memory into row segments.  They also run the combine tiles.
// A phase switch happens only between tiles, so no accumulator, TMA transaction or buffer is
// live across it (Section 4.2) and results are independent of the schedule.
//
// Every wait (mbarrier, dependency counter, ready word) is bounded: when it runs out the
// kernel records MOE_ETIMEOUT, raises the abort word, and all CTAs drain and return.
#include "moe_combine.cuh"
#include "moe_ptx.cuh"
#include "moe_sched.cuh"
#include <cuda_fp8.h>
#include <type_traits>

namespace moe {

constexpr int kGatherThreads = 128;                     // 4 gather warps
constexpr int kThreads = 512;                           // 16 warps, see the role list above
constexpr int kAHalfBytes = kTileM * kRowBytes;        // 128 activation rows of one k-block
constexpr int kBHalfBytes = 128 * kRowBytes;           // 128 weight rows of one k-block
constexpr int kBBytes = 2 * kBHalfBytes;               // 256 weight rows per stage
constexpr int kMaxStages = 5;                          // bf16: three 64 KB stages, fp8: four of 48 KB or (small tiles) five of 40 KB
// registers per thread of the control, gather and epilogue warpgroups (control + gather + 2 x epilogue = 4 x 128)
constexpr int kRegsControl = 64, kRegsGather = 64, kRegsEpilogue = 192;
constexpr int kRegsControlSmall = 96, kRegsGatherSmall = 96, kRegsEpilogueSmall = 160;
// what a launch's tiles need: bf16, e4m3, or e4m3 with small tiles only
enum Mode : int { kBf16 = 0, kF8 = 1, kF8Small = 2 };
constexpr int kAccCols = 256;                          // TMEM columns per accumulator

struct F8Big {
  float amax_x[2][2][4][32];                       // amax exchange between the two warps of a quadrant, tiles alternate
};
struct F8Small {
  alignas(16) unsigned char scale[16][256];        // ring of token scales, one slot per k-block
  float amax[2][8][64];                            // per warp and token, gate/up tiles alternate
};
template <int kMode>
struct SharedCtl {
  unsigned long long full[kMaxStages];             // the weights, and 128 arrivals of the gather threads (or of the producer in their place)
  unsigned long long empty[kMaxStages];
  // producer: the stage may be overwritten (by the gather warps; by the thread that loads boxes)
  unsigned long long goA[kMaxStages], goR[kMaxStages];
  unsigned long long tfull[2], tempty[2];
  unsigned long long pfull[2], pempty[2];          // fp8: per-k-block partial products, two 256-column buffers
  unsigned long long xbar[4];                      // fp8: amax exchange between the two warps of a quadrant (small tiles: [0], all eight)
  std::conditional_t<kMode == kF8Small, F8Small, F8Big> f8;
  unsigned long long ifull[kRing], iempty[kRing], done[kRing];
  unsigned long long taken[kRing];                 // the producer has started on the tile
  TileInfo info[kRing];
  unsigned tmem_base;
  alignas(16) unsigned char epi_scratch[8][2048];   // per epilogue warp: 32 rows x 64 bytes
  QueueTables qt;
};

template <int kMode>
struct Ring {
  static constexpr int kARows = kMode == kBf16 ? 256 : kMode == kF8 ? 128 : kWorkRowsFp8Small;
  static constexpr int kBOff = kARows * kRowBytes;       // activations first, then the 256 weight rows
  static constexpr int kSB = kBOff + kBBytes;
  static constexpr int kNS = kMode == kBf16 ? 3 : kMode == kF8 ? 4 : 5;
};
template <int kMode>
constexpr size_t kSmemBytes = 1024 + (size_t)Ring<kMode>::kNS * Ring<kMode>::kSB + sizeof(SharedCtl<kMode>);
static_assert(kSmemBytes<kBf16> <= 227 * 1024 && kSmemBytes<kF8> <= 227 * 1024 && kSmemBytes<kF8Small> <= 227 * 1024, "one SM");

// ------------------------------------------------------------------ FP8 (e4m3, fp32 block scales)
// instruction descriptors: D fp32, A/B e4m3, both K-major, M = 128 or (tiles of up to 64 rows) 64, N = 256.  With M = 64 the
// accumulator's rows lie 16 to a TMEM lane quadrant; the instruction takes as long, but half of the multipliers rest: under the
// 1000 W cap a 48-token decode launch went from 1535 us at 1.16 GHz to 1356 us at 1.42 GHz (2000 prefill tokens: 2511 -> 2342 us).
constexpr unsigned kIdescF8 = (1u << 4) | ((256u >> 3) << 17) | ((128u >> 4) << 24);
constexpr unsigned kIdescF8M64 = (1u << 4) | ((256u >> 3) << 17) | ((64u >> 4) << 24);
__device__ __forceinline__ int quadrant_rows(int rows) { return rows <= 64 ? 16 : 32; }

// Small tiles (a launch whose ops have up to 64 tokens each; tiles of up to 64 rows) run with the weight rows as the M operand,
// twice 128 of them, and the token rows as the N columns: tensor energy for the rows there are, and all eight epilogue warps share
// the work that a 16-row tile otherwise leaves to the two of one TMEM quadrant (a chain of 1050 clocks per k-block).  The hand-off costs
// hundreds of clocks whatever it carries, so four (tiles of more than 32 rows: two) k-blocks share one: half of TMEM holds their
// partials.  The token scales of every k-block are copied by the gather warps into a ring: what the epilogue has not read when
// a k-block's are written is two groups and the five k-blocks in the stages, of the ring's sixteen.
// Measured under the power cap (48 tokens, 200 experts of 256): 1245 -> 1108 us a pass at 1.58 -> 1.72 GHz, and
// 8..10 % on 1 to 64 tokens over 8 to 256 experts.  A weight byte is read once an op and leaves L2 first (1141 -> 1127 us;
// two ops on the same weights, 48 + 32 tokens on 8 active experts: 122 -> 115).
// Beyond 64 rows the scale of every column makes the epilogue longer than that of the tokens-as-M form, and a kernel that holds
// both forms spills.
constexpr unsigned kIdescF8M128 = (1u << 4) | ((128u >> 4) << 24);
__device__ __forceinline__ int small_cols(int rows) { return (rows + 15) & ~15; }
// columns set aside per k-block and weight half
__device__ __forceinline__ int small_slot(int rows) { return rows <= 32 ? 32 : 64; }
// Place of a token among the scales of a k-block: in blocks of 16, ordered so that the four that one thread's fragment
// needs lie together.
__device__ __forceinline__ int scale_index(int tok) { return (tok & ~15) | ((tok & 3) << 2) | ((tok >> 2) & 3); }

// One small e4m3 tile on an epilogue warp: weight half r = (warp - 8) / 4, TMEM lanes 32 q .. +31 (gate/up: 16 features, 8 even
// gate / 8 even up / 8 odd gate / 8 odd up rows; down: 32 features).  A fragment of 16 tokens holds, per token 4 j + lane % 4, rows
// lane / 4 and lane / 4 + 8 -- the gate and the up value of a feature, or two features -- as one register pair, of lanes 0..15 and of lanes
// 16..31.  kSlot: columns set aside per k-block and weight half; kseq: k-blocks so far.
template <int kSlot>
__device__ __forceinline__ bool epilogue_fp8_small(const Ctx& c, SharedCtl<kF8Small>* sc, OpDev* op, const TileInfo& ti, unsigned tmem,
                                                   int warp, int lane, unsigned& eph, unsigned& xph, unsigned& kseq) {
  constexpr int kGroup = 128 / kSlot, kChunks = kSlot / 16;
  const RunArgs& a = *c.a;
  const int q = warp & 3, half = (warp - 8) >> 2;
  const bool g1 = ti.kind != kDown;
  const int cols = small_cols(ti.rows);
  const int HB = a.H / 128, IB = a.I / 128;
  // weight scales: one per k-block and 128 rows of the matrix
  const float *sw0, *sw1;
  if (g1) {
    sw0 = op->s_gate_up + ((size_t)expert_of(ti) * (2 * IB) + ti.n) * HB;
    sw1 = sw0 + (size_t)IB * HB;
  } else {
    sw0 = sw1 = op->s_down + ((size_t)expert_of(ti) * HB + 2 * ti.n + half) * IB;
  }
  unsigned long long acc[kChunks][4][2];
#pragma unroll
  for (int i = 0; i < kChunks * 8; ++i) acc[i >> 3][(i >> 1) & 3][i & 1] = 0ull;
  float nw0 = sw0[0], nw1 = sw1[0];                 // the next k-block's weight scales
  unsigned lo[2][8], hi[2][8];                      // fragments of a chunk; those of the next travel while it is added in
  unsigned pb = 0;
  for (int kb0 = 0; kb0 < ti.kblocks; kb0 += kGroup, pb ^= 1u) {
    const int n = min(kGroup, ti.kblocks - kb0);
    if (!__all_sync(0xffffffffu, mbar_wait_inline(c, &sc->pfull[pb], (eph >> pb) & 1u, 19))) return false;
    eph ^= 1u << pb;
    tc_fence_after();
    unsigned taddr = tmem + pb * 256u + (unsigned)(half * kSlot) + ((unsigned)(q * 32) << 16);
    tc_ld_pairs(taddr, lo[0]);
    tc_ld_pairs(taddr + (16u << 16), hi[0]);
#pragma unroll 1
    for (int g = 0; g < n; ++g) {
      const unsigned long long w = f32x2(nw0, nw1);
      if (kb0 + g + 1 < ti.kblocks) { nw0 = sw0[kb0 + g + 1]; nw1 = sw1[kb0 + g + 1]; }
      const float* xs = reinterpret_cast<const float*>(sc->f8.scale[kseq++ & 15u]) + 4 * (lane & 3);
      float4 nx = *reinterpret_cast<const float4*>(xs);
#pragma unroll
      for (int ch = 0; ch < kChunks; ++ch) {
        if (ch * 16 >= cols) break;
        const float4 x = nx;
        tc_wait_ld();
        const bool more = ch + 1 < kChunks && (ch + 1) * 16 < cols;
        if (more) {
          tc_ld_pairs(taddr + (unsigned)((ch + 1) * 16), lo[(ch + 1) & 1]);
          tc_ld_pairs(taddr + (unsigned)((ch + 1) * 16) + (16u << 16), hi[(ch + 1) & 1]);
          nx = *reinterpret_cast<const float4*>(xs + (ch + 1) * 16);
        }
        const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const unsigned long long sw = mul_f32x2(f32x2(xv[j], xv[j]), w);
          acc[ch][j][0] = fma_f32x2(f32x2(__uint_as_float(lo[ch & 1][2 * j]), __uint_as_float(lo[ch & 1][2 * j + 1])), sw, acc[ch][j][0]);
          acc[ch][j][1] = fma_f32x2(f32x2(__uint_as_float(hi[ch & 1][2 * j]), __uint_as_float(hi[ch & 1][2 * j + 1])), sw, acc[ch][j][1]);
        }
      }
      taddr += 2u * kSlot;
      if (g + 1 < n) {
        tc_ld_pairs(taddr, lo[0]);
        tc_ld_pairs(taddr + (16u << 16), hi[0]);
      }
    }
    tc_fence_before();
    __syncwarp();                                   // every lane's TMEM and scale loads have completed
    if (lane == 0) mbar_arrive(&sc->pempty[pb]);
  }
  unsigned char* scratch = sc->epi_scratch[warp - 8];
  const unsigned scratch_addr = smem_u32(scratch);
  // stored row lane % 8 of matrix lane / 8 (8 tokens) is this token: the matrix' columns 2 i, 2 i + 1 are tokens i, i + 4
  const int row = (lane & ~7) + 4 * (lane & 1) + ((lane & 7) >> 1);
  if (!g1) {
    unsigned char* out = reinterpret_cast<unsigned char*>(op->D) + (size_t)ti.row0 * a.H * 2 +
                         (size_t)(ti.n * kTileN2 + half * 128 + q * 32) * 2;
#pragma unroll
    for (int p = 0; p < kChunks / 2; ++p) {
      if (p * 32 >= ti.rows) break;
      unsigned o[16];
#pragma unroll
      for (int j = 0; j < 4; ++j) {                 // matrix j: tokens 8 j .. + 7 of the pass
        const int ch = 2 * p + (j >> 1), k = 2 * (j & 1);
        const float2 e0 = f32x2_parts(acc[ch][k][0]), e1 = f32x2_parts(acc[ch][k + 1][0]);
        const float2 f0 = f32x2_parts(acc[ch][k][1]), f1 = f32x2_parts(acc[ch][k + 1][1]);
        o[j] = pack_bf16(e0.x, e1.x);
        o[4 + j] = pack_bf16(e0.y, e1.y);
        o[8 + j] = pack_bf16(f0.x, f1.x);
        o[12 + j] = pack_bf16(f0.y, f1.y);
      }
      store_features32(scratch, scratch_addr, o, row, out + (size_t)(p * 32) * a.H * 2, (size_t)a.H * 2, ti.rows - p * 32, lane);
    }
    return true;
  }
  // SwiGLU; per token the largest of this warp's 16 features, then of the tile's 128
  float* mine = sc->f8.amax[xph & 1u][warp - 8];
#pragma unroll
  for (int ch = 0; ch < kChunks; ++ch) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 e = f32x2_parts(acc[ch][j][0]), d = f32x2_parts(acc[ch][j][1]);
      const float v0 = __fdividef(e.x, 1.0f + __expf(-e.x)) * e.y, v1 = __fdividef(d.x, 1.0f + __expf(-d.x)) * d.y;
      acc[ch][j][0] = f32x2(v0, v1);                // the even and the odd feature
      float m = fmaxf(fabsf(v0), fabsf(v1));
#pragma unroll
      for (int s = 4; s < 32; s <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, s));
      if (lane < 4) mine[ch * 16 + 4 * j + lane] = m;
    }
  }
  // The eight warps meet here.  Like every wait it is bounded: a warp may have left because the launch was aborted.  One meeting a
  // tile is enough: a warp writes this half of amax again two tiles on, past the meeting that all come to after reading it.
  __syncwarp();
  if (lane == 0) mbar_arrive(&sc->xbar[0]);
  if (!__all_sync(0xffffffffu, mbar_wait_inline(c, &sc->xbar[0], xph & 1u, 20))) return false;
  const float(&all)[8][64] = sc->f8.amax[xph & 1u];
  xph ^= 1u;
  float inv[kSlot / 32];                            // of tokens lane, lane + 32
#pragma unroll
  for (int p = 0; p < kSlot / 32; ++p) {
    const int tok = 32 * p + lane;
    float amax = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) amax = fmaxf(amax, all[w][tok]);
    inv[p] = amax > 0.f ? 448.0f / amax : 0.0f;
    if (warp == 8 && tok < ti.rows) op->a_scale[(size_t)(ti.row0 + tok) * IB + ti.n] = amax > 0.f ? amax / 448.0f : 1.0f;
  }
  unsigned char* out = reinterpret_cast<unsigned char*>(op->A) + (size_t)ti.row0 * a.I + (size_t)(ti.n * kTileN1 + half * 64 + q * 16);
#pragma unroll
  for (int p = 0; p < kSlot / 32; ++p) {
    unsigned o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      o[j] = 0u;
#pragma unroll
      for (int s = 0; s < 2; ++s) {                 // 16-bit elements: the two neighbouring features of a token
        const int g = 2 * (j & 1) + s;
        const float2 v = f32x2_parts(acc[2 * p + (j >> 1)][g][0]);
        const float k = __shfl_sync(0xffffffffu, inv[p], 16 * (j >> 1) + 4 * g + (lane & 3));
        o[j] |= (unsigned)__nv_cvt_float2_to_fp8x2(make_float2(v.x * k, v.y * k), __NV_SATFINITE, __NV_E4M3) << (16 * s);
      }
    }
    __syncwarp();
    st_matrix4_trans(scratch_addr + row * 16, o[0], o[1], o[2], o[3]);
    __syncwarp();
    const uint4 v4 = *reinterpret_cast<const uint4*>(scratch + lane * 16);
    if (32 * p + lane < ti.rows) *reinterpret_cast<uint4*>(out + (size_t)(32 * p + lane) * a.I) = v4;
  }
  return true;
}

// The activation scales of one row of a tile: its own op's, or (paired form) its partner's when the row is tagged so.
__device__ __forceinline__ const float* row_scales(const Ctx& c, const OpDev* op, const TileInfo& ti, int row, bool valid) {
  const RunArgs& a = *c.a;
  if (ti.kind == kDown) return op->a_scale + (size_t)(ti.row0 + (valid ? row : 0)) * (a.I / 128);
  if (ti.kind == kGateUpDirect) return op->x_scale + (size_t)(ti.row0 + (valid ? row : 0)) * (a.H / 128);   // masked layout
  int tok = 0;
  const OpDev* src = op;
  if (valid) {
    const int v = op->gather_list[ti.row0 + row];
    const int tag = v >> kRowSlotShift, flat = v & kRowFlatMask;
    const int own_tag = op->paired ? slot_of(&a, ti.slot) : 0;
    if (op->paired && tag != own_tag && tag == slot_of(&a, op->partner)) src = &a.ops[op->partner];
    if (v >= 0 && (tag == own_tag || src != op) && flat < src->n_rows) tok = flat / a.k;
    else { src = op; report(c.st, MOE_EBOUNDS, slot_of(&a, ti.slot), ti.row0 + row, v, 1); }
  }
  return src->x_scale + (size_t)tok * (a.H / 128);
}

// The weight scales of a tile, one per k-block and 128 rows of the matrix.
__device__ __forceinline__ void weight_scales(const RunArgs& a, const OpDev* op, const TileInfo& ti, const float*& sw0, const float*& sw1) {
  const int HB = a.H / 128, IB = a.I / 128;
  if (ti.kind != kDown) {
    sw0 = op->s_gate_up + ((size_t)expert_of(ti) * (2 * IB) + ti.n) * HB;
    sw1 = sw0 + (size_t)IB * HB;
  } else {
    sw0 = op->s_down + ((size_t)expert_of(ti) * HB + 2 * ti.n) * IB;
    sw1 = sw0 + IB;
  }
}

// One e4m3 tile of up to 64 rows on the epilogue warps.  With M = 64 only 16 lanes of a TMEM quadrant hold rows, so a fragment load
// spreads 16 rows x 64 columns over the whole warp: row lane / 4 and the row eight below, columns 8 j + 2 (lane % 4) and the next as
// register pairs.  That is half of the registers and a quarter of the multiply-add instructions that a thread per row needs, and a
// k-block's two loads are in flight together; the partial buffer is handed back before they are multiplied in.  2000 tokens over 256
// experts: 2128 -> 2090 us a pass, 4096 + 512 paired: 3184 -> 3152.  (The same packed adds and early hand-back in the form of a thread per
// row, whose registers hold one chunk at a time, gave nothing: 3152 -> 3160.)
__device__ __forceinline__ bool epilogue_fp8_m64(const Ctx& c, SharedCtl<kF8>* sc, OpDev* op, const TileInfo& ti, unsigned tmem, int warp,
                                                 int lane, unsigned& eph, unsigned& xph) {
  const RunArgs& a = *c.a;
  const int q = warp & 3, ch = (warp - 8) >> 2;
  const bool g1 = ti.kind != kDown;
  const int IB = a.I / 128;
  const int r0 = q * 16 + (lane >> 2);              // and r0 + 8
  const float* sx0 = row_scales(c, op, ti, r0, r0 < ti.rows);
  const float* sx1 = row_scales(c, op, ti, r0 + 8, r0 + 8 < ti.rows);
  const float *sw0, *sw1;
  weight_scales(a, op, ti, sw0, sw1);
  unsigned long long acc[2][8][2];                  // [128-column half][8-column group][row]
#pragma unroll
  for (int i = 0; i < 32; ++i) acc[i >> 4][(i >> 1) & 7][i & 1] = 0ull;
  float nx0 = sx0[0], nx1 = sx1[0], nw0 = sw0[0], nw1 = sw1[0];      // of the next k-block
  const unsigned lane_addr = tmem + ((unsigned)(q * 32) << 16) + (unsigned)(ch * 64);
  for (int kb = 0; kb < ti.kblocks; ++kb) {
    const float s[2][2] = {{nx0 * nw0, nx1 * nw0}, {nx0 * nw1, nx1 * nw1}};
    if (kb + 1 < ti.kblocks) { nx0 = sx0[kb + 1]; nx1 = sx1[kb + 1]; nw0 = sw0[kb + 1]; nw1 = sw1[kb + 1]; }
    const int pb = kb & 1;
    if (!__all_sync(0xffffffffu, mbar_wait_inline(c, &sc->pfull[pb], (eph >> pb) & 1u, 19))) return false;
    eph ^= 1u << pb;
    tc_fence_after();
    unsigned p[2][32];
    tc_ld_frag64(lane_addr + (unsigned)(pb * 256), p[0]);
    tc_ld_frag64(lane_addr + (unsigned)(pb * 256 + 128), p[1]);
    tc_wait_ld();
    tc_fence_before();
    __syncwarp();                                   // every lane's TMEM loads have completed
    if (lane == 0) mbar_arrive(&sc->pempty[pb]);
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int r = 0; r < 2; ++r)
          acc[h][j][r] = fma_f32x2(f32x2(__uint_as_float(p[h][4 * j + 2 * r]), __uint_as_float(p[h][4 * j + 2 * r + 1])),
                                   f32x2(s[h][r], s[h][r]), acc[h][j][r]);
  }
  // rows leave through the warp's scratch, 16 bytes a lane; the 16-byte chunks of a row are rotated by XOR to keep banks apart
  unsigned char* scratch = sc->epi_scratch[warp - 8];
  const int fr = lane >> 2, fc = lane & 3;
  if (g1) {
    float amax[2] = {0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float2 g = f32x2_parts(acc[0][j][r]), u = f32x2_parts(acc[1][j][r]);
        const float v0 = __fdividef(g.x, 1.0f + __expf(-g.x)) * u.x, v1 = __fdividef(g.y, 1.0f + __expf(-g.y)) * u.y;
        acc[0][j][r] = f32x2(v0, v1);
        amax[r] = fmaxf(amax[r], fmaxf(fabsf(v0), fabsf(v1)));
      }
    float* mine = sc->f8.amax_x[xph & 1u][ch][q];
    const float* other = sc->f8.amax_x[xph & 1u][ch ^ 1][q];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      amax[r] = fmaxf(amax[r], __shfl_xor_sync(0xffffffffu, amax[r], 1));
      amax[r] = fmaxf(amax[r], __shfl_xor_sync(0xffffffffu, amax[r], 2));
      if (fc == 0) mine[fr + 8 * r] = amax[r];
    }
    mbar_arrive(&sc->xbar[q]);
    if (!__all_sync(0xffffffffu, mbar_wait_inline(c, &sc->xbar[q], xph, 20))) return false;
    xph ^= 1u;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const float m = fmaxf(amax[r], other[fr + 8 * r]);
      const float inv = m > 0.f ? 448.0f / m : 0.0f;
      const int row = fr + 8 * r;
      if (ch == 0 && fc == 0 && q * 16 + row < ti.rows)
        op->a_scale[(size_t)(ti.row0 + q * 16 + row) * IB + ti.n] = m > 0.f ? m / 448.0f : 1.0f;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float2 v = f32x2_parts(acc[0][j][r]);
        *reinterpret_cast<unsigned short*>(scratch + row * 64 + (((j >> 1) ^ ((row >> 1) & 3)) << 4) + (j & 1) * 8 + fc * 2) =
            (unsigned short)__nv_cvt_float2_to_fp8x2(make_float2(v.x * inv, v.y * inv), __NV_SATFINITE, __NV_E4M3);
      }
    }
    __syncwarp();
    unsigned char* out = reinterpret_cast<unsigned char*>(op->A) + (size_t)(ti.row0 + q * 16) * a.I + (size_t)(ti.n * kTileN1 + ch * 64);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int row = 8 * i + fr;
      const uint4 v4 = *reinterpret_cast<const uint4*>(scratch + row * 64 + ((fc ^ ((row >> 1) & 3)) << 4));
      if (q * 16 + row < ti.rows) *reinterpret_cast<uint4*>(out + (size_t)row * a.I + fc * 16) = v4;
    }
    __syncwarp();                                   // scratch free again
    return true;
  }
  unsigned char* out = reinterpret_cast<unsigned char*>(op->D) + ((size_t)(ti.row0 + q * 16) * a.H + (size_t)ti.n * kTileN2 + ch * 64) * 2;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int row = fr + 8 * r;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float2 v = f32x2_parts(acc[h][j][r]);
        *reinterpret_cast<unsigned*>(scratch + row * 128 + ((j ^ (row & 7)) << 4) + fc * 4) = pack_bf16(v.x, v.y);
      }
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int row = 4 * i + (lane >> 3), f = lane & 7;
      const uint4 v4 = *reinterpret_cast<const uint4*>(scratch + row * 128 + ((f ^ (row & 7)) << 4));
      if (q * 16 + row < ti.rows) *reinterpret_cast<uint4*>(out + ((size_t)row * a.H + h * 128) * 2 + f * 16) = v4;
    }
    __syncwarp();
  }
  return true;
}

// One e4m3 tile on the epilogue warps.  Thread = (accumulator row, 64-column slice of each
// 128-column half); its 128 fp32 accumulators stay in registers (the epilogue warps raise
// their register allowance for this).  Per k-block and half: partial * (activation scale of
// the row and k-block * weight scale of the half and k-block) is added in.  Then gate/up
// tiles apply SwiGLU and re-quantise the 128 outputs of the row to e4m3 with one fp32 scale
// (amax / 448) -- the one quantisation on the path -- and down tiles store bf16.
__device__ __forceinline__ bool epilogue_fp8(const Ctx& c, SharedCtl<kF8>* sc, OpDev* op, const TileInfo& ti,
                                             unsigned tmem, int warp, int lane, unsigned& eph,
                                             unsigned& xph) {
  const RunArgs& a = *c.a;
  const int q = warp & 3, ch = (warp - 8) >> 2;
  const int per_q = quadrant_rows(ti.rows);
  const int row = q * 32 + lane;
  const bool valid = row < ti.rows;
  const bool g1 = ti.kind != kDown;
  const int IB = a.I / 128;
  const unsigned lane_addr = tmem + ((unsigned)(q * 32) << 16);
  if (q * per_q >= ti.rows) {
    // No row of the tile lies in this warp's TMEM lane quadrant (both warps of a quadrant see
    // the same q): nothing to read, scale or store.  The warp still takes part in every partial
    // buffer hand-off, so that the barrier counts and phases stay those of a full tile.
    for (int kb = 0; kb < ti.kblocks; ++kb) {
      const int pb = kb & 1;
      if (!__all_sync(0xffffffffu, mbar_wait_inline(c, &sc->pfull[pb], (eph >> pb) & 1u, 19))) return false;
      eph ^= 1u << pb;
      if (lane == 0) mbar_arrive(&sc->pempty[pb]);
    }
    return true;
  }
  if (ti.rows <= 64) return epilogue_fp8_m64(c, sc, op, ti, tmem, warp, lane, eph, xph);
  const float* sx = row_scales(c, op, ti, row, valid);
  const float *sw0, *sw1;
  weight_scales(a, op, ti, sw0, sw1);
  float acc[128];                                 // [half][64]
#pragma unroll
  for (int i = 0; i < 128; ++i) acc[i] = 0.f;
  // scales of the next k-block are loaded one k-block ahead (three scalars in flight)
  float nfx = 0.f, nw0 = 0.f, nw1 = 0.f;
  if (ti.kblocks > 0) { nfx = sx[0]; nw0 = sw0[0]; nw1 = sw1[0]; }
  for (int kb = 0; kb < ti.kblocks; ++kb) {
    const float s0 = nfx * nw0, s1 = nfx * nw1;
    if (kb + 1 < ti.kblocks) { nfx = sx[kb + 1]; nw0 = sw0[kb + 1]; nw1 = sw1[kb + 1]; }
    const int pb = kb & 1;
    if (!__all_sync(0xffffffffu, mbar_wait_inline(c, &sc->pfull[pb], (eph >> pb) & 1u, 19))) return false;
    eph ^= 1u << pb;
    tc_fence_after();
    // four 32-column chunks (two per half), one TMEM load each: tcgen05.wait::ld waits for every load of the
    // thread, so a second load in flight only ever overlapped one chunk's FMAs; fewer, wider loads are faster
    // (the other warp of the scheduler partition fills the wait)
    const unsigned pbase = lane_addr + (unsigned)(pb * 256 + ch * 64);
    unsigned p[32];
#pragma unroll
    for (int cc = 0; cc < 4; ++cc) {
      tc_ld32(pbase + (unsigned)((cc >> 1) * 128 + (cc & 1) * 32), p);
      tc_wait_ld();
      const float s = (cc >> 1) ? s1 : s0;
#pragma unroll
      for (int i = 0; i < 32; ++i)
        acc[cc * 32 + i] = fmaf(__uint_as_float(p[i]), s, acc[cc * 32 + i]);
    }
    tc_fence_before();
    __syncwarp();                                 // every lane's TMEM loads have completed
    if (lane == 0) mbar_arrive(&sc->pempty[pb]); // one arrival per warp: the partial buffer may be overwritten
  }
  // the accumulator is complete
  if (g1) {
    float amax = 0.f;
#pragma unroll
    for (int i = 0; i < 64; ++i) {                // gate column i and up column i of this slice
      const float gv = acc[i];
      const float v = __fdividef(gv, 1.0f + __expf(-gv)) * acc[64 + i];
      acc[i] = v;
      amax = fmaxf(amax, fabsf(v));
    }
    // the row's 128 outputs live in two threads (ch = 0, 1): exchange the partial maxima
    sc->f8.amax_x[xph & 1u][ch][q][lane] = amax;
    mbar_arrive(&sc->xbar[q]);
    if (!__all_sync(0xffffffffu, mbar_wait_inline(c, &sc->xbar[q], xph, 20))) return false;
    amax = fmaxf(amax, sc->f8.amax_x[xph & 1u][ch ^ 1][q][lane]);
    xph ^= 1u;
    const float scale = amax > 0.f ? amax / 448.0f : 1.0f;
    const float inv = amax > 0.f ? 448.0f / amax : 0.0f;
    if (valid) {
      unsigned char* dst = static_cast<unsigned char*>((void*)op->A) + (size_t)(ti.row0 + row) * a.I +
                           (size_t)ti.n * 128 + ch * 64;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        unsigned w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int b0 = j * 16 + i * 4;
          const unsigned lo = __nv_cvt_float2_to_fp8x2(make_float2(acc[b0] * inv, acc[b0 + 1] * inv), __NV_SATFINITE, __NV_E4M3);
          const unsigned hi = __nv_cvt_float2_to_fp8x2(make_float2(acc[b0 + 2] * inv, acc[b0 + 3] * inv), __NV_SATFINITE, __NV_E4M3);
          w[i] = lo | (hi << 16);
        }
        reinterpret_cast<uint4*>(dst)[j] = make_uint4(w[0], w[1], w[2], w[3]);
      }
      if (ch == 0) op->a_scale[(size_t)(ti.row0 + row) * IB + ti.n] = scale;
    }
  } else if (valid) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      __nv_bfloat16* dst = op->D + (size_t)(ti.row0 + row) * a.H + (size_t)ti.n * kTileN2 + h * 128 + ch * 64;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        uint4 o4;
        __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(&o4);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          oh[i] = __floats2bfloat162_rn(acc[h * 64 + j * 8 + 2 * i], acc[h * 64 + j * 8 + 2 * i + 1]);
        reinterpret_cast<uint4*>(dst)[j] = o4;
      }
    }
  }
  return true;
}

// a warpgroup's registers per thread, of the launch's 128
template <int kMode, int kRegs, int kRegsSmall>
__device__ __forceinline__ void take_registers() {
  constexpr int n = kMode == kF8 ? kRegs : kMode == kF8Small ? kRegsSmall : 128;
  if constexpr (n < 128) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(n));
  else if constexpr (n > 128) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(n));
}

// The boxes of consecutive rows that a tile's k-block takes: of 8, 32, 128 or 256 rows, the smallest that holds them (small tiles: up to
// two of 32)
struct RowBoxes {
  int rows, boxes;
  __device__ __forceinline__ unsigned bytes() const { return (unsigned)(rows * boxes * kRowBytes); }
};
template <int kMode>
__device__ __forceinline__ RowBoxes row_boxes(int rows) {
  if (rows <= 8) return RowBoxes{8, 1};
  if (kMode == kF8Small) return RowBoxes{32, rows > 32 ? 2 : 1};
  return RowBoxes{rows <= 32 ? 32 : rows <= 128 ? 128 : 256, 1};
}

// ------------------------------------------------------------------ the persistent kernel
// which accumulator(s) a tile uses: a tile of up to 128 rows alternates between the two, a
// tile of up to 256 rows takes both (rows 0..127 -> accumulator 0, rows 128..255 -> 1).
// Every role walks the same tile sequence, so each derives this locally.
struct AccUse {
  int next = 0;
  __device__ __forceinline__ void take(int rows, bool& use0, bool& use1) {
    if (rows > kTileM) { use0 = use1 = true; }
    else { use0 = next == 0; use1 = !use0; next ^= 1; }
  }
};

template <int kMode>
__global__ void __launch_bounds__(kThreads, 1) moe_apk_kernel(const __grid_constant__ RunArgs args,
                                                              RunHead* rh) {
  constexpr bool kFp8 = kMode != kBf16, kSmall = kMode == kF8Small;
  constexpr int kKb = kFp8 ? 128 : kBlockK;     // K elements per stage (128 bytes per row either way)
  constexpr int kEl = kFp8 ? 1 : 2;             // bytes per element
  constexpr int kNS = Ring<kMode>::kNS, kBOff = Ring<kMode>::kBOff, kSB = Ring<kMode>::kSB;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* stages = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  SharedCtl<kMode>* sc = reinterpret_cast<SharedCtl<kMode>*>(stages + (size_t)kNS * kSB);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  Ctx c{&args, &args.g->status, 0u};

  if (threadIdx.x == 0) {
    for (int s = 0; s < kNS; ++s) {
      mbar_init(&sc->full[s], 1 + kGatherThreads);
      mbar_init(&sc->goA[s], 1);
      mbar_init(&sc->goR[s], 1);
      mbar_init(&sc->empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sc->tfull[s], 1);
      mbar_init(&sc->tempty[s], 256);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sc->pfull[s], 1);
      mbar_init(&sc->pempty[s], 8);
    }
    for (int s = 0; s < 4; ++s) mbar_init(&sc->xbar[s], kSmall ? 8 : 64);
    // a ring slot is released by the MMA thread, the committer, the producer and each gather warp
    for (int s = 0; s < kRing; ++s) {
      mbar_init(&sc->ifull[s], 1);
      mbar_init(&sc->iempty[s], 3 + kGatherThreads / 32);
      mbar_init(&sc->taken[s], 1);
      mbar_init(&sc->done[s], 256);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_proxy();
  }
  if (warp == 1) {   // TMEM: both accumulators (512 columns); this warp also frees them
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&sc->tmem_base)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  grid_dep_wait();             // everything above overlaps the kernel before this one
  if (warp == 0) begin_unit<false>(&args, &sc->qt, rh, lane, 1, Ring<kMode>::kARows);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned tmem = sc->tmem_base;
  c.run_off = sc->qt.run_off;
  if (warp == 2 && lane == 0) end_turn(&args, take_turn(&args), (int)gridDim.x);
  const bool watched = sc->qt.watched != 0;
  if (blockIdx.x == 0 && warp == 2) {
    clear_next_run(&args, rh, c.run_off, lane);
    if (lane == 0 && watched) finish_empty_ops(c, -1);
  }
  bool ended = true;           // false: this thread left its role because a wait gave up
  rh = reinterpret_cast<RunHead*>(reinterpret_cast<char*>(rh) + c.run_off);
  // The fp8 epilogue keeps 128 fp32 accumulators per thread: the two epilogue warpgroups take
  // registers from the two others (64 + 192 = 2 x 128 per thread pair).  Each role changes its
  // allowance at the top of its own branch, so the compiler can budget the branch by it.
  const auto control_regs = [] { take_registers<kMode, kRegsControl, kRegsControlSmall>(); };
  const auto gather_regs = [] { take_registers<kMode, kRegsGather, kRegsGatherSmall>(); };
  const auto epilogue_regs = [] { take_registers<kMode, kRegsEpilogue, kRegsEpilogueSmall>(); };

  if (warp == 0) {
    control_regs();
    // ============================================================ scheduler
    // The next tile is claimed while the current one is being loaded, so the claim's round trips do not drain the pipeline.
    ended = false;
    int islot = 0;
    unsigned iph = 0;
    TileInfo ti;
    bool need_ready = false, one = false;
    ti.kind = kEnd;
    ti.slot = ti.tile = ti.m = ti.row0 = ti.rows = ti.n = ti.kblocks = ti.expert = ti.cls = 0;
    ti.t_claim = 0;
    while (true) {
      claim_next<false, false>(c, &sc->qt, rh, lane, ti, need_ready, one);
      ti.kind = __shfl_sync(0xffffffffu, ti.kind, 0);      // the claim loops exit warp-uniformly
      const OpDev* op = &args.ops[ti.kind == kEnd ? args.slots[0] : ti.slot];
      // a free ring slot, the op ready, the tile's dependencies met
      if (!__all_sync(0xffffffffu, mbar_wait(c, &sc->iempty[islot], iph ^ 1u, 2))) break;
      if (ti.kind != kEnd && need_ready && !wait_op_ready(c, lane, ti)) ti.kind = kEnd;
      int ok = 1;
      if (lane == 0) {
        // a claimed tile only ever waits on tiles that were claimed before it
        if (ti.kind == kDown) ok = wait_counter(c, &g1_done_of(c, op)[ti.m], args.I / kTileN1, 3);
        if (ti.kind == kCombine) ok = wait_counter(c, &run_of(c, op)->gemm_done, op_down_tiles(&args, op), 4);
        if (!ok) ti.kind = kEnd;
        fence_async_proxy();
        sc->info[islot] = ti;
        __threadfence_block();
        mbar_arrive(&sc->ifull[islot]);
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (ti.kind == kEnd || !ok) { ended = ok; break; }
      if (!__all_sync(0xffffffffu, mbar_wait(c, &sc->taken[islot], iph, 26))) break;
      if (++islot == kRing) { islot = 0; iph ^= 1u; }
    }
  } else if (warp == 3) {
    control_regs();
    // ============================================================ producer
    // The weights of the tiles in the ring, and the go-ahead for those that bring the rows.  One thread runs the whole role, see elect_one.
    if (elect_one()) {
      ended = false;
      int islot = 0;
      unsigned iph = 0;
      unsigned stage = 0, par = 1;                         // parity of "stage is free"
      bool ready = false;                                  // the stage was seen free by the look-ahead test
      const unsigned stages0 = smem_u32(stages), full0 = smem_u32(&sc->full[0]), empty0 = smem_u32(&sc->empty[0]);
      while (true) {
        if (!mbar_wait(c, &sc->ifull[islot], iph, 21)) break;
        const int kind = sc->info[islot].kind, kblocks = sc->info[islot].kblocks, rows = sc->info[islot].rows;
        const int n = sc->info[islot].n, expert = expert_of(sc->info[islot]), slot = sc->info[islot].slot;
        // As in the CTA-pair kernel, the weights of an expert with one work tile leave L2 first (2000 tokens: 2075 -> 2038 us a pass, 4096 + 512
        // paired 3060 -> 3021, 512 on 64 experts 500 -> 485, 1000 + 200 unpaired 1744 -> 1713).  A kernel of its own for launches
        // without a second tile, with the whole producer warp choosing, was 0.9 % slower for the others.
        const unsigned long long policy = sc->info[islot].expert & kReadOnce ? l2_evict_first() : l2_evict_normal();
        if (kind == kEnd) { ended = true; break; }
        mbar_arrive(&sc->taken[islot]);
        mbar_arrive(&sc->iempty[islot]);
        if (++islot == kRing) { islot = 0; iph ^= 1u; }
        if (kind == kCombine) continue;
        const OpDev* op = &args.ops[slot];
        const bool g1 = kind != kDown;                     // gate/up weights
        const bool gathered = kind == kGateUp;             // activation rows come from the gather warps
        const CUtensorMap* tmw = kSmall ? (g1 ? &op->tm_p1 : &op->tm_p2) : (g1 ? &op->tm_w1 : &op->tm_w2);
        // the box of 256 weight rows of this tile, see OpDev
        const int c1 = kSmall || !g1 ? 0 : n * kTileN1;
        const int c2 = kSmall || g1 ? 0 : n * (kTileN2 / 128);
        const int c3 = !kSmall ? expert : g1 ? expert * 2 * args.I + n * kTileN1 : n * kTileN2 / 16;
        const int c4 = kSmall && !g1 ? expert : 0;
        const unsigned tx = (unsigned)kBBytes + (gathered ? 0u : row_boxes<kMode>(rows).bytes());
        const bool all_gather = gathered || kSmall;        // the gather warps arrive for every k-block (small tiles: with the scales)
        const unsigned go = all_gather ? smem_u32(&sc->goA[0]) : smem_u32(&sc->goR[0]), standin = all_gather ? 0u : (unsigned)kGatherThreads;
        bool fail = false;
        for (int kb = 0; kb < kblocks; ++kb) {
          if (!ready && !mbar_wait(c, &sc->empty[stage], par, 5)) { fail = true; break; }
          const unsigned nstage = stage + 1 == kNS ? 0u : stage + 1, npar = stage + 1 == kNS ? par ^ 1u : par;
          ready = single_issue_kblock(full0 + stage * 8u, tx, standin, go + stage * 8u, stages0 + stage * (unsigned)kSB + (unsigned)kBOff, tmw,
                                      kb * kKb, c1, c2, c3, c4, policy, empty0 + nstage * 8u, npar);
          stage = nstage;
          par = npar;
        }
        if (fail) break;
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    control_regs();
    // ============================================================ MMA issuer
    // One thread runs the whole role (see elect_one), and the barriers of the next k-block are tested while the MMAs of one are issued.  (The
    // whole warp in the loop, an election around each group and a wait for each of three barriers: 1090 clocks a k-block of up to 64
    // rows, 1240 above, now 1045 and 1190, of which the MMAs need 512; what is left is the partial buffers' way to the epilogue and back.)
    // With the scheduler, the loads of weights and those of rows on threads of their own: 48 tokens 1164 -> 1134 us a pass, 4096 + 512
    // paired 3412 -> 3389.
    if (elect_one()) {
      ended = false;
      unsigned stage = 0, par = 0, iph = 0, aph[2] = {0, 0}, pph = 0;
      int islot = 0;
      bool ready = false;                                  // the stage was seen full by the look-ahead test
      AccUse accs;
      const unsigned full0 = smem_u32(&sc->full[0]), empty0 = smem_u32(&sc->empty[0]), pfull0 = smem_u32(&sc->pfull[0]),
                     pempty0 = smem_u32(&sc->pempty[0]);
      const unsigned long long desc0 = umma_desc(smem_u32(stages), kRowBytes);
      while (true) {
        if (!mbar_wait(c, &sc->ifull[islot], iph, 6)) break;
        const int kind = sc->info[islot].kind;
        const int kblocks = sc->info[islot].kblocks;
        const int rows = sc->info[islot].rows;
        if (kind == kEnd) { ended = true; break; }
        bool fail = false;
        if (kFp8 && kind != kCombine) {
          // FP8 with fp32 block scales: the tensor core cannot apply a scale per 128-deep K block,
          // so every k-block (= one scale block) is multiplied into a FRESH partial buffer, one
          // per 128-column half of the weight tile (each half has a single weight scale), and the
          // epilogue warps scale-and-add it into their fp32 accumulators.
          const unsigned idesc8 = rows <= 64 ? kIdescF8M64 : kIdescF8;
          const unsigned idesc_small = kIdescF8M128 | ((unsigned)small_cols(rows) >> 3) << 17;
          const int slot = small_slot(rows), last_of_group = 128 / slot - 1;
          bool drained = false;                            // the next partial buffer was seen free
          for (int kb = 0; kb < kblocks; ++kb) {
            if (!ready && !mbar_wait(c, &sc->full[stage], par, 8)) { fail = true; break; }
            const unsigned nstage = stage + 1 == kNS ? 0u : stage + 1, npar = stage + 1 == kNS ? par ^ 1u : par;
            const unsigned long long xd = desc0 + stage * (unsigned)(kSB / 16), wd = xd + (unsigned)(kBOff / 16);
            if constexpr (kSmall) {
              const int g = kb & last_of_group, pb = (kb / (last_of_group + 1)) & 1;
              if (g == 0) {
                if (!mbar_wait(c, &sc->pempty[pb], ((pph >> pb) & 1u) ^ 1u, 18)) { fail = true; break; }
                pph ^= 1u << pb;
              }
              tc_fence_after();
              fence_async_proxy_smem();
              ready = f8_small_kblock(tmem + (unsigned)(pb * 256 + g * 2 * slot), wd, wd + (unsigned)(kBHalfBytes / 16), xd, idesc_small,
                                      (unsigned)slot, pfull0 + pb * 8u, g == last_of_group || kb + 1 == kblocks ? 1u : 0u,
                                      empty0 + stage * 8u, full0 + nstage * 8u, npar);
            } else {
              const unsigned pb = kb & 1u;                 // partial buffer of this k-block
              if (!drained && !mbar_wait(c, &sc->pempty[pb], ((pph >> pb) & 1u) ^ 1u, 18)) { fail = true; break; }
              pph ^= 1u << pb;
              tc_fence_after();
              fence_async_proxy_smem();
              // four MMAs of 32 e4m3 elements (32 bytes) each, partial full, stage empty
              f8_mma_kblock(tmem + pb * 256u, xd, wd, idesc8, pfull0 + pb * 8u, empty0 + stage * 8u, full0 + nstage * 8u, npar,
                            pempty0 + (pb ^ 1u) * 8u, ((pph >> (pb ^ 1u)) & 1u) ^ 1u, ready, drained);
            }
            stage = nstage;
            par = npar;
          }
          if (fail) break;
        } else if (kind != kCombine) {
          bool use0, use1;
          accs.take(rows, use0, use1);
          // A 256-row tile takes both accumulators: it waits for accumulator 1 only when its first
          // MMA into it is due, so the drain of accumulator 1 overlaps the tile's first MMAs.
          const bool pair = use0 && use1;
          if (use0 && !mbar_wait(c, &sc->tempty[0], aph[0] ^ 1u, 7)) break;
          if (use1 && !pair && !mbar_wait(c, &sc->tempty[1], aph[1] ^ 1u, 7)) break;
          tc_fence_after();
          const unsigned d0 = tmem + (use0 ? 0u : (unsigned)kAccCols);     // accumulator of rows 0..127
          for (int kb = 0; kb < kblocks; ++kb) {
            if (!mbar_wait(c, &sc->full[stage], par, 8)) { fail = true; break; }
            tc_fence_after();
            fence_async_proxy_smem();                      // cp.async-written rows -> tensor core reads
            const unsigned long long ad = desc0 + stage * (unsigned)(kSB / 16), bd = ad + (unsigned)(kBOff / 16);
#pragma unroll
            for (int k4 = 0; k4 < kBlockK / 16; ++k4)      // +32 bytes along K per step (>>4 = 2)
              tc_mma_bf16(d0, ad + 2ull * k4, bd + 2ull * k4, kIdesc, (kb | k4) ? 1u : 0u);
            if (pair) {                                    // rows 128..255 against the same weight tile
              if (kb == 0) {                               // accumulator 1 is needed from here on
                if (!mbar_wait(c, &sc->tempty[1], aph[1] ^ 1u, 7)) { fail = true; break; }
                tc_fence_after();
              }
              const unsigned long long ad1 = ad + (unsigned)(kAHalfBytes / 16);
#pragma unroll
              for (int k4 = 0; k4 < kBlockK / 16; ++k4)
                tc_mma_bf16(tmem + (unsigned)kAccCols, ad1 + 2ull * k4, bd + 2ull * k4, kIdesc, (kb | k4) ? 1u : 0u);
            }
            tc_commit(&sc->empty[stage]);                  // frees the stage when the MMAs retire
            if (++stage == kNS) { stage = 0; par ^= 1u; }
          }
          if (fail) break;
          if (use0) tc_commit(&sc->tfull[0]);              // accumulator(s) complete
          if (use1) tc_commit(&sc->tfull[1]);
          if (use0) aph[0] ^= 1u;
          if (use1) aph[1] ^= 1u;
        }
        mbar_arrive(&sc->iempty[islot]);
        if (++islot == kRing) { islot = 0; iph ^= 1u; }
      }
    }
    __syncwarp();
  } else if (warp >= 4 && warp < 4 + kGatherThreads / 32) {
    gather_regs();
    // ============================================================ gather warps (cp.async)
    // Rows of a gate/up tile are scattered tokens: row r of the tile is token
    // sorted_to_flat[row0 + r] / k.  Adjacent lanes copy one row slice (16 bytes each)
    // into the swizzled layout the tensor core reads.
    const int gt = threadIdx.x - 128;
    constexpr int kCpr = kRowBytes / 16;                  // 16-byte chunks per row slice
    constexpr int kRowsPerPass = kGatherThreads / kCpr;   // rows covered by one cp.async per thread
    constexpr int kPasses = Ring<kMode>::kARows / kRowsPerPass;
    const int chunk = gt % kCpr, rbase = gt / kCpr;       // rows rbase + kRowsPerPass * j
    // the swizzle XORs the 16-byte chunk index with the row's place in its 8-row group, which is the same in every pass
    static_assert(kRowsPerPass % 8 == 0 && kRowBytes == 128, "");
    const unsigned stages0 = smem_u32(stages), full0 = smem_u32(&sc->full[0]);
    const unsigned dst0 = stages0 + rbase * kRowBytes + ((chunk ^ (rbase & 7)) << 4);
    ended = false;
    int islot = 0;
    unsigned iph = 0, stage = 0, gmask = 0, rmask = 0, kiter = 0;      // kiter: k-blocks of all GEMM tiles so far
    while (true) {
      if (!__all_sync(0xffffffffu, mbar_wait(c, &sc->ifull[islot], iph, 13))) break;
      const int kind = sc->info[islot].kind;
      const int kblocks = sc->info[islot].kblocks;
      const int rows = sc->info[islot].rows, row0 = sc->info[islot].row0, slot = sc->info[islot].slot;
      __syncwarp();
      if (kind == kEnd) { ended = true; break; }
      if (lane == 0) mbar_arrive(&sc->iempty[islot]);
      if (++islot == kRing) { islot = 0; iph ^= 1u; }
      if (kind == kCombine) continue;
      const OpDev* op = &args.ops[slot];
      const RowBoxes rb = row_boxes<kMode>(rows);
      const bool fromx = kind == kGateUpDirect;           // masked layout: rows of x, otherwise of the packed intermediate
      const CUtensorMap* tma = rb.rows == 8    ? (fromx ? &op->tm_x8 : &op->tm_a8)
                               : rb.rows == 32 ? (fromx ? &op->tm_x32 : &op->tm_a32)
                               : rb.rows == 128 ? (fromx ? &op->tm_x128 : &op->tm_a128) : (fromx ? &op->tm_x256 : &op->tm_a256);
      if (kind != kGateUp && !kSmall) {   // consecutive rows, the smallest box that holds them
        bool fail = false;
        if (warp == 4 && elect_one()) {
          for (int kb = 0, s = (int)stage; kb < kblocks; ++kb) {
            if (!mbar_wait(c, &sc->goR[s], (rmask >> s) & 1u, 32)) { fail = true; break; }
            rmask ^= 1u << s;
            single_issue_rows(full0 + s * 8u, kb * kKb, stages0 + s * (unsigned)kSB, tma, row0, (unsigned)rb.boxes);
            if (++s == kNS) s = 0;
          }
        }
        if (__any_sync(0xffffffffu, fail)) break;
        kiter += (unsigned)kblocks;
        stage = kiter % (unsigned)kNS;
        continue;
      }
      // a paired op's gather list also holds rows of its partner, tagged with their slot: those come from
      // the partner's activations
      const bool paired = op->paired != 0;
      const OpDev* pop = paired ? &args.ops[op->partner] : op;
      const unsigned char* X = static_cast<const unsigned char*>(op->x) + chunk * 16;
      const unsigned char* Xp = static_cast<const unsigned char*>(pop->x) + chunk * 16;
      const size_t pitch = (size_t)args.H * kEl;
      const int n_gather = kind == kGateUp ? rows : 0;
      const unsigned char* src[kPasses];                  // this thread's 16 bytes of the row's first k-block
      const int n_rows = op->n_rows, n_rows_p = pop->n_rows;
      const int own_tag = paired ? slot_of(&args, slot) : 0, partner_tag = paired ? slot_of(&args, op->partner) : 0;
      bool bad = false;
#pragma unroll
      for (int j = 0; j < kPasses; ++j) {
        const int r = rbase + kRowsPerPass * j;
        const int v = r < n_gather ? op->gather_list[row0 + r] : 0;
        const int tag = v >> kRowSlotShift, flat = v & kRowFlatMask;
        const bool theirs = tag != own_tag;
        // an index the plan never wrote is reported below and its row is skipped
        const bool in_range = v >= 0 && (tag == own_tag || tag == partner_tag) && flat < (theirs ? n_rows_p : n_rows);
        bad |= r < n_gather && !in_range;
        src[j] = r < n_gather && in_range ? (theirs ? Xp : X) + (size_t)(flat / args.k) * pitch : nullptr;
      }
      if (bad) report(c.st, MOE_EBOUNDS, slot_of(&args, slot), row0, rows, 0);
      // a small e4m3 tile: the scale of token gt of every k-block
      const float* sx = nullptr;
      if (kSmall && gt < rows) {
        if (kind == kGateUp) {
          const int v = op->gather_list[row0 + gt];
          const int tag = v >> kRowSlotShift, flat = v & kRowFlatMask;
          const OpDev* from = tag != own_tag && tag == partner_tag ? pop : op;
          const bool in_range = v >= 0 && (tag == own_tag || from != op) && flat < from->n_rows;   // reported above if not
          sx = from->x_scale + (size_t)(in_range ? flat / args.k : 0) * (args.H / 128);
        } else {
          sx = kind == kDown ? op->a_scale + (size_t)(row0 + gt) * (args.I / 128) : op->x_scale + (size_t)(row0 + gt) * (args.H / 128);
        }
      }
      unsigned scale_at = 0;
      if constexpr (kSmall) scale_at = smem_u32(sc->f8.scale) + (unsigned)scale_index(gt & 63) * 4u;
      bool fail = false;
      for (int kb = 0; kb < kblocks; ++kb, ++kiter) {
        if (!__all_sync(0xffffffffu, mbar_wait(c, &sc->goA[stage], (gmask >> stage) & 1u, 14))) { fail = true; break; }
        gmask ^= 1u << stage;
        if (kSmall && kind != kGateUp && warp == 4 && elect_one())
          single_issue_rows(full0 + stage * 8u, kb * kKb, stages0 + stage * (unsigned)kSB, tma, row0, (unsigned)rb.boxes);
        if (kSmall && sx) cp_async_4(scale_at + (kiter & 15u) * 256u, sx + kb);
        const unsigned dst = dst0 + stage * (unsigned)kSB;
        const auto copy_row = [&](int j) {
          if (src[j]) cp_async_16(dst + j * (kRowsPerPass * kRowBytes), src[j] + (size_t)kb * kRowBytes);
        };
        copy_row(0);
        if (!kSmall || n_gather > kRowsPerPass) {        // most small tiles need one pass
#pragma unroll
          for (int j = 1; j < kPasses; ++j) copy_row(j);
        }
        cp_async_arrive_noinc(&sc->full[stage]);
        if (++stage == kNS) stage = 0;
      }
      if (fail) break;
    }
    cp_async_wait_all();
  } else if (warp == 2) {
    control_regs();
    // ============================================================ committer
    // Publishes a tile once all epilogue threads have arrived on the tile's barrier: the
    // barrier orders their stores before this warp's fence and release (cumulativity).
    ended = false;
    int islot = 0;
    unsigned iph = 0;
    while (true) {
      if (!__all_sync(0xffffffffu, mbar_wait(c, &sc->ifull[islot], iph, 16))) break;
      TileInfo ti;
      if (lane == 0) ti = sc->info[islot];
      const int kind = __shfl_sync(0xffffffffu, lane == 0 ? ti.kind : 0, 0);
      if (kind == kEnd) { ended = true; break; }
      if (!__all_sync(0xffffffffu, mbar_wait(c, &sc->done[islot], iph, 17))) break;
      if (lane == 0) {
        commit_tile<true>(c, rh, ti, watched);
        mbar_arrive(&sc->iempty[islot]);
      }
      __syncwarp();
      if (++islot == kRing) { islot = 0; iph ^= 1u; }
    }
  } else if (warp >= 8) {
    epilogue_regs();
    // ============================================================ epilogue (8 warps)
    // Warp w may read TMEM lanes 32 (w % 4) .. +31, i.e. accumulator rows of that quadrant.
    // The two warps of a quadrant split the columns of every accumulator the tile used.
    const int q = warp & 3;
    const int half = (warp - 8) >> 2;             // which half of the columns
    const int etid = threadIdx.x - 256;           // 0..255
    int islot = 0;
    unsigned iph = 0, aph[2] = {0, 0}, eph = 0, xph = 0, kseq = 0;
    AccUse accs;
    ended = false;
    unsigned char* scratch = sc->epi_scratch[warp - 8];
    const int srow = lane >> 2, schunk = lane & 3;          // this lane's part of a store
    while (true) {
      if (!__all_sync(0xffffffffu, mbar_wait_inline(c, &sc->ifull[islot], iph, 9))) break;
      const TileInfo ti = sc->info[islot];
      if (ti.kind == kEnd) { ended = true; break; }
      OpDev* op = &args.ops[ti.slot];
      bool ok = true;
      if (ti.kind == kCombine) {
        if constexpr (kSmall) combine_tokens_called(op, ti.row0, ti.row0 + ti.rows, args.k, args.H, etid, 256);
        else combine_tokens(op, ti.row0, ti.row0 + ti.rows, 0, args.H / 8, args.k, args.H, etid, 256, CombineNow{});
      } else if constexpr (kSmall) {
        ok = ti.rows <= 32 ? epilogue_fp8_small<32>(c, sc, op, ti, tmem, warp, lane, eph, xph, kseq)
                           : epilogue_fp8_small<64>(c, sc, op, ti, tmem, warp, lane, eph, xph, kseq);
      } else if constexpr (kFp8) {
        ok = epilogue_fp8(c, sc, op, ti, tmem, warp, lane, eph, xph);
      } else {
        bool use[2];
        accs.take(ti.rows, use[0], use[1]);
        const bool pair = use[0] && use[1];
        const bool g1 = ti.kind != kDown;
        const int passes = (g1 ? kTileN1 : kTileN2) / 64;      // 32-column passes per warp
        const size_t pitch = (size_t)(g1 ? args.I : args.H) * 2;
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          if (!use[b]) continue;
          ok = __all_sync(0xffffffffu, mbar_wait_inline(c, &sc->tfull[b], aph[b], 10));
          if (!ok) break;
          aph[b] ^= 1u;
          tc_fence_after();
          const int rbase = pair ? b * kTileM : 0;               // first tile row of this accumulator
          const int nrows = min(ti.rows - rbase, kTileM);
          if (q * 32 < nrows) {
            // 32 output columns (64 bytes of bf16) per pass.  Each lane owns one accumulator
            // row; the warp transposes the pass through its shared-memory scratch so that a
            // store instruction writes 8 rows x 64 contiguous bytes instead of 32 x 16.
            const unsigned taddr = tmem + (unsigned)b * kAccCols + ((unsigned)(q * 32) << 16);
            unsigned char* out = reinterpret_cast<unsigned char*>(g1 ? (void*)op->A : (void*)op->D) +
                                 (size_t)(ti.row0 + rbase + q * 32) * pitch +
                                 (size_t)ti.n * (g1 ? kTileN1 : kTileN2) * 2;
            const int rows_here = min(32, nrows - q * 32);
            // The TMEM load of pass p+1 is issued as soon as pass p has been converted, so its
            // latency hides behind the transpose and the stores of pass p.
            unsigned g[32], u[32];
            tc_ld32(taddr + (half * passes) * 32 + (g1 ? 0 : 0), g);
            if (g1) tc_ld32(taddr + 128 + (half * passes) * 32, u);
#pragma unroll 1
            for (int p = 0; p < passes; ++p) {
              const int pass = half * passes + p;
              uint4 o[4];
              __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(o);
              tc_wait_ld();
              if (g1) {
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                  const float a0 = silu_mul(__uint_as_float(g[2 * i]), __uint_as_float(u[2 * i]));
                  const float a1 = silu_mul(__uint_as_float(g[2 * i + 1]), __uint_as_float(u[2 * i + 1]));
                  oh[i] = __floats2bfloat162_rn(a0, a1);
                }
              } else {
#pragma unroll
                for (int i = 0; i < 16; ++i)
                  oh[i] = __floats2bfloat162_rn(__uint_as_float(g[2 * i]), __uint_as_float(g[2 * i + 1]));
              }
              if (p + 1 < passes) {
                tc_ld32(taddr + (pass + 1) * 32, g);
                if (g1) tc_ld32(taddr + 128 + (pass + 1) * 32, u);
              }
              __syncwarp();                                          // scratch free again
#pragma unroll
              for (int j = 0; j < 4; ++j)     // row `lane`, 16-byte chunk j (XOR keeps banks apart)
                *reinterpret_cast<uint4*>(scratch + lane * 64 + ((j ^ ((lane >> 1) & 3)) << 4)) = o[j];
              __syncwarp();
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const int r = 8 * j + srow;
                const uint4 v4 = *reinterpret_cast<const uint4*>(scratch + r * 64 + ((schunk ^ ((r >> 1) & 3)) << 4));
                if (r < rows_here)
                  *reinterpret_cast<uint4*>(out + (size_t)r * pitch + pass * 64 + schunk * 16) = v4;
              }
            }
          }
          tc_fence_before();
          mbar_arrive(&sc->tempty[b]);            // accumulator may be overwritten
        }
      }
      if (!ok) break;
      mbar_arrive(&sc->done[islot]);              // this thread's part of the tile is stored
      if (++islot == kRing) { islot = 0; iph ^= 1u; }
    }
  }

  // teardown: nothing is claimed any more.  Where a role gave up, asynchronous work may be under way: let it settle.  Then free TMEM
  tc_fence_before();
  if (__syncthreads_or(!ended)) __nanosleep(20000);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

template <int kMode>
static cudaError_t prepare_mode() {
  return cudaFuncSetAttribute(moe_apk_kernel<kMode>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes<kMode>);
}
cudaError_t prepare_run_kernel() {
  cudaError_t e = prepare_mode<kBf16>();
  if (e == cudaSuccess) e = prepare_mode<kF8>();
  return e == cudaSuccess ? prepare_mode<kF8Small>() : e;
}

template <int kMode>
static cudaError_t launch_mode(const RunArgs& args, RunHead* rh, int n_ctas, cudaStream_t stream) {
  return launch_after(moe_apk_kernel<kMode>, n_ctas, kThreads, kSmemBytes<kMode>, stream, args, rh);
}
cudaError_t launch_run(const RunArgs& args, RunHead* rh, int n_ctas, cudaStream_t stream) {
  return args.dtype != MOE_DTYPE_FP8_E4M3            ? launch_mode<kBf16>(args, rh, n_ctas, stream)
         : args.work_rows <= kWorkRowsFp8Small ? launch_mode<kF8Small>(args, rh, n_ctas, stream)
                                               : launch_mode<kF8>(args, rh, n_ctas, stream);
}

}  // namespace moe
