// Persistent whole-pass kernel for passes of at most 48 rows (batch 1, small batches, draft steps): one CTA per SM runs
// every phase of a model pass (embedding or draft-head input, all decoder layers, final norm,
// LM head with greedy choice) with grid barriers between dependent phases.
//
// Why: a 7B verify pass streams 13.2 GB of weights in about 2 ms at HBM speed; one layer is ~60 us.
// Nine separate launches per layer lose a large share of that to launch gaps, ramp-up and tails.
// Here each CTA owns a fixed slab of rows of every weight matrix (N / gridDim rows), and two
// producer threads stream those slabs through a shared-memory ring with TMA tiled loads
// (cp.async.bulk.tensor.2d, 128-byte swizzle, mbarrier transaction counts; one 4 KB box per
// instruction -- separate 512-byte bulk copies were measured to cap a CTA near 12 GB/s).  Weights do not depend on activations, so the
// producer runs ahead across phase boundaries: while the other warps sit in a grid barrier or in
// the attention phase, the ring is already filling with the next GEMM's weights.
//
// Every GEMM input lives in global memory already split into two bf16 planes (hi, lo) and already in
// the swizzled tile layout the tensor core reads, written by the epilogue that produced it, so a
// whole 256-k chunk of activations is one plain bulk copy (tiled TMA loads of 128-byte rows
// were measured to run out of request rate when activations shared them with the weights).  RMSNorm is folded around the GEMM: the producing epilogue stores split(h * gain) and
// the per-row sum of squares; the consuming epilogue multiplies its accumulators by 1/rms(row).
//
// The contraction runs on the 5th-generation tensor cores: one thread issues tcgen05.mma
// (M = 128 weight rows, N = 2 x the pass's rows, in a hi and a lo bf16 plane, K = 16) straight
// from the swizzled shared-memory tiles that TMA wrote, accumulating in tensor memory over the
// whole K range; tcgen05.commit releases ring stages and signals the finished accumulator.  (With
// mma.sync the same loop was bound by the latency of dependent register accumulators at about
// 40 % of the streaming rate.)
//
// Roles inside a CTA (12 warps):
//   warps 0, 3    weight producers, one thread each: both walk the static schedule of (phase, k chunk,
//                 k boxes, m tile) stages; warp 0 loads the even stages, warp 3 the odd ones (a single
//                 thread's mbarrier / TMA issue latency, about 700 cycles per stage, was the limit of the loops)
//   warp 1        stands for the thread block at the grid barriers, and produces activations: per GEMM phase (after the
//                 barrier that makes its input visible) copies the input planes chunk by chunk into shared memory
//   warp 2        one elected thread issues every tcgen05.mma and commit, in schedule order; the warp
//                 also owns the tensor-memory allocation
//   warps 4..11   workers: epilogues out of tensor memory (tcgen05.ld: one weight row per thread),
//                 attention (mma.sync on the 16-bit cache elements), row-wise phases
//
// Every wait (mbarrier, grid barrier) is bounded; when a bound is hit the kernel sets a status bit
// and carries on as if the wait had succeeded, so it always terminates.
#pragma once
#include <type_traits>

#include "ada_areas.h"
#include "ada_kernels.cuh"
#include "ada_ring.h"

namespace ada {

constexpr int kPassThreads = 12 * 32;
constexpr int kNumXWarps = 1;
constexpr int kNumCWarps = 8;                    // workers
constexpr int kFirstWorker = 4;                  // warp index of worker 0
constexpr int kKc = 256;                         // k elements per activation chunk = 4 boxes of 64
constexpr int kBoxK = 64;                        // box width: 64 bf16 = 128 bytes = one swizzle row
constexpr int kStageBytes = 32 * 1024;           // largest ring stage: kb boxes of [box_rows x 64 k], kb = 2 or 4
constexpr int kXBufs = 10;                       // activation buffers at most
// Activation boxes: 64 k of the pass's rows, hi rows then lo rows, padded to a multiple of 8 rows (TP): 256 TP bytes.  A buffer
// takes four boxes up to 40 rows, two beyond; as many buffers as fit the area are in flight.  (A stage of weights has no more
// boxes than a buffer, and stages are what the issuing thread's time goes into: 7B, 30 rows, 3500 us a pass with two boxes,
// 3263 with four.)
constexpr int kPassCtasMax = 160;                // CTAs at most
constexpr int kPassRowsMax = 48;                 // rows of a pass at most
constexpr int kXBytes = 80 * 1024;               // the buffers' area
__host__ __device__ constexpr int xbuf_boxes(int TP) { return TP <= 40 ? 4 : 2; }
__host__ __device__ constexpr int xbuf_bytes(int TP) { return xbuf_boxes(TP) * TP * 256; }
__host__ __device__ constexpr int xbuf_count(int TP) { return xbuf_bytes(TP) * kXBufs <= kXBytes ? kXBufs : kXBytes / xbuf_bytes(TP); }
// Tensor memory.  The tensor core drops what lies below the last bit of an accumulator at every addition, so an accumulator
// takes one section of K only (see Slab::per): two places of 2 TP columns per m tile take turns, and while the products fill
// one, the workers add the other to the sums so far (rounded to nearest), TP columns per m tile from kTmemSums on.  Two layers
// of 7B width, features of decode rows against 64-bit sums: 1.1e-5 off with one accumulator over K, 6.2e-6 so (7.0e-6 in the
// multi-row kernels, whose K splits are of up to 1365 k).  It costs 2 % of a pass (7B, 11 rows at context 3801: 4.95 -> 5.03 ms a block).
constexpr int kTmemCols = 512;
__host__ __device__ constexpr uint32_t acc_cols(uint32_t TP) { return (2 * TP + 31) & ~31u; }
constexpr uint32_t kTmemSums = 384;
static_assert(2 * 2 * acc_cols(kPassRowsMax) <= kTmemSums && kTmemSums + 2 * kPassRowsMax <= kTmemCols, "tensor memory");
constexpr int kRedBytes = (kPassRowsMax / 8) * 128 * 16;
constexpr int kMiscBytes = 6144;                 // mbarriers and small per-CTA arrays
// attention scratch lives where the activation buffers and the reduction buffer are (both idle
// during the attention phase); the ring is NOT reused: the producer keeps filling it meanwhile
constexpr int kAttnLoopBytes = kKeysAt + kNumCWarps * kKeysWarpBytes;   // q hi, q lo, new k, v rows; per warp 16 keys and 16 values
constexpr int kPassMaxSplits = 32;                // cache splits of a sequence at most (its split size is at least capacity / 32)
constexpr int kPartRow = 136;   // floats per row of a warp's partial result: 128 sums, m, l, padded so that a half-warp's fragment stores (4 rows x 4 column pairs) fall into 32 different banks
constexpr int kAttnPartBytes = 8 * 16 * kPartRow * 4;   // per-warp partial results
constexpr int kAttnBytes = kAttnPartBytes > kAttnLoopBytes ? kAttnPartBytes : kAttnLoopBytes;
// (a tensor-core read of 128 tile rows may run a few KB past the last ring stage: the areas below follow the ring)
static_assert(kAttnBytes <= kXBytes, "the attention scratch must not reach the area the pair's CTA writes");
constexpr int kScratchBytes = kXBytes + kRedBytes;
constexpr int kPassSmemBytes = 1024 + kRingBytes + kMiscBytes + kScratchBytes;   // 1 KB to align the ring
static_assert(kPassSmemBytes <= 227 * 1024, "shared memory budget");
constexpr int kSsStride = 256;   // CTAs at most; pairs of CTAs, three partials each (ss_slots)
// Partial sums of squares that a slab leaves per pass row: of its columns in groups of 32, the first two groups' sum and, where a
// slab has more than 64 columns, the third and the fourth, which are added to it one after the other.  A row's sum is made in the
// same order whatever phase or pass leaves it: another order moves the last bit of the row's scale, and with it 16-bit cache
// elements.  (Against trees over 64 columns and one partial for each: 7B verify of 5 rows 2659 -> 2671 us, 18 rows 2840 -> 2854,
// middle model 18 rows 785 -> 789.)
__host__ __device__ constexpr int ss_slots(int segs) { return segs > 1 ? 3 : 1; }
constexpr int kStatTimeout = 4;
constexpr unsigned kSpinLimit = 1u << 22;

struct LayerPtrs {
  const __nv_bfloat16 *wq, *wk, *wv, *wo, *wg, *wu, *wd, *na, *nm;
};

// Tensor maps (CUtensorMap, 128 bytes each) live in a device array, in this order:
//   7 per target layer (wq wk wv wo w_gate w_up w_down), 7 for the draft head's layer, then eagle_fc, lm_head.
// Dims {K, N}, box {64, rows of one m tile of that matrix's slabs}, 128-byte swizzle.
struct alignas(64) TensorMap128 {
  unsigned long long opaque[16];
};
// The row list of the pass in shared memory: the grid barriers' acquires empty level 1, so every phase that went through
// global memory for a position or a token paid a level-2 round trip per lookup.  Target pass: read from the Pass once.
// Draft steps: made here from the sequences' states, so that all steps run in one launch.
struct PassRows {
  int T, lmT, TP;                       // TP: rows of the activation tiles, T rounded up to a multiple of 8
  int seq[kPassRowsMax], pos[kPassRowsMax], tok[kPassRowsMax], out[kPassRowsMax], lm_row[kPassRowsMax], lm_out[kPassRowsMax];
  int choice[kPassRowsMax];             // target pass: the greedy choice after each row (CTA 0)
  // attention: the sequences that have rows
  int nseq, nitems;                     // items: (head, cache split) of every sequence
  int s_b[kMaxBatch], s_row0[kMaxBatch], s_rows[kMaxBatch], s_pos0[kMaxBatch], s_chunk[kMaxBatch], s_nsp[kMaxBatch];
  int s_item0[kMaxBatch + 1], s_part0[kMaxBatch];
  // draft steps: per sequence its draft length, pending position, first catch-up position, split size and newest draft token
  int n[kMaxBatch], j[kMaxBatch], p0[kMaxBatch], chunk[kMaxBatch], cur[kMaxBatch];
  float lp, cum;                        // log-probability of the newest token, of the draft (stopping rule)
};
enum { MAP_WQ = 0, MAP_WK, MAP_WV, MAP_WO, MAP_WG, MAP_WU, MAP_WD };

struct PassParams {
  const Pass *pass;            // prompt: the rows
  const TensorMap128 *maps;    // device array, see above
  int map_layer0;              // index of the first map of this pass's first layer
  int map_fc, map_lm;
  const LayerPtrs *layers;     // device array
  int n_layers;                // layers of this pass (target: L, draft head: 1)
  int cache_layers;            // layers in the KV pool (stride)
  int d, H, hd, F, V;
  float eps;
  const __nv_bfloat16 *embed, *final_norm;
  int mode;                    // 0 target pass over the pending tokens and drafts, 1 draft-head steps step0 .. (longest draft length) - 1
  int prompt;                  // 1: the rows of `pass` are a short prompt of one sequence (mode 0: greedy choice after the last
                               // row; mode 1: the draft head over its rows, no LM head)
  int step0;                   // draft: first step of this launch (0: catch-up rows of the one sequence)
  SeqState *st; int B;         // lengths and draft lengths of the sequences
  int *tok; int tok_stride;    // committed tokens, and positions between two sequences in tok and feat
  const int *draft;            // target pass: draft tokens [seq][nmax]
  int only_seq;                // target pass: the one sequence that takes part (-1: all)
  int accept;                  // target pass: accept afterwards (ada_step); results to
  int *acc_out, *emit_out, *nemit_out;
  float ddd_thr;               // < 0: the draft grows while its running log-probability is at least this (one sequence)
  // activations: fp32 residual stream and qkv; bf16 (hi, lo) planes of every GEMM input
  float *h, *qkv;              // [rows][d], [rows][3d]
  // each input is stored as tensor-core-ready tiles (see xstore): per 64 k one box of 2 TP rows
  __nv_bfloat16 *xa;              // K = d    h * gain of the norm that follows
  __nv_bfloat16 *at;              // K = d    attention output
  __nv_bfloat16 *ac;              // K = F    SwiGLU output
  __nv_bfloat16 *fc;              // K = 2d   draft-head input [e ; f]
  float *ss_part;              // [rows][kSsStride] partial sums of squares of h, see ss_slots
  float *feat; int cap;        // target features by position [seq][cap][d]
  float *dfeat; int nmax;      // draft features [seq][nmax][d]
  // attention
  const float2 *rope;
  __nv_bfloat16 *kpool, *vpool;
  const int *page_table; int pages_per_seq, page_size;
  float *attn_part;            // partial results per (sequence, head, split) and row of the sequence: [rows][hd] sums, then [rows] (m, l)
  int max_splits;              // attention splits of a sequence at most
  size_t attn_part_floats;     // where the (m, l) pairs start
  int *attn_cnt;               // [sequences][H] arrival counters (zero between passes)
  // LM head
  float4 *amax;                // [grid][kPassRowsMax]
  float *logits;               // optional [slot][V]
  int *tok_out; float2 *top_out; const int *forced;
  float *lp_out;               // optional [slot]: log softmax probability of the token written to tok_out
  float *tok_logit;            // scratch [slot]: logit of a forced token (lp_out with forced tokens)
  // sync
  unsigned *gbar;              // [0] grid barrier count, [16] CTAs that have left: both zero between launches
  Counters *cnt;
  int *steps_out;              // optional: the draft steps that the launch ran
  unsigned long long *phase_ns;  // optional [512]: [0] = start, [i+1] = time CTA 0 left barrier i (globaltimer)
};

// ---------------------------------------------------------------------------------- primitives

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
// ... without the arrival: bytes that the phase awaits beyond those of the arrival to come
__device__ __forceinline__ void mbar_expect_more(uint64_t *bar, unsigned bytes) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t *bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded wait; on give-up records a status bit and returns
// (*abort_flag is a per-CTA shared word: once any wait of the CTA has given up, later waits do not spin)
// non-blocking test of the same condition (cheaper than try_wait when the phase is already complete)
__device__ __forceinline__ bool mbar_test(uint64_t *bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// (the spin is kept out of line: the kernel's phases together exceed the instruction cache, so every
// copy of cold code that is not inlined into them makes the hot part smaller)
__device__ __noinline__ void mbar_spin(uint64_t *bar, unsigned parity, Counters *cnt, volatile int *abort_flag,
                                       unsigned limit = kSpinLimit) {
  for (unsigned i = 0; i < limit; ++i) {
    if (mbar_try(bar, parity)) return;
    if (*abort_flag) return;
    if (i > 64) __nanosleep(40);
  }
  *abort_flag = 1;
  atomicOr(&cnt->status, kStatTimeout);
}
__device__ __forceinline__ void mbar_wait(uint64_t *bar, unsigned parity, Counters *cnt, volatile int *abort_flag,
                                          unsigned limit = kSpinLimit) {
  if (mbar_test(bar, parity)) return;
  mbar_spin(bar, parity, cnt, abort_flag, limit);
}
// Where a wait gave up, copies into shared memory (this thread block's, or its peer's sums) may still be under way: the thread
// block stays for a millisecond, in which they land.  Called once, at a kernel's end.  (The compiler would otherwise write the loop out in
// 16 KB.)
__device__ __forceinline__ void await_copies(volatile int *abort_flag) {
  if (*abort_flag)
#pragma unroll 1
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);
}
__device__ __forceinline__ void bulk_g2s_hint(void *dst, const void *src, unsigned bytes, uint64_t *bar, uint64_t pol) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
               : "memory");
}
// Bulk copies read global memory through the async proxy: what this kernel's ordinary stores have written to it, here or (seen
// through a barrier) in another thread block, is ordered before the copies that this thread issues afterwards.  One fence a phase
// and reading thread: 0.2 to 0.5 % of a pass (as much as one by every writer before the barrier).
__device__ __forceinline__ void fence_global_copies() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
__device__ __forceinline__ void tma_load_2d(void *dst, const TensorMap128 *map, int x, int y, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}
// The same load with a level-2 eviction policy.  Weights are read once per pass: with evict-first they do not push the
// data that is read again (activation planes, partial sums, the cache) out of level 2.
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void tma_load_2d_hint(void *dst, const TensorMap128 *map, int x, int y, uint64_t *bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(smem_u32(bar)), "l"(pol)
      : "memory");
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}
// warp-level products on 16-bit halves with fp32 sums (attention): c[16 x 8] += a[16 x 16] b[16 x 8]
__device__ __forceinline__ void mma_f16_k16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                            uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// ---- tcgen05 (5th generation tensor cores, accumulators in tensor memory)
__device__ __forceinline__ void tmem_alloc(uint32_t *smem_slot, uint32_t ncols) {   // whole warp
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_slot)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {      // whole warp
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// K-major operand tile in shared memory, 128-byte swizzle: rows 128 B apart, 8-row groups 1024 B apart
__device__ __forceinline__ uint64_t umma_desc(uint32_t smem_addr) {
  return (uint64_t)((smem_addr >> 4) & 0x3FFFu) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// D(f32, tensor memory) (+)= A(bf16, smem) * B(bf16, smem)^T, M = 128 or 64, K = 16
// (M = 64 for slabs of at most 64 rows: the tensor core then reads half as much of the A tile)
__host__ __device__ constexpr uint32_t umma_idesc_mn(uint32_t m, uint32_t n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((m >> 4) << 24);
}
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// true in exactly one lane of the (converged) warp
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n .reg .pred P;\n elect.sync _|P, 0xffffffff;\n selp.b32 %0, 1, 0, P;\n}" : "=r"(pred));
  return pred != 0;
}
// arrive on an mbarrier once every tcgen05.mma issued so far by this thread has completed
__device__ __forceinline__ void umma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tmem_ld8_issue(uint32_t taddr, uint32_t (&r)[8]) {   // (valid after tcgen05.wait::ld)
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
// Sums of eight pass rows: those so far (where there are any, `more`) plus the accumulator's hi and lo parts, 8 + 8 columns of this
// thread's tensor-memory lane.
__device__ __forceinline__ void tmem_sum8(bool more, uint32_t sums, uint32_t hi, uint32_t lo, float (&v)[8]) {
  uint32_t a[8], b[8], c[8];
  tmem_ld8_issue(hi, a);
  tmem_ld8_issue(lo, b);
  if (more) {   // (warp-uniform)
    tmem_ld8_issue(sums, c);
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) c[i] = 0u;
  }
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(c[i]) + (__uint_as_float(a[i]) + __uint_as_float(b[i]));
}
__device__ __forceinline__ void named_bar(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// ---- thread-block cluster of two CTAs: the peer's shared memory and its mbarriers are addressable
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t peer_addr(const void *own_smem, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(own_smem)), "r"(rank));
  return r;
}
// 16 bytes into the peer's shared memory, counted on a barrier of the peer
__device__ __forceinline__ void st_async_peer(uint32_t addr, uint32_t bar, float a, float b, float c, float d) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr), "f"(a),
               "f"(b), "f"(c), "f"(d), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive_peer(uint32_t addr) {   // releases this CTA's earlier writes to the peer
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
__device__ __forceinline__ bool mbar_try_cluster(uint64_t *bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void cluster_sync_all() {   // every thread of both CTAs
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Activation tiles in global memory: for every 64 k one box of 2 TP rows x 128 bytes (rows 0 .. TP - 1 the hi plane of the
// pass rows, rows TP .. 2 TP - 1 the lo plane), with the 16-byte chunk index XORed with (row & 7): exactly what a
// 128-byte-swizzle K-major operand looks like in shared memory, so boxes are copied verbatim.
__device__ __forceinline__ size_t xtile(int TP, int t, int k) {
  const int kk = k & 63;
  return (size_t)(k >> 6) * (TP * 128) + (size_t)t * 64 + ((((kk >> 3) ^ (t & 7)) << 3) | (kk & 7));
}
__device__ __forceinline__ void xstore(__nv_bfloat16 *tiles, int TP, int t, int k, float v) {
  __nv_bfloat16 hi, lo;
  split_bf16(v, hi, lo);
  const size_t o = xtile(TP, t, k);
  tiles[o] = hi;
  tiles[o + TP * 64] = lo;   // row TP + t: same (row & 7)
}

// two neighbouring columns, k even
__device__ __forceinline__ void xstore2(__nv_bfloat16 *tiles, int TP, int t, int k, float x, float y) {
  __nv_bfloat162 hi, lo;
  split_bf16(x, hi.x, lo.x);
  split_bf16(y, hi.y, lo.y);
  const size_t o = xtile(TP, t, k);
  *reinterpret_cast<__nv_bfloat162 *>(tiles + o) = hi;
  *reinterpret_cast<__nv_bfloat162 *>(tiles + o + TP * 64) = lo;
}
__device__ __forceinline__ void xstore4(__nv_bfloat16 *tiles, int TP, int t, int k, float4 v) {   // k a multiple of 4
  __nv_bfloat16 hi[4], lo[4];
  split_bf16(v.x, hi[0], lo[0]); split_bf16(v.y, hi[1], lo[1]); split_bf16(v.z, hi[2], lo[2]); split_bf16(v.w, hi[3], lo[3]);
  const size_t o = xtile(TP, t, k);
  uint2 ph, pl;
  ph.x = (uint32_t)__bfloat16_as_ushort(hi[0]) | ((uint32_t)__bfloat16_as_ushort(hi[1]) << 16);
  ph.y = (uint32_t)__bfloat16_as_ushort(hi[2]) | ((uint32_t)__bfloat16_as_ushort(hi[3]) << 16);
  pl.x = (uint32_t)__bfloat16_as_ushort(lo[0]) | ((uint32_t)__bfloat16_as_ushort(lo[1]) << 16);
  pl.y = (uint32_t)__bfloat16_as_ushort(lo[2]) | ((uint32_t)__bfloat16_as_ushort(lo[3]) << 16);
  *reinterpret_cast<uint2 *>(tiles + o) = ph;
  *reinterpret_cast<uint2 *>(tiles + o + TP * 64) = pl;
}

// ---------------------------------------------------------------------------------- GEMM phases

enum { EPI_STORE_QKV = 0, EPI_RESID_H = 1, EPI_SWIGLU_ACT = 2, EPI_ARGMAX_LM = 3, EPI_STORE_H = 4 };

struct GemmDesc {
  int wmap[3];                      // tensor maps of the weight matrices (segments, or gate / up): index inside a layer's seven
  int nseg, Nseg, K, epi;
  const __nv_bfloat16 *xt;          // input tiles (xstore layout)
  int scale_inv_rms;                // accumulators are multiplied by 1/rms(row) of h (input was h * gain)
  int lm_rows;                      // input rows are pass->lm_row[i] (draft LM head)
  int split_k;                      // this GEMM may be cut along K as well (outputs of d columns: O, down, fc)
};

// Phase list.  Target: EMBED, then per layer QKV, ATTN, O, GATEUP, DOWN, then LM.
// Draft: EAGLE_IN, FC, then the same five, then LM (optional).
enum { PH_EMBED = 0, PH_EAGLE_IN, PH_FC, PH_QKV, PH_ATTN, PH_O, PH_GATEUP, PH_DOWN, PH_LM };

__device__ __forceinline__ int phase_count(const PassParams &p) {
  return (p.mode == 0 ? 1 : 2) + 5 * p.n_layers + (p.mode == 1 && p.prompt ? 0 : 1);
}
__device__ __forceinline__ int phase_kind(const PassParams &p, int idx, int &layer) {
  layer = 0;
  const int pre = p.mode == 0 ? 1 : 2;
  if (idx < pre) return p.mode == 0 ? PH_EMBED : (idx == 0 ? PH_EAGLE_IN : PH_FC);
  const int i = idx - pre;
  if (i < 5 * p.n_layers) {
    layer = i / 5;
    return PH_QKV + (i % 5);
  }
  return PH_LM;
}

__device__ __forceinline__ bool is_gemm(int kind) { return kind != PH_EMBED && kind != PH_EAGLE_IN && kind != PH_ATTN; }

__device__ __forceinline__ void make_gemm(const PassParams &p, int kind, GemmDesc &g) {
  g.nseg = 1; g.scale_inv_rms = 0; g.lm_rows = 0; g.split_k = 0;
  g.wmap[1] = g.wmap[2] = -1;
  switch (kind) {
    case PH_FC:
      g.wmap[0] = p.map_fc; g.Nseg = p.d; g.K = 2 * p.d; g.epi = EPI_STORE_H; g.split_k = 1; g.xt = p.fc;
      break;
    case PH_QKV:
      g.wmap[0] = MAP_WQ; g.wmap[1] = MAP_WK; g.wmap[2] = MAP_WV; g.nseg = 3; g.Nseg = p.d; g.K = p.d;
      g.epi = EPI_STORE_QKV; g.xt = p.xa; g.scale_inv_rms = 1;
      break;
    case PH_O:
      g.wmap[0] = MAP_WO; g.Nseg = p.d; g.K = p.d; g.epi = EPI_RESID_H; g.split_k = 1; g.xt = p.at;
      break;
    case PH_GATEUP:
      g.wmap[0] = MAP_WG; g.wmap[1] = MAP_WU; g.Nseg = p.F; g.K = p.d; g.epi = EPI_SWIGLU_ACT; g.xt = p.xa; g.scale_inv_rms = 1;
      break;
    case PH_DOWN:
      g.wmap[0] = MAP_WD; g.Nseg = p.d; g.K = p.F; g.epi = EPI_RESID_H; g.split_k = 1; g.xt = p.ac;
      break;
    default:   // PH_LM
      g.wmap[0] = p.map_lm; g.Nseg = p.V; g.K = p.d; g.epi = EPI_ARGMAX_LM; g.xt = p.xa;
      if (p.mode == 0) g.scale_inv_rms = 1;
      g.lm_rows = p.mode == 1 || p.prompt;
  }
}
// First tensor map of the layer a phase's map indices count from.
__device__ __forceinline__ int map_base(const PassParams &p, int kind, int layer) {
  return kind == PH_FC || kind == PH_LM ? 0 : p.map_layer0 + 7 * layer;
}
// Norm whose gain goes into the planes a phase writes (split(h * gain)); null = none: the next layer's, or the final one;
// the draft head has none after its layer.
__device__ __forceinline__ const __nv_bfloat16 *gain_after(const PassParams &p, int kind, int layer) {
  if (kind == PH_FC) return p.layers[layer].na;
  if (kind == PH_O) return p.layers[layer].nm;
  return layer + 1 < p.n_layers ? p.layers[layer + 1].na : (p.mode == 0 ? p.final_norm : nullptr);
}

// Row slab of this CTA.  A GEMM over nseg separate matrices of Nseg rows gives each matrix
// gridDim / nseg CTAs, so a slab never spans two matrices.  The slab is cut into at most two m
// tiles of box_rows <= 128 rows (the tensor map's box height, fixed per matrix at initialisation
// from the same arithmetic); SWIGLU: the two m tiles are the same row range of the gate and of the
// up matrix.  A ring stage holds kb boxes (kb * 64 k) of one m tile.
//
// GEMMs with only d output columns (O, down, the draft head's fc) would leave each CTA a slab of ~28
// rows: the tensor core then spends a whole instruction per 28 x 16 weights and every CTA re-reads the
// whole activation.  They are cut along K too: the two CTAs of a thread-block cluster share a slab of
// twice the rows, each takes one half of K (whole 256-k chunks); they exchange their sums through distributed shared memory and
// each finishes half of the pass rows.
struct Slab {
  int seg;          // matrix (segment) of this CTA
  int r0, rows;     // rows [r0, r0 + rows) inside that matrix
  int mtiles;       // accumulators in use (1 or 2)
  int box_rows;     // rows per m tile = box height of the tensor map
  int region;       // bytes of one box in shared memory (box_rows rounded up to 8, times 128)
  int kb;           // boxes per stage
  int m64;          // 1: M = 64 products (accumulator row i in lane (i % 16) + 32 * (i / 16))
  int ks, kj;       // K splits of this GEMM and this CTA's split
  int c0, c1;       // this CTA's 256-k chunks [c0, c1)
  int rot;          // ... which it walks from c0 + rot, around the end
  int per, nsec;    // chunks per section of K (in the order of the walk), sections
  int group;        // index of the slab (= group of ks CTAs)
  int segs, slabs;  // pieces of 64 columns that cover any slab (one or two), and slabs: a phase that leaves sums of squares leaves
                    // one per pass row and slab, of slabs of two pieces three (ss_slots)
};
__host__ __device__ __forceinline__ int slab_rpc(int Nseg, int nseg, int ncta) {
  const int cps = ncta / nseg;
  return (Nseg + cps - 1) / cps;
}
__host__ __device__ __forceinline__ int slab_box_rows(int rpc, bool swiglu) {
  const int mt = swiglu ? 1 : (rpc + 127) / 128;
  return (rpc + mt - 1) / mt;
}
// K splits for a GEMM of N output columns over K: 2 (the two CTAs of a cluster, which exchange their partial
// sums through distributed shared memory) if each split gets at least one 256-k chunk and a slab stays within
// one m tile (128 rows); else 1
__host__ __device__ __forceinline__ int slab_ksplit(int N, int K, int ncta) {
  const int nchunk = (K + kKc - 1) / kKc;
  const int groups = ncta / 2;
  if (groups < 1 || nchunk < 2) return 1;
  if ((N + groups - 1) / groups > 128) return 1;
  return 2;
}
__device__ __forceinline__ Slab make_slab(const GemmDesc &g, int cta, int ncta) {
  Slab s;
  const bool sw = g.epi == EPI_SWIGLU_ACT;
  const int nchunk = (g.K + kKc - 1) / kKc;
  s.ks = g.split_k ? slab_ksplit(g.Nseg, g.K, ncta) : 1;
  int rpc, li;
  if (s.ks > 1) {
    const int groups = ncta / s.ks;
    s.seg = 0;
    s.group = cta / s.ks;
    s.kj = cta - s.group * s.ks;
    rpc = (g.Nseg + groups - 1) / groups;
    li = s.group;
    const int per = (nchunk + s.ks - 1) / s.ks;
    s.c0 = s.kj * per;
    s.c1 = min(nchunk, s.c0 + per);
    if (s.group >= groups) { s.c0 = s.c1 = 0; li = groups; }   // CTAs beyond the last whole group idle
  } else {
    const int cps = ncta / g.nseg;                  // CTAs per matrix
    s.seg = cta / cps;
    li = cta - s.seg * cps;
    rpc = slab_rpc(g.Nseg, g.nseg, ncta);
    s.kj = 0; s.c0 = 0; s.c1 = nchunk; s.group = cta;
  }
  s.r0 = li * rpc;
  s.rows = (s.seg < g.nseg) ? max(0, min(g.Nseg, s.r0 + rpc) - s.r0) : 0;
  if (s.c1 <= s.c0) s.rows = 0;
  s.segs = (rpc + 63) / 64;
  s.slabs = (g.Nseg + rpc - 1) / rpc;
  s.box_rows = slab_box_rows(rpc, sw);
  s.mtiles = sw ? 2 : ((rpc + 127) / 128);
  if (!sw && s.rows <= s.box_rows) s.mtiles = 1;  // a short last slab may not reach the second tile
  s.region = ((s.box_rows + 7) & ~7) * 128;
  s.kb = s.region <= 8192 ? 4 : 2;   // a stage is at most 32 KB
  s.m64 = s.box_rows <= 64;
  // Four groups of CTAs start a quarter of K apart: all CTAs asking for the same 16 KB of activations at the same moment
  // queue at the few level-2 slices that hold them.  7B, 5 rows: QKV 20.1 -> 19.4 us, gate/up 32.8 -> 31.9 us per layer,
  // verify pass 3167 -> 3112 us; eight starts are no better, and K halves (already two starts) gain nothing.
  s.rot = s.ks == 1 && s.c1 > s.c0 ? ((cta & 3) * (s.c1 - s.c0)) >> 2 : 0;
  // Sections of 512 k, 32 additions to an accumulator; of 256 k where a CTA has 2048 or less, as the K splits of the multi-row
  // kernels are there (512 k throughout: features 4 % further off at d_model 512 and 1 % at 1536).  Of the shape alone: a row's
  // sums do not depend on the rows of its pass.
  const int nch = s.c1 - s.c0;
  s.per = nch <= 8 ? 1 : 2;
  s.nsec = nch <= 8 ? max(1, nch) : (nch + 1) >> 1;
  return s;
}
// A GEMM phase as a CTA sees it, for all layers: made once, in shared memory.  (Every role worked this out again after every
// barrier, 0.8 us of divisions and branches before the first request of a phase went out.)
struct PhaseGemm {
  GemmDesc g;
  Slab s;
};
constexpr int kPhaseGemms = PH_LM - PH_FC + 1;
// Parities of the two accumulator places after a phase of nsec sections, all but the last of which were handed on.
__device__ __forceinline__ uint32_t sections_done(uint32_t sphase, int nsec) {
  return sphase ^ (uint32_t)(((nsec >> 1) & 1) | ((((nsec - 1) >> 1) & 1) << 1));
}
// m tile mi -> weight map index and first row
__device__ __forceinline__ void tile_source(const GemmDesc &g, const Slab &s, int mi, int &map, int &row0) {
  if (g.epi == EPI_SWIGLU_ACT) { map = g.wmap[mi]; row0 = s.r0; }
  else { map = g.wmap[s.seg]; row0 = s.r0 + mi * s.box_rows; }
}

// ---------------------------------------------------------------------------------- grid barrier

// Warp 1 and the eight worker warps (288 threads) take part; the producers' and the issuer's warps do not.  Workers announce
// that their stores are done and later await the release; in between they may do what depends on no other CTA's results of the
// phase.  Warp 1 stands between them and the other CTAs.
__device__ __forceinline__ void named_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
constexpr int kBarThreads = (kNumXWarps + kNumCWarps) * 32;
__device__ __forceinline__ void phase_arrive() { named_arrive(2, kBarThreads); }
__device__ __forceinline__ void phase_await() { named_bar(4, kBarThreads); }

// One thread of the CTA: arrives with release semantics (a named barrier has ordered the other threads' writes before this
// thread; the release makes them visible with the count), polls with acquire loads until `target` arrivals.
__device__ __forceinline__ void grid_wait(unsigned *gbar, Counters *cnt, unsigned target, volatile int *abort_flag,
                                          unsigned limit = kSpinLimit) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(gbar) : "memory");
#pragma unroll 1
  for (unsigned i = 0; i < limit && !*abort_flag; ++i) {
    if (ld_acquire(gbar) >= target) return;
    if ((i & 63) == 63 && (ld_acquire(reinterpret_cast<const unsigned *>(&cnt->status)) & kStatTimeout)) break;
    if (i > 4096) __nanosleep(64);   // a barrier normally completes within a few polls
  }
  *abort_flag = 1;
  atomicOr(&cnt->status, kStatTimeout);
}

// optional fine-grained clock of CTA 0's first consumer lane: 4 stamps per phase after the 512 barrier stamps
__device__ __forceinline__ void stamp(const PassParams &p, int ph, int k, bool on) {
  if (on && p.phase_ns && ph < 500) {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    p.phase_ns[512 + 4 * ph + k] = t;
  }
}

// ---------------------------------------------------------------------------------- row lists

// Attention items of the sequences in s_* (one thread).  A sequence keeps the split size fixed when its prompt was read, in every
// pass and whatever the sequences beside it: the split a key falls in is part of the arithmetic.  (Split sizes chosen for a
// batch's draft step from all its sequences balance the items over the CTAs better, 0.6 % of a block of eight ragged sequences
// of 7B, but then a sequence's draft depends on its batch mates.)
__device__ __noinline__ void pass_items(PassRows *r, int H, int max_splits) {
  int item0 = 0, part0 = 0;
  for (int i = 0; i < r->nseq; ++i) {
    const int nkeys = r->s_pos0[i] + r->s_rows[i];
    r->s_nsp[i] = min(max_splits, (nkeys + r->s_chunk[i] - 1) / r->s_chunk[i]);
    r->s_item0[i] = item0; r->s_part0[i] = part0;
    item0 += H * r->s_nsp[i];
    part0 += H * r->s_nsp[i] * r->s_rows[i];
  }
  r->s_item0[r->nseq] = item0;
  r->nitems = item0;
}

// Stopping rule: the producers and the issuer run ahead of the steps up to the predicted length; past it they await the
// decision on each further step (the workers arrive on the barrier once per step from the predicted length on).
__device__ __noinline__ int await_length(uint64_t *step_bar, unsigned &decisions, const PassRows *rows, Counters *cnt,
                                         volatile int *abort_flag) {
  mbar_wait(step_bar, decisions & 1u, cnt, abort_flag);
  ++decisions;
  return *reinterpret_cast<const volatile int *>(&rows->n[0]);
}

// Rows of draft step `step` (Eq. 2; one thread).  Step 0: the catch-up rows p = p0 .. j - 1 of every sequence, row p pairs
// the target feature of p with the embedding of token p + 1, a sequence's last row feeds the LM head.  Step s >= 1: one row per
// sequence with n > s at position j + s - 1, its token the newest draft token.
__device__ __noinline__ void draft_rows_of_step(PassRows *r, const PassParams &p, int step) {
  int T = 0, ns = 0;
  for (int b = 0; b < p.B; ++b) {
    if (r->n[b] <= step) continue;
    const int first = step == 0 ? r->p0[b] : r->j[b] + step - 1, R = step == 0 ? r->j[b] - first : 1;
    r->s_b[ns] = b; r->s_row0[ns] = T; r->s_rows[ns] = R; r->s_pos0[ns] = first; r->s_chunk[ns] = r->chunk[b];
    for (int i = 0; i < R; ++i, ++T) {
      r->seq[T] = b;
      r->pos[T] = first + i;
      r->tok[T] = step == 0 ? p.tok[(size_t)b * p.tok_stride + first + i + 1] : r->cur[b];
    }
    r->lm_row[ns] = T - 1;
    r->lm_out[ns] = b * p.nmax + step;
    ++ns;
  }
  r->T = T; r->lmT = ns; r->nseq = ns; r->TP = (T + 7) & ~7;
  pass_items(r, p.H, p.max_splits);
}

// Rows of a target pass (Eq. 1; one warp): the pending token of every sequence that takes part, then its draft, positions
// j .. j + n.  A sequence that is full takes no further step.
__device__ __noinline__ void verify_rows(PassRows *r, const PassParams &p, bool record) {
  const int lane = threadIdx.x & 31;
  int R = 0, j = 0, chunk = 0;
  if (lane < p.B && (p.only_seq < 0 || lane == p.only_seq)) {
    const SeqState q = p.st[lane];
    if (q.len >= 1 && q.len + q.n + 1 <= p.cap) { R = q.n + 1; j = q.len - 1; chunk = max(32, q.chunk); }
  }
  int row0 = R;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, row0, o);
    if (lane >= o) row0 += v;
  }
  const int T = __shfl_sync(0xffffffffu, row0, 31);
  row0 -= R;
  const unsigned has = __ballot_sync(0xffffffffu, R > 0);
  if (R > 0) {
    const int i = __popc(has & ((1u << lane) - 1u));
    r->s_b[i] = lane; r->s_row0[i] = row0; r->s_rows[i] = R; r->s_pos0[i] = j; r->s_chunk[i] = chunk;
    if (record) p.st[lane].j_prev = j;
  }
  __syncwarp();
  const int ns = __popc(has);
  for (int t = lane; t < T; t += 32) {
    int i = 0;
    while (i + 1 < ns && t >= r->s_row0[i + 1]) ++i;
    const int b = r->s_b[i], k = t - r->s_row0[i], pos = r->s_pos0[i] + k;
    r->seq[t] = b; r->pos[t] = pos;
    r->tok[t] = k == 0 ? p.tok[(size_t)b * p.tok_stride + pos] : p.draft[b * p.nmax + k - 1];
    r->out[t] = b * (p.nmax + 1) + k;
  }
  if (lane == 0) {
    r->T = r->lmT = T; r->TP = (T + 7) & ~7; r->nseq = ns;
    pass_items(r, p.H, p.max_splits);
  }
}

// First catch-up position of a sequence that takes part in the draft steps of this launch (0 if the launch has no catch-up
// step), -1 for one that does not: no draft asked for, or more rows behind than a pass holds of a sequence.  One that is up
// to date (a second draft from the same state, e.g. after a label pass) computes the row of position j - 1 again -- same
// inputs, same cache row -- because its output yields the first draft token.
__device__ __forceinline__ int draft_first(const PassParams &p, const SeqState &q) {
  const int j = q.len - 1;
  if (q.n <= p.step0 || j < 1) return -1;
  if (p.step0 > 0) return 0;
  const int p0 = q.dlen == j ? j - 1 : q.dlen;
  return j - p0 < 1 || j - p0 > p.nmax + 1 || q.stale ? -1 : p0;
}

// The issuing warp between section sec - 1 of K and section sec, whose place must have been added up.
__device__ __noinline__ void next_section(uint64_t *secfull, uint64_t *secempty, int sec, uint32_t sphase, Counters *cnt, volatile int *abort_flag) {
  if (elect_one()) umma_commit(&secfull[(sec - 1) & 1]);
  __syncwarp();
  if (sec >= 2) {
    mbar_wait(&secempty[sec & 1], ((sphase >> (sec & 1)) ^ ((unsigned)(sec - 2) >> 1)) & 1u, cnt, abort_flag);
    tc_fence_after();
  }
}
// Column of the accumulators at `place` for rows t8 .. t8 + 7 of one m tile (t8 < TP) or of the second one.
__device__ __forceinline__ uint32_t acc_column(uint32_t place, int TP, int t8) {
  return place + (uint32_t)t8 + (t8 < TP ? 0u : acc_cols((uint32_t)TP) - (uint32_t)TP);
}
// All sections of K but the last, one after another under the products of the next (one worker warp; t_end = 0: it has no rows,
// but its arrivals must not run ahead of the sections).  Out of line: models whose K is one section jump over it.
__device__ __noinline__ uint32_t add_sections(uint64_t *secfull, uint64_t *secempty, uint32_t sphase, int nsec, int t_end, int TP,
                                              uint32_t taddr, uint32_t place, uint32_t sums, Counters *cnt, volatile int *abort_flag) {
#pragma unroll 1
  for (int q = 0; q + 1 < nsec; ++q) {
    mbar_wait(&secfull[q & 1], ((sphase >> (q & 1)) ^ ((unsigned)q >> 1)) & 1u, cnt, abort_flag);
    tc_fence_after();
#pragma unroll 1
    for (int t8 = 0; t8 < t_end; t8 += 8) {
      const uint32_t acc = acc_column(taddr + (uint32_t)(q & 1) * place, TP, t8);
      float v[8];
      uint32_t r[8];
      tmem_sum8(q > 0, sums + (uint32_t)t8, acc, acc + (uint32_t)TP, v);
#pragma unroll
      for (int u = 0; u < 8; ++u) r[u] = __float_as_uint(v[u]);
      tmem_st8(sums + (uint32_t)t8, r);
    }
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    tc_fence_before();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(&secempty[q & 1]);
  }
  return sections_done(sphase, nsec);
}

// ---------------------------------------------------------------------------------- the kernel

// PROMPT: the rows are a short prompt (p.prompt); a kernel of its own, for the extra tests cost the decode passes 1 %.
template <bool PROMPT>
__global__ void __launch_bounds__(kPassThreads, 1) k_pass(const __grid_constant__ PassParams p) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cta = blockIdx.x, ncta = gridDim.x;
  // Steps of the launch: the target's one pass, or the draft steps step0 .. the longest draft length (with the stopping
  // rule the length grows while the kernel runs, see `step_bar`).  Every thread reads the states here; CTA 0 changes them
  // after the first grid barrier only.
  int nstep = 0;
  if (PROMPT) {
    nstep = p.pass->T > 0 ? 1 : 0;
  } else if (p.mode == 0) {
    for (int b = 0; b < p.B; ++b) {
      const int len = p.st[b].len, n = p.st[b].n;
      if ((p.only_seq < 0 || b == p.only_seq) && len >= 1 && len + n + 1 <= p.cap) nstep = 1;
    }
    // no sequence takes part: nothing to verify, and accepting reports just that
    if (!nstep && p.accept && cta == 0 && tid < p.B)
      accept_sequence(p.st, p.tok, p.cap, p.tok_stride, nullptr, nullptr, p.nmax, tid, p.cnt, nullptr, 0, p.acc_out, p.emit_out,
                      p.nemit_out, nullptr);
  } else {
    for (int b = 0; b < p.B; ++b) {
      const SeqState q = p.st[b];
      if (draft_first(p, q) < 0) {
        if (q.n > p.step0 && q.len > 1 && cta == 0 && tid == 0) { p.st[b].n = 0; atomicOr(&p.cnt->status, kStatStale); }
        continue;
      }
      nstep = max(nstep, q.n);
    }
  }
  const int first_step = p.mode == 0 || PROMPT ? 0 : p.step0;
  if (!PROMPT && p.steps_out && nstep <= first_step && cta == 0 && tid == 0) *p.steps_out = 0;
  if (nstep <= first_step) return;

  extern __shared__ __align__(128) unsigned char pass_smem[];
  // swizzled TMA boxes need 1024-byte aligned bases
  unsigned char *const smem = pass_smem + ((1024u - (smem_u32(pass_smem) & 1023u)) & 1023u);
  unsigned char *ring = smem;
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kRingBytes);
  uint64_t *full = bars, *empty = bars + kSlots, *xfull = bars + 2 * kSlots, *xempty = bars + 2 * kSlots + kXBufs;
  float *inv_rms = reinterpret_cast<float *>(bars + 2 * kSlots + 2 * kXBufs + 8 + 2 * kNumCWarps);   // [rows] (after the single barriers)
  float *lps = inv_rms + kPassRowsMax;                                             // [8][16] sums of exponentials, for log-probabilities (one sequence)
  int *flag_s = reinterpret_cast<int *>(lps + kNumCWarps * 16);
  volatile int *abort_s = flag_s + 1;
  unsigned char *xbuf = smem + kRingBytes + kMiscBytes;
  float *red = reinterpret_cast<float *>(xbuf + kXBytes);   // [rows / 8][128 threads][4 rows] sums of the K-split pair's other CTA
  Top2 *topw = reinterpret_cast<Top2 *>(red);   // [8][rows] (LM head, which has no pairs)
  static_assert(8 * kPassRowsMax * sizeof(Top2) <= kRedBytes, "room for the warps' candidates");
  static_assert((2 * kSlots + 2 * kXBufs + 8 + 2 * kNumCWarps) * 8 + (kPassRowsMax + kNumCWarps * 16) * 4 + 16 + 4 * kFlight * 4 + sizeof(PassRows) + 8 + kPhaseGemms * sizeof(PhaseGemm) <= kMiscBytes, "misc area");

  uint64_t *accfull = xempty + kXBufs;                     // accumulator of the phase complete
  uint64_t *attn_bar = accfull + 1;                        // attention: per worker warp, its 16 keys and its 16 values have landed
  uint64_t *kbar = attn_bar + 2 * kNumCWarps;                           // K-split pair: the sums of the other CTA are here
  uint64_t *step_bar = kbar + 1;                           // stopping rule: the draft length after a step is decided
  uint64_t *secfull = step_bar + 1, *secempty = secfull + 2;   // the two places of the accumulators: a section of K is complete, has been added up by the eight workers
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(const_cast<int *>(abort_s) + 1);
  uint32_t *st_rec = tmem_slot + 1;   // [2 producers][offsets, ends][kFlight]: records of the stages in flight
  PassRows *rows = reinterpret_cast<PassRows *>(st_rec + 4 * kFlight);
  PhaseGemm *gemms = reinterpret_cast<PhaseGemm *>((reinterpret_cast<uintptr_t>(rows + 1) + 7) & ~(uintptr_t)7);   // by kind, PH_FC first
  if (tid == 0) {
    *abort_s = 0;
    for (int i = 0; i < kSlots; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < kXBufs; ++i) { mbar_init(&xfull[i], 1); mbar_init(&xempty[i], 1); }
    mbar_init(accfull, 1);
    for (int i = 0; i < 2 * kNumCWarps; ++i) mbar_init(attn_bar + i, 1);
    mbar_init(kbar, 1);
    mbar_init(step_bar, 1);
    for (int i = 0; i < 2; ++i) { mbar_init(&secfull[i], 1); mbar_init(&secempty[i], kNumCWarps); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) tmem_alloc(tmem_slot, kTmemCols);
  if (warp == kFirstWorker + 1 && lane < kPhaseGemms) {
    make_gemm(p, PH_FC + lane, gemms[lane].g);
    gemms[lane].s = make_slab(gemms[lane].g, cta, ncta);
  }
  if (warp == kFirstWorker) {
    if (PROMPT) {   // one sequence: groups of 16 rows, and the LM head after the last row only
      const Pass *ps = p.pass;
      const int T = ps->T, b = ps->row_seq[0];
      for (int t = lane; t < T; t += 32) {
        rows->seq[t] = b; rows->pos[t] = ps->row_pos[t]; rows->tok[t] = ps->row_tok[t];
      }
      if (lane < (T + 15) >> 4) {
        rows->s_b[lane] = b; rows->s_row0[lane] = 16 * lane; rows->s_rows[lane] = min(16, T - 16 * lane);
        rows->s_pos0[lane] = ps->row_pos[0] + 16 * lane; rows->s_chunk[lane] = max(32, ps->seq_chunk[b]);
      }
      __syncwarp();
      if (lane == 0) {
        rows->T = T; rows->TP = (T + 7) & ~7; rows->nseq = (T + 15) >> 4;
        rows->lmT = 1; rows->lm_row[0] = T - 1; rows->lm_out[0] = 0;
        pass_items(rows, p.H, p.max_splits);
      }
    } else if (p.mode == 0) {
      verify_rows(rows, p, cta == 0);
    } else {
      if (lane < p.B) {
        const SeqState q = p.st[lane];
        const int p0 = draft_first(p, q);
        rows->n[lane] = p0 < 0 ? 0 : q.n;
        rows->j[lane] = q.len - 1;
        rows->p0[lane] = p0;
        rows->chunk[lane] = max(32, q.chunk);
        rows->cur[lane] = first_step > 0 ? __ldcg(p.tok_out + lane * p.nmax + first_step - 1) : 0;
      }
      __syncwarp();
      if (lane == 0) draft_rows_of_step(rows, p, first_step);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // the two CTAs of a cluster arrive on each other's barriers later on: both must have initialised them
  cluster_sync_all();

  const int nphase = phase_count(p);
  if (p.phase_ns && cta == 0 && tid == 32) {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    p.phase_ns[0] = t;
  }

  // ================================================================= weight producer
  if (warp == 0 || warp == 3) {
    if (lane != 0) return;   // one thread produces (idle lanes walking the schedule would only steal its issue slots)
    const unsigned pidx = warp == 0 ? 0u : 1u;   // producer 0 loads the even stages, producer 1 the odd ones
    uint32_t *st_off = st_rec + pidx * 2 * kFlight, *st_end = st_off + kFlight;   // this producer's own record of the stages
    RingRetire rr;   // both producers place and retire every stage of the schedule (see ada_ring.h)
    rr.init();
    const uint64_t pol_w = l2_policy_evict_first();   // weights are read once per pass
    const int TP0 = *reinterpret_cast<const volatile int *>(&rows->TP);
    unsigned decisions = 0;
    for (int step = first_step; step < nstep || (p.ddd_thr < 0.f && step < await_length(step_bar, decisions, rows, p.cnt, abort_s)); ++step)
    for (int ph = 0; ph < nphase && !*abort_s; ++ph) {
      int layer;
      const int kind = phase_kind(p, ph, layer);
      if (!is_gemm(kind)) continue;
      const GemmDesc &g = gemms[kind - PH_FC].g;
      const Slab &s = gemms[kind - PH_FC].s;
      if (s.rows == 0) continue;
      // per-phase constants in registers (tensor map and first row of each m tile)
      int map0, map1, row0, row1;
      tile_source(g, s, 0, map0, row0);
      tile_source(g, s, s.mtiles - 1, map1, row1);
      map0 += map_base(p, kind, layer);
      map1 += map_base(p, kind, layer);
      const unsigned long long m0 = reinterpret_cast<unsigned long long>(p.maps + map0);
      const unsigned long long m1 = reinterpret_cast<unsigned long long>(p.maps + map1);
      // (a stage holds no more boxes than an activation buffer of the step; the steps after the first have one row per sequence)
      const int region = s.region, kb = min(s.kb, xbuf_boxes(step == first_step ? TP0 : 8)), mtiles = s.mtiles, K = g.K, c0 = s.c0, c1 = s.c1;
      int c = c0 + s.rot;
      const unsigned tx_box = (unsigned)(s.box_rows * 128);
      for (int i = c0; i < c1; ++i, c = c + 1 == c1 ? c0 : c + 1) {
        const int nbox = (min(kKc, K - c * kKc) + kBoxK - 1) / kBoxK;   // boxes that hold any k < K
        for (int b0 = 0; b0 < nbox; b0 += kb) {
          const int nb = min(kb, nbox - b0);
          for (int mi = 0; mi < mtiles; ++mi) {
            const uint32_t bytes = (uint32_t)(nb * region);
            const uint32_t off = rr.place(bytes, st_off, st_end);
            const unsigned j = rr.cur.n - 1, slot = j % kSlots;
            if ((j & 1u) != pidx) continue;   // the other producer's stage
            if (rr.pending != RingRetire::kNone) {   // stages are read in order: the newest retired one covers the rest
              mbar_wait(&empty[rr.pending % kSlots], (rr.pending / kSlots) & 1u, p.cnt, abort_s);
              rr.pending = RingRetire::kNone;
            }
            mbar_expect_tx(&full[slot], (unsigned)nb * tx_box);
            const uint32_t dst = smem_u32(ring) + off, bar = smem_u32(&full[slot]);
            const unsigned long long mp = mi ? m1 : m0;
            const int y = mi ? row1 : row0;
            for (int b = 0; b < nb; ++b)   // rows past the matrix and k past K read as zero; evict-first in level 2
              asm volatile(
                  "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(
                      dst + (uint32_t)(b * region)),
                  "l"(mp), "r"(c * kKc + (b0 + b) * kBoxK), "r"(y), "r"(bar), "l"(pol_w)
                  : "memory");
          }
        }
      }
    }
    return;
  }

  // ================================================================= tensor-core issuer (warp 2)
  // One elected thread issues every product, in schedule order (about 58 cycles per tcgen05.mma when the
  // products of a stage are issued back to back), so stages are also released in order.  M tile mi of section q of K
  // accumulates in the acc_cols(TP) tensor-memory columns from (mtiles (q & 1) + mi) acc_cols(TP) on.
  if (warp == 2) {
    {
      RingCursor cur{0, 0};
      int xslot = 0;           // activation buffer of the next box
      uint32_t xphase = 0;     // per buffer the parity of its next arrival
      const uint32_t ring_u = smem_u32(ring), xbuf_u = smem_u32(xbuf);
      // The tensor-core instructions take their operands from uniform registers.  Everything they and the branches around them
      // depend on is therefore worked out from the launch's parameters, or passes through a warp reduction, whose result the
      // compiler knows to be uniform; with a slab description or a step count read from memory each product took 80 cycles
      // to issue instead of 45, and the loops were bound by it (7B, 5 rows: QKV 22 400 of its 28 800 cycles).
      const int nsteps = (int)__reduce_max_sync(0xffffffffu, (unsigned)nstep);
      unsigned decisions = 0;
      uint32_t sphase = 0;     // per place of the accumulators the parity of its next release in this phase
      for (int step = first_step;
           step < nsteps || (p.ddd_thr < 0.f && step < (int)__reduce_max_sync(0xffffffffu, (unsigned)await_length(step_bar, decisions, rows, p.cnt, abort_s)));
           ++step, xslot = 0) {
      unsigned tp = 0;         // padded rows of the step
      for (int ph = 0; ph < nphase; ++ph) {
        int layer;
        const int kind = phase_kind(p, ph, layer);
        if (!is_gemm(kind)) continue;
        GemmDesc g;
        make_gemm(p, kind, g);
        const Slab s = make_slab(g, cta, ncta);
        const int K = g.K;
        if (s.rows == 0) continue;
        if (tp == 0) {   // (the rows of the step are known once its first activations have landed)
          mbar_wait(&xfull[xslot], (xphase >> xslot) & 1u, p.cnt, abort_s);
          tp = __reduce_max_sync(0xffffffffu, (unsigned)*reinterpret_cast<const volatile int *>(&rows->TP));
        }
        // A phase's products.  The padded row count is a constant in each form: box strides and the instruction descriptor
        // then need no registers that the tensor-core instructions could not take (with a row count read from memory gate/up
        // of 5 rows took 44.5 us, with one put into a uniform register by a reduction 33.5, as a constant 31.1).
        auto products = [&](auto rows_const) {
          constexpr uint32_t TP = decltype(rows_const)::value;
          constexpr int kxb = xbuf_boxes(TP), nx = xbuf_count(TP);   // boxes per activation buffer, buffers
          constexpr uint32_t xbox = TP * 256;
          const uint32_t idesc = umma_idesc_mn(s.m64 ? 64u : 128u, 2 * TP);
          const uint32_t region16 = (uint32_t)s.region >> 4;
          const int kb = min(s.kb, kxb);
          uint32_t started = 0;   // bit mi: the accumulator of m tile mi holds a product of this section
          uint32_t col = tmem_base;   // accumulators of the section
          const uint32_t step_cols = (uint32_t)s.mtiles * acc_cols(TP);
          int sec = 0, left = s.per;  // section, chunks left in it
          for (int i = s.c0, c = s.c0 + s.rot; i < s.c1; ++i, c = c + 1 == s.c1 ? s.c0 : c + 1) {
            if (left == 0) { next_section(secfull, secempty, ++sec, sphase, p.cnt, abort_s); col = tmem_base + (sec & 1 ? step_cols : 0u); started = 0; left = s.per; }
            --left;
            const int kleft = min(kKc, K - c * kKc);
            const int nbox = (kleft + kBoxK - 1) / kBoxK;
#pragma unroll 1
            for (int x0 = 0; x0 < nbox; x0 += kxb) {
              const int xend = min(nbox, x0 + kxb);
              const uint64_t bdesc0 = umma_desc(xbuf_u + (uint32_t)(xslot * xbuf_bytes(TP)));
              mbar_wait(&xfull[xslot], (xphase >> xslot) & 1u, p.cnt, abort_s);
              for (int b0 = x0; b0 < xend; b0 += kb) {
                const int nb = min(kb, xend - b0);
                for (int mi = 0; mi < s.mtiles; ++mi) {
                  const uint32_t off = cur.take((uint32_t)(nb * s.region));
                  const unsigned slot = (cur.n - 1) % kSlots, parity = ((cur.n - 1) / kSlots) & 1u;
                  const uint64_t adesc0 = umma_desc(ring_u + off);
                  const uint32_t dcol = col + (uint32_t)mi * acc_cols(TP);
                  mbar_wait(&full[slot], parity, p.cnt, abort_s);
                  tc_fence_after();
                  if (elect_one()) {   // one thread issues the stage's products and the commit that frees it
                    uint32_t acc = (started >> mi) & 1u;
                    uint64_t ad = adesc0, bd = bdesc0 + (uint64_t)((b0 - x0) * (xbox >> 4));
                    auto box = [&] {                                // 64 k: + 32 bytes per k16 step
                      umma_bf16(dcol, ad, bd, idesc, acc);
                      umma_bf16(dcol, ad + 2, bd + 2, idesc, 1);
                      umma_bf16(dcol, ad + 4, bd + 4, idesc, 1);
                      umma_bf16(dcol, ad + 6, bd + 6, idesc, 1);
                      ad += region16; bd += xbox >> 4; acc = 1;
                    };
                    for (int bi = 0; bi < nb; ++bi) {
                        const int nstep = min(4, (kleft - (b0 + bi) * kBoxK + 15) >> 4);   // k16 steps holding any k < K
                        if (nstep == 4) {
                          box();
                        } else {
                          for (int s4 = 0; s4 < nstep; ++s4) umma_bf16(dcol, ad + 2 * s4, bd + 2 * s4, idesc, s4 ? 1u : acc);
                          ad += region16; bd += xbox >> 4; acc = 1;
                        }
                      }
                    umma_commit(&empty[slot]);   // the stage is free once these products have read it
                  }
                  started |= 1u << mi;
                  __syncwarp();
                }
              }
              if (elect_one()) umma_commit(&xempty[xslot]);
              __syncwarp();
              xphase ^= 1u << xslot;
              xslot = xslot + 1 == nx ? 0 : xslot + 1;
            }
          }
        };
        // The same for K in whole chunks (all but odd sizes), with the boxes of a stage and the m tiles constants as well: what
        // a stage costs beside its products (offsets, waits, election, commits) is a chain of dependent instructions in this
        // one warp, 400 to 600 cycles a stage, and with the loops unrolled most of it goes.  Verify pass, before -> after:
        // middle model 778 -> 712 us, 13B 5339 -> 5080, 7B with 24 rows 3105 -> 2958, with 36 rows 3719 -> 3300.
        auto whole_chunks = [&](auto rows_const, auto boxes_const, auto tiles_const) {
          constexpr uint32_t TP = decltype(rows_const)::value;
          constexpr int kxb = xbuf_boxes(TP), nx = xbuf_count(TP);
          constexpr int KB = decltype(boxes_const)::value < kxb ? decltype(boxes_const)::value : kxb, MT = decltype(tiles_const)::value;
          constexpr uint32_t xbox16 = (TP * 256) >> 4;
          const uint32_t idesc = umma_idesc_mn(s.m64 ? 64u : 128u, 2 * TP);
          const uint32_t region16 = (uint32_t)s.region >> 4, bytes = (uint32_t)(KB * s.region);
          uint32_t acc = 0, col = tmem_base;        // accumulators of the section
          const int per = s.per * (4 / kxb);
          int sec = 0, left = per;                  // section, activation buffers left in it
          for (int n = (s.c1 - s.c0) * (4 / kxb); n > 0; --n) {   // activation buffers
            if (left == 0) {
              next_section(secfull, secempty, ++sec, sphase, p.cnt, abort_s);
              col = tmem_base + (sec & 1 ? MT * acc_cols(TP) : 0u);
              left = per; acc = 0;
            }
            --left;
            const uint64_t bdesc0 = umma_desc(xbuf_u + (uint32_t)(xslot * xbuf_bytes(TP)));
#pragma unroll
            for (int q = 0; q < kxb / KB * MT; ++q) {
              const int mi = q % MT, b0 = q / MT * KB;
              const uint32_t off = cur.take(bytes);
              const unsigned slot = (cur.n - 1) % kSlots;
              mbar_wait(&full[slot], ((cur.n - 1) / kSlots) & 1u, p.cnt, abort_s);
              // The activations last: a phase's first weights are there long before them, and all that leads to the products is done
              // when they land (the row count, too, is asked for once a pass).  Draft of four + verify, waiting for them first ->
              // so: small model 145 + 66.5 -> 139 + 64.5 us, middle model 331 + 717 -> 323 + 703, 7B 583 + 2663 -> 576 + 2628.
              if (q == 0) mbar_wait(&xfull[xslot], (xphase >> xslot) & 1u, p.cnt, abort_s);
              tc_fence_after();
              if (elect_one()) {
                const uint64_t ad = umma_desc(ring_u + off);
                const uint32_t dcol = col + (uint32_t)mi * acc_cols(TP);
#pragma unroll
                for (int b = 0; b < KB; ++b)
#pragma unroll
                  for (int k4 = 0; k4 < 4; ++k4)
                    umma_bf16(dcol, ad + (uint64_t)(b * region16) + 2 * k4, bdesc0 + (b0 + b) * xbox16 + 2 * k4, idesc, b0 + b + k4 > 0 ? 1u : acc);
                umma_commit(&empty[slot]);
                if (q + 1 == kxb / KB * MT) umma_commit(&xempty[xslot]);
              }
              __syncwarp();
            }
            acc = 1;
            xphase ^= 1u << xslot;
            xslot = xslot + 1 == nx ? 0 : xslot + 1;
          }
        };
        auto whole = [&](auto rows_const) {
          using std::integral_constant;
          if (s.kb == 4) {
            if (s.mtiles == 1) whole_chunks(rows_const, integral_constant<int, 4>{}, integral_constant<int, 1>{});
            else whole_chunks(rows_const, integral_constant<int, 4>{}, integral_constant<int, 2>{});
          } else {
            if (s.mtiles == 1) whole_chunks(rows_const, integral_constant<int, 2>{}, integral_constant<int, 1>{});
            else whole_chunks(rows_const, integral_constant<int, 2>{}, integral_constant<int, 2>{});
          }
        };
        auto dispatch = [&](auto &&form) {
          if (tp == 8) form(std::integral_constant<uint32_t, 8>{});
          else if (tp == 16) form(std::integral_constant<uint32_t, 16>{});
          else if (tp == 24) form(std::integral_constant<uint32_t, 24>{});
          else if (tp == 32) form(std::integral_constant<uint32_t, 32>{});
          else if (tp == 40) form(std::integral_constant<uint32_t, 40>{});
          else form(std::integral_constant<uint32_t, 48>{});
        };
        if (K % kKc == 0) dispatch(whole);
        else dispatch(products);
        if (elect_one()) umma_commit(accfull);
        __syncwarp();
        sphase = sections_done(sphase, s.nsec);
      }
      }
    }
    __syncwarp();
    // the workers signal when their last read of tensor memory is done
    tc_fence_before();
    named_bar(5, 32 + kNumCWarps * 32);
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
    return;
  }

  // ================================================================= grid barriers and activation producer (warp 1)
  // A small loop of its own: what follows a barrier's last poll is the release of the workers and the first copies of the next
  // phase's input, whose description was worked out before the barrier.  (As part of the workers' loop over the phases it was
  // 1950 clocks from the last poll to the first copy, most of them waits for instructions that every phase had to fetch again;
  // now 850.  Draft of four + its verify: small model 163 + 74.8 -> 148 + 64.7 us, middle model 352 + 783 -> 336 + 735, 7B 612 +
  // 2825 -> 595 + 2738.)
  if (warp == 1) {
    const uint64_t pol_x = l2_policy_evict_last();   // (every CTA reads the same input tiles)
    uint32_t xused = 0, xphase = 0;                  // buffers used before, parity of their next release
    unsigned target = 0, epoch = 0;
    for (int step = first_step; step < nstep; ++step) {
      const int TP = *reinterpret_cast<const volatile int *>(&rows->TP);
      const int kxb = xbuf_boxes(TP), nx = xbuf_count(TP);    // boxes per buffer, buffers (of this step)
      const unsigned xbytes = (unsigned)xbuf_bytes(TP);
      int xslot = 0;   // (all buffers are free between steps)
      const __nv_bfloat16 *src = nullptr;
      int beg = 0, end = 0, b = 0, parts = 0;        // boxes of this CTA's part of K, the next one, copies to make
      for (int ph = 0; ph < nphase; ++ph) {
        if (lane == 0 && parts > 0 && !*abort_s) {
          fence_global_copies();   // the input tiles that the phase before stored
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the buffers double as scratch of the workers
#pragma unroll 1
          for (int i = parts; i > 0; --i) {
            if ((xused >> xslot) & 1u) {
              mbar_wait(&xempty[xslot], (xphase >> xslot) & 1u, p.cnt, abort_s);
              xphase ^= 1u << xslot;
            }
            xused |= 1u << xslot;
            const unsigned bytes = (unsigned)(min(kxb, end - b) * TP * 256);
            mbar_expect_tx(&xfull[xslot], bytes);
            bulk_g2s_hint(xbuf + (size_t)xslot * xbytes, src + (size_t)b * (TP * 128), bytes, &xfull[xslot], pol_x);
            xslot = xslot + 1 == nx ? 0 : xslot + 1;
            b += kxb;
            if (b >= end) b = beg;
          }
        }
        __syncwarp();
        // the next phase's copies
        int layer;
        const int kind = phase_kind(p, ph, layer);
        parts = 0;
        if (ph + 1 < nphase) {
          const int next = phase_kind(p, ph + 1, layer);
          if (is_gemm(next)) {
            const GemmDesc &g = gemms[next - PH_FC].g;
            const Slab &s = gemms[next - PH_FC].s;
            src = g.xt;
            beg = s.c0 * (kKc / kBoxK);
            end = min(s.c1 * (kKc / kBoxK), (g.K + kBoxK - 1) / kBoxK);
            b = beg + s.rot * (kKc / kBoxK);
            parts = s.rows > 0 ? (end - beg + kxb - 1) / kxb : 0;
          }
        }
        for (int k = PROMPT && kind == PH_ATTN ? 2 : 1; k > 0; --k) {   // (a prompt's new cache rows have a barrier of their own)
          target += (unsigned)ncta;
          named_bar(2, kBarThreads);
          if (lane == 0) grid_wait(p.gbar, p.cnt, target, abort_s);
          __syncwarp();
          named_arrive(4, kBarThreads);
          ++epoch;
          if (p.phase_ns && cta == 0 && lane == 0 && epoch < 511) {
            unsigned long long t;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            p.phase_ns[epoch] = t;
          }
        }
      }
      if (p.mode == 1 && !PROMPT) {   // the next step's rows, and whether there is one
        named_bar(6, kBarThreads);
        if (p.ddd_thr < 0.f) nstep = *reinterpret_cast<const volatile int *>(&rows->n[0]);
      }
    }
    if (lane == 0) {
      if (!PROMPT && p.steps_out && cta == 0) *p.steps_out = nstep - first_step;
      // the last CTA to leave clears the barrier count for the next launch (all have passed the last barrier)
      if (atomicAdd(p.gbar + 16, 1u) == (unsigned)ncta - 1u) {
        p.gbar[0] = 0;
        p.gbar[16] = 0;
      }
    }
    return;
  }

  // ================================================================= workers
  const int cw = warp - kFirstWorker;         // worker warp index 0..7
  const int ctid = tid - kFirstWorker * 32;   // index among the 256 worker threads
  unsigned acc_phase = 0;   // GEMM phases of this CTA whose accumulator has been awaited
  unsigned attn_uses = 0;           // completed phases of this warp's two attention barriers
  // Keys and values of a worker warp: 16-key pieces cw, cw + 8, ... of an item's split, one bulk copy each into the warp's
  // own two buffers (a piece is contiguous in its cache page).  No warp waits for another inside an item.  The buffers lie over the
  // epilogues' sums of pass rows 16 and up (ada_areas.h): where there are such rows a warp's first pieces are requested behind
  // a barrier of the workers, else in the QKV phase.  (Behind that barrier but before the other CTAs' release, against behind the
  // release: verify of 7B 18 rows 2760 -> 2742 us, 22 rows at context 1900 3435 -> 3418; middle model 18 rows 788 -> 784.)
  __nv_bfloat16 *const wst = reinterpret_cast<__nv_bfloat16 *>(xbuf + kKeysAt + cw * kKeysWarpBytes);
  int pages = 0;                    // cache pages of the warp's pieces 32 i + lane of the current item
  auto attn_pages = [&](int sq, int kfirst, int kend, int i0) {   // (fetched 32 at a time: no copy waits for a table lookup)
    const int k0 = kfirst + 128 * (i0 + lane);
    pages = k0 < kend ? p.page_table[rows->s_b[sq] * p.pages_per_seq + k0 / kPageSize] : 0;
  };
  auto attn_issue = [&](int i, int kfirst, int hh, int layer, bool values, int page) {   // one lane
    const int k0 = kfirst + 128 * i;
    const unsigned bytes = (unsigned)(16 * p.hd * 2);
    const size_t off = ((((size_t)page * p.cache_layers + layer) * p.H + hh) * kPageSize + k0 % kPageSize) * p.hd;
    uint64_t *bar = attn_bar + 2 * cw + (values ? 1 : 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // earlier generic accesses to the buffer come first
    mbar_expect_tx(bar, bytes);
    // (a layer's cache rows are read once per pass: evict-first, like the weights)
    bulk_g2s_hint(wst + (values ? 16 * 128 : 0), (values ? p.vpool : p.kpool) + off, bytes, bar, l2_policy_evict_first());
  };
  unsigned kuses = 0;               // completed phases of the K-split pair barrier
  uint32_t sphase = 0;              // per place of the accumulators the parity of its next section of this phase

  for (int step = first_step; step < nstep; ++step) {
  const int T = rows->T, lmT = rows->lmT, TP = rows->TP;
  bool arrived = false;             // at a grid barrier whose release has not been awaited
  for (int ph = 0; ph < nphase; ++ph) {
    int layer;
    const int kind = phase_kind(p, ph, layer);

    // ------------------------------------------------------------- row-wise input phases
    if (kind == PH_EMBED || kind == PH_EAGLE_IN) {
      // EMBED: h = embedding rows, planes = split(h * gain of layer 0), partial sums of squares.
      // EAGLE_IN: planes of [e(token) ; feature] for the draft head's fc.  Column slices per CTA.
      // Sixteen lanes per pass row, 16 rows at once (row by row, each row waited for its own chain of lookups: 5 rows of the
      // small model took 6.6 us here); the row's sum of squares is a fixed shuffle tree over its lanes.
      const int width = kind == PH_EMBED ? p.d : 2 * p.d;
      const int cpc = (((width + ncta - 1) / ncta) + 3) & ~3;
      const int c0 = cta * cpc, c1 = min(width, c0 + cpc);
      const __nv_bfloat16 *gain = p.layers[0].na;
      const int l16 = ctid & 15;
      for (int t0 = 0; t0 < T; t0 += kNumCWarps * 2) {
        const int t = t0 + (ctid >> 4);
        float ss = 0.f;
        if (t < T) {
          const __nv_bfloat16 *e = p.embed + (size_t)rows->tok[t] * p.d;
          const float *f = step == 0 ? p.feat + ((size_t)rows->seq[t] * p.tok_stride + rows->pos[t]) * p.d
                                     : p.dfeat + ((size_t)rows->seq[t] * p.nmax + (step - 1)) * p.d;
#pragma unroll 4
          for (int c = c0 + l16; c < c1; c += 16) {
            if (kind == PH_EMBED) {
              const float v = __bfloat162float(e[c]);
              p.h[(size_t)t * p.d + c] = v;
              ss += v * v;
              xstore(p.xa, TP, t, c, v * __bfloat162float(gain[c]));
            } else {
              xstore(p.fc, TP, t, c, c < p.d ? __bfloat162float(e[c]) : __ldcg(f + (c - p.d)));
            }
          }
        }
        if (kind == PH_EMBED) {
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
          if (l16 == 0 && t < T) p.ss_part[t * kSsStride + cta] = ss;
        }
      }
      phase_arrive();
      arrived = true;
      continue;
    }

    // ------------------------------------------------------------- attention
    if (kind == PH_ATTN) {
      if (PROMPT) {
        phase_await();
        {
          const int half = p.hd >> 1, per_row = p.H * half, b = rows->seq[0];
          for (int i = cta * (kNumCWarps * 32) + ctid; i < T * per_row; i += ncta * (kNumCWarps * 32)) {
            const int r = i / per_row, e = i - r * per_row, hh = e / half, c = e - hh * half, pos = rows->pos[r];
            const float *kr = p.qkv + (size_t)r * 3 * p.d + p.d + hh * p.hd + c, *vr = kr + p.d;
            const float2 cs = p.rope[(size_t)pos * half + c];
            const float ka = __ldcg(kr), kb = __ldcg(kr + half), va = __ldcg(vr), vb = __ldcg(vr + half);
            const int page = p.page_table[b * p.pages_per_seq + pos / kPageSize], slot = pos % kPageSize, x7 = slot & 7;
            const size_t base = ((((size_t)page * p.cache_layers + layer) * p.H + hh) * kPageSize + slot) * p.hd;
            const int o0 = (((c >> 3) ^ x7) << 3) | (c & 7), o1 = ((((c + half) >> 3) ^ x7) << 3) | (c & 7);
            p.kpool[base + o0] = kv_store(ka * cs.x - kb * cs.y);
            p.kpool[base + o1] = kv_store(kb * cs.x + ka * cs.y);
            p.vpool[base + o0] = kv_store(va);
            p.vpool[base + o1] = kv_store(vb);
          }
        }
        phase_arrive();
        phase_await();
        if (lane == 0) fence_global_copies();   // the new cache rows
      }
      {
        // Items (sequence, head, KV split) round-robin over CTAs.  Worker warp w takes the 16-key pieces w, w + 8, ... of the
        // split for all 16 query rows with mma.sync: scores = q k^T (m16n8k16 per 16 channels, two tiles of 8 keys), online
        // softmax on the accumulator fragments, weighted values (m16n8k16 over the 16 keys per 8 channels).  Cache elements
        // are 16-bit halves and enter the products as they are; q and the softmax weights are fp32 and enter as a (hi, lo)
        // pair of halves, so each product is issued twice and the sums are fp32.
        //
        // The phase is bound by latency, so it is a short chain: the first pieces of a CTA's first item are requested during
        // the QKV phase's epilogue (old keys depend on no phase of this step; those of the draft steps before it lie a fence
        // back), a warp's next keys fly under its softmax and
        // values and its next values under its scores, the merge over the warps and the merge over the splits are one step
        // each with all loads in flight, and an item that is its head's only split writes the result straight away.
        // Phase per layer, 5 rows, before -> after: small model 10.2 -> 6.6 us (context 100), 7B 13.9 -> 9.5 us (512) and
        // 35.0 -> 21.7 us (3801), 13B 20.8 -> 13.4 us (1024); verify pass 3213 -> 3040, 3964 -> 3519, 5793 -> 5544 us.
        const int HD = p.hd, d = p.d, half = HD >> 1, hsh = HD == 128 ? 6 : 5;   // (half = 1 << hsh)
        // A prompt's groups of rows see each other's keys, so its rows go into the cache first, everything after a barrier.
        // The cache is cut into splits of a size fixed per sequence when its prompt was read (a multiple of 32 keys), so
        // the split a key falls in, and with it every sum of this phase, does not depend on how many rows a pass holds:
        // a row's result is the same bit for bit in a one-row pass and in a block of drafts.
        __half *qh_s = reinterpret_cast<__half *>(xbuf);                              // q hi [16][128], 16-byte chunks XORed with row & 7
        __half *ql_s = qh_s + 16 * 128;                                              // q lo, same layout
        __nv_bfloat16 *k_s = reinterpret_cast<__nv_bfloat16 *>(ql_s + 16 * 128);    // new rows, rotated [16][128]
        __nv_bfloat16 *v_s = k_s + 16 * 128;
        const __nv_bfloat16 *kst = wst, *vst = wst + 16 * 128;
        float *part_s = reinterpret_cast<float *>(xbuf);                              // [8 warps][16 rows][kPartRow], reuses the above
        const int g8r = lane >> 2, t4 = lane & 3;
        const uint32_t qh_u = smem_u32(qh_s), ql_u = smem_u32(ql_s);
        for (int item = cta, sq = 0; item < rows->nitems; item += ncta) {
          while (item >= rows->s_item0[sq + 1]) ++sq;
          const int b = rows->s_b[sq], R = rows->s_rows[sq], row0 = rows->s_row0[sq], pos0 = rows->s_pos0[sq];
          const int nkeys = pos0 + R, chunk = rows->s_chunk[sq], nsp = rows->s_nsp[sq];
          const int rel = item - rows->s_item0[sq], hh = rel / nsp, split = rel - hh * nsp;
          const int prow = rows->s_part0[sq] + hh * nsp * R;                          // first row of the head's partial results
          const int kbeg = split * chunk, kend = min(nkeys, kbeg + chunk);
          const int kfirst = kbeg + 16 * cw;
          if (item != cta || !keys_clear_of_sums(TP) || PROMPT) {   // (else the pieces were requested in the QKV phase)
            attn_pages(sq, kfirst, kend, 0);
            named_bar(3, kNumCWarps * 32);   // every warp has read what lay there: the QKV phase's sums, or the item before
            const int pg = __shfl_sync(0xffffffffu, pages, 0);
            if (lane == 0 && kfirst < kend) {
              attn_issue(0, kfirst, hh, layer, false, pg);
              attn_issue(0, kfirst, hh, layer, true, pg);
            }
          }
          // q (scaled) of the sequence's rows with rotary embedding as (hi, lo) halves; k and v of the rows that fall into
          // this split, which also stores them in the cache.  (A thread's loads in one round trip.)
          const float qscale = rsqrtf((float)HD);
          const int new0 = PROMPT ? 1 << 30 : pos0;   // first position whose key and value come from this pass's own sums
          const bool fresh_here = kend > new0;
          const int page_a = fresh_here ? p.page_table[b * p.pages_per_seq + pos0 / kPageSize] : 0;
          const int page_b = fresh_here ? p.page_table[b * p.pages_per_seq + (nkeys - 1) / kPageSize] : 0;
          // (The first item is worked out while the other CTAs arrive: verify of the middle model 730 -> 718 us, 7B 2708 -> 2690,
          // with the divisions by the head's width gone.)
          if (!PROMPT && item == cta) phase_await();
          for (int i0 = 0; i0 < R * half; i0 += 2 * kNumCWarps * 32) {
            float qa[2], qb[2], ka[2], kb[2], va[2], vb[2];
            float2 cs[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int i = i0 + u * kNumCWarps * 32 + ctid;
              const int r = i >> hsh, c = i & (half - 1);
              qa[u] = qb[u] = ka[u] = kb[u] = va[u] = vb[u] = 0.f;
              cs[u] = make_float2(1.f, 0.f);
              if (i < R * half) {
                cs[u] = p.rope[(size_t)(pos0 + r) * half + c];
                const float *qr = p.qkv + (size_t)(row0 + r) * 3 * d + hh * HD;
                qa[u] = __ldcg(qr + c); qb[u] = __ldcg(qr + c + half);
                if (pos0 + r >= kbeg && pos0 + r < kend && !PROMPT) {
                  ka[u] = __ldcg(qr + d + c); kb[u] = __ldcg(qr + d + c + half);
                  va[u] = __ldcg(qr + 2 * d + c); vb[u] = __ldcg(qr + 2 * d + c + half);
                }
              }
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int i = i0 + u * kNumCWarps * 32 + ctid;
              if (i >= R * half) continue;
              const int r = i >> hsh, c = i & (half - 1);
              const float q0 = (qa[u] * cs[u].x - qb[u] * cs[u].y) * qscale, q1 = (qb[u] * cs[u].x + qa[u] * cs[u].y) * qscale;
              const __half h0 = __float2half_rn(q0), h1 = __float2half_rn(q1);
              const int o0 = r * 128 + ((((c >> 3) ^ (r & 7)) << 3) | (c & 7));
              const int o1 = r * 128 + (((((c + half) >> 3) ^ (r & 7)) << 3) | (c & 7));
              qh_s[o0] = h0; qh_s[o1] = h1;
              ql_s[o0] = __float2half_rn(q0 - __half2float(h0)); ql_s[o1] = __float2half_rn(q1 - __half2float(h1));
              const int pos = pos0 + r;
              if (pos >= kbeg && pos < kend && !PROMPT) {
                const __nv_bfloat16 k0 = kv_store(ka[u] * cs[u].x - kb[u] * cs[u].y);   // 16-bit cache elements (see kv_store)
                const __nv_bfloat16 k1 = kv_store(kb[u] * cs[u].x + ka[u] * cs[u].y);
                const __nv_bfloat16 v0 = kv_store(va[u]), v1 = kv_store(vb[u]);
                k_s[o0] = k0; k_s[o1] = k1;      // (the staged rows have their chunks XORed by row & 7, like q)
                v_s[o0] = v0; v_s[o1] = v1;
                // (at most 16 rows: they lie in the page of the first row or in the page of the last)
                const int page = pos / kPageSize == pos0 / kPageSize ? page_a : page_b, slot = pos % kPageSize;
                const size_t base = ((((size_t)page * p.cache_layers + layer) * p.H + hh) * kPageSize + slot) * HD;
                // key and value rows are stored with their 16-byte chunks XORed by (slot & 7): copied verbatim to
                // shared memory, eight consecutive rows then sit in eight different bank groups (ldmatrix of 8 keys'
                // chunk, plain for the scores and transposed for the weighted values, is conflict-free)
                const int sw = slot & 7;
                p.kpool[base + ((((c >> 3) ^ sw) << 3) | (c & 7))] = k0;
                p.kpool[base + (((((c + half) >> 3) ^ sw) << 3) | (c & 7))] = k1;
                p.vpool[base + ((((c >> 3) ^ sw) << 3) | (c & 7))] = v0;
                p.vpool[base + (((((c + half) >> 3) ^ sw) << 3) | (c & 7))] = v1;
              }
            }
          }
          // running maxima, sums and outputs of rows g8r and g8r + 8 over this warp's keys
          float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
          float o[16][4];
#pragma unroll
          for (int nt = 0; nt < 16; ++nt) o[nt][0] = o[nt][1] = o[nt][2] = o[nt][3] = 0.f;
          named_bar(3, kNumCWarps * 32);   // staging visible
          for (int i = 0; kfirst + 128 * i < kend; ++i, ++attn_uses) {
            const int key0 = kfirst + 128 * i;
            // a key of this pass comes from the staged new rows, an older one from the copied cache rows; this lane supplies
            // the addresses of row (lane & 7) of both tiles of 8 keys.  Masked keys past the sequence read any finite row.
            const int ka_ = key0 + (lane & 7), kb_ = ka_ + 8;
            const int fa = min(ka_ - new0, R - 1), fb = min(kb_ - new0, R - 1);   // staged row, if >= 0
            const int swa = fa >= 0 ? fa & 7 : lane & 7, swb = fb >= 0 ? fb & 7 : lane & 7;
            if (((i + 1) & 31) == 0) attn_pages(sq, kfirst, kend, i + 1);
            const int pnext = __shfl_sync(0xffffffffu, pages, (i + 1) & 31);
            const bool more = lane == 0 && key0 + 128 < kend;
            mbar_wait(attn_bar + 2 * cw, attn_uses & 1u, p.cnt, abort_s);
            // ---- scores: 16 rows x 16 keys
            float sa[4] = {0.f, 0.f, 0.f, 0.f}, sb[4] = {0.f, 0.f, 0.f, 0.f};      // hi products
            float sal[4] = {0.f, 0.f, 0.f, 0.f}, sbl[4] = {0.f, 0.f, 0.f, 0.f};    // lo products: chains of their own
            {
              const uint32_t rowa = fa >= 0 ? smem_u32(k_s + fa * 128) : smem_u32(kst + (lane & 7) * HD);
              const uint32_t rowb = fb >= 0 ? smem_u32(k_s + fb * 128) : smem_u32(kst + ((lane & 7) + 8) * HD);
              const int arow = (lane & 7) + ((lane >> 3) & 1) * 8;
#pragma unroll 1
              for (int kp = 0; kp * 32 < HD; ++kp) {            // pairs of 16-channel steps
                {
                  uint32_t ka0, ka1, ka2, ka3, kb0, kb1, kb2, kb3;
                  ldmatrix_x4(rowa + (((kp * 4 + (lane >> 3)) ^ swa) << 4), ka0, ka1, ka2, ka3);
                  ldmatrix_x4(rowb + (((kp * 4 + (lane >> 3)) ^ swb) << 4), kb0, kb1, kb2, kb3);
#pragma unroll
                  for (int h2 = 0; h2 < 2; ++h2) {
                    const int ks = kp * 2 + h2;
                    const uint32_t aoff = (uint32_t)(arow * 256 + (((ks * 2 + (lane >> 4)) ^ (arow & 7)) << 4));
                    uint32_t a0, a1, a2, a3;
                    ldmatrix_x4(qh_u + aoff, a0, a1, a2, a3);
                    mma_f16_k16(sa, a0, a1, a2, a3, h2 ? ka2 : ka0, h2 ? ka3 : ka1);
                    mma_f16_k16(sb, a0, a1, a2, a3, h2 ? kb2 : kb0, h2 ? kb3 : kb1);
                    ldmatrix_x4(ql_u + aoff, a0, a1, a2, a3);
                    mma_f16_k16(sal, a0, a1, a2, a3, h2 ? ka2 : ka0, h2 ? ka3 : ka1);
                    mma_f16_k16(sbl, a0, a1, a2, a3, h2 ? kb2 : kb0, h2 ? kb3 : kb1);
                  }
                }
              }
            }
            __syncwarp();
            if (more) attn_issue(i + 1, kfirst, hh, layer, false, pnext);   // the next keys fly from here
#pragma unroll
            for (int j = 0; j < 4; ++j) { sa[j] += sal[j]; sb[j] += sbl[j]; }
            // ---- online softmax: this thread holds keys kc, kc + 1, kc + 8, kc + 9 of rows g8r and g8r + 8
            const int kc = key0 + 2 * t4;
            float p0[4] = {sa[0], sa[1], sb[0], sb[1]}, p1[4] = {sa[2], sa[3], sb[2], sb[3]};
            float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int k = kc + (j & 1) + 8 * (j >> 1);
              if (k >= kend || k > pos0 + g8r) p0[j] = -INFINITY;
              if (k >= kend || k > pos0 + g8r + 8) p1[j] = -INFINITY;
              mx0 = fmaxf(mx0, p0[j]); mx1 = fmaxf(mx1, p1[j]);
            }
            mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1)); mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
            mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2)); mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
            const float mn0 = fmaxf(m0, mx0), mn1 = fmaxf(m1, mx1);
            const float b0 = mn0 > -INFINITY ? mn0 : 0.f, b1 = mn1 > -INFINITY ? mn1 : 0.f;   // (a row that sees no key yet: all weights 0)
            const float c0 = __expf(m0 - b0), c1 = __expf(m1 - b1);
#pragma unroll
            for (int j = 0; j < 4; ++j) { p0[j] = __expf(p0[j] - b0); p1[j] = __expf(p1[j] - b1); }
            float ps0 = (p0[0] + p0[1]) + (p0[2] + p0[3]), ps1 = (p1[0] + p1[1]) + (p1[2] + p1[3]);
            ps0 += __shfl_xor_sync(0xffffffffu, ps0, 1); ps1 += __shfl_xor_sync(0xffffffffu, ps1, 1);
            ps0 += __shfl_xor_sync(0xffffffffu, ps0, 2); ps1 += __shfl_xor_sync(0xffffffffu, ps1, 2);
            l0 = l0 * c0 + ps0; l1 = l1 * c1 + ps1;
            const bool moved = (g8r < R && mn0 != m0) || (g8r + 8 < R && mn1 != m1);   // (rows past R hold whatever was in memory)
            m0 = mn0; m1 = mn1;
            // weights as (hi, lo) halves: a0 = row g8r keys 0..7, a1 = row g8r + 8 keys 0..7, a2, a3: keys 8..15
            uint32_t ah[4], al[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float x = (j & 1) ? p1[2 * (j >> 1)] : p0[2 * (j >> 1)], y = (j & 1) ? p1[2 * (j >> 1) + 1] : p0[2 * (j >> 1) + 1];
              const __half2 ph = __floats2half2_rn(x, y);
              const float2 pf = __half22float2(ph);
              const __half2 pl = __floats2half2_rn(x - pf.x, y - pf.y);
              ah[j] = *reinterpret_cast<const uint32_t *>(&ph);
              al[j] = *reinterpret_cast<const uint32_t *>(&pl);
            }
            if (__any_sync(0xffffffffu, moved)) {   // some running maximum moved: rescale the sums so far
#pragma unroll
              for (int nt = 0; nt < 16; ++nt) { o[nt][0] *= c0; o[nt][1] *= c0; o[nt][2] *= c1; o[nt][3] *= c1; }
            }
            mbar_wait(attn_bar + 2 * cw + 1, attn_uses & 1u, p.cnt, abort_s);
            // ---- values: out[16 rows][HD] += w[16 x 16 keys] v[16 keys x HD], two 8-channel tiles per load
            {
              const bool second = (lane >> 3) & 1;   // lanes 8..15 and 24..31 address keys 8..15
              const int fv = second ? fb : fa;
              const uint32_t vrow = fv >= 0 ? smem_u32(v_s + fv * 128) : smem_u32(vst + ((lane & 7) + (second ? 8 : 0)) * HD);
              const int vsw = second ? swb : swa;
#pragma unroll
              for (int c2 = 0; c2 < 8; ++c2) {
                if (c2 * 16 < HD) {
                  uint32_t v0, v1, v2, v3;   // (keys 0..7, keys 8..15) of channel tile 2 c2, then of tile 2 c2 + 1
                  ldmatrix_x4_trans(vrow + (((2 * c2 + (lane >> 4)) ^ vsw) << 4), v0, v1, v2, v3);
                  mma_f16_k16(o[2 * c2], ah[0], ah[1], ah[2], ah[3], v0, v1);
                  mma_f16_k16(o[2 * c2 + 1], ah[0], ah[1], ah[2], ah[3], v2, v3);
                  mma_f16_k16(o[2 * c2], al[0], al[1], al[2], al[3], v0, v1);
                  mma_f16_k16(o[2 * c2 + 1], al[0], al[1], al[2], al[3], v2, v3);
                }
              }
            }
            __syncwarp();
            if (more) attn_issue(i + 1, kfirst, hh, layer, true, pnext);
          }
          // per-warp partials -> shared, once every warp has left the staging areas
          named_bar(3, kNumCWarps * 32);
#pragma unroll
          for (int nt = 0; nt < 16; ++nt)
            if (nt * 8 < HD) {
              *reinterpret_cast<float2 *>(part_s + (cw * 16 + g8r) * kPartRow + nt * 8 + 2 * t4) = make_float2(o[nt][0], o[nt][1]);
              *reinterpret_cast<float2 *>(part_s + (cw * 16 + g8r + 8) * kPartRow + nt * 8 + 2 * t4) = make_float2(o[nt][2], o[nt][3]);
            }
          if (t4 == 0) {
            *reinterpret_cast<float2 *>(part_s + (cw * 16 + g8r) * kPartRow + 128) = make_float2(m0, l0);
            *reinterpret_cast<float2 *>(part_s + (cw * 16 + g8r + 8) * kPartRow + 128) = make_float2(m1, l1);
          }
          named_bar(3, kNumCWarps * 32);
          // merge over the eight warps in warp order, four channels of a row per thread and step
          const int q4n = HD >> 2;
          float *const po = p.attn_part;                                                   // [rows][HD]
          float2 *const pml = reinterpret_cast<float2 *>(p.attn_part + p.attn_part_floats); // [rows] (m, l)
#pragma unroll 1
          for (int i = ctid; i < R * q4n; i += kNumCWarps * 32) {
            const int r = i >> (hsh - 1), c = (i & (q4n - 1)) * 4;
            float2 ml[8];
            float4 ov[8];
#pragma unroll
            for (int w = 0; w < 8; ++w) {
              ml[w] = *reinterpret_cast<const float2 *>(part_s + (w * 16 + r) * kPartRow + 128);
              ov[w] = *reinterpret_cast<const float4 *>(part_s + (w * 16 + r) * kPartRow + c);
            }
            float M = -INFINITY, l = 0.f;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int w = 0; w < 8; ++w) M = fmaxf(M, ml[w].x);
#pragma unroll
            for (int w = 0; w < 8; ++w) {
              const float e = ml[w].x > -INFINITY ? __expf(ml[w].x - M) : 0.f;
              l += ml[w].y * e;
              x.x += ov[w].x * e; x.y += ov[w].y * e; x.z += ov[w].z * e; x.w += ov[w].w * e;
            }
            if (nsp == 1) {
              const float inv = 1.f / l;
              xstore4(p.at, TP, row0 + r, hh * HD + c, make_float4(x.x * inv, x.y * inv, x.z * inv, x.w * inv));
            } else {
              const size_t pr = (size_t)prow + split * R + r;
              __stcg(reinterpret_cast<float4 *>(po + pr * HD + c), x);
              if (c == 0) __stcg(pml + pr, make_float2(M, l));
            }
          }
          if (nsp > 1) {
            // the item that arrives last for this head merges the splits in split order
            named_bar(3, kNumCWarps * 32);
            if (ctid == 0) {
              int *const cnt_h = p.attn_cnt + sq * p.H + hh;
              int old;
              asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(old) : "l"(cnt_h) : "memory");
              *flag_s = old == nsp - 1;
              if (old == nsp - 1) *cnt_h = 0;
            }
            named_bar(3, kNumCWarps * 32);
            if (*flag_s) {
#pragma unroll 1
              for (int i = ctid; i < R * q4n; i += kNumCWarps * 32) {
                const int r = i >> (hsh - 1), c = (i & (q4n - 1)) * 4;
                float M = -INFINITY, l = 0.f;
                float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
                for (int s0 = 0; s0 < nsp; s0 += 4) {   // four splits' loads in flight together
                  float2 ml[4];
                  float4 ov[4];
#pragma unroll
                  for (int u = 0; u < 4; ++u) {
                    const size_t pr = (size_t)prow + (s0 + u) * R + r;
                    ml[u] = make_float2(-INFINITY, 0.f);
                    ov[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (s0 + u < nsp) {
                      ml[u] = __ldcg(pml + pr);
                      ov[u] = __ldcg(reinterpret_cast<const float4 *>(po + pr * HD + c));
                    }
                  }
                  float Mn = M;
#pragma unroll
                  for (int u = 0; u < 4; ++u) Mn = fmaxf(Mn, ml[u].x);
                  const float k = M > -INFINITY ? __expf(M - Mn) : 0.f;
                  l *= k; x.x *= k; x.y *= k; x.z *= k; x.w *= k;
                  M = Mn;
#pragma unroll
                  for (int u = 0; u < 4; ++u) {
                    const float e = ml[u].x > -INFINITY ? __expf(ml[u].x - M) : 0.f;
                    l += ml[u].y * e;
                    x.x += ov[u].x * e; x.y += ov[u].y * e; x.z += ov[u].z * e; x.w += ov[u].w * e;
                  }
                }
                const float inv = 1.f / l;
                xstore4(p.at, TP, row0 + r, hh * HD + c, make_float4(x.x * inv, x.y * inv, x.z * inv, x.w * inv));
              }
            }
          }
        }
      }
      if (!PROMPT && cta >= rows->nitems) phase_await();   // (nothing to do here)
      phase_arrive();
      arrived = true;
      continue;
    }

    // ------------------------------------------------------------- GEMM phases
    const GemmDesc &g = gemms[kind - PH_FC].g;
    const Slab &s = gemms[kind - PH_FC].s;
    const int Tg = g.lm_rows ? lmT : T;

    // ---- the epilogue straight out of tensor memory.  First what needs nothing from the phase before, while the other CTAs
    // arrive: old residual values are at least one barrier old.
    const bool has_ss = g.epi == EPI_RESID_H || g.epi == EPI_STORE_H;
    const bool sw = g.epi == EPI_SWIGLU_ACT;
    // thread <-> weight row: quarter = warp index mod 4 (the tensor-memory lanes this warp may read),
    // m tile = worker index / 4 (SWIGLU: the first four workers read both accumulators)
    const int quarter = warp & 3, mi = sw ? 0 : (cw >> 2);
    const int rloc = s.m64 ? (lane < 16 ? quarter * 16 + lane : 1 << 20) : quarter * 32 + lane;   // row inside the m tile
    const bool active_warp = s.rows > 0 && (sw ? cw < 4 : mi < s.mtiles);
    const int rslab = mi * s.box_rows + rloc;                   // row inside the slab
    const bool valid = active_warp && rloc < s.box_rows && rslab < s.rows;
    const int vrow = s.seg * g.Nseg + s.r0 + rslab;             // output column

    // K-split pair: CTA j of the pair finishes the pass rows j, j + 2, ...  Two neighbouring output columns go to a thread;
    // `odd` = 1 where the slab starts on an odd column.
    const bool pair = s.ks > 1 && s.rows > 0;
    const int t0 = pair ? s.kj : 0, tstep = pair ? 2 : 1, mine = s.rows > 0 ? (pair ? (Tg + 1 - s.kj) >> 1 : Tg) : 0;
    const int col0 = s.seg * g.Nseg + s.r0;                     // output column of slab row 0
    const int odd = s.r0 & 1;
    // QKV, SwiGLU: (pass row, even column and the next) over all 256 threads.  Residual rows: a warp takes 64 columns of one pass
    // row (an item), counted from the slab's first one, and leaves their sums of squares.  (With one column per thread, 32 columns of
    // a row per warp and step, a step was a chain of 400 to 700 clocks, two to four of them a phase, and the rows' sums went through
    // shared memory.  Verify: 7B 5 rows 2738 -> 2708 us, 11 rows 2918 -> 2840, 18 rows of three sequences 2975 -> 2875; middle model
    // 18 rows 853 -> 814.)
    const int pairs = (odd + s.rows + 1) >> 1, nflat = s.rows > 0 ? Tg * pairs : 0;
    const unsigned per_pair = ((1u << 22) + (unsigned)pairs - 1u) / (unsigned)max(1, pairs);   // e / pairs = e per_pair >> 22: e < 48 pairs, pairs <= 129
    const int segs = s.segs, nitem = mine * segs;
    // the next norm's gain and old residual values of the first items
    const __nv_bfloat16 *const gain = has_ss ? gain_after(p, kind, layer) : nullptr;
    constexpr int kAhead = 2;
    float2 hold[kAhead], gn[kAhead];
    auto item_old = [&](int wi, float2 &h, float2 &gv) {
      const int tq = wi / segs, r = (wi - tq * segs) * 64 + 2 * lane;
      const float *hp = p.h + (size_t)(t0 + tq * tstep) * p.d + col0 + r;
      h = make_float2(0.f, 0.f);
      gv = make_float2(1.f, 1.f);
      if (wi >= nitem) return;
      const bool in0 = r < s.rows, in1 = r + 1 < s.rows;
      if (g.epi == EPI_RESID_H) {
        if (in0) h.x = __ldcg(hp);
        if (in1) h.y = __ldcg(hp + 1);
      }
      if (gain) {
        if (in0) gv.x = __bfloat162float(gain[col0 + r]);
        if (in1) gv.y = __bfloat162float(gain[col0 + r + 1]);
      }
    };
    if (has_ss) {
#pragma unroll
      for (int k = 0; k < kAhead; ++k) item_old(cw + kNumCWarps * k, hold[k], gn[k]);
    }
    // the attention phase that follows: cache pages of the warp's pieces of this CTA's first item ...
    int at_kfirst = 0, at_hh = -1;
    if (kind == PH_QKV && keys_clear_of_sums(TP) && !PROMPT && cta < rows->nitems) {   // (more rows: the epilogue needs the area)
      int sq = 0;
      while (cta >= rows->s_item0[sq + 1]) ++sq;
      const int nsp = rows->s_nsp[sq], chunk = rows->s_chunk[sq], rel = cta - rows->s_item0[sq], hh = rel / nsp;
      const int kbeg = (rel - hh * nsp) * chunk, kend = min(rows->s_pos0[sq] + rows->s_rows[sq], kbeg + chunk);
      at_kfirst = kbeg + 16 * cw;
      attn_pages(sq, at_kfirst, kend, 0);
      if (at_kfirst < kend) at_hh = hh;
    }
    if (arrived) phase_await();
    const bool stamper = cta == 0 && ctid == 0;
    stamp(p, ph, 0, stamper);
    // 1/rms per row of h for phases whose input was h * gain (partials summed in CTA order)
    if (g.scale_inv_rms) {
      // partials of a row: left by the phase that wrote h, by the CTA of a pair that finishes the row (the embedding: by all CTAs)
      const int from = kind == PH_GATEUP ? PH_O : kind == PH_LM || layer > 0 ? PH_DOWN : p.mode == 0 ? PH_EMBED : PH_FC;
      const bool emb = from == PH_EMBED;
      const Slab &w = gemms[emb ? 0 : from - PH_FC].s;
      const int sh = !emb && w.ks > 1, slots = emb ? 1 : ss_slots(w.segs), n = (emb ? ncta : w.slabs) << sh;
      for (int r = 2 * cw; r < T; r += 2 * kNumCWarps) {   // two rows per warp and step; lanes stride over the CTAs (at most 256), all loads in flight, fixed shuffle tree
        float v0[8], v1[8];
        const int n0 = ((lane ^ r) & sh) ? 0 : n, n1 = r + 1 >= T || ((lane ^ (r + 1)) & sh) ? 0 : n;   // (CTA j of a pair: rows j, j + 2, ...)
        const float *q = p.ss_part + r * kSsStride + (lane >> sh) * slots;
        const int inc = (32 >> sh) * slots;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          v0[k] = lane + 32 * k < n0 ? __ldcg(q + k * inc) : 0.f;
          v1[k] = lane + 32 * k < n1 ? __ldcg(q + k * inc + kSsStride) : 0.f;
        }
        for (int j = 1; j < slots; ++j) {
          float u0[8], u1[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            u0[k] = lane + 32 * k < n0 ? __ldcg(q + k * inc + j) : 0.f;
            u1[k] = lane + 32 * k < n1 ? __ldcg(q + k * inc + j + kSsStride) : 0.f;
          }
#pragma unroll
          for (int k = 0; k < 8; ++k) { v0[k] += u0[k]; v1[k] += u1[k]; }
        }
        float s0 = 0.f, s1 = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) { s0 += v0[k]; s1 += v1[k]; }
        s0 = warp_sum(s0); s1 = warp_sum(s1);
        if (lane == 0) {
          inv_rms[r] = rsqrtf(s0 / (float)p.d + p.eps);
          if (r + 1 < T) inv_rms[r + 1] = rsqrtf(s1 / (float)p.d + p.eps);
        }
      }
      named_bar(3, kNumCWarps * 32);
    }
    if (kind == PH_LM) {
      // column slice of the feature rows: target f = h / rms * gain (kept per position); draft: the
      // head's own output rows (kept per step) -- both read by later passes
      const int cpc = (p.d + ncta - 1) / ncta;
      const int c0 = cta * cpc, c1 = min(p.d, c0 + cpc);
      for (int i = ctid; i < (p.mode == 0 ? T : Tg) * (c1 - c0); i += kNumCWarps * 32) {
        const int t = i / (c1 - c0), c = c0 + (i - t * (c1 - c0));
        if (p.mode == 0) {
          if (!p.feat) break;   // (packed start positions keep no features)
          const float v = (__ldcg(p.h + (size_t)t * p.d + c) * inv_rms[t]) * __bfloat162float(p.final_norm[c]);
          p.feat[((size_t)rows->seq[t] * p.cap + rows->pos[t]) * p.d + c] = v;
        } else {
          const int sr = rows->lm_row[t];
          p.dfeat[((size_t)rows->seq[sr] * p.nmax + step) * p.d + c] = __ldcg(p.h + (size_t)sr * p.d + c);
        }
      }
    }
    stamp(p, ph, 1, stamper);
    // accumulators of section q of K and this warp's m tile from taddr + (q & 1) place on, its sums from `sums` on
    const uint32_t cols = acc_cols((uint32_t)TP), place = (uint32_t)s.mtiles * cols;
    const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)mi * cols;
    const uint32_t sums = tmem_base + ((uint32_t)(quarter * 32) << 16) + kTmemSums + (uint32_t)(mi * TP);
    const int t_end = sw ? 2 * TP : TP;                  // (SwiGLU: the gate rows, then the up rows)
    if (s.nsec > 1 && s.rows > 0) sphase = add_sections(secfull, secempty, sphase, s.nsec, active_warp ? t_end : 0, TP, taddr, place, sums, p.cnt, abort_s);
    // (the cache rows of the draft steps before this one, under the products)
    if (kind == PH_QKV && step > first_step && lane == 0) fence_global_copies();
    if (s.rows > 0) {
      mbar_wait(accfull, acc_phase & 1u, p.cnt, abort_s);
      ++acc_phase;
      tc_fence_after();
    }
    if (kind == PH_QKV) {   // ... and its first keys and values (the products have read the last activation buffer)
      const int pg = __shfl_sync(0xffffffffu, pages, 0);
      if (lane == 0 && at_hh >= 0) {
        attn_issue(0, at_kfirst, at_hh, layer, false, pg);
        attn_issue(0, at_kfirst, at_hh, layer, true, pg);
      }
    }
    stamp(p, ph, 2, stamper);
    // The sums go through shared memory (the activation buffers are idle once the accumulator is complete), by pass row and
    // slab row, so that all eight warps take part however few rows the slab has (see nflat and nitem above).  (Each thread walking
    // the pass rows of its own weight row took 0.18 us a row.)
    //
    // K-split pair = the two CTAs of a cluster (same slab, same thread <-> row mapping): each finishes half of the pass rows
    // (CTA j of the pair rows j, j + 2, ...).  A thread sends its sums of the other rows into the peer's shared memory, to an
    // area nothing else uses, with stores that count their bytes on the peer's barrier; then it adds first half + second
    // half, whoever is faster.  (With plain stores and a releasing arrive the exchange took 1.7 to 2.4 us, most of it the
    // release; one CTA fetching all rows of the other and finishing them alone was no better.)
    // Per layer, 5 rows: 7B O 10.7 -> 8.6, down 19.6 -> 18.2 us; middle model 7.6 -> 6.4 and 11.4 -> 10.2 us.
    static_assert(kSumsRowBytes == 256 * sizeof(float), "rows of sums");
    float *const ys = reinterpret_cast<float *>(xbuf);    // [rows][256] accumulator values; SwiGLU: 128 gate, 128 up columns
    const bool sends = pair && cw < 4;
    if (sends && ctid == 0) mbar_expect_tx(kbar, (unsigned)(128 * 16 * (TP >> 3)));
    if (active_warp) {
      const unsigned other = (unsigned)(s.kj ^ 1);
      const uint32_t dst = peer_addr(red + ctid * 4, other), bar = peer_addr(kbar, other);
      const bool more = s.nsec > 1;
      const uint32_t last = taddr + (uint32_t)((s.nsec - 1) & 1) * place;   // the last section's accumulators
      float *y = ys + rslab;
#pragma unroll 1
      for (int t8 = 0; t8 < t_end; t8 += 8, y += 8 * 256) {
        if (t8 == TP) y = ys + 128 + rslab;
        const uint32_t acc = acc_column(last, TP, t8);   // accumulator column = pass row
        float v[8];
        tmem_sum8(more, sums + (uint32_t)t8, acc, acc + (uint32_t)TP, v);
        if (sends) {
          if (s.kj) st_async_peer(dst + (uint32_t)t8 * 256u, bar, v[0], v[2], v[4], v[6]);
          else st_async_peer(dst + (uint32_t)t8 * 256u, bar, v[1], v[3], v[5], v[7]);
        }
        if (valid) {
#pragma unroll
          for (int u = 0; u < 8; ++u) y[u * 256] = v[u];
        }
      }
    }
    tc_fence_before();
    if (sends) {
      bool ok = false;
      for (unsigned i = 0; i < kSpinLimit; ++i) {
        if (mbar_try_cluster(kbar, kuses & 1u)) { ok = true; break; }
        if (*abort_s) break;
        if (i > 64) __nanosleep(40);
      }
      if (!ok) { *abort_s = 1; atomicOr(&p.cnt->status, kStatTimeout); }
      if (valid) {
#pragma unroll 1
        for (int t8 = 0; t8 < TP; t8 += 8) {
          const float4 o = *reinterpret_cast<const float4 *>(red + t8 * 64 + ctid * 4);
          float *y = ys + (t8 + s.kj) * 256 + rslab;    // rows j, j + 2, j + 4, j + 6 of the eight
          if (s.kj) { y[0] = o.x + y[0]; y[512] = o.y + y[512]; y[1024] = o.z + y[1024]; y[1536] = o.w + y[1536]; }
          else { y[0] += o.x; y[512] += o.y; y[1024] += o.z; y[1536] += o.w; }
        }
      }
    }
    if (pair) ++kuses;
    const int epi = g.epi;
    if (has_ss) {
      named_bar(3, kNumCWarps * 32);
#pragma unroll 1
      for (int wi = cw, k = 0; wi < nitem; wi += kNumCWarps, ++k) {
        const int tq = wi / segs, sg = wi - tq * segs, r = sg * 64 + 2 * lane, t = t0 + tq * tstep;
        const bool in0 = r < s.rows, in1 = r + 1 < s.rows;
        float2 hn = k == 0 ? hold[0] : hold[1], gv = k == 0 ? gn[0] : gn[1];
        if (k >= kAhead) item_old(wi, hn, gv);   // (more items than were fetched ahead)
        const float *y = ys + t * 256 + r;
        hn.x = in0 ? hn.x + y[0] : 0.f;
        hn.y = in1 ? hn.y + y[1] : 0.f;
        float *hp = p.h + (size_t)t * p.d + col0 + r;
        if (in1 && !odd) {
          *reinterpret_cast<float2 *>(hp) = hn;
          xstore2(p.xa, TP, t, col0 + r, hn.x * gv.x, hn.y * gv.y);
        } else {
          if (in0) {
            hp[0] = hn.x;
            xstore(p.xa, TP, t, col0 + r, hn.x * gv.x);
          }
          if (in1) {
            hp[1] = hn.y;
            xstore(p.xa, TP, t, col0 + r + 1, hn.y * gv.y);
          }
        }
        // squares: each half of the piece as a tree over its 32 columns, the halves of a slab one after the other (those of a second
        // piece are left apart; ss_slots)
        float q = __fmul_rn(hn.x, hn.x), q1 = __fmul_rn(hn.y, hn.y);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
          q += __shfl_xor_sync(0xffffffffu, q, o);
          q1 += __shfl_xor_sync(0xffffffffu, q1, o);
        }
        q += q1;
        float *ss = p.ss_part + t * kSsStride + s.group * ss_slots(segs);
        if (sg == 0) {
          q += __shfl_xor_sync(0xffffffffu, q, 16);
          if (lane == 0) ss[0] = q;
        } else if ((lane & 15) == 0) {
          ss[1 + (lane >> 4)] = q;
        }
      }
    } else if (epi != EPI_ARGMAX_LM) {
      named_bar(3, kNumCWarps * 32);
#pragma unroll 1
      for (int e = ctid; e < nflat; e += kNumCWarps * 32) {
        const int t = (int)(((unsigned)e * per_pair) >> 22), r = 2 * (e - t * pairs) - odd;
        const bool in0 = r >= 0, in1 = r + 1 < s.rows;
        const float sc = inv_rms[t];
        const float *y = ys + t * 256 + r;
        float2 v = make_float2(in0 ? y[0] * sc : 0.f, in1 ? y[1] * sc : 0.f);
        if (sw) {
          v.x = (v.x / (1.f + __expf(-v.x))) * (in0 ? y[128] * sc : 0.f);
          v.y = (v.y / (1.f + __expf(-v.y))) * (in1 ? y[129] * sc : 0.f);
          if (in0 && in1) xstore2(p.ac, TP, t, col0 + r, v.x, v.y);
          else if (in0) xstore(p.ac, TP, t, col0 + r, v.x);
          else xstore(p.ac, TP, t, col0 + r + 1, v.y);
        } else {
          float *o = p.qkv + (size_t)t * 3 * p.d + col0 + r;
          if (in0 && in1) *reinterpret_cast<float2 *>(o) = v;
          else if (in0) o[0] = v.x;
          else o[1] = v.y;
        }
      }
    } else {
#pragma unroll 1
      for (int t = 0; t < Tg; ++t) {   // the warp's two largest logits of this pass row
        const int tr = g.lm_rows ? rows->lm_row[t] : t;   // (selected rows: output row t is pass row lm_row[t])
        const float sc = g.scale_inv_rms ? inv_rms[tr] : 1.f;
        const float y = valid ? ys[tr * 256 + rslab] * sc : 0.f;
        Top2 b;
        b.v1 = -INFINITY; b.i1 = 0x7fffffff; b.v2 = -INFINITY;
        if (valid) {
          if (p.logits) {
            const int slot_out = g.lm_rows ? rows->lm_out[t] : rows->out[t];
            p.logits[(size_t)slot_out * p.V + vrow] = y;
          }
          b.v1 = y; b.i1 = vrow;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) b = top2_shfl_xor(b, o);
        if (lane == 0) topw[cw * kPassRowsMax + t] = b;
        if (p.lp_out) {
          // for the log-probability of the chosen token: sum of exp(logit - warp maximum), and the logit of a
          // forced token where one is given
          const float e = warp_sum(valid ? __expf(y - b.v1) : 0.f);
          if (lane == 0) lps[cw * 16 + t] = e;
          if (valid && p.forced) {
            const int slot_out = g.lm_rows ? rows->lm_out[t] : rows->out[t];
            if (p.forced[slot_out] == vrow) p.tok_logit[slot_out] = y;
          }
        }
      }
    }
    if (epi == EPI_ARGMAX_LM) {
      named_bar(3, kNumCWarps * 32);
      if (ctid < Tg) {
        Top2 b = topw[ctid];
        for (int w = 1; w < kNumCWarps; ++w) b = top2_merge(b, topw[w * kPassRowsMax + ctid]);
        float se = 0.f;   // sum of exp(logit - this CTA's maximum) over the CTA's vocabulary rows
        if (p.lp_out)
          for (int w = 0; w < kNumCWarps; ++w) {
            const float mw = topw[w * kPassRowsMax + ctid].v1;
            if (mw > -INFINITY) se += lps[w * 16 + ctid] * __expf(mw - b.v1);
          }
        p.amax[(size_t)cta * kPassRowsMax + ctid] = make_float4(b.v1, __int_as_float(b.i1), b.v2, se);
      }
    }
    stamp(p, ph, 3, stamper);
    phase_arrive();
    arrived = true;

    if (g.epi != EPI_ARGMAX_LM) continue;
    phase_await();
    arrived = false;
    if (cta == 0 || p.mode == 1) {   // (every CTA needs the token of the next draft step)
      // greedy choice per row: the candidates of all CTAs merged (largest value, lowest index among equals, so
      // any merge order gives the same result).  Warp w takes rows 2w and 2w + 1 (of each 16), 16 lanes per row, each lane
      // the CTAs congruent to it mod 16 with all its loads in flight at once.
#pragma unroll 1
      for (int r0 = 0; r0 < Tg; r0 += 2 * kNumCWarps) {
      const int row = r0 + 2 * cw + (lane >> 4), l16 = lane & 15;
      Top2 b;
      b.v1 = -INFINITY; b.i1 = 0x7fffffff; b.v2 = -INFINITY;
      if (row < Tg) {
        float4 c4[10];
#pragma unroll
        for (int k = 0; k < 10; ++k) {
          const int i = l16 + 16 * k;
          c4[k] = i < ncta ? __ldcg(p.amax + (size_t)i * kPassRowsMax + row) : make_float4(-INFINITY, __int_as_float(0x7fffffff), -INFINITY, 0.f);
        }
#pragma unroll
        for (int k = 0; k < 10; ++k) {
          Top2 x; x.v1 = c4[k].x; x.i1 = __float_as_int(c4[k].y); x.v2 = c4[k].z;
          b = top2_merge(b, x);
        }
        for (int i = l16 + 160; i < ncta; i += 16) {   // grids beyond 160 CTAs
          const float4 c = __ldcg(p.amax + (size_t)i * kPassRowsMax + row);
          Top2 x; x.v1 = c.x; x.i1 = __float_as_int(c.y); x.v2 = c.z;
          b = top2_merge(b, x);
        }
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) b = top2_shfl_xor(b, o);
      float se = 0.f;   // sum over the vocabulary of exp(logit - maximum): the CTAs' sums rescaled to the global maximum
      if (p.lp_out) {
        if (row < Tg)
          for (int i = l16; i < ncta; i += 16) {
            const float4 c = __ldcg(p.amax + (size_t)i * kPassRowsMax + row);
            if (c.x > -INFINITY) se += c.w * __expf(c.x - b.v1);
          }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
      }
      if (row < Tg && l16 == 0) {
        const int slot_out = g.lm_rows ? rows->lm_out[row] : rows->out[row];
        const int token = p.forced ? p.forced[slot_out] : b.i1;
        // log softmax of the token that goes out: its logit minus (maximum + log of the sum)
        const float lp = p.lp_out ? (p.forced ? __ldcg(p.tok_logit + slot_out) - b.v1 : 0.f) - __logf(se) : 0.f;
        if (cta == 0) {
          p.tok_out[slot_out] = token;
          if (p.top_out) p.top_out[slot_out] = make_float2(b.v1, b.v2);
          if (p.lp_out) p.lp_out[slot_out] = lp;
        }
        if (p.mode == 1) { rows->cur[rows->s_b[row]] = token; rows->lp = lp; }
        else rows->choice[row] = token;
      }
      }
    }
  }
  // ---- accept (CTA 0; the rows' tokens past a sequence's first are its draft).  Row list and accepting in the pass instead of
  // launches before and after it: tiny model, a step of 4 drafts 235 -> 232 us, four sequences 287 -> 283 us.
  if (!PROMPT && p.mode == 0 && p.accept && cta == 0) {
    named_bar(3, kNumCWarps * 32);
    if (ctid < p.B) {
      int i = 0;
      while (i < rows->nseq && rows->s_b[i] != ctid) ++i;
      const bool part = i < rows->nseq;
      accept_sequence(p.st, p.tok, p.cap, p.tok_stride, part ? rows->tok + rows->s_row0[i] + 1 : nullptr,
                      part ? rows->choice + rows->s_row0[i] : nullptr, p.nmax, ctid, p.cnt, nullptr, 0, p.acc_out, p.emit_out, p.nemit_out,
                      nullptr);
    }
  }
  // ---- the next draft step: its rows, and with the stopping rule of Section 4 whether there is one.  Every CTA comes to
  // the same decision.
  if (p.mode == 1 && !PROMPT) {
    named_bar(3, kNumCWarps * 32);
    if (ctid == 0) {
      const int made = step + 1;
      int n = rows->n[0];
      if (p.ddd_thr < 0.f && made >= n) {
        // the running log-probability takes the new token's; at the predicted length and still at or above the
        // threshold the draft grows by one token, within n_max and the cache (len + n + 1 <= cap)
        rows->cum = (step == 0 ? 0.f : rows->cum) + rows->lp;
        const int room = p.cap - (rows->j[0] + 1) - 1;
        if (made < p.nmax && made < room && !(rows->cum < p.ddd_thr)) n = made + 1;
        *reinterpret_cast<volatile int *>(&rows->n[0]) = n;
        mbar_arrive(step_bar);
      } else if (p.ddd_thr < 0.f) {
        rows->cum = (step == 0 ? 0.f : rows->cum) + rows->lp;
      }
      if (p.ddd_thr < 0.f ? made < n : made < nstep) draft_rows_of_step(rows, p, made);
      else if (cta == 0) {   // the draft is complete
        for (int b = 0; b < p.B; ++b)
          if (rows->n[b] > 0 && p.step0 == 0) {
            p.st[b].dlen = rows->j[b];
            if (p.ddd_thr < 0.f) p.st[b].n = n;
          }
      }
    }
    named_bar(6, kBarThreads);
    if (p.ddd_thr < 0.f) nstep = rows->n[0];
  }
  if (arrived) phase_await();   // (a prompt's pass of the draft head ends with its layer)
  }
  // let warp 2 free the tensor memory once every worker has made its last read
  await_copies(abort_s);
  tc_fence_before();
  named_bar(5, 32 + kNumCWarps * 32);
}

// Self-test of the bounded waits: the same wait routines as the pass kernel, on a barrier nobody arrives at (mode 0:
// an mbarrier phase that never completes; mode 1: a grid-barrier count that is never reached), with a small limit.
// Both give up, set the time-out bit of the status word and return; result[mode] receives 1 when the wait returned.
__global__ void __launch_bounds__(kPassThreads, 1) k_wait_selftest(unsigned *gbar, Counters *cnt, unsigned limit, int mode,
                                                                   int *result) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5;
  if (tid == 0) {
    abort_flag = 0;
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (mode == 0) {
    if (tid == 0) {
      mbar_wait(&bar, 0u, cnt, &abort_flag, limit);
      await_copies(&abort_flag);
      result[0] = 1;
    }
  } else if (warp == 1) {   // as in the pass kernel: warp 1 stands for the CTA
    named_bar(2, kBarThreads);
    if (tid == 32) grid_wait(gbar, cnt, 2u * gridDim.x, &abort_flag, limit);   // one CTA arrives, two are awaited
    __syncwarp();
    named_arrive(4, kBarThreads);
    if (tid == 32) result[1] = 1;
  } else if (warp >= kFirstWorker) {
    phase_arrive();
    phase_await();
  }
}

}  // namespace ada
