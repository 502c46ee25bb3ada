// Device kernels of the adaptive speculative-decoding iteration (sm_100a).
//
// Numerics shared by all kernels: weights are bf16, KV caches 16-bit half (see kv_store); the residual
// stream, norms, softmax, every accumulator and every GEMM output are fp32.
// A GEMM input row x is carried as two bf16 rows hi = bf16(x), lo = bf16(x - hi);
// the tensor-core product W*hi + W*lo then equals W*x to ~2^-17 relative, which
// keeps logits within 2e-2 of an fp32 evaluation over 40 layers.  Every output
// element depends only on its own input row and on a fixed split of K, never on
// how many rows share the launch, so speculative and autoregressive runs of the
// library agree bit for bit.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "ada_ldlp.cuh"

namespace ada {

constexpr int kMaxBatch = 8;
constexpr int kPageSize = 64;   // positions per cache page (the configuration accepts no other): divisions by it are shifts
constexpr int kMaxRows = 1024;  // rows of one pass (all sequences together): a prompt chunk
constexpr int kAttnSplits = 8;  // KV splits per (sequence, head)
constexpr int kRowGroup = 16;   // rows of an m16 tile (attention of decode passes: the hi and the lo halves of 8 query rows)
constexpr int kTcRows = 88;     // rows of a decode pass of a batch at most (8 sequences x 11 rows)

// status bits (device status word)
constexpr int kStatKvFull = 1;
constexpr int kStatStale = 2;

struct SeqState {
  int len;     // committed tokens, the last one pending (its row is not in the target cache)
  int dlen;    // draft-cache rows computed from target features
  int n;       // draft length of this iteration
  int k_acc;   // accepted drafts of the last accept
  int j_prev;  // index of the pending token when the last verify started
  int n_emit;  // tokens emitted by the last accept
  int stale;   // draft head is behind by more rows than one pass holds
  int chunk;   // keys per attention split of this sequence's caches, fixed when its prompt was read (multiple of 32)
};

struct Counters {
  unsigned long long n_target, n_draft, n_waste, n_tokens;
  int status;
  int pad;
};

// Row list of the pass being computed.  Rows of one sequence are contiguous.
struct Pass {
  int T;                   // rows in this pass
  int lmT;                 // rows that go through the LM head (draft: one per active sequence)
  int row_seq[kMaxRows];
  int row_pos[kMaxRows];   // absolute position (RoPE angle, cache row)
  int row_tok[kMaxRows];   // token whose embedding enters the row
  int row_out[kMaxRows];   // output slot of the row
  int lm_row[kMaxRows];    // draft: pass row of LM row i
  int lm_out[kMaxRows];    // draft: output slot of LM row i
  int seq_row0[kMaxBatch];
  int seq_rows[kMaxBatch];
  int seq_chunk[kMaxBatch];   // keys per attention split of the sequence (SeqState::chunk)
  int4 seq_info[kMaxBatch];   // (seq_row0, seq_rows, seq_chunk, position of the first row): one load for the attention kernels
};

// Last step of every kernel that fills a row list.
__device__ __forceinline__ void pass_seal(Pass *pass, int B) {
  for (int b = 0; b < B; ++b) {
    const int r0 = pass->seq_row0[b], n = pass->seq_rows[b];
    pass->seq_info[b] = make_int4(r0, n, pass->seq_chunk[b], n > 0 ? pass->row_pos[r0] : 0);
  }
}

// KV-cache element: 16 bits per value like the weights, but IEEE half (11-bit significand) rather than bf16
// (8-bit): with bf16 keys and values the logits of a 32-layer stack were measured 0.03-0.05 away from the
// fp32 oracle (rounding of 2^-9 per layer), with half they stay inside the 2e-2 bound.  The pools are typed
// __nv_bfloat16 only as a 16-bit container; these three functions are the only ones that interpret the bits.
__device__ __forceinline__ __nv_bfloat16 kv_store(float x) {
  return __ushort_as_bfloat16(__half_as_ushort(__float2half_rn(x)));
}
__device__ __forceinline__ float kv_lo(uint32_t pair) { return __half2float(__ushort_as_half((unsigned short)(pair & 0xffffu))); }
__device__ __forceinline__ float kv_hi(uint32_t pair) { return __half2float(__ushort_as_half((unsigned short)(pair >> 16))); }

// Programmatic dependent launch.  A kernel launched with the programmatic-serialization attribute may start while the
// kernel before it in the stream still runs; pdl_wait returns once that kernel has completed and its writes are
// visible (at once if there is no such dependency).  Every thread of such a kernel waits before it touches memory
// another kernel writes and before it returns, so completion of a kernel implies completion of all before it.
// pdl_launch_dependents lets the kernel after this one begin its own prologue.  Before its wait such a kernel may read weights and
// the row list (Pass, page table): the chain of a pass begins with a kernel that is launched plainly after the one that makes the
// list and lets none start before it has completed, and the list is rewritten only after the chain.  (A kernel's lookups one behind
// the other, 0.4 to 1 us of its 3, then go on while the one before it finishes, and so do the first copies of old cache rows.  Verify
// of eight sequences: 16 layers of 2048 1242 -> 1134 us, 7B 4531 and 4530.  Prompts of 49 and 64 rows: 16 layers of 2048 1227 -> 1138
// and 1250 -> 1165 us, 13B 7168 -> 7038 and 7236 -> 7254, 7B 4125 -> 4167 and 4261 -> 4262.)
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void split_bf16(float x, __nv_bfloat16 &hi, __nv_bfloat16 &lo) {
  hi = __float2bfloat16_rn(x);
  lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// block-wide sum for blockDim.x <= 1024, result to all threads
__device__ __forceinline__ float block_sum(float v, float *sh) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  float t = 0.f;
  for (int i = 0; i < nw; ++i) t += sh[i];  // fixed order
  return t;
}

// ---------------------------------------------------------------------------------------------
// top-2 bookkeeping for the greedy choice: (v1, i1) best value / lowest index among equals, v2 second
struct Top2 {
  float v1;
  int i1;
  float v2;
};
__device__ __forceinline__ Top2 top2_merge(Top2 a, Top2 b) {
  Top2 r;
  const bool a_wins = (a.v1 > b.v1) || (a.v1 == b.v1 && a.i1 <= b.i1);
  if (a_wins) {
    r.v1 = a.v1; r.i1 = a.i1; r.v2 = fmaxf(a.v2, b.v1);
  } else {
    r.v1 = b.v1; r.i1 = b.i1; r.v2 = fmaxf(b.v2, a.v1);
  }
  return r;
}
__device__ __forceinline__ Top2 top2_shfl_xor(Top2 a, int m) {
  Top2 b;
  b.v1 = __shfl_xor_sync(0xffffffffu, a.v1, m);
  b.i1 = __shfl_xor_sync(0xffffffffu, a.i1, m);
  b.v2 = __shfl_xor_sync(0xffffffffu, a.v2, m);
  return top2_merge(a, b);
}

// ---------------------------------------------------------------------------------------------
// Epilogues of the multi-row GEMM (ada_gemm_tc.cuh).
enum { EPI_STORE = 0, EPI_RESID = 1, EPI_SWIGLU = 2, EPI_ARGMAX = 3 };

// Final greedy choice per row: merge the per-tile candidates in tile order.
// tok_out[slot] = argmax; top_out[slot] = (top1, top2).  forced (optional) overrides the token.
__global__ void k_argmax_final(const float4 *amax, int tiles, int TP, const Pass *pass, int use_lm_rows,
                               int *tok_out, float2 *top_out, const int *forced) {
  const int T = use_lm_rows ? pass->lmT : pass->T;
  const int t = blockIdx.x;
  if (t >= T) return;
  Top2 b;
  b.v1 = -INFINITY; b.i1 = 0x7fffffff; b.v2 = -INFINITY;
  for (int i0 = threadIdx.x; i0 < tiles; i0 += 4 * 32) {   // a lane's four candidates of a round in flight together
    float4 c[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      c[u] = i0 + 32 * u < tiles ? amax[(size_t)(i0 + 32 * u) * TP + t] : make_float4(-INFINITY, __int_as_float(0x7fffffff), -INFINITY, 0.f);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      Top2 x; x.v1 = c[u].x; x.i1 = __float_as_int(c[u].y); x.v2 = c[u].z;
      b = top2_merge(b, x);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) b = top2_shfl_xor(b, o);
  if (threadIdx.x == 0) {
    const int slot = use_lm_rows ? pass->lm_out[t] : pass->row_out[t];
    tok_out[slot] = forced ? forced[slot] : b.i1;
    if (top_out) top_out[slot] = make_float2(b.v1, b.v2);
  }
}

// ---------------------------------------------------------------------------------------------
// h[t][:] = embedding of row_tok[t]; planes = split(h * gain) of the first layer's norm; the row's sum of squares
// (slot 0 of the row's segments, the others zero: see the reduction kernels of the multi-row GEMM).
__global__ void k_embed(const Pass *pass, const __nv_bfloat16 *embed, float *h, int d, const __nv_bfloat16 *gain,
                        __nv_bfloat16 *xhi, __nv_bfloat16 *xlo, int ldx, float *ss_part, int ss_segs) {
  __shared__ float sh[32];
  const int t = blockIdx.x;
  if (t >= pass->T) return;
  const __nv_bfloat16 *__restrict__ e = embed + (size_t)pass->row_tok[t] * d;
  float *__restrict__ hr = h + (size_t)t * d;
  float ss = 0.f;
#pragma unroll 8
  for (int i = threadIdx.x; i < d; i += blockDim.x) {   // (loads of a row in flight together)
    const float v = __bfloat162float(e[i]);
    hr[i] = v;
    ss += v * v;
    __nv_bfloat16 hi, lo;
    split_bf16(v * __bfloat162float(gain[i]), hi, lo);
    xhi[(size_t)t * ldx + i] = hi;
    xlo[(size_t)t * ldx + i] = lo;
  }
  ss = block_sum(ss, sh);
  if (threadIdx.x < ss_segs) ss_part[(size_t)t * ss_segs + threadIdx.x] = threadIdx.x == 0 ? ss : 0.f;
}

// x = h / sqrt(mean(h^2) + eps) * gain  ->  hi/lo halves; optionally also fp32 rows to
// feat[(seq*cap + pos)][d] (the target feature f after the final norm).
__global__ void k_rmsnorm(const Pass *pass, const float *h, const __nv_bfloat16 *gain, float eps, int d,
                          __nv_bfloat16 *xhi, __nv_bfloat16 *xlo, int ldx, float *feat, int cap) {
  __shared__ float sh[32];
  const int t = blockIdx.x;
  if (t >= pass->T) return;
  // four elements per thread and step (d is a multiple of 64), the steps unrolled so that a row's loads are in
  // flight together: one element per step ran at one level-2 round trip per step
  const float4 *__restrict__ h4 = reinterpret_cast<const float4 *>(h + (size_t)t * d);
  const int d4 = d >> 2;
  float ss = 0.f;
#pragma unroll 4
  for (int i = threadIdx.x; i < d4; i += blockDim.x) {
    const float4 v = h4[i];
    ss += (v.x * v.x + v.y * v.y) + (v.z * v.z + v.w * v.w);
  }
  ss = block_sum(ss, sh);
  const float inv = rsqrtf(ss / (float)d + eps);
  float4 *__restrict__ fr =
      feat ? reinterpret_cast<float4 *>(feat + ((size_t)pass->row_seq[t] * cap + pass->row_pos[t]) * d) : nullptr;
  const uint2 *__restrict__ g4 = reinterpret_cast<const uint2 *>(gain);
  uint2 *__restrict__ oh = reinterpret_cast<uint2 *>(xhi + (size_t)t * ldx);
  uint2 *__restrict__ ol = reinterpret_cast<uint2 *>(xlo + (size_t)t * ldx);
#pragma unroll 4
  for (int i = threadIdx.x; i < d4; i += blockDim.x) {
    const float4 v = h4[i];
    const uint2 gg = g4[i];
    const __nv_bfloat162 g01 = *reinterpret_cast<const __nv_bfloat162 *>(&gg.x), g23 = *reinterpret_cast<const __nv_bfloat162 *>(&gg.y);
    float4 x;
    x.x = (v.x * inv) * __bfloat162float(g01.x); x.y = (v.y * inv) * __bfloat162float(g01.y);
    x.z = (v.z * inv) * __bfloat162float(g23.x); x.w = (v.w * inv) * __bfloat162float(g23.y);
    __nv_bfloat16 hi[4], lo[4];
    split_bf16(x.x, hi[0], lo[0]); split_bf16(x.y, hi[1], lo[1]);
    split_bf16(x.z, hi[2], lo[2]); split_bf16(x.w, hi[3], lo[3]);
    uint2 ph, pl;
    ph.x = (uint32_t)__bfloat16_as_ushort(hi[0]) | ((uint32_t)__bfloat16_as_ushort(hi[1]) << 16);
    ph.y = (uint32_t)__bfloat16_as_ushort(hi[2]) | ((uint32_t)__bfloat16_as_ushort(hi[3]) << 16);
    pl.x = (uint32_t)__bfloat16_as_ushort(lo[0]) | ((uint32_t)__bfloat16_as_ushort(lo[1]) << 16);
    pl.y = (uint32_t)__bfloat16_as_ushort(lo[2]) | ((uint32_t)__bfloat16_as_ushort(lo[3]) << 16);
    oh[i] = ph;
    ol[i] = pl;
    if (fr) fr[i] = x;
  }
}

// hi/lo halves of selected rows of h without normalisation (draft head output -> LM head);
// also keeps the fp32 row as the head's own feature for its next step.
__global__ void k_split_lm_rows(const Pass *pass, const float *h, int d, __nv_bfloat16 *xhi,
                                __nv_bfloat16 *xlo, int ldx, float *dfeat, int nmax, int step) {
  const int i = blockIdx.x;
  if (i >= pass->lmT) return;
  const int t = pass->lm_row[i];
  const int b = pass->row_seq[t];
  const float *__restrict__ hr = h + (size_t)t * d;
  float *__restrict__ fo = dfeat + ((size_t)b * nmax + step) * d;
  __nv_bfloat16 *__restrict__ oh = xhi + (size_t)i * ldx, *__restrict__ ol = xlo + (size_t)i * ldx;
#pragma unroll 8
  for (int c = threadIdx.x; c < d; c += blockDim.x) {   // (loads of eight steps in flight together)
    const float x = hr[c];
    __nv_bfloat16 hi, lo;
    split_bf16(x, hi, lo);
    oh[c] = hi;
    ol[c] = lo;
    fo[c] = x;
  }
}

// Keys per attention split of a sequence whose prompt has m tokens, in a cache of `cap` positions, for a model of H
// heads: as many splits as keep heads x splits within the persistent kernel's 148 CTAs (four at most: 32 heads -> 4,
// 40 heads -> 3) cover the prompt and the tokens expected after it (a quarter as many again, at least 256, within the
// capacity); at least 256 keys, and at least cap / 32 so that no sequence has more than 32 splits.  Chosen once per sequence, from its prompt
// alone: the split a key falls in must not depend on the shape of the pass that reads it (a one-row step and a block of
// drafts then sum in the same order).
__host__ __device__ __forceinline__ int attn_chunk_for_prompt(int m, int cap, int H) {
  const int grow = m / 4 > 256 ? m / 4 : 256;
  const int total = m + grow < cap ? m + grow : cap;
  int nsplit = H > 0 ? 148 / H : 4;
  nsplit = nsplit < 1 ? 1 : (nsplit > 4 ? 4 : nsplit);
  int chunk = ((total + nsplit - 1) / nsplit + 31) / 32 * 32;
  // 256 keys at least: eight warps take 128 of them in about a microsecond, merging splits takes two, and a context within
  // one split needs no merge (small model, context 100: attention phase 6.5 -> 4.6 us)
  int least = ((cap + 31) / 32 + 31) / 32 * 32;
  if (least < 256) least = 256;
  return chunk < least ? least : chunk;
}
// The multi-row attention kernel takes at most kAttnSplits splits per sequence: its split size is the sequence's, or
// cap / kAttnSplits if that is larger (again independent of the pass).
__host__ __device__ __forceinline__ int attn_rows_chunk(int seq_chunk, int cap) {
  const int least = ((cap + kAttnSplits - 1) / kAttnSplits + 31) / 32 * 32;
  const int c = seq_chunk < 32 ? 32 : seq_chunk;
  return c < least ? least : c;
}

// Merge the cache splits in split order and emit the attention output row as hi/lo halves.
template <int HD>
__global__ void k_attn_combine(const Pass *pass, const float *part, __nv_bfloat16 *xhi, __nv_bfloat16 *xlo,
                               int ldx, int cap) {
  pdl_launch_dependents();
  const int hh = blockIdx.x, t = blockIdx.y;
  const bool live = t < pass->T;
  const int4 si = live ? pass->seq_info[pass->row_seq[t]] : make_int4(0, 0, 0, 0);
  const int c = threadIdx.x;
  const float *base = part + (((size_t)hh * kAttnSplits) * kTcRows + t) * (HD + 2);
  const size_t sstride = (size_t)kTcRows * (HD + 2);
  const int nkeys = si.w + si.y;
  const int chunk = attn_rows_chunk(si.z, cap);
  pdl_wait();
  if (!live) return;
  const int nsp = (nkeys + chunk - 1) / chunk;  // splits that held keys (at most kAttnSplits)
  float ms[kAttnSplits], ls[kAttnSplits], os[kAttnSplits];
#pragma unroll
  for (int s = 0; s < kAttnSplits; ++s) {       // all loads first: one round trip
    ms[s] = -INFINITY; ls[s] = 0.f; os[s] = 0.f;
    if (s < nsp) { ms[s] = base[s * sstride + HD]; ls[s] = base[s * sstride + HD + 1]; os[s] = base[s * sstride + c]; }
  }
  float M = -INFINITY;
#pragma unroll
  for (int s = 0; s < kAttnSplits; ++s) M = fmaxf(M, ms[s]);
  float l = 0.f, o = 0.f;
#pragma unroll
  for (int s = 0; s < kAttnSplits; ++s)
    if (s < nsp) {
      const float e = __expf(ms[s] - M);
      l += ls[s] * e;
      o += os[s] * e;
    }
  const float x = o / l;
  __nv_bfloat16 hi, lo;
  split_bf16(x, hi, lo);
  xhi[(size_t)t * ldx + hh * HD + c] = hi;
  xlo[(size_t)t * ldx + hh * HD + c] = lo;
}

// ---------------------------------------------------------------------------------------------
// Draft-head input rows: X[t] = [embedding(row_tok[t]) ; feature] as hi/lo halves (K = 2d).
// Catch-up rows (step 0) read the target feature of their position; later steps read the head's
// own previous output dfeat[seq][step-1].
__global__ void k_eagle_input(const Pass *pass, const __nv_bfloat16 *embed, const float *feat, int feat_stride,
                              const float *dfeat, int nmax, int step, int d, __nv_bfloat16 *xhi,
                              __nv_bfloat16 *xlo, int ldx) {
  const int t = blockIdx.x;
  if (t >= pass->T) return;
  const int b = pass->row_seq[t];
  const __nv_bfloat16 *e = embed + (size_t)pass->row_tok[t] * d;
  const float *f = step == 0 ? feat + ((size_t)b * feat_stride + pass->row_pos[t]) * d
                             : dfeat + ((size_t)b * nmax + (step - 1)) * d;
  __nv_bfloat16 *__restrict__ oh = xhi + (size_t)t * ldx, *__restrict__ ol = xlo + (size_t)t * ldx;
  const __nv_bfloat16 *__restrict__ er = e;
  const float *__restrict__ fr = f;
#pragma unroll 8
  for (int i = threadIdx.x; i < d; i += blockDim.x) {   // (loads of eight steps in flight together)
    const __nv_bfloat16 ev = er[i];
    const float fv = fr[i];
    oh[i] = ev;
    ol[i] = __float2bfloat16_rn(0.f);
    __nv_bfloat16 hi, lo;
    split_bf16(fv, hi, lo);
    oh[d + i] = hi;
    ol[d + i] = lo;
  }
}

// ---------------------------------------------------------------------------------------------
// Length predictor (Eq. 3), class-logit form.  Stage 1: h[b] = ReLU(W1 [e(tok[len-2]) ; f[len-2]] + b1), four hidden units
// per block (see ada_ldlp.cuh; d is a multiple of 64 and every tensor 16-byte aligned).  7B widths, both stages: 28 us
// with a warp per unit and a plain launch of the second, 13.8 us now (with the launch overhead of separate calls).
__global__ void __launch_bounds__(kLdlpThreads) k_ldlp_hidden(const SeqState *st, const int *tok, const float *feat, int cap,
                                                              const __nv_bfloat16 *embed, const __nv_bfloat16 *w1,
                                                              const __nv_bfloat16 *b1, int d, int hid, float *hbuf) {
  pdl_launch_dependents();
  const int b = blockIdx.y, p = st[b].len - 2;
  if (p < 0) return;
  ldlp_hidden_block<true>(w1, b1, embed + (size_t)tok[(size_t)b * cap + p] * d, feat + ((size_t)b * cap + p) * d, d, hid,
                          blockIdx.x * kLdlpUnits, hbuf + (size_t)b * hid);
}

// Scalar form (Eq. 3), one residual block: hout = hin + ReLU(W_r hin + b_r).  One warp per unit.
__global__ void k_ldlp_block(const SeqState *st, const float *hin, float *hout, const __nv_bfloat16 *wr,
                             const __nv_bfloat16 *br, int hid) {
  pdl_launch_dependents();
  const int b = blockIdx.y;
  const int u = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  const __nv_bfloat16 *w = wr + (size_t)u * hid;
  LdlpRow row;
  const bool vec = (hid & 7) == 0 && (reinterpret_cast<uintptr_t>(wr) & 15) == 0;
  if (vec && u < hid) ldlp_out_ahead<true>(w, hid, row);
  pdl_wait();
  if (u >= hid || st[b].len < 2) return;
  const float *h = hin + (size_t)b * hid;
  const float s = vec ? ldlp_out_dot<true>(w, h, hid, row) : ldlp_out_dot<false>(w, h, hid, row);
  if (lane == 0) hout[(size_t)b * hid + u] = __ldcg(h + u) + fmaxf(s + __bfloat162float(br[u]), 0.f);
}

// Stage 2: z = W2 h + b2, then n = argmax + 1 (class form, lowest index among equals) or
// n = clip(round-half-even(z_0), k_min, n_max) (scalar form, Eq. 3), then the override and the clip to the
// cache capacity.  One CTA per sequence, one warp per output (16 warps: n_max <= 15).
__global__ void __launch_bounds__(512) k_ldlp_out(SeqState *st, const float *hbuf, const __nv_bfloat16 *w2, const __nv_bfloat16 *b2,
                                                  int hid, int nmax, int mode, int kmin, int cap, const int *force_n, int has_force,
                                                  float *zbuf, int *n_out, Counters *cnt) {
  __shared__ float zs[16];
  const int b = blockIdx.x, lane = threadIdx.x & 31, c = threadIdx.x >> 5;
  const int nz = mode == 0 ? nmax : 1;
  LdlpRow row;
  const bool vec = (hid & 7) == 0;
  if (vec && c < nz) ldlp_out_ahead<true>(w2 + (size_t)c * hid, hid, row);
  pdl_wait();
  const int len = st[b].len;
  if (len < 2) { if (threadIdx.x == 0) { st[b].n = 0; if (n_out) n_out[b] = 0; } return; }
  if (c < nz) {
    const __nv_bfloat16 *w = w2 + (size_t)c * hid;
    const float *h = hbuf + (size_t)b * hid;
    const float s = (vec ? ldlp_out_dot<true>(w, h, hid, row) : ldlp_out_dot<false>(w, h, hid, row)) + __bfloat162float(b2[c]);
    if (lane == 0) { zs[c] = s; zbuf[b * 16 + c] = s; }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float best = -INFINITY;
    int bi = 0;
    for (int i = 0; i < nz; ++i)
      if (zs[i] > best) { best = zs[i]; bi = i; }
    int n = bi + 1;
    if (mode != 0) n = (int)fminf(fmaxf(rintf(best), (float)kmin), (float)nmax);   // best = z_0
    if (has_force) n = force_n[b];
    const int room = cap - len - 1;  // the n + 1 tokens this iteration may commit must fit: len + n + 1 <= cap
    if (n > room) { n = room < 0 ? 0 : room; atomicOr(&cnt->status, kStatKvFull); }
    st[b].n = n;
    if (n_out) n_out[b] = n;
  }
}

// n[b] <- user array (separate-call API), with the same clip
__global__ void k_set_n(SeqState *st, const int *n_in, int B, int nmax, int cap, Counters *cnt) {
  const int b = threadIdx.x;
  if (b >= B) return;
  int n = n_in[b];
  n = max(0, min(n, nmax));
  const int room = cap - st[b].len - 1;
  if (n > room) { n = room < 0 ? 0 : room; atomicOr(&cnt->status, kStatKvFull); }
  st[b].n = n;
}

// ---------------------------------------------------------------------------------------------
// Row lists.  One thread block; B <= 8, rows <= kMaxRows.
//
// Verify (Eq. 1): rows of sequence b = pending token then its n drafts, positions j..j+n.
// tok[seq * tok_stride + position]: committed tokens (stride 0: all sequences are start positions of one text).
__global__ void k_rows_verify(Pass *pass, SeqState *st, const int *tok, int tok_stride, int cap, const int *draft, int nmax, int B,
                              int only_seq) {
  if (threadIdx.x != 0) return;
  int T = 0;
  for (int b = 0; b < B; ++b) {
    pass->seq_row0[b] = T;
    pass->seq_rows[b] = 0;
    pass->seq_chunk[b] = st[b].chunk;
    if (only_seq >= 0 && b != only_seq) continue;
    const int len = st[b].len;
    if (len < 1) continue;
    const int j = len - 1, n = st[b].n;
    if (len + n + 1 > cap) continue;  // a full sequence takes no further step
    st[b].j_prev = j;
    for (int i = 0; i <= n; ++i) {
      pass->row_seq[T] = b;
      pass->row_pos[T] = j + i;
      pass->row_tok[T] = i == 0 ? tok[(size_t)b * tok_stride + j] : draft[b * nmax + i - 1];
      pass->row_out[T] = b * (nmax + 1) + i;
      ++T;
    }
    pass->seq_rows[b] = n + 1;
  }
  pass->T = T;
  pass->lmT = T;
  pass_seal(pass, B);
}

// Prompt chunk: rows pos0..pos0+R-1 of sequence b, tokens from the committed-token array; the greedy choice (if one is
// asked for) is taken after the last row.
__global__ void k_rows_chunk(Pass *pass, const int *tok, int cap, int b, int pos0, int R, int tok_shift, int B, int chunk) {
  for (int i = threadIdx.x; i < R; i += blockDim.x) {
    pass->row_seq[i] = b;
    pass->row_pos[i] = pos0 + i;
    pass->row_tok[i] = tok[(size_t)b * cap + pos0 + i + tok_shift];
    pass->row_out[i] = i;
  }
  if (threadIdx.x != 0) return;
  for (int i = 0; i < B; ++i) {
    pass->seq_row0[i] = 0;
    pass->seq_rows[i] = i == b ? R : 0;
    pass->seq_chunk[i] = chunk;
    pass->seq_info[i] = make_int4(0, i == b ? R : 0, chunk, pos0);
  }
  pass->lm_row[0] = R - 1;
  pass->lm_out[0] = 0;
  pass->T = R;
  pass->lmT = 1;
}

// Draft (Eq. 2).  step 0: catch-up rows p = dlen..j-1 of every sequence with n >= 1; row p pairs the
// target feature of p with the embedding of token p+1; the last row feeds the LM head.
// step s >= 1: one row per sequence with n > s at position j+s-1, token = draft[s-1].
__global__ void k_rows_draft(Pass *pass, SeqState *st, const int *tok, int tok_stride, const int *draft, int nmax, int B,
                             int step, int max_rows, Counters *cnt) {
  if (threadIdx.x != 0) return;
  int T = 0, lmT = 0;
  for (int b = 0; b < B; ++b) {
    pass->seq_row0[b] = T;
    pass->seq_rows[b] = 0;
    pass->seq_chunk[b] = st[b].chunk;
    const int n = st[b].n, j = st[b].len - 1;
    if (n <= step || j < 1) continue;
    if (step == 0) {
      int R = j - st[b].dlen, p0 = st[b].dlen;
      // already up to date (a second draft from the same state, e.g. after a label pass): the row of position
      // j - 1 is computed again -- same inputs, same cache row -- because its output yields the first draft token
      if (R == 0) { R = 1; p0 = j - 1; }
      if (R < 1 || T + R > max_rows || st[b].stale) { st[b].n = 0; atomicOr(&cnt->status, kStatStale); continue; }
      for (int i = 0; i < R; ++i) {
        const int p = p0 + i;
        pass->row_seq[T] = b;
        pass->row_pos[T] = p;
        pass->row_tok[T] = tok[(size_t)b * tok_stride + p + 1];
        pass->row_out[T] = 0;
        ++T;
      }
      pass->seq_rows[b] = R;
      st[b].dlen = j;
    } else {
      pass->row_seq[T] = b;
      pass->row_pos[T] = j + step - 1;
      pass->row_tok[T] = draft[b * nmax + step - 1];
      pass->row_out[T] = 0;
      ++T;
      pass->seq_rows[b] = 1;
    }
    pass->lm_row[lmT] = T - 1;
    pass->lm_out[lmT] = b * nmax + step;
    ++lmT;
  }
  pass->T = T;
  pass->lmT = lmT;
  pass_seal(pass, B);
}

// ---------------------------------------------------------------------------------------------
// Accept (Eq. 1 and the footnote of Section 3.1) and roll-back of sequence b (one thread): draft[k] its draft, target[i] the
// target's choice after row i.  forced_count > 0 (force_commit): accept count - 1 drafts and take the bonus from forced_tok
// instead of the target's choice.
__device__ __forceinline__ void accept_sequence(SeqState *st, int *tok, int cap, int tok_stride, const int *draft, const int *target,
                                                int nmax, int b, Counters *cnt, const int *forced_tok, int forced_count,
                                                int *acc_out, int *emit_out, int *nemit_out, int *nused_out) {
  const int len = st[b].len;
  if (len < 1) return;
  const int n = st[b].n;
  const int j = st[b].j_prev;
  if (j != len - 1 || len + n + 1 > cap) {  // no verify ran for this sequence
    if (acc_out) acc_out[b] = 0;
    if (nemit_out) nemit_out[b] = 0;
    if (nused_out) nused_out[b] = n;
    st[b].n_emit = 0;
    return;
  }
  int k = 0;
  if (forced_count > 0) {
    k = forced_count - 1;
  } else {
    while (k < n && draft[k] == target[k]) ++k;
  }
  for (int i = 0; i <= k; ++i) {
    int t;
    if (forced_count > 0) t = forced_tok[i];
    else t = i < k ? draft[i] : target[k];
    tok[(size_t)b * tok_stride + j + 1 + i] = t;
    if (emit_out) emit_out[b * (nmax + 1) + i] = t;
  }
  st[b].len = j + k + 2;
  st[b].k_acc = k;
  st[b].n_emit = k + 1;
  if (n == 0) st[b].stale = (j + 1 - st[b].dlen) > nmax + 1;  // the head falls behind while not drafting
  if (acc_out) acc_out[b] = k;
  if (nemit_out) nemit_out[b] = k + 1;
  if (nused_out) nused_out[b] = n;
  if (forced_count == 0) {
    atomicAdd(&cnt->n_target, 1ull);
    atomicAdd(&cnt->n_draft, (unsigned long long)n);
    atomicAdd(&cnt->n_waste, (unsigned long long)(n - k));
    atomicAdd(&cnt->n_tokens, (unsigned long long)(k + 1));
  }
}
__global__ void k_accept(SeqState *st, int *tok, int cap, const int *draft, const int *target, int nmax, int B,
                         Counters *cnt, int only_seq, const int *forced_tok, int forced_count, int *acc_out,
                         int *emit_out, int *nemit_out, int *nused_out) {
  const int b = threadIdx.x;
  if (b >= B) return;
  if (only_seq >= 0 && b != only_seq) return;
  accept_sequence(st, tok, cap, cap, draft + b * nmax, target + b * (nmax + 1), nmax, b, cnt, forced_tok, forced_count, acc_out, emit_out,
                  nemit_out, nused_out);
}

// Small state edits used by prefill and force_commit.
__global__ void k_copy_prompt(int *tok, int cap, int b, const int *prompt, int m) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x)
    tok[(size_t)b * cap + i] = prompt[i];
}
__global__ void k_finish_prefill(SeqState *st, int *tok, int cap, int b, int m, int chunk, const int *first_tok_slot,
                                 int *user_out) {
  if (threadIdx.x != 0) return;
  const int t = first_tok_slot[0];
  tok[(size_t)b * cap + m] = t;
  st[b].len = m + 1;
  st[b].dlen = m - 1;
  st[b].n = 0; st[b].k_acc = 0; st[b].j_prev = -1; st[b].n_emit = 0; st[b].stale = 0;
  st[b].chunk = chunk;
  if (user_out) *user_out = t;
}
__global__ void k_rewind(SeqState *st, int b, int count, const int *forced_tok, int *draft, int nmax,
                         Counters *cnt) {
  if (threadIdx.x != 0) return;
  const int j = st[b].j_prev;
  if (j < 0) return;
  atomicAdd(&cnt->n_tokens, (unsigned long long)(count - st[b].n_emit));  // wraps correctly for negatives
  st[b].len = j + 1;
  st[b].n = count - 1;
  for (int i = 0; i + 1 < count; ++i) draft[b * nmax + i] = forced_tok[i];
}
__global__ void k_copy_i32(int *dst, const int *src, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) dst[i] = src[i];
}
// Results of a step to the caller's arrays (those that are not null), all in one launch.
struct CopyMany {
  int *dst[4];
  const int *src[4];
  int n[4];
};
__global__ void k_copy_many(const CopyMany c) {
  const int j = blockIdx.x;
  if (c.dst[j])
    for (int i = threadIdx.x; i < c.n[j]; i += blockDim.x) c.dst[j][i] = c.src[j][i];
}
// Label pass (Section 3.3 / the draft-length oracle of Section 2.3): full-length drafts for every sequence ...
__global__ void k_set_n_full(SeqState *st, int B, int nmax, int cap) {
  const int b = threadIdx.x;
  if (b >= B) return;
  const int room = cap - st[b].len - 1;
  st[b].n = st[b].len < 2 ? 0 : max(0, min(nmax, room));
}
// ... and, after the verify pass, the length of the longest draft prefix the target confirms.  Nothing is committed.
__global__ void k_label(const SeqState *st, const int *draft, const int *target, int nmax, int B, int *k_out) {
  const int b = threadIdx.x;
  if (b >= B) return;
  const int n = st[b].n;
  int k = 0;
  while (k < n && draft[b * nmax + k] == target[b * (nmax + 1) + k]) ++k;
  k_out[b] = k;
}

// Label collection over start positions (Section 3.3): sequence `seq` is put into the state it had when token j was
// pending (len = j + 1; the draft head's rows of true features up to dlen), with a full-length draft ahead; every
// other sequence of the batch sits the pass out.
__global__ void k_label_begin(SeqState *st, int seq, int B, int len_j, int dlen_j, int nmax, int cap) {
  const int b = threadIdx.x;
  if (b >= B) return;
  if (b != seq) { st[b].n = 0; return; }
  st[b].len = len_j;
  st[b].dlen = dlen_j;
  st[b].j_prev = -1;
  st[b].n = max(0, min(nmax, cap - len_j - 1));
}
// Rows of one sequence that the passes of a start position write, kept aside (restore = 0) and put back (1): cache rows and
// features of positions t0 .. t0 + nt - 1 of the target, cache rows of positions d0 .. d0 + nd - 1 of the draft head.  Block
// (row, layer; layer L: the draft head); `rows` holds nt rows per layer, then the draft head's, a row its keys and its values.
struct LabelRows {
  int t0, nt, d0, nd, L, H, hd;
  const int *pages;                      // page table of the sequence
  __nv_bfloat16 *tk, *tv, *dk, *dv, *rows;
  float *feat, *feat_rows;               // features of position 0, kept features
};
__global__ void __launch_bounds__(128) k_label_rows(const LabelRows a, int restore) {
  const int r = blockIdx.x, layer = blockIdx.y, d = a.H * a.hd;
  const bool head = layer == a.L;
  if (r >= (head ? a.nd : a.nt)) return;
  const int pos = (head ? a.d0 : a.t0) + r, page = a.pages[pos / kPageSize], slot = pos % kPageSize;
  const size_t base = head ? (size_t)page * a.H : ((size_t)page * a.L + layer) * a.H;
  uint4 *kept = reinterpret_cast<uint4 *>(a.rows + ((size_t)layer * a.nt + r) * 2 * d);
  for (int i = threadIdx.x; i < d / 8; i += 128) {
    const int hh = 8 * i / a.hd;
    const size_t o = ((base + hh) * kPageSize + slot) * a.hd + (8 * i - hh * a.hd);
    uint4 *k = reinterpret_cast<uint4 *>((head ? a.dk : a.tk) + o), *v = reinterpret_cast<uint4 *>((head ? a.dv : a.tv) + o);
    if (restore) { *k = kept[i]; *v = kept[d / 8 + i]; }
    else { kept[i] = *k; kept[d / 8 + i] = *v; }
  }
  if (layer == 0) {
    float *f = a.feat + (size_t)pos * d, *g = a.feat_rows + (size_t)r * d;
    for (int i = threadIdx.x; i < d; i += 128) {
      if (restore) f[i] = g[i];
      else g[i] = f[i];
    }
  }
}

// Label collection, packed: up to kMaxBatch start positions of one sequence as sequences of their own, which share the
// sequence's cache pages up to the one their first own row falls into (page0); from there on their pages are ones that the
// sequence does not use yet, with the rows before start position j copied.  The sequence's state and rows stay as they are.
struct LabelPlan {
  int G, seq, chunk;
  int j[kMaxBatch], dlen[kMaxBatch], n[kMaxBatch];
  int page0[kMaxBatch], npriv[kMaxBatch], free0[kMaxBatch];   // first private page, how many, the first of them counted from the table's end
};
__global__ void k_label_setup(const LabelPlan pl, SeqState *st, int *table, const int *page_table, int pages_per_seq) {
  const int v = blockIdx.x;
  const int *src = page_table + (size_t)pl.seq * pages_per_seq;
  for (int i = threadIdx.x; i < pages_per_seq; i += blockDim.x) {
    const int k = i - pl.page0[v];
    table[v * pages_per_seq + i] = k >= 0 && k < pl.npriv[v] ? src[pages_per_seq - 1 - (pl.free0[v] + k)] : src[i];
  }
  if (threadIdx.x == 0) {
    SeqState s;
    s.len = pl.j[v] + 1; s.dlen = pl.dlen[v]; s.n = pl.n[v]; s.k_acc = 0; s.j_prev = -1; s.n_emit = 0; s.stale = 0; s.chunk = pl.chunk;
    st[v] = s;
  }
}
// Rows before j of the private pages (at most two): block (head of a layer, start position, page).
__global__ void k_label_pages(const LabelPlan pl, const int *table, const int *page_table, int pages_per_seq, int heads, int hd,
                              __nv_bfloat16 *kpool, __nv_bfloat16 *vpool) {
  const int v = blockIdx.y, p0 = pl.page0[v] + blockIdx.z, slots = min(kPageSize, pl.j[v] - p0 * kPageSize);
  if ((int)blockIdx.z >= pl.npriv[v] || slots <= 0) return;
  const size_t unit = (size_t)kPageSize * hd;
  const size_t src = ((size_t)page_table[(size_t)pl.seq * pages_per_seq + p0] * heads + blockIdx.x) * unit;
  const size_t dst = ((size_t)table[v * pages_per_seq + p0] * heads + blockIdx.x) * unit;
  for (int i = threadIdx.x; i < slots * hd / 8; i += blockDim.x) {
    reinterpret_cast<uint4 *>(kpool + dst)[i] = reinterpret_cast<const uint4 *>(kpool + src)[i];
    reinterpret_cast<uint4 *>(vpool + dst)[i] = reinterpret_cast<const uint4 *>(vpool + src)[i];
  }
}
// Labels of the packed start positions (and, optionally, the drafts and the target's choices they came from).
__global__ void k_label_many(const SeqState *st, const int *draft, const int *target, int nmax, int *k_out, int *draft_out,
                             int *target_out) {
  const int v = blockIdx.x, i = threadIdx.x, n = st[v].n;
  if (i == 0) {
    int k = 0;
    while (k < n && draft[v * nmax + k] == target[v * (nmax + 1) + k]) ++k;
    k_out[v] = k;
  }
  if (draft_out && i < nmax) draft_out[v * nmax + i] = i < n ? draft[v * nmax + i] : -1;
  if (target_out && i <= nmax) target_out[v * (nmax + 1) + i] = i <= n ? target[v * (nmax + 1) + i] : -1;
}

__global__ void k_gather_n(const SeqState *st, int *out, int B) {
  if (threadIdx.x < B) out[threadIdx.x] = st[threadIdx.x].n;
}

}  // namespace ada
