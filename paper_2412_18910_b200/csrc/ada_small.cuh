// Decode passes of small models: a thread-block cluster of 16 CTAs per sequence runs a verify pass, or all draft steps of an
// iteration, and its CTAs hand their results to each other's shared memory.
//
// Why: a layer of such a model is a megabyte or two, so its passes in k_pass are nothing but phase changes of 64 CTAs, 3.7 us each at
// d_model 256: stores and a fence into level 2 (0.5), a count and the last poll of it (0.45), the copy of the activations into
// shared memory (0.7), products through tensor memory, sums, stores.  Here a phase's results go straight from the shared memory of
// the CTA that made them into that of the CTAs that read them (one bulk copy per reader, counted on the reader's mbarrier: 0.42 us
// from every CTA to every other for 1 KB in all, 0.5 for 4 KB; 16-byte st.async stores 0.52 and 0.74, reads of the peers' memory
// after a cluster barrier 0.75 and 0.87), and the products are warp-level ones (mma.sync: no descriptors, no commits, no tensor memory
// on the way; 24 clocks one behind the other).  What is left is a chain of dependent instructions, some eight clocks each, so the
// kernel does as little as it can between an exchange and the next: one copy per reader (a warp's copies are issued lane by lane, 100
// clocks each), gains and rotary factors in shared memory beforehand, a body of its own for draft steps of one row.
// Draft of four + verify of five rows, 2 layers of 256, vocabulary 4096, context 100: k_pass 134 + 62 us, here 50 + 42 (55 + 46 with candidates
// merged by five exchanges of three words and a thread walking all of its partial sums of attention); seven sequences 188 + 117 -> 57 +
// 46; verify with 8 layers 173 -> 120.
//
// Weights depend on no phase.  A layer's lie in shared memory (bulk copies as they are in memory, 118 KB a CTA at these sizes; those of the
// next layer's phase follow when the phase's products are done), draft steps keep them; the first 4096 rows of the LM head, 128 KB
// a CTA, stay in the registers of 8 warps.  (Through the load/store path to registers before each phase they came at 21 bytes a clock
// and SM: 33 us a draft step.)
//
// A phase's output columns are dealt to the CTAs in tiles of 16 weight rows, a CTA's tiles to its warps, K split among the warps
// of a tile (fixed by the shape), their sums added through shared memory in warp order.  Rows of a tile are chosen so that what belongs
// together meets in one thread: gate and up of a column, the two halves of a rotary pair.
//
// Sequences do not meet at all: a batch is a grid of clusters, each with its own lengths (seven run at once, an eighth after them).
//
// Phases and exchanges of a layer (ns = 16 / heads CTAs share a head):
//   QKV       the CTAs of head hh make its q, k, v (rotated), send them to each other and store the cache rows
//   attention CTA s of a head takes the 8-key pieces p with p % ns = s, its warps those dealt in turn; partial sums of all
//             heads to everyone, who merge them into the input of O
//   O, down   residual columns (kept by their CTA for the whole pass), input of the next GEMM and its sums of squares to everyone
//   gate/up   silu(gate) * up to everyone
//   LM head   the CTAs' two largest logits to everyone (draft) or to the first CTA (verify)
// Every output element depends only on its own row and on the shape: results do not depend on the rows or sequences beside it.
// Every wait is bounded; a wait that gave up sets the status bit (which ends the other CTAs' waits) and the rest of the kernel runs without
// waiting.  What that CTA then reads may be anything, so it sends nothing more, arms no barrier again, whose phase may not be complete, takes
// no token past the vocabulary, and the state of the sequence stays as it was; nobody leaves before all copies have landed.
#pragma once
#include "ada_pass.cuh"
#include "ada_small_shape.h"

namespace ada {

__device__ __forceinline__ void mma_bf16_k16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16_k8(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(b0));
}
__device__ __forceinline__ uint32_t movmatrix(uint32_t x) {   // transposes an 8 x 8 matrix of 16-bit elements held by the warp
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(x));
  return r;
}
// copy out of this CTA's shared memory into a CTA's of the cluster, counted on that CTA's barrier (cluster addresses)
__device__ __forceinline__ void bulk_s2c(uint32_t dst, uint32_t src, unsigned bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "r"(src),
               "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, unsigned bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ uint32_t map_rank(uint32_t own, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(own), "r"(rank));
  return r;
}

// Shared memory by 32-bit addresses (through generic pointers an access costs two to three instructions more, and the kernel's
// code is what its phases wait for).
__device__ __forceinline__ uint4 lds4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t lds_u(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float4 lds_f4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float2 lds_f2(uint32_t a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float lds_f(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts4(uint32_t a, uint4 v) {
  asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void sts_f4(uint32_t a, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void sts_f2(uint32_t a, float x, float y) {
  asm volatile("st.shared.v2.f32 [%0], {%1,%2};" ::"r"(a), "f"(x), "f"(y) : "memory");
}
__device__ __forceinline__ void sts_f(uint32_t a, float x) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(x) : "memory"); }
__device__ __forceinline__ void sts_h(uint32_t a, unsigned short x) { asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"(x) : "memory"); }
// The best of 32 candidates and the largest value among the others, as top2_merge gives them: the largest value, of equal ones the one
// of the lowest index.  (Integers in the order of the values; three reductions of the warp instead of five exchanges of three words.)
__device__ __forceinline__ int small_key(float v) {
  const int k = __float_as_int(v + 0.f);   // (-0 counts as 0)
  return k ^ ((k >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float small_unkey(int k) { return __int_as_float(k ^ ((k >> 31) & 0x7fffffff)); }
__device__ __forceinline__ Top2 small_best(Top2 c) {
  const int k = small_key(c.v1), best = __reduce_max_sync(0xffffffffu, k);
  Top2 r;
  r.i1 = __reduce_min_sync(0xffffffffu, k == best ? c.i1 : 0x7fffffff);
  r.v1 = small_unkey(best);
  r.v2 = small_unkey(__reduce_max_sync(0xffffffffu, small_key(k == best && c.i1 == r.i1 ? c.v2 : c.v1)));
  return r;
}
// Accepting is rare and serial: out of line.
__device__ __noinline__ void small_accept(const PassParams &p, int b, const int *draft, const int *target) {
  accept_sequence(p.st, p.tok, p.cap, p.tok_stride, draft, target, p.nmax, b, p.cnt, nullptr, 0, p.acc_out, p.emit_out, p.nemit_out, nullptr);
}
// Eight values of a row as their chunk: k 0 .. 3 to o, k 4 .. 7 to o + plane.
__device__ __forceinline__ uint4 small_split4(float a, float b, float c, float d) {
  __nv_bfloat162 h0, l0, h1, l1;
  split_bf16(a, h0.x, l0.x); split_bf16(b, h0.y, l0.y); split_bf16(c, h1.x, l1.x); split_bf16(d, h1.y, l1.y);
  return make_uint4(*reinterpret_cast<uint32_t *>(&h0), *reinterpret_cast<uint32_t *>(&l0), *reinterpret_cast<uint32_t *>(&h1),
                    *reinterpret_cast<uint32_t *>(&l1));
}
// Byte of element c (of eight) of a row's pieces: its hi part; the lo part lies 4 bytes on.
__device__ __forceinline__ int small_elem(int c, int plane) { return (c & 4 ? plane : 0) + (c & 2) * 4 + (c & 1) * 2; }

// DRAFT: all draft steps of an iteration; else the verify pass (p: as k_pass takes it).  Two kernels, so that the second's prologue runs
// beside the first, on other SMs.
template <bool DRAFT>
__global__ void __launch_bounds__(kSmThreads, 1) k_small(const __grid_constant__ PassParams p, const __grid_constant__ SmallShape z) {
  pdl_launch_dependents();
  constexpr int HD = kSmHd, HU = HD / 32, HALF = HD / 2, NTI = HD / 16;   // units and rotary pairs of a head, tiles of one of its q, k, v
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int rank = (int)cluster_rank(), b = blockIdx.x / kSmCtas;
  const int d = p.d, nd = d >> 4, F = p.F;

  extern __shared__ __align__(128) unsigned char small_smem[];
  unsigned char *const sm = small_smem + ((128u - (smem_u32(small_smem) & 127u)) & 127u);
  uint64_t *bars = reinterpret_cast<uint64_t *>(sm);
  static_assert(kSmBars * 8 <= 112, "barriers");
  static_assert(sizeof(Top2) + 4 <= kSmCandBytes, "candidates");
  volatile int *abort_s = reinterpret_cast<int *>(sm + 112);
  int *tok_s = reinterpret_cast<int *>(sm + 128);                       // tokens of the first rows
  int *choice_s = tok_s + kSmRowsMax;                                   // verify: the greedy choices
  float *flog = reinterpret_cast<float *>(choice_s + kSmRowsMax);       // logit of a forced token in this CTA's vocabulary rows
  float *lp_s = flog + kSmRowsMax;                                      // log-probability of the newest token
  Top2 *topw = reinterpret_cast<Top2 *>(sm + 1024);                     // [warps][rows]
  float *sew = reinterpret_cast<float *>(topw + kSmWarps * kSmRowsMax); // [warps][rows]
  int *pages = reinterpret_cast<int *>(sm + z.pages);
  const uint32_t sm0 = smem_u32(sm), scratch = sm0 + z.scratch, hown = sm0 + z.hown, rms0 = smem_u32(lp_s + 4);

  const bool has_d = rank < nd;                                         // tiles of d columns: one, the CTA's number
  const int hh = rank / z.ns, split = rank - hh * z.ns;                 // head of this CTA and its share of it
  const bool has_head = hh < p.H;
  const int qtiles = has_head ? (3 * NTI - split + z.ns - 1) / z.ns : 0;
  const int gtile0 = rank * z.gt, gtiles = max(0, min(F / 8 - gtile0, z.gt));
  const int ltile0 = rank * z.lt, ltiles = max(0, min(p.V / 16 - ltile0, z.lt));
  auto tiles_of = [&](int kind) { return kind == SM_QKV ? qtiles : kind == SM_GU ? gtiles : (int)has_d; };
  // ---- weights of a layer's phases: as they lie in memory, tile by tile, into shared memory (one warp)
  auto fetch_weights = [&](int kind, const LayerPtrs *lw) {
    const int rows = tiles_of(kind), K = kind == SM_FC ? 2 * d : kind == SM_DOWN ? F : d, bytes = 16 * K;    // of eight weight rows
    const uint32_t dst = sm0 + z.w[kind], bar = sm0 + 8 * (SMX_W + kind);
    if (lane == 0 && rows > 0) mbar_expect_tx(bars + SMX_W + kind, (unsigned)(2 * rows * bytes));
    __syncwarp();
    if (kind == SM_QKV || kind == SM_GU) {
      if (lane < 2 * rows) {
        const int i = lane >> 1, hf = lane & 1, m = split + z.ns * i, type = m / NTI;
        const __nv_bfloat16 *W = kind == SM_GU ? (hf ? lw->wu : lw->wg) : type == 0 ? lw->wq : type == 1 ? lw->wk : lw->wv;
        const int row = kind == SM_GU ? 8 * (gtile0 + i) : hh * HD + 8 * (m & (NTI - 1)) + hf * HALF;
        bulk_g2s(dst + lane * bytes, W + (size_t)row * K, bytes, bar);
      }
    } else if (lane == 0 && rows > 0) {
      const __nv_bfloat16 *W = kind == SM_FC ? z.w_fc : kind == SM_O ? lw->wo : lw->wd;
      bulk_g2s(dst, W + (size_t)16 * rank * K, 2 * bytes, bar);
    }
  };
  // ---- the LM head: rows g and g + 8 of two tiles of a warp stay in its registers (for as long as there are no more)
  uint4 w[4 * kSmLmUnits];
  auto load_lm = [&](int tile0) {
    const __nv_bfloat16 *A = z.w_lm + (size_t)(16 * (ltile0 + tile0 + 2 * warp) + g) * d + 8 * t;
#pragma unroll
    for (int i = 0; i < kSmLmUnits; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        w[4 * i + j] = make_uint4(0u, 0u, 0u, 0u);
        if (32 * i < d && tile0 + 2 * warp + (j >> 1) < ltiles) w[4 * i + j] = ldlp_load(A + (size_t)j * 8 * d + 32 * i);
      }
  };

  // ================================================================ before the wait: what depends on no other kernel
  if (tid == 0) {
    *abort_s = 0;
    for (int i = 0; i < kSmBars; ++i) mbar_init(bars + i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // which phases' weights have been asked for and not awaited yet: all of the first layer's
  uint32_t wpend = DRAFT ? 0x1fu : 0x1eu;
  if (warp < SM_LM && (wpend >> warp & 1u)) fetch_weights(warp, p.layers);
  // gains of this CTA's columns: of each layer the norm of attention and of the MLP, then the final one
#pragma unroll 1
  for (int i = tid; i < (2 * p.n_layers + 1) * 16; i += kSmThreads) {
    const int n = i >> 4;
    const __nv_bfloat16 *gp = n == 2 * p.n_layers ? p.final_norm : n & 1 ? p.layers[n >> 1].nm : p.layers[n >> 1].na;
    if (has_d) sts_f(sm0 + z.gains + i * 4, __bfloat162float(gp[rank * 16 + (i & 15)]));
  }
  load_lm(0);
  bool lm_first = true;                              // the registers hold the LM head's first round
  cluster_sync_all();                                // the barriers of all CTAs are initialised
  pdl_wait();

  // ================================================================ what this sequence does
  const SeqState q = p.st[b];
  for (int i = tid; i < p.pages_per_seq; i += kSmThreads) pages[i] = p.page_table[b * p.pages_per_seq + i];
  int nstep = 0, pos = 0, rows = 0;                  // passes; first position and rows of the first one
  bool refused = false;
  if (DRAFT) {
    pos = draft_first(p, q);
    if (pos >= 0) { nstep = q.n; rows = q.len - 1 - pos; }
    else refused = q.n > 0 && q.len > 1;
  } else if ((p.only_seq < 0 || b == p.only_seq) && q.len >= 1 && q.len + q.n + 1 <= p.cap) {
    nstep = 1; pos = q.len - 1; rows = q.n + 1;
  }
  // (all CTAs of the cluster come to the same)
  const int fresh0 = pos, T0 = rows;                 // cache rows from here on are made by this launch, T0 of them in its first pass
  if (tid < rows)
    tok_s[tid] = DRAFT ? p.tok[(size_t)b * p.tok_stride + pos + tid + 1]
               : tid == 0 ? p.tok[(size_t)b * p.tok_stride + pos] : p.draft[b * p.nmax + tid - 1];
  if (rows > 0) {
#pragma unroll 3
    for (int i = tid; i < z.cap_slots * HALF; i += kSmThreads)   // rotary factors of its positions
      if (pos + i / HALF < p.cap) {
        const float2 cs = p.rope[(size_t)pos * HALF + i];
        sts_f2(sm0 + z.rope + i * 8, cs.x, cs.y);
      }
  }
  __syncthreads();

  // phase clock of a profiled verify pass (of the first sequence): [0] its start, then the end of each phase
  auto stamp = [&](int i) {
    if (!DRAFT && p.phase_ns && blockIdx.x == 0 && tid == 0 && i < 512) {
      unsigned long long t;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      p.phase_ns[i] = t;
    }
  };
  stamp(0);

  // ---- exchanges
  uint32_t phases = 0;                               // per barrier the parity of its next completion (weights' among them)
  int sbuf = 0;
  uint32_t send = sm0 + z.send[0];
  // A buffer is written again three exchanges later: by then all that was sent from it has arrived (see SMX_X).
  int off = 0;                                       // this CTA has given up (looked at behind a barrier of the threads that waited)
  auto next_send = [&] { sbuf = sbuf == 2 ? 0 : sbuf + 1; send = sm0 + z.send[sbuf]; off = *abort_s; };
  auto arm = [&](int kind, int bytes) { if (tid == 0 && !off) mbar_expect_tx(bars + kind, (unsigned)bytes); };
  auto wait = [&](int kind) {
#pragma unroll 1
    for (unsigned i = 0; !mbar_try_cluster(bars + kind, (phases >> kind) & 1u) && !*abort_s; ++i) {
      if (i > 64) __nanosleep(40);
      if ((i & 63) == 63 && (i >= kSpinLimit || (ld_acquire(reinterpret_cast<const unsigned *>(&p.cnt->status)) & kStatTimeout))) {
        *abort_s = 1;
        atomicOr(&p.cnt->status, kStatTimeout);
      }
    }
    phases ^= 1u << kind;
  };
  auto wait_weights = [&](int kind) {
    if (wpend >> kind & 1u) {
      if (tiles_of(kind) > 0) wait(SMX_W + kind);
      wpend &= ~(1u << kind);
    }
  };
  // what this thread has written or read in shared memory comes before the copies that follow the barrier
  auto before_send = [&] {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
  };
  // One copy a lane and exchange: to CTA warp + 8 lane, and in QKV tile `qtile` to CTA `qdst` of the head.  (A warp's copies are issued lane
  // by lane, some 100 clocks each.)
  const uint32_t peer = map_rank(sm0, (uint32_t)min(warp + kSmWarps * lane, kSmCtas - 1));
  const int qe = warp + kSmWarps * lane, qtile = qe / z.ns, qm = split + z.ns * qtile;
  const bool qsends = qe < qtiles * z.ns;
  const uint32_t qpeer = map_rank(sm0, (uint32_t)min(hh * z.ns + qe - qtile * z.ns, kSmCtas - 1));
  auto copy_to_all = [&](int to, int bytes, int kind) {
    if (lane < kSmCtas / kSmWarps && !off) bulk_s2c(peer + to, send, (unsigned)bytes, peer + 8 * kind);
  };

  // ---- the first rows' input (row r: token tok_s[r], position first + r).  Verify: embedding rows, as residual and as input.  Draft:
  // [embedding ; feature]; catch-up rows pair the target feature of a position with the token after it (a later step has one
  // row, whose feature is the LM head's input of the step before and whose embedding row was fetched with its token).
  int xs = 1;                                        // which of the two X buffers holds the newest input
  if (nstep > 0) {
    const int T = T0, TS = small_stride(T), XB = small_xblock(T);
#pragma unroll 1
    for (int e = tid; e < T * nd; e += kSmThreads) {
      const int r = e / nd, tile = e - r * nd;
      const uint4 *ep = reinterpret_cast<const uint4 *>(p.embed + (size_t)small_token(tok_s[r], p.V) * d + tile * 16);
      const uint4 *gp = reinterpret_cast<const uint4 *>(p.layers[0].na + tile * 16);
      const float4 *fp = reinterpret_cast<const float4 *>(p.feat + ((size_t)b * p.tok_stride + pos + r) * d + tile * 16);
      const uint32_t x = sm0 + z.x[xs] + tile * XB;
      float ss = 0.f;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const uint4 er = ep[c];
        float v[8];
        if constexpr (!DRAFT) {
          float gv[8];
          ldlp_widen(er, v);
          ldlp_widen(gp[c], gv);
          if (tile == rank) {
            sts_f4(hown + (r * 16 + c * 8) * 4, make_float4(v[0], v[1], v[2], v[3]));
            sts_f4(hown + (r * 16 + c * 8) * 4 + 16, make_float4(v[4], v[5], v[6], v[7]));
          }
#pragma unroll
          for (int k = 0; k < 8; ++k) { ss += v[k] * v[k]; v[k] *= gv[k]; }
        } else {
          const uint32_t o = sm0 + z.e + ((tile * 2 + c) * 2 * TS + r) * 16;
          sts4(o, make_uint4(er.x, 0u, er.y, 0u));
          sts4(o + 16 * TS, make_uint4(er.z, 0u, er.w, 0u));
          const float4 f0 = fp[2 * c], f1 = fp[2 * c + 1];
          v[0] = f0.x; v[1] = f0.y; v[2] = f0.z; v[3] = f0.w; v[4] = f1.x; v[5] = f1.y; v[6] = f1.z; v[7] = f1.w;
        }
        sts4(x + (c * 2 * TS + r) * 16, small_split4(v[0], v[1], v[2], v[3]));
        sts4(x + (c * 2 * TS + TS + r) * 16, small_split4(v[4], v[5], v[6], v[7]));
      }
      sts_f(x + 64 * TS + r * 4, ss);
    }
    __syncthreads();
    stamp(1);
  }

  const int d4 = d >> 2, dr4 = kSmThreads / d4, dc4 = kSmThreads - dr4 * d4, r4 = tid / d4, c4 = tid - r4 * d4;   // walk over rows of d / 4
  int step = 0, nlen = q.n;                          // draft step, the draft's length
  int fT = T0;                                       // draft: rows that the feature is stored with
  float cum = 0.f;
  uint4 kf[HU], vf[HU];                              // attention: this thread's pieces of a key and its value

  // ---- one pass: its rows from position pos on.  ONE: a draft step of one row.  Draft: true if another step follows.
  auto run_pass = [&](auto one_const) -> bool {
    constexpr bool ONE = decltype(one_const)::value;
    const int T = ONE ? 1 : T0, TS = ONE ? 1 : small_stride(T0), XB = ONE ? small_xblock(1) : small_xblock(T0);
    const int nkeys = pos + T;
    const int PS = HD + 4, part_o = T * HD * 4, part = small_part(T);   // floats of a row of a warp's partial sums; bytes of a CTA's
    int l = 0;
    int arrive = -1;                                 // exchange that brings the phase's input (< 0: here already)
    // sums over the warps of a tile, of pass row r and weight row c
    auto sum_up = [&](int tile, int sh, int r, int c) {
      uint32_t s = scratch + (((tile << sh) * T + r) * kSmRed + c) * 4;
      float y = 0.f;
#pragma unroll 2
      for (int i = 1 << sh; i > 0; --i, s += T * kSmRed * 4) y += lds_f(s);
      return y;
    };
    auto rms_rows = [&] {   // 1/rms of the rows from the tiles' partial sums of squares (at most 16): a row to a warp, the last warps first
#pragma unroll 1
      for (int r = kSmWarps - 1 - warp; r < T; r += kSmWarps) {
        const float v = warp_sum(lane < nd ? lds_f(sm0 + z.x[xs] + lane * XB + 64 * TS + r * 4) : 0.f);
        if (lane == 0) sts_f(rms0 + r * 4, rsqrtf(v / (float)d + p.eps));
      }
    };
    auto cache_row = [&](int ps) {
      return ((((size_t)pages[ps / kPageSize] * p.cache_layers + l) * p.H + hh) * kPageSize + ps % kPageSize) * HD;
    };
    // A product: eight weight rows times 32 k of up to two pass rows.  The thread's sixteen bytes of weight row g are the whole first operand:
    // its rows 0 .. 7 are the weight rows at k 0, 1, 4, 5 of each chunk, its rows 8 .. 15 the same weight rows at k 2, 3, 6, 7; and of
    // the second operand's columns 0 and 1 are a pass row's hi and lo parts at the former k, 2 and 3 at the latter, 4 .. 7 the next
    // pass row's.  So the sum is in elements 0 and 1 of lane t = 0 and 2 and 3 of lane t = 1 (next row: t = 2 and 3).
    const int brow = g >> 2, bword = (g & 3) * 4;
    auto fold = [&](const float (&c)[4]) {
      const float v = t & 1 ? c[2] + c[3] : c[0] + c[1];
      return v + __shfl_xor_sync(0xffffffffu, v, 1);
    };
    auto phase = [&](auto kind_const) {
      // ============================================================== a phase: its input, its products
      constexpr int kind = decltype(kind_const)::value;
      // address of this thread's chunk t of unit 0, bytes from unit to unit, from k 0 .. 3 of a chunk to k 4 .. 7
      uint32_t x = sm0 + z.x[xs] + (t >> 1) * XB + (t & 1) * 32 * TS;
      int xu = 2 * XB, xh = 16 * TS;
      if constexpr (kind == SM_O) {
        // ---- attention: scores of eight rows with eight keys at a time, softmax, weighted values.  A head's chunks are taken in the order
        // 0, hd / 16, 1, hd / 16 + 1, ...: as the tiles make them.
        const int npiece = (nkeys + 7) >> 3, mine = has_head ? max(0, (npiece - split + z.ns - 1) / z.ns) : 0;   // pieces of this CTA
        auto load_old = [&](int ps) {   // this thread's key: position ps, its chunks 4 u + t
          const size_t row = cache_row(ps);
#pragma unroll
          for (int u = 0; u < HU; ++u) {
            const int c = ((2 * u + (t >> 1) + (t & 1) * NTI) ^ (ps & 7)) << 3;
            kf[u] = __ldcg(reinterpret_cast<const uint4 *>(p.kpool + row + c));
            vf[u] = __ldcg(reinterpret_cast<const uint4 *>(p.vpool + row + c));
          }
        };
        if (has_head) {
          {
            const int ps = 8 * (split + z.ns * warp) + g;   // the warp's first piece of old keys and values
            if (ps < fresh0) load_old(ps);
          }
          wait(SMX_Q);
          if (warp < mine) {
#pragma unroll 1
            for (int r0 = 0; r0 < T; r0 += 8) {
              float m = -INFINITY, L = 0.f;
              float o[HD / 8][4];                    // [2], [3]: the lo parts of the weights
#pragma unroll
              for (int i = 0; i < HD / 8; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
              const uint32_t qa = sm0 + z.q + t * 32 * TS + min(r0 + g, T - 1) * 16;
#pragma unroll 1
              for (int i = warp; i < mine; i += kSmWarps) {
                const int key0 = 8 * (split + z.ns * i), ps = key0 + g, f = ps - fresh0;
                if (f >= 0) {                        // made by this launch, or past the last key
#pragma unroll
                  for (int u = 0; u < HU; ++u) {
                    const int at = f < T0 ? (4 * u + t) * 16 * T0 + f * 16 : (4 * u + t) * 16 + f * NTI * 32;
                    kf[u] = vf[u] = make_uint4(0u, 0u, 0u, 0u);
                    if (ps < nkeys) {
                      kf[u] = lds4(sm0 + z.fk + at);
                      vf[u] = lds4(sm0 + z.fv + at);
                    }
                  }
                } else if (i != warp || r0 > 0) {
                  load_old(ps);
                }
                float s0[4] = {0.f, 0.f, 0.f, 0.f}, s1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int u = 0; u < HU; ++u) {
                  const uint4 a0 = lds4(qa + u * 128 * TS), a1 = lds4(qa + u * 128 * TS + 16 * TS);
                  mma_f16_k16(s0, a0.x, a0.y, a0.z, a0.w, kf[u].x, kf[u].y);
                  mma_f16_k16(s1, a1.x, a1.y, a1.z, a1.w, kf[u].z, kf[u].w);
                }
                // this thread: keys key0 + 2 t, + 1 of row r0 + g
                const int k = key0 + 2 * t, seen = min(pos + r0 + g, nkeys - 1);
                const float e0 = k <= seen ? (s0[0] + s1[0]) + (s0[2] + s1[2]) : -INFINITY;
                const float e1 = k + 1 <= seen ? (s0[1] + s1[1]) + (s0[3] + s1[3]) : -INFINITY;
                float mx = fmaxf(e0, e1);
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                const float mn = fmaxf(m, mx), base = mn > -INFINITY ? mn : 0.f;   // (a row that sees no key yet: weights 0)
                const float f0 = __expf(m - base), w0 = __expf(e0 - base), w1 = __expf(e1 - base);
                m = mn;
                float s = w0 + w1;
                s += __shfl_xor_sync(0xffffffffu, s, 1);
                s += __shfl_xor_sync(0xffffffffu, s, 2);
                L = L * f0 + s;
                // weights as (hi, lo) halves: rows 0 .. 7 and 8 .. 15 of the product
                const __half2 wh = __floats2half2_rn(w0, w1);
                const float2 whf = __half22float2(wh);
                const __half2 wl = __floats2half2_rn(w0 - whf.x, w1 - whf.y);
                const uint32_t ah = *reinterpret_cast<const uint32_t *>(&wh), al = *reinterpret_cast<const uint32_t *>(&wl);
                if (i != warp) {
#pragma unroll
                  for (int n = 0; n < HD / 8; ++n) { o[n][0] *= f0; o[n][1] *= f0; o[n][2] *= f0; o[n][3] *= f0; }
                }
                // block n of unit u: elements 2 n, + 1 of the chunks 4 u + t, transposed so that a thread has two keys of a channel
#pragma unroll
                for (int u = 0; u < HU; ++u) {
                  mma_f16_k8(o[4 * u], ah, al, movmatrix(vf[u].x));
                  mma_f16_k8(o[4 * u + 1], ah, al, movmatrix(vf[u].y));
                  mma_f16_k8(o[4 * u + 2], ah, al, movmatrix(vf[u].z));
                  mma_f16_k8(o[4 * u + 3], ah, al, movmatrix(vf[u].w));
                }
              }
              // this warp's partial sums (the products' sums that lay there were read before the exchange)
              if (r0 + g < T) {
                const uint32_t pw = scratch + ((warp * T + r0 + g) * PS + 8 * ((t >> 1) + (t & 1) * NTI)) * 4;
#pragma unroll
                for (int n = 0; n < HD / 8; n += 2)
                  sts_f4(pw + (16 * (n >> 2) + 2 * (n & 3)) * 4, make_float4(o[n][0] + o[n][2], o[n][1] + o[n][3], o[n + 1][0] + o[n + 1][2], o[n + 1][1] + o[n + 1][3]));
                if (t == 0) sts_f2(scratch + ((warp * T + r0 + g) * PS + HD) * 4, m, L);
              }
            }
          }
        }
        __syncthreads();
        next_send();
        // Adds up to N partial sums, `step` bytes apart, to those so far, in order: (m, l) at ml, four channels at o.  (One a lane, merged by
        // exchanges, took three times as long for five rows.)
        auto merge = [&](auto slots, uint32_t ml, uint32_t o, int step, int n, float4 &y, float &M, float &L) {
          constexpr int N = decltype(slots)::value;
          float2 v[N];
          float4 ov[N];
#pragma unroll
          for (int k = 0; k < N; ++k) {
            v[k] = make_float2(-INFINITY, 0.f);
            ov[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (k < n) { v[k] = lds_f2(ml + k * step); ov[k] = lds_f4(o + k * step); }
          }
          const float M0 = M;
#pragma unroll
          for (int k = 0; k < N; ++k) M = fmaxf(M, v[k].x);
          const float base = M > -INFINITY ? M : 0.f, f0 = __expf(M0 - base);
          L *= f0;
          y.x *= f0; y.y *= f0; y.z *= f0; y.w *= f0;
#pragma unroll
          for (int k = 0; k < N; ++k) {
            const float f = __expf(v[k].x - base);
            L += v[k].y * f;
            y.x += ov[k].x * f; y.y += ov[k].y * f; y.z += ov[k].z * f; y.w += ov[k].w * f;
          }
        };
        if (has_head) {
          // over the warps, four channels of a row per thread
          const int nw = min(mine, kSmWarps);
#pragma unroll 1
          for (int e = tid; e < T * (HD / 4); e += kSmThreads) {
            const int r = e / (HD / 4), c = (e & (HD / 4 - 1)) * 4;
            const uint32_t pr = scratch + r * PS * 4;
            float M = -INFINITY, L = 0.f;
            float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
            for (int k = 0; k < nw; k += 4)
              merge(std::integral_constant<int, 4>{}, pr + k * T * PS * 4 + HD * 4, pr + k * T * PS * 4 + c * 4, T * PS * 4, nw - k, y, M, L);
            sts_f4(send + (r * HD + c) * 4, y);
            if (c == 0) sts_f2(send + part_o + r * 8, M, L);
          }
        }
        arm(SMX_A, small_expect(z.heads, part));
        before_send();
        copy_to_all(has_head ? z.ac + rank * part : kSmNone, has_head ? part : kSmNoneBytes, SMX_A);
        wait(SMX_A);
        // over the CTAs of each head, by every CTA for itself: O's input
        auto merge_head = [&](int r, int c) {
          const uint32_t src = sm0 + z.ac + 4 * c / HD * z.ns * part, ch = (r * HD + (4 * c & (HD - 1))) * 4;
          float M = -INFINITY, L = 0.f;
          float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
          for (int k = 0; k < z.ns; k += 4)
            merge(std::integral_constant<int, 4>{}, src + k * part + part_o + 8 * r, src + k * part + ch, part, z.ns - k, y, M, L);
          const float inv = 1.f / L;
          sts4(sm0 + z.e + ((c >> 1) * 2 * TS + (c & 1) * TS + r) * 16, small_split4(y.x * inv, y.y * inv, y.z * inv, y.w * inv));
        };
        if (ONE) {
          if (tid < d4) merge_head(0, tid);
        } else {
#pragma unroll 1
          for (int r = r4, c = c4; r < T;) {
            merge_head(r, c);
            r += dr4; c += dc4;
            if (c >= d4) { c -= d4; ++r; }
          }
        }
        __syncthreads();
        stamp(5 * l + 3);                            // attention
        x = sm0 + z.e + t * 32 * TS;
        xu = 128 * TS;
      } else {
        if (arrive >= 0) wait(arrive);
        if constexpr (kind == SM_DOWN) {
          x = sm0 + z.ac + t * 32 * TS;
          xu = 128 * TS;
        }
      }
      // Products with the 16 weight rows of a tile, sums into shared memory: [row][16 weight rows].  Activations lie in chunks of eight k,
      // of each 16 bytes a row for k 0 .. 3 and, behind them, for k 4 .. 7.
      if (!ONE) wait_weights(kind);
      const int sh = z.shift[kind];
      if ((warp >> sh) < tiles_of(kind)) {
        const int K = kind == SM_FC ? 2 * d : kind == SM_DOWN ? F : d, n = (K + 31) >> 5, u0 = warp & ((1 << sh) - 1);
        const uint32_t pw = sm0 + z.w[kind] + ((warp >> sh) * 16 + g) * 2 * K + t * 16;
        // fc: the first half of K are embeddings, the second the feature, stored with the rows of the step before
        const int eu = kind == SM_FC ? d >> 5 : 0;
        if constexpr (kind == SM_FC) {
          const int fS = small_stride(fT), FB = small_xblock(fT);
          x = sm0 + z.x[xs] + (t >> 1) * FB + (t & 1) * 32 * fS + (step == 0 ? 0 : fT - 1) * 16 - eu * 2 * FB;
          xu = 2 * FB; xh = 16 * fS;
        }
        constexpr int NP = ONE ? 1 : 2;              // pairs of rows at a time
#pragma unroll 1
        for (int r0 = 0; r0 < T; r0 += 2 * NP) {
          int r[NP];
#pragma unroll
          for (int i = 0; i < NP; ++i) r[i] = min(r0 + 2 * i + brow, T - 1) * 16 + bword;
          float s0[NP][4], s1[NP][4];
#pragma unroll
          for (int i = 0; i < NP; ++i) s0[i][0] = s0[i][1] = s0[i][2] = s0[i][3] = s1[i][0] = s1[i][1] = s1[i][2] = s1[i][3] = 0.f;
#pragma unroll 2
          for (int u = u0; u < n; u += 1 << sh) {
            uint4 w0 = make_uint4(0u, 0u, 0u, 0u), w1 = w0;
            uint32_t b0[NP], b1[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) b0[i] = b1[i] = 0u;
            if (kind != SM_DOWN || 32 * u + 8 * t < K) {   // (d is whole units)
              const bool emb = kind == SM_FC && u < eu;
              const uint32_t at = emb ? sm0 + z.e + t * 32 * TS + u * 128 * TS : x + u * xu;
              const int hf = emb ? 16 * TS : xh;
              w0 = lds4(pw + u * 64);
              w1 = lds4(pw + u * 64 + 16 * K);
#pragma unroll
              for (int i = 0; i < NP; ++i) { b0[i] = lds_u(at + r[i]); b1[i] = lds_u(at + r[i] + hf); }
            }
#pragma unroll
            for (int i = 0; i < NP; ++i) {
              mma_bf16_k16(s0[i], w0.x, w0.y, w0.z, w0.w, b0[i], b1[i]);
              mma_bf16_k16(s1[i], w1.x, w1.y, w1.z, w1.w, b0[i], b1[i]);
            }
          }
#pragma unroll
          for (int i = 0; i < NP; ++i) {
            const float y0 = fold(s0[i]), y1 = fold(s1[i]);
            const int rr = r0 + 2 * i + (t >> 1);    // lanes t = 0 and 2: weight row g, t = 1 and 3: weight row g + 8
            if (rr < T) sts_f(scratch + ((warp * T + rr) * kSmRed + g + 8 * (t & 1)) * 4, t & 1 ? y1 : y0);
          }
        }
      }
      if constexpr (kind == SM_QKV || kind == SM_GU) rms_rows();   // (the norm that the sums carry)
      __syncthreads();
      // ============================================================== what becomes of the sums
      next_send();
      if (!DRAFT && l + 1 < p.n_layers && !off) {    // the same phase's weights of the next layer
        wpend |= 1u << kind;
        if (warp == kSmWarps - 1) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          fetch_weights(kind, p.layers + l + 1);
        }
      }
      if constexpr (kind == SM_QKV) {
        const int n = qtiles * T;
#pragma unroll 1
        for (int tr = tid >> 3; tr < n; tr += kSmThreads / 8) {   // eight lanes: the columns of one (tile, row) and their partners
          int r = 0, tile = tr;
          if (!ONE) { tile = 0; r = tr; while (r >= T) { r -= T; ++tile; } }
          const int c = lane & 7, m = split + z.ns * tile, type = m / NTI, i = m & (NTI - 1), ps = pos + r;
          float2 cs = make_float2(1.f, 0.f);
          if (type < 2) cs = lds_f2(sm0 + z.rope + ((ps - fresh0) * HALF + 8 * i + c) * 8);
          const float inv = lds_f(rms0 + r * 4), v0 = sum_up(tile, sh, r, c) * inv, v1 = sum_up(tile, sh, r, c + 8) * inv;
          const float a0 = type < 2 ? v0 * cs.x - v1 * cs.y : v0, a1 = type < 2 ? v1 * cs.x + v0 * cs.y : v1;
          uint32_t o = send + tile * 64 * TS + r * 16;            // chunks 8 i .. and 8 i + hd / 2 ..
          if (type == 0) {
            const float qscale = rsqrtf((float)HD), q0 = a0 * qscale, q1 = a1 * qscale;
            const __half h0 = __float2half_rn(q0), h1 = __float2half_rn(q1);
            o += small_elem(c, 16 * TS);
            sts_h(o, __half_as_ushort(h0));
            sts_h(o + 4, __half_as_ushort(__float2half_rn(q0 - __half2float(h0))));
            sts_h(o + 32 * TS, __half_as_ushort(h1));
            sts_h(o + 32 * TS + 4, __half_as_ushort(__float2half_rn(q1 - __half2float(h1))));
          } else {
            const __nv_bfloat16 k0 = kv_store(a0), k1 = kv_store(a1);
            sts_h(o + c * 2, __bfloat16_as_ushort(k0));
            sts_h(o + 16 * T + c * 2, __bfloat16_as_ushort(k1));
            __nv_bfloat16 *row = (type == 1 ? p.kpool : p.vpool) + cache_row(ps) + c;
            row[(i ^ (ps & 7)) << 3] = k0;
            row[((i + NTI) ^ (ps & 7)) << 3] = k1;
          }
        }
        if (has_head) arm(SMX_Q, 4 * HD * (T + TS));
        before_send();
        // a tile to every CTA of the head: of q 32 TS bytes a chunk, of k and v 16 bytes a row and chunk, behind those of the steps before
        if (qsends && !off) {
          const int type = qm / NTI, i = qm & (NTI - 1), to = type == 0 ? z.q + i * 64 * TS : (type == 1 ? z.fk : z.fv) + (pos - fresh0) * NTI * 32 + i * 32 * T;
          bulk_s2c(qpeer + to, send + qtile * 64 * TS, type == 0 ? 64 * TS : 32 * T, qpeer + 8 * SMX_Q);
        }
      } else if constexpr (kind == SM_GU) {
        const int n = gtiles * T;
#pragma unroll 1
        for (int tr = tid >> 3; tr < n; tr += kSmThreads / 8) {
          int r = 0, tile = tr;
          if (!ONE) { tile = 0; r = tr; while (r >= T) { r -= T; ++tile; } }
          const int c = lane & 7;
          const float inv = lds_f(rms0 + r * 4), y = sum_up(tile, sh, r, c) * inv, u = sum_up(tile, sh, r, c + 8) * inv;
          __nv_bfloat16 hi, lo;
          split_bf16((y / (1.f + __expf(-y))) * u, hi, lo);
          const uint32_t o = send + (tile * 2 * TS + r) * 16 + small_elem(c, 16 * TS);
          sts_h(o, __bfloat16_as_ushort(hi));
          sts_h(o + 4, __bfloat16_as_ushort(lo));
        }
        arrive = SMX_AC;
        arm(SMX_AC, F * 4 * TS);
        before_send();
        if (gtiles > 0) copy_to_all(z.ac + gtile0 * 32 * TS, gtiles * 32 * TS, SMX_AC);
      } else {
        // fc, O, down: this CTA's columns of the residual rows; the next input and its sums of squares to everyone
        const int norm = kind == SM_FC ? 0 : kind == SM_O ? 2 * l + 1 : 2 * l + 2;   // that follows (the draft head has none after its layer)
        constexpr bool gain = kind != SM_DOWN || !DRAFT;
#pragma unroll 1
        for (int r = warp; r < T; r += kSmWarps) {   // a row to a warp, its halves each every other partial sum
          const int c = lane & 15;
          const uint32_t h = hown + (r * 16 + c) * 4;
          const float gv = gain ? lds_f(sm0 + z.gains + (norm * 16 + c) * 4) : 1.f, old = kind != SM_FC ? lds_f(h) : 0.f;
          uint32_t s = scratch + (((lane >> 4) * T + r) * kSmRed + c) * 4;
          float y = 0.f;
#pragma unroll 4
          for (int i = lane >> 4; i < 1 << sh; i += 2, s += 2 * T * kSmRed * 4) y += lds_f(s);
          y += __shfl_xor_sync(0xffffffffu, y, 16);
          if (!has_d) y = 0.f;
          if (kind != SM_FC) y = old + y;
          if (lane < 16) {
            sts_f(h, y);
            __nv_bfloat16 hi, lo;
            split_bf16(y * gv, hi, lo);
            const uint32_t o = send + ((c >> 3) * 2 * TS + r) * 16 + small_elem(c & 7, 16 * TS);
            sts_h(o, __bfloat16_as_ushort(hi));
            sts_h(o + 4, __bfloat16_as_ushort(lo));
          }
          if (gain) {
            float ss = y * y;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
            if (lane == 0) sts_f(send + 64 * TS + r * 4, ss);
          }
        }
        xs ^= 1;
        arrive = kind == SM_FC ? SMX_X : kind == SM_O ? SMX_O : SMX_D;
        arm(arrive, small_expect(nd, XB));
        before_send();
        copy_to_all(has_d ? z.x[xs] + rank * XB : kSmNone, has_d ? XB : kSmNoneBytes, arrive);
      }
      stamp(5 * l + (kind == SM_QKV ? 2 : kind + 2));
    };
    if constexpr (DRAFT) phase(std::integral_constant<int, SM_FC>{});
#pragma unroll 1
    for (; l < (DRAFT ? 1 : p.n_layers); ++l) {
      phase(std::integral_constant<int, SM_QKV>{});
      phase(std::integral_constant<int, SM_O>{});
      phase(std::integral_constant<int, SM_GU>{});
      phase(std::integral_constant<int, SM_DOWN>{});
    }
    wait(SMX_D);

    // ================================================================ LM head and greedy choice
    const int row0 = DRAFT ? T - 1 : 0, Tg = DRAFT ? 1 : T;                // rows (draft: the last one)
    const int out0 = DRAFT ? b * p.nmax + step : b * (p.nmax + 1);         // output slot of the first row
    const bool lps = DRAFT && p.lp_out;
    if (!DRAFT) rms_rows();
    if (lps && tid == 0) *flog = -INFINITY;
    if (!DRAFT || lps) __syncthreads();
    {
      const uint32_t x = sm0 + z.x[xs] + (t >> 1) * XB + (t & 1) * 32 * TS + row0 * 16;
      const uint32_t red = scratch + warp * Tg * 2 * kSmRed * 4;   // this warp's sums: [row][2 tiles of 16 weight rows]
      Top2 *const tw = topw + warp * kSmRowsMax;
      float *const sw = sew + warp * kSmRowsMax;
#pragma unroll 1
      for (int round = 0; round < ltiles; round += kSmLmRound) {
        if (ltiles > kSmLmRound && (round > 0 || !lm_first)) load_lm(round);
        lm_first = false;                            // (with more rounds than one the registers hold another by the next pass)
#pragma unroll 1
        for (int r0 = 0; r0 < Tg; r0 += 2) {
          const uint32_t px = x + min(r0 + brow, Tg - 1) * 16 + bword;
          float s[4][4];
#pragma unroll
          for (int n = 0; n < 4; ++n) s[n][0] = s[n][1] = s[n][2] = s[n][3] = 0.f;
#pragma unroll
          for (int i = 0; i < kSmLmUnits; ++i)
            if (32 * i < d) {
              const uint32_t b0 = lds_u(px + i * 2 * XB), b1 = lds_u(px + i * 2 * XB + 16 * TS);
#pragma unroll
              for (int n = 0; n < 4; ++n) mma_bf16_k16(s[n], w[4 * i + n].x, w[4 * i + n].y, w[4 * i + n].z, w[4 * i + n].w, b0, b1);
            }
          float y[4];
#pragma unroll
          for (int n = 0; n < 4; ++n) y[n] = fold(s[n]);
          if (r0 + (t >> 1) < Tg) {                  // lanes t = 0 and 2 store weight rows g and 16 + g, t = 1 and 3 the others
            const uint32_t o = red + ((r0 + (t >> 1)) * 2 * kSmRed + g + 8 * (t & 1)) * 4;
            sts_f(o, t & 1 ? y[1] : y[0]);
            sts_f(o + 64, t & 1 ? y[3] : y[2]);
          }
        }
        __syncwarp();
        const bool own = round + 2 * warp + (lane >> 4) < ltiles;
        const int v0 = 16 * (ltile0 + round + 2 * warp) + lane;
#pragma unroll 1
        for (int r = 0; r < Tg; ++r) {               // a lane: one vocabulary row of the warp's two tiles
          Top2 c;
          c.v1 = c.v2 = -INFINITY; c.i1 = 0x7fffffff;
          if (own) {
            float y = lds_f(red + (r * 2 * kSmRed + lane) * 4);
            if (!DRAFT) y *= lds_f(rms0 + r * 4);
            if (!DRAFT && p.logits) p.logits[(size_t)(out0 + r) * p.V + v0] = y;
            if (lps && p.forced && p.forced[out0 + r] == v0) flog[r] = y;
            c.v1 = y; c.i1 = v0;
          }
          const float y = c.v1;
          c = small_best(c);
          float s = 0.f;
          if (lps) s = warp_sum(own ? __expf(y - c.v1) : 0.f);   // sum of exp(logit - maximum)
          if (lane == 0) {
            if (round == 0) {
              tw[r] = c;
              sw[r] = s;
            } else {
              const Top2 before = tw[r];
              tw[r] = top2_merge(before, c);
              const float mx = tw[r].v1;
              if (lps) sw[r] = (before.v1 > -INFINITY ? sw[r] * __expf(before.v1 - mx) : 0.f) + (c.v1 > -INFINITY ? s * __expf(c.v1 - mx) : 0.f);
            }
          }
        }
        __syncwarp();
      }
      if (ltiles <= 0 && lane < Tg) {
        tw[lane].v1 = tw[lane].v2 = -INFINITY; tw[lane].i1 = 0x7fffffff;
        sw[lane] = 0.f;
      }
    }
    __syncthreads();
    next_send();
    // candidates of the warps, then of the CTAs: a row to a warp, a candidate to a lane
    const bool takes = DRAFT || rank == 0;
#pragma unroll 1
    for (int stage = 0; stage < (takes ? 2 : 1); ++stage) {
      if (stage == 1) wait(SMX_C);
#pragma unroll 1
      for (int r = warp; r < Tg; r += kSmWarps) {
        Top2 c;
        c.v1 = c.v2 = -INFINITY; c.i1 = 0x7fffffff;
        float cs = 0.f, fl = -INFINITY;
        if (lane < (stage == 0 ? kSmWarps : kSmCtas)) {
          if (stage == 0) {
            c = topw[lane * kSmRowsMax + r];
            if (lps) { cs = sew[lane * kSmRowsMax + r]; fl = flog[r]; }
          } else {
            const uint32_t cp = sm0 + z.cand + lane * 32 * Tg + r * 32;
            const float4 v = lds_f4(cp);
            c.v1 = v.x; c.i1 = __float_as_int(v.y); c.v2 = v.z; cs = v.w;
            if (lps) fl = lds_f(cp + 16);
          }
        }
        const float own = c.v1;
        c = small_best(c);
        if (lps) {
          cs = warp_sum(own > -INFINITY ? cs * __expf(own - c.v1) : 0.f);
          fl = warp_max(fl);
        }
        if (stage == 0) {
          if (lane == 0) {
            sts_f4(send + r * 32, make_float4(c.v1, __int_as_float(c.i1), c.v2, cs));
            sts_f4(send + r * 32 + 16, make_float4(fl, 0.f, 0.f, 0.f));
          }
          continue;
        }
        const int token = DRAFT && p.forced ? p.forced[out0 + r] : small_token(c.i1, p.V);
        if constexpr (DRAFT) {               // the embedding row of the next step
#pragma unroll 1
          for (int c8 = lane; c8 < d / 8; c8 += 32) {
            const uint4 er = *reinterpret_cast<const uint4 *>(p.embed + (size_t)small_token(token, p.V) * d + c8 * 8);
            sts4(sm0 + z.e + c8 * 32, make_uint4(er.x, 0u, er.y, 0u));
            sts4(sm0 + z.e + c8 * 32 + 16, make_uint4(er.z, 0u, er.w, 0u));
          }
        }
        if (lane == 0) {
          const float lp = lps ? (p.forced ? fl - c.v1 : 0.f) - __logf(cs) : 0.f;
          choice_s[r] = token;
          if (lps) *lp_s = lp;
          if (rank == 0) {
            p.tok_out[out0 + r] = token;
            if (p.top_out) p.top_out[out0 + r] = make_float2(c.v1, c.v2);
            if (lps) p.lp_out[out0 + r] = lp;
          }
        }
      }
      if (stage == 1) break;
      if (takes) arm(SMX_C, kSmCtas * 32 * Tg);
      before_send();
      if (DRAFT) copy_to_all(z.cand + rank * 32 * Tg, 32 * Tg, SMX_C);
      else if (tid == 0 && !off) bulk_s2c(peer + z.cand + rank * 32 * Tg, send, 32 * Tg, peer + 8 * SMX_C);   // (to CTA 0)
      // this CTA's columns of the feature rows: the target's, by position, or the head's own output
      if (has_d && (DRAFT || p.feat))        // (packed start positions keep no features)
#pragma unroll 1
        for (int e = tid; e < Tg * 16; e += kSmThreads) {
          const int r = e >> 4, col = e & 15;
          const float h = lds_f(hown + ((row0 + r) * 16 + col) * 4);
          if (DRAFT) p.dfeat[((size_t)b * p.nmax + step) * d + rank * 16 + col] = h;
          else p.feat[((size_t)b * p.cap + pos + r) * d + rank * 16 + col] = (h * lds_f(rms0 + r * 4)) * lds_f(sm0 + z.gains + (2 * p.n_layers * 16 + col) * 4);
        }
    }
    if (!takes) return false;                // (verify: only the first CTA goes on)
    __syncthreads();
    bool another = false;
    if (DRAFT) {
      // ---- the next draft step; with the stopping rule, whether there is one (every CTA comes to the same decision)
      if (p.ddd_thr < 0.f) {
        cum = (step == 0 ? 0.f : cum) + *lp_s;
        const int made = step + 1, room = p.cap - q.len - 1;
        if (made >= nlen && made < p.nmax && made < room && !(cum < p.ddd_thr)) nlen = made + 1;
        nstep = nlen;
      }
      ++step;
      fT = T;
      pos += T;
      another = step < nstep;
    }
    return another;
  };

  bool more = nstep > 0;
  if (more && DRAFT && T0 == 1) {
    for (int k = 0; k < SM_LM; ++k) wait_weights(k);
  } else if (more) {
    more = run_pass(std::false_type{});
  }
  if constexpr (DRAFT) {
#pragma unroll 1
    while (more) more = run_pass(std::true_type{});
  }
  // ================================================================ the sequence's state
  // (a pass has exchanged results with every CTA of the cluster, so all of them have read the state; without one they meet first)
  if (nstep == 0) {
    for (int k = 0; k < SM_LM; ++k) wait_weights(k);   // no copy may outlive the CTA
    cluster_sync_all();
  }
  if (rank == 0 && tid == 0) {
    if (nstep > 0) stamp(5 * p.n_layers + 2);        // LM head and choice
    SeqState *const st = p.st + b;
    const bool lost = *abort_s != 0;                 // (the choices may be anything: as if no pass had run)
    if (DRAFT) {
      if (refused) { st->n = 0; atomicOr(&p.cnt->status, kStatStale); }
      if (nstep > 0 && !lost) {
        st->dlen = q.len - 1;
        if (p.ddd_thr < 0.f) st->n = nlen;
      }
      if (p.steps_out) atomicMax(p.steps_out, nstep);
    } else {
      if (nstep > 0) st->j_prev = lost ? -1 : fresh0;
      if (p.accept) small_accept(p, b, nstep > 0 ? tok_s + 1 : nullptr, nstep > 0 ? choice_s : nullptr);
    }
  }
  // No CTA leaves while copies into its memory, or out of it, are under way: all that were sent have been awaited by their readers.  Where one
  // gave up it tells the others, and all of them stay, when the last has stopped sending, until what was sent has landed.
  __syncthreads();
  if (*abort_s) {
    if (tid < kSmCtas) asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], 1;" ::"r"(map_rank(sm0 + 112, (uint32_t)tid)) : "memory");
    asm volatile("fence.acq_rel.cluster;" ::: "memory");
    __syncwarp();
  }
  asm volatile("barrier.cluster.arrive.relaxed.aligned;\n barrier.cluster.wait.aligned;" ::: "memory");   // (nothing else is published here)
  await_copies(abort_s);
}

}  // namespace ada
