// Attention of a prompt pass (rows of one sequence at consecutive positions) on the 5th-generation tensor cores: two tiles
// of 128 query rows of one head per CTA over all keys up to their own, 64 keys (one cache page) at a time.
//
//   warps 0..3, 4..7  softmax of row tile 0 and 1, thread = query row (tensor-memory lane)
//   warp 8            producer: a page's keys and values by TMA, two stages
//   warp 9            one elected thread issues the products; owns the tensor memory (512 columns)
//
// Per page and row tile: scores S[128 x 64] = q_hi K^T + q_lo K^T (queries as fp16 hi and lo tiles in shared memory, keys
// K-major as they lie in the cache); the softmax warps read S, keep running maxima and sums, and write the weights back to
// tensor memory as fp16 hi and lo operands; O[128 x hd] = w_hi V + w_lo V (weights from tensor memory, values as the MN-major
// operand).  O of a page is added to fp32 sums in registers, rescaled whenever a maximum moved, so nothing is ever rescaled
// in tensor memory and the sums are rounded to nearest.  While one tile is in its softmax the products of the other run.
// Cache rows have their 16-byte chunks XORed with slot & 7: boxes of 64 rows x 128 bytes, copied verbatim, are the
// 128-byte-swizzle layout that the tensor core reads.
//
// No split of the keys and no merge: a prompt pass has rows enough.  The result is normalised and written as the planes of
// the O projection.  Row tiles with the most keys start first.  Every wait is bounded.
// 7B, layer of 1000 rows at positions 1000 .. 1999, before -> after: 245 us on mma.sync (tensor products at 200 TFLOP/s) -> 87 us.
// What bounds it now is a page's chain, 2.4 us for both tiles: 1.7 us of products (hi and lo parts; 64 keys are a narrow N for
// queries that are read from shared memory each time) with the softmax in turn.  Scores a page ahead and sums kept in
// tensor memory made 333 tokens of 16 layers of 2048 2.5 % faster, but hundreds of additions in one accumulator are less exact.
#pragma once
#include <type_traits>

#include "ada_gemm_pair.cuh"

namespace ada {

constexpr int kPaThreads = 12 * 32;               // (the last two warps only make up the warpgroup that hands registers over)
constexpr int kPaRows = 256;                      // query rows of a CTA: two tiles of 128
constexpr int kPaStages = 2;

template <int HD>
struct PaShape {
  static constexpr int kHalves = HD / 64;         // 64-channel boxes of a row
  static constexpr int kBox = 64 * 128;           // bytes of a box: 64 keys x 64 channels
  static constexpr int kQBox = 128 * 128;         // the same of a query tile: 128 rows
  static constexpr int kStage = 2 * kHalves * kBox;        // keys, then values
  static constexpr int kQTile = 2 * kHalves * kQBox;       // hi boxes, then lo boxes
  static constexpr int kSmemBytes = 1024 + 2 * kQTile + kPaStages * kStage + 256;
};
static_assert(PaShape<128>::kSmemBytes <= 227 * 1024, "shared memory budget");

struct AttnPromptArgs {
  const float *q;                          // [T][H * HD], scaled, rotated
  const TensorMap128 *kmap, *vmap;         // cache pools as rows of HD elements: box {64 channels, 64 rows}, no swizzle
  const int *pages;                        // page table of the sequence
  int L, layer, H, T, pos0;
  __nv_bfloat16 *xhi, *xlo; int ldx;
  Counters *cnt;
};

// K-major fp16 operands, M = 128, fp32 sums; bt: B is MN-major
__host__ __device__ constexpr uint32_t pa_idesc(uint32_t n, bool bt) {
  return (1u << 4) | (bt ? 1u << 16 : 0u) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}
// MN-major operand, 128-byte swizzle: 64-element groups `lbo` bytes apart, groups of 8 k-rows 1024 bytes apart
__device__ __forceinline__ uint64_t pa_desc_mn(uint32_t smem_addr, uint32_t lbo) {
  return (uint64_t)((smem_addr >> 4) & 0x3FFFu) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// D (+)= A B^T with A in tensor memory (row r in lane r, two k per column)
__device__ __forceinline__ void umma_f16_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(tmem_d),
      "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ float pa_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

template <int HD>
__global__ void __launch_bounds__(kPaThreads, 1) k_attn_prompt(const AttnPromptArgs a) {
  using Sh = PaShape<HD>;
  pdl_launch_dependents();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int hh = blockIdx.y, r0 = (gridDim.x - 1 - blockIdx.x) * kPaRows;   // longest first
  extern __shared__ __align__(128) unsigned char pa_smem[];
  unsigned char *const smem = pa_smem + ((1024u - (smem_u32(pa_smem) & 1023u)) & 1023u);
  unsigned char *const stages = smem + 2 * Sh::kQTile;
  uint64_t *const bars = reinterpret_cast<uint64_t *>(stages + kPaStages * Sh::kStage);
  uint64_t *const full = bars, *const empty = bars + 2, *const sfull = bars + 4, *const pready = bars + 6, *const ofull = bars + 8,
           *const qready = bars + 10;                                        // sfull .. qready: per row tile
  uint32_t *const tmem_slot = reinterpret_cast<uint32_t *>(bars + 12);
  volatile int *const abort_s = reinterpret_cast<int *>(tmem_slot + 1);
  // pages that a row tile sees (none if it has no rows)
  auto tiles_of = [&](int i) {
    const int first = r0 + 128 * i;
    return first < a.T ? (a.pos0 + min(a.T, first + 128) - 1) / kPageSize + 1 : 0;
  };
  const int n0 = tiles_of(0), n1 = tiles_of(1), nmax = max(n0, n1);
  if (tid == 0) {
    *abort_s = 0;
    for (int i = 0; i < 2; ++i) {
      mbar_init(&full[i], 1); mbar_init(&empty[i], 1); mbar_init(&sfull[i], 1); mbar_init(&ofull[i], 1);
      mbar_init(&pready[i], 4); mbar_init(&qready[i], 4);                    // four softmax warps each
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 9) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();                  // queries and the new cache rows come from the kernel before this one

  // a softmax thread holds its row's sums: 256 x 224 + 128 x 56 registers = the 384 x 168 of the launch
  if (warp >= 8) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
  if (warp == 8) {
    // ------------------------------------------------------------- producer
    if (lane == 0) {
#pragma unroll 1
      for (int t = 0; t < nmax; ++t) {
        const int s = t & 1;
        if (t >= 2) mbar_wait_inline(&empty[s], ((unsigned)(t >> 1) & 1u) ^ 1u, a.cnt, abort_s);
        if (*abort_s) break;
        const int row = ((a.pages[t] * a.L + a.layer) * a.H + hh) * kPageSize;
        unsigned char *st = stages + s * Sh::kStage;
        mbar_expect_tx(&full[s], (unsigned)Sh::kStage);
#pragma unroll
        for (int h = 0; h < Sh::kHalves; ++h) {
          tma_load_2d(st + h * Sh::kBox, a.kmap, h * 64, row, &full[s]);
          tma_load_2d(st + (Sh::kHalves + h) * Sh::kBox, a.vmap, h * 64, row, &full[s]);
        }
      }
    }
  } else if (warp == 9) {
    // ------------------------------------------------------------- tensor-core issuer
    const uint32_t id_s = pa_idesc(64, false), id_o = pa_idesc(HD, true);
    auto scores = [&](int i, int t) {    // S of row tile i against page t
      if (t == 0) mbar_wait_inline(&qready[i], 0u, a.cnt, abort_s);
      mbar_wait_inline(&full[t & 1], (unsigned)(t >> 1) & 1u, a.cnt, abort_s);
      tc_fence_after();
      if (elect_one()) {
        const uint32_t q = smem_u32(smem + i * Sh::kQTile), k = smem_u32(stages + (t & 1) * Sh::kStage), d = tmem_base + 256u * i;
        uint32_t acc = 0;
#pragma unroll
        for (int pl = 1; pl >= 0; --pl)    // lo first: an addition drops what lies below the accumulator's last bit
#pragma unroll
          for (int h = 0; h < Sh::kHalves; ++h) {
            const uint64_t ad = umma_desc(q + (uint32_t)((pl * Sh::kHalves + h) * Sh::kQBox)), bd = umma_desc(k + (uint32_t)(h * Sh::kBox));
#pragma unroll
            for (int k4 = 0; k4 < 4; ++k4) { umma_bf16(d, ad + 2 * k4, bd + 2 * k4, id_s, acc); acc = 1; }
          }
        umma_commit(&sfull[i]);
      }
      __syncwarp();
    };
    auto values = [&](int i, int t, bool last_use) {   // O of row tile i for page t
      mbar_wait_inline(&pready[i], (unsigned)t & 1u, a.cnt, abort_s);
      tc_fence_after();
      if (elect_one()) {
        const uint32_t v = smem_u32(stages + (t & 1) * Sh::kStage + Sh::kHalves * Sh::kBox), d = tmem_base + 256u * i + 128u;
        uint32_t acc = 0;
#pragma unroll
        for (int pl = 1; pl >= 0; --pl)
#pragma unroll
          for (int k4 = 0; k4 < 4; ++k4) {   // 16 keys
            umma_f16_ta(d, tmem_base + 256u * i + 64u + 32u * pl + 8u * k4, pa_desc_mn(v + (uint32_t)(k4 * 2048), Sh::kBox), id_o, acc);
            acc = 1;
          }
        umma_commit(&ofull[i]);
        if (last_use) umma_commit(&empty[t & 1]);
      }
      __syncwarp();
    };
#pragma unroll 1
    for (int t = -1; t < nmax; ++t)
#pragma unroll 1
      for (int i = 0; i < 2; ++i) {
        const int n = i ? n1 : n0;
        if (t >= n) continue;
        if (t >= 0) values(i, t, i == 1 || t >= n1);
        // (the softmax warps have read S of page t before they wrote its weights)
        if (t + 1 < n) scores(i, t + 1);
      }
  }
  } else {
    // ------------------------------------------------------------- softmax, thread = query row
    asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
    const int i = warp >> 2, w4 = warp & 3, n = i ? n1 : n0;
    if (n > 0) {
      constexpr float kLog2e = 1.4426950408889634f;
      const int first = r0 + 128 * i;
      {   // queries of the tile as fp16 hi and lo boxes, a row per warp and step
        unsigned char *q = smem + i * Sh::kQTile;
        constexpr int LPR = HD / 4;             // lanes per row
#pragma unroll 4
        for (int r = w4 * 32 + lane / LPR; r < w4 * 32 + 32; r += 32 / LPR) {
          const int c = (lane % LPR) * 4;
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (first + r < a.T) v = *reinterpret_cast<const float4 *>(a.q + (size_t)(first + r) * a.H * HD + hh * HD + c);
          v.x *= kLog2e; v.y *= kLog2e; v.z *= kLog2e; v.w *= kLog2e;   // scores in units of log 2
          const __half2 h0 = __floats2half2_rn(v.x, v.y), h1 = __floats2half2_rn(v.z, v.w);
          const float2 f0 = __half22float2(h0), f1 = __half22float2(h1);
          const __half2 l0 = __floats2half2_rn(v.x - f0.x, v.y - f0.y), l1 = __floats2half2_rn(v.z - f1.x, v.w - f1.y);
          unsigned char *p = q + (c >> 6) * Sh::kQBox + r * 128 + ((((c & 63) >> 3) ^ (r & 7)) << 4) + (c & 7) * 2;
          *reinterpret_cast<uint2 *>(p) = make_uint2(*reinterpret_cast<const uint32_t *>(&h0), *reinterpret_cast<const uint32_t *>(&h1));
          *reinterpret_cast<uint2 *>(p + Sh::kHalves * Sh::kQBox) =
              make_uint2(*reinterpret_cast<const uint32_t *>(&l0), *reinterpret_cast<const uint32_t *>(&l1));
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the tensor core reads them
        __syncwarp();
        if (lane == 0) mbar_arrive(&qready[i]);
      }
      const uint32_t tm = tmem_base + 256u * i + ((uint32_t)(w4 * 32) << 16);
      const int row = first + w4 * 32 + lane, pos = a.pos0 + row;
      float o[HD];
#pragma unroll
      for (int c = 0; c < HD; ++c) o[c] = 0.f;
      float m = -INFINITY, l = 0.f;
      auto add_o = [&](int t) {           // O of page t
        mbar_wait_inline(&ofull[i], (unsigned)t & 1u, a.cnt, abort_s);
        tc_fence_after();
#pragma unroll
        for (int c0 = 0; c0 < HD; c0 += 32) {
          uint32_t v[32];
          tmem_ld32_issue(tm + 128u + (uint32_t)c0, v);
          tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < 32; ++c) o[c0 + c] += __uint_as_float(v[c]);
        }
      };
      auto softmax_page = [&](auto masked, int key0) {   // S of a page -> weights
        constexpr bool kMasked = decltype(masked)::value;
        float mx = m;
#pragma unroll 1
        for (int hf = 0; hf < 2; ++hf) {
          uint32_t v[32];
          tmem_ld32_issue(tm + 32u * hf, v);
          tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < 32; ++c)
            mx = fmaxf(mx, kMasked && key0 + hf * 32 + c > pos ? -INFINITY : __uint_as_float(v[c]));
        }
        // (every row sees key 0, so its maximum is finite from the first page on)
        if (__any_sync(0xffffffffu, mx != m)) {
          const float k = pa_exp2(m - mx);
          l *= k;
#pragma unroll
          for (int c = 0; c < HD; ++c) o[c] *= k;
          m = mx;
        }
        // (rolled, as the loop above: a CTA sees few pages, and unrolled the loops were waits for instructions as much as work;
        // 333 rows, 16 layers of 2048: 2053 -> 2029 us a prompt)
#pragma unroll 1
        for (int q4 = 0; q4 < 4; ++q4) {   // 16 keys
          float v[16];
          uint32_t ph[8], pl[8];
          tmem_ld16(tm + 16u * q4, v);
#pragma unroll
          for (int c = 0; c < 16; c += 2) {
            float x = pa_exp2(v[c] - m), y = pa_exp2(v[c + 1] - m);
            if constexpr (kMasked) {
              if (key0 + q4 * 16 + c > pos) x = 0.f;
              if (key0 + q4 * 16 + c + 1 > pos) y = 0.f;
            }
            l += x + y;
            const __half2 h = __floats2half2_rn(x, y);
            const float2 f = __half22float2(h);
            const __half2 lo = __floats2half2_rn(x - f.x, y - f.y);
            ph[c >> 1] = *reinterpret_cast<const uint32_t *>(&h);
            pl[c >> 1] = *reinterpret_cast<const uint32_t *>(&lo);
          }
          tmem_st8(tm + 64u + 8u * q4, ph);
          tmem_st8(tm + 96u + 8u * q4, pl);
        }
      };
#pragma unroll 1
      for (int t = 0;; ++t) {
        if (t > 0) add_o(t - 1);
        if (t == n) break;
        mbar_wait_inline(&sfull[i], (unsigned)t & 1u, a.cnt, abort_s);
        tc_fence_after();
        const int key0 = t * kPageSize;
        const bool masked = key0 + kPageSize - 1 > a.pos0 + first + w4 * 32;   // (warp-uniform) some row does not see the whole page
        if (masked) softmax_page(std::true_type{}, key0);
        else softmax_page(std::false_type{}, key0);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&pready[i]);
      }
      if (row < a.T) {
        const float inv = 1.f / l;
        __nv_bfloat16 *ph = a.xhi + (size_t)row * a.ldx + hh * HD, *pl = a.xlo + (size_t)row * a.ldx + hh * HD;
#pragma unroll
        for (int c = 0; c < HD; c += 8) {
          uint32_t h[4], lo[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            __nv_bfloat162 x, y;
            split_bf16(o[c + 2 * e] * inv, x.x, y.x);
            split_bf16(o[c + 2 * e + 1] * inv, x.y, y.y);
            h[e] = *reinterpret_cast<const uint32_t *>(&x);
            lo[e] = *reinterpret_cast<const uint32_t *>(&y);
          }
          *reinterpret_cast<uint4 *>(ph + c) = make_uint4(h[0], h[1], h[2], h[3]);
          *reinterpret_cast<uint4 *>(pl + c) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
      }
    }
  }
  // every read of tensor memory is done: free it
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  await_copies(abort_s);
  if (warp == 9) tmem_dealloc(tmem_base, 512);
}

}  // namespace ada
