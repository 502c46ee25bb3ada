// GEMM of the prompt passes on pairs of CTAs (tcgen05, cta_group::2):
//   Y[t][n] = sum_k X[t][k] * W[n][k],  X as bf16 hi and lo planes, W bf16 [N][K],  up to kPromptRows rows t.
//
// A prompt pass has hundreds of rows, so it is bound by the tensor cores (two products per weight and row: hi and lo)
// and, on the way there, by what level 2 can hand to shared memory.  Two CTAs of a cluster therefore work on one tile of
// 256 weight rows x 2 nb prompt rows: each holds 128 of the weight rows and nb of the prompt rows (both planes), and the
// products read both CTAs' shared memory.  Per 64 k a CTA loads 16 KB of weights and 256 nb bytes of planes for
// 4 x 2 products of 256 x 2 nb x 16: 47 bytes per clock at nb = 128, where the tile of one CTA with 128 rows of either
// operand (k_gemm_tc<88> for the few rows of a decode pass) would need twice that.  hi and lo products add into the same
// accumulator, whose 2 nb columns leave room in tensor memory for a second one: the epilogue of a tile runs under the
// products of the next (persistent grid, one pair per two SMs, tiles dealt in a fixed order with the token tiles of a
// weight tile side by side so that its weights cross HBM once).
//
// Where the last tiles would leave most pairs idle (86 gate/up tiles of 256 rows on 74 pairs take the time of 148), the tiles
// from `whole` on are cut: every pair gets a run of as many accumulators, which may begin and end inside a tile.  A tile's first boxes
// are the end of a pair's run, its last ones the beginning of another's (or whole runs between): those leave their fp32 sums in memory,
// and the pair that has the first boxes adds them up in order and finishes the tile.  By then they have long been there: all runs begin
// together.  7B, level 2 cold: gate/up of 205 rows 106 -> 81 us, of 512 159 -> 146, QKV of 205 63 -> 58; 13B QKV of 1024 258 -> 239, down 255
// -> 206.  With token tiles side by side no longer, weights cross HBM more than once (13B QKV of 512 168 -> 323 MB; kept in level 2
// instead of passing through it they were slower, 129 -> 134 us).
//
//   warp 0      producer, one thread per CTA: weight box and plane boxes of its half of the tile into a ring of stages;
//               the bytes of both CTAs are counted on the leader's (even CTA's) barrier
//   warp 1      leader only: one elected thread issues the products and commits to both CTAs' barriers
//   warp 2      owns the tensor memory (512 columns in each CTA)
//   warps 4..11 epilogue: thread = one weight row (tensor-memory lane) x nb of the tile's prompt rows
//
// The accumulator of the tensor cores drops what lies below its last bit at every addition: over K = 4096, hi and lo in
// one accumulator, sums came out 8e-6 short (measured; 2.5e-5 over K = 11008).  So an accumulator takes a few boxes of 64 k
// only (GemmPairArgs::chunk, see pair_chunk), in each the lo products before the hi ones; the epilogue warps add it to fp32
// sums in their registers (round to nearest) while the products go on in the other accumulator.
//
// Epilogues (template parameter): PART leaves fp32 sums of a K split for k_reduce_h (O, down, the draft head's fc: their
// consumer needs the sums of squares of whole rows); QKV applies 1/rms, rotary embedding and writes q and the cache rows;
// SWIGLU applies 1/rms and silu(gate) * up and writes the planes of the next GEMM.  The two values a thread needs there
// (rows i and i + hd/2 of a head; gate and up of a column) sit in two lanes of the same CTA and are exchanged through
// shared memory.  Every wait is bounded.
//
// A launch of a short prompt runs each part of this code once or twice, so its size is time: loops that are not worked through many
// times a tile (waits, the producer's and the issuer's, the stores) are kept rolled.  70..78 KB -> 30..45 KB: four layers of 2048 and 333
// rows 686 -> 677 us, 7B 205 rows 1183 -> 1168 (with k_attn_prompt 84 -> 42 KB).
#pragma once
#include "ada_gemm_tc.cuh"

namespace ada {

constexpr int kPairThreads = 12 * 32;
constexpr int kPairStageMax = kTcABytes + 2 * 128 * 128;      // weight box + hi and lo boxes of 128 prompt rows
constexpr int kPairRing = 4 * kPairStageMax;                  // 192 KB
constexpr int kPairSlots = 8;                                 // barrier pairs (stages in flight at most)
constexpr int kPairXchBytes = 8 * 16 * 32 * 4;                // exchange of values between epilogue warps
constexpr int kPairInfoBytes = 256 * 16;                      // per prompt row of the tile: 1/rms, position, cache offset
constexpr int kPairSmemBytes = 1024 + kPairRing + kPairXchBytes + kPairInfoBytes + 256;
static_assert(kPairSmemBytes <= 227 * 1024, "shared memory budget");

enum { PAIR_PART = 0, PAIR_QKV = 1, PAIR_SWIGLU = 2 };

struct GemmPairArgs {
  const TensorMap128 *wmap[3];             // PART, QKV: box {64 k, 128 rows}; SWIGLU (gate, up): box {64 k, 64 rows}
  const TensorMap128 *xhi_map, *xlo_map;   // planes, box {64 k, nb rows}
  int nseg, Nseg, K;
  int T;                                   // rows of the pass (known on the host)
  int nb;                                  // prompt rows per CTA and tile: 32, 40, .. 128
  int token_tiles, weight_tiles, S;        // S: K splits (PART only)
  int chunk;                               // 64-k boxes per accumulator
  int whole;                               // tiles (and splits) dealt whole; the rest (S = 1) in equal runs to all pairs
  float *cut; int *cut_flags;              // ... sums of a tile's cut-off parts [CTA][prompt row][128 weight rows]; per CTA and epilogue warp
                                           // 1 when they are there (zero between launches)
  float *part; int part_rows;              // PART: [S][part_rows][Nseg]
  // QKV and SWIGLU
  const float *ss_part; float eps; int d;
  __nv_bfloat16 *ohi, *olo; int ldo;       // SWIGLU: planes of the next GEMM's input
  const float2 *rope; float *qout;         // QKV
  __nv_bfloat16 *kpool, *vpool;
  const int *page_table; int pages_per_seq, L, layer, H, hd;
  float qscale;
  const Pass *pass;
  Counters *cnts;
};

__device__ __forceinline__ void tmem_alloc_pair(uint32_t *smem_slot, uint32_t ncols) {   // one warp of each CTA of the pair
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_slot)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// D (+)= A B^T over both CTAs' shared memory: M = 256 (128 rows in each), N as in idesc (half of the rows of B in each)
__device__ __forceinline__ void umma_bf16_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// arrive on the barrier at this offset in both CTAs once the products issued so far have completed
__device__ __forceinline__ void umma_commit_pair(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
                   smem_u32(bar)),
               "h"((unsigned short)3)
               : "memory");
}
// 16 consecutive accumulator columns of this thread's tensor-memory lane
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
// load into this CTA's shared memory whose bytes are counted on a barrier of either CTA of the pair (cluster address)
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const TensorMap128 *map, int x, int y, uint32_t bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3}], "
      "[%4], %5;" ::"r"(dst),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(bar), "l"(pol)
      : "memory");
}

// mbar_wait with the spin inlined: a call could not be made from the epilogue warps, whose registers are all in use
__device__ __forceinline__ void mbar_wait_inline(uint64_t *bar, unsigned parity, Counters *cnt, volatile int *abort_flag) {
#pragma unroll 1
  for (unsigned i = 0; i < kSpinLimit; ++i) {
    if (mbar_try(bar, parity) || *abort_flag) return;
    if (i > 64) __nanosleep(40);
  }
  *abort_flag = 1;
  atomicOr(&cnt->status, kStatTimeout);
}

// x / (1 + e^-x) without a branch, so that a thread's quotients overlap (with the rounded division, which branches for its
// special cases, they took half of a SwiGLU tile's epilogue).  The approximate quotient is off by a few units in the last
// place; its remainder is exact in one fused operation, and adding remainder / divisor leaves it within 0.51 units of the
// quotient, as the rounded division does within 0.5.  Below -80, where the divisor would outgrow the reciprocal and the result
// lies between -1.5e-33 and 0, it is 0; above 88 the divisor is 1 and the result x.  Infinities and not-a-number give what the
// division gives (+inf, NaN, NaN).  Epilogue of a 7B tile of 256 rows: 17.0 -> 13.6 thousand clocks.
__device__ __forceinline__ float silu(float x) {
  const float d = 1.f + __expf(-x), r = __fdividef(1.f, d), q = x * r, z = fmaf(fmaf(-q, d, x), r, q);
  return x > 88.f ? x : x < -80.f ? x * 0.f : z;
}

__device__ __forceinline__ uint4 pack8(const __nv_bfloat162 (&v)[4]) {
  uint32_t u[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) u[k] = *reinterpret_cast<const uint32_t *>(&v[k]);
  return make_uint4(u[0], u[1], u[2], u[3]);
}

// CUT: with tiles that pairs share (a kernel of its own: as a branch of one it cost the others 1.6 us a launch).
template <int EPI, bool CUT>
__global__ void __launch_bounds__(kPairThreads, 1) k_gemm_pair(const GemmPairArgs a) {
  pdl_launch_dependents();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_rank();
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  constexpr bool sw = EPI == PAIR_SWIGLU;

  extern __shared__ __align__(128) unsigned char pair_smem[];
  unsigned char *const smem = pair_smem + ((1024u - (smem_u32(pair_smem) & 1023u)) & 1023u);
  float *xch = reinterpret_cast<float *>(smem + kPairRing);                                 // [8 warps][16][32]
  float *t_inv = reinterpret_cast<float *>(smem + kPairRing + kPairXchBytes);               // [256]
  int *t_pos = reinterpret_cast<int *>(t_inv + 256);                                        // [256]
  size_t *t_base = reinterpret_cast<size_t *>(t_pos + 256);                                 // [256]
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kPairRing + kPairXchBytes + kPairInfoBytes);
  uint64_t *full = bars, *empty = bars + kPairSlots, *accfull = bars + 2 * kPairSlots, *accempty = accfull + 2;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(accempty + 2);
  volatile int *abort_s = reinterpret_cast<int *>(tmem_slot + 1);

  const int stage_bytes = kTcABytes + 2 * a.nb * 128;
  const int nstage = min(kPairSlots, kPairRing / stage_bytes);
  const int N = 2 * a.nb;
  const int kboxes = (a.K + 63) >> 6;
  const int items = a.token_tiles * a.weight_tiles * a.S;
  const int tiles_per_seg = sw ? a.weight_tiles : a.weight_tiles / a.nseg;
  // The pair's work, a tile and a range of its boxes at a time: whole tiles (or K splits) dealt in turn, then, of the tiles from `whole`
  // on, a run of accumulators as long as every other pair's, which may start and end inside a tile.
  const int kruns = CUT ? (kboxes + a.chunk - 1) / a.chunk : 0, whole = CUT ? a.whole : items;
  auto run_begin = [&](int p) { return p * ((items - whole) * kruns) / npairs; };
  struct Work { int item, kb0, kb1, next, run, end; };
  auto first_work = [&](Work &w) {
    w.next = pair;
    if (CUT) { w.run = run_begin(pair); w.end = run_begin(pair + 1); }
  };
  auto next_work = [&](Work &w) {
    if (w.next < whole) {
      w.item = w.next;
      const int split = w.item / (a.token_tiles * a.weight_tiles);
      w.kb0 = split * kboxes / a.S; w.kb1 = (split + 1) * kboxes / a.S;
      w.next += npairs;
      return true;
    }
    if (!CUT || w.run >= w.end) return false;
    const int i = w.run / kruns, c0 = w.run - i * kruns, c1 = min(kruns, c0 + w.end - w.run);
    w.item = whole + i;
    w.kb0 = c0 * a.chunk; w.kb1 = min(kboxes, c1 * a.chunk);
    w.run += c1 - c0;
    return true;
  };

  if (tid == 0) {
    *abort_s = 0;
    for (int i = 0; i < kPairSlots; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&accfull[i], 1); mbar_init(&accempty[i], 16); }   // eight epilogue warps of each CTA
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 2) tmem_alloc_pair(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();   // both CTAs' barriers are initialised before either counts on the other's
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // item -> split, weight tile (segment and first row), token tile
  auto decode = [&](int item, int &seg, int &tile, int &tok0, int &split) {
    const int tt = item % a.token_tiles, rest = item / a.token_tiles;
    const int wt = rest % a.weight_tiles;
    split = rest / a.weight_tiles;
    seg = sw ? 0 : wt / tiles_per_seg;
    tile = sw ? wt : wt - seg * tiles_per_seg;
    tok0 = tt * N;
  };

  // the epilogue warps hold a tile's sums: 256 x 224 + 128 x 56 registers = the 384 x 168 of the launch
  if (warp < 4) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
  if (warp == 0 && lane == 0) {
    // ------------------------------------------------------------- producer (both CTAs)
    const uint64_t pol_w = l2_policy_evict_first(), pol_x = l2_policy_evict_last();
    const unsigned tx = 2u * (unsigned)stage_bytes;   // both CTAs' boxes (rows past a matrix arrive as zeros)
    int slot = 0, it = 0;
    bool waited = false;
    Work wk;
    for (first_work(wk); next_work(wk);) {
      int seg, tile, tok0, split;
      decode(wk.item, seg, tile, tok0, split);
      const int kb0 = wk.kb0, kb1 = wk.kb1;
      const TensorMap128 *m0 = sw ? a.wmap[0] : a.wmap[seg];
      const int row = sw ? tile * 128 + (int)rank * 64 : tile * 256 + (int)rank * 128;
      const int xrow = tok0 + (int)rank * a.nb;
      auto load_w = [&](int kb, int s) {
        const uint32_t st = smem_u32(smem) + (uint32_t)(s * stage_bytes), bar = peer_addr(&full[s], 0);
        if (rank == 0) mbar_expect_tx(&full[s], tx);
        tma_load_2d_pair(st, m0, kb * 64, row, bar, pol_w);
        if (sw) tma_load_2d_pair(st + kTcABytes / 2, a.wmap[1], kb * 64, row, bar, pol_w);
      };
      auto load_x = [&](int kb, int s) {
        const uint32_t st = smem_u32(smem) + (uint32_t)(s * stage_bytes) + kTcABytes, bar = peer_addr(&full[s], 0);
        tma_load_2d_pair(st, a.xhi_map, kb * 64, xrow, bar, pol_x);
        tma_load_2d_pair(st + (uint32_t)(a.nb * 128), a.xlo_map, kb * 64, xrow, bar, pol_x);
      };
      int kb = kb0;
      if (!waited) {
        // the first stages' weights depend on no kernel: they fly while the grid before this one finishes
        waited = true;
        const int nfirst = min(nstage, kb1 - kb0);
#pragma unroll 1
        for (int i = 0; i < nfirst; ++i) load_w(kb0 + i, i);
        pdl_wait();
#pragma unroll 1
        for (int i = 0; i < nfirst; ++i) load_x(kb0 + i, i);
        kb += nfirst; it = nfirst; slot = nfirst % nstage;
      }
#pragma unroll 1
      for (; kb < kb1; ++kb, ++it) {
        if (it >= nstage) mbar_wait_inline(&empty[slot], ((unsigned)(it / nstage) & 1u) ^ 1u, a.cnts, abort_s);
        if (*abort_s) break;
        load_w(kb, slot);
        load_x(kb, slot);
        slot = slot + 1 == nstage ? 0 : slot + 1;
      }
    }
    if (!waited) pdl_wait();
    // the last stages' releases are not awaited here: the leader's products have completed before the CTAs meet below
  } else {
    pdl_wait();
  }
  __syncwarp();

  if (warp == 1 && rank == 0) {
    // ------------------------------------------------------------- tensor-core issuer (leader)
    const uint32_t idesc = umma_idesc_mn(256u, (uint32_t)N);
    // operands from values that are the same in all lanes as far as the compiler can see, and no loop over the 16-k steps of
    // a whole box: products whose operands have to be fetched from a lane first issue at 80 clocks each (512 rows, 7B:
    // 15.9 -> 14.9 ms a prompt; 333 rows, 16 layers of 2048: 2296 -> 2130 us)
    const uint32_t tb = __reduce_max_sync(0xffffffffu, tmem_base), sb = __reduce_max_sync(0xffffffffu, smem_u32(smem));
    int slot = 0, it = 0, n = 0;   // n: accumulators filled so far
    Work wk;
    for (first_work(wk); next_work(wk);) {
      const int kb0 = wk.kb0, kb1 = wk.kb1;
      for (int kc = kb0; kc < kb1; kc += a.chunk, ++n) {
        const int buf = n & 1, kc1 = min(kb1, kc + a.chunk);
        if (n >= 2) mbar_wait_inline(&accempty[buf], ((unsigned)(n >> 1) & 1u) ^ 1u, a.cnts, abort_s);
        tc_fence_after();
        const uint32_t dcol = tb + (uint32_t)buf * 256;
#pragma unroll 1
        for (int kb = kc; kb < kc1; ++kb, ++it) {
          mbar_wait_inline(&full[slot], (unsigned)(it / nstage) & 1u, a.cnts, abort_s);
          tc_fence_after();
          if (elect_one()) {
            const uint32_t st = sb + (uint32_t)(slot * stage_bytes);
            const uint64_t ad = umma_desc(st), bh = umma_desc(st + kTcABytes), bl = umma_desc(st + kTcABytes + (uint32_t)(a.nb * 128));
            const uint32_t acc = kb > kc ? 1u : 0u;
            if (kb * 64 + 64 <= a.K) {
#pragma unroll
              for (int k4 = 0; k4 < 4; ++k4) umma_bf16_pair(dcol, ad + 2 * k4, bl + 2 * k4, idesc, k4 > 0 ? 1u : acc);
#pragma unroll
              for (int k4 = 0; k4 < 4; ++k4) umma_bf16_pair(dcol, ad + 2 * k4, bh + 2 * k4, idesc, 1u);
            } else {
              const int nstep = (a.K - kb * 64 + 15) >> 4;   // k16 steps holding any k < K
#pragma unroll 1
              for (int k4 = 0; k4 < nstep; ++k4) umma_bf16_pair(dcol, ad + 2 * k4, bl + 2 * k4, idesc, k4 > 0 ? 1u : acc);
#pragma unroll 1
              for (int k4 = 0; k4 < nstep; ++k4) umma_bf16_pair(dcol, ad + 2 * k4, bh + 2 * k4, idesc, 1u);
            }
            umma_commit_pair(&empty[slot]);
          }
          __syncwarp();
          slot = slot + 1 == nstage ? 0 : slot + 1;
        }
        if (elect_one()) umma_commit_pair(&accfull[buf]);
        __syncwarp();
      }
    }
  }

  } else {
    // ------------------------------------------------------------- epilogue (both CTAs)
    asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
    pdl_wait();
    const int quarter = warp & 3, ch = (warp - 4) >> 2, etid = tid - 128;    // ch: which nb columns of the tile
    int n = 0;
    // the other value of a pair: gate / up are 64 lanes apart, rotary pairs hd / 2
    const int dist = sw ? 2 : (a.hd == 128 ? 2 : 1);       // in warps
    // Exchange area of a warp: [16 prompt rows][32 weight rows].  Thread gid of the four warps reads eight weight rows (w0, and those `dist`
    // warps on) of prompt row gid / 8; the warps whose areas the same eight threads read have their groups of four swapped, so
    // that the eight read from different banks.
    float *own_at = xch + (ch * 4 + quarter) * 16 * 32;
    const int gid = etid & 127, wq = sw || a.hd == 128 ? (gid & 7) >> 2 : ((gid & 7) >> 2) * 2;
    const float *low_at = xch + (ch * 4 + wq) * 16 * 32 + (gid >> 3) * 32 + 8 * (gid & 3), *high_at = low_at + dist * 16 * 32;
    auto xch_swap = [](int q) { return ((q ^ (q >> 1)) & 1) << 2; };
    auto row_info = [&](int tok0, int Tl) {
      // per prompt row of the tile: 1/rms of its residual stream and, for keys and values, where its cache row starts
      for (int i = etid; i < Tl; i += 256) {
        t_inv[i] = inv_rms_of(a.ss_part, tok0 + i, a.d, a.eps);
        if (!sw) {
          const int pos = a.pass->row_pos[tok0 + i], b = a.pass->row_seq[tok0 + i];
          t_pos[i] = pos;
          const int page = a.page_table[b * a.pages_per_seq + pos / kPageSize];
          t_base[i] = (((size_t)page * a.L + a.layer) * a.H * kPageSize + (size_t)(pos % kPageSize)) * a.hd;
        }
      }
    };
    Work wk;
    for (first_work(wk); next_work(wk);) {
      int seg, tile, tok0, split;
      decode(wk.item, seg, tile, tok0, split);
      const int kb0 = wk.kb0, kb1 = wk.kb1;
      const int Tl = min(N, a.T - tok0);
      float sum[4][32];
#pragma unroll
      for (int blk = 0; blk < 4; ++blk)
#pragma unroll
        for (int i = 0; i < 32; ++i) sum[blk][i] = 0.f;
      for (int kc = kb0; kc < kb1; kc += a.chunk, ++n) {
        const int buf = n & 1;
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * 256 + ch * a.nb);
        mbar_wait_inline(&accfull[buf], (unsigned)(n >> 1) & 1u, a.cnts, abort_s);
        tc_fence_after();
#pragma unroll
        for (int blk = 0; blk < 4; ++blk)
          if (blk * 32 < a.nb) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              float v[16];
              tmem_ld16(taddr + (uint32_t)(blk * 32 + h * 16), v);
#pragma unroll
              for (int i = 0; i < 16; ++i) sum[blk][h * 16 + i] += v[i];
            }
          }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_peer(peer_addr(&accempty[buf], 0));
        if (EPI != PAIR_PART && kc == 0) row_info(tok0, Tl);   // (under the products of the chunks that follow)
      }
      if constexpr (CUT) {
        // A tile cut by the runs' ends: the pair that has its first boxes, the last of its run, finishes it; the others, for which it is the
        // first of theirs, leave their sums in memory.  A warp takes what the same warp of the other pairs left.
        const size_t at = (size_t)(ch * a.nb) * 128 + quarter * 32 + lane;
        const int ew = warp - 4;
        if (kb0 > 0) {
          float *o = a.cut + (size_t)blockIdx.x * N * 128 + at;
#pragma unroll
          for (int blk = 0; blk < 16; ++blk)
            if (blk * 8 < a.nb) {
#pragma unroll
              for (int i = 0; i < 8; ++i) __stcg(o + (size_t)(blk * 8 + i) * 128, sum[blk >> 2][(blk & 3) * 8 + i]);
            }
          __syncwarp();
          if (lane == 0) asm volatile("st.release.gpu.global.s32 [%0], 1;" ::"l"(a.cut_flags + blockIdx.x * 8 + ew) : "memory");
          continue;
        }
        if (kb1 < kboxes) {
          const int tile_end = (wk.item - whole + 1) * kruns;
#pragma unroll 1
          for (int p = pair + 1; run_begin(p) < tile_end; ++p) {
            const int cta = 2 * p + (int)rank;
            int *flag = a.cut_flags + cta * 8 + ew;
            if (lane == 0) {
              for (unsigned i = 0;; ++i) {
                if (ld_acquire(reinterpret_cast<const unsigned *>(flag)) == 1u || *abort_s) break;
                if (i > 64) __nanosleep(40);
                if (i == kSpinLimit) { *abort_s = 1; atomicOr(&a.cnts->status, kStatTimeout); }
              }
            }
            __syncwarp();
            const float *q = a.cut + (size_t)cta * N * 128 + at;
#pragma unroll
            for (int blk = 0; blk < 4; ++blk)
              if (blk * 32 < a.nb) {
                float v[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = blk * 32 + (i & ~7) < a.nb ? __ldcg(q + (size_t)(blk * 32 + i) * 128) : 0.f;
#pragma unroll
                for (int i = 0; i < 32; ++i) sum[blk][i] += v[i];
              }
            __syncwarp();
            if (lane == 0) *flag = 0;
          }
        }
      }
      if constexpr (EPI == PAIR_PART) {
        // By way of the warp's exchange area, 16 prompt rows at a time, so that a lane stores four weight rows of a prompt row at once.
        const int row4 = tile * 256 + (int)rank * 128 + quarter * 32 + 4 * (lane & 7), rows = min(a.nb, Tl - ch * a.nb);
        float *pp = a.part + ((size_t)split * a.part_rows + tok0 + ch * a.nb + (lane >> 3)) * a.Nseg + row4;
#pragma unroll 1
        for (int b16 = 0; b16 * 16 < rows; ++b16) {
          __syncwarp();
#pragma unroll
          for (int b = 0; b < 8; ++b)
            if (b == b16) {
#pragma unroll
              for (int k = 0; k < 16; ++k) own_at[k * 32 + lane] = sum[b >> 1][(b & 1) * 16 + k];
            }
          __syncwarp();
#pragma unroll
          for (int k = 0; k < 16; k += 4, pp += (size_t)4 * a.Nseg)
            if (b16 * 16 + k + (lane >> 3) < rows && row4 < a.Nseg)
              __stcg(reinterpret_cast<float4 *>(pp), *reinterpret_cast<const float4 *>(own_at + k * 32 + 4 * lane));
        }
      } else {
        // A thread finishes eight neighbouring weight rows (and the eight that they are paired with) of one of 16 prompt rows, so that what
        // it stores are 16 bytes or more and a row's information is read once.  (Two
        // weight rows of four prompt rows a thread: the tile of a CTA took 6.3 thousand clocks at nb = 64 for 3.9 now, SwiGLU, and 19 for 17 at nb
        // = 128, queries; four layers of 2048 and 333 rows 677 -> 665 us, 7B 205 rows 1169 -> 1153.)
        const int half = a.hd >> 1, gr = gid & 7, w0 = sw || a.hd == 128 ? 8 * gr : 64 * (gr >> 2) + 8 * (gr & 3);
        const int row = (sw ? tile * 128 + (int)rank * 64 : tile * 256 + (int)rank * 128) + w0;   // first weight row inside its matrix
        const int hh = sw ? 0 : row / a.hd, il = sw ? 0 : row - hh * a.hd;                         // head, index of the first pair
        const size_t head_off = (size_t)hh * kPageSize * a.hd;
        named_bar(3, 256);   // the rows' information is complete
        float4 cs[4];        // rotary factors of the block, requested a block ahead
        auto rotary = [&](int tb) {
          if constexpr (!sw) {
            const float4 *f = reinterpret_cast<const float4 *>(a.rope + (size_t)t_pos[min(tb + (gid >> 3), Tl - 1)] * half + il);
#pragma unroll
            for (int k = 0; k < 4; ++k) cs[k] = seg < 2 ? __ldg(f + k) : make_float4(1.f, 0.f, 1.f, 0.f);
          }
        };
        rotary(ch * a.nb);
        // One body for all blocks (only the writes of the sums, which are registers, exist once per block): the code runs a few
        // times per launch, and eight copies of it were mostly waits for instructions -- 35 thousand clocks for a CTA's first
        // tile against 14 for the next.
#pragma unroll 1
        for (int b16 = 0; b16 * 16 < min(a.nb, Tl - ch * a.nb); ++b16) {     // (uniform over the four warps that exchange)
          const int tb = ch * a.nb + b16 * 16, i = tb + (gid >> 3);
          named_bar(1 + ch, 128);
#pragma unroll
          for (int b = 0; b < 8; ++b)
            if (b == b16) {
#pragma unroll
              for (int k = 0; k < 16; ++k) own_at[k * 32 + (lane ^ xch_swap(quarter))] = sum[b >> 1][(b & 1) * 16 + k];
            }
          named_bar(1 + ch, 128);
          float x[8], y[8];        // (gate, up) or rows (i, i + hd / 2)
          const float inv = t_inv[i];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const float4 u = *reinterpret_cast<const float4 *>(low_at + ((4 * k) ^ xch_swap(wq))), v = *reinterpret_cast<const float4 *>(high_at + ((4 * k) ^ xch_swap(wq + dist)));
            x[4 * k] = u.x * inv; x[4 * k + 1] = u.y * inv; x[4 * k + 2] = u.z * inv; x[4 * k + 3] = u.w * inv;
            y[4 * k] = v.x * inv; y[4 * k + 1] = v.y * inv; y[4 * k + 2] = v.z * inv; y[4 * k + 3] = v.w * inv;
          }
          float4 c[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) c[k] = cs[k];
          if ((b16 + 1) * 16 < a.nb) rotary(tb + 16);
          if (row >= a.Nseg || i >= min(Tl, (ch + 1) * a.nb)) continue;
          if constexpr (sw) {
            __nv_bfloat162 hi[4], lo[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              split_bf16(silu(x[2 * k]) * y[2 * k], hi[k].x, lo[k].x);
              split_bf16(silu(x[2 * k + 1]) * y[2 * k + 1], hi[k].y, lo[k].y);
            }
            const size_t o = (size_t)(tok0 + i) * a.ldo + row;
            *reinterpret_cast<uint4 *>(a.ohi + o) = pack8(hi);
            *reinterpret_cast<uint4 *>(a.olo + o) = pack8(lo);
          } else {
            float v0[8], v1[8];   // (values: x and y as they are)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              v0[2 * k] = x[2 * k] * c[k].x - y[2 * k] * c[k].y; v0[2 * k + 1] = x[2 * k + 1] * c[k].z - y[2 * k + 1] * c[k].w;
              v1[2 * k] = y[2 * k] * c[k].x + x[2 * k] * c[k].y; v1[2 * k + 1] = y[2 * k + 1] * c[k].z + x[2 * k + 1] * c[k].w;
            }
            if (seg == 0) {
              float *q = a.qout + (size_t)(tok0 + i) * a.d + hh * a.hd + il;
#pragma unroll
              for (int k = 0; k < 8; k += 4) {
                *reinterpret_cast<float4 *>(q + k) = make_float4(v0[k] * a.qscale, v0[k + 1] * a.qscale, v0[k + 2] * a.qscale, v0[k + 3] * a.qscale);
                *reinterpret_cast<float4 *>(q + half + k) = make_float4(v1[k] * a.qscale, v1[k + 1] * a.qscale, v1[k + 2] * a.qscale, v1[k + 3] * a.qscale);
              }
            } else {
              const int s7 = t_pos[i] & 7;
              __nv_bfloat16 *pool = (seg == 1 ? a.kpool : a.vpool) + t_base[i] + head_off;
              __nv_bfloat162 p0[4], p1[4];
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                p0[k].x = kv_store(v0[2 * k]); p0[k].y = kv_store(v0[2 * k + 1]);
                p1[k].x = kv_store(v1[2 * k]); p1[k].y = kv_store(v1[2 * k + 1]);
              }
              *reinterpret_cast<uint4 *>(pool + (((il >> 3) ^ s7) << 3)) = pack8(p0);
              *reinterpret_cast<uint4 *>(pool + ((((il + half) >> 3) ^ s7) << 3)) = pack8(p1);
            }
          }
        }
        named_bar(3, 256);   // the rows' information is rewritten for the next tile
      }
    }
  }

  // both CTAs are done with each other's barriers and with tensor memory
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  await_copies(abort_s);
  cluster_sync_all();
  tc_fence_after();
  if (warp == 2) tmem_dealloc_pair(tmem_base, 512);
}

}  // namespace ada
