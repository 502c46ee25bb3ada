// Shape of the work of k_small (ada_small.cuh): what each CTA of a cluster does, where everything lies in its shared memory, and who sends
// in which exchange.  Plain C++, so that a host program can follow the exchanges (tests/small_model.cpp).
#pragma once
#ifndef __CUDACC__
#define __host__
#define __device__
#endif

struct __nv_bfloat16;

namespace ada {

constexpr int kSmCtas = 16;                 // CTAs of a cluster
constexpr int kSmWarps = 8;
constexpr int kSmThreads = kSmWarps * 32;
constexpr int kSmHd = 64;                   // width of a head
constexpr int kSmRowsMax = 16;              // rows of a sequence in one pass at most (n_max + 1)
constexpr int kSmLmUnits = 8;               // units of 32 k of the LM head: two tiles of a warp stay in its registers
constexpr int kSmLmRound = 2 * kSmWarps;    // its tiles that are there at a time
// Vocabulary at most: beyond 4096 rows the LM head no longer stays in the registers, and sixteen SMs read it at 40 GB/s each.  Draft of
// four + verify, k_pass -> here: 4096 rows 134 + 62 -> 55 + 46 us, 8192 142 + 64 -> 71 + 50, 16 384 144 + 67 -> 95 + 60, 32 768 150 +
// 69 -> 155 + 83.
constexpr int kSmVocabMax = 16384;
constexpr int kSmCandBytes = 16;            // a warp's candidate for a row, with its sum of exponentials
constexpr int kSmRed = 20;                  // floats per row of a warp's 16 sums (an 8 x 4 fragment then stores into 32 banks)
enum { SM_FC = 0, SM_QKV, SM_O, SM_GU, SM_DOWN, SM_LM, kSmKinds };                        // phases with products
// Exchanges: fc, q k v, attention, O, gate/up, down, candidates; then the weights of a layer's phases.
//
// Every CTA takes part in X, A, O, D and a draft's C: one that has nothing to send (no columns of d, no head) sends 16 bytes that nobody
// reads, when it has read all that came before.  So whoever has awaited one of these exchanges knows that all CTAs have done everything
// before it.  (Q is among the CTAs of a head, C of a verify pass goes to CTA 0, and AC, which all await, comes from the CTAs with tiles
// of gate/up only.)
//
//   place      written by       read by                            written again by senders who have awaited
//   x[i]       X, O, D in turn  fc (the feature), QKV, gate/up,    C (X), A (O), O (D): sent after the last product with what
//              into either      LM head                            the buffer held
//   q          Q                attention                          D of the layer before, X of the same step
//   fk, fv     Q                attention                          D of the layer before; a draft step's rows have their own place
//   ac         A                merging for O                      O
//              AC               down                               D, in a draft C
//   cand       C                the choice                         X
//   send[i]    this CTA         its own copies                     (this CTA, three exchanges on) the next of X, A, O, D, C but one's own,
//                               which every CTA sends when it has received them
//   barrier    its exchange     this CTA                           an exchange that this CTA sends when it has awaited the one before: a phase's
//                               bytes may come before this CTA has armed it, but never while the phase before it is not complete
//
// A CTA whose wait gave up takes no part any more: it arms and sends nothing, all others' waits end by the status word, and all meet at the
// kernel's end, where they are told and stay until every copy has landed.
//
// (tests/small_model.cpp runs the CTAs through it in any order.)
enum { SMX_X = 0, SMX_Q, SMX_A, SMX_O, SMX_AC, SMX_D, SMX_C, SMX_W, kSmBars = SMX_W + SM_LM };

// Shape of the work and places in shared memory (bytes from the aligned start), worked out on the host.
struct SmallShape {
  int ns;                                   // CTAs per head (whole ones)
  int qt, gt, lt;                           // tiles of a CTA at most: QKV, gate/up (8 columns each), vocabulary (of d columns it has one)
  int heads;                                // CTAs that have a share of a head: the first ones
  int shift[SM_LM];                         // by kind of phase, log2 of the warps that share a tile's K
  int cap_slots;                            // fresh cache rows kept in shared memory
  const __nv_bfloat16 *w_fc, *w_lm;
  int pages, hown, gains, rope, x[2], e, ac, q, fk, fv, cand, send[3], scratch, w[SM_LM], total;
};

__host__ __device__ inline int small_align(int x) { return (x + 127) & ~127; }

// Rows that a chunk of activations is stored for: odd, so that the loads of eight lanes, two rows of four neighbouring chunks, fall into
// different banks.
__host__ __device__ inline int small_stride(int T) { return T | 1; }
// Bytes of a CTA's 16 columns of an input X with the rows' partial sums of squares behind them: one copy to each CTA.
__host__ __device__ inline int small_xblock(int T) { return 64 * small_stride(T) + ((4 * T + 15) & ~15); }
// Bytes of a CTA's partial sums of its head: of each row hd sums, then of each row (maximum, sum).
__host__ __device__ inline int small_part(int T) { return T * kSmHd * 4 + ((T * 8 + 15) & ~15); }
// A token as an index of the vocabulary: a candidate is read from memory that others fill, and nobody has where a wait gave up.
__host__ __device__ inline int small_token(int i, int V) { return (unsigned)i < (unsigned)V ? i : 0; }
constexpr int kSmNone = 1008, kSmNoneBytes = 16;   // where, and how much, a CTA without a share sends
// Bytes of an exchange whose first n CTAs send `bytes` each.
__host__ __device__ inline int small_expect(int n, int bytes) { return n * bytes + (kSmCtas - n) * kSmNoneBytes; }
constexpr int kSmSmemMax = 227 * 1024;
// False if the kernel's plan does not hold the shape.  d_model up to 256 (a CTA has one tile of 16 columns of d) and heads of 64 are what
// the plan was written for, not where k_pass gets faster: draft of four + verify of five rows at context 100, us, d_model 256 in four heads
// 48 + 40 here, in two heads of 128 139 + 65 on k_pass, d_model 320 148 + 68; seven sequences 48 + 41, 182 + 112, 195 + 114; an eighth
// makes a second round of clusters: 89 + 75, 184 + 110, 198 + 116.
__host__ inline bool small_shape(int L, int d, int H, int hd, int F, int V, int nmax, int pages_per_seq, SmallShape &z) {
  if (H > kSmCtas || nmax + 1 > kSmRowsMax || hd != kSmHd || d > 16 * kSmCtas || V > kSmVocabMax) return false;
  const int R = nmax + 1, Rs = small_stride(R), slots = 2 * nmax + 1;
  z.ns = kSmCtas / H;
  z.qt = (3 * hd / 16 + z.ns - 1) / z.ns;
  z.gt = (F / 8 + kSmCtas - 1) / kSmCtas;
  z.lt = (V / 16 + kSmCtas - 1) / kSmCtas;
  z.heads = H * z.ns;
  // as many warps to a tile as there are, no more than K has units
  const int tiles[SM_LM] = {1, z.qt, 1, z.gt, 1}, K[SM_LM] = {2 * d, d, d, d, F};
  for (int k = 0; k < SM_LM; ++k) {
    const int units = (K[k] + 31) / 32;
    int l = 0;
    while ((2 << l) * tiles[k] <= kSmWarps && (2 << l) <= units) ++l;
    if (tiles[k] << l > kSmWarps) return false;
    z.shift[k] = l;
  }
  z.cap_slots = slots;
  const int part = small_part(R);
  int at = small_align(1024 + kSmWarps * kSmRowsMax * (kSmCandBytes));   // barriers, row information; candidates of the warps
  auto take = [&](int bytes) { const int p = at; at += small_align(bytes); return p; };
  z.pages = take(pages_per_seq * 4);
  z.hown = take(R * 16 * 4);
  z.gains = take((2 * L + 1) * 16 * 4);
  z.rope = take(slots * hd / 2 * 8);
  for (int i = 0; i < 2; ++i) z.x[i] = take(d / 16 * small_xblock(R));
  const int acb = 4 * Rs * F, rcv = H * z.ns * part;
  z.ac = take(acb > rcv ? acb : rcv);
  z.q = take(4 * Rs * hd);
  z.fk = take(2 * hd * slots);
  z.fv = take(2 * hd * slots);
  z.cand = take(kSmCtas * R * 32);
  int sb = part;
  auto up = [&](int v) { if (v > sb) sb = v; };
  up(small_xblock(R)); up(z.gt * 32 * Rs); up(z.qt * 64 * Rs); up(32 * R);
  for (int i = 0; i < 3; ++i) z.send[i] = take(sb);
  // the products' sums, behind them the embeddings (draft) or attention's result, whose readers write no sums of their own over them; the
  // warps' partial sums of attention over both
  const int red = small_align(kSmWarps * R * kSmRed * 4);
  int sc = red + 4 * Rs * d;
  auto upc = [&](int v) { if (v > sc) sc = v; };
  upc(kSmWarps * R * (hd + 4) * 4); upc(kSmWarps * R * 2 * kSmRed * 4);
  z.scratch = take(sc);
  z.e = z.scratch + red;
  for (int k = 0; k < SM_LM; ++k) z.w[k] = take(tiles[k] * 32 * K[k]);
  z.total = at + 128;
  return z.total <= kSmSmemMax;
}

}  // namespace ada
