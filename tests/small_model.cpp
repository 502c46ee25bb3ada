// Host model of the exchanges of k_small (csrc/ada_small.cuh, places and participants from csrc/ada_small_shape.h): the 16 CTAs of a
// cluster and the copies between them take their steps in any order.  Checked at every step:
//   - a copy lands on no bytes that its receiver has still to read for something earlier than what it brings
//   - bytes reach a barrier in the phase that they are meant for
//   - a CTA writes no buffer that a copy of its own has still to read
//   - all CTAs come to the end, and nothing is under way when they leave
// Where a wait gives up (in any CTA, at any time; the status word then ends the other CTAs' waits) what arrives is of no use to anyone.  Checked
// instead:
//   - no barrier is armed again before its phase is complete
//   - nothing is under way to or from a CTA that has left
// usage: small_model d heads F V n_max rows layers draft(0: verify, else steps) silent trials [gives_up]
//   silent 1: CTAs without a share say nothing (an order that must be found wrong for narrow models)
//   gives_up 1: a wait of each trial gives up; 2: and its CTA goes on arming and sending; 3: it does not, but it alone stays for a while, before
//   it meets the others at the end (2 and 3 must be found wrong)
//        small_model token V i [i ...]   -> the vocabulary row that is read for candidate i
// prints "ok" and returns 0, "refused" (3) for a shape that the kernel does not take, or the first violation (1)
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <vector>
#include "ada_small_shape.h"
using namespace ada;

enum Kind { READ, WRITE, ARM, SEND, WAIT };
struct Op {
  Kind kind;
  int ex, inst;              // exchange and its how-many-th instance
  int at, bytes;             // place in this CTA (READ, WRITE, source of SEND); bytes expected (ARM)
  int dst, to;               // SEND: receiver and place there
};
struct Copy { int src, at, bytes, dst, to, ex, inst; };
struct Bar { int phase = 0, pending = 1, tx = 0; };

static SmallShape z;
static int d, H, F, V, nmax, rows, layers, steps, silent;

// What CTA `rank` does, in order.
static std::vector<Op> program(int rank) {
  std::vector<Op> o;
  int inst[kSmBars] = {0}, xs = 1, sbuf = 0;
  const int cols = d / 16;
  const bool has_d = rank < cols, has_head = rank < z.heads;
  const int hh = rank / z.ns, split = rank % z.ns, ntile = kSmHd / 16;
  const int qtiles = has_head ? (3 * ntile - split + z.ns - 1) / z.ns : 0;
  const int gtile0 = rank * z.gt, gtiles = std::max(0, std::min(F / 8 - gtile0, z.gt));
  auto read = [&](int at, int bytes) { o.push_back({READ, 0, 0, at, bytes, 0, 0}); };
  auto wait = [&](int ex) { o.push_back({WAIT, ex, inst[ex]++, 0, 0, 0, 0}); };
  auto write = [&](int bytes) { o.push_back({WRITE, 0, 0, z.send[sbuf], bytes, 0, 0}); };
  auto all = [&](int ex, int n, bool has, int to, int bytes) {   // the first n CTAs send `bytes` each
    o.push_back({ARM, ex, inst[ex], 0, silent ? n * bytes : small_expect(n, bytes), 0, 0});
    for (int c = 0; c < kSmCtas && (has || !silent); ++c)
      o.push_back({SEND, ex, inst[ex], z.send[sbuf], has ? bytes : kSmNoneBytes, c, has ? to : kSmNone});
  };
  auto next = [&] { sbuf = sbuf == 2 ? 0 : sbuf + 1; };
  int pos = 0;
  for (int step = 0; step < (steps ? steps : 1); ++step) {
    const int T = step ? 1 : rows, TS = small_stride(T), XB = small_xblock(T), part = small_part(T), X = cols * XB;
    int arrive = -1;
    if (steps) {   // fc: the feature lies with the rows of the step before
      if (has_d) read(z.x[xs], cols * small_xblock(step <= 1 ? rows : 1));
      next();
      write(XB);
      xs ^= 1;
      all(SMX_X, cols, has_d, z.x[xs] + rank * XB, XB);
      arrive = SMX_X;
    }
    for (int l = 0; l < (steps ? 1 : layers); ++l) {
      if (arrive >= 0) wait(arrive);
      read(z.x[xs], X);
      next();
      if (qtiles) write(qtiles * 64 * TS);
      if (has_head) o.push_back({ARM, SMX_Q, inst[SMX_Q], 0, 4 * kSmHd * (T + TS), 0, 0});
      for (int e = 0; e < qtiles * z.ns; ++e) {
        const int tile = e / z.ns, m = split + z.ns * tile, type = m / ntile, i = m % ntile;
        const int to = type == 0 ? z.q + i * 64 * TS : (type == 1 ? z.fk : z.fv) + pos * ntile * 32 + i * 32 * T;
        o.push_back({SEND, SMX_Q, inst[SMX_Q], z.send[sbuf] + tile * 64 * TS, type == 0 ? 64 * TS : 32 * T, hh * z.ns + e % z.ns, to});
      }
      if (has_head) {
        wait(SMX_Q);
        read(z.q, 4 * kSmHd * TS);
        read(z.fk, 2 * kSmHd * (pos + T));
        read(z.fv, 2 * kSmHd * (pos + T));
      }
      next();
      if (has_head) write(part);
      all(SMX_A, z.heads, has_head, z.ac + rank * part, part);
      wait(SMX_A);
      read(z.ac, z.heads * part);
      next();
      write(XB);
      xs ^= 1;
      all(SMX_O, cols, has_d, z.x[xs] + rank * XB, XB);
      wait(SMX_O);
      read(z.x[xs], X);
      next();
      if (gtiles) write(gtiles * 32 * TS);
      o.push_back({ARM, SMX_AC, inst[SMX_AC], 0, F * 4 * TS, 0, 0});
      for (int c = 0; c < kSmCtas && gtiles; ++c) o.push_back({SEND, SMX_AC, inst[SMX_AC], z.send[sbuf], gtiles * 32 * TS, c, z.ac + gtile0 * 32 * TS});
      wait(SMX_AC);
      if (has_d) read(z.ac, F * 4 * TS);
      next();
      write(XB);
      xs ^= 1;
      all(SMX_D, cols, has_d, z.x[xs] + rank * XB, XB);
      arrive = SMX_D;
    }
    wait(SMX_D);
    read(z.x[xs], X);
    const int Tg = steps ? 1 : T;
    next();
    write(32 * Tg);
    if (steps) {
      all(SMX_C, kSmCtas, true, z.cand + rank * 32 * Tg, 32 * Tg);
      wait(SMX_C);
      read(z.cand, kSmCtas * 32 * Tg);
    } else {
      if (rank == 0) o.push_back({ARM, SMX_C, 0, 0, kSmCtas * 32 * Tg, 0, 0});
      o.push_back({SEND, SMX_C, 0, z.send[sbuf], 32 * Tg, 0, z.cand + rank * 32 * Tg});
      if (rank == 0) { wait(SMX_C); read(z.cand, kSmCtas * 32 * Tg); }
    }
    pos += T;
  }
  return o;
}

static bool meet(int a, int an, int b, int bn) { return a < b + bn && b < a + an; }

int main(int argc, char **argv) {
  if (argc > 2 && !strcmp(argv[1], "token")) {
    for (int i = 3; i < argc; ++i) printf("%d ", small_token((int)strtoll(argv[i], nullptr, 0), atoi(argv[2])));
    return 0;
  }
  if (argc < 11) return 2;
  d = atoi(argv[1]); H = atoi(argv[2]); F = atoi(argv[3]); V = atoi(argv[4]); nmax = atoi(argv[5]); rows = atoi(argv[6]); layers = atoi(argv[7]);
  steps = atoi(argv[8]); silent = atoi(argv[9]);
  const int trials = atoi(argv[10]), gives_up = argc > 11 ? atoi(argv[11]) : 0;
  if (!small_shape(layers, d, H, H > 0 ? d / H : 0, F, V, nmax, 8, z)) { printf("refused\n"); return 3; }
  if (rows > nmax + 1 || steps > nmax) return 2;
  std::vector<Op> prog[kSmCtas];
  std::vector<size_t> wait_at[kSmCtas][kSmBars];   // where a CTA awaits an exchange's instances
  for (int c = 0; c < kSmCtas; ++c) {
    prog[c] = program(c);
    for (size_t i = 0; i < prog[c].size(); ++i)
      if (prog[c][i].kind == WAIT) wait_at[c][prog[c][i].ex].push_back(i);
      else if ((prog[c][i].kind == READ || prog[c][i].kind == WRITE) && prog[c][i].at + prog[c][i].bytes > z.total) { printf("past the end\n"); return 1; }
  }
  std::mt19937 rng(12345);
  for (int trial = 0; trial < trials; ++trial) {
    Bar bar[kSmCtas][kSmBars];
    size_t pc[kSmCtas] = {0};
    std::vector<Copy> fly;
    // CTAs run by a priority that changes now and then; copies land at random, early in some trials and late in others
    int prio[kSmCtas];
    for (int c = 0; c < kSmCtas; ++c) prio[c] = c;
    std::shuffle(prio, prio + kSmCtas, rng);
    const unsigned land = trial % 3 == 0 ? 1 : trial % 3 == 1 ? 8 : 64, change = trial % 2 ? 40 : 4000;
    bool status = false, given[kSmCtas] = {false};   // a wait has given up; in this CTA
    int countdown = gives_up ? (int)(rng() % 50000) : -1;
    auto complete = [&](int c, int e) {
      Bar &b = bar[c][e];
      if (b.pending == 0 && b.tx == 0) { ++b.phase; b.pending = 1; }
    };
    auto reaches = [&](int c, int e, int inst, const char *what) {
      if (status || bar[c][e].phase == inst) return true;
      printf("trial %d: %s for instance %d of exchange %d come to CTA %d in phase %d\n", trial, what, inst, e, c, bar[c][e].phase);
      return false;
    };
    for (;;) {
      if (rng() % change == 0) std::shuffle(prio, prio + kSmCtas, rng);
      int c = -1;
      for (int i = 0; i < kSmCtas && c < 0; ++i) {
        const int k = prio[i];
        if (pc[k] == prog[k].size()) continue;
        const Op &o = prog[k][pc[k]];
        if (o.kind != WAIT || bar[k][o.ex].phase > o.inst || given[k]) { c = k; continue; }
        if (gives_up && (status ? fly.empty() || rng() % 16 == 0 : countdown-- <= 0)) { status = given[k] = true; c = k; }
      }
      if (!fly.empty() && (c < 0 || rng() % land == 0)) {
        const size_t i = rng() % fly.size();
        const Copy f = fly[i];
        fly[i] = fly.back();
        fly.pop_back();
        const auto &w = wait_at[f.dst][f.ex];
        const size_t known = f.inst < (int)w.size() ? w[f.inst] : prog[f.dst].size();
        for (size_t k = pc[f.dst]; k < known && !status; ++k) {
          const Op &o = prog[f.dst][k];
          if (o.kind == READ && meet(o.at, o.bytes, f.to, f.bytes)) {
            printf("trial %d: exchange %d of CTA %d lands on what CTA %d has still to read\n", trial, f.ex, f.src, f.dst);
            return 1;
          }
        }
        if (!reaches(f.dst, f.ex, f.inst, "bytes")) return 1;
        bar[f.dst][f.ex].tx -= f.bytes;
        complete(f.dst, f.ex);
        continue;
      }
      if (c < 0) break;
      const Op &o = prog[c][pc[c]++];
      const bool off = given[c] && gives_up != 2;    // it takes no part any more
      if (o.kind == WRITE && !status) {
        for (const Copy &f : fly)
          if (f.src == c && meet(o.at, o.bytes, f.at, f.bytes)) {
            printf("trial %d: CTA %d writes what its copy for exchange %d has still to read\n", trial, c, f.ex);
            return 1;
          }
      } else if (o.kind == ARM && !off) {
        if (!reaches(c, o.ex, o.inst, "its own bytes")) return 1;
        if (bar[c][o.ex].pending == 0) { printf("trial %d: CTA %d arms exchange %d twice in a phase\n", trial, c, o.ex); return 1; }
        bar[c][o.ex].tx += o.bytes;
        --bar[c][o.ex].pending;
        complete(c, o.ex);
      } else if (o.kind == SEND && !off) {
        fly.push_back({c, o.at, o.bytes, o.dst, o.to, o.ex, o.inst});
      }
      // at the end all meet; where a wait gave up, all (3: only its CTA, and before they meet) stay until what is under way has landed
      bool all = true;
      for (int k = 0; k < kSmCtas; ++k) all = all && pc[k] == prog[k].size();
      if (gives_up == 3 && given[c] && pc[c] == prog[c].size())
        fly.erase(std::remove_if(fly.begin(), fly.end(), [&](const Copy &f) { return f.src == c || f.dst == c; }), fly.end());
      if (all && gives_up < 3 && status) fly.clear();
      if (all && !fly.empty()) {
        printf("trial %d: a copy from CTA %d to CTA %d is under way when they have left\n", trial, fly[0].src, fly[0].dst);
        return 1;
      }
    }
    for (int c = 0; c < kSmCtas; ++c)
      if (pc[c] != prog[c].size()) { printf("trial %d: CTA %d waits for exchange %d for ever\n", trial, c, prog[c][pc[c]].ex); return 1; }
  }
  printf("ok\n");
  return 0;
}
