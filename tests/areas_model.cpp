// Host model of the shared-memory area of csrc/ada_areas.h: eight worker warps, in random order, go from the products of a QKV phase
// of T rows to their first keys.  They write their sums, meet, read them row by row, and request their keys where the kernel does:
// before the sums where keys_clear_of_sums says so, else after a barrier behind the last read.  A copy may land at once or never
// be seen: it must not meet a row that any warp has still to write or to read.
// usage: areas_model T head_bytes trials  -> "ok" or the first violation; exit code 1 on error
#include <cstdio>
#include <cstdlib>
#include <random>
#include "ada_areas.h"
using namespace ada;

int main(int argc, char **argv) {
  if (argc < 4) return 2;
  const int T = atoi(argv[1]), piece = 16 * atoi(argv[2]), trials = atoi(argv[3]), TP = (T + 7) & ~7;
  const bool early = keys_clear_of_sums(TP);
  constexpr int kWarps = 8;
  std::mt19937 rng(T);
  for (int trial = 0; trial < trials; ++trial) {
    int state[kWarps] = {0}, row[kWarps] = {0};   // 0 start, 1 writes its sums, 2 met, 3 reads, 4 read, 5 met again, 6 requested
    auto at_least = [&](int s) { for (int w = 0; w < kWarps; ++w) if (state[w] < s) return false; return true; };
    auto request = [&](int w) {   // overlap with a row that somebody still needs?
      for (int o = 0; o < kWarps; ++o)
        for (int t = state[o] == 3 ? row[o] : 0; t < TP && state[o] < 4; ++t)
          for (int v = 0; v < 2; ++v) {
            const int beg = kKeysAt + w * kKeysWarpBytes + v * kKeysWarpBytes / 2;
            if (beg < (t + 1) * kSumsRowBytes && t * kSumsRowBytes < beg + piece) {
              printf("T %d: keys of warp %d land on row %d, which warp %d needs\n", T, w, t, o);
              return false;
            }
          }
      return true;
    };
    for (int steps = 0; !at_least(6);) {
      if (++steps > 1000000) { printf("T %d: no end\n", T); return 1; }
      const int w = (int)(rng() % kWarps);
      switch (state[w]) {
        case 0: if (early && !request(w)) return 1; state[w] = 1; break;
        case 1: state[w] = 2; break;
        case 2: if (at_least(2)) { state[w] = 3; row[w] = 0; } break;
        case 3: if (++row[w] == TP) state[w] = early ? 6 : 4; break;
        case 4: state[w] = 5; break;
        case 5: if (at_least(5)) { if (!request(w)) return 1; state[w] = 6; } break;
      }
    }
  }
  printf("ok\n");
  return 0;
}
