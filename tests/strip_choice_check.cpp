// The tile of a strip launch for pairs of unequal length, run by
// tests/test_strip_choice.py: the strips that follow one another are those of the
// longer sequence, the rows those of the shorter.  Exit status 0 on success.
#include "../paper_2205_07610_gb300/csrc/ga_kx.cu"

#include <cstdio>

using namespace ga;

int main() {
  int failed = 0;
  auto tile_of = [&](int mode, int64_t m, int64_t n, int64_t pairs) {
    const int64_t R = std::min(m, n), C = std::max(m, n);
    int64_t strips[kKxWidths], chain[kKxWidths];
    for (int w = 0; w < kKxWidths; ++w) {
      strips[w] = pairs * ((C + kx_width(w) - 1) / kx_width(w));
      chain[w] = kx_chain(R, C, w);
      // the pair's strips start kKxLag rows after one another
      if (chain[w] != R + kKxLag * (C / kx_width(w))) ++failed;
    }
    return kx_choose(mode, false, chain, strips, 152);
  };
  struct Pair {
    int64_t m, n;
    int tile;
  };
  // cycles of one pair at K = 4 / 12 (94 and 155 a row): 700 x 40,000 1.75e6 / 1.04e6,
  // 2,000 x 40,000 1.87e6 / 1.24e6; 20,000 x 20,000 2.7e6 / 3.6e6
  for (const Pair &p : {Pair{700, 40000, kKx12}, {40000, 700, kKx12}, {2000, 40000, kKx12}, {20000, 20000, kKx4}}) {
    const int tile = tile_of(1, p.m, p.n, 1);
    if (tile != p.tile) {
      std::printf("failed: %lld x %lld takes tile %d, not %d\n", (long long)p.m, (long long)p.n, tile, p.tile);
      ++failed;
    }
  }
  return failed != 0;
}
