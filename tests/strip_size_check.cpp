// Size decisions of the strip launches (paper_2205_07610_gb300/csrc/ga_kx.h) on
// totals beyond 32 bits, run by tests/test_strip_sizes.py: a total that wrapped would
// pass for a small launch, and the task list would be written past its end.
// Exit status 0 on success; the first failure is printed.
#include "../paper_2205_07610_gb300/csrc/ga_kx.cu"

#include <cstdio>

using namespace ga;

int main() {
  int failed = 0;
  auto check = [&](bool ok, const char *what) {
    if (!ok && !failed++) std::printf("failed: %s\n", what);
  };
  struct Search {
    int64_t pairs, shorter, longer;
  };
  // one query of 200,000 residues against 11 million targets of 40 (wraps to 12.1
  // million strips of 256 columns); 2,048 queries of one residue against 2,048
  // targets of 262,144 (wraps to 0); one beyond the limit; the limit; ordinary sizes
  const Search cases[] = {{11000000, 40, 200000}, {1 << 22, 1, 262144}, {(1 << 20) + 1, 1, 262144},
                          {1 << 20, 1, 262144},   {1 << 20, 300, 360}};
  const bool fits4[] = {false, false, false, true, true};
  for (int k = 0; k < 5; ++k) {
    const Search &c = cases[k];
    LongSums s{};
    int64_t strips[kKxWidths], chain[kKxWidths];
    for (int w = 0; w < kKxWidths; ++w) {
      s.strips[w] += (unsigned long long)c.pairs * (unsigned long long)((c.longer + kx_width(w) - 1) / kx_width(w));
      strips[w] = (int64_t)s.strips[w];
      chain[w] = kx_chain(c.shorter, c.longer, w);
      check(strips[w] / c.pairs == (c.longer + kx_width(w) - 1) / kx_width(w), "strip totals are not cut off");
    }
    check(kx_fits(kKx4, c.longer, strips[0], c.pairs * (c.shorter + 1), (4ll << 30) / 8) == fits4[k],
          "a launch of 256-column strips");
    for (const bool profile : {false, true})
      for (int mode = 0; mode < 3; ++mode) {
        const int tile = kx_choose(mode, profile, chain, strips, 152);
        const int64_t n = strips[kKxTileK[tile] / 4 - 1];
        check(!kx_fits(tile, c.longer, n, 0, 1) || n <= kKxMaxTasks, "the chosen tile's tasks");
      }
  }
  check(!kx_fits(kKx4, 262145, 1025, 0, 1), "strips of one pair");
  check(!kx_fits(kKx4, 1000, 4, 2, 1), "edge words");
  return failed != 0;
}
