// ga_bandfull.cuh -- band doubling decided by the exact score.
//
// For a pair whose exact global score S* is known, most attempts of the doubling
// need not be run.  The certificate accepts the half-width w when the score S(w)
// of its region reaches UB(w), the bound on every path that visits a diagonal
// outside the band (ga_banded.cuh).  S(w) <= S*, so S* < UB(w) rejects; and when
// S* > UB(w) no optimal path leaves the band, so S(w) = S* is accepted.  Only S* =
// UB(w) depends on whether an optimal path stays inside: that attempt is run.
//
// When the exact score is the cheaper way.  A band attempt runs on one warp, m +
// D (n / 1024) iterations of 400 cycles and more, and a wide one takes 30 ms
// (20,000 residues, w = 4,096); the strips of the full matrix (ga_strip.cuh) spread
// over the chip and take 1.4 ms for one such pair.  So a call whose full matrices
// fit the time of its first attempts runs them alone, and otherwise a pair that
// fails goes to the strips once its windows are long (the rules stand in BandRun,
// ga_api.cu).  GB300, pairs of 1k..20k from w = 1,024: 30 pairs 46 -> 1.7 ms, 300
// pairs 52 -> 9.5, 1,500 pairs 63 -> 31.
#pragma once

#include "ga_banded.cuh"

namespace ga {

struct BandVerdictParams {
  const int64_t *q_off, *t_off;
  const int32_t *list;       // pair ids; entries range[0] .. range[1] - 1
  const int32_t *range;
  const int32_t *w_next;     // per pair: the next half-width to decide; null: w0 / default_w0
  const int32_t *w0;
  int32_t default_w0;
  int32_t alpha, beta, sigma_max_pos;
  const int32_t *scores;     // exact scores (INT32_MIN: a wait ran out)
  int32_t *w_used;           // nullable
  unsigned long long *retries, *cells;
  int32_t *tie_list, *tie_count;  // pairs whose attempt has to be run,
  int32_t *tie_w;                 // and per pair its half-width
};

// A warp per pair: the doubling from the pair's width.  Counts what the attempts
// would have: rejected ones, and the region's cells of every attempt.
template <int K>
__global__ void band_verdict_kernel(const __grid_constant__ BandVerdictParams p) {
  const int t = threadIdx.x & 31;
  const int count = p.range[1] - p.range[0];
  for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < count; i += (gridDim.x * blockDim.x) >> 5) {
    const int pid = p.list[p.range[0] + i];
    const int m = (int)(p.q_off[pid + 1] - p.q_off[pid]), n = (int)(p.t_off[pid + 1] - p.t_off[pid]);
    const int dn = n - m, nb = (n + K - 1) / K;
    const int S = p.scores[pid];
    int w = p.w_next ? p.w_next[pid] : p.w0 ? p.w0[pid] : p.default_w0;
    if (w < 0) w = 0;
    unsigned long long cells = 0;
    unsigned tries = 0;
    if (S == INT32_MIN) {
      if (t == 0 && p.w_used) p.w_used[pid] = -1;
      continue;
    }
    for (;;) {
      const int64_t lo = (int64_t)(dn < 0 ? dn : 0) - w, hi = (int64_t)(dn > 0 ? dn : 0) + w;
      const bool covers = (lo <= -m) && (hi >= n);
      int64_t ub = INT64_MIN;
      if (lo - 1 >= -m) ub = ::max(ub, band_ub(m, n, p.sigma_max_pos, p.alpha, p.beta, lo - 1));
      if (hi + 1 <= n) ub = ::max(ub, band_ub(m, n, p.sigma_max_pos, p.alpha, p.beta, hi + 1));
      if (!covers && (int64_t)S == ub) {
        if (t == 0) {
          p.tie_list[atomicAdd(p.tie_count, 1)] = pid;
          p.tie_w[pid] = w;
        }
        break;
      }
      for (int b = t; b < nb; b += 32) {  // the region's cells: block b's rows times its columns
        const int64_t cb = (int64_t)K * b;
        const int64_t wlo = ::max((int64_t)1, cb + 1 - hi), whi = ::min((int64_t)m, cb + K - lo);
        cells += (unsigned long long)(whi - wlo + 1) * (unsigned long long)::min((int64_t)K, n - cb);
      }
      if (covers || (int64_t)S > ub) {
        if (t == 0 && p.w_used) p.w_used[pid] = w;
        break;
      }
      ++tries;
      w = (w == 0) ? 1 : 2 * w;
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) cells += __shfl_xor_sync(0xffffffffu, cells, o);
    if (t == 0) {
      if (tries) atomicAdd(p.retries, (unsigned long long)tries);
      if (cells) atomicAdd(p.cells, cells);
    }
  }
}

}  // namespace ga
