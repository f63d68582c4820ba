// ga_reads.cuh -- a small batch of short pairs in one launch (alphabets of <= 4
// symbols, sigma_max + alpha <= kKxMaxStep): a warp per pair validates it,
// classifies it and computes it as one strip (ga_strip.cuh).
//
// Why.  A batch of a thousand reads is 2e7 cells, 2 us of the chip's ALU rate;
// through the planned path it is a dozen small kernels (packing, validation,
// keys, a counting sort), three host round trips and one launch per tile width,
// each with a few warps.  A plan's graph of the same batch holds 40 kernels.  Here
// nothing is packed or sorted, and the rows of a pair are the latency of a lone
// strip: 1,000 pairs of 150 x 150 in one call 135 -> 58 us, 1,000 pairs of 100..300
// in a plan's graph 560 -> 44 us (GB300, the call and the wait for it).  Larger batches go the planned way, whose tiles pad less and hold two
// pairs a lane (the limits stand beside the two callers).
//
// Strips of 256, 512 or 768 columns (K = 4, 8, 12) by the longer sequence, with
// the one-op column chain: a batch leaves a scheduler one to four warps.  Pairs
// longer than 768 residues are only counted: the caller plans those alone; a plan
// whose capacity admits one never comes here.
#pragma once

#include "ga_strip.cuh"

namespace ga {

constexpr int kKrMaxLen = 768;
constexpr int kKrWarps = 4;

struct KRParams {
  const uint8_t *q_codes, *t_codes;
  const int64_t *q_off, *t_off;
  int32_t npairs;
  int32_t plan;         // offsets and lengths checked as a plan checks them
  int64_t cap;          // plan: residues at or beyond this position are not read
  int32_t max_len;      // plan: longest sequence
  uint32_t tables[16];  // table words as in KAParams
  int32_t A, alpha, beta;
  int32_t *scores;
  int32_t *status;
  unsigned long long *cells;
  int32_t *computed;    // pairs computed here
  int32_t *left;        // pairs longer than kKrMaxLen
  int64_t *ends;        // q_off[0], q_off[npairs], t_off[0], t_off[npairs]
};

// 0: sequence k is fine, 2: its offsets are not, 3: beyond the plan's capacity
// (validate_kernel and plan_validate_kernel in ga_prep.cuh).
__device__ __forceinline__ int kr_check(const KRParams &p, const int64_t *off, int64_t s, int64_t e) {
  const int64_t first = off[0], last = off[p.npairs];
  if (p.plan) {
    if (first < 0 || s < first || e < s || e > last) return 2;
    return (e > p.cap || e - s > p.max_len) ? 3 : 0;
  }
  const int64_t total = last > 0 ? last : 0;
  const int64_t start = first > 0 ? (first < total ? first : total) : 0;
  return (s < start || e < s || e > total) ? 2 : 0;
}

template <int MODE>
__global__ void __launch_bounds__(32 * kKrWarps, 4) kr_kernel(const __grid_constant__ KRParams p) {
  __shared__ uint2 ring_s[kKrWarps][kKxRing + 34];
  __shared__ uint32_t in_s[kKrWarps][33];
  const int warp = threadIdx.x >> 5, t = threadIdx.x & 31;
  const int pid = blockIdx.x * kKrWarps + warp;
  if (pid >= p.npairs) return;
  if (pid == 0 && t == 0) {
    p.ends[0] = p.q_off[0];
    p.ends[1] = p.q_off[p.npairs];
    p.ends[2] = p.t_off[0];
    p.ends[3] = p.t_off[p.npairs];
  }
  const int64_t qs = p.q_off[pid], qe = p.q_off[pid + 1], ts = p.t_off[pid], te = p.t_off[pid + 1];
  const int qb = kr_check(p, p.q_off, qs, qe), tb = kr_check(p, p.t_off, ts, te);
  int status = GA_OK, val = 0;
  if (qb || tb) {
    status = (qb == 2 || tb == 2) ? GA_ERR_ARG : GA_ERR_RANGE;
  } else if (::max(qe - qs, te - ts) > kKrMaxLen) {
    if (t == 0) atomicAdd(p.left, 1);
    return;
  } else {
    const int m = (int)(qe - qs), n = (int)(te - ts);
    if (m == 0 || n == 0) {
      // the closed form, and the other sequence's codes are still checked
      int bad = 0;
      for (int i = t; i < m; i += 32) bad |= p.q_codes[qs + i] >= p.A;
      for (int i = t; i < n; i += 32) bad |= p.t_codes[ts + i] >= p.A;
      if (__any_sync(0xffffffffu, bad)) status = GA_ERR_RESIDUE;
      val = MODE == kModeGlobal && m + n > 0 ? -(p.alpha + p.beta * (m + n - 1)) : 0;
    } else {
      KXView v;
      v.sw = m > n;
      v.R = v.sw ? n : m;
      v.C = v.sw ? m : n;
      v.row = v.sw ? p.t_codes + ts : p.q_codes + qs;
      v.col = v.sw ? p.q_codes + qs : p.t_codes + ts;
      v.nstrips = 1;
      v.A = p.A;
      v.alpha = p.alpha;
      v.beta = p.beta;
      v.edges = nullptr;
      const uint32_t *tab = p.tables + (v.sw ? 8 : 0);
      constexpr bool kFc = MODE != kModeSemi;
      uint2 *ring = ring_s[warp];
      uint32_t *in = in_s[warp];
      if (v.C <= 256)
        val = kx_strip<MODE, 4, kFc, false, 1>(v, 0, t, ring, in, ring, nullptr, nullptr, tab, status, KXNoHook{});
      else if (v.C <= 512)
        val = kx_strip<MODE, 8, kFc, false, 1>(v, 0, t, ring, in, ring, nullptr, nullptr, tab, status, KXNoHook{});
      else
        val = kx_strip<MODE, 12, kFc, false, 1>(v, 0, t, ring, in, ring, nullptr, nullptr, tab, status, KXNoHook{});
      if (t == 0 && !status) {  // (as planning counts: pairs without an invalid code)
        atomicAdd(p.cells, (unsigned long long)m * (unsigned long long)n);
        atomicAdd(p.computed, 1);
      }
    }
  }
  if (t == 0) {
    p.scores[pid] = status ? INT32_MIN : val;
    if (status) set_status(p.status, status);
  }
}

}  // namespace ga
