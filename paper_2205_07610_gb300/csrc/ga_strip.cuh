// ga_strip.cuh -- strips of long pairs as tasks: one warp computes one strip of
// 64 K columns of one pair, the strips of a pair run on different warps at the
// same time, each about a hundred rows behind its left neighbour.
//
// Cells are packed int16x2 relative to a per-lane, per-half int32 base as in
// ga_longpk.cuh (the left 32 K columns of the strip in the low halves, the
// right 32 K columns, 32 rows behind, in the high halves).  Rows are the
// shorter sequence, so a pair has as many strips and as few rows as possible.
//
// What bounds the row step, and why the loop looks as it does.  One row of a
// lane's K packed columns is 4 ALU + 2 FMA operations a column (one more each
// with the one-op column chain), and the ALU pipe takes one of a warp's
// instructions every two cycles.  A launch that leaves a scheduler one warp is
// bound by the latency of the row step instead.  So the loop has no checks and
// no branches: rows before the first and past the last one are ordinary rows
// with a table word that leaves the state alone (virtual rows, below), lane 0's
// left input is joined by a byte permute whose selector is lane-dependent, the
// left edge comes as one packed word per row, relative to lane 0's base, and the
// loads of the next row are issued a row ahead.
//   Lone warp, cycles a row (GB300): 90 at K = 4, 115 at K = 8, 155 at 12, 220 at
// 16, 265 at 20, against 440 at K = 8 for the strips that publish their edges
// through a fence and a counter: one 20k x 20k pair 6.1 -> 1.4 ms.  48 pairs of
// 5k..20k residues 62 -> 3.0 ms (48 warps before).  Full chip, K = 16 without the
// chain: 71 ALU instructions a row at 78 % of the ALU pipe, 11.3 cycles a packed
// column; 2,000 pairs of 1k..20k 106 -> 42 ms (one warp per pair before, so the
// longest pair set the time).  Protein pairs (10,000 of about 360 residues): 5.5
// -> 0.9 ms against the int32 kernel whose profile was built byte by byte.
//   The register limit matters: without a stated minimum of one block per SM
// ptxas holds the loop to 128 registers and a lone K = 4 step takes 125 cycles;
// more resident blocks at fewer registers were slower throughout (2,000 pairs:
// 41 ms at 3 blocks per SM, 43 at 4, 47 at 5).
//
// Virtual rows.  A lane-half before its first row sees sigma = 0 (local, semi-
// global: row 0 is all 0) or sigma = -beta (global: H(0, j) = H(0, j - 1) -
// beta for every column but the first, which belongs to lane 0 of strip 0 and
// has no virtual rows): E(1, j) = H(0, j) - alpha and H(0, j) reproduce
// themselves and no F exceeds H(0, j), because alpha >= beta.  Past its last
// row a lane-half runs pad rows (sigma = 0) that no result reads and that never
// exceed the largest real cell.  The loop ends when the last real column has
// run its last row, so global mode's H(R, C) is what its owner holds then.
//
// Last column of semi-global mode: see ga_longpk.cuh.
//
// Edges.  The right edge of a strip (H and the outgoing F per row) goes to the
// next strip through one 8-byte word per row in global memory: H (32 bits),
// H - F (16 bits; alpha >= H - F >= beta), and the number of the strip that
// wrote it (16 bits).  A word is written and read whole, so its tag says that
// it is valid and neither side needs a fence or a progress counter (a fence
// every 32 rows stood in the way of the next rows).  All strips of a pair share
// one buffer: strip s reads row r before it overwrites it for strip s + 1.
//
// Order.  Tasks are claimed from one list in which every strip of a pair comes
// after its left neighbour, so the strip that a warp waits for was claimed
// before by a running warp, whatever blocks are resident.  Every wait is
// bounded by globaltimer; one that runs out marks the pair GA_ERR_TIMEOUT.
//
// Substitution scores: alphabets of <= 4 symbols as in ga_inter.cuh (a selector
// per column, a table word per row), larger ones from a profile of the strip in
// shared memory, P[c][x] = sigma(row residue c, column x) as int8.
#pragma once

#include "ga_dp.cuh"
#include "ga_kx.h"
#include "ga_longpk.cuh"

namespace ga {

constexpr int kKxWarps = 4;
constexpr int kKxMaxStep = 128;       // largest sigma_max + alpha (relative int16 cells)
constexpr int kKxRing = 64;           // row entries (+ a mirror of the first 34)
constexpr int kKxSigRow = 9;          // words of a score vector in shared memory (32 bytes, odd stride)
constexpr int64_t kKxWaitNs = 10ll * 1000 * 1000 * 1000;

struct KXPairState {  // one per pair, zeroed before the launch
  int32_t score, done, status, nstrips;  // nstrips: set by the task list
};

struct KXParams {
  const uint8_t *q_codes, *t_codes;
  const int64_t *q_off, *t_off;  // null: one pair of m x n residues, task = strip
  int32_t m, n;
  const int32_t *sorted;         // pair ids; list entry i is sorted[range[0] + i]
  const int32_t *range;
  const int2 *tasks;             // (list entry, strip)
  int32_t ntasks;
  const int32_t *ntasks_dev;     // the count on the device instead (nullable)
  const int64_t *edge_off;       // per list entry: its first edge word
  unsigned long long *edges;     // zeroed before the launch
  KXPairState *state;            // per list entry
  int32_t *counter;
  int32_t *scores;
  int32_t *status;               // nullable
  int64_t nt, q0;                // cross chunk: pair p = (q0 + p/nt, p%nt); batch: nt = 0
  uint32_t tables[16];           // table words as in KAParams
  int8_t sigma[32 * 32];         // A*A row-major sigma(query, target)
  int32_t A, alpha, beta;
};

__device__ __forceinline__ unsigned long long kx_ld(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void kx_st(unsigned long long *p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

template <int K>
struct StripState {
  uint32_t H[K], E[K];
  uint32_t Hdiag, Hleft, Fin;
  uint32_t D;     // base difference to the left neighbour, added to what it sends
  uint32_t Z;     // local: the zero of Eq. H relative to the bases
  uint32_t best;  // local: running maximum, relative
};

// Row update.  FC: a one-op chain across the columns (local and global mode,
// where every column's gap open alpha >= beta).  With X(j) = max(Hdiag + sigma, E
// [, Z in local mode]) the H of a column is max(X(j), F(j)), and since F(j) -
// alpha <= F(j) - beta the gap entering the next column is F(j+1) = max(F(j) -
// beta, X(j) - alpha): it no longer waits for H(j).  One more ALU and one more FMA
// operation per packed column, for a chain of one operation per column instead of
// three.
template <int MODE, int K, bool FC, class SigFn, class NaFn>
__device__ __forceinline__ uint32_t strip_row(StripState<K> &s, uint32_t NB, uint32_t NAc, SigFn SIG, NaFn NA) {
  static_assert(!FC || MODE != kModeSemi, "semi-global frees the last column's gap open");
#pragma unroll
  for (int j = K - 1; j >= 1; --j) s.H[j] = __vadd2(s.H[j - 1], SIG(j));
  s.H[0] = __vadd2(s.Hdiag, SIG(0));
  uint32_t F = s.Fin;
#pragma unroll
  for (int j = 0; j < K; ++j) {
    if constexpr (FC) {
      const uint32_t X = MODE == kModeLocal ? __vimax3_s16x2(s.H[j], s.E[j], s.Z) : __vmaxs2(s.H[j], s.E[j]);
      const uint32_t Fj = F;
      F = __viaddmax_s16x2(F, NB, __vadd2(X, NAc));
      s.H[j] = __vmaxs2(X, Fj);
      s.E[j] = __viaddmax_s16x2(s.E[j], NB, __vadd2(s.H[j], NAc));
    } else {
      s.H[j] = __vimax3_s16x2(s.H[j], s.E[j], F);
      const uint32_t A = __vadd2(s.H[j], NA(j));
      if constexpr (MODE == kModeLocal) s.E[j] = __vimax3_s16x2(__vadd2(s.E[j], NB), A, s.Z);
      else s.E[j] = __viaddmax_s16x2(s.E[j], NB, A);
      F = __viaddmax_s16x2(F, NB, A);
    }
    if constexpr (MODE == kModeLocal) {
      if ((j & 1) == 1) s.best = __vimax3_s16x2(s.best, s.H[j - 1], s.H[j]);
      else if (j == K - 1) s.best = __vmaxs2(s.best, s.H[j]);
    }
  }
  return F;
}

// Profile bytes of a lane's K columns in one half: word q of lane t at word
// 32 q + t of the row's half, so a warp's loads hit 32 consecutive words when
// its lanes are on one row.
template <int K>
constexpr int kx_prof_row = 64 * K;  // bytes of a profile row: low half, then high half

// One pair as the strip function sees it: rows and columns, the scoring, the
// edge words of rows 0 .. R.
struct KXView {
  const uint8_t *row, *col;
  int R, C, sw, nstrips;
  int A, alpha, beta;
  unsigned long long *edges;
};

struct KXNoHook {
  __device__ __forceinline__ void operator()(int) const {}
};

// Strip s of a pair; returns its contribution to the score (local: best H; semi-
// global: max of row R; global: H(R, C) in the last strip).  tables: the table
// words of the 4 row codes (no profile); sig: the score vectors of the column
// residues, SIGW words apart (profile).  on_rows(n) is called when rows 1 .. n of
// the right edge have been written.
template <int MODE, int K, bool FC, bool PROF, int SIGW, class OnRows>
__device__ __forceinline__ int kx_strip(const KXView &v, int s, int t, uint2 *ring, uint32_t *in, uint2 *out,
                                        uint8_t *prof, const uint32_t *sig, const uint32_t *tables, int &status,
                                        OnRows on_rows) {
  constexpr int WH = 32 * K, W = 64 * K, NQ = K / 4;
  constexpr unsigned FULL = 0xffffffffu;
  static_assert(K % 4 == 0, "profile words");
  static_assert(kKxMaxStep * (kKwRenorm + 2 * K + 8) < 32000 - 256, "relative int16 cells of this tile width");
  const int R = v.R, C = v.C, A = v.A, alpha = v.alpha, beta = v.beta;
  const int col0 = s * W, ncol = ::min(W, C - col0);
  const bool edge_out = s + 1 < v.nstrips;
  const uint32_t NB = pk16(-beta, -beta), NAc = pk16(-alpha, -alpha);
  const uint32_t NEGV = pk16(kNeg16, kNeg16);
  auto h0 = [&](int c) -> int { return (MODE == kModeGlobal && c > 0) ? -alpha - beta * (c - 1) : 0; };
  int bad = 0;  // a residue code >= A

  // (codes are read past L1: the server's buffers are refilled while its kernel
  // runs)
  // ---- columns: selectors, or the strip's profile ---------------------------
  uint32_t sel[PROF ? 1 : K];
  uint32_t na[MODE == kModeSemi ? K : 1];
  StripState<K> st;
  int b[2] = {h0(col0 + t * K + 1), h0(col0 + WH + t * K + 1)};
#pragma unroll
  for (int j = 0; j < K; ++j) {
    const int c0 = t * K + j, c1 = c0 + WH;
    if constexpr (!PROF) {
      const int x0 = c0 < ncol ? (int)__ldcg(v.col + col0 + c0) : -1, x1 = c1 < ncol ? (int)__ldcg(v.col + col0 + c1) : -1;
      bad |= (x0 >= A) | (x1 >= A);
      // pad columns replicate a table byte's sign: sigma in {0, -1}
      const uint32_t n0 = x0 >= 0 ? (uint32_t)(x0 & 3) : 8u, n0s = x0 >= 0 ? (uint32_t)((x0 & 3) + 8) : 8u;
      const uint32_t n1 = x1 >= 0 ? (uint32_t)((x1 & 3) + 4) : 12u, n1s = x1 >= 0 ? (uint32_t)((x1 & 3) + 12) : 12u;
      sel[j] = n0 | (n0s << 4) | (n1 << 8) | (n1s << 12);
    }
    if constexpr (MODE == kModeSemi) na[j] = pk16(col0 + c0 == C - 1 ? 0 : -alpha, col0 + c1 == C - 1 ? 0 : -alpha);
    const int hv = (MODE == kModeGlobal) ? -beta * j : 0;  // H(0, first + j) - b
    const int ev = (MODE == kModeLocal) ? 0 : hv - alpha;  // local: E' = max(E, 0)
    st.H[j] = pk16(hv, hv);
    st.E[j] = pk16(ev, ev);
  }
  if constexpr (PROF) {
    // 4 columns x 4 row residues at a time: the columns' score vectors over
    // the row residue (a row of sig) transposed by byte permutes; row A serves
    // virtual and pad rows, pad columns (the zero row A of sig) are 0.
    const uint32_t rowA = (MODE == kModeGlobal) ? 0x01010101u * (uint32_t)(uint8_t)(-beta) : 0u;
    uint32_t *pw = reinterpret_cast<uint32_t *>(prof);
#pragma unroll 1
    for (int q = 0; q < 2 * NQ; ++q) {
      const int cb = (q / NQ) * WH + t * K + 4 * (q % NQ);
      const uint32_t *sg[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int x = cb + i < ncol ? (int)__ldcg(v.col + col0 + cb + i) : A;
        bad |= cb + i < ncol && x >= A;
        sg[i] = sig + ::min(x, A) * SIGW;
      }
      uint32_t *dst = pw + (q / NQ) * (WH / 4) + (q % NQ) * 32 + t;
#pragma unroll 1
      for (int c = 0; c < A; c += 4) {
        const uint32_t a0 = sg[0][c >> 2], a1 = sg[1][c >> 2], a2 = sg[2][c >> 2], a3 = sg[3][c >> 2];
        const uint32_t l01 = prmt(a0, a1, 0x5140u), l23 = prmt(a2, a3, 0x5140u);
        const uint32_t h01 = prmt(a0, a1, 0x7362u), h23 = prmt(a2, a3, 0x7362u);
        dst[c * (W / 4)] = prmt(l01, l23, 0x5410u);
        if (c + 1 < A) dst[(c + 1) * (W / 4)] = prmt(l01, l23, 0x7632u);
        if (c + 2 < A) dst[(c + 2) * (W / 4)] = prmt(h01, h23, 0x5410u);
        if (c + 3 < A) dst[(c + 3) * (W / 4)] = prmt(h01, h23, 0x7632u);
      }
      dst[A * (W / 4)] = rowA;
    }
  }
  st.Z = 0;
  st.best = 0;
  st.D = pk16(t == 0 ? 0 : h0(col0 + t * K + 1 - K) - b[0], h0(col0 + WH + t * K + 1 - K) - b[1]);
  int best_abs = 0, rowmax = 0;

  // ---- rows: table words (or profile row offsets), 32 at a time -------------
  const uint32_t virt = PROF ? (uint32_t)(A * W)
                             : (MODE == kModeGlobal) ? 0x01010101u * (uint32_t)(uint8_t)(-beta) : 0u;
  auto read_code = [&](int bb) -> int {  // row 32bb + 1 + t, -1 past the last
    const int r = 32 * bb + t;
    return r < R ? (int)__ldcg(v.row + r) : -1;
  };
  auto row_word = [&](int c) -> uint32_t {
    if constexpr (PROF) {
      bad |= c >= A;
      return (uint32_t)((c < 0 || c >= A) ? A : c) * (uint32_t)W;
    } else {
      bad |= c >= A;
      return c < 0 ? 0u : tables[c & 3];
    }
  };
  auto put_row = [&](int x, uint32_t lo, uint32_t hi) {
    ring[x] = make_uint2(lo, hi);
    if (x < 34) ring[x + kKxRing] = make_uint2(lo, hi);
  };
  put_row((-t) & (kKxRing - 1), virt, virt);  // rows 0 .. -31 of both halves
  uint32_t prev_word = virt;                  // the row words 32 rows back
  int next_code = read_code(0);

  // ---- the left edge ---------------------------------------------------------
  bool gave_up = false;
  const unsigned long long tag = (unsigned long long)s << 48;  // written by strip s - 1
  auto ready = [&](unsigned long long e) { return (e & 0xffff000000000000ull) == tag; };
  // entry of row r for every lane that has one, after waiting for it
  auto wait_edge = [&](int r, unsigned long long e) -> unsigned long long {
    const bool need = r <= R;
    if (__all_sync(FULL, !need || ready(e)) || gave_up) return e;
    uint64_t t0 = 0;
    for (unsigned spin = 0;; ++spin) {
      if (need && !ready(e)) e = kx_ld(v.edges + r);
      if (__all_sync(FULL, !need || ready(e))) return e;
      if ((spin & 15) == 15) {
        const uint64_t now = __shfl_sync(FULL, sv_now(), 0);
        if (t0 == 0) t0 = now;
        else if (now - t0 > (uint64_t)kKxWaitNs) {
          gave_up = true;
          return e;
        }
        __nanosleep(64);
      }
    }
  };
  auto edge_abs = [&](unsigned long long e, int &h, int &f) {
    h = (int)(uint32_t)e;
    f = h - (int)((e >> 32) & 0xffffu);
  };
  const int h00 = h0(col0 + t * K) - b[0], h01 = h0(col0 + WH + t * K) - b[1];
  st.Hdiag = pk16(h00, h01);
  st.Hleft = st.Hdiag;
  st.Fin = NEGV;
  unsigned long long edge = 0;  // rows 2 .. 33, then 32 more a batch
  {
    int h = 0, f = 0;
    if (s == 0) {
      h = (MODE == kModeGlobal) ? -alpha : 0;
      f = h - alpha;
    } else {
      edge_abs(wait_edge(1, 0), h, f);
      if (2 + t <= R) edge = kx_ld(v.edges + 2 + t);
    }
    if (t == 0) {
      st.Hleft = pk16(h - b[0], h01);
      st.Fin = pk16(f - b[0], kNeg16);
    }
  }

  // left inputs: what the left lane sends; for lane 0 the left edge (H | F << 16)
  // in the low half and lane 31's low half in the high half
  const uint32_t sel_h = t == 0 ? 0x5410u : 0x7654u, sel_f = t == 0 ? 0x5432u : 0x7654u;
  const int left = (t + 31) & 31;
  const bool keep_out = t == 31 && edge_out;
  const uint8_t *plo = prof + 4 * t, *phi = prof + WH + 4 * t;
  const int nit = R + (ncol + K - 1) / K - 1;

  auto flush = [&](int it0) {  // lane 31's high-half rows of the batch before it0
    const int b31 = __shfl_sync(FULL, b[1], 31);
    const int r = it0 - 94 + t;
    if (r >= 1 && r <= R) {
      const uint2 o = out[t];
      const int h = hi16(o.x);
      kx_st(v.edges + r, (unsigned long long)(uint32_t)(h + b31) |
                             ((unsigned long long)(uint32_t)(h - hi16(o.y)) << 32) |
                             ((unsigned long long)(s + 1) << 48));
    }
  };

  for (int it0 = 0; it0 < nit; it0 += 32) {
    __syncwarp();
    if (edge_out) {
      flush(it0);
      on_rows(it0 - 63);
    }
    if ((it0 & (kKwRenorm - 1)) == 0 && it0 > 0) {
      if constexpr (MODE == kModeSemi)
        if (!edge_out) rowmax = pk_drop_free_end<K>(st.H, st.E, st.Hdiag, NAc, ncol - 1 - t * K, WH, b, rowmax);
      // move each half's base to its current H of the first column
      const int d0 = lo16(st.H[0]), d1 = hi16(st.H[0]);
      if constexpr (MODE == kModeLocal) {
        best_abs = ::max(best_abs, ::max(lo16(st.best) + b[0], hi16(st.best) + b[1]));
        st.best = NEGV;
      }
      b[0] += d0;
      b[1] += d1;
      const uint32_t dl = pk16(-d0, -d1);
#pragma unroll
      for (int j = 0; j < K; ++j) {
        st.H[j] = __vadd2(st.H[j], dl);
        st.E[j] = __vadd2(st.E[j], dl);
      }
      // (the left inputs can be -inf, past the last row of the left edge)
      const uint32_t dp = pk16(d0, d1);
      st.Hdiag = __vmaxs2(__vsubss2(st.Hdiag, dp), NEGV);
      st.Hleft = __vmaxs2(__vsubss2(st.Hleft, dp), NEGV);
      st.Fin = __vmaxs2(__vsubss2(st.Fin, dp), NEGV);
      if constexpr (MODE == kModeLocal) {  // the zero of Eq. H under the new bases
        st.Z = pk16(::max(-b[0], kNeg16), ::max(-b[1], kNeg16));
#pragma unroll
        for (int j = 0; j < K; ++j) st.E[j] = __vmaxs2(st.E[j], st.Z);
      }
      const int nb0 = __shfl_sync(FULL, b[0], left), nb1 = __shfl_sync(FULL, b[1], left);
      st.D = t == 0 ? pk16(0, nb0 - b[1]) : pk16(nb0 - b[0], nb1 - b[1]);
    }
    // lane 0's left inputs of this batch, rows it0 + 2 .. it0 + 33
    {
      const int r = it0 + 2 + t, b0 = __shfl_sync(FULL, b[0], 0);
      int h, f;
      if (s == 0) {
        h = (MODE == kModeGlobal) ? -alpha - beta * (r - 1) : 0;
        f = h - alpha;
      } else {
        edge = wait_edge(r, edge);
        edge_abs(edge, h, f);
        if (r + 32 <= R) edge = kx_ld(v.edges + r + 32);
      }
      in[t] = r <= R ? pk16(h - b0, f - b0) : NEGV;
    }
    {
      const uint32_t w = row_word(next_code);
      put_row((it0 + 1 + t) & (kKxRing - 1), w, prev_word);
      prev_word = w;
      next_code = read_code(it0 / 32 + 1);
    }
    __syncwarp();
    const uint2 *rp = ring + ((it0 - t + 1) & (kKxRing - 1));
    // n row steps.  EVENT (semi-global, the iterations in which some lane-half is
    // at row R): the row's maximum is taken there.
    auto rows = [&](int n, auto event_tag) {
      constexpr bool EVENT = decltype(event_tag)::value;
      uint2 w = rp[0];
      uint32_t lw = in[0];
      uint32_t gl[PROF ? NQ : 1], gh[PROF ? NQ : 1];
      auto load_prof = [&](uint2 o) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          gl[q] = *reinterpret_cast<const uint32_t *>(plo + o.x + 128 * q);
          gh[q] = *reinterpret_cast<const uint32_t *>(phi + o.y + 128 * q);
        }
      };
      if constexpr (PROF) {
        load_prof(w);
        w = rp[1];
      }
#pragma unroll 2
      for (int k = 0; k < n; ++k) {
        const uint32_t lnext = in[k + 1];
        uint32_t F;
        auto na_of = [&](int j) -> uint32_t {
          if constexpr (MODE == kModeSemi) return na[j];
          else return NAc;
        };
        if constexpr (PROF) {
          uint32_t cl[NQ], ch[NQ];
#pragma unroll
          for (int q = 0; q < NQ; ++q) {
            cl[q] = gl[q];
            ch[q] = gh[q];
          }
          load_prof(w);  // the next row's profile words, the row after's offsets
          w = rp[k + 2];
          F = strip_row<MODE, K, FC>(
              st, NB, NAc, [&](int j) -> uint32_t { return prmt(cl[j >> 2], ch[j >> 2], sext_sel<CellS16x2>(j & 3)); },
              na_of);
        } else {
          const uint2 wn = rp[k + 1];
          F = strip_row<MODE, K, FC>(
              st, NB, NAc, [&](int j) -> uint32_t { return prmt(w.x, w.y, sel[j]); }, na_of);
          w = wn;
        }
        const uint32_t H = st.H[K - 1];
        if constexpr (EVENT) {
          const int rlo = it0 + k - t + 1, rhi = rlo - 32;
          if (rlo == R || rhi == R) {
            uint32_t mx = st.H[0];
#pragma unroll
            for (int j = 1; j < K; ++j) mx = __vmaxs2(mx, st.H[j]);
            rowmax = ::max(rowmax, rhi == R ? hi16(mx) + b[1] : lo16(mx) + b[0]);
          }
        }
        if (keep_out) out[k] = make_uint2(H, F);
        st.Hdiag = st.Hleft;
        const uint32_t hs = __shfl_sync(FULL, H, left), fs = __shfl_sync(FULL, F, left);
        st.Hleft = __vadd2(prmt(lw, hs, sel_h), st.D);
        st.Fin = __vadd2(prmt(lw, fs, sel_f), st.D);
        lw = lnext;
      }
    };
    const int n = ::min(32, nit - it0);
    if (MODE == kModeSemi && it0 + 32 >= R) rows(n, std::true_type{});
    else rows(n, std::false_type{});
  }
  __syncwarp();
  if (edge_out) {  // rows of the last two batches (nit = R + 63: rows up to R)
    const int last0 = ((nit + 31) / 32) * 32;
    flush(last0);
    on_rows(R);
  }
  if (__any_sync(FULL, bad)) status = GA_ERR_RESIDUE;
  if (gave_up) status = GA_ERR_TIMEOUT;
  if constexpr (MODE == kModeLocal) {
    best_abs = ::max(best_abs, ::max(lo16(st.best) + b[0], hi16(st.best) + b[1]));
    return group_max<32>(best_abs);
  } else if constexpr (MODE == kModeSemi) {
    return group_max<32>(rowmax);
  } else {
    // the owner of column C ran row R last
    const int oc = ncol - 1, oh = oc >= WH ? 1 : 0, ol = (oc - oh * WH) / K, oj = (oc - oh * WH) % K;
    uint32_t g = st.H[0];
#pragma unroll
    for (int j = 1; j < K; ++j)
      if (j == oj) g = st.H[j];
    return __shfl_sync(FULL, oh ? hi16(g) + b[1] : lo16(g) + b[0], ol);
  }
}

template <int MODE, int K, bool FC, bool PROF>
__global__ void __launch_bounds__(32 * kKxWarps, 1) kx_kernel(const __grid_constant__ KXParams p) {
  extern __shared__ __align__(16) uint8_t kx_smem[];
  __shared__ uint2 ring_s[kKxWarps][kKxRing + 34];
  __shared__ uint32_t in_s[kKxWarps][33];
  __shared__ uint2 out_s[kKxWarps][32];
  const int warp = threadIdx.x >> 5, t = threadIdx.x & 31;
  uint8_t *prof = kx_smem + (size_t)warp * (size_t)(p.A + 1) * kx_prof_row<K>;
  // score vectors: row x of sig_s[sw] holds the scores of column residue x
  // against every row residue (sw: rows are the target); row A is 0
  __shared__ uint32_t sig_s[PROF ? 2 : 1][PROF ? 32 * kKxSigRow : 1];
  if constexpr (PROF) {
    for (int i = threadIdx.x; i < 2 * 32 * 32; i += blockDim.x) {
      const int sw = i >> 10, x = (i >> 5) & 31, c = i & 31;
      const int8_t g = (x < p.A && c < p.A) ? (sw ? p.sigma[x * p.A + c] : p.sigma[c * p.A + x]) : (int8_t)0;
      reinterpret_cast<int8_t *>(sig_s[sw])[x * 4 * kKxSigRow + c] = g;
    }
    __syncthreads();
  }
  const int ntasks = p.ntasks_dev ? *p.ntasks_dev : p.ntasks;
  for (;;) {
    int task = 0;
    if (t == 0) task = atomicAdd(p.counter, 1);
    task = __shfl_sync(0xffffffffu, task, 0);
    if (task >= ntasks) break;
    int li = 0, s = task, m = p.m, n = p.n, pid = 0;
    int64_t qs = 0, ts = 0, eo = 0;
    if (p.tasks) {
      const int2 tk = p.tasks[task];
      li = tk.x;
      s = tk.y;
      pid = p.sorted[p.range[0] + li];
      const int64_t qi = p.nt ? p.q0 + pid / p.nt : pid, ti = p.nt ? pid % p.nt : pid;
      qs = p.q_off[qi];
      ts = p.t_off[ti];
      m = (int)(p.q_off[qi + 1] - qs);
      n = (int)(p.t_off[ti + 1] - ts);
      eo = p.edge_off[li];
    }
    KXView v;
    v.sw = m > n;  // rows: the shorter sequence
    v.R = v.sw ? n : m;
    v.C = v.sw ? m : n;
    v.row = v.sw ? p.t_codes + ts : p.q_codes + qs;
    v.col = v.sw ? p.q_codes + qs : p.t_codes + ts;
    v.nstrips = (v.C + 64 * K - 1) / (64 * K);
    v.edges = p.edges + eo;
    v.A = p.A;
    v.alpha = p.alpha;
    v.beta = p.beta;
    int status = GA_OK;
    const int val = kx_strip<MODE, K, FC, PROF, kKxSigRow>(v, s, t, ring_s[warp], in_s[warp], out_s[warp], prof,
                                                           sig_s[PROF ? v.sw : 0], p.tables + (v.sw ? 8 : 0), status,
                                                           KXNoHook{});
    if (t == 0) {
      KXPairState *ps = p.state + li;
      bool finish = v.nstrips == 1;
      int score = val;
      if (!finish) {
        if (status) atomicCAS(&ps->status, 0, status);
        if (MODE == kModeGlobal) {
          if (s + 1 == v.nstrips) atomicExch(&ps->score, val);
        } else {
          atomicMax(&ps->score, val);
        }
        __threadfence();
        if (atomicAdd(&ps->done, 1) + 1 == v.nstrips) {
          __threadfence();
          finish = true;
          score = atomicAdd(&ps->score, 0);
          status = atomicAdd(&ps->status, 0);
        }
      }
      if (finish) {
        p.scores[pid] = status ? INT32_MIN : score;
        if (status && p.status) set_status(p.status, status);
      }
    }
    __syncwarp();
  }
}

}  // namespace ga
