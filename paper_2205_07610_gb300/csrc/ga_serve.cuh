// ga_serve.cuh -- strip-task kernel: one warp computes one strip of 512
// columns of one pair; the strips of a pair run on different warps (and
// SMs) at the same time, each a few dozen rows behind its left neighbour.
//
// This is the paper's multi-stage partitioning of a long alignment (Sec. 3.1:
// submatrices of the target computed left to right) spread over warps
// instead of run by one thread group in sequence: the right edge of strip s
// (H and the outgoing F of its last column, per row) is written to global
// memory in batches of 32 rows and published through a per-strip progress
// counter (release); strip s+1 waits (acquire, bounded) until the rows it
// is about to read are published.  Rows are the shorter sequence, columns
// the longer one.
//
// Tasks come from two device-resident rings: strip 0 of each request from
// the producer's ring (host or init kernel), strip s+1 from a continuation
// ring that the warp running strip s fills once it has published the first
// kSvContRows edge rows, so the next strip rarely waits.  A warp claims a
// task only when an entry is there, continuations first, so a claim is always
// made by a running warp, and the producer of every edge a warp waits on (strip
// s of the same request) was claimed earlier by a warp that is running: the
// waits end without any assumption about which blocks are resident.  A claim
// decrements the ring's count of unclaimed entries and only then draws a ticket:
// a compare-and-swap of the ring head, with 2,400 warps polling it, let one claim
// through per microsecond (9,728 requests of 512 residues 8.6 ms).  While few
// entries wait, a warp whose scheduler already runs strips hangs back
// kSvShareNs for each of them, so that idle schedulers take the entries: the
// strips of a request move at the pace of the slowest (8 requests of 20k
// residues took 500 cycles a row with strips wherever a poll found them).
// Every wait is
// bounded (globaltimer): an edge wait that runs out marks the request
// GA_ERR_TIMEOUT and continues; a warp without work exits once no request
// is in flight and `stop` is set or it has idled for idle_ns, and in any
// case after wait_ns without a claimable task.
//
// A request completes when its last strip finishes: that warp writes the
// score to `out` (if set) and a completion record (id, score, status, seq)
// to the completion ring, seq last.
//
// Substitution scores come from a per-warp int8 profile of the strip in
// shared memory, P[c][x] = sigma(row residue c, column x), for any alphabet
// of <= 31 symbols (Sec. 3.1, "scoring profile").
//
// Cells.  A request whose scoring has sigma_max + alpha <= kKxMaxStep runs the
// packed strips of ga_strip.cuh (8 columns per lane and half, 512 a strip), its
// edges as their self-validating words in one buffer per request, zeroed by the
// warp of strip 0 before it queues strip 1.  Other scorings run the int32 strip
// (sv_strip) with one edge buffer per strip and progress counters.
//
// Alphabets of <= 4 symbols take their scores from column selectors, larger ones
// from the strip's profile.  No request runs the one-op column chain, although a
// lone strip's row takes 115 instead of 172 cycles with it: a service mixes modes
// and alphabets, and with ten row loops instead of six in flight the instruction
// caches thrash (4,000 mixed requests below 15k residues: 12.7 ms with both
// variants, 8.2 with the chain alone, 7.7 without it; one mode and alphabet: 7.1).
//
// Measured on GB300: a burst of 4,000 requests (median length 1,000, up to
// 50,000) 31 -> 19 ms against strips that published their edges through a fence
// and a counter every 32 rows and claimed tasks by compare-and-swap; 9,728
// requests of 512 residues 8.6 -> 0.8 ms; 8 requests of 40k residues 20 -> 8 ms.
#pragma once

#include "ga_dp.cuh"
#include "ga_strip.cuh"

namespace ga {

constexpr int kSvK = 16;
constexpr int kSvKp = 8;          // packed strips: 8 packed columns per lane and half
constexpr int kSvW = 32 * kSvK;  // columns per strip
constexpr int kSvWarps = 4;      // warps per block
constexpr int kSvMaxStrips = 128;
constexpr int kSvMaxLen = kSvMaxStrips * kSvW;  // longer sequence <= 65536
constexpr int kSvContRows = 96;  // edge rows published before the next strip is queued

struct SvScoring {
  int32_t A, alpha, beta;
  int32_t packed;         // 1: packed strips (sigma_max + alpha <= kKxMaxStep)
  int8_t sigma[32 * 32];  // sigma(query code, target code), A x A row-major
  // rows = query / rows = target: table words of the row codes (alphabets of <= 4
  // symbols), score vectors of the column residues over the row residue (row A: 0)
  uint32_t tables[2][4];
  int8_t vec[2][32][32];
};

struct SvRequest {
  const uint8_t *q;     // device codes
  const uint8_t *t;
  int2 *edges;          // int32 strips: (nstrips - 1) edges of R + 1 int2; packed ones share R + 1 words
  int32_t *out;         // nullable: the score is also stored here
  int64_t id;
  int32_t m, n;
  int32_t mode, scoring;
  int32_t nstrips;
  int32_t score;        // local / semi: max over strips (starts 0); global: from the last strip
  int32_t strips_done;
  int32_t status;
  int32_t pad[2];
  int32_t progress[kSvMaxStrips];  // rows of each strip's edge published
};

struct SvCompletion {
  int64_t id;
  int32_t score, status;
  int64_t seq;   // index + 1, written last
  int64_t slot;  // request slot (host bookkeeping)
};

// Counters shared by the warps, each on a line of its own.
struct SvCtl {
  struct Line64 {
    unsigned long long v, pad[15];
  };
  struct Line32 {
    int32_t v, pad[31];
  };
  Line64 head, tail;            // task ring: tickets drawn; entries published (by the producer)
  Line64 seen;                  // entries of the task ring already added to `ready`
  Line64 cont_head, cont_tail;  // continuation ring: tickets drawn, entries reserved
  Line32 ready, cont_ready;     // unclaimed entries of the two rings (transiently below zero)
  Line64 comp_count, admitted, completed;
  int32_t busy[1024];           // strips running per scheduler (SM id * 4 + warp of the block)
};
constexpr int kSvShareNs = 2000;
constexpr int kSvPlenty = 32;   // unclaimed entries beyond which nobody hangs back

struct SvParams {
  SvRequest *req;
  const SvScoring *scorings;
  const int2 *tasks;  // (slot, strip)
  int64_t task_cap;
  SvCtl *ctl;
  SvCompletion *comp;  // nullable
  int64_t comp_cap;
  const int32_t *stop;
  // continuation queue: strip s+1 of a request, pushed by the warp running
  // strip s once that strip has published kSvContRows edge rows (at most one
  // unclaimed continuation per request, so cont_cap >= requests in flight)
  int2 *cont;
  unsigned long long *cont_seq;  // entry i holds a task once cont_seq[i % cap] == i + 1
  int64_t cont_cap;
  int64_t idle_ns;
  int64_t wait_ns;
  int32_t prof_bytes;  // per warp: (max A + 1) * kSvW (real residues, one pad / virtual row)
};

__device__ __forceinline__ int sv_ld_acquire(const int32_t *p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long sv_ld_acquire64(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void sv_st_release(int32_t *p, int v) {
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void sv_st_release64(unsigned long long *p, unsigned long long v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ int sv_ld_sys(const int32_t *p) {
  int v;
  asm volatile("ld.relaxed.sys.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Bounded wait until *flag >= need (acquire): true once it is, false when
// limit_ns of globaltimer time pass first.  The poll backs off from 32 ns to
// 2 us of __nanosleep.
__device__ __forceinline__ bool sv_wait_at_least(const int32_t *flag, int need, uint64_t limit_ns) {
  if (sv_ld_acquire(flag) >= need) return true;
  const uint64_t t0 = sv_now();
  unsigned ns = 32;
  while (sv_ld_acquire(flag) < need) {
    if (sv_now() - t0 > limit_ns) return false;
    __nanosleep(ns);
    if (ns < 2048) ns *= 2;
  }
  return true;
}

// Queues a continuation (one lane).
__device__ __forceinline__ void sv_push(const SvParams &p, int slot, int strip) {
  const unsigned long long idx = atomicAdd(&p.ctl->cont_tail.v, 1ull);
  const int64_t e = (int64_t)(idx % (unsigned long long)p.cont_cap);
  p.cont[e] = make_int2(slot, strip);
  __threadfence();
  sv_st_release64(p.cont_seq + e, idx + 1);
  __threadfence();
  atomicAdd(&p.ctl->cont_ready.v, 1);
}

// Takes one unclaimed entry off a ring's count: true when there was one.  A
// ticket drawn after that is below the number of entries published.
__device__ __forceinline__ bool sv_take(int32_t *ready) {
  if (atomicSub(ready, 1) > 0) {
    __threadfence();
    return true;
  }
  atomicAdd(ready, 1);
  return false;
}

struct SvView {
  const uint8_t *rowraw, *colraw;
  int2 *edges;
  int R, C, sw, A, alpha, beta, nstrips, packed;
  const int8_t *sigma;
};

// One strip of one request; returns the strip's contribution to the score
// (local: best H; semi: max of row R; global: H(R, C) on the lane that owns
// column C, else INT_MIN).
template <int MODE>
__device__ int sv_strip(const SvParams &p, SvRequest *rq, int slot, const SvView &v, int s, int t,
                        uint8_t *prof, uint8_t *colc, int2 *in_ring, int2 *out_ring,
                        uint32_t *row_ring) {
  using Cell = CellS32;
  using T = int32_t;
  constexpr int K = kSvK, W = kSvW;
  constexpr int kNeg = kNeg32;
  const int R = v.R, C = v.C, A = v.A, alpha = v.alpha, beta = v.beta;
  const T NB = -beta;
  const int col0 = s * W;
  const int2 *edge_in = (s > 0) ? v.edges + (size_t)(s - 1) * (size_t)(R + 1) : nullptr;
  int2 *edge_out = (s + 1 < v.nstrips) ? v.edges + (size_t)s * (size_t)(R + 1) : nullptr;

  // ---- column codes and the strip's profile ---------------------------
  for (int x = t; x < W; x += 32) {
    const int col = col0 + x;
    int c = A;  // pad
    if (col < C) {
      c = __ldcg(v.colraw + col);
      if (c >= A) {
        atomicCAS(&rq->status, 0, GA_ERR_RESIDUE);
        c = A;
      }
    }
    colc[x] = (uint8_t)c;
  }
  __syncwarp();
  // rows c < A only: pad rows (beyond R) are never computed, pad columns
  // (beyond C) read 0 from their own entries
  for (int e = t; e < A * W; e += 32) {
    const int c = e / W, x = e - c * W;
    const int cc = colc[x];
    int val = 0;
    if (c < A && cc < A) val = v.sw ? v.sigma[cc * A + c] : v.sigma[c * A + cc];
    prof[e] = (uint8_t)(int8_t)val;
  }

  T na[MODE == kModeSemi ? K : 1];
  T H[K], E[K];
#pragma unroll
  for (int j = 0; j < K; ++j) {
    const int col = col0 + t * K + j;
    if constexpr (MODE == kModeSemi) na[j] = (col == C - 1) ? 0 : -alpha;
    H[j] = (MODE == kModeGlobal) ? ::max(-alpha - beta * col, kNeg) : 0;  // H(0, col+1)
    E[j] = ::max(H[j] - alpha, kNeg);
  }
  const int ocol = C - 1 - col0 - t * K;  // local index of column C, if in this tile
  T best = 0;
  int rowmax = 0, gscore = INT_MIN;

  auto left_row = [&](int r) -> int2 {  // (H(r, col0), F(r, col0+1))
    int2 lv;
    if (s == 0) {
      lv.x = (MODE == kModeGlobal) ? ((r == 0) ? 0 : ::max(-alpha - beta * (r - 1), kNeg)) : 0;
      lv.y = ::max(lv.x - alpha, kNeg);
    } else {
      lv = in_ring[(r - 1) & 63];
    }
    return lv;
  };
  // rows 32b+1 .. 32b+32 of the left edge -> in_ring, after waiting for them
  auto load_batch = [&](int b) {
    if (s == 0) return;
    const int need = ::min(R, 32 * b + 32);
    if (32 * b + 1 > R) return;
    const int32_t *pp = &rq->progress[s - 1];
    if (t == 0 && !sv_wait_at_least(pp, need, (uint64_t)p.wait_ns)) atomicCAS(&rq->status, 0, GA_ERR_TIMEOUT);
    __syncwarp();
    (void)sv_ld_acquire(pp);  // every lane orders its edge loads after the flag
    const int r = 32 * b + 1 + t;
    if (r <= R) in_ring[(r - 1) & 63] = __ldcg(edge_in + r);
  };
  auto fill_rows = [&](int b) {  // row codes, 4 batches of 32 in flight
    const int r = 32 * b + 1 + t;
    uint32_t c = (uint32_t)A;
    if (r <= R) {
      c = __ldcg(v.rowraw + r - 1);
      if (c >= (uint32_t)A) {  // reported; any in-range row keeps the profile read in bounds
        atomicCAS(&rq->status, 0, GA_ERR_RESIDUE);
        c = 0;
      }
    }
    row_ring[r & 127] = c;
  };
  bool queued = false;  // strip s+1 queued
  auto publish = [&](int rows) {  // edge rows 1..rows are in global memory
    __threadfence();
    __syncwarp();
    if (t == 0) {
      sv_st_release(&rq->progress[s], rows);
      if (!queued && rows >= ::min(R, kSvContRows)) sv_push(p, slot, s + 1);
    }
    queued = queued || rows >= ::min(R, kSvContRows);
  };

  load_batch(0);
  fill_rows(0);
  fill_rows(1);
  __syncwarp();

  const int h00 = (MODE == kModeGlobal && col0 > 0) ? ::max(-alpha - beta * (col0 - 1), kNeg) : 0;
  int hdt = 0;  // H(0, col0 + t*K)
  if constexpr (MODE == kModeGlobal)
    hdt = (col0 + t * K == 0) ? 0 : ::max(-alpha - beta * (col0 + t * K - 1), kNeg);
  const int2 l1 = left_row(1);
  T Hdiag = (t == 0) ? h00 : hdt;
  T Hleft = (t == 0) ? l1.x : hdt;
  T Fin = (t == 0) ? l1.y : kNeg;

  const int nit = R + 31;
  int flushed = 0;  // edge rows 1..flushed are in global memory
  for (int it = 0; it < nit; ++it) {
    if ((it & 31) == 0) {
      __syncwarp();
      load_batch(it / 32 + 1);
      fill_rows(it / 32 + 2);
      if (it >= 32 && edge_out) {  // lane 31's rows stored since the last flush: .. it-31
        const int r = flushed + 1 + t;
        if (r <= it - 31) edge_out[r] = out_ring[(r - 1) & 31];
        flushed = it - 31;
        publish(flushed);
      }
      __syncwarp();
    }
    const int r = it - t + 1;
    T Hout, Fout;
    if ((unsigned)(r - 1) < (unsigned)R) {
      const uint32_t rv = row_ring[r & 127];
      const uint4 *pr = reinterpret_cast<const uint4 *>(prof + (size_t)rv * W + t * K);
      const uint4 q4 = *pr;
      const uint32_t w[4] = {q4.x, q4.y, q4.z, q4.w};
      Fout = dp_row<Cell, MODE, K>(
          H, E, Hdiag, Fin, NB, best,
          [&](int j) -> T { return (T)prmt(w[j >> 2], 0u, sext_sel<Cell>(j & 3)); },
          [&](int j) -> T {
            if constexpr (MODE == kModeSemi) return na[j];
            else return -alpha;
          });
      Hout = H[K - 1];
      if (r == R) {
        if constexpr (MODE == kModeGlobal) {
          if (ocol >= 0 && ocol < K) {
            T g = H[0];
#pragma unroll
            for (int j = 1; j < K; ++j)
              if (j == ocol) g = H[j];
            gscore = g;
          }
        } else if constexpr (MODE == kModeSemi) {
#pragma unroll
          for (int j = 0; j < K; ++j) rowmax = ::max(rowmax, H[j]);
        }
      }
    } else {
      Hout = H[K - 1];
      Fout = kNeg;
    }
    if (t == 31 && r >= 1 && r <= R) out_ring[(r - 1) & 31] = make_int2(Hout, Fout);
    Hdiag = Hleft;
    Hleft = __shfl_up_sync(0xffffffffu, Hout, 1);
    Fin = __shfl_up_sync(0xffffffffu, Fout, 1);
    if (t == 0) {
      const int2 lv = (it + 2 <= R) ? left_row(it + 2) : make_int2(0, kNeg);
      Hleft = lv.x;
      Fin = lv.y;
    }
  }
  __syncwarp();
  if (edge_out) {  // remaining lane-31 rows, then the whole edge is published
    const int r = flushed + 1 + t;
    if (r <= R) edge_out[r] = out_ring[(r - 1) & 31];
    publish(R);
  }
  __syncwarp();
  if constexpr (MODE == kModeLocal) return group_max<32>(best);
  else if constexpr (MODE == kModeSemi) return group_max<32>(rowmax);
  else return __reduce_max_sync(0xffffffffu, gscore);
}

// One packed strip of one request: kx_strip, and the next strip queued once
// kSvContRows rows of the right edge are written.
template <int MODE, bool PROF>
__device__ __forceinline__ int sv_strip_pk(const SvParams &p, SvRequest *rq, int slot, const SvView &v,
                                           const SvScoring *sc, int s, int t, uint2 *ring, uint32_t *in, uint2 *out,
                                           uint8_t *prof) {
  KXView k;
  k.row = v.rowraw;
  k.col = v.colraw;
  k.R = v.R;
  k.C = v.C;
  k.sw = v.sw;
  k.nstrips = v.nstrips;
  k.A = v.A;
  k.alpha = v.alpha;
  k.beta = v.beta;
  k.edges = reinterpret_cast<unsigned long long *>(v.edges);
  if (s == 0 && k.nstrips > 1) {
    for (int r = t; r <= k.R; r += 32) k.edges[r] = 0;
    __syncwarp();
  }
  bool queued = false;
  auto on_rows = [&](int rows) {
    if (queued || rows < ::min(k.R, kSvContRows)) return;
    queued = true;
    __syncwarp();
    if (t == 0) sv_push(p, slot, s + 1);  // its fence also orders strip 0's zeroed edge words
  };
  int status = GA_OK;
  const int val = kx_strip<MODE, kSvKp, false, PROF, 8>(k, s, t, ring, in, out, prof,
                                                     reinterpret_cast<const uint32_t *>(sc->vec[v.sw]),
                                                     sc->tables[v.sw], status, on_rows);
  if (t == 0 && status) atomicCAS(&rq->status, 0, status);
  return val;
}

template <int MODE>
__device__ __forceinline__ int sv_packed(const SvParams &p, SvRequest *rq, int slot, const SvView &v, const SvScoring *sc, int s, int t,
                         uint2 *ring, uint32_t *in, uint2 *out, uint8_t *prof) {
  return v.A <= 4 ? sv_strip_pk<MODE, false>(p, rq, slot, v, sc, s, t, ring, in, out, prof)
                  : sv_strip_pk<MODE, true>(p, rq, slot, v, sc, s, t, ring, in, out, prof);
}

__global__ void __launch_bounds__(32 * kSvWarps, 4) ks_kernel(const __grid_constant__ SvParams p) {
  extern __shared__ __align__(16) uint8_t sv_smem[];
  // Static shared memory is kept small so that four blocks fit on an SM
  // with a 24-symbol profile: a strip's column codes are needed only while
  // its profile is built, before the left-edge ring is first written, so
  // the two share their bytes.
  __shared__ int2 in_ring_s[kSvWarps][64];
  __shared__ int2 out_ring_s[kSvWarps][32];
  __shared__ __align__(8) uint32_t row_ring_s[kSvWarps][2 * (kKxRing + 34)];
  static_assert(sizeof(in_ring_s[0]) >= kSvW, "column codes fit in the left-edge ring");
  const int warp = threadIdx.x >> 5, t = threadIdx.x & 31;
  uint8_t *prof = sv_smem + (size_t)warp * (size_t)p.prof_bytes;
  uint8_t *colc = reinterpret_cast<uint8_t *>(in_ring_s[warp]);
  unsigned smid;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
  int32_t *busy = &p.ctl->busy[(smid * kSvWarps + warp) & 1023];

  for (;;) {
    // ---- claim the next task (lane 0), bounded idle wait ----------------
    int slot = -1, strip = 0, quit = 0;
    if (t == 0) {
      SvCtl *ctl = p.ctl;
      uint64_t idle0 = 0, avail0 = 0;
      unsigned ns = 64;
      for (;;) {
        // entries that the producer has published since the last look
        const unsigned long long tl = sv_ld_acquire64(&ctl->tail.v);
        if (tl > *(volatile unsigned long long *)&ctl->seen.v) {
          const unsigned long long old = atomicMax(&ctl->seen.v, tl);
          if (old < tl) {
            __threadfence();
            atomicAdd(&ctl->ready.v, (int32_t)(tl - old));
          }
        }
        const int cont = *(volatile int32_t *)&ctl->cont_ready.v, fresh = *(volatile int32_t *)&ctl->ready.v;
        const uint64_t now = sv_now();
        if (cont > 0 || fresh > 0) {
          bool go = ::max(cont, 0) + ::max(fresh, 0) >= kSvPlenty;
          if (!go) {
            const int running = *(volatile int32_t *)busy;
            if (!avail0) avail0 = now;
            go = running <= 0 || now - avail0 >= (uint64_t)running * kSvShareNs;
          }
          if (go) {
            // continuations first: they belong to requests already running
            if (cont > 0 && sv_take(&ctl->cont_ready.v)) {
              const unsigned long long h = atomicAdd(&ctl->cont_head.v, 1ull);
              const int64_t e = (int64_t)(h % (unsigned long long)p.cont_cap);
              // (as many entries are published as tickets were drawn, but entry h
              // may be one whose warp is between reserving and publishing it; one that
              // never shows is not read: the warp leaves, its request stays open)
              bool there;
              while (!(there = sv_ld_acquire64(p.cont_seq + e) == h + 1) && sv_now() - now < (uint64_t)p.wait_ns) {
              }
              if (!there) {
                quit = 1;
                break;
              }
              const int2 tk = __ldcg(p.cont + e);
              slot = tk.x;
              strip = tk.y;
              break;
            }
            if (fresh > 0 && sv_take(&ctl->ready.v)) {
              const unsigned long long h = atomicAdd(&ctl->head.v, 1ull);
              const int2 tk = __ldcg(p.tasks + (int64_t)(h % (unsigned long long)p.task_cap));
              slot = tk.x;
              strip = tk.y;
              break;
            }
          }
          idle0 = 0;
          ns = 64;
          __nanosleep(ns);
          continue;
        }
        avail0 = 0;
        // no task: leave once nothing is in flight and the producer has
        // stopped (or has been quiet for idle_ns)
        const bool drained = sv_ld_acquire64(&ctl->admitted.v) == *(volatile unsigned long long *)&ctl->completed.v;
        if (drained && sv_ld_sys(p.stop)) {
          quit = 1;
          break;
        }
        if (!idle0) idle0 = now;
        else if (drained && now - idle0 > (uint64_t)p.idle_ns) {
          quit = 1;
          break;
        } else if (now - idle0 > (uint64_t)p.wait_ns) {  // nothing claimable for wait_ns
          quit = 1;
          break;
        }
        __nanosleep(ns);
        if (ns < 1024) ns *= 2;
      }
      if (!quit) atomicAdd(busy, 1);
    }
    quit = __shfl_sync(0xffffffffu, quit, 0);
    if (quit) break;
    slot = __shfl_sync(0xffffffffu, slot, 0);
    strip = __shfl_sync(0xffffffffu, strip, 0);

    SvRequest *rq = p.req + slot;
    const int m = __ldcg(&rq->m), n = __ldcg(&rq->n);
    const int mode = __ldcg(&rq->mode), sc = __ldcg(&rq->scoring);
    SvView v;
    v.sw = m > n;
    v.R = v.sw ? n : m;
    v.C = v.sw ? m : n;
    v.rowraw = v.sw ? (const uint8_t *)__ldcg((const unsigned long long *)&rq->t)
                    : (const uint8_t *)__ldcg((const unsigned long long *)&rq->q);
    v.colraw = v.sw ? (const uint8_t *)__ldcg((const unsigned long long *)&rq->q)
                    : (const uint8_t *)__ldcg((const unsigned long long *)&rq->t);
    v.nstrips = __ldcg(&rq->nstrips);
    v.edges = (int2 *)__ldcg((const unsigned long long *)&rq->edges);
    v.A = __ldcg(&p.scorings[sc].A);
    v.alpha = __ldcg(&p.scorings[sc].alpha);
    v.beta = __ldcg(&p.scorings[sc].beta);
    v.sigma = p.scorings[sc].sigma;
    v.packed = __ldcg(&p.scorings[sc].packed);

    int val;
    if (v.R == 0 || v.C == 0) {  // closed forms, any mode
      const int len = v.R + v.C;
      val = (mode == kModeGlobal && len) ? -(v.alpha + v.beta * (len - 1)) : 0;
    } else if (v.packed) {
      uint2 *ring = reinterpret_cast<uint2 *>(row_ring_s[warp]), *out = reinterpret_cast<uint2 *>(out_ring_s[warp]);
      uint32_t *in = reinterpret_cast<uint32_t *>(in_ring_s[warp]);
      const SvScoring *scp = p.scorings + sc;
      val = mode == kModeLocal    ? sv_packed<kModeLocal>(p, rq, slot, v, scp, strip, t, ring, in, out, prof)
            : mode == kModeGlobal ? sv_packed<kModeGlobal>(p, rq, slot, v, scp, strip, t, ring, in, out, prof)
                                  : sv_packed<kModeSemi>(p, rq, slot, v, scp, strip, t, ring, in, out, prof);
    } else if (mode == kModeLocal) {
      val = sv_strip<kModeLocal>(p, rq, slot, v, strip, t, prof, colc, in_ring_s[warp],
                                 out_ring_s[warp], row_ring_s[warp]);
    } else if (mode == kModeGlobal) {
      val = sv_strip<kModeGlobal>(p, rq, slot, v, strip, t, prof, colc, in_ring_s[warp],
                                  out_ring_s[warp], row_ring_s[warp]);
    } else {
      val = sv_strip<kModeSemi>(p, rq, slot, v, strip, t, prof, colc, in_ring_s[warp],
                                out_ring_s[warp], row_ring_s[warp]);
    }
    if (t == 0) {
      atomicSub(busy, 1);
      if (mode == kModeGlobal) {
        if (strip + 1 == v.nstrips || v.R == 0 || v.C == 0) atomicExch(&rq->score, val);
      } else {
        atomicMax(&rq->score, val);
      }
      __threadfence();
      const int done = atomicAdd(&rq->strips_done, 1) + 1;
      if (done == v.nstrips) {
        __threadfence();
        atomicAdd(&p.ctl->completed.v, 1ull);
        const int score = atomicAdd(&rq->score, 0);
        const int status = atomicAdd(&rq->status, 0);
        int32_t *out = (int32_t *)__ldcg((const unsigned long long *)&rq->out);
        if (out) *out = status ? INT_MIN : score;
        if (p.comp) {
          const unsigned long long idx = atomicAdd(&p.ctl->comp_count.v, 1ull);
          SvCompletion *c = p.comp + (int64_t)(idx % (unsigned long long)p.comp_cap);
          c->id = __ldcg(&rq->id);
          c->score = status ? INT_MIN : score;
          c->status = status;
          c->slot = slot;
          __threadfence_system();
          *(volatile int64_t *)&c->seq = (int64_t)idx + 1;
        }
      }
    }
    __syncwarp();
  }
}

}  // namespace ga
