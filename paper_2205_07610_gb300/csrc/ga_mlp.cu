// ga_mlp.cu -- training and inference kernels of the band predictor's
// network and their C ABI (include/gotoh_band.h).  Not part of the paper.
//
// Training is one launch for all of its steps (mlp_train_kernel): one cluster
// of blocks that keeps the parameters on chip and sums every gradient over the
// batch in sample order (deterministic, no atomics).
#include <cooperative_groups.h>

#include <cmath>
#include <vector>

#include "../../include/gotoh_band.h"
#include "ga_common.cuh"
#include "ga_mlp.cuh"
#include "ga_pool.h"

namespace ga {

// Dynamic shared memory of the per-sample kernels: the parameters as float,
// then per thread two columns of 64 activations ([unit][thread] layout, so
// that a warp touches 32 consecutive words).
constexpr int kParamsPadded = kMlpParamsPadded;
__host__ __device__ constexpr size_t mlp_smem_bytes(int threads) {
  return sizeof(float) * ((size_t)kParamsPadded + 2 * (size_t)kMlpH * (size_t)threads);
}

// Thread per sample: y = net(x).  Inputs are rows of 32 floats.
__global__ void __launch_bounds__(128) mlp_forward_kernel(const uint16_t *__restrict__ wb,
                                                          const float *__restrict__ x, int64_t n,
                                                          float *__restrict__ y) {
  extern __shared__ float ws[];
  const int T = blockDim.x;
  float *a1 = ws + kParamsPadded + threadIdx.x, *a2 = a1 + kMlpH * T;
  stage_params(wb, ws);
  __syncthreads();
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < n;
       b += (int64_t)gridDim.x * blockDim.x) {
    const float *xv = x + b * kMlpIn;
    for (int o = 0; o < kMlpH; ++o) a1[o * T] = unit1(ws, o, xv, 1);
    for (int o = 0; o < kMlpH; ++o) a2[o * T] = fmaxf(unit2(ws, o, a1, T), 0.f);
    y[b] = output(ws, a2, T);
  }
}

struct AdamArgs {
  float lr, beta1, beta2, eps;
  int update;  // 0: gradient (and loss) only
};

struct TrainParams {
  const uint16_t *wb_in;   // bf16 parameters of a gradient-only call (update == 0)
  float *master;           // float32 parameters, moments and bf16 copy (update != 0)
  float *adam_m, *adam_v;
  uint16_t *wb;
  const float *x;          // [nsamples][32]
  const float *target;
  const int32_t *idx;      // [steps][B], or null: samples 0 .. B - 1
  int64_t nsamples;
  int32_t steps, B;
  float inv_b;             // 1 / B
  const float2 *coef;      // per step: 1 / (1 - beta1^t), 1 / (1 - beta2^t)
  float *grad_out, *loss_out;
  int32_t *status;
  AdamArgs a;
};

// All Adam steps (or one gradient) in one launch of one cluster of NC blocks.
//
// What bounds it: a step is a chain of dependent sums, not work (1.3 MFMA at a
// batch of 256).  The sums keep the order of the plain loops (a unit's dot
// product in index order, a parameter's gradient in sample order), so every
// result is the same float32 value whatever the cluster size; the shortest
// possible step is then 32 + 64 + 64 + 64 dependent multiply-adds of a sample,
// 256 of a parameter, and two exchanges.  Two launches per step with a thread
// per sample and a thread per parameter took 265 us per step at a batch of 256
// (2 blocks, then 50 blocks of uncoalesced column reads); this takes 10.6 us, of
// which 2.6 us are the forward and backward pass, 2.3 us the gradients (both at one
// shared-memory wavefront per cycle), 1.1 us Adam, and 3 us the exchanges.
//
// Split.  Chunks of 256 samples.  Forward and backward: each block owns SP =
// 256 / NC samples, a warp four of them: lane l computes units l and l + 32 of
// its warp's samples, so a layer needs only __syncwarp and every weight read
// serves four samples.  Gradients: block (p, q) of a 4 x NC/4 grid owns the
// parameters of 16 units o = 16p.. and 1/(NC/4) of the inputs i of W1 and W2, a
// 2 x 2 tile per thread, with the master value and both moments in registers
// for the whole run.  The exchanges are bulk copies between the blocks' shared
// memories, counted by an mbarrier of the receiver: a block's samples of one group
// of units are one piece for each block that owns parameters of those units, and a
// block's new weights are one tile for every other block.  (Stored value by value
// into the receivers, 53 KB a step and block in pieces of 64 bytes, between cluster
// barriers, the exchanges took 7 us: 13.8 us a step.)  The two waits order
// everything: a block sends activations only after it has every block's weights,
// and weights only after it has every block's activations, so what is overwritten
// has been read, and no piece of a step is counted in the phase of another.  That
// takes a piece from every block: one that holds no sample of a chunk sends 16 bytes
// that nobody reads.  Chunks without new weights end in a cluster barrier instead.  The
// next chunk's inputs are loaded a chunk ahead.  The last warp takes the biases,
// the head and the loss.
constexpr int kTrChunk = 256;  // samples per chunk

template <int NC>
struct TrainShape {
  static constexpr int Q = NC / 4;                  // blocks along the inputs of a layer
  static constexpr int I1 = kMlpIn / Q, I2 = kMlpH / Q;  // input columns of W1 and W2 per block
  static constexpr int SP = kTrChunk / NC;          // samples per block and chunk
  static constexpr int T = 8 * SP;                  // threads: 4 samples x 32 lanes per warp
  static constexpr int N2 = 8 * (I2 / 2), N1 = 8 * (I1 / 2);  // threads with a tile of W2, of W1
  static constexpr int PER = kTrChunk / T;          // staged samples per thread
  static_assert(N2 + N1 + 32 <= T && PER * I1 == 16, "roles");
  // Weights: W1 and W2 as the tiles of the blocks that own them (16 units x I1 or
  // I2 inputs, padded rows), so that a block's new weights are one piece.  Row and
  // tile strides keep row reads by 8 lanes and column reads by 32 conflict-free.
  static constexpr int RS1 = I1 + 4, RS2 = I2 + 4, TS1 = 16 * RS1, TS2 = 16 * RS2 + (I2 == 16 ? 16 : 0);
  static constexpr int oW1 = 0, oW2 = oW1 + NC * TS1, oB1 = oW2 + NC * TS2, oB2 = oB1 + kMlpH, oW3 = oB2 + kMlpH,
                       oB3 = oW3 + kMlpH, kWeights = oB3 + 4;
  static constexpr int kAct = 4 * (kMlpIn + 3 * kMlpH);  // floats per warp: x, h1, h2, d2 of 4 samples
  // what the block sends: per group of units, its samples' rows
  static constexpr int GS = SP * 16 + 16, GS1 = SP * I2 + (I2 == 16 ? 16 : 0);
  static constexpr int oS2 = kWeights + (T / 32) * kAct, oS1 = oS2 + 4 * GS, oSH = oS1 + 4 * GS, oSA = oSH + 4 * GS,
                       oSY = oSA + Q * GS1, oSR = oSY + SP;
  // what it receives, a row per sample of the chunk
  static constexpr int oD2 = oSR + SP, oD1 = oD2 + 16 * kTrChunk,
                       oH2 = oD1 + 16 * kTrChunk, oH1 = oH2 + 16 * kTrChunk, oX = oH1 + I2 * kTrChunk,
                       oDY = oX + I1 * kTrChunk, oR = oDY + kTrChunk, oBar = oR + kTrChunk, oUnread = oBar + 4,
                       kFloats = oUnread + 4;
  static_assert(oW2 % 4 == 0 && oB1 % 4 == 0 && kWeights % 4 == 0 && GS % 4 == 0 && GS1 % 4 == 0 && oBar % 4 == 0,
                "16-byte pieces");
  static constexpr __device__ __forceinline__ int w1(int o, int i) {
    return oW1 + (o / 16 * Q + i / I1) * TS1 + o % 16 * RS1 + i % I1;
  }
  static constexpr __device__ __forceinline__ int w2(int o, int i) {
    return oW2 + (o / 16 * Q + i / I2) * TS2 + o % 16 * RS2 + i % I2;
  }
  // Position of parameter k.
  static __device__ __forceinline__ int slot(int k) {
    if (k < kOffB1) return w1(k / kMlpIn, k % kMlpIn);
    if (k < kOffW2) return oB1 + (k - kOffB1);
    if (k < kOffB2) return w2((k - kOffW2) / kMlpH, (k - kOffW2) % kMlpH);
    if (k < kOffW3) return oB2 + (k - kOffB2);
    if (k < kOffB3) return oW3 + (k - kOffW3);
    return oB3;
  }
  static constexpr size_t kSmem = sizeof(float) * kFloats;
  static_assert(kSmem <= 227 * 1024, "shared memory");
};

__device__ __forceinline__ float tr_bf16(float w) { return bf16_bits_to_f32(f32_to_bf16_bits(w)); }

struct TrState {  // one parameter's float32 value and moments
  float w, m, v;
};

__device__ __forceinline__ void tr_adam(TrState &s, float g, const AdamArgs &a, float2 c) {
  s.m = fmaf(a.beta1, s.m, (1.f - a.beta1) * g);
  s.v = fmaf(a.beta2, s.v, (1.f - a.beta2) * g * g);
  const float mhat = s.m * c.x, vhat = s.v * c.y;
  s.w = s.w - a.lr * mhat / (sqrtf(vhat) + a.eps);
}

// Dot products of two units with four samples: z[u][s] += sum_k W[u][k] x[s][k] in
// index order; W0 and W1 point to the units' rows in the first of the tiles of I
// inputs, TS apart.
template <int N, int I, int TS>
__device__ __forceinline__ void tr_layer(const float *W0, const float *W1, const float *x, float (&z)[2][4]) {
#pragma unroll 4
  for (int k = 0; k < N; k += 4) {
    const int at = k / I * TS + k % I;
    const float4 wa = *reinterpret_cast<const float4 *>(W0 + at);
    const float4 wc = *reinterpret_cast<const float4 *>(W1 + at);
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const float4 v = *reinterpret_cast<const float4 *>(x + s * N + k);
      z[0][s] = fmaf(wa.w, v.w, fmaf(wa.z, v.z, fmaf(wa.y, v.y, fmaf(wa.x, v.x, z[0][s]))));
      z[1][s] = fmaf(wc.w, v.w, fmaf(wc.z, v.z, fmaf(wc.y, v.y, fmaf(wc.x, v.x, z[1][s]))));
    }
  }
}

// Pieces between the blocks' shared memories: one bulk copy each, counted in bytes
// by an mbarrier of the receiver.
__device__ __forceinline__ uint32_t tr_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t tr_peer(uint32_t addr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void tr_copy(int rank, const float *dst, const float *src, int floats, const uint64_t *bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(tr_peer(tr_addr(dst), rank)), "r"(tr_addr(src)), "r"(4 * floats), "r"(tr_peer(tr_addr(bar), rank))
               : "memory");
}
__device__ __forceinline__ void tr_bar_init(uint64_t *bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tr_addr(bar)) : "memory");
}
__device__ __forceinline__ void tr_expect(uint64_t *bar, int bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tr_addr(bar)), "r"(bytes) : "memory");
}
// False: the limit ran out (2 s; nothing of the kernel waits that long).
__device__ __forceinline__ bool tr_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok = 0;
  const long long start = clock64();
  while (!ok && clock64() - start < (1ll << 32))
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        "selp.b32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(tr_addr(bar)), "r"(parity)
        : "memory");
  return ok != 0;
}
// Shared memory written by this thread may be the source of a bulk copy.
__device__ __forceinline__ void tr_publish() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

template <int NC>
__global__ void __launch_bounds__(TrainShape<NC>::T, 1) mlp_train_kernel(const __grid_constant__ TrainParams p) {
  using S = TrainShape<NC>;
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) float tr_smem[];
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), tid = threadIdx.x, l = tid & 31, warp = tid >> 5;
  const int bp = rank / S::Q, bq = rank % S::Q;
  float *W = tr_smem;
  uint64_t *bar_a = reinterpret_cast<uint64_t *>(tr_smem + S::oBar), *bar_w = bar_a + 1;
  float *xs = tr_smem + S::kWeights + warp * S::kAct, *h1s = xs + 4 * kMlpIn, *h2s = h1s + 4 * kMlpH,
        *d2s = h2s + 4 * kMlpH;
  const bool upd = p.a.update != 0;

  for (int k = tid; k < kMlpParams; k += S::T)
    W[S::slot(k)] = upd ? tr_bf16(p.master[k]) : bf16_bits_to_f32(p.wb_in[k]);

  // ---- the parameters of this thread --------------------------------------
  // role 0: 2 x 2 tile of W2, 1: of W1, 2: one parameter or the loss, 3: none
  int role = 3, par[4] = {-1, -1, -1, -1};  // parameter indices
  // staged columns (a row per sample): units and inputs, with their row lengths
  const float *pu = tr_smem, *pv = tr_smem;
  int su = 16, sv = 16;
  bool sum_only = false, is_loss = false;
  if (tid < S::N2) {
    role = 0;
    const int o = 2 * (tid / (S::I2 / 2)), i = 2 * (tid % (S::I2 / 2));
    pu = tr_smem + S::oD2 + o;
    pv = tr_smem + S::oH1 + i;
    sv = S::I2;
    for (int e = 0; e < 4; ++e) par[e] = kOffW2 + (16 * bp + o + (e >> 1)) * kMlpH + S::I2 * bq + i + (e & 1);
  } else if (tid < S::N2 + S::N1) {
    role = 1;
    const int r = tid - S::N2, o = 2 * (r / (S::I1 / 2)), i = 2 * (r % (S::I1 / 2));
    pu = tr_smem + S::oD1 + o;
    pv = tr_smem + S::oX + i;
    sv = S::I1;
    for (int e = 0; e < 4; ++e) par[e] = kOffW1 + (16 * bp + o + (e >> 1)) * kMlpIn + S::I1 * bq + i + (e & 1);
  } else if (tid < S::N2 + S::N1 + 32) {
    const int r = l & 15;
    if (bq == 0) {
      role = 2;
      sum_only = l >= 16;
      par[0] = (sum_only ? kOffB2 : kOffW3) + 16 * bp + r;
      pu = tr_smem + (sum_only ? S::oD2 + r : S::oDY);
      su = sum_only ? 16 : 1;
      pv = tr_smem + S::oH2 + r;
    } else if (bq == 1 && l < 16) {
      role = 2;
      sum_only = true;
      par[0] = kOffB1 + 16 * bp + r;
      pu = tr_smem + S::oD1 + r;
    } else if (bq == 1 && bp == 0 && l == 16) {
      role = 2;
      sum_only = true;
      par[0] = kOffB3;
      pu = tr_smem + S::oDY;
      su = 1;
    } else if (bq == 1 && bp == 0 && l == 17) {
      role = 2;
      is_loss = true;
      pu = pv = tr_smem + S::oR;
      su = sv = 1;
    }
  }
  TrState st[4] = {};
  if (upd)
    for (int e = 0; e < 4; ++e)
      if (par[e] >= 0) st[e] = TrState{p.master[par[e]], p.adam_m[par[e]], p.adam_v[par[e]]};

  // ---- inputs of one chunk, loaded a chunk ahead ---------------------------
  float xv[4], tv = 0.f, xc[S::PER][S::I1];  // own samples (lane = input), target of sample l % 4, staged columns
  uint32_t ok = 0;                           // bits 0..3: the warp's samples are valid
  int bad_idx = 0;
  // the index is only loaded here; it is checked where the inputs are read, so
  // that nothing waits for it (kNone: no sample at this place)
  constexpr int32_t kNone = INT32_MIN;
  auto sample_of = [&](int step, int c0, int b) -> int32_t {
    if (step >= p.steps || b >= ::min(kTrChunk, p.B - c0)) return kNone;
    return p.idx ? p.idx[(int64_t)step * p.B + c0 + b] : c0 + b;
  };
  auto own_base = [&](int cb) -> int {  // first sample of this warp in a chunk of cb, or >= cb
    const int spc = ((cb + NC - 1) / NC + 3) & ~3;
    return 4 * warp < spc ? rank * spc + 4 * warp : kTrChunk;
  };
  int32_t own_s[4], con_s[S::PER];
  auto read_idx = [&](int step, int c0) {
    const int sb = own_base(::min(kTrChunk, p.B - c0));
#pragma unroll
    for (int s = 0; s < 4; ++s) own_s[s] = sample_of(step, c0, sb + s);
#pragma unroll
    for (int j = 0; j < S::PER; ++j) con_s[j] = sample_of(step, c0, tid + j * S::T);
  };
  auto read_x = [&]() {
    ok = 0;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const bool in = own_s[s] >= 0 && own_s[s] < p.nsamples;
      xv[s] = in ? p.x[(int64_t)own_s[s] * kMlpIn + l] : 0.f;
      ok |= (in ? 1u : 0u) << s;
      if ((l & 3) == s) tv = in ? p.target[own_s[s]] : 0.f;
    }
#pragma unroll
    for (int j = 0; j < S::PER; ++j) {
      const bool in = con_s[j] >= 0 && con_s[j] < p.nsamples;
      bad_idx |= !in && con_s[j] != kNone;
#pragma unroll
      for (int i = 0; i < S::I1; ++i) xc[j][i] = in ? p.x[(int64_t)con_s[j] * kMlpIn + S::I1 * bq + i] : 0.f;
    }
  };
  read_idx(0, 0);
  read_x();
  if (tid == 0) {
    tr_bar_init(bar_a);
    tr_bar_init(bar_w);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  cluster.sync();  // every block of the cluster runs, its weights and barriers are in place
  uint32_t parity_a = 0;
  bool late = false;  // a wait has run out
  // bytes of the weights that the other blocks send
  constexpr int kOwnTiles = 16 * (S::RS1 + S::RS2);
  const int w_bytes = 4 * ((NC - 1) * kOwnTiles + (bq == 0 ? 3 : 4) * 32 + (bq == 1 ? 3 : 4) * 16 + (rank == 1 ? 0 : 4));

  // bytes of a chunk's activations: of a full one, of the rest
  const int row_bytes = 4 * (S::I2 + 32 + (bq == 0 ? 17 : 0) + (rank == 1 ? 2 : 0));
  const int rest = p.B % kTrChunk, rest_spc = ((rest + NC - 1) / NC + 3) & ~3;
  const int a_bytes_full = row_bytes * kTrChunk;
  const int a_bytes_rest =
      rest ? row_bytes * ((rest + 3) & ~3) + 16 * (NC - (rest + rest_spc - 1) / rest_spc) : 0;

  for (int step = 0; step < p.steps; ++step) {
    if (upd && tid == 0) tr_expect(bar_w, w_bytes);
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    const float2 coef = upd ? p.coef[step] : make_float2(0.f, 0.f);
    for (int c0 = 0; c0 < p.B; c0 += kTrChunk) {
      const int cb = ::min(kTrChunk, p.B - c0);
      const int sb = own_base(cb);
      if (tid == 0) tr_expect(bar_a, cb == kTrChunk ? a_bytes_full : a_bytes_rest);
      // ---- forward and backward of this warp's four samples -----------------
#pragma unroll
      for (int j = 0; j < S::PER; ++j)
#pragma unroll
        for (int i = 0; i < S::I1; i += 4)
          *reinterpret_cast<float4 *>(tr_smem + S::oX + (tid + j * S::T) * S::I1 + i) =
              make_float4(xc[j][i], xc[j][i + 1], xc[j][i + 2], xc[j][i + 3]);
#pragma unroll
      for (int s = 0; s < 4; ++s) xs[s * kMlpIn + l] = xv[s];
      const float target = tv;
      const uint32_t valid = ok;
      const bool last = c0 + kTrChunk >= p.B;
      read_idx(last ? step + 1 : step, last ? 0 : c0 + kTrChunk);
      __syncwarp();
      if (sb < cb) {
        float z[2][4], h1[2][4], h2[2][4], d2[2][4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          z[0][s] = W[S::oB1 + l];
          z[1][s] = W[S::oB1 + l + 32];
        }
        tr_layer<kMlpIn, S::I1, S::TS1>(W + S::w1(l, 0), W + S::w1(l + 32, 0), xs, z);
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int s = 0; s < 4; ++s) h1s[s * kMlpH + l + 32 * u] = h1[u][s] = fmaxf(z[u][s], 0.f);
        __syncwarp();
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          z[0][s] = W[S::oB2 + l];
          z[1][s] = W[S::oB2 + l + 32];
        }
        tr_layer<kMlpH, S::I2, S::TS2>(W + S::w2(l, 0), W + S::w2(l + 32, 0), h1s, z);
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int s = 0; s < 4; ++s) h2s[s * kMlpH + l + 32 * u] = h2[u][s] = fmaxf(z[u][s], 0.f);
        __syncwarp();
        float y = W[S::oB3];
        const float *hv = h2s + (l & 3) * kMlpH;
#pragma unroll 4
        for (int o = 0; o < kMlpH; o += 4) {
          const float4 w = *reinterpret_cast<const float4 *>(W + S::oW3 + o);
          const float4 v = *reinterpret_cast<const float4 *>(hv + o);
          y = fmaf(w.w, v.w, fmaf(w.z, v.z, fmaf(w.y, v.y, fmaf(w.x, v.x, y))));
        }
        const bool mine = (valid >> (l & 3)) & 1u;
        const float r = mine ? y - target : 0.f, dy = mine ? r * p.inv_b : 0.f;
        float dys[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) dys[s] = __shfl_sync(0xffffffffu, dy, s);
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int s = 0; s < 4; ++s)
            d2s[s * kMlpH + l + 32 * u] = d2[u][s] = h2[u][s] > 0.f ? dys[s] * W[S::oW3 + l + 32 * u] : 0.f;
        __syncwarp();
#pragma unroll
        for (int s = 0; s < 4; ++s) z[0][s] = z[1][s] = 0.f;
#pragma unroll 2
        for (int o = 0; o < kMlpH; o += 4) {
          float wa[4], wc[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            wa[j] = W[S::w2(o + j, l)];
            wc[j] = W[S::w2(o + j, l + 32)];
          }
#pragma unroll
          for (int s = 0; s < 4; ++s) {
            const float4 d = *reinterpret_cast<const float4 *>(d2s + s * kMlpH + o);
            z[0][s] = fmaf(d.w, wa[3], fmaf(d.z, wa[2], fmaf(d.y, wa[1], fmaf(d.x, wa[0], z[0][s]))));
            z[1][s] = fmaf(d.w, wc[3], fmaf(d.z, wc[2], fmaf(d.y, wc[1], fmaf(d.x, wc[0], z[1][s]))));
          }
        }
        // ---- staged for the blocks that own the parameters -------------------
        const int row = 4 * warp;
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const bool keep = (valid >> s) & 1u;  // an invalid sample adds nothing
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int unit = l + 32 * u, at = unit / 16 * S::GS + (row + s) * 16 + unit % 16;
            tr_smem[S::oS2 + at] = keep ? d2[u][s] : 0.f;
            tr_smem[S::oS1 + at] = keep && h1[u][s] > 0.f ? z[u][s] : 0.f;
            tr_smem[S::oSH + at] = keep ? h2[u][s] : 0.f;
            tr_smem[S::oSA + unit / S::I2 * S::GS1 + (row + s) * S::I2 + unit % S::I2] = keep ? h1[u][s] : 0.f;
          }
        }
        if (l < 4) {  // the head's error signal, the error
          tr_smem[S::oSY + row + l] = dy;
          tr_smem[S::oSR + row + l] = r;
        }
        tr_publish();
      }
      __syncthreads();
      {
        // this block's rows: b0 .. b0 + n of the chunk
        const int spc = ((cb + NC - 1) / NC + 3) & ~3, b0 = rank * spc;
        const int n = ::min(spc, ::max(0, (cb - b0 + 3) & ~3));
        if (n > 0) {
          // a kind of piece per warp, a block per lane
          const int d = l, kind = warp, dp = d / S::Q, dq = d % S::Q;
          if (d < NC && kind < 4) {
            if (kind == 0) tr_copy(d, tr_smem + S::oD2 + b0 * 16, tr_smem + S::oS2 + dp * S::GS, 16 * n, bar_a);
            else if (kind == 1) tr_copy(d, tr_smem + S::oD1 + b0 * 16, tr_smem + S::oS1 + dp * S::GS, 16 * n, bar_a);
            else if (kind == 2)
              tr_copy(d, tr_smem + S::oH1 + b0 * S::I2, tr_smem + S::oSA + dq * S::GS1, S::I2 * n, bar_a);
            else if (dq == 0) {
              tr_copy(d, tr_smem + S::oH2 + b0 * 16, tr_smem + S::oSH + dp * S::GS, 16 * n, bar_a);
              tr_copy(d, tr_smem + S::oDY + b0, tr_smem + S::oSY, n, bar_a);
            } else if (d == 1) {
              tr_copy(d, tr_smem + S::oDY + b0, tr_smem + S::oSY, n, bar_a);
              tr_copy(d, tr_smem + S::oR + b0, tr_smem + S::oSR, n, bar_a);
            }
          }
        } else if (warp == 0 && l < NC) {
          tr_copy(l, tr_smem + S::oUnread, tr_smem + S::oSY, 4, bar_a);
        }
      }
      read_x();  // the next chunk's inputs arrive while the gradients run
      if (!late) late = !tr_wait(bar_a, parity_a);
      parity_a ^= 1;
      // ---- gradients, in sample order ---------------------------------------
      if (role < 2) {
        // eight samples are loaded while the eight before them are summed
        float2 a[8], c[8];
        auto load8 = [&](int b) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            a[j] = *reinterpret_cast<const float2 *>(pu + (b + j) * 16);
            c[j] = *reinterpret_cast<const float2 *>(pv + (b + j) * sv);
          }
        };
        load8(0);
        int b = 0;
        for (; b + 8 <= cb; b += 8) {
          float2 a0[8], c0v[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            a0[j] = a[j];
            c0v[j] = c[j];
          }
          load8(::min(b + 8, kTrChunk - 8));
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            acc[0] = fmaf(a0[j].x, c0v[j].x, acc[0]);
            acc[1] = fmaf(a0[j].x, c0v[j].y, acc[1]);
            acc[2] = fmaf(a0[j].y, c0v[j].x, acc[2]);
            acc[3] = fmaf(a0[j].y, c0v[j].y, acc[3]);
          }
        }
        for (; b < cb; ++b) {
          const float2 e = *reinterpret_cast<const float2 *>(pu + b * 16);
          const float2 f = *reinterpret_cast<const float2 *>(pv + b * sv);
          acc[0] = fmaf(e.x, f.x, acc[0]);
          acc[1] = fmaf(e.x, f.y, acc[1]);
          acc[2] = fmaf(e.y, f.x, acc[2]);
          acc[3] = fmaf(e.y, f.y, acc[3]);
        }
      } else if (role == 2) {
#pragma unroll 8
        for (int b = 0; b < cb; ++b) acc[0] = fmaf(pu[b * su], sum_only ? 1.f : pv[b * sv], acc[0]);
      }
      if (last) {
        if (is_loss && p.loss_out) p.loss_out[step] = late ? NAN : 0.5f * acc[0] / (float)p.B;
        if (p.grad_out)
          for (int e = 0; e < 4; ++e)
            if (par[e] >= 0) p.grad_out[par[e]] = late ? NAN : acc[e];  // (no status to set)
        if (upd && role < 2) {
          float n[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            tr_adam(st[e], acc[e], p.a, coef);
            n[e] = tr_bf16(st[e].w);
          }
          *reinterpret_cast<float2 *>(W + S::slot(par[0])) = make_float2(n[0], n[1]);
          *reinterpret_cast<float2 *>(W + S::slot(par[2])) = make_float2(n[2], n[3]);
        } else if (upd && role == 2 && !is_loss) {
          tr_adam(st[0], acc[0], p.a, coef);
          W[S::slot(par[0])] = tr_bf16(st[0].w);
        }
      }
      if (last && upd) {
        // the new weights to every other block; what it received has been read
        tr_publish();
        __syncthreads();
        const int d = l, kind = warp;
        if (d < NC && d != rank) {
          const float *w2 = W + S::oW2 + rank * S::TS2, *w1 = W + S::oW1 + rank * S::TS1;
          if (kind == 0) tr_copy(d, w2, w2, 16 * S::RS2, bar_w);
          else if (kind == 1) tr_copy(d, w1, w1, 16 * S::RS1, bar_w);
          else if (kind == 2 && bq < 2) {
            const float *v = W + (bq == 0 ? S::oB2 : S::oB1) + 16 * bp;
            tr_copy(d, v, v, 16, bar_w);
          } else if (kind == 3 && (bq == 0 || rank == 1)) {
            const float *v = W + (bq == 0 ? S::oW3 + 16 * bp : S::oB3);
            tr_copy(d, v, v, bq == 0 ? 16 : 4, bar_w);
          }
        }
        if (!late) late = !tr_wait(bar_w, (uint32_t)step & 1u);
      } else if (!last) {
        cluster.sync();  // everything read before it is overwritten
      }
    }
  }
  cluster.sync();  // no block leaves while another copies from or to it
  if (late && p.status) set_status(p.status, GA_ERR_CUDA);
  if (bad_idx && p.status) set_status(p.status, GA_ERR_ARG);
  if (upd)
    for (int e = 0; e < 4; ++e)
      if (par[e] >= 0) {
        p.master[par[e]] = st[e].w;
        p.adam_m[par[e]] = st[e].m;
        p.adam_v[par[e]] = st[e].v;
        p.wb[par[e]] = f32_to_bf16_bits(st[e].w);
      }
}

// Cast of a float32 parameter vector to bf16 (round to nearest even).
__global__ void mlp_cast_kernel(const float *__restrict__ master, uint16_t *__restrict__ wb, int n) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) wb[k] = f32_to_bf16_bits(master[k]);
}


namespace {

constexpr int kMlpThreads = 128;
constexpr size_t kParamSmem = mlp_smem_bytes(kMlpThreads);

int mlp_smem_ok() {  // per call: the attribute belongs to the current device
  int ok = 0;
  {
    ok = cudaFuncSetAttribute(mlp_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kParamSmem) == cudaSuccess;
  }
  return ok;
}

struct Scratch {
  cudaStream_t s;
  void *p = nullptr;
  Scratch(cudaStream_t st, size_t bytes) : s(st) {
    if (pool_malloc(&p, bytes, s) != cudaSuccess) p = nullptr;
  }
  ~Scratch() {
    if (p) cudaFreeAsync(p, s);
  }
};

template <int NC>
cudaError_t launch_train(const TrainParams &p, cudaStream_t s, bool only_if_it_fits, bool *launched) {
  using S = TrainShape<NC>;
  *launched = false;
  cudaError_t e = cudaFuncSetAttribute(mlp_train_kernel<NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::kSmem);
  if (e == cudaSuccess && NC > 8)
    e = cudaFuncSetAttribute(mlp_train_kernel<NC>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(NC);
  cfg.blockDim = dim3(S::T);
  cfg.dynamicSmemBytes = S::kSmem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = NC;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (only_if_it_fits) {
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, mlp_train_kernel<NC>, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      return cudaSuccess;
    }
  }
  *launched = true;
  return cudaLaunchKernelEx(&cfg, mlp_train_kernel<NC>, p);
}

// Cluster size: 8 blocks below 32 samples a step, where a chunk keeps few warps
// busy (GB300, us per step, 16 / 8 blocks: 6.9 / 6.7 at 16 samples, 7.1 / 7.3 at
// 32, 7.7 / 8.1 at 64, 7.8 / 9.1 at 95); 8 is also the portable size where a device
// places no cluster of 16.  The results are the same.
cudaError_t enqueue_train(const TrainParams &p, cudaStream_t s) {
  bool launched = false;
  if (p.B >= 32) {
    const cudaError_t e = launch_train<16>(p, s, true, &launched);
    if (e != cudaSuccess || launched) return e;
  }
  return launch_train<8>(p, s, false, &launched);
}

}  // namespace
}  // namespace ga

using namespace ga;

extern "C" {

int ga_mlp_forward(const uint16_t *params_bf16, const float *x, int64_t n, float *y, void *stream) {
  if (n < 0 || (n > 0 && (!params_bf16 || !x || !y))) return GA_ERR_ARG;
  if (n == 0) return GA_OK;
  if (!mlp_smem_ok()) return GA_ERR_CUDA;
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return GA_ERR_CUDA;
  const int64_t want = (n + kMlpThreads - 1) / kMlpThreads;
  const int grid = (int)(want < (int64_t)nsm * 8 ? want : (int64_t)nsm * 8);
  mlp_forward_kernel<<<grid, kMlpThreads, kParamSmem, (cudaStream_t)stream>>>(params_bf16, x, n, y);
  return cudaGetLastError() == cudaSuccess ? GA_OK : GA_ERR_CUDA;
}

int ga_mlp_loss_grad(const uint16_t *params_bf16, const float *x, const float *target, int32_t n,
                     float *grad, float *loss, void *stream) {
  if (n <= 0 || !params_bf16 || !x || !target || !grad) return GA_ERR_ARG;
  TrainParams p{};
  p.wb_in = params_bf16;
  p.x = x;
  p.target = target;
  p.nsamples = n;
  p.steps = 1;
  p.B = n;
  p.inv_b = 1.0f / (float)n;
  p.grad_out = grad;
  p.loss_out = loss;
  return enqueue_train(p, (cudaStream_t)stream) == cudaSuccess ? GA_OK : GA_ERR_CUDA;
}

int ga_mlp_train(float *master, uint16_t *params_bf16, float *adam_m, float *adam_v, const float *x,
                 const float *target, int64_t nsamples, const int32_t *batch_idx, int32_t steps,
                 int32_t batch, int32_t step0, float lr, float beta1, float beta2, float eps,
                 float *losses, void *stream) {
  if (!master || !params_bf16 || !adam_m || !adam_v || !x || !target || !batch_idx) return GA_ERR_ARG;
  if (nsamples <= 0 || steps < 0 || batch <= 0 || batch > (1 << 20) || step0 < 0) return GA_ERR_ARG;
  if (!(lr > 0.f) || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f) || !(eps >= 0.f))
    return GA_ERR_ARG;
  if (steps == 0) return GA_OK;
  cudaStream_t s = (cudaStream_t)stream;
  Scratch st(s, 256 + sizeof(float2) * (size_t)steps);
  if (!st.p) return GA_ERR_OOM;
  int32_t *status = (int32_t *)st.p;
  float2 *coef = (float2 *)((char *)st.p + 256);
  std::vector<float2> h_coef((size_t)steps);  // bias corrections, in double on the host
  for (int k = 0; k < steps; ++k) {
    const double t = (double)step0 + k + 1;
    h_coef[k] = make_float2((float)(1.0 / (1.0 - std::pow((double)beta1, t))),
                            (float)(1.0 / (1.0 - std::pow((double)beta2, t))));
  }
  if (cudaMemsetAsync(status, 0, sizeof(int32_t), s) != cudaSuccess ||
      cudaMemcpyAsync(coef, h_coef.data(), sizeof(float2) * h_coef.size(), cudaMemcpyHostToDevice, s) != cudaSuccess)
    return GA_ERR_CUDA;
  TrainParams p{};
  p.master = master;
  p.adam_m = adam_m;
  p.adam_v = adam_v;
  p.wb = params_bf16;
  p.x = x;
  p.target = target;
  p.idx = batch_idx;
  p.nsamples = nsamples;
  p.steps = steps;
  p.B = batch;
  p.inv_b = 1.0f / (float)batch;
  p.coef = coef;
  p.loss_out = losses;
  p.status = status;
  p.a = AdamArgs{lr, beta1, beta2, eps, 1};
  if (enqueue_train(p, s) != cudaSuccess) return GA_ERR_CUDA;
  int32_t h = 0;
  if (cudaMemcpyAsync(&h, status, sizeof(int32_t), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return GA_ERR_CUDA;
  return h ? h : GA_OK;
}

int ga_mlp_cast(const float *master, uint16_t *params_bf16, void *stream) {
  if (!master || !params_bf16) return GA_ERR_ARG;
  mlp_cast_kernel<<<(kMlpParams + 255) / 256, 256, 0, (cudaStream_t)stream>>>(master, params_bf16,
                                                                                 kMlpParams);
  return cudaGetLastError() == cudaSuccess ? GA_OK : GA_ERR_CUDA;
}

}  // extern "C"
