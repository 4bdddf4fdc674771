// bf16 routing on the tcgen05 tensor cores.
//
//   predict (Eqs. pr2_predict, pr2_route; Algorithm 2 first two steps):
//     [p_old | b] = h [W ; W_p]^T   (fp32 accumulators in TMEM, K = d),
//     z = p_old + b, rho_hat = Softmax(z), idx = TopK(rho_hat, k), gates = rho_hat[idx],
//     p_old optionally written as the feature-cache logits.
//   replay (Sec. 4.1 "Replay During Training"):
//     p = h W^T, rho = Softmax(p), gates = rho[idx_in]   (no top-k, no predictor).
//
// A 128-token tile is handled by a cluster of S CTAs (S = 1, 2, 4 or 8) that split K = d.  Each
// tcgen05.mma costs the same issue time for any N <= 256 (one M=128 x N x K=16 step), so a lone
// tile's chain of d/16 MMAs, not bandwidth, bounds it, and only a K split shortens that chain:
// CTA r multiplies K blocks [r KB/S, (r+1) KB/S) into a partial [128 x NB] fp32 accumulator
// (NB = 2N columns [p_old | b] for predict, N for replay and loss).  The widest split whose
// clusters are all resident at once is taken, for any N and any number of K blocks: when it had
// to divide them (and N into sixteens) predict of 1000 tokens, d = 2048, took 25.3 us with N = 80
// (now 9.6), 35.9 with N = 144 (13.1), 26 with N = 256 (17.5), 53.7 with N = 256 and d = 7168
// (24.8), 29 with N = 128 and d = 2112 (11.5); loss T = 600, N = 160 27.9 (15.3).  With S = 2 and
// N > 128 predict splits the two passes over K instead (below).  When the tiles outnumber the SMs
// (S = 1), each CTA takes half the pipeline stages so that two run on an SM side by side, one
// CTA's loads and finishing overlapping the other's MMAs (RouteTcArgs::compact; predict T = 32768,
// N = 128, d = 2048 51.7 us against 61.8 with one CTA per SM and rows by warps).
//
// Warp roles: warp 0 = TMA producer, warp 1 = TMEM owner and MMA issuer, warps 2..5 = epilogue
// (by warps, below: all sixteen).
// With S > 1 the partials are reduce-scattered by rows through distributed shared memory: CTA q
// receives rows [q 128/S, (q+1) 128/S) of every CTA's partial, stored [source][column/4][row][4]
// so that each warp store moves contiguous bytes, in as many rounds of columns as shared memory
// asks for (predict: two or three from N = 176 on); rows beyond the batch are not moved.  Two ways
// to finish the rows:
//  - by warps (CTAs of sixteen warps; all but the next line): the warps bring the rows into row
//    order in shared memory, summing the S copies once, in source order (deterministic), and each
//    then finishes whole rows, a lane holding 2, 4 or 8 experts (N <= 64, 128, 256).  predict: the
//    top k + 1 come out one by one by warp maxima (redux.sync) over orderable 32-bit values.
//    loss: the dKL/dz rows leave transposed through shared memory.  Short chains of ALU work per
//    element bound this, not the shuffles or reductions, so it is the number of warps that counts:
//    calls by threads / six warps / sixteen, N = 128: predict T = 4001 16.5 / 16.2 / 14.0 us,
//    T = 600 12.9 / 11.1 / 10.2; loss T_c = 2048 18.9 / 21.1 / 17.7; by threads / sixteen warps
//    replay T = 4001 12.4 / 10.6, T = 256 9.2 / 7.5; predict T = 4096, N = 64 11.1 / 9.2, T = 8192
//    (S = 2) 22.2 / 20.5, T = 7000, N = 64, S = 2 13.4 / 12.9 (14.1 with four experts per lane);
//    S = 1: predict N = 256, T = 12000 46.7 / 44.5, loss T_c = 12000 54.3 / 52.4.
//  - by threads (predict and replay with S = 1 and N <= 128, or two CTAs per SM): one of 128
//    threads finishes its row straight from TMEM, without the pass through shared memory (predict
//    N = 64, T = 15000 25.7 us against 28.6 by warps; replay N = 256 with two CTAs per SM T = 40000
//    80.3 against 81.9 with one and rows by warps).  It reduces its experts to a max, a sum of
//    exp(z - max) and (predict) its top-16 by 64-bit keys (orderable z bits, inverted expert
//    index: z descending, ties to the lower expert), built by bitonic sorting 16 experts at a time
//    and merging, in one pass with a running (online) softmax sum.
// Selection is on z in fp32 (softmax is monotone, so the order equals the order of rho_hat).
#include <float.h>

#include <mutex>

#include "pr2_device.cuh"
#include "pr2_internal.h"

namespace pr2 {
namespace {

constexpr int kThreads = 192;                    // rows finished by threads
constexpr int kWarpThreads = 512;                // rows finished by warps
constexpr int kBK = 64;                          // bf16 elements per 128-byte swizzle row
constexpr int kATileBytes = kTileM * kBK * 2;    // 16 KB
constexpr int kKeep = kMaxTopK + 1;              // top-(k+1) kept for the margin
constexpr int kMaxSplit = 8;
static_assert(kMaxSplit == kRouteMaxSplit, "histogram rows per routing tile");
constexpr int kMaxStages = 12;
constexpr int kStageBudget = 192 * 1024;    // pipeline stages of a CTA alone on its SM
constexpr int kCompactBudget = 96 * 1024;   // two CTAs per SM (more token tiles than SMs)
constexpr int kFinishBudget = 224 * 1024;   // exchange and finishing of a CTA alone on its SM
constexpr int kAlignSlack = 1024, kBarBytes = 256;
constexpr int kMostSmem = kAlignSlack + kFinishBudget + kBarBytes;  // no launch takes more

struct RouteSmemLayout {
  int stages;
  int b_rows;        // rows of the weight tile: 2N (predict) or N (replay, loss)
  int passes;        // passes over K: 2 streams [W] then [W_p] (predict, N > 128), else 1
  int pass_rows;     // weight rows of a stage: b_rows / passes
  int stage_bytes;   // A + B
  int acc_cols;      // accumulator columns of a CTA (pass split: those of one pass)
  int xcols;         // split > 1: columns of a partial row that one round of the exchange moves
  int frows;         // rows finished at once: all 128 / S, or (S = 1, N > 208) half of them
  int bar_offset;    // after all stages (and after what the exchange and the rows take)
  int total;         // dynamic smem bytes requested (incl. 1 KB alignment slack)
};

__host__ __device__ inline RouteSmemLayout route_layout(int N, int mode, int split, bool compact) {
  RouteSmemLayout L;
  const bool predict = mode == kModePredict;
  L.b_rows = predict ? 2 * N : N;
  // Predict with more than 128 experts: [W; W_p] would make 80 KB stages (two in flight at
  // most), so the router and the predictor weights stream in two passes over K instead, each
  // stage holding N weight rows; h is read twice, but four stages overlap loads and MMAs.
  L.passes = (L.b_rows > 256 && N % 32 == 0) ? 2 : 1;
  L.pass_rows = L.b_rows / L.passes;
  L.stage_bytes = kATileBytes + L.pass_rows * kBK * 2;
  L.stages = (compact ? kCompactBudget : kStageBudget) / L.stage_bytes;
  if (L.stages > kMaxStages) L.stages = kMaxStages;
  if (L.stages < 2) L.stages = 2;
  L.bar_offset = L.stages * L.stage_bytes;
  L.acc_cols = L.passes == 2 && split == 2 ? N : L.b_rows;
  L.xcols = split > 1 ? L.acc_cols : 0;
  L.frows = kTileM / split;
  if (!compact) {
    // After the K blocks the stages' bytes hold the received copies [S][xcols/4][128/S][4] fp32,
    // in as few rounds as fit, then the rows in row order (loss: and as bf16).
    const int row = (L.b_rows / 4 + 1) * 16 + (mode == kModeLoss ? N * 2 + 8 : 0);
    while (L.frows * row > kFinishBudget) L.frows /= 2;
    for (int n = 2; L.xcols * kTileM * 4 + L.frows * row > kFinishBudget; ++n)
      L.xcols = ((L.acc_cols + n - 1) / n + 15) & ~15;
    const int need = L.xcols * kTileM * 4 + L.frows * row;
    if (need > L.bar_offset) L.bar_offset = (need + 15) & ~15;
  }
  L.total = kAlignSlack + L.bar_offset + kBarBytes;
  return L;
}

__host__ __device__ inline uint32_t tmem_cols_for(int cols) {
  uint32_t c = 32;
  while (c < static_cast<uint32_t>(cols)) c <<= 1;
  return c;
}

// Compare-exchange leaving the larger key in a.
__device__ __forceinline__ void cas_desc(uint64_t& a, uint64_t& b) {
  const bool sw = b > a;
  const uint64_t hi = sw ? b : a;
  const uint64_t lo = sw ? a : b;
  a = hi;
  b = lo;
}

// Bitonic sort of 16 keys into descending order.
__device__ __forceinline__ void sort16_desc(uint64_t (&v)[16]) {
#pragma unroll
  for (int kk = 2; kk <= 16; kk <<= 1)
#pragma unroll
    for (int j = kk >> 1; j > 0; j >>= 1)
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int l = i ^ j;
        if (l > i) {
          if ((i & kk) == 0)
            cas_desc(v[i], v[l]);
          else
            cas_desc(v[l], v[i]);
        }
      }
}

// top <- the 16 largest of top and c, both sorted descending (c is clobbered): the elementwise
// max of top and reversed c is a bitonic sequence holding them, then a bitonic merge sorts it.
__device__ __forceinline__ void merge16_desc(uint64_t (&top)[16], const uint64_t (&c)[16]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) top[i] = top[i] > c[15 - i] ? top[i] : c[15 - i];
#pragma unroll
  for (int j = 8; j > 0; j >>= 1)
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int l = i ^ j;
      if (l > i) cas_desc(top[i], top[l]);
    }
}

// 64-bit key ordering (z descending, expert ascending).  An empty slot is key 0, below every
// real key.
__device__ __forceinline__ uint64_t topk_key(float z, int e) {
  const uint32_t u = __float_as_uint(z);
  const uint32_t ord = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
  return (static_cast<uint64_t>(ord) << 32) | static_cast<uint32_t>(~static_cast<uint32_t>(e));
}
__device__ __forceinline__ float key_z(uint64_t key) {
  const uint32_t ord = static_cast<uint32_t>(key >> 32);
  return __uint_as_float((ord & 0x80000000u) ? (ord & 0x7fffffffu) : ~ord);
}
__device__ __forceinline__ int key_e(uint64_t key) {
  return static_cast<int>(~static_cast<uint32_t>(key));
}

// Write a finished predict row: idx and gates of the k best keys (divided by their sum under
// PR2_F_NORMALIZE_TOPK); returns the near-tie flag rho_hat_(k) - rho_hat_(k+1) <
// PR2_NEAR_TIE_GAP, always on the unnormalised probabilities.
__device__ __forceinline__ bool predict_write(const uint64_t (&key)[16], float mx, float inv_s,
                                              int64_t t, const RouteTcArgs& a) {
  int32_t* irow = a.idx_out + t * a.k;
  float* grow = a.gates + t * a.k;
  float pr[kKeep];
  float sk = 0.f;
#pragma unroll
  for (int j = 0; j < kKeep; ++j) {
    pr[j] = expf(key_z(key[j]) - mx) * inv_s;
    if (j < a.k) sk += pr[j];
  }
  const float sc = a.norm ? 1.0f / sk : 1.0f;
  float pk = 0.f, pk1 = 0.f;
#pragma unroll
  for (int j = 0; j < kKeep; ++j) {
    if (j < a.k) {
      irow[j] = key_e(key[j]);
      grow[j] = pr[j] * sc;
    }
    if (j == a.k - 1) pk = pr[j];
    if (j == a.k) pk1 = pr[j];
  }
  return (a.k < a.N) && (pk - pk1 < (float)PR2_NEAR_TIE_GAP);
}

// Orderable bits of z (z descending = bits descending), at least 1: 0 marks a removed expert.
__device__ __forceinline__ uint32_t order_bits(float z) {
  const uint32_t u = __float_as_uint(z);
  const uint32_t ord = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
  return ord > 1u ? ord : 1u;
}
__device__ __forceinline__ float order_value(uint32_t ord) {
  return __uint_as_float((ord & 0x80000000u) ? (ord & 0x7fffffffu) : ~ord);
}
// kE floats of shared or global memory from p (aligned to their size, at most 16 bytes).
template <int kE>
__device__ __forceinline__ void load_vec(const float* p, float (&v)[kE]) {
  if constexpr (kE == 2) {
    const float2 x = *reinterpret_cast<const float2*>(p);
    v[0] = x.x;
    v[1] = x.y;
  } else {
#pragma unroll
    for (int q = 0; q < kE; q += 4) {
      const float4 x = *reinterpret_cast<const float4*>(p + q);
      v[q] = x.x;
      v[q + 1] = x.y;
      v[q + 2] = x.z;
      v[q + 3] = x.w;
    }
  }
}
template <int kE>
__device__ __forceinline__ void store_vec(float* p, const float (&v)[kE]) {
  if constexpr (kE == 2) {
    *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
  } else {
#pragma unroll
    for (int q = 0; q < kE; q += 4)
      *reinterpret_cast<float4*>(p + q) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
  }
}
// Warp-wide operations on kRB rows at once: a warp issues in order, so each step is written for all
// rows before the next one.
template <int kRB>
__device__ __forceinline__ void warp_add(float (&v)[kRB]) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    float w[kRB];
#pragma unroll
    for (int j = 0; j < kRB; ++j) w[j] = __shfl_xor_sync(0xffffffffu, v[j], o);
#pragma unroll
    for (int j = 0; j < kRB; ++j) v[j] += w[j];
  }
}
template <int kRB>
__device__ __forceinline__ void warp_max(uint32_t (&v)[kRB]) {
#pragma unroll
  for (int j = 0; j < kRB; ++j) v[j] = __reduce_max_sync(0xffffffffu, v[j]);
}

// Finishes kRB predict rows by one warp (N <= 32 kE).  Row j: [p_old | b] of 2 N floats at rows[j] in
// shared memory, token t[j] (live[j]: inside the batch).  Lane l holds experts kE l .. kE l + kE - 1,
// sorted once; the top k + 1 then come out one by one, the lane whose head equals the warp's
// maximum giving it (the lowest such lane: z descending, ties to the lower expert).  Writes p_old,
// idx, gates (divided by their sum under PR2_F_NORMALIZE_TOPK), counts the experts into `hist`
// (with `count`) and returns the number of rows with rho_hat_(k) - rho_hat_(k+1) <
// PR2_NEAR_TIE_GAP, always on the unnormalised probabilities.
template <int kRB, int kE>
__device__ __forceinline__ int finish_predict_rows(const float* const (&rows)[kRB],
                                                   const int64_t (&t)[kRB],
                                                   const bool (&live)[kRB], const RouteTcArgs& a,
                                                   bool count, int (&hist)[kMaxExperts]) {
  const int lane = threadIdx.x & 31;
  const bool in = lane * kE < a.N;
  uint32_t key[kRB][kE];
  uint32_t ids[kRB];  // the lane's experts in the order of its keys, 4 bits each
  uint32_t head[kRB];
  float mx[kRB], sum[kRB], my_z[kRB], zs[kRB][kE];
  int my_e[kRB];
#pragma unroll
  for (int j = 0; j < kRB; ++j) {
    float z[kE];
    uint32_t id[kE];
#pragma unroll
    for (int q = 0; q < kE; ++q) id[q] = q;
    if (in) {
      float b[kE];
      load_vec<kE>(rows[j] + lane * kE, z);
      load_vec<kE>(rows[j] + a.N + lane * kE, b);
      if (a.logits_or_probs != nullptr && live[j])
        store_vec<kE>(a.logits_or_probs + t[j] * a.N + lane * kE, z);
#pragma unroll
      for (int q = 0; q < kE; ++q) z[q] += b[q];
#pragma unroll
      for (int q = 0; q < kE; ++q) key[j][q] = order_bits(z[q]);
    } else {
#pragma unroll
      for (int q = 0; q < kE; ++q) {
        z[q] = -INFINITY;
        key[j][q] = 0u;
      }
    }
    // odd-even transposition: neighbours swap only when out of order, so equal values keep theirs
#pragma unroll
    for (int ph = 0; ph < kE; ++ph)
#pragma unroll
      for (int q = ph & 1; q + 1 < kE; q += 2) {
        const bool sw = key[j][q + 1] > key[j][q];
        const uint32_t k0 = key[j][q], i0 = id[q];
        key[j][q] = sw ? key[j][q + 1] : k0;
        key[j][q + 1] = sw ? k0 : key[j][q + 1];
        id[q] = sw ? id[q + 1] : i0;
        id[q + 1] = sw ? i0 : id[q + 1];
      }
    ids[j] = 0u;
#pragma unroll
    for (int q = 0; q < kE; ++q) ids[j] |= id[q] << (4 * q);
    head[j] = key[j][0];
#pragma unroll
    for (int q = 0; q < kE; ++q) zs[j][q] = z[q];
    my_z[j] = 0.f;
    my_e[j] = 0;
  }
  warp_max<kRB>(head);
#pragma unroll
  for (int j = 0; j < kRB; ++j) {
    mx[j] = fmaxf(order_value(head[j]), -FLT_MAX);
    sum[j] = 0.f;
    if (in)
#pragma unroll
      for (int q = 0; q < kE; ++q) sum[j] += expf(zs[j][q] - mx[j]);
  }
  warp_add<kRB>(sum);
  const int rounds = a.k < a.N ? a.k + 1 : a.k;
  for (int r = 0; r < rounds; ++r) {
    unsigned has[kRB];
    int e[kRB];
    if (r > 0) {
#pragma unroll
      for (int j = 0; j < kRB; ++j) head[j] = key[j][0];
      warp_max<kRB>(head);
    }
#pragma unroll
    for (int j = 0; j < kRB; ++j) has[j] = __ballot_sync(0xffffffffu, key[j][0] == head[j]);
#pragma unroll
    for (int j = 0; j < kRB; ++j)
      e[j] = __shfl_sync(0xffffffffu, lane * kE + static_cast<int>(ids[j] & 15u), __ffs(has[j]) - 1);
#pragma unroll
    for (int j = 0; j < kRB; ++j) {
      if (lane == r) {
        my_z[j] = order_value(head[j]);
        my_e[j] = e[j];
      }
      if (lane == e[j] / kE) {
#pragma unroll
        for (int q = 0; q < kE - 1; ++q) key[j][q] = key[j][q + 1];
        key[j][kE - 1] = 0u;
        ids[j] >>= 4;
      }
    }
  }
  float pr[kRB], sk[kRB], pk[kRB], pk1[kRB];
#pragma unroll
  for (int j = 0; j < kRB; ++j) {
    pr[j] = expf(my_z[j] - mx[j]) * (1.0f / sum[j]);
    sk[j] = lane < a.k ? pr[j] : 0.f;
  }
  if (a.norm) warp_add<kRB>(sk);
#pragma unroll
  for (int j = 0; j < kRB; ++j) pk[j] = __shfl_sync(0xffffffffu, pr[j], a.k - 1);
#pragma unroll
  for (int j = 0; j < kRB; ++j) pk1[j] = __shfl_sync(0xffffffffu, pr[j], a.k);  // k <= 8
  int ties = 0;
#pragma unroll
  for (int j = 0; j < kRB; ++j) {
    if (live[j] && lane < a.k) {
      a.idx_out[t[j] * a.k + lane] = my_e[j];
      a.gates[t[j] * a.k + lane] = a.norm ? pr[j] * (1.0f / sk[j]) : pr[j];
      if (count) atomicAdd(&hist[my_e[j]], 1);
    }
    ties += (live[j] && a.k < a.N && pk[j] - pk1[j] < (float)PR2_NEAR_TIE_GAP) ? 1 : 0;
  }
  return ties;
}

// kRB replay rows finished by one warp: row j's logits are N floats at rows[j] (lane l: experts
// kE l ..), lane s < k holds cached slot s in es[j] (-1: none, out of range or repeated).  Writes
// the gates (divided by their sum over the valid slots under PR2_F_NORMALIZE_TOPK) and, where
// asked for, the row of rho.
template <int kRB, int kE>
__device__ __forceinline__ void finish_replay_rows(const float* const (&rows)[kRB],
                                                   const int (&es)[kRB], const int64_t (&t)[kRB],
                                                   const bool (&live)[kRB], const RouteTcArgs& a) {
  const int lane = threadIdx.x & 31;
  const bool in = lane * kE < a.N;
  float z[kRB][kE];
  uint32_t head[kRB];
  float sum[kRB], g[kRB], sk[kRB];
#pragma unroll
  for (int j = 0; j < kRB; ++j) {
    float c = -FLT_MAX;
    if (in) {
      load_vec<kE>(rows[j] + lane * kE, z[j]);
    } else {
#pragma unroll
      for (int q = 0; q < kE; ++q) z[j][q] = -FLT_MAX;
    }
#pragma unroll
    for (int q = 0; q < kE; ++q) c = fmaxf(c, z[j][q]);
    head[j] = order_bits(c);
  }
  warp_max<kRB>(head);
#pragma unroll
  for (int j = 0; j < kRB; ++j) {
    const float mx = fmaxf(order_value(head[j]), -FLT_MAX);
    const float zg = es[j] >= 0 ? rows[j][es[j]] : 0.f;
    float part = 0.f;
#pragma unroll
    for (int q = 0; q < kE; q += 2) {
      z[j][q] = expf(z[j][q] - mx);
      z[j][q + 1] = expf(z[j][q + 1] - mx);
      part += z[j][q] + z[j][q + 1];
    }
    sum[j] = in ? part : 0.f;
    g[j] = es[j] >= 0 ? expf(zg - mx) : 0.f;
  }
  warp_add<kRB>(sum);
#pragma unroll
  for (int j = 0; j < kRB; ++j) sk[j] = g[j] = g[j] * (1.0f / sum[j]);
  if (a.norm) warp_add<kRB>(sk);
#pragma unroll
  for (int j = 0; j < kRB; ++j) {
    if (!live[j]) continue;
    if (lane < a.k) a.gates[t[j] * a.k + lane] = a.norm && sk[j] > 0.f ? g[j] * (1.0f / sk[j]) : g[j];
    if (a.logits_or_probs != nullptr && in) {
      const float inv = 1.0f / sum[j];
#pragma unroll
      for (int q = 0; q < kE; ++q) z[j][q] *= inv;
      store_vec<kE>(a.logits_or_probs + t[j] * a.N + lane * kE, z[j]);
    }
  }
}

// kRB rows of the predictive loss (Eq. pr2_loss, Algorithm 3) finished by one warp: row j's
// predictor logits b are N floats at rows[j] (lane l: experts kE l ..), its p_old and teacher
// values (row pos[t] of rho) po[j], tr[j]:
//   standard: prediction Softmax(v), v = p_old + b;  target rho
//   delta:    prediction Softmax(b);  target Softmax(u), u = log rho - p_old
// KL_t = sum_j tgt_j (log tgt_j - log pred_j);  dKL_t/dv_j = pred_j - tgt_j, rounded to bf16 and
// written to gs[j] (shared memory).  Exponentials and logarithms use the hardware approximations
// (__expf, __logf: a few ulp over the ranges met here, far inside the loss's tolerance).
template <int kRB, int kE>
__device__ __forceinline__ void finish_loss_rows(const float* const (&rows)[kRB],
                                                 const float (&po)[kRB][kE],
                                                 const float (&tr)[kRB][kE],
                                                 const bool (&use)[kRB], const int64_t (&t)[kRB],
                                                 uint32_t* const (&gs)[kRB], const RouteTcArgs& a) {
  const int lane = threadIdx.x & 31;
  const bool delta = a.delta != 0, in = lane * kE < a.N;
  float v[kRB][kE], lt[kRB][kE], tg[kRB][kE], s1[kRB], s2[kRB], kl[kRB];
  uint32_t m1[kRB], m2[kRB];  // row maxima (order_bits: no NaN among the candidates)
#pragma unroll
  for (int j = 0; j < kRB; ++j) {
    float c1 = -FLT_MAX, c2 = -FLT_MAX;
    float b[kE];
    if (in) {
      load_vec<kE>(rows[j] + lane * kE, b);
    } else {
#pragma unroll
      for (int q = 0; q < kE; ++q) b[q] = 0.f;
    }
#pragma unroll
    for (int q = 0; q < kE; ++q) {
      const bool ok = in && use[j];
      v[j][q] = ok ? (delta ? b[q] : po[j][q] + b[q]) : -INFINITY;
      tg[j][q] = ok ? tr[j][q] : 0.f;
      lt[j][q] = ok && tr[j][q] > 0.f ? __logf(tr[j][q]) - (delta ? po[j][q] : 0.f) : -INFINITY;
      c1 = fmaxf(c1, v[j][q]);
      c2 = fmaxf(c2, lt[j][q]);
    }
    m1[j] = order_bits(c1);
    m2[j] = order_bits(c2);
  }
  warp_max<kRB>(m1);
  if (delta) warp_max<kRB>(m2);
#pragma unroll
  for (int j = 0; j < kRB; ++j) {
    s1[j] = s2[j] = 0.f;
#pragma unroll
    for (int q = 0; q < kE; ++q) {
      s1[j] += __expf(v[j][q] - order_value(m1[j]));
      if (delta) s2[j] += __expf(lt[j][q] - order_value(m2[j]));
    }
  }
  warp_add<kRB>(s1);
  if (delta) warp_add<kRB>(s2);
#pragma unroll
  for (int j = 0; j < kRB; ++j) {
    const float l1 = order_value(m1[j]) + __logf(s1[j]);  // log normalisers
    const float l2 = delta ? order_value(m2[j]) + __logf(s2[j]) : 0.f;
    float g[kE];
    kl[j] = 0.f;
#pragma unroll
    for (int q = 0; q < kE; ++q) {
      const float lp = v[j][q] - l1;  // log prediction
      const float ltq = lt[j][q] - l2;
      const float tgt = delta ? (tg[j][q] > 0.f ? __expf(ltq) : 0.f) : tg[j][q];
      if (tgt > 0.f) kl[j] += tgt * (ltq - lp);
      g[q] = in && use[j] ? __expf(lp) - tgt : 0.f;
    }
    if (in)
#pragma unroll
      for (int q = 0; q < kE; q += 2) gs[j][q / 2] = pack_bf16x2(g[q], g[q + 1]);
  }
  warp_add<kRB>(kl);
#pragma unroll
  for (int j = 0; j < kRB; ++j)
    if (lane == 0 && t[j] < a.T) a.kl_tok[t[j]] = use[j] ? kl[j] : 0.f;
}

// kE: experts of a lane where rows are finished by warps (2, 4 or 8: N <= 32 kE); 0: by threads.
template <int kMode, int split, int kE>
__global__ void __launch_bounds__(kE > 0 ? kWarpThreads : kThreads, 1)
    route_tc_kernel(const __grid_constant__ CUtensorMap tm_h,
                    const __grid_constant__ CUtensorMap tm_w,
                    const __grid_constant__ CUtensorMap tm_wp, RouteTcArgs a) {
  constexpr bool predict = kMode == kModePredict;
  constexpr bool loss = kMode == kModeLoss;
  constexpr bool by_warps = kE > 0;
  extern __shared__ __align__(16) uint8_t smem_raw[];
  const int N = a.N, k = a.k;
  const RouteSmemLayout L = route_layout(N, kMode, split, a.compact != 0);
  // 1024-B aligned base, kept as an offset into the shared array so the compiler knows every
  // derived pointer is shared memory.
  const uint32_t pad = (1024u - (smem_u32(smem_raw) & 1023u)) & 1023u;
  uint8_t* smem = smem_raw + pad;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + L.bar_offset);
  uint64_t* empty = full + L.stages;
  uint64_t* acc_full = empty + L.stages;
  uint64_t* drain = acc_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int rank = split > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  const int t0 = (blockIdx.x / split) * kTileM;
  const int nb4 = L.b_rows / 4;             // float4 columns of a partial row
  // Pass split: predict whose weights stream in two passes (N > 128) run by a 2-CTA cluster in
  // which CTA r streams pass r ([W], then [W_p]) over all of K; the two column halves of every
  // row then meet in the CTA that finishes it and are not summed: half the exchange of a K split.
  const bool psplit = predict && L.passes == 2 && split == 2;
  const int KB = a.d / kBK;                 // K blocks, of which this CTA takes [kb0, kb1)
  const int kb0 = psplit ? 0 : rank * KB / split;
  const int kb1 = psplit ? KB : (rank + 1) * KB / split;
  const int npass = psplit ? 1 : L.passes;  // passes this CTA streams
  const int pass0 = psplit ? rank : 0;      // the first of them
  const uint32_t ncols = tmem_cols_for(L.acc_cols);

  if (threadIdx.x == 0) {
    for (int s = 0; s < L.stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tm_h);
    tma_prefetch_desc(&tm_w);
    if (predict) tma_prefetch_desc(&tm_wp);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, ncols);
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // h, the weights and the cached route may come from the previous kernels.  With late_wait
  // the caller guarantees they are complete already (the kernel before is a grouped GEMM whose
  // own inputs came after them), so the CTAs start on the SMs that GEMM frees and wait for it
  // only before they exit: a kernel launched after this one then sees the GEMM's results too.
  if (!a.late_wait) pdl_wait();
  pdl_trigger();

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer ----------------
      const uint32_t bytes = static_cast<uint32_t>(L.stage_bytes);
      uint32_t issued = 0, last_par = 0;
      int stage = 0;
      uint32_t phase = 0;
      const uint64_t keep = l2_policy_evict_last();    // weights are re-read by every tile
      const uint64_t once = l2_policy_evict_first();   // h is read once
      bool ok = true;
      for (int pass = pass0; pass < pass0 + npass && ok; ++pass)
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!mbar_wait(&empty[stage], phase ^ 1u, abort_flag, a.status)) {
          ok = false;
          break;
        }
        uint8_t* sa = smem + stage * L.stage_bytes;
        uint8_t* sb = sa + kATileBytes;
        mbar_arrive_expect_tx(&full[stage], bytes);
        tma_load_2d_hint(sa, &tm_h, &full[stage], kb * kBK, t0, once);
        if (!predict || L.passes == 1) {  // replay never takes two passes
          tma_load_2d_hint(sb, &tm_w, &full[stage], kb * kBK, 0, keep);
          if (predict) tma_load_2d_hint(sb + N * kBK * 2, &tm_wp, &full[stage], kb * kBK, 0, keep);
        } else if (pass == 0) {
          // Each map is named directly: with one pointer selected between the two maps here,
          // even the replay kernel's mainloop (which never gets here) ran 25 % slower.
          tma_load_2d_hint(sb, &tm_w, &full[stage], kb * kBK, 0, keep);
        } else {
          tma_load_2d_hint(sb, &tm_wp, &full[stage], kb * kBK, 0, keep);
        }
        issued |= 1u << stage;
        last_par = (last_par & ~(1u << stage)) | (phase << stage);
        if (++stage == L.stages) {
          stage = 0;
          phase ^= 1u;
        }
      }
      // Drain: every issued copy must have landed before the stages are reused or the CTA exits.
      for (int s = 0; s < L.stages; ++s)
        if ((issued >> s) & 1u)
          mbar_wait_slow(&full[s], (last_par >> s) & 1u, nullptr, nullptr, kDrainLimitNs);
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      // ---------------- MMA issuer ----------------
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int pass = pass0; pass < pass0 + npass && ok; ++pass)
      for (int kb = kb0; kb < kb1 && ok; ++kb) {
        if (!mbar_wait(&full[stage], phase, abort_flag, a.status)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t sa = smem_u32(smem + stage * L.stage_bytes);
        const uint32_t sb = sa + kATileBytes;
#pragma unroll
        for (int kk = 0; kk < kBK / 16; ++kk) {
          const uint64_t adesc = umma_desc_sw128(sa + kk * 32);
          const uint32_t acc = (kb > kb0 || kk > 0) ? 1u : 0u;
          if (!predict || L.passes == 1) {  // replay never takes two passes
            for (int n0 = 0; n0 < L.b_rows; n0 += 256) {
              const int nc = (L.b_rows - n0) < 256 ? (L.b_rows - n0) : 256;
              const uint64_t bdesc = umma_desc_sw128(sb + n0 * (kBK * 2) + kk * 32);
              umma_bf16(tmem + n0, adesc, bdesc, umma_idesc_bf16(kTileM, nc), acc);
            }
          } else {  // pass p fills accumulator columns [p N, (p + 1) N): p_old, then b
            umma_bf16(tmem + (psplit ? 0 : pass * L.pass_rows), adesc,
                      umma_desc_sw128(sb + kk * 32), umma_idesc_bf16(kTileM, L.pass_rows), acc);
          }
        }
        umma_commit(&empty[stage]);
        if (++stage == L.stages) {
          stage = 0;
          phase ^= 1u;
        }
      }
      if (ok) umma_commit(acc_full);
      umma_commit(drain);
      mbar_wait_slow(drain, 0, nullptr, nullptr, kDrainLimitNs);
    }
    __syncwarp();
  }

  // ---------------- epilogue ----------------
  const bool epi = warp >= 2 && warp < 6;
  // predict: experts of the rows this CTA finishes, for the dispatch that follows
  __shared__ int hist_s[kMaxExperts];
  const bool count = predict && a.hist != nullptr;
  if (count && epi) {  // (by warps: the barriers below order it before the counting)
    for (int e = threadIdx.x - 64; e < N; e += 128) hist_s[e] = 0;
    if (!by_warps) named_bar_sync(1, 128);
  }
  const int q = warp & 3;
  const int row = q * 32 + lane;  // TMEM lane of this thread
  const uint32_t trow = tmem + (static_cast<uint32_t>(q * 32) << 16);
  const int64_t t = static_cast<int64_t>(t0) + row;  // split = 1: this thread's row
  const bool live = epi && t < a.T;

  // replay: cached indices, validated (range, duplicates) while the K blocks run
  int e_s[kMaxTopK];
  bool bad = false;
  if (kMode == kModeReplay && !by_warps) {
#pragma unroll
    for (int s = 0; s < kMaxTopK; ++s) {
      int e = -1;
      if (live && s < k) {
        e = a.idx_in[t * k + s];
        bool ok = e >= 0 && e < N;
#pragma unroll
        for (int s2 = 0; s2 < kMaxTopK; ++s2)
          if (s2 < s && e_s[s2] == e) ok = false;
        if (!ok) {
          bad = true;
          e = -1;
        }
      }
      e_s[s] = e;
    }
  }

  // finished by warps: the CTA's kR rows, frows of them at once, fper of those by each warp, kRB
  // at a time; replay: cached slot `lane` of each row, -1 if it does not count; loss: p_old and
  // teacher values (row pos[t] of rho).  The first kRB rows' are loaded while the K blocks run.
  constexpr int kR = kTileM / split;
  constexpr int kRows = kR / (kWarpThreads / 32);
  constexpr int kLane = by_warps ? kE : 2;
  constexpr int kHeld = loss && split < 4 ? 8 : 16;  // logits a lane holds at once (registers)
  constexpr int kRB = kRows * kLane > kHeld ? kHeld / kLane : kRows;
  const int frows = split > 1 ? kR : L.frows, fper = split > 1 ? kRows : L.frows / 16;
  const int64_t tc = static_cast<int64_t>(t0) + rank * kR;  // token of the CTA's row 0
  float po_w[kRB][kLane], tr_w[kRB][kLane];
  bool use_w[kRB];
  int es_w[kRB];
  auto load_rows = [&](int r0) {  // of the CTA's rows r0 .. r0 + kRB - 1
    if constexpr (kMode == kModeReplay) {
      bool wrong = false;
#pragma unroll
      for (int j = 0; j < kRB; ++j) {
        const bool in = tc + r0 + j < a.T && lane < k;
        es_w[j] = in ? a.idx_in[(tc + r0 + j) * k + lane] : -1;
      }
#pragma unroll
      for (int j = 0; j < kRB; ++j) {
        const int e = es_w[j];
        bool ok = e >= 0 && e < N;
#pragma unroll
        for (int s2 = 0; s2 < kMaxTopK - 1; ++s2) {
          // a repeat counts against its later slot; an entry out of range repeats nothing
          const int other = __shfl_sync(0xffffffffu, e, s2);
          if (s2 < lane && other == e) ok = false;
        }
        wrong = wrong || (tc + r0 + j < a.T && lane < k && !ok);
        if (!ok) es_w[j] = -1;
      }
      if (wrong && a.status != nullptr) atomicOr(a.status, PR2_STATUS_BAD_INDEX);
    }
    if constexpr (loss) {
      int32_t pw[kRB];
#pragma unroll
      for (int j = 0; j < kRB; ++j)
        pw[j] = tc + r0 + j < a.T && a.pos != nullptr ? a.pos[tc + r0 + j] : 0;
#pragma unroll
      for (int j = 0; j < kRB; ++j) {
        const int64_t tj = tc + r0 + j;
        const int64_t r = a.pos != nullptr ? static_cast<int64_t>(pw[j]) : tj;
        use_w[j] = tj < a.T && r >= 0 && r < a.T_rho;
        if (tj < a.T && !use_w[j] && lane == 0 && a.status != nullptr)
          atomicOr(a.status, PR2_STATUS_BAD_INDEX);
#pragma unroll
        for (int c = 0; c < kLane; ++c) po_w[j][c] = tr_w[j][c] = 0.f;
        if (use_w[j] && lane * kLane < N) {
          load_vec<kLane>(a.p_old + tj * N + lane * kLane, po_w[j]);
          load_vec<kLane>(a.rho + r * N + lane * kLane, tr_w[j]);
        }
      }
    }
  };
  if (by_warps) load_rows(warp * fper);
  bool have = false;
  if (epi || by_warps) {
    // tcgen05.ld is warp-collective: the whole warp reads TMEM or none of it does.
    have = __all_sync(0xffffffffu, mbar_wait(acc_full, 0, abort_flag, a.status));
    if (have) tc_fence_after();
  }
  // Columns [c, c + 16) of this thread's row.
  auto load16 = [&](int c, uint32_t (&r)[16]) {
    tmem_ld16(trow + c, r);
    tmem_wait_ld(r);
  };

  if constexpr (by_warps) {
    const int pitch = (nb4 + 1) * 4;  // floats of a row: 8 rows in turn take 8 bank groups
    float4* recv = reinterpret_cast<float4*>(smem);  // [S][columns of a round / 4][kR]
    float* rm = reinterpret_cast<float*>(smem + L.xcols * kTileM * 4);  // the rows in row order
    if constexpr (split > 1) {
      // Reduce-scatter by rows: this TMEM row goes to CTA row / kR as its row row % kR, into the
      // slot of source `rank`; the four warps of a lane quadrant share its columns.  Rows beyond
      // the batch are not moved (a decode batch fills a few rows of its tile); a warp of such
      // rows skips its loads too.
      const uint32_t dst = static_cast<uint32_t>(row / kR);
      const bool in_batch = static_cast<int64_t>(t0) + row < a.T;
      const bool move = have && static_cast<int64_t>(t0) + q * 32 < a.T;
      for (int x0 = 0; x0 < L.acc_cols; x0 += L.xcols) {
        const int xn = L.acc_cols - x0 < L.xcols ? L.acc_cols - x0 : L.xcols;
        cluster_sync();  // every CTA is done with its K blocks (the round before): recv is free
        if (move) {
          const uint32_t rbase = mapa_shared(
              smem_u32(recv + rank * (xn / 4) * kR + (row - static_cast<int>(dst) * kR)), dst);
          for (int c0 = (warp >> 2) * 32; c0 < xn; c0 += 32 * (kWarpThreads / 128)) {
            uint32_t r0[16], r1[16];
            const bool two = c0 + 16 < xn;  // a multiple of 16, not always of 32
            tmem_ld16(trow + x0 + c0, r0);
            if (two) tmem_ld16(trow + x0 + c0 + 16, r1);
            tmem_wait_ld(r0);
            if (two) reg_fence(r1);
            if (in_batch) {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                st_cluster_v4(rbase + static_cast<uint32_t>(((c0 / 4 + j) * kR) * 16), r0[4 * j],
                              r0[4 * j + 1], r0[4 * j + 2], r0[4 * j + 3]);
            }
            if (two && in_batch) {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                st_cluster_v4(rbase + static_cast<uint32_t>(((c0 / 4 + 4 + j) * kR) * 16), r1[4 * j],
                              r1[4 * j + 1], r1[4 * j + 2], r1[4 * j + 3]);
            }
          }
        }
        cluster_sync();  // every partial row has landed
        // all sixteen warps bring the copies into row order: summed once, in source order, or
        // (pass split) source 1's columns behind source 0's
        const int n4 = (xn / 4) * kR;
        for (int i = threadIdx.x; i < n4; i += kWarpThreads) {
          float4 v = recv[i];
          float4* to = reinterpret_cast<float4*>(rm + (i % kR) * pitch) + x0 / 4 + i / kR;
          if (psplit) {
            to[N / 4] = recv[n4 + i];
          } else {
#pragma unroll
            for (int src = 1; src < split; ++src) {
              const float4 w = recv[src * n4 + i];
              v.x += w.x;
              v.y += w.y;
              v.z += w.z;
              v.w += w.w;
            }
          }
          *to = v;
        }
      }
    }
    // the bf16 dKL/dz rows (loss) meet in shared memory
    uint8_t* gsb = reinterpret_cast<uint8_t*>(rm + frows * pitch);
    const int gpitch = N * 2 + 8;
    int ties = 0;
    for (int f0 = 0; f0 < kR; f0 += frows) {  // rows f0 .. f0 + frows - 1 of the CTA
      __syncthreads();  // split = 1: every K block, copy and earlier row is done with the stages
      if constexpr (split == 1) {
        if (have && row >= f0 && row < f0 + frows) {  // whole warps: frows is 64 or 128
          float4* to = reinterpret_cast<float4*>(rm + (row - f0) * pitch);
          for (int c0 = (warp >> 2) * 16; c0 < L.b_rows; c0 += 16 * (kWarpThreads / 128)) {
            uint32_t r[16];
            tmem_ld16(trow + c0, r);
            tmem_wait_ld(r);
#pragma unroll
            for (int j = 0; j < 4; ++j)
              to[c0 / 4 + j] =
                  make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]),
                              __uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3]));
          }
        }
        __syncthreads();
      }
      const bool good = *abort_flag == 0;
      for (int j0 = 0; j0 < fper; j0 += kRB) {
        const int fr = warp * fper + j0;  // of the frows rows in shared memory
        if (f0 > 0 || j0 > 0) load_rows(f0 + fr);
        const float* rows[kRB];
        int64_t ts[kRB];
        bool lv[kRB];
#pragma unroll
        for (int j = 0; j < kRB; ++j) {
          rows[j] = rm + (fr + j) * pitch;
          ts[j] = tc + f0 + fr + j;
          lv[j] = good && ts[j] < a.T;
        }
        if constexpr (predict) {
          if (good && ts[0] < a.T)
            ties += finish_predict_rows<kRB, kLane>(rows, ts, lv, a, count, hist_s);
        } else if constexpr (kMode == kModeReplay) {
          if (ts[0] < a.T) finish_replay_rows<kRB, kLane>(rows, es_w, ts, lv, a);
        } else {
          uint32_t* gs[kRB];
#pragma unroll
          for (int j = 0; j < kRB; ++j) {
            gs[j] = reinterpret_cast<uint32_t*>(gsb + (fr + j) * gpitch + lane * (kLane * 2));
            use_w[j] = use_w[j] && good;
          }
          finish_loss_rows<kRB, kLane>(rows, po_w, tr_w, use_w, ts, gs, a);
        }
      }
      if constexpr (loss) {
        // ... and leave transposed, 2 frows bytes per expert: thread (e, part) 8 rows of expert e
        __syncthreads();
        const int parts = frows / 8;
        for (int i = threadIdx.x; i < N * parts; i += kWarpThreads) {
          const int e = i / parts, r0 = i % parts * 8;
          uint32_t w[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const uint8_t* at = gsb + (r0 + 2 * r) * gpitch + e * 2;
            w[r] = *reinterpret_cast<const uint16_t*>(at) |
                   static_cast<uint32_t>(*reinterpret_cast<const uint16_t*>(at + gpitch)) << 16;
          }
          *reinterpret_cast<uint4*>(a.gt + static_cast<int64_t>(e) * a.Tpad + tc + f0 + r0) =
              make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
    }
    if constexpr (predict) {
      if (lane == 0 && ties != 0 && a.near_tie != nullptr)
        atomicAdd(reinterpret_cast<unsigned long long*>(a.near_tie),
                  static_cast<unsigned long long>(ties));
      if (count) {  // every row of this CTA counted: publish its histogram row (zeros included)
        __syncthreads();
        int32_t* hrow = a.hist + static_cast<int64_t>(blockIdx.x) * N;
        for (int e = threadIdx.x; e < N; e += kWarpThreads) hrow[e] = hist_s[e];
      }
    }
    tc_fence_before();
  }
  // One pass over this thread's experts, 16 at a time: running max m and sum of exp(z - m),
  // (predict) the top-16 keys, (replay) the z of the cached slots.
  if (epi && !loss && !by_warps) {
    bool tie = false;
    float m = -FLT_MAX, sum = 0.f;
    uint64_t top[16];
    float z_s[kMaxTopK];
#pragma unroll
    for (int j = 0; j < 16; ++j) top[j] = 0ull;
#pragma unroll
    for (int s = 0; s < kMaxTopK; ++s) z_s[s] = 0.f;
    if (have) {
      float* lrow = (predict && a.logits_or_probs != nullptr && live) ? a.logits_or_probs + t * N
                                                                      : nullptr;
      for (int c0 = 0; c0 < N; c0 += 16) {
        float z[16];
        if (predict) {
          uint32_t rp[16], rb[16];
          load16(c0, rp);
          load16(N + c0, rb);
          if (lrow != nullptr) {
            float4* dst = reinterpret_cast<float4*>(lrow + c0);
#pragma unroll
            for (int j = 0; j < 4; ++j)
              dst[j] = make_float4(__uint_as_float(rp[4 * j]), __uint_as_float(rp[4 * j + 1]),
                                   __uint_as_float(rp[4 * j + 2]), __uint_as_float(rp[4 * j + 3]));
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) z[j] = __uint_as_float(rp[j]) + __uint_as_float(rb[j]);
        } else {
          uint32_t rp[16];
          load16(c0, rp);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            z[j] = __uint_as_float(rp[j]);
#pragma unroll
            for (int s = 0; s < kMaxTopK; ++s)
              if (e_s[s] == c0 + j) z_s[s] = z[j];
          }
        }
        float cm = z[0];
#pragma unroll
        for (int j = 1; j < 16; ++j) cm = fmaxf(cm, z[j]);
        const float nm = fmaxf(m, cm);
        float cs = 0.f;
#pragma unroll
        for (int j = 0; j < 16; ++j) cs += expf(z[j] - nm);
        sum = sum * expf(m - nm) + cs;
        m = nm;
        if (predict) {
          uint64_t ck[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) ck[j] = topk_key(z[j], c0 + j);
          sort16_desc(ck);
          merge16_desc(top, ck);
        }
      }
    }
    const float mx = m;
    const float inv_s = 1.0f / sum;
    if (predict) {
      if (have && live) {
        tie = predict_write(top, mx, inv_s, t, a);
        if (count)
#pragma unroll
          for (int j = 0; j < kMaxTopK; ++j)
            if (j < k) atomicAdd(&hist_s[key_e(top[j])], 1);
      }
    } else if (!loss) {
      if (have && live) {
        float* grow = a.gates + t * k;
        float gv[kMaxTopK];
        float sk = 0.f;
#pragma unroll
        for (int s = 0; s < kMaxTopK; ++s) {
          gv[s] = (s < k && e_s[s] >= 0) ? expf(z_s[s] - mx) * inv_s : 0.f;
          sk += gv[s];
        }
        const float sc = (a.norm && sk > 0.f) ? 1.0f / sk : 1.0f;  // over the valid slots
#pragma unroll
        for (int s = 0; s < kMaxTopK; ++s)
          if (s < k) grow[s] = gv[s] * sc;
        if (bad && a.status != nullptr) atomicOr(a.status, PR2_STATUS_BAD_INDEX);
      }
      if (have && a.logits_or_probs != nullptr) {
        float* prow = a.logits_or_probs + t * N;
        for (int c0 = 0; c0 < N; c0 += 16) {
          uint32_t rp[16];
          load16(c0, rp);
          if (live) {
            float4* dst = reinterpret_cast<float4*>(prow + c0);
#pragma unroll
            for (int j = 0; j < 4; ++j)
              dst[j] = make_float4(expf(__uint_as_float(rp[4 * j]) - mx) * inv_s,
                                   expf(__uint_as_float(rp[4 * j + 1]) - mx) * inv_s,
                                   expf(__uint_as_float(rp[4 * j + 2]) - mx) * inv_s,
                                   expf(__uint_as_float(rp[4 * j + 3]) - mx) * inv_s);
          }
        }
      }
    }
    const unsigned ties = __ballot_sync(0xffffffffu, tie);
    if (lane == 0 && ties != 0u && a.near_tie != nullptr)
      atomicAdd(reinterpret_cast<unsigned long long*>(a.near_tie),
                static_cast<unsigned long long>(__popc(ties)));
    if (count) {  // every row of this CTA counted: publish its histogram row (zeros included)
      named_bar_sync(1, 128);
      int32_t* hrow = a.hist + static_cast<int64_t>(blockIdx.x) * N;
      for (int e = threadIdx.x - 64; e < N; e += 128) hrow[e] = hist_s[e];
    }
    tc_fence_before();
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, ncols);
  }
  if (a.late_wait) pdl_wait();
}

// The limit is the kernel's, not the launch's: the same for every shape, so that a call of another
// shape on another host thread cannot lower it between this and a launch.
template <int kMode, int kSplit, int kE>
cudaError_t set_smem_attr() {
  const cudaError_t err = cudaFuncSetAttribute(
      route_tc_kernel<kMode, kSplit, kE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSmem);
  if (err != cudaSuccess) return err;
  // all of the SM's unified L1 / shared storage as shared memory, so that two compact CTAs fit
  return cudaFuncSetAttribute(route_tc_kernel<kMode, kSplit, kE>,
                              cudaFuncAttributePreferredSharedMemoryCarveout,
                              cudaSharedmemCarveoutMaxShared);
}

template <int kMode, int kSplit, int kE>
cudaError_t launch_kernel(const CUtensorMap& tm_h, const CUtensorMap& tm_w,
                          const CUtensorMap& tm_wp, const RouteTcArgs& a, int tiles,
                          cudaStream_t st, int* max_clusters) {
  if (kE > 0 && a.compact != 0) return cudaErrorInvalidValue;  // no room for the rows
  cudaError_t err = set_smem_attr<kMode, kSplit, kE>();
  if (err != cudaSuccess) return err;
  const int smem = route_layout(a.N, kMode, kSplit, a.compact != 0).total;
  if (smem > kMostSmem) return cudaErrorInvalidValue;
  const dim3 block(kE > 0 ? kWarpThreads : kThreads);
  if (max_clusters != nullptr) {  // occupancy query only
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(tiles * kSplit);
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kSplit;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(max_clusters, route_tc_kernel<kMode, kSplit, kE>,
                                          &cfg);
  }
  return launch_pdl(route_tc_kernel<kMode, kSplit, kE>, dim3(tiles * kSplit), block, smem, st,
                    kSplit, tm_h, tm_w, tm_wp, a);
}

template <int kMode, int kSplit>
cudaError_t launch_split(const CUtensorMap& tm_h, const CUtensorMap& tm_w,
                         const CUtensorMap& tm_wp, const RouteTcArgs& a, int tiles,
                         cudaStream_t st, int* max_clusters) {
  if constexpr (kSplit == 1 && kMode != kModeLoss)
    if (a.compact != 0 || a.N <= 128)
      return launch_kernel<kMode, 1, 0>(tm_h, tm_w, tm_wp, a, tiles, st, max_clusters);
  if (a.N > 128)
    return launch_kernel<kMode, kSplit, 8>(tm_h, tm_w, tm_wp, a, tiles, st, max_clusters);
  if (a.N > 64)
    return launch_kernel<kMode, kSplit, 4>(tm_h, tm_w, tm_wp, a, tiles, st, max_clusters);
  return launch_kernel<kMode, kSplit, 2>(tm_h, tm_w, tm_wp, a, tiles, st, max_clusters);
}

template <int kMode>
cudaError_t launch_splits(const CUtensorMap& tm_h, const CUtensorMap& tm_w,
                          const CUtensorMap& tm_wp, const RouteTcArgs& a, int split, int tiles,
                          cudaStream_t st, int* max_clusters) {
  switch (split) {
    case 1: return launch_split<kMode, 1>(tm_h, tm_w, tm_wp, a, tiles, st, max_clusters);
    case 2: return launch_split<kMode, 2>(tm_h, tm_w, tm_wp, a, tiles, st, max_clusters);
    case 4: return launch_split<kMode, 4>(tm_h, tm_w, tm_wp, a, tiles, st, max_clusters);
    case 8: return launch_split<kMode, 8>(tm_h, tm_w, tm_wp, a, tiles, st, max_clusters);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_any(int mode, const CUtensorMap& tm_h, const CUtensorMap& tm_w,
                       const CUtensorMap& tm_wp, const RouteTcArgs& a, int split, int tiles,
                       cudaStream_t st, int* max_clusters) {
  switch (mode) {
    case kModeReplay:
      return launch_splits<kModeReplay>(tm_h, tm_w, tm_wp, a, split, tiles, st, max_clusters);
    case kModePredict:
      return launch_splits<kModePredict>(tm_h, tm_w, tm_wp, a, split, tiles, st, max_clusters);
    case kModeLoss:
      return launch_splits<kModeLoss>(tm_h, tm_w, tm_wp, a, split, tiles, st, max_clusters);
    default: return cudaErrorInvalidValue;
  }
}

// CTAs of route_tc_kernel<mode, 1> with the compact layout that fit on one SM by its shared
// memory, registers, threads and TMEM columns (0 on error).  Counted from the kernel's attributes and the
// device limits: the occupancy query answers 1 for this kernel although two CTAs do run on
// one SM side by side (a per-CTA %smid / %globaltimer record of a T = 32768 launch).
template <int kMode>
int compact_blocks_per_sm(int N) {
  if (set_smem_attr<kMode, 1, 0>() != cudaSuccess) return 0;
  cudaFuncAttributes fa{};
  if (cudaFuncGetAttributes(&fa, route_tc_kernel<kMode, 1, 0>) != cudaSuccess) return 0;
  int dev = 0, smem_sm = 0, reserved = 0, regs_sm = 0, threads_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) !=
          cudaSuccess ||
      cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) !=
          cudaSuccess ||
      cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev) !=
          cudaSuccess ||
      cudaDeviceGetAttribute(&threads_sm, cudaDevAttrMaxThreadsPerMultiProcessor, dev) !=
          cudaSuccess)
    return 0;
  const size_t smem = route_layout(N, kMode, 1, true).total + fa.sharedSizeBytes +
                      static_cast<size_t>(reserved);
  const int regs = ((fa.numRegs + 7) / 8) * 8 * kThreads;  // allocated per warp in 256s
  int n = static_cast<int>(static_cast<size_t>(smem_sm) / smem);
  if (regs > 0 && regs_sm / regs < n) n = regs_sm / regs;
  if (threads_sm / kThreads < n) n = threads_sm / kThreads;
  // each CTA holds its accumulator columns for its whole life: more CTAs than fit in the SM's
  // 512 TMEM columns would only wait in tcgen05.alloc for a neighbour to leave
  const int b_rows = route_layout(N, kMode, 1, true).b_rows;
  const int by_tmem = static_cast<int>(512u / tmem_cols_for(b_rows));
  if (by_tmem < n) n = by_tmem;
  return n;
}

// Clusters of `split` CTAs of this kernel that can be resident at once (0 on error), cached
// per device and shape.
int max_active_clusters(int mode, int split, int N, bool compact = false) {
  struct Entry {
    int dev, mode, split, N, compact, clusters;
  };
  static std::mutex mu;
  static Entry cache[64];
  static int used = 0;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  std::lock_guard<std::mutex> lock(mu);
  for (int i = 0; i < used; ++i)
    if (cache[i].dev == dev && cache[i].mode == mode && cache[i].split == split &&
        cache[i].N == N && cache[i].compact == static_cast<int>(compact))
      return cache[i].clusters;
  int clusters = 0;
  if (compact) {  // clusters of one CTA: CTAs per SM, times the SMs
    const int per_sm = mode == kModePredict ? compact_blocks_per_sm<kModePredict>(N)
                                            : compact_blocks_per_sm<kModeReplay>(N);
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess)
      clusters = per_sm * sms;
    (void)cudaGetLastError();
  } else {
    RouteTcArgs probe{};
    probe.N = N;
    CUtensorMap none{};
    const cudaError_t err =
        launch_any(mode, none, none, none, probe, split, 1, nullptr, &clusters);
    if (err != cudaSuccess) {
      (void)cudaGetLastError();
      clusters = 0;
    }
  }
  if (used < 64) cache[used++] = Entry{dev, mode, split, N, static_cast<int>(compact), clusters};
  return clusters;
}

}  // namespace

bool route_compact(int T, int N, int mode, int num_sms) {
  const int tiles = (T + kTileM - 1) / kTileM;
  if (tiles <= num_sms) return false;
  const RouteSmemLayout L = route_layout(N, mode, 1, true);
  if (L.stages * L.stage_bytes > kCompactBudget) return false;  // not even two stages fit
  if (2 * tmem_cols_for(L.b_rows) > 512) return false;           // two accumulators in TMEM
  return max_active_clusters(mode, 1, N, true) >= 2 * num_sms;
}

// The widest cluster whose CTAs are all resident at once and have at least one K block each.
int route_split(int T, int N, int d, int mode, int num_sms) {
  const int tiles = (T + kTileM - 1) / kTileM;
  for (int s = kMaxSplit; s > 1; s >>= 1) {
    if (d / kBK < s || tiles * s > num_sms) continue;
    if (max_active_clusters(mode, s, N) < tiles) continue;  // must fit in one wave
    return s;
  }
  return 1;
}

cudaError_t launch_route_tc(int mode, const CUtensorMap& tm_h, const CUtensorMap& tm_w,
                            const CUtensorMap& tm_wp, const RouteTcArgs& a, int split,
                            cudaStream_t st) {
  if (a.T == 0) return cudaSuccess;
  if (split < 1 || split > kMaxSplit || a.d / kBK < split || (a.compact != 0 && split != 1))
    return cudaErrorInvalidValue;
  const int tiles = (a.T + kTileM - 1) / kTileM;
  return launch_any(mode, tm_h, tm_w, tm_wp, a, split, tiles, st, nullptr);
}

}  // namespace pr2
