// fp32 grouped expert GEMMs (exact fp32 FMA; the fp32 layer needs a 1e-4 tolerance, which
// TF32 tensor cores cannot meet).  Same tile table as the tensor-core path.
//   gate/up: H[r, c] = silu(X[r] . Wg_e[c]) * (X[r] . Wu_e[c])      (App. E.2, SwiGLU)
//   down:    Y[r, c] = H[r] . Wd_e[c]
// A block computes BM rows x BN columns of one M-tile.  Both operands are K-contiguous, so K
// blocks of the rows and of the weight rows travel as 16-byte cp.async copies through a ring of
// kStages stages in shared memory (the routed gate/up GEMM gathers its rows from h through perm
// here: no permuted copy of h exists), and a thread accumulates a TM x TN register tile (twice
// for gate and up) from float4 reads along K.  The row pitch of BK + 4 floats puts the 16-byte
// words of eight consecutive rows on distinct banks.  K that is not a multiple of 4 (a ragged
// expert width) copies 4 bytes at a time instead, its rows being unaligned.  Every output is one
// chain of FMAs in ascending K.
//
// What bounds it: the FMA issue rate for large layers, and the chain of K blocks at small ones;
// hence two tile sizes (launch_expert_simt).  A rollout + replay step of the T = 256, d = 128,
// m = 256, N = 8, k = 2 layer took 79 us when only these kernels had changed and 5203 us with one thread
// per output column walking its weight row by uncoalesced 4-byte loads for every row of the
// tile, behind a launch that wrote a permuted copy of h.
#include "pr2_device.cuh"
#include "pr2_internal.h"

namespace pr2 {
namespace {

constexpr int kStages = 3;

template <int BM, int BN, int TM, int TN, int BK, bool kSwiglu>
struct SimtTile {
  static constexpr int kThreads = (BM / TM) * (BN / TN);
  static constexpr int kRows = BM + BN * (kSwiglu ? 2 : 1);  // A rows, then weight rows
  static constexpr int kPitch = BK + 4;
  static constexpr int kVecs = kRows * (BK / 4);             // 16-byte words of a stage
  static constexpr int kLoads = kVecs / kThreads;
  static constexpr int kStageFloats = kRows * kPitch;
  static constexpr int kSmem = kStages * kStageFloats * 4;
  static_assert(kVecs % kThreads == 0 && BM % 8 == 0 && BN % 8 == 0, "whole rounds of copies");
  static_assert(kSmem <= 48 * 1024, "static shared memory");
};

template <int BM, int BN, int TM, int TN, int BK, bool kSwiglu>
__global__ void __launch_bounds__((SimtTile<BM, BN, TM, TN, BK, kSwiglu>::kThreads))
    expert_simt_kernel(SimtArgs g, int col_blocks) {
  using S = SimtTile<BM, BN, TM, TN, BK, kSwiglu>;
  __shared__ __align__(16) float smem[kStages * S::kStageFloats];
  constexpr int kSub = kMinTileRows / BM;  // row blocks of one M-tile
  pdl_wait();
  pdl_trigger();
  // mt < max_tiles by the grid; a dispatch that timed out leaves the table unwritten.  The three
  // loads are in flight together.
  const int row_block = static_cast<int>(blockIdx.x) / col_blocks;
  const int mt = row_block / kSub;
  const int nm = *g.num_tiles;
  const TileEntry te = g.tiles[mt];
  if (status_timed_out(g.status) || mt >= nm) return;
  const int K = g.K, n_out = g.n_out;
  const float* __restrict__ A = g.A;
  const bool shared = te.expert >= g.N;
  const float* __restrict__ W0 = shared ? g.S0 : g.W0;
  const float* __restrict__ W1 = shared ? g.S1 : g.W1;
  const int64_t wrow0 = static_cast<int64_t>(shared ? te.expert - g.N : te.expert) * n_out;
  const int r0 = (row_block % kSub) * BM;
  if (r0 >= te.rows) return;
  const int c0 = (static_cast<int>(blockIdx.x) % col_blocks) * BN;
  // row numbers are 32 unsigned bits (TileEntry); times unsigned lengths, one wide multiply each
  const uint32_t out_row0 = static_cast<uint32_t>(te.out_row0);
  const int tid = threadIdx.x;
  const bool vec = K % 4 == 0;  // rows of 16-byte words (every base is 16-byte aligned)

  // This thread's copies of a stage: row kRow of [A rows; W0 rows; W1 rows], words kc.. of it.
  const float* src[S::kLoads];
  uint32_t on = 0;
#pragma unroll
  for (int i = 0; i < S::kLoads; ++i) {
    const int v = tid + i * S::kThreads;
    const int row = v / (BK / 4), kc = (v % (BK / 4)) * 4;
    src[i] = A;
    if (row < BM) {
      if (r0 + row < te.rows) {
        // gate/up: the token at this place (shared experts: the token itself); down: its H row
        const uint32_t p = (kSwiglu ? static_cast<uint32_t>(te.a_row0) : out_row0) + (r0 + row);
        const uint32_t at = kSwiglu && !shared ? static_cast<uint32_t>(g.perm[p] / g.k) : p;
        src[i] = A + static_cast<uint64_t>(at) * static_cast<uint32_t>(K) + kc;
        on |= 1u << i;
      }
    } else {
      const int c = c0 + (row - BM) % BN;
      if (c < n_out) {
        src[i] = (row - BM < BN ? W0 : W1) + (wrow0 + c) * K + kc;
        on |= 1u << i;
      }
    }
  }
  const uint32_t sbase = smem_u32(smem);
  auto issue = [&](int kb) {
    const uint32_t st = sbase + static_cast<uint32_t>(kb % kStages) * S::kStageFloats * 4;
    const int k0 = kb * BK;
#pragma unroll
    for (int i = 0; i < S::kLoads; ++i) {
      const int v = tid + i * S::kThreads;
      const int row = v / (BK / 4), kc = (v % (BK / 4)) * 4;
      const uint32_t dst = st + static_cast<uint32_t>(row * S::kPitch + kc) * 4;
      const bool live = (on >> i) & 1u;
      if (vec) {
        const bool in = live && k0 + kc < K;
        cp_async_16(dst, in ? src[i] + k0 : A, in ? 16u : 0u);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const bool in = live && k0 + kc + j < K;
          cp_async_4(dst + 4 * j, in ? src[i] + k0 + j : A, in ? 4u : 0u);
        }
      }
    }
  };

  // Threads of a warp: 8 columns x 4 rows, so that a warp's reads of a stage touch eight
  // consecutive weight rows and four consecutive A rows.
  constexpr int kTx = BN / TN, kTy = BM / TM;
  constexpr int kWx = kTx / 8;
  const int lane = tid & 31, warp = tid >> 5;
  const int tx = (lane & 7) + 8 * (warp % kWx);
  const int ty = (lane >> 3) + 4 * (warp / kWx);
  float acc0[TM][TN], acc1[kSwiglu ? TM : 1][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      acc0[i][j] = 0.f;
      if (kSwiglu) acc1[i][j] = 0.f;
    }
  const int KB = (K + BK - 1) / BK;
#pragma unroll
  for (int s = 0; s < kStages - 1; ++s) {
    if (s < KB) issue(s);
    cp_async_commit();
  }
  for (int kb = 0; kb < KB; ++kb) {
    cp_async_wait<kStages - 2>();
    __syncthreads();  // stage kb has landed for every thread, stage kb - 1 is free
    if (kb + kStages - 1 < KB) issue(kb + kStages - 1);
    cp_async_commit();
    const float* sa = smem + (kb % kStages) * S::kStageFloats;
    const float* sb = sa + BM * S::kPitch;
    const float* su = sb + BN * S::kPitch;
#pragma unroll
    for (int kk = 0; kk < BK; kk += 4) {
      float4 a[TM], b[TN], u[kSwiglu ? TN : 1];
#pragma unroll
      for (int i = 0; i < TM; ++i)
        a[i] = *reinterpret_cast<const float4*>(sa + (ty + kTy * i) * S::kPitch + kk);
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        b[j] = *reinterpret_cast<const float4*>(sb + (tx + kTx * j) * S::kPitch + kk);
        if (kSwiglu) u[j] = *reinterpret_cast<const float4*>(su + (tx + kTx * j) * S::kPitch + kk);
      }
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          acc0[i][j] = fmaf(a[i].x, b[j].x, acc0[i][j]);
          acc0[i][j] = fmaf(a[i].y, b[j].y, acc0[i][j]);
          acc0[i][j] = fmaf(a[i].z, b[j].z, acc0[i][j]);
          acc0[i][j] = fmaf(a[i].w, b[j].w, acc0[i][j]);
          if (kSwiglu) {
            acc1[i][j] = fmaf(a[i].x, u[j].x, acc1[i][j]);
            acc1[i][j] = fmaf(a[i].y, u[j].y, acc1[i][j]);
            acc1[i][j] = fmaf(a[i].z, u[j].z, acc1[i][j]);
            acc1[i][j] = fmaf(a[i].w, u[j].w, acc1[i][j]);
          }
        }
    }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int r = r0 + ty + kTy * i;
    if (r >= te.rows) continue;
    float* orow = g.out + static_cast<uint64_t>(out_row0 + r) * static_cast<uint32_t>(n_out);
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int c = c0 + tx + kTx * j;
      if (c < n_out) {
        const float v = acc0[i][j];
        orow[c] = kSwiglu ? v / (1.0f + expf(-v)) * acc1[i][j] : v;
      }
    }
  }
}

template <int BM, int BN, int TM, int TN, int BK>
cudaError_t launch_tile(bool swiglu, const SimtArgs& g, cudaStream_t st) {
  const int col_blocks = (g.n_out + BN - 1) / BN;
  const int64_t blocks = static_cast<int64_t>(col_blocks) * g.max_tiles * (kMinTileRows / BM);
  if (blocks > INT32_MAX) return cudaErrorInvalidValue;
  const dim3 grid(static_cast<unsigned>(blocks));
  const int threads = SimtTile<BM, BN, TM, TN, BK, true>::kThreads;
  auto* kern = swiglu ? expert_simt_kernel<BM, BN, TM, TN, BK, true>
                      : expert_simt_kernel<BM, BN, TM, TN, BK, false>;
  return launch_pdl(kern, grid, dim3(threads), 0, st, 1, g, col_blocks);
}

}  // namespace

cudaError_t launch_expert_simt(bool swiglu, const SimtArgs& g, int64_t rows, int num_sms,
                               cudaStream_t st) {
  if (g.max_tiles <= 0) return cudaSuccess;
  // 32 x 64 blocks (4 x 4 per thread) read a third fewer bytes of shared memory per FMA than
  // 32 x 32 ones (4 x 2), but only once they fill the GPU five times over; below that the shorter
  // chains win by their number.  A rollout + replay step, 32 x 32 / 32 x 64 / 64 x 64: T = 2048,
  // d = m = 512, N = 64, k = 8 1609 / 1473 / 1641 us; T = 600, m = 300 460 / 436 / 509; T = 2048,
  // d = m = 256, N = 32, k = 4 262 / 256 / 290; T = 300, d = m = 400, N = 40, k = 4 202 / 260 / 239.
  // Larger register tiles (8 x 4, 8 x 8) and packed FMAs (fma.rn.f32x2, even and odd K apart) gave
  // nothing: 1556 and 1541 at the first of these sizes, the FMA pipe at 55 to 60 % either way.
  const int64_t wide = ((rows + 31) / 32) * ((g.n_out + 63) / 64);
  return wide >= 5 * static_cast<int64_t>(num_sms)
             ? launch_tile<32, 64, 4, 4, 16>(swiglu, g, st)
             : launch_tile<32, 32, 4, 2, 32>(swiglu, g, st);
}

}  // namespace pr2
