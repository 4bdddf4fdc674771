// fp32 routing kernels (exact fp32 SIMT arithmetic; TF32 tensor cores would not meet the fp32
// tolerance).  One warp per kTok tokens.
//   predict (Eqs. pr2_predict, pr2_route): z = h W^T + h W_p^T, rho_hat = Softmax(z),
//            idx = TopK(rho_hat, k) (ties to the lower expert), gates = rho_hat[idx].
//   replay  (Sec. 4.1 "Replay During Training"): rho = Softmax(h W^T), gates = rho[idx_in].
// PR2_F_NORMALIZE_TOPK divides a token's gates by their sum (over its valid slots).
//
// The warp takes eight experts at a time: their weight rows are read as float4 along d, all of
// them in flight, and the eight (predict: sixteen) dot products are summed over the lanes together,
// a step halving both the values and the lanes that share one (9 shuffles for 8 sums instead of
// 40).  Small layers are bound by that latency, large ones by the weight rows that every token
// reads from L2, which kTok = 4 tokens of a warp then share.
#include <float.h>

#include "route_epilogue.cuh"

namespace pr2 {
namespace {

constexpr int kWarps = 2;

template <bool kPredict, int kTok>
__global__ void __launch_bounds__(kWarps * 32)
    route_simt_kernel(int T, int d, int N, int k, const float* __restrict__ h,
                      const float* __restrict__ W, const float* __restrict__ Wp,
                      const int32_t* __restrict__ idx_in, int32_t* __restrict__ idx_out,
                      float* __restrict__ gates, float* __restrict__ aux,
                      unsigned long long* near_tie, int32_t* status, int norm, int late_wait) {
  // late_wait: the inputs are complete already (see pr2_moe_replay_forward); the kernel before is
  // waited for only before leaving, so that a kernel after this one sees its results too
  if (!late_wait) pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const int t0 = (blockIdx.x * kWarps + (threadIdx.x >> 5)) * kTok;
  if (t0 < T) {
    const float* ht[kTok];
#pragma unroll
    for (int q = 0; q < kTok; ++q)
      ht[q] = h + static_cast<int64_t>(t0 + q < T ? t0 + q : t0) * d;
    // z for experts e = j*32 + lane lives in zr[j]; p (router part alone) in pr[j].
    float zr[kTok][kRoutePerLane], pr[kTok][kRoutePerLane];
    const int src = ((lane & 4) << 2) | ((lane & 2) << 2) | ((lane & 1) << 2);
#pragma unroll
    for (int j = 0; j < kRoutePerLane; ++j) {
#pragma unroll
      for (int q = 0; q < kTok; ++q) {
        zr[q][j] = -FLT_MAX;
        pr[q][j] = 0.f;
      }
      for (int g = 0; g < 4; ++g) {
        const int e0 = j * 32 + g * 8;
        if (e0 >= N) break;
        float p[kTok][8], b[kTok][8];
#pragma unroll
        for (int q = 0; q < kTok; ++q)
#pragma unroll
          for (int l = 0; l < 8; ++l) p[q][l] = b[q][l] = 0.f;
        for (int i = 4 * lane; i < d; i += 128) {
          float4 x[kTok];
#pragma unroll
          for (int q = 0; q < kTok; ++q) x[q] = *reinterpret_cast<const float4*>(ht[q] + i);
#pragma unroll
          for (int l = 0; l < 8; ++l) {
            const int64_t at = static_cast<int64_t>(e0 + l < N ? e0 + l : e0) * d + i;
            const float4 w = __ldg(reinterpret_cast<const float4*>(W + at));
#pragma unroll
            for (int q = 0; q < kTok; ++q)
              p[q][l] = fmaf(x[q].w, w.w, fmaf(x[q].z, w.z, fmaf(x[q].y, w.y, fmaf(x[q].x, w.x, p[q][l]))));
            if (kPredict) {
              const float4 v = __ldg(reinterpret_cast<const float4*>(Wp + at));
#pragma unroll
              for (int q = 0; q < kTok; ++q)
                b[q][l] = fmaf(x[q].w, v.w, fmaf(x[q].z, v.z, fmaf(x[q].y, v.y, fmaf(x[q].x, v.x, b[q][l]))));
            }
          }
        }
#pragma unroll
        for (int q = 0; q < kTok; ++q) {
          const float ps = __shfl_sync(0xffffffffu, warp_sum8(p[q]), src);
          const float bs = kPredict ? __shfl_sync(0xffffffffu, warp_sum8(b[q]), src) : 0.f;
          if ((lane >> 3) == g && e0 + (lane & 7) < N) {
            pr[q][j] = ps;
            zr[q][j] = ps + bs;
          }
        }
      }
    }
#pragma unroll
    for (int q = 0; q < kTok; ++q) {
      if (t0 + q < T) {
        const bool tie = route_warp_finish(kPredict, t0 + q, N, k, zr[q], pr[q], idx_in, idx_out,
                                           gates, aux, status, norm != 0);
        if (tie && lane == 0 && near_tie != nullptr) atomicAdd(near_tie, 1ull);
      }
    }
  }
  if (late_wait) pdl_wait();
}

}  // namespace

cudaError_t launch_route_simt(const pr2_dims& dm, bool predict, const float* h, const float* W,
                              const float* Wp, const int32_t* idx_in, int32_t* idx_out,
                              float* gates, float* aux, int64_t* near_tie, int32_t* status,
                              bool late_wait, cudaStream_t st) {
  const int T = static_cast<int>(dm.T);
  if (T == 0) return cudaSuccess;
  // four tokens per warp where the weight rows weigh more than the parallelism (rollout + replay
  // step, one / four: T = 600, N = 64, d = 512 528 / 506 us; T = 2048, N = 32, d = 256 291 / 291;
  // T = 1000, N = 16, d = 128 132 / 138; T = 256, N = 8, d = 128 54 / 60)
  const bool four = T >= 512 && static_cast<int64_t>(dm.N) * dm.d >= 16384;
  const int per_block = kWarps * (four ? 4 : 1);
  auto* kern = predict ? (four ? route_simt_kernel<true, 4> : route_simt_kernel<true, 1>)
                       : (four ? route_simt_kernel<false, 4> : route_simt_kernel<false, 1>);
  return launch_pdl(kern, dim3((T + per_block - 1) / per_block), dim3(kWarps * 32), 0, st, 1, T,
                    dm.d, dm.N, dm.k, h, W, Wp, idx_in, idx_out, gates, aux,
                    reinterpret_cast<unsigned long long*>(near_tie), status,
                    (dm.flags & PR2_F_NORMALIZE_TOPK) ? 1 : 0, late_wait ? 1 : 0);
}

}  // namespace pr2
