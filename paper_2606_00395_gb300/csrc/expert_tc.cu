// Grouped expert GEMMs on the tcgen05 tensor cores (bf16 operands, fp32 accumulation in TMEM).
//
// The gated-MLP expert of App. E.2 with the SwiGLU activation, over the rows that dispatch
// grouped by expert (and over every token for a shared expert):
//   phase 0, gate/up:  H[r, :] = silu(X[r] Wg_e^T) * (X[r] Wu_e^T)   (K = d, 128 H columns / job)
//   phase 1, down:     Y[r, :] = H[r] Wd_e^T                         (K = m, 256 Y columns / job)
// where X[r] = h[perm[r] / k] is the token that dispatch placed at row r.
//
// Both products are computed transposed: the weights are the M operand and the tile's rows the N
// operand.  A job multiplies 256 weight rows (two M = 128 halves: gate and up, or 2 x 128 Y
// columns) with the up to kRows rows of its tile, so a K block of 64 brings 32 KB of weights and
// 128 B per row into shared memory for 2 x 4 MMAs of N = the rows rounded up to 16.
//
// What bounds it: at large experts the ~64 B per clk that an SM takes in from L2, then the power
// limit; below ~200 rows per expert the weight stream from HBM; just above 256 rows the intake
// again, because an expert of 270 rows is two tiles of ~136, each with its 32 KB of weights per K
// block for half the MMAs (DeepSeek-V3-shaped launch: 4022 us at T = 7200, where 5 of 256 experts are
// above 256 rows, 5282 at 8192, 123 of them, 7242 at 14000).  Rows as M = 128 against N
// = 256 weight rows (the layout before) bring 48 KB per 4 MMAs of 128 x 256 x 16, 750 clk of
// intake for 512 clk of MMA; 256 x 256 bring 64 KB per 8 of them, 1024 for 1024.  An expert of up
// to 256 rows reads its weights from L2 once instead of 2-3 times, and N follows its row count
// where M padded to 128 (20 % of the rows at 256 per expert).  Layer calls, before -> after
// (same box, alternating): T = 3001 Qwen3-shaped replay 283.6 -> 267.9 us, T = 32768 2030 -> 1917,
// T = 8192 DeepSeek-V3-shaped with its shared expert (two launches more before) 6319 -> 5887.
//
// Persistent kernel: one CTA per SM walks its list of jobs, every phase-0 job before every
// phase-1 job, tile-major, so the CTAs running at the same time share the weights of the same few
// experts through L2.  A phase-1 job waits until the phase-0 epilogues of its tile have counted
// themselves done (an acquire on a per-tile counter).  No phase-0 job waits on another job and
// every CTA is resident (cooperative launch), so the waits end.
//
// Weights and rows travel in two rings of 128-byte-swizzled K-major stages, each with its own
// producers, so that the weight stream from HBM runs further ahead than the rows, which come from
// L2.  The weight ring's stages are the 16 KB halves of a K block; both rings' copies of a K block
// complete one barrier, because every further wait costs the MMA warp ~80 clk per K block (three
// waits: 1227 clk per K block of the DeepSeek-V3-shaped launch, one: 1149).  Warp roles (warp w
// runs on SM sub-partition w % 4):
//   warps 0-2, 4  row producers (128 threads): every thread copies one 16-byte column chunk of
//              every 16th row with cp.async, written to its swizzled position, straight from h
//              through perm (phase 0), from h (shared experts) or from H (phase 1).
//   warp 3     TMEM owner and tcgen05.mma issuer.  No producer shares its sub-partition.
//   warp 5     TMA producer of the weight ring.
//   warps 6-13 epilogue (two warps per TMEM lane quadrant): TMEM lane = weight row, column = row.
//   warp 14    watches the per-tile counters ahead of the row producers.
//
// TMEM: accumulator columns [0, 256) hold the first weight half (gate), [256, 512) the second
// (up), one column per row of the tile.  Columns fall into two row halves, 0 = rows 0-127 and
// 1 = rows 128-255, each with its own full / empty barriers.  A job of at most 128 rows uses one
// of them, alternating, so that its epilogue overlaps the next job's MMAs.  A larger job uses
// both; its last K block is multiplied for row half 0 first, and its first one likewise if half 1
// is still being drained, so that the epilogue of one half overlaps MMAs of the other (three such K
// blocks overlap more, but MMAs of N = 128 take more shared-memory reads per FLOP: T = 3001 replay
// 272.5 us with three, 265.9 with one, 271.2 with none).
#include "pr2_device.cuh"
#include "pr2_internal.h"

namespace pr2 {
namespace {

constexpr int kThreads = 480;
constexpr int kWarpMma = 3;
constexpr int kWarpB = 5;
constexpr int kEpiWarp0 = 6;
constexpr int kEpiWarps = 8;
constexpr int kWarpReady = 14;
constexpr int kBK = 64;
constexpr int kGatherThreads = 128;          // warps 0-2 and 4
constexpr int kWHalf = 128 * kBK * 2;        // 16 KB: one M = 128 half of a weight stage
constexpr int kHalfRows = 128;               // rows of one TMEM row half
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kAccCols = 256;           // columns of one weight half's accumulator
constexpr int kRel = 8;                      // full and release barriers, one per K block mod 8
constexpr int kOutPitch = 128 * 2 + 16;      // row pitch of an epilogue buffer (distinct banks)
constexpr int kOutBuf = 16 * kOutPitch;      // 16 rows x 128 bf16 columns

// kRows = most rows of a tile.  256: 7 x 16 KB of weights + 3 x 32 KB of rows.  128 (decode
// batches, whose experts serve a few rows each): 10 x 16 KB of weights + 3 x 16 KB of rows.
template <int kRows>
struct Ring {
  static constexpr int kStagesW = kRows == 256 ? 7 : 10;  // weight halves, two per K block
  static constexpr int kStagesR = 3;
  static constexpr int kRStage = kRows * kBK * 2;
  static constexpr int kRRing = kStagesW * kWHalf;  // offset of the row ring
  static constexpr int kOut = kRRing + kStagesR * kRStage;      // epilogue buffers
  static constexpr int kBarOffset = kOut + 4 * kOutBuf;  // two per side
  static constexpr int kSmemBytes = 1024 + kBarOffset + 256;
  static_assert(kStagesW / 2 + 1 < kRel && kStagesR < kRel, "a ring could see a release twice");
  static_assert((2 * kRel + 5) * 8 + 8 <= 256, "barrier area");
};

// Stage release.  The MMA thread commits once per K block, to rel[n % kRel] for the n-th K block.
// A producer with P stages per K block and a ring of S stages may refill a ring's stage for its
// n-th stage once the K block of stage n - S, number (n - S) / P, has completed: that is phase
// j / kRel of rel[j % kRel].  That barrier cannot be a phase further on: its next completion is
// K block j + kRel, whose data this producer has not issued yet (S / P + 1 < kRel).
template <int S, int P>
struct ReleaseCursor {
  int n = 0;  // stages issued so far
  __device__ __forceinline__ bool wait(uint64_t* rel, volatile int* abort_flag, int32_t* status) {
    if (n < S) return true;
    const int j = (n - S) / P;
    return mbar_wait(&rel[j % kRel], static_cast<uint32_t>(j / kRel) & 1u, abort_flag, status);
  }
  __device__ __forceinline__ void advance() { ++n; }
};

struct Job {
  int phase;  // 0: gate/up + SwiGLU, 1: down, -1: no such job
  int mt;     // tile (entry of the tile table)
  int nt;     // block of weight rows
};

// The jobs of one CTA: job(t) for t = 0, 1, ... until phase -1.  Phase-0 jobs are dealt round
// robin.  CTAs that get one fewer of them take `early` phase-1 jobs each before the others
// join (as many as one phase-0 job costs in K blocks), and the rest is dealt round robin.
struct Schedule {
  int n1, n2;    // jobs per tile in phase 0 / 1
  int P0, P1;    // jobs of each phase
  int own0;      // phase-0 jobs of this CTA
  int late;      // CTAs 0 .. late - 1 have one phase-0 job more than the others (0: all the same)
  int early, taken;  // early phase-1 jobs per such CTA, and in all
  __device__ __forceinline__ void init(int nm, int n1_, int n2_, int kb0, int kb1) {
    const int G = static_cast<int>(gridDim.x), b = static_cast<int>(blockIdx.x);
    n1 = n1_;
    n2 = n2_;
    P0 = nm * n1;
    P1 = nm * n2;
    own0 = b < P0 ? (P0 - b + G - 1) / G : 0;
    late = P0 % G;
    early = late != 0 ? (kb0 + kb1 / 2) / kb1 : 0;
    const int64_t all = static_cast<int64_t>(early) * (G - late);
    taken = late != 0 ? static_cast<int>(all < P1 ? all : P1) : 0;
  }
  __device__ __forceinline__ Job job(int t) const {
    const int G = static_cast<int>(gridDim.x), b = static_cast<int>(blockIdx.x);
    if (t < own0) {
      const int f = b + t * G;
      return Job{0, f / n1, f % n1};
    }
    int u = t - own0;
    int f;
    if (b >= late && u < early) {
      f = u * (G - late) + (b - late);
      if (f >= taken) return Job{-1, 0, 0};
    } else {
      if (b >= late) u -= early;
      f = taken + u * G + b;
      if (f >= P1) return Job{-1, 0, 0};
    }
    return Job{1, f / n2, f % n2};
  }
};

__device__ __forceinline__ int round16(int n) { return (n + 15) & ~15; }

// Row producer (warps 0-2, 4; 128 threads; each row stage registers 128 arrivals with its K block).  Thread
// `tid` copies, for every K block, the 16-byte chunk c = tid % 8 of tile rows r = tid / 8 + 16 i.
// In the 128-byte swizzled K-major stage, chunk c of row r sits at r * 128 + ((c ^ (r % 8)) * 16),
// and r % 8 is the same for all rows of a thread.  After its copies of a stage the thread
// registers an arrival that fires when they have landed; the MMA thread, after acquiring the
// barrier, fences the stage into the async proxy.  Rows between the tile's count and its
// multiple of 16 are zero-filled.  The next job's table entry is loaded when a job starts and its
// perm entries halfway through the job, as raw values turned into pointers only when that job
// starts, so no load result is waited for while the ring needs refilling.
template <int kRows>
__device__ __forceinline__ void row_producer(const MlpArgs& ma, const Schedule& sch, uint8_t* smem,
                                             uint64_t* full, uint64_t* rel_bar,
                                             const int* jobs_ready, volatile int* abort_flag) {
  using R = Ring<kRows>;
  constexpr int kPer = kRows / 16;  // rows of a thread
  const int tid = threadIdx.x < 96 ? threadIdx.x : threadIdx.x - 32;  // warps 0-2, 4
  const int c = tid & 7;
  const int r0 = tid >> 3;
  const uint32_t soff = static_cast<uint32_t>(r0 * 128 + ((c ^ (r0 & 7)) << 4));
  const __nv_bfloat16* h = static_cast<const __nv_bfloat16*>(ma.h);
  const __nv_bfloat16* H = static_cast<const __nv_bfloat16*>(ma.H);
  const uint64_t keep = l2_policy_evict_last();  // h: every token row is read k times and more
  auto entry = [&](const Job& j) {
    return j.phase >= 0 ? ma.tiles[j.mt] : TileEntry{0, 0, 0, 0};
  };
  // tokens of a phase-0 tile's rows (rows beyond the tile: 0, they are zero-filled)
  auto fetch = [&](const TileEntry& te, int32_t (&slot)[kPer]) {
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int row = r0 + 16 * i;
      slot[i] = 0;
      if (row < te.rows)
        slot[i] = te.expert < ma.N ? ma.perm[te.a_row0 + row] : (te.a_row0 + row) * ma.k;
    }
  };
  int32_t slot[kPer], slot_next[kPer];
#pragma unroll
  for (int i = 0; i < kPer; ++i) slot[i] = slot_next[i] = 0;
  int t = 0;
  Job job = sch.job(0), next = sch.job(1);
  TileEntry te = entry(job), te_next = entry(next);
  if (job.phase == 0) fetch(te, slot);
  int stage = 0;
  ReleaseCursor<R::kStagesR, 1> rc;
  bool ok = true;
  while (job.phase >= 0 && ok) {
    const Job after = sch.job(t + 2);
    const TileEntry te_after = entry(after);  // used by the next job's fetch
    const int n = round16(te.rows);
    const __nv_bfloat16* src[kPer];
    if (job.phase == 0) {
#pragma unroll
      for (int i = 0; i < kPer; ++i)
        src[i] = h + static_cast<int64_t>(slot[i] / ma.k) * ma.d + c * 8;
    } else {
      // H rows of this tile: written by other CTAs' phase-0 epilogues (plain stores, read here
      // by plain asynchronous copies behind the acquire)
      while (ld_acquire_cta(jobs_ready) <= t) {
        if (*abort_flag) {
          ok = false;
          break;
        }
        __nanosleep(32);
      }
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int row = r0 + 16 * i;
        src[i] = H + static_cast<int64_t>(te.out_row0 + (row < te.rows ? row : 0)) * ma.m + c * 8;
      }
    }
    const int KB = job.phase ? ma.m / kBK : ma.d / kBK;
    const int kb_fetch = KB / 2;
    for (int kb = 0; kb < KB && ok; ++kb) {
      if (!rc.wait(rel_bar, abort_flag, ma.status)) {
        ok = false;
        break;
      }
      uint64_t* bar = &full[rc.n % kRel];
      rc.advance();
      const uint32_t dst = smem_u32(smem + R::kRRing + stage * R::kRStage) + soff;
      if (job.phase == 0) {
#pragma unroll
        for (int i = 0; i < kPer; ++i)
          if (16 * i < n)
            cp_async_16_hint(dst + i * 2048, src[i] + kb * kBK, r0 + 16 * i < te.rows ? 16u : 0u,
                             keep);
      } else {
#pragma unroll
        for (int i = 0; i < kPer; ++i)
          if (16 * i < n)
            cp_async_16(dst + i * 2048, src[i] + kb * kBK, r0 + 16 * i < te.rows ? 16u : 0u);
      }
      cp_async_arrive_noinc(bar);
      if (++stage == R::kStagesR) stage = 0;
      if (kb == kb_fetch && next.phase == 0) fetch(te_next, slot_next);
    }
#pragma unroll
    for (int i = 0; i < kPer; ++i) slot[i] = slot_next[i];
    job = next;
    te = te_next;
    next = after;
    te_next = te_after;
    ++t;
  }
  cp_async_commit();
  cp_async_wait<0>();  // nothing may still be writing shared memory when the CTA leaves
}

template <int kRows>
__global__ void __launch_bounds__(kThreads, 1)
    expert_tc_kernel(const __grid_constant__ CUtensorMap tm_g,
                     const __grid_constant__ CUtensorMap tm_u,
                     const __grid_constant__ CUtensorMap tm_d,
                     const __grid_constant__ CUtensorMap tm_sg,
                     const __grid_constant__ CUtensorMap tm_su,
                     const __grid_constant__ CUtensorMap tm_sd, MlpArgs ma) {
  using R = Ring<kRows>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + R::kBarOffset);  // [kRel]
  uint64_t* rel = full + kRel;               // [kRel]
  uint64_t* acc_full = rel + kRel;           // [2], one per row half
  uint64_t* acc_empty = acc_full + 2;        // [2]
  uint64_t* drain = acc_empty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kRel; ++s) {
      mbar_init(&full[s], kGatherThreads + 1);  // the row copies, and the weights' expect_tx
      mbar_init(&rel[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], kEpiWarps);  // one arrival per epilogue warp
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tm_g);
    tma_prefetch_desc(&tm_u);
    tma_prefetch_desc(&tm_d);
  }
  if (warp == kWarpMma) {
    tmem_alloc(tmem_slot, kTmemCols);
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();  // the tile table and the route come from the previous kernels
  pdl_trigger();
  __shared__ int nm_s;
  __shared__ int jobs_ready;  // jobs [0, jobs_ready) of this CTA may read their rows
  if (threadIdx.x == 0) {
    jobs_ready = 0;
    const int nm = *ma.num_tiles;  // in flight with the status word
    nm_s = status_timed_out(ma.status) || nm < 0 ? 0 : (nm > ma.max_tiles ? ma.max_tiles : nm);
  }
  __syncthreads();
  Schedule sch;  // dispatch's tile count, never above the host bound; 0 after a timeout
  sch.init(nm_s, (ma.m + 127) / 128, (ma.d + 255) / 256, ma.d / kBK, ma.m / kBK);

  if (warp < 3 || warp == 4) {
    row_producer<kRows>(ma, sch, smem, full, rel, &jobs_ready, abort_flag);
  } else if (warp == kWarpB && lane == 0) {
    // ---------------- TMA producer of the weight ring ----------------
    // Weights are reused only by the tiles of their expert, which run at about the same time, so
    // they take the normal L2 policy (an evict_last hint on them pushes out h, H and Y, which
    // later tiles and kernels read again).
    int stage = 0;
    int n = 0;  // K blocks issued
    ReleaseCursor<R::kStagesW, 2> rcw;
    bool ok = true;
    // the next job's expert is loaded while this job streams
    Job next = sch.job(0);
    int e_next = next.phase >= 0 ? ma.tiles[next.mt].expert : 0;
    for (int t = 0; next.phase >= 0 && ok; ++t) {
      const Job job = next;
      const int e = e_next;
      next = sch.job(t + 1);
      if (next.phase >= 0) e_next = ma.tiles[next.mt].expert;
      const bool shared = e >= ma.N;
      const int es = shared ? e - ma.N : e;
      const int wrow = job.phase == 0 ? es * ma.m + job.nt * 128 : es * ma.d + job.nt * 256;
      const int KB = job.phase ? ma.m / kBK : ma.d / kBK;
      for (int kb = 0; kb < KB && ok; ++kb) {
        uint64_t* bar = &full[n % kRel];
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          if (!rcw.wait(rel, abort_flag, ma.status)) {
            ok = false;
            break;
          }
          rcw.advance();
          uint8_t* sw = smem + stage * kWHalf;
          if (half == 0) {
            mbar_arrive_expect_tx(bar, 2 * kWHalf);
            ++n;
          }
          // each map is named directly: a selected map pointer slows the loop
          if (job.phase == 0) {
            if (!shared) {
              if (half == 0) tma_load_2d(sw, &tm_g, bar, kb * kBK, wrow);
              else tma_load_2d(sw, &tm_u, bar, kb * kBK, wrow);
            } else {
              if (half == 0) tma_load_2d(sw, &tm_sg, bar, kb * kBK, wrow);
              else tma_load_2d(sw, &tm_su, bar, kb * kBK, wrow);
            }
          } else if (!shared) {
            tma_load_2d(sw, &tm_d, bar, kb * kBK, wrow + half * 128);
          } else {
            tma_load_2d(sw, &tm_sd, bar, kb * kBK, wrow + half * 128);
          }
          if (++stage == R::kStagesW) stage = 0;
        }
      }
    }
    // no copy may still be landing when the CTA leaves (the MMA thread may have given up)
    for (int j = n > kRel ? n - kRel : 0; j < n; ++j)
      mbar_wait_slow(&full[j % kRel], static_cast<uint32_t>(j / kRel) & 1u, nullptr, nullptr,
                     kDrainLimitNs);
  } else if (warp == kWarpMma) {
    // ---------------- MMA issuer: the whole warp in step, one elected lane issues ----------------
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
    const uint32_t lo_w = umma_lo(smem_u32(smem)), lo_r = umma_lo(smem_u32(smem + R::kRRing));
    constexpr uint32_t kLoW = kWHalf / 16, kLoR = R::kRStage / 16;
    int sw_i = 0, sr_i = 0;          // weight half and row stage the next K block arrives in
    int ka = 0;                      // K blocks acquired
    int kn = 0;                      // K blocks released: K block kn through rel[kn % kRel]
    int half_next = 0;               // row half of the next small job
    uint32_t par_empty = 0;          // bit h: parity of acc_empty[h] that was last waited for
    bool ok = true;
    // the next K block's stages: descriptor words of its weight halves and rows
    struct Stage {
      uint32_t w0, w1, r;
    };
    auto acquire = [&](Stage& st) {
      const bool in = mbar_wait(&full[ka % kRel], static_cast<uint32_t>(ka / kRel) & 1u, abort_flag,
                                ma.status);
      ++ka;
      st.w0 = lo_w + sw_i * kLoW;
      if (++sw_i == R::kStagesW) sw_i = 0;
      st.w1 = lo_w + sw_i * kLoW;
      if (++sw_i == R::kStagesW) sw_i = 0;
      st.r = lo_r + sr_i * kLoR;
      if (++sr_i == R::kStagesR) sr_i = 0;
      if (!__all_sync(0xffffffffu, in)) return false;
      fence_proxy_async_smem();  // rows written by cp.async (generic proxy)
      tc_fence_after();
      return true;
    };
    // a K block's MMAs for the rows from row0 on (0 or 128; N = rows by idesc) into columns acc0..,
    // then a commit to `bar` (nullable) by the same thread
    auto multiply = [&](const Stage& st, int row0, uint32_t idesc, int acc0, bool first,
                        uint64_t* bar) {
      const uint32_t d0 = tm + acc0, d1 = d0 + kAccCols;
      const uint32_t b = st.r + row0 * (128 / 16);
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < kBK / 16; ++kk) {
          const uint64_t bd = umma_desc_lo(b + 2 * kk);
          const uint32_t acc = (!first || kk > 0) ? 1u : 0u;
          umma_bf16(d0, umma_desc_lo(st.w0 + 2 * kk), bd, idesc, acc);
          umma_bf16(d1, umma_desc_lo(st.w1 + 2 * kk), bd, idesc, acc);
        }
        if (bar != nullptr) umma_commit(bar);
      }
      __syncwarp();
    };
    auto next_rel = [&]() { return &rel[kn++ % kRel]; };  // releases the oldest K block's stages
    auto wait_empty = [&](int h) {
      const uint32_t par = ((par_empty >> h) & 1u) ^ 1u;
      par_empty ^= 1u << h;
      const bool in = mbar_wait(&acc_empty[h], par, abort_flag, ma.status);
      if (!__all_sync(0xffffffffu, in)) return false;
      tc_fence_after();
      return true;
    };
    auto commit = [&](uint64_t* bar) {
      if (elect_one()) umma_commit(bar);
      __syncwarp();
    };
    Job job = sch.job(0);
    int rows = job.phase >= 0 ? ma.tiles[job.mt].rows : 0;
    for (int t = 0; job.phase >= 0 && ok; ++t) {
      const int n = __shfl_sync(0xffffffffu, round16(rows), 0);
      const int KB = job.phase ? ma.m / kBK : ma.d / kBK;
      job = sch.job(t + 1);
      const int rows_next = job.phase >= 0 ? ma.tiles[job.mt].rows : 0;
      const uint32_t idesc = umma_idesc_bf16(128, n);
      Stage st;
      if (kRows <= kHalfRows || n <= kHalfRows) {
        const int h = half_next;
        half_next ^= 1;
        ok = wait_empty(h) && acquire(st);
        for (int kb = 0; kb < KB && ok; ++kb) {
          multiply(st, 0, idesc, h * kHalfRows, kb == 0, next_rel());
          if (kb + 1 < KB) ok = acquire(st);
        }
        if (ok) commit(&acc_full[h]);
      } else {
        constexpr uint32_t idesc0 = umma_idesc_bf16(128, kHalfRows);
        const uint32_t idesc1 = umma_idesc_bf16(128, n - kHalfRows);
        ok = wait_empty(0);
        int kb = 0;
        const uint32_t par1 = ((par_empty >> 1) & 1u) ^ 1u;
        const bool free1 = __all_sync(0xffffffffu, mbar_test_wait(&acc_empty[1], par1));
        if (ok && KB > 1 && !free1) {
          // half 1 is still being drained: the first K block's half 0 goes ahead
          ok = acquire(st);
          if (ok) multiply(st, 0, idesc0, 0, true, nullptr);
          if (ok) ok = wait_empty(1);
          if (ok) multiply(st, kHalfRows, idesc1, kHalfRows, true, next_rel());
          kb = 1;
        } else if (ok) {
          ok = wait_empty(1);
        }
        if (ok) ok = acquire(st);
        for (; kb < KB - 1 && ok; ++kb) {
          multiply(st, 0, idesc, 0, kb == 0, next_rel());
          ok = acquire(st);
        }
        if (ok) {
          multiply(st, 0, idesc0, 0, kb == 0, &acc_full[0]);
          multiply(st, kHalfRows, idesc1, kHalfRows, kb == 0, next_rel());
          commit(&acc_full[1]);
        }
      }
      rows = rows_next;
    }
    commit(drain);
    mbar_wait_slow(drain, 0, nullptr, nullptr, kDrainLimitNs);
  } else if (warp == kWarpReady) {
    // ---- watcher: job after job, the H rows of a phase-1 job's tile are complete ----
    // (it runs ahead of the row producers, which then need no round trip to L2 of their own)
    if (lane == 0) {
      const int need = kEpiWarps * sch.n1;
      bool ok = true;
      for (int t = 0; ok; ++t) {
        const Job job = sch.job(t);
        if (job.phase < 0) break;
        if (job.phase == 1) {
          const int* cnt = ma.ready + job.mt;
          const uint64_t t0 = globaltimer_ns();
          while (ld_acquire_gpu(cnt) < need) {
            if (*abort_flag || globaltimer_ns() - t0 > kWaitLimitNs) {
              *abort_flag = 1;
              if (ma.status != nullptr) atomicOr(ma.status, PR2_STATUS_TIMEOUT);
              ok = false;
              break;
            }
            __nanosleep(64);
          }
        }
        if (ok) st_release_cta(&jobs_ready, t + 1);
      }
    }
  } else if (warp >= kEpiWarp0) {
    // ---- epilogue: TMEM lane 32 (w % 4) + lane = weight row, column = row of the tile ----
    // The quadrant's two warps are sides 0 and 1; the four warps of a side take 16 rows of the tile
    // at a time: phase 0, 128 columns of H from both accumulators, the sides taking turns; phase
    // 1, 128 columns of Y from accumulator `side`.  The values come out of TMEM as fragments with
    // the rows along registers, are transposed by stmatrix into one of the side's two [16][128]
    // bf16 buffers and leave as 16-byte stores, 256 contiguous bytes per row: 25 clk per tile row
    // at T = 32768, where 2-byte stores straight from registers took 31-37 and kept the load /
    // store unit from the row copies, 64-byte row segments per warp 23-29, and bulk copies out of
    // the buffer 54-85 (~1300 clk until a chunk's copies had read it).
    const int q = warp & 3;
    const int side = (warp - kEpiWarp0) >> 2;
    const int st_id = ((warp - kEpiWarp0) & 3) * 32 + lane;  // this thread among its side's 128
    const uint32_t tq = tmem + (static_cast<uint32_t>(q * 32) << 16);
    const uint32_t obuf = smem_u32(smem + R::kOut + side * 2 * kOutBuf);
    // stmatrix: row lane % 8, columns 32 q + 8 (lane / 8)..; read back: row st_id / 16, 16-byte
    // word st_id % 16 (both: rows 8.. follow)
    const uint32_t ost = static_cast<uint32_t>((lane & 7) * kOutPitch + q * 64 + (lane >> 3) * 16);
    const uint32_t old = static_cast<uint32_t>((st_id >> 4) * kOutPitch + (st_id & 15) * 16);
    uint32_t sel = 0;  // buffer of the next chunk
    uint32_t par_full = 0;
    int half_next = 0;
    bool ok = true;
    Job job = sch.job(0);
    TileEntry te = job.phase >= 0 ? ma.tiles[job.mt] : TileEntry{0, 0, 0, 0};
    for (int t = 0; job.phase >= 0 && ok; ++t) {
      const Job next = sch.job(t + 1);
      const TileEntry te_next = next.phase >= 0 ? ma.tiles[next.mt] : TileEntry{0, 0, 0, 0};
      const int n = round16(te.rows);
      const bool big = kRows > kHalfRows && n > kHalfRows;
      const int ld = job.phase == 0 ? ma.m : ma.d;
      const int col0 = (job.phase == 0 ? job.nt * 128 : job.nt * 256 + side * 128) + (st_id & 15) * 8;
      const bool live = col0 < ld;  // this thread's 8 columns (ld % 64 == 0) or none
      __nv_bfloat16* out = static_cast<__nv_bfloat16*>(job.phase == 0 ? ma.H : ma.Y) +
                           static_cast<int64_t>(te.out_row0) * ld + col0;
      for (int ev = 0; ev < (big ? 2 : 1); ++ev) {
        int h = ev;
        if (!big) {
          h = half_next;
          half_next ^= 1;
        }
        // a whole side leaves its loop or none of it does (it meets at a barrier below)
        const bool in = mbar_wait(&acc_full[h], (par_full >> h) & 1u, abort_flag, ma.status);
        if (!named_bar_and(1 + side, 128, in)) {
          ok = false;
          break;
        }
        par_full ^= 1u << h;
        tc_fence_after();
        const int row0 = ev * kHalfRows;  // first tile row of this half
        const int cols = n - row0 < kHalfRows ? n - row0 : kHalfRows;
        const uint32_t tacc = tq + h * kHalfRows;
        const int step = job.phase == 0 ? 32 : 16;
        for (int c0 = job.phase == 0 ? side * 16 : 0; c0 < cols; c0 += step) {
          uint32_t pk[2][4];  // [8 rows][8 columns]: column j of rows 8 i.. in pk[i][j / 8]
          if (job.phase == 0) {
            uint32_t g0[8], g1[8], u0[8], u1[8];
            tmem_ld_frag(tacc + c0, g0);
            tmem_ld_frag(tacc + c0 + (16u << 16), g1);
            tmem_ld_frag(tacc + kAccCols + c0, u0);
            tmem_ld_frag(tacc + kAccCols + c0 + (16u << 16), u1);
            tmem_wait_ld8(g0, g1);
            reg_fence8(u0, u1);
            auto act = [](uint32_t g, uint32_t u) {
              const float x = __uint_as_float(g);
              return __fdividef(x, 1.0f + __expf(-x)) * __uint_as_float(u);
            };
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
              for (int j = 0; j < 2; ++j) {
                pk[i][j] = pack_bf16x2(act(g0[4 * i + 2 * j], u0[4 * i + 2 * j]),
                                       act(g0[4 * i + 2 * j + 1], u0[4 * i + 2 * j + 1]));
                pk[i][2 + j] = pack_bf16x2(act(g1[4 * i + 2 * j], u1[4 * i + 2 * j]),
                                           act(g1[4 * i + 2 * j + 1], u1[4 * i + 2 * j + 1]));
              }
          } else {
            uint32_t y0[8], y1[8];
            tmem_ld_frag(tacc + side * kAccCols + c0, y0);
            tmem_ld_frag(tacc + side * kAccCols + c0 + (16u << 16), y1);
            tmem_wait_ld8(y0, y1);
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
              for (int j = 0; j < 2; ++j) {
                pk[i][j] = pack_bf16x2(__uint_as_float(y0[4 * i + 2 * j]),
                                       __uint_as_float(y0[4 * i + 2 * j + 1]));
                pk[i][2 + j] = pack_bf16x2(__uint_as_float(y1[4 * i + 2 * j]),
                                           __uint_as_float(y1[4 * i + 2 * j + 1]));
              }
          }
          const uint32_t buf = obuf + sel * kOutBuf;
          sel ^= 1u;
          stmatrix_x4_trans(buf + ost, pk[0][0], pk[0][1], pk[0][2], pk[0][3]);
          stmatrix_x4_trans(buf + ost + 8 * kOutPitch, pk[1][0], pk[1][1], pk[1][2], pk[1][3]);
          // (the other buffer's reads are behind this barrier too: the next chunk may write it)
          named_bar_sync(1 + side, 128);
          uint32_t v0[4], v1[4];
          ld_shared_v4(buf + old, v0);
          ld_shared_v4(buf + old + 8 * kOutPitch, v1);
          const int r = row0 + c0 + (st_id >> 4);
          if (live && r < te.rows) st_global_v4(out + static_cast<int64_t>(r) * ld, v0);
          if (live && r + 8 < te.rows) st_global_v4(out + static_cast<int64_t>(r + 8) * ld, v1);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[h]);
      }
      if (ok && job.phase == 0) {  // H rows before the count
        __threadfence();
        __syncwarp();
        if (lane == 0) atomicAdd(ma.ready + job.mt, 1);
      }
      job = next;
      te = te_next;
    }
  }
  __syncthreads();
  if (warp == kWarpMma) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

template <int kRows>
cudaError_t launch_rows(const ExpertMaps& tm, const MlpArgs& a, int num_sms, cudaStream_t st) {
  const int64_t per_tile = (a.m + 127) / 128 + (a.d + 255) / 256;
  const int64_t bound = a.max_tiles * per_tile;
  const int grid = static_cast<int>(bound < num_sms ? bound : num_sms);
  auto* kernel = expert_tc_kernel<kRows>;
  constexpr int smem = Ring<kRows>::kSmemBytes;
  cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (err != cudaSuccess) return err;
  // CTAs wait on one another: a cooperative launch guarantees that all of them are resident (one
  // per SM at this shared-memory size).
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  err = cudaLaunchKernelEx(&cfg, kernel, tm.gate, tm.up, tm.down, tm.s_gate, tm.s_up, tm.s_down, a);
  if (err == cudaSuccess) return err;
  (void)cudaGetLastError();  // cooperative + programmatic serialization refused: drop the latter
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, tm.gate, tm.up, tm.down, tm.s_gate, tm.s_up, tm.s_down, a);
}

}  // namespace

// Tiles of 128 rows leave 48 KB more for the weight ring, tiles of 256 read an expert's weights and
// issue its MMAs once for twice the rows.  Replay layer of the Qwen3 shape, 128 / 256 rows, by mean
// rows per expert: even routes 53 209.5 / 215.1 us, 69 213.4 / 218.7, 98 221.5 / 225.6, 119 231.5 /
// 232.0, 131 249.1 / 235.9; Zipf(1.2) routes 32 207.7 / 212.6, 48 220 / 217.2, 64 230.6 / 223.3, 96
// 259.8 / 245.5.  The line lies where the loss on either side is the same.  (One kernel that picks
// the layout on the device by how many experts have more than 128 rows took 2 us more at every
// size: more code to fetch after weights that flush L2.)
int expert_tile_rows(int64_t rows, int N) {
  return rows <= static_cast<int64_t>(N) * 64 ? 128 : 256;
}

cudaError_t launch_expert_tc(const ExpertMaps& tm, const MlpArgs& a, int tile_rows, int num_sms,
                             cudaStream_t st) {
  if (a.max_tiles <= 0) return cudaSuccess;
  if (a.perm == nullptr || a.k <= 0 || a.ready == nullptr) return cudaErrorInvalidValue;
  return tile_rows == 128 ? launch_rows<128>(tm, a, num_sms, st)
                          : launch_rows<256>(tm, a, num_sms, st);
}

}  // namespace pr2
