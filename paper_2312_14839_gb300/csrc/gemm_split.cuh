// The weight-gradient GEMMs C[m][n] += sum_k A[m][k] B[n][k] of every layer in one launch on the tensor
// cores, K split over CTAs, the split sums added to C with TMA reductions.
// Pipeline (per CTA): thread 0 issues the TMA copies of up to kStages K chunks ahead (one mbarrier per
// stage counts the bytes), thread 32 waits for each stage, issues its four MMAs and commits them
// to the stage's "empty" mbarrier, which releases the stage to the producer. A final commit
// signals the epilogue, which all 8 warps share. Two CTAs fit an SM, so one CTA's epilogue overlaps the
// other's loads and MMAs. Every wait is bounded: on expiry the CTA raises an error
// bit, waits (bounded) for the copies it issued, skips the epilogue, frees its TMEM and returns.
#pragma once

#include "tc_gemm.cuh"

namespace bhem {
namespace tc {

constexpr int kBN = 128;          // columns per CTA tile
constexpr int kStages = 3;        // 32 KB each
constexpr int kStageA = kBM * kBK * 2, kStageB = kBN * kBK * 2, kStage = kStageA + kStageB;
constexpr size_t kGemmSmem = (size_t)kStages * kStage + 1024;   // + base alignment
constexpr int kStageWarp = 2 * 2048;   // epilogue: two FP32 tiles of 32 rows x 16 columns per warp
static_assert(kStage % 1024 == 0, "every operand tile starts on a 1024-byte swizzle atom");
static_assert(kStages * kStage >= 8 * kStageWarp, "the epilogue's tiles fit the freed stages");
constexpr int kMaxGroups = 4;

// One GEMM of the launch: maps of A [M][K] and B [N][K] (boxes of 64 columns x 128 rows, reads outside
// are zero) and of C [M][N] (boxes of 16 columns x 32 rows, writes outside are dropped).
struct GemmGroup {
  CUtensorMap a, b, c;
};
struct GemmSet {
  GemmGroup g[kMaxGroups];
  int n[kMaxGroups];                // columns of C, a multiple of 16
  int tiles_n[kMaxGroups];          // column tiles
  int first[kMaxGroups + 1];        // first tile (blockIdx.x) of each group
  int kchunks;                      // ceil(K / kBK), the same for every group
  int kchunks_per_split;            // K chunks of one blockIdx.y (the host makes every split non-empty)
  unsigned polls;                   // bound of every mbarrier wait
  int* err;                         // error word; err_bit is raised when a wait expires
  int err_bit;
};

// What bounds it: the operands' way from L2 (64 KB a chunk and tile pair against 0.26 us of MMAs) and, with
// small K per CTA, the split sums' reductions, so one launch takes every layer's tiles and splits K no finer
// than fills the SMs twice over.
__global__ void __launch_bounds__(kThreads, 2)
k_gemm_split(const __grid_constant__ GemmSet set) {
  extern __shared__ unsigned char tc_smem_raw[];
  __shared__ __align__(8) uint64_t bar_full[kStages];
  __shared__ __align__(8) uint64_t bar_empty[kStages];
  __shared__ __align__(8) uint64_t bar_done;
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort, s_consumed, s_issued;
  volatile int* abort_flag = &s_abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t raw = smem_addr(tc_smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  int grp = 0;
  while (grp + 1 < kMaxGroups && (int)blockIdx.x >= set.first[grp + 1]) ++grp;
  const int tile = blockIdx.x - set.first[grp];
  const int m0 = tile / set.tiles_n[grp] * kBM, n0 = tile % set.tiles_n[grp] * kBN;
  const int N = set.n[grp];
  const GemmGroup& G = set.g[grp];
  const int kc0 = blockIdx.y * set.kchunks_per_split;
  const int nk = min(set.kchunks, kc0 + set.kchunks_per_split) - kc0;
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_addr(&bar_full[s]), 1);
      mbar_init(smem_addr(&bar_empty[s]), 1);
    }
    mbar_init(smem_addr(&bar_done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    s_abort = 0;
    s_consumed = 0;
    s_issued = 0;
  }
  if (warp == 0) tmem_alloc<kBN>(smem_addr(&tmem_slot));
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  if (tid == 0) {
    // producer: TMA copies of K chunk i into stage i % kStages once the MMAs of chunk i - kStages are done
    int i = 0;
    for (; i < nk; ++i) {
      const int s = i % kStages;
      if (i >= kStages && !mbar_wait_parity(smem_addr(&bar_empty[s]), ((i / kStages) - 1) & 1, set.polls)) {
        *abort_flag = 1;
        break;
      }
      if (*abort_flag) break;
      const uint32_t fb = smem_addr(&bar_full[s]);
      mbar_arrive_expect_tx(fb, kStage);
      const uint32_t sa = base + s * kStage, sb = sa + kStageA;
      const int k0 = (kc0 + i) * kBK;
      tma_load_2d(sa, &G.a, fb, k0, m0);
      tma_load_2d(sb, &G.b, fb, k0, n0);
    }
    s_issued = i;
  } else if (tid == 32) {
    // MMA issuer: four K = 16 MMAs per chunk into the TMEM accumulator
    constexpr uint32_t idesc = idesc_bf16(kBM, kBN);
    int i = 0;
    for (; i < nk; ++i) {
      const int s = i % kStages;
      if (!mbar_wait_parity(smem_addr(&bar_full[s]), (i / kStages) & 1, set.polls)) {
        *abort_flag = 1;
        break;
      }
      tc_fence_after();
      const uint32_t sa = base + s * kStage, sb = sa + kStageA;
#pragma unroll
      for (int j = 0; j < kBK / 16; ++j) {
        const uint64_t da = smem_desc_sw128(sa + 32 * j);
        const uint64_t db = smem_desc_sw128(sb + 32 * j);
        mma_bf16_ss(tmem, da, db, idesc, i > 0 || j > 0);
      }
      mma_commit(smem_addr(&bar_empty[s]));
    }
    s_consumed = i;
    mma_commit(smem_addr(&bar_done));
  }
  // every thread: wait for the last MMA (a CTA with nothing consumed still gets the commit)
  if (!mbar_wait_parity(smem_addr(&bar_done), 0, set.polls)) *abort_flag = 1;
  __syncthreads();
  const bool aborted = *abort_flag != 0;
  if (aborted) {
    if (tid == 0) {
      atomicOr(set.err, set.err_bit);
      // copies issued but not consumed, and the final commit, are still landing in shared
      // memory: wait for them before the CTA exits
      for (int i = s_consumed; i < s_issued; ++i)
        mbar_wait_parity(smem_addr(&bar_full[i % kStages]), (i / kStages) & 1, kDrainPolls);
      mbar_wait_parity(smem_addr(&bar_done), 0, kDrainPolls);
    }
  } else if (nk > 0) {
    // epilogue: the two warps of a TMEM lane quarter take 64 columns each, in steps of 32: two loads and
    // one wait, two staged tiles once the previous step's reductions have read them, one proxy fence and
    // one bulk group
    tc_fence_after();
    const int quarter = warp & 3, part = warp >> 2;
    const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16);
    const uint32_t stg = base + (uint32_t)warp * kStageWarp;
    unsigned char* stg_g = tc_smem_raw + (stg - raw);
    const int y = m0 + quarter * 32;
#pragma unroll 1
    for (int cb = part * (kBN / 2); cb < (part + 1) * (kBN / 2); cb += 32) {
      if (n0 + cb >= N) break;
      const int ng = n0 + cb + 16 < N ? 2 : 1;
      uint32_t r[2][16];
      tmem_ld16_async(lane_addr + (uint32_t)cb, r[0]);
      if (ng == 2) tmem_ld16_async(lane_addr + (uint32_t)(cb + 16), r[1]);
      tmem_ld_wait();
      if (cb > part * (kBN / 2)) {
        if (lane == 0) bulk_wait_read<0>();
        __syncwarp();
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (h >= ng) break;
        uint4* d = reinterpret_cast<uint4*>(stg_g + h * 2048 + lane * 64);
#pragma unroll
        for (int k = 0; k < 4; ++k) d[k] = make_uint4(r[h][4 * k], r[h][4 * k + 1], r[h][4 * k + 2], r[h][4 * k + 3]);
      }
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        for (int h = 0; h < ng; ++h) tma_reduce_add_2d(&G.c, stg + (uint32_t)h * 2048u, n0 + cb + 16 * h, y);
        bulk_commit();
      }
      __syncwarp();
    }
    if (lane == 0) bulk_wait_all();
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc<kBN>(tmem);
}

// Launches the `tiles` tiles of a set for K columns, K split over at most ksplit CTAs per tile.
inline cudaError_t launch_gemm_split(GemmSet& set, int tiles, long long K, int ksplit, cudaStream_t st) {
  static bool attr_set[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (!attr_set[dev & 63]) {
    e = cudaFuncSetAttribute(k_gemm_split, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGemmSmem);
    if (e != cudaSuccess) return e;
    attr_set[dev & 63] = true;
  }
  set.kchunks = (int)((K + kBK - 1) / kBK);
  if (ksplit < 1) ksplit = 1;
  set.kchunks_per_split = (set.kchunks + ksplit - 1) / ksplit;
  const int splits = (set.kchunks + set.kchunks_per_split - 1) / set.kchunks_per_split;
  k_gemm_split<<<dim3(tiles, splits), kThreads, kGemmSmem, st>>>(set);
  return cudaGetLastError();
}

}  // namespace tc
}  // namespace bhem
