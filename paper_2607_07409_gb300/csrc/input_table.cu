// The GRU input table G = E W_ih^T [V, 3H] float32 (head preparation): the
// one product of the library with a large M, and the only one bound by the
// tensor cores (2 V 3H D operations against V D 2 + V 3H 4 bytes: 3.8 TFLOP
// and 3.1 GB for the 151936 x 4096 embedding of a 1024-wide GRU).
//
// CTA pairs (cta_group::2): a pair computes a 256 x 256 tile, each CTA
// holding 128 rows of E and 128 rows of W_ih per 64-wide K chunk. One CTA
// alone (128 x 256) would move 48 KB into and 48 KB out of its shared memory
// for every 512 tensor-core cycles, more than the 128 bytes per cycle that
// shared memory has, and read 27 TB/s from L2 over the chip; a pair halves
// W_ih's share (32 KB per CTA). Persistent pairs walk the tiles with the W_ih
// tiles fastest, so that the pairs running at one time share a few row blocks
// of E and all of W_ih (25 MB) in L2: E is read from memory once.
//
// Measured at V = 151936, D = 4096, H = 1024: 2.78 ms, 1.38 PFLOP/s; 32.2 ms
// with one launch of 24 CTAs per 128 rows of E, as it was before.
//
// Roles: warp 0 loads (TMA, a ring of 6 K chunks), warp 1 issues the MMAs (the
// pair's even CTA), warps 4..11 keep the sums and store. The tensor cores
// accumulate a segment of 512 along K at a time in one of two TMEM buffers;
// the sum warps add the segments in registers (128 columns per thread) under
// the next segment's products, rounding to nearest, where one accumulator over
// all of K truncates at every step (error against float64 at D = 4096 4.4e-6
// with one accumulator, 4.8e-7 with segments, for 5 % more time). A tile's stores
// (TMA, through a 4 KB staging buffer per warp) run under the next tile.
#include <algorithm>

#include "dels_device.cuh"

namespace dels {

namespace {

constexpr int kTM = 256, kTN = 256;          // a pair's tile
constexpr int kTK = 64;                      // K chunk (one 128-byte swizzled row)
constexpr int kChunkBytes = 128 * 128;       // 128 rows of one K chunk
constexpr int kRing = 6;                     // K chunks of E and of W_ih that the stages hold
constexpr int kSegChunks = 8;                // K chunks accumulated in TMEM before they are added up
constexpr int kStoreWarps = 8;               // two per TMEM lane quadrant, 128 columns each
constexpr int kStoreBytes = 32 * 128;        // one staging buffer: 32 rows x 32 floats
constexpr int kSumWarp0 = 4;                 // after the loading, issuing and two idle warps of the first warpgroup
constexpr int kThreads = (kSumWarp0 + kStoreWarps) * 32;
// Registers: 168 per thread at launch (12 warps); the first warpgroup keeps
// 56 and the two that hold the sums take 224 (128 x 56 + 256 x 224 = 384 x 168).
constexpr int kRegsFew = 56, kRegsMany = 224;
constexpr int kTableSmem = 2 * kRing * kChunkBytes + kStoreWarps * kStoreBytes + 256 + 1024;

__device__ __forceinline__ void tmem_alloc2(uint32_t* smem_dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_dst)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc2(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_mma2_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive on `bar` (the same offset) in both CTAs of the pair when the MMAs
// issued so far complete.
__device__ __forceinline__ void tc_commit2(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}
// 2-D load into this CTA's shared memory, completing on a barrier of the
// pair given by its cluster address.
__device__ __forceinline__ void tma_load_2d_pair(void* dst, const CUtensorMap* map, uint32_t bar, int x, int y,
                                                 uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4}], [%2], %5;" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d_pair(void* dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z,
                                                 uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4, %5}], [%2], %6;" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, const void* src, int x, int y, uint64_t policy) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group.L2::cache_hint [%0, {%2, %3}], [%1], %4;" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(smem_u32(src)), "r"(x), "r"(y), "l"(policy)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// Grid: whole pairs. mE, mW: boxes of C K chunks x 128 rows; mG: 32 x 32
// (all 128-byte swizzled). Rows past V, columns past O and the K tail read as
// zero and are clipped by the store.
template <int C>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    k_input_table(const __grid_constant__ CUtensorMap mE, const __grid_constant__ CUtensorMap mW,
                  const __grid_constant__ CUtensorMap mG, int V, int O, int D, int* status, uint64_t budget_ns) {
  constexpr int kStages = kRing / C;
  constexpr int kStageBytes = 2 * C * kChunkBytes;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  uint8_t* staging = smem + kStages * kStageBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(staging + kStoreWarps * kStoreBytes);
  uint64_t* full = bars;                 // [kStages], the even CTA's: both CTAs' bytes
  uint64_t* empty = bars + kStages;      // [kStages], in each CTA
  uint64_t* accf = empty + kStages;      // [2], in each CTA
  uint64_t* acce = accf + 2;             // [2], the even CTA's: both CTAs' store warps
  uint64_t* mmadone = acce + 2;          // the even CTA's, after an abort
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mmadone + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();

  if (threadIdx.x == 0) {
    pdl_trigger();
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&full[i], 2);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&accf[i], 1);
      mbar_init(&acce[i], 2 * kStoreWarps);
    }
    mbar_init(mmadone, 1);
    *abort_flag = 0;
    fence_mbarrier_init();
    tma_prefetch_desc(&mE);
    tma_prefetch_desc(&mW);
    tma_prefetch_desc(&mG);
  }
  if (warp == 1) tmem_alloc2(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();   // barriers initialised and TMEM held in both CTAs
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();           // the predecessor may still be writing E, W_ih or reading G

  const int nt = (O + kTN - 1) / kTN;
  const int tiles = ((V + kTM - 1) / kTM) * nt;
  const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
  const int chunks = (D + kTK - 1) / kTK;
  const int fills = (chunks + C - 1) / C;                // stages per tile; the last may hold fewer chunks
  constexpr int kSegFills = kSegChunks / C;
  const int segs = (fills + kSegFills - 1) / kSegFills;  // accumulations per tile

  if (warp < kSumWarp0) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsFew));
    if (warp == 0) {
      if (lane == 0) {
        const uint64_t pol_e = l2_policy_evict_normal();
        const uint64_t pol_w = l2_policy_evict_last();   // read by every pair for every row block
        int f = 0;
        bool ok = true;
        for (int t = pair; t < tiles && ok; t += pairs) {
          const uint64_t deadline = globaltimer_ns() + budget_ns;   // of each tile: a table may take longer
          const int m0 = (t / nt) * kTM + (int)rank * 128, n0 = (t % nt) * kTN + (int)rank * 128;
          for (int k = 0; k < fills; ++k, ++f) {
            const int s = f % kStages;
            ok = mbar_wait(&empty[s], ((f / kStages) & 1) ^ 1, deadline, abort_flag);
            if (!ok) break;
            const uint32_t bar = cluster_map(smem_u32(&full[s]), 0);
            if (rank == 0)
              mbar_arrive_expect_tx(&full[s], 2u * kStageBytes);   // both CTAs' loads
            else
              mbar_arrive_remote(bar);
            uint8_t* dst = smem + s * kStageBytes;
            if constexpr (C == 1) {
              tma_load_2d_pair(dst, &mE, bar, k * kTK, m0, pol_e);
              tma_load_2d_pair(dst + kStageBytes / 2, &mW, bar, k * kTK, n0, pol_w);
            } else {
              tma_load_3d_pair(dst, &mE, bar, 0, m0, k * C, pol_e);
              tma_load_3d_pair(dst + kStageBytes / 2, &mW, bar, 0, n0, k * C, pol_w);
            }
          }
        }
        // after an abort, wait (bounded) for the loads issued to land
        if (!ok && rank == 0) {
          const uint64_t dd = globaltimer_ns() + 100000000ull;
          volatile int dummy = 0;
          for (int k = max(0, f - kStages); k < f; ++k) mbar_wait(&full[k % kStages], (k / kStages) & 1, dd, &dummy);
        }
      }
    } else if (warp == 1) {
      if (lane == 0 && rank == 0) {
        const uint32_t idesc = idesc_bf16_f32(kTM, kTN);
        int f = 0, i = 0;
        bool ok = true;
        for (int t = pair; t < tiles && ok; t += pairs) {
          const uint64_t deadline = globaltimer_ns() + budget_ns;
          for (int k = 0; k < fills && ok; ++i) {
            const int buf = i & 1;
            ok = mbar_wait_cluster(&acce[buf], ((i >> 1) & 1) ^ 1, deadline, abort_flag);
            if (!ok) break;
            tc_fence_after();
            const uint32_t d = tmem + (uint32_t)(buf * kTN);
            const int k0 = k, k1 = min(fills, k + kSegFills);
            for (; k < k1; ++k, ++f) {
              const int s = f % kStages;
              ok = mbar_wait_cluster(&full[s], (f / kStages) & 1, deadline, abort_flag);
              if (!ok) break;
              tc_fence_after();
              const uint32_t ea = smem_u32(smem + s * kStageBytes), wa = ea + kStageBytes / 2;
#pragma unroll
              for (int kk = 0; kk < C * kTK / 16; ++kk) {
                const uint32_t off = (kk / 4) * kChunkBytes + (kk % 4) * 32;
                if (C == 1 || k * C + kk / 4 < chunks)
                  tc_mma2_f16(d, smem_desc_sw128(ea + off), smem_desc_sw128(wa + off), idesc,
                              (k > k0 || kk > 0) ? 1u : 0u);
              }
              tc_commit2(&empty[s]);
            }
            if (ok) tc_commit2(&accf[buf]);
          }
        }
        if (!ok) {
          tc_commit2(mmadone);   // the MMAs issued have completed before TMEM is freed
          volatile int dummy = 0;
          mbar_wait(mmadone, 0, globaltimer_ns() + 100000000ull, &dummy);
        }
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsMany));
    const int q = warp & 3;                                    // TMEM lane quadrant
    const int half = (warp - kSumWarp0) >> 2;                  // columns [128 half, 128 half + 128)
    uint8_t* stage = staging + (warp - kSumWarp0) * kStoreBytes;
    const uint64_t pol = l2_policy_evict_first();
    int i = 0;
    bool ok = true;
    for (int t = pair; t < tiles && ok; t += pairs) {
      const uint64_t deadline = globaltimer_ns() + budget_ns;
      float sum[kTN / 2];
#pragma unroll
      for (int x = 0; x < kTN / 2; ++x) sum[x] = 0.f;
      for (int sg = 0; sg < segs; ++sg, ++i) {
        const int buf = i & 1;
        ok = mbar_wait(&accf[buf], (i >> 1) & 1, deadline, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint32_t base = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * kTN + half * (kTN / 2));
#pragma unroll
        for (int c = 0; c < kTN / 64; ++c) {
          float acc[32];
          tmem_ld_32x32b_x32(base + (uint32_t)(c * 32), acc);
          tmem_ld_wait();
#pragma unroll
          for (int x = 0; x < 32; ++x) sum[c * 32 + x] += acc[x];
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_remote(cluster_map(smem_u32(&acce[buf]), 0));
      }
      if (!ok) break;
      const int m0 = (t / nt) * kTM + (int)rank * 128 + q * 32, n0 = (t % nt) * kTN + half * (kTN / 2);
#pragma unroll
      for (int c = 0; c < kTN / 64; ++c) {
        if (n0 + c * 32 < O) {                                 // not whole chunks past the table's width
          // the staging buffer's previous store has been read out
          if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          __syncwarp();
          float4* dst = reinterpret_cast<float4*>(stage + lane * 128);
#pragma unroll
          for (int k = 0; k < 8; ++k)
            dst[k ^ (lane & 7)] =
                make_float4(sum[c * 32 + 4 * k], sum[c * 32 + 4 * k + 1], sum[c * 32 + 4 * k + 2], sum[c * 32 + 4 * k + 3]);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0 && m0 < V) tma_store_2d(&mG, stage, n0 + c * 32, m0, pol);
        }
      }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync_all();   // no arrival, MMA or load of the pair is outstanding in either CTA
  if (threadIdx.x == 0 && *abort_flag) raise_status(status, DELS_STATUS_TIMEOUT);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc2(tmem, 512);
  }
}

}  // namespace

cudaError_t launch_input_table(const uint16_t* E, const uint16_t* W, float* G, int V, int O, int D, int* status,
                               int sms, cudaStream_t s) {
  CUtensorMap mE, mW, mG;
  // Two K chunks per stage, each operand's as one 3-D box whose rows are
  // 256-byte spans, where the width is whole chunks (the 3-D view has no
  // ragged tail): 2.64 ms for the table above before its segments, against
  // 4.55 ms with one chunk (128-byte spans) per box, which the loads bind (30
  // GB at 6.6 TB/s).
  const bool pair = D % kTK == 0;
  auto load_map = [&](CUtensorMap* m, const uint16_t* x, int rows) {
    return pair ? encode_tmap_3d(m, x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, kTK, (uint64_t)rows, (uint64_t)(D / kTK),
                                 (uint64_t)D * 2, 2 * kTK, kTK, 128, 2, CU_TENSOR_MAP_SWIZZLE_128B)
                : encode_tmap_2d(m, x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (uint64_t)D, (uint64_t)rows,
                                 (uint64_t)D * 2, kTK, 128, CU_TENSOR_MAP_SWIZZLE_128B);
  };
  if (!load_map(&mE, E, V) || !load_map(&mW, W, O) ||
      !encode_tmap_2d(&mG, G, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, (uint64_t)O, (uint64_t)V, (uint64_t)O * 4, 32, 32,
                      CU_TENSOR_MAP_SWIZZLE_128B))
    return cudaErrorInvalidValue;
  auto kern = pair ? k_input_table<2> : k_input_table<1>;
  cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), kTableSmem);
  if (e != cudaSuccess) return e;
  const long long tiles = ((long long)(V + kTM - 1) / kTM) * ((O + kTN - 1) / kTN);
  const int pairs = (int)std::min<long long>(tiles, std::max(1, sms / 2));
  return launch_pdl(kern, dim3(2 * pairs), dim3(kThreads), kTableSmem, s, mE, mW, mG, V, O, D, status,
                    kWaitBudgetNs);
}

}  // namespace dels
