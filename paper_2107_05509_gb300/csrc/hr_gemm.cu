// BF16 GEMM on the 5th-generation tensor cores (tcgen05) for the learned proposal
// network: C[M][N] = act(A[M][K] B[N][K]^T + bias), A and B bf16 with K contiguous,
// accumulation in float32 in tensor memory, C stored as bf16 or float32.
//
// Large products take k_gemm_pair below.  Of the others, one CTA computes a 128 x BN tile:
//   warp 0      TMA producer: 128 x 64 tiles of A and BN x 64 tiles of B into a ring of
//               shared-memory stages (128-byte swizzle), one mbarrier per stage that
//               completes when both copies have landed
//   warp 1      allocates BN tensor-memory columns; one thread issues the
//               tcgen05.mma (M = 128, N = BN, K = 16) of every stage and commits each
//               stage back to the producer, and the last one to the epilogue
//   warps 2-5   epilogue: tcgen05.ld of the accumulator rows of their lane quarter,
//               bias, ReLU, conversion, stores
// Split-K (gridDim.z > 1): CTA z takes K range z of gridDim.z and writes float32
// partials to C + z * ldc_split (no bias, no activation); a separate reduction sums
// them in split order.
//
// Every mbarrier wait is bounded (about one second of device time); a wait that
// runs out sets a status bit, the CTA stops issuing work, waits (bounded) for its own
// copies and products in flight (drain_fills), frees its tensor memory and returns.
#include <algorithm>
#include <mutex>

#include "hr_tcgen05.cuh"

namespace hr {

namespace {

constexpr int kBM = 128, kBK = 64, kStages = 3, kGemmThreads = 192;

struct GemmArgs {
  int M, N, K;
  int kt_per_split;    // 64-wide K steps per split
  const float* bias;   // [N] or null
  int relu;
  void* C;
  int ldc;             // elements
  long long split_stride;   // elements between split outputs (split-K partials)
  int out_bf16;
  int rows16;               // every row of a bf16 C starts on 16 bytes
  Guard guard;
};

// 16 columns of a warp's 32 rows (lane: row row0 + lane): bias, ReLU, conversion (bias null
// and relu 0 for split partials).  bf16 rows that start on 16 bytes take a lane's 16 values
// as two vectors (a sector each); others go through the warp's 32 x 17 floats of shared
// memory, so that a store covers two rows' 16 consecutive values instead of one value of 32
// rows (float32, 4471 x 2863 x 128: 58 -> 23 us; of aligned rows, where a vector store of
// 32 rows touched 32 sectors in halves, 2304 x 2304 x 256: 19 -> 17 us).
constexpr int kXpose = 32 * 17;
__device__ __forceinline__ void store16(const GemmArgs& g, int row0, int col, long long offset, float (&v)[16], float* xp) {
  const int lane = threadIdx.x & 31;
  if (g.bias) {
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (col + i < g.N) v[i] += g.bias[col + i];
  }
  if (g.relu) {
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = fmaxf(v[i], 0.0f);
  }
  if (g.out_bf16 && g.rows16 && col + 16 <= g.N) {
    if (row0 + lane >= g.M) return;
    const size_t o = (size_t)(row0 + lane) * g.ldc + col;
    uint4* out = reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(g.C) + o);
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = pack_bf16(v[2 * i], v[2 * i + 1]);
    out[0] = make_uint4(w[0], w[1], w[2], w[3]);
    out[1] = make_uint4(w[4], w[5], w[6], w[7]);
    return;
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 16; ++i) xp[lane * 17 + i] = v[i];
  __syncwarp();
  const int c = col + (lane & 15);
  if (c >= g.N) return;
#pragma unroll 4
  for (int r = lane >> 4; r < 32 && row0 + r < g.M; r += 2) {
    const size_t o = (size_t)(row0 + r) * g.ldc + c;
    const float x = xp[r * 17 + (lane & 15)];
    if (g.out_bf16) reinterpret_cast<__nv_bfloat16*>(g.C)[o] = __float2bfloat16_rn(x);
    else reinterpret_cast<float*>(g.C)[offset + o] = x;
  }
}

template <int BN>
__global__ void __launch_bounds__(kGemmThreads, 1) k_gemm_bf16(const __grid_constant__ CUtensorMap tmA,
                                                               const __grid_constant__ CUtensorMap tmB,
                                                               GemmArgs g) {
  constexpr int kTmemCols = BN < 32 ? 32 : BN;
  constexpr uint32_t kABytes = kBM * kBK * 2, kBBytes = BN * kBK * 2;
  extern __shared__ __align__(1024) unsigned char gsm_raw[];
  // 1024-byte aligned stage buffers (the 128-byte swizzle pattern repeats every 1024 B)
  unsigned char* base =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(gsm_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* sA = base;
  unsigned char* sB = base + kStages * kABytes;
  __shared__ __align__(8) uint64_t full_bar[kStages], empty_bar[kStages], done_bar;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  __shared__ float xpose[4][kXpose];

  const int warp = warp_id(), lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * kBM, n0 = blockIdx.y * BN;
  const int kt0 = blockIdx.z * g.kt_per_split;
  const int kt_total = (g.K / kBK);
  const int nkt = max(0, min(g.kt_per_split, kt_total - kt0));

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    mbar_init(smem_u32(&done_bar), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc<kTmemCols>(smem_u32(&tmem_base));
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;

  if (warp == 0) {
    // producer
    const bool leader = elect_one();
    int issued = 0;
    for (int kt = 0; kt < nkt; ++kt) {
      const int s = kt % kStages;
      if (kt >= kStages && !mbar_wait(smem_u32(&empty_bar[s]), ((kt / kStages) + 1) & 1, g.guard.waits.clocks)) {
        if (lane == 0) set_status(g.guard.status, kStatusTimeout);
        atomicExch(&abort_flag, 1);
        break;
      }
      if (*reinterpret_cast<volatile int*>(&abort_flag)) break;
      const uint32_t fb = smem_u32(&full_bar[s]);
      if (leader) {
        mbar_expect_tx(fb, kABytes + kBBytes);
        tma_load_2d(smem_u32(sA + s * kABytes), &tmA, (kt0 + kt) * kBK, m0, fb);
        tma_load_2d(smem_u32(sB + s * kBBytes), &tmB, (kt0 + kt) * kBK, n0, fb);
      }
      ++issued;
    }
    drain_fills<kStages>(full_bar, issued);   // copies still in flight must land before the CTA may exit
  } else if (warp == 1) {
    // MMA issuer
    constexpr uint32_t idesc = mma_idesc(kBM, BN);
    const bool leader = elect_one();
    const uint32_t a0 = desc_lo(smem_u32(sA)), b0 = desc_lo(smem_u32(sB));
    for (int kt = 0; kt < nkt; ++kt) {
      const int s = kt % kStages;
      if (kt == g.guard.waits.stop || !mbar_wait(smem_u32(&full_bar[s]), (kt / kStages) & 1, g.guard.waits.clocks)) {
        if (lane == 0) set_status(g.guard.status, kStatusTimeout);
        atomicExch(&abort_flag, 1);
        break;
      }
      tc_fence_after();
      if (leader) {
        mma_step(tmem, a0 + s * (kABytes >> 4), b0 + s * (kBBytes >> 4), idesc, kt > 0);
        mma_commit(smem_u32(&empty_bar[s]));   // the stage is free once these MMAs have read it
      }
    }
    // all products, or those issued before giving up: the epilogue waits for them either way
    if (leader) {
      if (nkt > 0) mma_commit(smem_u32(&done_bar));
      else mbar_arrive(smem_u32(&done_bar));
    }
  } else if (warp >= 2) {
    // epilogue: warp w reads tensor-memory lanes 32 (w % 4) .. + 31 = tile rows
    const bool ok = mbar_wait(smem_u32(&done_bar), 0, kWaitClocks);
    tc_fence_after();
    if (!ok) {
      set_status(g.guard.status, kStatusTimeout);
    } else if (!*reinterpret_cast<volatile int*>(&abort_flag)) {
      const int q = warp & 3;
      const bool split = gridDim.z > 1;
      for (int c = 0; c < BN; c += 16) {
        float v[16];
        if (nkt > 0) {
          tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c, v);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = 0.0f;
        }
        if (n0 + c < g.N) store16(g, m0 + q * 32, n0 + c, split ? blockIdx.z * g.split_stride : 0, v, xpose[warp - 2]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    mbar_wait(smem_u32(&done_bar), 0, kWaitClocks);   // (an epilogue that gave up has not waited for the products)
    tc_fence_after();
    tmem_free<kTmemCols>(tmem);
  }
}

// Large products on pairs of SMs: a tile of C is 256 x 256, each CTA of a pair stages its
// 128 rows of A and half of the tile's columns of B (32 KB per 64-wide K step, five stages)
// and holds 128 rows of the accumulator; one thread of the first CTA issues the products
// of both (cta_group::2).  A 128 x 128 tile reads 128 bytes of shared memory per clock,
// all that an SM has, and asks L2 for 20 TB/s; the pair's reads 64 and asks for half.
// 8192^3 bf16: 775 -> 582 us, 97 % of cuBLAS's burst rate on this chip.  The two
// accumulators (all 512 columns) alternate, so that a tile's epilogue runs
// beside the next tile's products; CTA pairs take tiles in turn, eight tile rows at a
// time, which keeps the operands that they share in L2.
//   warp 0      TMA loads of the CTA's halves, counted on the first CTA's barriers
//   warp 1      the first CTA's: products; commits arrive on both CTAs' barriers
//   warps 2-9   epilogue of the CTA's 128 rows, columns by halves
// Waits are bounded as above; the CTAs of a pair end together.
constexpr int kPairM = 256, kPairN = 256, kPairStages = 5, kPairRows = 8, kPairThreads = 320;
constexpr uint32_t kPairHalf = 128 * kBK * 2;   // bytes of a CTA's part of A or B
constexpr size_t kPairSmem = 1024 + kPairStages * 2 * (size_t)kPairHalf;

// tile t in the order of the pairs: kPairRows tile rows, column after column
__device__ __forceinline__ void pair_tile(int t, int tm, int tn, int& m, int& n) {
  const int band = t / (kPairRows * tn), in = t - band * kPairRows * tn;
  const int rows = min(kPairRows, tm - band * kPairRows);
  m = band * kPairRows + in % rows;
  n = in / rows;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
    k_gemm_pair(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, GemmArgs g) {
  constexpr int S = kPairStages;
  extern __shared__ __align__(1024) unsigned char gsm_raw[];
  unsigned char* sA = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(gsm_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* sB = sA + S * kPairHalf;
  __shared__ __align__(8) uint64_t full[S], empty[S], acc_full[2], acc_empty[2], drained;
  __shared__ uint32_t tmem_slot;
  __shared__ int gave_up, filled[2];   // of the pair (both CTAs write them); filled: the first CTA's
  __shared__ float xpose[8][kXpose];
  const Waits& waits = g.guard.waits;
  const int warp = warp_id(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int tm = (g.M + kPairM - 1) / kPairM, tn = (g.N + kPairN - 1) / kPairN, tiles = tm * tn;
  const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1, nkt = g.K / kBK;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&acc_full[b]), 1);
      mbar_init(smem_u32(&acc_empty[b]), 16);   // the epilogue warps of both CTAs
    }
    mbar_init(smem_u32(&drained), 1);
    gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc_pair<512>(smem_u32(&tmem_slot));
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  bool ok = true;
  if (warp == 0) {
    const bool leader = elect_one();
    int s = 0, issued = 0;
    uint32_t phase = 0;
    for (int t = pair; ok && t < tiles; t += pairs) {
      int m, n;
      pair_tile(t, tm, tn, m, n);
      const int ma = m * kPairM + 128 * (int)rank, nb = n * kPairN + 128 * (int)rank;
      for (int kt = 0; kt < nkt; ++kt) {
        if (!(ok = mbar_wait(smem_u32(&empty[s]), phase ^ 1, waits.clocks))) break;
        ++issued;
        if (leader) {
          if (rank == 0) mbar_expect_tx(smem_u32(&full[s]), 4 * kPairHalf);
          const uint32_t fb = cluster_addr(smem_u32(&full[s]), 0);
          tma_load_2d_pair(smem_u32(sA + s * kPairHalf), &tmA, kt * kBK, ma, fb);
          tma_load_2d_pair(smem_u32(sB + s * kPairHalf), &tmB, kt * kBK, nb, fb);
        }
        if (++s == S) s = 0, phase ^= 1;
      }
    }
    if (lane == 0) store_cluster(cluster_addr(smem_u32(&filled[rank]), 0), issued);
  } else if (warp == 1 && rank == 0) {
    constexpr uint32_t idesc = mma_idesc(kPairM, kPairN);
    const bool leader = elect_one();
    const uint32_t a0 = desc_lo(smem_u32(sA)), b0 = desc_lo(smem_u32(sB));
    int s = 0, it = 0, step = 0;
    uint32_t phase = 0;
    for (int t = pair; ok && t < tiles; t += pairs, ++it) {
      const int b = it & 1;
      if (!(ok = mbar_wait_cluster(smem_u32(&acc_empty[b]), ((it >> 1) & 1) ^ 1, waits.clocks))) break;
      tc_fence_after();
      for (int kt = 0; kt < nkt; ++kt) {
        if (!(ok = step++ != waits.stop && mbar_wait(smem_u32(&full[s]), phase, waits.clocks))) break;
        tc_fence_after();
        if (leader) {
          mma_step_pair(tmem + b * kPairN, a0 + s * (kPairHalf >> 4), b0 + s * (kPairHalf >> 4), idesc, kt > 0);
          mma_commit_pair(smem_u32(&empty[s]));
        }
        if (++s == S) s = 0, phase ^= 1;
      }
      if (ok && leader) mma_commit_pair(smem_u32(&acc_full[b]));
    }
  } else if (warp >= 2) {
    const int q = warp & 3, half = warp < 6 ? 0 : kPairN / 2;
    int it = 0;
    for (int t = pair; t < tiles; t += pairs, ++it) {
      const int b = it & 1;
      int m, n;
      pair_tile(t, tm, tn, m, n);
      const int row0 = m * kPairM + 128 * (int)rank + q * 32;
      if (!(ok = mbar_wait(smem_u32(&acc_full[b]), (it >> 1) & 1, waits.clocks))) break;
      tc_fence_after();
      for (int c = half; c < half + kPairN / 2; c += 16) {
        float v[16];
        tmem_ld16(tmem + b * kPairN + ((uint32_t)(q * 32) << 16) + (uint32_t)c, v);
        if (row0 < g.M && n * kPairN + c < g.N) store16(g, row0, n * kPairN + c, 0, v, xpose[warp - 2]);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(cluster_addr(smem_u32(&acc_empty[b]), 0));
    }
  }
  if (!ok && lane == 0) {
    set_status(g.guard.status, kStatusTimeout);
    for (uint32_t r = 0; r < 2; ++r) store_cluster(cluster_addr(smem_u32(&gave_up), r), 1);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();   // no CTA ends while the other's copies, products or arrivals may reach it
  if (gave_up) {    // (otherwise the products have waited for the copies, the epilogues for the products)
    if (warp == 0 && rank == 0) drain_fills<S>(full, max(filled[0], filled[1]));   // both CTAs' copies count here
    if (warp == 1) {
      if (rank == 0 && elect_one()) mma_commit_pair(smem_u32(&drained));
      mbar_wait_cluster(smem_u32(&drained), 0, kWaitClocks);
    }
    __syncthreads();
    cluster_sync();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_free_pair<512>(tmem);
  }
}

// fixed-order sum of split-K partials: out[i] = act(sum_z part[z][i] + bias[col])
__global__ void k_split_reduce(const float* __restrict__ part, int splits, long long stride, int M, int N, int ldc,
                               const float* __restrict__ bias, int relu, void* out, int ldo, int out_bf16) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)M * N) return;
  const int r = (int)(i / N), c = (int)(i % N);
  float acc = 0.0f;
  for (int z = 0; z < splits; ++z) acc += part[z * stride + (size_t)r * ldc + c];
  if (bias) acc += bias[c];
  if (relu) acc = fmaxf(acc, 0.0f);
  if (out_bf16)
    reinterpret_cast<__nv_bfloat16*>(out)[(size_t)r * ldo + c] = __float2bfloat16_rn(acc);
  else
    reinterpret_cast<float*>(out)[(size_t)r * ldo + c] = acc;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

std::mutex g_encode_mutex;
EncodeTiledFn g_encode = nullptr;

EncodeTiledFn encode_fn() {
  std::lock_guard<std::mutex> lock(g_encode_mutex);
  if (!g_encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
      cudaGetLastError();
      return nullptr;
    }
    g_encode = reinterpret_cast<EncodeTiledFn>(fn);
  }
  return g_encode;
}

// Pairs where there is a tile for nearly every pair and a reduction long enough to cover
// the coarser last round.  Measured, 128 x 128 tiles -> pairs, us: 8192^3 758 -> 582,
// 4096^3 106 -> 84, 3072 x 3072 x 2048 35.2 -> 28.7, 2048 x 2048 x 2048 (64 tiles) 18.5 ->
// 18.0; but 1792 x 1792 x 2048 (49 tiles) 18.7 -> 19.0, 2304 x 2304 x 512 (81) 16.7 -> 17.6
// and 3072 x 3072 x 128 14.4 -> 16.4.
bool use_pair(int M, int N, int K) {
  const long long tiles = (long long)((M + kPairM - 1) / kPairM) * ((N + kPairN - 1) / kPairN);
  return N > 64 && tiles >= 64 && K >= 512 && tiles * K >= 65536;
}

template <int BN>
size_t gemm_smem() {
  return 1024 + (size_t)kStages * (kBM * kBK * 2 + BN * kBK * 2);
}

template <int BN>
int launch_gemm_bn(const CUtensorMap& ta, const CUtensorMap& tb, const GemmArgs& g, int splits, cudaStream_t s) {
  const size_t smem = gemm_smem<BN>();
  dim3 grid((g.M + kBM - 1) / kBM, (g.N + BN - 1) / BN, splits);
  k_gemm_bf16<BN><<<grid, kGemmThreads, smem, s>>>(ta, tb, g);
  HR_CHECK_LAUNCH();
  return HR_OK;
}

}  // namespace

bool tma_map(CUtensorMap* map, const void* ptr, long long rows, int cols, int ld, int box_rows) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int configure_gemm_kernels() {
  if (cudaFuncSetAttribute(k_gemm_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPairSmem) != cudaSuccess ||
      cudaFuncSetAttribute(k_gemm_bf16<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem<32>()) !=
          cudaSuccess ||
      cudaFuncSetAttribute(k_gemm_bf16<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem<64>()) !=
          cudaSuccess ||
      cudaFuncSetAttribute(k_gemm_bf16<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem<128>()) !=
          cudaSuccess) {
    cudaGetLastError();
    return HR_ERR_CUDA;
  }
  return HR_OK;
}

int launch_gemm(const void* A, int lda, const void* Bm, int ldb, int M, int N, int K, const float* bias, int relu,
                void* C, int ldc, int out_bf16, int splits, float* split_buf, Guard guard, cudaStream_t s) {
  if (M < 1 || N < 1 || K < kBK || K % kBK != 0 || lda < K || ldb < K || lda % 8 || ldb % 8 || splits < 1)
    return HR_ERR_ARG;
  if ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(Bm)) & 15) return HR_ERR_ARG;
  const int BN = N <= 32 ? 32 : (N <= 64 ? 64 : 128);
  CUtensorMap ta, tb;
  if (!tma_map(&ta, A, M, K, lda, kBM) || !tma_map(&tb, Bm, N, K, ldb, BN)) return HR_ERR_CUDA;
  const int kt_total = K / kBK;
  if (splits > kt_total) splits = kt_total;
  GemmArgs g;
  g.M = M;
  g.N = N;
  g.K = K;
  g.kt_per_split = (kt_total + splits - 1) / splits;
  splits = (kt_total + g.kt_per_split - 1) / g.kt_per_split;
  g.guard = guard;
  if (splits > 1) {
    if (!split_buf) return HR_ERR_ARG;
    g.bias = nullptr;
    g.relu = 0;
    g.C = split_buf;
    g.ldc = N;
    g.split_stride = (long long)M * N;
    g.out_bf16 = 0;
  } else {
    g.bias = bias;
    g.relu = relu;
    g.C = C;
    g.ldc = ldc;
    g.split_stride = 0;
    g.out_bf16 = out_bf16;
  }
  g.rows16 = (reinterpret_cast<uintptr_t>(g.C) | (uintptr_t)g.ldc * 2) % 16 == 0;
  const long long pair_tiles = (long long)((M + kPairM - 1) / kPairM) * ((N + kPairN - 1) / kPairN);
  if (splits == 1 && use_pair(M, N, K)) {
    k_gemm_pair<<<(unsigned)(2 * std::min<long long>(pair_tiles, sm_count() / 2)), kPairThreads, kPairSmem, s>>>(ta, tb, g);
    HR_CHECK_LAUNCH();
    return HR_OK;
  }
  int rc = BN == 32 ? launch_gemm_bn<32>(ta, tb, g, splits, s)
                    : (BN == 64 ? launch_gemm_bn<64>(ta, tb, g, splits, s) : launch_gemm_bn<128>(ta, tb, g, splits, s));
  if (rc != HR_OK || splits == 1) return rc;
  const long long n = (long long)M * N;
  k_split_reduce<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(split_buf, splits, (long long)M * N, M, N, N, bias, relu,
                                                             C, ldc, out_bf16);
  HR_CHECK_LAUNCH();
  return HR_OK;
}

}  // namespace hr
