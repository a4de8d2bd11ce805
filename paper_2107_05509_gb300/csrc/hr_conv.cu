// Convolutions of the proposal network on the 5th-generation tensor cores without
// column matrices: 3x3, stride 2, padding 1, NHWC bf16, float32 accumulation.
//
//   k_conv_fwd    Y = relu(W * X + b): a tile is 128 output pixels x Cout; its A operand
//                 (pixels x 64 of the 9 Cin products) is gathered from X straight into
//                 swizzled shared memory, 16 bytes (8 channels of one tap) per copy
//   k_conv_dgrad  dX through one parity class of input pixels: pixel (2i + py, 2j + px) is
//                 read by 1, 2 or 4 of the taps, each from the output pixel (i + dy, j +
//                 dx); a tap's product dPre W_tap has its own accumulator columns, is
//                 rounded to bf16 and added in tap order (the rounding of a bf16 column
//                 matrix and its gather), and the ReLU mask of the layer below is applied
//   k_wgrad       dW^T = cols^T dPre and db: both operands MN-major (the reduction runs
//                 over pixels, the slow dimension of both), so nothing is transposed;
//                 the columns are gathered as in the forward, or (dense layers) loaded
//
// A column matrix is 9 / 4 of its input in values and was written and read once per
// product; the gather reads the input itself (the overlapping taps from L1 and L2).
// What bounds it now is L1's data path: the copies write shared memory one 32-byte
// sector per clock (73 % of its wavefronts in the first layer), whichever instruction
// makes them and whether one or two CTAs share an SM.  For 1024 views: forward 7.4 ms
// (of which 6.8 in column matrices) -> 0.45 ms, backward 15.5 ms -> 1.1 ms.
//
// Roles of a CTA's warps: 0 TMA loads of the other operand, 1 the product's issue, 2-9
// two groups of epilogue warps (taking tiles in turn), 10-17 the gather, each warp filling
// whole stages in turn (a stage costs its warp a wait for the slot, one for the copies and
// a proxy fence, about a microsecond in all, which eight warps hide).  Stages of the
// ring run on from tile to tile and the accumulators are double-buffered, so that a
// tile's epilogue runs beside the next tiles' products.  Every mbarrier wait is bounded;
// one that runs out sets a status bit, its role stops, the others' waits run out
// likewise, copies and products in flight are waited for and tensor memory is freed.
#include <algorithm>

#include "hr_tcgen05.cuh"

namespace hr {

namespace {

typedef __nv_bfloat16 bf16;

constexpr int kGatherWarp = 10, kGatherWarps = 8, kThreads = 32 * (kGatherWarp + kGatherWarps);
constexpr int kTileM = 128, kStep = 64;   // pixels per tile, products per stage
constexpr uint32_t kABytes = kTileM * kStep * 2;

// 16-byte copy global -> shared, zeros when !in
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool in) {
  const int n = in ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
// the warp's copies have landed and are visible to the tensor core's reads: the stage is
// full as far as this warp is concerned
__device__ __forceinline__ void finish_stage(uint64_t* full) {
  asm volatile("cp.async.wait_all;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(smem_u32(full));
}

__device__ __forceinline__ void store32(void* p, const uint32_t (&w)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]),
               "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}
__device__ __forceinline__ void load32(const void* p, uint32_t (&w)[8]) {
  asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
               : "l"(p));
}

// Where a tile's rows and products lie in the gathered tensor: row (v, i, j) of a grid of
// Ho x Ho per view (Ho = 1 << lo <= 128), product k = (tap k >> lc, channel k & (C - 1));
// the value is src[v][stride i + dy][stride j + dx][channel], zero outside the view's
// side Hs = 1 << ls and for taps >= ntap.  Ho is a power of two, so the rows of an aligned
// group of 64 or 128 lie the same way from the group's first row in every group: their
// offsets are worked out once, into shared memory.
struct Gather {
  const bf16* src;
  int lc, ls, lo, stride, ntap;
  int M;                  // rows
  signed char dy[9], dx[9];
};
// (offset in elements, row, column) from the group's first pixel
__device__ __forceinline__ int4 gather_row(const Gather& g, int r) {
  const int j = r & ((1 << g.lo) - 1), i = (r >> g.lo) & ((1 << g.lo) - 1), v = r >> (2 * g.lo);
  const int y = g.stride * i, x = g.stride * j;
  return make_int4(((v << (2 * g.ls)) + (y << g.ls) + x) << g.lc, y, x, 0);
}
// the group at `row0` (a multiple of its size): its first pixel's address, y its row
__device__ __forceinline__ const bf16* gather_base(const Gather& g, int row0, int& y) {
  const int i = (row0 >> g.lo) & ((1 << g.lo) - 1), v = row0 >> (2 * g.lo);
  y = g.stride * i;
  return g.src + ((((size_t)v << (2 * g.ls)) + ((size_t)y << g.ls)) << g.lc);
}

// The stages in flight hold every gathered pixel 9 / 4 times, so their unique bytes do
// not cover the latency of memory: one thread asks L2 for the pixels of the tiles (or
// steps) ahead.  `bytes` a multiple of 16, p 16-byte aligned.
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
// the pixels that output rows [row0, row0 + n) read first (n rows of the grid are n
// stride^2 consecutive pixels)
__device__ __forceinline__ void prefetch_rows(const Gather& g, int row0, int n) {
  if (row0 >= g.M) return;
  int y;
  const bf16* p = gather_base(g, row0, y);
  prefetch_l2(p, (uint32_t)(min(n, g.M - row0) * g.stride * g.stride) << (g.lc + 1));
}
constexpr int kAheadTiles = 3, kAheadSteps = 16;

// Gather warps at work: at most one per stage.  Warp w fills stages n = w, w + G, ...; a
// wait for slot n % S asks whether the barrier's phase of one parity is complete, which
// is only unambiguous once fill n - 2 S has been used up.  Its previous fill n - G waited
// for the use of fill n - G - S, and fills are used in order, so G <= S makes it certain.
template <int S>
__host__ __device__ constexpr int gather_warps() {
  return S < kGatherWarps ? S : kGatherWarps;
}

struct Ring {   // position in the ring of stages
  int s = 0;
  uint32_t phase = 0;
  template <int S>
  __device__ __forceinline__ void next() {
    if (++s == S) {
      s = 0;
      phase ^= 1;
    }
  }
};

__device__ __forceinline__ unsigned char* align1024(unsigned char* p) {
  return reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

// Units of work: a tile of 128 rows, BN of the output's channels, and (dgrad) one parity
// class of pixels; the classes and channel blocks of a tile run one after another, so
// that their gathers of the same pixels hit L1 and L2.
struct ConvClass {
  int ntap, py, px;
  int btap[4];            // row of each tap in the weights' map
  signed char dy[4], dx[4];
};
struct ConvArgs {
  Gather g;
  int tiles, nkt;         // K-steps per accumulator (a tap's in dgrad, all in fwd)
  int last16;             // K = 16 groups of the last step that hold products
  int nblocks, nclass;    // units per tile
  int C;                  // the output's channels
  const float* bias;      // fwd
  bf16* out;              // fwd [M][C]; dgrad [NV][2 Ho][2 Ho][C]
  const bf16* mask;       // dgrad: the layer's activations (ReLU mask), out's layout
  ConvClass cls[4];
  Guard guard;
};

// What the roles need of each K-step of a tile, worked out once per block into shared
// memory (a tile of the first layer has two steps: per-tile and per-step arithmetic in
// every role's loop took longer than the step itself)
struct Step {
  int off, dy, dx;   // dgrad: the gather's offset (tap and first channel), in pixels
  int tx, ty;        // the weights' tile
  int acc;           // accumulator column
  int groups;        // K = 16 groups that hold products
  int flags;         // 1 first of a unit, 2 last of a unit, 4 first of an accumulator
};
constexpr int kMaxSteps = 40;

template <int BN, bool DGRAD>
struct ConvCfg {
  static constexpr int kAcc = DGRAD ? 4 * BN : BN;   // a class has up to four taps
  static constexpr int kCols = 2 * kAcc < 32 ? 32 : 2 * kAcc;
  static_assert(kCols <= 512, "tensor memory");
  static constexpr uint32_t kBBytes = BN * kStep * 2;
  static constexpr int kStages = BN >= 128 ? 6 : 8;
  static constexpr size_t kSmem = 1024 + kStages * (size_t)(kABytes + kBBytes);
};

template <int BN, bool DGRAD>
__global__ void __launch_bounds__(kThreads, 1) k_conv(const __grid_constant__ CUtensorMap tmB, const __grid_constant__ ConvArgs c) {
  typedef ConvCfg<BN, DGRAD> Cfg;
  constexpr int S = Cfg::kStages;
  extern __shared__ __align__(1024) unsigned char raw[];
  unsigned char* sA = align1024(raw);
  unsigned char* sB = sA + S * kABytes;
  __shared__ __align__(8) uint64_t full[S], empty[S], acc_full[2], acc_empty[2], drained;
  __shared__ uint32_t tmem_slot;
  __shared__ int gave_up;
  const Waits& waits = c.guard.waits;
  __shared__ float sbias[BN];
  __shared__ int4 rows[kTileM];
  __shared__ Step steps[kMaxSteps];
  if (threadIdx.x < kTileM) rows[threadIdx.x] = gather_row(c.g, threadIdx.x);
  const int warp = warp_id(), lane = threadIdx.x & 31;
  const int per_tile = DGRAD ? c.nblocks * c.nclass : 1;
  const int T = DGRAD ? c.nblocks * 9 * c.nkt : c.nkt;   // steps per tile (the classes' taps are all nine)
  if (threadIdx.x == 32) {
    int n = 0;
    for (int u = 0; u < per_tile; ++u) {
      const ConvClass& k = c.cls[DGRAD ? u % c.nclass : 0];
      const int m = DGRAD ? c.nkt * k.ntap : c.nkt;
      for (int st = 0; st < m && n < kMaxSteps; ++st, ++n) {
        Step& e = steps[n];
        const int tap = DGRAD ? st / c.nkt : 0, kt = DGRAD ? st % c.nkt : st;
        e.dy = DGRAD ? k.dy[tap] : 0;
        e.dx = DGRAD ? k.dx[tap] : 0;
        e.off = (((e.dy << c.g.ls) + e.dx) << c.g.lc) + kt * kStep;
        e.tx = kt * kStep;
        e.ty = DGRAD ? k.btap[tap] + (u / c.nclass) * BN : 0;
        e.acc = tap * BN;
        e.groups = !DGRAD && st == m - 1 ? c.last16 : kStep / 16;
        e.flags = (st == 0 ? 1 : 0) | (st == m - 1 ? 2 : 0) | (kt == 0 ? 4 : 0);
      }
    }
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(smem_u32(&full[s]), 2);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&acc_full[b]), 1);
      mbar_init(smem_u32(&acc_empty[b]), 128);
    }
    mbar_init(smem_u32(&drained), 1);
    gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (!DGRAD && threadIdx.x < BN) sbias[threadIdx.x] = c.bias[threadIdx.x];
  if (warp == 1) tmem_alloc<Cfg::kCols>(smem_u32(&tmem_slot));
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  bool ok = true;
  int filled = 0;   // stages whose copies warp 0 has asked for
  if (warp == 0) {
    // the weights' tiles, and the prefetches
    const bool leader = elect_one();
    Ring r;
    for (int tile = blockIdx.x; ok && tile < c.tiles; tile += gridDim.x) {
      const long long ahead = tile + (long long)kAheadTiles * gridDim.x;
      if (leader && ahead < c.tiles) {
        const int row0 = (int)ahead * kTileM;
        prefetch_rows(c.g, row0, kTileM);
        if (DGRAD)   // the mask of the tile's 4 x 128 pixels
          prefetch_l2(c.mask + (size_t)row0 * 4 * c.C, (uint32_t)min(kTileM, c.g.M - row0) * 8 * c.C);
      }
      for (int st = 0; st < T; ++st, r.next<S>()) {
        const int x = steps[st].tx, y = steps[st].ty;
        if (!(ok = mbar_wait(smem_u32(&empty[r.s]), r.phase ^ 1, waits.clocks))) break;
        ++filled;
        const uint32_t fb = smem_u32(&full[r.s]);
        if (leader) {
          mbar_expect_tx(fb, Cfg::kBBytes);
          tma_load_2d(smem_u32(sB + r.s * Cfg::kBBytes), &tmB, x, y, fb);
        }
      }
    }
  } else if (warp == 1) {
    constexpr uint32_t idesc = mma_idesc(kTileM, BN);
    const bool leader = elect_one();
    const uint32_t a0 = desc_lo(smem_u32(sA)), b0 = desc_lo(smem_u32(sB));
    Ring r;
    int it = -1, step = 0;
    for (int tile = blockIdx.x; ok && tile < c.tiles; tile += gridDim.x)
      for (int st = 0; st < T; ++st, r.next<S>()) {
        const Step e = steps[st];
        if (e.flags & 1) {
          ++it;
          if (!(ok = mbar_wait(smem_u32(&acc_empty[it & 1]), ((it >> 1) & 1) ^ 1, waits.clocks))) break;
        }
        if (!(ok = step++ != waits.stop && mbar_wait(smem_u32(&full[r.s]), r.phase, waits.clocks))) break;
        tc_fence_after();
        if (leader) {
          const uint32_t a = a0 + r.s * (kABytes >> 4), b = b0 + r.s * (Cfg::kBBytes >> 4);
          const uint32_t d = tmem + (it & 1) * Cfg::kAcc + e.acc;
          if (e.groups == kStep / 16) {
            mma_step(d, a, b, idesc, !(e.flags & 4));
          } else {
            for (int k = 0; k < e.groups; ++k) mma_bf16(d, a + 2 * k, b + 2 * k, idesc, !(e.flags & 4) || k > 0);
          }
          mma_commit(smem_u32(&empty[r.s]));
          if (e.flags & 2) mma_commit(smem_u32(&acc_full[it & 1]));
        }
      }
  } else if (warp >= 2 && warp < kGatherWarp) {
    const int q = warp & 3, grp = (warp - 2) >> 2;   // tensor-memory lanes 32 q .. of this warp
    int it = 0;
    for (int tile = blockIdx.x; ok && tile < c.tiles; tile += gridDim.x)
      for (int u = 0; ok && u < per_tile; ++u, ++it) {
        const int b = it & 1, use = it >> 1;
        if (b != grp) continue;
        const int row = tile * kTileM + q * 32 + lane;
        const bool in = row < c.g.M;
        size_t o = (size_t)row * c.C;
        int ntap = 1;
        uint32_t y[DGRAD ? BN / 2 : 1];
        if (DGRAD) {
          const ConvClass& k = c.cls[u % c.nclass];
          ntap = k.ntap;
          const int j = row & ((1 << c.g.lo) - 1), i = (row >> c.g.lo) & ((1 << c.g.lo) - 1), v = row >> (2 * c.g.lo);
          const int side = 2 << c.g.lo;
          o = (((size_t)v * side + 2 * i + k.py) * side + 2 * j + k.px) * c.C + (u / c.nclass) * BN;
          // the row's mask, on its way while the products run
#pragma unroll
          for (int n = 0; n < BN; n += 16)
            if (in) load32(c.mask + o + n, *reinterpret_cast<uint32_t(*)[8]>(&y[n / 2]));
        }
        if (!(ok = mbar_wait(smem_u32(&acc_full[b]), use & 1, waits.clocks))) break;
        tc_fence_after();
        const uint32_t t0 = tmem + b * Cfg::kAcc + ((uint32_t)(q * 32) << 16);
#pragma unroll
        for (int n = 0; n < BN; n += 16) {
          float x[16];
          tmem_ld16(t0 + n, x);
          uint32_t w[8];
          if (!DGRAD) {
#pragma unroll
            for (int e = 0; e < 16; ++e) x[e] = fmaxf(x[e] + sbias[n + e], 0.0f);
          } else {
#pragma unroll
            for (int e = 0; e < 16; ++e) x[e] = __bfloat162float(__float2bfloat16_rn(x[e]));
            for (int t = 1; t < ntap; ++t) {
              float z[16];
              tmem_ld16(t0 + t * BN + n, z);
#pragma unroll
              for (int e = 0; e < 16; ++e) x[e] += __bfloat162float(__float2bfloat16_rn(z[e]));
            }
          }
#pragma unroll
          for (int e = 0; e < 8; ++e) w[e] = pack_bf16(x[2 * e], x[2 * e + 1]);
          if (DGRAD) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {   // activations are >= 0: non-zero bits are positive values
              if (!(y[n / 2 + e] & 0x7fffu)) w[e] &= 0xffff0000u;
              if (!(y[n / 2 + e] & 0x7fff0000u)) w[e] &= 0x0000ffffu;
            }
          }
          if (in) store32(c.out + o + n, w);
        }
        tc_fence_before();
        mbar_arrive(smem_u32(&acc_empty[b]));
      }
  } else if (warp >= kGatherWarp && warp < kGatherWarp + gather_warps<S>()) {
    // lane's 16-byte column of a row, 8 lanes per row, rows rr, rr + 4, ... of the tile;
    // every G-th stage
    constexpr int G = gather_warps<S>();
    const int q = lane & 7, rr = lane >> 3;
    const int Hs = 1 << c.g.ls, C = 1 << c.g.lc;
    int tile = blockIdx.x, st = warp - kGatherWarp;
    Ring r;
    r.s = st;
    for (;;) {
      for (; st >= T; st -= T) tile += gridDim.x;
      if (tile >= c.tiles) break;
      int yb, off, dy = 0, dx = 0;
      const bf16* base = gather_base(c.g, tile * kTileM, yb);
      const int left = c.g.M - tile * kTileM;
      bool tv = true;
      if (DGRAD) {
        off = steps[st].off + 8 * q;
        dy = steps[st].dy;
        dx = steps[st].dx;
      } else {
        const int k = st * kStep + 8 * q, tap = k >> c.g.lc;
        tv = tap < c.g.ntap;
        if (tv) {   // tap = 3 (dy + 1) + dx + 1
          dy = (tap * 11) >> 5;
          dx = tap - 3 * dy - 1;
          dy -= 1;
        }
        off = ((dy << c.g.ls) + dx) * C + (k & (C - 1));
      }
      const bool used = DGRAD || q < 2 * steps[st].groups;   // the others are not read
      if (!(ok = mbar_wait(smem_u32(&empty[r.s]), r.phase ^ 1, waits.clocks))) break;
      if (used) {
        const bf16* p = base + off;
        const int y0 = tv ? yb + dy : Hs;   // Hs: every row is outside
        uint32_t dst = smem_u32(sA) + r.s * kABytes + rr * 128;
#pragma unroll 8
        for (int rw = rr; rw < kTileM; rw += 4, dst += 512) {
          const int4 o = rows[rw];
          const bool in = (unsigned)(y0 + o.y) < (unsigned)Hs && (unsigned)(o.z + dx) < (unsigned)Hs && rw < left;
          cp16(dst + ((q ^ (rw & 7)) << 4), in ? p + o.x : c.g.src, in);
        }
      }
      finish_stage(&full[r.s]);
      st += G;
      if ((r.s += G) >= S) {
        r.s -= S;
        r.phase ^= 1;
      }
    }
  }
  if (!ok && lane == 0) {
    set_status(c.guard.status, kStatusTimeout);
    gave_up = 1;
  }
  tc_fence_before();
  __syncthreads();
  if (gave_up) {   // (otherwise the products have waited for the copies, the epilogue for the products)
    if (warp == 0) drain_fills<S>(full, filled);
    if (warp == 1) {
      if (elect_one()) mma_commit(smem_u32(&drained));
      mbar_wait(smem_u32(&drained), 0, kWaitClocks);
    }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_free<Cfg::kCols>(tmem);
  }
}

// dW^T tile: 128 products x BN outputs over the pixels of one split.  Stage: 64 pixels x
// 128 products (two blocks of 64) and 64 pixels x BN outputs, both rows of 128 bytes per
// pixel.  The column sums of dPre (the bias gradient) are taken from the staged tiles by
// the epilogue's warps of the first product tile's CTAs.
constexpr int kMaxSplits = 128;
struct WgradArgs {
  Gather g;               // GATHER: the columns
  const bf16* dpre;
  int steps_total, steps_per_split, splits;
  int K, N;               // products (rows of dW^T), outputs
  float* part;            // [splits][K][N]
  float* bias_part;       // [splits][N]
  Guard guard;
};

template <int BN>
struct WgradCfg {
  static constexpr int kBBlocks = BN > 64 ? 2 : 1;
  static constexpr uint32_t kBBytes = kBBlocks * 64 * 128;
  static constexpr int kStages = BN > 64 ? 6 : 8;
  static constexpr size_t kSmem = 1024 + kStages * (size_t)(kABytes + kBBytes);
};

template <int BN, bool GATHER>
__global__ void __launch_bounds__(kThreads, 1) k_wgrad(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                                                       const __grid_constant__ WgradArgs c) {
  typedef WgradCfg<BN> Cfg;
  constexpr int S = Cfg::kStages;
  constexpr int kCols = BN < 32 ? 32 : BN;
  extern __shared__ __align__(1024) unsigned char raw[];
  unsigned char* sA = align1024(raw);
  unsigned char* sB = sA + S * kABytes;
  __shared__ __align__(8) uint64_t full[S], empty[S], done;
  __shared__ uint32_t tmem_slot;
  __shared__ int gave_up;
  const Waits& waits = c.guard.waits;
  __shared__ float sbias[BN];
  __shared__ int4 rows[kStep];
  if (GATHER && threadIdx.x < kStep) rows[threadIdx.x] = gather_row(c.g, threadIdx.x);
  // columns beyond the products are zeros, written once: the gather leaves them alone
  // (56 of the first layer's 128)
  if (GATHER && ((int)blockIdx.x + 1) * 128 > (c.g.ntap << c.g.lc)) {
    for (uint32_t i = threadIdx.x; i < S * kABytes / 16; i += kThreads) reinterpret_cast<uint4*>(sA)[i] = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  const int warp = warp_id(), lane = threadIdx.x & 31;
  const int k0 = blockIdx.x * 128, split = blockIdx.y, n0 = blockIdx.z * BN;
  const int s0 = split * c.steps_per_split, steps = max(0, min(c.steps_per_split, c.steps_total - s0));
  const bool bias = blockIdx.x == 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(smem_u32(&full[s]), GATHER ? 2 : 1);
      mbar_init(smem_u32(&empty[s]), 1 + (bias ? 4 : 0));
    }
    mbar_init(smem_u32(&done), 1);
    gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc<kCols>(smem_u32(&tmem_slot));
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  bool ok = true;
  int filled = 0;   // stages whose copies warp 0 has asked for
  if (warp == 0) {
    const bool leader = elect_one();
    Ring r;
    for (int st = 0; st < steps; ++st, r.next<S>()) {
      if (!(ok = mbar_wait(smem_u32(&empty[r.s]), r.phase ^ 1, waits.clocks))) break;
      ++filled;
      const uint32_t fb = smem_u32(&full[r.s]);
      const int row = (s0 + st) * kStep;
      if (!leader) continue;
      if (GATHER && st + kAheadSteps < steps) {
        const int row1 = row + kAheadSteps * kStep;
        prefetch_rows(c.g, row1, kStep);
        if (row1 < c.g.M) prefetch_l2(c.dpre + (size_t)row1 * c.N, (uint32_t)min(kStep, c.g.M - row1) * 2 * c.N);
      }
      mbar_expect_tx(fb, Cfg::kBBytes + (GATHER ? 0 : kABytes));
      for (int h = 0; h < Cfg::kBBlocks; ++h)
        tma_load_2d(smem_u32(sB + r.s * Cfg::kBBytes + h * 8192), &tmB, n0 + 64 * h, row, fb);
      if (!GATHER)
        for (int h = 0; h < 2; ++h) tma_load_2d(smem_u32(sA + r.s * kABytes + h * 8192), &tmA, k0 + 64 * h, row, fb);
    }
  } else if (warp == 1) {
    constexpr uint32_t idesc = mma_idesc(128, BN, true);
    const bool leader = elect_one();
    const uint32_t a0 = desc_mn_lo(smem_u32(sA), 8192), b0 = desc_mn_lo(smem_u32(sB), 8192);
    Ring r;
    for (int st = 0; st < steps; ++st, r.next<S>()) {
      if (!(ok = st != waits.stop && mbar_wait(smem_u32(&full[r.s]), r.phase, waits.clocks))) break;
      tc_fence_after();
      const uint32_t a = a0 + r.s * (kABytes >> 4), b = b0 + r.s * (Cfg::kBBytes >> 4);
      if (leader) {
#pragma unroll
        for (int k = 0; k < kStep / 16; ++k)   // 16 pixels: two groups of 8 rows of 128 bytes
          mma_bf16(tmem, a + k * (2048 >> 4), b + k * (2048 >> 4), idesc, st > 0 || k > 0);
        mma_commit(smem_u32(&empty[r.s]));
      }
    }
    if (!ok) *reinterpret_cast<volatile int*>(&gave_up) = 1;   // before the epilogue is released
    __syncwarp();
    // all products, or those issued before giving up: the epilogue waits for them either way
    if (leader) {
      if (steps > 0) mma_commit(smem_u32(&done));
      else mbar_arrive(smem_u32(&done));
    }
  } else if (warp >= 2 && warp < 6) {
    const int t = threadIdx.x - 64;   // 0 .. 127
    if (bias) {
      // thread: outputs 2 p, 2 p + 1 of the stage's rows h, h + step, ...
      constexpr int kPairs = BN / 2, kRows = 128 / kPairs;
      const int p = t % kPairs, h = t / kPairs;
      float a = 0.0f, b = 0.0f;
      Ring r;
      for (int st = 0; st < steps; ++st, r.next<S>()) {
        if (!(ok = mbar_wait(smem_u32(&full[r.s]), r.phase, waits.clocks))) break;
        const unsigned char* tile = sB + r.s * Cfg::kBBytes + (p >> 5) * 8192;
        const int ch = (p & 31) >> 2, in = (p & 3) * 4;   // 16-byte column and byte within it
#pragma unroll 8
        for (int row = h; row < kStep; row += kRows) {
          const uint32_t w = *reinterpret_cast<const uint32_t*>(tile + row * 128 + ((ch ^ (row & 7)) << 4) + in);
          a += __uint_as_float(w << 16);
          b += __uint_as_float(w & 0xffff0000u);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&empty[r.s]));
      }
      // the row groups' sums in order
      for (int g = 0; g < kRows; ++g) {
        if (h == g) {
          sbias[p * 2] = g ? sbias[p * 2] + a : a;
          sbias[p * 2 + 1] = g ? sbias[p * 2 + 1] + b : b;
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
      }
      if (t < BN && n0 + t < c.N) c.bias_part[(size_t)split * c.N + n0 + t] = sbias[t];
    }
    const bool got = mbar_wait(smem_u32(&done), 0, kWaitClocks);
    tc_fence_after();
    ok = got && ok;
    if (ok && !*reinterpret_cast<volatile int*>(&gave_up)) {
      const int q = warp & 3, row = k0 + q * 32 + lane;
      float* out = c.part + ((size_t)split * c.K + row) * c.N + n0;
      for (int n = 0; n < BN; n += 16) {
        float x[16];
        if (steps > 0) {
          tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + n, x);
        } else {
#pragma unroll
          for (int e = 0; e < 16; ++e) x[e] = 0.0f;
        }
        if (row < c.K && n0 + n < c.N) {
#pragma unroll
          for (int e = 0; e < 16; e += 4) *reinterpret_cast<float4*>(out + n + e) = make_float4(x[e], x[e + 1], x[e + 2], x[e + 3]);
        }
      }
    }
  } else if (GATHER && warp >= kGatherWarp && warp < kGatherWarp + gather_warps<S>()) {
    // 16 lanes per pixel (16 chunks of 8 products), rows rr, rr + 2, ... of the stage;
    // every G-th stage
    constexpr int G = gather_warps<S>();
    const int q = lane & 15, rr = lane >> 4;
    const int Hs = 1 << c.g.ls, C = 1 << c.g.lc;
    const int k = k0 + 8 * q, tap = k >> c.g.lc, ch = k & (C - 1);
    const bool tv = tap < c.g.ntap;   // columns beyond the products are zeros
    const int dy = tv ? c.g.dy[tap] : 0, dx = tv ? c.g.dx[tap] : 0, off = ((dy << c.g.ls) + dx) * C + ch;
    Ring r;
    r.s = warp - kGatherWarp;
    for (int st = warp - kGatherWarp; st < steps; st += G) {
      const int row0 = (s0 + st) * kStep, left = c.g.M - row0;
      int yb;
      const bf16* p = gather_base(c.g, row0, yb) + off;
      const int y0 = yb + dy;
      if (!(ok = mbar_wait(smem_u32(&empty[r.s]), r.phase ^ 1, waits.clocks))) break;
      if (tv) {
        uint32_t dst = smem_u32(sA) + r.s * kABytes + (q >> 3) * 8192 + rr * 128;
#pragma unroll 8
        for (int rw = rr; rw < kStep; rw += 2, dst += 256) {
          const int4 o = rows[rw];
          const bool in = (unsigned)(y0 + o.y) < (unsigned)Hs && (unsigned)(o.z + dx) < (unsigned)Hs && rw < left;
          cp16(dst + (((q & 7) ^ (rw & 7)) << 4), in ? p + o.x : c.g.src, in);
        }
      }
      finish_stage(&full[r.s]);
      if ((r.s += G) >= S) {
        r.s -= S;
        r.phase ^= 1;
      }
    }
  }
  if (!ok && lane == 0) {
    set_status(c.guard.status, kStatusTimeout);
    gave_up = 1;
  }
  tc_fence_before();
  __syncthreads();
  if (gave_up) {   // (otherwise the products have waited for the copies)
    if (warp == 0) drain_fills<S>(full, filled);
    __syncthreads();
  }
  if (warp == 1) {
    mbar_wait(smem_u32(&done), 0, kWaitClocks);   // (an epilogue that gave up has not waited for the products)
    tc_fence_after();
    tmem_free<kCols>(tmem);
  }
}

// dW[n][k] = sum over splits of part[split][k][n], db[n] likewise.  A block takes 8
// products x 32 outputs: warp g adds splits g, g + 16, ... (eight independent loads per
// split), then the 16 warps' sums are added in warp order (a fixed order for every call).
constexpr int kRedK = 8, kRedWarps = 16;
__global__ void __launch_bounds__(32 * kRedWarps) k_wgrad_reduce(const float* __restrict__ part, const float* __restrict__ bias_part,
                                                                int splits, int K, int N, float* __restrict__ dW,
                                                                float* __restrict__ db) {
  __shared__ float red[kRedWarps][kRedK + 1][33];
  const int kb = blockIdx.x * kRedK, nb = blockIdx.y * 32, lane = threadIdx.x & 31, g = threadIdx.x >> 5, n = nb + lane;
  const bool bias = blockIdx.x == 0;
  float acc[kRedK + 1] = {};
  if (n < N)
    for (int z = g; z < splits; z += kRedWarps) {
#pragma unroll
      for (int k = 0; k < kRedK; ++k)
        if (kb + k < K) acc[k] += part[((size_t)z * K + kb + k) * N + n];
      if (bias) acc[kRedK] += bias_part[(size_t)z * N + n];
    }
#pragma unroll
  for (int k = 0; k <= kRedK; ++k) red[g][k][lane] = acc[k];
  __syncthreads();
  const int t = threadIdx.x;
  if (t < 32 * (kRedK + 1)) {
    const int k = t < 32 * kRedK ? t % kRedK : kRedK, i = t < 32 * kRedK ? t / kRedK : t - 32 * kRedK;
    float s = 0.0f;
    for (int w = 0; w < kRedWarps; ++w) s += red[w][k][i];
    if (nb + i < N) {
      if (k < kRedK) {
        if (kb + k < K) dW[(size_t)(nb + i) * K + kb + k] = s;
      } else if (bias) {
        db[nb + i] = s;
      }
    }
  }
}

int ilog2(int x) {
  int l = 0;
  while ((1 << l) < x) ++l;
  return l;
}

Gather conv_gather(const bf16* src, int NV, int C, int Hin) {
  Gather g;
  g.src = src;
  g.lc = ilog2(C);
  g.ls = ilog2(Hin);
  g.lo = g.ls - 1;
  g.stride = 2;
  g.ntap = 9;
  g.M = NV << (2 * g.lo);
  for (int t = 0; t < 9; ++t) {
    g.dy[t] = (signed char)(t / 3 - 1);
    g.dx[t] = (signed char)(t % 3 - 1);
  }
  return g;
}

template <int BN, bool DGRAD>
int launch_conv(const CUtensorMap& tb, const ConvArgs& c, cudaStream_t s) {
  k_conv<BN, DGRAD><<<std::min(c.tiles, sm_count()), kThreads, ConvCfg<BN, DGRAD>::kSmem, s>>>(tb, c);
  HR_CHECK_LAUNCH();
  return HR_OK;
}

template <int BN>
int launch_wgrad_bn(const CUtensorMap& ta, const CUtensorMap& tb, const WgradArgs& c, bool gather, cudaStream_t s) {
  const dim3 grid((unsigned)((c.K + 127) / 128), (unsigned)c.splits, (unsigned)((c.N + BN - 1) / BN));
  if (gather)
    k_wgrad<BN, true><<<grid, kThreads, WgradCfg<BN>::kSmem, s>>>(ta, tb, c);
  else
    k_wgrad<BN, false><<<grid, kThreads, WgradCfg<BN>::kSmem, s>>>(ta, tb, c);
  HR_CHECK_LAUNCH();
  return HR_OK;
}

// dW [N][K] and db [N] of a layer from dPre [rows][N]; the columns gathered (ta unused)
// or a plain [rows][K] matrix
int launch_wgrad(const CUtensorMap& ta, WgradArgs c, const bf16* dPre, long long rows, bool gather, float* dW, float* db,
                 float* part, size_t part_floats, cudaStream_t s) {
  CUtensorMap tb;
  if (!tma_map(&tb, dPre, rows, c.N, c.N, 64)) return HR_ERR_CUDA;
  c.dpre = dPre;
  const int BN = c.N <= 32 ? 32 : (c.N <= 64 ? 64 : 128);
  const int tiles = ((c.K + 127) / 128) * ((c.N + BN - 1) / BN);
  c.steps_total = (int)((rows + kStep - 1) / kStep);
  // Two rounds of one block per SM (their stages fill its shared memory), each with at
  // least eight steps.  The tensor core's running sums are truncated, so a split's length
  // is also the result's error: one round of blocks with chains twice as long measured 2 % less
  // time and up to 2.6 times the error (second layer, 4096 images: 6e-6 of the
  // gradient's norm instead of 2e-6).
  int splits = std::min(std::min((2 * sm_count() + tiles - 1) / tiles, kMaxSplits), std::max(1, c.steps_total / 8));
  c.steps_per_split = (c.steps_total + splits - 1) / splits;
  c.splits = (c.steps_total + c.steps_per_split - 1) / c.steps_per_split;
  while (c.splits > 1 && (size_t)c.splits * ((size_t)c.K + 1) * c.N > part_floats) {   // (never, at the network's sizes)
    c.steps_per_split *= 2;
    c.splits = (c.steps_total + c.steps_per_split - 1) / c.steps_per_split;
  }
  c.part = part;
  c.bias_part = part + (size_t)c.splits * c.K * c.N;
  const int rc = BN == 32 ? launch_wgrad_bn<32>(ta, tb, c, gather, s)
                          : (BN == 64 ? launch_wgrad_bn<64>(ta, tb, c, gather, s) : launch_wgrad_bn<128>(ta, tb, c, gather, s));
  if (rc != HR_OK) return rc;
  k_wgrad_reduce<<<dim3((unsigned)((c.K + kRedK - 1) / kRedK), (unsigned)((c.N + 31) / 32)), 32 * kRedWarps, 0, s>>>(
      c.part, c.bias_part, c.splits, c.K, c.N, dW, db);
  HR_CHECK_LAUNCH();
  return HR_OK;
}

template <class F>
bool smem_ok(F* kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}
template <int BN>
bool configure_bn() {
  return smem_ok(k_conv<BN, false>, ConvCfg<BN, false>::kSmem) && smem_ok(k_wgrad<BN, true>, WgradCfg<BN>::kSmem) && smem_ok(k_wgrad<BN, false>, WgradCfg<BN>::kSmem);
}

}  // namespace

int configure_conv_kernels() {
  if (!configure_bn<32>() || !configure_bn<64>() || !configure_bn<128>() ||
      !smem_ok(k_conv<32, true>, ConvCfg<32, true>::kSmem) || !smem_ok(k_conv<64, true>, ConvCfg<64, true>::kSmem)) {
    cudaGetLastError();
    return HR_ERR_CUDA;
  }
  return HR_OK;
}

int launch_conv_fwd(const void* X, int NV, int Hin, int Cin, const void* W, int Kp, const float* bias, int Cout, void* Y,
                    Guard guard, cudaStream_t s) {
  CUtensorMap tb;
  if (!tma_map(&tb, W, Cout, Kp, Kp, Cout)) return HR_ERR_CUDA;
  ConvArgs c = {};
  c.g = conv_gather(static_cast<const bf16*>(X), NV, Cin, Hin);
  c.tiles = (c.g.M + kTileM - 1) / kTileM;
  const int K = 9 * Cin;
  c.nkt = (K + kStep - 1) / kStep;
  c.last16 = (K - (c.nkt - 1) * kStep + 15) / 16;
  c.nblocks = c.nclass = 1;
  c.C = Cout;
  c.bias = bias;
  c.out = static_cast<bf16*>(Y);
  c.guard = guard;
  return Cout == 32 ? launch_conv<32, false>(tb, c, s)
                    : (Cout == 64 ? launch_conv<64, false>(tb, c, s) : launch_conv<128, false>(tb, c, s));
}

int launch_conv_dgrad(const void* dPre, int NV, int Hin, int Cin, const void* wT, int Cout, const void* X, void* dX, Guard guard,
                      cudaStream_t s) {
  CUtensorMap tb;
  const int BN = Cin == 32 ? 32 : 64;   // four taps' accumulators, twice: 8 BN columns
  if (!tma_map(&tb, wT, 9 * Cin, Cout, Cout, BN)) return HR_ERR_CUDA;
  ConvArgs c = {};
  c.g.src = static_cast<const bf16*>(dPre);
  c.g.lc = ilog2(Cout);
  c.g.lo = c.g.ls = ilog2(Hin) - 1;
  c.g.stride = 1;
  c.g.M = NV << (2 * c.g.lo);
  c.tiles = (c.g.M + kTileM - 1) / kTileM;
  c.nkt = Cout / kStep;
  c.out = static_cast<bf16*>(dX);
  c.mask = static_cast<const bf16*>(X);
  c.guard = guard;
  c.C = Cin;
  c.nblocks = Cin / BN;
  c.nclass = 4;
  for (int q = 0; q < 4; ++q) {
    // pixel y = 2 i + py is read by tap ky from output row (y + 1 - ky) / 2: ky = 1 (row i)
    // when even, ky = 0 (row i + 1) and ky = 2 (row i) when odd; columns likewise
    ConvClass& k = c.cls[q];
    k.py = q >> 1;
    k.px = q & 1;
    for (int ky = 0; ky < 3; ++ky)
      for (int kx = 0; kx < 3; ++kx) {
        if (((k.py + 1 - ky) & 1) || ((k.px + 1 - kx) & 1)) continue;
        const int t = k.ntap++;
        k.dy[t] = (signed char)((k.py + 1 - ky) / 2);
        k.dx[t] = (signed char)((k.px + 1 - kx) / 2);
        k.btap[t] = (ky * 3 + kx) * Cin;
      }
  }
  return BN == 32 ? launch_conv<32, true>(tb, c, s) : launch_conv<64, true>(tb, c, s);
}

int launch_conv_wgrad(const void* X, int NV, int Hin, int Cin, int Kp, const void* dPre, int Cout, float* dW, float* db,
                      float* part, size_t part_floats, Guard guard, cudaStream_t s) {
  WgradArgs c = {};
  c.g = conv_gather(static_cast<const bf16*>(X), NV, Cin, Hin);
  c.K = Kp;
  c.N = Cout;
  c.guard = guard;
  const CUtensorMap none = {};
  return launch_wgrad(none, c, static_cast<const bf16*>(dPre), c.g.M, true, dW, db, part, part_floats, s);
}

int launch_dense_wgrad(const void* x, long long rows, int K, const void* dPre, int N, float* dW, float* db, float* part,
                       size_t part_floats, Guard guard, cudaStream_t s) {
  CUtensorMap ta;
  if (!tma_map(&ta, x, rows, K, K, 64)) return HR_ERR_CUDA;
  WgradArgs c = {};
  c.K = K;
  c.N = N;
  c.guard = guard;
  return launch_wgrad(ta, c, static_cast<const bf16*>(dPre), rows, false, dW, db, part, part_floats, s);
}

}  // namespace hr
