// The two dense products of an attention layer's reverse pass (paper Section 3.3.4's gradient through Eq. 7) on the
// 5th-generation tensor cores, for bf16 models: with dz the gradient of Z = h W in bf16 (hidden 128 and 256: both in one
// kernel, k_dhw_umma; hidden 512, whose dW takes the tensor memory of four SMs, one after the other),
//   dh = dz W^T   the transform kernel's roles and tiles (xrl_xform_umma.cuh) with W itself as the K-major operand
//                 and an fp32 result, which leaves masked by the ReLU of h (what the next layer down needs);
//   dW += h^T dz  reduces over the rows, so both operands are used as they lie in memory, which tcgen05.mma reads as
//                 MN-major operands, and the result stays in tensor memory while the CTA walks its range of rows
//                 (hidden 512: a 256 x 256 quarter per CTA, all 512 columns).  The CTAs' results meet in the gradient by
//                 TMA reductions (fp32 add in L2).
// Both are bound by HBM: 8 H bytes per row (dh: 4 H in, 4 H out) and 4 H bytes per row (dW); together, with dz and h read
// once, 8 H.
//
// Every wait on an mbarrier is bounded; on expiry the kernel records XRL_ERR_TIMEOUT, drains its own copies in
// flight, frees its tensor memory and returns.
#include "xrl_xform_umma.cuh"

namespace xrl {

using namespace umma;
using namespace xform;

namespace {

constexpr int kThreads = 192;            // warp 0 TMA, warp 1 MMA, warps 2..5 epilogue

__device__ __forceinline__ void tma_reduce_add_2d(const CUtensorMap* map, uint32_t src, int x, int y) {
  asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%2, %3}], [%1];"
               ::"l"(map), "r"(src), "r"(x), "r"(y) : "memory");
}

// 32 fp32 columns of a thread's row into a staging tile of 128 rows x 128 bytes, 128-byte swizzle
__device__ __forceinline__ void stage_row(uint8_t* tile, int row, const uint32_t (&v)[32]) {
  uint8_t* p = tile + row * 128;
#pragma unroll
  for (int j = 0; j < 8; ++j)
    *reinterpret_cast<uint4*>(p + ((j ^ (row & 7)) << 4)) = make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
}

// ---- dh = dz W^T at hidden 512 ----------------------------------------------------------------------------------
// (a CTA: 128 columns of dh for every 128-row tile of its share, four CTAs side by side)
constexpr int WIDE = 512, NS = 128, SLICES = WIDE / NS;
using DhCfg = Cfg<NS, WIDE, true>;
__global__ void __launch_bounds__(kThreads, 1)
k_dh_umma(const __grid_constant__ CUtensorMap map_g, const __grid_constant__ CUtensorMap map_w,
          const __grid_constant__ CUtensorMap map_o, const bf16* __restrict__ h, int rows, int32_t* status) {
  using C = DhCfg;
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t base = smem_u32(smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int num_tiles = (rows + BM - 1) / BM;
  const int col0 = int(blockIdx.x) % SLICES * NS, first = int(blockIdx.x) / SLICES, step = int(gridDim.x) / SLICES;
  if ((base & 1023u) != 0) {
    if (threadIdx.x == 0) raise(status, XRL_ERR_UNSUPPORTED);
    return;
  }
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_TMEM);
  if (threadIdx.x == 0) {
    tmem_slot[1] = 0;
    init_barriers<C>(base, 128);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(uint32_t(C::TMEM_COLS)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if (warp == 0) {
    if (lane == 0) {
      load_w<C>(base, &map_w, col0);
      enter();
      uint32_t it = 0;
      if (!produce_tiles<C>(base, &map_g, first, step, num_tiles, it)) {
        raise(status, XRL_ERR_TIMEOUT);
        drain_producer<C>(base, it, 0);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      uint32_t it = 0, lt = 0;
      if (!mma_tiles<C, NS>(base, tmem_base, first, step, num_tiles, it, lt, 0)) raise(status, XRL_ERR_TIMEOUT);
    }
  } else {
    const int q = warp & 3, row_in_tile = q * 32 + lane;
    const bool leader = threadIdx.x == 64;
    volatile uint32_t* abort_flag = tmem_slot + 1;
    uint32_t lt = 0;
    enter();
    // The features whose ReLU masks the result: this thread's row of a tile, 32 columns (64 bytes) per chunk, asked for a
    // whole tile ahead (2 NS bytes of them in registers: asked for one chunk ahead the four warps wait for them; 256
    // columns per CTA, 990 k rows: 0.448 instead of 0.351 ms).
    uint4 hn[NS / 32][4];
    auto features = [&](int tile, int c, uint4 (&f)[4]) {
      const int64_t r = int64_t(tile) * BM + row_in_tile;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        f[j] = make_uint4(0u, 0u, 0u, 0u);
        if (tile < num_tiles && r < rows)
          f[j] = __ldg(reinterpret_cast<const uint4*>(h + size_t(r) * WIDE + col0 + c * 32) + j);
      }
    };
#pragma unroll
    for (int c = 0; c < NS / 32; ++c) features(first, c, hn[c]);
    for (int tile = first; tile < num_tiles; tile += step, ++lt) {
      const int buf = lt & 1;
      uint32_t okw = 1;
      if (lane == 0) okw = mbar_wait(C::bar_acc_full(base, buf), (lt >> 1) & 1) ? 1u : 0u;
      okw = __shfl_sync(0xFFFFFFFFu, okw, 0);
      if (!okw && lane == 0) { *abort_flag = 1; raise(status, XRL_ERR_TIMEOUT); }
      epi_barrier();
      if (*abort_flag) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + (uint32_t(q * 32) << 16) + uint32_t(buf * C::ACC_COLS);
#pragma unroll
      for (int c = 0; c < NS / 32; ++c) {
        uint32_t v[32];
        tc_ld32(taddr + c * 32, v);
        tc_wait_ld();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float f[8];
          unpack(hn[c][j], f);
#pragma unroll
          for (int t = 0; t < 8; ++t) v[8 * j + t] = f[t] > 0.f ? v[8 * j + t] : 0u;
        }
        features(tile + step, c, hn[c]);
        if (leader) tma_wait_read<1>();          // the store issued two chunks ago has read this staging tile
        epi_barrier();
        stage_row(smem + C::OFF_OUT + (c & 1) * STAGE_BYTES, row_in_tile, v);
        fence_async_smem();
        epi_barrier();
        if (leader) {
          tma_store_2d(&map_o, base + C::OFF_OUT + (c & 1) * STAGE_BYTES, col0 + c * 32, tile * BM);
          tma_commit();
        }
      }
      tc_fence_before();
      mbar_arrive(C::bar_acc_empty(base, buf));
    }
    if (leader) tma_wait_all();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                 ::"r"(tmem_base), "r"(uint32_t(C::TMEM_COLS)) : "memory");
  }
}

// ---- dW += h^T dz at hidden 512 ---------------------------------------------------------------------------------
constexpr int RB = 64;                   // rows per stage: 64-row blocks of h and of dz, in boxes of 64 columns
constexpr int S = 256, SIDE = WIDE / S;  // side of the square of dW a CTA accumulates
struct DwCfg {
  static constexpr int CHUNK = RB * 128;                 // 64 rows x 64 columns
  static constexpr int OPERAND = (S / 64) * CHUNK;       // one operand of a stage
  static constexpr int STAGES = 3;
  static constexpr int OFF_OUT = STAGES * 2 * OPERAND;
  static constexpr int OFF_BAR = OFF_OUT + 2 * STAGE_BYTES;
  static constexpr int OFF_TMEM = OFF_BAR + 8 * (2 * STAGES + 1);
  static constexpr int SMEM_BYTES = OFF_TMEM + 16;
  static constexpr int HALVES = S / 128;                 // M = 128 rows of dW per instruction
  static constexpr int TMEM_COLS = HALVES * S;
  static_assert(SMEM_BYTES <= 227 * 1024, "shared memory of one SM");
};

// Shared-memory matrix descriptor of an MN-major, 128-byte-swizzled operand: rows (the reduction index) of 128 bytes,
// 8-row groups 1,024 bytes apart, 64-column chunks `chunk` bytes apart.
__device__ __forceinline__ uint64_t smem_desc_mn(uint32_t addr, uint32_t chunk) {
  return uint64_t((addr & 0x3FFFFu) >> 4) | (uint64_t(chunk >> 4) << 16) | (uint64_t(1024 >> 4) << 32) |
         (uint64_t(1) << 46) | (uint64_t(2) << 61);
}

__global__ void __launch_bounds__(kThreads, 1)
k_dw_umma(const __grid_constant__ CUtensorMap map_h, const __grid_constant__ CUtensorMap map_g,
          const __grid_constant__ CUtensorMap map_o, float* __restrict__ dW, int rows, bool use_tma, int32_t* status) {
  using C = DwCfg;
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t base = smem_u32(smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if ((base & 1023u) != 0) {
    if (threadIdx.x == 0) raise(status, XRL_ERR_UNSUPPORTED);
    return;
  }
  // CTA = (range of 64-row blocks, square of dW); the squares of a range side by side
  constexpr int squares = SIDE * SIDE;
  const int part = int(blockIdx.x) / squares, parts = int(gridDim.x) / squares;
  const int a0 = (int(blockIdx.x) % squares) / SIDE * S, b0 = int(blockIdx.x) % SIDE * S;
  const int blocks = (rows + RB - 1) / RB;
  const int blk0 = int(int64_t(blocks) * part / parts), blk1 = int(int64_t(blocks) * (part + 1) / parts);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_TMEM);
  auto bar_full = [&](int s) { return base + C::OFF_BAR + 8u * s; };
  auto bar_empty = [&](int s) { return base + C::OFF_BAR + 8u * (C::STAGES + s); };
  const uint32_t bar_done = base + C::OFF_BAR + 8u * (2 * C::STAGES);
  if (threadIdx.x == 0) {
    tmem_slot[1] = 0;
    for (int s = 0; s < C::STAGES; ++s) { mbar_init(bar_full(s), 1); mbar_init(bar_empty(s), 1); }
    mbar_init(bar_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(uint32_t(C::TMEM_COLS)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  enter();
  const int nblk = blk1 - blk0;            // >= 1: the launch has at most one part per block

  if (warp == 0) {
    if (lane == 0) {
      bool ok = true;
      int i = 0;
      for (; i < nblk; ++i) {
        const int s = i % C::STAGES, round = i / C::STAGES;
        if (round > 0 && !mbar_wait(bar_empty(s), (round - 1) & 1)) { ok = false; break; }
        mbar_expect_tx(bar_full(s), 2 * C::OPERAND);
        const uint32_t at = base + s * 2 * C::OPERAND;
        for (int c = 0; c < S / 64; ++c) {
          tma_load_2d(at + c * C::CHUNK, &map_h, a0 + c * 64, (blk0 + i) * RB, bar_full(s));
          tma_load_2d(at + C::OPERAND + c * C::CHUNK, &map_g, b0 + c * 64, (blk0 + i) * RB, bar_full(s));
        }
      }
      if (!ok) {                           // let the loads already issued land before the shared memory goes away
        raise(status, XRL_ERR_TIMEOUT);
        for (int j = i > C::STAGES ? i - C::STAGES : 0; j < i; ++j) mbar_wait(bar_full(j % C::STAGES), (j / C::STAGES) & 1);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // fp32 accumulators, bf16 x bf16, both operands MN-major (bits 15, 16), M = 128, N = S
      constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | (uint32_t(S >> 3) << 17) |
                                 (uint32_t(128 >> 4) << 24);
      bool ok = true;
      for (int i = 0; i < nblk; ++i) {
        const int s = i % C::STAGES;
        if (!mbar_wait(bar_full(s), (i / C::STAGES) & 1)) { ok = false; break; }
        tc_fence_after();
        const uint32_t at = base + s * 2 * C::OPERAND;
#pragma unroll
        for (int ks = 0; ks < RB / 16; ++ks)             // 16 rows = two 8-row groups per instruction
#pragma unroll
          for (int m = 0; m < C::HALVES; ++m)
            tc_mma(tmem_base + uint32_t(m * S), smem_desc_mn(at + m * 2 * C::CHUNK + ks * 2048, C::CHUNK),
                   smem_desc_mn(at + C::OPERAND + ks * 2048, C::CHUNK), idesc, (i | ks) != 0 ? 1u : 0u);
        tc_commit(bar_empty(s));
      }
      if (ok) tc_commit(bar_done);
      else raise(status, XRL_ERR_TIMEOUT);
    }
  } else {
    const int q = warp & 3, row = q * 32 + lane;
    const bool leader = threadIdx.x == 64;
    volatile uint32_t* abort_flag = tmem_slot + 1;
    // the whole range is multiplied first: the limit of one wait, several times over
    uint32_t okw = 1;
    if (lane == 0) {
      okw = 0;
      for (int t = 0; t < 4 && !okw; ++t) okw = mbar_wait(bar_done, 0) ? 1u : 0u;
    }
    okw = __shfl_sync(0xFFFFFFFFu, okw, 0);
    if (!okw && lane == 0) { *abort_flag = 1; raise(status, XRL_ERR_TIMEOUT); }
    epi_barrier();
    if (!*abort_flag) {
      tc_fence_after();
      const uint32_t taddr = tmem_base + (uint32_t(q * 32) << 16);
      for (int c = 0; c < C::HALVES * (S / 32); ++c) {
        const int m = c / (S / 32), cc = c % (S / 32);
        uint32_t v[32];
        tc_ld32(taddr + m * S + cc * 32, v);
        tc_wait_ld();
        if (use_tma) {
          if (leader) tma_wait_read<1>();
          epi_barrier();
          stage_row(smem + C::OFF_OUT + (c & 1) * STAGE_BYTES, row, v);
          fence_async_smem();
          epi_barrier();
          if (leader) {
            tma_reduce_add_2d(&map_o, base + C::OFF_OUT + (c & 1) * STAGE_BYTES, b0 + cc * 32, a0 + m * 128);
            tma_commit();
          }
        } else {
          float* o = dW + size_t(a0 + m * 128 + row) * WIDE + b0 + cc * 32;
#pragma unroll
          for (int t = 0; t < 32; ++t) atomicAdd(o + t, __uint_as_float(v[t]));
        }
      }
      if (leader) tma_wait_all();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                 ::"r"(tmem_base), "r"(uint32_t(C::TMEM_COLS)) : "memory");
  }
}

// ---- both products in one pass: dh = dz W^T and dW += h^T dz for H = 128 and 256 -----------------------------------
// A CTA takes 128 columns of h (H / 128 CTAs side by side per tile of rows): their 128 x H part of dW stays in tensor memory
// for the whole range of tiles, and the same 128 columns of dh are computed tile by tile into two more accumulators.  A
// 128-row tile of dz (64-column chunks through a ring) is then read once from memory for both products - as the K-major
// operand of dh and, the same bytes, as the MN-major operand of dW - and so is the tile of h, which is dW's other operand
// and the ReLU mask of dh.  W's 128 rows are resident.  One kernel per product read both twice: 990 k rows of 256,
// 0.163 + 0.365 -> 0.341 ms per layer; 183 k rows 41 + 65 -> 66 us.
template <int H> struct PCfg {
  static constexpr int KC = H / KCH, HALVES = H / 128;
  static constexpr int W_CHUNK = 128 * 128, W_BYTES = KC * W_CHUNK;
  static constexpr int RING = 4, H_STAGES = 2, H_STAGE = 2 * STAGE_BYTES;
  static constexpr int OFF_DZ = W_BYTES;
  static constexpr int OFF_H = OFF_DZ + RING * STAGE_BYTES;
  static constexpr int OFF_OUT = OFF_H + H_STAGES * H_STAGE;
  static constexpr int OFF_BAR = OFF_OUT + 2 * STAGE_BYTES;
  static constexpr int NUM_BARS = 2 + 2 * RING + 2 * H_STAGES + 4;
  static constexpr int OFF_TMEM = OFF_BAR + 8 * NUM_BARS;
  static constexpr int SMEM_BYTES = OFF_TMEM + 16;
  static constexpr int TMEM_COLS = 512;                  // dW: H columns, then two accumulators of 128
  static_assert(SMEM_BYTES <= 227 * 1024 && H + 256 <= 512, "shared and tensor memory of one SM");
};

template <int H>
__global__ void __launch_bounds__(kThreads, 1)
k_dhw_umma(const __grid_constant__ CUtensorMap map_g, const __grid_constant__ CUtensorMap map_h,
           const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_dh,
           const __grid_constant__ CUtensorMap map_dw, float* __restrict__ dW, int rows, bool use_tma, int32_t* status) {
  using C = PCfg<H>;
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t base = smem_u32(smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if ((base & 1023u) != 0) {
    if (threadIdx.x == 0) raise(status, XRL_ERR_UNSUPPORTED);
    return;
  }
  const int num_tiles = (rows + BM - 1) / BM;
  const int a0 = int(blockIdx.x) % C::HALVES * 128, first = int(blockIdx.x) / C::HALVES, step = int(gridDim.x) / C::HALVES;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_TMEM);
  const uint32_t bars = base + C::OFF_BAR, bar_w = bars, bar_done = bars + 8;
  auto dz_full = [&](uint32_t s) { return bars + 8u * (2 + s); };
  auto dz_empty = [&](uint32_t s) { return bars + 8u * (2 + C::RING + s); };
  auto h_full = [&](uint32_t s) { return bars + 8u * (2 + 2 * C::RING + s); };
  auto h_empty = [&](uint32_t s) { return bars + 8u * (2 + 2 * C::RING + C::H_STAGES + s); };
  auto acc_full = [&](uint32_t b) { return bars + 8u * (2 + 2 * C::RING + 2 * C::H_STAGES + b); };
  auto acc_empty = [&](uint32_t b) { return bars + 8u * (2 + 2 * C::RING + 2 * C::H_STAGES + 2 + b); };
  if (threadIdx.x == 0) {
    tmem_slot[1] = 0;
    mbar_init(bar_w, 1);
    mbar_init(bar_done, 1);
    for (uint32_t s = 0; s < C::RING; ++s) { mbar_init(dz_full(s), 1); mbar_init(dz_empty(s), 1); }
    // a tile of h is free once the products have read it and each epilogue warp has taken its mask
    for (uint32_t s = 0; s < C::H_STAGES; ++s) { mbar_init(h_full(s), 1); mbar_init(h_empty(s), 5); }
    for (uint32_t b = 0; b < 2; ++b) { mbar_init(acc_full(b), 1); mbar_init(acc_empty(b), 128); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(uint32_t(C::TMEM_COLS)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      mbar_expect_tx(bar_w, C::W_BYTES);
      for (int kc = 0; kc < C::KC; ++kc) tma_load_2d(base + kc * C::W_CHUNK, &map_w, kc * KCH, a0, bar_w);
      enter();
      bool ok = true;
      uint32_t it = 0, lt = 0;
      for (int tile = first; tile < num_tiles && ok; tile += step, ++lt) {
        const uint32_t hs = lt % C::H_STAGES, hr = lt / C::H_STAGES;
        if (hr > 0 && !mbar_wait(h_empty(hs), (hr - 1) & 1)) { ok = false; break; }
        mbar_expect_tx(h_full(hs), C::H_STAGE);
        for (int c = 0; c < 2; ++c)
          tma_load_2d(base + C::OFF_H + hs * C::H_STAGE + c * STAGE_BYTES, &map_h, a0 + c * KCH, tile * BM, h_full(hs));
        for (int kc = 0; kc < C::KC; ++kc, ++it) {
          const uint32_t s = it % C::RING, round = it / C::RING;
          if (round > 0 && !mbar_wait(dz_empty(s), (round - 1) & 1)) { ok = false; break; }
          mbar_expect_tx(dz_full(s), STAGE_BYTES);
          tma_load_2d(base + C::OFF_DZ + s * STAGE_BYTES, &map_g, kc * KCH, tile * BM, dz_full(s));
        }
      }
      if (!ok) {                             // let the loads already issued land before the shared memory goes away
        raise(status, XRL_ERR_TIMEOUT);
        for (uint32_t j = it > C::RING ? it - C::RING : 0; j < it; ++j) mbar_wait(dz_full(j % C::RING), (j / C::RING) & 1);
        for (uint32_t j = lt > C::H_STAGES ? lt - C::H_STAGES : 0; j < lt; ++j)
          mbar_wait(h_full(j % C::H_STAGES), (j / C::H_STAGES) & 1);
        mbar_wait(bar_w, 0);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // fp32 accumulators, bf16 x bf16: dh K-major both, M = N = 128; dW MN-major both (bits 15, 16), M = 128, N = 64
      constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(128 >> 4) << 24);
      constexpr uint32_t idesc_dh = idesc | (uint32_t(128 >> 3) << 17);
      constexpr uint32_t idesc_dw = idesc | (1u << 15) | (1u << 16) | (uint32_t(64 >> 3) << 17);
      bool ok = mbar_wait(bar_w, 0);
      uint32_t it = 0, lt = 0;
      for (int tile = first; tile < num_tiles && ok; tile += step, ++lt) {
        const uint32_t hs = lt % C::H_STAGES, buf = lt & 1, use = lt >> 1;
        if (use > 0 && !mbar_wait(acc_empty(buf), (use - 1) & 1)) { ok = false; break; }
        if (!mbar_wait(h_full(hs), (lt / C::H_STAGES) & 1)) { ok = false; break; }
        const uint32_t acc = tmem_base + uint32_t(H) + buf * 128u, h_at = base + C::OFF_H + hs * C::H_STAGE;
        for (int kc = 0; kc < C::KC; ++kc, ++it) {
          const uint32_t s = it % C::RING, at = base + C::OFF_DZ + s * STAGE_BYTES;
          if (!mbar_wait(dz_full(s), (it / C::RING) & 1)) { ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int k = 0; k < KCH / 16; ++k)
            tc_mma(acc, smem_desc(at + k * 32), smem_desc(base + kc * C::W_CHUNK + k * 32), idesc_dh, (kc | k) != 0 ? 1u : 0u);
#pragma unroll
          for (int ks = 0; ks < BM / 16; ++ks)         // 16 rows = two 8-row groups per instruction
            tc_mma(tmem_base + uint32_t(kc * KCH), smem_desc_mn(h_at + ks * 2048, STAGE_BYTES),
                   smem_desc_mn(at + ks * 2048, STAGE_BYTES), idesc_dw, (lt | uint32_t(ks)) != 0 ? 1u : 0u);
          tc_commit(dz_empty(s));
        }
        if (!ok) break;
        tc_commit(h_empty(hs));
        tc_commit(acc_full(buf));
      }
      if (ok) tc_commit(bar_done);
      else raise(status, XRL_ERR_TIMEOUT);
    }
  } else {
    const int q = warp & 3, row = q * 32 + lane;
    const bool leader = threadIdx.x == 64;
    volatile uint32_t* abort_flag = tmem_slot + 1;
    uint32_t lt = 0, stores = 0;
    enter();
    // a 32-column piece of a thread's row, out through the staging tile whose store of two pieces ago has read it
    auto stage_out = [&](const uint32_t (&v)[32], auto store) {
      if (leader) tma_wait_read<1>();
      epi_barrier();
      stage_row(smem + C::OFF_OUT + (stores & 1) * STAGE_BYTES, row, v);
      fence_async_smem();
      epi_barrier();
      if (leader) {
        store(base + C::OFF_OUT + (stores & 1) * STAGE_BYTES);
        tma_commit();
      }
      ++stores;
    };
    // the outcome of a wait, agreed on by the four warps
    auto agreed = [&](bool ok) {
      if (!ok && lane == 0) { *abort_flag = 1; raise(status, XRL_ERR_TIMEOUT); }
      epi_barrier();
      return *abort_flag == 0;
    };
    bool run = true;
    for (int tile = first; tile < num_tiles; tile += step, ++lt) {
      const uint32_t hs = lt % C::H_STAGES, buf = lt & 1;
      // this thread's 128 features of h (every lane waits: each has to see the copy's bytes itself)
      run = agreed(mbar_wait(h_full(hs), (lt / C::H_STAGES) & 1));
      if (!run) break;
      uint4 f[2][8];
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int j = 0; j < 8; ++j)
          f[c][j] = *reinterpret_cast<const uint4*>(smem + C::OFF_H + hs * C::H_STAGE + c * STAGE_BYTES + row * 128 + ((j ^ (row & 7)) << 4));
      __syncwarp();
      if (lane == 0) mbar_arrive(h_empty(hs));
      bool ok = true;
      if (lane == 0) ok = mbar_wait(acc_full(buf), (lt >> 1) & 1);
      run = agreed(__shfl_sync(0xFFFFFFFFu, int(ok), 0) != 0);
      if (!run) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + (uint32_t(q * 32) << 16) + uint32_t(H) + buf * 128u;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t v[32];
        tc_ld32(taddr + c * 32, v);
        tc_wait_ld();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float x[8];
          unpack(f[c >> 1][(c & 1) * 4 + j], x);
#pragma unroll
          for (int t = 0; t < 8; ++t) v[8 * j + t] = x[t] > 0.f ? v[8 * j + t] : 0u;
        }
        if (c == 3) {
          tc_fence_before();
          mbar_arrive(acc_empty(buf));
        }
        stage_out(v, [&](uint32_t src) { tma_store_2d(&map_dh, src, a0 + c * 32, tile * BM); });
      }
    }
    if (run) {
      bool ok = true;
      if (lane == 0) ok = mbar_wait(bar_done, 0);
      run = agreed(__shfl_sync(0xFFFFFFFFu, int(ok), 0) != 0);
    }
    if (run) {
      tc_fence_after();
      const uint32_t taddr = tmem_base + (uint32_t(q * 32) << 16);
      for (int c = 0; c < H / 32; ++c) {
        uint32_t v[32];
        tc_ld32(taddr + c * 32, v);
        tc_wait_ld();
        if (use_tma) {
          stage_out(v, [&](uint32_t src) { tma_reduce_add_2d(&map_dw, src, c * 32, a0); });
        } else {
          float* o = dW + size_t(a0 + row) * H + c * 32;
#pragma unroll
          for (int t = 0; t < 32; ++t) atomicAdd(o + t, __uint_as_float(v[t]));
        }
      }
    }
    if (leader) tma_wait_all();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                 ::"r"(tmem_base), "r"(uint32_t(C::TMEM_COLS)) : "memory");
  }
}

// 2-D fp32 tensor [rows x cols] row-major, box [128 rows x 32 columns], 128-byte swizzle
bool make_map_f32(CUtensorMap* m, void* ptr, uint64_t rows, uint64_t cols) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 4};
  cuuint32_t box[2] = {32, 128};
  cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, ptr, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

int launch_dh(const void* h, const void* dzb, const void* W, float* dh, int32_t rows, int32_t* status, cudaStream_t st) {
  static bool attr_set[64] = {};
  if (!ensure_dynamic_smem(k_dh_umma, DhCfg::SMEM_BYTES, attr_set)) return -1;
  CUtensorMap mg, mw, mo;
  if (!make_map(&mg, dzb, uint64_t(rows), WIDE, BM) || !make_map(&mw, W, WIDE, WIDE, NS) ||
      !make_map_f32(&mo, dh, uint64_t(rows), WIDE))
    return -1;
  const int tiles = (rows + BM - 1) / BM, groups = kNumSMs / SLICES;
  launch(k_dh_umma, (tiles < groups ? tiles : groups) * SLICES, kThreads, DhCfg::SMEM_BYTES, st,
         mg, mw, mo, static_cast<const bf16*>(h), rows, status);
  return 1;
}

int launch_dw(const void* h, const void* dzb, float* dW, int32_t rows, int32_t* status, cudaStream_t st) {
  static bool attr_set[64] = {};
  if (!ensure_dynamic_smem(k_dw_umma, DwCfg::SMEM_BYTES, attr_set)) return -1;
  const bool aligned = (reinterpret_cast<uintptr_t>(dW) & 15) == 0;    // the caller's buffer may sit on any 4-byte boundary
  CUtensorMap mh, mg, mo;
  if (!make_map(&mh, h, uint64_t(rows), WIDE, RB) || !make_map(&mg, dzb, uint64_t(rows), WIDE, RB)) return -1;
  if (aligned) { if (!make_map_f32(&mo, dW, WIDE, WIDE)) return -1; }
  else mo = mh;
  constexpr int squares = SIDE * SIDE;
  // at least eight blocks per CTA: every CTA ends with a reduction of its whole square of dW into the gradient
  const int blocks = (rows + RB - 1) / RB, want = (blocks + 7) / 8, most = kNumSMs / squares;
  launch(k_dw_umma, (want < most ? want : most) * squares, kThreads, DwCfg::SMEM_BYTES, st,
         mh, mg, mo, dW, rows, aligned, status);
  return 1;
}

template <int H>
int launch_dhw(const void* h, const void* dzb, const void* W, float* dh, float* dW, int32_t rows, int32_t* status, cudaStream_t st) {
  using C = PCfg<H>;
  static bool attr_set[64] = {};
  if (!ensure_dynamic_smem(k_dhw_umma<H>, C::SMEM_BYTES, attr_set)) return -1;
  const bool aligned = (reinterpret_cast<uintptr_t>(dW) & 15) == 0;    // the caller's buffer may sit on any 4-byte boundary
  CUtensorMap mg, mh, mw, mo, md;
  if (!make_map(&mg, dzb, uint64_t(rows), H, BM) || !make_map(&mh, h, uint64_t(rows), H, BM) ||
      !make_map(&mw, W, H, H, 128) || !make_map_f32(&mo, dh, uint64_t(rows), H))
    return -1;
  if (aligned) { if (!make_map_f32(&md, dW, H, H)) return -1; }
  else md = mo;
  // at least two tiles per CTA: every CTA ends with a reduction of its part of dW into the gradient
  const int tiles = (rows + BM - 1) / BM, want = (tiles + 1) / 2, most = kNumSMs / C::HALVES;
  launch(k_dhw_umma<H>, (want < most ? want : most) * C::HALVES, kThreads, C::SMEM_BYTES, st,
         mg, mh, mw, mo, md, dW, rows, aligned, status);
  return 1;
}

}  // namespace

// bf16 models of hidden 128, 256 or 512 (the widths whose dz is kept in bf16 for these products)
bool bwd_umma_supported(const Dims& d) {
  return d.dtype == XRL_BF16 && (d.H == 128 || d.H == 256 || d.H == 512) && encode_fn() != nullptr;
}
// dh [rows x H] = dzb W^T where h > 0, else 0, and dW [H x H] += h^T dzb.  Returns kernels launched, or -1.
int launch_bwd_umma(const Dims& d, const void* h, const void* dzb, const void* W, float* dh, float* dW, int32_t rows,
                    int32_t* status, cudaStream_t st) {
  if (rows <= 0) return 0;
  int a, b;
  switch (d.H) {
    case 128:
      return launch_dhw<128>(h, dzb, W, dh, dW, rows, status, st);
    case 256:
      return launch_dhw<256>(h, dzb, W, dh, dW, rows, status, st);
    case WIDE:
      a = launch_dw(h, dzb, dW, rows, status, st);
      b = launch_dh(h, dzb, W, dh, rows, status, st);
      break;
    default: return -1;
  }
  return a < 0 || b < 0 ? -1 : a + b;
}

}  // namespace xrl
