// Device code of the tensor-core node transform (paper Eq. 7, Z = h W with the per-head attention
// half-scores taken from the fp32 accumulators), shared by the kernel that runs one layer per launch
// and by the kernel that runs all layers of a small step in one launch: shared-memory layout and the
// three roles (TMA producer, MMA issuer, epilogue) as routines over a CTA's tiles.  The counters a
// role passes by reference carry the positions in the stage ring and in the accumulator pair from one
// call to the next, so that a role can be called once per layer on the same barriers.
#pragma once

#include "xrl_umma.cuh"

namespace xrl {
namespace xform {

using namespace umma;

constexpr int BM = 128;                 // rows per tile (UMMA M)
constexpr int STAGE_BYTES = BM * 128;   // one A stage / one output staging tile: 128 rows x 128 B

// NS: output columns a CTA computes (its slice of W, resident in shared memory); KP: input width padded to whole
// 64-element chunks (the TMA unit fills what lies beyond the matrix with zeros).  NS = KP = H for hidden 128 and 256.
// STAGED: two staging tiles for an epilogue that leaves through the TMA unit.
template <int NS, int KP = NS, bool STAGED = false> struct Cfg {
  static_assert(NS % 32 == 0 && NS >= 32 && NS <= 256 && KP % KCH == 0, "tile shapes of tcgen05.mma and of the swizzle");
  static constexpr int KC = KP / KCH;                   // K chunks
  static constexpr int NC = (NS + KCH - 1) / KCH;       // output column chunks
  static constexpr int W_CHUNK_BYTES = NS * 128;        // N rows x 128 B
  static constexpr int W_BYTES = KC * W_CHUNK_BYTES;
  static constexpr int STAGES = (W_BYTES > 64 * 1024 ? 6 : 8) - (STAGED ? 2 : 0);
  static constexpr int ACC_COLS = NS <= 32 ? 32 : NS <= 64 ? 64 : NS <= 128 ? 128 : 256;
  static constexpr int TMEM_COLS = 2 * ACC_COLS;        // two fp32 accumulators of N columns, a power of two apart
  static constexpr int OFF_A = W_BYTES;
  static constexpr int OFF_OUT = OFF_A + STAGES * STAGE_BYTES;
  static constexpr int OFF_AVEC = OFF_OUT + (STAGED ? 2 * STAGE_BYTES : 0);
  static constexpr int OFF_BAR = OFF_AVEC + 2 * NS * 4;
  static constexpr int NUM_BARS = 1 + 2 * STAGES + 4;
  static constexpr int OFF_TMEM = OFF_BAR + NUM_BARS * 8;   // [0] TMEM base address, [1] abort flag
  static constexpr int SMEM_BYTES = OFF_TMEM + 16;
  static_assert(SMEM_BYTES <= 227 * 1024, "shared memory of one SM");

  __device__ static uint32_t bar_w(uint32_t base) { return base + OFF_BAR; }
  __device__ static uint32_t bar_a_full(uint32_t base, int s) { return base + OFF_BAR + 8u * (1 + s); }
  __device__ static uint32_t bar_a_empty(uint32_t base, int s) { return base + OFF_BAR + 8u * (1 + STAGES + s); }
  __device__ static uint32_t bar_acc_full(uint32_t base, int b) { return base + OFF_BAR + 8u * (1 + 2 * STAGES + b); }
  __device__ static uint32_t bar_acc_empty(uint32_t base, int b) {
    return base + OFF_BAR + 8u * (1 + 2 * STAGES + 2 + b);
  }
};

// One thread: barriers of the layout above (`frees` arrivals of the epilogue free an accumulator).
template <typename C> __device__ __forceinline__ void init_barriers(uint32_t base, int frees) {
  mbar_init(C::bar_w(base), 1);
  for (int s = 0; s < C::STAGES; ++s) { mbar_init(C::bar_a_full(base, s), 1); mbar_init(C::bar_a_empty(base, s), 1); }
  for (int b = 0; b < 2; ++b) { mbar_init(C::bar_acc_full(base, b), 1); mbar_init(C::bar_acc_empty(base, b), frees); }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  fence_async_smem();
}

// One thread: rows col0 .. col0 + NS - 1 of W^T (K-major bf16) into the start of shared memory; completion on bar_w.
template <typename C> __device__ __forceinline__ void load_w(uint32_t base, const CUtensorMap* map_w, int col0 = 0) {
  mbar_expect_tx(C::bar_w(base), C::W_BYTES);
  for (int kc = 0; kc < C::KC; ++kc) tma_load_2d(base + kc * C::W_CHUNK_BYTES, map_w, kc * KCH, col0, C::bar_w(base));
}

// One thread: the A tiles first, first + step, ... < num_tiles through the stage ring.  False on a timeout.
template <typename C>
__device__ __forceinline__ bool produce_tiles(uint32_t base, const CUtensorMap* map_h, int first, int step,
                                              int num_tiles, uint32_t& it) {
  for (int tile = first; tile < num_tiles; tile += step) {
    for (int kc = 0; kc < C::KC; ++kc, ++it) {
      const int s = it % C::STAGES;
      const uint32_t round = it / C::STAGES;
      if (round > 0 && !mbar_wait(C::bar_a_empty(base, s), (round - 1) & 1)) return false;
      mbar_expect_tx(C::bar_a_full(base, s), STAGE_BYTES);
      tma_load_2d(base + C::OFF_A + s * STAGE_BYTES, map_h, kc * KCH, tile * BM, C::bar_a_full(base, s));
    }
  }
  return true;
}

// After a producer timeout: let the loads already issued land before the CTA's shared memory goes away.
template <typename C> __device__ __forceinline__ void drain_producer(uint32_t base, uint32_t it, uint32_t w_parity) {
  const uint32_t first = it > uint32_t(C::STAGES) ? it - C::STAGES : 0;
  for (uint32_t j = first; j < it; ++j) mbar_wait(C::bar_a_full(base, j % C::STAGES), (j / C::STAGES) & 1);
  mbar_wait(C::bar_w(base), w_parity);
}

// One thread: tcgen05.mma (M = 128, N = NS, K = 16) over the same tiles, alternating between the two
// accumulators; waits for W (phase w_parity of bar_w) first.  False on a timeout.
template <typename C, int NS>
__device__ __forceinline__ bool mma_tiles(uint32_t base, uint32_t tmem_base, int first, int step, int num_tiles,
                                          uint32_t& it, uint32_t& lt, uint32_t w_parity) {
  constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(NS >> 3) << 17) |
                             (uint32_t(BM >> 4) << 24);   // fp32 accum, bf16 x bf16, K-major both
  if (!mbar_wait(C::bar_w(base), w_parity)) return false;
  tc_fence_after();
  for (int tile = first; tile < num_tiles; tile += step, ++lt) {
    const int buf = lt & 1;
    const uint32_t use = lt >> 1;
    if (use > 0 && !mbar_wait(C::bar_acc_empty(base, buf), (use - 1) & 1)) return false;
    tc_fence_after();
    const uint32_t tmem_d = tmem_base + uint32_t(buf * C::ACC_COLS);
    for (int kc = 0; kc < C::KC; ++kc, ++it) {
      const int s = it % C::STAGES;
      if (!mbar_wait(C::bar_a_full(base, s), (it / C::STAGES) & 1)) return false;
      tc_fence_after();
      const uint32_t a_addr = base + C::OFF_A + s * STAGE_BYTES;
      const uint32_t b_addr = base + kc * C::W_CHUNK_BYTES;
#pragma unroll
      for (int k = 0; k < KCH / 16; ++k)
        tc_mma(tmem_d, smem_desc(a_addr + k * 32), smem_desc(b_addr + k * 32), idesc, (kc | k) != 0 ? 1u : 0u);
      tc_commit(C::bar_a_empty(base, s));       // the stage is free once these MMAs have read it
    }
    tc_commit(C::bar_acc_full(base, buf));      // the accumulator is complete
  }
  return true;
}

__device__ __forceinline__ void fma_pair(unsigned long long& acc, uint32_t z0, uint32_t z1, float s0, float s1) {
  unsigned long long z, s;
  asm("mov.b64 %0, {%1, %2};" : "=l"(z) : "r"(z0), "r"(z1));
  asm("mov.b64 %0, {%1, %2};" : "=l"(s) : "f"(s0), "f"(s1));
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(z), "l"(s));
}
__device__ __forceinline__ float pair_sum(unsigned long long a) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a));
  return lo + hi;
}

// Groups of four epilogue warps on one tile: two where its halves are whole 32-column pieces and heads, else one.
__host__ __device__ constexpr int epilogue_groups(int NS, int d) { return NS % 64 == 0 && (NS / 2) % d == 0 ? 2 : 1; }

// The epilogue warps (two groups of four from CTA warp 2 on; warp q = warp & 3 of a group reads tensor-memory lanes
// [32 q, 32 q + 32)): per tile the half-scores from the fp32 accumulators and Z rounded to bf16, a lane per row, written
// straight from registers in whole 32-byte sectors.  With `groups` = 2 a group takes half of every tile's columns.  With one
// group per tile the two take tiles in turn, an accumulator each, where a CTA has all of a power of two of columns (one head at
// 64, 128 or 256: 1.02 M rows 58, 93 and 184 us per layer with an idle second group, 51, 89 and 178 in turn; four warps and
// TMA stores 76, 95 and 180); elsewhere the second group has nothing to do (both storing rows of other lengths at once: 192 with
// three heads 134 -> 140 us, 160, 224, 96 and 32 +1 to +3 %, slices of 320 to 512 +1 to +3 %).  No barrier between the
// warps: each waits for the accumulator and frees it on its own.
// (Through swizzled staging tiles and TMA stores, two CTA barriers and a proxy fence per 64 columns, four warps took 3.3 us
// per 128 x 256 tile, which held the large steps' transform to what 148 such epilogues can do: 2.8 M rows 0.58 -> 0.49 ms,
// 4.1 M 0.79 -> 0.73, 124 k rows of 192 26.6 -> 22.1 us, the all-layers kernel of a small step 65.5 -> 61.8.  Eight warps
// with a staging tile per group and TMA stores: 0.51 and 0.72 ms, the steps within 1.5 %.  The node update's epilogue, which
// has no half-scores, is slower this way: 0.41 -> 0.63 ms at 4.1 M rows.)
// A timeout sets the abort word behind the tensor-memory slot and raises XRL_ERR_TIMEOUT.
// The CTA's NS columns are the matrix's columns col0 ... (Z: rows of z_row bytes from column col0 on) and their heads (of `d`
// columns, whole heads within the NS) go to scores[row * score_stride + 0 ...]; columns and heads from `cols_left` on do not
// exist.  scores = nullptr: none are taken.  ROUNDED: the half-scores are those of Z as stored (rounded), not of the
// accumulators.  HD: the head width where it is known (16, 32 or 64; half-scores then leave in pieces of up to 32 bytes), or 0.
template <typename C, int NS, bool ROUNDED, int HD>
__device__ __forceinline__ void epilogue_tiles(uint8_t* smem, uint32_t base, uint32_t tmem_base, char* __restrict__ Z,
                                               int z_row, float2* __restrict__ scores, int score_stride, int rows, int d,
                                               int groups, int first, int step, int num_tiles, uint32_t& lt, int32_t* status,
                                               int cols_left = NS) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int q = warp & 3, grp = (warp - 2) >> 2;
  constexpr bool kTurns = NS == C::KC * KCH && (NS & (NS - 1)) == 0;
  if (!kTurns && grp >= groups) { lt += num_tiles > first ? (num_tiles - first + step - 1) / step : 0; return; }
  const int row_in_tile = q * 32 + lane;
  const int c0 = groups == 2 ? grp * (NS / 2) : 0, c1 = groups == 2 ? c0 + NS / 2 : NS;
  const float* avec = reinterpret_cast<const float*>(smem + C::OFF_AVEC);
  volatile uint32_t* abort_flag = reinterpret_cast<uint32_t*>(smem + C::OFF_TMEM) + 1;
  for (int tile = first; tile < num_tiles; tile += step, ++lt) {
    const int buf = lt & 1;
    if (kTurns && groups == 1 && buf != grp) continue;
    uint32_t ok = 1;
    if (lane == 0) ok = mbar_wait(C::bar_acc_full(base, buf), (lt >> 1) & 1) ? 1u : 0u;
    ok = __shfl_sync(0xFFFFFFFFu, ok, 0);
    if (!ok) {
      if (lane == 0) { *abort_flag = 1; raise(status, XRL_ERR_TIMEOUT); }
      break;
    }
    tc_fence_after();
    const uint32_t taddr = tmem_base + (uint32_t(q * 32) << 16) + uint32_t(buf * C::ACC_COLS);
    const int64_t grow = int64_t(tile) * BM + row_in_tile;
    const bool live = grow < rows;
    char* zr = Z + grow * z_row;
    float2* sr = scores + grow * score_stride;
    unsigned long long ss = 0ull, sd = 0ull;
    int head = c0 / d, left = d;               // columns left in the current head
    uint32_t sc[8];                            // (HD) half-scores of up to four heads
#pragma unroll 2
    for (int c = c0; c < c1; c += 32) {
      uint32_t v[32];
      tc_ld32(taddr + c, v);
      tc_wait_ld();
      if (c + 32 >= c1) {                      // everything this warp needs has left tensor memory
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(C::bar_acc_empty(base, buf));
      }
      uint32_t pk[16];
#pragma unroll
      for (int t = 0; t < 16; ++t) pk[t] = pack_bf16x2(__uint_as_float(v[2 * t]), __uint_as_float(v[2 * t + 1]));
      if (ROUNDED) {                           // Z as it will be stored
#pragma unroll
        for (int t = 0; t < 16; ++t) { v[2 * t] = pk[t] << 16; v[2 * t + 1] = pk[t] & 0xFFFF0000u; }
      }
#pragma unroll
      for (int g = 0; g < 4; ++g) {            // eight columns at a time
        const float4* as = reinterpret_cast<const float4*>(avec + c + g * 8);
        const float4* ad = reinterpret_cast<const float4*>(avec + NS + c + g * 8);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float4 s4 = as[e], d4 = ad[e];
          const uint32_t* z = &v[g * 8 + e * 4];
          fma_pair(ss, z[0], z[1], s4.x, s4.y); fma_pair(sd, z[0], z[1], d4.x, d4.y);
          fma_pair(ss, z[2], z[3], s4.z, s4.w); fma_pair(sd, z[2], z[3], d4.z, d4.w);
        }
        if (HD == 0) {
          left -= 8;
          if (left == 0) {
            if (live && scores != nullptr && c + g * 8 < cols_left) sr[head] = make_float2(pair_sum(ss), pair_sum(sd));
            ss = sd = 0ull; ++head; left = d;
          }
        } else if ((c - c0 + g * 8 + 8) % (HD == 0 ? 8 : HD) == 0) {        // a head ends here
          const int slot = (c - c0 + g * 8) / (HD == 0 ? 8 : HD) & 3;
          const uint32_t x = __float_as_uint(pair_sum(ss)), y = __float_as_uint(pair_sum(sd));
          ss = sd = 0ull;
#pragma unroll
          for (int t = 0; t < 4; ++t)
            if (slot == t) { sc[2 * t] = x; sc[2 * t + 1] = y; }
          if (slot == 3 || c + g * 8 + 8 >= c1) {
            float2* p = sr + head;             // (four heads, two or one: a piece's start is a multiple of its size)
            if (live) {
              if (slot == 3) store32(p, sc[0], sc[1], sc[2], sc[3], sc[4], sc[5], sc[6], sc[7]);
              else if (slot == 0) *reinterpret_cast<uint2*>(p) = make_uint2(sc[0], sc[1]);
              else *reinterpret_cast<uint4*>(p) = make_uint4(sc[0], sc[1], sc[2], sc[3]);
            }
            head += slot + 1;
          }
        }
      }
      if (live && c < cols_left) {
        store32(zr + c * 2, pk[0], pk[1], pk[2], pk[3], pk[4], pk[5], pk[6], pk[7]);
        store32(zr + c * 2 + 32, pk[8], pk[9], pk[10], pk[11], pk[12], pk[13], pk[14], pk[15]);
      }
    }
  }
}

}  // namespace xform
}  // namespace xrl
