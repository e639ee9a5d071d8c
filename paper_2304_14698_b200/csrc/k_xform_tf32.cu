// Dense node transform of a graph-attention layer, Z = h W (paper Eq. 7), for fp32 storage on the 5th-generation tensor
// cores: every operand is split into hi = tf32(x) and lo = tf32(x - hi), and Z = lo_h hi_W + hi_h lo_W + hi_h hi_W
// accumulates in fp32 (tcgen05.mma kind::tf32; the dropped lo lo term is below 2^-22 of a product).
//
// One persistent CTA per SM.  Both splits of a slice of W^T (NS output columns, all K inputs) stay in shared memory for the
// whole launch (128 KB at hidden 128).  Eight loader warps bring 128-row tiles of h in 32-column chunks, two chunks ahead
// in registers, split them and write both parts into a two-stage ring of 128-byte-swizzled tiles; one thread issues the
// products into one of two accumulators in tensor memory; four epilogue warps take the half-scores from the accumulators
// and store Z through a swizzled staging tile by TMA.  Bound by HBM (8 H bytes per row) once the pipeline is full; steps of
// tens of thousands of rows are two tiles per SM, i.e. fill and drain.  The same arithmetic on mma.sync (k_xform_tf32x3)
// waits on shared-memory fragment loads: 29.5 us per layer of 36 k rows at hidden 128, here 14.3, with the same error against
// 64 bits (1.3e-6 of the embeddings).
//
// Every wait on an mbarrier is bounded; on expiry the kernel records XRL_ERR_TIMEOUT, frees its tensor memory and returns.
#include "xrl_umma.cuh"

namespace xrl {

using namespace umma;

namespace {

constexpr int BM = 128;                      // rows per tile
constexpr int KC32 = 32;                     // fp32 columns per 128-byte swizzle row
constexpr int TILE = BM * 128;               // one part of a chunk: 128 rows x 128 bytes
constexpr int kLoaders = 8;                  // loader warps
constexpr int kThreads = 32 * (1 + 4 + kLoaders);
constexpr int STAGES = 2;

template <int NS, int K> struct TCfg {
  static constexpr int KC = K / KC32;                       // chunks
  static constexpr int W_PART = KC * NS * 128;              // one part of W's slice
  static constexpr int OFF_A = 2 * W_PART;
  static constexpr int OFF_OUT = OFF_A + STAGES * 2 * TILE;
  static constexpr int OFF_AVEC = OFF_OUT + 2 * TILE;
  static constexpr int OFF_BAR = OFF_AVEC + 2 * NS * 4;
  static constexpr int OFF_TMEM = OFF_BAR + 8 * (2 * STAGES + 4);
  static constexpr int SMEM_BYTES = OFF_TMEM + 16;
  static constexpr int ACC_COLS = NS <= 32 ? 32 : NS <= 64 ? 64 : 128;
  static constexpr int TMEM_COLS = 2 * ACC_COLS;
  static_assert(NS % 32 == 0 && NS <= 128 && K % KC32 == 0 && SMEM_BYTES <= 227 * 1024, "tile shapes");
};

__device__ __forceinline__ float to_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}
__device__ __forceinline__ void split4(const float4& v, float4& hi, float4& lo) {
  hi = make_float4(to_tf32(v.x), to_tf32(v.y), to_tf32(v.z), to_tf32(v.w));
  lo = make_float4(to_tf32(v.x - hi.x), to_tf32(v.y - hi.y), to_tf32(v.z - hi.z), to_tf32(v.w - hi.w));
}
__device__ __forceinline__ void tc_mma_tf32(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(acc) : "memory");
}

template <int NS, int K>
__global__ void __launch_bounds__(kThreads, 1)
k_xform_tf32(const float* __restrict__ h, const float* __restrict__ Wt, const __grid_constant__ CUtensorMap map_z,
             const float* __restrict__ a_src, const float* __restrict__ a_dst, float2* __restrict__ scores, int heads,
             int rows, int d, int slices, int32_t* status) {
  using C = TCfg<NS, K>;
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t base = smem_u32(smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int num_tiles = (rows + BM - 1) / BM;
  const int slice = int(blockIdx.x) % slices, first = int(blockIdx.x) / slices, step = int(gridDim.x) / slices;
  const int col0 = slice * NS;
  if ((base & 1023u) != 0) {
    if (threadIdx.x == 0) raise(status, XRL_ERR_UNSUPPORTED);
    return;
  }
  auto bar_full = [&](int s) { return base + C::OFF_BAR + 8u * s; };
  auto bar_empty = [&](int s) { return base + C::OFF_BAR + 8u * (STAGES + s); };
  auto bar_acc_full = [&](int b) { return base + C::OFF_BAR + 8u * (2 * STAGES + b); };
  auto bar_acc_empty = [&](int b) { return base + C::OFF_BAR + 8u * (2 * STAGES + 2 + b); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_TMEM);
  float* avec = reinterpret_cast<float*>(smem + C::OFF_AVEC);
  if (threadIdx.x == 0) {
    tmem_slot[1] = 0;
    for (int s = 0; s < STAGES; ++s) { mbar_init(bar_full(s), 32 * kLoaders); mbar_init(bar_empty(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(bar_acc_full(b), 1); mbar_init(bar_acc_empty(b), 128); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  // attention vectors pre-multiplied by log2(e): the half-scores are consumed by an exp2 softmax
  for (int t = threadIdx.x; t < NS; t += kThreads) {
    avec[t] = a_src[col0 + t] * kLog2e;
    avec[NS + t] = a_dst[col0 + t] * kLog2e;
  }
  // both parts of W^T's rows col0 .. col0 + NS - 1, in the operand layout
  for (int t = threadIdx.x; t < NS * (K / 4); t += kThreads) {
    const int n = t / (K / 4), p = t - n * (K / 4);          // 16-byte piece p of row n
    const float4 v = __ldg(reinterpret_cast<const float4*>(Wt + size_t(col0 + n) * K) + p);
    float4 hi, lo;
    split4(v, hi, lo);
    const int at = (p >> 3) * NS * 128 + n * 128 + (((p & 7) ^ (n & 7)) << 4);
    *reinterpret_cast<float4*>(smem + at) = hi;
    *reinterpret_cast<float4*>(smem + C::W_PART + at) = lo;
  }
  fence_async_smem();
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(uint32_t(C::TMEM_COLS)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  enter();

  if (warp == 0) {
    // ---- MMA issuer -------------------------------------------------------------------------------
    if (lane == 0) {
      constexpr uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | (uint32_t(NS >> 3) << 17) | (uint32_t(BM >> 4) << 24);
      bool ok = true;
      uint32_t it = 0, lt = 0;
      for (int tile = first; tile < num_tiles && ok; tile += step, ++lt) {
        const int buf = lt & 1;
        if ((lt >> 1) > 0 && !mbar_wait(bar_acc_empty(buf), ((lt >> 1) - 1) & 1)) { ok = false; break; }
        tc_fence_after();
        const uint32_t acc = tmem_base + uint32_t(buf * C::ACC_COLS);
        for (int kc = 0; kc < C::KC; ++kc, ++it) {
          const int s = it % STAGES;
          if (!mbar_wait(bar_full(s), (it / STAGES) & 1)) { ok = false; break; }
          tc_fence_after();
          const uint32_t ah = base + C::OFF_A + s * 2 * TILE, al = ah + TILE;
          const uint32_t bh = base + kc * NS * 128, bl = bh + C::W_PART;
#pragma unroll
          for (int k = 0; k < KC32 / 8; ++k) {
            tc_mma_tf32(acc, smem_desc(al + k * 32), smem_desc(bh + k * 32), idesc, (kc | k) != 0 ? 1u : 0u);
            tc_mma_tf32(acc, smem_desc(ah + k * 32), smem_desc(bl + k * 32), idesc, 1u);
            tc_mma_tf32(acc, smem_desc(ah + k * 32), smem_desc(bh + k * 32), idesc, 1u);
          }
          tc_commit(bar_empty(s));
        }
        if (ok) tc_commit(bar_acc_full(buf));
      }
      if (!ok) raise(status, XRL_ERR_TIMEOUT);
    }
  } else if (warp <= 4) {
    // ---- epilogue ---------------------------------------------------------------------------------
    const int q = warp & 3, row_in_tile = q * 32 + lane;
    const bool leader = threadIdx.x == 32;
    volatile uint32_t* abort_flag = tmem_slot + 1;
    uint32_t lt = 0, stores = 0;
    for (int tile = first; tile < num_tiles; tile += step, ++lt) {
      const int buf = lt & 1;
      uint32_t okw = 1;
      if (lane == 0) okw = mbar_wait(bar_acc_full(buf), (lt >> 1) & 1) ? 1u : 0u;
      okw = __shfl_sync(0xFFFFFFFFu, okw, 0);
      if (!okw && lane == 0) { *abort_flag = 1; raise(status, XRL_ERR_TIMEOUT); }
      epi_barrier();
      if (*abort_flag) break;
      tc_fence_after();
      const uint32_t taddr = tmem_base + (uint32_t(q * 32) << 16) + uint32_t(buf * C::ACC_COLS);
      const int64_t grow = int64_t(tile) * BM + row_in_tile;
      const bool live = grow < rows;
      float ss = 0.f, sd = 0.f;
      int head = col0 / d, left = d;             // (whole heads per slice, or no scores are taken)
      for (int c = 0; c < NS / 32; ++c, ++stores) {
        uint32_t v[32];
        tc_ld32(taddr + c * 32, v);
        tc_wait_ld();
#pragma unroll
        for (int g = 0; g < 4; ++g) {              // half-scores, eight columns at a time
          const float4* as = reinterpret_cast<const float4*>(avec + c * 32 + g * 8);
          const float4* ad = reinterpret_cast<const float4*>(avec + NS + c * 32 + g * 8);
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float4 s4 = as[e], d4 = ad[e];
            const uint32_t* z = &v[g * 8 + e * 4];
            ss = fmaf(__uint_as_float(z[0]), s4.x, ss); sd = fmaf(__uint_as_float(z[0]), d4.x, sd);
            ss = fmaf(__uint_as_float(z[1]), s4.y, ss); sd = fmaf(__uint_as_float(z[1]), d4.y, sd);
            ss = fmaf(__uint_as_float(z[2]), s4.z, ss); sd = fmaf(__uint_as_float(z[2]), d4.z, sd);
            ss = fmaf(__uint_as_float(z[3]), s4.w, ss); sd = fmaf(__uint_as_float(z[3]), d4.w, sd);
          }
          left -= 8;
          if (left == 0) {
            if (live && scores != nullptr) scores[grow * heads + head] = make_float2(ss, sd);
            ss = 0.f; sd = 0.f; ++head; left = d;
          }
        }
        // the two staging tiles alternate from store to store: this one's last store must have read it
        if (leader) tma_wait_read<1>();
        epi_barrier();
        uint8_t* p = smem + C::OFF_OUT + (stores & 1) * TILE + row_in_tile * 128;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          *reinterpret_cast<uint4*>(p + ((j ^ (row_in_tile & 7)) << 4)) = make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        fence_async_smem();
        epi_barrier();
        if (leader) {
          tma_store_2d(&map_z, base + C::OFF_OUT + (stores & 1) * TILE, col0 + c * 32, tile * BM);
          tma_commit();
        }
      }
      tc_fence_before();
      mbar_arrive(bar_acc_empty(buf));
    }
    if (leader) tma_wait_all();
  } else {
    // ---- loaders: chunk i of this CTA's sequence of (tile, chunk) pairs, four 16-byte pieces per thread -------------
    const int t = threadIdx.x - 160;
    const int my_tiles = first < num_tiles ? (num_tiles - first + step - 1) / step : 0;
    const int total = my_tiles * C::KC;
    auto fetch = [&](int i, float4 (&v)[4]) {
      const int tile = first + (i / C::KC) * step, kc = i % C::KC;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int idx = t + 256 * u, row = idx >> 3, p = idx & 7;
        const int64_t r = int64_t(tile) * BM + row;
        v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < total && r < rows) v[u] = *(reinterpret_cast<const float4*>(h + size_t(r) * K + kc * KC32) + p);
      }
    };
    float4 a[4], b[4];
    fetch(0, a);
    fetch(1, b);
    bool ok = true;
    auto put = [&](int i, float4 (&v)[4]) {
      const int s = i % STAGES, round = i / STAGES;
      if (round > 0 && !mbar_wait(bar_empty(s), (round - 1) & 1)) { raise(status, XRL_ERR_TIMEOUT); ok = false; return; }
      uint8_t* hi_t = smem + C::OFF_A + s * 2 * TILE;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int idx = t + 256 * u, row = idx >> 3, p = idx & 7;
        float4 hi, lo;
        split4(v[u], hi, lo);
        const int at = row * 128 + ((p ^ (row & 7)) << 4);
        *reinterpret_cast<float4*>(hi_t + at) = hi;
        *reinterpret_cast<float4*>(hi_t + TILE + at) = lo;
      }
      fence_async_smem();
      mbar_arrive(bar_full(s));
      fetch(i + 2, v);
    };
    for (int i = 0; i < total && ok; i += 2) {
      put(i, a);
      if (ok && i + 1 < total) put(i + 1, b);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                 ::"r"(tmem_base), "r"(uint32_t(C::TMEM_COLS)) : "memory");
  }
}

template <int NS, int K>
int launch_h(const Dims& d, const float* h, const LayerWeights& lw, float* Z, float2* scores, int64_t rows, int32_t* status,
             cudaStream_t st) {
  using C = TCfg<NS, K>;
  static bool attr_set[64] = {};
  if (!ensure_dynamic_smem(k_xform_tf32<NS, K>, C::SMEM_BYTES, attr_set)) return -1;
  EncodeTiledFn fn = encode_fn();
  if (!fn) return -1;
  CUtensorMap mz;
  cuuint64_t dims[2] = {cuuint64_t(K), cuuint64_t(rows)};
  cuuint64_t strides[1] = {cuuint64_t(K) * 4};
  cuuint32_t box[2] = {KC32, BM};
  cuuint32_t estr[2] = {1, 1};
  if (fn(&mz, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, Z, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
         CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return -1;
  const int slices = K / NS, tiles = int((rows + BM - 1) / BM), groups = kNumSMs / slices;
  const int head = d.H / d.K;
  const bool whole = slices == 1 || NS % head == 0;      // else a head crosses a slice's end: half-scores from Z afterwards
  launch(k_xform_tf32<NS, K>, (tiles < groups ? tiles : groups) * slices, kThreads, C::SMEM_BYTES, st,
      h, static_cast<const float*>(lw.Wt), mz, lw.a_src, lw.a_dst, whole ? scores : nullptr, d.K, int(rows), head, slices, status);
  return whole ? 1 : 0;
}

}  // namespace

// fp32 storage, hidden 32, 64, 96, 128 (whole rows per CTA), 192, 256 (slices of 64 columns).  Returns 1 when the half-scores
// were taken too, 0 when k_scores has to follow, -1 when the shape is not handled.
int launch_xform_tf32(const Dims& d, const float* h, const LayerWeights& lw, float* Z, float2* scores, int64_t rows,
                      int32_t* status, cudaStream_t st) {
  if (d.dtype != XRL_FP32 || rows <= 0) return -1;
#define TF32_CASE(H_, NS_) \
  case H_: return launch_h<NS_, H_>(d, h, lw, Z, scores, rows, status, st);
  switch (d.H) {
    TF32_CASE(32, 32) TF32_CASE(64, 64) TF32_CASE(96, 96) TF32_CASE(128, 128) TF32_CASE(192, 64) TF32_CASE(256, 64)
    default: return -1;
  }
#undef TF32_CASE
}

}  // namespace xrl
