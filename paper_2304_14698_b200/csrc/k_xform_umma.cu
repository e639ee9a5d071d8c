// Dense node transform of a graph-attention layer on the 5th-generation tensor cores:
// Z = h W (paper Eq. 7, the "W h_j" term) for bf16 storage, fp32 accumulation in tensor memory,
// with the per-head attention half-scores s_src = a_src . Z_k, s_dst = a_dst . Z_k taken from the
// fp32 accumulators in the epilogue.
//
// One persistent CTA per SM.  W^T (the K-major B operand, bf16) stays resident in shared memory; 128-row tiles of h
// stream through a ring of TMA-loaded, 128-byte-swizzled stages; one thread issues tcgen05.mma (M = 128, N = NS,
// K = 16) into one of two accumulator buffers in tensor memory; eight epilogue warps read the accumulators back
// (tcgen05.ld), form the half-scores, round Z to bf16 and write it from registers, whole sectors per lane.
// The op moves 2 H b bytes per node against 2 H^2 flops: up to hidden 256 it is bound by HBM, not by the tensor
// pipe, so the design goal is to keep loads and stores streaming.
//
// Hidden sizes: every multiple of 32 up to 512 (what the library supports).  Up to 256 a CTA holds all of W (128 KB at
// 256) and computes whole rows.  Above, W no longer fits one SM (512 KB at 512): a CTA keeps a slice of 128 output columns
// (128 KB at 512) for the whole launch and the CTAs of a row tile's slices run side by side, so that its second
// to fourth reading of h comes from L2.  Widths that are not a multiple of 64 leave the last chunk
// of the way in to the TMA unit's bounds (zeros); on the way out pieces of 32 columns beyond the width are not written.
// Measured: hidden 192, 124 k rows, 0.286 ms per layer with the CUDA-core product plus 0.052 ms for the half-scores
// -> 0.022 ms (95 MB: 4.3 TB/s); hidden 256, 4.1 M rows, 0.73 ms (4.5 GB: 6.2 TB/s), 2.8 M rows 0.58 -> 0.49 ms.
//
// Every wait on an mbarrier is bounded; on expiry the kernel records XRL_ERR_TIMEOUT, drains its
// own copies in flight, frees its tensor memory and returns.
#include "xrl_xform_umma.cuh"

namespace xrl {

using namespace umma;
using namespace xform;

namespace {

constexpr int kThreads = 320;           // warp 0 TMA, warp 1 MMA, warps 2..9 epilogue

template <int NS, int KP, bool ROUNDED, int HD>
__global__ void __launch_bounds__(kThreads, 1)
k_xform_umma(const __grid_constant__ CUtensorMap map_h, const __grid_constant__ CUtensorMap map_w,
             char* __restrict__ Z, int z_row, const float* __restrict__ a_src,
             const float* __restrict__ a_dst, float2* __restrict__ scores, int score_stride,
             int rows, int H, int d, int slices, int32_t* status) {
  using C = Cfg<NS, KP>;
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t base = smem_u32(smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int num_tiles = (rows + BM - 1) / BM;
  // slices = 1 up to hidden 256; else CTA = (row tile group, slice of NS columns), slices of a tile side by side
  const int slice = int(blockIdx.x) % slices, first = int(blockIdx.x) / slices, step = int(gridDim.x) / slices;
  const int col0 = slice * NS, cols = min(NS, H - col0);

  if ((base & 1023u) != 0) {               // the swizzled tiles need 1024-byte alignment
    if (threadIdx.x == 0) raise(status, XRL_ERR_UNSUPPORTED);
    return;
  }
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_TMEM);
  float* avec = reinterpret_cast<float*>(smem + C::OFF_AVEC);

  if (threadIdx.x == 0) {
    tmem_slot[1] = 0;
    init_barriers<C>(base, 4 * epilogue_groups(NS, d));
  }
  // attention vectors pre-multiplied by log2(e): the half-scores are consumed by an exp2 softmax
  for (int t = threadIdx.x; t < NS; t += kThreads) {
    avec[t] = t < cols ? a_src[col0 + t] * kLog2e : 0.f;
    avec[NS + t] = t < cols ? a_dst[col0 + t] * kLog2e : 0.f;
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
    // ---- TMA producer ---------------------------------------------------------------------------
    if (lane == 0) {
      load_w<C>(base, &map_w, col0);
      enter();
      uint32_t it = 0;
      if (!produce_tiles<C>(base, &map_h, first, step, num_tiles, it)) {
        raise(status, XRL_ERR_TIMEOUT);
        drain_producer<C>(base, it, 0);
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer -----------------------------------------------------------------------------
    if (lane == 0) {
      enter();
      uint32_t it = 0, lt = 0;
      if (!mma_tiles<C, NS>(base, tmem_base, first, step, num_tiles, it, lt, 0)) raise(status, XRL_ERR_TIMEOUT);
    }
  } else {
    // ---- epilogue: two groups of four warps ----------------------------------------------------------
    uint32_t lt = 0;
    enter();
    epilogue_tiles<C, NS, ROUNDED, HD>(smem, base, tmem_base, Z + col0 * 2, z_row, scores ? scores + col0 / d : nullptr,
                                       score_stride, rows, d, epilogue_groups(NS, d), first, step, num_tiles, lt, status, cols);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                 ::"r"(tmem_base), "r"(uint32_t(C::TMEM_COLS)) : "memory");
  }
}

// Widths 128 and 256 take the half-scores from the fp32 accumulators, the others from Z as it is stored (both are
// fixed per model, so that the forward and the reverse pass of a model see the same scores).
template <int NS, int KP, int HD = 0>
int launch_h(const Dims& d, const void* h, const LayerWeights& lw, void* Z, float* scores,
             Window win, int32_t* status, cudaStream_t st) {
  using C = Cfg<NS, KP>;
  constexpr bool kRounded = !(NS == KP && (NS == 128 || NS == 256));
  static bool attr_set[64] = {};
  if (!ensure_dynamic_smem(k_xform_umma<NS, KP, kRounded, HD>, C::SMEM_BYTES, attr_set)) return -1;
  const int64_t rows = int64_t(win.row_end) - win.row_begin;
  const size_t off = size_t(win.row_begin - win.win_base), H = size_t(d.H);
  const bf16* hp = static_cast<const bf16*>(h) + off * H;
  const size_t zrow = z_row_bytes(d);                    // H * 2, or H * 2 + 8 K when the pairs follow the row
  char* zp = static_cast<char*>(Z) + off * zrow;
  float2* sc = d.zmerged ? reinterpret_cast<float2*>(zp + H * 2)
                         : reinterpret_cast<float2*>(scores) + off * d.K;
  const int sc_stride = d.zmerged ? int(zrow / 8) : d.K;
  const int head = d.H / d.K, slices = (d.H + NS - 1) / NS;
  // a head that crosses a slice's end has its half-scores taken from Z afterwards
  const bool whole_heads = slices == 1 || NS % head == 0;
  CUtensorMap mh, mw;
  if (!make_map(&mh, hp, uint64_t(rows), H, BM) || !make_map(&mw, lw.Wt, H, H, NS)) return -1;
  const int tiles = int((rows + BM - 1) / BM);
  const int groups = kNumSMs / slices, grid = (tiles < groups ? tiles : groups) * slices;
  launch(k_xform_umma<NS, KP, kRounded, HD>, grid, kThreads, C::SMEM_BYTES, st,
      mh, mw, zp, int(zrow), lw.a_src, lw.a_dst, whole_heads ? sc : nullptr, sc_stride, int(rows), d.H, head, slices, status);
  return whole_heads ? 1 : 1 + launch_scores(d, Z, lw, scores, win, st);
}

}  // namespace

bool xform_umma_supported(const Dims& d) {
  return d.dtype == XRL_BF16 && d.H % 32 == 0 && d.H <= 512 && encode_fn() != nullptr;
}

// Returns the number of kernels launched, or -1 if the tensor maps could not be built.
int launch_xform_umma(const Dims& d, const void* h, const LayerWeights& lw, void* Z, float* scores,
                      Window win, int32_t* status, cudaStream_t st) {
  if (int64_t(win.row_end) - win.row_begin <= 0) return 0;
#define XFORM_CASE(H_, NS_, KP_) \
  case H_: return launch_h<NS_, KP_>(d, h, lw, Z, scores, win, status, st);
  // heads of 16, 32 or 64 columns in the usual widths (their half-scores leave in 32-byte pieces)
#define XFORM_HEADS(H_, HD_) \
  if (d.H == H_ && d.H / d.K == HD_) return launch_h<H_, H_, HD_>(d, h, lw, Z, scores, win, status, st);
  XFORM_HEADS(128, 16) XFORM_HEADS(128, 32) XFORM_HEADS(128, 64) XFORM_HEADS(256, 16) XFORM_HEADS(256, 32) XFORM_HEADS(256, 64)
#undef XFORM_HEADS
  switch (d.H) {
    XFORM_CASE(32, 32, 64) XFORM_CASE(64, 64, 64) XFORM_CASE(96, 96, 128) XFORM_CASE(128, 128, 128)
    XFORM_CASE(160, 160, 192) XFORM_CASE(192, 192, 192) XFORM_CASE(224, 224, 256) XFORM_CASE(256, 256, 256)
    XFORM_CASE(288, 128, 320) XFORM_CASE(320, 128, 320) XFORM_CASE(352, 128, 384) XFORM_CASE(384, 128, 384)
    XFORM_CASE(416, 128, 448) XFORM_CASE(448, 128, 448) XFORM_CASE(480, 128, 512) XFORM_CASE(512, 128, 512)
    default: return -1;
  }
#undef XFORM_CASE
}

}  // namespace xrl
