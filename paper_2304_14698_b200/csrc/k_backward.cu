// Reverse pass of the agent's forward path for the PPO objective of the paper's Section 3.3.4
// (Eq. 3 clipped objective, Eq. 4 value loss, Eq. 5 their sum with an entropy term): the loss over the
// environments of a mini-batch, then the gradient with respect to every weight, layer by layer backwards
// through the heads, Eq. 8, the k attention layers of Eq. 7 and Eq. 6.
//
// What is in this file: the forward pass of xrl_ppo_grad keeps every layer's input, Z rows and half-scores
// (nothing is recomputed here); the reverse of Eq. 7 runs row-wise kernels (a warp per destination row:
// k_aggregate_bwd_rows, k_scores_bwd_rows) with generic fallbacks (k_aggregate_bwd, k_scores_bwd) for head
// counts that do not divide 32; the two dense products of a layer, dW = h_in^T dz and dh_in = dz W^T, run on
// the tensor cores (k_bwd_umma.cu) for bf16 models of hidden 128, 256 or 512 and on CUDA-core tiles (k_atb_tile,
// k_gwt and the forward product's kernel) otherwise.  Gradients are fp32; sums over rows are collected
// with floating-point atomics, so the last bits of a gradient depend on the order in which the hardware
// serves them.  Activations saved by the forward pass are read in their storage type.  On the tensor-core
// path the half-score terms (ds a) are added into the bf16 copy of dz that the products read (`dzb`) only:
// the fp32 `dz` buffer is then left without them and must not be read afterwards.
// ReLU'(0) = 0, LeakyReLU'(0) = 0.2; the clipped objective has the slope of whichever term of its min is
// the smaller one.
#include <algorithm>

#include "xrl_agg_tma.cuh"
#include "xrl_heads.cuh"

namespace xrl {

namespace {

__device__ __forceinline__ float lrelu(float x) { return fmaxf(x, 0.2f * x); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}

// Z rows and half-score pairs of a layer, in either layout (pairs behind the rows, or in their own array).
template <typename T> struct ZView {
  const char* z; size_t row_bytes; const float2* pairs; int pair_stride;   // pairs[i * pair_stride + k]
  __device__ __forceinline__ const T* row(int32_t i) const { return reinterpret_cast<const T*>(z + size_t(i) * row_bytes); }
  __device__ __forceinline__ float2 pair(int32_t i, int k) const { return pairs[size_t(i) * pair_stride + k]; }
};

constexpr int kMaxPerLane = 16;          // hidden <= 512

// ---- Eq. 7, reverse: one warp per destination row ---------------------------------------------------
// in : dh_out [N x H] fp32 (gradient of the layer's output), h_out (its output, for the ReLU), Z / pairs
// out: dz [N x H] fp32 += alpha * dpre (scattered to the gathered rows, atomics), ds_src [N x K] += (atomics),
//      ds_dst [N x K] = (own row), db [H] += (atomics, one per CTA and column)
template <typename T>
__global__ void __launch_bounds__(256)
k_aggregate_bwd(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col, ZView<T> zv,
                const T* __restrict__ h_out, const float* __restrict__ dh_out, float* __restrict__ dz,
                float* __restrict__ ds_src, float* __restrict__ ds_dst, float* __restrict__ db, int N, int H,
                int K) {
  enter();
  extern __shared__ float sm_db[];                 // [H] per-CTA sums of dpre
  for (int c = threadIdx.x; c < H; c += blockDim.x) sm_db[c] = 0.f;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const int d = H / K, NF = H / 32;
  for (int32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < N; i += warps) {
    float dp[kMaxPerLane];
#pragma unroll
    for (int f = 0; f < kMaxPerLane; ++f) {
      dp[f] = 0.f;
      if (f < NF) {
        const int c = lane + 32 * f;
        dp[f] = to_float(h_out[size_t(i) * H + c]) > 0.f ? dh_out[size_t(i) * H + c] : 0.f;
        atomicAdd(&sm_db[c], dp[f]);
      }
    }
    const int32_t e0 = rowptr[i], deg = rowptr[i + 1] - e0;
    // softmax statistics per head (every lane keeps all K heads; K is small)
    for (int k0 = 0; k0 < K; ++k0) {
      const float sd = zv.pair(i, k0).y;
      float mx = -INFINITY;
      for (int t = lane; t <= deg; t += 32) {
        const int32_t j = t < deg ? col[e0 + t] : i;
        mx = fmaxf(mx, lrelu(zv.pair(j, k0).x + sd));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
      float sum = 0.f;
      for (int t = lane; t <= deg; t += 32) {
        const int32_t j = t < deg ? col[e0 + t] : i;
        sum += exp2f(lrelu(zv.pair(j, k0).x + sd) - mx);
      }
      sum = warp_sum(sum);
      const float inv = 1.f / sum;
      // dal_t = sum over the head's features of dpre * z_j; dot = sum_t alpha_t dal_t
      float dot = 0.f;
      for (int t = 0; t <= deg; ++t) {
        const int32_t j = t < deg ? col[e0 + t] : i;
        const T* zj = zv.row(j);
        float part = 0.f;
#pragma unroll
        for (int f = 0; f < kMaxPerLane; ++f)
          if (f < NF) {
            const int c = lane + 32 * f;
            if (c / d == k0) part += dp[f] * to_float(zj[c]);
          }
        const float dal = warp_sum(part);
        const float al = exp2f(lrelu(zv.pair(j, k0).x + sd) - mx) * inv;
        dot += al * dal;
      }
      float dsd = 0.f;
      for (int t = 0; t <= deg; ++t) {
        const int32_t j = t < deg ? col[e0 + t] : i;
        const T* zj = zv.row(j);
        float part = 0.f;
#pragma unroll
        for (int f = 0; f < kMaxPerLane; ++f)
          if (f < NF) {
            const int c = lane + 32 * f;
            if (c / d == k0) part += dp[f] * to_float(zj[c]);
          }
        const float dal = warp_sum(part);
        const float e = zv.pair(j, k0).x + sd;          // (times log2 e: the sign is what matters below)
        const float al = exp2f(lrelu(e) - mx) * inv;
        const float de = al * (dal - dot) * (e > 0.f ? 1.f : 0.2f);
        dsd += de;
        if (lane == 0) atomicAdd(&ds_src[size_t(j) * K + k0], de);
#pragma unroll
        for (int f = 0; f < kMaxPerLane; ++f)
          if (f < NF) {
            const int c = lane + 32 * f;
            if (c / d == k0) atomicAdd(&dz[size_t(j) * H + c], al * dp[f]);
          }
      }
      if (lane == 0) ds_dst[size_t(i) * K + k0] = dsd;
    }
  }
  __syncthreads();
  for (int c = threadIdx.x; c < H; c += blockDim.x)
    if (sm_db[c] != 0.f) atomicAdd(&db[c], sm_db[c]);
}

// ---- half-scores, reverse: dz += ds_src a_src + ds_dst a_dst; da_src += ds_src z; da_dst += ds_dst z -----
template <typename T>
__global__ void __launch_bounds__(256)
k_scores_bwd(ZView<T> zv, const float* __restrict__ ds_src, const float* __restrict__ ds_dst,
             const float* __restrict__ a_src, const float* __restrict__ a_dst, float* __restrict__ dz,
             float* __restrict__ da_src, float* __restrict__ da_dst, int N, int H, int K) {
  enter();
  extern __shared__ float sm_da[];                 // [2H]
  for (int c = threadIdx.x; c < 2 * H; c += blockDim.x) sm_da[c] = 0.f;
  __syncthreads();
  const int d = H / K;
  const int rows_per_cta = (N + gridDim.x - 1) / gridDim.x;
  const int r0 = blockIdx.x * rows_per_cta, r1 = min(N, r0 + rows_per_cta);
  for (int c = threadIdx.x; c < H; c += blockDim.x) {
    const int k = c / d;
    const float as = a_src[c], ad = a_dst[c];
    float accs = 0.f, accd = 0.f;
    for (int i = r0; i < r1; ++i) {
      const float gs = ds_src[size_t(i) * K + k], gd = ds_dst[size_t(i) * K + k];
      const float z = to_float(zv.row(i)[c]);
      dz[size_t(i) * H + c] += gs * as + gd * ad;
      accs += gs * z;
      accd += gd * z;
    }
    sm_da[c] = accs;
    sm_da[H + c] = accd;
  }
  __syncthreads();
  for (int c = threadIdx.x; c < H; c += blockDim.x) {
    atomicAdd(&da_src[c], sm_da[c]);
    atomicAdd(&da_dst[c], sm_da[H + c]);
  }
}

// ---- the same two kernels for the usual shapes: K divides 32 and H = 32 NF (every width) --------------------
// (hidden 192, K 4, fp32, 1.2 k rows: 7 + 4 us per layer where the generic pair took 82 + 80)
// A lane owns NF consecutive features, all of one head (32 / K lanes per head): a head's reductions stay inside
// its group of lanes, all heads proceed at once, rows move as 4- to 16-byte pieces, and the scattered sums
// go out as vector atomics.
// Both add the columns that a CTA's warps keep (db; da_src, da_dst) from a slot per warp, and the second kernel gives a warp two
// rows at least: additions into one shared row, and one global one per column and eight rows, took 56 us for 7 k rows of 512
// (now 11; the first kernel 32 -> 23).
constexpr int kBwdWarps = 8;
// (NF values side by side, on the boundary that every lane's have: the power of two in their size, 16 at most)
constexpr int chunk_align(int bytes) { return bytes % 16 == 0 ? 16 : bytes % 8 == 0 ? 8 : bytes % 4 == 0 ? 4 : 2; }
// Rows whose units are all off, lanes whose are, and half-scores without a gradient add nothing and are passed over at the
// widths of a power of two.  The other widths, which the generic pair served first, take them as that pair does: 0 times an
// infinite feature is no number, and the gradient shows it.
template <int NF> constexpr bool kPassOver = (NF & (NF - 1)) == 0;
template <typename T, int NF> struct alignas(chunk_align(int(sizeof(T)) * NF)) Chunk { T v[NF]; };

template <typename T, int NF>
__device__ __forceinline__ void load_chunk(const T* p, float (&f)[NF]) {
  const Chunk<T, NF> c = *reinterpret_cast<const Chunk<T, NF>*>(p);
#pragma unroll
  for (int t = 0; t < NF; ++t) f[t] = to_float(c.v[t]);
}
template <int NF>
__device__ __forceinline__ void store_chunk(float* p, const float (&f)[NF]) {
  Chunk<float, NF> c;
#pragma unroll
  for (int t = 0; t < NF; ++t) c.v[t] = f[t];
  *reinterpret_cast<Chunk<float, NF>*>(p) = c;
}
template <int NF>
__device__ __forceinline__ void atomic_add_chunk(float* p, const float (&v)[NF]) {
  if constexpr (NF % 4 == 0) {
#pragma unroll
    for (int q = 0; q < NF / 4; ++q)
      atomicAdd(reinterpret_cast<float4*>(p) + q, make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]));
  } else if constexpr (NF % 2 == 0) {
#pragma unroll
    for (int q = 0; q < NF / 2; ++q) atomicAdd(reinterpret_cast<float2*>(p) + q, make_float2(v[2 * q], v[2 * q + 1]));
  } else {
#pragma unroll
    for (int q = 0; q < NF; ++q) atomicAdd(p + q, v[q]);
  }
}

// GATHER: nothing is scattered; every entry's (alpha, de) goes to its place in the transposed lists `tl` and the masked
// gradient dpre replaces dh_out (unless it arrives masked), for k_dz_gather to collect.
template <typename T, int NF, bool GATHER>
__global__ void __launch_bounds__(256)
k_aggregate_bwd_rows(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col, ZView<T> zv,
                     const T* __restrict__ h_out, float* __restrict__ dh_out, bool masked, float* __restrict__ dz,
                     float* __restrict__ ds_src, float* __restrict__ ds_dst, float* __restrict__ db, int N, int K,
                     BwdLists tl) {
  enter();
  constexpr int H = 32 * NF;
  __shared__ __align__(16) float sm_db[kBwdWarps][H];             // each warp's sums
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const int lph = 32 / K, k = lane / lph;            // lanes per head, this lane's head
  const bool leader = (lane % lph) == 0;
  float dbr[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) dbr[f] = 0.f;
  for (int32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < N; i += warps) {
    float dp[NF];
    {
      float g[NF], ho[NF];
      load_chunk<float, NF>(dh_out + size_t(i) * H + lane * NF, g);
      load_chunk<T, NF>(h_out + size_t(i) * H + lane * NF, ho);
#pragma unroll
      for (int f = 0; f < NF; ++f) { dp[f] = ho[f] > 0.f ? g[f] : 0.f; dbr[f] += dp[f]; }
      if (GATHER && !masked) store_chunk<NF>(dh_out + size_t(i) * H + lane * NF, dp);
    }
    bool live = false;
#pragma unroll
    for (int f = 0; f < NF; ++f) live = live || dp[f] != 0.f;
    if (!GATHER && kPassOver<NF> && !__any_sync(0xFFFFFFFFu, live)) continue;   // (ds is zeroed)
    const int32_t e0 = rowptr[i], deg = rowptr[i + 1] - e0;
    const int32_t self_entry = GATHER ? tl.rowptr[i] + i : 0;
    const float sd = zv.pair(i, k).y;
    // One sweep over the row's neighbours and the row itself (entry `deg`) takes, per head, the score e_t, the
    // product dal_t = dpre . z_t, and with a running maximum the sums  sum_t 2^(e_t - mx)  and
    // sum_t 2^(e_t - mx) dal_t; the first kCache entries keep (e_t, dal_t) in registers for the second sweep,
    // which turns them into d e_t and the scattered sums (later entries are read and multiplied again).
    constexpr int kCache = 4;
    float ce[kCache], cd[kCache];
    float mx = -INFINITY, sum = 0.f, dotu = 0.f;
    auto product = [&](const Chunk<T, NF>& zc, float& dal) {
      float part = 0.f;
#pragma unroll
      for (int f = 0; f < NF; ++f) part = fmaf(dp[f], to_float(zc.v[f]), part);
      for (int o = lph >> 1; o > 0; o >>= 1) part += __shfl_xor_sync(0xFFFFFFFFu, part, o);
      dal = part;
    };
    auto score_and_product = [&](int32_t j, float& eraw, float& dal) {
      const Chunk<T, NF> zc = *reinterpret_cast<const Chunk<T, NF>*>(zv.row(j) + lane * NF);
      eraw = zv.pair(j, k).x + sd;
      product(zc, dal);
    };
    auto accumulate = [&](float eraw, float dal) {
      const float e = lrelu(eraw);
      if (e > mx) {
        const float sc = exp2f(mx - e);
        sum = fmaf(sum, sc, kPassOver<NF> ? 1.f : 1.f + (e - e)); dotu = fmaf(dotu, sc, dal); mx = e;
      } else {
        const float w = exp2f(e - mx);
        sum += w; dotu = fmaf(w, dal, dotu);
      }
    };
    const int32_t c0 = lane < deg ? col[e0 + lane] : i;      // the first 32 entries (the row itself after the last)
    {
      // the first kCache rows are fetched together (entries past the last one repeat it: always a valid row)
      Chunk<T, NF> zc[kCache];
#pragma unroll
      for (int t = 0; t < kCache; ++t) {
        const int32_t j = __shfl_sync(0xFFFFFFFFu, c0, min(t, deg));
        zc[t] = *reinterpret_cast<const Chunk<T, NF>*>(zv.row(j) + lane * NF);
        ce[t] = zv.pair(j, k).x;
      }
#pragma unroll
      for (int t = 0; t < kCache; ++t) {
        ce[t] += sd;
        cd[t] = 0.f;
        if (t <= deg) {
          product(zc[t], cd[t]);
          accumulate(ce[t], cd[t]);
        }
      }
    }
    for (int base = 0; base <= deg; base += 32) {
      const int idx = base + lane;
      const int32_t cj = base == 0 ? c0 : (idx < deg ? col[e0 + idx] : i);
      const int cnt = min(32, deg + 1 - base);
      for (int t = (base == 0 ? kCache : 0); t < cnt; ++t) {
        const int32_t j = __shfl_sync(0xFFFFFFFFu, cj, t);
        float eraw, dal;
        score_and_product(j, eraw, dal);
        accumulate(eraw, dal);
      }
    }
    const float inv = 1.f / sum;
    const float dot = dotu * inv;
    float dsd = 0.f;
    auto scatter = [&](int32_t j, int t, float eraw, float dal) {
      const float al = exp2f(lrelu(eraw) - mx) * inv;
      const float de = al * (dal - dot) * (eraw > 0.f ? 1.f : 0.2f);
      dsd += de;
      if (GATHER) {
        const int32_t at = t < deg ? tl.inv[e0 + t] : self_entry;
        if (leader) tl.entry[size_t(at) * K + k] = make_float2(al, de);
        return;
      }
      if (leader && de != 0.f) atomicAdd(&ds_src[size_t(j) * K + k], de);
      if (live || (!kPassOver<NF> && al != al)) {
        float v[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) v[f] = al * dp[f];
        atomic_add_chunk<NF>(dz + size_t(j) * H + lane * NF, v);
      }
    };
#pragma unroll
    for (int t = 0; t < kCache; ++t)
      if (t <= deg) scatter(__shfl_sync(0xFFFFFFFFu, c0, t), t, ce[t], cd[t]);
    for (int base = 0; base <= deg; base += 32) {
      const int idx = base + lane;
      const int32_t cj = base == 0 ? c0 : (idx < deg ? col[e0 + idx] : i);
      const int cnt = min(32, deg + 1 - base);
      for (int t = (base == 0 ? kCache : 0); t < cnt; ++t) {
        const int32_t j = __shfl_sync(0xFFFFFFFFu, cj, t);
        float eraw, dal;
        score_and_product(j, eraw, dal);
        scatter(j, base + t, eraw, dal);
      }
    }
    if (leader) ds_dst[size_t(i) * K + k] = dsd;
  }
  store_chunk<NF>(&sm_db[threadIdx.x >> 5][lane * NF], dbr);
  __syncthreads();
  for (int c = threadIdx.x; c < H; c += blockDim.x) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kBwdWarps; ++w) v += sm_db[w][c];
    if (v != 0.f) atomicAdd(&db[c], v);
  }
}

// dz += ds_src a_src + ds_dst a_dst per row and head, da_src / da_dst += ds z.  With `dzb` (tensor-core
// products follow) the completed row goes to dzb in bf16 and the fp32 dz is NOT updated.
template <typename T, int NF>
__global__ void __launch_bounds__(256)
k_scores_bwd_rows(ZView<T> zv, const float* __restrict__ ds_src, const float* __restrict__ ds_dst,
                  const float* __restrict__ a_src, const float* __restrict__ a_dst, float* __restrict__ dz,
                  bf16* __restrict__ dzb, float* __restrict__ da_src, float* __restrict__ da_dst, int N, int K) {
  enter();
  constexpr int H = 32 * NF;
  __shared__ __align__(16) float sm_da[kBwdWarps][2 * H];         // each warp's sums
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const int k = lane / (32 / K);
  float as[NF], ad[NF], accs[NF], accd[NF];
  load_chunk<float, NF>(a_src + lane * NF, as);
  load_chunk<float, NF>(a_dst + lane * NF, ad);
#pragma unroll
  for (int f = 0; f < NF; ++f) { accs[f] = 0.f; accd[f] = 0.f; }
  for (int32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < N; i += warps) {
    const float gs = ds_src[size_t(i) * K + k], gd = ds_dst[size_t(i) * K + k];
    float z[NF], g[NF];
    load_chunk<float, NF>(dz + size_t(i) * H + lane * NF, g);
    if (!kPassOver<NF> || gs != 0.f || gd != 0.f) {
      load_chunk<T, NF>(zv.row(i) + lane * NF, z);
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        g[f] += gs * as[f] + gd * ad[f];
        accs[f] = fmaf(gs, z[f], accs[f]);
        accd[f] = fmaf(gd, z[f], accd[f]);
      }
      if (dzb == nullptr) store_chunk<NF>(dz + size_t(i) * H + lane * NF, g);
    }
    if (dzb != nullptr) {                             // the tensor-core products read dz in bf16
      Chunk<bf16, NF> c;
#pragma unroll
      for (int f = 0; f < NF; ++f) c.v[f] = __float2bfloat16(g[f]);
      *reinterpret_cast<Chunk<bf16, NF>*>(dzb + size_t(i) * H + lane * NF) = c;
    }
  }
  store_chunk<NF>(&sm_da[threadIdx.x >> 5][lane * NF], accs);
  store_chunk<NF>(&sm_da[threadIdx.x >> 5][H + lane * NF], accd);
  __syncthreads();
  for (int c = threadIdx.x; c < 2 * H; c += blockDim.x) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kBwdWarps; ++w) v += sm_da[w][c];
    if (v != 0.f) atomicAdd(c < H ? &da_src[c] : &da_dst[c - H], v);
  }
}

// ---- the heads' weight gradients: C += A^T B for every dense layer of the heads and Eq. 8, in one launch ---------
// A [rows x Ka], B [rows x Nb], fp32, any shapes; colsum (optional) += the column sums of B (the bias gradient).  64 x 64
// output tile per CTA, the rows cut into chunks, partial products added with atomics.  These products are small (hundreds of
// rows): what they cost is the chain of row steps of one CTA, so chunks are short, and seven launches became one (432 graphs,
// hidden 256: 0.178 -> 0.009 ms; 1,024 graphs 0.361 -> 0.019 ms).
struct GradTask { const float *A, *B; float *C, *colsum; int lda, ldb, ldc, rows, Ka, Nb, tiles_a, tiles_b, chunk, first; };
constexpr int kMaxTasks = 8;
struct GradTasks { GradTask t[kMaxTasks]; int n; };
__global__ void __launch_bounds__(256)
k_head_grads(const __grid_constant__ GradTasks tasks) {
  enter();
  __shared__ float As[16][64 + 1];
  __shared__ float Bs[16][64 + 1];
  int which = 0;
  while (which + 1 < tasks.n && int(blockIdx.x) >= tasks.t[which + 1].first) ++which;
  const GradTask& k = tasks.t[which];
  const int local = int(blockIdx.x) - k.first, ta = local % k.tiles_a, tb = (local / k.tiles_a) % k.tiles_b;
  const int z = local / (k.tiles_a * k.tiles_b);
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int a0 = ta * 64, b0 = tb * 64, Ka = k.Ka, Nb = k.Nb;
  const int r_begin = z * k.chunk, r_end = min(k.rows, r_begin + k.chunk);
  float acc[4][4] = {};
  const bool sums = k.colsum != nullptr && ta == 0 && ty == 0;     // the first row of CTAs also sums B's columns
  float csum[4] = {0.f, 0.f, 0.f, 0.f};
  float ra[4], rb[4];                                              // the next sixteen rows travel during the products
  auto fetch = [&](int r0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int t = tid + 256 * q, r = r0 + (t >> 6), c = t & 63;
      ra[q] = r < r_end && a0 + c < Ka ? __ldg(k.A + size_t(r) * k.lda + a0 + c) : 0.f;
      rb[q] = r < r_end && b0 + c < Nb ? __ldg(k.B + size_t(r) * k.ldb + b0 + c) : 0.f;
    }
  };
  if (r_begin < r_end) fetch(r_begin);
  for (int r0 = r_begin; r0 < r_end; r0 += 16) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int t = tid + 256 * q;
      As[t >> 6][t & 63] = ra[q];
      Bs[t >> 6][t & 63] = rb[q];
    }
    __syncthreads();
    if (r0 + 16 < r_end) fetch(r0 + 16);
#pragma unroll
    for (int rr = 0; rr < 16; ++rr) {
      float a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) { a[u] = As[rr][ty * 4 + u]; b[u] = Bs[rr][tx * 4 + u]; }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(a[u], b[v], acc[u][v]);
      if (sums) {
#pragma unroll
        for (int v = 0; v < 4; ++v) csum[v] += b[v];
      }
    }
    __syncthreads();
  }
  if (sums) {
#pragma unroll
    for (int v = 0; v < 4; ++v)
      if (b0 + tx * 4 + v < Nb && csum[v] != 0.f) atomicAdd(&k.colsum[b0 + tx * 4 + v], csum[v]);
  }
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int ka = a0 + ty * 4 + u, nb = b0 + tx * 4 + v;
      if (ka < Ka && nb < Nb && acc[u][v] != 0.f) atomicAdd(&k.C[size_t(ka) * k.ldc + nb], acc[u][v]);
    }
}

// ---- the same product for the layers' weights: dW [H x H] += A^T B, A = h_in [rows x H], B = dz [rows x H] fp32 --------
// TILE x TILE outputs per CTA, 8 x 8 per thread (two 4-wide groups in each direction: conflict-free 16-byte reads of
// shared memory), 16 rows per step with the next step's pieces already in registers.  The product reduces over the
// rows, so all parallelism beyond the H x H / TILE^2 tiles comes from cutting the rows into chunks (grid.z) whose
// results meet in vector atomics; 64-row tiles of 4 x 4 outputs per thread with chunks of 2,048 rows left half the SMs
// without work at 36 k rows (0.333 ms per layer at H = 128; now 0.031, with dh = dz W^T 0.065 -> 0.029).  Bound by FFMA issue.  fp32 FMA chains as before, shorter ones per chunk.
constexpr int kAtbRows = 16;
template <typename TA, int TILE>
__global__ void __launch_bounds__((TILE / 8) * (TILE / 8))
k_atb_tile(const TA* __restrict__ A, const float* __restrict__ Bm, float* __restrict__ Cout, int rows, int H,
           int rows_per_chunk, bool vec) {
  enter();
  constexpr int NTX = TILE / 8, NT = NTX * NTX;
  constexpr int PIECES = kAtbRows * TILE / 4 / NT;     // 4-wide pieces per thread, operand and step
  __shared__ __align__(16) float As[kAtbRows][TILE];
  __shared__ __align__(16) float Bs[kAtbRows][TILE];
  const int tid = threadIdx.x, ty = tid / NTX, tx = tid % NTX;
  const int a0 = blockIdx.x * TILE, b0 = blockIdx.y * TILE;
  const int r_begin = blockIdx.z * rows_per_chunk, r_end = min(rows, r_begin + rows_per_chunk);
  float acc[8][8];
#pragma unroll
  for (int u = 0; u < 8; ++u)
#pragma unroll
    for (int v = 0; v < 8; ++v) acc[u][v] = 0.f;
  Chunk<TA, 4> ra[PIECES];
  float4 rb[PIECES];
  auto fetch = [&](int r0) {
#pragma unroll
    for (int it = 0; it < PIECES; ++it) {
      const int idx = tid + it * NT, rr = r0 + idx / (TILE / 4), c = (idx % (TILE / 4)) * 4;
#pragma unroll
      for (int t = 0; t < 4; ++t) ra[it].v[t] = TA(0.f);
      rb[it] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (rr < r_end) {
        if (a0 + c < H) ra[it] = *reinterpret_cast<const Chunk<TA, 4>*>(A + size_t(rr) * H + a0 + c);
        if (b0 + c < H) rb[it] = *reinterpret_cast<const float4*>(Bm + size_t(rr) * H + b0 + c);
      }
    }
  };
  if (r_begin < r_end) fetch(r_begin);
  for (int r0 = r_begin; r0 < r_end; r0 += kAtbRows) {
#pragma unroll
    for (int it = 0; it < PIECES; ++it) {
      const int idx = tid + it * NT, rr = idx / (TILE / 4), c = (idx % (TILE / 4)) * 4;
      *reinterpret_cast<float4*>(&As[rr][c]) =
          make_float4(to_float(ra[it].v[0]), to_float(ra[it].v[1]), to_float(ra[it].v[2]), to_float(ra[it].v[3]));
      *reinterpret_cast<float4*>(&Bs[rr][c]) = rb[it];
    }
    __syncthreads();
    if (r0 + kAtbRows < r_end) fetch(r0 + kAtbRows);
#pragma unroll
    for (int rr = 0; rr < kAtbRows; ++rr) {
      float a[8], b[8];
      *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(&As[rr][ty * 4]);
      *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(&As[rr][TILE / 2 + ty * 4]);
      *reinterpret_cast<float4*>(b) = *reinterpret_cast<const float4*>(&Bs[rr][tx * 4]);
      *reinterpret_cast<float4*>(b + 4) = *reinterpret_cast<const float4*>(&Bs[rr][TILE / 2 + tx * 4]);
#pragma unroll
      for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int v = 0; v < 8; ++v) acc[u][v] = fmaf(a[u], b[v], acc[u][v]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 8; ++u)
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const int m = a0 + (u < 4 ? ty * 4 + u : TILE / 2 + ty * 4 + u - 4), n = b0 + g * (TILE / 2) + tx * 4;
      if (m >= H || n >= H) continue;
      float* o = Cout + size_t(m) * H + n;
      if (vec) {
        atomicAdd(reinterpret_cast<float4*>(o), make_float4(acc[u][4 * g], acc[u][4 * g + 1], acc[u][4 * g + 2], acc[u][4 * g + 3]));
      } else {                                         // (the caller's gradient buffer may sit on any 4-byte boundary)
#pragma unroll
        for (int t = 0; t < 4; ++t) atomicAdd(o + t, acc[u][4 * g + t]);
      }
    }
}

// ---- out = G W^T: G [rows x Hn] fp32, W [Hk x Hn] (storage type, row-major [in x out]) -> out [rows x Hk] ----
// (k_xform_simt's order of loads: 5.4 k rows of 512, 149 -> 96 us)
template <typename TW>
__global__ void __launch_bounds__(256)
k_gwt(const float* __restrict__ G, const TW* __restrict__ W, float* __restrict__ out, int rows, int Hk, int Hn) {
  enter();
  __shared__ __align__(16) float Gs[16][64 + 4];
  __shared__ __align__(16) float Ws[16][64 + 4];
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int r0 = blockIdx.x * 64, k0 = blockIdx.y * 64;
  float acc[4][4] = {};
  // four columns of one row of each operand per thread and step (the widths are multiples of 32), the next step's in flight
  // during the arithmetic
  const int rr = tid >> 2, cc0 = (tid & 3) * 4;
  const bool g_ok = r0 + rr < rows, w_ok = k0 + rr < Hk;
  const float* gp = G + size_t(g_ok ? r0 + rr : 0) * Hn + cc0;
  const TW* wp = W + size_t(w_ok ? k0 + rr : 0) * Hn + cc0;
  float g[4] = {}, w[4] = {};
  if (g_ok) load_chunk<float, 4>(gp, g);
  if (w_ok) load_chunk<TW, 4>(wp, w);
  for (int c0 = 0; c0 < Hn; c0 += 16) {
#pragma unroll
    for (int t = 0; t < 4; ++t) { Gs[cc0 + t][rr] = g[t]; Ws[cc0 + t][rr] = w[t]; }
    __syncthreads();
    if (c0 + 16 < Hn) {
      if (g_ok) load_chunk<float, 4>(gp + c0 + 16, g);
      if (w_ok) load_chunk<TW, 4>(wp + c0 + 16, w);
    }
#pragma unroll
    for (int cc = 0; cc < 16; ++cc) {
      const float4 a4 = *reinterpret_cast<const float4*>(&Gs[cc][ty * 4]), b4 = *reinterpret_cast<const float4*>(&Ws[cc][tx * 4]);
      const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(a[u], b[v], acc[u][v]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int r = r0 + ty * 4 + u, k = k0 + tx * 4 + v;
      if (r < rows && k < Hk) out[size_t(r) * Hk + k] = acc[u][v];
    }
}

// the sixteen dense entries of Eq. 6's input, one thread per node: [sum of the edge attributes | own shape]
template <typename T>
__global__ void __launch_bounds__(256)
k_embed_inputs(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col, const T* __restrict__ shape,
               const T* __restrict__ eattr, float* __restrict__ xs, int N) {
  enter();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  float x[2 * kS];
#pragma unroll
  for (int s = 0; s < kS; ++s) x[s] = 0.f;
  for (int32_t e = rowptr[i]; e < rowptr[i + 1]; ++e) {
    float v[kS];
    load_chunk<T, kS>(eattr ? eattr + size_t(e) * kS : shape + size_t(col[e]) * kS, v);
#pragma unroll
    for (int s = 0; s < kS; ++s) x[s] += v[s];
  }
  load_chunk<T, kS>(shape + size_t(i) * kS, reinterpret_cast<float(&)[kS]>(x[kS]));
  store_chunk<2 * kS>(xs + size_t(i) * 2 * kS, x);
}

// ---- Eq. 6, reverse: dW0 += x^T dpre, db0 += dpre, x_i = [edge sum | one-hot op | own shape] -------------
// A warp owns 64 columns (two per lane) and walks its share of the rows eight at a time: the next eight rows' gradients
// (256 bytes each), operators and dense inputs (k_embed_inputs; one coalesced 512-byte load) are asked for before the
// current eight are used, so no barrier and no staging of the gradients stands between memory and the multiplies.  The
// sixteen dense products accumulate in registers, the one-hot block in the warp's own shared-memory copy [T x 64] of
// that part of dW0 (a plain add per row and column: nobody else touches the copy; shared-memory float atomics cost far
// more than the adds).  Bound by issue: 16 packed FMA and as many others per row and 64 columns.  Staging 64-row tiles of all
// columns for 512 threads between two barriers took 0.94 ms at 990 k rows and hidden 256, this takes 0.45 (1.0 GB: 0.16 ms).
constexpr int kEmbBwdRows = 8;                     // rows in flight per warp
struct EmbBwdStage { float x[kEmbBwdRows][2 * kS]; int32_t op[kEmbBwdRows]; };
template <typename T>
__global__ void __launch_bounds__(128)
k_embed_bwd(const float* __restrict__ xs, const int32_t* __restrict__ op, const T* __restrict__ h0,
            const float* __restrict__ dh0, bool masked, float* __restrict__ dW0, float* __restrict__ db0, int N, int H, int Tn) {
  enter();
  extern __shared__ __align__(16) float sm_embed[];
  const int warps = blockDim.x >> 5, wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
  EmbBwdStage& stg = reinterpret_cast<EmbBwdStage*>(sm_embed)[wib];
  float* oh = sm_embed + warps * (sizeof(EmbBwdStage) / sizeof(float)) + size_t(wib) * Tn * 64;   // [Tn x 64]
  for (int t = lane; t < Tn * 64; t += 32) oh[t] = 0.f;
  const int c = blockIdx.y * 64 + 2 * lane;        // H is a multiple of 32: the last group may hold 32 columns only
  const bool on = c < H;
  // packed fp32 (two products per instruction): acc[c][t] = inputs 2t, 2t + 1 of column c
  aggtma::F2 acc[2][kS];
#pragma unroll
  for (int t = 0; t < kS; ++t) acc[0][t] = acc[1][t] = aggtma::make_f2(0.f, 0.f);
  const int64_t step = int64_t(gridDim.x) * warps * kEmbBwdRows;
  float2 g[kEmbBwdRows], gn[kEmbBwdRows];
  float4 xn;
  int32_t on_op = 0;
  auto fetch = [&](int64_t r0) {
    const float* p = dh0 + size_t(r0) * H + c;
    const T* q = h0 + size_t(r0) * H + c;
    const bool whole = on && r0 + kEmbBwdRows <= N;
#pragma unroll
    for (int u = 0; u < kEmbBwdRows; ++u) {
      const bool live = whole || (on && r0 + u < N);
      gn[u] = make_float2(0.f, 0.f);
      if (live) gn[u] = __ldg(reinterpret_cast<const float2*>(p + u * H));
      if (!masked && live) {
        float ho[2];
        load_chunk<T, 2>(q + u * H, ho);
        if (!(ho[0] > 0.f)) gn[u].x = 0.f;
        if (!(ho[1] > 0.f)) gn[u].y = 0.f;
      }
    }
    // lane t: piece t of the eight rows' inputs (four 16-byte pieces per row)
    xn = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r0 + (lane >> 2) < N) xn = __ldg(reinterpret_cast<const float4*>(xs + size_t(r0) * 2 * kS) + lane);
    if (lane < kEmbBwdRows) on_op = r0 + lane < N ? min(max(__ldg(op + r0 + lane), 0), Tn - 1) * 64 : 0;   // (pack reports bad ids)
  };
  int64_t r0 = (int64_t(blockIdx.x) * warps + wib) * kEmbBwdRows;
  if (r0 < N) fetch(r0);
  for (; r0 < N; r0 += step) {
    __syncwarp();                                  // the previous eight rows' inputs have been read
    reinterpret_cast<float4*>(&stg.x[0][0])[lane] = xn;
    if (lane < kEmbBwdRows) stg.op[lane] = on_op;
#pragma unroll
    for (int u = 0; u < kEmbBwdRows; ++u) g[u] = gn[u];
    __syncwarp();
    if (r0 + step < N) fetch(r0 + step);
    // two rows at a time: everything they read from shared memory is asked for before their sums are stored (the
    // compiler keeps reads behind stores that may alias them); rows past the end hold zeros
#pragma unroll
    for (int u = 0; u < kEmbBwdRows; u += 2) {
      ulonglong2 x[2][4];                          // pairs of inputs as they lie
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        x[0][v] = reinterpret_cast<const ulonglong2*>(stg.x[u])[v];
        x[1][v] = reinterpret_cast<const ulonglong2*>(stg.x[u + 1])[v];
      }
      const int2 o = *reinterpret_cast<const int2*>(&stg.op[u]);
      float2* p0 = reinterpret_cast<float2*>(oh + o.x) + lane;
      float2* p1 = reinterpret_cast<float2*>(oh + o.y) + lane;
      float2 v0 = *p0, v1 = *p1;
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        const aggtma::F2 ga = aggtma::make_f2(g[u + w].x, g[u + w].x), gb = aggtma::make_f2(g[u + w].y, g[u + w].y);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const aggtma::F2 xa{x[w][v].x}, xb{x[w][v].y};
          aggtma::fma2(acc[0][2 * v], xa, ga); aggtma::fma2(acc[0][2 * v + 1], xb, ga);
          aggtma::fma2(acc[1][2 * v], xa, gb); aggtma::fma2(acc[1][2 * v + 1], xb, gb);
        }
      }
      v0.x += g[u].x; v0.y += g[u].y;
      if (o.x == o.y) v1 = v0;
      v1.x += g[u + 1].x; v1.y += g[u + 1].y;
      *p0 = v0;
      *p1 = v1;
    }
  }
  // the CTA's warps share the columns: their registers meet in shared memory, one input at a time, and go to global memory
  // once per CTA
  __syncthreads();
  const float* oh0 = sm_embed + warps * (sizeof(EmbBwdStage) / sizeof(float));
  float* red = sm_embed + warps * (sizeof(EmbBwdStage) / sizeof(float)) + size_t(warps) * Tn * 64;  // [warps][64]
  const int cc = blockIdx.y * 64 + int(threadIdx.x & 63);
#pragma unroll
  for (int s = 0; s < 2 * kS; ++s) {
    float lo, hi, v[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      aggtma::split_f2(acc[e][s >> 1], lo, hi);
      v[e] = s & 1 ? hi : lo;
    }
    reinterpret_cast<float2*>(red + wib * 64)[lane] = make_float2(v[0], v[1]);
    __syncthreads();
    for (int k = threadIdx.x; k < 64; k += blockDim.x) {
      float t = 0.f;
      for (int w = 0; w < warps; ++w) t += red[w * 64 + k];
      const int col = blockIdx.y * 64 + k;
      if (col < H && t != 0.f) atomicAdd(dW0 + size_t(s < kS ? s : kS + Tn + (s - kS)) * H + col, t);
    }
    __syncthreads();
  }
  // the one-hot block; every row has one operator, so the block's columns sum to the bias gradient
  float bias = 0.f;
  for (int t = threadIdx.x; t < Tn * 64; t += blockDim.x) {       // (a thread keeps one column: blockDim is 64 or 128)
    float v = 0.f;
    for (int w = 0; w < warps; ++w) v += oh0[size_t(w) * Tn * 64 + t];
    const int col = blockIdx.y * 64 + (t & 63);
    if (col < H && v != 0.f) atomicAdd(&dW0[size_t(kS + (t >> 6)) * H + col], v);
    bias += v;
  }
  if (cc < H && bias != 0.f) atomicAdd(&db0[cc], bias);
}

// ---- the heads --------------------------------------------------------------------------------------------------
// The forward part is the forward path's own kernels (readout, k_global_update, k_policy_value_hidden) with the per-graph sums
// and hidden activations kept; what follows turns d(out) into the gradients of the hidden pre-activations (d1, d2) and of
// the inputs.  The weights' gradients are products of those per-row buffers (X^T D1, Y1^T D2, ...), taken afterwards by
// k_head_grads (which also sums the columns of D for the biases).
using heads::Mlp;

// y1, y2 -> d1, d2 of one row of a head whose output's gradient is dout (all in shared memory; y2, d2 for hid2 > 0 only)
__device__ __forceinline__ void mlp_hidden_bwd(const Mlp& m, const float* y1, const float* y2, float dout, float* d1, float* d2) {
  if (m.hid2 <= 0) {
    for (int c = threadIdx.x; c < m.hid; c += blockDim.x) d1[c] = y1[c] > 0.f ? m.w2[c] * dout : 0.f;
    __syncthreads();
  } else {
    for (int c = threadIdx.x; c < m.hid2; c += blockDim.x) d2[c] = y2[c] > 0.f ? m.w2[c] * dout : 0.f;
    __syncthreads();
    heads::rows_dot<1>(m.Wh, m.hid, m.hid2, d2, 0, [&](int, int k, float v) { d1[k] = y1[k] > 0.f ? v : 0.f; });
  }
}

// ---- per environment: Eq. 3-5, d J / d logit of its graphs, value head forward and reverse -----------------
// loss[4] += {J, L_clip, L_vf, L_ent} (atomics); dlogit [B]; demb [B x H] = the value head's share (plain
// stores: a graph belongs to one environment); the value head's per-row buffers vu [2H], vy1, vy2, vd1, vd2,
// vdout; logp_out [num_envs].  Two CTAs per environment, side by side: blockIdx.y 0 the policy's part, 1 the value head's
// (one after the other: 19 us instead of 16 at 6 environments of hidden 128, 32 instead of 29.5 at hidden 256).
struct EnvBufs { float *vu, *vy1, *vy2, *vd1, *vd2, *vdout; };

__global__ void __launch_bounds__(1024)
k_ppo_env(const float* __restrict__ logit, const int32_t* __restrict__ env_off,
          const uint8_t* __restrict__ mask, const int32_t* __restrict__ action, const float* __restrict__ logp_old,
          const float* __restrict__ adv, const float* __restrict__ ret, float eps, float c1, float c2, Mlp vm,
          EnvBufs eb, int H, int A, int num_envs, float* __restrict__ loss, float* __restrict__ dlogit,
          float* __restrict__ demb, float* __restrict__ logp_out, int32_t* status) {
  enter();
  extern __shared__ __align__(16) float sm[];
  const int e = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
  float* scratch = sm;                              // [4 blockDim]
  float* du = scratch + 4 * nt;                     // [2H]
  float* y1 = du + 2 * H;                           // [hid], padded
  float* y2 = y1 + heads::row_stride(vm.hid);       // [hid2], padded
  float* d1 = y2 + heads::row_stride(vm.hid2);      // [hid], padded
  float* d2 = d1 + heads::row_stride(vm.hid);       // [hid2]
  const int32_t cur = env_off[e];
  const int32_t C = env_off[e + 1] - cur - 1;
  const uint8_t* mk = mask + size_t(e) * A;
  const float inv_ne = 1.f / float(num_envs);
  auto valid = [&](int a) { return a == A || (a < C && mk[a]); };
  auto lg = [&](int a) { return logit[a == A ? cur : cur + 1 + a]; };
  const int act = action[e];
  if (act < 0 || act > A || !valid(act)) {          // the same for every thread of both CTAs
    if (tid == 0 && blockIdx.y == 0) raise(status, XRL_ERR_INVALID_ARG);
    return;
  }
  if (blockIdx.y == 0) {
    // masked softmax statistics
    float mx = -INFINITY;
    for (int a = tid; a <= A; a += nt)
      if (valid(a)) mx = fmaxf(mx, lg(a));
    mx = heads::block_max(mx, scratch);
    float se = 0.f;
    for (int a = tid; a <= A; a += nt)
      if (valid(a)) se += expf(lg(a) - mx);
    const float sum = heads::block_sum(se, scratch);
    const float lsum = logf(sum);
    float pl = 0.f;                                   // sum_a p_a log p_a
    for (int a = tid; a <= A; a += nt)
      if (valid(a)) { const float lp = lg(a) - mx - lsum; pl += expf(lp) * lp; }
    const float plogp = heads::block_sum(pl, scratch);
    const float logp = lg(act) - mx - lsum;
    const float ratio = expf(logp - logp_old[e]);
    const float clipped = fminf(fmaxf(ratio, 1.f - eps), 1.f + eps);
    const float t1 = ratio * adv[e], t2 = clipped * adv[e];
    const float dlogp = (t1 <= t2) ? -adv[e] * ratio * inv_ne : 0.f;
    for (int a = tid; a <= A; a += nt) {
      if (a < A && a >= C) continue;                  // no graph behind a padded slot
      const int32_t g = a == A ? cur : cur + 1 + a;
      float dl = 0.f;
      if (valid(a)) {
        const float lp = lg(a) - mx - lsum, p = expf(lp);
        dl = dlogp * ((a == act ? 1.f : 0.f) - p) + c2 * inv_ne * p * (lp - plogp);
      }
      dlogit[g] = dl;
    }
    if (tid == 0) {
      const float lc = -(t1 <= t2 ? t1 : t2) * inv_ne, le = plogp * inv_ne;
      atomicAdd(&loss[1], lc); atomicAdd(&loss[3], le);
      atomicAdd(&loss[0], lc + c2 * le);
      if (logp_out) logp_out[e] = logp;
    }
    return;
  }
  // value head over [ current graph | mean of the valid candidates ]: its input and first layer come from the launch that
  // scores the policy, whose CTAs share the layer (one CTA here read all of its weights)
  float cnt = 0.f;
  for (int a = tid; a < min(C, A); a += nt) cnt += mk[a] ? 1.f : 0.f;
  for (int c = tid; c < vm.hid; c += nt) y1[c] = eb.vy1[size_t(e) * vm.hid + c];
  const float nv = heads::block_sum(cnt, scratch);
  float contrib = 0.f;
  if (vm.hid2 <= 0) {
    for (int c = tid; c < vm.hid; c += nt) contrib += y1[c] * vm.w2[c];
  } else {
    heads::dense_rows<1>(y1, 0, vm.hid, vm.Wh, vm.hid2, vm.hid2, vm.bh, scratch, [&](int, int c, float y) {
      y2[c] = fmaxf(y, 0.f);
      contrib += fmaxf(y, 0.f) * vm.w2[c];
    });
  }
  const float v = heads::block_sum(contrib, scratch) + vm.b2[0];
  const float dv = c1 * 2.f * (v - ret[e]) * inv_ne;
  mlp_hidden_bwd(vm, y1, y2, dv, d1, d2);
  heads::rows_dot<1>(vm.W1, 2 * H, vm.hid, d1, 0, [&](int, int k, float x) { du[k] = x; });
  for (int c = tid; c < vm.hid; c += nt) eb.vd1[size_t(e) * vm.hid + c] = d1[c];
  for (int c = tid; c < vm.hid2; c += nt) {
    eb.vy2[size_t(e) * vm.hid2 + c] = y2[c];
    eb.vd2[size_t(e) * vm.hid2 + c] = d2[c];
  }
  // the value head's share of every graph's gradient (the current graph's, then the candidates'), four columns per thread
  const int HV = H >> 2;
  for (int i = tid; i < (C + 1) * HV; i += nt) {
    const int a = i / HV - 1, c = (i - (a + 1) * HV) * 4;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a < 0) s = *reinterpret_cast<const float4*>(du + c);
    else if (mk[a] && nv > 0.f) s = make_float4(du[H + c] / nv, du[H + c + 1] / nv, du[H + c + 2] / nv, du[H + c + 3] / nv);
    *reinterpret_cast<float4*>(demb + size_t(cur + 1 + a) * H + c) = s;
  }
  if (tid == 0) {
    eb.vdout[e] = dv;
    const float lv = (v - ret[e]) * (v - ret[e]) * inv_ne;
    atomicAdd(&loss[2], lv);
    atomicAdd(&loss[0], c1 * lv);
  }
}

// ---- per graph, reverse: policy head, then Eq. 8; GP graphs per CTA, so that every weight is loaded once for all of them ---
// in : demb (the value head's share), dlogit, emb, py1, py2   out: pd1, pd2, dpre [B x H] (gradient of Eq. 8's
// pre-activation), dr [B x H] (gradient of the graph's readout sum)
template <int GP>
__global__ void __launch_bounds__(1024)
k_graph_bwd(const float* __restrict__ emb, const float* __restrict__ dlogit, Mlp pm,
            const float* __restrict__ py1, const float* __restrict__ py2, const float* __restrict__ demb,
            const float* __restrict__ Wg, float* __restrict__ pd1, float* __restrict__ pd2,
            float* __restrict__ dpre, float* __restrict__ dr, int H, int B) {
  enter();
  extern __shared__ float sm[];
  const int tid = threadIdx.x, nt = blockDim.x;
  float* d1 = sm;                                   // [GP][hid]
  float* d2 = d1 + GP * pm.hid;                     // [GP][hid2]
  float* dx = d2 + GP * pm.hid2;                    // [GP][H]
  const int first = blockIdx.x * GP, rows = min(GP, B - first);
  const int hl = pm.hid2 > 0 ? pm.hid2 : pm.hid;    // the last hidden layer
  const float* yl = pm.hid2 > 0 ? py2 : py1;
  float* dl = pm.hid2 > 0 ? d2 : d1;
  float* pdl = pm.hid2 > 0 ? pd2 : pd1;
  for (int i = tid; i < GP * hl; i += nt) {
    const int g = i / hl, c = i - g * hl;
    float v = 0.f;
    if (g < rows) {
      v = yl[size_t(first + g) * hl + c] > 0.f ? pm.w2[c] * dlogit[first + g] : 0.f;
      pdl[size_t(first + g) * hl + c] = v;
    }
    dl[i] = v;
  }
  __syncthreads();
  if (pm.hid2 > 0)
    heads::rows_dot<GP>(pm.Wh, pm.hid, pm.hid2, d2, pm.hid2, [&](int g, int k, float v) {
      float d = 0.f;
      if (g < rows) {
        d = py1[size_t(first + g) * pm.hid + k] > 0.f ? v : 0.f;
        pd1[size_t(first + g) * pm.hid + k] = d;
      }
      d1[g * pm.hid + k] = d;
    });
  heads::rows_dot<GP>(pm.W1, H, pm.hid, d1, pm.hid, [&](int g, int k, float v) { dx[g * H + k] = v; });
  for (int i = tid; i < GP * H; i += nt) {
    const int g = i / H;
    float d = 0.f;
    if (g < rows) {
      const size_t at = size_t(first) * H + i;
      d = emb[at] > 0.f ? demb[at] + dx[i] : 0.f;
      dpre[at] = d;
    }
    dx[i] = d;
  }
  __syncthreads();
  heads::rows_dot<GP>(Wg, H, H, dx, H, [&](int g, int k, float v) {
    if (g < rows) dr[size_t(first + g) * H + k] = v;
  });
}

// the readout is a plain sum: every node receives its graph's gradient, masked by the ReLU of its features (four columns
// per thread; H % 4 == 0)
template <typename T>
__global__ void k_readout_bwd(const float* __restrict__ dr, const int32_t* __restrict__ seg_id, const T* __restrict__ h,
                              float* __restrict__ dh, int64_t n_quads, int H) {
  enter();
  const int q = H >> 2;
  for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < n_quads; t += int64_t(gridDim.x) * blockDim.x) {
    const int64_t i = t / q;
    const int c = int(t - i * q);
    const float4 g = reinterpret_cast<const float4*>(dr + size_t(seg_id[i]) * H)[c];
    float ho[4];
    load_chunk<T, 4>(h + 4 * t, ho);
    reinterpret_cast<float4*>(dh)[t] = make_float4(ho[0] > 0.f ? g.x : 0.f, ho[1] > 0.f ? g.y : 0.f, ho[2] > 0.f ? g.z : 0.f,
                                                   ho[3] > 0.f ? g.w : 0.f);
  }
}

// the tasks of k_head_grads
struct TaskList {
  GradTasks tasks{};
  int ctas = 0;
  void add(const float* A, int lda, const float* B, int ldb, float* C, int ldc, int rows, int Ka, int Nb, float* colsum) {
    if (rows <= 0 || Ka <= 0 || Nb <= 0) return;
    GradTask& t = tasks.t[tasks.n++];
    t = GradTask{A, B, C, colsum, lda, ldb, ldc, rows, Ka, Nb, (Ka + 63) / 64, (Nb + 63) / 64, chunk_rows(rows), ctas};
    ctas += t.tiles_a * t.tiles_b * ((rows + t.chunk - 1) / t.chunk);
  }
  // one head's layers from its per-row buffers
  void add_mlp(const float* X, int in, int rows, int hid, int hid2, const float* Y1, const float* Y2, const float* D1,
               const float* D2, const float* dout, float* gW1, float* gb1, float* gWh, float* gbh, float* gw2, float* gb2) {
    add(X, in, D1, hid, gW1, hid, rows, in, hid, gb1);
    if (hid2 > 0) add(Y1, hid, D2, hid2, gWh, hid2, rows, hid, hid2, gbh);
    add(hid2 > 0 ? Y2 : Y1, hid2 > 0 ? hid2 : hid, dout, 1, gw2, 1, rows, hid2 > 0 ? hid2 : hid, 1, gb2);
  }
  // 64 rows per chunk, more where that would make more than 64 chunks
  static int chunk_rows(int64_t rows) { return int(std::max<int64_t>(64, ((rows + 63) / 64 + 15) & ~int64_t(15))); }
};

template <int GP>
int graph_bwd(const Dims& d, const float* emb, const float* dlogit, const Mlp& pm, const float* py1, const float* py2,
              const float* demb, const float* Wg, float* pd1, float* pd2, float* dpre, float* dr, int32_t B, cudaStream_t st) {
  static bool attr[64] = {};
  const size_t smem = sizeof(float) * size_t(GP) * (d.H + d.Hm + d.Hm2);
  if (smem > 48 * 1024 && !ensure_dynamic_smem(k_graph_bwd<GP>, 227 * 1024, attr)) return -1;
  launch(k_graph_bwd<GP>, (B + GP - 1) / GP, 1024, smem, st, emb, dlogit, pm, py1, py2, demb, Wg, pd1, pd2, dpre, dr, d.H, B);
  return 1;
}

// Generalised advantage estimates: one thread per trajectory, backwards over its T steps (a first-order
// recurrence; trajectories are laid out step-major, [T x M], so that the threads of a warp read neighbours)
__global__ void k_gae(const float* __restrict__ reward, const float* __restrict__ values,
                      const uint8_t* __restrict__ done, float gamma, float lambda, int T, int M,
                      float* __restrict__ adv, float* __restrict__ ret) {
  enter();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= M) return;
  float run = 0.f, vnext = values[size_t(T) * M + j];
  for (int t = T - 1; t >= 0; --t) {
    const float nd = done[size_t(t) * M + j] ? 0.f : 1.f;
    const float v = values[size_t(t) * M + j];
    const float delta = reward[size_t(t) * M + j] + gamma * vnext * nd - v;
    run = delta + gamma * lambda * nd * run;
    adv[size_t(t) * M + j] = run;
    ret[size_t(t) * M + j] = run + v;
    vnext = v;
  }
}

}  // namespace

// ---- launchers ------------------------------------------------------------------------------------------
// ---- weights of a rank's means in the data-parallel exchange --------------------------------------------
// buf = [grad * n | loss[0..3] * n | n] before the caller's sum all-reduce; grad, loss = buf / buf[last] after it.
namespace {
template <typename F>
__global__ void k_grad_weigh(const F* __restrict__ grad, int64_t count, const F* __restrict__ loss, F n,
                             F* __restrict__ buf) {
  enter();
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < count) buf[i] = grad[i] * n;
  else if (i < count + 4) buf[i] = loss[i - count] * n;
  else if (i == count + 4) buf[i] = n;
}
template <typename F>
__global__ void k_grad_unweigh(const F* __restrict__ buf, int64_t count, F* __restrict__ grad, F* __restrict__ loss) {
  enter();
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const F total = buf[count + 4];
  if (i < count) grad[i] = buf[i] / total;
  else if (i < count + 4) loss[i - count] = buf[i] / total;
}
}  // namespace

int launch_grad_weigh(int elem_bytes, const void* grad, int64_t count, const void* loss, int64_t n, void* buf,
                      cudaStream_t st) {
  const unsigned blocks = unsigned((count + 5 + 255) / 256);
  if (elem_bytes == 8)
    launch(k_grad_weigh<double>, blocks, 256, 0, st, static_cast<const double*>(grad), count,
                                                 static_cast<const double*>(loss), double(n), static_cast<double*>(buf));
  else
    launch(k_grad_weigh<float>, blocks, 256, 0, st, static_cast<const float*>(grad), count,
                                                static_cast<const float*>(loss), float(n), static_cast<float*>(buf));
  return 1;
}
int launch_grad_unweigh(int elem_bytes, const void* buf, int64_t count, void* grad, void* loss, cudaStream_t st) {
  const unsigned blocks = unsigned((count + 4 + 255) / 256);
  if (elem_bytes == 8)
    launch(k_grad_unweigh<double>, blocks, 256, 0, st, static_cast<const double*>(buf), count, static_cast<double*>(grad),
                                                   static_cast<double*>(loss));
  else
    launch(k_grad_unweigh<float>, blocks, 256, 0, st, static_cast<const float*>(buf), count, static_cast<float*>(grad),
                                                  static_cast<float*>(loss));
  return 1;
}

int launch_gae(const float* reward, const float* values, const uint8_t* done, float gamma, float lambda, int32_t T,
               int32_t M, float* adv, float* ret, cudaStream_t st) {
  if (T <= 0 || M <= 0) return 0;
  launch(k_gae, unsigned((M + 127) / 128), 128, 0, st, reward, values, done, gamma, lambda, T, M, adv, ret);
  return 1;
}

// every piece of the heads' workspace starts on a 16-byte boundary (some are read as float4)
static size_t up4(size_t n) { return (n + 3) & ~size_t(3); }
size_t ppo_heads_workspace_floats(const Dims& d, int64_t B, int64_t num_envs) {
  const size_t H = d.H, Hm = d.Hm, Hm2 = d.Hm2, b = size_t(B), e = size_t(num_envs);
  return up4(b * (H + d.Dg)) + 4 * up4(b * H) + 2 * up4(b) + 2 * up4(b * Hm) + 2 * up4(b * Hm2) +
         up4(e * 2 * H) + 2 * up4(e * Hm) + 2 * up4(e * Hm2) + up4(e);
}

// The gradient of every row of the last layer's features, masked by their ReLU, from that of the graphs' sums.
static int launch_readout_bwd(const Dims& d, const float* dr, const int32_t* seg_id, const void* hL, float* dh, int64_t N,
                              cudaStream_t st) {
  const int64_t ne = N * (d.H / 4);
  if (ne <= 0) return 0;
  const unsigned grid = unsigned(std::min<int64_t>((ne + 255) / 256, int64_t(kNumSMs) * 64));
  if (d.dtype == XRL_BF16) launch(k_readout_bwd<bf16>, grid, 256, 0, st, dr, seg_id, static_cast<const bf16*>(hL), dh, ne, d.H);
  else launch(k_readout_bwd<float>, grid, 256, 0, st, dr, seg_id, static_cast<const float*>(hL), dh, ne, d.H);
  return 1;
}

// Forward from the readout's sums (of chunks: partial_off = the graphs' first chunks, nblocks = 0; or of the last layer's
// blocks of rows: partial_off = the graphs' first rows) to the logits, Eq. 3-5, and the reverse pass down to the gradient of the last
// layer's node features (dh [N x H]), or, without dh, to that of the graphs' sums (*dr_out [B x H], in ws).  ws:
// ppo_heads_workspace_floats floats.
int launch_ppo_heads(const Dims& d, const DevWeights& w, float* grad_base, const float* w_base, const void* hL,
                     const float* partial, const int32_t* partial_off, int32_t nblocks, int block_shift,
                     const int32_t* seg_id, const float* g0,
                     const int32_t* env_off,
                     const uint8_t* mask, const int32_t* action, const float* logp_old, const float* adv,
                     const float* ret, float eps, float c1, float c2, int32_t B, int32_t num_envs, int64_t N,
                     float* ws, float* loss, float* dh, const float** dr_out, float* logp_out, int32_t* status,
                     cudaStream_t st) {
  if (B <= 0 || num_envs <= 0) return 0;
  const size_t H = d.H, Hm = d.Hm, Hm2 = d.Hm2, HU = H + d.Dg;
  float* p = ws;
  auto take = [&](size_t n) { float* q = p; p += up4(n); return q; };
  // what a bad action leaves unwritten for its environment (the kernel stops there) comes first and is cleared
  float* demb = take(size_t(B) * H);
  float* dlogit = take(B);
  EnvBufs eb;
  eb.vu = take(size_t(num_envs) * 2 * H);
  eb.vy1 = take(size_t(num_envs) * Hm); eb.vd1 = take(size_t(num_envs) * Hm);
  eb.vy2 = take(size_t(num_envs) * Hm2); eb.vd2 = take(size_t(num_envs) * Hm2);
  eb.vdout = take(num_envs);
  float* const cleared_end = p;
  float* U = take(size_t(B) * HU);
  float* emb = take(size_t(B) * H);
  float* dpre = take(size_t(B) * H);
  float* dr = take(size_t(B) * H);
  float* logit = take(B);
  float* py1 = take(size_t(B) * Hm);
  float* pd1 = take(size_t(B) * Hm);
  float* py2 = take(size_t(B) * Hm2);
  float* pd2 = take(size_t(B) * Hm2);
  auto gp = [&](const float* q) { return grad_base + (q - w_base); };     // same place in the gradient blob
  const Mlp vm{w.vW1, w.vb1, w.vWh, w.vbh, w.vw2, w.vb2, d.Hm, d.Hm2};
  const Mlp pm{w.pW1, w.pb1, w.pWh, w.pbh, w.pw2, w.pb2, d.Hm, d.Hm2};
  int n = 0;
  cudaMemsetAsync(ws, 0, sizeof(float) * size_t(cleared_end - ws), st);
  int k = nblocks > 0 ? launch_global_update_blocks(d, partial, partial_off, nblocks, block_shift, g0, w, emb, B, st, U)
                      : launch_global_update(d, partial, partial_off, g0, w, emb, B, st, U);
  if (k < 0) return -1;
  n += k;
  k = launch_policy_value_hidden(d, w, emb, logit, B, py1, py2, env_off, mask, num_envs, eb.vy1, st, eb.vu);
  if (k < 0) return -1;
  n += k;
  const size_t env_smem = sizeof(float) * (4 * 1024 + 2 * H + 2 * heads::row_stride(d.Hm) + 2 * heads::row_stride(d.Hm2));
  launch(k_ppo_env, dim3(unsigned(num_envs), 2), 1024, env_smem, st, logit, env_off, mask, action, logp_old, adv, ret, eps, c1, c2, vm, eb, d.H,
                                              d.A, num_envs, loss, dlogit, demb, logp_out, status);
  ++n;
  // graphs per CTA: as few as leave every CTA an SM of its own, at most eight
  const int64_t per = (int64_t(B) + kNumSMs - 1) / kNumSMs;
#define GRAPH_BWD(G_) graph_bwd<G_>(d, emb, dlogit, pm, py1, py2, demb, w.Wg, pd1, pd2, dpre, dr, B, st)
  k = per <= 1 ? GRAPH_BWD(1) : per <= 2 ? GRAPH_BWD(2) : per <= 4 ? GRAPH_BWD(4) : GRAPH_BWD(8);
#undef GRAPH_BWD
  if (k < 0) return -1;
  n += k;
  TaskList tl;
  tl.add(U, int(HU), dpre, d.H, gp(w.Wg), d.H, B, int(HU), d.H, gp(w.bg));
  tl.add_mlp(emb, d.H, B, d.Hm, d.Hm2, py1, py2, pd1, pd2, dlogit, gp(w.pW1), gp(w.pb1), gp(w.pWh), gp(w.pbh), gp(w.pw2),
             gp(w.pb2));
  tl.add_mlp(eb.vu, 2 * d.H, num_envs, d.Hm, d.Hm2, eb.vy1, eb.vy2, eb.vd1, eb.vd2, eb.vdout, gp(w.vW1), gp(w.vb1), gp(w.vWh),
             gp(w.vbh), gp(w.vw2), gp(w.vb2));
  launch(k_head_grads, tl.ctas, 256, 0, st, tl.tasks);
  ++n;
  *dr_out = dr;
  if (dh != nullptr) n += launch_readout_bwd(d, dr, seg_id, hL, dh, N, st);
  return n;
}

static bool bwd_rows_kernels(const Dims& d) {
  return 32 % d.K == 0;
}
bool bwd_leaves_masked(const Dims& d) { return bwd_rows_kernels(d) && bwd_umma_supported(d); }

// One attention layer backwards: dh_out -> (dW, da_src, da_dst, db) and dh_in.  Z / scores hold the layer's
// forward transform of h_in; dz [N x H] and ds [2 N K] are scratch.  With dr (rows_gather_supported models with lists only)
// the gradient of a row's output is its graph's row of dr, and dh_out is scratch.
int launch_gat_layer_bwd(const Dims& d, const int32_t* rowptr, const int32_t* col, const void* Z, const float* scores,
                         const void* h_in, const void* h_out, float* dh_out, bool masked, const float* dr,
                         const int32_t* seg_id, float* dh_in, float* dz, float* ds, void* dz_store, const BwdLists* lists, const LayerWeights& lw, float* gW, float* ga_src,
                         float* ga_dst, float* gb, int32_t N, int32_t* status, cudaStream_t st) {
  if (N <= 0) return 0;
  const int H = d.H, K = d.K;
  const bool gather = lists != nullptr;      // dz by producer from the lists (every entry written, nothing to clear)
  if (!gather) {
    cudaMemsetAsync(dz, 0, sizeof(float) * size_t(N) * H, st);
    cudaMemsetAsync(ds, 0, sizeof(float) * size_t(N) * K * 2, st);
  }
  float* ds_src = ds;
  float* ds_dst = ds + size_t(N) * K;
  const size_t zrow = z_row_bytes(d);
  const int grid_rows = int(std::min<int64_t>((int64_t(N) + 7) / 8, int64_t(kNumSMs) * 8));
  const int grid_sums = int(std::min<int64_t>((int64_t(N) + 15) / 16, int64_t(kNumSMs) * 4));
  const int grid_cols = int(std::min<int64_t>((int64_t(N) + 255) / 256, int64_t(kNumSMs) * 2));
  // dW on CUDA cores: 128-wide tiles where they fit H (one CTA of 256 threads per SM: 160 registers; held to 128
  // registers and two CTAs the launch takes 35.6 us instead of 33.6 at 36 k rows), else 64-wide ones (six CTAs of 64
  // threads per SM); the rows in as many chunks as fill the SMs, at least 64 rows each
  const bool wide_atb = H % 128 == 0;
  const int atb_side = wide_atb ? H / 128 : (H + 63) / 64;
  const int atb_chunks = std::max(1, (wide_atb ? 1 : 6) * kNumSMs / (atb_side * atb_side));
  const int chunk = std::max(64, int(((int64_t(N) + atb_chunks - 1) / atb_chunks + 15) & ~int64_t(15)));
  dim3 g_atb(unsigned(atb_side), unsigned(atb_side), unsigned((N + chunk - 1) / chunk));
  const bool vec = (reinterpret_cast<uintptr_t>(gW) & 15) == 0;
  dim3 g_gwt(unsigned((N + 63) / 64), unsigned((H + 63) / 64));
  const int NF = H / 32;
  const bool rows_kernels = bwd_rows_kernels(d);
  // bf16 models of hidden 128, 256 or 512 take both products on the tensor cores, from a bf16 copy of dz
  const bool mma = rows_kernels && bwd_umma_supported(d) && dz_store != nullptr;
  bf16* dzb = mma ? static_cast<bf16*>(dz_store) : nullptr;
#define BWD_ROWS(TY_, NF_)                                                                                     \
  do {                                                                                                         \
    launch(k_aggregate_bwd_rows<TY_, NF_, false>, grid_rows, 256, 0, st,                                           \
        rowptr, col, zv, static_cast<const TY_*>(h_out), dh_out, masked, dz, ds_src, ds_dst, gb, N, K, BwdLists{});  \
    launch(k_scores_bwd_rows<TY_, NF_>, grid_sums, 256, 0, st, zv, ds_src, ds_dst, lw.a_src, lw.a_dst, dz, dzb,    \
                                                           ga_src, ga_dst, N, K);                              \
  } while (0)
#define BWD_GATHER(TY_, NF_)                                                                                   \
  do {                                                                                                         \
    const int k_ = launch_rows_gather(d, *lists, rowptr, col, Z, scores, h_out, dh_out, masked, dr, seg_id, ds_dst, gb, N, \
                                      status, st);                                                             \
    if (k_ < 0) {                            /* (it reads rows: the graphs' gradients are written out first) */   \
      if (dr != nullptr) launch_readout_bwd(d, dr, seg_id, h_out, dh_out, N, st);                              \
      launch(k_aggregate_bwd_rows<TY_, NF_, true>, grid_rows, 256, 0, st, rowptr, col, zv,                     \
             static_cast<const TY_*>(h_out), dh_out, masked || dr != nullptr, nullptr, nullptr, ds_dst, gb, N, K, *lists); \
    }                                                                                                          \
    if (launch_dz_gather(d, *lists, dh_out, Z, zrow, ds_dst, lw, mma ? dz_store : static_cast<void*>(dz), ga_src, ga_dst, \
                         N, status, st) < 0)                                                                   \
      return -1;                                                                                               \
  } while (0)
#define BWD_BODY(TY_)                                                                                          \
  do {                                                                                                         \
    ZView<TY_> zv;                                                                                             \
    zv.z = static_cast<const char*>(Z); zv.row_bytes = zrow;                                                   \
    zv.pairs = d.zmerged ? reinterpret_cast<const float2*>(static_cast<const char*>(Z) + size_t(H) * sizeof(TY_)) \
                         : reinterpret_cast<const float2*>(scores);                                          \
    zv.pair_stride = d.zmerged ? int(zrow / 8) : K;                                                            \
    if (gather) {                                                                                              \
      if (NF == 4) BWD_GATHER(TY_, 4); else BWD_GATHER(TY_, 8);                                                \
    } else if (rows_kernels) {                                                                                 \
      switch (NF) {                                                                                            \
        case 1: BWD_ROWS(TY_, 1); break;                                                                       \
        case 2: BWD_ROWS(TY_, 2); break;                                                                       \
        case 3: BWD_ROWS(TY_, 3); break;                                                                       \
        case 4: BWD_ROWS(TY_, 4); break;                                                                       \
        case 5: BWD_ROWS(TY_, 5); break;                                                                       \
        case 6: BWD_ROWS(TY_, 6); break;                                                                       \
        case 7: BWD_ROWS(TY_, 7); break;                                                                       \
        case 8: BWD_ROWS(TY_, 8); break;                                                                       \
        case 9: BWD_ROWS(TY_, 9); break;                                                                       \
        case 10: BWD_ROWS(TY_, 10); break;                                                                     \
        case 11: BWD_ROWS(TY_, 11); break;                                                                     \
        case 12: BWD_ROWS(TY_, 12); break;                                                                     \
        case 13: BWD_ROWS(TY_, 13); break;                                                                     \
        case 14: BWD_ROWS(TY_, 14); break;                                                                     \
        case 15: BWD_ROWS(TY_, 15); break;                                                                     \
        default: BWD_ROWS(TY_, 16); break;                                                                     \
      }                                                                                                        \
    } else {                                                                                                   \
      launch(k_aggregate_bwd<TY_>, grid_rows, 256, sizeof(float) * H, st,                                          \
          rowptr, col, zv, static_cast<const TY_*>(h_out), dh_out, dz, ds_src, ds_dst, gb, N, H, K);           \
      launch(k_scores_bwd<TY_>, grid_cols, 256, sizeof(float) * 2 * H, st, zv, ds_src, ds_dst, lw.a_src, lw.a_dst, \
                                                                       dz, ga_src, ga_dst, N, H, K);           \
    }                                                                                                          \
    if (mma) {                                                                                                 \
      if (launch_bwd_umma(d, h_in, dzb, lw.W, dh_in, gW, N, status, st) < 0) return -1;                        \
    } else {                                                                                                   \
      if (wide_atb)                                                                                            \
        launch(k_atb_tile<TY_, 128>, g_atb, 256, 0, st, static_cast<const TY_*>(h_in), dz, gW, N, H, chunk, vec);  \
      else                                                                                                     \
        launch(k_atb_tile<TY_, 64>, g_atb, 64, 0, st, static_cast<const TY_*>(h_in), dz, gW, N, H, chunk, vec);    \
      /* from 8,192 rows on the 128 x 128 tiles of the forward product have CTAs for every SM */               \
      if (N >= 8192 && H > 64)                                                                                 \
        launch_rows_times_matrix(d, dz, lw.Wt, dh_in, N, st);                                                  \
      else                                                                                                     \
        launch(k_gwt<TY_>, g_gwt, 256, 0, st, dz, static_cast<const TY_*>(lw.W), dh_in, N, H, H);                  \
    }                                                                                                          \
  } while (0)
  if (d.dtype == XRL_BF16) BWD_BODY(bf16); else BWD_BODY(float);
#undef BWD_ROWS
#undef BWD_GATHER
#undef BWD_BODY
  return 4;
}

// The model shapes xrl_ppo_grad takes: a copy of the one-hot block of W0's gradient ([T x H]) and eight rows of all columns
// within 227 KB.  A limit of the interface: the kernel below keeps 64 columns of that block per warp and would take any.
size_t embed_bwd_smem_bytes(const Dims& d) {
  return sizeof(float) * (size_t(d.T) * d.H + 8 * size_t(d.H) + 8 * 2 * kS) + sizeof(int32_t) * 8;
}

int launch_embed_bwd(const Dims& d, const int32_t* rowptr, const int32_t* col, const int32_t* op, const void* shape,
                     const void* eattr, const void* h0, const float* dh0, bool masked, float* xs, float* gW0, float* gb0,
                     int32_t N, cudaStream_t st) {
  if (N <= 0) return 0;
  // four warps per CTA, two where their copies would not fit (T <= 256: two always do); CTAs for every SM's shared memory (at most 16 warps' worth)
  const size_t per_warp = sizeof(EmbBwdStage) + sizeof(float) * (size_t(d.T) * 64 + 64), room = size_t(220) * 1024;
  const int warps = 4 * per_warp <= room ? 4 : 2;
  const size_t smem = warps * per_warp;
  const int groups = (d.H + 63) / 64;
  const int per_sm = int(std::max<size_t>(1, std::min<size_t>(16 / warps, room / (smem + 1024))));
  const int64_t want = (int64_t(N) + warps * kEmbBwdRows - 1) / (warps * kEmbBwdRows);
  const dim3 grid(unsigned(std::min<int64_t>(want, std::max(1, kNumSMs * per_sm / groups))), unsigned(groups));
  const unsigned grid_x = unsigned((int64_t(N) + 255) / 256);
  // the opt-in is the kernel's ceiling for every later launch: ask for all an SM has, once per device
  constexpr int kSmemCeiling = 227 * 1024;
  if (d.dtype == XRL_BF16) {
    static bool attr[64] = {};
    if (!ensure_dynamic_smem(k_embed_bwd<bf16>, kSmemCeiling, attr)) return -1;
    launch(k_embed_inputs<bf16>, grid_x, 256, 0, st, rowptr, col, static_cast<const bf16*>(shape),
                                                 static_cast<const bf16*>(eattr), xs, N);
    launch(k_embed_bwd<bf16>, grid, 32 * warps, smem, st, xs, op, static_cast<const bf16*>(h0), dh0, masked, gW0, gb0, N, d.H, d.T);
  } else {
    static bool attr[64] = {};
    if (!ensure_dynamic_smem(k_embed_bwd<float>, kSmemCeiling, attr)) return -1;
    launch(k_embed_inputs<float>, grid_x, 256, 0, st, rowptr, col, static_cast<const float*>(shape),
                                                  static_cast<const float*>(eattr), xs, N);
    launch(k_embed_bwd<float>, grid, 32 * warps, smem, st, xs, op, static_cast<const float*>(h0), dh0, masked, gW0, gb0, N, d.H, d.T);
  }
  return 2;
}

}  // namespace xrl
