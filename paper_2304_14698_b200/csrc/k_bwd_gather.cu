// An attention layer's reverse pass (paper Eq. 7), gathered by producer in place of scattered:
//   dz_j = sum over the rows i that read j (and j itself) of alpha_ij dpre_i  +  ds_src_j a_src + ds_dst_j a_dst
// with ds_src_j = sum of the score gradients de_ij of the same entries, and da_src += ds_src z, da_dst += ds_dst z.
//
// k_rows_gather (512-byte Z rows; k_aggregate_bwd_rows otherwise) takes the softmax's reverse row by row and leaves
// (alpha, de) of every entry in the order of the transposed lists built here: for producer j its own entry first, then its
// readers'; so the weights k_dz_gather needs are one contiguous run per list, fetched with a bulk copy, and the dpre rows
// come through the TMA unit's gather4 into a per-warp ring, as in the forward aggregate.
// Scattering alpha dpre into an fp32 dz with vector atomics instead cost a zeroed buffer, its read-modify-write
// through DRAM (1 KB per row each way at hidden 256) and a second kernel that read it all again for the ds terms.
// Both kernels are bound by HBM: per row H x 4 bytes of dpre and Z once, 8 K bytes per entry; the second also writes the
// result (2 H in bf16).  990 k rows, hidden 256: scatter 1.065 + half-score terms 0.463 + clearing 0.16 ms per layer ->
// 0.350 + 0.443 ms.
//
// Every wait is bounded; on expiry the warp records XRL_ERR_TIMEOUT and stops.
#include "xrl_agg_tma.cuh"

namespace xrl {

using namespace umma;
using namespace aggtma;

namespace {

constexpr int TW = 4;                // warps per CTA
constexpr int G = 2;                 // k_dz_gather: groups of four rows in flight per warp
constexpr int LIST = 96;             // list capacity per piece, a multiple of 8

// ---- transposed lists ------------------------------------------------------------------------------------------
// (the slots that rows own are rowptr[0] .. rowptr[N] - 1: a batch that was reported bad may have been given others, before
// them when its first graph has edges and no nodes, or behind)
__global__ void k_t_count(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col, int32_t N, int32_t E,
                          int32_t* __restrict__ cnt) {
  enter();
  const int32_t e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < E && e >= __ldg(rowptr) && e < __ldg(rowptr + N)) atomicAdd(&cnt[col[e]], 1);
}
// cnt holds the counts on entry and zeros on return; inv[e]: where the entry of slot e sits (every list is preceded by
// its producer's own entry, so entry number = list position + producer + 1)
__global__ void k_t_fill(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col, int32_t N,
                         const int32_t* __restrict__ rowptr_t, int32_t* __restrict__ cnt, int32_t* __restrict__ col_t,
                         int32_t* __restrict__ inv) {
  enter();
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  for (int32_t e = rowptr[i]; e < rowptr[i + 1]; ++e) {
    const int32_t j = col[e], q = rowptr_t[j] + atomicSub(&cnt[j], 1) - 1;
    col_t[q] = i;
    inv[e] = q + j + 1;
  }
}

// ---- one warp per block of producers ----------------------------------------------------------------------------
// A lane owns columns 4 lane .. 4 lane + 3 of each group of 128 (conflict-free 16-byte reads of a gathered row).
template <int NV> struct Layout {
  static constexpr int ROW = 512 * NV;                    // bytes of a dpre row
  __host__ __device__ static int group_bytes(int K) { return 4 * ROW + 4 * 8 * K; }
  __host__ __device__ static int slot_bytes(int K) { return (group_bytes(K) + 127) & ~127; }   // (TMA: 128-byte steps)
  // ring, then the barriers, row pointers and list
  __host__ __device__ static int warp_bytes(int K) {
    return (G * slot_bytes(K) + 8 * G + 4 * (BR + 1 + 3) + 4 * (LIST + 4) + 127) & ~127;
  }
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

__device__ __forceinline__ float4 load4f(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 load4f(const bf16* p) {
  const uint2 t = __ldg(reinterpret_cast<const uint2*>(p));
  return make_float4(__uint_as_float(t.x << 16), __uint_as_float(t.x & 0xFFFF0000u), __uint_as_float(t.y << 16),
                     __uint_as_float(t.y & 0xFFFF0000u));
}
__device__ __forceinline__ void store4f(float* p, const float4& v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void store4f(bf16* p, const float4& v) {
  *reinterpret_cast<uint2*>(p) = make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
}

template <typename T, int NV>
__global__ void __launch_bounds__(TW * 32, 5)
k_dz_gather(const __grid_constant__ CUtensorMap map_dp, const float* __restrict__ dpre, const float2* __restrict__ entry,
            const int32_t* __restrict__ rowptr_t, const int32_t* __restrict__ col_t, const char* __restrict__ Z,
            size_t z_row, const float* __restrict__ ds_dst, const float* __restrict__ a_src,
            const float* __restrict__ a_dst, T* __restrict__ dz, float* __restrict__ da_src, float* __restrict__ da_dst,
            int32_t N, int32_t K, int32_t br_shift, int32_t* status) {
  enter();
  constexpr int H = 128 * NV;
  using L = Layout<NV>;
  extern __shared__ __align__(128) uint8_t gsm[];
  float* sm_da = reinterpret_cast<float*>(gsm + size_t(TW) * L::warp_bytes(K));      // [2 H]
  float* sm_a = sm_da + 2 * H;                                                        // [2 H] a_src, a_dst
  for (int c = threadIdx.x; c < 2 * H; c += blockDim.x) {
    sm_da[c] = 0.f;
    sm_a[c] = c < H ? __ldg(a_src + c) : __ldg(a_dst + c - H);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint8_t* mine = gsm + size_t(wib) * L::warp_bytes(K);
  const uint32_t gbytes = L::group_bytes(K), sbytes = L::slot_bytes(K);
  const uint32_t ring = smem_u32(mine), bar_base = ring + G * sbytes;
  int32_t* rp = reinterpret_cast<int32_t*>(mine + G * sbytes + 8 * G);
  int32_t* item = rp + BR + 4;                             // (16-byte aligned: 8 G + 144 bytes behind the ring)
  const int br = 1 << br_shift;
  float4 accs[NV], accd[NV];
  int head[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    accs[v] = accd[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    head[v] = (v * 128 + lane * 4) / (H / K);
  }
  if (lane == 0) {
    for (int g = 0; g < G; ++g) mbar_init(bar_base + 8 * g, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  __syncwarp();
  uint32_t slot = 0, par = 0;
  bool alive = true;
  const int64_t step = int64_t((gridDim.x * blockDim.x) >> 5) << br_shift;
  for (int64_t r0 = int64_t((blockIdx.x * blockDim.x + threadIdx.x) >> 5) << br_shift; r0 < N && alive; r0 += step) {
    const int nr = int(min(int64_t(br), N - r0));
    __syncwarp();
    if (lane < nr) rp[lane] = __ldg(rowptr_t + r0 + lane);
    if (lane == 0) rp[nr] = __ldg(rowptr_t + r0 + nr);
    __syncwarp();
    // the row's Z and score gradients are asked for one row ahead
    float4 zn[NV];
    float gdn[NV];
    auto prefetch = [&](int row) {
      const size_t j = size_t(r0 + min(row, nr - 1));
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        zn[v] = load4f(reinterpret_cast<const T*>(Z + j * z_row) + v * 128 + lane * 4);
        gdn[v] = __ldg(ds_dst + j * K + head[v]);
      }
    };
    prefetch(0);
    // dz row, da sums; acc: sum alpha dpre, des: sum de per head
    auto finish = [&](int row, float4 (&acc)[NV], const float (&des)[NV]) {
      float4 z[NV];
      float gd[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) { z[v] = zn[v]; gd[v] = gdn[v]; }
      prefetch(row + 1);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const float4 as = *reinterpret_cast<const float4*>(sm_a + v * 128 + lane * 4);
        const float4 ad = *reinterpret_cast<const float4*>(sm_a + H + v * 128 + lane * 4);
        acc[v].x += des[v] * as.x + gd[v] * ad.x;
        acc[v].y += des[v] * as.y + gd[v] * ad.y;
        acc[v].z += des[v] * as.z + gd[v] * ad.z;
        acc[v].w += des[v] * as.w + gd[v] * ad.w;
        accs[v].x = fmaf(des[v], z[v].x, accs[v].x); accd[v].x = fmaf(gd[v], z[v].x, accd[v].x);
        accs[v].y = fmaf(des[v], z[v].y, accs[v].y); accd[v].y = fmaf(gd[v], z[v].y, accd[v].y);
        accs[v].z = fmaf(des[v], z[v].z, accs[v].z); accd[v].z = fmaf(gd[v], z[v].z, accd[v].z);
        accs[v].w = fmaf(des[v], z[v].w, accs[v].w); accd[v].w = fmaf(gd[v], z[v].w, accd[v].w);
        store4f(dz + size_t(r0 + row) * H + v * 128 + lane * 4, acc[v]);
      }
    };
    auto add = [&](float4& a, float w, const float4& x) {
      a.x = fmaf(w, x.x, a.x); a.y = fmaf(w, x.y, a.y); a.z = fmaf(w, x.z, a.z); a.w = fmaf(w, x.w, a.w);
    };
    int rs = 0;
    while (rs < nr && alive) {
      const int32_t eb = rp[rs];
      const bool fits = (rs + lane < nr) && (lane + 1 + rp[rs + lane + 1] - eb <= LIST);
      const uint32_t fmask = __ballot_sync(0xFFFFFFFFu, fits);
      const int cnt = (fmask == 0xFFFFFFFFu) ? 32 : __ffs(~fmask) - 1;
      const float2* ent = entry + size_t(int64_t(eb) + r0 + rs) * K;     // the list's entries, in its order
      if (cnt == 0) {                      // more readers than the list holds: plain loads
        const int n = rp[rs + 1] - eb;
        float4 acc[NV];
        float des[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) { acc[v] = make_float4(0.f, 0.f, 0.f, 0.f); des[v] = 0.f; }
        for (int t = 0; t <= n; ++t) {
          const int32_t i = t == 0 ? int32_t(r0) + rs : __ldg(col_t + eb + t - 1);
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            const float2 w = __ldg(ent + size_t(t) * K + head[v]);
            add(acc[v], w.x, load4f(dpre + size_t(i) * H + v * 128 + lane * 4));
            des[v] += w.y;
          }
        }
        finish(rs, acc, des);
        rs += 1;
        continue;
      }
      __syncwarp();
      const int total = cnt + (rp[rs + cnt] - eb);
      if (lane < cnt) {
        const int e0 = rp[rs + lane] - eb, n = rp[rs + lane + 1] - eb - e0;
        int pos = lane + e0;
        item[pos++] = int32_t(r0) + rs + lane;
        for (int t = 0; t < n; ++t) item[pos++] = __ldg(col_t + eb + e0 + t);
      }
      if (lane < 4) item[total + lane] = int32_t(r0) + rs;               // pad the last group
      __syncwarp();
      const int ngroups = (total + 3) / 4;
      // (the entry array is padded by four entries, so that the last group's copy stays inside it)
      auto issue = [&](int gi, uint32_t s) {
        const uint32_t bar = bar_base + 8 * s, at = ring + s * sbytes;
        mbar_expect_tx(bar, gbytes);
        const int4 it = *reinterpret_cast<const int4*>(&item[gi * 4]);
        tma_gather4(at, &map_dp, it.x, it.y, it.z, it.w, bar);
        bulk_load(at + 4 * L::ROW, ent + size_t(gi) * 4 * K, 32 * K, bar);
      };
      if (lane == 0) {
        uint32_t s = slot;
        for (int gi = 0; gi < min(G, ngroups); ++gi) { issue(gi, s); s = (s + 1 == G) ? 0 : s + 1; }
      }
      int gi = 0, w = 4;
      uint32_t dp = ring + slot * sbytes + lane * 16, wp = ring + slot * sbytes + 4 * L::ROW;
      if (!wait_all_lanes(bar_base + 8 * slot, par)) alive = false;
      for (int rr = 0; rr < cnt; ++rr) {
        const int n = rp[rs + rr + 1] - rp[rs + rr];
        float4 acc[NV];
        float des[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) { acc[v] = make_float4(0.f, 0.f, 0.f, 0.f); des[v] = 0.f; }
        for (int t = 0; t <= n; ++t) {
          uint4 raw[NV];
          float2 wt[NV];
#pragma unroll
          for (int v = 0; v < NV; ++v) { raw[v] = lds128(dp + v * 512); wt[v] = lds64(wp + head[v] * 8); }
          dp += L::ROW; wp += 8 * K;
          if (--w == 0) {                   // group finished: refill its slot, move on, wait for the next one
            __syncwarp();
            if (lane == 0 && gi + G < ngroups) issue(gi + G, slot);
            ++gi;
            if (++slot == G) { slot = 0; par ^= 1; }
            dp = ring + slot * sbytes + lane * 16;
            wp = ring + slot * sbytes + 4 * L::ROW;
            w = 4;
            if (gi < ngroups && alive && !wait_all_lanes(bar_base + 8 * slot, par)) alive = false;
          }
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            add(acc[v], wt[v].x, make_float4(__uint_as_float(raw[v].x), __uint_as_float(raw[v].y),
                                             __uint_as_float(raw[v].z), __uint_as_float(raw[v].w)));
            des[v] += wt[v].y;
          }
        }
        finish(rs + rr, acc, des);
      }
      if (w != 4) {                          // the list ended inside a group: retire it without waiting
        __syncwarp();
        if (++slot == G) { slot = 0; par ^= 1; }
      }
      rs += cnt;
    }
  }
  if (!alive) {
    if (lane == 0) raise(status, XRL_ERR_TIMEOUT);
    for (int t = 0; t < 100; ++t) __nanosleep(10000);     // give copies still in flight time to land
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    float* s = sm_da + v * 128 + lane * 4;
    atomicAdd(s, accs[v].x); atomicAdd(s + 1, accs[v].y); atomicAdd(s + 2, accs[v].z); atomicAdd(s + 3, accs[v].w);
    s += H;
    atomicAdd(s, accd[v].x); atomicAdd(s + 1, accd[v].y); atomicAdd(s + 2, accd[v].z); atomicAdd(s + 3, accd[v].w);
  }
  __syncthreads();
  for (int c = threadIdx.x; c < H; c += blockDim.x) {
    if (sm_da[c] != 0.f) atomicAdd(&da_src[c], sm_da[c]);
    if (sm_da[H + c] != 0.f) atomicAdd(&da_dst[c], sm_da[H + c]);
  }
}

// ---- one warp per block of destination rows: the softmax's reverse ----------------------------------------------
// For row i with entries t = itself, producers: e_t, dal_t = dpre_i . z_t per head, alpha = softmax(LeakyReLU(e)),
// de_t = alpha_t (dal_t - sum alpha dal) LeakyReLU'(e_t); (alpha_t, de_t) go to the entry's place in the transposed
// lists, sum de_t to ds_dst, dpre to the bias gradient.  The Z rows (and half-score pairs) come through the forward
// aggregate's ring of gather4 copies; the row's own gradient is asked for one row ahead.  With `masked` dh arrives as
// dpre; otherwise the ReLU of h_out is applied here and dpre replaces dh.  With `dr` (the last layer) the gradient of a row's
// output is its graph's row of dr - the readout is a plain sum - and dh is only written: a pass over all rows that wrote
// it for this one to read took 0.29 ms at 990 k rows of 256.
// A warp per row with plain loads waits three dependent round trips per row (990 k rows, hidden 256: 1.00 ms).
constexpr int RG = 2, RGQ = 2, RGV = 4 * RGQ;     // ring: two groups of eight rows
constexpr int kKeep = 4;                           // entries whose score and product stay in registers

template <int K, bool MERGED> struct alignas(128) RowSmem {
  static constexpr int ROW = MERGED ? 512 + 8 * K : 512;
  uint8_t z[RG][RGV][ROW];
  float2 sc[MERGED ? 1 : RG][RGV][K];
  unsigned long long bar[RG];
  int32_t rp[BR + 1];
  alignas(16) int32_t item[LIST + RGV];
  int32_t entry[LIST];
};

template <typename T, int K, bool MERGED>
__global__ void __launch_bounds__(TW * 32, 5)
k_rows_gather(const __grid_constant__ CUtensorMap map_z, const __grid_constant__ CUtensorMap map_s,
              const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col, const T* __restrict__ Z,
              const float2* __restrict__ scores, const T* __restrict__ h_out, float* __restrict__ dh, bool masked,
              const float* __restrict__ dr, const int32_t* __restrict__ seg_id, const BwdLists tl, float* __restrict__ ds_dst,
              float* __restrict__ db, int32_t N, int32_t br_shift, int32_t* status) {
  enter();
  using Smem = RowSmem<K, MERGED>;
  constexpr int VEC = VecOf<T>::N, NP = VEC / 2, H = 32 * VEC, LPH = 32 / K;
  constexpr uint32_t ZR = Smem::ROW, SR = MERGED ? ZR : 8 * K;
  constexpr uint32_t GROUP_BYTES = RGV * (512 + K * 8), ZG = RGV * ZR, SG = RGV * SR;
  constexpr int ZS = int(ZR / sizeof(T));
  extern __shared__ __align__(128) uint8_t gsm[];
  Smem& sm = reinterpret_cast<Smem*>(gsm)[threadIdx.x >> 5];
  float* sm_db = reinterpret_cast<float*>(gsm + sizeof(Smem) * TW);      // [H]
  for (int c = threadIdx.x; c < H; c += blockDim.x) sm_db[c] = 0.f;
  __syncthreads();
  const int lane = threadIdx.x & 31, c0 = lane * VEC, head = lane / LPH;
  const bool leader = (lane % LPH) == 0;
  const uint32_t z_base = smem_u32(&sm.z[0][0][0]), s_base = smem_u32(&sm.sc[0][0][0]);
  const uint32_t z_lane = z_base + lane * 16, s_lane = MERGED ? z_base + 512 + head * 8 : s_base + head * 8;
  const uint32_t bar_base = smem_u32(&sm.bar[0]);
  const int br = 1 << br_shift;
  F2 dbr[NP];
#pragma unroll
  for (int t = 0; t < NP; ++t) dbr[t] = make_f2(0.f, 0.f);
  if (lane == 0) {
    for (int g = 0; g < RG; ++g) mbar_init(bar_base + 8 * g, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  __syncwarp();
  uint32_t slot = 0, par = 0;
  bool alive = true;
  auto issue = [&](int gi, uint32_t s) {
    const uint32_t bar = bar_base + 8 * s;
    mbar_expect_tx(bar, GROUP_BYTES);
#pragma unroll
    for (int q = 0; q < RGQ; ++q) {
      const int4 it = *reinterpret_cast<const int4*>(&sm.item[gi * RGV + q * 4]);
      tma_gather4(z_base + s * ZG + q * 4 * ZR, &map_z, it.x, it.y, it.z, it.w, bar);
      if (!MERGED) tma_gather4(s_base + s * SG + q * 4 * SR, &map_s, it.x, it.y, it.z, it.w, bar);
    }
  };
  const int64_t step = int64_t((gridDim.x * blockDim.x) >> 5) << br_shift;
  for (int64_t r0 = int64_t((blockIdx.x * blockDim.x + threadIdx.x) >> 5) << br_shift; r0 < N && alive; r0 += step) {
    const int nr = int(min(int64_t(br), N - r0));
    uint4 gn[VEC / 4], hn = make_uint4(0u, 0u, 0u, 0u);        // the next row's gradient (and output, for its ReLU)
    const int32_t my_graph = dr != nullptr && lane < nr ? __ldg(seg_id + r0 + lane) : 0;
    auto prefetch = [&](int row) {
      const size_t at = size_t(r0 + row) * H + c0;
      const float* g = dr != nullptr ? dr + size_t(__shfl_sync(0xFFFFFFFFu, my_graph, row)) * H + c0 : dh + at;
#pragma unroll
      for (int t = 0; t < VEC / 4; ++t) gn[t] = *reinterpret_cast<const uint4*>(g + 4 * t);
      if (!masked) hn = __ldg(reinterpret_cast<const uint4*>(h_out + at));
    };
    // the row's dpre as register pairs; asks for the next row's
    auto take = [&](int row, F2 (&dp)[NP]) {
      float g[VEC];
#pragma unroll
      for (int t = 0; t < VEC / 4; ++t) {
        g[4 * t] = __uint_as_float(gn[t].x); g[4 * t + 1] = __uint_as_float(gn[t].y);
        g[4 * t + 2] = __uint_as_float(gn[t].z); g[4 * t + 3] = __uint_as_float(gn[t].w);
      }
      if (!masked) {
        float ho[VEC];
        unpack(hn, ho);
#pragma unroll
        for (int t = 0; t < VEC; ++t) g[t] = ho[t] > 0.f ? g[t] : 0.f;
        float4* o = reinterpret_cast<float4*>(dh + size_t(r0 + row) * H + c0);
#pragma unroll
        for (int t = 0; t < VEC / 4; ++t) o[t] = make_float4(g[4 * t], g[4 * t + 1], g[4 * t + 2], g[4 * t + 3]);
      }
      if (row + 1 < nr) prefetch(row + 1);
#pragma unroll
      for (int t = 0; t < NP; ++t) { dp[t] = make_f2(g[2 * t], g[2 * t + 1]); add2(dbr[t], dp[t]); }
    };
    // dpre . z over the lanes of a head
    auto product = [&](const F2 (&dp)[NP], const uint4& raw) {
      F2 z[NP], s = make_f2(0.f, 0.f);
      to_pairs(raw, z);
#pragma unroll
      for (int t = 0; t < NP; ++t) fma2(s, dp[t], z[t]);
      float lo, hi;
      split_f2(s, lo, hi);
      float v = lo + hi;
#pragma unroll
      for (int o = LPH >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
      return v;
    };
    // running sums of 2^(e - m) and 2^(e - m) dal; the reference m moves only when a score exceeds it by 32
    auto accumulate = [&](float e, float dal, float& m, float& l, float& dot) {
      const float ev = lrelu(e);
      if (ev > m + 32.f) {
        const float sc = fast_exp2(m - ev);
        l *= sc; dot *= sc; m = ev;
      }
      const float p = fast_exp2(ev - m);
      l += p;
      dot = fmaf(p, dal, dot);
    };
    auto finish = [&](float e, float dal, float m, float inv, float dot) {
      const float al = fast_exp2(lrelu(e) - m) * inv;
      return make_float2(al, al * (dal - dot) * (e > 0.f ? 1.f : 0.2f));
    };
    __syncwarp();
    if (lane < nr) sm.rp[lane] = __ldg(rowptr + r0 + lane);
    if (lane == 0) sm.rp[nr] = __ldg(rowptr + r0 + nr);
    const int32_t my_entry = lane < nr ? __ldg(tl.rowptr + r0 + lane) + int32_t(r0) + lane : 0;   // the row's own
    prefetch(0);
    __syncwarp();
    int rs = 0;
    while (rs < nr && alive) {
      const int32_t eb = sm.rp[rs];
      const bool fits = (rs + lane < nr) && (lane + 1 + sm.rp[rs + lane + 1] - eb <= LIST);
      const uint32_t fmask = __ballot_sync(0xFFFFFFFFu, fits);
      const int cnt = (fmask == 0xFFFFFFFFu) ? 32 : __ffs(~fmask) - 1;
      if (cnt == 0) {
        // more producers than the list holds: plain loads; (e, dal) wait in the entry between the two sweeps
        const int n = sm.rp[rs + 1] - eb;
        const int32_t own = __shfl_sync(0xFFFFFFFFu, my_entry, rs);
        F2 dp[NP];
        take(rs, dp);
        float m = 0.f, l = 0.f, dot = 0.f, sd = 0.f, dsd = 0.f;
        for (int t = 0; t <= n; ++t) {
          const int32_t j = t == 0 ? int32_t(r0) + rs : __ldg(col + eb + t - 1);
          const float2 pr = MERGED ? __ldg(reinterpret_cast<const float2*>(Z + size_t(j) * ZS + H) + head)
                                   : __ldg(scores + size_t(j) * K + head);
          const float dal = product(dp, __ldg(reinterpret_cast<const uint4*>(Z + size_t(j) * ZS + c0)));
          if (t == 0) { sd = pr.y; m = lrelu(pr.x + sd); }
          const float e = pr.x + sd;
          accumulate(e, dal, m, l, dot);
          if (leader) tl.entry[size_t(t == 0 ? own : __ldg(tl.inv + eb + t - 1)) * K + head] = make_float2(e, dal);
        }
        const float inv = 1.f / l;
        dot *= inv;
        if (leader) {
          for (int t = 0; t <= n; ++t) {
            float2* p = tl.entry + size_t(t == 0 ? own : __ldg(tl.inv + eb + t - 1)) * K + head;
            const float2 w = finish(p->x, p->y, m, inv, dot);
            *p = w;
            dsd += w.y;
          }
          ds_dst[size_t(r0 + rs) * K + head] = dsd;
        }
        rs += 1;
        continue;
      }
      __syncwarp();
      const int total = cnt + (sm.rp[rs + cnt] - eb);
      const int32_t own = __shfl_sync(0xFFFFFFFFu, my_entry, (rs + lane) & 31);
      if (lane < cnt) {
        const int e0 = sm.rp[rs + lane] - eb, n = sm.rp[rs + lane + 1] - eb - e0;
        int pos = lane + e0;
        sm.item[pos] = int32_t(r0) + rs + lane;
        sm.entry[pos++] = own;
        for (int t = 0; t < n; ++t) {
          sm.item[pos] = __ldg(col + eb + e0 + t);
          sm.entry[pos++] = __ldg(tl.inv + eb + e0 + t);
        }
      }
      if (lane < RGV) sm.item[total + lane] = int32_t(r0) + rs;          // pad the last group
      __syncwarp();
      const int ngroups = (total + RGV - 1) / RGV;
      if (lane == 0) {
        uint32_t s = slot;
        for (int gi = 0; gi < min(RG, ngroups); ++gi) { issue(gi, s); s = (s + 1 == RG) ? 0 : s + 1; }
      }
      int gi = 0, w = RGV, li = 0;           // group, vectors left in it, position in the list
      uint32_t zp = z_lane + slot * ZG, sp = s_lane + slot * SG;
      if (!wait_all_lanes(bar_base + 8 * slot, par)) alive = false;
      auto next = [&](uint4& raw, float2& sc) {
        raw = lds128(zp);
        sc = lds64(sp);
        zp += ZR; sp += SR;
        if (--w == 0) {
          __syncwarp();
          if (lane == 0 && gi + RG < ngroups) issue(gi + RG, slot);
          ++gi;
          if (++slot == RG) { slot = 0; par ^= 1; }
          zp = z_lane + slot * ZG;
          sp = s_lane + slot * SG;
          w = RGV;
          if (gi < ngroups && alive && !wait_all_lanes(bar_base + 8 * slot, par)) alive = false;
        }
      };
      for (int rr = 0; rr < cnt; ++rr) {
        const int n = sm.rp[rs + rr + 1] - sm.rp[rs + rr];
        F2 dp[NP];
        take(rs + rr, dp);
        uint4 raw;
        float2 sc;
        float ce[kKeep], cd[kKeep];
        next(raw, sc);
        const float sd = sc.y;
        ce[0] = sc.x + sd;
        cd[0] = product(dp, raw);
        float m = lrelu(ce[0]), l = 1.f, dot = cd[0], dsd = 0.f;
#pragma unroll
        for (int t = 1; t < kKeep; ++t) {
          ce[t] = 0.f; cd[t] = 0.f;
          if (t <= n) {
            next(raw, sc);
            ce[t] = sc.x + sd;
            cd[t] = product(dp, raw);
            accumulate(ce[t], cd[t], m, l, dot);
          }
        }
        for (int t = kKeep; t <= n; ++t) {    // the rest waits in its entries
          next(raw, sc);
          const float e = sc.x + sd, dal = product(dp, raw);
          accumulate(e, dal, m, l, dot);
          if (leader) tl.entry[size_t(sm.entry[li + t]) * K + head] = make_float2(e, dal);
        }
        const float inv = 1.f / l;
        dot *= inv;
        if (leader) {
#pragma unroll
          for (int t = 0; t < kKeep; ++t)
            if (t <= n) {
              const float2 v = finish(ce[t], cd[t], m, inv, dot);
              tl.entry[size_t(sm.entry[li + t]) * K + head] = v;
              dsd += v.y;
            }
          for (int t = kKeep; t <= n; ++t) {
            float2* p = tl.entry + size_t(sm.entry[li + t]) * K + head;
            const float2 v = finish(p->x, p->y, m, inv, dot);
            *p = v;
            dsd += v.y;
          }
          ds_dst[size_t(r0 + rs + rr) * K + head] = dsd;
        }
        li += n + 1;
      }
      if (w != RGV) {                          // the list ended inside a group: retire it without waiting
        __syncwarp();
        if (++slot == RG) { slot = 0; par ^= 1; }
      }
      rs += cnt;
    }
  }
  if (!alive) {
    if (lane == 0) raise(status, XRL_ERR_TIMEOUT);
    for (int t = 0; t < 100; ++t) __nanosleep(10000);
  }
#pragma unroll
  for (int t = 0; t < NP; ++t) {
    float lo, hi;
    split_f2(dbr[t], lo, hi);
    atomicAdd(&sm_db[c0 + 2 * t], lo);
    atomicAdd(&sm_db[c0 + 2 * t + 1], hi);
  }
  __syncthreads();
  for (int c = threadIdx.x; c < H; c += blockDim.x)
    if (sm_db[c] != 0.f) atomicAdd(&db[c], sm_db[c]);
}

// rows of `cols` elements, boxes of one row (gather4)
bool make_gather_map(CUtensorMap* m, const void* ptr, CUtensorMapDataType dt, uint32_t elem, uint64_t rows, uint32_t cols) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {uint64_t(cols) * elem};
  cuuint32_t box[2] = {cols, 1};
  cuuint32_t estr[2] = {1, 1};
  return fn(m, dt, 2, const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

int gather_grid(int32_t N, int shift) {
  const int64_t per_cta = int64_t(TW) << shift, want = (int64_t(N) + per_cta - 1) / per_cta;
  return int(want < int64_t(kNumSMs) * 5 ? want : int64_t(kNumSMs) * 5);
}

template <typename T, int K, bool MERGED>
int launch_rows_k(const BwdLists& t, const int32_t* rowptr, const int32_t* col, const void* Z, const float* scores,
                  const void* h_out, float* dh, bool masked, const float* dr, const int32_t* seg_id, float* ds_dst, float* gb,
                  int32_t N, int32_t* status, cudaStream_t st) {
  static bool attr[64] = {};
  constexpr int H = 32 * VecOf<T>::N;
  const size_t smem = sizeof(RowSmem<K, MERGED>) * TW + sizeof(float) * H;
  if (!ensure_dynamic_smem(k_rows_gather<T, K, MERGED>, int(smem), attr)) return -1;
  CUtensorMap mz, ms;
  if (MERGED) {
    if (!make_merged_map(&mz, Z, uint64_t(N), 512 + 8 * K)) return -1;
    ms = mz;
  } else if (!make_gather_map(&mz, Z, sizeof(T) == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                              sizeof(T), uint64_t(N), H) ||
             !make_gather_map(&ms, scores, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, uint64_t(N), 2 * K)) {
    return -1;
  }
  const int shift = aggregate_block_shift(N);
  launch(k_rows_gather<T, K, MERGED>, gather_grid(N, shift), TW * 32, smem, st,
      mz, ms, rowptr, col, static_cast<const T*>(Z), reinterpret_cast<const float2*>(scores), static_cast<const T*>(h_out), dh,
      masked, dr, seg_id, t, ds_dst, gb, N, shift, status);
  return 1;
}

template <typename T, int NV>
int launch_nv(const BwdLists& t, const float* dpre, const void* Z, size_t z_row, const float* ds_dst,
              const LayerWeights& lw, void* dz, float* ga_src, float* ga_dst, int32_t N, int32_t K, int32_t* status,
              cudaStream_t st) {
  using L = Layout<NV>;
  static bool attr[64] = {};
  const size_t smem = size_t(L::warp_bytes(K)) * TW + sizeof(float) * 512 * NV;
  // (the opt-in is the kernel's ceiling for every K: ask for the largest)
  if (!ensure_dynamic_smem(k_dz_gather<T, NV>, L::warp_bytes(16) * TW + int(sizeof(float)) * 512 * NV, attr)) return -1;
  CUtensorMap m;
  if (!make_gather_map(&m, dpre, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, uint64_t(N), 128 * NV)) return -1;
  const int shift = aggregate_block_shift(N);
  launch(k_dz_gather<T, NV>, gather_grid(N, shift), TW * 32, smem, st,
      m, dpre, t.entry, t.rowptr, t.col, static_cast<const char*>(Z), z_row, ds_dst, lw.a_src, lw.a_dst, static_cast<T*>(dz),
      ga_src, ga_dst, N, K, shift, status);
  return 1;
}

}  // namespace

// Hidden 128 or 256 (dpre rows of 512 or 1,024 bytes: a gather4 box holds at most 256 elements), an even number of heads
// that divides 32 (an entry's weights are then a multiple of 16 bytes).
bool bwd_gather_supported(const Dims& d) {
  return (d.H == 128 || d.H == 256) && d.K >= 2 && 32 % d.K == 0 && d.K <= 16 && encode_fn() != nullptr;
}

// Transposed lists of a CSR with E slots; scratch: N + scan_workspace_ints(N) ints.
int launch_bwd_lists(const int32_t* rowptr, const int32_t* col, int32_t N, int32_t E, const BwdLists& t, int32_t* scratch,
                     cudaStream_t st) {
  if (N <= 0) return 0;
  int32_t* cnt = scratch;
  cudaMemsetAsync(cnt, 0, sizeof(int32_t) * size_t(N), st);
  if (E > 0) launch(k_t_count, (E + 255) / 256, 256, 0, st, rowptr, col, N, E, cnt);
  const int n = launch_exclusive_scan(cnt, t.rowptr, N, scratch + N, st);
  launch(k_t_fill, (N + 255) / 256, 256, 0, st, rowptr, col, N, t.rowptr, cnt, t.col, t.inv);
  return n + 2;
}

int launch_dz_gather(const Dims& d, const BwdLists& t, const float* dpre, const void* Z, size_t z_row, const float* ds_dst,
                     const LayerWeights& lw, void* dz, float* ga_src, float* ga_dst, int32_t N, int32_t* status,
                     cudaStream_t st) {
#define DZ_ARGS t, dpre, Z, z_row, ds_dst, lw, dz, ga_src, ga_dst, N, d.K, status, st
  if (d.dtype == XRL_BF16) return d.H == 256 ? launch_nv<bf16, 2>(DZ_ARGS) : launch_nv<bf16, 1>(DZ_ARGS);
  return d.H == 256 ? launch_nv<float, 2>(DZ_ARGS) : launch_nv<float, 1>(DZ_ARGS);
#undef DZ_ARGS
}

// The softmax's reverse over 512-byte Z rows (hidden 256 in bf16 with the pairs behind the rows, 128 in fp32); -1: other
// shapes.
bool rows_gather_supported(const Dims& d) {
  return bwd_gather_supported(d) && (d.zmerged || (d.dtype == XRL_FP32 && d.H == 128)) && (d.K == 4 || d.K == 8 || d.K == 16);
}
int launch_rows_gather(const Dims& d, const BwdLists& t, const int32_t* rowptr, const int32_t* col, const void* Z,
                       const float* scores, const void* h_out, float* dh, bool masked, const float* dr, const int32_t* seg_id,
                       float* ds_dst, float* gb, int32_t N, int32_t* status, cudaStream_t st) {
#define ROWS_ARGS t, rowptr, col, Z, scores, h_out, dh, masked, dr, seg_id, ds_dst, gb, N, status, st
#define ROWS_CASE(KK)                                                                    \
  case KK:                                                                               \
    if (d.zmerged) return launch_rows_k<bf16, KK, true>(ROWS_ARGS);                      \
    if (d.dtype == XRL_FP32 && d.H == 128) return launch_rows_k<float, KK, false>(ROWS_ARGS); \
    return -1;
  switch (d.K) {
    ROWS_CASE(4) ROWS_CASE(8) ROWS_CASE(16)
    default: return -1;
  }
#undef ROWS_CASE
#undef ROWS_ARGS
}

}  // namespace xrl
