// Row-wise kernels of the encoder (paper Section 3.4): the node-update layer (Eq. 6), the
// attention half-scores, and the edge-score / segment-softmax / weighted-aggregate step of a
// graph-attention layer (Eq. 7).  One group of LPR lanes owns one destination row and moves it as 16-byte vectors: VPL per
// lane in the first two, one in the attention kernel (which splits longer rows into slabs of columns); 32 / LPR rows share
// a warp.
#include "xrl_agg_tma.cuh"

namespace xrl {

namespace {

constexpr int kRowThreads = 256;

// 8 shape features of one node as floats (all lanes of a group read the same address).
__device__ __forceinline__ void load_shape(const float* shape, int32_t node, float (&f)[kS]) {
  const float4 a = __ldg(reinterpret_cast<const float4*>(shape + size_t(node) * kS));
  const float4 b = __ldg(reinterpret_cast<const float4*>(shape + size_t(node) * kS) + 1);
  f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
}
__device__ __forceinline__ void load_shape(const bf16* shape, int32_t node, float (&f)[kS]) {
  unpack(__ldg(reinterpret_cast<const uint4*>(shape + size_t(node) * kS)), f);
}

// ---- Eq. 6: h0_i = ReLU(W0^T [ sum_{j->i} shape_j | onehot(op_i) | shape_i ] + b0) -----------
// (with attributes on the edges, Section 3.3.2 as written, the sum runs over the in-edges' own attributes)
// The one-hot block of the product is a row lookup of W0; the two shape blocks are a 16 x H
// dense map kept in shared memory as fp32.  A warp takes 8 rows at a time in two phases: first a lane per row
// gathers the row's sixteen dense inputs (row pointers, producers, their shape features: a chain of dependent
// loads, 8 chains side by side), then the warp's lanes share each row's columns, reading the inputs back from
// shared memory; the lookups of W0 for up to four rows are issued before the first is used.
constexpr int kEmbedWarps = kRowThreads / 32;
constexpr int kEmbedRows = 8;        // rows a warp takes at a time
struct EmbedStage { float x[kEmbedRows][2 * kS]; int32_t op[kEmbedRows]; };

template <typename T, int LPR, int VPL>
__global__ void __launch_bounds__(kRowThreads)
k_embed(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
        const int32_t* __restrict__ op, const T* __restrict__ shape, const T* __restrict__ W0,
        const float* __restrict__ b0, T* __restrict__ h, int H, int Tn, Window win,
        const int32_t* __restrict__ row_list, const T* __restrict__ eattr) {
  constexpr int VEC = VecOf<T>::N;
  constexpr int RPW = 32 / LPR;
  extern __shared__ __align__(16) float smem[];
  EmbedStage& stg = reinterpret_cast<EmbedStage*>(smem)[threadIdx.x >> 5];
  float* Wd = smem + kEmbedWarps * (sizeof(EmbedStage) / sizeof(float));   // [2*kS][H]
  float* bs = Wd + 2 * kS * H;                                             // [H]
  for (int t = threadIdx.x; t < 2 * kS * H; t += blockDim.x) {
    const int s = t / H, c = t - s * H;
    const int src_row = (s < kS) ? s : (kS + Tn + (s - kS));
    Wd[t] = to_float(W0[size_t(src_row) * H + c]);
  }
  for (int t = threadIdx.x; t < H; t += blockDim.x) bs[t] = b0[t];
  // only weights are read above; as the kernel's first statement the wait cost the one-vector bf16 kernels 47 registers and their
  // third CTA per SM (179 k rows of hidden 64 65.9 us instead of 59.8, of 128 171.9 instead of 166.5)
  enter();
  __syncthreads();

  const int NV = H / VEC;
  const int lane = threadIdx.x & 31, sub = lane / LPR, sl = lane % LPR;
  const int warps_total = (gridDim.x * blockDim.x) >> 5;
  const int warp_id = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  // fp32 rows with one vector of columns per lane: the lane's 16 x VEC slice of the dense map and its bias stay in registers
  // (read from shared memory per row, the map makes the kernel wait on shared-memory bandwidth)
  constexpr bool REGW = VPL == 1 && VEC == 4;
  float wreg[REGW ? 2 * kS : 1][VEC], breg[VEC];
  if (REGW && sl < NV) {
#pragma unroll
    for (int s = 0; s < 2 * kS; ++s)
#pragma unroll
      for (int t = 0; t < VEC; ++t) wreg[REGW ? s : 0][t] = Wd[s * H + sl * VEC + t];
#pragma unroll
    for (int t = 0; t < VEC; ++t) breg[t] = bs[sl * VEC + t];
  }
  for (int64_t r0 = int64_t(win.row_begin) + int64_t(warp_id) * kEmbedRows; r0 < win.row_end;
       r0 += int64_t(warps_total) * kEmbedRows) {
    const int nr = int(min(int64_t(kEmbedRows), win.row_end - r0));
    __syncwarp();
    if (lane < nr) {
      const int32_t out_row = int32_t(r0) + lane;
      const int32_t row = row_list ? __ldg(row_list + out_row) : out_row;   // listed rows are written densely
      float x[kS];
#pragma unroll
      for (int s = 0; s < kS; ++s) x[s] = 0.f;
      const int32_t e0 = __ldg(rowptr + row), e1 = __ldg(rowptr + row + 1);
      for (int32_t e = e0; e < e1; ++e) {
        float f[kS];
        if (eattr) load_shape(eattr, e, f);            // attributes on the edges, already in slot order
        else load_shape(shape, __ldg(col + e), f);     // the producer's shape features
#pragma unroll
        for (int s = 0; s < kS; ++s) x[s] += f[s];
      }
      float own[kS];
      load_shape(shape, row, own);
#pragma unroll
      for (int s = 0; s < kS; ++s) { stg.x[lane][s] = x[s]; stg.x[lane][kS + s] = own[s]; }
      // an operator id outside the table was reported by the packer; clamped here so that nothing is read
      // outside W0 if the caller encodes such a batch anyway
      stg.op[lane] = min(max(__ldg(op + row), 0), Tn - 1);
    }
    __syncwarp();
    constexpr int U = (VPL >= 4) ? 1 : (VPL == 2 ? 2 : 4);     // rows whose lookups are in flight together
    for (int rb = sub; rb < nr; rb += RPW * U) {
      float acc[U][VPL][VEC];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int rr = rb + u * RPW;
        if (rr < nr) {
          const T* lookup = W0 + size_t(kS + stg.op[rr]) * H;
#pragma unroll
          for (int v = 0; v < VPL; ++v) {
            const int vi = v * LPR + sl;
            if (vi < NV) load_vec(lookup + vi * VEC, acc[u][v]);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int rr = rb + u * RPW;
        if (rr >= nr) continue;
        float x[2 * kS];
#pragma unroll
        for (int s = 0; s < 2 * kS; s += 4) {
          const float4 v4 = *reinterpret_cast<const float4*>(&stg.x[rr][s]);
          x[s] = v4.x; x[s + 1] = v4.y; x[s + 2] = v4.z; x[s + 3] = v4.w;
        }
        T* out = h + size_t(int32_t(r0) + rr - win.win_base) * H;
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
          const int vi = v * LPR + sl;
          if (vi < NV) {
            const int c0 = vi * VEC;
            if (REGW) {
#pragma unroll
              for (int t = 0; t < VEC; ++t) acc[u][v][t] += breg[t];
#pragma unroll
              for (int s = 0; s < 2 * kS; ++s)
#pragma unroll
                for (int t = 0; t < VEC; ++t) acc[u][v][t] = fmaf(x[s], wreg[REGW ? s : 0][t], acc[u][v][t]);
            } else {
#pragma unroll
              for (int t = 0; t < VEC; ++t) acc[u][v][t] += bs[c0 + t];
#pragma unroll
              for (int s = 0; s < 2 * kS; ++s)
#pragma unroll
                for (int t = 0; t < VEC; ++t) acc[u][v][t] = fmaf(x[s], Wd[s * H + c0 + t], acc[u][v][t]);
            }
#pragma unroll
            for (int t = 0; t < VEC; ++t) acc[u][v][t] = fmaxf(acc[u][v][t], 0.f);
            store_vec(out + c0, acc[u][v]);
          }
        }
      }
    }
  }
}

// ---- attention half-scores from Z (used when the transform kernel does not emit them) ------
// s_src[i,k] = log2(e) a_src[k] . Z[i, head k],  s_dst[i,k] = log2(e) a_dst[k] . Z[i, head k]
// (stored pre-multiplied by log2(e): the aggregate kernel then needs exp2 only)
// A row group takes R rows at a time (their loads in flight together) with its columns of a_src and a_dst in registers.  The
// lanes of a head's q vectors (q = the power of two in their number) add up by shuffles, the first of which leaves one of
// the two sums per lane; heads of more than one such run add the runs through shared memory.  (A row at a time, a lane adding
// its head's vectors one by one: 384 us per layer of 323 k rows of 512 with one head, now 151.)
template <typename T, int LPR, int VPL>
__global__ void __launch_bounds__(kRowThreads)
k_scores(const T* __restrict__ Z, const float* __restrict__ a_src, const float* __restrict__ a_dst,
         float2* __restrict__ scores, int H, int K, Window win) {
  enter();
  constexpr int VEC = VecOf<T>::N;
  constexpr int RPW = 32 / LPR;
  constexpr int WARPS = kRowThreads / 32;
  constexpr int R = VPL >= 2 ? 2 : 4;
  __shared__ float2 part[WARPS][RPW][R][LPR * VPL];
  const int NV = H / VEC, vph = H / K / VEC;
  const int lane = threadIdx.x & 31, sub = lane / LPR, sl = lane % LPR, wib = threadIdx.x >> 5;
  const int warps_total = (gridDim.x * blockDim.x) >> 5;
  const int warp_id = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int q = vph & -vph;
  if (q > LPR) q = LPR;
  const int qs = __ffs(q) - 1, runs = vph >> qs;          // runs of q vectors per head
  float as[VPL][VEC], ad[VPL][VEC];
#pragma unroll
  for (int v = 0; v < VPL; ++v)
#pragma unroll
    for (int t = 0; t < VEC; ++t) {
      const int c = (v * LPR + sl) * VEC + t;
      as[v][t] = c < H ? __ldg(a_src + c) : 0.f;
      ad[v][t] = c < H ? __ldg(a_dst + c) : 0.f;
    }
  for (int64_t r0 = int64_t(win.row_begin) + int64_t(warp_id) * (RPW * R); r0 < win.row_end;
       r0 += int64_t(warps_total) * (RPW * R)) {
    float f[R][VPL][VEC];
#pragma unroll
    for (int u = 0; u < R; ++u)
#pragma unroll
      for (int v = 0; v < VPL; ++v) {
        const int64_t row = r0 + sub * R + u;
        const int vi = v * LPR + sl;
#pragma unroll
        for (int t = 0; t < VEC; ++t) f[u][v][t] = 0.f;
        if (row < win.row_end && vi < NV) load_vec(Z + size_t(row - win.win_base) * H + vi * VEC, f[u][v]);
      }
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const int64_t row = r0 + sub * R + u;
      float2* out = scores + size_t(row - win.win_base) * K;
#pragma unroll
      for (int v = 0; v < VPL; ++v) {
        const int vi = v * LPR + sl;
        float ps = 0.f, pd = 0.f;
#pragma unroll
        for (int t = 0; t < VEC; ++t) {
          ps = fmaf(f[u][v][t], as[v][t], ps);
          pd = fmaf(f[u][v][t], ad[v][t], pd);
        }
        if (q == 1) {
          part[wib][sub][u][vi] = make_float2(ps, pd);
        } else {                                          // lanes of even vectors: the sum for s_src, odd: for s_dst
          const bool odd = (sl & 1) != 0;
          float x = (odd ? pd : ps) + __shfl_xor_sync(0xFFFFFFFFu, odd ? ps : pd, 1);
#pragma unroll
          for (int o = 2; o < LPR; o <<= 1)
            if (o < q) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
          if (runs == 1) {
            if ((sl & (q - 1)) < 2 && vi < NV && row < win.row_end)
              reinterpret_cast<float*>(out + (vi >> qs))[odd ? 1 : 0] = x * kLog2e;
          } else if ((sl & (q - 1)) < 2) {
            reinterpret_cast<float*>(&part[wib][sub][u][vi >> qs])[odd ? 1 : 0] = x;
          }
        }
      }
    }
    if (runs > 1 || q == 1) {
      __syncwarp();
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const int64_t row = r0 + sub * R + u;
        if (row < win.row_end)
          for (int k = sl; k < K; k += LPR) {
            float ss = 0.f, sd = 0.f;
            for (int v = k * runs; v < (k + 1) * runs; ++v) {
              const float2 p = part[wib][sub][u][v];
              ss += p.x;
              sd += p.y;
            }
            scores[size_t(row - win.win_base) * K + k] = make_float2(ss * kLog2e, sd * kLog2e);
          }
      }
      __syncwarp();
    }
  }
}

// ---- Eq. 7: edge scores, softmax over producers + self, weighted sum of Z rows, bias, ReLU ---
// A warp takes blocks of 32 consecutive destination rows: row pointers and producer ids of the
// whole block are fetched with a few coalesced loads into shared memory, so that the per-row work
// starts straight at the gathers of Z.  The half-scores arrive already multiplied by log2(e)
// (LeakyReLU commutes with a positive factor), so the softmax weights are plain exp2.  Producers
// are taken two at a time, the first two asked for with the row's own vector.
constexpr int kAggBlockRows = 32;
constexpr int kAggColCap = 224;       // producer ids cached per block of rows

__device__ __forceinline__ float lrelu(float x) { return fmaxf(x, 0.2f * x); }
__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// READOUT (several rows per warp only): the last layer fused with the per-graph sum of Eq. 8 (hidden 128 in bf16, 299 k rows:
// 51 + 19 -> 51 us; with a row per warp, hidden 192, 124 k rows, 46 + 10 -> 59 us: the sums do not fit the registers of four
// CTAs per SM), in the layout of the TMA kernel's fused variant (blocks of `block_rows` = 2^k rows from row 0 on: the rows of
// a block's first graph to partial[block], those of a graph that starts inside it to partial[nblocks + graph]).  READOUT = 2
// stores the rows as well; the sum is of the rows as they are stored either way, as the readout's and the delta path's are.
// ZERO (bf16 rows of more than 32 vectors): the ReLU of what is no number - a row that an infinite feature has reached - is 0, as
// in the definition; the one inside the rounding, which shorter bf16 rows have, keeps it (a step of 256 k rows of 320 1,139 us
// with that one, 1,144 with this).
template <typename T, int LPR, int READOUT, bool ZERO>
__global__ void __launch_bounds__(kRowThreads, 4)
k_aggregate(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
            const T* __restrict__ Z, const float2* __restrict__ scores,
            const float* __restrict__ bias, T* __restrict__ h_out, int H, int K, Window win,
            const int32_t* __restrict__ self_idx, int block_rows, int slab_vecs, const int32_t* __restrict__ seg_id,
            float* __restrict__ partial, int32_t nblocks) {
  enter();
  constexpr int VEC = VecOf<T>::N;
  constexpr int RPW = 32 / LPR;
  constexpr int WARPS = kRowThreads / 32;
  __shared__ int32_t s_rp[WARPS][kAggBlockRows + 1];
  __shared__ int32_t s_col[WARPS][kAggColCap];
  const int NV = H / VEC, d = H / K;
  const int lane = threadIdx.x & 31, sub = lane / LPR, sl = lane % LPR, wib = threadIdx.x >> 5;
  const int warps_total = (gridDim.x * blockDim.x) >> 5;
  const int warp_id = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;

  // one vector per lane; rows of more than 32 vectors are split into gridDim.y slabs of columns (every slab weighs the
  // producers anew; two vectors per lane one after the other, in groups of one to four producers, took 356 us per layer of
  // 323 k rows of 512 with one head, slabs 240)
  const int vi = int(blockIdx.y) * slab_vecs + sl;
  const bool on = sl < slab_vecs && vi < NV;
  const int c0 = on ? vi * VEC : 0, head = c0 / d;
  float bs[VEC];
#pragma unroll
  for (int t = 0; t < VEC; ++t) bs[t] = __ldg(bias + c0 + t);

  // blocks of rows: as many rows (up to 32) as keep the block's producer ids within the cache;
  // a single row with more producers than that is walked straight from global memory
  // block_rows <= kAggBlockRows rows per warp and pass: fewer when the batch is small, so that every
  // warp of the grid has work
  int64_t r0 = int64_t(win.row_begin) + int64_t(warp_id) * block_rows;
  while (r0 < win.row_end) {
    const int nr = int(min(int64_t(block_rows), win.row_end - r0));
    __syncwarp();                                   // the previous block's reads are done
    if (lane < nr) s_rp[wib][lane] = __ldg(rowptr + r0 + lane);
    if (lane == 0) s_rp[wib][nr] = __ldg(rowptr + r0 + nr);
    __syncwarp();
    const int32_t eb = s_rp[wib][0];
    const int ne = min(s_rp[wib][nr] - eb, kAggColCap);
    for (int t = lane; t < ne; t += 32) s_col[wib][t] = __ldg(col + eb + t);
    __syncwarp();

    // The 32 / LPR rows of a warp go through one code path together: producers two at a time up to
    // the largest count among the rows, the first two asked for together with the row's own
    // vector, packed fp32 arithmetic, a reference exponent that moves only when a score exceeds it by 32.  Rows of
    // different degrees taking their own branches through groups of 1 to 4 producers executed 115 warp instructions
    // per row at 58 % issue utilisation (hidden 128 bf16, 299 k rows of mean degree 1.1: 0.057 ms; now
    // 0.053.  Asking for the next rows' vectors one step ahead costs a resident CTA per SM: 0.066).
    constexpr int NP = VEC / 2;
    const T* zlane = Z + c0;
    const float2* slane = scores + head;
    // (READOUT) the running sum of the current graph's rows, one per row group of the warp
    const int32_t myseg = READOUT && lane < nr ? __ldg(seg_id + r0 + lane) : 0;
    int32_t cur = -1;
    bool first_seg = true;
    aggtma::F2 sum[NP];
    auto clear = [&]() {
#pragma unroll
      for (int t = 0; t < NP; ++t) sum[t] = aggtma::make_f2(0.f, 0.f);
    };
    auto flush = [&]() {
      float* dst = partial + size_t(first_seg ? int32_t(r0 / block_rows) : nblocks + cur) * H + c0;
#pragma unroll
      for (int t = 0; t < NP; ++t) {
        float lo, hi;
        aggtma::split_f2(sum[t], lo, hi);
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1) {
          lo += __shfl_xor_sync(0xFFFFFFFFu, lo, o);
          hi += __shfl_xor_sync(0xFFFFFFFFu, hi, o);
        }
        if (sub == 0 && on) *reinterpret_cast<float2*>(dst + 2 * t) = make_float2(lo, hi);
      }
      first_seg = false;
      clear();
    };
    if (READOUT) clear();
    for (int base = 0; base < nr; base += RPW) {
      const int rr = base + sub;
      const bool live = on && rr < nr;
      int e0 = 0, n = 0;
      if (live) { e0 = s_rp[wib][rr] - eb; n = s_rp[wib][rr + 1] - eb - e0; }
      const int nmax = RPW == 1 ? n : __reduce_max_sync(0xFFFFFFFFu, n);
      const int32_t lrow = int32_t(r0) + rr - win.win_base;
      const int32_t* js = e0 + n <= kAggColCap ? &s_col[wib][e0] : col + eb + e0;
      float2 self = make_float2(0.f, 0.f);
      uint4 raw = make_uint4(0u, 0u, 0u, 0u), qa, qb;
      float ea, eo;
      if (live) {
        const int32_t srow = self_idx ? __ldg(self_idx + int32_t(r0) + rr) : lrow;   // where the row's own Z lives
        self = __ldg(slane + size_t(srow) * K);
        raw = __ldg(reinterpret_cast<const uint4*>(zlane + size_t(srow) * H));
      }
      auto pair = [&](int t) {                        // producers t, t + 1
        ea = eo = -INFINITY;
        qa = qb = make_uint4(0u, 0u, 0u, 0u);
        if (t < n) {
          const int32_t j = js[t] - win.win_base;
          ea = __ldg(&slane[size_t(j) * K].x);
          qa = __ldg(reinterpret_cast<const uint4*>(zlane + size_t(j) * H));
        }
        if (t + 1 < n) {
          const int32_t j = js[t + 1] - win.win_base;
          eo = __ldg(&slane[size_t(j) * K].x);
          qb = __ldg(reinterpret_cast<const uint4*>(zlane + size_t(j) * H));
        }
      };
      if (nmax > 0) pair(0);
      const float sd = self.y;
      float m = lrelu(self.x + sd), l = 1.f;          // the self term opens the softmax
      aggtma::F2 acc[NP];
      aggtma::to_pairs(raw, acc);
      for (int t = 0; t < nmax; t += 2) {
        if (t > 0) pair(t);
        const float ev0 = lrelu(ea + sd), ev1 = lrelu(eo + sd), evm = fmaxf(ev0, ev1);
        if (evm > m + 32.f) aggtma::raise_reference<NP>(evm, m, l, acc);
        // (absent producers weigh 0 by their place and not by their score, which is no number where the row's is infinite)
        const float p0 = t < n ? fast_exp2(ev0 - m) : 0.f, p1 = t + 1 < n ? fast_exp2(ev1 - m) : 0.f;
        l += p0 + p1;
        aggtma::F2 z[NP];
        aggtma::to_pairs(qa, z);
        const aggtma::F2 w0 = aggtma::make_f2(p0, p0), w1 = aggtma::make_f2(p1, p1);
#pragma unroll
        for (int q = 0; q < NP; ++q) aggtma::fma2(acc[q], w0, z[q]);
        aggtma::to_pairs(qb, z);
#pragma unroll
        for (int q = 0; q < NP; ++q) aggtma::fma2(acc[q], w1, z[q]);
      }
      const float inv = __fdividef(1.f, l);
      if constexpr (READOUT == 0) {
        if constexpr (ZERO) {
          uint32_t w[4];
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            aggtma::F2 v = aggtma::make_f2(bs[2 * t], bs[2 * t + 1]);
            aggtma::fma2(v, acc[t], aggtma::make_f2(inv, inv));
            float lo, hi;
            aggtma::split_f2(v, lo, hi);
            w[t] = pack_bf16x2(lo, hi);
            asm("max.bf16x2 %0, %0, %1;" : "+r"(w[t]) : "r"(0u));      // (of a number and none: the number)
          }
          if (live) *reinterpret_cast<uint4*>(h_out + size_t(lrow) * H + c0) = make_uint4(w[0], w[1], w[2], w[3]);
        } else if (live) {
          aggtma::finish_row(h_out + size_t(lrow) * H + c0, acc, inv, bs);
        }
      } else {
        aggtma::F2 o[NP];
        if constexpr (READOUT == 1) aggtma::to_pairs(aggtma::row_as_stored(acc, inv, bs), o);
        else if (live) aggtma::to_pairs(aggtma::finish_row(h_out + size_t(lrow) * H + c0, acc, inv, bs), o);
        const int32_t g0 = __shfl_sync(0xFFFFFFFFu, myseg, base), g1 = __shfl_sync(0xFFFFFFFFu, myseg, min(base + RPW, nr) - 1);
        if (g0 == cur && g1 == cur) {
          if (live)
#pragma unroll
            for (int t = 0; t < NP; ++t) aggtma::add2(sum[t], o[t]);
        } else {                                 // a graph begins here: row by row
          for (int s = 0; s < RPW && base + s < nr; ++s) {
            const int32_t g = __shfl_sync(0xFFFFFFFFu, myseg, base + s);
            if (g != cur) {
              if (cur >= 0) flush();
              cur = g;
            }
            if (live && sub == s)
#pragma unroll
              for (int t = 0; t < NP; ++t) aggtma::add2(sum[t], o[t]);
          }
        }
      }
    }
    if (READOUT && cur >= 0) flush();
    r0 += int64_t(warps_total) * block_rows;
  }
}

// ---- dispatch on the row geometry ------------------------------------------------------------
struct RowGeom { int lpr, vpl; };

template <typename T>
RowGeom row_geom(int H) {
  const int nv = H / VecOf<T>::N;
  if (nv <= 8) return {8, 1};
  if (nv <= 16) return {16, 1};        // (12 vectors, hidden 96: a row per warp took 66 us per layer of 194 k rows, two 43)
  const int vpl = (nv + 31) / 32;
  return {32, vpl <= 1 ? 1 : (vpl == 2 ? 2 : 4)};
}

RowGeom row_geom_of(const Dims& d) { return d.dtype == XRL_BF16 ? row_geom<bf16>(d.H) : row_geom<float>(d.H); }

int row_grid(int64_t rows, int rpw) {
  const int64_t warps = (rows + rpw - 1) / rpw;
  const int64_t blocks = (warps + (kRowThreads / 32) - 1) / (kRowThreads / 32);
  const int64_t cap = int64_t(kNumSMs) * 8;
  return int(blocks < 1 ? 1 : (blocks > cap ? cap : blocks));
}

#define XRL_ROW_DISPATCH(TY_, H, CALL)                                         \
  do {                                                                       \
    const RowGeom g_ = row_geom<TY_>(H);                                       \
    if (g_.lpr == 8) { CALL(TY_, 8, 1); }                                      \
    else if (g_.lpr == 16) { CALL(TY_, 16, 1); }                               \
    else if (g_.vpl == 1) { CALL(TY_, 32, 1); }                                \
    else if (g_.vpl == 2) { CALL(TY_, 32, 2); }                                \
    else { CALL(TY_, 32, 4); }                                                 \
  } while (0)

}  // namespace

// one opt-in record per instantiation of k_embed (ensure_dynamic_smem keeps one flag array per kernel)
static int embed_slot(size_t elem, int lpr, int vpl) {
  return (elem == 2 ? 5 : 0) + (lpr == 8 ? 0 : lpr == 16 ? 1 : vpl == 1 ? 2 : vpl == 2 ? 3 : 4);
}

int launch_embed(const Dims& d, const int32_t* rowptr, const int32_t* col, const int32_t* op,
                 const void* shape, const DevWeights& w, void* h, Window win, cudaStream_t st,
                 const int32_t* row_list, const void* eattr) {
  const int64_t rows = int64_t(win.row_end) - win.row_begin;
  if (rows <= 0) return 0;
  const size_t smem = sizeof(EmbedStage) * kEmbedWarps + sizeof(float) * size_t(2 * kS + 1) * d.H;
  static bool attr_set[10][64] = {};
#define CALL(TY_, LPR, VPL)                                                                        \
  if (smem > 48 * 1024 &&                                                                          \
      !ensure_dynamic_smem(k_embed<TY_, LPR, VPL>, int(smem), attr_set[embed_slot(sizeof(TY_), LPR, VPL)])) return -1; \
  launch(k_embed<TY_, LPR, VPL>, row_grid(rows, kEmbedRows), kRowThreads, smem, st,                            \
      rowptr, col, op, static_cast<const TY_*>(shape), static_cast<const TY_*>(w.W0), w.b0,   \
      static_cast<TY_*>(h), d.H, d.T, win, row_list, static_cast<const TY_*>(eattr))
  if (d.dtype == XRL_BF16) XRL_ROW_DISPATCH(bf16, d.H, CALL);
  else XRL_ROW_DISPATCH(float, d.H, CALL);
#undef CALL
  return 1;
}

int launch_scores(const Dims& d, const void* Z, const LayerWeights& lw, float* scores, Window win,
                  cudaStream_t st) {
  const int64_t rows = int64_t(win.row_end) - win.row_begin;
  if (rows <= 0) return 0;
#define CALL(TY_, LPR, VPL)                                                                        \
  launch(k_scores<TY_, LPR, VPL>, row_grid(rows, 32 / LPR * (VPL >= 2 ? 2 : 4)), kRowThreads, 0, st,                        \
      static_cast<const TY_*>(Z), lw.a_src, lw.a_dst, reinterpret_cast<float2*>(scores), d.H, d.K, win)
  if (d.dtype == XRL_BF16) XRL_ROW_DISPATCH(bf16, d.H, CALL);
  else XRL_ROW_DISPATCH(float, d.H, CALL);
#undef CALL
  return 1;
}

int launch_aggregate(const Dims& d, const int32_t* rowptr, const int32_t* col, const void* Z,
                     const float* scores, const float* bias, void* h_out,
                     Window win, int64_t buf_rows, int32_t* status, cudaStream_t st,
                     const int32_t* self_idx, const int32_t* seg_id, float* partial) {
  const int64_t rows = int64_t(win.row_end) - win.row_begin;
  if (rows <= 0) return 0;
  {   // 512-byte rows with 4 | K: gathers by the TMA engine
    const int k = launch_aggregate_tma(d, rowptr, col, Z, scores, bias, h_out, win, buf_rows, seg_id, partial, status, st,
                                       self_idx);
    if (k >= 0 || d.zmerged) return k;       // with merged rows there is no other kernel to fall back to
  }
  if (partial != nullptr && (win.row_begin != 0 || win.win_base != 0 || row_geom_of(d).lpr > 16)) return -1;
  // rows per warp and pass: the 32 of a full block, fewer for small batches (a multiple of the rows a
  // warp holds at once); with the sums the blocks that their layout has
  const int64_t warps_avail = int64_t(kNumSMs) * 8 * (kRowThreads / 32);
  const int64_t sum_rows = int64_t(1) << aggregate_block_shift(rows);
  const int nv = d.H / (d.dtype == XRL_BF16 ? VecOf<bf16>::N : VecOf<float>::N), slabs = (nv + 31) / 32,
            slab_vecs = (nv + slabs - 1) / slabs;
#define CALL_(TY_, LPR, RO_, ZERO_, br_)                                                           \
  launch(k_aggregate<TY_, LPR, RO_, ZERO_>, dim3(unsigned(row_grid(rows, int(br_))), unsigned(slabs)), kRowThreads, 0, st, \
         rowptr, col, static_cast<const TY_*>(Z), reinterpret_cast<const float2*>(scores), bias,   \
         static_cast<TY_*>(h_out), d.H, d.K, win, self_idx, int(br_), slab_vecs, seg_id, partial,  \
         int32_t((rows + sum_rows - 1) / sum_rows))
#define CALL(TY_, LPR, VPL)                                                                        \
  do {                                                                                             \
    const int rpw_ = 32 / LPR;                                                                     \
    int64_t br_ = (rows * slabs + warps_avail - 1) / warps_avail;                                          \
    br_ = ((br_ + rpw_ - 1) / rpw_) * rpw_;                                                        \
    if (br_ > kAggBlockRows) br_ = kAggBlockRows;                                                  \
    if (slabs > 1) CALL_(TY_, 32, 0, sizeof(TY_) == 2, br_);                                       \
    else if (LPR > 16 || partial == nullptr) CALL_(TY_, LPR, 0, false, br_);                       \
    else if (h_out == nullptr) CALL_(TY_, LPR, (LPR <= 16 ? 1 : 0), false, sum_rows);              \
    else CALL_(TY_, LPR, (LPR <= 16 ? 2 : 0), false, sum_rows);                                    \
  } while (0)
  if (d.dtype == XRL_BF16) XRL_ROW_DISPATCH(bf16, d.H, CALL);
  else XRL_ROW_DISPATCH(float, d.H, CALL);
#undef CALL
#undef CALL_
  return 1;
}

}  // namespace xrl
