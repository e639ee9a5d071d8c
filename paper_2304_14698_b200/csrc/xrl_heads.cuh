// Device code of the dense layers at the end of the path (Eq. 8's W_g, the policy and value MLPs), shared by the heads'
// forward kernels and by the training step's: matrix-vector products by a whole CTA, for one or several input rows at a
// time, and block-wide reductions.  Every sum runs in an order fixed by the launch shape.
#pragma once

#include "xrl_internal.cuh"

namespace xrl {
namespace heads {

// A head's MLP (Section 3.3.2): out = w2 . ReLU(W1^T x + b1) + b2, or with a second hidden width hid2 > 0
// out = w2 . ReLU(Wh^T ReLU(W1^T x + b1) + bh) + b2.
struct Mlp { const float *W1, *b1, *Wh, *bh, *w2, *b2; int hid, hid2; };

constexpr int kThreads = 1024;

// Rows of x in shared memory start `row_stride` floats apart, on 16-byte boundaries.
__host__ __device__ inline int row_stride(int n) { return (n + 3) & ~3; }

// y[g][c] = bias[c] + sum_k x[g][k] W[k * ld + c] for the GP rows of x and c < ncols, by all threads of the block.  A
// weight is loaded once for the GP rows: launches of many rows are bound by these loads (264 KB of W_g per graph at
// hidden 256), launches of few by their latency, so up to D of them are in flight per thread.  With fewer columns than
// threads the k range is cut into P = blockDim / CP contiguous parts (CP = columns per pass, a power of two), added in part
// order.  `part`: GP * blockDim floats of scratch; emit(g, c, y) runs once per output; ends with a barrier.
template <int GP, typename Emit>
__device__ __forceinline__ void dense_rows(const float* x, int xs, int in, const float* __restrict__ W, int ld, int ncols,
                                           const float* __restrict__ bias, float* part, Emit emit) {
  constexpr int D = GP == 1 ? 32 : GP <= 4 ? 16 : 8;
  const int nt = blockDim.x, tid = threadIdx.x;
  int CP = 32;
  while (CP < ncols && CP < nt) CP <<= 1;
  const int P = nt / CP, cl = tid % CP, p = tid / CP;
  const int chunk = ((in + P - 1) / P + 3) & ~3, k0 = min(in, p * chunk), k1 = min(in, k0 + chunk);
  for (int c0 = 0; c0 < ncols; c0 += CP) {
    const int c = c0 + cl;
    float acc[GP];
#pragma unroll
    for (int g = 0; g < GP; ++g) acc[g] = 0.f;
    if (c < ncols) {
      const float* w0 = W + c;
      int k = k0;
      for (; k + D <= k1; k += D) {
        float w[D];
#pragma unroll
        for (int t = 0; t < D; ++t) w[t] = __ldg(w0 + size_t(k + t) * ld);
#pragma unroll
        for (int g = 0; g < GP; ++g)
#pragma unroll
          for (int t = 0; t < D; t += 4) {
            const float4 v = *reinterpret_cast<const float4*>(x + g * xs + k + t);
            acc[g] = fmaf(v.x, w[t], acc[g]); acc[g] = fmaf(v.y, w[t + 1], acc[g]);
            acc[g] = fmaf(v.z, w[t + 2], acc[g]); acc[g] = fmaf(v.w, w[t + 3], acc[g]);
          }
      }
      for (; k + 4 <= k1; k += 4) {
        float w[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) w[t] = __ldg(w0 + size_t(k + t) * ld);
#pragma unroll
        for (int g = 0; g < GP; ++g) {
          const float4 v = *reinterpret_cast<const float4*>(x + g * xs + k);
          acc[g] = fmaf(v.x, w[0], acc[g]); acc[g] = fmaf(v.y, w[1], acc[g]);
          acc[g] = fmaf(v.z, w[2], acc[g]); acc[g] = fmaf(v.w, w[3], acc[g]);
        }
      }
      for (; k < k1; ++k) {
        const float w = __ldg(w0 + size_t(k) * ld);
#pragma unroll
        for (int g = 0; g < GP; ++g) acc[g] = fmaf(x[g * xs + k], w, acc[g]);
      }
    }
    if (P == 1) {
      if (c < ncols) {
        const float b = bias[c];
#pragma unroll
        for (int g = 0; g < GP; ++g) emit(g, c, b + acc[g]);
      }
    } else {
#pragma unroll
      for (int g = 0; g < GP; ++g) part[(g * P + p) * CP + cl] = acc[g];
      __syncthreads();
      for (int t = tid; t < GP * CP; t += nt) {
        const int g = t / CP, cc = t % CP;
        if (c0 + cc < ncols) {
          float y = bias[c0 + cc];
          for (int q = 0; q < P; ++q) y += part[(g * P + q) * CP + cc];
          emit(g, c0 + cc, y);
        }
      }
    }
    __syncthreads();
  }
}

// The sums over a warp's lanes of V = 2^k values each: value i ends up in lanes i * 32 / V and up.  Every step
// halves the values that a lane carries: V - 1 + log2(32 / V) shuffles where a tree per value takes 5 V, the same additions.
template <int V>
__device__ __forceinline__ float warp_sums(float (&v)[V], int lane) {
  int o = 16;
#pragma unroll
  for (int n = V / 2; n > 0; n >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const float keep = up ? v[i + n] : v[i], send = up ? v[i] : v[i + n];
      v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, o);
    }
  }
  float s = v[0];
  for (; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
  return s;
}

// out[g][k] = sum_c W[k * ncols + c] v[g][c] for the GP rows of v (in shared memory, vs floats apart): a warp per R rows of
// W, lanes along the columns, 4 R loads in flight.  The chain of passes over W's rows bounds it, then the shuffles
// (two rows a warp and a tree per sum: k_graph_bwd of 324 graphs of 256 33 us, now 16; k_ppo_env 37 -> 32).
// emit(g, k, value) runs in one lane; ends with a barrier.
template <int GP, typename Emit>
__device__ __forceinline__ void rows_dot(const float* __restrict__ W, int nrows, int ncols, const float* v, int vs, Emit emit) {
  constexpr int R = GP == 1 ? 8 : GP <= 4 ? 4 : 2, V = R * GP;
  static_assert((V & (V - 1)) == 0 && V <= 32, "");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int k = R * warp; k < nrows; k += R * nw) {
    const float* w0 = W + size_t(k) * ncols;
    const int last = nrows - 1 - k;                   // (rows past the end: the last one again)
    float a[V];
#pragma unroll
    for (int i = 0; i < V; ++i) a[i] = 0.f;
    int c = lane;
    for (; c + 96 < ncols; c += 128) {
      float p[R][4];
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int t = 0; t < 4; ++t) p[r][t] = __ldg(w0 + size_t(min(r, last)) * ncols + c + 32 * t);
#pragma unroll
      for (int g = 0; g < GP; ++g)
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const float x = v[g * vs + c + 32 * t];
#pragma unroll
          for (int r = 0; r < R; ++r) a[r * GP + g] = fmaf(p[r][t], x, a[r * GP + g]);
        }
    }
    for (; c < ncols; c += 32) {
      float p[R];
#pragma unroll
      for (int r = 0; r < R; ++r) p[r] = __ldg(w0 + size_t(min(r, last)) * ncols + c);
#pragma unroll
      for (int g = 0; g < GP; ++g) {
        const float x = v[g * vs + c];
#pragma unroll
        for (int r = 0; r < R; ++r) a[r * GP + g] = fmaf(p[r], x, a[r * GP + g]);
      }
    }
    const float s = warp_sums<V>(a, lane);
    const int i = lane / (32 / V), r = i / GP;
    if (lane % (32 / V) == 0 && r <= last) emit(i % GP, k + r, s);
  }
  __syncthreads();
}

// Block-wide sum in a fixed order (lanes of a warp by a shuffle tree, then the warps' sums by one warp's
// shuffle tree): the same for the same blockDim, two barriers.  Every thread contributes v and gets the sum;
// `scratch` holds at least 32 floats.  blockDim is a multiple of 32.
__device__ inline float block_sum(float v, float* scratch) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  if (lane == 0) scratch[wid] = v;
  __syncthreads();
  float r = lane < nw ? scratch[lane] : 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xFFFFFFFFu, r, o);
  __syncthreads();
  return r;
}
__device__ inline float block_max(float v, float* scratch) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
  if (lane == 0) scratch[wid] = v;
  __syncthreads();
  float r = lane < nw ? scratch[lane] : -INFINITY;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) r = fmaxf(r, __shfl_xor_sync(0xFFFFFFFFu, r, o));
  __syncthreads();
  return r;
}

// The value head's input of one environment, u = [emb(current) | mean of the valid candidates' emb] (2 H floats; H a
// multiple of 4), by all threads: part p of blockDim / (H / 4) adds candidates p, p + P, ... in order, four columns per
// thread, the parts in order.  scratch: 4 blockDim floats.  Returns the number of valid candidates; ends with a barrier.
__device__ inline float value_input(const float* __restrict__ emb, int32_t cur, int32_t C, const uint8_t* __restrict__ mk, int A,
                                    int H, float* u, float* scratch) {
  const int nt = blockDim.x, tid = threadIdx.x, HV = H >> 2, P = nt / HV, cv = tid % HV, p = tid / HV;
  const int n = min(C, A);
  const bool wide = (reinterpret_cast<uintptr_t>(emb) & 15) == 0;      // (the caller's buffer: any 4-byte boundary)
  float cnt = 0.f;
  for (int a = tid; a < n; a += nt) cnt += mk[a] ? 1.f : 0.f;
  const float nv = block_sum(cnt, scratch);
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  if (p < P)
    for (int a = p; a < n; a += 4 * P) {
      float4 v[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        v[t] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (a + t * P < n && mk[a + t * P]) {
          const float* r = emb + size_t(cur + 1 + a + t * P) * H + 4 * cv;
          v[t] = wide ? *reinterpret_cast<const float4*>(r) : make_float4(r[0], r[1], r[2], r[3]);
        }
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) { s.x += v[t].x; s.y += v[t].y; s.z += v[t].z; s.w += v[t].w; }
    }
  if (p < P) *reinterpret_cast<float4*>(scratch + size_t(p) * H + 4 * cv) = s;
  __syncthreads();
  for (int c = tid; c < H; c += nt) {
    float t = 0.f;
    for (int q = 0; q < P; ++q) t += scratch[q * H + c];
    u[c] = emb[size_t(cur) * H + c];
    u[H + c] = nv > 0.f ? t / nv : 0.f;
  }
  __syncthreads();
  return nv;
}

}  // namespace heads
}  // namespace xrl
