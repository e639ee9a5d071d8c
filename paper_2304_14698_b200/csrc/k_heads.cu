// Per-graph readout and global update (paper Eq. 8), the policy and value heads with
// invalid-action masking and No-Op (Sections 3.3.2, 3.3.3), and the categorical draw.
// Every reduction runs in a fixed order (no floating-point atomics), so results are
// reproducible run to run.
#include <algorithm>

#include "xrl_heads.cuh"

namespace xrl {

using namespace heads;

namespace {

constexpr int kRoThreads = 256;

// ---- readout, stage 1: column sums of one chunk of consecutive rows of one graph -------------
template <typename T>
__global__ void __launch_bounds__(kRoThreads)
k_readout(const T* __restrict__ h, const int32_t* __restrict__ chunk_row0,
          const int32_t* __restrict__ chunk_row1, int32_t chunk_begin, float* __restrict__ partial,
          int H, int32_t win_base, const int32_t* __restrict__ remap) {
  enter();
  constexpr int VEC = VecOf<T>::N;
  extern __shared__ float red[];                 // [RG][H]
  const int NV = H / VEC;
  const int RG = kRoThreads / NV;                // row groups working in parallel
  const int32_t chunk = chunk_begin + blockIdx.x;
  const int32_t r0 = chunk_row0[chunk], r1 = chunk_row1[chunk];
  const int vi = threadIdx.x % NV, rg = threadIdx.x / NV;
  float acc[VEC];
#pragma unroll
  for (int t = 0; t < VEC; ++t) acc[t] = 0.f;
  if (rg < RG) {
    int32_t r = r0 + rg;
    for (; r + 3 * RG < r1; r += 4 * RG) {
      float f[4][VEC];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        load_vec(h + size_t(remap ? __ldg(remap + r + u * RG) : r + u * RG - win_base) * H + vi * VEC, f[u]);
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int t = 0; t < VEC; ++t) acc[t] += f[u][t];
    }
    for (; r < r1; r += RG) {
      float f[VEC];
      load_vec(h + size_t(remap ? __ldg(remap + r) : r - win_base) * H + vi * VEC, f);
#pragma unroll
      for (int t = 0; t < VEC; ++t) acc[t] += f[t];
    }
#pragma unroll
    for (int t = 0; t < VEC; ++t) red[rg * H + vi * VEC + t] = acc[t];
  }
  __syncthreads();
  for (int c = threadIdx.x; c < H; c += kRoThreads) {
    float s = 0.f;
    for (int g = 0; g < RG; ++g) s += red[g * H + c];
    partial[size_t(chunk) * H + c] = s;
  }
}

// ---- Eq. 8: emb_g = ReLU(Wg^T [ sum of the graph's partial sums | g0_g ] + bg), GP graphs per CTA -------------------
// Where a graph's partial sums lie: BLOCKS = false: rows off[g] .. off[g + 1] - 1 of `partial` (readout chunks).
// BLOCKS = true, after the aggregate kernel fused with the readout: off = node offsets; the partial of the block in which
// the graph starts (if it does not start at the block's first row), then the partials of the following blocks whose first
// row belongs to the graph.  The rows are added in P interleaved parts, four columns per thread, and the parts in order: a
// fixed order for a given launch shape.  U_out (optional): the sums with g0 behind them, [B x (H + Dg)].
template <int GP, bool BLOCKS>
__global__ void __launch_bounds__(kThreads)
k_global_update(const float* __restrict__ partial, const int32_t* __restrict__ off, int32_t nblocks, int bshift,
                const float* __restrict__ g0, const float* __restrict__ Wg, const float* __restrict__ bg,
                float* __restrict__ emb, float* __restrict__ U_out, int H, int Dg, int B) {
  enter();
  extern __shared__ __align__(16) float u[];     // [GP][xs], then scratch
  const int xs = row_stride(H + Dg), nt = blockDim.x, tid = threadIdx.x;
  int32_t* filled = reinterpret_cast<int32_t*>(u + GP * xs);       // [GP] parts of each graph that hold any row
  float* part = u + GP * xs + row_stride(GP);
  const int32_t first = blockIdx.x * GP;
  const int HV = H >> 2, NG = nt / HV, P = NG >= GP ? NG / GP : 1;
  const int cv = tid % HV, grp = tid / HV;
  auto range = [&](int32_t g, int32_t& b0, int32_t& b1) {         // rows b0 .. b1 of `partial`
    const int32_t start = off[g], end = off[g + 1];
    if (BLOCKS) {
      b0 = 0; b1 = -1;
      if (end > start) {
        b0 = start >> bshift;
        if (start & ((1 << bshift) - 1)) ++b0;
        b1 = (end - 1) >> bshift;
      }
    } else {
      b0 = start; b1 = end - 1;
    }
  };
  if (grp < NG)
    for (int t = grp; t < GP * P; t += NG) {
      const int gl = t / P, p = t - gl * P;
      if (first + gl >= B) break;
      int32_t b0, b1;
      range(first + gl, b0, b1);
      if (p == 0 && cv == 0) filled[gl] = min(P, max(0, b1 - b0 + 1));
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int32_t b = b0 + p; b <= b1; b += 8 * P) {
        float4 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (b + q * P <= b1) v[q] = *reinterpret_cast<const float4*>(partial + size_t(b + q * P) * H + 4 * cv);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) { s.x += v[q].x; s.y += v[q].y; s.z += v[q].z; s.w += v[q].w; }
      }
      *reinterpret_cast<float4*>(part + size_t(t) * H + 4 * cv) = s;
    }
  __syncthreads();
  for (int i = tid; i < GP * xs; i += nt) {
    const int gl = i / xs, c = i - gl * xs;
    const int32_t g = first + gl;
    float v = 0.f;
    if (g < B && c < H) {
      if (BLOCKS) {
        const int32_t start = off[g];
        if (off[g + 1] > start && (start & ((1 << bshift) - 1))) v = partial[size_t(nblocks + g) * H + c];
      }
      for (int q = 0, n = filled[gl]; q < n; ++q) v += part[size_t(gl * P + q) * H + c];
    } else if (g < B && c < H + Dg) {
      v = g0 ? g0[size_t(g) * Dg + (c - H)] : 0.f;
    }
    u[i] = v;
    if (U_out != nullptr && g < B && c < H + Dg) U_out[size_t(g) * (H + Dg) + c] = v;
  }
  __syncthreads();
  dense_rows<GP>(u, xs, H + Dg, Wg, H, H, bg, part, [&](int g, int c, float y) {
    if (first + g < B) emb[size_t(first + g) * H + c] = fmaxf(y, 0.f);
  });
}

// The rest of a head's MLP behind its first layer: y1 = ReLU(W1^T x + b1) is given (hid floats in shared memory, on a
// 16-byte boundary; y2: hid2 floats); all threads return the result.
__device__ float mlp_tail(const float* y1, const Mlp& m, float* scratch) {
  float contrib = 0.f;
  if (m.hid2 <= 0) {
    for (int c = threadIdx.x; c < m.hid; c += blockDim.x) contrib += y1[c] * m.w2[c];
  } else {
    dense_rows<1>(y1, 0, m.hid, m.Wh, m.hid2, m.hid2, m.bh, scratch,
                  [&](int, int c, float y) { contrib += fmaxf(y, 0.f) * m.w2[c]; });
  }
  return block_sum(contrib, scratch) + m.b2[0];
}

// ---- policy scores of all graphs and the value head's first layer, in one launch ----------------------------------
// CTAs [0, policy_ctas): policy MLP of GP graphs each, one scalar per graph.  y1_out / y2_out (optional): its hidden
// activations.  CTAs policy_ctas + e * VC + ch compute chunk ch (hid / VC columns) of the value head's first layer for
// environment e, y1v[e] = ReLU(W1^T [emb(current) | mean of the valid candidates' emb] + b1), the candidate mean taken
// inside the CTA: the 2H x hid weights are then read by VC CTAs instead of by the one CTA of the environment.
template <int GP>
__global__ void __launch_bounds__(kThreads)
k_policy_value_hidden(const float* __restrict__ emb, const Mlp pm, float* __restrict__ logit, int H, int32_t B,
                      int policy_ctas, float* __restrict__ y1_out, float* __restrict__ y2_out,
                      const int32_t* __restrict__ env_off, const uint8_t* __restrict__ mask, int A, const Mlp vm,
                      float* __restrict__ y1v, int VC, float* __restrict__ u_out) {
  enter();
  extern __shared__ __align__(16) float sm[];
  const int nt = blockDim.x, tid = threadIdx.x;
  if (int(blockIdx.x) < policy_ctas) {
    const int xs = row_stride(H), ys = row_stride(pm.hid), zs = row_stride(pm.hid2);
    float* x = sm;                               // [GP][xs]
    float* y1 = x + GP * xs;                     // [GP][ys]
    float* y2 = y1 + GP * ys;                    // [GP][zs]
    float* part = y2 + GP * zs;                  // [GP * nt]
    const int32_t first = blockIdx.x * GP;
    for (int i = tid; i < GP * xs; i += nt) {
      const int g = i / xs, c = i - g * xs;
      x[i] = first + g < B && c < H ? emb[size_t(first + g) * H + c] : 0.f;
    }
    __syncthreads();
    dense_rows<GP>(x, xs, H, pm.W1, pm.hid, pm.hid, pm.b1, part, [&](int g, int c, float y) {
      y1[g * ys + c] = fmaxf(y, 0.f);
      if (y1_out != nullptr && first + g < B) y1_out[size_t(first + g) * pm.hid + c] = fmaxf(y, 0.f);
    });
    const float* last = y1;
    int ls = ys, width = pm.hid;
    if (pm.hid2 > 0) {
      dense_rows<GP>(y1, ys, pm.hid, pm.Wh, pm.hid2, pm.hid2, pm.bh, part, [&](int g, int c, float y) {
        y2[g * zs + c] = fmaxf(y, 0.f);
        if (y2_out != nullptr && first + g < B) y2_out[size_t(first + g) * pm.hid2 + c] = fmaxf(y, 0.f);
      });
      last = y2; ls = zs; width = pm.hid2;
    }
    const int lane = tid & 31, warp = tid >> 5;  // a warp per graph
    if (warp < GP && first + warp < B) {
      float v = 0.f;
      for (int c = lane; c < width; c += 32) v = fmaf(last[warp * ls + c], pm.w2[c], v);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
      if (lane == 0) logit[first + warp] = v + pm.b2[0];
    }
    return;
  }
  float* u = sm;                                 // [2H]
  float* scratch = sm + 2 * H;                   // [4 blockDim]
  const int32_t e = (int32_t(blockIdx.x) - policy_ctas) / VC, ch = (int32_t(blockIdx.x) - policy_ctas) % VC;
  const int32_t cur = env_off[e];
  value_input(emb, cur, env_off[e + 1] - cur - 1, mask + size_t(e) * A, A, H, u, scratch);
  if (u_out != nullptr && ch == 0)
    for (int c = tid; c < 2 * H; c += nt) u_out[size_t(e) * 2 * H + c] = u[c];
  const int CW = (vm.hid + VC - 1) / VC, c_lo = ch * CW, ncols = min(CW, vm.hid - c_lo);
  if (ncols > 0)
    dense_rows<1>(u, 0, 2 * H, vm.W1 + c_lo, vm.hid, ncols, vm.b1 + c_lo, scratch,
                  [&](int, int c, float y) { y1v[size_t(e) * vm.hid + c_lo + c] = fmaxf(y, 0.f); });
}

// ---- Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) -----------------------------------------
struct U4 { uint32_t x, y, z, w; };
__device__ U4 philox4x32_10(uint32_t k0, uint32_t k1, U4 c) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = U4{hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0};
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c;
}

__device__ unsigned long long block_sum_u64(unsigned long long v, unsigned long long* scratch) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  if (lane == 0) scratch[wid] = v;
  __syncthreads();
  unsigned long long r = lane < nw ? scratch[lane] : 0ull;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xFFFFFFFFu, r, o);
  __syncthreads();
  return r;
}

// Categorical draw from fp32 probabilities p[0..A1) with integer arithmetic only.
// scratch: blockDim.x + 1 unsigned 64-bit words.  Every thread returns the action.
__device__ int32_t sample_row(const float* __restrict__ p, int A1, uint64_t seed, uint64_t step,
                              uint32_t env, unsigned long long* scratch) {
  const int tid = threadIdx.x, nt = blockDim.x;
  // contiguous slice per thread so that prefix order = index order
  const int per = (A1 + nt - 1) / nt;
  const int a0 = min(A1, tid * per), a1 = min(A1, a0 + per);
  unsigned long long mine = 0;
  for (int a = a0; a < a1; ++a) mine += (unsigned long long)floorf(p[a] * 4294967296.0f);
  const unsigned long long Q = block_sum_u64(mine, scratch);
  if (Q == 0) return A1 - 1;
  const U4 r = philox4x32_10(uint32_t(seed), uint32_t(seed >> 32),
                             U4{env, uint32_t(step), uint32_t(step >> 32), 0u});
  const unsigned long long r64 = (unsigned long long)r.x | ((unsigned long long)r.y << 32);
  const unsigned long long t = __umul64hi(r64, Q);
  // exclusive prefix of the per-thread totals: scan inside each warp, then over the warp totals
  // (integer sums: any association gives the same result)
  {
    const int lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
    unsigned long long incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += y;
    }
    __syncthreads();                            // scratch is free again after block_sum_u64
    if (lane == 31) scratch[wid] = incl;
    __syncthreads();
    unsigned long long wbase = 0;
    for (int w = 0; w < wid && w < nw; ++w) wbase += scratch[w];
    __syncthreads();
    scratch[tid] = wbase + incl - mine;
    if (tid == 0) scratch[nt] = (unsigned long long)(A1 - 1);
  }
  __syncthreads();
  unsigned long long run = scratch[tid];
  if (run <= t && t < run + mine) {              // exactly one thread owns t
    for (int a = a0; a < a1; ++a) {
      run += (unsigned long long)floorf(p[a] * 4294967296.0f);
      if (run > t) { scratch[nt] = (unsigned long long)a; break; }
    }
  }
  __syncthreads();
  const int32_t act = int32_t(scratch[nt]);
  __syncthreads();
  return act;
}

// ---- per environment: masked softmax, the value MLP behind its first layer, optional draw ----------------------------
// A thread keeps its entries' scores in registers up to kKeep per thread; the rest is read again.
constexpr int kKeep = 2;
__global__ void __launch_bounds__(1024)
k_env_policy(const float* __restrict__ logit, const int32_t* __restrict__ env_off, const uint8_t* __restrict__ mask,
             const Mlp vmlp, float* __restrict__ probs, float* __restrict__ value, int32_t* __restrict__ action, int A,
             uint64_t seed, uint64_t step, int32_t* status, const float* __restrict__ y1v) {
  enter();
  extern __shared__ __align__(16) unsigned long long sm64[];   // [nt + 2] u64, then floats
  const int nt = blockDim.x, tid = threadIdx.x;
  float* scratch = reinterpret_cast<float*>(sm64 + nt + 2);   // [nt]
  float* y1 = scratch + nt;                                   // [hid]
  const int32_t e = blockIdx.x;
  const int32_t cur = env_off[e];
  const int32_t C = env_off[e + 1] - cur - 1;
  const uint8_t* mk = mask + size_t(e) * A;
  float* pr = probs + size_t(e) * (A + 1);
  // the value head's first layer is asked for before the softmax needs its barriers
  for (int c = tid; c < vmlp.hid; c += nt) y1[c] = __ldg(y1v + size_t(e) * vmlp.hid + c);

  // masked softmax over the valid candidates and No-Op (index A, scored by the current graph)
  auto score = [&](int a) -> float {             // -inf: excluded
    if (a == A) return logit[cur];
    return a < C && mk[a] ? logit[cur + 1 + a] : -INFINITY;
  };
  float kept[kKeep];
  float mx = -INFINITY;
#pragma unroll
  for (int t = 0; t < kKeep; ++t) {
    const int a = tid + t * nt;
    kept[t] = -INFINITY;
    if (a <= A) {
      if (a < A && a >= C && mk[a]) raise(status, XRL_ERR_INVALID_ARG);
      kept[t] = score(a);
      mx = fmaxf(mx, kept[t]);
    }
  }
  for (int a = tid + kKeep * nt; a <= A; a += nt) {
    if (a < A && a >= C && mk[a]) raise(status, XRL_ERR_INVALID_ARG);
    mx = fmaxf(mx, score(a));
  }
  mx = block_max(mx, scratch);
  float se = 0.f;
  bool drop[kKeep];                              // an excluded entry is exactly 0 whatever the maximum is
#pragma unroll
  for (int t = 0; t < kKeep; ++t) {
    const int a = tid + t * nt;
    drop[t] = a > A || (a < A && !(a < C && mk[a]));
    kept[t] = drop[t] ? 0.f : expf(kept[t] - mx);
    se += kept[t];
  }
  for (int a = tid + kKeep * nt; a <= A; a += nt) {
    const bool valid = (a == A) || (a < C && mk[a]);
    const float ex = valid ? expf(score(a) - mx) : 0.f;
    pr[a] = ex;
    se += ex;
  }
  const float denom = block_sum(se, scratch);
#pragma unroll
  for (int t = 0; t < kKeep; ++t)
    if (tid + t * nt <= A) pr[tid + t * nt] = kept[t] / denom;
  for (int a = tid + kKeep * nt; a <= A; a += nt) pr[a] = pr[a] / denom;     // each thread rewrites its own entries

  const float v = mlp_tail(y1, vmlp, scratch);
  if (tid == 0) value[e] = v;

  if (action != nullptr) {
    __syncthreads();                              // probs of this row are written by this block
    const int32_t act = sample_row(pr, A + 1, seed, step, uint32_t(e), sm64);
    if (tid == 0) action[e] = act;
  }
}

__global__ void __launch_bounds__(1024)
k_sample(const float* __restrict__ probs, int A1, uint64_t seed, uint64_t step,
         int32_t* __restrict__ action) {
  enter();
  extern __shared__ unsigned long long sm64[];
  const int32_t e = blockIdx.x;
  const int32_t act = sample_row(probs + size_t(e) * A1, A1, seed, step, uint32_t(e), sm64);
  if (threadIdx.x == 0) action[e] = act;
}

// Seeded initial weights: element i of the blob is bound * u_i, u_i = (w >> 8) * 2^-23 - 1 in [-1, 1) with w the
// first word of Philox4x32-10(key = seed, counter = (i, 0, 0, 1)); every step is exact in fp32 except the one
// product, so any IEEE implementation gives the same bits.  (Counter word 3 = 1 keeps this stream apart from
// the action draws, which use 0.)
__global__ void k_init_weights(float* __restrict__ blob, int64_t first, int64_t count, float bound, uint32_t k0,
                               uint32_t k1) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= count) return;
  const uint64_t i = uint64_t(first + t);
  const U4 r = philox4x32_10(k0, k1, U4{uint32_t(i), uint32_t(i >> 32), 0u, 1u});
  const float u = __fsub_rn(__fmul_rn(float(r.x >> 8), 1.1920928955078125e-07f), 1.0f);
  blob[first + t] = __fmul_rn(bound, u);
}

__global__ void k_to_float_bf16(const bf16* __restrict__ src, float* __restrict__ dst, int64_t n) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = __bfloat162float(src[i]);
}

// dst = storage-type copy of src [rows x cols]; dst_t (optional) = its transpose [cols x rows]
template <typename T>
__global__ void k_round_weights(const float* __restrict__ src, T* __restrict__ dst,
                                T* __restrict__ dst_t, int rows, int cols) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= rows * cols) return;
  const int r = i / cols, c = i - r * cols;
  const T v = T(src[i]);
  dst[i] = v;
  if (dst_t != nullptr) dst_t[size_t(c) * rows + r] = v;
}

// Graphs per CTA: as few as leave every CTA an SM of its own (each then waits for its weights once, and every weight is
// loaded once for all of a CTA's graphs), at most 16, within the shared memory that `bytes(GP)` says.  Measured (Eq. 8 and
// the policy scores, hidden 256): 2,945 graphs 0.081 + 0.058 ms with a CTA of 256 threads per graph, 1,024 graphs 0.048 +
// 0.030 ms.
template <typename Bytes> int graphs_per_cta(int64_t B, Bytes bytes) {
  int gp = 1;
  while (gp < 16 && (B + gp - 1) / gp > kNumSMs && bytes(2 * gp) <= size_t(200) * 1024) gp <<= 1;
  return gp;
}

int pow2_threads(int want) {          // power of two in [32, 1024] (block_sum needs a power of two)
  int t = 32;
  while (t < want && t < 1024) t <<= 1;
  return t;
}

}  // namespace

int launch_readout(const Dims& d, const void* h, const int32_t* chunk_row0, const int32_t* chunk_row1,
                   int32_t chunk_begin, int32_t chunk_end, float* partial, int32_t win_base,
                   cudaStream_t st, const int32_t* remap) {
  const int n = chunk_end - chunk_begin;
  if (n <= 0) return 0;
  if (d.dtype == XRL_BF16) {
    const int RG = kRoThreads / (d.H / 8);
    launch(k_readout<bf16>, n, kRoThreads, sizeof(float) * size_t(RG) * d.H, st,
        static_cast<const bf16*>(h), chunk_row0, chunk_row1, chunk_begin, partial, d.H, win_base, remap);
  } else {
    const int RG = kRoThreads / (d.H / 4);
    launch(k_readout<float>, n, kRoThreads, sizeof(float) * size_t(RG) * d.H, st,
        static_cast<const float*>(h), chunk_row0, chunk_row1, chunk_begin, partial, d.H, win_base, remap);
  }
  return 1;
}

namespace {
template <int GP, bool BLOCKS>
int global_update(const Dims& d, const float* partial, const int32_t* off, int32_t nblocks, int shift, const float* g0,
                  const DevWeights& w, float* emb, float* U_out, int32_t B, size_t smem, cudaStream_t st, int nt = kThreads) {
  static bool attr[64] = {};
  if (smem > 48 * 1024 && !ensure_dynamic_smem(k_global_update<GP, BLOCKS>, 227 * 1024, attr)) return -1;
  launch(k_global_update<GP, BLOCKS>, (B + GP - 1) / GP, nt, smem, st, partial, off, nblocks, shift, g0, w.Wg, w.bg, emb,
                                                                         U_out, d.H, d.Dg, B);
  return 1;
}
template <bool BLOCKS>
int launch_update(const Dims& d, const float* partial, const int32_t* off, int32_t nblocks, int shift, const float* g0,
                  const DevWeights& w, float* emb, float* U_out, int32_t B, cudaStream_t st) {
  if (B <= 0) return 0;
  // rows of u, then scratch: the parts of the block sums (max(groups, GP) rows of H), the parts of the dense map
  auto bytes = [&](int gp) {
    const size_t rows = size_t(std::max(kThreads / (d.H / 4), gp)) * d.H, parts = size_t(gp) * kThreads;
    return sizeof(float) * (size_t(gp) * row_stride(d.H + d.Dg) + row_stride(gp) + std::max(rows, parts));
  };
  int gp = graphs_per_cta(B, bytes);
  // two graphs per CTA (up to two per SM) are slower than four, and than one each on fewer threads where W_g is small: 220
  // graphs, hidden 64 / 128 / 256 / 512: 5.4 / 7.4 / 12.6 / 32.9 us, four 5.2 / 6.8 / 11.5 / 27.9, one 4.3 / 6.2 / 12.2 / 36.8
  if (gp == 2) {
    if (d.H <= 128) return global_update<1, BLOCKS>(d, partial, off, nblocks, shift, g0, w, emb, U_out, B, bytes(1), st, 256);
    gp = 4;
  }
#define UPDATE_CASE(G_) case G_: return global_update<G_, BLOCKS>(d, partial, off, nblocks, shift, g0, w, emb, U_out, B, bytes(G_), st);
  switch (gp) { UPDATE_CASE(1) UPDATE_CASE(4) UPDATE_CASE(8) default: UPDATE_CASE(16) }
#undef UPDATE_CASE
}
template <int GP>
int policy_value(const Dims& d, const Mlp& pm, const Mlp& vm, const float* emb, float* logit, int32_t B, float* y1_out,
                 float* y2_out, const int32_t* env_off, const uint8_t* mask, int32_t num_envs, float* y1v, int VC, size_t smem,
                 cudaStream_t st, float* u_out) {
  static bool attr[64] = {};
  if (smem > 48 * 1024 && !ensure_dynamic_smem(k_policy_value_hidden<GP>, 227 * 1024, attr)) return -1;
  const int pc = (B + GP - 1) / GP;
  launch(k_policy_value_hidden<GP>, pc + num_envs * VC, kThreads, smem, st, emb, pm, logit, d.H, B, pc, y1_out, y2_out, env_off,
                                                                        mask, d.A, vm, y1v, VC, u_out);
  return 1;
}
}  // namespace

int launch_global_update(const Dims& d, const float* partial, const int32_t* graph_chunk_off,
                         const float* g0, const DevWeights& w, float* emb, int32_t B, cudaStream_t st, float* U_out) {
  return launch_update<false>(d, partial, graph_chunk_off, 0, 0, g0, w, emb, U_out, B, st);
}

int launch_global_update_blocks(const Dims& d, const float* partial, const int32_t* node_off, int32_t nblocks,
                                int block_shift, const float* g0, const DevWeights& w, float* emb, int32_t B,
                                cudaStream_t st, float* U_out) {
  return launch_update<true>(d, partial, node_off, nblocks, block_shift, g0, w, emb, U_out, B, st);
}

// Policy scores of all graphs (logit [B]; y1_out / y2_out optional) and, for num_envs > 0, the first layer of the value
// head (y1v [num_envs x Hm]; its input u_out [num_envs x 2 H] is optional).
int launch_policy_value_hidden(const Dims& d, const DevWeights& w, const float* emb, float* logit, int32_t B, float* y1_out,
                               float* y2_out, const int32_t* env_off, const uint8_t* mask, int32_t num_envs, float* y1v,
                               cudaStream_t st, float* u_out) {
  const Mlp pm{w.pW1, w.pb1, w.pWh, w.pbh, w.pw2, w.pb2, d.Hm, d.Hm2};
  const Mlp vm{w.vW1, w.vb1, w.vWh, w.vbh, w.vw2, w.vb2, d.Hm, d.Hm2};
  auto bytes = [&](int gp) {
    const size_t policy = size_t(gp) * (row_stride(d.H) + row_stride(d.Hm) + row_stride(d.Hm2) + kThreads);
    return sizeof(float) * std::max(policy, size_t(2 * d.H + 4 * kThreads));
  };
  const int gp = graphs_per_cta(B, bytes);
  // the value CTAs of an environment share its first layer: eight while they find SMs of their own beside the others'
  const int VC = num_envs <= 8 ? 8 : num_envs <= 32 ? 4 : num_envs <= 128 ? 2 : 1;
#define POLICY_CASE(G_) \
  case G_: return policy_value<G_>(d, pm, vm, emb, logit, B, y1_out, y2_out, env_off, mask, num_envs, y1v, VC, bytes(G_), st, u_out);
  switch (gp) { POLICY_CASE(1) POLICY_CASE(2) POLICY_CASE(4) POLICY_CASE(8) default: POLICY_CASE(16) }
#undef POLICY_CASE
}

int launch_heads(const Dims& d, const DevWeights& w, const float* emb, const int32_t* env_off,
                 const uint8_t* mask, int32_t B, int32_t num_envs, float* logit_ws, float* probs,
                 float* value, int32_t* action, uint64_t seed, uint64_t step, int32_t* status,
                 cudaStream_t st) {
  if (B <= 0 || num_envs <= 0) return 0;
  const Mlp vm{w.vW1, w.vb1, w.vWh, w.vbh, w.vw2, w.vb2, d.Hm, d.Hm2};
  float* y1v = logit_ws + B;                      // [num_envs x Hm], behind the per-graph logits
  if (launch_policy_value_hidden(d, w, emb, logit_ws, B, nullptr, nullptr, env_off, mask, num_envs, y1v, st) < 0) return -1;
  int want = std::max({d.A + 1, d.Hm, 256});      // enough threads to split the value head's dense map
  if (num_envs <= kNumSMs && d.Hm2 > 0) want = 1024;     // (an SM per environment: more parts, shorter chains)
  const int nt = pow2_threads(want);
  const size_t smem = sizeof(unsigned long long) * size_t(nt + 2) + sizeof(float) * size_t(nt + d.Hm);
  launch(k_env_policy, num_envs, nt, smem, st, logit_ws, env_off, mask, vm, probs, value, action, d.A, seed, step, status, y1v);
  return 2;
}

int launch_sample(const float* probs, int32_t num_envs, int32_t A1, uint64_t seed, uint64_t step,
                  int32_t* action, cudaStream_t st) {
  if (num_envs <= 0) return 0;
  const int nt = pow2_threads(A1);
  launch(k_sample, num_envs, nt, sizeof(unsigned long long) * size_t(nt + 1), st, probs, A1, seed, step,
                                                                              action);
  return 1;
}

int launch_init_weights(float* blob, int64_t first, int64_t count, float bound, uint64_t seed, cudaStream_t st) {
  if (count <= 0) return 0;
  k_init_weights<<<unsigned((count + 255) / 256), 256, 0, st>>>(blob, first, count, bound, uint32_t(seed),
                                                                uint32_t(seed >> 32));
  return 1;
}

int launch_to_float(const void* src, int dtype, float* dst, int64_t n, cudaStream_t st) {
  if (n <= 0) return 0;
  if (dtype == XRL_BF16) {
    k_to_float_bf16<<<unsigned((n + 255) / 256), 256, 0, st>>>(static_cast<const bf16*>(src), dst, n);
    return 1;
  }
  cudaMemcpyAsync(dst, src, sizeof(float) * size_t(n), cudaMemcpyDeviceToDevice, st);
  return 0;
}

int launch_round_weights(const float* src, void* dst, void* dst_t, int rows, int cols, int dtype,
                         cudaStream_t st) {
  const int n = rows * cols;
  if (dtype == XRL_BF16)
    k_round_weights<bf16><<<(n + 255) / 256, 256, 0, st>>>(src, static_cast<bf16*>(dst),
                                                          static_cast<bf16*>(dst_t), rows, cols);
  else
    k_round_weights<float><<<(n + 255) / 256, 256, 0, st>>>(src, static_cast<float*>(dst),
                                                           static_cast<float*>(dst_t), rows, cols);
  return 1;
}

}  // namespace xrl
