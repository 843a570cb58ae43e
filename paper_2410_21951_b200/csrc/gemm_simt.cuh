// Plain FMA matrix products C[m,n] = sum_k A[m,k] * W[n,k] with fused epilogues.
// This is the arithmetic of the fp32 model type (no tensor-core rounding); the
// bf16 model type uses the tensor-core kernels and only falls back to this
// file for shapes those do not cover.
#pragma once
#include "common.cuh"

namespace vadusa {

// ---- epilogues: called with the fp32 accumulator, one element at a time (operator()) or
// four consecutive features of one token at a time (vec4; n is a multiple of 4) ----------

// q/k/v projection (verify step, per layer): + bias, round to T; q goes to a dense buffer,
// k and v go straight to the paged cache at the node's slot (kv_row[m], written by the
// embedding kernel of the same pass; -1: the row is not scored).
template <typename T>
struct EpiQKV {
  const float* bias;
  T* q;
  T* pool;                      // KV pool of this layer
  const long long* kv_row;      // [M] element offset of the row's K slot for head 0
  long long kv_stride;          // elements from a K row to the V row of the same head
  int tile_elems;               // elements between heads: 64 * head_dim
  int head_dim, d;
  __device__ __forceinline__ long long kv_elem(long long row, int n) const {
    const int c = n - d, kv = c >= d, cc = c - kv * d, h = cc / head_dim;
    return row + kv * kv_stride + (long long)h * tile_elems + (cc - h * head_dim);
  }
  __device__ __forceinline__ void operator()(int, int m, int n, float acc) const {
    const T r = from_f<T>(acc + bias[n]);
    if (n < d) { q[(long long)m * d + n] = r; return; }
    const long long row = kv_row[m];
    if (row >= 0) pool[kv_elem(row, n)] = r;
  }
  __device__ __forceinline__ void vec4(int, int m, int n, float4 a) const {
    const float4 b = *reinterpret_cast<const float4*>(bias + n);
    if (n < d) { store4<T>(q + (long long)m * d + n, a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); return; }
    const long long row = kv_row[m];
    if (row >= 0) store4<T>(pool + kv_elem(row, n), a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
  }
  // CH consecutive tokens m .. m+count-1 of one feature n (all loads first, then the stores)
  template <int CH>
  __device__ __forceinline__ void col(int, int m, int n, const float* v, int count) const {
    const float b = bias[n];
    if (n < d) {
#pragma unroll
      for (int j = 0; j < CH; ++j)
        if (j < count) q[(long long)(m + j) * d + n] = from_f<T>(v[j] + b);
      return;
    }
    long long rows[CH];
#pragma unroll
    for (int j = 0; j < CH; ++j) rows[j] = j < count ? kv_row[m + j] : -1;
    const long long off = kv_elem(0, n);
#pragma unroll
    for (int j = 0; j < CH; ++j)
      if (rows[j] >= 0) pool[rows[j] + off] = from_f<T>(v[j] + b);
  }
};

// output projection / second feed-forward matrix: x += acc + bias (fp32 residual stream)
struct EpiResidual {
  const float* bias;
  float* x;
  int ld;
  __device__ __forceinline__ void operator()(int, int m, int n, float acc) const {
    x[(long long)m * ld + n] += acc + bias[n];
  }
  __device__ __forceinline__ void vec4(int, int m, int n, float4 a) const {
    const float4 b = *reinterpret_cast<const float4*>(bias + n);
    float4* p = reinterpret_cast<float4*>(x + (long long)m * ld + n);
    float4 v = *p;
    v.x += a.x + b.x; v.y += a.y + b.y; v.z += a.z + b.z; v.w += a.w + b.w;
    *p = v;
  }
  template <int CH>
  __device__ __forceinline__ void col(int, int m, int n, const float* v, int count) const {
    const float b = bias[n];
    float xv[CH];
#pragma unroll
    for (int j = 0; j < CH; ++j) xv[j] = j < count ? x[(long long)(m + j) * ld + n] : 0.f;
#pragma unroll
    for (int j = 0; j < CH; ++j)
      if (j < count) x[(long long)(m + j) * ld + n] = xv[j] + (v[j] + b);
  }
};

// EpiResidual that also leaves, per row and group of 128 features, the mean and the sum of squared
// deviations of the updated residual stream (the LayerNorm-fused product reads them).  vec4 must be
// called by all 32 lanes of a warp with the same row m and n = (a multiple of 128) + 4 * lane.
struct EpiResidualStats {
  const float* bias;
  float* x;
  int ld;
  float2* stats;          // [rows][ld / 128]
  __device__ __forceinline__ void operator()(int, int m, int n, float acc) const {
    x[(long long)m * ld + n] += acc + bias[n];
  }
  __device__ __forceinline__ void vec4(int, int m, int n, float4 a) const {
    const float4 b = *reinterpret_cast<const float4*>(bias + n);
    float4* p = reinterpret_cast<float4*>(x + (long long)m * ld + n);
    float4 v = *p;
    v.x += a.x + b.x; v.y += a.y + b.y; v.z += a.z + b.z; v.w += a.w + b.w;
    *p = v;
    float s = (v.x + v.y) + (v.z + v.w);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float mu = s * (1.0f / 128.0f);
    const float d0 = v.x - mu, d1 = v.y - mu, d2 = v.z - mu, d3 = v.w - mu;
    float q = (d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    if ((threadIdx.x & 31) == 0) stats[(long long)m * (ld >> 7) + (n >> 7)] = make_float2(mu, q);
  }
  template <int CH>
  __device__ __forceinline__ void col(int z, int m, int n, const float* v, int count) const {
    EpiResidual{bias, x, ld}.template col<CH>(z, m, n, v, count);     // no statistics on this path
  }
};

// first feed-forward matrix: relu(acc + bias) rounded to T
template <typename T>
struct EpiRelu {
  const float* bias;
  T* out;
  int ld;
  __device__ __forceinline__ void operator()(int, int m, int n, float acc) const {
    out[(long long)m * ld + n] = from_f<T>(fmaxf(acc + bias[n], 0.f));
  }
  __device__ __forceinline__ void vec4(int, int m, int n, float4 a) const {
    const float4 b = *reinterpret_cast<const float4*>(bias + n);
    store4<T>(out + (long long)m * ld + n, fmaxf(a.x + b.x, 0.f), fmaxf(a.y + b.y, 0.f), fmaxf(a.z + b.z, 0.f),
              fmaxf(a.w + b.w, 0.f));
  }
  template <int CH>
  __device__ __forceinline__ void col(int, int m, int n, const float* v, int count) const {
    const float b = bias[n];
#pragma unroll
    for (int j = 0; j < CH; ++j)
      if (j < count) out[(long long)(m + j) * ld + n] = from_f<T>(fmaxf(v[j] + b, 0.f));
  }
};

// vocabulary heads: fp32 logits; z selects the draft head
struct EpiLogits {
  float* out;
  int ld;
  long long z_stride;
  __device__ __forceinline__ void operator()(int z, int m, int n, float acc) const {
    out[z * z_stride + (long long)m * ld + n] = acc;
  }
  __device__ __forceinline__ void vec4(int z, int m, int n, float4 a) const {
    *reinterpret_cast<float4*>(out + z * z_stride + (long long)m * ld + n) = a;
  }
  template <int CH>
  __device__ __forceinline__ void col(int z, int m, int n, const float* v, int count) const {
#pragma unroll
    for (int j = 0; j < CH; ++j)
      if (j < count) out[z * z_stride + (long long)(m + j) * ld + n] = v[j];
  }
};

// draft residual block (Sec. III-A.1): z = h + SiLU(acc + bias), rounded to T; z selects the head
template <typename T>
struct EpiDraftHidden {
  const float* bias;     // [heads][d]
  const T* h;            // [batch][d]
  T* out;                // [heads][batch][d]
  int d, batch;
  __device__ __forceinline__ void operator()(int z, int m, int n, float acc) const {
    const float t = acc + bias[z * d + n];
    const float s = t / (1.0f + expf(-t));
    out[((long long)z * batch + m) * d + n] = from_f<T>(to_f<T>(h[(long long)m * d + n]) + s);
  }
};

// the same with the heads' matrices stacked along the feature axis: n = head * d + column
template <typename T>
struct EpiDraftHiddenFlat {
  const float* bias;     // [heads * d]
  const T* h;            // [batch][d]
  T* out;                // [heads][batch][d]
  int d, batch;
  __device__ __forceinline__ void operator()(int, int m, int n, float acc) const {
    const int head = n / d, col = n - head * d;
    const float t = acc + bias[n];
    const float s = t / (1.0f + expf(-t));
    out[((long long)head * batch + m) * d + col] = from_f<T>(to_f<T>(h[(long long)m * d + col]) + s);
  }
  __device__ __forceinline__ void vec4(int z, int m, int n, float4 a) const {
    (*this)(z, m, n, a.x); (*this)(z, m, n + 1, a.y); (*this)(z, m, n + 2, a.z); (*this)(z, m, n + 3, a.w);
  }
  template <int CH>
  __device__ __forceinline__ void col(int z, int m, int n, const float* v, int count) const {
#pragma unroll
    for (int j = 0; j < CH; ++j)
      if (j < count) (*this)(z, m + j, n, v[j]);
  }
};

// ---- kernels ----------------------------------------------------------------------
// LayerNorm of the fp32 rows that make the operand of a product (few-token kernel only).
struct RowNorm {
  const float* g;        // [K] gain (null: the operand is used as it is)
  const float* b;        // [K] shift
  float* y;              // if not null: the blocks of the first features also store the normalised rows ([M][K])
  float eps;
};

constexpr int kFewTokens = 128;          // tokens up to which the few-token kernel serves
constexpr int kFewNormK = 512;           // longest row it normalises itself (four float4 per lane and token)

// Four consecutive elements as floats; beyond the end: zeros.
template <typename T> __device__ __forceinline__ float4 ld4(const T* p, bool in);
template <> __device__ __forceinline__ float4 ld4<float>(const float* p, bool in) {
  return in ? *reinterpret_cast<const float4*>(p) : make_float4(0.f, 0.f, 0.f, 0.f);
}
template <> __device__ __forceinline__ float4 ld4<bf16>(const bf16* p, bool in) {
  if (!in) return make_float4(0.f, 0.f, 0.f, 0.f);
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                     __uint_as_float(v.y & 0xffff0000u));
}

// Few tokens (up to kFewTokens): a warp makes 4 tokens x 4 features, its lanes take K in pieces of 4 and the 16 sums meet in
// one butterfly of 16 shuffles.  Nothing goes through shared memory and no barrier is in the way: at these sizes a launch
// is bound by the latency of its loads (the 64 x 64 tile kernel walked K in steps of 16 behind two barriers each, 4 to 18
// blocks on the device: 18 us at K = 256, 60 us at K = 1024 against 3 and 4 us here, 16 tokens of the fp32 model).  A
// warp holds all of its four rows between its lanes, so LayerNorm needs no kernel of its own: the statistics are eight warp
// sums.  Weights of the first 512 columns are fetched before the upstream kernel has finished.
// Block: 4 warps, `mw` (1, 2 or 4) of them along the tokens, the others along the features.
// grid = (ceil(N / (16 / mw)), ceil(M / (4 mw)), batches).  K a multiple of 4.
template <typename T, typename Epi, bool LN>
__global__ void __launch_bounds__(128) gemm_few_kernel(const T* A, const T* __restrict__ W, int M, int N, int K, long long a_z,
                                                       long long w_z, int mw, Epi epi, RowNorm rn) {
  const int z = blockIdx.z, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  A += z * a_z; W += z * w_z;
  const int nw = 4 / mw;
  const int m0 = (blockIdx.y * mw + warp % mw) * 4, n0 = (blockIdx.x * nw + warp / mw) * 4;
  constexpr int G = 4;                                   // pieces of 128 columns per group
  float4 w[G][4];
#pragma unroll
  for (int c = 0; c < G; ++c)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = 128 * c + 4 * lane;
      w[c][j] = ld4<T>(W + (long long)(n0 + j) * K + k, k < K && n0 + j < N);
    }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (m0 >= M || n0 >= N) return;
  float acc[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) acc[i] = 0.f;
  auto mac = [&](const float4* x, const float4* ww) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float t = acc[4 * i + j];
        t = fmaf(x[i].x, ww[j].x, t); t = fmaf(x[i].y, ww[j].y, t);
        t = fmaf(x[i].z, ww[j].z, t); t = fmaf(x[i].w, ww[j].w, t);
        acc[4 * i + j] = t;
      }
  };
  if constexpr (LN) {
    float4 x[G][4];
    float s[4] = {0.f, 0.f, 0.f, 0.f}, q[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < G; ++c)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int k = 128 * c + 4 * lane;
        x[c][i] = ld4<T>(A + (long long)(m0 + i) * K + k, k < K && m0 + i < M);
      }
    float4 g[G], b[G];
#pragma unroll
    for (int c = 0; c < G; ++c) {
      const int k = 128 * c + 4 * lane;
      g[c] = ld4<float>(rn.g + k, k < K); b[c] = ld4<float>(rn.b + k, k < K);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
      for (int c = 0; c < G; ++c) s[i] += (x[c][i].x + x[c][i].y) + (x[c][i].z + x[c][i].w);
      s[i] = warp_sum(s[i]) / (float)K;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
      for (int c = 0; c < G; ++c) {
        if (128 * c + 4 * lane >= K) continue;
        const float d0 = x[c][i].x - s[i], d1 = x[c][i].y - s[i], d2 = x[c][i].z - s[i], d3 = x[c][i].w - s[i];
        q[i] += (d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3);
      }
      q[i] = 1.0f / sqrtf(warp_sum(q[i]) / (float)K + rn.eps);
    }
#pragma unroll
    for (int c = 0; c < G; ++c) {
      if (128 * c >= K) break;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float4& v = x[c][i];
        v = make_float4((v.x - s[i]) * q[i] * g[c].x + b[c].x, (v.y - s[i]) * q[i] * g[c].y + b[c].y,
                        (v.z - s[i]) * q[i] * g[c].z + b[c].z, (v.w - s[i]) * q[i] * g[c].w + b[c].w);
        const int k = 128 * c + 4 * lane;
        if (rn.y && n0 == 0 && k < K && m0 + i < M) *reinterpret_cast<float4*>(rn.y + (long long)(m0 + i) * K + k) = v;
      }
      mac(x[c], w[c]);                                   // (beyond K the weights are zero)
    }
  } else {
    for (int k0 = 0;;) {
      float4 x[G][4];
#pragma unroll
      for (int c = 0; c < G; ++c)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int k = k0 + 128 * c + 4 * lane;
          x[c][i] = ld4<T>(A + (long long)(m0 + i) * K + k, k < K && m0 + i < M);
        }
#pragma unroll
      for (int c = 0; c < G; ++c) mac(x[c], w[c]);
      k0 += 128 * G;
      if (k0 >= K) break;
#pragma unroll
      for (int c = 0; c < G; ++c)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int k = k0 + 128 * c + 4 * lane;
          w[c][j] = ld4<T>(W + (long long)(n0 + j) * K + k, k < K && n0 + j < N);
        }
    }
  }
  // sums over the lanes; lane l ends with value l >> 1 (token (l >> 3), feature (l >> 1) & 3)
  float r8[8], r4[4], r2[2], r1;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float keep = (lane & 16) ? acc[i + 8] : acc[i], give = (lane & 16) ? acc[i] : acc[i + 8];
    r8[i] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float keep = (lane & 8) ? r8[i + 4] : r8[i], give = (lane & 8) ? r8[i] : r8[i + 4];
    r4[i] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float keep = (lane & 4) ? r4[i + 2] : r4[i], give = (lane & 4) ? r4[i] : r4[i + 2];
    r2[i] = keep + __shfl_xor_sync(0xffffffffu, give, 4);
  }
  {
    const float keep = (lane & 2) ? r2[1] : r2[0], give = (lane & 2) ? r2[0] : r2[1];
    r1 = keep + __shfl_xor_sync(0xffffffffu, give, 2);
  }
  r1 += __shfl_xor_sync(0xffffffffu, r1, 1);
  const int m = m0 + (lane >> 3), n = n0 + ((lane >> 1) & 3);
  if (!(lane & 1) && m < M && n < N) epi(z, m, n, r1);
}

// Many tokens: 64x64 tile, K step 16, 256 threads, 4x4 outputs per thread.  K must be a multiple of 16.
// grid = (ceil(N/64), ceil(M/64), batches); A and W advance by a_z / w_z elements per batch.  Two shared-memory buffers: the
// next step's operands are on their way while a step is multiplied, one barrier per step.
template <typename T, typename Epi>
__global__ void __launch_bounds__(256) gemm_simt_kernel(const T* A, const T* __restrict__ W,
                                                        int M, int N, int K, long long a_z, long long w_z, Epi epi) {
  __shared__ float As[2][16][64 + 4];
  __shared__ float Ws[2][16][64 + 4];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int z = blockIdx.z;
  A += z * a_z; W += z * w_z;
  const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int lr = threadIdx.x >> 2, lk = (threadIdx.x & 3) * 4;   // loader: row 0..63, k offset 0,4,8,12
  const T* ap = A + (long long)(m0 + lr) * K + lk;
  const T* wp = W + (long long)(n0 + lr) * K + lk;
  const bool am = m0 + lr < M, wn = n0 + lr < N;
  float acc[4][4] = {};
  float4 a4 = ld4<T>(ap, am), w4 = ld4<T>(wp, wn);
  int buf = 0;
  for (int k0 = 0; k0 < K; k0 += 16, buf ^= 1) {
    As[buf][lk][lr] = a4.x; As[buf][lk + 1][lr] = a4.y; As[buf][lk + 2][lr] = a4.z; As[buf][lk + 3][lr] = a4.w;
    Ws[buf][lk][lr] = w4.x; Ws[buf][lk + 1][lr] = w4.y; Ws[buf][lk + 2][lr] = w4.z; Ws[buf][lk + 3][lr] = w4.w;
    __syncthreads();
    const bool more = k0 + 16 < K;
    a4 = ld4<T>(ap + k0 + 16, am && more);
    w4 = ld4<T>(wp + k0 + 16, wn && more);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float4 a = *reinterpret_cast<const float4*>(&As[buf][k][ty * 4]), w = *reinterpret_cast<const float4*>(&Ws[buf][k][tx * 4]);
      const float av[4] = {a.x, a.y, a.z, a.w}, wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], wv[j], acc[i][j]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + ty * 4 + i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx * 4 + j;
      if (n < N) epi(z, m, n, acc[i][j]);
    }
  }
}

}  // namespace vadusa
