// Fitting of the draft heads with the base model frozen (paper Sec. II-A: the i-th draft head is supervised by
// a cross-entropy loss multiplied by lambda^i; Sec. III-A.2: heads trained with a fixed base model).  Not on
// the decoding path: fp32 master copies of the heads, fp32 results; after every step the heads in the weight blob are
// rewritten in the model dtype.
//
// The five products of a step run on the tensor cores with fp32 operands cut into three bf16 parts, a = a1 + a2 + a3
// (24 significant bits: each part is the rounded rest of the ones before), and the products a1 b1, a1 b2, a2 b1, a2 b2,
// a1 b3, a3 b1 summed in fp32; what is dropped is below 2^-26 of a product.  A tensor-core accumulation cuts its sum off
// where an fp32 addition rounds, an error that grows with the number of instructions behind one accumulator: the a1 b1
// products go round three accumulators and all the small ones into a fourth, which are added at the end (one accumulator for
// everything left six times the error of the fp32 FMA form in the updated weights; this leaves the same).  (Plain fp32 FMA tiles took 240 us per product
// at 512 tokens, 1.34 ms per step.)  The parts of an array lie behind one another, [part][head][row][column], written by
// whoever makes the array; each is read in its natural layout, whichever side of a product it is on: rows along K as a
// K-major operand, rows along the output as an MN-major one, so nothing is transposed.
#pragma once
#include "tc.cuh"

namespace vadusa {

constexpr int kFitTile = 128;                                    // rows and columns of an output tile
constexpr int kFitThreads = 512;
constexpr int kFitPart = kFitTile * 64 * 2;                      // one part of one operand for a 64-wide K step

template <int NA, int NB> struct FitCfg {
  static constexpr int kStageBytes = (NA + NB) * kFitPart;
  static constexpr int kStages = NA + NB > 4 ? 2 : 3;
  static constexpr int kSmem = kStages * kStageBytes + 1024 /*alignment*/ + 128 /*barriers*/;
};

// Shared-memory descriptor of an MN-major tile: 64-element columns (128 bytes, 128-byte swizzle) of 64 K rows each, the
// next 64 columns 8192 bytes on; 8 K rows are 1024 bytes.  Advancing 16 K rows adds 2048 bytes.
__device__ __forceinline__ uint64_t fit_desc_mn(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (512ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}

// C[r][c] = sum over k of A(r, k) B(c, k) per head; A and B in NA and NB parts (1: exact in bf16, or 3).
// AMN / BMN: the operand lies with its rows along K ([k][r]), else [r][k].  a_heads / b_heads: heads of the array (1: shared).
// grid = (ceil(C / 128), ceil(R / 128), heads), kFitThreads threads; warp roles as in gemm_tc_kernel, sixteen warps for the
// epilogue (a block has the SM to itself, and Adam's divisions and root are 130 instructions per weight).  A K step brings the parts of
// both operands once (up to 96 KB) and feeds up to 24 instructions from them: 64 bytes per cycle and SM from L2 at the full
// tensor rate, where separate passes over the pairs of parts would want 128.
template <int NA, int NB, bool AMN, bool BMN, typename Epi>
__global__ void __launch_bounds__(kFitThreads) fit_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                                                     int R, int C, int K, int a_heads, int b_heads, Epi epi, uint32_t* err) {
  using Cfg = FitCfg<NA, NB>;
  constexpr int S = Cfg::kStages;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bars = base + S * Cfg::kStageBytes;             // full[S], empty[S], accumulator, tmem holder
  const uint32_t full0 = bars, empty0 = bars + 8 * S, accum = bars + 16 * S, holder = accum + 8;
  volatile uint32_t* holder_ptr = reinterpret_cast<volatile uint32_t*>(smem_raw + (holder - smem_u32(smem_raw)));
  const int warp = warp_index(), lane = threadIdx.x & 31, head = blockIdx.z;
  const int c0 = blockIdx.x * kFitTile, r0 = blockIdx.y * kFitTile, nk = (K + 63) / 64;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
    mbar_init(accum, 1);
    mbar_fence_init();
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
  }
  if (warp == 1) { tmem_alloc(holder, 4 * kFitTile); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *holder_ptr;
  grid_dep_wait();
  grid_dep_launch();

  if (warp == 0 && elect_one()) {
    auto load = [&](uint32_t dst, const CUtensorMap* map, uint32_t bar, bool mn, int row0, int k0, int z) {
      if (mn) {
        tma_load_3d(dst, map, bar, row0, k0, z);
        tma_load_3d(dst + kFitPart / 2, map, bar, row0 + 64, k0, z);
      } else {
        tma_load_3d(dst, map, bar, k0, row0, z);
      }
    };
    for (int i = 0; i < nk; ++i) {
      const int s = i % S;
      if (i >= S && !mbar_wait(empty0 + 8 * s, ((i / S) - 1) & 1, err)) break;
      mbar_expect_tx(full0 + 8 * s, Cfg::kStageBytes);
      const uint32_t st = base + s * Cfg::kStageBytes;
      for (int p = 0; p < NA; ++p) load(st + p * kFitPart, &tmA, full0 + 8 * s, AMN, r0, 64 * i, p * a_heads + (a_heads > 1 ? head : 0));
      for (int p = 0; p < NB; ++p) load(st + (NA + p) * kFitPart, &tmB, full0 + 8 * s, BMN, c0, 64 * i, p * b_heads + (b_heads > 1 ? head : 0));
    }
  }
  if (warp == 1 && elect_one()) {
    constexpr uint32_t idesc = umma_idesc_bf16(kFitTile, kFitTile) | (AMN ? 1u << 15 : 0u) | (BMN ? 1u << 16 : 0u);
    for (int i = 0; i < nk; ++i) {
      const int s = i % S;
      if (!mbar_wait(full0 + 8 * s, (i / S) & 1, err)) break;
      tc_fence_after();
      const uint32_t a = base + s * Cfg::kStageBytes, b = a + NA * kFitPart;
#pragma unroll
      for (int pa = 0; pa < NA; ++pa)
#pragma unroll
        for (int pb = 0; pb < NB; ++pb) {
          if (pa + pb > 2) continue;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint32_t aa = a + pa * kFitPart + (AMN ? 2048 : 32) * k, bb = b + pb * kFitPart + (BMN ? 2048 : 32) * k;
            const bool main = pa + pb == 0;
            const int g = 4 * i + k;
            umma_bf16(tmem + kFitTile * (main ? g % 3 : 3), AMN ? fit_desc_mn(aa) : umma_desc_k_sw128(aa),
                      BMN ? fit_desc_mn(bb) : umma_desc_k_sw128(bb), idesc,
                      main ? g >= 3 : !(g == 0 && pa == 0 && pb == (NB > 1 ? 1 : 0)) && !(g == 0 && NB == 1 && pa == 1));
          }
        }
      umma_commit(empty0 + 8 * s);
    }
    umma_commit(accum);
  }
  __syncwarp();
  const bool done = mbar_wait(accum, 0, err);
  tc_fence_after();
  // the tile goes through the (idle) ring: a thread has a row of it, memory wants a warp per row.  The updates that read and
  // write 38 bytes per weight took 100-200 us with a row per thread.
  float* tile = reinterpret_cast<float*>(smem_raw + (base - smem_u32(smem_raw)));
  constexpr int LD = kFitTile + 4;
  const uint32_t trow = tmem + ((uint32_t)(32 * warp) << 16);
  if (done && warp < 4) {
#pragma unroll 1
    for (int c = 0; c < kFitTile; c += 32) {
      float v[32], t[32];
      tmem_ld32(trow + c, v);
#pragma unroll 1
      for (int q = 1; q < 4; ++q) {
        tmem_ld32(trow + kFitTile * q + c, t);
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] += t[j];
      }
      float4* o = reinterpret_cast<float4*>(tile + (32 * warp + lane) * LD + c);
#pragma unroll
      for (int i = 0; i < 8; ++i) o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
  }
  __syncthreads();
  if (done) {
    const int c = c0 + 4 * lane;                                 // C is a multiple of 4: whole pieces
    constexpr int U = Epi::kRows;
#pragma unroll 1
    for (int i = 8 * warp; i < 8 * warp + 8; i += U) {
      typename Epi::In in[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int r = r0 + i + u;
        if (r < R && c < C) epi.load(head, r, c, in[u]);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int r = r0 + i + u;
        if (r < R && c < C) epi.finish(head, r, c, *reinterpret_cast<const float4*>(tile + (i + u) * LD + 4 * lane), in[u]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, 4 * kFitTile);
}

// The three parts of eight values, one 16-byte store each; `stride` elements between the parts.
__device__ __forceinline__ void store_parts8(bf16* p, long long stride, const float* v) {
  uint32_t o[3][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float2 x = make_float2(v[2 * i], v[2 * i + 1]);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(x.x, x.y);
      o[q][i] = *reinterpret_cast<const uint32_t*>(&h);
      x.x -= __bfloat162float(h.x); x.y -= __bfloat162float(h.y);
    }
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) *reinterpret_cast<uint4*>(p + q * stride) = make_uint4(o[q][0], o[q][1], o[q][2], o[q][3]);
}

// The three parts of four values, one 8-byte store each.
__device__ __forceinline__ void store_parts4(bf16* p, long long stride, float4 v) {
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    *reinterpret_cast<uint2*>(p + q * stride) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
    v.x -= __bfloat162float(a.x); v.y -= __bfloat162float(a.y); v.z -= __bfloat162float(b.x); v.w -= __bfloat162float(b.y);
  }
}
__device__ __forceinline__ float4 ldf4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// ---- epilogues: four consecutive columns of a row; load() of kRows rows first, then finish() --------------------------

// pre = acc + b (kept for the backward pass); z = h + SiLU(pre), in parts.  r = token, c = feature.
struct FitHidden {
  static constexpr int kRows = 4;
  struct In { float4 h; };
  const float *b, *h;            // [heads][d], [T][d]
  float* pre;                    // [heads][T][d]
  bf16* z;                       // [3][heads][T][d]
  int T, d, heads;
  __device__ __forceinline__ void load(int, int r, int c, In& in) const { in.h = ldf4(h + (long long)r * d + c); }
  __device__ __forceinline__ void finish(int head, int r, int c, float4 a, const In& in) const {
    const long long at = ((long long)head * T + r) * d + c;
    const float4 bb = ldf4(b + head * d + c);
    a.x += bb.x; a.y += bb.y; a.z += bb.z; a.w += bb.w;
    *reinterpret_cast<float4*>(pre + at) = a;
    store_parts4(z + at, (long long)heads * T * d,
                 make_float4(in.h.x + a.x / (1.0f + expf(-a.x)), in.h.y + a.y / (1.0f + expf(-a.y)),
                             in.h.z + a.z / (1.0f + expf(-a.z)), in.h.w + a.w / (1.0f + expf(-a.w))));
  }
};

// Plain fp32 rows.
struct FitStore {
  static constexpr int kRows = 4;
  struct In {};
  float* out;                    // [heads][rows][cols]
  int rows, cols;
  __device__ __forceinline__ void load(int, int, int, In&) const {}
  __device__ __forceinline__ void finish(int head, int r, int c, float4 a, const In&) const {
    *reinterpret_cast<float4*>(out + ((long long)head * rows + r) * cols + c) = a;
  }
};

// dpre = dz * SiLU'(pre), in parts.  r = token, c = feature.
struct FitDpre {
  static constexpr int kRows = 4;
  struct In { float4 t; };
  const float* pre;              // [heads][T][d]
  bf16* dpre;                    // [3][heads][T][d]
  int T, d, heads;
  __device__ __forceinline__ void load(int head, int r, int c, In& in) const { in.t = ldf4(pre + ((long long)head * T + r) * d + c); }
  static __device__ __forceinline__ float slope(float t) {
    const float s = 1.0f / (1.0f + expf(-t));
    return s * (1.0f + t * (1.0f - s));
  }
  __device__ __forceinline__ void finish(int head, int r, int c, float4 a, const In& in) const {
    store_parts4(dpre + ((long long)head * T + r) * d + c, (long long)heads * T * d,
                 make_float4(a.x * slope(in.t.x), a.y * slope(in.t.y), a.z * slope(in.t.z), a.w * slope(in.t.w)));
  }
};

// One Adam step on a parameter (beta 0.9 / 0.999, eps 1e-8; c1, c2 = 1 - beta^t).
__device__ __forceinline__ float adam_step(float p, float g, float& m, float& v, float lr, float c1, float c2) {
  m = 0.9f * m + 0.1f * g;
  v = 0.999f * v + 0.001f * g * g;
  return p - lr * (m / c1) / (sqrtf(v / c2) + 1e-8f);
}

// The accumulator is the gradient: Adam on the fp32 master, the deployed weight and the master's parts rewritten (the
// gradient itself never goes to memory).
template <typename T>
struct FitAdam {
  static constexpr int kRows = 4;
  struct In { float4 p, m, v; };
  float *p, *m, *v;              // [heads][rows][cols]
  T* deployed;
  bf16* parts;                   // [3][heads][rows][cols]
  int rows, cols, heads;
  float lr, c1, c2;
  __device__ __forceinline__ void load(int head, int r, int c, In& in) const {
    const long long at = ((long long)head * rows + r) * cols + c;
    in.p = ldf4(p + at); in.m = ldf4(m + at); in.v = ldf4(v + at);
  }
  __device__ __forceinline__ void finish(int head, int r, int c, float4 g, In in) const {
    const long long at = ((long long)head * rows + r) * cols + c;
    in.p.x = adam_step(in.p.x, g.x, in.m.x, in.v.x, lr, c1, c2); in.p.y = adam_step(in.p.y, g.y, in.m.y, in.v.y, lr, c1, c2);
    in.p.z = adam_step(in.p.z, g.z, in.m.z, in.v.z, lr, c1, c2); in.p.w = adam_step(in.p.w, g.w, in.m.w, in.v.w, lr, c1, c2);
    *reinterpret_cast<float4*>(p + at) = in.p;
    *reinterpret_cast<float4*>(m + at) = in.m;
    *reinterpret_cast<float4*>(v + at) = in.v;
    store4<T>(deployed + at, in.p.x, in.p.y, in.p.z, in.p.w);
    store_parts4(parts + at, (long long)heads * rows * cols, in.p);
  }
};

// Weights of the model dtype -> fp32 masters and their parts.  n a multiple of 8.
template <typename T>
__global__ void fit_masters_kernel(const T* __restrict__ src, float* __restrict__ dst, bf16* __restrict__ parts, long long n) {
  const long long i = 8 * ((long long)blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n) return;
  float v[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) { v[j] = to_f<T>(src[i + j]); dst[i + j] = v[j]; }
  store_parts8(parts + i, n, v);
}

// Hidden states as fp32 and as operand parts (one part where they are bf16 already); the last block counts every head's
// targets (>= 0).  n a multiple of 8.
template <typename T>
__global__ void __launch_bounds__(256) fit_inputs_kernel(const T* src, float* __restrict__ hf, bf16* __restrict__ parts, long long n,
                                                         const int32_t* targets, int tokens, int heads, int32_t* __restrict__ count) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (blockIdx.x == gridDim.x - 1) {
    __shared__ int s[8];
    for (int hd = 0; hd < heads; ++hd) {
      int c = 0;
      for (int t = threadIdx.x; t < tokens; t += blockDim.x) c += targets[(long long)t * heads + hd] >= 0 ? 1 : 0;
      c = __reduce_add_sync(0xffffffffu, c);
      __syncthreads();
      if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = c;
      __syncthreads();
      if (threadIdx.x == 0) {
        int tot = 0;
        for (int w = 0; w < 8; ++w) tot += s[w];
        count[hd] = tot;
      }
    }
    return;
  }
  const long long i = 8 * ((long long)blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n) return;
  float v[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) { v[j] = to_f<T>(src[i + j]); hf[i + j] = v[j]; }
  if (sizeof(T) == 2) {
    uint32_t o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
      o[j] = *reinterpret_cast<const uint32_t*>(&h);
    }
    *reinterpret_cast<uint4*>(parts + i) = make_uint4(o[0], o[1], o[2], o[3]);
  } else {
    store_parts8(parts + i, n, v);
  }
}

// One block per (position, head): softmax of the logits row over the vocabulary, the row's cross-entropy, and, in parts, the
// row of d loss / d logits = lambda^(head+1) / count * (p - onehot) (zero for a position without a target and in the padding
// columns).
__global__ void __launch_bounds__(256) fit_softmax_ce_kernel(const float* logits, const int32_t* targets,
                                                             const int32_t* count, int T, int heads, int vocab,
                                                             int ld, float lambda, bf16* __restrict__ dl /*[3][heads][T][ld]*/,
                                                             float* __restrict__ ce) {
  __shared__ float red[2][8];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int t = blockIdx.x, head = blockIdx.y, tid = threadIdx.x;
  const long long at = ((long long)head * T + t) * ld, part = (long long)heads * T * ld;
  const float* row = logits + at;
  const int tg = targets[(long long)t * heads + head];
  const bool live = tg >= 0 && tg < vocab;
  auto block_reduce = [&](float v, bool is_max, int buf) -> float {
    for (int o = 16; o > 0; o >>= 1) {
      const float u = __shfl_xor_sync(0xffffffffu, v, o);
      v = is_max ? fmaxf(v, u) : v + u;
    }
    if ((tid & 31) == 0) red[buf][tid >> 5] = v;
    __syncthreads();
    float r = is_max ? -INFINITY : 0.f;
    for (int w = 0; w < 8; ++w) r = is_max ? fmaxf(r, red[buf][w]) : r + red[buf][w];
    return r;
  };
  float mx = -INFINITY, sum = 0.f, w = 0.f, inv = 0.f;
  if (live) {
    for (int j = tid; j < vocab; j += blockDim.x) mx = fmaxf(mx, row[j]);
    mx = block_reduce(mx, true, 0);
    for (int j = tid; j < vocab; j += blockDim.x) sum += expf(row[j] - mx);
    sum = block_reduce(sum, false, 1);
    w = 1.0f;
    for (int i = 0; i <= head; ++i) w *= lambda;
    w /= (float)count[head];
    inv = 1.0f / sum;
  }
  if (tid == 0) ce[(long long)head * T + t] = live ? logf(sum) + mx - row[tg] : 0.f;
  for (int j0 = 8 * tid; j0 < ld; j0 += 8 * blockDim.x) {
    float g[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = j0 + j;
      g[j] = live && c < vocab ? w * (expf(row[c] - mx) * inv - (c == tg ? 1.0f : 0.0f)) : 0.f;
    }
    store_parts8(dl + at + j0, part, g);
  }
}

// x < ceil(d / 32): db[head][j] = sum_t dpre[head][t][j] (32 rows of threads take every 32nd position, summed in a fixed
// order), then Adam on the bias.  The last x: the loss.  loss[1 + head] = mean cross-entropy of the head over its targets;
// loss[0] = sum_i lambda^(i+1) loss[1 + i], fixed summation order.  grid = (ceil(d / 32) + 1, heads), 1024 threads.
__global__ void __launch_bounds__(1024) fit_bias_kernel(const bf16* dpre /*[3][heads][T][d]*/, int T, int d, int heads,
                                                       float* p, float* m, float* v, float* __restrict__ deployed, float lr,
                                                       float c1, float c2, const float* ce, const int32_t* count, float lambda,
                                                       float* __restrict__ loss) {
  __shared__ float red[32][33];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  if (blockIdx.x == gridDim.x - 1) {
    if (blockIdx.y != 0 || !loss) return;
    float total = 0.f, w = 1.f;
    for (int hd = 0; hd < heads; ++hd) {
      float s = 0.f;
      for (int t = threadIdx.x; t < T; t += blockDim.x) s += ce[(long long)hd * T + t];
      s = warp_sum(s);
      __syncthreads();
      if (tx == 0) red[0][ty] = s;
      __syncthreads();
      float tot = 0.f;
      for (int q = 0; q < 32; ++q) tot += red[0][q];
      const float mean = count[hd] > 0 ? tot / (float)count[hd] : 0.f;
      w *= lambda;
      total += w * mean;
      if (threadIdx.x == 0) loss[1 + hd] = mean;
    }
    if (threadIdx.x == 0) loss[0] = total;
    return;
  }
  const int j = blockIdx.x * 32 + tx, head = blockIdx.y;
  const long long part = (long long)heads * T * d;
  float s = 0.f;
  if (j < d) {
    const bf16* q = dpre + (long long)head * T * d + j;
#pragma unroll 4
    for (int t = ty; t < T; t += 32) {
      const long long o = (long long)t * d;
      s += (to_f<bf16>(q[o + 2 * part]) + to_f<bf16>(q[o + part])) + to_f<bf16>(q[o]);
    }
  }
  red[ty][tx] = s;
  __syncthreads();
  if (ty == 0 && j < d) {
    float g = 0.f;
    for (int q = 0; q < 32; ++q) g += red[q][tx];
    const int i = head * d + j;
    float mi = m[i], vi = v[i];
    const float np_ = adam_step(p[i], g, mi, vi, lr, c1, c2);
    m[i] = mi; v[i] = vi; p[i] = np_;
    deployed[i] = np_;
  }
}

}  // namespace vadusa
