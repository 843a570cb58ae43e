// Block-level selection helpers, the keys of a base-head row (with the top-p nucleus), the root sample and the
// draft heads' top-k (paper Sec. II-A: the base head gives the first next token, draft head i the top-k
// candidates of depth i).  Up to kSelectWide tokens a block of a few warps serves, beyond it 1024 threads (16 tokens per
// thread at a 16 000-entry vocabulary).
#pragma once
#include "rng.cuh"

namespace vadusa {

constexpr int kSelectWide = 4096;
inline int select_threads(int vocab) { return vocab <= kSelectWide ? 256 : 1024; }

struct Best { float v; int i; };

__device__ __forceinline__ Best better(Best a, Best b) {
  if (b.i < 0) return a;
  if (a.i < 0) return b;
  return precedes(a.v, a.i, b.v, b.i) ? a : b;
}

// fp32 -> uint32 that orders like the value (-0 counted as +0); every finite value and -inf map above 0.
__device__ __forceinline__ uint32_t ordered_bits(float v) {
  const uint32_t u = __float_as_uint(__fadd_rn(v, 0.0f));
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float from_ordered_bits(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// First element of the block in the order "larger value, then lower id" (i < 0: none).
// scratch: 32 Best entries of shared memory.  Result is the same in every thread.  The value travels as
// its ordered bit pattern, so a warp needs two reduction instructions: the largest value, then the lowest
// id among the lanes that hold it.
__device__ __forceinline__ Best block_first(Best x, Best* scratch) {
  const uint32_t none = 0xffffffffu;
  uint32_t k = x.i < 0 ? 0u : ordered_bits(x.v);
  uint32_t wk = __reduce_max_sync(0xffffffffu, k);
  uint32_t wi = __reduce_min_sync(0xffffffffu, (x.i >= 0 && k == wk) ? (uint32_t)x.i : none);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if (lane == 0) scratch[warp] = Best{__uint_as_float(wk), (int)wi};
  __syncthreads();
  const bool have = lane < nw && scratch[lane].i != (int)none;
  k = have ? __float_as_uint(scratch[lane].v) : 0u;
  const uint32_t id = have ? (uint32_t)scratch[lane].i : none;
  wk = __reduce_max_sync(0xffffffffu, k);
  wi = __reduce_min_sync(0xffffffffu, (have && k == wk) ? id : none);
  if (wi == none) return Best{0.f, -1};
  return Best{from_ordered_bits(wk), (int)wi};
}

__device__ __forceinline__ float block_sum(float x, float* scratch) {
  x = warp_sum(x);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if (lane == 0) scratch[warp] = x;
  __syncthreads();
  float r = (lane < nw) ? scratch[lane] : 0.f;
  return warp_sum(r);
}

__device__ __forceinline__ float block_max(float x, float* scratch) {
  x = warp_max(x);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if (lane == 0) scratch[warp] = x;
  __syncthreads();
  float r = (lane < nw) ? scratch[lane] : -INFINITY;
  return warp_max(r);
}

__device__ __forceinline__ bool nucleus_on(const SamplingDev& sp) {
  return sp.temperature != 0.f && sp.top_p < 1.0f;
}

// Sums of eight values per lane over the warp; lane l returns the sum of value l & 7 (nine shuffles instead of forty:
// each of the first three steps halves the values a lane carries).
template <typename V> __device__ __forceinline__ V warp_sum8(const V* v, int lane) {
  V a[4], b[2], c;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const V keep = (lane & 4) ? v[i + 4] : v[i], give = (lane & 4) ? v[i] : v[i + 4];
    a[i] = keep + __shfl_xor_sync(0xffffffffu, give, 4);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const V keep = (lane & 2) ? a[i + 2] : a[i], give = (lane & 2) ? a[i] : a[i + 2];
    b[i] = keep + __shfl_xor_sync(0xffffffffu, give, 2);
  }
  const V keep = (lane & 1) ? b[1] : b[0], give = (lane & 1) ? b[0] : b[1];
  c = keep + __shfl_xor_sync(0xffffffffu, give, 1);
  c += __shfl_xor_sync(0xffffffffu, c, 8);
  c += __shfl_xor_sync(0xffffffffu, c, 16);
  return c;
}

// Shared scratch of the selection routines (32 warps at most).
struct SelectScratch {
  Best best[32];
  float f[32];
  float mass[2][32][8];
  int count[2][32][8];
  int scan[1024];     // (ties at the edge of the nucleus)
};

// The top-p nucleus of softmax(logits / T), in the order "larger logit, then lower id": the prefix of tokens whose
// mass ahead of them is below top_p (the crossing token included).  The mass strictly above a value falls as the value
// grows, so the nucleus is everything above the smallest value v* whose mass above is still below top_p, plus the
// tokens AT v* while (mass above v*) + (ties with a lower id) * p* stays below top_p.  v* is searched on the ordered
// bit pattern of the value: every round splits the interval in eight and sums mass and token count per part in one
// pass over the row (each thread over its own tokens, fixed order), until the interval holds one token or one value:
// three or four rounds for a thousand tokens, where bisection took 32 block-wide sums (36 us of a 49 us launch at
// 1025 tokens).  The first interval is what the peak alone decides: below max + T ln((1 - top_p) Z / vocab) all tokens
// together weigh less than 1 - top_p.
//   val[]   in: logits (EOS masked) in shared memory;  prob[] out: exp((val - max) / T)
// On return token j is inside iff bits(val[j]) > lo, where `tied` tells that the tokens at hi (the only ones in
// (lo, hi]) are tied and `above` is their mass ahead; without ties everything above lo is inside.
struct Nucleus { uint32_t lo, hi; float above, limit; bool tied; };

__device__ Nucleus nucleus_of(const float* val, float* prob, int vocab, const SamplingDev& sp, SelectScratch& sc) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = (int)blockDim.x >> 5;
  float mx = -INFINITY;
  for (int j = tid; j < vocab; j += blockDim.x) mx = fmaxf(mx, val[j]);
  mx = block_max(mx, sc.f);
  float z = 0.f;
  for (int j = tid; j < vocab; j += blockDim.x) {
    const float p = expf((val[j] - mx) * sp.inv_temperature);
    prob[j] = p;
    z += p;
  }
  z = block_sum(z, sc.f);
  Nucleus n;
  n.limit = sp.top_p * z;
  n.above = 0.f;
  n.hi = ordered_bits(mx);                       // mass above the largest value: 0 < limit
  n.tied = false;
  // (a margin below the bound of the comment, so that rounding cannot put v* under it)
  const float cut = mx + sp.temperature * (logf((1.0f - sp.top_p) * z / (float)vocab) - 0.01f);
  n.lo = cut > -INFINITY ? ordered_bits(cut) : 0u;
  if (n.lo >= n.hi) n.lo = n.hi - 1u;
  for (int round = 0;; ++round) {
    // parts of the interval (lo, hi]: part k = (lo + k 2^s, lo + (k + 1) 2^s]
    const uint32_t range = n.hi - n.lo;
    const int s = range <= 8u ? 0 : 29 - __clz((int)(range - 1u));
    float m[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    int c[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int j = tid; j < vocab; j += blockDim.x) {
      const uint32_t b = ordered_bits(val[j]);
      if (b > n.lo && b <= n.hi) {
        const uint32_t k = (b - n.lo - 1u) >> s;
        const float p = prob[j];
#pragma unroll
        for (int i = 0; i < 8; ++i) { m[i] += k == (uint32_t)i ? p : 0.f; c[i] += k == (uint32_t)i ? 1 : 0; }
      }
    }
    const float wm = warp_sum8<float>(m, lane);
    const int wc = warp_sum8<int>(c, lane);
    const int buf = round & 1;                   // two buffers: one barrier per round
    if (lane < 8) { sc.mass[buf][warp][lane] = wm; sc.count[buf][warp][lane] = wc; }
    __syncthreads();
    float pm = 0.f;
    int pc = 0;
    for (int w = 0; w < nw; ++w) { pm += sc.mass[buf][w][lane & 7]; pc += sc.count[buf][w][lane & 7]; }
    // from the top part down to the first whose lower end has at least `limit` above it (the same in every thread)
    float above = n.above;
    int part = 7, cnt = 0;
    for (;; --part) {
      const float with = above + __shfl_sync(0xffffffffu, pm, part);
      cnt = __shfl_sync(0xffffffffu, pc, part);
      if (with >= n.limit || part == 0) break;
      above = with;
    }
    const uint32_t lo = n.lo + ((uint32_t)part << s), width = 1u << s;
    if (n.hi - lo > width) n.hi = lo + width;
    n.lo = lo;
    n.above = above;
    if (cnt <= 1) break;
    if (n.hi - n.lo <= 1u) { n.tied = true; break; }
  }
  return n;
}

// Gumbel noise of a row's tokens into noise[] (shared memory; each thread its own tokens j = tid + i * blockDim.x).  It
// depends on the position alone, so a kernel can form it while the product that makes the logits still runs.  With the
// nucleus on, few tokens need a key: row_keys makes their noise itself and this does nothing.
__device__ __forceinline__ void row_noise(int vocab, uint64_t rs, const SamplingDev& sp, float* noise) {
  if (nucleus_on(sp) || sp.temperature == 0.f) return;
  for (int j = threadIdx.x; j < vocab; j += blockDim.x) noise[j] = gumbel_of(rs, j);
}

// Keys of one base-head row in shared memory: key[j] = logit / T + noise (or the logit alone), -inf outside the
// nucleus.  key[] holds row_noise of the row on entry.  val[] (nucleus only) gets the logits as the sampler sees them.
// All threads; ends with a barrier.
__device__ void row_keys(const BaseRow row, int vocab, uint64_t rs, const SamplingDev& sp, bool noise, float* key, float* val,
                         SelectScratch& sc) {
  const int tid = threadIdx.x;
  if (!nucleus_on(sp)) {
#pragma unroll 4
    for (int j = tid; j < vocab; j += blockDim.x) {
      const float l = masked_logit(row[j], j, sp);
      key[j] = (sp.temperature == 0.f || !noise || l == -INFINITY) ? l : __fadd_rn(__fmul_rn(l, sp.inv_temperature), key[j]);
    }
    __syncthreads();
    return;
  }
#pragma unroll 4
  for (int j = tid; j < vocab; j += blockDim.x) val[j] = masked_logit(row[j], j, sp);
  __syncthreads();
  const Nucleus n = nucleus_of(val, key, vocab, sp, sc);        // key[] holds the probabilities for now
  if (!n.tied) {
    for (int j = tid; j < vocab; j += blockDim.x)
      key[j] = ordered_bits(val[j]) > n.lo ? key_of(val[j], j, rs, sp, noise) : -INFINITY;
  } else {
    // ties at v* = hi: earlier ids with the same value, by contiguous chunks of ids
    const int chunk = (vocab + (int)blockDim.x - 1) / (int)blockDim.x, j0 = tid * chunk, j1 = min(vocab, j0 + chunk);
    int mine = 0;
    for (int j = j0; j < j1; ++j) mine += ordered_bits(val[j]) == n.hi ? 1 : 0;
    __syncthreads();
    sc.scan[tid] = mine;
    __syncthreads();
    int before = 0;
    for (int t = 0; t < tid; ++t) before += sc.scan[t];
    for (int j = j0; j < j1; ++j) {
      const uint32_t b = ordered_bits(val[j]);
      bool inside = b > n.hi;
      if (b == n.hi) { inside = n.above + (float)before * key[j] < n.limit; ++before; }
      key[j] = inside ? key_of(val[j], j, rs, sp, noise) : -INFINITY;
    }
  }
  __syncthreads();
}

// The token that comes first in key order.  Same result in every thread.
__device__ __forceinline__ int first_key(const float* key, int vocab, SelectScratch& sc) {
  Best mine{0.f, -1};
  for (int j = threadIdx.x; j < vocab; j += blockDim.x) mine = better(mine, Best{key[j], j});
  const Best top = block_first(mine, sc.best);
  return top.i < 0 ? 0 : top.i;
}

// Dynamic shared memory of a kernel that calls row_keys.
inline size_t row_keys_smem(int ld, const SamplingDev& sp) {
  return (size_t)ld * sizeof(float) * (sp.temperature != 0.f && sp.top_p < 1.0f ? 2 : 1);
}

// grid = (n_draft_heads + 1, batch).  blockIdx.x < n_draft_heads: the head's top-k ids in
// descending logit order (EOS masked), written to topk[b][head][0..k).  Last x: the root.
// Top-k: every thread keeps the best of its own tokens; the k-th best of those maxima is a bound that at least k
// tokens reach, and only tokens of the k threads at or before it can be among the first k: a few dozen candidates,
// ranked by counting.  Three block barriers whatever k (one barrier pair per rank took 6.8 us per launch at 1025
// tokens, 73 us at 16001).
__global__ void __launch_bounds__(1024) draft_select_kernel(
    const float* __restrict__ dlogits /*[heads][batch][ld]*/, const float* __restrict__ logits_star /*[batch][ld]*/,
    int ld, int vocab, int batch, int n_heads, int k, const int32_t* __restrict__ ctx_len,
    const int32_t* __restrict__ nvalid, SamplingDev sp, int32_t* __restrict__ topk, int32_t* __restrict__ root) {
  constexpr int kCand = 512;
  extern __shared__ float keys[];              // the root's row only
  __shared__ SelectScratch sc;
  __shared__ unsigned long long s_cand[kCand], s_bound;
  __shared__ int s_n;
  const int b = blockIdx.y, head = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = (int)blockDim.x >> 5;
  if (head == n_heads) {
    // (the context length is not written by the products of the draft heads: readable before they end)
    const uint64_t rs = noise_row_state(sp.seed, b, __ldcg(ctx_len + b));
    row_noise(vocab, rs, sp, keys);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (nvalid[b] == 0) return;
    row_keys(base_row(logits_star + (long long)b * ld, sp, b), vocab, rs, sp, true, keys, keys + ld, sc);
    const int r = first_key(keys, vocab, sc);
    if (tid == 0) root[b] = r;
    return;
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const float* row = dlogits + ((long long)head * batch + b) * ld;
  int32_t* out = topk + ((long long)b * n_heads + head) * k;
  // a token in the order "larger logit, then lower id" as one number, larger first; 0: none
  auto pack = [&](float v, int j) { return ((unsigned long long)ordered_bits(v) << 32) | (uint32_t)~j; };
  unsigned long long mine = 0ull;
#pragma unroll 8
  for (int j = tid; j < vocab; j += blockDim.x) {
    const unsigned long long t = pack(masked_logit(row[j], j, sp), j);
    mine = t > mine ? t : mine;
  }
  if (nvalid[b] == 0) return;
  // the k best thread maxima of every warp, in order
  uint32_t left = (uint32_t)(mine >> 32);
  const uint32_t low = (uint32_t)mine;
  for (int r = 0; r < k; ++r) {
    const uint32_t wk = __reduce_max_sync(0xffffffffu, left);
    const uint32_t wl = __reduce_max_sync(0xffffffffu, left == wk ? low : 0u);
    if (lane == 0) s_cand[warp * k + r] = wk == 0u ? 0ull : ((unsigned long long)wk << 32) | wl;
    if (left == wk && low == wl) left = 0u;
  }
  if (tid == 0) { s_bound = 0ull; s_n = 0; }
  __syncthreads();
  // the k-th of all of them: k < vocab, and every warp lists min(k, its threads that hold a token)
  const int nmax = nw * k;
  if (tid < nmax) {
    const unsigned long long t = s_cand[tid];
    int before = 0;
#pragma unroll 8
    for (int o = 0; o < nmax; ++o) before += s_cand[o] > t ? 1 : 0;
    if (before == k - 1 && t != 0ull) s_bound = t;
  }
  __syncthreads();
  // candidates: tokens at or before the bound
  const unsigned long long bound_t = s_bound;
  if (mine != 0ull && mine >= bound_t)
    for (int j = tid; j < vocab; j += blockDim.x) {
      const unsigned long long t = pack(masked_logit(row[j], j, sp), j);
      if (t < bound_t) continue;
      const int at = atomicAdd(&s_n, 1);
      if (at < kCand) s_cand[at] = t;
    }
  __syncthreads();
  const int n = s_n;
  if (n <= kCand) {
    for (int t = tid; t < n; t += blockDim.x) {
      const unsigned long long own = s_cand[t];
      int before = 0;
#pragma unroll 4
      for (int o = 0; o < n; ++o) before += s_cand[o] > own ? 1 : 0;
      if (before < k) out[before] = (int)~(uint32_t)own;
    }
    return;
  }
  // more candidates than fit (a vocabulary far beyond the decoding path's, or no bound): one pass per rank
  Best bound{INFINITY, -1};
  for (int r = 0; r < k; ++r) {
    Best m{0.f, -1};
    for (int j = tid; j < vocab; j += blockDim.x) {
      const float v = masked_logit(row[j], j, sp);
      if (bound.i >= 0 && !precedes(bound.v, bound.i, v, j)) continue;
      m = better(m, Best{v, j});
    }
    bound = block_first(m, sc.best);
    if (tid == 0) out[r] = bound.i < 0 ? 0 : bound.i;
  }
}

}  // namespace vadusa
