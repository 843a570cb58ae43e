// Tree-masked decode attention over the paged KV cache, plain FMA arithmetic.
// Node n of sequence b attends to every cached position < ctx_len[b] and to the tree
// slots ctx_len[b] + m whose bit m is set in anc[n] (its ancestors and itself); tree
// nodes' K/V rows sit in the cache behind the context (paper Sec. II-A, tree attention).
#pragma once
#include "common.cuh"

namespace vadusa {

template <typename T> __device__ __forceinline__ float4 att_ld4(const T* p);
template <> __device__ __forceinline__ float4 att_ld4<float>(const float* p) { return *reinterpret_cast<const float4*>(p); }
template <> __device__ __forceinline__ float4 att_ld4<bf16>(const bf16* p) {
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                     __uint_as_float(v.y & 0xffff0000u));
}

// grid = (heads, batch, ceil(N / NG)): NG nodes of one (head, sequence) per block.  The eight warps take the keys in
// chunks of 32 (fetched by rows into the warp's own shared memory; a lane forms the scores of one key for all NG nodes, then
// the lanes turn to the features and add the weighted V rows), each with running maxima and sums of its own; they are
// merged once at the end.  A short context is one chunk per warp: three dependent loads and one block barrier (17 us before,
// with a block per head that staged 64-key pages one after another).  Rows read straight into the lanes that own them
// touch 32 lines per load: 9 us for 16 nodes over 120-200 keys, about 4 us through shared memory.
// NG = 4 while the blocks are few, 8 when they fill the device several times (half the K/V reads).
// Dynamic shared memory: att_simt_smem(DH).
inline int att_simt_smem(int dh) { return 8 * 32 * (dh + 4) * 4; }

template <typename T, int DH, int NG>
__global__ void __launch_bounds__(256) tree_attention_simt_kernel(
    const T* q, const T* pool, const int32_t* __restrict__ block_table,
    const int32_t* ctx_len, const int32_t* nvalid, TreeView tree, KvGeom geom,
    int d_model, float scale, int ahead /*rows inside the context may be read before the upstream kernel ends: not while prefilling*/,
    T* __restrict__ out, uint32_t* err) {
  constexpr int R = DH / 32;
  __shared__ float4 Qs[NG][DH / 4];
  __shared__ float4 Ps[8][NG][8];             // a warp's weights: [node][32 keys]
  extern __shared__ float4 stage[];           // [8 warps][32 keys][DH + 4] fp32; at the end the warps' sums [8][NG][DH]
  __shared__ float Ms[8][NG], Ls[8][NG];
  const int h = blockIdx.x, b = blockIdx.y, N = tree.n_nodes, n0 = NG * blockIdx.z;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // lengths and the context's rows were there before the projection that precedes this kernel: fetched while it runs
  const int nv = __ldcg(nvalid + b), S = __ldcg(ctx_len + b);
  constexpr int U = DH / 4;                                  // four-element units of a row
  const int total = nv > 0 ? S + nv : 0;
  float4 kr[U];
  long long blk = -1;
  auto fetch_keys = [&](int t0) {
    blk = kv_block_of(block_table, geom, b, t0, err);
    if (blk < 0) return;                                     // uniform over the warp
    const T* Kg = pool + geom.elem(blk, 0, h, t0 % kKvBlock);
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const int u = lane + 32 * i;                           // slots past the tree hold stale data
      kr[i] = t0 + u / U < total ? att_ld4<T>(Kg + 4 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  const bool early = ahead && 32 * warp + 32 <= S && nv > 0;
  if (early) fetch_keys(32 * warp);
  unsigned long long alo[NG], ahi[NG];
#pragma unroll
  for (int i = 0; i < NG; ++i) {
    alo[i] = ahi[i] = 0ull;
    if (n0 + i < nv) tree.anc_of(b, n0 + i, alo[i], ahi[i]);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  for (int i = threadIdx.x; i < NG * DH / 4; i += 256) {
    const int n = i / (DH / 4), e = i % (DH / 4);
    Qs[n][e] = n0 + n < N ? att_ld4<T>(q + ((long long)b * N + n0 + n) * d_model + h * DH + 4 * e) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float O[NG][R], mrun[NG], lrun[NG];
#pragma unroll
  for (int i = 0; i < NG; ++i) {
    mrun[i] = -INFINITY; lrun[i] = 0.f;
#pragma unroll
    for (int c = 0; c < R; ++c) O[i][c] = 0.f;
  }
  __syncthreads();
  for (int t0 = 32 * warp; t0 < total; t0 += 256) {
    if (!(early && t0 == 32 * warp)) fetch_keys(t0);
    if (blk < 0) continue;
    const int t = t0 + lane, nk = min(32, total - t0);
    const T* Vg = pool + geom.elem(blk, 1, h, t0 % kKvBlock);
    const bool live = t < total;
    float s[NG], v[32][R];
#pragma unroll
    for (int i = 0; i < NG; ++i) s[i] = 0.f;
    {
      float4* st = stage + warp * 32 * (U + 1);
#pragma unroll
      for (int i = 0; i < U; ++i) {
        const int u = lane + 32 * i;
        st[(u / U) * (U + 1) + u % U] = kr[i];
      }
      // V rows: on their way during the scores
#pragma unroll
      for (int j = 0; j < 32; ++j)
#pragma unroll
        for (int c = 0; c < R; ++c) v[j][c] = j < nk ? to_f<T>(Vg[j * DH + lane + 32 * c]) : 0.f;
      __syncwarp();
#pragma unroll
      for (int e = 0; e < U; ++e) {
        const float4 k4 = st[lane * (U + 1) + e];
#pragma unroll
        for (int i = 0; i < NG; ++i) {
          const float4 qq = Qs[i][e];
          s[i] = fmaf(qq.x, k4.x, s[i]); s[i] = fmaf(qq.y, k4.y, s[i]);
          s[i] = fmaf(qq.z, k4.z, s[i]); s[i] = fmaf(qq.w, k4.w, s[i]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      const bool vis = n0 + i < nv && (t < S || (live && bit_at(alo[i], ahi[i], t - S)));
      const float x = vis ? s[i] * scale : -INFINITY;
      const float mnew = fmaxf(mrun[i], warp_max(x));
      const float p = mnew == -INFINITY ? 0.f : expf(x - mnew);
      const float corr = mrun[i] == -INFINITY ? 0.f : expf(mrun[i] - mnew);
      lrun[i] = lrun[i] * corr + warp_sum(p);
      mrun[i] = mnew;
      reinterpret_cast<float*>(&Ps[warp][i][0])[lane] = p;
#pragma unroll
      for (int c = 0; c < R; ++c) O[i][c] *= corr;
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int i = 0; i < NG; ++i) {
        const float4 p = Ps[warp][i][j];
#pragma unroll
        for (int c = 0; c < R; ++c) {
          O[i][c] = fmaf(p.x, v[4 * j][c], O[i][c]); O[i][c] = fmaf(p.y, v[4 * j + 1][c], O[i][c]);
          O[i][c] = fmaf(p.z, v[4 * j + 2][c], O[i][c]); O[i][c] = fmaf(p.w, v[4 * j + 3][c], O[i][c]);
        }
      }
    __syncwarp();
  }
  __syncthreads();                                           // (the staging areas become the exchange)
  float* Os = reinterpret_cast<float*>(stage);
#pragma unroll
  for (int i = 0; i < NG; ++i) {
    if (lane == 0) { Ms[warp][i] = mrun[i]; Ls[warp][i] = lrun[i]; }
#pragma unroll
    for (int c = 0; c < R; ++c) Os[(warp * NG + i) * DH + lane + 32 * c] = O[i][c];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < NG * DH; i += 256) {
    const int n = i / DH, e = i % DH;
    if (n0 + n >= N) continue;
    float m = -INFINITY;
#pragma unroll
    for (int w = 0; w < 8; ++w) m = fmaxf(m, Ms[w][n]);
    float l = 0.f, o = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      const float f = Ms[w][n] == -INFINITY ? 0.f : expf(Ms[w][n] - m);
      l = fmaf(Ls[w][n], f, l);
      o = fmaf(Os[(w * NG + n) * DH + e], f, o);
    }
    out[((long long)b * N + n0 + n) * d_model + h * DH + e] = from_f<T>(n0 + n < nv && l > 0.f ? o / l : 0.f);
  }
}

}  // namespace vadusa
