// Tree-masked decode attention over the paged bf16 KV cache on the tcgen05 tensor cores
// (head_dim 64).  Node n of sequence b attends to every cached position < ctx_len[b] and to
// the tree slots ctx_len[b] + m whose bit m is set in anc[n] (paper Sec. II-A, tree attention).
//
// One CTA per (head, sequence, tile of 64 nodes, KV split); the splits of one (head, sequence, tile) form a
// cluster.  Trees of up to 128 nodes carry two 64-bit ancestor words per node.
// The 64 query rows are stored twice in the 128-row Q operand, so the scores of row r appear in
// TMEM lanes r and r + 64: warps 0-1 (lanes 0..63) work on keys 0..31 of every 64-key page,
// warps 2-3 (lanes 64..127) on keys 32..63.  Per page:
//   S = Q K^T      tcgen05.mma, A = Q tile, B = K tile, D in one of three TMEM score buffers (columns
//                  0..63 / 64..127 / 128..191), issued by a warp of its own up to three pages ahead of
//                  P V, so that neither the softmax nor the other issuer waits for it
//   softmax        each thread reads its 32 scores, keeps a scaling maximum of its own for its key
//                  half of the row, and the weights go back to TMEM as
//                  two bf16 halves (p = hi + lo, 16 significant bits) over the score columns,
//                  zero in the other thread's key range.  (Weights rounded to bf16 once would save the lo
//                  product, 4 % of a batch-64 launch, and take the logits of a 12-layer pass over contexts of
//                  up to 3000 tokens from 1.5e-2 to 2.05e-2 away from an fp64 evaluation.)
//   O += P V       tcgen05.mma with A from TMEM (hi then lo), B = V tile (MN-major), accumulating
//                  in TMEM columns 192..255; lanes r and r + 64 hold the two key-halves' sums
// The scaling maximum of a row only moves when the page maximum exceeds it by more than 2^6
// (p <= 64 is harmless in fp32 / bf16); then the row's accumulator is rescaled in TMEM.
// At the end rows r and r + 64 are brought to a common scale and added; splits are merged through an exchange area in global
// memory (L2) in a fixed order.
// K and V tiles have rings of their own: a K tile is free as soon as its Q K^T has completed, a V tile after
// its P V.  "Scores ready", "weights ready" and "P V done" have one mbarrier per score buffer: a buffer's next
// use cannot begin before the waiter of the current one has passed, so no parity wait can fall a round behind.
// Warps: 0-3 softmax, warp 4 TMA producer, warp 5 TMEM owner / P V issuer, warp 6 Q K^T issuer.
#pragma once
#include <type_traits>

#include "tc.cuh"

namespace vadusa {

constexpr int kAttStagesK = 4;                                               // K tiles leave their ring after Q K^T,
constexpr int kAttStagesV = 6;                                               // V tiles after P V: rings of their own
constexpr int kAttThreads = 224;
constexpr int kAttTileBytes = 64 * 64 * 2;                                   // one K or V page tile
constexpr int kAttRingBytes = (kAttStagesK + kAttStagesV) * kAttTileBytes;   // 80 KB; also holds the output exchange
constexpr int kAttSmemBytes = 2 * kAttTileBytes /*Q, 128 rows*/ + kAttRingBytes + 1024 /*sums, maxima*/ +
                              1024 /*alignment*/ + 256 /*barriers*/;
constexpr int kAttBlocks = 64;                                               // block ids kept in shared memory
constexpr float kAttRescaleStep = 6.0f;                                      // log2 units

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
        "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// D[tmem] (+)= A[tmem] * B[smem] for one K step of 16 elements (A: lane = row, 8 columns of bf16 pairs).
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"((uint32_t)accumulate)
      : "memory");
}

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Two independent fp32 operations in one instruction (each half rounds as the scalar form does).
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\t"
      "mov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 fadd2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "add.rn.f32x2 rd, ra, rb;\n\t"
      "mov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 fsub2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "sub.rn.f32x2 rd, ra, rb;\n\t"
      "mov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}

__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

__global__ void __launch_bounds__(kAttThreads, 2) tree_attention_tc_kernel(
    const __grid_constant__ CUtensorMap tmQ,    // q [1][batch * n_nodes][d_model], box 64 x 64
    const __grid_constant__ CUtensorMap tmKV,   // pool [layers][blocks * 2 * heads * 64][64], box 64 x 64
    int layer, const int32_t* __restrict__ block_table, const int32_t* __restrict__ ctx_len,
    const int32_t* __restrict__ nvalid, const int32_t* __restrict__ order /*may be null*/, TreeView tree, KvGeom geom,
    int d_model, float scale_log2e, int splits, int ahead /*pages inside the context may be read before the upstream kernel ends*/,
    bf16* __restrict__ out, float* __restrict__ xch /*split exchange area*/, uint32_t* err) {
  constexpr int SK = kAttStagesK, SV = kAttStagesV;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - smem_u32(smem_raw));
  const uint32_t q_addr = base, ring = base + 2 * kAttTileBytes, ring_v = ring + SK * kAttTileBytes;
  uint8_t* ring_ptr = base_ptr + 2 * kAttTileBytes;
  float* lx = reinterpret_cast<float*>(ring_ptr + kAttRingBytes);            // end of the kernel: [128] partial sums, [128] scaling maxima
  const uint32_t bars = ring + kAttRingBytes + 1024;
  const uint32_t full_k0 = bars, empty_k0 = bars + 8 * SK, full_v0 = bars + 16 * SK, empty_v0 = full_v0 + 8 * SV,
                 bar_q = bars + 16 * (SK + SV), bar_s0 = bar_q + 8, bar_p0 = bar_q + 32,
                 bar_o0 = bar_q + 56, holder = bar_q + 80;     // scores ready / weights ready / P V done: one each per score
                                                               // buffer, so that a phase parity is never one round behind
  volatile uint32_t* holder_ptr = reinterpret_cast<volatile uint32_t*>(ring_ptr + kAttRingBytes + 1024 + 16 * (SK + SV) + 80);

  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  __shared__ int s_blk[kAttBlocks];           // block ids of the first pages
  const int h = blockIdx.x, split = blockIdx.z;
  const int N = tree.n_nodes;

  if (tid == 0) {
    for (int s = 0; s < 2 * (SK + SV); ++s) mbar_init(bars + 8 * s, 1);       // full / empty of the K and V rings
    mbar_init(bar_q, 1); mbar_init(bar_s0, 1); mbar_init(bar_s0 + 8, 1); mbar_init(bar_s0 + 16, 1);
    for (int j = 0; j < 3; ++j) { mbar_init(bar_p0 + 8 * j, 128); mbar_init(bar_o0 + 8 * j, 1); }
    mbar_fence_init();
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmKV);
  }
  __syncthreads();
  // the producer fetches lengths, block ids and first pages while the other warps may still wait for tensor memory that
  // the CTAs before them hold
  uint32_t tmem = 0;
  if (warp != 4) {
    if (warp == 5) { tmem_alloc(holder, 256); tmem_relinquish(); }
    tc_fence_before();
    asm volatile("bar.sync 1, 192;" ::: "memory");
    tc_fence_after();
    tmem = *holder_ptr;
  }

  // Lengths, order and block ids were written before the projection that precedes this kernel (L2 loads: it may still be
  // running); so were, in a decoding pass, the pages that lie inside the context.  q and the tree's own rows come from it.
  // blockIdx.y = (sequence, tile of 64 nodes); longest sequences first
  const int ntile = (N + 63) >> 6, qt = (int)blockIdx.y % ntile, node0 = 64 * qt;
  const int b = order ? __ldcg(order + blockIdx.y / ntile) : (int)blockIdx.y / ntile;
  const int nv = __ldcg(nvalid + b), ctx = __ldcg(ctx_len + b);
  const int total = ctx + nv;
  const int npages = nv > 0 ? (total + kKvBlock - 1) / kKvBlock : 0;
  const int per = (npages + splits - 1) / splits;
  const int p0 = split * per, p1 = min(npages, p0 + per);
  const int ntiles = max(0, p1 - p0);

  float m_use = -INFINITY, l_run = 0.f;       // softmax threads: scaling maximum (log2 units) and partial sum

  if (warp == 4) {
    // ---- TMA producer (one lane); the block ids of this CTA's pages are fetched by the whole warp first
    for (int i = lane; i < min(ntiles, kAttBlocks); i += 32) {
      const long long v = kv_block_of(block_table, geom, b, (p0 + i) * kKvBlock, err);
      s_blk[i] = v < 0 ? 0 : (int)v;          // flagged; stay inside the pool
    }
    __syncwarp();
    if (elect_one() && ntiles > 0) {
      auto row_of = [&](int i) {
        long long blk;
        if (i < kAttBlocks) {
          blk = s_blk[i];
        } else {
          blk = kv_block_of(block_table, geom, b, (p0 + i) * kKvBlock, err);
          if (blk < 0) blk = 0;
        }
        return (int)((blk * 2 * geom.n_heads + h) * kKvBlock);
      };
      auto load_k = [&](int i, int row) {
        mbar_expect_tx(full_k0 + 8 * (i % SK), kAttTileBytes);
        tma_load_3d(ring + (i % SK) * kAttTileBytes, &tmKV, full_k0 + 8 * (i % SK), 0, row, layer);
      };
      auto load_v = [&](int i, int row) {
        mbar_expect_tx(full_v0 + 8 * (i % SV), kAttTileBytes);
        tma_load_3d(ring_v + (i % SV) * kAttTileBytes, &tmKV, full_v0 + 8 * (i % SV), 0, row + geom.n_heads * kKvBlock, layer);
      };
      // the rings' first fill, while the projection is still running (750 tokens at batch 1: 123.5 -> 119.2 ms)
      const int inside = ahead ? min(ntiles, max(0, ctx / kKvBlock - p0)) : 0;
      const int ek = min(inside, SK), ev = min(inside, SV);
      for (int i = 0; i < ev; ++i) {
        const int row = row_of(i);
        if (i < ek) load_k(i, row);
        load_v(i, row);
      }
      grid_dep_wait();
      mbar_expect_tx(bar_q, 2 * kAttTileBytes);
      tma_load_3d(q_addr, &tmQ, bar_q, h * 64, b * N + node0, 0);
      tma_load_3d(q_addr + kAttTileBytes, &tmQ, bar_q, h * 64, b * N + node0, 0);      // the same rows again: lanes 64..127
      for (int i = ek; i < ntiles; ++i) {
        const int row = row_of(i);
        if (i >= SK && !mbar_wait(empty_k0 + 8 * (i % SK), ((i / SK) - 1) & 1, err)) break;   // timed out (recorded): stop issuing
        load_k(i, row);
        if (i < ev) continue;
        if (i >= SV && !mbar_wait(empty_v0 + 8 * (i % SV), ((i / SV) - 1) & 1, err)) break;
        load_v(i, row);
      }
    }
    __syncwarp();
    grid_dep_wait();
  } else if (warp == 5) {
    // ---- P V issuer (one lane): O += P(i) V(i) as soon as the softmax threads have stored P(i)
    grid_dep_wait();
    if (elect_one()) {
      constexpr uint32_t idesc_pv = umma_idesc_bf16(128, 64) | (1u << 16);     // B (V tile) is MN-major
      for (int i = 0; i < ntiles; ++i) {
        if (!mbar_wait(bar_p0 + 8 * (i % 3), (i / 3) & 1, err)) break;
        if (!mbar_wait(full_v0 + 8 * (i % SV), (i / SV) & 1, err)) break;
        tc_fence_after();
        const uint32_t va = ring_v + (i % SV) * kAttTileBytes, pa = tmem + 64 * (i % 3);
#pragma unroll
        for (int k = 0; k < 4; ++k)          // 16 keys per step: 8 TMEM columns of A, 16 rows (2048 bytes) of V
          umma_bf16_ts(tmem + 192, pa + 8 * k, umma_desc_k_sw128(va + 2048 * k), idesc_pv, (i | k) != 0);
#pragma unroll
        for (int k = 0; k < 4; ++k)          // the lo halves of the weights
          umma_bf16_ts(tmem + 192, pa + 32 + 8 * k, umma_desc_k_sw128(va + 2048 * k), idesc_pv, true);
        umma_commit(empty_v0 + 8 * (i % SV));
        umma_commit(bar_o0 + 8 * (i % 3));
      }
    }
  } else if (warp == 6) {
    // ---- Q K^T issuer (one lane): S(i) = Q K(i)^T into score buffer i % 3, up to three pages ahead of P V
    grid_dep_wait();
    if (elect_one()) {
      constexpr uint32_t idesc_qk = umma_idesc_bf16(128, 64);
      bool ok = ntiles == 0 || mbar_wait(bar_q, 0, err);
      for (int i = 0; i < ntiles && ok; ++i) {
        // the buffer held P(i - 3): free once P(i - 3) V(i - 3) has completed
        if (i >= 3 && !mbar_wait(bar_o0 + 8 * (i % 3), ((i - 3) / 3) & 1, err)) break;
        const int s = i % SK;
        if (!mbar_wait(full_k0 + 8 * s, (i / SK) & 1, err)) break;
        tc_fence_after();
        const uint32_t ka = ring + s * kAttTileBytes;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          umma_bf16(tmem + 64 * (i % 3), umma_desc_k_sw128(q_addr + 32 * k), umma_desc_k_sw128(ka + 32 * k), idesc_qk, k != 0);
        umma_commit(empty_k0 + 8 * s);                     // the K tile is free once these MMAs have read it
        umma_commit(bar_s0 + 8 * (i % 3));
      }
    }
  } else {
    // ---- softmax: thread tid owns TMEM lane tid = query row (tid & 63), keys 32*half .. 32*half+31 of each page
    grid_dep_wait();
    const int row = tid & 63, half = tid >> 6;
    unsigned long long alo = 0ull, ahi = 0ull;                     // ancestor-or-self bits of this row's node
    if (node0 + row < nv) tree.anc_of(b, node0 + row, alo, ahi);
    const uint32_t trow = tmem + ((uint32_t)(32 * warp) << 16);
    for (int i = 0; i < ntiles; ++i) {
      if (!mbar_wait(bar_s0 + 8 * (i % 3), (i / 3) & 1, err)) break;
      tc_fence_after();
      const uint32_t tsp = trow + 64 * (i % 3);       // this page's score / weight buffer
      float sc[32];
      tmem_ld32(tsp + 32 * half, sc);
      {
        // the weights' columns of the other key half are zero in this lane; written here, they are off the path from the
        // maximum to the weights (the scores of this lane are in registers by now)
        const uint32_t zero[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          tmem_st8(tsp + 16 * (1 - half) + 8 * u, zero);
          tmem_st8(tsp + 32 + 16 * (1 - half) + 8 * u, zero);
        }
      }
      const int key0 = (p0 + i) * kKvBlock + 32 * half;
      if (key0 + 32 > ctx) {
        // bit j of vis: key key0 + j is visible (context, or an ancestor-or-self tree node; the ancestor
        // word has no bits at or above the node count).  Selects, not branches: the rows of a warp differ.
        const int rel = key0 - ctx;           // > -32 here
        uint32_t vis;
        if (rel >= 0) vis = rel < 128 ? bits32_at(alo, ahi, rel) : 0u;
        else vis = ((1u << (-rel)) - 1u) | (uint32_t)(alo << (-rel));
#pragma unroll
        for (int j = 0; j < 32; ++j) sc[j] = ((vis >> j) & 1u) ? sc[j] : -INFINITY;
      }                                       // else: all 32 keys inside the context, every key visible
      float mx4[4];                           // four chains of three-input maxima over eight scores each
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        mx4[c] = fmax3(sc[8 * c], sc[8 * c + 1], sc[8 * c + 2]);
        mx4[c] = fmax3(mx4[c], sc[8 * c + 3], sc[8 * c + 4]);
        mx4[c] = fmax3(mx4[c], sc[8 * c + 5], sc[8 * c + 6]);
        mx4[c] = fmaxf(mx4[c], sc[8 * c + 7]);
      }
      float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
      if ((p0 + i + 1) * kKvBlock > total && tid < 64) {   // rows of V past the tree may hold anything: zero them
        const int valid = total - (p0 + i) * kKvBlock;
        mbar_wait(full_v0 + 8 * (i % SV), (i / SV) & 1, err);      // the V tile has landed before rows of it are cleared
        if (tid >= valid) {
          uint4* vr = reinterpret_cast<uint4*>(ring_ptr + (SK + i % SV) * kAttTileBytes + tid * 128);
#pragma unroll
          for (int c = 0; c < 8; ++c) vr[c] = make_uint4(0, 0, 0, 0);
        }
        fence_proxy_async_smem();
      }
      // each key half of a row keeps its own scaling maximum (the halves accumulate in separate TMEM lanes
      // and are brought to a common scale once, at the end)
      mx *= scale_log2e;                      // raw scores; the (positive) scale moves into the exponent
      // move the scaling maximum only when the page maximum exceeds it by more than the step
      float factor = 1.f;
      if (mx > m_use + kAttRescaleStep || m_use == -INFINITY) {
        factor = (m_use == -INFINITY) ? 0.f : fast_exp2(m_use - mx);
        if (mx > -INFINITY) m_use = mx;
      }
      if (i > 0 && __any_sync(0xffffffffu, factor != 1.f)) {
        // rescale this row's accumulator, once the previous page's P V has completed
        if (!mbar_wait(bar_o0 + 8 * ((i - 1) % 3), ((i - 1) / 3) & 1, err)) break;
        tc_fence_after();
#pragma unroll 1
        for (int hh = 0; hh < 4; ++hh) {
          float ot[16];
          tmem_ld16(trow + 192 + 16 * hh, ot);
          uint32_t ob[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) ob[e] = __float_as_uint(ot[e] * factor);
          tmem_st16(trow + 192 + 16 * hh, ob);
        }
      }
      l_run *= factor;
      float2 psum4[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};   // four chains of pairs
      const float m_sub = (m_use == -INFINITY) ? 0.f : m_use;      // no visible key yet: every score is -inf, p = 0
      const float2 sc2 = make_float2(scale_log2e, scale_log2e), nm2 = make_float2(-m_sub, -m_sub);
      // this thread's 32 keys sit in columns 16*half .. 16*half+15 of each 32-column group, stored eight at a time
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        uint32_t hv[8], lv[8];
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) {
          // two keys per instruction where the pipe has a paired form (fma, add, sub)
          const int q = 8 * u + jj;
          const float2 x = ffma2(make_float2(sc[2 * q], sc[2 * q + 1]), sc2, nm2);
          const float2 pp = make_float2(fast_exp2(x.x), fast_exp2(x.y));
          psum4[q & 3] = fadd2(psum4[q & 3], pp);
          hv[jj] = pack_bf16(pp.x, pp.y);
          const float2 hh = make_float2(__uint_as_float(hv[jj] << 16), __uint_as_float(hv[jj] & 0xffff0000u));
          const float2 ll = fsub2(pp, hh);
          lv[jj] = pack_bf16(ll.x, ll.y);
        }
        tmem_st8(tsp + 16 * half + 8 * u, hv);
        tmem_st8(tsp + 32 + 16 * half + 8 * u, lv);
      }
      {
        const float2 s01 = fadd2(psum4[0], psum4[1]), s23 = fadd2(psum4[2], psum4[3]);
        const float2 st = fadd2(s01, s23);
        l_run += st.x + st.y;
      }
      tmem_st_wait();
      tc_fence_before();
      mbar_arrive(bar_p0 + 8 * (i % 3));
    }
    if (ntiles > 0) { mbar_wait(bar_o0 + 8 * ((ntiles - 1) % 3), ((ntiles - 1) / 3) & 1, err); tc_fence_after(); }
  }
  __syncwarp();
  grid_dep_launch();
  __syncthreads();                            // the ring is idle from here on (every MMA has completed)

  // ---- output: the rows' two key halves, each with a sum and a scaling maximum, meet in the ring; half a row for each of
  // 128 threads, and tensor memory is given back before the merge (per launch, one thread a row before -> now: batch 8
  // 23.3 -> 22.2 us, batch 32 with 2,340 context tokens 77.2 -> 75.5, batch 64 with 1,300 104.8 -> 102.4)
  float* Ox = reinterpret_cast<float*>(ring_ptr);          // [2][64 rows][64], row r rotated by 4r columns
  if (warp < 4) {
    const uint32_t to = tmem + ((uint32_t)(32 * warp) << 16) + 192;
    lx[tid] = l_run;
    lx[128 + tid] = m_use;
    float4* dst = reinterpret_cast<float4*>(Ox + tid * 64);
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      float o[32];
      tmem_ld32(to + 32 * hh, o);
#pragma unroll
      for (int e = 0; e < 8; ++e)
        dst[(8 * hh + e + tid) & 15] = ntiles > 0 ? make_float4(o[4 * e], o[4 * e + 1], o[4 * e + 2], o[4 * e + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 5) tmem_dealloc(tmem, 256);                  // the accumulator is in shared memory: room for the next CTA
  const int orow = tid >> 1, oh = tid & 1;                 // 128 threads: half a row each
  float4 o4[8];
  if (tid < 128) {
    const float m0 = lx[128 + orow], m1 = lx[192 + orow], mm = fmaxf(m0, m1);
    const float w0 = m0 == -INFINITY ? 0.f : fast_exp2(m0 - mm), w1 = m1 == -INFINITY ? 0.f : fast_exp2(m1 - mm);
    l_run = lx[orow] * w0 + lx[64 + orow] * w1;
    m_use = mm;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int at = (8 * oh + c + orow) & 15;             // (rows r and r + 64 have the same rotation)
      const float4 x = reinterpret_cast<const float4*>(Ox + orow * 64)[at], y = reinterpret_cast<const float4*>(Ox + (64 + orow) * 64)[at];
      o4[c] = make_float4(x.x * w0 + y.x * w1, x.y * w0 + y.y * w1, x.z * w0 + y.z * w1, x.w * w0 + y.w * w1);
    }
  }
  if (splits == 1) {
    if (tid < 128 && node0 + orow < N) {
      const float inv = (node0 + orow < nv && l_run > 0.f) ? 1.f / l_run : 0.f;
      uint4* dst = reinterpret_cast<uint4*>(out + ((long long)b * N + node0 + orow) * d_model + h * 64 + 32 * oh);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float4 x = o4[2 * c], y = o4[2 * c + 1];
        dst[c] = make_uint4(pack_bf16(x.x * inv, x.y * inv), pack_bf16(x.z * inv, x.w * inv), pack_bf16(y.x * inv, y.y * inv),
                            pack_bf16(y.z * inv, y.w * inv));
      }
    }
  } else {
    // this split's result goes to its slot of the exchange area in global memory (it stays in L2):
    // O [64 nodes][64] fp32, then the row sums l[64] and scaling maxima m[64]; the splits of one (head,
    // sequence) meet at a cluster barrier and are merged in a fixed order
    constexpr int kSlot = 64 * 64 + 128;
    float* mine = xch + ((long long)(blockIdx.y * gridDim.x + blockIdx.x) * splits + split) * kSlot;
    if (tid < 128) {
      float4* dst = reinterpret_cast<float4*>(mine + orow * 64 + 32 * oh);
#pragma unroll
      for (int c = 0; c < 8; ++c) dst[c] = o4[c];
      if (oh == 0) { mine[64 * 64 + orow] = l_run; mine[64 * 64 + 64 + orow] = m_use; }
    }
    cluster_sync_all();                        // release / acquire: the peers' slots are visible
    // CTA `split` finishes nodes [split*per_n, (split+1)*per_n): 16 threads per node, four consecutive features each.  All of a
    // thread's nodes (one with eight splits, two with four, four with two) are requested before the first is merged: one
    // round trip to L2 instead of up to four (batch 8, two splits: 14.4 -> 12.9 us per launch).
    const float* first = xch + (long long)(blockIdx.y * gridDim.x + blockIdx.x) * splits * kSlot;
    auto merge = [&](auto splits_c) {
      constexpr int PP = decltype(splits_c)::value, TT = 8 / PP;
      const int e4 = (tid & 15) * 4, n = split * (64 / PP) + (tid >> 4);
      float mm[TT][PP], ll[TT][PP];
      float4 oo[TT][PP];
#pragma unroll
      for (int u = 0; u < TT; ++u)
#pragma unroll
        for (int p = 0; p < PP; ++p) {
          const float* sl = first + (long long)p * kSlot;
          mm[u][p] = __ldcg(sl + 64 * 64 + 64 + n + 8 * u);
          ll[u][p] = __ldcg(sl + 64 * 64 + n + 8 * u);
          oo[u][p] = __ldcg(reinterpret_cast<const float4*>(sl + (n + 8 * u) * 64 + e4));
        }
#pragma unroll
      for (int u = 0; u < TT; ++u) {
        float M = -INFINITY, L = 0.f;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int p = 0; p < PP; ++p) M = fmaxf(M, mm[u][p]);
#pragma unroll
        for (int p = 0; p < PP; ++p) {
          const float w = (mm[u][p] == -INFINITY) ? 0.f : exp2f(mm[u][p] - M);
          L = fmaf(ll[u][p], w, L);
          o.x = fmaf(oo[u][p].x, w, o.x); o.y = fmaf(oo[u][p].y, w, o.y); o.z = fmaf(oo[u][p].z, w, o.z); o.w = fmaf(oo[u][p].w, w, o.w);
        }
        const int node = node0 + n + 8 * u;
        if (node < N) {
          const float inv = (node < nv && L > 0.f) ? 1.f / L : 0.f;
          uint2 v;
          v.x = pack_bf16(o.x * inv, o.y * inv);
          v.y = pack_bf16(o.z * inv, o.w * inv);
          *reinterpret_cast<uint2*>(out + ((long long)b * N + node) * d_model + h * 64 + e4) = v;
        }
      }
    };
    if (tid < 128) {
      if (splits == 8) merge(std::integral_constant<int, 8>{});
      else if (splits == 4) merge(std::integral_constant<int, 4>{});
      else merge(std::integral_constant<int, 2>{});
    }
  }
}

}  // namespace vadusa
