// Tolerance verification (Algorithm 1), choice of the longest / leftmost accepted
// path (Sec. II-C) and the commit of its K/V rows into the cache.
#pragma once
#include "select.cuh"

namespace vadusa {

struct AcceptOut {            // optional user-visible outputs (any may be null)
  int32_t* accept_len;        // [batch]
  int32_t* path_nodes;        // [batch][kMaxPath]
  int32_t* path_tokens;       // [batch][kMaxPath]
  long long* kv_slots;        // [batch][kMaxPath]
  unsigned long long* edge_bits;  // [batch][edge_words]
  long long edge_words;       // 1 (trees of up to 64 nodes) or 2 (a full word: the struct's bytes key the graph cache)
  int32_t* next_root;         // [batch]
};

struct SeqState {             // device state of the batch (all [batch] unless noted)
  int32_t* ctx_len;
  int32_t* nvalid;            // tree nodes scored for the sequence this iteration (0: inactive)
  int32_t* gen_count;         // tokens generated so far
  int32_t* commit_base;       // ctx_len as the acceptance saw it: the commit's blocks read this while one of them moves ctx_len on
  int32_t* commit_nv;         // the same of nvalid
  int32_t* node_ok;           // [batch][kMaxNodes]: the node is among its parent's draws
  int32_t* node_top;          // [batch][kMaxNodes]: the node's first draw, where accept_kernel forms it
  int32_t* out_tokens;        // [batch][out_cap] generated tokens (may be null)
  int32_t* done_count;        // [3] scalars: sequences that reached the target, iterations finished, blocks arrived in this one
  int32_t* progress;          // pinned host memory [2] that gets (iterations finished, sequences done) after every commit, or null
  int out_cap;
  int target;                 // stop a sequence after this many tokens (0: never)
  unsigned long long* stats;  // [2][kStatDepth][kStatTopk]: acceptance tests applied / passed, by (draft head, rank)
};

// (a grid of more than two blocks of 512 per SM is bound by throughput: smaller blocks, fewer barriers' worth of idling)
inline int accept_threads(int vocab, int blocks) { return vocab > kSelectWide ? 1024 : blocks <= 4 * 148 ? 512 : 256; }

// grid = (most inner nodes of a tree, batch): one block per node that has children; or (nodes, batch) with inner = null: a
// block per node, which then also leaves the node's first draw (the token that continues the sequence if it wins).  The draws of every such node are
// formed at once, whether or not it turns out to be accepted (the keys of its logits row predict absolute position
// ctx_len + depth + 1): child token c is accepted iff fewer than tau tokens precede it in key order (and it lies in the
// nucleus).  commit_kernel walks the tree.  Bound by latency: one block per sequence that formed the keys of one
// accepted parent after another and walked the tree took 18-26 us at 1025 tokens (three or four parents, 16 block barriers
// each), 178 us with the nucleus at 2049, 945 us at 16001.  Few tokens per thread (the two logarithms of a token's noise
// are a chain of 400 cycles) and short code (it runs once per block, from a cold instruction cache) matter more than the
// operations.  The noise is formed, and everything but the logits is read, while the product that makes the logits still
// runs: that product waits for its own predecessors before it lets this kernel start.
// Dynamic shared memory: row_keys_smem.  accept_threads(vocab) threads.
__global__ void __launch_bounds__(1024) accept_kernel(
    const float* __restrict__ logits, int ld, int vocab, const int32_t* tokens, TreeView tree,
    const int32_t* __restrict__ inner /*[kMaxNodes] per tree, -1 behind the last; or null*/, SamplingDev sp, SeqState st) {
  extern __shared__ float keys[];          // [ld] keys, then [ld] logits (nucleus only)
  __shared__ SelectScratch sc;
  __shared__ int s_node[kMaxNodes], s_tok[kMaxNodes], s_cnt[kMaxNodes], s_n, s_depth;
  const int b = blockIdx.y, N = tree.n_nodes, tid = threadIdx.x, lane = tid & 31;
  const int to = tree.off(b);
  // (L2 loads: these were written by kernels before the one that may still be running)
  const int nv = __ldcg(st.nvalid + b), S = __ldcg(st.ctx_len + b);
  const int p = inner ? inner[(tree.per_seq ? b * kMaxNodes : 0) + blockIdx.x] : (int)blockIdx.x;
  int par = -1, tok = 0, dep = 0;
  if (tid < N) {
    par = tree.parent[to + tid]; dep = tree.depth[to + tid];
    tok = __ldcg(tokens + (long long)b * N + tid);
  }
  if (tid == 0) s_n = 0;
  __syncthreads();
  const bool live = p >= 0 && p < nv;
  if (live && tid < nv) {
    if (tid == p) s_depth = dep;
    if (par == p) { const int i = atomicAdd(&s_n, 1); s_node[i] = tid; s_tok[i] = tok; s_cnt[i] = 0; }
  }
  __syncthreads();
  const uint64_t rs = noise_row_state(sp.seed, b, S + s_depth + 1);
  if (live && sp.accept_rule == 0) row_noise(vocab, rs, sp, keys);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (blockIdx.x == 0 && tid == 0) { st.commit_base[b] = S; st.commit_nv[b] = nv; }
  if (!live) return;
  row_keys(base_row(logits + ((long long)b * N + p) * ld, sp, b), vocab, rs, sp, sp.accept_rule == 0, keys, keys + ld, sc);
  const int nchild = s_n;
#pragma unroll 1
  for (int i = 0; i < nchild; ++i) {
    const int c = s_tok[i];
    if (c < 0 || c >= vocab) continue;     // not a speech token: never accepted
    const float kc = keys[c];
    int cnt = 0;
#pragma unroll 4
    for (int j = tid; j < vocab; j += blockDim.x) cnt += precedes(keys[j], j, kc, c) ? 1 : 0;
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0 && cnt) atomicAdd(&s_cnt[i], cnt);
  }
  __syncthreads();
  if (tid < nchild) {
    const int c = s_tok[tid];
    st.node_ok[b * kMaxNodes + s_node[tid]] = c >= 0 && c < vocab && s_cnt[tid] < sp.tau && keys[c] > -INFINITY ? 1 : 0;
  }
  if (!inner) {
    const int first = first_key(keys, vocab, sc);
    if (tid == 0) st.node_top[b * kMaxNodes + p] = first;
  }
}

// One thread per sequence, after it has counted the sequence's end: the last of the batch tells the host.
__device__ __forceinline__ void report_progress(const SeqState& st) {
  if (!st.progress) return;
  __threadfence();
  if (atomicAdd(st.done_count + 2, 1) != (int)gridDim.y - 1) return;
  st.done_count[2] = 0;
  const int it = st.done_count[1] + 1;
  st.done_count[1] = it;
  const unsigned long long both = (uint32_t)it | ((unsigned long long)(uint32_t)atomicAdd(st.done_count, 0) << 32);
  *reinterpret_cast<volatile unsigned long long*>(st.progress) = both;
}

// floats of the carried logits that one block of commit_kernel copies
constexpr int kCommitLogits = 4096;

// grid = (n_layers + ceil(ld / kCommitLogits) + 1, batch).  Every block finds the winner for itself: a node is accepted
// iff it and all its ancestors are among their parents' draws (one mask test per node), the deepest accepted node wins,
// the smallest index among equally deep ones.  Then
//   x < n_layers: move the K/V rows of the winning path of layer x from slot base + path[j] to slot base + j, 16 bytes per
//     thread and step; a thread always handles the same 16-byte column of every row, and rows are read in ascending j
//     no later than they are overwritten;
//   the next blocks: carry the winner's hidden state and logits, 16 bytes per thread and step;
//   the last: outputs, statistics, the sequence's new state.  A sequence whose path commits EOS (when EOS is not
//     masked) or reaches the token target becomes inactive (nvalid = 0).
// next_root: accept_kernel has left it with the node (have_top), or the last block draws it here.
// Dynamic shared memory: row_keys_smem if it has to draw, else none.
template <typename T>
__global__ void __launch_bounds__(1024) commit_kernel(
    T* __restrict__ pool, KvGeom geom, const int32_t* __restrict__ block_table, SeqState st, int n_layers, TreeView tree,
    const int32_t* tokens, SamplingDev sp, const int32_t* __restrict__ forced_best, int have_top, AcceptOut out,
    const T* __restrict__ hfinal, int d_model, const float* __restrict__ logits, int ld, int vocab,
    T* __restrict__ hstar, float* __restrict__ logits_star, uint32_t* err) {
  extern __shared__ float keys[];
  __shared__ unsigned long long s_anc[kMaxNodes][2];
  __shared__ int s_depth[kMaxNodes], s_path[kMaxPath], s_top[kMaxNodes / 32], s_end;
  __shared__ uint32_t s_edge[kMaxNodes / 32], s_acc[kMaxNodes / 32];
  const int b = blockIdx.y, N = tree.n_nodes, tid = threadIdx.x, warp = tid >> 5;
  const int to = tree.off(b);
  int par = -1, dep = 0, tok = -1;
  unsigned long long a0 = ~0ull, a1 = ~0ull;
  if (tid < N) {
    par = tree.parent[to + tid]; dep = tree.depth[to + tid];
    tree.anc_of(b, tid, a0, a1);
    tok = __ldcg(tokens + (long long)b * N + tid);     // (written before the product of the vocabulary head)
    s_anc[tid][0] = a0; s_anc[tid][1] = a1;
    s_depth[tid] = dep;
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int nv = st.commit_nv[b], S = st.commit_base[b];
  const int fb = forced_best ? forced_best[b] : -1;
  const bool ok = tid == 0 || (tid < N && par >= 0 && st.node_ok[b * kMaxNodes + tid] != 0);
  const int nlog = (ld + kCommitLogits - 1) / kCommitLogits, part = (int)blockIdx.x - n_layers;
  if (nv == 0) {
    if (part != nlog) return;
    if (tid == 0) {
      if (out.accept_len) out.accept_len[b] = 0;
      if (out.edge_bits) for (int w = 0; w < (int)out.edge_words; ++w) out.edge_bits[b * out.edge_words + w] = 0ull;
      if (out.next_root) out.next_root[b] = -1;
      report_progress(st);
    }
    if (tid < kMaxPath) {
      if (out.path_nodes) out.path_nodes[b * kMaxPath + tid] = -1;
      if (out.path_tokens) out.path_tokens[b * kMaxPath + tid] = -1;
      if (out.kv_slots) out.kv_slots[b * kMaxPath + tid] = -1;
    }
    return;
  }
  const bool forced = fb >= 0 && fb < nv;
  if (tid < kMaxNodes) {
    const uint32_t e = __ballot_sync(0xffffffffu, ok && tid < nv);
    if ((tid & 31) == 0) s_edge[warp] = e;
  }
  if (tid == 0) s_end = kMaxPath;
  __syncthreads();
  bool acc = false;
  if (tid < kMaxNodes) {
    const unsigned long long e0 = s_edge[0] | ((unsigned long long)s_edge[1] << 32), e1 = s_edge[2] | ((unsigned long long)s_edge[3] << 32);
    acc = tid < nv && (fb < 0 ? ((a0 & ~e0) | (a1 & ~e1)) == 0ull : tid == 0);
    const uint32_t w = __ballot_sync(0xffffffffu, acc);
    // deepest first, then the smallest index
    const int top = __reduce_max_sync(0xffffffffu, acc ? (dep << 8) | (255 - tid) : 0);
    if ((tid & 31) == 0) { s_acc[warp] = w; s_top[warp] = top; }
  }
  __syncthreads();
  int best = forced ? fb : 255 - (max(max(s_top[0], s_top[1]), max(s_top[2], s_top[3])) & 255);
  // the path is the winner's ancestors, a node per depth
  const bool on = tid < nv && bit_at(s_anc[best][0], s_anc[best][1], tid) && dep < kMaxPath;
  if (on) {
    s_path[dep] = tid;
    // EOS not masked: the sequence ends with the first EOS on the path; what follows it is dropped
    if (!sp.eos_masked && tok == sp.eos_id) atomicMin(&s_end, dep);
  }
  int len = min(s_depth[best] + 1, kMaxPath);
  __syncthreads();
  const bool eos = s_end < len;
  if (eos) { len = s_end + 1; best = s_path[s_end]; }

  if (part >= 0 && part < nlog) {
    const long long m = (long long)b * N + best;
    // (d_model and ld are multiples of 64 and 128: whole 16-byte pieces)
    const uint4* hs = reinterpret_cast<const uint4*>(hfinal + m * d_model);
    uint4* hd = reinterpret_cast<uint4*>(hstar + (long long)b * d_model);
    if (part == 0)
      for (int i = tid; i < d_model * (int)sizeof(T) / 16; i += blockDim.x) hd[i] = hs[i];
    const uint4* ls = reinterpret_cast<const uint4*>(logits + m * ld);
    uint4* l = reinterpret_cast<uint4*>(logits_star + (long long)b * ld);
    const int end = min(ld, (part + 1) * kCommitLogits) / 4;
#pragma unroll 4
    for (int i = part * (kCommitLogits / 4) + tid; i < end; i += blockDim.x) l[i] = ls[i];
    return;
  }
  if (part == nlog) {
    int g = 0;
    if (st.out_tokens || tid == 0) g = st.gen_count[b];
    if (tid < kMaxPath) {
      const bool in = tid < len;
      if (out.path_nodes) out.path_nodes[b * kMaxPath + tid] = in ? s_path[tid] : -1;
      if (out.kv_slots) {
        long long slot = -1;
        if (in) {
          const long long blk = kv_block_of(block_table, geom, b, S + tid, err);
          slot = blk < 0 ? -1 : blk * kKvBlock + (S + tid) % kKvBlock;
        }
        out.kv_slots[b * kMaxPath + tid] = slot;
      }
      if (out.path_tokens && !in) out.path_tokens[b * kMaxPath + tid] = -1;
    }
    if (on && dep < len) {
      if (out.path_tokens) out.path_tokens[b * kMaxPath + dep] = tok;
      if (st.out_tokens && g + dep < st.out_cap) st.out_tokens[(long long)b * st.out_cap + g + dep] = tok;
    }
    // tests applied and passed, by (draft head, rank)
    if (st.stats && fb < 0 && tid < nv && par >= 0 && ((s_acc[par >> 5] >> (par & 31)) & 1u)) {
      const int d = dep - 1, r = tree.rank[to + tid];
      if (d < kStatDepth && r >= 0 && r < kStatTopk) {
        atomicAdd(st.stats + d * kStatTopk + r, 1ull);
        if (acc) atomicAdd(st.stats + (kStatDepth + d) * kStatTopk + r, 1ull);
      }
    }
    __syncthreads();                             // (every thread has read gen_count)
    if (tid == 0) {
      st.ctx_len[b] = S + len;
      st.gen_count[b] = g + len;
      if (eos || (st.target > 0 && g + len >= st.target)) { st.nvalid[b] = 0; atomicAdd(st.done_count, 1); }
      if (out.accept_len) out.accept_len[b] = len;
      if (out.edge_bits)
        for (int w = 0; w < (int)out.edge_words; ++w)
          out.edge_bits[b * out.edge_words + w] = s_acc[2 * w] | ((unsigned long long)s_acc[2 * w + 1] << 32);
      report_progress(st);
    }
    if (out.next_root && have_top) {
      if (tid == 0) out.next_root[b] = st.node_top[b * kMaxNodes + best];
    } else if (out.next_root) {
      __shared__ SelectScratch sc;
      const uint64_t rs = noise_row_state(sp.seed, b, S + len);
      row_noise(vocab, rs, sp, keys);
      row_keys(base_row(logits + ((long long)b * N + best) * ld, sp, b), vocab, rs, sp, true, keys, keys + ld, sc);
      const int next = first_key(keys, vocab, sc);
      if (tid == 0) out.next_root[b] = next;
    }
    return;
  }
  __shared__ long long s_src[kMaxPath], s_dst[kMaxPath];
  if (tid < kMaxPath) {
    const int j = tid;
    long long src = -1, dst = -1;
    if (j < len) {
      const int node = s_path[j];
      if (node != j) {
        const long long bs = kv_block_of(block_table, geom, b, S + node, err);
        const long long bd = kv_block_of(block_table, geom, b, S + j, err);
        if (bs >= 0 && bd >= 0) {
          src = geom.elem(bs, 0, 0, (S + node) % kKvBlock);
          dst = geom.elem(bd, 0, 0, (S + j) % kKvBlock);
        }
      }
    }
    s_src[j] = src; s_dst[j] = dst;
  }
  __syncthreads();
  T* lp = pool + (long long)blockIdx.x * geom.layer_stride;
  const int cpr = geom.head_dim * (int)sizeof(T) / 16;            // 16-byte chunks per row
  const int chunks = 2 * geom.n_heads * cpr;
  const long long row_stride = (long long)kKvBlock * geom.head_dim;   // elements between (kv, head) tiles
  for (int c = tid; c < chunks; c += blockDim.x) {
    const int tile = c / cpr, cc = c % cpr;
    for (int j0 = 1; j0 < len; j0 += 4) {                         // four rows in flight
      uint4 v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (j0 + i < len && s_src[j0 + i] >= 0) v[i] = *(reinterpret_cast<const uint4*>(lp + s_src[j0 + i] + tile * row_stride) + cc);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (j0 + i < len && s_src[j0 + i] >= 0) *(reinterpret_cast<uint4*>(lp + s_dst[j0 + i] + tile * row_stride) + cc) = v[i];
    }
  }
}

// Prefill bookkeeping.  gather: row r of the pass gets the block-table row of its sequence.
__global__ void prefill_gather_kernel(const int32_t* __restrict__ block_table, const int32_t* seq_of,
                                      int max_blocks, int32_t* __restrict__ out) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int r = blockIdx.x, b = seq_of[r];
  for (int i = threadIdx.x; i < max_blocks; i += blockDim.x) out[(long long)r * max_blocks + i] = block_table[(long long)b * max_blocks + i];
}

// pick: rows m[i] of the attention outputs and of the residual stream, one behind the other.  grid = rows.
template <typename T>
__global__ void prefill_pick_kernel(const int32_t* m, const T* o, const float* x, int d, T* __restrict__ a, float* __restrict__ xg) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const long long i = blockIdx.x, r = m[i];
  for (int c = threadIdx.x; c < d * (int)sizeof(T) / 16; c += blockDim.x)
    reinterpret_cast<uint4*>(a + i * d)[c] = reinterpret_cast<const uint4*>(o + r * d)[c];
  for (int c = threadIdx.x; c < d / 4; c += blockDim.x)
    reinterpret_cast<float4*>(xg + i * d)[c] = reinterpret_cast<const float4*>(x + r * d)[c];
}

// finish: what the last token of a prefix leaves, as its sequence's state: hidden state, base-head logits, context length.
// by_row: hidden state and logits lie at the token's row of the pass (m), else at the index of the prefix.  grid = ends.
template <typename T>
__global__ void prefill_finish_kernel(const int32_t* m, const int32_t* seq, const int32_t* len, int by_row, const T* hfinal,
                                      int d_model, const float* logits, int ld, T* __restrict__ hstar,
                                      float* __restrict__ logits_star, int32_t* __restrict__ ctx_len) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int i = blockIdx.x, b = seq[i];
  const long long r = by_row ? m[i] : i;
  for (int c = threadIdx.x; c < d_model * (int)sizeof(T) / 16; c += blockDim.x)
    reinterpret_cast<uint4*>(hstar + (long long)b * d_model)[c] = reinterpret_cast<const uint4*>(hfinal + r * d_model)[c];
  for (int c = threadIdx.x; c < ld / 4; c += blockDim.x)
    reinterpret_cast<float4*>(logits_star + (long long)b * ld)[c] = reinterpret_cast<const float4*>(logits + r * ld)[c];
  if (threadIdx.x == 0) ctx_len[b] = len[i];
}

}  // namespace vadusa
