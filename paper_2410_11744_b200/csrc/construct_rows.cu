// Construction of the draft token tree with one CTA of 1024 threads per request: the form for large batches of large trees,
// whose rows leave the clusters of construct.cu no room for hot CTAs.  A draw takes 7.4 us here (vocabulary 32000) and
// 3.4 in such a cluster, but 15 clusters run at once against 148 CTAs: 38 trees of 2047 distinct rows take 15.2 ms here
// and 20.8 there, 148 of them 15.3 and 68.7.
//
// What is computed is what construct.cu computes.  A "slot" (v, position, attempt) is the next sampling at a position.
//   greedy:    the whole block scans the slots (<= 4096) for the largest v, loads the position's row, strikes out the
//     tokens of its children and draws.
//   threshold: layer by layer; a position's row stays in registers while it draws.
// The residual lives in registers (thread t owns float4 chunks t, t + 1024, ...); a draw is an inverse-CDF search in token
// order (row totals, then one block scan).  The tokens a position has used are struck out in constant time whatever their
// number: every thread looks at one or two nodes of the tree, and where a node is a child of the position it sets the
// token's bit in the word of the thread that owns the token; after a barrier a thread zeroes what its word marks.
// What bounds it: block barriers, some twenty a draw.
#include "vocab_ops.cuh"

namespace dyspec {

namespace {

constexpr int kVThreads = 1024;
constexpr int kMaxChunks = 8;

struct VocabScratch {          // shared memory used by the helpers below
  double rows[kMaxChunks][32];
  double rowtot[kMaxChunks];
  double scan[32];
  int pick;
  float pub[2];
};

__device__ __forceinline__ void load_row(float4 (&R)[kMaxChunks], const float* row, int vocab) {
  const int n_vec = vocab >> 2;
#pragma unroll
  for (int k = 0; k < kMaxChunks; ++k) {
    const int v4 = k * kVThreads + int(threadIdx.x);
    R[k] = v4 < n_vec ? __ldg(reinterpret_cast<const float4*>(row) + v4) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// Element `token` of the row: its owner reads (and optionally zeroes) it and publishes it; every
// thread gets the value.  Contains block barriers.
__device__ __forceinline__ float take_element(float4 (&R)[kMaxChunks], int token, bool zero_it, VocabScratch& s) {
  const int y4 = token >> 2, yk = y4 / kVThreads, yt = y4 - yk * kVThreads, ye = token & 3;
  if (int(threadIdx.x) == yt) {
    float val = 0.f;
#pragma unroll
    for (int k = 0; k < kMaxChunks; ++k) {
      if (k == yk) {
        val = ye == 0 ? R[k].x : ye == 1 ? R[k].y : ye == 2 ? R[k].z : R[k].w;
        if (zero_it) {
          if (ye == 0) R[k].x = 0.f; else if (ye == 1) R[k].y = 0.f; else if (ye == 2) R[k].z = 0.f; else R[k].w = 0.f;
        }
      }
    }
    s.pub[0] = val;
  }
  __syncthreads();
  const float v = s.pub[0];
  __syncthreads();
  return v;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Inverse-CDF draw in token order: the first token v with cumsum(R)[v] > u * sum(R) (the last token if
// rounding leaves none).  Row totals come from one reduction, then one block scan inside the row that
// holds the crossing.  The sums are carried in fp64: tokens of a 32000-word vocabulary have CDF
// intervals of ~1e-5 and less, which fp32 prefix sums (error ~1e-6 of the total) would not resolve
// reproducibly; fp64 runs at half the fp32 rate on this part and the draw is a few dozen adds per
// thread.  Returns the token; `total` receives sum(R).  Contains block barriers.
__device__ __forceinline__ int sample_inverse_cdf(const float4 (&R)[kMaxChunks], int vocab, float u, double& total,
                                                  VocabScratch& s) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_chunks = ((vocab >> 2) + kVThreads - 1) / kVThreads;
#pragma unroll
  for (int k = 0; k < kMaxChunks; ++k) {
    const double w_ = warp_sum_d((double(R[k].x) + double(R[k].y)) + (double(R[k].z) + double(R[k].w)));
    if (lane == 0) s.rows[k][warp] = w_;
  }
  __syncthreads();
  if (warp < kMaxChunks) {
    const double w_ = warp_sum_d(s.rows[warp][lane]);
    if (lane == 0) s.rowtot[warp] = w_;
  }
  if (tid == 0) s.pick = 0x7fffffff;
  __syncthreads();
  double tot = 0.0;
#pragma unroll
  for (int k = 0; k < kMaxChunks; ++k) tot += s.rowtot[k];
  total = tot;
  const double target = double(u) * tot;
  int krow = n_chunks - 1;
  double before = 0.0;
  {
    double acc = 0.0;
    bool found = false;
#pragma unroll
    for (int k = 0; k < kMaxChunks; ++k) {
      if (k < n_chunks && !found) {
        if (acc + s.rowtot[k] > target) { krow = k; before = acc; found = true; }
        else acc += s.rowtot[k];
      }
    }
    if (!found) before = acc - s.rowtot[n_chunks - 1];
  }
  double mine = 0.0;
  float4 rv = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int k = 0; k < kMaxChunks; ++k)
    if (k == krow) rv = R[k];
  mine = (double(rv.x) + double(rv.y)) + (double(rv.z) + double(rv.w));
  double incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  __syncthreads();
  if (lane == 31) s.scan[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const double w_ = s.scan[lane];
    double x = w_;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double t = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += t;
    }
    s.scan[lane] = x - w_;                                     // mass of the warps before this one
  }
  __syncthreads();
  double cum = before + s.scan[warp] + (incl - mine);          // mass before this thread's 4 tokens
  const int v0 = (krow * kVThreads + tid) * 4;
  int pick = 0x7fffffff;
  const float e4[4] = {rv.x, rv.y, rv.z, rv.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    cum += double(e4[e]);
    if (pick == 0x7fffffff && v0 + e < vocab && cum > target) pick = v0 + e;
  }
  if (pick != 0x7fffffff) atomicMin(&s.pick, pick);
  __syncthreads();
  const int y = min(s.pick, vocab - 1);
  __syncthreads();
  return y;
}

struct TreeOut {
  int32_t* parents;
  int32_t* tokens;
  float* values;
  float* child_values;
  int32_t* rows;
};

__device__ __forceinline__ void write_node(const TreeOut& o, size_t base, int k, int parent, int token, float v, float cv,
                                           int row) {
  o.parents[base + k] = parent;
  o.tokens[base + k] = token;
  o.values[base + k] = v;
  o.child_values[base + k] = cv;
  o.rows[base + k] = row;
}

}  // namespace

__global__ void __launch_bounds__(kVThreads, 1)
build_tree_greedy_rows_kernel(const float* __restrict__ draft_table, int n_rows, int vocab, const float* __restrict__ uniforms,
                         int n_uniforms, const int32_t* __restrict__ root_row, int m, TreeOut out,
                         int32_t* __restrict__ n_nodes_out) {
  extern __shared__ __align__(16) uint8_t csm[];
  // slots: value, position, attempt; per node: row id, token, the position it was drawn at
  const int max_slots = 2 * m + 2;
  double* s_v = reinterpret_cast<double*>(csm);                     // [max_slots]   (-1 = taken); fp64 like the draws
  int16_t* s_pos = reinterpret_cast<int16_t*>(s_v + max_slots);     // [max_slots]
  int16_t* s_att = s_pos + max_slots;                               // [max_slots]
  int32_t* s_row = reinterpret_cast<int32_t*>(s_att + max_slots + (max_slots & 1));   // [m + 1]
  int32_t* s_tok = s_row + (m + 1);                                 // [m + 1]
  int16_t* s_ppos = reinterpret_cast<int16_t*>(s_tok + (m + 1));    // [m + 1] the position (parent) a node was drawn at
  __shared__ uint32_t s_kill[kVThreads];                            // bit 4 k + e of word t: element e of thread t's chunk k is used up
  __shared__ VocabScratch s_vs;
  __shared__ double s_bv[33];
  __shared__ int s_bi[33];

  const int r = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t base = size_t(r) * (m + 1);
  if (tid == 0) {
    s_row[0] = ((root_row[r] % n_rows) + n_rows) % n_rows;        // non-negative remainder: any int32 maps to a row
    s_tok[0] = 0;
    s_ppos[0] = -1;
    s_v[0] = 1.0; s_pos[0] = 0; s_att[0] = 0;
    write_node(out, base, 0, -1, 0, 1.f, 1.f, s_row[0]);
  }
  __syncthreads();
  int n_slots = 1, n_created = 0;

  for (int step = 0; step < m; ++step) {
    // ---- the slot with the largest value (ties: lowest index = pushed first)
    double bv = -1.0;
    int bi = 0x7fffffff;
    for (int i = tid; i < n_slots; i += kVThreads) {
      const double v_ = s_v[i];
      if (v_ > bv) { bv = v_; bi = i; }                          // i increases: the first of equal values is kept
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double tv = __shfl_xor_sync(0xffffffffu, bv, o);
      const int ti = __shfl_xor_sync(0xffffffffu, bi, o);
      if (tv > bv || (tv == bv && ti < bi)) { bv = tv; bi = ti; }
    }
    __syncthreads();
    if (lane == 0) { s_bv[warp] = bv; s_bi[warp] = bi; }
    __syncthreads();
    if (warp == 0) {
      double v_ = s_bv[lane];
      int i_ = s_bi[lane];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double tv = __shfl_xor_sync(0xffffffffu, v_, o);
        const int ti = __shfl_xor_sync(0xffffffffu, i_, o);
        if (tv > v_ || (tv == v_ && ti < i_)) { v_ = tv; i_ = ti; }
      }
      if (lane == 0) { s_bv[32] = v_; s_bi[32] = i_; }
    }
    __syncthreads();
    if (s_bv[32] < 0.0) break;                                   // no live slot (cannot happen before m nodes exist)
    const int slot = s_bi[32];
    const double v = s_v[slot];
    const int pos = s_pos[slot], attempt = s_att[slot];
    const int prow = s_row[pos];
    __syncthreads();
    if (tid == 0) s_v[slot] = -1.0;

    // ---- residual of the position: its row with the tokens of its existing children zeroed
    float4 R[kMaxChunks];
    load_row(R, draft_table + size_t(prow) * vocab, vocab);
    if (attempt > 0) {                                           // (a first sampling has nothing to strike out)
      s_kill[tid] = 0u;
      __syncthreads();
      for (int c = 1 + tid; c <= n_created; c += kVThreads)
        if (s_ppos[c] == pos) {
          const int yc = s_tok[c], y4 = yc >> 2;
          atomicOr(&s_kill[y4 % kVThreads], 1u << ((y4 / kVThreads) * 4 + (yc & 3)));
        }
      __syncthreads();
      const uint32_t kill = s_kill[tid];
      if (kill) {
#pragma unroll
        for (int k = 0; k < kMaxChunks; ++k) {
          if ((kill >> (4 * k)) & 1u) R[k].x = 0.f;
          if ((kill >> (4 * k + 1)) & 1u) R[k].y = 0.f;
          if ((kill >> (4 * k + 2)) & 1u) R[k].z = 0.f;
          if ((kill >> (4 * k + 3)) & 1u) R[k].w = 0.f;
        }
      }
    }
    double total;
    const float u = uniforms[draft_uniform_index(uint32_t(prow), uint32_t(attempt), uint32_t(n_uniforms))];
    const int y = sample_inverse_cdf(R, vocab, u, total, s_vs);
    const float py = take_element(R, y, false, s_vs);
    const double rr = total > 0.0 ? double(py) / total : 0.0;

    // ---- the new node and the two slots it opens
    const int k = ++n_created;
    if (tid == 0) {
      const int krow = int(draft_child_hash(uint32_t(prow), uint32_t(y)) % uint32_t(n_rows));
      s_row[k] = krow;
      s_tok[k] = y;
      s_ppos[k] = int16_t(pos);
      write_node(out, base, k, pos, y, float(v), float(v * rr), krow);
      int ns = n_slots;
      if (1.0 - rr > 0.0) { s_v[ns] = v * (1.0 - rr); s_pos[ns] = int16_t(pos); s_att[ns] = int16_t(attempt + 1); ++ns; }
      s_v[ns] = v * rr; s_pos[ns] = int16_t(k); s_att[ns] = 0;
    }
    n_slots += (1.0 - rr > 0.0) ? 2 : 1;
    __syncthreads();
  }
  if (tid == 0) n_nodes_out[r] = n_created + 1;
}

__global__ void __launch_bounds__(kVThreads, 1)
build_tree_threshold_rows_kernel(const float* __restrict__ draft_table, int n_rows, int vocab, const float* __restrict__ uniforms,
                            int n_uniforms, const int32_t* __restrict__ root_row, float threshold, int max_nodes,
                            TreeOut out, int32_t* __restrict__ n_nodes_out) {
  extern __shared__ __align__(16) uint8_t csm[];
  int32_t* s_row = reinterpret_cast<int32_t*>(csm);                 // [max_nodes + 1]
  double* s_cv = reinterpret_cast<double*>(csm + ((size_t(max_nodes + 1) * 4 + 7) & ~size_t(7)));   // [max_nodes + 1] value of the first sampling under a node
  __shared__ VocabScratch s_vs;

  const int r = blockIdx.x, tid = threadIdx.x;
  const size_t base = size_t(r) * (max_nodes + 1);
  if (tid == 0) {
    s_row[0] = ((root_row[r] % n_rows) + n_rows) % n_rows;        // non-negative remainder: any int32 maps to a row
    s_cv[0] = 1.0;
    write_node(out, base, 0, -1, 0, 1.f, 1.f, s_row[0]);
  }
  __syncthreads();
  int n_created = 0;
  int layer_begin = 0, layer_end = 1;                               // nodes [layer_begin, layer_end) are the current leaves
  while (layer_begin < layer_end && n_created < max_nodes) {
    for (int node = layer_begin; node < layer_end && n_created < max_nodes; ++node) {
      double v = s_cv[node];
      if (!(v >= double(threshold))) continue;
      const int prow = s_row[node];
      float4 R[kMaxChunks];
      load_row(R, draft_table + size_t(prow) * vocab, vocab);
      int attempt = 0;
      while (v >= double(threshold) && n_created < max_nodes) {
        double total;
        const float u = uniforms[draft_uniform_index(uint32_t(prow), uint32_t(attempt), uint32_t(n_uniforms))];
        const int y = sample_inverse_cdf(R, vocab, u, total, s_vs);
        const float py = take_element(R, y, true, s_vs);            // drawn tokens leave the residual
        const double rr = total > 0.0 ? double(py) / total : 0.0;
        const int k = ++n_created;
        if (tid == 0) {
          const int krow = int(draft_child_hash(uint32_t(prow), uint32_t(y)) % uint32_t(n_rows));
          s_row[k] = krow;
          s_cv[k] = v * rr;
          write_node(out, base, k, node, y, float(v), float(v * rr), krow);
        }
        v = v * (1.0 - rr);
        ++attempt;
        if (!(1.0 - rr > 0.0)) break;
      }
    }
    __syncthreads();
    layer_begin = layer_end;
    layer_end = n_created + 1;
  }
  if (tid == 0) n_nodes_out[r] = n_created + 1;
}

size_t build_tree_greedy_smem(int m) {
  const size_t max_slots = 2 * size_t(m) + 2;          // value (8 bytes) + position and attempt (2 + 2) per slot
  return 12 * max_slots + 10 * size_t(m + 1) + 64;     // row and token (4 + 4) + the 2-byte position per node
}

cudaError_t launch_build_tree_greedy_rows(const float* draft_table, int n_rows, int vocab, const float* uniforms, int n_uniforms,
                                     const int32_t* root_row, int n_req, int m, int32_t* parents, int32_t* tokens,
                                     float* values, float* child_values, int32_t* rows, int32_t* n_nodes,
                                     cudaStream_t stream) {
  if (n_req <= 0) return cudaSuccess;
  const size_t smem = build_tree_greedy_smem(m);
  static DynSmemGrant grant;
  if (cudaError_t e = grant.ensure(build_tree_greedy_rows_kernel, smem); e != cudaSuccess) return e;
  TreeOut out{parents, tokens, values, child_values, rows};
  build_tree_greedy_rows_kernel<<<n_req, kVThreads, smem, stream>>>(draft_table, n_rows, vocab, uniforms, n_uniforms, root_row, m,
                                                               out, n_nodes);
  return cudaGetLastError();
}

cudaError_t launch_build_tree_threshold_rows(const float* draft_table, int n_rows, int vocab, const float* uniforms,
                                        int n_uniforms, const int32_t* root_row, int n_req, float threshold, int max_nodes,
                                        int32_t* parents, int32_t* tokens, float* values, float* child_values, int32_t* rows,
                                        int32_t* n_nodes, cudaStream_t stream) {
  if (n_req <= 0) return cudaSuccess;
  const size_t smem = size_t(max_nodes + 1) * 12 + 16;
  TreeOut out{parents, tokens, values, child_values, rows};
  build_tree_threshold_rows_kernel<<<n_req, kVThreads, smem, stream>>>(draft_table, n_rows, vocab, uniforms, n_uniforms, root_row,
                                                                  threshold, max_nodes, out, n_nodes);
  return cudaGetLastError();
}

}  // namespace dyspec
