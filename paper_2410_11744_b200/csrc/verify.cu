// Verification of a draft token tree against the target model (Algorithm 3: multi-branch rejection
// sampling along the tree), on the device, so that the step after the tree attention needs no host
// round trip.
//
// A thread-block cluster of C CTAs (1024 threads each) walks one request's tree from node 0; CTA c owns the c-th
// part of the vocabulary.  All CTAs hold the same scalars and take the same decisions, so the walk itself
// needs no exchange.  As long as the FIRST branch of the current node is accepted the walk needs two numbers
// per node, Target(node, y) and Draft(node, y), not the rows: these are fetched for all first branches at
// once, so a node of the walk costs a shared-memory read instead of a round trip to memory.  Only at a
// first rejection -- or where a token has to be drawn -- the rows are loaded: the target row's part into
// registers (the residual R; thread t owns the float4 chunks t, t + 1024, ... of the part) and the draft
// row's part D into shared memory in the same interleaved order.  Both carry a scalar scale instead of
// being renormalised in place:
//   reject y:  R <- max(R sR - D sD, 0), sR <- 1 / sum(R);  D[y] <- 0, sD <- sD / (1 - D[y] sD)
// so a rejection costs one pass over the registers and one exchange: every CTA sends its part of the sum (and, the
// owner of the next branch's token, R and D there) to all others, one cluster barrier, and all add the parts in
// the same order.  "D is all zero" is an exact test on the count of non-zero draft entries.  The final
// token is drawn from R by inverse CDF in token order: the parts' fp64 sums are exchanged and the CTA
// that holds the crossing searches its part.  The random numbers are inputs (one acceptance number
// per node, one sampling number per node), so the caller's generator decides reproducibility.
//
// What bounds it: memory latency and block barriers.  With one CTA a request and the walk's numbers fetched one by one (the
// rows then take 5500 cycles to arrive, the draw 8700, 32 conversions to fp64 a thread among them, and every node of
// the walk 1000) a 64-node tree at vocabulary 32000 took 12 - 16 us back to back, 8 trees of 256 nodes 22.5; now 8 - 12 and
// 18.4.  75 requests and more still get one CTA each and take what they took: 148 trees of 64 nodes 24.6 (without a
// cluster's barriers, which would make it 26.7).
#include "common.cuh"

namespace dyspec {

namespace {

constexpr int kVThreads = 1024;
constexpr int kMaxChunks = 8;              // 4096-token chunks of a row, vocabulary <= 32768
constexpr int kMaxParts = 8;

struct __align__(16) Part {                // what a CTA tells the others
  float sum, count, ry, dy;                // a rejection: part of sum(R), of the non-zero draft entries; R and D at the next branch's token
};
struct VerifyScratch {
  Part part[2][kMaxParts];                 // by exchange parity: a CTA can be one exchange ahead at most
  double draw[kMaxParts];
  double warp_d[kMaxChunks][32];
  double chunk_d[kMaxChunks];
  float warp_f[2][32];
  float ry, dy;
  int n_child, pick;
};

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float element(const float4& v, int e) { return e == 0 ? v.x : e == 1 ? v.y : e == 2 ? v.z : v.w; }

constexpr int kTakeOver = -1, kLeafNode = -2;

}  // namespace

// K = chunks of a CTA's part.
template <int K>
__global__ void __launch_bounds__(kVThreads, 1)
verify_tree_kernel(const int32_t* __restrict__ parents, const int32_t* __restrict__ tokens,
                   const float* __restrict__ draft_probs, const float* __restrict__ target_probs,
                   const float* __restrict__ accept_u, const float* __restrict__ sample_u,
                   const int32_t* __restrict__ node_offsets, int max_nodes, int vocab, int bonus_at_leaf,
                   int32_t* __restrict__ out_tokens, int32_t* __restrict__ out_nodes, int32_t* __restrict__ out_count,
                   int max_out, int32_t* status) {
  extern __shared__ __align__(16) uint8_t vsm[];
  float4* s_d = reinterpret_cast<float4*>(vsm);                                   // draft row's part, [chunk][thread]
  int32_t* s_par = reinterpret_cast<int32_t*>(vsm + size_t(K) * kVThreads * 16);  // [n] parents of the request
  int32_t* s_tok = s_par + max_nodes;                                             // [n] tokens of the nodes
  float* s_acc = reinterpret_cast<float*>(s_tok + max_nodes);                     // [n] acceptance numbers
  int32_t* s_first = reinterpret_cast<int32_t*>(s_acc + max_nodes);               // [n] first branch
  int32_t* s_go = s_first + max_nodes;                                            // [n] the first branch when it is accepted, else kTakeOver, kLeafNode
  __shared__ VerifyScratch s;
  __shared__ int16_t s_child[2048];

  const uint32_t rank = cluster_ctarank();
  uint32_t n_cta;
  asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(n_cta));
  const int r = int(blockIdx.x / n_cta), C = int(n_cta);
  auto sync_parts = [&] {                   // all CTAs of the request (one alone: cluster barriers cost it 2 us a call)
    if (C > 1) cluster_sync_all();
    else __syncthreads();
  };
  const int node0 = node_offsets[r], n = node_offsets[r + 1] - node0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_vec = vocab >> 2;                                  // float4 chunks in a row
  const int vec0 = int(rank) * K * kVThreads;                    // the part's first
  const bool writer = rank == 0 && tid == 0;
  int n_out = 0;
  if (n <= 0 || n > max_nodes) {            // max_nodes sized the shared arrays: a larger request is refused
    if (writer) {
      out_count[r] = 0;
      if (n > max_nodes && status) atomicCAS(status, 0, DYSPEC_ERR_INVALID_ARG);
    }
    return;                                 // (all CTAs of the request)
  }
  if (C > 1) cluster_arrive();              // "this CTA has started": only then may the others write its shared memory
  bool bad = false;
  for (int i = tid; i < n; i += kVThreads) {
    int p_ = parents[node0 + i];
    if (p_ < -1 || p_ >= i) { p_ = -1; bad = true; }
    s_par[i] = p_;
    s_tok[i] = tokens[node0 + i];
    s_acc[i] = accept_u[node0 + i];
    s_first[i] = 0x7fffffff;
    s_go[i] = kLeafNode;
  }
  if (bad && status) atomicCAS(status, 0, DYSPEC_ERR_BAD_TREE);
  __syncthreads();
  // first branches (node 0 is nobody's), and whether the walk may pass through them without the rows
  for (int i = tid; i < n; i += kVThreads)
    if (i > 0 && s_par[i] >= 0) atomicMin(&s_first[s_par[i]], i);
  __syncthreads();
  for (int p = tid; p < n; p += kVThreads) {
    const int i = s_first[p];
    if (i == 0x7fffffff) continue;
    const int y = s_tok[i];
    int go = kTakeOver;                                          // (not a token: the block path reports it)
    if (y >= 0 && y < vocab) {
      const float ry = __ldg(target_probs + size_t(node0 + p) * vocab + y);
      const float dy = __ldg(draft_probs + size_t(node0 + p) * vocab + y);
      const float ratio = dy > 0.f ? ry / dy : (ry > 0.f ? INFINITY : 0.f);
      if (s_acc[i] <= ratio) go = i;
    }
    s_go[p] = go;
  }
  __syncthreads();
  if (C > 1) cluster_wait();                // (here, where every path passes; the loads above hide it)

  auto emit = [&](int token, int node) {
    if (writer && n_out < max_out) { out_tokens[size_t(r) * max_out + n_out] = token; out_nodes[size_t(r) * max_out + n_out] = node; }
    ++n_out;
  };
  int cur = 0, parity = 0;
  for (int step = 0; step <= n; ++step) {                        // at most n moves; bounded in any case
    // ---- fast path: follow first branches for as long as they are accepted
    int go = s_go[cur];
    for (int hop = 0; hop <= n && go >= 0; ++hop) {
      emit(s_tok[go], go);
      cur = go;
      go = s_go[cur];
    }
    const bool leaf = go == kLeafNode;
    if (leaf && !bonus_at_leaf) break;                           // as printed: the loop runs while there are branches

    // ---- R <- Target(cur, .) in registers, D <- Draft(cur, .) in shared memory
    float4 R[K];
    const float4* t_row = reinterpret_cast<const float4*>(target_probs + size_t(node0 + cur) * vocab);
    const float4* d_row = reinterpret_cast<const float4*>(draft_probs + size_t(node0 + cur) * vocab);
    float nnz_f = 0.f;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int v4 = vec0 + k * kVThreads + tid;
      R[k] = v4 < n_vec ? __ldg(t_row + v4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (!leaf) {
      constexpr int kAtOnce = K < 4 ? K : 4;                     // (registers: the whole part of D beside R would spill)
#pragma unroll
      for (int k0 = 0; k0 < K; k0 += kAtOnce) {
        float4 d[kAtOnce];
#pragma unroll
        for (int k = 0; k < kAtOnce; ++k) {
          const int v4 = vec0 + (k0 + k) * kVThreads + tid;
          d[k] = v4 < n_vec ? __ldg(d_row + v4) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int k = 0; k < kAtOnce; ++k) {
          nnz_f += (d[k].x > 0.f) + (d[k].y > 0.f) + (d[k].z > 0.f) + (d[k].w > 0.f);
          s_d[(k0 + k) * kVThreads + tid] = d[k];
        }
      }
    }
    int n_child = 0;
    float ry = 0.f, dy = 0.f;
    if (!leaf) {
      // the branches of `cur`, in index order (one warp; the others wait for their rows)
      __syncthreads();                                           // the list of the node before may still be read
      if (warp == 0) {
        int cnt = 0;
        for (int c0 = 0; c0 < n; c0 += 128) {
          uint32_t m[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = c0 + 32 * u + lane;
            m[u] = __ballot_sync(0xffffffffu, i > 0 && i < n && s_par[i] == cur);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if ((m[u] >> lane) & 1u) s_child[cnt + __popc(m[u] & ((1u << lane) - 1u))] = int16_t(c0 + 32 * u + lane);
            cnt += __popc(m[u]);
          }
        }
        if (lane == 0) s.n_child = cnt;
      }
      const int y = min(max(s_tok[s_first[cur]], 0), vocab - 1);
      ry = __ldg(target_probs + size_t(node0 + cur) * vocab + y);
      dy = __ldg(draft_probs + size_t(node0 + cur) * vocab + y);
      __syncthreads();
      n_child = s.n_child;
    }
    float sR = 1.f, sD = 1.f;
    int nnz = -1;                                                // not counted yet
    bool moved = false;
    for (int b = 0; b < n_child; ++b) {
      const int child = s_child[b];
      int y = s_tok[child];
      if (y < 0 || y >= vocab) {                                 // not a token: report it, carry on with a legal index
        if (writer && status) atomicCAS(status, 0, DYSPEC_ERR_INVALID_ARG);
        y = min(max(y, 0), vocab - 1);
      }
      const float ratio = dy > 0.f ? ry / dy : (ry > 0.f ? INFINITY : 0.f);
      if (s_acc[child] <= ratio) {
        emit(y, child);
        cur = child;
        moved = true;
        break;
      }
      // ---- rejected: R <- norm(max(R - D, 0)); D[y] <- 0; stop if D is all zero; D <- norm(D)
      float part = 0.f;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const float4 d = s_d[k * kVThreads + tid];
        R[k].x = fmaxf(R[k].x * sR - d.x * sD, 0.f);
        R[k].y = fmaxf(R[k].y * sR - d.y * sD, 0.f);
        R[k].z = fmaxf(R[k].z * sR - d.z * sD, 0.f);
        R[k].w = fmaxf(R[k].w * sR - d.w * sD, 0.f);
        part += (R[k].x + R[k].y) + (R[k].z + R[k].w);
      }
      {                                                          // D[y] <- 0 (each thread reads its own entries of D only)
        const int v = (y >> 2) - vec0;
        if (v >= 0 && v < K * kVThreads && (v & (kVThreads - 1)) == tid) reinterpret_cast<float*>(&s_d[v])[y & 3] = 0.f;
      }
      // the next branch's token: its owner's R and D
      const int y2 = b + 1 < n_child ? min(max(s_tok[s_child[b + 1]], 0), vocab - 1) : 0;
      const int v2 = (y2 >> 2) - vec0;
      if (v2 >= 0 && v2 < K * kVThreads && (v2 & (kVThreads - 1)) == tid) {
        float4 mine = R[0];
#pragma unroll
        for (int k = 1; k < K; ++k)
          if (v2 >= k * kVThreads) mine = R[k];
        s.ry = element(mine, y2 & 3);
        s.dy = element(s_d[v2], y2 & 3);
      }
      part = warp_sum(part);
      const float cnt = nnz < 0 ? warp_sum(nnz_f) : 0.f;
      if (lane == 0) { s.warp_f[0][warp] = part; s.warp_f[1][warp] = cnt; }
      __syncthreads();
      if (warp == 0) {
        const float a = warp_sum(s.warp_f[0][lane]), c = warp_sum(s.warp_f[1][lane]);
        if (lane < C) {
          const uint32_t to = map_to_cta(smem_u32(&s.part[parity][rank]), uint32_t(lane));
          asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(to), "f"(a), "f"(c), "f"(s.ry), "f"(s.dy) : "memory");
        }
      }
      __syncwarp();
      sync_parts();
      float tot = 0.f, all = 0.f;
      for (int c = 0; c < C; ++c) { tot += s.part[parity][c].sum; all += s.part[parity][c].count; }
      const Part own = s.part[parity][(y2 >> 2) / (K * kVThreads)];
      parity ^= 1;
      sR = tot > 0.f ? 1.f / tot : 1.f;
      if (nnz < 0) nnz = int(all + 0.5f);
      if (dy > 0.f) --nnz;
      if (nnz <= 0) break;
      sD = sD / (1.f - dy);
      ry = own.ry * sR;
      dy = own.dy * sD;
    }
    if (moved) continue;

    // ---- no branch accepted (or a leaf with the bonus token): draw the token from R by inverse CDF in token order: the
    // first token v with cumsum(R)[v] > u * sum(R) (the last token if rounding leaves none).  The sums are
    // carried in fp64: tokens of a 32000-word vocabulary have CDF intervals of ~1e-5 and less, which fp32
    // prefix sums (error ~1e-6 of the total) would not resolve reproducibly.
    const float u = sample_u[node0 + cur];
    for (int attempt = 0; attempt < 2; ++attempt) {
      {
        // K sums over 32 lanes: the values are halved log2(K) times (a lane's upper bits choose its chunk), then plain steps
        double v[K];
#pragma unroll
        for (int k = 0; k < K; ++k) v[k] = (double(R[k].x) + double(R[k].y)) + (double(R[k].z) + double(R[k].w));
        int o = 16;
#pragma unroll
        for (int w = K / 2; w >= 1; w >>= 1, o >>= 1) {
          const bool upper = lane & o;
#pragma unroll
          for (int k = 0; k < w; ++k) {
            const double give = upper ? v[k] : v[k + w], keep = upper ? v[k + w] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
          }
        }
#pragma unroll
        for (int q = 16 / K; q > 0; q >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], q);
        if (lane % (32 / K) == 0) s.warp_d[lane / (32 / K)][warp] = v[0];
      }
      if (tid == 0) s.pick = 0x7fffffff;
      __syncthreads();
      if (warp < K) {
        const double w_ = warp_sum(s.warp_d[warp][lane]);
        if (lane == 0) s.chunk_d[warp] = w_;
      }
      __syncthreads();
      if (warp == 0 && lane < C) {
        double mine = 0.0;
#pragma unroll
        for (int k = 0; k < K; ++k) mine += s.chunk_d[k];
        st_dsmem_f64(map_to_cta(smem_u32(&s.draw[rank]), uint32_t(lane)), mine);
      }
      __syncwarp();
      sync_parts();
      double total = 0.0;
      for (int c = 0; c < C; ++c) total += s.draw[c];
      if (attempt > 0 || total > 0.0) {
        // the part with the crossing (the last one with tokens if there is none), then its chunk
        const double target = double(u) * total;
        const int last = (n_vec - 1) / (K * kVThreads);
        int owner = last;
        double before = 0.0;
        for (int c = 0; c <= last; ++c) {
          if (before + s.draw[c] > target || c == last) { owner = c; break; }
          before += s.draw[c];
        }
        if (int(rank) == owner) {
          const int n_chunks = min(K, (n_vec - vec0 + kVThreads - 1) / kVThreads);
          int kc = n_chunks - 1;
          bool found = false;
#pragma unroll
          for (int k = 0; k < K; ++k)
            if (k < n_chunks - 1 && !found) {
              if (before + s.chunk_d[k] > target) { kc = k; found = true; }
              else before += s.chunk_d[k];
            }
          float4 rv = R[0];
#pragma unroll
          for (int k = 1; k < K; ++k)
            if (k == kc) rv = R[k];
          const double mine = (double(rv.x) + double(rv.y)) + (double(rv.z) + double(rv.w));
          double incl = mine;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const double t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
          }
          double excl = __shfl_up_sync(0xffffffffu, incl, 1);
          if (lane == 0) excl = 0.0;
          double in_front = lane < warp ? s.warp_d[kc][lane] : 0.0;    // the warps before this one
          in_front = warp_sum(in_front);
          double cum = before + in_front + excl;                 // mass before this thread's 4 tokens
          const int v0 = (vec0 + kc * kVThreads + tid) * 4;
          int pick = 0x7fffffff;
          const float e4[4] = {rv.x, rv.y, rv.z, rv.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            cum += double(e4[e]);
            if (pick == 0x7fffffff && v0 + e < vocab && cum > target) pick = v0 + e;
          }
          if (pick != 0x7fffffff) atomicMin(&s.pick, pick);
          __syncthreads();
          if (tid == 0 && n_out < max_out) {
            out_tokens[size_t(r) * max_out + n_out] = min(s.pick, vocab - 1);
            out_nodes[size_t(r) * max_out + n_out] = -1;
          }
        }
        break;
      }
      // nothing left: fall back to Target
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int v4 = vec0 + k * kVThreads + tid;
        R[k] = v4 < n_vec ? __ldg(t_row + v4) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
      sync_parts();                                              // everyone has read the parts of the first attempt
    }
    ++n_out;
    break;
  }
  if (writer) out_count[r] = min(n_out, max_out);
  if (C > 1) cluster_sync_all();                                 // nobody leaves while its shared memory may be written
}

namespace {
template <int K>
cudaError_t launch_parts(int C, const int32_t* parents, const int32_t* tokens, const float* draft_probs, const float* target_probs,
                         const float* accept_u, const float* sample_u, const int32_t* node_offsets, int n_req, int max_nodes,
                         int vocab, int bonus_at_leaf, int32_t* out_tokens, int32_t* out_nodes, int32_t* out_count, int max_out,
                         int32_t* status, cudaStream_t stream) {
  const size_t smem = size_t(K) * kVThreads * 16 + size_t(max_nodes) * 20;
  static DynSmemGrant grant;
  if (cudaError_t e = grant.ensure(verify_tree_kernel<K>, smem); e != cudaSuccess) return e;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = unsigned(C);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(n_req) * unsigned(C));
  cfg.blockDim = dim3(kVThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = C > 1 ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, verify_tree_kernel<K>, parents, tokens, draft_probs, target_probs, accept_u, sample_u,
                                           node_offsets, max_nodes, vocab, bonus_at_leaf, out_tokens, out_nodes, out_count,
                                           max_out, status);
  return e != cudaSuccess ? e : cudaGetLastError();
}
}  // namespace

cudaError_t launch_verify_tree(const int32_t* parents, const int32_t* tokens, const float* draft_probs,
                               const float* target_probs, const float* accept_u, const float* sample_u,
                               const int32_t* node_offsets, int n_req, int max_nodes, int vocab, int bonus_at_leaf,
                               int32_t* out_tokens, int32_t* out_nodes, int32_t* out_count, int max_out, int32_t* status,
                               cudaStream_t stream) {
  if (n_req <= 0) return cudaSuccess;
  // As many CTAs a request as leave every CTA a chunk of its own, while all requests still run at once: 15 clusters of 8 and 33 - 36 of
  // 4 do, not the 18 and 37 that the SMs would make (vocabulary 32000, 18 trees of 256 nodes: 33 us in two waves of 8, 19 with
  // clusters of 4; 37: 29 in two waves of 4, 22 with clusters of 2).
  const int n_chunks = (vocab + 4 * kVThreads - 1) / (4 * kVThreads);
  static ClusterRoom room;
  int C = 8, K = 1;
  while (C > 1 && (C >= 2 * n_chunks || n_req > room.ask(verify_tree_kernel<8>, kVThreads, C))) C /= 2;
  auto go = [&](auto launch) {
    return launch(C, parents, tokens, draft_probs, target_probs, accept_u, sample_u, node_offsets, n_req, max_nodes, vocab,
                  bonus_at_leaf, out_tokens, out_nodes, out_count, max_out, status, stream);
  };
  for (;; C /= 2) {
    while (K * C < n_chunks) K *= 2;
    const cudaError_t e = K == 1 ? go(launch_parts<1>) : K == 2 ? go(launch_parts<2>) : K == 4 ? go(launch_parts<4>) : go(launch_parts<8>);
    if (e != cudaErrorInvalidClusterSize || C == 1) return e;
    (void)cudaGetLastError();            // a share of a device whose SMs hold no cluster of this size: a smaller one
  }
}

}  // namespace dyspec
