// Depth-first renumbering of a token tree (App. C: DySpec orders the tree tokens by DFS, which
// approximates heavy-path order, so that the attention mask touches few b x b blocks).
//
// One CTA per request.  new index of node i = its position in the pre-order walk that visits roots
// and the children of every node in increasing old index.  No thread walks the tree: the CTA builds
// the Euler tour of the forest as a linked list (an "enter" and an "exit" element per node) and ranks it.
//
//   1. previous sibling of every node, in index order.  A warp looks at 32 consecutive nodes and groups equal
//      parents with match.any; the last lane of each group records itself in a byte table [parent][chunk] and
//      sets the chunk's bit in the parent's word; the first lane of each group finds the nearest earlier
//      chunk of the same parent by a count of leading zeros.  (The bits say which bytes of the table are
//      valid, so it needs no clearing.)  Roots are the children of a virtual node n.
//   2. first child / next sibling follow from that, and with them the tour:
//        enter(i) -> enter(first child of i), or exit(i) for a leaf
//        exit(i)  -> enter(next sibling of i), or exit(parent of i), or the end of the list
//   3. list ranking with weight 1 on enter elements: S(e) = number of enter elements from e to the
//      end, so the pre-order index of node i is n - S(enter(i)).  Up to 256 nodes by pointer jumping over all elements,
//      ceil(log2(2 n)) rounds.  Larger trees: seven elements in 32 are splitters, those that a
//      multiplication modulo a power of two (a bijection, so a splitter's number gives its element back) takes
//      below a bound.  A thread walks from each splitter to the next one (5 steps on average, some 30 at
//      most), the splitters alone are ranked by pointer jumping in eight warps, and every element adds its
//      distance.
// Measured back to back, us: random trees of 65, 128, 200 nodes 4.0, 3.9, 4.4 (with splitters 5.1, 4.4, 5.0); of 512, 1024 and
// 2048 nodes 5.6, 8.3, 13.0 (without them 6.1, 9.8, 18.1).
//
// A parent outside {-1} U [0, i) makes that node a root and reports DYSPEC_ERR_BAD_TREE, as in the
// mask builder.
#include "common.cuh"
#include "dfs_layout.h"

namespace dyspec {

namespace {
constexpr uint32_t kNone = 0xFFFFu;
constexpr int kJumpThreads = 256;                 // (a launch of more than kJumpAll nodes has more threads)

__device__ __forceinline__ uint32_t jumped(const uint32_t* cur, int k) {
  const uint32_t v = cur[k], to = v >> 16;
  if (to == kNone) return v;
  const uint32_t b = cur[to];
  return (b & 0xFFFF0000u) | ((v & 0xFFFFu) + (b & 0xFFFFu));
}
}  // namespace

__global__ void __launch_bounds__(1024, 1)
dfs_reorder_kernel(const int32_t* __restrict__ parents, const ReqInfo* __restrict__ reqs, int single_n,
                   int32_t* __restrict__ order, int32_t* __restrict__ new_of_old, int32_t* __restrict__ new_parents,
                   int32_t* status) {
  extern __shared__ __align__(16) uint8_t ro_smem[];
  // No early launch of dependents here: the kernel that follows is normally the mask builder, which
  // reads its parent array (this kernel's output) before it waits on its predecessor.  Without the
  // trigger the stream serialises the two completely.
  int node0 = 0, n = single_n;
  if (reqs != nullptr) {
    node0 = reqs[blockIdx.x].node0;
    n = reqs[blockIdx.x].n_nodes;
  }
  if (n <= 0) return;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarps = nthr >> 5;
  const int n_chunks = (n + 31) >> 5;
  const int E = 2 * n;                                              // tour elements: enter(i) = i, exit(i) = n + i
  const DfsLayout l(n);
  int16_t* s_par = reinterpret_cast<int16_t*>(ro_smem + l.par);     // [n] parent, n for a root
  uint16_t* s_fc = reinterpret_cast<uint16_t*>(ro_smem + l.fc);     // [n] first child
  uint16_t* s_ns = reinterpret_cast<uint16_t*>(ro_smem + l.ns);     // [n] next sibling
  uint32_t* s_chunks = reinterpret_cast<uint32_t*>(ro_smem + l.chunks); // [n + 1][2] bit c: the parent has a child in chunk c
  uint8_t* s_table = ro_smem + l.table;                             // [n + 1][n_chunks] lane of the parent's last child in the chunk
  uint16_t* s_next = reinterpret_cast<uint16_t*>(ro_smem + l.next); // [E] the tour
  uint32_t* s_at = reinterpret_cast<uint32_t*>(ro_smem + l.at);     // [E] number of the segment's splitter << 16 | enter elements of the segment before it
  const Splitters sp(E);
  uint32_t* cur = reinterpret_cast<uint32_t*>(ro_smem + l.jump);    // an element (n <= kJumpAll) or the number of a splitter ahead << 16 | enter elements up to it
  uint32_t* nxt = cur + (n <= kJumpAll ? E : sp.count);
  bool bad = false;

#pragma unroll 2
  for (int i = tid; i < n; i += nthr) {
    int parent = __ldg(parents + node0 + i);
    if (parent < -1 || parent >= i) {
      parent = -1;
      bad = true;
    }
    s_par[i] = int16_t(parent < 0 ? n : parent);
    s_fc[i] = uint16_t(kNone);
    s_ns[i] = uint16_t(kNone);
  }
  for (int k = tid; k < 2 * (n + 1); k += nthr) s_chunks[k] = 0u;
  __syncthreads();

  // ---- 1. siblings (at most two chunks a warp: n <= 2 nthr)
  uint32_t grp[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int c = warp + j * nwarps, i = c * 32 + lane;
    grp[j] = 0u;
    if (c < n_chunks) {
      const int key = i < n ? int(s_par[i]) : -1 - lane;            // lanes past the end match nobody
      grp[j] = __match_any_sync(0xffffffffu, key);
      if (i < n && lane == 31 - __clz(grp[j])) {
        s_table[key * n_chunks + c] = uint8_t(lane);
        atomicOr(&s_chunks[2 * key + (c >> 5)], 1u << (c & 31));
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int c = warp + j * nwarps, i = c * 32 + lane;
    if (i < n) {
      const int key = s_par[i];
      const uint32_t lower = grp[j] & ((1u << lane) - 1u);
      int prev = -1;
      if (lower) {
        prev = c * 32 + 31 - __clz(lower);
      } else {
        const uint2 m = reinterpret_cast<const uint2*>(s_chunks)[key];
        const uint32_t below = (1u << (c & 31)) - 1u, lo = c < 32 ? m.x & below : m.x, hi = c < 32 ? 0u : m.y & below;
        const int before = hi ? 63 - __clz(hi) : 31 - __clz(lo);    // nearest earlier chunk, -1: none
        if (before >= 0) prev = before * 32 + s_table[key * n_chunks + before];
      }
      if (prev >= 0) s_ns[prev] = uint16_t(i);
      else if (key < n) s_fc[key] = uint16_t(i);
    }
  }
  __syncthreads();

  // ---- 2. Euler tour
  auto next_of = [&](int e) -> uint32_t {
    if (e < n) return s_fc[e] != kNone ? uint32_t(s_fc[e]) : uint32_t(n + e);
    const int i = e - n;
    return s_ns[i] != kNone ? uint32_t(s_ns[i]) : s_par[i] < n ? uint32_t(n + s_par[i]) : kNone;
  };

  // ---- 3. list ranking
  if (n <= kJumpAll) {                                              // after round r an element points 2^r steps ahead
    for (int e = tid; e < E; e += nthr) cur[e] = (next_of(e) << 16) | (e < n ? 1u : 0u);
    __syncthreads();
    for (int span = 1; span < E; span <<= 1) {
      for (int e = tid; e < E; e += nthr) nxt[e] = jumped(cur, e);
      __syncthreads();
      uint32_t* t = cur; cur = nxt; nxt = t;
    }
  } else {
    // A thread walks from each of its splitters to the next one (the tour starts at one: element 0) ...
    for (int e = tid; e < E; e += nthr) s_next[e] = uint16_t(next_of(e));
    __syncthreads();
    for (int k = tid; k < sp.count; k += nthr) {
      uint32_t e = sp.element(k), enters = 0;
      if (e >= uint32_t(E)) continue;
      int to;
      do {                                                          // at most E steps: the tour has no cycle
        s_at[e] = (uint32_t(k) << 16) | enters;
        enters += e < uint32_t(n) ? 1u : 0u;
        e = s_next[e];
        to = sp.number(e);
      } while (e != kNone && to >= sp.count);
      cur[k] = ((e != kNone ? uint32_t(to) : kNone) << 16) | enters;
    }
    __syncthreads();
    // ... and the splitters jump: after round r one points 2^r segments ahead (or to the end) and holds their enter elements.
    // (Eight warps: with all 32 a round costs their barrier and four times the instruction issue.)
    for (int span = 1; span < sp.exist; span <<= 1) {
      if (tid < kJumpThreads) {
        for (int k = tid; k < sp.count; k += kJumpThreads)
          if (sp.element(k) < uint32_t(E)) nxt[k] = jumped(cur, k);
        asm volatile("bar.sync 1, %0;" ::"n"(kJumpThreads) : "memory");
      }
      uint32_t* t = cur; cur = nxt; nxt = t;
    }
    __syncthreads();
  }

  grid_dependency_wait();     // outputs may still be in use by the kernel before this one in the stream
  if (bad && status) atomicCAS(status, 0, DYSPEC_ERR_BAD_TREE);
  auto preorder = [&](int i) {                                      // n - (enter elements from enter(i) to the end)
    if (n <= kJumpAll) return n - int(cur[i] & 0xFFFFu);
    const uint32_t a = s_at[i];
    return n - int(cur[a >> 16] & 0xFFFFu) + int(a & 0xFFFFu);
  };
  for (int i = tid; i < n; i += nthr) {
    const int pre = preorder(i), parent = s_par[i];
    if (new_of_old) new_of_old[node0 + i] = pre;
    if (order) order[node0 + pre] = i;
    if (new_parents) new_parents[node0 + pre] = parent < n ? preorder(parent) : -1;
  }
}

cudaError_t launch_dfs_reorder(const int32_t* parents, const ReqInfo* reqs, int n_req, int single_n, int max_n,
                               int32_t* order, int32_t* new_of_old, int32_t* new_parents, int32_t* status,
                               cudaStream_t stream) {
  if (n_req <= 0 || max_n <= 0) return cudaSuccess;
  const size_t smem = size_t(DfsLayout(max_n).bytes);            // 160 KB at 2048 nodes
  static DynSmemGrant grant;
  if (cudaError_t e = grant.ensure(dfs_reorder_kernel, smem); e != cudaSuccess) return e;
  int threads = ((max_n + 31) / 32) * 32;
  if (threads < 128) threads = 128;
  if (threads > 1024) threads = 1024;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(n_req));
  cfg.blockDim = dim3(unsigned(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, dfs_reorder_kernel, parents, reqs, single_n, order, new_of_old, new_parents,
                                     status);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace dyspec

// ---------------------------------------------------------------------------------------------------
// Block count of a packed tree mask (App. C.1, Table 5): the number of block x block tiles that hold
// at least one visible (query, key) pair.  One thread per tile of the lower triangle.
// ---------------------------------------------------------------------------------------------------
namespace dyspec {

__global__ void mask_block_count_kernel(const uint32_t* __restrict__ bits, int n, int W, int block,
                                        unsigned long long* __restrict__ count) {
  const int nb = (n + block - 1) / block;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  bool hit = false;
  if (idx < nb * nb) {
    const int rb = idx / nb, cb = idx - rb * nb;
    if (cb <= rb) {                       // ancestors have smaller indices: nothing above the diagonal
      const int wpb = block >> 5;         // words per block column
      uint32_t any = 0u;
      for (int r = rb * block; r < min(n, (rb + 1) * block); ++r)
        for (int w = 0; w < wpb; ++w) any |= bits[size_t(r) * W + cb * wpb + w];
      hit = any != 0u;
    }
  }
  const uint32_t votes = __ballot_sync(0xffffffffu, hit);
  if ((threadIdx.x & 31) == 0 && votes) atomicAdd(count, (unsigned long long)__popc(votes));
}

cudaError_t launch_mask_block_count(const uint32_t* bits, int n, int W, int block, unsigned long long* count,
                                    cudaStream_t stream) {
  cudaError_t e = cudaMemsetAsync(count, 0, sizeof(unsigned long long), stream);
  if (e != cudaSuccess || n <= 0) return e;
  const int nb = (n + block - 1) / block;
  const int threads = 256, blocks = (nb * nb + threads - 1) / threads;
  mask_block_count_kernel<<<blocks, threads, 0, stream>>>(bits, n, W, block, count);
  return cudaGetLastError();
}

}  // namespace dyspec
