// Parent array -> packed ancestor bitmasks and depths (Sec. 2, the mask(A) equation, plus the self bit).
//
// First, per 32 nodes (one word of a row) and by one warp in registers: which ancestors of a node lie in its own
// word, and the first one that does not (pointer doubling with shuffles, at most five rounds).  Then one thread
// per node walks from word to word to its root: parents have smaller indices, so it meets every word at
// most once and stores it whole.  A warp's 32 rows are put together in shared memory (rows padded to an odd
// number of words, so that the 32 threads' stores spread over the banks) and leave as one contiguous piece.
// Rows are independent, so a request is cut into CTAs of up to 512 rows.
// The walk takes as many steps as a node has words with ancestors: at most its depth (some 20 for a random
// recursive tree of 2048 nodes) and at most n / 32 (a chain).  Completing all rows together by
// pointer jumping on bitsets in one CTA per request, the earlier form of this kernel, took 1.6, 2.6, 5.1
// and 5.4 us for random trees of 64, 512, 1024 and 2048 nodes back to back (2048: 18 us alone); now 1.2, 1.8, 2.4 and 3.6
// (4 alone).  (Walking from parent to parent without the
// words costs a chain of 2048 nodes 113 us.)
// Optionally the kernel emits, per node, which 64-key tiles of the tree its row touches
// (bit t of node_tiles[i] = row i has a visible key in columns [64 t, 64 t + 64)); the attention
// kernel ORs these over a query tile and skips key tiles no row of it can see (App. C).
// A parent index outside {-1} U [0, i) makes that node a root and reports DYSPEC_ERR_BAD_TREE.
#include "common.cuh"

namespace dyspec {

namespace {
constexpr int kMaskRows = 512;            // rows (threads) of a CTA at most

// The work of one CTA: rows [blockDim blockIdx.y, + blockDim) of request (node0, n).
__device__ __forceinline__ void build_tree_mask_body(const int32_t* __restrict__ parents, int node0, int n,
                                                     uint32_t* __restrict__ bits, int32_t* __restrict__ depths,
                                                     uint32_t* __restrict__ node_tiles, int W, int32_t* status) {
  extern __shared__ __align__(16) uint8_t mask_smem[];
  trigger_dependents();   // the attention kernel may start streaming K/V now; it waits for us before it reads the mask
  const int nthr = int(blockDim.x), row0 = int(blockIdx.y) * nthr;
  if (row0 >= n) return;
  const int row_end = min(n, row0 + nthr);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int pitch = W + 1;
  const int n_words = (row_end + 31) >> 5;
  uint2* s_node = reinterpret_cast<uint2*>(mask_smem);          // [32 n_words] ancestors in the node's own word; the first one below it (or -1)
  uint32_t* s_rows = reinterpret_cast<uint32_t*>(s_node + 32 * n_words) + warp * 32 * pitch;   // [32][pitch], this warp's
  bool bad = false;
  {
    const int step = nthr & ~31;                                 // whole warps (blockDim is a multiple of 32)
    int i = warp * 32 + lane;
    int parent = i < row_end ? __ldg(parents + node0 + i) : -1;
    for (int w = warp; w < n_words; w += nthr >> 5) {
      const int ahead = i + step < row_end ? __ldg(parents + node0 + i + step) : -1;
      if (parent < -1 || parent >= i) {
        bad = bad || i < row_end;
        parent = -1;
      }
      uint32_t mine = 1u << lane;                                // the path from the node up to, not with, lane `up`
      int up = parent >= w * 32 ? parent & 31 : -1, below = parent;   // `below` counts once up < 0
      while (__any_sync(0xffffffffu, up >= 0)) {                 // every lane's path doubles: at most five rounds
        const int src = up >= 0 ? up : lane;
        const uint32_t m = __shfl_sync(0xffffffffu, mine, src);
        const int u = __shfl_sync(0xffffffffu, up, src), b = __shfl_sync(0xffffffffu, below, src);
        if (up >= 0) {
          mine |= m;
          up = u;
          below = b;
        }
      }
      s_node[i] = make_uint2(mine, uint32_t(below));
      i += step;
      parent = ahead;
    }
  }
  for (int k = lane; k < 32 * pitch; k += 32) s_rows[k] = 0u;
  __syncthreads();

  const int i = row0 + tid;
  uint32_t tiles = 0u;
  int depth = -1;
  if (i < row_end) {
    uint32_t* row = s_rows + lane * pitch;
    for (int a = i; a >= 0;) {                                   // every step goes to a lower word
      const uint2 nd = s_node[a];
      row[a >> 5] = nd.x;
      tiles |= 1u << (a >> 6);
      depth += __popc(nd.x);
      a = int(nd.y);
    }
  }
  __syncwarp();

  // Launched with programmatic dependent launch: everything above only read `parents` and worked in
  // shared memory, so it may overlap the tail of the kernel before it in the stream.  The outputs may
  // still be in use by that kernel (the mask of the previous call): wait for it before writing.
  grid_dependency_wait();
  if (bad && status) atomicCAS(status, 0, DYSPEC_ERR_BAD_TREE);
  if (i < row_end) {
    if (depths) depths[node0 + i] = depth;
    if (node_tiles) node_tiles[node0 + i] = tiles;
  }
  const int first = row0 + warp * 32, rows = min(32, row_end - first), W4 = W >> 2;
  uint4* out = reinterpret_cast<uint4*>(bits) + size_t(node0 + first) * W4;
  for (int k = lane; k < rows * W4; k += 32) {
    const int r = k / W4, w = (k - r * W4) * 4;
    const uint32_t* x = s_rows + r * pitch + w;
    out[k] = make_uint4(x[0], x[1], x[2], x[3]);
  }
}
}  // namespace

// Request list in a plan's device table (or one request given by its size).
__global__ void __launch_bounds__(kMaskRows)
build_tree_mask_kernel(const int32_t* __restrict__ parents, const ReqInfo* __restrict__ reqs, int single_n,
                       uint32_t* __restrict__ bits, int32_t* __restrict__ depths, uint32_t* __restrict__ node_tiles,
                       int W, int32_t* status) {
  int node0 = 0, n = single_n;
  if (reqs != nullptr) {
    node0 = reqs[blockIdx.x].node0;
    n = reqs[blockIdx.x].n_nodes;
  }
  build_tree_mask_body(parents, node0, n, bits, depths, node_tiles, W, status);
}

// Request list passed by value (kernel parameter space): a ragged batch without a plan, one launch for
// up to kMaskBatchMax requests, one status word per request.
__global__ void __launch_bounds__(kMaskRows)
build_tree_mask_batch_kernel(const int32_t* __restrict__ parents, const __grid_constant__ MaskBatch batch,
                             uint32_t* __restrict__ bits, int32_t* __restrict__ depths, int W, int32_t* status) {
  const int node0 = batch.node0[blockIdx.x], n = batch.node0[blockIdx.x + 1] - node0;
  build_tree_mask_body(parents, node0, n, bits, depths, nullptr, W, status ? status + batch.first_req + blockIdx.x : nullptr);
}

namespace {
// Launch shape and programmatic dependent launch, the same for both kernels.  A CTA takes up to 512 rows: the attention kernel that follows starts early and wants whole SMs, and every SM that holds
// a mask CTA waiting for its predecessor is one it cannot have yet (with 128 rows a CTA a call of 512 nodes came out
// 0.5 % slower although its mask was there sooner).
struct MaskLaunch {
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = {};
  MaskLaunch(int n_req, int max_n, int W, cudaStream_t stream) {
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    const int all = (max_n + 31) & ~31, rows = all < kMaskRows ? all : kMaskRows;
    cfg.gridDim = dim3(unsigned(n_req), unsigned((max_n + rows - 1) / rows));
    cfg.blockDim = dim3(unsigned(rows));
    cfg.dynamicSmemBytes = size_t(all) * 8 + size_t(rows) * size_t(W + 1) * 4;   // at most 146 KB
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  }
};
}  // namespace

cudaError_t launch_build_tree_mask_batch(const int32_t* parents, const MaskBatch& batch, int n_req, int max_n, uint32_t* bits,
                                         int32_t* depths, int W, int32_t* status, cudaStream_t stream) {
  if (n_req <= 0 || max_n <= 0) return cudaSuccess;
  const MaskLaunch m(n_req, max_n, W, stream);
  static DynSmemGrant grant;
  if (cudaError_t e = grant.ensure(build_tree_mask_batch_kernel, m.cfg.dynamicSmemBytes); e != cudaSuccess) return e;
  const cudaError_t e = cudaLaunchKernelEx(&m.cfg, build_tree_mask_batch_kernel, parents, batch, bits, depths, W, status);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_build_tree_mask(const int32_t* parents, const ReqInfo* reqs, int n_req, int single_n, int max_n,
                                   uint32_t* bits, int32_t* depths, uint32_t* node_tiles, int W, int32_t* status,
                                   cudaStream_t stream) {
  if (n_req <= 0 || max_n <= 0) return cudaSuccess;
  const MaskLaunch m(n_req, max_n, W, stream);
  static DynSmemGrant grant;
  if (cudaError_t e = grant.ensure(build_tree_mask_kernel, m.cfg.dynamicSmemBytes); e != cudaSuccess) return e;
  const cudaError_t e = cudaLaunchKernelEx(&m.cfg, build_tree_mask_kernel, parents, reqs, single_n, bits, depths, node_tiles, W,
                                           status);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace dyspec
