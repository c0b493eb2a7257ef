// Construction of the draft token tree on the device (Sec. 4.1-4.3, Algorithm 1; App. B, Algorithm 2).
//
// The draft model is a table lookup: the distribution that follows a tree position is row
// f(row of the parent, token) of `draft_table`, and the uniform number of the j-th sampling at a
// position is entry g(row, j) of `uniforms` (vocab_ops.cuh).  So what the j-th sampling at a position
// yields -- its token and that token's residual probability -- is a function of the position's row
// and j alone: positions with the same row share one stream of draws.
//
//   greedy (Algorithm 1):   take the position whose next sampling has the largest estimated acceptance
//     rate v (ties: the one opened first), create the node of that draw, leave v (1 - r) at the position
//     and v r at the new node, r = the drawn token's probability in the residual (the row with the
//     tokens drawn before zeroed, renormalised); m times.
//   threshold (Algorithm 2): layer by layer, each position keeps drawing while v >= t.
//
// Deciding which draw comes next is a serial chain over all nodes, and so is one row's stream of
// draws; but streams of different rows are independent of each other and of the order in which the
// tree takes them.  One thread-block cluster per request therefore splits the work by role:
//
//   planner  (warp 0 of CTA 0)  the serial part only.  Open positions lie in shared memory, 32 lists of them with
//            a lane's best in its registers and the best of all in a scalar; the two values a step makes are
//            compared with that scalar, so only a step that turns to another position needs reductions (two).
//   helpers  (warps 1 and 2 of CTA 0)  one node behind it.  One finds the child's row in a hash table of the rows
//            met so far and orders the row's load and first draws where it is new; the other orders further
//            draws ahead of their use (more of them the longer a stream has become).
//   fetcher and loaders (9 warps of a worker CTA)  row -> 64 leaf sums in fp64, every worker CTA a share of them, kept in the
//            shared memory of the CTA that draws from the row.
//   drawers  (4 warps of a worker CTA)   a draw by one warp: scan of the 64 leaf sums, then of the one leaf
//            that the number falls into (read again from L1 / L2, the tokens drawn before struck out).
//            Only that leaf is summed anew (never by subtraction), so a draw touches 2 KB instead of the row's 128.
//   hot CTAs  (up to three of a cluster)  each takes over one row whose stream runs long: the best-first tree of a
//            flat row is a star, and most of its draws are one serial stream (up to 762 of 768 draws on
//            language-model rows).  The row moves into shared memory with prefix sums over sub-blocks of 8
//            tokens (per chunk of 1024) and over the chunks, as unevaluated pairs of doubles (error 2^-100 of
//            the row's sum), which a draw updates by subtraction; when the residual has fallen below 2^-40
//            of the sum the tables were built from, they are built again.  No scan is left in a draw: two
//            compares with a ballot and eight tokens.  It runs ahead of the orders, which only say where its
//            draws go.
//
// Messages are single words that validate themselves (a draw's record in CTA 0, a load order or a ring
// entry in a worker CTA; written through distributed shared memory), and no hand-over needs a block barrier.
// What a message does not carry itself is ordered by a release and an acquire inside CTA 0: a node's event, behind which
// lie its value and the token of its draw, from the planner to the helpers; the number of nodes opened, behind which
// lie the rows, their entries and first records, from the opener to the orderer; and a hot CTA's buffer of
// draws, in both directions.  Every wait is bounded; when one runs out the request reports 0 nodes and DYSPEC_ERR_TIMEOUT.
//
// Measured on a B200 (vocabulary 32000, 256 language-model rows): one greedy tree of 768 nodes 5466 us with
// the whole row re-read and re-summed by one block per node, 343 - 410 us now; eight threshold trees of 512
// nodes 2518 -> 300 us.  What bounds it: single warps' chains of dependent instructions, about four cycles
// each -- the hot stream's 900 cycles a draw (chunk 240, sub-block 165, token 260, tables 210), the planner's
// 500 a step, about 150 us for the first 127 nodes, whose draws are still cold (2600 cycles a draw in a stream).
//
// Batches of trees with too many rows for this split go to the one-CTA form (construct_rows.cu); launch_tree says when.
#include "vocab_ops.cuh"

namespace dyspec {

cudaError_t launch_build_tree_greedy_rows(const float* draft_table, int n_rows, int vocab, const float* uniforms, int n_uniforms,
                                          const int32_t* root_row, int n_req, int m, int32_t* parents, int32_t* tokens,
                                          float* values, float* child_values, int32_t* rows, int32_t* n_nodes,
                                          cudaStream_t stream);
cudaError_t launch_build_tree_threshold_rows(const float* draft_table, int n_rows, int vocab, const float* uniforms,
                                             int n_uniforms, const int32_t* root_row, int n_req, float threshold, int max_nodes,
                                             int32_t* parents, int32_t* tokens, float* values, float* child_values,
                                             int32_t* rows, int32_t* n_nodes, cudaStream_t stream);

namespace {

constexpr int kLeaves = 64;            // leaf sums per row; a leaf is 128 K tokens, K = 1, 2, 4 by vocabulary
constexpr int kDrawWarps = 4;
constexpr int kLoadWarps = 8, kBatch = 2 * kLoadWarps;         // leaves that come in with one copy: two for each warp that sums
constexpr int kMaxStages = 4;
constexpr int kRoles = 3;              // planner and two helpers; then the drawers, the fetcher, the loaders
constexpr int kTreeThreads = 32 * (kRoles + kDrawWarps + 1 + kLoadWarps);
// Draws used of a row before a hot CTA takes it over.  The root's row (with three hot CTAs) goes to the first at once: every
// path starts there.  The second is given away early, the last one late, to a row that is sure to run on.
// (6 and 14, or 4 and 8, are as good on average, but now and then give a place away to a row that stops, and the long one
// stays with the drawers: 486 and 1457 us where 10 and 20 take 395 and 351.  A fourth hot CTA leaves three
// workers: 127 nodes 123 us instead of 96.)
constexpr int kHotSoon = 10, kHotAfter = 20;
constexpr int kHotLeast = 10;          // trees up to this size have no hot CTA: its tables would not be ready in time
constexpr int kHotRing = 32;           // orders to a hot CTA in flight (at most kMaxAhead - 1 + 16)
constexpr int kHotAhead = 256;         // draws a hot CTA may have ready before they are ordered
constexpr int kMaxHot = 3;
constexpr int kSub = 8, kChunk = 1024, kChunks = 32;          // hot tables: tokens per sub-block, per chunk; chunks
constexpr int kSubs = kChunk / kSub / 32;                     // sub-blocks of a chunk per lane
constexpr int kShortTree = 96;         // nodes x CTAs of a cluster up to which no second wave of clusters pays
constexpr int kMaxAhead = 8;           // draws of a row that may be ordered before they are used
constexpr uint32_t kEmpty = 0xFFFFFFFFu;
constexpr uint32_t kPatientNs = 1000000;     // waits with a limit below this look at the clock at every probe
constexpr uint32_t kFollow = 0x80000000u;   // slot: the record after this one, not linked yet when the slot was written
constexpr int kMaxRecords = 8192;      // 13 bits of a ring entry

// One draw: r (all ones = not drawn yet), token, record of the row's next draw.
struct __align__(16) DrawRecord {
  unsigned long long r_bits;
  uint32_t token;
  uint32_t next;
};

struct __align__(16) EntryState {      // helper's view of a row's stream
  uint16_t consumed, ordered;
  uint32_t last;                       // last record ordered
  uint32_t ring;                       // cluster address of the ring that takes its orders
  uint32_t el_unit;                    // index in its worker CTA << 8 | ring number
};

// Shared-memory layout (the same in every CTA of the cluster; a part a CTA does not use has no bytes).
struct TreeLayout {
  int nodes_pad;                       // m + 1 rounded up to whole groups of 32
  int max_entries, entries_local;      // distinct rows: in all, per worker CTA
  int n_workers, first_worker, n_hot;  // hot CTAs follow CTA 0, the workers follow them
  int n_records, open_records, hash_size, ring_size, ring_shift, n_stages;
  // byte offsets
  int rec, open, note, first, rec_owner, hash_row, hash_val, entry;
  int stage, sums, load_row, attempts, number, ring, log;
  int hot_row, hot_sub, hot_ring, hot_pub, hot_number;
  int bytes;
};

__host__ __device__ inline bool root_is_hot(const TreeLayout& l) { return l.n_hot >= 3; }

__host__ __device__ inline int first_loaded(const TreeLayout& l) { return root_is_hot(l) ? 1 : 0; }   // first entry that the workers see

struct TreeArgs {
  const float* table;
  const float* uniforms;
  const int32_t* root_row;
  int n_rows, vocab, n_uniforms, m;
  uint32_t rows_inverse;               // floor(2^32 / n_rows), at most 2^32 - 1
  float threshold;                     // threshold algorithm only
  uint32_t wait_limit_ns;              // of the planner's waits, at most kWaitLimitNs
  int32_t* status;                     // may be null
  int32_t* parents;
  int32_t* tokens;
  float* values;
  float* child_values;
  int32_t* rows;
  int32_t* n_nodes;
  TreeLayout lay;
};

// Words that another warp or CTA writes: relaxed accesses, single-copy atomic at their size.
__device__ __forceinline__ uint32_t ld_relaxed(const void* p) {
  uint32_t v;
  asm volatile("ld.relaxed.cluster.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long ld_relaxed64(const void* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(const void* p, uint32_t v) {
  asm volatile("st.relaxed.cluster.shared::cta.u32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ void st_relaxed64(const void* p, unsigned long long v) {
  asm volatile("st.relaxed.cluster.shared::cta.u64 [%0], %1;" ::"r"(smem_u32(p)), "l"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_acquire(const void* p) {
  uint32_t v;
  asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(const void* p, uint32_t v) {
  asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_acquire64(const void* p) {
  unsigned long long v;
  asm volatile("ld.acquire.cta.shared::cta.u64 %0, [%1];" : "=l"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ void st_release64(const void* p, unsigned long long v) {
  asm volatile("st.release.cta.shared::cta.u64 [%0], %1;" ::"r"(smem_u32(p)), "l"(v) : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t cluster_addr, uint32_t v) {
  asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_remote64(uint32_t cluster_addr, unsigned long long v) {
  asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(cluster_addr), "l"(v) : "memory");
}

// Polls `ready` (warp-uniform) until it holds; false once the limit has passed.  For the planner and the helpers, whose flag
// never rises; the others use poll(), which ends with the tree.
// kPatient: hundreds of probes before the clock is looked at, and seldom then; else (a limit below a millisecond) at every probe.
template <bool kPatient = true, typename F>
__device__ __forceinline__ bool wait_until(F ready, const uint32_t* exit_flag, uint32_t limit_ns = uint32_t(kWaitLimitNs)) {
#pragma unroll 1
  for (int i = 0; i < (kPatient ? 512 : 1); ++i)
    if (ready()) return true;
  const uint64_t t0 = global_timer_ns();
  for (uint32_t spins = 1;; ++spins) {
    if (ready()) return true;
    if (ld_relaxed(exit_flag)) return false;
    if ((!kPatient || (spins & 255u) == 0) && global_timer_ns() - t0 >= limit_ns) return false;
  }
}

// The same for a wait that may be long or in vain in ordinary operation.
template <typename F>
__device__ __forceinline__ bool poll(F ready, const uint32_t* exit_flag) {
  uint64_t t0 = 0;
  for (uint32_t spins = 1;; ++spins) {
    if (ready()) return true;
    if (ld_relaxed(exit_flag)) return false;
    if ((spins & 1023u) == 0) {
      const uint64_t now = global_timer_ns();
      if (t0 == 0) t0 = now;
      if (now - t0 > 4 * kWaitLimitNs) return false;
    }
  }
}

__device__ __forceinline__ uint32_t ld_remote(uint32_t cluster_addr) {
  uint32_t v;
  asm volatile("ld.relaxed.cluster.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(cluster_addr) : "memory");
  return v;
}

// Lane with the largest value v (v >= 0, or -1 for none; ties: the smallest sequence number); `best` = that value.
__device__ __forceinline__ int warp_best(double v, uint32_t seq, double& best) {
  const int hi = __double2hiint(v);                            // grows with v; negative for -1
  const uint32_t lo = uint32_t(__double2loint(v));
  const int mh = __reduce_max_sync(0xffffffffu, hi);
  bool c = hi == mh;
  uint32_t b = __ballot_sync(0xffffffffu, c);
  if (b & (b - 1)) {
    const uint32_t ml = __reduce_max_sync(0xffffffffu, c ? lo : 0u);
    c = c && lo == ml;
    b = __ballot_sync(0xffffffffu, c);
    if (b & (b - 1)) {
      const uint32_t ms = __reduce_min_sync(0xffffffffu, c ? seq : kEmpty);
      b = __ballot_sync(0xffffffffu, c && seq == ms);
    }
  }
  const int src = __ffs(b) - 1;
  best = __hiloint2double(mh, int(__shfl_sync(0xffffffffu, lo, src)));
  return src;
}

struct Draw { double r; uint32_t next; };

// The record that `slot` stands for and its content, when it has been drawn.
template <bool kPatient>
__device__ __forceinline__ bool wait_draw(const DrawRecord* recs, uint32_t& slot, Draw& d, const uint32_t* exit_flag, uint32_t limit_ns) {
  if (slot & kFollow) {
    const uint32_t prev = slot & ~kFollow;
    uint32_t nx = kEmpty;
    if (!wait_until<kPatient>([&] { nx = ld_relaxed(&recs[prev].next); return nx != kEmpty; }, exit_flag, limit_ns)) return false;
    slot = nx;
  }
  const uint32_t at = smem_u32(recs + slot);
  unsigned long long rb = 0, tn = 0;                           // two words that are each read at once: r; token and next record
  if (!wait_until<kPatient>([&] {
        asm volatile("ld.volatile.shared.v2.u64 {%0, %1}, [%2];" : "=l"(rb), "=l"(tn) : "r"(at) : "memory");
        return rb != ~0ull && uint32_t(tn) != kEmpty;
      }, exit_flag, limit_ns))
    return false;
  d.r = __longlong_as_double((long long)rb);
  d.next = uint32_t(tn >> 32);
  return true;
}

struct __align__(16) OpenSlot {        // greedy: an open position; threshold: value of the first sampling under a node
  double v;                            // value of the position's next sampling; -1: none
  uint32_t seq;                        // order of opening
  uint32_t slot;                       // record of that sampling (or the one before it and kFollow)
};
struct __align__(16) NodeNote {
  double v;                            // value the node was created with
  uint32_t event;                      // parent position << 13 | record of the draw (all ones = not created)
  uint32_t row;                        // written by the helper that reads the event
};

struct Shared {                        // pointers into one CTA's shared memory
  DrawRecord* rec;
  OpenSlot* open;                      // greedy: position p at [p % 32][p / 32]; threshold: node k at [k]
  NodeNote* note;
  uint32_t *first, *rec_owner, *hash_row;
  uint32_t* hash_val;                  // entry << 16 | first record
  EntryState* entry;
};

__device__ __forceinline__ Shared planner_view(uint8_t* sm, const TreeLayout& l) {
  Shared s;
  s.rec = reinterpret_cast<DrawRecord*>(sm + l.rec);
  s.open = reinterpret_cast<OpenSlot*>(sm + l.open);
  s.note = reinterpret_cast<NodeNote*>(sm + l.note);
  s.first = reinterpret_cast<uint32_t*>(sm + l.first);
  s.rec_owner = reinterpret_cast<uint32_t*>(sm + l.rec_owner);
  s.hash_row = reinterpret_cast<uint32_t*>(sm + l.hash_row);
  s.hash_val = reinterpret_cast<uint32_t*>(sm + l.hash_val);
  s.entry = reinterpret_cast<EntryState*>(sm + l.entry);
  return s;
}

// A node for the helpers (one lane, which has seen the draw).
__device__ __forceinline__ void announce(const Shared& s, int k, int pos, uint32_t rec, double v) {
  s.note[k].v = v;                               // (read at the end only)
  st_release(&s.note[k].event, (uint32_t(pos) << 13) | rec);
}

// Algorithm 1's order.  Returns the number of nodes created, -1 when a wait ran out.
// One warp, so every instruction of a step counts about four cycles.
template <bool kPatient>
__device__ int plan_greedy(const TreeArgs& a, const Shared& s, const uint32_t* exit_flag) {
  const int lane = threadIdx.x & 31, per_lane = a.lay.nodes_pad >> 5;
  double c_v = -1.0, rest_v = -1.0;              // the best open position p with p % 32 == lane; the best of all: both without the current one
  uint32_t c_seq = kEmpty;
  int c_pos = 0, rest_pos = 0;
  double v = 1.0;                                // the current position, its next sampling's value and record (kEmpty: a helper names it)
  int pos = 0;
  uint32_t slot = kEmpty;
  auto insert = [&](int p, double val, uint32_t seq, uint32_t rec) {
    if (lane == (p & 31)) {
      s.open[(p & 31) * per_lane + (p >> 5)] = OpenSlot{val, seq, rec};
      if (val > c_v) { c_v = val; c_seq = seq; c_pos = p; }    // (opened last: it loses a tie)
    }
  };
  int n = 0;
  while (n < a.m) {
    if (slot == kEmpty && !wait_until<kPatient>([&] { slot = ld_relaxed(&s.first[pos]); return slot != kEmpty; }, exit_flag, a.wait_limit_ns)) return -1;
    Draw d;
    if (!wait_draw<kPatient>(s.rec, slot, d, exit_flag, a.wait_limit_ns)) return -1;
    const int k = ++n;
    if (lane == 0) announce(s, k, pos, slot, v);
    const double left = 1.0 - d.r;
    double stay = v * left, child = v * d.r;
    if (!(left > 0.0)) stay = -1.0;
    if (!(child >= 0.0)) child = -1.0;           // (NaN: never taken)
    const uint32_t next = d.next != kEmpty ? d.next : (slot | kFollow);
    // (equal values: the one opened first; the rest was opened before either)
    if (stay >= child && stay > rest_v) {        // the same position again
      insert(k, child, 2u * k + 1u, kEmpty);
      if (child > rest_v) { rest_v = child; rest_pos = k; }
      v = stay;
      slot = next;
    } else if (child > stay && child > rest_v) { // straight on to the new node
      insert(pos, stay, 2u * k, next);
      if (stay > rest_v) { rest_v = stay; rest_pos = pos; }
      v = child;
      pos = k;
      slot = kEmpty;
    } else {                                     // another position: take it out of its lane's list, find the best of the others
      insert(pos, stay, 2u * k, next);
      insert(k, child, 2u * k + 1u, kEmpty);
      if (rest_v < 0.0) break;                   // no open position
      v = rest_v;
      pos = rest_pos;
      __syncwarp();
      const int src = pos & 31, at = pos >> 5;
      OpenSlot* list = s.open + src * per_lane;
      slot = list[at].slot;
      double o_v = -1.0;
      uint32_t o_seq = kEmpty;
      int o_at = lane;
      for (int j = lane; j < per_lane; j += 32) {              // one round up to 1024 nodes, two beyond
        const double x = list[j].v;
        const uint32_t q = list[j].seq;
        if (j != at && (x > o_v || (x == o_v && q < o_seq))) { o_v = x; o_seq = q; o_at = j; }
      }
      if (lane == 0) list[at].v = -1.0;
      double top;
      const int from = warp_best(o_v, o_seq, top);
      const uint32_t top_seq = __shfl_sync(0xffffffffu, o_seq, from);
      const int top_at = __shfl_sync(0xffffffffu, o_at, from);
      if (lane == src) { c_v = top; c_seq = top_seq; c_pos = top_at * 32 + src; }
      const int who = warp_best(c_v, c_seq, rest_v);
      rest_pos = __shfl_sync(0xffffffffu, c_pos, who);
      __syncwarp();
    }
  }
  return n;
}

// Algorithm 2's order: positions in index order (which is layer order) draw while v >= t.
template <bool kPatient>
__device__ int plan_threshold(const TreeArgs& a, const Shared& s, const uint32_t* exit_flag) {
  const int lane = threadIdx.x & 31;
  const double t = double(a.threshold);
  if (lane == 0) s.open[0].v = 1.0;
  __syncwarp();
  int n = 0;
  for (int pos = 0; pos <= n && n < a.m; ++pos) {
    double v = s.open[pos].v;
    if (!(v >= t)) continue;
    uint32_t slot = kEmpty;
    if (!wait_until<kPatient>([&] { slot = ld_relaxed(&s.first[pos]); return slot != kEmpty; }, exit_flag, a.wait_limit_ns)) return -1;
    while (v >= t && n < a.m) {
      Draw d;
      if (!wait_draw<kPatient>(s.rec, slot, d, exit_flag, a.wait_limit_ns)) return -1;
      const int k = ++n;
      if (lane == 0) {
        st_relaxed64(&s.open[k].v, (unsigned long long)__double_as_longlong(v * d.r));
        announce(s, k, pos, slot, v);
      }
      v = v * (1.0 - d.r);
      if (!(1.0 - d.r > 0.0)) break;
      slot = d.next != kEmpty ? d.next : (slot | kFollow);
    }
    __syncwarp();
  }
  return n;
}

// Sends the orders for the next `n` draws of a row, to be put into records rec, rec + 1, ... (whole warp, n <= 32).  Two warps
// send to the workers' rings.
__device__ __forceinline__ void send_orders(const TreeLayout& l, uint32_t* s_tail, uint32_t ring, uint32_t el_unit, uint32_t rec, int n) {
  const int lane = threadIdx.x & 31;
  const uint32_t unit = el_unit & 0xFFu;
  uint32_t i = 0;
  if (lane == 0) i = atomicAdd(&s_tail[unit], uint32_t(n));
  i = __shfl_sync(0xffffffffu, i, 0) + uint32_t(lane);
  const bool hot = unit >= 8 * kDrawWarps;
  const uint32_t mask = hot ? uint32_t(kHotRing - 1) : uint32_t(l.ring_size - 1), shift = hot ? 5u : uint32_t(l.ring_shift);
  if (lane < n) st_remote(ring + (i & mask) * 4, (((i >> shift) & 1u) << 31) | ((el_unit >> 8) << 13) | (rec + uint32_t(lane)));
}

// The next node for a helper warp; false when the tree is complete (or a wait ran out).
__device__ __forceinline__ bool next_event(const Shared& s, int m, int k, uint32_t& ev, const uint32_t* s_final, const uint32_t* exit_flag) {
  bool over = false;
  const bool got = wait_until([&] {
    if (k <= m) {
      ev = ld_acquire(&s.note[k].event);
      if (ev != kEmpty) return true;
    }
    const uint32_t fin = ld_relaxed(s_final);
    over = fin != kEmpty && uint32_t(k) > fin;
    return over;
  }, exit_flag);
  return got && !over;
}

// Helper 1: rows of new nodes.  `hot_addr` (both helpers): the hot CTAs' hand-over words, at the same offset in each.
template <bool kGreedy>
__device__ __forceinline__ void run_opener(const TreeArgs& a, const Shared& s, uint8_t* sm, uint32_t* s_tail, uint32_t hot_addr, uint32_t* s_opened,
                                           const uint32_t* s_final, const uint32_t* exit_flag, int req) {
  const TreeLayout& l = a.lay;
  const int lane = threadIdx.x & 31;
  const double t = double(a.threshold);
  int n_entries = 0, n_records = 0;
  int next_worker = 0, next_el = 0;              // round robin over the worker CTAs
  const uint32_t sm_addr = smem_u32(sm);
  const uint32_t n_buckets = uint32_t(l.hash_size) >> 5;

  // Names node k's first record: that of the row's entry, created (and its load ordered) when the row is new.
  auto open_row = [&](int k, uint32_t row) {
    uint32_t b = ((row * 2654435769u) >> 16) & (n_buckets - 1);
    for (uint32_t tries = 0; tries < n_buckets; ++tries, b = (b + 1) & (n_buckets - 1)) {
      const uint32_t h = s.hash_row[b * 32 + lane], hv = s.hash_val[b * 32 + lane];
      const uint32_t hit = __ballot_sync(0xffffffffu, h == row);
      if (hit) {
        if (lane == __ffs(hit) - 1) st_relaxed(&s.first[k], hv & 0xFFFFu);
        break;
      }
      const uint32_t open = __ballot_sync(0xffffffffu, h == kEmpty);
      if (open) {
        // one record is due to every row still to come; the rest of the pool lets the first draws run ahead
        const int e = n_entries++, spare = l.open_records - n_records - (l.max_entries - e);
        const int rec0 = n_records, want = 1 + max(0, min(kGreedy ? 1 : 3, spare));
        n_records += want;
        const int w = next_worker, el = next_el;
        if (++next_worker == l.n_workers) { next_worker = 0; ++next_el; }
        const uint32_t cta = uint32_t(w + l.first_worker);
        const bool hot = k == 0 && root_is_hot(l);             // no draw of it is ordered elsewhere, and no worker needs the row
        if (hot) {
          if (lane == 0) { st_remote(map_to_cta(hot_addr + 4, 1u), 0u); st_remote(map_to_cta(hot_addr, 1u), row); }
        } else if (lane < l.n_workers) st_remote(map_to_cta(sm_addr + l.load_row + e * 4, uint32_t(l.first_worker + lane)), row);
        const EntryState st{0, uint16_t(want), uint32_t(rec0 + want - 1),
                            hot ? map_to_cta(sm_addr + l.hot_ring, 1u) : map_to_cta(sm_addr + l.ring + (el % kDrawWarps) * l.ring_size * 4, cta),
                            hot ? uint32_t(8 * kDrawWarps) : (uint32_t(el) << 8) | uint32_t(w * kDrawWarps + el % kDrawWarps)};
        if (lane < want) {
          s.rec_owner[rec0 + lane] = (uint32_t(e) << 16) | uint32_t(lane);
          if (lane + 1 < want) st_relaxed(&s.rec[rec0 + lane].next, uint32_t(rec0 + lane + 1));
        }
        if (lane == 0) {
          const int at = b * 32 + __ffs(open) - 1;
          s.entry[e] = st;
          s.hash_row[at] = row;
          s.hash_val[at] = (uint32_t(e) << 16) | uint32_t(rec0);
          st_relaxed(&s.first[k], uint32_t(rec0));
        }
        __syncwarp();
        send_orders(l, s_tail, st.ring, st.el_unit, uint32_t(rec0), want);
        break;
      }
    }
    __syncwarp();
  };

  const int32_t rr0 = a.root_row[req];
  const uint32_t row0 = uint32_t(((rr0 % a.n_rows) + a.n_rows) % a.n_rows);      // non-negative remainder: any int32 maps to a row
  if (lane == 0) s.note[0].row = row0;
  if (a.m > 0) open_row(0, row0);
  __syncwarp();
  if (lane == 0) st_release(s_opened, 1u);       // nodes opened: what the whole warp wrote for them is in front of this
  uint32_t ev = kEmpty;
  for (int k = 1; next_event(s, a.m, k, ev, s_final, exit_flag); ++k) {
    const uint32_t rec = ev & 0x1FFFu, prow = s.note[ev >> 13].row;
    const uint32_t y = ld_relaxed(&s.rec[rec].token);          // drawn: the planner has used it
    // row of the child: the remainder by the prepared inverse
    const uint32_t h = draft_child_hash(prow, y);
    uint32_t row = h - __umulhi(h, a.rows_inverse) * uint32_t(a.n_rows);
    while (row >= uint32_t(a.n_rows)) row -= uint32_t(a.n_rows);                 // (the quotient is at most two short)
    if (lane == 0) s.note[k].row = row;
    bool expand = k < a.m;
    if (!kGreedy) expand = __longlong_as_double((long long)ld_relaxed64(&s.open[k].v)) >= t;   // (written before the event)
    if (expand) open_row(k, row);
    __syncwarp();
    if (lane == 0) st_release(s_opened, uint32_t(k) + 1u);
  }
}

// Helper 2: a used draw lets its row's stream run on.
template <bool kGreedy>
__device__ __forceinline__ void run_orderer(const TreeArgs& a, const Shared& s, uint8_t* sm, uint32_t* s_tail, uint32_t hot_addr,
                                            const uint32_t* s_opened, const uint32_t* s_final, const uint32_t* exit_flag) {
  const TreeLayout& l = a.lay;
  const int lane = threadIdx.x & 31;
  int next_rec = l.open_records, n_hot = root_is_hot(l) ? 1 : 0;
  const uint32_t sm_addr = smem_u32(sm);
  uint32_t ev = kEmpty, opened = 0;
  for (int k = 1; next_event(s, a.m, k, ev, s_final, exit_flag); ++k) {
    // the draw's row was opened with the position or before it; the opener may only just have named the record
    if (opened <= (ev >> 13) && !wait_until([&] { opened = ld_acquire(s_opened); return opened > (ev >> 13); }, exit_flag)) return;
    const uint32_t owner = s.rec_owner[ev & 0x1FFFu];
    const int e = int(owner >> 16);
    EntryState st = s.entry[e];
    if ((owner & 0xFFFFu) == st.consumed) {
      const int c = ++st.consumed;
      if (n_hot < l.n_hot && c >= (n_hot + 1 < l.n_hot ? kHotSoon : kHotAfter) && (st.el_unit & 0xFFu) < 8 * kDrawWarps) {
        // to a hot CTA: the row and the records of the draws ordered so far
        const uint32_t cta = uint32_t(1 + n_hot), at = map_to_cta(hot_addr, cta), pos = ev >> 13;
        uint32_t r = ld_relaxed(&s.first[pos]), mine = r;
        for (int i = 1; i < int(st.ordered); ++i) {
          r = ld_relaxed(&s.rec[r].next);
          if (lane == i) mine = r;
        }
        if (lane < int(st.ordered)) st_remote(at + 8 + lane * 4, mine);
        if (lane == 0) { st_remote(at + 4, st.ordered); st_remote(at, s.note[pos].row); }
        st.ring = map_to_cta(sm_addr + l.hot_ring, cta);
        st.el_unit = uint32_t(8 * kDrawWarps + n_hot);
        ++n_hot;
      }
      // One record is due to every node still to come; the rest of the pool lets streams run further ahead the longer they
      // are.  A hot stream, whose draws are there before they are ordered, gets its orders 16 at a time.
      const bool hot = (st.el_unit & 0xFFu) >= 8 * kDrawWarps;
      const int lead = int(st.ordered) - c;
      int add = hot ? (lead < kMaxAhead ? 16 : 0) : max(0, min(2 + c, kMaxAhead) - lead);
      if (add > 0) {
        add = min(add, max(lead < 1 ? 1 : 0, l.n_records - next_rec - (a.m - k) - 1));
        if (add > 0) {
          if (lane < add) {
            const uint32_t rec = uint32_t(next_rec + lane);
            s.rec_owner[rec] = (uint32_t(e) << 16) | uint32_t(st.ordered + lane);
            st_relaxed(&s.rec[lane ? rec - 1 : st.last].next, rec);
          }
          send_orders(l, s_tail, st.ring, st.el_unit, uint32_t(next_rec), add);
          st.ordered = uint16_t(st.ordered + add);
          next_rec += add;
          st.last = uint32_t(next_rec - 1);
        }
      }
      if (lane == 0) s.entry[e] = st;
    }
    __syncwarp();
  }
}

// Row -> 64 leaf sums.  Every worker CTA sums its share of the leaves of every row (a row is then there after a quarter of
// the time) and sends the sums to the CTA that draws from the row.  One thread brings the shares in with bulk copies, up to
// four batches of 16 leaves ahead; 8 warps convert to fp64 (16 values a clock and SM: what bounds it) and reduce.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

template <int K>
__device__ __forceinline__ void run_fetcher(const TreeArgs& a, uint8_t* sm, int worker, unsigned long long* s_full, unsigned long long* s_empty,
                                            const uint32_t* s_never, const uint32_t* exit_flag) {
  const TreeLayout& l = a.lay;
  if ((threadIdx.x & 31) != 0) return;
  constexpr int kLeafTokens = 128 * K;
  const uint32_t* s_row = reinterpret_cast<const uint32_t*>(sm + l.load_row);
  const uint32_t stage0 = smem_u32(sm) + uint32_t(l.stage);
  const int leaf0 = kLeaves * worker / l.n_workers, leaf1 = kLeaves * (worker + 1) / l.n_workers;
  uint32_t stage = 0, round = 0, issued = 0;
  bool go = true;
  for (int e = first_loaded(l); go && e < l.max_entries; ++e) {
    uint32_t row = kEmpty;                                     // idle until a row is ordered or the tree is finished
    go = poll([&] { row = ld_relaxed(s_row + e); return row != kEmpty; }, exit_flag);
    for (int first = leaf0; go && first < leaf1; first += kBatch) {
      const uint32_t full = smem_u32(s_full + stage);
      if (round > 0 && !poll([&] { return mbar_test_wait(smem_u32(s_empty + stage), (round - 1) & 1u); }, exit_flag)) { go = false; break; }
      const int begin = first * kLeafTokens, end = min(min(first + kBatch, leaf1) * kLeafTokens, a.vocab);
      if (end > begin) {
        const uint32_t bytes = uint32_t(end - begin) * 4u;
        mbar_expect_tx(full, bytes);
        bulk_load(stage0 + stage * uint32_t(kBatch * kLeafTokens * 4), a.table + size_t(row) * a.vocab + begin, bytes, full);
      } else {
        mbar_arrive(full);
      }
      ++issued;
      if (++stage == uint32_t(l.n_stages)) { stage = 0; ++round; }
    }
    if (go && e % l.n_workers == worker)
      st_relaxed(reinterpret_cast<uint32_t*>(sm + l.number) + e / l.n_workers,
                 __float_as_uint(__ldg(a.uniforms + draft_uniform_index(row, 0u, uint32_t(a.n_uniforms)))));
  }
  // no copy may be under way when the block ends
  for (uint32_t k = 0; k < uint32_t(l.n_stages) && k < issued; ++k) {
    if (stage == 0) { stage = uint32_t(l.n_stages); --round; }
    --stage;
    poll([&] { return mbar_test_wait(smem_u32(s_full + stage), round & 1u); }, s_never);
  }
}

template <int K>
__device__ __forceinline__ void run_loader(const TreeArgs& a, uint8_t* sm, int lw, int worker, unsigned long long* s_full, unsigned long long* s_empty,
                                           const uint32_t* exit_flag) {
  const TreeLayout& l = a.lay;
  const int lane = threadIdx.x & 31, n_vec = a.vocab >> 2;
  const uint32_t sums = smem_u32(sm) + uint32_t(l.sums);
  const int leaf0 = kLeaves * worker / l.n_workers, leaf1 = kLeaves * (worker + 1) / l.n_workers;
  uint32_t stage = 0, round = 0;
  int el = first_loaded(l) / l.n_workers, owner = first_loaded(l) % l.n_workers;
  for (int e = first_loaded(l); e < l.max_entries; ++e) {
    const uint32_t dst = map_to_cta(sums + uint32_t(el) * (kLeaves * 8), uint32_t(l.first_worker + owner));
    if (++owner == l.n_workers) { owner = 0; ++el; }
    for (int first = leaf0; first < leaf1; first += kBatch) {
      if (!poll([&] { return mbar_test_wait(smem_u32(s_full + stage), round & 1u); }, exit_flag)) return;
      const float4* src = reinterpret_cast<const float4*>(sm + l.stage) + stage * (kBatch * K * 32);
      double q[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {                            // leaves first + 2 lw, + 1
        q[j] = 0.0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const int v4 = ((2 * lw + j) * K + k) * 32 + lane;
          float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
          if (first + 2 * lw + j < leaf1 && first * K * 32 + v4 < n_vec) x = src[v4];
          q[j] += (double(x.x) + double(x.y)) + (double(x.z) + double(x.w));
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(s_empty + stage));
      if (++stage == uint32_t(l.n_stages)) { stage = 0; ++round; }
      const bool upper = lane & 16;                            // two sums over 32 lanes: halves swap, then plain steps
      double b = upper ? q[1] : q[0];
      b += __shfl_xor_sync(0xffffffffu, upper ? q[0] : q[1], 16);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
      const int leaf = first + 2 * lw + (upper ? 1 : 0);
      if ((lane & 15) == 0 && leaf < leaf1) st_remote64(dst + uint32_t(leaf) * 8, (unsigned long long)__double_as_longlong(b));
    }
  }
}

// Draws, one warp each, in the order in which the helpers asked for them.
template <int K>
__device__ __forceinline__ void run_drawer(const TreeArgs& a, uint8_t* sm, int dw, int worker, uint32_t (*s_mask)[32], uint32_t* s_log_n,
                                           const uint32_t* exit_flag) {
  constexpr int kLane = 4 * K, kLeaf = 32 * kLane;             // consecutive tokens of a lane, of a leaf
  const TreeLayout& l = a.lay;
  const int lane = threadIdx.x & 31, n_vec = a.vocab >> 2;
  const uint32_t* ring = reinterpret_cast<const uint32_t*>(sm + l.ring) + dw * l.ring_size;
  const uint32_t* s_row = reinterpret_cast<const uint32_t*>(sm + l.load_row);
  unsigned long long* s_sums = reinterpret_cast<unsigned long long*>(sm + l.sums);
  uint32_t* s_att = reinterpret_cast<uint32_t*>(sm + l.attempts);
  uint32_t* s_log = reinterpret_cast<uint32_t*>(sm + l.log);
  uint32_t* s_num = reinterpret_cast<uint32_t*>(sm + l.number);
  const uint32_t rec_base = map_to_cta(smem_u32(sm) + l.rec, 0);
  for (uint32_t i = 0;; ++i) {
    const uint32_t at = i & uint32_t(l.ring_size - 1), phase = (i >> l.ring_shift) & 1u;
    uint32_t msg = kEmpty;
    if (!poll([&] { msg = ld_relaxed(ring + at); return msg != kEmpty && (msg >> 31) == phase; }, exit_flag)) return;
    const uint32_t el = (msg >> 13) & 0xFFFu, rec = msg & 0x1FFFu;
    uint32_t row = kEmpty, ub = kEmpty;
    if (!poll([&] { row = ld_relaxed(s_row + el * l.n_workers + worker); return row != kEmpty; }, exit_flag)) return;
    const uint32_t att = s_att[el];
    const float u_next = __ldg(a.uniforms + draft_uniform_index(row, att + 1, uint32_t(a.n_uniforms)));   // arrives behind this draw
    unsigned long long* sums = s_sums + size_t(el) * kLeaves;
    unsigned long long b0 = 0, b1 = 0;
    if (!poll([&] {                                            // (may be cut short: the tree can be finished before the row is there)
          b0 = ld_relaxed64(sums + 2 * lane);
          b1 = ld_relaxed64(sums + 2 * lane + 1);
          ub = ld_relaxed(s_num + el);
          return __all_sync(0xffffffffu, b0 != ~0ull && b1 != ~0ull && ub != kEmpty) != 0;
        }, exit_flag))
      return;
    const float u = __uint_as_float(ub);

    // ---- the leaf: prefix sums over the 64 leaf sums, two per lane
    const double s0 = __longlong_as_double((long long)b0), s1 = __longlong_as_double((long long)b1);
    double incl = s0 + s1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    double excl = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) excl = 0.0;
    const double total = __shfl_sync(0xffffffffu, incl, 31);
    const double target = double(u) * total;
    const uint32_t over = __ballot_sync(0xffffffffu, incl > target);
    const bool none = over == 0u;                              // rounding (or an empty residual) left no crossing: the last token
    const int hit = none ? 0 : __ffs(over) - 1;
    const bool second = !(excl + s0 > target);
    int leaf = __shfl_sync(0xffffffffu, 2 * lane + (second ? 1 : 0), hit);
    const double before = __shfl_sync(0xffffffffu, second ? excl + s0 : excl, hit);
    if (none) leaf = (a.vocab - 1) / kLeaf;

    // ---- its tokens, those drawn before struck out
    const float4* src = reinterpret_cast<const float4*>(a.table + size_t(row) * a.vocab);
    float4 x[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int v4 = (leaf * 32 + lane) * K + k;
      x[k] = v4 < n_vec ? __ldg(src + v4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (att > 0) {
      s_mask[dw][lane] = 0u;
      __syncwarp();
      const uint32_t n_log = ld_relaxed(s_log_n);
      const uint32_t want = (el << 16) | uint32_t(leaf * kLeaf);
#pragma unroll 4
      for (uint32_t j = lane; j < n_log; j += 32) {
        const uint32_t off = ld_relaxed(s_log + j) - want;     // token within the leaf
        if (off < uint32_t(kLeaf)) atomicOr(&s_mask[dw][off / kLane], 1u << (off % kLane));
      }
      __syncwarp();
      const uint32_t dead = s_mask[dw][lane];
      if (dead) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
          if ((dead >> (4 * k)) & 1u) x[k].x = 0.f;
          if ((dead >> (4 * k + 1)) & 1u) x[k].y = 0.f;
          if ((dead >> (4 * k + 2)) & 1u) x[k].z = 0.f;
          if ((dead >> (4 * k + 3)) & 1u) x[k].w = 0.f;
        }
      }
    }
    double q[K], mine = 0.0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      q[k] = (double(x[k].x) + double(x[k].y)) + (double(x[k].z) + double(x[k].w));
      mine += q[k];
    }
    double pre = mine;                                         // inclusive prefix sums over the lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double t = __shfl_up_sync(0xffffffffu, pre, o);
      if (lane >= o) pre += t;
    }
    double pex = __shfl_up_sync(0xffffffffu, pre, 1);
    if (lane == 0) pex = 0.0;
    const uint32_t cross = __ballot_sync(0xffffffffu, before + pre > target);
    int owner = __ffs(cross) - 1;
    if (none) {
      owner = ((a.vocab - 1) % kLeaf) / kLane;
    } else if (cross == 0u) {                                  // rounding between the two levels: the leaf's last mass
      const uint32_t some = __ballot_sync(0xffffffffu, mine > 0.0);
      owner = some ? 31 - __clz(some) : 0;
    }
    if (lane == owner) {
      // quad, then token; where rounding leaves no crossing, the lane's last token with mass
      double cum = before + pex, at_quad = -INFINITY;
      int kp = -1, last = 0, pe = 0;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (kp < 0 && cum + q[k] > target) { kp = k; at_quad = cum; }
        if (q[k] > 0.0) last = k;
        cum += q[k];
      }
      if (kp < 0) kp = last;
      if (none) kp = ((a.vocab - 1) % kLane) >> 2;
      float4 f = x[0];
#pragma unroll
      for (int k = 1; k < K; ++k)
        if (k == kp) f = x[k];
      const double f0 = f.x, f1 = f.y, f2 = f.z, c0 = at_quad + f0, c1 = c0 + f1, c2 = c1 + f2, c3 = c2 + double(f.w);
      if (c0 > target) pe = 0;
      else if (c1 > target) pe = 1;
      else if (c2 > target) pe = 2;
      else if (c3 > target) pe = 3;
      else pe = f.w > 0.f ? 3 : f.z > 0.f ? 2 : f.y > 0.f ? 1 : 0;
      if (none) pe = (a.vocab - 1) & 3;
      const int y = min(leaf * kLeaf + owner * kLane + 4 * kp + pe, a.vocab - 1);
      const float py = pe == 0 ? f.x : pe == 1 ? f.y : pe == 2 ? f.z : f.w;
      const double r = total > 0.0 ? double(py) / total : 0.0;
      st_remote64(rec_base + rec * 16, (unsigned long long)__double_as_longlong(r));
      st_remote(rec_base + rec * 16 + 8, uint32_t(y));
      // ---- the token leaves the row
      s_log[atomicAdd(s_log_n, 1u)] = (el << 16) | uint32_t(y);
      s_att[el] = att + 1;
      s_num[el] = __float_as_uint(u_next);
      if (pe == 0) f.x = 0.f; else if (pe == 1) f.y = 0.f; else if (pe == 2) f.z = 0.f; else f.w = 0.f;
      const double quad = (double(f.x) + double(f.y)) + (double(f.z) + double(f.w));
      mine = 0.0;
#pragma unroll
      for (int k = 0; k < K; ++k) mine += k == kp ? quad : q[k];
    }
    __syncwarp();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    if (lane == 0) sums[leaf] = (unsigned long long)__double_as_longlong(mine);
    __syncwarp();
  }
}

// ---- hot CTA: one row's stream from a copy of the row and prefix sums in shared memory ----
struct __align__(16) Pair { double hi, lo; };   // hi + lo, unevaluated
struct __align__(16) Published { double sum; unsigned long long word; };   // residual sum; phase, token, probability
__device__ __forceinline__ Pair add(Pair a, Pair b) {
  const double s = a.hi + b.hi, t = s - a.hi;
  const double e = (a.hi - (s - t)) + (b.hi - t);            // Knuth's two-sum
  return Pair{s, e + (a.lo + b.lo)};
}
__device__ __forceinline__ Pair take_off(Pair a, double p) { // the sum holds p: a.hi >= p, Dekker's fast two-sum
  const double s = a.hi - p;
  return Pair{s, a.lo + ((a.hi - s) - p)};
}
__device__ __forceinline__ Pair shfl_up_pair(Pair v, int o) {
  return Pair{__shfl_up_sync(0xffffffffu, v.hi, o), __shfl_up_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ Pair scan(Pair v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const Pair t = shfl_up_pair(v, o);
    if (lane >= o) v = add(t, v);
  }
  return v;
}

// Prefix sums over the sub-blocks of chunk c (one warp; lane = kSubs sub-blocks).  Sub-block kSubs l + j of a chunk lies at [j][l].
__device__ __forceinline__ void build_chunk(const float* s_row, Pair* s_sub, int c, int lane) {
  Pair v[kSubs];
#pragma unroll
  for (int j = 0; j < kSubs; ++j) {
    v[j] = Pair{0.0, 0.0};
    const float* x = s_row + c * kChunk + (kSubs * lane + j) * kSub;
#pragma unroll
    for (int i = 0; i < kSub; ++i) v[j] = add(v[j], Pair{double(x[(i + lane) & (kSub - 1)]), 0.0});   // (any order; rotated: fewer bank conflicts)
    if (j) v[j] = add(v[j - 1], v[j]);
  }
  const Pair upto = shfl_up_pair(scan(v[kSubs - 1], lane), 1);
#pragma unroll
  for (int j = 0; j < kSubs; ++j) s_sub[(c * kSubs + j) * 32 + lane] = lane ? add(upto, v[j]) : v[j];
}

__device__ __forceinline__ void run_hot(const TreeArgs& a, uint8_t* sm, const uint32_t* s_hot, uint32_t* s_go, const uint32_t* exit_flag) {
  const TreeLayout& l = a.lay;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* s_row = reinterpret_cast<float*>(sm + l.hot_row);
  Pair* s_sub = reinterpret_cast<Pair*>(sm + l.hot_sub);
  const uint32_t* ring = reinterpret_cast<const uint32_t*>(sm + l.hot_ring);
  Published* s_pub = reinterpret_cast<Published*>(sm + l.hot_pub);
  const uint32_t rec_base = map_to_cta(smem_u32(sm) + l.rec, 0);
  // ---- one thread waits for a row: its number and how many draws have been ordered elsewhere (each word validates itself)
  if (tid == 0) {
    uint32_t row = kEmpty, n_prev = kEmpty;
    if (!poll([&] { row = ld_relaxed(s_hot); n_prev = ld_relaxed(s_hot + 1); return row != kEmpty && n_prev != kEmpty; }, exit_flag))
      row = kEmpty;
    s_go[0] = row;
    s_go[1] = n_prev;
    s_go[2] = 0u;                                              // draws taken out of the buffer
  }
  __syncthreads();
  const uint32_t row = s_go[0], n_prev = s_go[1];
  if (row == kEmpty) return;                                   // the whole block
  const float4* src = reinterpret_cast<const float4*>(a.table + size_t(row) * a.vocab);
  for (int i = tid; i < kChunks * kChunk / 4; i += kTreeThreads)
    reinterpret_cast<float4*>(s_row)[i] = i < (a.vocab >> 2) ? __ldg(src + i) : make_float4(0.f, 0.f, 0.f, 0.f);
  float* s_num = reinterpret_cast<float*>(sm + l.hot_number);
  for (int i = tid; i < a.m; i += kTreeThreads)
    s_num[i] = __ldg(a.uniforms + draft_uniform_index(row, n_prev + uint32_t(i), uint32_t(a.n_uniforms)));
  bool good = true;
  uint32_t prev = kEmpty, gone = kEmpty;                       // (a draw ordered elsewhere may still be under way)
  if (warp == 0 && lane < int(n_prev)) {
    good = poll([&] { prev = ld_relaxed(s_hot + 2 + lane); return prev != kEmpty; }, exit_flag);
    if (good) good = poll([&] { gone = ld_remote(rec_base + (prev & (kMaxRecords - 1)) * 16 + 8); return gone != kEmpty; }, exit_flag);
  }
  __syncthreads();
  if (gone != kEmpty) s_row[gone] = 0.f;
  __syncthreads();
  for (int c = warp; c < kChunks; c += kTreeThreads / 32) build_chunk(s_row, s_sub, c, lane);
  __syncthreads();
  if (warp == 1) {                                             // divides, waits for the order and sends
    if (lane != 0) return;
    for (uint32_t i = 0; i < uint32_t(a.m); ++i) {
      const Published* from = s_pub + (i & (kHotAhead - 1));
      const uint32_t* order = ring + (i & (kHotRing - 1));
      const uint32_t made = (i / kHotAhead) & 1u, asked = (i / kHotRing) & 1u;
      unsigned long long w = 0;
      if (!poll([&] { w = ld_acquire64(&from->word); return uint32_t(w >> 63) == made; }, exit_flag)) return;
      const double sum = from->sum, p = double(__uint_as_float(uint32_t(w)));
      st_release(s_go + 2, i + 1);                             // read: the place may be written again
      const double r = sum > 0.0 ? p / sum : 0.0;
      uint32_t msg = kEmpty;
      if (!poll([&] { msg = ld_relaxed(order); return msg != kEmpty && (msg >> 31) == asked; }, exit_flag)) return;
      const uint32_t rec = msg & 0x1FFFu;
      st_remote64(rec_base + rec * 16, (unsigned long long)__double_as_longlong(r));
      st_remote(rec_base + rec * 16 + 8, uint32_t(w >> 32) & 0x7FFFu);
    }
    return;
  }
  if (warp != 0 || !__all_sync(0xffffffffu, good)) return;

  // ---- the stream.  Lane c holds the prefix sum over chunks 0 .. c.
  Pair upto = scan(s_sub[(lane * kSubs + kSubs - 1) * 32 + 31], lane);
  Pair total{__shfl_sync(0xffffffffu, upto.hi, 31), __shfl_sync(0xffffffffu, upto.lo, 31)};
  double built = total.hi;
  uint32_t taken = 0;
  float u_next = s_num[0];
  for (uint32_t i = 0; i < uint32_t(a.m); ++i) {               // ahead of the orders, as far as the buffer goes
    const uint32_t at = i & (kHotAhead - 1), phase = (i / kHotAhead) & 1u;
    if (i - taken >= uint32_t(kHotAhead) &&
        !poll([&] { taken = ld_acquire(s_go + 2); return i - taken < uint32_t(kHotAhead); }, exit_flag))
      return;
    const uint32_t stop = ld_relaxed(exit_flag);
    const float u = u_next;
    u_next = s_num[min(i + 1, uint32_t(a.m - 1))];
    const double sum = total.hi + total.lo, target = double(u) * sum;
    const double mine = upto.hi + upto.lo;
    // chunk, then sub-block, then token: the first whose prefix sum exceeds the target
    const uint32_t in_chunk = __ballot_sync(0xffffffffu, mine > target);
    const bool none = in_chunk == 0u;                          // rounding (or an empty residual) left no crossing: the last token
    const int c = none ? (a.vocab - 1) / kChunk : __ffs(in_chunk) - 1;
    const double up = __shfl_sync(0xffffffffu, mine, (c - 1) & 31), before = c ? up : 0.0;
    Pair q[kSubs];
    double w[kSubs];
#pragma unroll
    for (int j = 0; j < kSubs; ++j) q[j] = s_sub[(c * kSubs + j) * 32 + lane];
#pragma unroll
    for (int j = 0; j < kSubs; ++j) w[j] = before + (q[j].hi + q[j].lo);
    const uint32_t in_sub = __ballot_sync(0xffffffffu, w[kSubs - 1] > target);
    const double left = __shfl_up_sync(0xffffffffu, w[kSubs - 1], 1);
    double from = lane ? left : before;                        // prefix sum in front of this lane's crossing sub-block
    int sub = kSubs * lane;
#pragma unroll
    for (int j = 0; j < kSubs - 1; ++j)
      if (!(w[j] > target)) { from = w[j]; sub = kSubs * lane + j + 1; }
    const int who = in_sub ? __ffs(in_sub) - 1 : 31;
    sub = __shfl_sync(0xffffffffu, sub, who);
    from = __shfl_sync(0xffffffffu, from, who);
    if (none) sub = ((a.vocab - 1) % kChunk) / kSub;
    float* xs = s_row + c * kChunk + sub * kSub;
    // two tokens per lane, lanes 0 .. 3 (the others repeat them): prefix sums in front of each pair
    constexpr int kPairs = kSub / 2;
    static_assert(kPairs == 4, "three lanes in front at most");
    constexpr uint32_t kPairLanes = (1u << kPairs) - 1u;
    const int t = lane & (kPairs - 1);
    const float2 x = reinterpret_cast<const float2*>(xs)[t];
    const double d0 = x.x, d1 = x.y, both = d0 + d1;
    double z1 = __shfl_up_sync(0xffffffffu, both, 1, kPairs), z2 = __shfl_up_sync(0xffffffffu, both, 2, kPairs),
           z3 = __shfl_up_sync(0xffffffffu, both, 3, kPairs);    // (three at once: a step of a scan waits for the one before)
    if (t < 1) z1 = 0.0;
    if (t < 2) z2 = 0.0;
    if (t < 3) z3 = 0.0;
    const double at_pair = from + (z3 + (z2 + z1));
    const bool h0 = at_pair + d0 > target, h1 = at_pair + both > target;
    const uint32_t b0 = __ballot_sync(0xffffffffu, h0), b1 = __ballot_sync(0xffffffffu, h1) & kPairLanes;
    int lt = __ffs(b1) - 1, pick = 2 * lt + (((b0 >> (lt & 31)) & 1u) ? 0 : 1);
    double p = __shfl_sync(0xffffffffu, h0 ? d0 : d1, lt & 31);
    if (none || b1 == 0u) {                                    // rounding left no crossing: the last token with mass
      const uint32_t m = __ballot_sync(0xffffffffu, x.x > 0.f || x.y > 0.f) & kPairLanes, m1 = __ballot_sync(0xffffffffu, x.y > 0.f);
      lt = m ? 31 - __clz(m) : 0;
      pick = 2 * lt + int((m1 >> lt) & 1u);
      if (none) pick = (a.vocab - 1) & (kSub - 1);
      p = double(xs[pick]);
    }
    const int y = min(c * kChunk + sub * kSub + pick, a.vocab - 1);
    // the token leaves the row: every prefix sum from it on
    __syncwarp();
    if (lane == 0) {
      xs[pick] = 0.f;
      s_pub[at].sum = sum;
      st_release64(&s_pub[at].word, ((unsigned long long)phase << 63) | ((unsigned long long)y << 32) |
                                        (unsigned long long)__float_as_uint(float(p)));
    }
    total = take_off(total, p);
    const Pair cut = take_off(upto, p);
    if (lane >= c) upto = cut;
#pragma unroll
    for (int j = 0; j < kSubs; ++j) {
      q[j] = take_off(q[j], p);
      if (kSubs * lane + j >= sub) s_sub[(c * kSubs + j) * 32 + lane] = q[j];
    }
    __syncwarp();
    if (stop) return;
    // rare: what is left is small against the tables' rounding, or no number (a token that was none may just have left)
    if (!(total.hi + total.lo >= built * 0x1p-40)) {
      for (int k = 0; k < kChunks; ++k) build_chunk(s_row, s_sub, k, lane);
      __syncwarp();
      upto = scan(s_sub[(lane * kSubs + kSubs - 1) * 32 + 31], lane);
      total = Pair{__shfl_sync(0xffffffffu, upto.hi, 31), __shfl_sync(0xffffffffu, upto.lo, 31)};
      built = total.hi;
    }
  }
}

template <bool kGreedy, int K>
__global__ void __launch_bounds__(kTreeThreads, 1)
build_tree_kernel(const __grid_constant__ TreeArgs a) {
  extern __shared__ __align__(16) uint8_t csm[];
  __shared__ uint32_t s_exit, s_never, s_final, s_opened, s_log_n;       // (planner and helper do not listen to s_exit)
  __shared__ uint32_t s_tail[8 * kDrawWarps + kMaxHot];
  __shared__ uint32_t s_hot[2 + 32], s_go[3];
  __shared__ uint32_t s_mask[kDrawWarps][32];
  __shared__ __align__(8) unsigned long long s_full[kMaxStages], s_empty[kMaxStages];
  const TreeLayout& l = a.lay;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = cluster_ctarank();
  uint32_t n_cta;
  asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(n_cta));
  const int req = int(blockIdx.x / n_cta);
  const bool planner_cta = rank == 0, worker_cta = int(rank) >= l.first_worker, hot_cta = !planner_cta && !worker_cta;

  // ---- every word that another warp or CTA will write starts as "not there yet"
  if (tid == 0) { s_exit = 0u; s_never = 0u; s_final = kEmpty; s_opened = 0u; s_log_n = 0u; }
  if (tid < kMaxStages) {
    mbar_init(smem_u32(s_full + tid), 1);
    mbar_init(smem_u32(s_empty + tid), kLoadWarps);
    fence_barrier_init();
  }
  if (tid < 8 * kDrawWarps + kMaxHot) s_tail[tid] = 0u;
  if (tid < 2 + 32) s_hot[tid] = kEmpty;
  auto fill = [&](int off, int words, uint32_t v) {
    uint32_t* p = reinterpret_cast<uint32_t*>(csm + off);
    for (int i = tid; i < words; i += kTreeThreads) p[i] = v;
  };
  if (planner_cta) {
    fill(l.rec, l.n_records * 4, kEmpty);
    fill(l.note, l.nodes_pad * 4, kEmpty);
    for (int i = tid; i < l.nodes_pad; i += kTreeThreads) reinterpret_cast<OpenSlot*>(csm + l.open)[i] = OpenSlot{-1.0, kEmpty, kEmpty};
    fill(l.first, l.nodes_pad, kEmpty);
    fill(l.hash_row, l.hash_size, kEmpty);
  }
  if (worker_cta) {
    fill(l.load_row, l.max_entries, kEmpty);
    fill(l.sums, l.entries_local * kLeaves * 2, kEmpty);
    fill(l.number, l.entries_local, kEmpty);
    fill(l.attempts, l.entries_local, 0u);
    fill(l.ring, kDrawWarps * l.ring_size, kEmpty);
    fill(l.log, l.n_records, kEmpty);
  }
  if (hot_cta) {
    fill(l.hot_ring, kHotRing, kEmpty);
    fill(l.hot_pub, kHotAhead * int(sizeof(Published)) / 4, kEmpty);
  }
  __syncthreads();
  cluster_sync_all();

  const Shared s = planner_view(csm, l);
  if (hot_cta) {
    run_hot(a, csm, s_hot, s_go, &s_exit);
  } else if (warp == 0) {
    if (planner_cta) {
      const bool patient = a.wait_limit_ns >= kPatientNs;
      const int n = kGreedy ? (patient ? plan_greedy<true>(a, s, &s_never) : plan_greedy<false>(a, s, &s_never))
                            : (patient ? plan_threshold<true>(a, s, &s_never) : plan_threshold<false>(a, s, &s_never));
      __syncwarp();
      if (lane == 0) {
        a.n_nodes[req] = n + 1;                                // 0: a wait ran out
        if (n < 0 && a.status) atomicCAS(a.status, 0, DYSPEC_ERR_TIMEOUT);
        st_relaxed(&s_final, n < 0 ? 0u : uint32_t(n));
      }
      for (uint32_t c = uint32_t(lane); c < n_cta; c += 32) st_remote(map_to_cta(smem_u32(&s_exit), c), 1u);
    }
  } else if (warp == 1) {
    if (planner_cta) run_opener<kGreedy>(a, s, csm, s_tail, smem_u32(s_hot), &s_opened, &s_final, &s_never, req);
  } else if (warp == 2) {
    if (planner_cta) run_orderer<kGreedy>(a, s, csm, s_tail, smem_u32(s_hot), &s_opened, &s_final, &s_never);
  } else if (worker_cta) {
    if (warp < kRoles + kDrawWarps) run_drawer<K>(a, csm, warp - kRoles, int(rank) - l.first_worker, s_mask, &s_log_n, &s_exit);
    else if (warp == kRoles + kDrawWarps) run_fetcher<K>(a, csm, int(rank) - l.first_worker, s_full, s_empty, &s_never, &s_exit);
    else run_loader<K>(a, csm, warp - kRoles - kDrawWarps - 1, int(rank) - l.first_worker, s_full, s_empty, &s_exit);
  }
  __syncwarp();
  cluster_sync_all();                                          // nobody leaves while its shared memory may be written

  if (planner_cta) {                                           // the tree, from the planner's and the helper's notes
    const int n = int(s_final);
    const size_t base = size_t(req) * (a.m + 1);
    for (int k = tid; k <= n; k += kTreeThreads) {
      const NodeNote note = s.note[k];
      const DrawRecord rc = s.rec[k ? note.event & 0x1FFFu : 0u];
      a.parents[base + k] = k ? int32_t(note.event >> 13) : -1;
      a.tokens[base + k] = k ? int32_t(rc.token) : 0;
      a.values[base + k] = k ? float(note.v) : 1.f;
      a.child_values[base + k] = k ? float(note.v * __longlong_as_double((long long)rc.r_bits)) : 1.f;
      a.rows[base + k] = int32_t(note.row);
    }
  }
}

// Cluster of C CTAs: CTA 0 plans, n_hot take over long streams, the others load and draw (one CTA does it all when C = 1).
bool tree_layout(int nodes, int n_rows, int leaf_bytes, int C, int n_hot, TreeLayout& l) {
  l.nodes_pad = (nodes + 1 + 31) & ~31;
  l.max_entries = nodes + 1 < n_rows ? nodes + 1 : n_rows;
  l.n_hot = n_hot;
  l.first_worker = C > 1 ? 1 + n_hot : 0;
  l.n_workers = C - l.first_worker;
  l.entries_local = (l.max_entries + l.n_workers - 1) / l.n_workers;
  const int per_drawer = (l.entries_local + kDrawWarps - 1) / kDrawWarps;
  l.ring_shift = 5;
  while ((1 << l.ring_shift) < per_drawer * kMaxAhead) ++l.ring_shift;
  l.ring_size = 1 << l.ring_shift;
  l.hash_size = 32;
  while (l.hash_size < 2 * l.max_entries) l.hash_size *= 2;
  // Records: one per row to open and one per node is what the tree can need; the rest lets draws run ahead.
  l.n_stages = kMaxStages;
  int open_ahead = 4, run_ahead = nodes + 4 * l.max_entries;
  for (;;) {
    l.open_records = l.max_entries * open_ahead;
    l.n_records = l.open_records + nodes + 1 + run_ahead;
    int at = 0;
    auto take = [&](int bytes) { const int o = at; at = (at + bytes + 15) & ~15; return o; };
    l.rec = take(l.n_records * 16);
    l.open = take(l.nodes_pad * int(sizeof(OpenSlot)));
    l.note = take(l.nodes_pad * int(sizeof(NodeNote)));
    l.first = take(l.nodes_pad * 4);
    l.rec_owner = take(l.n_records * 4);
    l.hash_row = take(l.hash_size * 4);
    l.hash_val = take(l.hash_size * 4);
    l.entry = take(l.max_entries * int(sizeof(EntryState)));
    l.bytes = at;
    if (C > 1) at = 0;                                         // the other CTAs hold none of the above
    l.stage = take(l.n_stages * kBatch * leaf_bytes);
    l.sums = take(l.entries_local * kLeaves * 8);
    l.load_row = take(l.max_entries * 4);
    l.attempts = take(l.entries_local * 4);
    l.number = take(l.entries_local * 4);
    l.ring = take(kDrawWarps * l.ring_size * 4);
    l.log = take(l.n_records * 4);
    if (at > l.bytes) l.bytes = at;
    at = 0;
    l.hot_row = take(n_hot ? kChunks * kChunk * 4 : 0);
    l.hot_sub = take(n_hot ? kChunks * kChunk / kSub * int(sizeof(Pair)) : 0);
    l.hot_ring = take(n_hot ? kHotRing * 4 : 0);
    l.hot_pub = take(n_hot ? kHotAhead * int(sizeof(Published)) : 0);
    l.hot_number = take(n_hot ? nodes * 4 : 0);
    if (at > l.bytes) l.bytes = at;
    if (l.bytes <= 224 * 1024 && l.n_records <= kMaxRecords) return true;
    if (l.n_stages > 2) l.n_stages = 2;
    else if (run_ahead > nodes) run_ahead = nodes;
    else if (open_ahead > 2) open_ahead = 2;
    else if (run_ahead > 64) run_ahead /= 2;
    else if (open_ahead > 1) open_ahead = 1;
    else if (l.n_stages > 1) l.n_stages = 1;
    else return false;
  }
}

template <bool kGreedy, int K>
cudaError_t launch_tree(const TreeArgs& a, int n_req, int C, cudaStream_t stream) {
  static DynSmemGrant grant;
  if (cudaError_t e = grant.ensure(build_tree_kernel<kGreedy, K>, size_t(a.lay.bytes)); e != cudaSuccess) return e;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = unsigned(C);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(n_req) * unsigned(C));
  cfg.blockDim = dim3(kTreeThreads);
  cfg.dynamicSmemBytes = size_t(a.lay.bytes);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, build_tree_kernel<kGreedy, K>, a);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// The general form, one CTA a request (construct_rows.cu).
template <bool kGreedy>
cudaError_t launch_rows(const TreeArgs& a, int n_req, cudaStream_t stream) {
  return kGreedy ? launch_build_tree_greedy_rows(a.table, a.n_rows, a.vocab, a.uniforms, a.n_uniforms, a.root_row, n_req, a.m,
                                                 a.parents, a.tokens, a.values, a.child_values, a.rows, a.n_nodes, stream)
                 : launch_build_tree_threshold_rows(a.table, a.n_rows, a.vocab, a.uniforms, a.n_uniforms, a.root_row, n_req,
                                                    a.threshold, a.m, a.parents, a.tokens, a.values, a.child_values, a.rows,
                                                    a.n_nodes, stream);
}

template <bool kGreedy>
cudaError_t launch_tree(TreeArgs a, int n_req, cudaStream_t stream) {
  const int K = a.vocab <= kLeaves * 128 ? 1 : a.vocab <= kLeaves * 256 ? 2 : 4, leaf_bytes = 512 * K;
  auto fits = [&](int c) {
    for (int hot = c == 8 ? kMaxHot : c == 4 ? 1 : 0; hot >= 0; --hot)
      if ((hot == 0 || a.m > kHotLeast) && tree_layout(a.m, a.n_rows, leaf_bytes, c, hot, a.lay)) return true;
    return false;
  };
  // The largest cluster for which the SMs suffice, n_req C <= 148.  (15 clusters of 8 run at once and fewer than 36 of 4, an SM's
  // neighbours being what they are, but 16 - 18 requests in two waves of 8 take 150 - 290 us for 127 nodes and with clusters of
  // 4 120 - 290, 37 take 230 - 310 in two waves of 4 and 340 - 460 with clusters of 2.)
  int C = 8;
  while (C > 1 && int64_t(n_req) * C > kDefaultSMs) C /= 2;
  // Short trees: all at once.  (18 trees of 8 nodes: 37 us with clusters of 4, 61 - 66 in two waves of 8; of 16 nodes 45 - 54
  // and 48 - 68.  37 of 8: 43 with clusters of 2, 67 in two waves of 4; of 16 70 and 100; at 64 nodes two waves win.)
  static ClusterRoom room;
  while (C > 2 && a.m * C <= kShortTree && n_req > room.ask(build_tree_kernel<kGreedy, 4>, kTreeThreads, C)) C /= 2;
  // Trees with too many rows for that: the next larger cluster that has room for a hot CTA, in as many waves as it takes.
  // (24 trees of 768 distinct rows: 1.0 ms with clusters of 8, 2.3 with 4 and no hot CTA, 5.6 one CTA each; 148 of
  // them: 4.5 - 5.4, 11 and 5.6; 148 of 300 rows: 1.3 - 1.7 with clusters of 4, 3.5 with 2, 2.1 one CTA each.)
  if (!fits(C) || (C == 4 && a.m > kHotLeast && a.lay.n_hot == 0)) {
    const bool four = C < 4 && fits(4) && a.lay.n_hot > 0;
    C = four ? 4 : 8;
    if (!fits(C)) return launch_rows<kGreedy>(a, n_req, stream);
  }
  // How many requests clusters of 8 finish while 148 CTAs build one tree each depends on the hot CTAs that the rows leave room for.
  // (Vocabulary 16000 - 32000.  Three or two, up to 1550 rows: 148 trees in 0.8 - 1.04 of the single CTAs' time.  One, up to some
  // 1850: 75 in 0.5 - 0.8, 148 in 0.8 - 1.4, 300, three waves of CTAs, in 0.6 - 0.95.  None: 30 in 0.9, 38 in 1.3, 148 in 4.5.)
  const int together = a.lay.n_hot >= 2 ? kDefaultSMs : a.lay.n_hot == 1 ? 105 : 30;
  if (C == 8 && n_req > int64_t(together) * ((n_req + kDefaultSMs - 1) / kDefaultSMs)) return launch_rows<kGreedy>(a, n_req, stream);
  a.rows_inverse = uint32_t((1ull << 32) / uint64_t(a.n_rows) - (a.n_rows == 1 ? 1 : 0));
  for (;;) {
    const cudaError_t e = K == 1   ? launch_tree<kGreedy, 1>(a, n_req, C, stream)
                          : K == 2 ? launch_tree<kGreedy, 2>(a, n_req, C, stream)
                                   : launch_tree<kGreedy, 4>(a, n_req, C, stream);
    // a share of a device whose SMs hold no cluster of this size: a smaller one, if the tree fits there
    if (e != cudaErrorInvalidClusterSize || C == 1) return e;
    (void)cudaGetLastError();
    C /= 2;
    if (!fits(C)) return launch_rows<kGreedy>(a, n_req, stream);
  }
}

}  // namespace

cudaError_t launch_build_tree_greedy(const float* draft_table, int n_rows, int vocab, const float* uniforms, int n_uniforms,
                                     const int32_t* root_row, int n_req, int m, int32_t* parents, int32_t* tokens,
                                     float* values, float* child_values, int32_t* rows, int32_t* n_nodes,
                                     uint32_t wait_limit_ns, int32_t* status, cudaStream_t stream) {
  if (n_req <= 0) return cudaSuccess;
  return launch_tree<true>(TreeArgs{draft_table, uniforms, root_row, n_rows, vocab, n_uniforms, m, 0u, 0.f, wait_limit_ns, status, parents, tokens, values,
                                    child_values, rows, n_nodes, TreeLayout{}}, n_req, stream);
}

cudaError_t launch_build_tree_threshold(const float* draft_table, int n_rows, int vocab, const float* uniforms,
                                        int n_uniforms, const int32_t* root_row, int n_req, float threshold, int max_nodes,
                                        int32_t* parents, int32_t* tokens, float* values, float* child_values, int32_t* rows,
                                        int32_t* n_nodes, uint32_t wait_limit_ns, int32_t* status, cudaStream_t stream) {
  if (n_req <= 0) return cudaSuccess;
  return launch_tree<false>(TreeArgs{draft_table, uniforms, root_row, n_rows, vocab, n_uniforms, max_nodes, 0u, threshold, wait_limit_ns, status, parents,
                                     tokens, values, child_values, rows, n_nodes, TreeLayout{}}, n_req, stream);
}

}  // namespace dyspec
