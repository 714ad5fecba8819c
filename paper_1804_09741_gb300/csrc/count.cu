// K2: enumerate every weakly connected k-vertex set once, classify it by one
// table read, add it to the histogram (Problem 1 of Sec. 1; Sec. 3.1, 3.2).
//
// Enumeration (extension scheme of ESU, the "Fanmod" method of Table 1): a set
// is produced from its smallest vertex, the root v.  The root's candidate list
// is {u in delta(v) : u > v}; choosing a candidate w appends to the remaining
// candidates the exclusive neighbours of w -- neighbours larger than v that are
// neither in the current set nor adjacent to it.  With k-1 vertices chosen,
// every remaining candidate completes one k-set.
//
// GPU mapping (one warp = one depth-first walk, lanes cooperate):
//  * per warp a "relation word" lab[u] for every vertex: bits 2p, 2p+1 hold the
//    A/B/C relation (Sec. 2) of u to the vertex at position p of the current
//    set.  Pushing w at position p scans delta(w) above the root coalesced
//    (the row-scan strategy of Sec. 3.1), ORs its relation bits into lab[u]
//    and, with one ballot, appends to the candidate stack every u with no
//    relation to the earlier positions (exclusive neighbour).  Popping clears
//    the same bits.  Words are 8, 16 or 32 bits (see LabT): the bits above the
//    first k-2 positions are slots for the (k-1)-th choices;
//  * candidate lists of all levels live in one per-warp stack: level p+1's list
//    is the unused tail of level p's list followed by the newly appended
//    exclusive neighbours, so no list is ever copied;
//  * the current level's state (cursor, ends, key prefix) lives in warp-uniform
//    registers; suspended levels wait in a small per-warp stack in shared
//    memory;
//  * choosing the (k-1)-th vertex finishes its k-sets in place, for up to GS
//    choices at once: the choices' rows, concatenated over the lanes, mark
//    each choice's slot in its neighbours' words and classify the exclusive
//    neighbours (their word is the arc code to the choice); then one pass over
//    the remaining candidates classifies every choice's leaves from the words
//    (key prefix OR word) and clears the slots again -- no per-subgraph
//    adjacency test; one match_any groups the pass's lanes for every choice
//    at once (tag: the candidate's word, which fixes its key for each choice,
//    plus the number of choices it is a leaf of), and a group of equal keys
//    shares one table read; k = 6 launches with many blocks per graph match
//    three choices at a time instead (see kWideTailBlocksPerGraph); at k = 6,
//    short candidate lists let several choices share one pass, a (choice,
//    candidate) pair per lane;
//  * MT_METHOD_CELLS, the automatic choice at every k, stops one level
//    earlier and counts the last two vertices per pair of cells (Algorithm 1 of
//    Sec. 3; see pair_level below);
//  * histograms: per-block shared-memory 32-bit counters for k <= 5 (13 / 199
//    / 9,364 classes), the graph's 64-bit global counters for k = 6 (a
//    one-graph count spreads its blocks over kHistCopies copies of them and
//    folds the copies afterwards), both updated with reductions that return
//    nothing (PTX red).
//
// Work items are (graph, root, first-level branch range) or, for expensive
// branches, (graph, root, branch, second-level choice range); a planner sizes
// them from per-branch cost estimates.  Hub graphs whose candidate stacks
// ((k-2) x max degree + 32 entries per warp) would leave few warps in shared
// memory keep the stacks in per-warp slices of global memory.  Blocks work
// graph by graph, warps take the items of the block's current graph from that
// graph's queue, and a warp that runs out takes halves of its block-mates'
// remaining ranges (work donation).
#include <algorithm>
#include <type_traits>

#include "count.cuh"

namespace mt {

struct Hdr {
  uint32_t err;
  uint32_t pad[3];
};

// The planner's result for one graph: its estimated work, and its items
// [base, base + count) of the launch's array with the queue's head.
struct GraphPlan {
  double est;
  uint32_t count, base;
  uint32_t qhead, pad;
};

static_assert(sizeof(GraphPlan) % 8 == 0, "zeroed in 8-byte words");

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kTargetItemsPerWarp = 64;
// Cell method: an item's least estimated work, below which fetching it and
// marking its root's neighbours costs more than the warps it feeds give.  One
// graph on a GB300: k = 4 (n = 2,000) 97 us at 128 against 113 at 32 and 140 at
// 512; k = 5 (n = 112 / 310 / 343) 127 / 177 / 115 us at 128, 151 / 225 / 138 at
// 512, 114 / 173 / 115 near 10, n = 1,500 indifferent; k = 3 (n = 20,000) 131 us at
// 1,024, 151 at 512.
template <int K>
constexpr double kCellsItemFloor = K == 3 ? 1024.0 : 128.0;
// Adds one warp may make to a shared 32-bit histogram between two flushes of
// it by exchange (enumeration path, k <= 5; see `ladd` in k_count).
constexpr int kLeafBudget = 1 << 25;
// The same for the cell method, whose adds also come in larger steps: one list's
// pairs (at most 2^24, or they go to the graph's counters), 32 rows' arcs, and the
// list's exclusive counts.  Those are charged as the rows are read but added at the
// list's end, so a flush in between leaves them uncharged: at most one list's per
// warp, each below 2^20 (larger ones go to the graph's counters), and one class
// takes few of a list's (cell, code) counts.  So a counter stays below 32 warps x
// (2 x 2^24 and a few 2^20) < 2^31.
constexpr int kCellBudget = 1 << 24;
// Items a block's warps can hand to each other at once (work donation).
constexpr int kDonSlots = 32;
// Bounds of the waits of work donation: lock attempts, idle polls, and the
// idle time (ns) after which a warp gives up and reports kErrWaitLimit.
constexpr int kLockTries = 1 << 24;
constexpr int kIdlePolls = 1 << 28;
constexpr unsigned long long kIdleNs = 60ull * 1000 * 1000 * 1000;  // default; mt_set_wait_limit

// Idle-wait limit (ns) given to the launches enqueued from now on.
static unsigned long long g_idle_ns = kIdleNs;

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
constexpr int kMaxWarpsPerBlock = 32;
// k = 6 launches with at most this many blocks per histogram (copy) group a
// tail batch's lanes with one match for all of a group's choices; launches over
// fewer graphs match three choices at a time.  A block works on one graph at a time, so with
// few graphs many blocks add into the same global histogram; there the single
// match's finer groups (more leaders, each adding for every choice) sent 29%
// more reduction sectors to L2 and ran slower.  Measured on 152 blocks, k = 6
// batches of 2 .. 33 graphs run 22% .. 1.5% faster with three choices per
// match, 49 alike, 65 3% slower.
constexpr int kWideTailBlocksPerGraph = 3;
// A one-graph k = 6 count spreads its blocks over this many copies of the
// graph's histogram (block b adds into copy b mod kHistCopies), folded into the
// caller's histogram by k_fold_copies: ~19 blocks per copy on 152 SMs instead
// of all blocks on the same counters.  Measured on the k = 6 workload graph and
// three of its nulls (n = 800, m = 3,200): 16.0-16.4 ms per count without
// copies, 5.6-5.8 ms with 8, histograms identical.
constexpr int kHistCopies = 8;
// Per-warp stack of suspended DFS levels: (cursor, choice end, tail end, key, vertex).
constexpr int kLevelBytes = 128;

__device__ __forceinline__ float choose_f(int x, int r) {
  if (x < r) return 0.f;
  float c = 1.f;
  for (int i = 0; i < r; ++i) c = c * (float)(x - i) / (float)(i + 1);
  return c;
}

// Estimated work of a first-level branch whose second-level candidate list has
// x1 entries, whose degrees add up to w1.  Per-subgraph method: about
// C(x1, k-2) sets of k-1 vertices, each touching its candidates once.  Cell
// method: a fixed cost (64) for each (k-2)-set, and its list; the third-level
// lists (x1^2 / 2 + w1 entries together) are the k = 5 sets' lists and the number
// of k = 6 sets.  With x1 alone a k = 6 branch that reaches a hub was estimated
// 160 times too low, and its block ran on after the others (SMs active 2.2 to
// 4.1 million cycles on one graph of n = 800).
template <int K, bool CB>
__device__ __forceinline__ float branch_cost(int x1, float w1) {
  const float x = (float)x1;
  if (!CB) return 1.f + x + choose_f(x1, K - 2) * (K >= 4 ? 2.f : 1.f);
  if (K == 3) return 8.f + x;
  if (K == 4) return 72.f + 2.f * x;
  const float l2 = 0.5f * x * x + w1;
  return K == 5 ? 8.f + 65.f * x + l2 : 8.f + x + l2 * (64.f + x);
}

// Offset of position p's 2p bits in an extension-order key of k vertices:
// later positions sit lower, so the k-sets below one (k-2)-set differ only in
// the low bits of their keys and read nearby table slots.
__host__ __device__ constexpr int key_off(int k, int p) { return k * (k - 1) - p * (p + 1); }

// Histogram reductions without a returned value (PTX red): the issuing warp
// never waits for them.
__device__ __forceinline__ void red_add_global(unsigned long long* p, unsigned long long v) {
  asm volatile("red.global.add.u64 [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "l"(v)
               : "memory");
}
__device__ __forceinline__ void red_add_shared(int* p, int v) {
  asm volatile("red.shared.add.s32 [%0], %1;" ::"r"((unsigned)__cvta_generic_to_shared(p)), "r"(v)
               : "memory");
}

// First index in sorted packed entries [lo, hi) whose vertex is > x.
__device__ __forceinline__ int first_above(const uint32_t* __restrict__ ucol, int lo, int hi,
                                           int x) {
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if ((int)(__ldg(&ucol[mid]) & kVertexMask) > x) hi = mid; else lo = mid + 1;
  }
  return lo;
}

// ------------------------------------------------------------------ planner
//
// Two launches: the graphs' estimated work, then their items.  A branch's
// estimate takes the neighbours of its vertex above the root as its new
// candidates, common neighbours counted twice: that bounds the second-level list
// (ranges past its end are empty items) and needs one binary search where exact
// counts took a search per neighbour.  Measured on a GB300, one k = 5 graph
// (n = 1,500): 400 us before, 40 now;
// 512 graphs of n = 300 at k = 3: 590 us before, 130 now.

// Sum of the neighbours' degrees of every vertex (the cell method at k >= 5).
__global__ void __launch_bounds__(256) k_plan_degsum(const DevGraph* __restrict__ graphs, int nmax,
                                                     int32_t* dsum) {
  const DevGraph G = graphs[blockIdx.y];
  const int lane = threadIdx.x & 31;
  const int nwarps = (int)(gridDim.x * (blockDim.x >> 5));
  for (int v = blockIdx.x * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5); v < G.n;
       v += nwarps) {
    int sum = 0;
    for (int i = G.urow[v] + lane; i < G.urow[v + 1]; i += 32) {
      const int u = (int)(G.ucol[i] & kVertexMask);
      sum += G.urow[u + 1] - G.urow[u];
    }
    for (int d = 16; d; d >>= 1) sum += __shfl_xor_sync(kFull, sum, d);
    if (lane == 0) dsum[(int64_t)blockIdx.y * nmax + v] = sum;
  }
}

// Branch of entry e (a forward entry of root v, whose row is [rs, re)): its
// cost, and x = the bound of its second-level list.  dsum: this graph's sums of
// the neighbours' degrees; the degrees of the root's later neighbours are taken
// as the row's mean.
template <int K, bool CB>
__device__ __forceinline__ float entry_cost(const DevGraph& G, const int32_t* __restrict__ dsum,
                                            int v, int rs, int re, int e, int& x) {
  const int u = (int)(__ldg(&G.ucol[e]) & kVertexMask);
  const int ue = __ldg(&G.urow[u + 1]);
  x = (re - e - 1) + (ue - first_above(G.ucol, __ldg(&G.urow[u]), ue, v));
  float w = 0.f;
  if (CB && K >= 5)
    w = (float)__ldg(&dsum[u]) + (float)(re - e - 1) * ((float)__ldg(&dsum[v]) / (float)(re - rs));
  return branch_cost<K, CB>(x, w);
}

template <int K, bool CB>
__global__ void __launch_bounds__(256) k_plan_total(const DevGraph* __restrict__ graphs,
                                                    GraphPlan* gp,
                                                    const int32_t* __restrict__ dsum_all, int nmax,
                                                    int root_begin, int root_end) {
  __shared__ double red[8];
  const DevGraph G = graphs[blockIdx.y];
  const int32_t* dsum = dsum_all + (int64_t)blockIdx.y * nmax;
  const int r0 = max(root_begin, G.root_begin), r1 = min(root_end, G.root_end);
  double local = 0.0;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < G.nu; e += gridDim.x * blockDim.x) {
    const int v = __ldg(&G.usrc[e]);
    if (v < r0 || v >= r1) continue;
    const int rs = __ldg(&G.urow[v]);
    int x;
    if (e >= rs + __ldg(&G.ufwd[v]))
      local += entry_cost<K, CB>(G, dsum, v, rs, __ldg(&G.urow[v + 1]), e, x);
  }
  for (int d = 16; d; d >>= 1) local += __shfl_xor_sync(kFull, local, d);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = local;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
    if (s > 0.0) atomicAdd(&gp[blockIdx.y].est, s);
  }
}

// How the roots are cut into items.
struct SplitArgs {
  double split_cost, split_scale, target_items, items_factor, floor;
  uint64_t items_max;
  int root_begin, root_end;
};

// A warp takes 32 branches of a root at a time, a lane each (hub roots have more
// and are spread over the grid's z).  Branches above twice the threshold T are
// cut into second-level ranges; the others form first-level ranges, a new one
// wherever the running cost passes a multiple of T, next to a cut branch and
// every 32 branches.  A graph's items start at the sum of the
// bounds of the graphs before it (every block adds them up: G is at most some
// hundreds) and are handed out by an atomic counter.
template <int K, bool CB>
__global__ void __launch_bounds__(256) k_plan_items(const DevGraph* __restrict__ graphs, int ng,
                                                    GraphPlan* gp,
                                                    const int32_t* __restrict__ dsum_all, int nmax,
                                                    Item* items, Hdr* hdr, SplitArgs a) {
  __shared__ double red[8];
  __shared__ unsigned long long redb[8];
  __shared__ float s_T;
  __shared__ uint32_t s_base;
  const int g = blockIdx.y;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double local = 0.0;
  for (int h = threadIdx.x; h < ng; h += blockDim.x) local += gp[h].est;
  for (int d = 16; d; d >>= 1) local += __shfl_xor_sync(kFull, local, d);
  if (lane == 0) red[wid] = local;
  __syncthreads();
  if (threadIdx.x == 0) {
    double total = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) total += red[i];
    // root-split threshold: explicit, or the automatic one scaled; never so small
    // that the items exceed their budget
    const double t_auto = fmax(total / a.target_items, a.floor);
    double T = a.split_cost > 0.0 ? a.split_cost : t_auto * a.split_scale;
    T = fmax(fmax(T, total / (a.items_factor * a.target_items)), 1.0);
    s_T = (float)T;
  }
  __syncthreads();
  const float T = s_T, inv_T = 1.f / T;
  unsigned long long before = 0;
  for (int h = threadIdx.x; h < g; h += blockDim.x)
    before += (unsigned long long)(gp[h].est / (double)T * 1.001) +
              2ull * (unsigned)(graphs[h].nu / 2) + 16ull;
  for (int d = 16; d; d >>= 1) before += __shfl_xor_sync(kFull, before, d);
  if (lane == 0) redb[wid] = before;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long b = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) b += redb[i];
    s_base = (uint32_t)min(b, (unsigned long long)a.items_max);
    if (blockIdx.x == 0 && blockIdx.z == 0) gp[g].base = s_base;
  }
  __syncthreads();
  const uint32_t base = s_base;
  const DevGraph G = graphs[g];
  const int32_t* dsum = dsum_all + (int64_t)g * nmax;
  const int r0 = max(max(a.root_begin, G.root_begin), 0);
  const int r1 = min(min(a.root_end, G.root_end), G.n);
  const int nwarps = (int)(gridDim.x * (blockDim.x >> 5));
  for (int v = r0 + (int)(blockIdx.x * (blockDim.x >> 5)) + wid; v < r1; v += nwarps) {
    const int rs = __ldg(&G.urow[v]), re = __ldg(&G.urow[v + 1]);
    const int f = rs + __ldg(&G.ufwd[v]);
    const int dplus = re - f;
    auto put = [&](uint32_t at, int j1a, int j1b, int a2, int b2) {
      const uint64_t pos = (uint64_t)base + at;
      if (pos < a.items_max) {
        Item it;
        it.root = (uint32_t)v;
        it.j1a = (uint16_t)j1a;
        it.j1b = (uint16_t)j1b;
        it.a2 = (uint16_t)a2;
        it.b2 = (uint16_t)b2;
        it.a3 = 0;
        it.b3 = 0xFFFF;
        items[pos] = it;
      } else {
        atomicOr(&hdr->err, kErrStackOverflow);
      }
    };
    for (int jb = 32 * (int)blockIdx.z; jb < dplus; jb += 32 * (int)gridDim.z) {
      const int n = min(32, dplus - jb);
      const int j = jb + lane;
      float c = 0.f;
      int x = 0;
      if (lane < n) c = entry_cost<K, CB>(G, dsum, v, rs, re, f + j, x);
      const bool cut = K >= 4 && lane < n && c > 2.f * T && x >= 2;
      int r2 = 0, ns = 0;
      if (cut) {
        const int nch = min((int)ceilf(fminf(c * inv_T, 65536.f)), x);
        r2 = (x + nch - 1) / nch;
        ns = (x + r2 - 1) / r2;
      }
      float sum = cut ? 0.f : c;
      for (int d = 1; d < 32; d <<= 1) {
        const float y = __shfl_up_sync(kFull, sum, d);
        if (lane >= d) sum += y;
      }
      const int step = (int)fminf((sum - (cut ? 0.f : c)) * inv_T, 1e9f);
      const int step_before = __shfl_up_sync(kFull, step, 1);
      const unsigned cuts = __ballot_sync(kFull, cut);
      const bool start = lane < n && !cut &&
                         (lane == 0 || (cuts >> (lane - 1) & 1u) || step != step_before);
      const unsigned ends = cuts | __ballot_sync(kFull, start);
      const int mine = start ? 1 : ns;
      const int incl = warp_incl_scan(mine);
      uint32_t at = 0;
      const int all = __shfl_sync(kFull, incl, 31);
      if (lane == 0 && all) at = atomicAdd(&gp[g].count, (uint32_t)all);
      at = __shfl_sync(kFull, at, 0);
      if (start) {
        const unsigned later = lane == 31 ? 0u : ends >> (lane + 1);
        const int end = later ? lane + __ffs(later) : n;
        put(at + incl - 1, j, jb + end, 0, 0xFFFF);
      }
      for (unsigned q = cuts; q; q &= q - 1) {
        const int l = __ffs(q) - 1;
        const int ns_l = __shfl_sync(kFull, ns, l), r_l = __shfl_sync(kFull, r2, l);
        const int x_l = __shfl_sync(kFull, x, l);
        const uint32_t at_l = at + (uint32_t)(__shfl_sync(kFull, incl, l) - ns_l);
        for (int t = lane; t < ns_l; t += 32)
          put(at_l + t, jb + l, jb + l + 1, t * r_l, min(t * r_l + r_l, x_l));
      }
    }
  }
}

// ------------------------------------------------------------------ enumerator

// Relation words: 2 bits per earlier position.  The first k-2 positions take
// 2(k-2) bits; the slots above them let several (k-1)-th choices be marked at
// once: 8 bits for k <= 4 (3 and 2 slots), 16 bits for k = 5 (5 slots), 32 bits
// for k = 6 (8 slots used).  The cell method needs only two flag bits above
// them: 8 bits up to k = 5, 16 bits for k = 6.
template <int K, bool CB>
using LabT = typename std::conditional<
    (K <= 4 || (CB && K <= 5)), uint8_t,
    typename std::conditional<(K == 5 || CB), uint16_t, uint32_t>::type>::type;

// Neighbour entries as the enumerator reads them: the graph's 32-bit entries
// (vertex in bits 0..29, arc code in bits 30..31) or, in the shared-memory copy
// the cell method makes of graphs of fewer than 2^14 vertices, 16-bit ones
// (vertex in bits 0..13, code in bits 14..15).  2^14 is what the format holds; the
// layout rule stops making copies earlier (near n = 4,000 at two arcs per vertex).
__device__ __forceinline__ int ent_vertex(uint32_t e) { return (int)(e & kVertexMask); }
__device__ __forceinline__ uint32_t ent_code(uint32_t e) { return e >> 30; }
constexpr int kMaxVertices16 = 1 << 14;
__device__ __forceinline__ int ent_vertex(uint16_t e) { return (int)(e & 0x3FFFu); }
__device__ __forceinline__ uint32_t ent_code(uint16_t e) { return (uint32_t)e >> 14; }

// Row segments of the cell method: entries one lane reads at a time.  Rows of
// the 16-bit copy start at multiples of kSeg entries and are padded with zeros.
constexpr int kSeg = 8;

template <typename LT, typename ET>
struct WarpCtx {
  // 32-bit entries: row x is [urow[x], urow[x + 1]).  16-bit ones: urow[x] holds
  // its start / kSeg (bits 16..31) and its length.
  const int32_t* urow;   // shared-memory copy of the graph or global memory
  const ET* ucol;
  LT* lab;
  uint16_t* buf;
  int cap;
  int root;
  int lane;
  uint32_t* err;
  __device__ __forceinline__ void row(int x, int& rs, int& re) const {
    if (sizeof(ET) == 2) {
      const uint32_t r = (uint32_t)urow[x];
      rs = (int)(r >> 16) * kSeg;
      re = rs + (int)(r & 0xFFFFu);
    } else {
      rs = urow[x];
      re = urow[x + 1];
    }
  }
};

// First index in sorted packed entries [lo, hi) whose vertex is > x.
template <typename ET>
__device__ __forceinline__ int first_above_p(const ET* ucol, int lo, int hi, int x) {
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (ent_vertex(ucol[mid]) > x) hi = mid; else lo = mid + 1;
  }
  return lo;
}

// Push x at position p: OR its relation bits into lab[] of its neighbours above
// the root and append the exclusive ones (no relation to positions 0..p-1, the
// bits in `low`; bits above it may be stale) at stack index e.  Returns the
// new end of the candidate list.
template <typename LT, typename ET>
__device__ __forceinline__ int push_vertex(const WarpCtx<LT, ET>& w, int x, int p, int e,
                                           uint32_t low) {
  int rs, re;
  w.row(x, rs, re);
  const int start = (re - rs > 32) ? first_above_p(w.ucol, rs, re, w.root) : rs;
  const unsigned lt = (1u << w.lane) - 1u;
  int cnt = 0;
  for (int b = start; b < re; b += 32) {
    const int i = b + w.lane;
    bool ex = false;
    int u = 0;
    if (i < re) {
      const ET ent = w.ucol[i];
      u = ent_vertex(ent);
      if (u > w.root) {
        const LT old = w.lab[u];
        w.lab[u] = (LT)(old | (ent_code(ent) << (2 * p)));
        ex = ((uint32_t)old & low) == 0;
      }
    }
    const unsigned bal = __ballot_sync(kFull, ex);
    if (ex) {
      const int pos = e + cnt + __popc(bal & lt);
      if (pos < w.cap) w.buf[pos] = (uint16_t)u;
      else atomicOr(w.err, kErrStackOverflow);
    }
    cnt += __popc(bal);
  }
  __syncwarp();
  const int ne = e + cnt;
  return ne < w.cap ? ne : w.cap;
}

// Pop the vertex x at position p: clear its relation bits again.
template <typename LT, typename ET>
__device__ __forceinline__ void pop_vertex(const WarpCtx<LT, ET>& w, int x, int p) {
  int rs, re;
  w.row(x, rs, re);
  const int start = (re - rs > 32) ? first_above_p(w.ucol, rs, re, w.root) : rs;
  const LT clear = (LT)~(3u << (2 * p));
  for (int b = start; b < re; b += 32) {
    const int i = b + w.lane;
    if (i < re) {
      const int u = ent_vertex(w.ucol[i]);
      if (u > w.root) w.lab[u] &= clear;
    }
  }
  __syncwarp();
}

// A warp moves a block's shared counters to the graph's by exchange (rare, and
// called from several places: kept out of line).
__device__ __noinline__ void move_hist(int32_t* s_hist, unsigned long long* ghist, int C, int lane) {
  for (int i = lane; i < C; i += 32) {
    const int x = atomicExch(&s_hist[i], 0);
    if (x) atomicAdd(&ghist[i], (unsigned long long)(long long)x);
  }
}

// hist[i] += the copies' counts of class i (a one-graph k = 6 count; see
// kHistCopies).  Counts are two's-complement 64-bit sums, so the cell method's
// negative corrections fold correctly.
__global__ void __launch_bounds__(256) k_fold_copies(unsigned long long* __restrict__ hist,
                                                     const unsigned long long* __restrict__ copies,
                                                     int ncopies, uint32_t C, uint32_t stride) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < C; i += gridDim.x * blockDim.x) {
    unsigned long long sum = 0;
    for (int c = 0; c < ncopies; ++c) sum += copies[(size_t)c * stride + i];
    if (sum) hist[i] += sum;
  }
}

struct CountArgs {
  const DevGraph* graphs;
  const Item* items;
  GraphPlan* gp;             // per graph: its items and its queue's head
  Hdr* hdr;
  const uint32_t* table;
  const uint16_t* xclass;    // compact k = 6 table: prefix key -> class of the first 4 vertices
  const uint8_t* xmap;       //   and its word relabelling (256 bytes per prefix key)
  void* lab_global;
  void* stack_global;        // per-warp candidate stacks when they live in global memory
  void* kept;                // per-warp kept lists of the cell method, or null
  size_t kept_bytes;
  unsigned long long* hist_copies;  // copies 1 .. copies-1 of a one-graph k = 6 histogram
  int copies;                // 1 = every block adds into the graph's own histogram
  uint32_t copy_stride;      // elements between two copies
  int G, nmax, cap;
  uint32_t classes;
  int graph_bytes, hist_bytes, lab_bytes, buf_bytes, cell_bytes, map_bytes;
  unsigned long long idle_ns;  // a warp waiting for donated work gives up after this
};

// Cells of the last two positions (combinatorial counting): a relation word to
// the k-2 chosen vertices has 2(k-2) bits.  The cells of one list are numbered
// when there are at most kNumbered.
template <int K>
constexpr int kCells = 1 << (2 * (K - 2));
constexpr int kNumbered = 64;
// Kept lists (see keep_list): arcs of one list, and the choices and members that
// a list must have for it to be worth noting.  Launches over 8 and more graphs use
// them (for one graph they lost, 756 : 837 us; 2 to 7 are untried, but for 4 at k = 6,
// 4.6 : 4.5 ms) when the degrees give long lists and an item holds enough sets to
// share one.  Measured on a GB300, count phase without and with, ms:
//  * by degree, 257 graphs, k = 5: 142 21.0 : 16.3, 106 10.7 : 9.3, 70 8.4 : 7.9, 61
//    4.3 : 4.3, 57 3.3 : 3.6; 65 graphs, k = 6: 53 72.6 : 69.1, 45 28.5 : 27.7, 42
//    10.9 : 11.1;
//  * by estimated sets per item, k = 5: the workload graph (n = 1,500) at 6.7 (8 graphs)
//    3.86 : 4.00, 7.6 4.30 : 4.29, 8.4 4.77 : 4.56, 13 7.4 : 5.8, 217 (257 graphs) 116 :
//    85; n = 700 at 7 3.79 : 3.85, 10 4.97 : 4.38; n = 400 at 7 2.70 : 2.86, 14 5.2 : 4.8; a
//    hub of degree 400 in a sparse background at 3 1.85 : 1.95, 12 6.4 : 5.3; hubs of 64 to
//    200 and small graphs, at 0.4 to 4, lost 5 to 8%;
//  * k = 6: the workload graph (n = 800) at 26 (8 graphs) 8.9 : 8.5, 210 (65) 71.3 : 67.9;
//    n = 500 at 15 5.18 : 5.02; a hub of degree 150 at 16 5.3 : 5.1; hubs of 44 and 80, at 1 to
//    12, lost 6 to 10%; n = 300, degree 46, at 17 to 109 0.984 to 0.993.  Dense graphs,
//    whose lists have more arcs than are kept, lose 2%.
// Server rounds are indifferent (1,420 : 1,415 requests/s).  Kernels of their own: the
// tests for kept lists in the common one cost the other lists 8 to 13%.
constexpr int kKeptArcs = 1024;
constexpr int kKeepGraphs = 8;
constexpr int kKeepDegree5 = 64, kKeepDegree6 = 44;
constexpr double kKeepSets5 = 8.0, kKeepSets6 = 16.0;  // per item
constexpr int kKeepChoices = 8, kKeepLength = 32;

// Persistent enumerator.  A thread block works on one graph at a time: its
// warps take that graph's items from the graph's queue.  A warp that finds the
// queue empty waits for work donated by the block's other warps: a busy warp
// that sees an idle one hands over half of its remaining first- or
// second-level choices as a new item.  When every warp is idle and nothing is
// left to take, the block flushes its shared histogram, picks the next graph
// that still has items and (GC) copies that graph's CSR into shared memory.
// SG: the candidate stacks live in per-warp slices of global memory (graphs
// with hubs so large that shared-memory stacks would leave few warps).
// KEPT: (k-2)-sets below one list share what is kept of it (keep_list).
template <int K, bool GC, bool LS, bool COMB, bool SG = false, bool KEPT = false>
__global__ void __launch_bounds__(kMaxWarpsPerBlock * 32, 1) k_count(CountArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_cur_g;
  __shared__ int s_scan[33];
  __shared__ int s_idle, s_ndon, s_lock;  // work donation (see above)
  __shared__ uint32_t s_don[kDonSlots * 4];  // donated items, 4 words each
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int nwarps = blockDim.x >> 5;
  const unsigned lanes_below = (1u << lane) - 1u;
  int since = 0;  // this warp's enumeration adds since its last flush
  int kept_n = 0, kept_at = 0;  // cell method: arcs kept for the current parent list (keep_list)
  bool bad_id = false;  // a table read gave an id out of range (k = 6, cell method)
  int dead = 0;         // cell method: words [0, dead) are marked LM
  unsigned char* sp = smem;
  int32_t* s_urow = (int32_t*)sp;
  // the cell method's copy of the graph has 16-bit entries
  using ET = typename std::conditional<COMB && GC, uint16_t, uint32_t>::type;
  ET* s_ucol = (ET*)(sp + (GC ? ((a.nmax + 1) * 4 + 15) / 16 * 16 : 0));
  sp += a.graph_bytes;
  int32_t* s_hist = (int32_t*)sp;
  sp += a.hist_bytes;
  const int sbuf = SG ? 0 : a.buf_bytes;  // stack bytes in this warp's shared slice
  unsigned char* mine =
      sp + (size_t)wid * ((LS ? a.lab_bytes : 0) + sbuf + (COMB ? a.cell_bytes : 0) +
                          kLevelBytes + a.map_bytes);
  int* lvs = (int*)(mine + (LS ? a.lab_bytes : 0) + sbuf + (COMB ? a.cell_bytes : 0));
  // compact k = 6 table: the current 4-vertex prefix's word relabelling
  uint8_t* xmw = (uint8_t*)lvs + kLevelBytes;
  const bool cpt = K == 6 && a.xclass != nullptr;
  const bool wide_tail = K <= 5 || (int)gridDim.x <= kWideTailBlocksPerGraph * a.G * a.copies;
  using LT = LabT<K, COMB>;
  // each warp's relation words start on a 16-byte boundary (lab_bytes is a
  // multiple of 16), so 32-bit atomics on them are aligned
  LT* lab = LS ? (LT*)mine
               : (LT*)((char*)a.lab_global + ((size_t)blockIdx.x * nwarps + wid) * a.lab_bytes);
  uint16_t* buf =
      SG ? (uint16_t*)((char*)a.stack_global + ((size_t)blockIdx.x * nwarps + wid) * a.buf_bytes)
         : (uint16_t*)(mine + (LS ? a.lab_bytes : 0));
  // cell method: counts per cell (choices in the low, tail in the high 16
  // bits), counts per numbered cell, exclusive neighbours per (numbered cell,
  // code), the arc queue, the length of the cell list and the list
  uint32_t* ct = (uint32_t*)(mine + (LS ? a.lab_bytes : 0) + sbuf);
  uint32_t* sc = ct + kCells<K>;
  uint32_t* xs = sc + kNumbered;
  uint32_t* qb = xs + 3 * kNumbered;
  int* ncell = (int*)(qb + 64);
  uint16_t* cl = (uint16_t*)(ncell + 4);
  uint32_t* kept_ex = (uint32_t*)((char*)a.kept + ((size_t)blockIdx.x * nwarps + wid) *
                                                       a.kept_bytes);
  uint32_t* kept_arcs = kept_ex + a.cap;
  const uint32_t C = a.classes;

  if (LS)
    for (int i = lane; i < a.nmax; i += 32) lab[i] = 0;
  if (COMB) {
    for (int i = lane; i < kCells<K>; i += 32) ct[i] = 0;
    for (int i = lane; i < 3 * kNumbered; i += 32) xs[i] = 0;
    if (lane == 0) *ncell = 0;
  }
  if (K <= 5)
    for (int i = tid; i <= (int)C; i += blockDim.x) s_hist[i] = 0;  // C: catch slot
  if (tid == 0) {
    s_cur_g = (int)(((int64_t)blockIdx.x * a.G) / gridDim.x);
    s_idle = 0;
    s_ndon = 0;
    s_lock = 0;
  }
  __syncthreads();

  // Block-local lock of the donation slots (lane 0 of a warp only).
  auto block_lock = [&]() -> bool {
    for (int i = 0; i < kLockTries; ++i) {
      if (atomicCAS(&s_lock, 0, 1) == 0) {
        __threadfence_block();
        return true;
      }
      __nanosleep(32);
    }
    atomicOr(&a.hdr->err, kErrWaitLimit);
    return false;
  };
  auto block_unlock = [&]() {
    __threadfence_block();
    atomicExch(&s_lock, 0);
  };
  volatile int* v_idle = &s_idle;
  volatile int* v_ndon = &s_ndon;
  volatile uint32_t* v_don = s_don;

  WarpCtx<LT, ET> w;
  w.lab = lab;
  w.buf = buf;
  w.cap = a.cap;
  w.lane = lane;
  w.err = &a.hdr->err;

  int g = s_cur_g;
  while (g >= 0) {
    const DevGraph* Gp = a.graphs + g;
    if (GC) {
      const int n = Gp->n, nu = Gp->nu;
      const int32_t* grow = Gp->urow;
      const uint32_t* gcol = Gp->ucol;
      if (COMB) {
        // rows start at multiples of kSeg entries, padded with zeros; an entry
        // per thread, so that the loads of a whole copy are in flight together
        const int32_t* gsrc = Gp->usrc;
        uint4* words = (uint4*)s_ucol;
        const int nwords = (int)((unsigned char*)s_hist - (unsigned char*)s_ucol) / 16;
        for (int i = tid; i < nwords; i += blockDim.x) words[i] = make_uint4(0, 0, 0, 0);
        for (int i = tid; i <= n; i += blockDim.x)
          s_urow[i] = i < n ? (grow[i + 1] - grow[i] + kSeg - 1) / kSeg : 0;
        __syncthreads();
        block_exclusive_scan(s_urow, n + 1, s_scan);
        for (int i = tid; i < nu; i += blockDim.x) {
          const int x = gsrc[i];
          const uint32_t ent = gcol[i];
          s_ucol[s_urow[x] * kSeg + (i - grow[x])] =
              (ET)(ent_vertex(ent) | (ent_code(ent) << 14));
        }
        __syncthreads();
        for (int i = tid; i < n; i += blockDim.x)
          s_urow[i] = (int32_t)(((uint32_t)s_urow[i] << 16) | (uint32_t)(grow[i + 1] - grow[i]));
      } else {
        for (int i = tid; i <= n; i += blockDim.x) s_urow[i] = grow[i];
        for (int i = tid; i < nu; i += blockDim.x) s_ucol[i] = (ET)gcol[i];
      }
      w.urow = s_urow;
      w.ucol = s_ucol;
    } else {
      w.urow = Gp->urow;
      w.ucol = (const ET*)Gp->ucol;
    }
    __syncthreads();
    unsigned long long* ghist = Gp->hist;
    if (K == 6 && a.copies > 1) {  // one graph: this block's copy of its histogram
      const int cp = (int)(blockIdx.x % (unsigned)a.copies);
      if (cp) ghist = a.hist_copies + (size_t)(cp - 1) * a.copy_stride;
    }
    const int32_t* ufwd = Gp->ufwd;
    const uint32_t nitems = a.gp[g].count;
    const Item* my_items = a.items + a.gp[g].base;

    // Adds of the cell method, which may be negative (corrections).  For k <= 5
    // the shared 32-bit counters take deltas below 2^20 under the add budget
    // below; larger ones and k = 6 go to the graph's 64-bit counters (two's
    // complement).
    auto cadd = [&](uint32_t id, long long delta, bool direct) {
      const bool ok = id < C;
      bad_id |= !ok;
      if (K <= 5 && !direct && delta < (1ll << 20) && delta > -(1ll << 20))
        red_add_shared(&s_hist[min(id, C)], (int)delta);
      else
        red_add_global(&ghist[ok ? id : 0u], ok ? (unsigned long long)delta : 0ull);
    };

    // Positive adds of the enumeration path.  For k <= 5 the shared 32-bit
    // counters take them without returning the old value; each warp counts
    // what it added since it last flushed and, past kLeafBudget, moves the
    // whole shared histogram to the graph's 64-bit counters by exchange
    // (adds of other warps stay in the counters).  A counter then never holds
    // more than warps x (kLeafBudget + one choice's adds) < 2^31.
    // (An id out of range, which a valid table never holds, lands in the
    // shared catch slot C, checked at the flush; for k = 6 it adds nothing and
    // is recorded in `bad_id`, reported when the thread exits.  Neither form
    // branches on the table read, so the reads of several slots overlap.)
    auto ladd = [&](uint32_t id, int d) {
      if (K <= 5) {
        red_add_shared(&s_hist[min(id, C)], d);
      } else {
        const bool ok = id < C;
        bad_id |= !ok;
        red_add_global(&ghist[ok ? id : 0u], ok ? (unsigned long long)d : 0ull);
      }
    };
    auto leaf_budget = [&](int adds) {
      if (K <= 5) {
        if (since >= (COMB ? kCellBudget : kLeafBudget)) {
          move_hist(s_hist, ghist, (int)C, lane);
          since = 0;
        }
        since += adds;
      }
    };

    // Compact table: load the relabelling of words to the canonical order of the
    // first four vertices (positions 1..3 sit in key bits 18..29); returns their
    // class, in place.
    auto load_prefix = [&](uint32_t key) -> uint32_t {
      const uint32_t xk = key >> 18;
      ((uint2*)xmw)[lane] = __ldg((const uint2*)(a.xmap + (size_t)xk * 256) + lane);
      uint32_t c4 = __ldg(&a.xclass[xk]);
      if (c4 >= 199u) {  // a disconnected prefix, which the enumeration never forms
        atomicOr(w.err, kErrStackOverflow);
        c4 = 0;
      }
      __syncwarp();
      return c4 << 18;
    };

    // The rows of up to 32 list members buf[cb ..] (c1 the list's end) in segments
    // of kSeg entries, one per lane.  A lane counts its segment's exclusive
    // neighbours (word 0) per arc code in bytes 1..3 of one register and notes the
    // entries inside E (words above LM).  Vertices up to the root carry word LM,
    // neither exclusive nor in E, and so does the padding (vertex 0).  `meta`
    // describes a member; `seg` gets a segment's member (its lane), meta, first
    // entry, counts and hits.  Returns the number of segments.
    auto walk_rows = [&](int cb, int c1, auto&& meta_of, auto&& seg) {
      constexpr uint32_t LM = (1u << (2 * (K - 2))) - 1u;
      const int i = cb + lane;
      const bool vy = i < c1;
      int rs = 0, re = 0, ns = 0;
      uint32_t meta = 0;
      if (vy) {
        const int y = buf[i];
        w.row(y, rs, re);
        if (re - rs > 4 * kSeg)
          rs += max(min(first_above_p(w.ucol, rs, re, w.root), re - 1) - rs, 0) / kSeg * kSeg;
        ns = max((re - rs + kSeg - 1) / kSeg, 1);
        meta = meta_of(y);
      }
      const int pre = warp_incl_scan(ns) - ns;
      const int total = __shfl_sync(kFull, pre + ns, 31);
      leaf_budget(total * kSeg * 3);
      for (int q0 = 0; q0 < total; q0 += 32) {
        // the lane's member: the rows that start before the batch, and up to the
        // lane within it (every row has a segment)
        const unsigned at = (unsigned)(pre - q0);
        const unsigned starts = __reduce_or_sync(kFull, vy && at < 32u ? 1u << at : 0u);
        const int before = __popc(__ballot_sync(kFull, vy && pre < q0));
        const int own = before + __popc(starts & (lanes_below | (1u << lane))) - 1;
        const int sg = q0 + lane - __shfl_sync(kFull, pre, own);
        const int first = __shfl_sync(kFull, rs, own) + sg * kSeg;
        const int last = __shfl_sync(kFull, re, own);
        const uint32_t my = __shfl_sync(kFull, meta, own);
        uint32_t cnt = 0, hits = 0;
        if (q0 + lane < total) {
          __align__(16) ET ent[kSeg];
          if (sizeof(ET) == 2) {
            *(uint4*)ent = *(const uint4*)(w.ucol + first);
          } else {
#pragma unroll
            for (int j = 0; j < kSeg; ++j) ent[j] = first + j < last ? w.ucol[first + j] : (ET)0;
          }
          uint32_t l[kSeg];
#pragma unroll
          for (int j = 0; j < kSeg; ++j) l[j] = lab[ent_vertex(ent[j])];
#pragma unroll
          for (int j = 0; j < kSeg; ++j) {
            if (l[j] == 0) cnt += 1u << (8 * ent_code(ent[j]));
            if (l[j] > LM) hits |= 1u << j;
          }
        }
        seg(own, my, first, cnt, hits);
      }
    };

    // The arcs inside a list and its members' exclusive neighbours, kept for the
    // (k-2)-sets that add one member x to the k-3 vertices chosen so far: all of
    // them share the list's tail, and only the vertices that x brings have rows
    // yet to be read.  Noted per member: its exclusive neighbours per arc code
    // (10 bits each), in stack order; per arc: its two ends and its code.  Gives
    // up (and the sets read all rows) on rows or arcs past what fits.
    auto keep_list = [&](int c, int e) -> bool {
      constexpr uint32_t LM = (1u << (2 * (K - 2))) - 1u;
      constexpr uint32_t INC = LM + 1u, INT = 2u * INC;
      for (int b = c + lane; b < e; b += 32) lab[buf[b]] |= (LT)INT;
      __syncwarp();
      int n = 0;
      bool ok = true;
      for (int cb = c; cb < e && ok; cb += 32) {
        // these 32: INC; later ones INT, earlier ones no longer flagged
        const int i = cb + lane;
        bool wide = false;
        if (i < e) {
          const int y = buf[i];
          int rs, re;
          w.row(y, rs, re);
          wide = re - rs > 1023;
          lab[y] ^= (LT)(INC | INT);
        }
        sc[lane] = 0;
        ok = !__any_sync(kFull, wide);
        __syncwarp();
        if (ok)
          walk_rows(cb, e, [&](int y) { return (uint32_t)y; },
                    [&](int own, uint32_t y, int first, uint32_t cnt, uint32_t hits) {
                      if (cnt)
                        atomicAdd(&sc[own], ((cnt >> 8) & 0xFFu) | ((cnt >> 6) & 0x3FC00u) |
                                                ((cnt >> 4) & 0xFF00000u));
                      while (__any_sync(kFull, hits != 0)) {
                        bool put = false;
                        uint32_t q = 0;
                        if (hits) {
                          const ET en = w.ucol[first + __ffs(hits) - 1];
                          hits &= hits - 1;
                          const int u = ent_vertex(en);
                          put = ((uint32_t)lab[u] & INT) || u > (int)y;
                          q = y | ((uint32_t)u << 14) | (ent_code(en) << 28);
                        }
                        const unsigned bal = __ballot_sync(kFull, put);
                        const int at = n + __popc(bal & lanes_below);
                        if (put && at < kKeptArcs) kept_arcs[at] = q;
                        n += __popc(bal);
                      }
                    });
        ok = ok && n <= kKeptArcs;
        __syncwarp();
        if (i < e) {
          kept_ex[i] = sc[lane];
          lab[buf[i]] &= (LT)LM;
        }
        __syncwarp();
      }
      if (!ok)
        for (int b = c + lane; b < e; b += 32) lab[buf[b]] &= (LT)LM;
      __syncwarp();
      kept_n = n;
      kept_at = 0;
      return ok;
    };

    // Exclusive neighbours of lanes' list members, per code, to the counters of
    // their cells' numbers.  Both forms add atomically, like the kept lists'
    // corrections: votes and shuffles order no memory between the lanes.
    auto add_exclusive = [&](uint32_t num, uint32_t n1, uint32_t n2, uint32_t n3) {
      const bool some = (n1 | n2 | n3) != 0;
      const uint32_t num0 = __shfl_sync(kFull, num, 0);
      if (__all_sync(kFull, !some || num == num0)) {
        const uint32_t s12 = __reduce_add_sync(kFull, n1 | (n2 << 16));
        const uint32_t s3 = __reduce_add_sync(kFull, n3);
        if (lane == 0) {
          red_add_shared((int*)&xs[3 * num0], (int)(s12 & 0xFFFFu));
          red_add_shared((int*)&xs[3 * num0 + 1], (int)(s12 >> 16));
          red_add_shared((int*)&xs[3 * num0 + 2], (int)s3);
        }
      } else if (some) {
        if (n1) atomicAdd(&xs[3 * num], n1);
        if (n2) atomicAdd(&xs[3 * num + 1], n2);
        if (n3) atomicAdd(&xs[3 * num + 2], n3);
      }
    };

    // Combinatorial counting of the last two positions (Algorithm 1 of Sec. 3
    // on the enumerator's (k-2)-set X with candidate list E = buf[c, e) whose
    // choices are buf[c, ce)): the k-sets below X are the pairs {y, z}, y a
    // choice and z after it in E, plus {y, u} with u an exclusive neighbour of
    // y.  Without an arc between y and z the class depends only on the cells
    // (relation words to X) of y and z, so those pairs are counted per cell
    // pair; arcs inside E are corrected one by one; {y, u} depends only on y's
    // cell and the arc code between y and u, so exclusive neighbours are
    // counted per (cell, code).
    // Bound by instruction issue (75% of cycles on the k = 5 workload: 68
    // candidates and 6 cells per X).  A lane per row segment
    // needs one search and no ballots for 8 entries where a lane per entry
    // needed a 5-step search and a match for each 32; the k = 5 batch (257 graphs)
    // went from 260 to 187 ms, the k = 6 one (65 graphs) from 112 to 71 ms.
    // `ke` > 0 (KEPT): the arcs inside buf[c, ke) and its exclusive neighbours are
    // kept (see keep_list), and only the rows of buf[ke, ce) are read.
    auto pair_level = [&](int c, int ce, int e, uint32_t P, int ke) {
      constexpr int NB = 2 * (K - 2);
      constexpr uint32_t LM = (1u << NB) - 1u;
      constexpr uint32_t INC = 1u << NB, INT = 2u << NB;
      constexpr int OFF2 = key_off(K, K - 2), OFF1 = key_off(K, K - 1);
      if (c >= ce) return;
      if (cpt) P = load_prefix(P);
      auto word = [&](uint32_t lam) -> uint32_t { return cpt ? (uint32_t)xmw[lam] : lam; };
      // 1. cells of the choices and of the tail; flag E's members
      for (int b = c; b < e; b += 32) {
        const int i = b + lane;
        const bool v = i < e;
        uint32_t lam = 0, tag = 0xFFFFFFFFu;
        bool inc = false;
        if (v) {
          const int u = buf[i];
          lam = (uint32_t)lab[u] & LM;
          inc = i < ce;
          lab[u] = (LT)(lam | (inc && (!KEPT || i >= ke) ? INC : INT));  // INC: its row is read
          tag = lam | (inc ? 0x10000u : 0u);
        }
        const unsigned peers = __match_any_sync(kFull, tag);
        if (v && !(peers & lanes_below)) {
          const uint32_t old = atomicAdd(&ct[lam], (uint32_t)__popc(peers) << (inc ? 0 : 16));
          if (old == 0) cl[atomicAdd(ncell, 1)] = (uint16_t)lam;
        }
      }
      __syncwarp();
      const int r = *ncell;
      // the cells are numbered (ct becomes cell -> number, sc holds the counts)
      // unless a huge X has more than fit (never at k <= 5)
      const bool numbered = kCells<K> <= kNumbered || r <= kNumbered;
      if (numbered) {
        for (int ia = lane; ia < r; ia += 32) {
          const uint32_t lam = cl[ia];
          sc[ia] = ct[lam];
          ct[lam] = (uint32_t)ia;
        }
        __syncwarp();
      }
      if (KEPT && ke && !numbered) {  // the kept counts are added up per number
        for (int i = c + lane; i < min(ke, ce); i += 32)
          lab[buf[i]] = (LT)(((uint32_t)lab[buf[i]] & LM) | INC);
        ke = 0;
        __syncwarp();
      }
      // 2. pairs without an arc, per cell pair
      const long long npairs = (long long)(ce - c) * (e - c);
      const bool direct = npairs > kCellBudget;  // deltas past the shared counters' budget
      leaf_budget(direct ? 0 : (int)npairs);
      auto cell_pair = [&](uint32_t la, uint32_t pa, uint32_t lb, uint32_t pb, bool same) {
        const long long ca = pa & 0xFFFFu, ta = pa >> 16, cb = pb & 0xFFFFu, tb = pb >> 16;
        const long long cnt = same ? ca * (ca - 1) / 2 + ca * ta : ca * cb + ca * tb + cb * ta;
        if (cnt)
          cadd(__ldg(&a.table[P | (word(la) << OFF2) | (word(lb) << OFF1)]), cnt, direct);
      };
      if (numbered) {
        // the unordered pairs (ia, ia + d mod r), d = 0 .. r/2, over the lanes
        const uint32_t inv = (1u << 20) / (uint32_t)r + 1u;  // exact below 2^20 / r
        const int np = r * (r / 2 + 1);
        for (int idx = lane; idx < np; idx += 32) {
          const int d = (int)(((uint32_t)idx * inv) >> 20);
          const int ia = idx - d * r;
          int ib = ia + d;
          if (ib >= r) ib -= r;
          if (2 * d != r || ia < ib) cell_pair(cl[ia], sc[ia], cl[ib], sc[ib], d == 0);
        }
      } else {
        for (int ia = 0; ia < r; ++ia)
          for (int ib = ia + lane; ib < r; ib += 32)
            cell_pair(cl[ia], ct[cl[ia]], cl[ib], ct[cl[ib]], ia == ib);
      }
      // An arc inside E (cells of the two ends, arc code) moves one pair from its
      // cell pair's class to its own; 32 are added at once.
      auto add_arcs = [&](bool v, uint32_t q) {
        const unsigned peers = __match_any_sync(kFull, v ? q : 0xFFFFFFFFu);
        if (v && !(peers & lanes_below)) {
          const uint32_t base = P | (word(q & LM) << OFF2);
          const uint32_t lz = word((q >> 8) & LM);
          const uint32_t from = __ldg(&a.table[base | (lz << OFF1)]);
          const uint32_t to = __ldg(&a.table[base | ((lz | ((q >> 16) << NB)) << OFF1)]);
          const int cnt = __popc(peers);
          cadd(to, cnt, false);
          cadd(from, -cnt, false);
        }
      };
      int qn = 0;  // arcs waiting in qb
      auto flush_arcs = [&](int n) {
        __syncwarp();
        add_arcs(lane < n, lane < n ? qb[lane] : 0u);
        __syncwarp();
      };
      // 3. kept arcs whose ends are both still in the list; members leave it from
      //    the front, and so do their arcs
      if (KEPT && ke)
        for (int b = kept_at; b < kept_n; b += 32) {
          uint32_t q = 0;
          bool v = false;
          if (b + lane < kept_n) {
            const uint32_t k = kept_arcs[b + lane];
            const uint32_t ly = lab[k & 0x3FFFu], lz = lab[(k >> 14) & 0x3FFFu];
            v = ly > LM && lz > LM;
            q = (ly & LM) | ((lz & LM) << 8) | ((k >> 28) << 16);
          }
          if (!__any_sync(kFull, v)) {
            if (b == kept_at && b + 32 <= kept_n) kept_at += 32;
            continue;
          }
          leaf_budget(64);
          add_arcs(v, q);
        }
      // 4. the other choices' rows: exclusive neighbours are counted per (number
      //    of the choice's cell, code), arcs inside E wait in a queue until 32 are
      //    there
      for (int cb = KEPT ? max(c, ke) : c; cb < ce; cb += 32)
        walk_rows(cb, ce,
                  [&](int y) {
                    const uint32_t lam = (uint32_t)lab[y] & LM;
                    return (uint32_t)y | (lam << 16) | ((numbered ? ct[lam] : 0u) << 24);
                  },
                  [&](int own, uint32_t my, int first, uint32_t cnt, uint32_t hits) {
          if (numbered) {
            add_exclusive(my >> 24, (cnt >> 8) & 0xFFu, (cnt >> 16) & 0xFFu, cnt >> 24);
          } else {
            for (uint32_t j = 1; j <= 3; ++j) {
              const uint32_t n = (cnt >> (8 * j)) & 0xFFu;
              if (n)
                cadd(__ldg(&a.table[P | (word((my >> 16) & LM) << OFF2) | ((j << NB) << OFF1)]), n,
                     false);
            }
          }
          while (__any_sync(kFull, hits != 0)) {
            bool put = false;
            uint32_t q = 0;
            if (hits) {
              const ET en = w.ucol[first + __ffs(hits) - 1];
              hits &= hits - 1;
              const int u = ent_vertex(en);
              const uint32_t lu = lab[u], code = ent_code(en);
              // a pair of two choices whose rows are read once, from its smaller
              // vertex
              put = (lu & INT) || u > (int)(my & 0xFFFFu);
              q = ((my >> 16) & LM) | ((lu & LM) << 8) | (code << 16);
              // a member whose row was read before x brought this choice counts
              // the choice among its exclusive neighbours (the arc seen from it)
              if (KEPT && ke && (lu & INT))
                atomicSub(&xs[3 * ct[lu & LM] + (code == 3u ? 3u : 3u - code) - 1u], 1u);
            }
            const unsigned bal = __ballot_sync(kFull, put);
            if (put) qb[qn + __popc(bal & lanes_below)] = q;
            qn += __popc(bal);
            if (qn >= 32) {
              flush_arcs(32);
              qn -= 32;
              const uint32_t t = lane < qn ? qb[32 + lane] : 0u;
              __syncwarp();
              if (lane < qn) qb[lane] = t;
            }
          }
        });
      if (qn) flush_arcs(qn);
      // 5. the kept members' exclusive neighbours
      if (KEPT && ke) {
        uint32_t sum = 0;
        for (int b = c; b < ke; b += 32) {
          const int i = b + lane;
          uint32_t num = 0, ex = 0;
          if (i < ke) {
            num = ct[(uint32_t)lab[buf[i]] & LM];
            ex = kept_ex[i];
          }
          add_exclusive(num, ex & 0x3FFu, (ex >> 10) & 0x3FFu, ex >> 20);
          sum += (ex & 0x3FFu) + ((ex >> 10) & 0x3FFu) + (ex >> 20);
        }
        leaf_budget((int)__reduce_add_sync(kFull, sum));
      }
      __syncwarp();
      if (numbered)
        for (int i = lane; i < 3 * r; i += 32) {
          const uint32_t n = xs[i];
          if (n) {
            const int ia = i / 3;
            const uint32_t code = (uint32_t)(i - 3 * ia + 1);
            cadd(__ldg(&a.table[P | (word(cl[ia]) << OFF2) | ((code << NB) << OFF1)]), n, false);
            xs[i] = 0;
          }
        }
      // 6. clear flags and cells
      for (int b = c; b < e; b += 32) {
        const int i = b + lane;
        if (i < e) lab[buf[i]] &= (LT)LM;
      }
      for (int ia = lane; ia < r; ia += 32) ct[cl[ia]] = 0;
      __syncwarp();
      if (lane == 0) *ncell = 0;
      __syncwarp();
    };

    // Lane 0: wait, idle, for a donated item (1) or for the whole block to be
    // idle with nothing left to take (0).
    auto take_donation = [&](uint4& raw) -> int {
      if (!block_lock()) return 0;
      *v_idle = *v_idle + 1;
      block_unlock();
      const unsigned long long t0 = global_ns();
      for (int poll = 0; poll < kIdlePolls; ++poll) {
        if (*v_ndon > 0 || *v_idle == nwarps) {
          if (!block_lock()) return 0;
          int r = -1;
          const int nd = *v_ndon;
          if (nd > 0) {
            raw.x = v_don[4 * (nd - 1)];
            raw.y = v_don[4 * (nd - 1) + 1];
            raw.z = v_don[4 * (nd - 1) + 2];
            raw.w = v_don[4 * (nd - 1) + 3];
            *v_ndon = nd - 1;
            *v_idle = *v_idle - 1;
            r = 1;
          } else if (*v_idle == nwarps) {
            r = 0;
          }
          block_unlock();
          if (r >= 0) return r;
        }
        if (global_ns() - t0 > a.idle_ns) break;
        __nanosleep(256);
      }
      atomicOr(&a.hdr->err, kErrWaitLimit);
      return 0;
    };
    // The warp's next item: the graph's queue, then donated items.
    auto next_item = [&](Item& out) -> bool {
      uint32_t idx = 0;
      if (lane == 0) idx = atomicAdd(&a.gp[g].qhead, 1u);
      idx = __shfl_sync(kFull, idx, 0);
      if (idx < nitems) {
        out = my_items[idx];
        return true;
      }
      uint4 raw = make_uint4(0, 0, 0, 0);
      int got = 0;
      if (lane == 0) got = take_donation(raw);
      got = __shfl_sync(kFull, got, 0);
      if (!got) return false;
      raw.x = __shfl_sync(kFull, raw.x, 0);
      raw.y = __shfl_sync(kFull, raw.y, 0);
      raw.z = __shfl_sync(kFull, raw.z, 0);
      raw.w = __shfl_sync(kFull, raw.w, 0);
      memcpy(&out, &raw, sizeof(Item));
      return true;
    };

    while (true) {
      Item it;
      if (!next_item(it)) break;
      const int v = (int)it.root;
      w.root = v;
      int re, f;
      w.row(v, f, re);
      f += __ldg(&ufwd[v]);
      const int dplus = re - f;
      if (COMB) {  // words of the vertices up to the root: LM (see pair_level)
        constexpr LT LM = (LT)((1u << (2 * (K - 2))) - 1u);
        for (int i = dead + lane; i <= v; i += 32) lab[i] = LM;
        for (int i = v + 1 + lane; i < dead; i += 32) lab[i] = 0;
        dead = v + 1;
        __syncwarp();
      }
      const int j1a = it.j1a, j1b = it.j1b;
      // push the root at position 0: every forward neighbour gets its relation
      // bits; candidates j1a.. go to the stack.
      for (int b = f; b < re; b += 32) {
        const int i = b + lane;
        if (i < re) {
          const ET ent = w.ucol[i];
          const int u = ent_vertex(ent);
          lab[u] |= (LT)ent_code(ent);
          const int q = i - f - j1a;
          if (q >= 0) {
            if (q < w.cap) buf[q] = (uint16_t)u;
            else atomicOr(w.err, kErrStackOverflow);
          }
        }
      }
      __syncwarp();
      // the current level's state lives in (warp-uniform) registers; the
      // levels above it wait in the per-warp stack `lvs`
      int cur_e = min(dplus - j1a, w.cap);
      int cur_c = 0, cur_ce = min(j1b - j1a, cur_e);
      uint32_t cur_key = 0;
      const bool has2 = it.b2 != 0xFFFF, has3 = it.b3 != 0xFFFF;
      // The enumerator's slot codes (bits of positions k-2 and up) are not
      // cleared by row scans: the tail pass writes each candidate back
      // without them, and a candidate list is cleaned once when its level
      // (k-2 positions chosen) is entered; every other reader masks them.
      bool fresh = true;
      // cell method: the end of the list at level k-3 while its arcs are kept;
      // `decide`: it has just been entered
      int kept = 0;
      bool decide = false;
      uint32_t xpre = 0;  // compact table: class of the current 4-vertex prefix, in place
      int L = 1;
      auto pop_level = [&]() {
        L -= 1;
        const int* sv = lvs + 5 * L;
        cur_c = sv[0];
        cur_ce = sv[1];
        cur_e = sv[2];
        cur_key = (uint32_t)sv[3];
        pop_vertex(w, sv[4], L);
      };
      while (true) {
        const int c = cur_c, ce = cur_ce, e = cur_e;
        const uint32_t key = cur_key;
        if (COMB && L == K - 2) {
          pair_level(c, ce, e, key, kept);
          if (L == 1) break;
          pop_level();
          continue;
        }
        if (!COMB && L == K - 2) {
          // Choosing the (k-1)-th vertex finishes its k-sets in place, for up
          // to GS consecutive choices at once (as many as the relation word
          // has free 2-bit slots, at most 8: 3, 2, 5, 8 for k = 3..6): choice
          // g marks its row into slot g above the first k-2 positions' bits,
          // so one pass over the shared candidate tail classifies every
          // choice's leaves.
          if (c >= ce) {
            if (L == 1) break;
            pop_level();
            continue;
          }
          constexpr int NB = 2 * (K - 2);
          constexpr uint32_t LM = (1u << NB) - 1u;
          constexpr int OFF1 = key_off(K, K - 1);
          constexpr int OFF2 = key_off(K, K - 2);
          if (fresh) {
            // a new candidate list: clear slot codes left by earlier rows
            for (int b = c; b < e; b += 32) {
              const int i = b + lane;
              if (i < e) {
                const int u = buf[i];
                lab[u] = (LT)((uint32_t)lab[u] & LM);
              }
            }
            __syncwarp();
            fresh = false;
            if (cpt) xpre = load_prefix(key);
          }
          // slots left in the relation word above the first k-2 positions
          constexpr int GS = (8 * (int)sizeof(LT) - NB) / 2 < 8 ? (8 * (int)sizeof(LT) - NB) / 2 : 8;
          static_assert(COMB || GS >= 2, "at least two slots per relation word");
          const int ng = min(GS, ce - c);
          cur_c = c + ng;
          // lane g < ng: choice g's key prefix and its row above the root
          uint32_t Pg = 0;
          int rs_g = 0, len_g = 0;
          if (lane < ng) {
            const int y = buf[c + lane];
            Pg = cpt ? xpre | ((uint32_t)xmw[(uint32_t)lab[y] & LM] << OFF2)
                     : key | ((uint32_t)(lab[y] & LM) << OFF2);
            int r0, r1;
            w.row(y, r0, r1);
            rs_g = (r1 - r0 > 32) ? first_above_p(w.ucol, r0, r1, w.root) : r0;
            len_g = r1 - rs_g;
          }
          // qs[g] = where choice g's row starts in the concatenation
          int qs[GS + 1];
          qs[0] = 0;
#pragma unroll
          for (int gg = 0; gg < GS; ++gg) qs[gg + 1] = qs[gg] + __shfl_sync(kFull, len_g, gg);
          const int tot = qs[GS];
          leaf_budget(ng * (e - c - 1) + tot);
          // (a) the group's rows, concatenated over the lanes: choice g sets
          //     slot g of its neighbours (a 32-bit atomic OR on the word that
          //     holds the relation word, as two choices may share a
          //     neighbour); an exclusive neighbour u (no relation to the first
          //     k-2 vertices) completes a k-set keyed by the choice's prefix
          //     and the arc code between the choice and u, counted per
          //     (choice, code) group of the pass
          {
            constexpr int PER = 4 / (int)sizeof(LT);  // relation words per 32-bit word
            uint32_t* lab32 = (uint32_t*)lab;
            for (int b = 0; b < tot; b += 32) {
              const int q = b + lane;
              int gg = 0, off = 0;
#pragma unroll
              for (int t = 1; t < GS; ++t)
                if (q >= qs[t]) {
                  gg = t;
                  off = qs[t];
                }
              const int rs = __shfl_sync(kFull, rs_g, gg);
              const uint32_t pg = __shfl_sync(kFull, Pg, gg);
              bool ex = false;
              uint32_t code = 0;
              if (q < tot) {
                const ET ent = w.ucol[rs + (q - off)];
                const int u = ent_vertex(ent);
                code = ent_code(ent);
                if (u > w.root) {
                  const uint32_t old = (uint32_t)lab[u];
                  atomicOr(&lab32[u / PER],
                           (code << (NB + 2 * gg)) << (8 * (int)sizeof(LT) * (u % PER)));
                  ex = (old & LM) == 0;
                }
              }
              const unsigned peers = __match_any_sync(kFull, ex ? (uint32_t)(gg * 4) + code : 0xFFFFFFFFu);  // (choice, code)
              if (ex && !(peers & lanes_below))
                ladd(__ldg(&a.table[pg | ((code << NB) << OFF1)]), __popc(peers));
            }
            __syncwarp();
          }
          // (b) the candidates after the group's first choice; those after
          //     choice g are its leaves, keyed by their word to the first k-2
          //     vertices plus slot g; equal keys of a batch share a table read
          const int lc = e - c - 1;  // candidates after the group's first choice
          if (K == 6 && lc <= 16 && ng > 1) {
            // A short list (common at k = 6, where lists average 20
            // candidates; measured no better at k = 5): P choices per pass,
            // 32 / P lanes each, every lane one (choice, candidate) pair; the
            // match groups equal full keys, so pairs of different choices with
            // the same key share a read.
            const int P = lc <= 4 ? 8 : (lc <= 8 ? 4 : 2);
            const int lw = P == 8 ? 2 : (P == 4 ? 3 : 4);  // log2 of the lanes per choice
            const int h = lane >> lw, idx = lane & ((1 << lw) - 1);
            const bool v0 = idx < lc;
            const int u0 = v0 ? buf[c + 1 + idx] : 0;
            const uint32_t lt = v0 ? (uint32_t)lab[u0] : 0u;
            __syncwarp();  // the other choices' lanes read the word too
            if (v0 && h == 0) lab[u0] = (LT)(lt & LM);
            const uint32_t lb = cpt ? (uint32_t)xmw[lt & LM] : (lt & LM);
            for (int p0 = 0; p0 < ng; p0 += P) {
              const int gg = p0 + h;
              const uint32_t pg = __shfl_sync(kFull, Pg, gg & 31);
              const bool vg = v0 && gg < ng && idx + 1 > gg;
              const uint32_t key = pg | ((lb | ((lt >> (2 * gg)) & (3u << NB))) << OFF1);
              const unsigned peers = __match_any_sync(kFull, vg ? key : 0xFFFFFFFFu);
              if (vg && !(peers & lanes_below)) ladd(__ldg(&a.table[key]), __popc(peers));
            }
            __syncwarp();
            continue;
          }
          uint32_t pgs[GS];
#pragma unroll
          for (int gg = 0; gg < GS; ++gg) pgs[gg] = __shfl_sync(kFull, Pg, gg);
          for (int b = c + 1; b < e; b += 32) {
            const int i0 = b + lane;
            const bool v0 = i0 < e;
            const int u0 = v0 ? buf[i0] : 0;
            const uint32_t lt = v0 ? (uint32_t)lab[u0] : 0u;
            if (v0) lab[u0] = (LT)(lt & LM);
            const int rel = v0 ? i0 - c : 0;  // candidate is after choice g iff rel > g
            const uint32_t lb = cpt ? (uint32_t)xmw[lt & LM] : (lt & LM);
            if (wide_tail) {
              // One match groups the batch's lanes for every choice of the
              // group (k <= 5, and k = 6 launches over many graphs).  A leaf's
              // key for choice g is a function of the candidate's relation word
              // (its bits to the first k-2 vertices and the group's slot
              // codes), and the candidate is a leaf of choices 0 .. vc-1,
              // vc = min(ng, rel); lanes with equal word and vc have equal keys
              // for every choice, and the leader of such a group classifies it
              // for each of its vc choices.
              constexpr int WB = NB + 2 * GS;  // relation-word bits in use (<= 24)
              const uint32_t vc = (uint32_t)min(ng, rel);
              const uint32_t tag = (lt & ((1u << WB) - 1u)) | (vc << WB);
              const unsigned peers = __match_any_sync(kFull, vc ? tag : 0xFFFFFFFFu);
              if (vc && !(peers & lanes_below)) {
                const int cnt = __popc(peers);
                uint32_t id[GS];
#pragma unroll
                for (int gg = 0; gg < GS; ++gg)
                  id[gg] = gg < (int)vc
                               ? __ldg(&a.table[pgs[gg] | ((lb | ((lt >> (2 * gg)) & (3u << NB))) << OFF1)])
                               : 0u;
#pragma unroll
                for (int gg = 0; gg < GS; ++gg)
                  if (gg < (int)vc) ladd(id[gg], cnt);
              }
            } else {
              // k = 6 over few graphs: one match groups the lanes for M = 3
              // choices at once, so a leader adds for at most three.  The tag
              // holds M fields of NB + 2 bits, the leaf's word for a choice it
              // is a leaf of and 0 otherwise (a candidate is adjacent to the
              // first k-2 vertices, so its word is never 0: at most 30 tag
              // bits, so no tag is all ones), and a group's leader classifies
              // it for each choice it is a leaf of.
              constexpr int FB = NB + 2;
              constexpr int M = (31 / FB) < GS ? (31 / FB) : GS;
#pragma unroll
              for (int g0 = 0; g0 < GS; g0 += M) {
                if (g0 < ng) {
                  uint32_t tag = 0, wdv[M];
                  bool vv[M];
                  bool any = false;
#pragma unroll
                  for (int t = 0; t < M; ++t) {
                    const int gg = g0 + t;
                    vv[t] = gg < ng && rel > gg;
                    wdv[t] = lb | ((lt >> (2 * gg)) & (3u << NB));
                    tag |= (vv[t] ? wdv[t] : 0u) << (FB * t);
                    any |= vv[t];
                  }
                  const unsigned peers = __match_any_sync(kFull, any ? tag : 0xFFFFFFFFu);
                  if (any && !(peers & lanes_below)) {
                    const int cnt = __popc(peers);
                    uint32_t id[M];
#pragma unroll
                    for (int t = 0; t < M; ++t)
                      id[t] = vv[t] ? __ldg(&a.table[pgs[(g0 + t) % GS] | (wdv[t] << OFF1)]) : 0u;
#pragma unroll
                    for (int t = 0; t < M; ++t)
                      if (vv[t]) ladd(id[t], cnt);
                  }
                }
              }
            }
          }
          __syncwarp();
          continue;
        }
        if (c < ce) {
          // work donation: with an idle warp in the block, hand the second
          // half of this level's remaining choices over as a new item (a
          // range of this level under the current choices of the levels above).
          // At k = 6 that includes the third level: one second-level choice that
          // reaches a hub can hold more work than a warp's share of a launch.
          int cee = ce;
          if (KEPT && L == K - 3 && decide) {
            decide = false;
            kept = ce - c >= kKeepChoices && e - c >= kKeepLength && keep_list(c, e) ? e : 0;
          }
          if (L <= 3 && L < K - 2 && ce - c >= 2) {
            int hungry = 0;
            if (lane == 0) hungry = *v_idle > 0 && *v_ndon < kDonSlots;
            hungry = __shfl_sync(kFull, hungry, 0);
            if (hungry) {
              const int mid = c + (ce - c + 1) / 2;
              int ok = 0;
              if (lane == 0) {
                Item d;
                d.root = (uint32_t)v;
                d.a2 = d.a3 = 0;
                d.b2 = d.b3 = 0xFFFF;
                if (L == 1) {
                  d.j1a = (uint16_t)(j1a + mid);
                  d.j1b = (uint16_t)(j1a + ce);
                } else {
                  const int c1 = lvs[5] - 1;  // index of the first-level choice
                  d.j1a = (uint16_t)(j1a + c1);
                  d.j1b = (uint16_t)(j1a + c1 + 1);
                  if (L == 2) {
                    d.a2 = (uint16_t)(mid - (c1 + 1));
                    d.b2 = (uint16_t)(ce - (c1 + 1));
                  } else {
                    const int c2 = lvs[10] - 1;  // and of the second-level choice
                    d.a2 = (uint16_t)(c2 - (c1 + 1));
                    d.b2 = (uint16_t)(c2 - c1);
                    d.a3 = (uint16_t)(mid - (c2 + 1));
                    d.b3 = (uint16_t)(ce - (c2 + 1));
                  }
                }
                if (block_lock()) {
                  const int nd = *v_ndon;
                  if (nd < kDonSlots) {
                    uint4 raw;
                    memcpy(&raw, &d, sizeof(Item));
                    v_don[4 * nd] = raw.x;
                    v_don[4 * nd + 1] = raw.y;
                    v_don[4 * nd + 2] = raw.z;
                    v_don[4 * nd + 3] = raw.w;
                    *v_ndon = nd + 1;
                    ok = 1;
                  }
                  block_unlock();
                }
              }
              ok = __shfl_sync(kFull, ok, 0);
              if (ok) cee = mid;
            }
          }
          const int x = buf[c];
          const uint32_t nkey = key | (((uint32_t)lab[x] & ((1u << (2 * L)) - 1u)) << key_off(K, L));
          const int ne = push_vertex(w, x, L, e, (1u << (2 * (K - 2))) - 1u);
          if (lane == 0) {
            int* sv = lvs + 5 * L;
            sv[0] = c + 1;
            sv[1] = cee;
            sv[2] = e;
            sv[3] = (int)key;
            sv[4] = x;
          }
          __syncwarp();
          cur_c = c + 1;
          cur_ce = ne;
          cur_e = ne;
          cur_key = nkey;
          if (L == 1 && has2) {
            cur_c = c + 1 + it.a2;
            cur_ce = min(c + 1 + (int)it.b2, ne);
          }
          if (K == 6 && L == 2 && has3) {
            cur_c = c + 1 + it.a3;
            cur_ce = min(c + 1 + (int)it.b3, ne);
          }
          L += 1;
          if (L == K - 2) fresh = true;
          if (KEPT && L == K - 3) decide = true;
        } else {
          if (L == 1) break;
          pop_level();
        }
      }
      // pop the root
      for (int b = f; b < re; b += 32) {
        const int i = b + lane;
        if (i < re) lab[ent_vertex(w.ucol[i])] &= (LT)~3u;
      }
      __syncwarp();
    }
    // this graph's queue is empty: flush, then move to a graph with items left
    __syncthreads();
    since = 0;
    if (K <= 5) {
      for (int i = tid; i < (int)C; i += blockDim.x) {
        const int32_t x = s_hist[i];
        if (x) {
          atomicAdd(&ghist[i], (unsigned long long)(long long)x);
          s_hist[i] = 0;
        }
      }
      if (tid == 0 && s_hist[C] != 0) {
        atomicOr(w.err, kErrStackOverflow);
        s_hist[C] = 0;
      }
    }
    if (tid == 0) {
      s_idle = 0;
      s_ndon = 0;
      int next = -1;
      for (int t = 1; t <= a.G; ++t) {
        const int g2 = (g + t) % a.G;
        if (*(volatile uint32_t*)&a.gp[g2].qhead < a.gp[g2].count) {
          next = g2;
          break;
        }
      }
      s_cur_g = next;
    }
    __syncthreads();
    g = s_cur_g;
  }
  if (bad_id) atomicOr(&a.hdr->err, kErrStackOverflow);
}

// ------------------------------------------------------------------ host side

static size_t round16(size_t x) { return (x + 15) & ~(size_t)15; }

// The kernel of a launch shape.  Kept lists: words and graph in shared memory.
template <int K, bool CB>
static const void* pick_kernel_kc(bool gc, bool ls, bool sg) {
  if (sg) return ls ? (const void*)k_count<K, false, true, CB, true>
                    : (const void*)k_count<K, false, false, CB, true>;
  if (gc) return ls ? (const void*)k_count<K, true, true, CB> : (const void*)k_count<K, true, false, CB>;
  return ls ? (const void*)k_count<K, false, true, CB> : (const void*)k_count<K, false, false, CB>;
}

template <int K>
static const void* pick_kernel_k(bool gc, bool ls, bool cb, bool sg) {
  return cb ? pick_kernel_kc<K, true>(gc, ls, sg) : pick_kernel_kc<K, false>(gc, ls, sg);
}

static const void* pick_kernel(const CountPlan& p) {
  if (p.keep)
    return p.K == 5 ? (const void*)k_count<5, true, true, true, false, true>
                    : (const void*)k_count<6, true, true, true, false, true>;
  switch (p.K) {
    case 3: return pick_kernel_k<3>(p.gcache, p.lab_smem, p.comb, p.stack_global);
    case 4: return pick_kernel_k<4>(p.gcache, p.lab_smem, p.comb, p.stack_global);
    case 5: return pick_kernel_k<5>(p.gcache, p.lab_smem, p.comb, p.stack_global);
    default: return pick_kernel_k<6>(p.gcache, p.lab_smem, p.comb, p.stack_global);
  }
}

mt_status count_configure_tuned(CountPlan* p, int K, int G, int nmax, int dmax, int64_t fwd_bound,
                                int64_t entry_stride, uint32_t classes, const mt_tuning* tuning,
                                bool compact, int method, double sets) {
  if (tuning) method = tuning->method;
  if (K < 3 || K > 6 || G < 1 || nmax < 1) return MT_EINVAL;
  const double split_cost = tuning ? tuning->split_cost : 0.0;
  const int warps_per_block = tuning ? tuning->warps_per_block : 0;
  p->K = K;
  p->G = G;
  p->nmax = nmax;
  p->dmax = dmax;
  p->fwd_bound = fwd_bound;
  p->entry_stride = entry_stride > 0 ? entry_stride : 1;
  p->classes = classes;
  p->split_cost = split_cost;
  p->split_scale = (tuning && tuning->split_scale > 0.0) ? tuning->split_scale : 1.0;
  p->items_factor = tuning ? 5.0 : 1.25;
  // The stack holds the root's forward list and the exclusive neighbours of the
  // vertices at positions 1..k-3 (positions k-2 and k-1 are finished in place),
  // each at most one row: k-2 rows of at most dmax entries.
  p->cap = (tuning && tuning->stack_cap > 0) ? tuning->stack_cap
                                             : std::max(K - 2, 1) * std::max(dmax, 1) + 32;
  if (p->cap > 65535) return MT_EUNSUPPORTED;
  p->nu_cap = (int)p->entry_stride;
  // The library's own choice counts the same histogram from the (k-2)-sets
  // instead of from every k-set.  Measured on a GB300, per-subgraph against
  // cells: k = 6 one graph (n = 800) 2.3 : 1.2 ms, 65 of them 135 : 71 ms; k = 5
  // one graph (n = 1,500) 2.4 : 0.88 ms, 257 of them 526 : 187 ms; k = 4 n = 239 /
  // 2,000 / 3,646 59 : 59, 235 : 119, 455 : 163 us; k = 3 n = 122 / 300 / 20,000
  // 57 : 58, 58 : 60, 289 : 144 us.
  if (method == kAutoMethod) method = MT_METHOD_CELLS;
  else if (compact && method == MT_METHOD_CELLS)
    return MT_EUNSUPPORTED;
  p->comb = method == MT_METHOD_CELLS;
  p->compact = compact;
  if (compact && K != 6) return MT_EUNSUPPORTED;
  p->map_bytes = compact ? 256 : 0;
  const size_t lab_elem = (K <= 4 || (p->comb && K <= 5)) ? 1 : ((K == 5 || p->comb) ? 2 : 4);
  const size_t lab_bytes = round16((size_t)nmax * lab_elem);
  const size_t cells = (size_t)1 << (2 * (K - 2));
  const size_t cell_bytes =
      p->comb ? round16(cells * 4) + (kNumbered * 4 + 64) * 4 + 16 +
                    round16(std::min<size_t>(cells, p->cap) * 2)
              : 0;
  const size_t buf_bytes = round16((size_t)p->cap * 2) + cell_bytes + kLevelBytes + p->map_bytes;
  // k <= 5: one 32-bit counter per class plus a catch slot for invalid ids
  const size_t hist_bytes = K <= 5 ? round16(((size_t)classes + 1) * 4) : 0;
  // the cell method's copy has 16-bit entries and rows padded to segments
  const size_t graph_bytes =
      round16((size_t)(nmax + 1) * 4) +
      (p->comb ? round16(((size_t)p->nu_cap + (size_t)nmax * (kSeg - 1)) * 2 + kSeg * 2)
               : round16((size_t)p->nu_cap * 4));
  const bool copy_fits16 = nmax < kMaxVertices16;
  int dev = 0, sms = 0, max_smem = 0;
  MT_CUDA_TRY(cudaGetDevice(&dev));
  MT_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  MT_CUDA_TRY(cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  const size_t budget = (size_t)max_smem - 1024;
  const int want = warps_per_block > 0 ? std::min(warps_per_block, kMaxWarpsPerBlock)
                                       : kMaxWarpsPerBlock;
  // Layout: the one that fits the most warps (>= 16 if any does), and on a tie
  // the first of: graph copy and relation words in shared memory, relation
  // words only, graph only, neither.  More warps beat the graph copy: rows
  // read through L1 cost less than the warps the copy displaces.
  // The cell method spends its time on rows and words instead: 27 warps with
  // words and copy count a k = 5 batch (n = 1,500, 257 graphs) in 187 ms, 32
  // with words only in 216 ms, 32 with the copy only in 223 ms.
  struct Opt { bool gc, ls; };
  const Opt opts[4] = {{true, true}, {false, true}, {true, false}, {false, false}};
  bool found = false;
  for (int pass = 0; pass < 2 && !found; ++pass) {
    const int min_w = pass == 0 ? std::min(want, 16) : 1;
    int best_score = 0;
    for (const Opt& o : opts) {
      if (o.gc && p->comb && !copy_fits16) continue;
      const size_t fixed = (o.gc ? graph_bytes : 0) + hist_bytes;
      const size_t per = (o.ls ? lab_bytes : 0) + buf_bytes;
      int w = want;
      while (w > min_w && fixed + (size_t)w * per > budget) --w;
      const int score = w * (!p->comb ? 4 : !o.ls ? 2 : o.gc ? 5 : 4);
      if (fixed + (size_t)w * per <= budget && score > best_score) {
        p->gcache = o.gc;
        p->lab_smem = o.ls;
        p->warps_per_block = w;
        p->smem_bytes = fixed + (size_t)w * per;
        found = true;
        best_score = score;
      }
    }
  }
  // Graphs with hubs so large that no shared-memory layout holds 16 warps'
  // candidate stacks: the stacks go to per-warp slices of global memory
  // (L1/L2-cached), with the relation words in shared memory when they fit.
  const size_t stack_bytes = round16((size_t)p->cap * 2);
  p->stack_global = false;
  if (!found || p->warps_per_block < std::min(want, 16)) {
    int best_w = found ? p->warps_per_block : 0;
    for (const bool ls : {true, false}) {
      const size_t per = (ls ? lab_bytes : 0) + buf_bytes - stack_bytes;
      int w = want;
      while (w > 1 && hist_bytes + (size_t)w * per > budget) --w;
      if (hist_bytes + (size_t)w * per <= budget && w > best_w) {
        p->gcache = false;
        p->lab_smem = ls;
        p->stack_global = true;
        p->warps_per_block = w;
        p->smem_bytes = hist_bytes + (size_t)w * per;
        found = true;
        best_w = w;
      }
    }
  }
  if (!found) return MT_EUNSUPPORTED;
  p->graph_bytes = p->gcache ? graph_bytes : 0;
  p->hist_bytes = hist_bytes;
  p->lab_bytes = lab_bytes;
  p->buf_bytes = buf_bytes - cell_bytes - kLevelBytes - p->map_bytes;
  p->cell_bytes = cell_bytes;
  // (one block per SM, as in every layout that keeps lists)
  p->keep = K >= 5 && p->comb && p->gcache && p->lab_smem && G >= kKeepGraphs &&
            dmax >= (K == 5 ? kKeepDegree5 : kKeepDegree6) &&
            sets >= (K == 5 ? kKeepSets5 : kKeepSets6) * sms * p->warps_per_block *
                        kTargetItemsPerWarp;
  const void* kern = pick_kernel(*p);
  // the limit belongs to the kernel, not to this plan: a smaller plan made before
  // a batch runs must not lower it
  MT_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)budget));
  int occ = 0;
  MT_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, p->warps_per_block * 32,
                                                            p->smem_bytes));
  if (occ < 1) return MT_EUNSUPPORTED;
  p->blocks = sms * occ;
  const double target = (double)p->blocks * p->warps_per_block * kTargetItemsPerWarp;
  p->items_max = (uint64_t)(target * p->items_factor * 1.01) + 16 * (uint64_t)G +
                 2 * (uint64_t)fwd_bound + 4096;
  size_t off = 0;
  p->off_hdr = off; off += 256;
  p->off_gp = off; off += round16((size_t)G * sizeof(GraphPlan));
  p->off_dsum = off;
  if (p->comb && K >= 5) off += round16((size_t)G * nmax * 4);
  p->off_items = off; off += round16(p->items_max * sizeof(Item));
  p->off_lab = off;
  if (!p->lab_smem) off += (size_t)p->blocks * p->warps_per_block * lab_bytes;
  p->off_stack = off;
  if (p->stack_global) off += (size_t)p->blocks * p->warps_per_block * p->buf_bytes;
  off = (off + 255) & ~(size_t)255;
  p->off_kept = off;
  p->kept_bytes = 0;
  if (p->keep) {
    p->kept_bytes = (((size_t)p->cap + kKeptArcs) * 4 + 127) & ~(size_t)127;
    off += (size_t)p->blocks * p->warps_per_block * p->kept_bytes;
  }
  p->ws_bytes = off + 256;
  return MT_OK;
}

double estimate_sets(int K, int n, const int32_t* deg, const int32_t* row_ptr, const int32_t* col) {
  double sets = 0.0;
  if (K == 5)
    for (int v = 0; v < n; ++v) sets += 0.5 * deg[v] * (deg[v] - 1.0);
  if (K == 6)
    for (int v = 0; v < n; ++v) {
      const double d = deg[v];
      double ends = 0.0;
      for (int32_t e = row_ptr[v]; e < row_ptr[v + 1]; ++e) ends += deg[col[e]] - 1.0;
      sets += d * (d - 1.0) * (d - 2.0) / 6.0 + (d - 1.0) * ends;
    }
  return sets;
}

void plan_info(const CountPlan& p, int32_t* warps_per_block, int32_t* blocks, int32_t* stack_cap,
               uint32_t* layout) {
  if (warps_per_block) *warps_per_block = p.warps_per_block;
  if (blocks) *blocks = p.blocks;
  if (stack_cap) *stack_cap = p.cap;
  if (layout)
    *layout = (p.gcache ? 1u : 0u) | (p.lab_smem ? 2u : 0u) | (p.stack_global ? 4u : 0u) |
              (p.keep ? 8u : 0u);
}

uint32_t* count_err_ptr(const CountPlan& p, void* ws) {
  return &((Hdr*)((char*)ws + p.off_hdr))->err;
}
uint32_t* count_nitems_ptr(const CountPlan& p, void* ws) {
  return &((GraphPlan*)((char*)ws + p.off_gp))->count;
}

// Start of a one-graph launch: its descriptor, which travels as a kernel argument
// so that a captured launch holds it and reads no host memory at replay, and
// zeros in header and plan (`words` 8-byte words).  One kernel for both: in place
// of the header's memset it costs nothing, beside it a k = 3 count of n = 300 took
// 76 us, not 69.
__global__ void __launch_bounds__(32) k_begin(DevGraph* dst, DevGraph src,
                                              unsigned long long* hdr, int words) {
  if (threadIdx.x == 0) *dst = src;
  for (int i = threadIdx.x; i < words; i += blockDim.x) hdr[i] = 0;
}

template <int K>
static cudaError_t enqueue_k(const CountPlan& p, void* ws, DevGraph* graphs, const DevGraph* one,
                             const TableView& table, int32_t rb, int32_t re, cudaStream_t s,
                             unsigned long long* copies_base, int copies, uint32_t copy_stride) {
  char* base = (char*)ws;
  Hdr* hdr = (Hdr*)(base + p.off_hdr);
  GraphPlan* gp = (GraphPlan*)(base + p.off_gp);
  Item* items = (Item*)(base + p.off_items);
  void* lab = base + p.off_lab;
  // header and graph plans are neighbours
  const size_t zeros = p.off_gp - p.off_hdr + (size_t)p.G * sizeof(GraphPlan);
  cudaError_t e = cudaSuccess;
  if (one)
    k_begin<<<1, 32, 0, s>>>(graphs, *one, (unsigned long long*)(base + p.off_hdr),
                             (int)(zeros / 8));
  else
    e = cudaMemsetAsync(base + p.off_hdr, 0, zeros, s);
  if (e != cudaSuccess) return e;
  SplitArgs sa;
  sa.split_cost = p.split_cost;
  sa.split_scale = p.split_scale;
  sa.target_items = (double)p.blocks * p.warps_per_block * kTargetItemsPerWarp;
  sa.items_factor = p.items_factor;
  sa.floor = p.comb ? kCellsItemFloor<K> : 1.0;
  sa.items_max = p.items_max;
  sa.root_begin = rb;
  sa.root_end = re;
  const int ex = (int)std::min<int64_t>((p.entry_stride + 255) / 256, 4096);
  // one warp per root, until the grid holds some thousands of blocks
  const int rx = std::max(1, std::min((p.nmax + 7) / 8, std::max(2048 / p.G, 4)));
  const int rz = std::max(1, std::min(8, std::min((p.dmax + 31) / 32, 2048 / (rx * p.G))));
  int32_t* dsum = (int32_t*)(base + p.off_dsum);
  if (p.comb) {
    if (K >= 5) k_plan_degsum<<<dim3(rx, p.G), 256, 0, s>>>(graphs, p.nmax, dsum);
    // One graph whose whole work is below the items' floor whatever its rows are:
    // the threshold is the floor (an upper bound of the total stands for it).
    const double most = (double)(p.entry_stride / 2 + 1) * (72.0 + 4.0 * p.dmax);
    const bool known = K <= 4 && p.G == 1 && p.split_cost == 0.0 && p.split_scale == 1.0 &&
                       most <= sa.floor * sa.target_items;
    if (!known) k_plan_total<K, true><<<dim3(ex, p.G), 256, 0, s>>>(graphs, gp, dsum, p.nmax, rb, re);
    k_plan_items<K, true><<<dim3(rx, p.G, rz), 256, 0, s>>>(graphs, p.G, gp, dsum, p.nmax, items, hdr,
                                                        sa);
  } else {
    k_plan_total<K, false><<<dim3(ex, p.G), 256, 0, s>>>(graphs, gp, dsum, p.nmax, rb, re);
    k_plan_items<K, false><<<dim3(rx, p.G, rz), 256, 0, s>>>(graphs, p.G, gp, dsum, p.nmax, items, hdr,
                                                         sa);
  }
  if (!p.lab_smem) {
    e = cudaMemsetAsync(lab, 0, (size_t)p.blocks * p.warps_per_block * p.lab_bytes, s);
    if (e != cudaSuccess) return e;
  }
  CountArgs a;
  a.graphs = graphs;
  a.items = items;
  a.gp = gp;
  a.hdr = hdr;
  a.table = table.slots;
  a.xclass = p.compact ? table.xclass : nullptr;
  a.xmap = p.compact ? table.xmap : nullptr;
  a.map_bytes = (int)p.map_bytes;
  a.idle_ns = g_idle_ns;
  a.lab_global = lab;
  a.stack_global = base + p.off_stack;
  a.kept = p.kept_bytes ? base + p.off_kept : nullptr;
  a.kept_bytes = p.kept_bytes;
  a.hist_copies = copies_base;
  a.copies = copies;
  a.copy_stride = copy_stride;
  a.G = p.G;
  a.nmax = p.nmax;
  a.cap = p.cap;
  a.classes = p.classes;
  a.graph_bytes = (int)p.graph_bytes;
  a.hist_bytes = (int)p.hist_bytes;
  a.lab_bytes = (int)p.lab_bytes;
  a.buf_bytes = (int)p.buf_bytes;
  a.cell_bytes = (int)p.cell_bytes;
  const unsigned threads = p.warps_per_block * 32;
  void* args[] = {&a};
  return cudaLaunchKernel(pick_kernel(p), dim3(p.blocks), dim3(threads), args, p.smem_bytes, s);
}

mt_status count_enqueue(const CountPlan& p, void* ws, DevGraph* graphs, const DevGraph* one,
                        const TableView& table, int32_t root_begin, int32_t root_end,
                        cudaStream_t s, unsigned long long* copies_base, int copies,
                        uint32_t copy_stride) {
  if (copies > 1 && (p.K != 6 || p.G != 1 || !copies_base)) return MT_EINVAL;
  if (one && p.G != 1) return MT_EINVAL;
  cudaError_t e;
  switch (p.K) {
    case 3: e = enqueue_k<3>(p, ws, graphs, one, table, root_begin, root_end, s, nullptr, 1, 0); break;
    case 4: e = enqueue_k<4>(p, ws, graphs, one, table, root_begin, root_end, s, nullptr, 1, 0); break;
    case 5: e = enqueue_k<5>(p, ws, graphs, one, table, root_begin, root_end, s, nullptr, 1, 0); break;
    default:
      e = enqueue_k<6>(p, ws, graphs, one, table, root_begin, root_end, s, copies_base, copies,
                       copy_stride);
      break;
  }
  if (e != cudaSuccess) {
    set_last_error(cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? MT_ENOMEM : MT_ECUDA;
  }
  return MT_OK;
}

// Histogram copies of a one-graph count (see kHistCopies).
static int count_hist_copies(const CountPlan& p) { return p.K == 6 && p.G == 1 ? kHistCopies : 1; }

// Scratch of a one-graph count: plan workspace + the DevGraph + a histogram +
// the histogram's extra copies.
static size_t count_scratch_bytes(const CountPlan& p, uint32_t C) {
  return p.ws_bytes + 256 + (size_t)count_hist_copies(p) * round16((size_t)C * 8);
}

// Give up g's scratch: the library's own goes back to the pool on `s`, or stays
// with the handle when a captured count uses it.  The caller has waited for the
// counts that use it.
static void drop_scratch(mt_graph* g, cudaStream_t s) {
  if (g->ws && g->ws_owned) {
    if (g->ws_captured) g->captured_ws.push_back(g->ws);
    else pool_free(g->ws, s);
    g->ws_captured = false;
  }
  g->ws = nullptr;
  g->ws_bytes = 0;
}

// Plain one-graph count with the workspace cached in the graph handle.
static mt_status count_one(const mt_graph* gc, const mt_table* t, uint64_t* hist,
                           int32_t rb, int32_t re, const mt_tuning* tuning, cudaStream_t s) {
  mt_graph* g = const_cast<mt_graph*>(gc);
  const int K = table_k(t);
  const uint32_t C = table_classes(t);
  CountPlan p;
  MT_TRY(count_configure_tuned(&p, K, 1, g->n, g->dmax, g->nu / 2 + 1, std::max(g->nu, 1), C,
                               tuning, table_compact(t)));
  // workspace: plan scratch + the DevGraph + a device histogram
  const size_t need = count_scratch_bytes(p, C);
  if (!g->ws_owned && g->ws_bytes < need) {
    set_last_error("attached workspace holds " + std::to_string(g->ws_bytes) +
                   " bytes, this count needs " + std::to_string(need));
    return MT_EINVAL;
  }
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  MT_CUDA_TRY(cudaStreamIsCapturing(s, &cap));
  const bool captured = cap != cudaStreamCaptureStatusNone;
  if (g->ws_bytes < need) {
    // scratch outlives a captured launch, so it is not allocated by one
    if (captured) {
      set_last_error("the first count of a graph allocates scratch: not under stream capture");
      return MT_ECUDA;
    }
    // an earlier count may still use the old scratch, on any stream
    if (g->ws) MT_CUDA_TRY(cudaDeviceSynchronize());
    drop_scratch(g, s);
    MT_CUDA_TRY(pool_alloc(&g->ws, need, s));
    g->ws_bytes = need;
  }
  if (captured && g->ws_owned) g->ws_captured = true;
  if (!g->ev0) {
    MT_CUDA_TRY(cudaEventCreate(&g->ev0));
    MT_CUDA_TRY(cudaEventCreate(&g->ev1));
  }
  char* base = (char*)g->ws;
  DevGraph* dg = (DevGraph*)(base + p.ws_bytes);
  cudaPointerAttributes attr;
  bool dev_hist = cudaPointerGetAttributes(&attr, hist) == cudaSuccess &&
                  (attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged);
  cudaGetLastError();
  if (dev_hist && attr.type == cudaMemoryTypeDevice) {
    int dev = 0;
    MT_CUDA_TRY(cudaGetDevice(&dev));
    if (attr.device != dev) {  // this device's kernels would write another GPU's memory
      set_last_error("hist is memory of device " + std::to_string(attr.device) +
                     ", the current device is " + std::to_string(dev));
      return MT_EINVAL;
    }
  }
  unsigned long long* dh =
      dev_hist ? (unsigned long long*)hist : (unsigned long long*)(base + p.ws_bytes + 256);
  // a part of the roots: sets belong to their smallest original vertex
  const bool part = rb > 0 || re < g->n;
  if (part && g->n >= K && rb < re) {
    if (original_scratch_bytes(g) > p.ws_bytes - p.off_items) return MT_EOVERFLOW;
    MT_TRY(graph_build_original(g, base + p.off_items, s));  // before the items are written
  }
  const DevGraph hg = dev_view(g, dh, part);
  MT_CUDA_TRY(cudaMemsetAsync(dh, 0, (size_t)C * 8, s));
  if (g->n >= K && rb < re) {
    const int copies = count_hist_copies(p);
    const uint32_t stride = (uint32_t)(round16((size_t)C * 8) / 8);
    unsigned long long* cbase = (unsigned long long*)(base + p.ws_bytes + 256) + stride;
    MT_CUDA_TRY(cudaEventRecord(g->ev0, s));
    if (copies > 1)
      MT_CUDA_TRY(cudaMemsetAsync(cbase, 0, (size_t)(copies - 1) * stride * 8, s));
    MT_TRY(count_enqueue(p, g->ws, dg, &hg, table_view(t), rb, re, s, cbase, copies, stride));
    if (copies > 1) {
      const unsigned fb = (unsigned)std::min<uint32_t>((C + 255) / 256, 152u * 8u);
      k_fold_copies<<<fb, 256, 0, s>>>(dh, cbase, copies - 1, C, stride);
      MT_CUDA_TRY(cudaGetLastError());
    }
    MT_CUDA_TRY(cudaEventRecord(g->ev1, s));
  } else {
    // no launch: the status word and the item count are read all the same
    MT_CUDA_TRY(cudaMemsetAsync(base + p.off_hdr, 0, p.off_gp - p.off_hdr + sizeof(GraphPlan), s));
    MT_CUDA_TRY(cudaEventRecord(g->ev0, s));
    MT_CUDA_TRY(cudaEventRecord(g->ev1, s));
  }
  if (!dev_hist) {
    MT_CUDA_TRY(cudaMemcpyAsync(hist, dh, (size_t)C * 8, cudaMemcpyDeviceToHost, s));
  }
  g->stats_valid = true;
  g->off_err = (size_t)((char*)count_err_ptr(p, g->ws) - base);
  g->off_nitems = (size_t)((char*)count_nitems_ptr(p, g->ws) - base);
  if (!dev_hist) {
    uint32_t err = 0;
    MT_CUDA_TRY(cudaMemcpyAsync(&err, base + g->off_err, 4, cudaMemcpyDeviceToHost, s));
    MT_CUDA_TRY(cudaStreamSynchronize(s));
    if (err) return (err & kErrWaitLimit) ? MT_ETIMEOUT : MT_EOVERFLOW;
  }
  return MT_OK;
}

}  // namespace mt

using namespace mt;

extern "C" {

mt_status mt_count_roots(const mt_graph* g, const mt_table* t, int32_t root_begin,
                         int32_t root_end, uint64_t* hist, void* stream) {
  if (!g || !t || !hist) return MT_EINVAL;
  if (root_begin < 0) root_begin = 0;
  if (root_end > g->n) root_end = g->n;
  return count_one(g, t, hist, root_begin, root_end, nullptr, (cudaStream_t)stream);
}

mt_status mt_count(const mt_graph* g, const mt_table* t, uint64_t* hist, void* stream) {
  if (!g || !t || !hist) return MT_EINVAL;
  return count_one(g, t, hist, 0, g->n, nullptr, (cudaStream_t)stream);
}

mt_status mt_count_tuned(const mt_graph* g, const mt_table* t, uint64_t* hist,
                         const mt_tuning* tuning, void* stream) {
  if (!g || !t || !hist) return MT_EINVAL;
  if (tuning && (tuning->split_cost < 0 || tuning->split_scale < 0 ||
                 tuning->warps_per_block < 0 || tuning->warps_per_block > 32 ||
                 tuning->stack_cap < 0 || tuning->stack_cap > 65535 ||
                 tuning->method < 0 || tuning->method > 1))
    return MT_EINVAL;
  return count_one(g, t, hist, 0, g->n, tuning, (cudaStream_t)stream);
}

mt_status mt_set_wait_limit(uint64_t ns) {
  g_idle_ns = ns ? (unsigned long long)ns : kIdleNs;
  return MT_OK;
}

mt_status mt_workspace_query(const mt_graph* g, int k, size_t* bytes) {
  if (!g || !bytes) return MT_EINVAL;
  if (k < 3 || k > 6) return MT_EUNSUPPORTED;
  CountPlan p;
  MT_TRY(count_configure_tuned(&p, k, 1, g->n, g->dmax, g->nu / 2 + 1, std::max(g->nu, 1),
                               kNumClasses[k], nullptr));
  *bytes = count_scratch_bytes(p, kNumClasses[k]);
  return MT_OK;
}

mt_status mt_count_launch_info(const mt_graph* g, int k, int32_t* warps_per_block,
                               int32_t* blocks, int32_t* stack_cap, uint32_t* layout) {
  if (!g) return MT_EINVAL;
  if (k < 3 || k > 6) return MT_EUNSUPPORTED;
  CountPlan p;
  MT_TRY(count_configure_tuned(&p, k, 1, g->n, g->dmax, g->nu / 2 + 1, std::max(g->nu, 1),
                               kNumClasses[k], nullptr));
  plan_info(p, warps_per_block, blocks, stack_cap, layout);
  return MT_OK;
}

mt_status mt_set_workspace(mt_graph* g, void* ws, size_t bytes) {
  if (!g) return MT_EINVAL;
  if (ws) {
    cudaPointerAttributes attr;
    const bool dev = cudaPointerGetAttributes(&attr, ws) == cudaSuccess &&
                     attr.type == cudaMemoryTypeDevice;
    cudaGetLastError();
    if (!dev || ((uintptr_t)ws & 255u) || bytes == 0) {
      set_last_error("mt_set_workspace: ws must be device memory, 256-byte aligned, non-empty");
      return MT_EINVAL;
    }
  }
  // an earlier count may still use the current scratch, on any stream of the
  // graph's device
  DeviceScope on(g->device);
  MT_CUDA_TRY(cudaDeviceSynchronize());
  drop_scratch(g, nullptr);
  g->ws = ws;
  g->ws_bytes = ws ? bytes : 0;
  g->ws_owned = ws == nullptr;
  g->stats_valid = false;
  return MT_OK;
}

mt_status mt_count_stats(const mt_graph* g, uint64_t* items, uint32_t* err, float* ms) {
  if (!g) return MT_EINVAL;
  uint32_t it = 0, er = 0;
  float t = 0.f;
  if (g->stats_valid) {
    MT_CUDA_TRY(cudaEventSynchronize(g->ev1));
    MT_CUDA_TRY(cudaMemcpy(&it, (char*)g->ws + g->off_nitems, 4, cudaMemcpyDeviceToHost));
    MT_CUDA_TRY(cudaMemcpy(&er, (char*)g->ws + g->off_err, 4, cudaMemcpyDeviceToHost));
    MT_CUDA_TRY(cudaEventElapsedTime(&t, g->ev0, g->ev1));
  }
  if (items) *items = it;
  if (err) *err = er;
  if (ms) *ms = t;
  return MT_OK;
}

}  // extern "C"
