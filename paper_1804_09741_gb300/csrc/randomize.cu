// K3: degree-preserving directed arc swaps (the null model of Sec. 1, step (c);
// the paper names no randomisation model, the reading is the switch of Milo et
// al.).  Attempts run in order, exactly as the sequential definition:
//   attempt t draws arc positions e1 = floor(r1 m / 2^64), e2 = floor(r2 m / 2^64)
//   with r1, r2 = SplitMix64 outputs 2t and 2t+1 of the graph's seed; arcs
//   (a->b) at e1 and (c->d) at e2 become (a->d), (c->b) unless e1 == e2, a == c,
//   b == d, a == d, c == b, or (a->d) or (c->b) is already an arc.
// A swap keeps the source of each position, so the out-CSR shape is unchanged:
// only the destinations move, and the builder re-sorts the rows afterwards.
//
// GPU mapping: one thread block per graph.  The arc array (src<<16 | dst) and a
// hash set of the present arcs sit in shared memory (global memory for graphs
// too large for it); the block fills them in parallel.  Then 256 threads run
// the attempts in windows of 64 (128 threads, 32 for small graphs), four threads
// per attempt (one per arc that it looks up or replaces; a warp has new arcs or
// old ones), while two warps draw the next attempts' positions, which do not
// depend on the graph:
//  * speculation: every attempt is evaluated against the state at the start of
//    the window (the two arcs at its positions, the checks, whether the two new
//    arcs are present);
//  * resolution: an attempt's speculative outcome is its sequential outcome
//    unless an earlier attempt of the window that the speculation accepted wrote
//    one of its two positions, or inserted or erased one of the two arcs it
//    looks up.  Accepted attempts set their bit in two small tables hashed by
//    position and by arc; an attempt reads the bits of its own four entries and
//    compares itself with the earlier attempts it finds there, so hash
//    collisions cost a comparison and no lost attempt;
//  * the attempts before the first unsafe one are applied together (their
//    positions and arcs are disjoint), and the next window starts at it.
// The outcome is that of the attempts run one after another.  What bounds it is
// the latency of one window after another: at m = 6,000 a window passes 44.5
// attempts (two attempts of a window overlap with probability about 4 / m; 128
// wide it would pass 50) and takes 1.4 us.  One graph of m = 6,000, 60,000
// attempts: 7.2 ms with one warp, 32 attempts and bucket scans by every lane,
// 2.1 ms now; 511 graphs of m = 1,500: 6.0 ms, 1.5 in windows of 64, 1.1 in windows
// of 32.
//
// Set: 2^bb buckets of 8 slots (two 16-byte reads), 2 to 4 keys per bucket on
// average; a key lives in the first bucket of its probe sequence (home bucket,
// then the next ones) that had a free slot when it was inserted, and every
// bucket counts the keys that passed over it, so a lookup moves on only past
// buckets with a count.  Only membership matters to the attempts, not where a
// key is stored, so the results are those of the sequential definition.
//
// SplitMix64 (Steele, Lea and Flood, OOPSLA 2014, public-domain reference
// generator): state advances by the golden gamma 0x9E3779B97F4A7C15, output =
// mix(state) with the variant-13 mix; output i of seed s is mix(s + (i+1)*gamma).
#include "graph.cuh"
#include "trace.cuh"

namespace mt {

constexpr uint32_t kEmpty = 0xFFFFFFFFu;
constexpr unsigned kWarp = 0xFFFFFFFFu;

__device__ __forceinline__ uint64_t sm64_mix(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Layout of one graph's randomiser state (in 32-bit words): the entry array
// (arcs, or the dyad lists) padded to 4 words, the buckets, their counts (16
// bits each).
struct RandLayout {
  int bb;          // log2 of the number of buckets (>= 1)
  size_t t_off;    // first slot
  size_t c_off;    // first count word
  size_t words;    // total
};

__host__ __device__ inline RandLayout rand_layout(int32_t m) {
  RandLayout L;
  int bb = 1;
  while ((4ll << bb) < (m > 0 ? m : 1)) ++bb;  // at most 4 keys per bucket on average
  L.bb = bb;
  L.t_off = ((size_t)(m > 0 ? m : 1) + 3) & ~(size_t)3;
  L.c_off = L.t_off + ((size_t)8 << bb);
  L.words = (L.c_off + ((size_t)1 << bb) / 2 + 3) & ~(size_t)3;
  return L;
}

// Reads of the state: another thread of the block may have written it, and the
// set's global-memory form is updated by atomics, so that form reads past L1.
template <bool GM, typename T>
__device__ __forceinline__ T state_read(const T* p) {
  return GM ? __ldcg(p) : *p;
}

// A bucket's 8 slots.
struct BucketRow {
  uint4 a, b;
  __device__ __forceinline__ bool has(uint32_t key) const {
    return a.x == key || a.y == key || a.z == key || a.w == key || b.x == key || b.y == key ||
           b.z == key || b.w == key;
  }
  // bits of the slots holding `key`
  __device__ __forceinline__ unsigned mask(uint32_t key) const {
    return (a.x == key ? 1u : 0u) | (a.y == key ? 2u : 0u) | (a.z == key ? 4u : 0u) |
           (a.w == key ? 8u : 0u) | (b.x == key ? 16u : 0u) | (b.y == key ? 32u : 0u) |
           (b.z == key ? 64u : 0u) | (b.w == key ? 128u : 0u);
  }
  // index of the first slot holding `key`, or -1
  __device__ __forceinline__ int find(uint32_t key) const {
    int at = -1;
    if (b.w == key) at = 7;
    if (b.z == key) at = 6;
    if (b.y == key) at = 5;
    if (b.x == key) at = 4;
    if (a.w == key) at = 3;
    if (a.z == key) at = 2;
    if (a.y == key) at = 1;
    if (a.x == key) at = 0;
    return at;
  }
};

template <bool GM>
struct BucketSet {
  uint32_t* t;     // (1 << bb) x 8 slots
  uint32_t* cnt;   // keys that passed over each bucket, two 16-bit counts per word
  int bb;
  uint32_t bmask;
  __device__ __forceinline__ uint32_t home(uint32_t key) const {
    return (key * 0x9E3779B1u) >> (32 - bb);
  }
  __device__ __forceinline__ BucketRow row(uint32_t b) const {
    const uint4* r = (const uint4*)t + 2 * b;
    return BucketRow{state_read<GM>(r), state_read<GM>(r + 1)};
  }
  __device__ __forceinline__ bool passed(uint32_t b) const {
    return ((state_read<GM>(cnt + (b >> 1)) >> (16 * (b & 1u))) & 0xFFFFu) != 0;
  }

  // Whether `key` is in a bucket after b (called when b has a count).
  __device__ __noinline__ bool contains_after(uint32_t key, uint32_t b) const {
    for (uint32_t i = 0; i < bmask; ++i) {
      b = (b + 1) & bmask;
      if (row(b).find(key) >= 0) return true;
      if (!passed(b)) break;
    }
    return false;
  }

  // Insert a key known to be absent (several threads at once).
  __device__ __noinline__ void insert(uint32_t key) const {
    uint32_t b = home(key);
    for (uint32_t i = 0; i <= bmask; ++i) {
      for (int at = row(b).find(kEmpty); at >= 0; at = row(b).find(kEmpty))
        if (atomicCAS(&t[8 * b + at], kEmpty, key) == kEmpty) return;
      atomicAdd(&cnt[b >> 1], 1u << (16 * (b & 1u)));
      b = (b + 1) & bmask;
    }
  }

  // Erase a key that is present but not in its home bucket b (several threads
  // at once, insertions too: keys do not move).
  __device__ __noinline__ void erase_after(uint32_t key, uint32_t b) const {
    for (uint32_t i = 0; i < bmask; ++i) {
      atomicSub(&cnt[b >> 1], 1u << (16 * (b & 1u)));
      b = (b + 1) & bmask;
      const int at = row(b).find(key);
      if (at >= 0) {
        t[8 * b + at] = kEmpty;
        return;
      }
    }
  }
};

// Shared-memory working set of the windows.
constexpr int kWindow = 64;      // attempts per window at most, four threads each
template <int WN>
constexpr int kRunners = 4 * WN;
template <int WN>
constexpr int kRandThreads = kRunners<WN> + 64;  // two warps draw
// Graphs of fewer arcs run windows of 32: little of a wider one passes (20 of 32
// attempts at m = 1,500, 24 of 64), and it takes half the warps.  Randomise phase of
// 1 and 511 null graphs, 32 against 64, ms: m = 1,500 0.72 : 0.85 and 1.00 : 1.45, 2,500
// 1.01 : 1.08 and 2.25 : 2.52, 3,000 1.32 : 1.36 and 2.90 : 3.08, 3,500 1.72 : 1.68 and
// 3.83 : 3.79, 4,000 2.18 : 2.01 and 4.85 : 4.61, 6,000 2.39 : 2.20 and 5.36 : 5.34.
constexpr int kWideArcs = 3000;
constexpr int kDraws = 256;      // attempts per buffer of drawn positions
constexpr int kKeyTab = 512, kPosTab = 512;
struct RandWindow {
  uint4 keys[kWindow];           // of an accepted attempt: new arcs, old arcs
  uint2 pos[kWindow];            //   and its positions
  uint2 ktab[kKeyTab];           // bits of the accepted attempts by arc (hashed)
  uint2 ptab[kPosTab];           //   and by position
  uint2 draws[2][kDraws];
  uint32_t accepted[2][4];       // accepted attempts, a bit per even lane of the new keys'
                                 // warps; windows alternate
  int first_bad[2];              // first unsafe attempt
};

__device__ __forceinline__ uint32_t key_slot(uint32_t key) {
  return (key * 0x85EBCA6Bu) >> 23;  // 32 - log2(kKeyTab)
}

// The even bits of x, together.
__device__ __forceinline__ uint32_t squeeze(uint32_t x) {
  x &= 0x55555555u;
  x = (x | x >> 1) & 0x33333333u;
  x = (x | x >> 2) & 0x0F0F0F0Fu;
  x = (x | x >> 4) & 0x00FF00FFu;
  return (x | x >> 8) & 0xFFFFu;
}

// Barrier of the threads that run the attempts.
template <int WN>
__device__ __forceinline__ void run_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(kRunners<WN>) : "memory");
}

// Threads 0 .. kRunners<WN> - 1: the attempts whose positions are draws[0..n), in
// order.  Thread 2j + q of the first half holds new key q of the window's attempt
// j (to be absent), of the second half old key q (a warp does one of the two).
// `Pol::make` derives from the two entries an attempt's validity, its keys and
// the two new entries.
template <class Pol, bool GM, int WN>
__device__ __forceinline__ void run_draws(const Pol& pol, uint32_t* ent, const BucketSet<GM>& S,
                                          RandWindow& W, const uint2* draws, int n) {
  const bool fresh = threadIdx.x < 2 * WN;
  const int j = (threadIdx.x >> 1) & (WN - 1), q = threadIdx.x & 1;
  const int half = j >> 5;
  const unsigned bit = 1u << (j & 31);
  for (int t = 0, w = 0; t < n; w ^= 1) {
    const int cnt = min(WN, n - t);
    // speculation; `valid`: the outcome depends on the graph, `tried`: its keys
    // are looked up
    uint2 e = make_uint2(0, 0);
    if (j < cnt) e = draws[t + j];
    const bool valid = e.x != e.y;
    uint32_t k1 = 0, k2 = 0, o1 = 0, o2 = 0, w1 = 0, w2 = 0;
    bool tried = false;
    if (valid)
      tried = pol.make(state_read<GM>(ent + e.x), state_read<GM>(ent + e.y), k1, k2, o1, o2, w1,
                       w2);
    const uint32_t key = fresh ? (q ? k2 : k1) : (q ? o2 : o1);
    const uint32_t pos = q ? e.y : e.x;
    const uint32_t ks = key_slot(key), ps = pos & (kPosTab - 1);
    const uint32_t h = S.home(key);
    const BucketRow r = S.row(h);
    int at;  // new key: a free slot of its home bucket; old key: its slot (only
             // this attempt may erase it, so the slot stays valid)
    if (fresh) {
      // new keys of one window prefer different slots of a bucket
      const unsigned slots = r.mask(kEmpty);
      at = slots ? (__ffs((slots | slots << 8) >> (j & 7)) - 1 + j) & 7 : -1;
      bool there = r.has(key);
      if (tried && !there && S.passed(h)) there = S.contains_after(key, h);
      const unsigned hit = __ballot_sync(kWarp, there);
      const bool acc = tried && ((hit >> (threadIdx.x & 30)) & 3u) == 0;
      const unsigned accs = __ballot_sync(kWarp, acc && q == 0);
      if ((threadIdx.x & 31) == 0) W.accepted[w][threadIdx.x >> 5] = accs;
      if (acc) {
        if (q == 0) W.pos[j] = e;
        else W.keys[j] = make_uint4(k1, k2, o1, o2);
        atomicOr((uint32_t*)&W.ktab[ks] + half, bit);
      }
    } else {
      // marked whether accepted or not; whoever reads the marks looks at
      // `accepted`
      at = r.find(key);
      if (tried) {
        atomicOr((uint32_t*)&W.ktab[ks] + half, bit);
        atomicOr((uint32_t*)&W.ptab[ps] + half, bit);
      }
    }
    run_sync<WN>();
    // the accepted attempts: one bit per pair of lanes of the new keys' warps
    const uint4 av = *(const uint4*)W.accepted[w];
    const uint32_t alo = squeeze(av.x) | squeeze(av.y) << 16;
    const uint32_t ahi = squeeze(av.z) | squeeze(av.w) << 16;
    const bool acc = ((half ? ahi : alo) & bit) != 0;
    // earlier accepted attempts that may overlap: by arc for the new keys, by
    // position for the old ones
    bool unsafe = false;
    if (fresh ? tried : valid) {
      const uint2 c = fresh ? W.ktab[ks] : W.ptab[ps];
      uint32_t lo = c.x & alo, hi = c.y & ahi;
      if (half == 0) {
        lo &= bit - 1u;
        hi = 0;
      } else {
        hi &= bit - 1u;
      }
      while (lo | hi) {
        const int i = lo ? __ffs(lo) - 1 : 31 + __ffs(hi);
        if (lo) lo &= lo - 1;
        else hi &= hi - 1;
        bool same;
        if (fresh) {
          const uint4 k = W.keys[i];
          same = key == k.x || key == k.y || key == k.z || key == k.w;
        } else {
          const uint2 p = W.pos[i];
          same = pos == p.x || pos == p.y;
        }
        if (same) {
          unsafe = true;
          break;
        }
      }
    }
    const unsigned bad = __ballot_sync(kWarp, unsafe);
    if (bad && (threadIdx.x & 31) == 0)
      atomicMin(&W.first_bad[w], j + ((__ffs(bad) - 1) >> 1));
    run_sync<WN>();
    // attempts before the first unsafe one (the first of a window is never
    // unsafe) are applied, and the marks go.  A free slot that another key took,
    // or a bucket without one, sends a key the slow way.
    const int p = min(W.first_bad[w], cnt);
    if (threadIdx.x == 0) W.first_bad[w ^ 1] = kWindow;
    const bool apply = acc && j < p;
    if (fresh) {
      if (acc) W.ktab[ks] = make_uint2(0, 0);
      if (apply && (at < 0 || atomicCAS(&S.t[8 * h + at], kEmpty, key) != kEmpty)) S.insert(key);
    } else {
      if (tried) {
        W.ktab[ks] = make_uint2(0, 0);
        W.ptab[ps] = make_uint2(0, 0);
      }
      if (apply) {
        ent[pos] = q ? w2 : w1;
        if (at >= 0) S.t[8 * h + at] = kEmpty;
        else S.erase_after(key, h);
      }
    }
    run_sync<WN>();
    t += p;
  }
}

// The attempts of one graph, by the whole block: kRunners threads run the drawn
// attempts of one buffer while the others draw the next buffer's positions.
template <int WN, class Pol, bool GM>
__device__ void run_attempts(const Pol& pol, uint32_t* ent, const BucketSet<GM>& S, RandWindow& W,
                             uint64_t attempts) {
  const int tid = threadIdx.x;
  for (int i = tid; i < kKeyTab; i += blockDim.x) W.ktab[i] = make_uint2(0, 0);
  for (int i = tid; i < kPosTab; i += blockDim.x) W.ptab[i] = make_uint2(0, 0);
  if (tid < 2) W.first_bad[tid] = kWindow;
  if (tid < 8) W.accepted[tid >> 2][tid & 3] = 0;  // the words of absent warps stay 0
  auto draw = [&](uint64_t t0, int buf, int first, int step) {
    for (int j = first; j < kDraws && t0 + j < attempts; j += step)
      pol.draw(t0 + j, W.draws[buf][j].x, W.draws[buf][j].y);
  };
  draw(0, 0, tid, blockDim.x);
  __syncthreads();
  int buf = 0;
  for (uint64_t t0 = 0; t0 < attempts; t0 += kDraws, buf ^= 1) {
    if (tid < kRunners<WN>) {
      const int n = (int)(attempts - t0 < (uint64_t)kDraws ? attempts - t0 : kDraws);
      run_draws<Pol, GM, WN>(pol, ent, S, W, W.draws[buf], n);
      if (tid == 0) W.first_bad[0] = kWindow;
    } else {
      draw(t0 + kDraws, buf ^ 1, tid - kRunners<WN>, blockDim.x - kRunners<WN>);
    }
    __syncthreads();
  }
}

// Degree-preserving arc swaps: attempt t's positions are SplitMix64 outputs
// 2t and 2t+1 scaled to [0, m); entries and keys are arcs (src << 16 | dst).
struct ArcSwap {
  uint64_t seed, m;
  __device__ void draw(uint64_t t, uint32_t& e1, uint32_t& e2) const {
    const uint64_t gamma = 0x9E3779B97F4A7C15ull;
    e1 = (uint32_t)__umul64hi(sm64_mix(seed + (2 * t + 1) * gamma), m);
    e2 = (uint32_t)__umul64hi(sm64_mix(seed + (2 * t + 2) * gamma), m);
  }
  __device__ bool make(uint32_t A, uint32_t B, uint32_t& k1, uint32_t& k2, uint32_t& o1,
                       uint32_t& o2, uint32_t& w1, uint32_t& w2) const {
    const uint32_t sa = A >> 16, da = A & 0xFFFFu, sc = B >> 16, dc = B & 0xFFFFu;
    if (sa == sc || da == dc || sa == dc || sc == da) return false;
    k1 = w1 = (sa << 16) | dc;
    k2 = w2 = (sc << 16) | da;
    o1 = A;
    o2 = B;
    return true;
  }
};

struct RandArgs {
  int32_t n, m, G;
  const int32_t* row_ptr;  // shared out-CSR shape
  const int32_t* col0;     // destinations of the source graph (CSR order)
  const uint64_t* seeds;   // G seeds
  uint64_t swaps;
  int32_t* col_out;        // G x m destinations after the swaps (rows unsorted)
  uint32_t* gscratch;      // per-graph state when it does not fit shared memory
};

__device__ __forceinline__ int row_of(const int32_t* row_ptr, int n, int e) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (row_ptr[mid] <= e) lo = mid; else hi = mid - 1;
  }
  return lo;
}

template <bool GM, int WN>
__global__ void __launch_bounds__(kRandThreads<WN>) k_randomize(RandArgs a) {
  extern __shared__ __align__(16) uint32_t rsm[];
  __shared__ RandWindow W;
  const int g = blockIdx.x;
  const int m = a.m, n = a.n;
  const RandLayout L = rand_layout(m);
  uint32_t* arcs = GM ? a.gscratch + (size_t)g * L.words : rsm;
  const BucketSet<GM> S{arcs + L.t_off, arcs + L.c_off, L.bb, (1u << L.bb) - 1u};
  for (size_t i = threadIdx.x; i < L.c_off - L.t_off; i += blockDim.x) S.t[i] = kEmpty;
  for (size_t i = threadIdx.x; i < L.words - L.c_off; i += blockDim.x) S.cnt[i] = 0;
  for (int e = threadIdx.x; e < m; e += blockDim.x)
    arcs[e] = ((uint32_t)row_of(a.row_ptr, n, e) << 16) | (uint32_t)a.col0[e];
  __syncthreads();
  for (int e = threadIdx.x; e < m; e += blockDim.x) S.insert(arcs[e]);
  __syncthreads();
  if (m > 0) {
    const ArcSwap pol{a.seeds[g], (uint64_t)m};
    run_attempts<WN>(pol, arcs, S, W, a.swaps);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < m; e += blockDim.x)
    a.col_out[(size_t)g * m + e] = (int32_t)(state_read<GM>(arcs + e) & 0xFFFFu);
}

// Dyad-preserving variant (swap mutual pairs and one-way arcs separately; the
// reading of the null model that keeps reciprocity): the arcs are split, in CSR
// order, into singles (u->v without v->u) and mutual dyads {u,v} (listed once,
// from the smaller end).  Attempt t takes SplitMix64 outputs 3t, 3t+1, 3t+2:
// the first picks the list (singles if floor(r*(S+D)/2^64) < S), the other two
// pick two entries; (a,b), (c,d) become (a,d), (c,b) unless the entries
// coincide, a == c, b == d, a == d, c == b, or a new pair is already adjacent in
// either direction.  The set holds the unordered adjacent pairs (min<<16|max).
struct DyadArgs {
  int32_t n, m, G;
  const int32_t* row_ptr;  // shared out-CSR shape (sorted rows)
  const int32_t* col0;
  const uint64_t* seeds;
  uint64_t attempts;
  int32_t* col_out;        // G x m destinations, rows unsorted
  int32_t* scratch;        // G x (2m + n + 2) ints
  uint32_t* gscratch;      // per-graph state when it does not fit shared memory
};

__device__ __forceinline__ bool has_arc(const int32_t* row_ptr, const int32_t* col, int a, int b) {
  int lo = row_ptr[a], hi = row_ptr[a + 1];
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    const int x = col[mid];
    if (x == b) return true;
    if (x < b) lo = mid + 1; else hi = mid;
  }
  return false;
}

__device__ __forceinline__ uint32_t pair_key(uint32_t u, uint32_t v) {
  return u < v ? (u << 16) | v : (v << 16) | u;
}

// Dyad-preserving swaps: attempt t takes SplitMix64 outputs 3t, 3t+1, 3t+2 (the
// list, then two entries of it); entries are (u << 16 | v) of the singles
// [0, S) and the mutual dyads [S, S + D), keys the unordered adjacent pairs.
struct DyadSwap {
  uint64_t seed, S, D;
  __device__ void draw(uint64_t t, uint32_t& e1, uint32_t& e2) const {
    const uint64_t gamma = 0x9E3779B97F4A7C15ull;
    const uint64_t r0 = sm64_mix(seed + (3 * t + 1) * gamma);
    const uint64_t r1 = sm64_mix(seed + (3 * t + 2) * gamma);
    const uint64_t r2 = sm64_mix(seed + (3 * t + 3) * gamma);
    const bool single = __umul64hi(r0, S + D) < S;
    const uint64_t len = single ? S : D;
    const uint32_t base_l = single ? 0u : (uint32_t)S;
    e1 = base_l + (uint32_t)__umul64hi(r1, len);
    e2 = base_l + (uint32_t)__umul64hi(r2, len);
  }
  __device__ bool make(uint32_t A, uint32_t B, uint32_t& k1, uint32_t& k2, uint32_t& o1,
                       uint32_t& o2, uint32_t& w1, uint32_t& w2) const {
    const uint32_t pa = A >> 16, pb = A & 0xFFFFu, pc = B >> 16, pd = B & 0xFFFFu;
    if (pa == pc || pb == pd || pa == pd || pc == pb) return false;
    k1 = pair_key(pa, pd);
    k2 = pair_key(pc, pb);
    o1 = pair_key(pa, pb);
    o2 = pair_key(pc, pd);
    w1 = (pa << 16) | pd;
    w2 = (pc << 16) | pb;
    return true;
  }
};

template <bool GM, int WN>
__global__ void __launch_bounds__(kRandThreads<WN>) k_randomize_dyads(DyadArgs a) {
  extern __shared__ __align__(16) uint32_t dsm[];
  __shared__ RandWindow W;
  __shared__ int scan_tmp[33];
  const int g = blockIdx.x;
  const int m = a.m, n = a.n;
  const RandLayout L = rand_layout(m);
  // singles [0, S), dyads [S, S + D)
  uint32_t* lists = GM ? a.gscratch + (size_t)g * L.words : dsm;
  const BucketSet<GM> Sset{lists + L.t_off, lists + L.c_off, L.bb, (1u << L.bb) - 1u};
  int32_t* fs = a.scratch + (size_t)g * (2 * (size_t)m + n + 2);
  int32_t* fd = fs + m + 1;
  int32_t* cur = fd + m + 1;
  for (size_t i = threadIdx.x; i < L.c_off - L.t_off; i += blockDim.x) Sset.t[i] = kEmpty;
  for (size_t i = threadIdx.x; i < L.words - L.c_off; i += blockDim.x) Sset.cnt[i] = 0;
  for (int v = threadIdx.x; v < n; v += blockDim.x) cur[v] = 0;
  // kinds of the arcs, in CSR order
  for (int e = threadIdx.x; e < m; e += blockDim.x) {
    const int v = row_of(a.row_ptr, n, e), u = a.col0[e];
    const bool rev = has_arc(a.row_ptr, a.col0, u, v);
    fs[e] = rev ? 0 : 1;
    fd[e] = (rev && v < u) ? 1 : 0;
  }
  if (threadIdx.x == 0) {
    fs[m] = 0;
    fd[m] = 0;
  }
  __syncthreads();
  const int S = (int)block_exclusive_scan(fs, m + 1, scan_tmp);
  const int D = (int)block_exclusive_scan(fd, m + 1, scan_tmp);
  for (int e = threadIdx.x; e < m; e += blockDim.x) {
    const bool single = fs[e + 1] != fs[e];
    const bool dyad = fd[e + 1] != fd[e];
    if (single || dyad) {
      const uint32_t v = (uint32_t)row_of(a.row_ptr, n, e), u = (uint32_t)a.col0[e];
      if (single) lists[fs[e]] = (v << 16) | u;
      else lists[S + fd[e]] = (v << 16) | u;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < S + D; i += blockDim.x)
    Sset.insert(pair_key(lists[i] >> 16, lists[i] & 0xFFFFu));
  __syncthreads();
  if (S + D > 0) {
    const DyadSwap pol{a.seeds[g], (uint64_t)S, (uint64_t)D};
    run_attempts<WN>(pol, lists, Sset, W, a.attempts);
  }
  __syncthreads();
  // arcs back into the rows of the fixed out-CSR shape (order inside a row is
  // arbitrary; the builder sorts)
  int32_t* out = a.col_out + (size_t)g * m;
  for (int i = threadIdx.x; i < S + D; i += blockDim.x) {
    const uint32_t x = state_read<GM>(lists + i);
    const int u = (int)(x >> 16), v = (int)(x & 0xFFFFu);
    out[a.row_ptr[u] + atomicAdd(&cur[u], 1)] = v;
    if (i >= S) out[a.row_ptr[v] + atomicAdd(&cur[v], 1)] = u;
  }
}

size_t dyad_scratch_ints(int32_t n, int32_t m) { return 2 * (size_t)m + (size_t)n + 2; }

// Shared memory of one graph's randomiser state, and whether it fits a block.
size_t rand_smem_bytes(int32_t m) { return rand_layout(m).words * 4; }

static bool rand_fits_smem(int32_t m) {
  int dev = 0, max_smem = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return rand_smem_bytes(m) <= (size_t)max_smem - sizeof(RandWindow) - 2048;
}

// Scratch (uint32 words) that G randomisations need when their state does not
// fit shared memory (0 when it does).
size_t rand_gscratch_words(int32_t m, int G) {
  return rand_fits_smem(m) ? 0 : (size_t)G * rand_layout(m).words;
}

template <typename Args>
static cudaError_t launch_rand(void (*narrow)(Args), void (*wide)(Args), void (*in_global)(Args),
                               Args& a, int32_t m, int G, uint32_t* gscratch, cudaStream_t s) {
  a.gscratch = gscratch;
  if (!rand_fits_smem(m)) {
    if (!gscratch) return cudaErrorInvalidValue;
    in_global<<<G, kRandThreads<64>, 0, s>>>(a);
    return cudaGetLastError();
  }
  void (*in_smem)(Args) = m < kWideArcs ? narrow : wide;
  const size_t smem = rand_smem_bytes(m);
  // the limit is the function's, shared by launches of other sizes: always the
  // largest this rule lets through
  int dev = 0, max_smem = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute((const void*)in_smem, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             max_smem - (int)sizeof(RandWindow) - 2048);
  if (e != cudaSuccess) return e;
  in_smem<<<G, m < kWideArcs ? kRandThreads<32> : kRandThreads<64>, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_randomize_dyads(int32_t n, int32_t m, int G, const int32_t* row_ptr,
                                   const int32_t* col0, const uint64_t* seeds, uint64_t attempts,
                                   int32_t* col_out, int32_t* scratch, uint32_t* gscratch,
                                   cudaStream_t s) {
  DyadArgs a;
  a.n = n; a.m = m; a.G = G;
  a.row_ptr = row_ptr; a.col0 = col0; a.seeds = seeds; a.attempts = attempts;
  a.col_out = col_out; a.scratch = scratch;
  return launch_rand(k_randomize_dyads<false, 32>, k_randomize_dyads<false, 64>,
                     k_randomize_dyads<true, 64>, a, m, G, gscratch, s);
}

// Enqueue G randomisations of the graph (row_ptr, col0) into col_out.
cudaError_t launch_randomize(int32_t n, int32_t m, int G, const int32_t* row_ptr,
                             const int32_t* col0, const uint64_t* seeds, uint64_t swaps,
                             int32_t* col_out, uint32_t* gscratch, cudaStream_t s) {
  RandArgs a;
  a.n = n; a.m = m; a.G = G;
  a.row_ptr = row_ptr; a.col0 = col0; a.seeds = seeds; a.swaps = swaps;
  a.col_out = col_out;
  return launch_rand(k_randomize<false, 32>, k_randomize<false, 64>, k_randomize<true, 64>, a, m, G, gscratch, s);
}

}  // namespace mt

using namespace mt;

extern "C" {

mt_status mt_randomize(const mt_graph* src, uint64_t seed, uint64_t swaps, void* stream,
                       mt_graph** out) {
  if (!src || !out) return MT_EINVAL;
  TraceRange tr("mt_randomize");
  cudaStream_t s = (cudaStream_t)stream;
  mt_graph* g = nullptr;
  MT_TRY(graph_alloc(src->n, src->m, s, &g));
  const size_t m1 = (size_t)(src->m > 0 ? src->m : 1);
  const size_t gwords = rand_gscratch_words(src->m, 1);
  char* scratch = nullptr;
  cudaError_t e = pool_alloc((void**)&scratch, m1 * 4 + 16 + gwords * 4 + 16, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(g->row_ptr, src->row_ptr, (3 * (size_t)src->n + 2) * 4,
                        cudaMemcpyDeviceToDevice, s);  // row_ptr, rank, off
  int32_t* col_tmp = (int32_t*)scratch;
  uint64_t* d_seed = (uint64_t*)(scratch + ((m1 * 4 + 15) & ~(size_t)15));
  uint32_t* gscr = gwords ? (uint32_t*)((char*)d_seed + 16) : nullptr;
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_seed, &seed, 8, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess)
    e = launch_randomize(src->n, src->m, 1, src->row_ptr, src->col, d_seed, swaps, col_tmp, gscr, s);
  if (e != cudaSuccess) {
    set_last_error(cudaGetErrorString(e));
    pool_free(scratch, s);
    graph_release(g, s);
    return MT_ECUDA;
  }
  mt_status st = graph_build_sync(g, col_tmp, true, s);
  pool_free(scratch, s);
  if (st != MT_OK) {
    graph_release(g, s);
    return st;
  }
  *out = g;
  return MT_OK;
}

mt_status mt_randomize_dyads(const mt_graph* src, uint64_t seed, uint64_t attempts, void* stream,
                             mt_graph** out) {
  if (!src || !out) return MT_EINVAL;
  TraceRange tr("mt_randomize_dyads");
  cudaStream_t s = (cudaStream_t)stream;
  mt_graph* g = nullptr;
  MT_TRY(graph_alloc(src->n, src->m, s, &g));
  const size_t m1 = (size_t)(src->m > 0 ? src->m : 1);
  const size_t sc = dyad_scratch_ints(src->n, src->m);
  const size_t gwords = rand_gscratch_words(src->m, 1);
  char* scratch = nullptr;
  cudaError_t e = pool_alloc((void**)&scratch, (m1 + sc) * 4 + 64 + gwords * 4 + 16, s);
  int32_t* col_tmp = (int32_t*)scratch;
  int32_t* dsc = col_tmp + m1;
  uint64_t* d_seed = (uint64_t*)(((uintptr_t)(dsc + sc) + 15) & ~(uintptr_t)15);
  uint32_t* gscr = gwords ? (uint32_t*)((char*)d_seed + 16) : nullptr;
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(g->row_ptr, src->row_ptr, (3 * (size_t)src->n + 2) * 4,
                        cudaMemcpyDeviceToDevice, s);  // row_ptr, rank, off
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_seed, &seed, 8, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess)
    e = launch_randomize_dyads(src->n, src->m, 1, src->row_ptr, src->col, d_seed, attempts,
                               col_tmp, dsc, gscr, s);
  if (e != cudaSuccess) {
    set_last_error(cudaGetErrorString(e));
    pool_free(scratch, s);
    graph_release(g, s);
    return MT_ECUDA;
  }
  mt_status st = graph_build_sync(g, col_tmp, true, s);
  pool_free(scratch, s);
  if (st != MT_OK) {
    graph_release(g, s);
    return st;
  }
  *out = g;
  return MT_OK;
}

}  // extern "C"
