// K1: the isomorphism table ISO of Sec. 3.2, built on the device.
//
// Keys are "extension-order keys": position p >= 1 of the enumerated vertex
// sequence owns the 2p bits starting at k(k-1) - p(p+1) (the last position
// lowest); inside them bits 2q / 2q+1 (q < p) say whether the arcs q->p /
// p->q exist.  For every key the builder
//  1. expands it to an 8x8 bit matrix (row i in byte i, column j in bit j),
//  2. walks all k! orderings of the vertices by adjacent transpositions
//     (Steinhaus-Johnson-Trotter order; each step swaps two neighbouring rows
//     and the same two columns) and keeps the numerically smallest matrix --
//     the order of the 8x8 values is the order of the canonical-layout masks,
//     because both lay the off-diagonal entries out row-major,
//  3. marks the key's own canonical-layout mask in a bitmap when it is its
//     own minimum and weakly connected.
// A popcount prefix over the bitmap then ranks the connected canonical masks
// (dense id = rank), and a last pass replaces each slot by the id of its
// canonical mask, or 0xFFFFFFFF for disconnected patterns.
//
// At k = 6 steps 2 and 3 run over the 9,608 x 2^10 keys whose first five
// vertices are in canonical order only, and the other rows of the table are
// permuted copies (see "k = 6 through its 5-vertex prefixes").
#include <algorithm>
#include <numeric>
#include <vector>

#include "graph.cuh"
#include "trace.cuh"

struct mt_table {
  int k = 0;
  uint32_t classes = 0;
  int device = 0;
  uint64_t nkeys = 0;
  uint32_t* table = nullptr;        // device, nkeys
  uint32_t* class_masks = nullptr;  // device, classes
  // compact k = 6 form (see build_compact6): `table` holds the slots of
  // (prefix class, relabelled words) instead of one slot per key
  bool compact = false;
  uint16_t* xclass = nullptr;       // device, 4096: prefix key -> class of the first 4 vertices
  uint8_t* xmap = nullptr;          // device, 4096 x 256: prefix key -> word relabelling
};

namespace mt {

__constant__ uint8_t c_sjt[6][120];  // per k <= 5: transposition positions p (swap p, p+1)

// Positions of the adjacent transpositions that take the identity through all
// k! permutations (Steinhaus-Johnson-Trotter with directions).
static std::vector<uint8_t> sjt_sequence(int k) {
  std::vector<int> perm(k), dir(k, -1);
  std::iota(perm.begin(), perm.end(), 0);
  std::vector<uint8_t> out;
  while (true) {
    int best = -1, bi = -1;
    for (int i = 0; i < k; ++i) {
      int j = i + dir[perm[i]];
      if (j < 0 || j >= k) continue;
      if (perm[j] < perm[i] && perm[i] > best) {
        best = perm[i];
        bi = i;
      }
    }
    if (bi < 0) break;
    int j = bi + dir[perm[bi]];
    out.push_back((uint8_t)std::min(bi, j));
    std::swap(perm[bi], perm[j]);
    for (int x = best + 1; x < k; ++x) dir[x] = -dir[x];
  }
  return out;
}

__device__ __forceinline__ uint64_t key_to_matrix(uint32_t key, int k) {
  uint64_t x = 0;
  for (int p = 1; p < k; ++p) {
    const int off = k * (k - 1) - p * (p + 1);
    for (int q = 0; q < p; ++q) {
      if ((key >> (off + 2 * q)) & 1u) x |= 1ull << (8 * q + p);      // q -> p
      if ((key >> (off + 2 * q + 1)) & 1u) x |= 1ull << (8 * p + q);  // p -> q
    }
  }
  return x;
}

__device__ __forceinline__ uint32_t matrix_to_mask(uint64_t x, int k) {
  uint32_t m = 0;
  for (int i = 0; i < k; ++i) {
    const uint32_t row = (uint32_t)(x >> (8 * i)) & 0xFFu;
    const uint32_t r = (row & ((1u << i) - 1u)) | ((row >> (i + 1)) << i);
    m |= r << (i * (k - 1));
  }
  return m;
}

__device__ __forceinline__ bool matrix_connected(uint64_t x, int k) {
  // undirected adjacency rows: a[i] = row i | column i
  uint32_t a[8];
  for (int i = 0; i < k; ++i) {
    uint32_t r = (uint32_t)(x >> (8 * i)) & 0xFFu;
    uint32_t c = 0;
    for (int j = 0; j < k; ++j) c |= (uint32_t)((x >> (8 * j + i)) & 1ull) << j;
    a[i] = r | c;
  }
  uint32_t seen = 1u, frontier = 1u;
  while (frontier) {
    uint32_t nxt = 0;
    for (int i = 0; i < k; ++i)
      if ((frontier >> i) & 1u) nxt |= a[i];
    nxt &= ~seen;
    seen |= nxt;
    frontier = nxt;
  }
  return seen == (1u << k) - 1u;
}

__device__ __forceinline__ uint64_t swap_adjacent(uint64_t x, int p) {
  // rows p and p+1 (bytes)
  uint64_t t = ((x >> (8 * p)) ^ (x >> (8 * p + 8))) & 0xFFull;
  x ^= (t << (8 * p)) | (t << (8 * p + 8));
  // columns p and p+1 (bits p, p+1 of every byte)
  t = ((x >> 1) ^ x) & (0x0101010101010101ull << p);
  x ^= t | (t << 1);
  return x;
}

template <int K>
__global__ void __launch_bounds__(256) k_canon(uint32_t* table, uint32_t* bitmap, uint64_t nkeys,
                                               int nsteps) {
  for (uint64_t key = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; key < nkeys;
       key += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t x0 = key_to_matrix((uint32_t)key, K);
    uint64_t x = x0, best = x0;
    for (int s = 0; s < nsteps; ++s) {
      x = swap_adjacent(x, c_sjt[K][s]);
      best = x < best ? x : best;
    }
    const uint32_t canon = matrix_to_mask(best, K);
    table[key] = canon;
    if (best == x0 && matrix_connected(x0, K))
      atomicOr(&bitmap[canon >> 5], 1u << (canon & 31u));
  }
}

// prefix[q] = number of set bits in the bitmap's 128-bit groups 0..q-1 (one
// uint4 each; a rank adds the group's own words); tile sums first.
constexpr int kScanThreads = 256, kScanPer = 16, kScanTile = kScanThreads * kScanPer;

__device__ __forceinline__ int popc4(uint4 v) {
  return __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
}

__global__ void k_tile_popc(const uint4* bitmap, size_t ngroups, int32_t* tile_sum) {
  __shared__ int red[kScanThreads / 32];
  const size_t base = (size_t)blockIdx.x * kScanTile;
  int s = 0;
  for (int i = 0; i < kScanPer; ++i) {
    size_t w = base + (size_t)i * kScanThreads + threadIdx.x;
    if (w < ngroups) s += popc4(bitmap[w]);
  }
  for (int d = 16; d; d >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, d);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int i = 0; i < kScanThreads / 32; ++i) t += red[i];
    tile_sum[blockIdx.x] = t;
  }
}

__global__ void __launch_bounds__(1024) k_scan_single(int32_t* data, int count) {
  __shared__ int tmp[33];
  block_exclusive_scan(data, count, tmp);
}

// A warp scans 32 consecutive groups at a time, so its reads and writes are
// coalesced; the tile's warps take the tile's slices in order.
__global__ void k_tile_prefix(const uint4* bitmap, size_t ngroups, const int32_t* tile_off,
                              int32_t* prefix) {
  constexpr int kWarps = kScanThreads / 32, kSlice = kScanTile / kWarps;
  __shared__ int wsum[kWarps];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const size_t base = (size_t)blockIdx.x * kScanTile + (size_t)wid * kSlice;
  int loc[kSlice / 32];
  int s = 0;
  for (int i = 0; i < kSlice / 32; ++i) {
    const size_t w = base + (size_t)i * 32 + lane;
    const int c = w < ngroups ? popc4(bitmap[w]) : 0;
    const int inc = warp_incl_scan(c);
    loc[i] = s + inc - c;
    s += __shfl_sync(0xFFFFFFFFu, inc, 31);
  }
  if (lane == 0) wsum[wid] = s;
  __syncthreads();
  int off = tile_off[blockIdx.x];
  for (int i = 0; i < wid; ++i) off += wsum[i];
  for (int i = 0; i < kSlice / 32; ++i) {
    const size_t w = base + (size_t)i * 32 + lane;
    if (w < ngroups) prefix[w] = off + loc[i];
  }
}

// Rank of bit c among the set bits, or kNoClass when it is not set.
__device__ __forceinline__ uint32_t rank_of(const uint4* bitmap, const int32_t* prefix,
                                            uint32_t c) {
  const uint4 v = bitmap[c >> 7];
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  const uint32_t at = (c >> 5) & 3u, bit = 1u << (c & 31u);
  uint32_t r = (uint32_t)prefix[c >> 7], own = 0;
#pragma unroll
  for (uint32_t i = 0; i < 4; ++i) {
    if (i < at) r += __popc(w[i]);
    if (i == at) own = w[i];
  }
  return (own & bit) ? r + __popc(own & (bit - 1u)) : kNoClass;
}

// table[key] = rank of the canonical mask that k_canon or k_sub_canon left there.
__global__ void k_assign(uint32_t* table, uint64_t nkeys, const uint4* bitmap,
                         const int32_t* prefix) {
  for (uint64_t key = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; key < nkeys;
       key += (uint64_t)gridDim.x * blockDim.x)
    table[key] = rank_of(bitmap, prefix, table[key]);
}

// The set bits of the bitmap in ascending order.
__global__ void k_bit_list(const uint4* bitmap, size_t ngroups, const int32_t* prefix,
                           uint32_t* out, uint32_t count) {
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < ngroups;
       q += (size_t)gridDim.x * blockDim.x) {
    const uint4 v = bitmap[q];
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t r = (uint32_t)prefix[q];
    for (int i = 0; i < 4; ++i)
      for (uint32_t bits = w[i]; bits; bits &= bits - 1u, ++r)
        if (r < count) out[r] = (uint32_t)(q * 128 + i * 32 + __ffs(bits) - 1);
  }
}

static cudaError_t launch_rank(const uint32_t* bitmap, size_t ngroups, int32_t* tiles,
                               int32_t* prefix, cudaStream_t s) {
  const unsigned ntiles = (unsigned)((ngroups + kScanTile - 1) / kScanTile);
  const uint4* bits = (const uint4*)bitmap;
  k_tile_popc<<<ntiles, kScanThreads, 0, s>>>(bits, ngroups, tiles);
  k_scan_single<<<1, 1024, 0, s>>>(tiles, (int)ntiles);
  k_tile_prefix<<<ntiles, kScanThreads, 0, s>>>(bits, ngroups, tiles, prefix);
  return cudaGetLastError();
}

// --------------------------------------------- k = 6 through its 5-vertex prefixes
//
// A 6-vertex key is a 5-vertex prefix X (key bits 10..29, itself a 5-vertex
// extension-order key) and the sixth vertex's word z (bits 0..9).  Relabelling
// X into the canonical order of its own class and z's fields with it leaves the
// class of the whole unchanged, so only 9,608 x 2^10 of the 2^30 keys (one
// prefix per 5-vertex digraph, connected or not) go through the k! orderings;
// every other row of 1,024 slots is one of theirs with its slots permuted.
// Measured on a GB300, table, count and read-out of one 800-vertex graph: 910
// ms with all 2^30 keys walked (893 ms of it k_canon<6>), 8.0 ms this way: 3.1
// of it allocating and freeing 4 GiB, 1.1 writing the table (3.8 TB/s), 1.25 the
// canonical masks, 1.1 the count.

constexpr int kP5Keys = 1 << 20;      // 5-vertex prefix keys
constexpr uint32_t kP5Classes = 9608; // 5-vertex digraphs up to isomorphism
constexpr int kP5Low = 10;            // bits of the sixth vertex's word

// For every prefix key: its canonical mask and the ordering sigma that reaches
// it (new position i holds old vertex sigma(i), 3 bits each); marks the
// canonical masks.
__global__ void __launch_bounds__(256) k_prefix5(uint32_t* canon, uint16_t* sigma,
                                                 uint32_t* bitmap, int nsteps) {
  const uint32_t xk = blockIdx.x * blockDim.x + threadIdx.x;
  if (xk >= (uint32_t)kP5Keys) return;
  const uint64_t x0 = key_to_matrix(xk, 5);
  uint64_t x = x0, best = x0;
  uint32_t at = 0 | (1 << 3) | (2 << 6) | (3 << 9) | (4 << 12), best_at = at;
  for (int s = 0; s < nsteps; ++s) {
    const int p = c_sjt[5][s];
    x = swap_adjacent(x, p);
    const uint32_t t = ((at >> (3 * p)) ^ (at >> (3 * p + 3))) & 7u;
    at ^= (t << (3 * p)) | (t << (3 * p + 3));
    if (x < best) {
      best = x;
      best_at = at;
    }
  }
  const uint32_t c = matrix_to_mask(best, 5);
  canon[xk] = c;
  sigma[xk] = (uint16_t)best_at;
  if (best == x0) atomicOr(&bitmap[c >> 5], 1u << (c & 31u));
}

// 5-vertex canonical mask -> the prefix key with that very matrix.
__device__ __forceinline__ uint32_t mask5_to_key(uint32_t mask) {
  uint32_t key = 0;
  for (int p = 1; p < 5; ++p)
    for (int q = 0; q < p; ++q) {
      const int off = 20 - p * (p + 1) + 2 * q;
      key |= ((mask >> (q * 4 + p - 1)) & 1u) << off;        // q -> p
      key |= ((mask >> (p * 4 + q)) & 1u) << (off + 1);      // p -> q
    }
  return key;
}

// Orderings that can reach a 6-vertex digraph's least mask.  The last vertex's
// row is the mask's highest, so the last vertex has the least out-degree d and
// its d successors come first: d! (5 - d)! orderings for each such vertex, 12 to
// 120 instead of 720.  Per d, the adjacent transpositions that walk S_d on
// positions 0..d-1 times S_(5-d) on positions d..4.
struct LastWalks {
  int32_t first[7];   // of d's transpositions in `at`; first[6] is the end
  uint8_t at[320];
};
__constant__ LastWalks c_last;

static LastWalks last_walks() {
  LastWalks w{};
  int n = 0;
  for (int d = 0; d <= 5; ++d) {
    w.first[d] = n;
    const std::vector<uint8_t> left = sjt_sequence(d), right = sjt_sequence(5 - d);
    for (size_t i = 0; i <= left.size(); ++i) {
      for (uint8_t p : right) w.at[n++] = (uint8_t)(d + p);
      if (i < left.size()) w.at[n++] = left[i];
    }
  }
  w.first[6] = n;
  return w;
}

// Canonical masks of the 6-vertex keys above the class prefixes (sub[class][z]);
// marks the connected ones.  Disconnected patterns get mask 0, which is not
// connected and so is never marked.  Bound by its integer operations: walking
// all 720 orderings took 7.5 ms, these take 1.25 ms.
__global__ void __launch_bounds__(256) k_sub_canon(uint32_t* sub, const uint32_t* masks5,
                                                   uint32_t* bitmap) {
  __shared__ LastWalks walks;
  for (int i = threadIdx.x; i < (int)sizeof(LastWalks) / 4; i += blockDim.x)
    ((uint32_t*)&walks)[i] = ((const uint32_t*)&c_last)[i];
  __syncthreads();
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (kP5Classes << kP5Low)) return;
  const uint32_t key =
      (mask5_to_key(masks5[i >> kP5Low]) << kP5Low) | (i & ((1u << kP5Low) - 1u));
  const uint64_t x0 = key_to_matrix(key, 6);
  uint32_t c = 0;
  if (matrix_connected(x0, 6)) {
    int d = 6;
    for (int v = 0; v < 6; ++v) d = min(d, __popc((uint32_t)(x0 >> (8 * v)) & 0xFFu));
    uint64_t best = ~0ull;
    for (int v = 0; v < 6; ++v) {
      const uint32_t succ = (uint32_t)(x0 >> (8 * v)) & 0xFFu;
      if (__popc(succ) != d) continue;
      // successors of v, the others, v: old vertex of each position, 4 bits each
      uint32_t at = (uint32_t)v << 20;
      int lo = 0, hi = d;
      for (int u = 0; u < 6; ++u)
        if (u != v) at |= (uint32_t)u << (4 * ((succ >> u) & 1u ? lo++ : hi++));
      uint64_t x = 0;
#pragma unroll
      for (int p = 0; p < 6; ++p) {
        const uint32_t row = (uint32_t)(x0 >> (8 * ((at >> (4 * p)) & 15u))) & 0xFFu;
        uint32_t r = 0;
#pragma unroll
        for (int q = 0; q < 6; ++q) r |= ((row >> ((at >> (4 * q)) & 15u)) & 1u) << q;
        x |= (uint64_t)r << (8 * p);
      }
      best = x < best ? x : best;
      for (int s = walks.first[d]; s < walks.first[d + 1]; ++s) {
        x = swap_adjacent(x, walks.at[s]);
        best = x < best ? x : best;
      }
    }
    c = matrix_to_mask(best, 6);
    const uint32_t bit = 1u << (c & 31u);
    // about six keys share a mask: most find the bit set
    if (!(*(volatile uint32_t*)&bitmap[c >> 5] & bit)) atomicOr(&bitmap[c >> 5], bit);
  }
  sub[i] = c;
}

// out[row * 1024 + z] = sub[class of the row's prefix][z relabelled]; row r's
// prefix key is r, or prefix_of[r >> 8] << 8 | (r & 255) for the compact form's
// rows.  One warp per row, four neighbouring slots per lane and store.
__global__ void __launch_bounds__(256) k_expand(uint32_t* __restrict__ out,
                                                const uint32_t* __restrict__ sub,
                                                const uint32_t* __restrict__ class5,
                                                const uint16_t* __restrict__ sigma,
                                                const int32_t* __restrict__ prefix_of,
                                                uint32_t nrows) {
  const int lane = threadIdx.x & 31;
  const uint32_t warps = gridDim.x * (blockDim.x >> 5);
  for (uint32_t r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < nrows; r += warps) {
    const uint32_t xk = prefix_of ? ((uint32_t)prefix_of[r >> 8] << 8) | (r & 255u) : r;
    const uint32_t* row = sub + ((size_t)class5[xk] << kP5Low);
    const uint32_t sg = sigma[xk];
    int to[5];  // where z's field q goes
#pragma unroll
    for (int q = 0; q < 5; ++q) to[q] = 0;
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
      for (int q = 0; q < 5; ++q)
        if (((sg >> (3 * i)) & 7u) == (uint32_t)q) to[q] = 2 * i;
    // z = step * 128 + lane * 4 + t: t is field 0, the lane fields 1, 2 and the
    // low bit of 3, the step the high bit of 3 and field 4
    const uint32_t zl = ((lane & 3u) << to[1]) | (((lane >> 2) & 3u) << to[2]) |
                        ((uint32_t)(lane >> 4) << to[3]);
    uint4* o = (uint4*)(out + ((size_t)r << kP5Low)) + lane;
#pragma unroll
    for (int step = 0; step < 8; ++step) {
      const uint32_t z = zl | ((uint32_t)(step & 1) << (to[3] + 1)) |
                         ((uint32_t)(step >> 1) << to[4]);
      uint4 v;
      v.x = __ldg(row + z);
      v.y = __ldg(row + (z | (1u << to[0])));
      v.z = __ldg(row + (z | (2u << to[0])));
      v.w = __ldg(row + (z | (3u << to[0])));
      o[step * 32] = v;
    }
  }
}

// Upload k's transposition sequence (always the same bytes), after checking that
// the walk visits every ordering exactly once.
static mt_status upload_sjt(int k, cudaStream_t s, int* nsteps) {
  const std::vector<uint8_t> seq = sjt_sequence(k);
  std::vector<uint32_t> seen;
  uint32_t p = 0x543210u & ((1u << (4 * k)) - 1u);  // 4 bits per position
  seen.push_back(p);
  for (uint8_t q : seq) {
    const uint32_t t = ((p >> (4 * q)) ^ (p >> (4 * q + 4))) & 15u;
    p ^= (t << (4 * q)) | (t << (4 * q + 4));
    seen.push_back(p);
  }
  std::sort(seen.begin(), seen.end());
  size_t fact = 1;
  for (int i = 2; i <= k; ++i) fact *= i;
  if (seq.size() + 1 != fact || std::unique(seen.begin(), seen.end()) != seen.end())
    return MT_ECUDA;
  MT_CUDA_TRY(cudaMemcpyToSymbolAsync(c_sjt, seq.data(), seq.size(), (size_t)k * 120,
                                      cudaMemcpyHostToDevice, s));
  *nsteps = (int)seq.size();
  return MT_OK;
}

static int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// Scratch of one build, one stream-ordered allocation.
struct TableScratch {
  char* mem = nullptr;
  size_t off = 0, bytes = 0;
  uint32_t *bitmap = nullptr, *bitmap5 = nullptr;  // connected 6- (or k-), 5-vertex masks
  size_t ngroups = 0, ngroups5 = 0, zeroed = 0;
  int32_t *prefix = nullptr, *prefix5 = nullptr, *tiles = nullptr;
  uint32_t *sub = nullptr, *class5 = nullptr, *masks5 = nullptr;
  uint16_t* sigma = nullptr;
  int32_t* reps = nullptr;  // compact form: representative 4-vertex prefix keys
};

static cudaError_t scratch_alloc(TableScratch* x, int k, cudaStream_t s) {
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off += (bytes + 255) & ~(size_t)255;
    return o;
  };
  x->ngroups = (size_t)std::max<uint64_t>((1ull << (k * (k - 1))) / 128, 1);
  x->ngroups5 = k == 6 ? kP5Keys / 128 : 0;
  const size_t tiles = (x->ngroups + kScanTile - 1) / kScanTile;
  const size_t o_b = take(x->ngroups * 16), o_b5 = take(x->ngroups5 * 16);
  x->zeroed = off;
  const size_t o_p = take(x->ngroups * 4), o_p5 = take(x->ngroups5 * 4), o_t = take(tiles * 4);
  const size_t o_s = take(k == 6 ? ((size_t)kP5Classes << kP5Low) * 4 : 0);
  const size_t o_c = take(k == 6 ? (size_t)kP5Keys * 4 : 0);
  const size_t o_m = take(k == 6 ? (size_t)kP5Classes * 4 : 0);
  const size_t o_g = take(k == 6 ? (size_t)kP5Keys * 2 : 0);
  const size_t o_r = take(k == 6 ? 256 * 4 : 0);
  cudaError_t e = pool_alloc((void**)&x->mem, off, s);
  if (e != cudaSuccess) return e;
  x->bitmap = (uint32_t*)(x->mem + o_b);
  x->bitmap5 = (uint32_t*)(x->mem + o_b5);
  x->prefix = (int32_t*)(x->mem + o_p);
  x->prefix5 = (int32_t*)(x->mem + o_p5);
  x->tiles = (int32_t*)(x->mem + o_t);
  x->sub = (uint32_t*)(x->mem + o_s);
  x->class5 = (uint32_t*)(x->mem + o_c);
  x->masks5 = (uint32_t*)(x->mem + o_m);
  x->sigma = (uint16_t*)(x->mem + o_g);
  x->reps = (int32_t*)(x->mem + o_r);
  return cudaMemsetAsync(x->mem, 0, x->zeroed, s);
}

// The 5-vertex classes and the dense ids above them (x->sub, x->class5,
// x->sigma), and the class list.
static cudaError_t launch_sub6(const TableScratch& x, uint32_t* class_masks, int nsteps5, int sms,
                               cudaStream_t s) {
  const LastWalks walks = last_walks();
  cudaError_t e = cudaMemcpyToSymbolAsync(c_last, &walks, sizeof(walks), 0, cudaMemcpyHostToDevice,
                                          s);
  if (e != cudaSuccess) return e;
  k_prefix5<<<kP5Keys / 256, 256, 0, s>>>(x.class5, x.sigma, x.bitmap5, nsteps5);
  e = launch_rank(x.bitmap5, x.ngroups5, x.tiles, x.prefix5, s);
  if (e != cudaSuccess) return e;
  const uint4* b5 = (const uint4*)x.bitmap5;
  const uint4* b6 = (const uint4*)x.bitmap;
  k_bit_list<<<32, 256, 0, s>>>(b5, x.ngroups5, x.prefix5, x.masks5, kP5Classes);
  k_assign<<<sms * 8, 256, 0, s>>>(x.class5, kP5Keys, b5, x.prefix5);
  const uint32_t nsub = kP5Classes << kP5Low;
  k_sub_canon<<<(nsub + 255) / 256, 256, 0, s>>>(x.sub, x.masks5, x.bitmap);
  e = launch_rank(x.bitmap, x.ngroups, x.tiles, x.prefix, s);
  if (e != cudaSuccess) return e;
  k_assign<<<sms * 16, 256, 0, s>>>(x.sub, nsub, b6, x.prefix);
  k_bit_list<<<sms * 8, 256, 0, s>>>(b6, x.ngroups, x.prefix, class_masks, kNumClasses[6]);
  return cudaGetLastError();
}

// Number of set bits of a ranked bitmap, read back to `out[0..4]` (prefix of
// the last group, then its words).
static cudaError_t read_total(const uint32_t* bitmap, const int32_t* prefix, size_t ngroups,
                              uint32_t* out, cudaStream_t s) {
  cudaError_t e = cudaMemcpyAsync(out, prefix + ngroups - 1, 4, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(out + 1, bitmap + 4 * (ngroups - 1), 16, cudaMemcpyDeviceToHost, s);
  return e;
}
static uint32_t total_of(const uint32_t* r) {
  uint32_t t = r[0];
  for (int i = 1; i < 5; ++i) t += (uint32_t)__builtin_popcount(r[i]);
  return t;
}

static void table_drop(mt_table* t) {
  if (t->table) cudaFree(t->table);
  if (t->class_masks) cudaFree(t->class_masks);
  if (t->xclass) cudaFree(t->xclass);
  if (t->xmap) cudaFree(t->xmap);
  delete t;
}

static mt_status table_done(mt_table* t, mt_table** out) {
  cudaGetDevice(&t->device);
  handle_born(t->device);
  *out = t;
  return MT_OK;
}

static mt_status build_table(int k, cudaStream_t s, mt_table** out) {
  const uint64_t nkeys = 1ull << (k * (k - 1));
  int nsteps = 0;  // k = 6 walks the orderings of its 5-vertex prefixes
  MT_TRY(upload_sjt(std::min(k, 5), s, &nsteps));
  mt_table* t = new mt_table();
  t->k = k;
  t->nkeys = nkeys;
  t->classes = kNumClasses[k];
  TableScratch x;
  cudaError_t e = cudaMalloc(&t->table, nkeys * 4);
  if (e == cudaSuccess) e = cudaMalloc(&t->class_masks, (size_t)t->classes * 4);
  if (e == cudaSuccess) e = scratch_alloc(&x, k, s);
  if (e == cudaSuccess) {
    const int sms = sm_count();
    const int grid = (int)std::min<uint64_t>((nkeys + 255) / 256, (uint64_t)sms * 16);
    if (k == 6) {
      e = launch_sub6(x, t->class_masks, nsteps, sms, s);
      if (e == cudaSuccess)
        k_expand<<<sms * 8, 256, 0, s>>>(t->table, x.sub, x.class5, x.sigma, nullptr, kP5Keys);
    } else {
      switch (k) {
        case 3: k_canon<3><<<grid, 256, 0, s>>>(t->table, x.bitmap, nkeys, nsteps); break;
        case 4: k_canon<4><<<grid, 256, 0, s>>>(t->table, x.bitmap, nkeys, nsteps); break;
        default: k_canon<5><<<grid, 256, 0, s>>>(t->table, x.bitmap, nkeys, nsteps); break;
      }
      e = launch_rank(x.bitmap, x.ngroups, x.tiles, x.prefix, s);
      const uint4* bits = (const uint4*)x.bitmap;
      k_assign<<<grid, 256, 0, s>>>(t->table, nkeys, bits, x.prefix);
      k_bit_list<<<(unsigned)((x.ngroups + 255) / 256), 256, 0, s>>>(
          bits, x.ngroups, x.prefix, t->class_masks, t->classes);
    }
    if (e == cudaSuccess) e = cudaGetLastError();
  }
  // the numbers of canonical masks must equal the closed-form counts
  uint32_t got[5] = {0}, got5[5] = {0};
  if (e == cudaSuccess) e = read_total(x.bitmap, x.prefix, x.ngroups, got, s);
  if (e == cudaSuccess && k == 6) e = read_total(x.bitmap5, x.prefix5, x.ngroups5, got5, s);
  pool_free(x.mem, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    set_last_error(cudaGetErrorString(e));
    table_drop(t);
    return e == cudaErrorMemoryAllocation ? MT_ENOMEM : MT_ECUDA;
  }
  if (total_of(got) != t->classes || (k == 6 && total_of(got5) != kP5Classes)) {
    set_last_error("table builder found " + std::to_string(total_of(got)) + " classes");
    table_drop(t);
    return MT_ECUDA;
  }
  return table_done(t, out);
}

// ---------------------------------------------------------- compact k = 6 form
//
// The k = 6 table has 2^30 slots (4 GiB), but a key is three parts: the first
// four vertices X (positions 0..3, 12 key bits), the fifth vertex's word y (8
// bits) and the sixth's z (10 bits).  Relabelling X into a canonical order of
// its own (one of the 199 weakly connected 4-vertex classes; X is connected in
// every enumerated set) and the words with it leaves the class of the whole
// unchanged, so a table indexed by (class of X, relabelled y, relabelled z)
// holds every class: 199 x 2^18 slots (208 MB).  Per prefix key it needs the
// class of X and the relabelling of an 8-bit word (4 two-bit fields, one per
// vertex of X); the sixth vertex's field for the fifth vertex is not moved.

constexpr int kXKeys = 1 << 12;          // prefix keys (positions 1..3 of a 6-vertex key)
constexpr int kXClasses = 199;           // weakly connected 4-vertex classes
constexpr int kXLow = 18;                // bits of y and z in a 6-vertex key

// The 4-vertex prefix of a 6-vertex key, as an 8x8 bit matrix.
__device__ __forceinline__ uint64_t xkey_matrix(uint32_t xk) { return key_to_matrix(xk << kXLow, 6); }

// For every prefix key: the smallest 4-vertex canonical-layout mask over the 24
// orderings sigma (new position i holds old vertex sigma(i)), the ordering that
// reaches it, and whether X is weakly connected.  Marks the connected minima.
__global__ void k_xprefix(uint16_t* xcanon, uint8_t* xsigma, uint32_t* xbits, int32_t* xrep) {
  const int xk = blockIdx.x * blockDim.x + threadIdx.x;
  if (xk >= kXKeys) return;
  const uint64_t x0 = xkey_matrix((uint32_t)xk);
  uint32_t best = 0xFFFFFFFFu, best_sigma = 0;
  for (int c = 0; c < 24; ++c) {
    // the c-th ordering of 4 vertices (factorial number system)
    int avail[4] = {0, 1, 2, 3}, sig[4];
    int r = c;
    for (int i = 0, f = 6; i < 4; ++i) {
      const int d = r / f;
      r %= f;
      sig[i] = avail[d];
      for (int j = d; j < 3 - i; ++j) avail[j] = avail[j + 1];
      f = i < 3 ? f / (3 - i) : 1;
    }
    uint64_t y = 0;
    for (int i = 0; i < 4; ++i)
      for (int j = 0; j < 4; ++j)
        if ((x0 >> (8 * sig[i] + sig[j])) & 1ull) y |= 1ull << (8 * i + j);
    const uint32_t mask = matrix_to_mask(y, 4);
    if (mask < best) {
      best = mask;
      best_sigma = (uint32_t)(sig[0] | (sig[1] << 2) | (sig[2] << 4) | (sig[3] << 6));
    }
  }
  xcanon[xk] = (uint16_t)best;
  xsigma[xk] = (uint8_t)best_sigma;
  const bool conn = matrix_connected(x0, 4);
  if (conn) atomicOr(&xbits[best >> 5], 1u << (best & 31u));
  // the prefix key whose own matrix is the canonical one represents the class
  if (conn && matrix_to_mask(x0, 4) == best) xrep[best] = xk;
}

// Class of each prefix key (rank of its canonical mask among the connected
// ones; 0xFFFF if X is disconnected) and the relabelling of all 256 words.
__global__ void k_xtables(const uint16_t* xcanon, const uint8_t* xsigma, const uint32_t* xbits,
                          uint16_t* xclass, uint8_t* xmap) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= kXKeys * 256) return;
  const int xk = t >> 8, w = t & 255;
  const uint32_t sg = xsigma[xk];
  uint32_t out = 0;
  for (int i = 0; i < 4; ++i) out |= ((w >> (2 * ((sg >> (2 * i)) & 3u))) & 3u) << (2 * i);
  xmap[t] = (uint8_t)out;
  if (w == 0) {
    const uint32_t c = xcanon[xk];
    const bool conn = matrix_connected(xkey_matrix((uint32_t)xk), 4);
    uint32_t rank = 0;
    for (uint32_t q = 0; q < (c >> 5); ++q) rank += __popc(xbits[q]);
    rank += __popc(xbits[c >> 5] & ((1u << (c & 31u)) - 1u));
    xclass[xk] = conn ? (uint16_t)rank : (uint16_t)0xFFFFu;
  }
}

// Representative prefix key of each class, in class order.
__global__ void k_xreps(const uint32_t* xbits, const int32_t* xrep, int32_t* reps) {
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  int r = 0;
  for (uint32_t c = 0; c < kXKeys && r < kXClasses; ++c)
    if ((xbits[c >> 5] >> (c & 31u)) & 1u) reps[r++] = xrep[c];
}

static mt_status build_compact6(cudaStream_t s, mt_table** out) {
  int nsteps5 = 0;
  MT_TRY(upload_sjt(5, s, &nsteps5));
  mt_table* t = new mt_table();
  t->k = 6;
  t->classes = kNumClasses[6];
  t->compact = true;
  t->nkeys = (uint64_t)kXClasses << kXLow;
  TableScratch x;
  uint16_t* xcanon = nullptr;
  uint8_t* xsigma = nullptr;
  uint32_t* xbits = nullptr;
  int32_t* xrep = nullptr;
  cudaError_t e = cudaMalloc(&t->table, t->nkeys * 4);
  if (e == cudaSuccess) e = cudaMalloc(&t->class_masks, (size_t)t->classes * 4);
  if (e == cudaSuccess) e = cudaMalloc(&t->xclass, kXKeys * 2);
  if (e == cudaSuccess) e = cudaMalloc(&t->xmap, kXKeys * 256);
  if (e == cudaSuccess) e = scratch_alloc(&x, 6, s);
  if (e == cudaSuccess) e = cudaMallocAsync(&xcanon, kXKeys * 2, s);
  if (e == cudaSuccess) e = cudaMallocAsync(&xsigma, kXKeys, s);
  if (e == cudaSuccess) e = cudaMallocAsync(&xbits, kXKeys / 8, s);
  if (e == cudaSuccess) e = cudaMallocAsync(&xrep, kXKeys * 4, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(xbits, 0, kXKeys / 8, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(x.reps, 0, kXClasses * 4, s);
  int32_t nreps = 0;
  if (e == cudaSuccess) {
    const int sms = sm_count();
    e = launch_sub6(x, t->class_masks, nsteps5, sms, s);
    k_xprefix<<<kXKeys / 256, 256, 0, s>>>(xcanon, xsigma, xbits, xrep);
    k_xtables<<<kXKeys, 256, 0, s>>>(xcanon, xsigma, xbits, t->xclass, t->xmap);
    k_xreps<<<1, 32, 0, s>>>(xbits, xrep, x.reps);
    if (e == cudaSuccess)
      k_expand<<<sms * 8, 256, 0, s>>>(t->table, x.sub, x.class5, x.sigma, x.reps,
                                       (uint32_t)kXClasses << (kXLow - kP5Low));
    if (e == cudaSuccess) e = cudaGetLastError();
  }
  // the numbers of classes: connected 4-vertex, all 5-vertex, connected 6-vertex
  uint32_t got[5] = {0}, got5[5] = {0};
  std::vector<uint32_t> hb(kXKeys / 32);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(hb.data(), xbits, kXKeys / 8, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = read_total(x.bitmap, x.prefix, x.ngroups, got, s);
  if (e == cudaSuccess) e = read_total(x.bitmap5, x.prefix5, x.ngroups5, got5, s);
  if (xcanon) cudaFreeAsync(xcanon, s);
  if (xsigma) cudaFreeAsync(xsigma, s);
  if (xbits) cudaFreeAsync(xbits, s);
  if (xrep) cudaFreeAsync(xrep, s);
  pool_free(x.mem, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  for (uint32_t w : hb) nreps += __builtin_popcount(w);
  if (e != cudaSuccess) {
    set_last_error(cudaGetErrorString(e));
    table_drop(t);
    return e == cudaErrorMemoryAllocation ? MT_ENOMEM : MT_ECUDA;
  }
  if (nreps != kXClasses || total_of(got) != t->classes || total_of(got5) != kP5Classes) {
    set_last_error("compact table: " + std::to_string(nreps) + " prefix classes, " +
                   std::to_string(total_of(got)) + " classes");
    table_drop(t);
    return MT_ECUDA;
  }
  return table_done(t, out);
}

TableView table_view(const mt_table* t) {
  TableView v;
  v.slots = t->table;
  v.xclass = t->compact ? t->xclass : nullptr;
  v.xmap = t->compact ? t->xmap : nullptr;
  return v;
}
bool table_compact(const mt_table* t) { return t->compact; }

int table_k(const mt_table* t) { return t->k; }
uint32_t table_classes(const mt_table* t) { return t->classes; }

}  // namespace mt

using namespace mt;

extern "C" {

mt_status mt_table_build(int k, void* stream, mt_table** out) {
  if (!out) return MT_EINVAL;
  if (k < 3 || k > 6) return MT_EUNSUPPORTED;
  TraceRange tr("mt_table_build");
  return build_table(k, (cudaStream_t)stream, out);
}

mt_status mt_table_build_compact(int k, void* stream, mt_table** out) {
  if (!out) return MT_EINVAL;
  if (k != 6) return MT_EUNSUPPORTED;
  TraceRange tr("mt_table_build_compact");
  return build_compact6((cudaStream_t)stream, out);
}

mt_status mt_table_is_compact(const mt_table* t, int* compact) {
  if (!t || !compact) return MT_EINVAL;
  *compact = t->compact ? 1 : 0;
  return MT_OK;
}

mt_status mt_table_free(mt_table* t) {
  if (!t) return MT_OK;
  const int device = t->device;
  DeviceScope on(device);
  cudaDeviceSynchronize();
  table_drop(t);
  handle_died(device);
  return MT_OK;
}

mt_status mt_table_k(const mt_table* t, int* k) {
  if (!t || !k) return MT_EINVAL;
  *k = t->k;
  return MT_OK;
}

mt_status mt_table_num_classes(const mt_table* t, uint32_t* out) {
  if (!t || !out) return MT_EINVAL;
  *out = t->classes;
  return MT_OK;
}

mt_status mt_table_class_masks(const mt_table* t, uint32_t* masks) {
  if (!t || !masks) return MT_EINVAL;
  MT_CUDA_TRY(cudaMemcpy(masks, t->class_masks, (size_t)t->classes * 4, cudaMemcpyDeviceToHost));
  return MT_OK;
}

mt_status mt_table_entries(const mt_table* t, uint64_t first, uint64_t count, uint32_t* ids) {
  if (!t || (!ids && count)) return MT_EINVAL;
  if (first > t->nkeys || count > t->nkeys - first) return MT_EINVAL;
  if (count == 0) return MT_OK;
  MT_CUDA_TRY(cudaMemcpy(ids, t->table + first, count * 4, cudaMemcpyDeviceToHost));
  return MT_OK;
}

}  // extern "C"
