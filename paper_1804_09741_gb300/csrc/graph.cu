// Graph loading and the device graph builder.
//
// The undirected neighbour CSR of Sec. 2 (for each vertex v the sorted set
// delta(v) = A(v) u B(v) u C(v), each entry tagged with which of the arcs v->u,
// u->v exist) is built from a directed out-CSR whose rows may be unsorted, in
// four launches over all graphs of a batch:
//  * every arc puts an entry into its tail's and its head's row (k_scatter; the
//    rows' places are prefix sums of in + out degree);
//  * a warp sorts a row and merges the two entries of a mutual pair (k_rows);
//  * one block per graph adds up the rows' lengths (k_lengths);
//  * a warp moves a row to its place and notes the row vertex of each entry and
//    the index of the first neighbour larger than the row's (k_place).
// The vertices are numbered by `rank` in it.  The counting kernels own a set by
// its smallest number; the directed CSR keeps the original numbers.
//
// One block per graph, a thread per vertex or arc with a scan of its whole row,
// took 1,254 us for one graph of n = 20,000, m = 120,000, and 95 us for n =
// 2,000, m = 8,000, on latency alone; these launches take
// 85 us and 30 us.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>

#include "graph.cuh"
#include "trace.cuh"

namespace mt {

namespace {
thread_local std::string g_last_error;
}

void set_last_error(const std::string& s) { g_last_error = s; }

// ------------------------------------------------------------------ builder

constexpr unsigned kAll = 0xFFFFFFFFu;

__device__ __forceinline__ int row_of(const int32_t* row_ptr, int n, int e) {
  // largest v with row_ptr[v] <= e (rows may be empty)
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (row_ptr[mid] <= e) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__global__ void __launch_bounds__(256) k_scatter(BuildArgs a) {
  const size_t g = blockIdx.y;
  const int32_t* col = a.col_in + g * a.m;
  int32_t* cursor = a.cursor + g * a.n;
  uint32_t* tmp = a.tmp + g * 2 * a.m;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < a.m; e += gridDim.x * blockDim.x) {
    const int x = __ldg(&a.rank[row_of(a.row_ptr, a.n, e)]), y = __ldg(&a.rank[col[e]]);
    if (x == y) atomicOr(&a.stats[g].err, kErrSelfLoop);
    tmp[__ldg(&a.off[x]) + atomicAdd(&cursor[x], 1)] = (uint32_t)y | (1u << 30);  // x -> y
    tmp[__ldg(&a.off[y]) + atomicAdd(&cursor[y], 1)] = (uint32_t)x | (1u << 31);  // y <- x
  }
}

// Sort a row of d packed entries in place by vertex, entries of one vertex
// merged (their code bits or-ed); returns the number left.  `dup` is set when one
// code bit appears twice.  Up to 32 entries sit in the lanes' registers and
// count the smaller ones; longer rows go through two bitmaps of the vertices
// (`bits`, 2 x words, all zero before and after), one per direction.
__device__ __forceinline__ int sort_row(uint32_t* row, int d, uint32_t* bits, int words, int lane,
                                        bool& dup) {
  if (d <= 32) {
    const uint32_t x = lane < d ? row[lane] : 0xFFFFFFFFu;
    const uint32_t id = x & kVertexMask;
    uint32_t code = x >> 30;
    unsigned less = 0;
    bool first = lane < d;
    for (int i = 0; i < d; ++i) {
      const uint32_t y = __shfl_sync(kAll, x, i), yid = y & kVertexMask;
      if (yid < id) less |= 1u << i;
      if (yid == id && i != lane && lane < d) {
        dup |= (code & (y >> 30)) != 0;
        if (i < lane) first = false;
        code |= y >> 30;
      }
    }
    const unsigned firsts = __ballot_sync(kAll, first);
    __syncwarp();
    if (first) row[__popc(less & firsts)] = id | (code << 30);
    return __popc(firsts);
  }
  for (int i = lane; i < d; i += 32) {
    const uint32_t x = row[i], id = x & kVertexMask;
    for (int q = 0; q < 2; ++q)
      if ((x >> (30 + q)) & 1u)
        dup |= (atomicOr(&bits[q * words + (id >> 5)], 1u << (id & 31u)) >> (id & 31u)) & 1u;
  }
  __syncwarp();
  int at = 0;
  for (int w0 = 0; w0 < words; w0 += 32) {
    const int w = w0 + lane;
    uint32_t b0 = 0, b1 = 0;
    if (w < words) {
      b0 = bits[w];
      b1 = bits[words + w];
      bits[w] = bits[words + w] = 0;
    }
    const int c = __popc(b0 | b1);
    const int incl = warp_incl_scan(c);
    int pos = at + incl - c;
    for (uint32_t left = b0 | b1; left; left &= left - 1) {
      const int i = __ffs(left) - 1;
      row[pos++] = (uint32_t)(32 * w + i) | (((b0 >> i) & 1u) << 30) | (((b1 >> i) & 1u) << 31);
    }
    at += __shfl_sync(kAll, incl, 31);
  }
  __syncwarp();
  return at;
}

// Shared memory of one warp's bitmaps.
static __host__ __device__ int bitmap_words(int n) { return (n + 31) / 32; }

__global__ void k_rows(BuildArgs a) {
  extern __shared__ uint32_t sbits[];
  const size_t g = blockIdx.y;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int words = bitmap_words(a.n);
  uint32_t* bits = sbits + (size_t)wid * 2 * words;
  for (int i = lane; i < 2 * words; i += 32) bits[i] = 0;
  __syncwarp();
  bool dup = false;
  // neighbouring rows (of similar length, longest first) in different blocks
  for (int v = wid * (int)gridDim.x + (int)blockIdx.x; v < a.n; v += nw * (int)gridDim.x) {
    const int o = __ldg(&a.off[v]);
    const int c = sort_row(a.tmp + g * 2 * a.m + o, __ldg(&a.off[v + 1]) - o, bits, words, lane, dup);
    if (lane == 0) a.urow[g * (a.n + 1) + v] = c;
  }
  if (dup) atomicOr(&a.stats[g].err, kErrDuplicateArc);
}

__global__ void __launch_bounds__(1024) k_lengths(BuildArgs a) {
  __shared__ int scan_tmp[33];
  __shared__ int s_dmax;
  const size_t g = blockIdx.x;
  int32_t* urow = a.urow + g * (a.n + 1);
  if (threadIdx.x == 0) {
    s_dmax = 0;
    urow[a.n] = 0;
  }
  __syncthreads();
  int most = 0;
#pragma unroll 8
  for (int v = threadIdx.x; v < a.n; v += blockDim.x) most = max(most, urow[v]);
  most = __reduce_max_sync(kAll, most);
  if ((threadIdx.x & 31) == 0) atomicMax(&s_dmax, most);
  __syncthreads();
  const long long nu = block_exclusive_scan(urow, a.n + 1, scan_tmp);
  if (threadIdx.x == 0) {
    a.stats[g].nu = (int32_t)nu;
    a.stats[g].dmax = s_dmax;
  }
}

__global__ void __launch_bounds__(256) k_place(BuildArgs a) {
  const size_t g = blockIdx.y;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int32_t* urow = a.urow + g * (a.n + 1);
  uint32_t* ucol = a.ucol + g * 2 * a.m;
  int32_t* usrc = a.usrc + g * 2 * a.m;
  for (int v = wid * (int)gridDim.x + (int)blockIdx.x; v < a.n; v += nw * (int)gridDim.x) {
    const uint32_t* row = a.tmp + g * 2 * a.m + __ldg(&a.off[v]);
    const int u0 = urow[v], d = urow[v + 1] - u0;
    int below = 0;
    for (int i = lane; i < d; i += 32) {
      const uint32_t x = row[i];
      ucol[u0 + i] = x;
      usrc[u0 + i] = v;
      below += (int)(x & kVertexMask) < v;
    }
    below = __reduce_add_sync(kAll, below);
    if (lane == 0) a.ufwd[g * a.n + v] = below;
  }
}

// The launches' y dimension is the graph, of which a grid has at most 65,535.
constexpr int kGridGraphs = 65535;

cudaError_t launch_build(const BuildArgs& all, cudaStream_t s) {
  if (all.G <= 0) return cudaSuccess;
  cudaError_t e = cudaMemsetAsync(all.cursor, 0, (size_t)all.G * all.n * 4, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(all.stats, 0, (size_t)all.G * sizeof(BuildStats), s);
  // 8 warps of bitmaps, 4 for graphs of more than 48,000 vertices
  const size_t per_warp = (size_t)bitmap_words(all.n) * 8;
  const int warps = per_warp * 8 > 96 * 1024 ? 4 : 8;
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute((const void*)k_rows, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             96 * 1024);
  if (e != cudaSuccess) return e;
  for (int g0 = 0; g0 < all.G; g0 += kGridGraphs) {
    BuildArgs a = all;
    a.G = std::min(all.G - g0, kGridGraphs);
    const size_t n0 = (size_t)g0 * a.n, m0 = (size_t)g0 * a.m;
    a.col_in += m0;
    a.tmp += 2 * m0;
    a.cursor += n0;
    a.urow += n0 + g0;
    a.ucol += 2 * m0;
    a.usrc += 2 * m0;
    a.ufwd += n0;
    a.stats += g0;
    const int most = std::max(1, 8192 / a.G);  // blocks per graph
    if (a.m > 0) k_scatter<<<dim3(std::min((a.m + 255) / 256, most), a.G), 256, 0, s>>>(a);
    k_rows<<<dim3(std::min((a.n + warps - 1) / warps, most), a.G), warps * 32, per_warp * warps,
             s>>>(a);
    k_lengths<<<a.G, 1024, 0, s>>>(a);
    k_place<<<dim3(std::min((a.n + 7) / 8, most), a.G), 256, 0, s>>>(a);
  }
  return cudaGetLastError();
}

// Sorted rows of a directed CSR.  Duplicate arcs are left to k_rows.
__global__ void k_sort_cols(int n, const int32_t* __restrict__ row_ptr,
                            const int32_t* __restrict__ in, int32_t* out) {
  extern __shared__ uint32_t sbits[];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int words = bitmap_words(n);
  uint32_t* bits = sbits + (size_t)wid * 2 * words;
  for (int i = lane; i < 2 * words; i += 32) bits[i] = 0;
  __syncwarp();
  bool dup = false;
  for (int v = wid * (int)gridDim.x + (int)blockIdx.x; v < n; v += nw * (int)gridDim.x) {
    const int o = row_ptr[v], d = row_ptr[v + 1] - o;
    uint32_t* row = (uint32_t*)out + o;
    for (int i = lane; i < d; i += 32) row[i] = (uint32_t)in[o + i] | (1u << 30);
    __syncwarp();
    const int c = sort_row(row, d, bits, words, lane, dup);
    __syncwarp();
    for (int i = lane; i < c; i += 32) row[i] &= kVertexMask;
  }
}

// In + out degree of every vertex (deg zeroed before).
__global__ void __launch_bounds__(256) k_degrees(int n, int m, const int32_t* __restrict__ row_ptr,
                                                 const int32_t* __restrict__ col, int32_t* deg) {
  const int t0 = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
  for (int v = t0; v < n; v += step) atomicAdd(&deg[v], row_ptr[v + 1] - row_ptr[v]);
  for (int e = t0; e < m; e += step) atomicAdd(&deg[col[e]], 1);
}

// One block: the vertices' numbers in the undirected CSR, by descending degree
// (degrees of 4,095 and more are one class), and the places of their rows before
// merging.  A set belongs to its smallest number, so hubs are roots: their
// neighbours are off the lists of every later root, and the rows that a list's
// members are read for are the short ones.  On the k = 5 workload graph (ids half
// in this order already) the rows of a 3-set's choices hold 453 entries above the
// root, 742 in the original numbering: the 257-graph batch counted in 138 ms, 194
// in the original numbering.
constexpr int kDegreeBins = 4096;
__global__ void __launch_bounds__(1024) k_rank(int n, const int32_t* __restrict__ deg,
                                               int32_t* rank, int32_t* off) {
  __shared__ int scan_tmp[33];
  __shared__ int32_t bins[kDegreeBins];
  for (int i = threadIdx.x; i < kDegreeBins; i += blockDim.x) bins[i] = 0;
  __syncthreads();
#pragma unroll 4
  for (int v = threadIdx.x; v < n; v += blockDim.x)
    atomicAdd(&bins[kDegreeBins - 1 - min(deg[v], kDegreeBins - 1)], 1);
  __syncthreads();
  block_exclusive_scan(bins, kDegreeBins, scan_tmp);
#pragma unroll 4
  for (int v = threadIdx.x; v < n; v += blockDim.x) {
    const int d = deg[v];
    const int r = atomicAdd(&bins[kDegreeBins - 1 - min(d, kDegreeBins - 1)], 1);
    rank[v] = r;
    off[r] = d;
  }
  if (threadIdx.x == 0) off[n] = 0;
  __syncthreads();
  block_exclusive_scan(off, n + 1, scan_tmp);
}

// ------------------------------------------------------------------ device memory of the handles

// Graphs, their scratch and the builder's come from a pool per device that keeps
// up to kPoolKeep bytes between allocations while any graph or table there is alive:
// with the runtime's own calls one load, count and free of a small graph spent
// 0.4 ms in cudaMalloc, cudaFree (50 us each) and in returning stream-ordered
// scratch to the system at every synchronisation (85 us).  What the pool keeps goes
// back to the system with the last handle, and before an allocation fails.
constexpr uint64_t kPoolKeep = 128ull << 20;
constexpr int kPoolDevices = 64;

namespace {
std::mutex g_pool_mu;
cudaMemPool_t g_pools[kPoolDevices] = {};
int64_t g_live_handles[kPoolDevices] = {};
}  // namespace

void handle_born(int device) {
  std::lock_guard<std::mutex> lock(g_pool_mu);
  if (device >= 0 && device < kPoolDevices) ++g_live_handles[device];
}

void handle_died(int device) {
  std::lock_guard<std::mutex> lock(g_pool_mu);
  if (device < 0 || device >= kPoolDevices || --g_live_handles[device] > 0 || !g_pools[device])
    return;
  DeviceScope on(device);
  cudaDeviceSynchronize();  // the frees are stream-ordered: until then nothing can be trimmed
  cudaMemPoolTrimTo(g_pools[device], 0);
}

cudaError_t pool_alloc(void** out, size_t bytes, cudaStream_t s) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kPoolDevices) return cudaErrorInvalidDevice;
  cudaMemPool_t pool = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_pool_mu);
    if (!g_pools[dev]) {
      cudaMemPoolProps props = {};
      props.allocType = cudaMemAllocationTypePinned;
      props.location.type = cudaMemLocationTypeDevice;
      props.location.id = dev;
      cudaMemPool_t p = nullptr;
      e = cudaMemPoolCreate(&p, &props);
      if (e != cudaSuccess) return e;
      uint64_t keep = kPoolKeep;
      e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
      if (e != cudaSuccess) {
        cudaMemPoolDestroy(p);
        return e;
      }
      g_pools[dev] = p;
    }
    pool = g_pools[dev];
  }
  e = cudaMallocFromPoolAsync(out, bytes, pool, s);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    cudaMemPoolTrimTo(pool, 0);
    e = cudaMallocFromPoolAsync(out, bytes, pool, s);
  }
  return e;
}

void pool_free(void* p, cudaStream_t s) {
  if (p) cudaFreeAsync(p, s);
}

// ------------------------------------------------------------------ handles

DevGraph dev_view(const mt_graph* g, unsigned long long* hist, bool original) {
  DevGraph d;
  d.n = g->n;
  d.m = g->m;
  d.nu = g->nu;
  d.root_begin = 0;
  d.root_end = g->n;
  d.pad = 0;
  d.row_ptr = g->row_ptr;
  d.col = g->col;
  d.urow = original ? g->orig_urow : g->urow;
  d.ucol = original ? g->orig_ucol : g->ucol;
  d.usrc = original ? g->orig_usrc : g->usrc;
  d.ufwd = original ? g->orig_ufwd : g->ufwd;
  d.hist = hist;
  return d;
}

// Ints of one undirected CSR: urow, ucol, usrc, ufwd.
static size_t undirected_ints(int32_t n, size_t m1) { return 2 * (size_t)n + 1 + 4 * m1; }

static size_t graph_ints(int32_t n, int32_t m, bool pooled) {
  const size_t m1 = (size_t)(m > 0 ? m : 1);
  return 3 * (size_t)n + 2 + m1 + undirected_ints(n, m1) * (pooled ? 1 : 2);
}

size_t graph_device_bytes(int32_t n, int32_t m) { return graph_ints(n, m, true) * 4 + 256; }

// Allocate the device arrays of a graph with n vertices and m arcs on `s`.
// Graphs of the server (`pooled`) count root ranges of the ranked numbering only
// and have no arrays in the original one.
static mt_status graph_alloc_impl(int32_t n, int32_t m, bool pooled, cudaStream_t s,
                                  mt_graph** out) {
  mt_graph* g = new mt_graph();
  g->n = n;
  g->m = m;
  const size_t m1 = (size_t)(m > 0 ? m : 1);
  cudaError_t e = cudaGetDevice(&g->device);
  if (e == cudaSuccess) e = pool_alloc(&g->mem, graph_ints(n, m, pooled) * 4 + 256, s);
  if (e != cudaSuccess) {
    delete g;
    set_last_error(cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? MT_ENOMEM : MT_ECUDA;
  }
  handle_born(g->device);
  g->mem_stats = (BuildStats*)g->mem;
  int32_t* p = (int32_t*)((char*)g->mem + 256);
  g->row_ptr = p; p += n + 1;  // row_ptr, rank and off are copied together
  g->rank = p; p += n;
  g->off = p; p += n + 1;
  g->col = p; p += m1;
  g->urow = p; p += n + 1;
  g->ucol = (uint32_t*)p; p += 2 * m1;
  g->usrc = p; p += 2 * m1;
  g->ufwd = p; p += n;
  if (!pooled) {
    g->orig_urow = p; p += n + 1;
    g->orig_ucol = (uint32_t*)p; p += 2 * m1;
    g->orig_usrc = p; p += 2 * m1;
    g->orig_ufwd = p;
  }
  *out = g;
  return MT_OK;
}

mt_status graph_alloc(int32_t n, int32_t m, cudaStream_t s, mt_graph** out) {
  return graph_alloc_impl(n, m, false, s, out);
}

// Free a graph's memory on `s`, behind everything that uses it there.
static void graph_free_on(mt_graph* g, cudaStream_t s) {
  {
    DeviceScope on(g->device);
    pool_free(g->mem, s);
    if (g->ws && g->ws_owned) pool_free(g->ws, s);
    for (void* p : g->captured_ws) pool_free(p, s);
  }
  if (g->ev0) cudaEventDestroy(g->ev0);
  if (g->ev1) cudaEventDestroy(g->ev1);
  const int device = g->device;
  delete g;
  handle_died(device);
}

void graph_release(mt_graph* g, cudaStream_t s) {
  if (g) graph_free_on(g, s);
}

// What a device build needs to be safe, in whole-array passes that the compiler
// vectorises: sizes, monotone rows, ids in range.  `sorted`: every row strictly
// ascending (and so without duplicates): the array falls only where a row starts.
static mt_status check_csr(int32_t n, int32_t m, const int32_t* row_ptr, const int32_t* col,
                           bool* sorted) {
  if (!row_ptr || (m > 0 && !col) || n < 1 || m < 0) return MT_EINVAL;
  if (n > kMaxVertices) return MT_EUNSUPPORTED;
  if (row_ptr[0] != 0 || row_ptr[n] != m) return MT_EINVAL;
  unsigned down = 0;
  for (int32_t v = 0; v < n; ++v) down |= (unsigned)(row_ptr[v + 1] < row_ptr[v]);
  if (down) return MT_EINVAL;
  unsigned outside = 0, falls = 0, starts = 0;
  for (int32_t e = 0; e < m; ++e) outside |= (unsigned)((uint32_t)col[e] >= (uint32_t)n);
  if (outside) return MT_EINVAL;
  for (int32_t e = 1; e < m; ++e) falls += (unsigned)(col[e] <= col[e - 1]);
  for (int32_t v = 0; v < n; ++v) {
    const int32_t a = row_ptr[v];
    if (a > 0 && a < row_ptr[v + 1]) starts += (unsigned)(col[a] <= col[a - 1]);
  }
  *sorted = falls == starts;
  return MT_OK;
}

static bool has_self_loop(int32_t n, const int32_t* row_ptr, const int32_t* col) {
  unsigned loops = 0;
  for (int32_t v = 0; v < n; ++v)
    for (int32_t e = row_ptr[v]; e < row_ptr[v + 1]; ++e) loops |= (unsigned)(col[e] == v);
  return loops != 0;
}

mt_status validate_csr(int32_t n, int32_t m, const int32_t* row_ptr, const int32_t* col) {
  bool sorted = false;
  MT_TRY(check_csr(n, m, row_ptr, col, &sorted));
  return has_self_loop(n, row_ptr, col) ? MT_EINVAL : MT_OK;
}

// Enqueue the load of a checked CSR on `s`: upload, build, stats into `st` (host
// memory; pinned, the call does not wait for the device).
static mt_status graph_load_enqueue(int32_t n, int32_t m, const int32_t* row_ptr,
                                    const int32_t* col, bool sorted, bool pooled, cudaStream_t s,
                                    BuildStats* st, mt_graph** out) {
  mt_graph* g = nullptr;
  MT_TRY(graph_alloc_impl(n, m, pooled, s, &g));
  // unsorted rows are uploaded beside and sorted into place; sorted ones go there
  int32_t* up = nullptr;
  cudaError_t e = cudaSuccess;
  if (!sorted) e = pool_alloc((void**)&up, (size_t)m * 4, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(g->row_ptr, row_ptr, (size_t)(n + 1) * 4, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess && m > 0)
    e = cudaMemcpyAsync(sorted ? g->col : up, col, (size_t)m * 4, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = graph_build_enqueue(g, sorted ? nullptr : up, false, s, st);
  pool_free(up, s);
  if (e != cudaSuccess) {
    set_last_error(cudaGetErrorString(e));
    graph_release(g, s);
    return e == cudaErrorMemoryAllocation ? MT_ENOMEM : MT_ECUDA;
  }
  *out = g;
  return MT_OK;
}

// The stats of a finished build into the handle (MT_EINVAL: a duplicate arc or a
// self-loop).
mt_status graph_take_stats(mt_graph* g, const BuildStats& st) {
  if (st.err) return MT_EINVAL;
  g->nu = st.nu;
  g->dmax = st.dmax;
  return MT_OK;
}

mt_status graph_load_begin(int32_t n, int32_t m, const int32_t* row_ptr, const int32_t* col,
                           cudaStream_t s, BuildStats* st, mt_graph** out) {
  bool sorted = false;
  MT_TRY(check_csr(n, m, row_ptr, col, &sorted));
  return graph_load_enqueue(n, m, row_ptr, col, sorted, true, s, st, out);
}

// The build reports self-loops and duplicate arcs (on the host the look for
// self-loops was 93 us of a 120,000-arc graph's load); where it cannot run, the
// host looks, so that a malformed graph is MT_EINVAL all the same.
static mt_status graph_load(int32_t n, int32_t m, const int32_t* row_ptr, const int32_t* col,
                            cudaStream_t s, mt_graph** out) {
  bool sorted = false;
  MT_TRY(check_csr(n, m, row_ptr, col, &sorted));
  mt_graph* g = nullptr;
  BuildStats st{};
  mt_status r = graph_load_enqueue(n, m, row_ptr, col, sorted, false, s, &st, &g);
  if (r != MT_OK) return has_self_loop(n, row_ptr, col) ? MT_EINVAL : r;
  const cudaError_t e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    set_last_error(cudaGetErrorString(e));
    r = MT_ECUDA;
  } else {
    r = graph_take_stats(g, st);
  }
  if (r != MT_OK) {
    graph_release(g, s);
    return r;
  }
  *out = g;
  return MT_OK;
}

// Enqueue the build of the undirected CSR of `g` from its row_ptr and its
// destinations.  `unsorted` (device, m): destinations to be sorted into g->col
// first; nullptr when g->col holds them.  `ranked`: g->rank and g->off are filled
// in already (a null graph's degrees are its source's).  The stats go to
// g->mem_stats and, if given, to `st` (host).
cudaError_t graph_build_enqueue(mt_graph* g, const int32_t* unsorted, bool ranked, cudaStream_t s,
                                BuildStats* st) {
  const int n = g->n, m = g->m;
  const size_t m1 = (size_t)(m > 0 ? m : 1);
  void* scratch = nullptr;
  cudaError_t e = pool_alloc(&scratch, (2 * m1 + (size_t)n) * 4, s);
  if (e != cudaSuccess) return e;
  BuildArgs a;
  a.n = n; a.m = m; a.G = 1;
  a.row_ptr = g->row_ptr;
  a.col_in = g->col;
  a.rank = g->rank;
  a.off = g->off;
  a.stats = g->mem_stats;
  a.tmp = (uint32_t*)scratch;
  a.cursor = (int32_t*)(a.tmp + 2 * m1);
  a.urow = g->urow; a.ucol = g->ucol; a.usrc = g->usrc; a.ufwd = g->ufwd;
  if (unsorted && m > 0) {
    const size_t per_warp = (size_t)bitmap_words(n) * 8;
    const int warps = per_warp * 8 > 96 * 1024 ? 4 : 8;
    e = cudaFuncSetAttribute((const void*)k_sort_cols, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             96 * 1024);
    if (e == cudaSuccess)
      k_sort_cols<<<std::min((n + warps - 1) / warps, 8192), warps * 32, per_warp * warps, s>>>(
          n, g->row_ptr, unsorted, g->col);
    a.col_in = unsorted;  // with its duplicates, which k_rows reports
  }
  if (e == cudaSuccess && !ranked) {
    e = cudaMemsetAsync(a.cursor, 0, (size_t)n * 4, s);
    k_degrees<<<std::min((std::max(n, m) + 255) / 256, 2048), 256, 0, s>>>(n, m, g->row_ptr,
                                                                           a.col_in, a.cursor);
    k_rank<<<1, 1024, 0, s>>>(n, a.cursor, g->rank, g->off);
  }
  if (e == cudaSuccess) e = launch_build(a, s);
  if (e == cudaSuccess && st)
    e = cudaMemcpyAsync(st, a.stats, sizeof(BuildStats), cudaMemcpyDeviceToHost, s);
  pool_free(scratch, s);
  return e;
}

mt_status graph_build_sync(mt_graph* g, const int32_t* unsorted, bool ranked, cudaStream_t s) {
  BuildStats st{};
  cudaError_t e = graph_build_enqueue(g, unsorted, ranked, s, &st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    set_last_error(cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? MT_ENOMEM : MT_ECUDA;
  }
  return graph_take_stats(g, st);
}

// One block: the original numbering's "ranks" and places of rows.
__global__ void __launch_bounds__(1024) k_orig_layout(int n, const int32_t* __restrict__ rank,
                                                      const int32_t* __restrict__ off,
                                                      int32_t* id, int32_t* ooff) {
  __shared__ int scan_tmp[33];
  for (int v = threadIdx.x; v < n; v += blockDim.x) {
    id[v] = v;
    ooff[v] = off[rank[v] + 1] - off[rank[v]];
  }
  if (threadIdx.x == 0) ooff[n] = 0;
  __syncthreads();
  block_exclusive_scan(ooff, n + 1, scan_tmp);
}

size_t original_scratch_bytes(const mt_graph* g) {
  const size_t m1 = (size_t)(g->m > 0 ? g->m : 1);
  return (2 * m1 + 3 * (size_t)g->n + 1) * 4 + sizeof(BuildStats) + 256;
}

mt_status graph_build_original(mt_graph* g, void* scratch, cudaStream_t s) {
  if (g->has_orig) return MT_OK;
  const int n = g->n, m = g->m;
  const size_t m1 = (size_t)(m > 0 ? m : 1);
  BuildArgs a;
  a.n = n; a.m = m; a.G = 1;
  a.row_ptr = g->row_ptr;
  a.col_in = g->col;
  a.stats = (BuildStats*)scratch;
  a.tmp = (uint32_t*)((char*)scratch + 256);
  a.cursor = (int32_t*)(a.tmp + 2 * m1);
  int32_t* id = a.cursor + n;
  int32_t* ooff = id + n;
  a.rank = id;
  a.off = ooff;
  a.urow = g->orig_urow; a.ucol = g->orig_ucol; a.usrc = g->orig_usrc; a.ufwd = g->orig_ufwd;
  k_orig_layout<<<1, 1024, 0, s>>>(n, g->rank, g->off, id, ooff);
  MT_CUDA_TRY(cudaGetLastError());
  MT_CUDA_TRY(launch_build(a, s));
  // built when the stream gets there; under capture nothing runs now
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  MT_CUDA_TRY(cudaStreamIsCapturing(s, &cap));
  g->has_orig = cap == cudaStreamCaptureStatusNone;
  return MT_OK;
}

}  // namespace mt

using namespace mt;

extern "C" {

const char* mt_status_str(mt_status s) {
  switch (s) {
    case MT_OK: return "ok";
    case MT_EINVAL: return "invalid argument or malformed graph";
    case MT_EUNSUPPORTED: return "unsupported size (k outside 3..6, n > 65535 or degree too large)";
    case MT_ENOMEM: return "out of memory";
    case MT_ECUDA: return "CUDA error";
    case MT_ETIMEOUT: return "bounded device wait expired";
    case MT_EOVERFLOW: return "device stack or queue overflow";
    case MT_EBUSY: return "admission refused (budget or slots)";
  }
  return "unknown status";
}

const char* mt_last_error(void) { return g_last_error.c_str(); }

mt_status mt_graph_load_csr(int32_t n, int32_t m, const int32_t* row_ptr, const int32_t* col,
                            void* stream, mt_graph** out) {
  if (!out) return MT_EINVAL;
  TraceRange tr("mt_graph_load_csr");
  return graph_load(n, m, row_ptr, col, (cudaStream_t)stream, out);
}

mt_status mt_graph_free(mt_graph* g) {
  if (!g) return MT_OK;
  // counts on any stream of the graph's device may still use it, and the pool
  // orders memory it takes back behind the freeing stream's work only
  DeviceScope on(g->device);
  cudaDeviceSynchronize();
  graph_free_on(g, nullptr);
  return MT_OK;
}

mt_status mt_graph_info(const mt_graph* g, int32_t* n, int32_t* m, int32_t* m_undirected,
                        int32_t* max_degree) {
  if (!g) return MT_EINVAL;
  if (n) *n = g->n;
  if (m) *m = g->m;
  if (m_undirected) *m_undirected = g->nu / 2;
  if (max_degree) *max_degree = g->dmax;
  return MT_OK;
}

mt_status mt_graph_copy_csr(const mt_graph* g, int32_t* row_ptr, int32_t* col, void* stream) {
  if (!g || !row_ptr || (g->m > 0 && !col)) return MT_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  MT_CUDA_TRY(cudaMemcpyAsync(row_ptr, g->row_ptr, (size_t)(g->n + 1) * 4,
                              cudaMemcpyDeviceToHost, s));
  if (g->m > 0)
    MT_CUDA_TRY(cudaMemcpyAsync(col, g->col, (size_t)g->m * 4, cudaMemcpyDeviceToHost, s));
  MT_CUDA_TRY(cudaStreamSynchronize(s));
  return MT_OK;
}

}  // extern "C"
