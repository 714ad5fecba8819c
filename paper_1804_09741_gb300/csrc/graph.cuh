// Host-side graph handle and the device graph builder (sorted CSR + labelled
// undirected CSR) shared by the loader, the randomiser and the batch path.
#pragma once

#include <vector>

#include "common.cuh"

namespace mt {

// Per-graph results of the builder.
struct BuildStats {
  int32_t nu;
  int32_t dmax;
  uint32_t err;
  int32_t pad;
};

}  // namespace mt

struct mt_graph {
  int32_t n = 0, m = 0;
  int32_t nu = 0, dmax = 0;    // filled after the build (host copy of the stats)
  int device = 0;
  int32_t* row_ptr = nullptr;  // device, n+1
  int32_t* rank = nullptr;     // device, n: each vertex's number in the undirected CSR
  int32_t* off = nullptr;      // device, n+1: prefix sums of in + out degree by number
  int32_t* col = nullptr;      // device, m (sorted rows)
  int32_t* urow = nullptr;     // device, n+1
  uint32_t* ucol = nullptr;    // device, 2m (nu used)
  int32_t* usrc = nullptr;     // device, 2m
  int32_t* ufwd = nullptr;     // device, n
  // the undirected CSR in the original numbering, which root ranges are in;
  // built by the first count that needs it
  int32_t* orig_urow = nullptr;
  uint32_t* orig_ucol = nullptr;
  int32_t* orig_usrc = nullptr;
  int32_t* orig_ufwd = nullptr;
  bool has_orig = false;
  void* mem = nullptr;         // one allocation backing all of the above
  mt::BuildStats* mem_stats = nullptr;  // device: what the build found, at its start

  // Counting scratch, grown on demand by mt_count, or the caller's buffer
  // attached by mt_set_workspace (ws_owned false: never grown or freed here).
  // Scratch that a captured count uses stays until the handle goes: its CUDA
  // graph may be replayed after a larger count has moved on to another buffer.
  void* ws = nullptr;
  size_t ws_bytes = 0;
  bool ws_owned = true;
  bool ws_captured = false;         // a captured count uses ws
  std::vector<void*> captured_ws;   // earlier ones
  // Where the last count left its error word and item count inside `ws`.
  bool stats_valid = false;
  size_t off_err = 0, off_nitems = 0;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
};

namespace mt {

// Makes `device` the current one while in scope: what is waited for and the
// legacy stream that memory is returned on are the current device's.
class DeviceScope {
 public:
  explicit DeviceScope(int device) {
    if (cudaGetDevice(&before_) != cudaSuccess) before_ = device;
    if (before_ != device) cudaSetDevice(device);
    device_ = device;
  }
  ~DeviceScope() {
    if (before_ != device_) cudaSetDevice(before_);
  }
  DeviceScope(const DeviceScope&) = delete;
  DeviceScope& operator=(const DeviceScope&) = delete;

 private:
  int before_ = 0, device_ = 0;
};

// Pointers of G graphs of equal degrees laid out with fixed strides.
struct BuildArgs {
  int32_t n, m, G;
  const int32_t* row_ptr;   // n+1, shared by all graphs
  const int32_t* col_in;    // destinations, rows in any order, stride m
  const int32_t* rank;      // n, shared
  const int32_t* off;       // n+1, shared
  uint32_t* tmp;            // scratch 2m per graph
  int32_t* cursor;          // scratch n per graph
  int32_t* urow;            // n+1 per graph
  uint32_t* ucol;           // 2m per graph
  int32_t* usrc;            // 2m per graph
  int32_t* ufwd;            // n per graph
  BuildStats* stats;        // one per graph
};

// Enqueue the builder.
cudaError_t launch_build(const BuildArgs& a, cudaStream_t s);
cudaError_t graph_build_enqueue(mt_graph* g, const int32_t* unsorted, bool ranked, cudaStream_t s,
                                BuildStats* st);
mt_status graph_build_sync(mt_graph* g, const int32_t* unsorted, bool ranked, cudaStream_t s);
mt_status graph_alloc(int32_t n, int32_t m, cudaStream_t s, mt_graph** out);

// Enqueue the build of g's undirected CSR in the original numbering, unless it is
// there; `scratch` holds original_scratch_bytes.
size_t original_scratch_bytes(const mt_graph* g);
mt_status graph_build_original(mt_graph* g, void* scratch, cudaStream_t s);

// Device memory of handles and their scratch, in the order of stream `s`.
cudaError_t pool_alloc(void** out, size_t bytes, cudaStream_t s);
void pool_free(void* p, cudaStream_t s);
void handle_born(int device);
void handle_died(int device);

DevGraph dev_view(const mt_graph* g, unsigned long long* hist, bool original = false);

// Host-side checks of a CSR (MT_OK, MT_EINVAL or MT_EUNSUPPORTED).
mt_status validate_csr(int32_t n, int32_t m, const int32_t* row_ptr, const int32_t* col);

// Enqueue the load of a valid graph for the server, in the order of `s`; the
// handle is ready when `s` is done and graph_take_stats accepts `st` (pinned).
// Release it with graph_release on a stream.
mt_status graph_load_begin(int32_t n, int32_t m, const int32_t* row_ptr, const int32_t* col,
                           cudaStream_t s, BuildStats* st, mt_graph** out);
mt_status graph_take_stats(mt_graph* g, const BuildStats& st);
void graph_release(mt_graph* g, cudaStream_t s);
size_t graph_device_bytes(int32_t n, int32_t m);

}  // namespace mt
