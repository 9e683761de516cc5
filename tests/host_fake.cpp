// The host side of the library (api.cu, noalloc.cu, compiled as plain C++) over a CUDA
// runtime and kernel launchers that do nothing but keep books: device memory is host memory,
// a launch records its arguments, and any allocation can be made to fail.  What the host
// decides - routes, launch shapes, what is checked, what is held - is printed for
// test_host_decisions.py; no kernel's work is done here.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <utility>
#include <vector>

#include "band.cuh"
#include "fronts.cuh"
#include "gsofa.h"
#include "internal.cuh"

// ---------------------------------------------------------------- what a scenario sets
static int g_band_left = 0, g_band_right = 0;      // what the scan measures, for every matrix
static long long g_reach = 1000000;                // entries that a sampled row reaches
static int g_per_row = 3;                          // entries of a row
static int g_blocks = 0;                           // a dissection: it falls into closed blocks
static int g_fail_count = 0, g_fail_at = -1;       // the g_fail_at-th pool allocation from now on fails
static std::map<void*, size_t> g_held;             // pool memory: bytes by block
static size_t g_now = 0, g_peak = 0;
static int g_stuck = 0;                            // streams that never finish
static std::vector<std::pair<const char*, size_t>> g_pinned_blocks, g_in_flight;  // pinned memory; what copies of a stuck stream use
static void copied(const void* host, size_t n) {
  for (auto& b : g_pinned_blocks) {
    if ((const char*)host < b.first || (const char*)host >= b.first + b.second) continue;
    for (auto& f : g_in_flight)
      if (f.first < (const char*)host + n && (const char*)host < f.first + f.second && !g_stuck) std::puts("in flight");
    if (g_stuck) g_in_flight.push_back({(const char*)host, n});
  }
}

// ---------------------------------------------------------------- CUDA runtime
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 227 * 1024;
  return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { *p = (cudaMemPool_t)1; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t, cudaMemPoolAttr, void* v) { *(uint64_t*)v = 0; return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)270 << 30; return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) {
  *p = nullptr;
  if (g_fail_at >= 0 && g_fail_count++ == g_fail_at) return cudaErrorMemoryAllocation;
  *p = std::calloc(1, n);
  if (!*p) return cudaErrorMemoryAllocation;
  g_held[*p] = n;
  g_now += n;
  if (g_now > g_peak) g_peak = g_now;
  return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
  auto it = g_held.find(p);
  if (it != g_held.end()) {
    g_now -= it->second;
    g_held.erase(it);
  }
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = n < (size_t)1 << 30 ? std::calloc(1, n) : nullptr;
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) {
  const cudaError_t e = cudaMalloc(p, n);
  if (*p) g_pinned_blocks.push_back({(const char*)*p, n});
  return e;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) { *d = h; return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  copied(k == cudaMemcpyDeviceToHost ? d : s, n);
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaStreamQuery(cudaStream_t) { return g_stuck ? cudaErrorNotReady : cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)1; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) { *s = cudaStreamCaptureStatusNone; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)1; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* f, cudaEvent_t, cudaEvent_t) { *f = 1.f; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = const_cast<void*>(s); return cudaSuccess; }
}

// ---------------------------------------------------------------- kernel launchers
namespace gsofa {

size_t trav_smem_bytes(int32_t n, int32_t, int32_t cap, int l16) { return (size_t)(l16 ? 2 : 4) * (n + 2 * (size_t)cap); }
int32_t trav_smem_max_S(int32_t n, size_t, int) { return n <= 65533 ? n : 32768; }
int trav_smem_static_bytes() { return 0; }
int trav_smem_occupancy(int, size_t, int) { return 1; }
int trav_class_occupancy(int, int warps_per_sm, int, int) { return warps_per_sm / CLASS_WARPS_PER_CTA; }
size_t trav_class_smem(int, int, int) { return 0; }
size_t scan_tmp_bytes(int32_t) { return 64; }
size_t scan_tmp_bytes_long(int64_t) { return 64; }

cudaError_t launch_init_counters(DevCounters* c, cudaStream_t) { std::memset(c, 0, sizeof(*c)); return cudaSuccess; }
cudaError_t launch_validate(int32_t, const int32_t*, const int32_t*, DevCounters*, cudaStream_t) {
  std::puts("validate");
  return cudaSuccess;
}
cudaError_t launch_validate_batch(const MatDesc*, int32_t, int64_t, DevCounters*, cudaStream_t) {
  std::puts("validate_batch");
  return cudaSuccess;
}
cudaError_t launch_trav_smem(const TravArgs&, int grid, int, int, cudaStream_t) {
  std::printf("trav_smem %d\n", grid);
  return cudaSuccess;
}
cudaError_t launch_trav_class(const TravArgs&, int grid, int, int, cudaStream_t) {
  std::printf("trav_class %d\n", grid);
  return cudaSuccess;
}
cudaError_t launch_fill_i32(int32_t*, int64_t, int32_t, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_iota_desc(int32_t*, int32_t, int32_t, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_build_ell(int32_t, const int32_t*, const int32_t*, int4*, DevCounters*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_build_ellw(int32_t, const int32_t*, const int32_t*, int4*, DevCounters*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_build_ell_batch(const MatDesc*, int32_t, int64_t, int4*, DevCounters*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_supernode_flags(int32_t, int32_t, const uint32_t*, const int64_t*, const int32_t*, const int32_t*, int32_t*,
                                   DevCounters*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_supernode_batch(const MatDesc*, int32_t, int64_t, int32_t, const uint32_t*, const int64_t*, const int32_t*,
                                   const int32_t*, int32_t*, int32_t*, DevCounters*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_compact(int32_t, const uint32_t*, const int64_t*, const int32_t*, const int32_t*, const int64_t*,
                           const int64_t*, int32_t*, int32_t*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_compact_long(int64_t, const uint32_t*, const int64_t*, const int32_t*, const int32_t*, const int64_t*,
                                const int64_t*, int32_t*, int32_t*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_scan_i32_i64(const int32_t*, int64_t*, int32_t, void*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_scan_i32_i64_long(const int32_t*, int64_t*, int64_t, void*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_rebase_rowptr(const MatDesc*, int32_t, int64_t, const int64_t*, int64_t*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_scatter_starts(int32_t, const int32_t*, const int64_t*, int32_t*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_scatter_starts_batch(const MatDesc*, int32_t, int64_t, const int32_t*, const int64_t*, int32_t*,
                                        cudaStream_t) { return cudaSuccess; }

cudaError_t launch_band_scan(const BandArgs& a, cudaStream_t) {
  std::puts("band_scan");
  for (int m = 0; m < a.nmats; m++) {
    a.band[2 * m] = g_band_left;
    a.band[2 * m + 1] = g_band_right;
    if (a.entries) a.entries[m] = g_per_row * (a.mats ? a.mats[m] : a.one).n;
  }
  a.ctr->nnz = (unsigned long long)g_per_row * (unsigned long long)a.rows;
  a.ctr->spread = a.ctr->nnz * (unsigned long long)(g_band_left > g_band_right ? g_band_left : g_band_right) / 2;
  return cudaSuccess;
}
cudaError_t launch_band_reach(const BandArgs& a, bool, cudaStream_t) {
  for (int m = 0; m < a.sampled; m++) {
    a.reach[m].entries = (unsigned long long)(g_reach * a.reach_rows);
    a.reach[m].levels = 5u * (uint32_t)a.reach_rows;
  }
  a.ctr->stretch = (a.one.n + 31) / 32;
  return cudaSuccess;
}
cudaError_t launch_band_elim(const BandArgs& a, int count, int C, int, size_t, cudaStream_t) {
  const BandMat& d = a.mats ? a.mats[a.first] : a.one;
  std::printf("band_elim %d %d left %d right %d\n", count, C, d.LB, d.UB);
  return cudaSuccess;
}
cudaError_t launch_band_count(const BandArgs&, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_band_expand(const BandArgs&, cudaStream_t) { return cudaSuccess; }

cudaError_t launch_front_blocks(const FrontLevel&, cudaStream_t) { std::puts("front_blocks"); return cudaSuccess; }
// blocks of 500 vertices that leave nothing for a next level, or none
cudaError_t launch_front_above(const FrontLevel& l, cudaStream_t) {
  if (!g_blocks) l.ctr->overflow = 1;
  for (int b = 0; g_blocks && 500 * b < l.n; b++) {
    l.ctr->nblocks = b + 1;
    l.b_first[b] = 500 * b;
    l.b_size[b] = l.n - 500 * b < 500 ? l.n - 500 * b : 500;
  }
  return cudaSuccess;
}
cudaError_t launch_front_reduce(const FrontLevel&, int32_t, const FrontMat*, const uint32_t*, int32_t*, int32_t*, int32_t*,
                                int32_t*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_front_whole(const FrontLevel&, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_front_iota(int32_t*, int32_t, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_front_gids(const FrontLevel&, int32_t, int32_t*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_front_count(const FrontEmit&, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_front_expand(const FrontEmit&, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_front_elim(const FrontArgs&, int count, int C, int, size_t, cudaStream_t) {
  std::printf("front_elim %d %d held %zu\n", count, C, g_now);
  return cudaSuccess;
}

}  // namespace gsofa

// ---------------------------------------------------------------- scenarios
// arguments: key=value
int main(int argc, char** argv) {
  std::map<std::string, long long> v;
  for (int i = 1; i < argc; i++) {
    const std::string s = argv[i];
    const size_t at = s.find('=');
    v[s.substr(0, at)] = std::atoll(s.c_str() + at + 1);
  }
  auto get = [&](const char* k, long long d) { return v.count(k) ? v[k] : d; };
  const int32_t n = (int32_t)get("n", 100);
  const int count = (int)get("count", 1);  // above 1: one batch
  g_band_left = (int)get("left", 0);
  g_band_right = (int)get("right", 0);
  g_fail_at = (int)get("fail_at", -1);
  g_blocks = (int)get("blocks", 0);
  g_reach = get("reach", 1000000);
  g_per_row = (int)get("per_row", 3);
  gsofa_options o;
  gsofa_default_options(&o);
  o.max_ctas = (int32_t)get("max_ctas", 0);
  o.mem_budget_bytes = get("budget", 0);
  std::vector<int32_t> rp((size_t)(get("rows", n) + 1), 0), ci(1, 0);
  std::vector<gsofa_result> out(count);
  int rc;
  auto call = [&] {
    if (count > 1) {
      std::vector<int32_t> ns(count, n);
      std::vector<const int32_t*> rps(count, rp.data()), cis(count, ci.data());
      return gsofa_batch(count, ns.data(), rps.data(), cis.data(), &o, nullptr, out.data());
    }
    return gsofa_symbolic_device(n, rp.data(), ci.data(), &o, nullptr, &out[0]);
  };
  if (get("stuck", 0)) {  // a call whose wait runs out before the one that is looked at
    g_stuck = 1;
    std::printf("first rc %d\n", call());
    g_stuck = 0;
  }
  if (get("counts", 0)) {
    std::vector<int32_t> a(n), b(n), c(n);
    rc = gsofa_row_counts_noalloc(n, rp.data(), ci.data(), a.data(), b.data(), c.data(), nullptr);
  } else {
    rc = call();
  }
  std::printf("rc %d\n", rc);
  if (rc == GSOFA_OK && !get("counts", 0))
    for (auto& r : out) gsofa_free(&r);
  std::printf("held %zu\n", g_now);
  return 0;
}
