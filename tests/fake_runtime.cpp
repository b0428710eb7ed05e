// A CUDA runtime and a device pool on the host, linked with the library's own
// objects (without its pool): calls queue nothing, but every block that queued
// work may use stays busy until its stream is waited for, and the k-th
// allocation or the k-th queued call can be made to fail.  What is reported:
// blocks given back while busy, blocks never given back, copies whose kind
// does not fit their source.  Runs without a GPU; no kernel is executed.
//
//   program SCENARIO         every allocation, then every call, fails in turn
//   program SCENARIO SIZE    the smallest pool in which it does not run out of
//                            memory, as it is and with no blocks of SIZE bytes
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <set>
#include <string>
#include <vector>

#include <cuda_runtime.h>
int atomicOr(int *, int);  // (named by device code of the header)
#include "internal.cuh"

namespace {

using Streams = std::set<cudaStream_t>;
struct Block {
  size_t bytes;
  Streams busy;
  int kind;  // 0 pool, 1 caller's device memory, 2 page-locked
};
std::map<char *, Block> blocks;
std::map<cudaStream_t, Streams> waits;  // streams whose work a stream waits for
std::vector<std::string> found;
long allocs, calls, fail_alloc = -1, fail_call = -1;
size_t budget = ~(size_t)0, used, refused = ~(size_t)0;
cudaError_t last = cudaSuccess;
cudaStream_t launch_stream;

std::map<char *, Block>::iterator block_of(const void *p) {
  auto it = blocks.upper_bound((char *)p);
  if (it == blocks.begin()) return blocks.end();
  --it;
  return (char *)p < it->first + it->second.bytes ? it : blocks.end();
}
void use(const void *p, cudaStream_t s) {
  auto it = block_of(p);
  if (it != blocks.end()) it->second.busy.insert(s);
}
void use_all(cudaStream_t s) {
  for (auto &b : blocks) b.second.busy.insert(s);
}
bool injected() { return calls++ == fail_call; }
void give_back(void *p, bool ordered, const char *who) {
  auto it = blocks.find((char *)p);
  if (it == blocks.end()) {
    found.push_back(std::string(who) + ": no such block");
    return;
  }
  if (!ordered && !it->second.busy.empty())
    found.push_back(std::string(who) + ": block of " + std::to_string(it->second.bytes) + " bytes in use");
  if (it->second.kind == 0) used -= it->second.bytes;
  std::free(it->first);
  blocks.erase(it);
}
void *take(size_t bytes, int kind) {
  if (bytes == 0) bytes = 1;
  void *p = std::calloc(1, bytes);
  blocks[(char *)p] = Block{bytes, {}, kind};
  if (kind == 0) used += bytes;
  return p;
}

}  // namespace

extern "C" {
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  Streams done = waits[s];
  done.insert(s);
  for (auto &b : blocks)
    for (cudaStream_t d : done) b.second.busy.erase(d);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind k, cudaStream_t s) {
  if (injected()) return cudaErrorUnknown;
  const auto b = block_of(src);
  if (k == cudaMemcpyDeviceToDevice && (b == blocks.end() || b->second.kind == 2))
    found.push_back("a copy between device buffers from host memory");
  use(dst, s);
  use(src, s);
  std::memcpy(dst, src, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void *dst, const void *src, size_t n, cudaMemcpyKind) {
  std::memcpy(dst, src, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t s) {
  if (injected()) return cudaErrorUnknown;
  use(p, s);
  std::memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaLaunchCooperativeKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t s) {
  if (injected()) return cudaErrorUnknown;
  use_all(s);
  return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, CUstream_st *s) {
  launch_stream = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *s) {
  *(cudaStream_t *)s = launch_stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *) {
  *k = nullptr;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t s) {
  if (injected()) return last = cudaErrorUnknown;
  use_all(s);
  return cudaSuccess;
}
void **__cudaRegisterFatBinary(void *) {
  static void *h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
const char *cudaGetErrorString(cudaError_t) { return "made to fail"; }
cudaError_t cudaGetDevice(int *d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrL2CacheSize ? 128 << 20 : 152;
  return cudaSuccess;
}
struct Event {
  Streams s;
};
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
  if (injected()) return cudaErrorUnknown;
  *e = (cudaEvent_t) new Event;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  delete (Event *)e;
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  if (injected()) return cudaErrorUnknown;
  ((Event *)e)->s = waits[s];
  ((Event *)e)->s.insert(s);
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  if (injected()) return cudaErrorUnknown;
  waits[s].insert(((Event *)e)->s.begin(), ((Event *)e)->s.end());
  return cudaSuccess;
}
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.f;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  *s = (cudaStream_t)std::malloc(1);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return injected() ? cudaErrorUnknown : cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *, const void *) { return cudaErrorUnknown; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
  *p = std::calloc(1, n);
  return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n) {
  *p = std::calloc(1, n);
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { return cudaFree(p); }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
  std::memset(a, 0, sizeof(*a));
  const auto b = block_of(p);
  a->type = b == blocks.end() ? cudaMemoryTypeUnregistered : b->second.kind == 2 ? cudaMemoryTypeHost : cudaMemoryTypeDevice;
  a->devicePointer = const_cast<void *>(p);
  return cudaSuccess;
}
// what the loop over the CSR uses is not here: its calls end with an error
cudaError_t cudaGetSymbolAddress(void **, const void *) { return cudaErrorNotSupported; }
cudaError_t cudaGraphAddNode(cudaGraphNode_t *, cudaGraph_t, const cudaGraphNode_t *, const cudaGraphEdgeData *, size_t,
                             cudaGraphNodeParams *) {
  return cudaErrorNotSupported;
}
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle *, cudaGraph_t, unsigned, unsigned) {
  return cudaErrorNotSupported;
}
cudaError_t cudaGraphCreate(cudaGraph_t *, unsigned) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t *, const cudaGraphEdgeData *,
                                          size_t, cudaStreamCaptureMode) {
  return cudaErrorNotSupported;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) { return cudaErrorNotSupported; }
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t, cudaStreamCaptureStatus *, unsigned long long *, cudaGraph_t *,
                                     const cudaGraphNode_t **, const cudaGraphEdgeData **, size_t *) {
  return cudaErrorNotSupported;
}
cudaError_t cudaStreamUpdateCaptureDependencies(cudaStream_t, cudaGraphNode_t *, const cudaGraphEdgeData *, size_t,
                                                unsigned) {
  return cudaErrorNotSupported;
}
}

namespace msf {
void *pool_alloc(size_t bytes, int *err) {
  if (allocs++ == fail_alloc || used + bytes > budget || bytes == refused) {
    *err = MSF_ERR_OOM;
    return nullptr;
  }
  *err = MSF_OK;
  return take(bytes, 0);
}
void pool_free(void *p) {
  if (p) give_back(p, false, "pool_free");
}
void pool_free_after(void *p, cudaStream_t) {
  if (p) give_back(p, true, "pool_free_after");
}
int PinnedWords::take(size_t want) {
  if (allocs++ == fail_alloc) return MSF_ERR_OOM;
  p = (unsigned *)::take(want, 2);
  bytes = want;
  return MSF_OK;
}
PinnedWords::~PinnedWords() {
  if (p) give_back(p, false, "pinned words");
}
std::string message;
void set_error(const std::string &m) { message = m; }
int fail(int code, const std::string &m) {
  message = m;
  return code;
}
int cuda_fail(cudaError_t e, const char *) { return e == cudaErrorMemoryAllocation ? MSF_ERR_OOM : MSF_ERR_CUDA; }
const char *last_error_cstr() { return message.c_str(); }
int sm_count() { return 152; }
DeviceShare::DeviceShare(int64_t, int64_t) : sms(152) {}
DeviceShare::~DeviceShare() {}
Options &options() {
  static Options o;
  return o;
}
}  // namespace msf

int main(int argc, char **argv) {
  const std::string name = argc > 1 ? argv[1] : "";
  const bool host = name.find("host") != std::string::npos;    // arrays in pageable memory
  const bool locked = name.find("locked") != std::string::npos;  // read in place
  if (locked) msf::options().host_input = 1;
  std::vector<void *> own;
  auto array = [&](size_t bytes) {
    void *p = host ? std::calloc(1, bytes) : take(bytes, locked ? 2 : 1);
    own.push_back(p);
    return p;
  };
  std::function<int()> call;
  // the graph: n vertices, m edges (or slots), all arrays zero
  auto graph = [&](int64_t n, int64_t m, bool csr, std::function<int(msf_graph *)> then) {
    auto *s = (int32_t *)array((size_t)m * 4), *d = (int32_t *)array((size_t)m * 4);
    void *w = array((size_t)m * 4);
    int64_t *rp = nullptr;
    if (csr) {
      rp = (int64_t *)array((size_t)(n + 1) * 8);
      for (int64_t i = 1; i <= n; ++i) rp[i] = m;
    }
    call = [=]() -> int {
      msf_graph *g = nullptr;
      int rc = msf_build_csr(n, m, s, d, rp, w, MSF_F32, 0, nullptr, &g);
      if (rc == MSF_OK && then) rc = then(g);
      msf_free(g);
      return rc;
    };
  };
  auto batch = [&](std::vector<int64_t> nv, std::vector<int64_t> ne) {
    static std::vector<int64_t> vo, eo;
    vo = {0}, eo = {0};
    for (size_t i = 0; i < nv.size(); ++i) vo.push_back(vo.back() + nv[i]), eo.push_back(eo.back() + ne[i]);
    const int64_t n = vo.back(), m = eo.back();
    auto *s = (int32_t *)array((size_t)m * 4), *d = (int32_t *)array((size_t)m * 4);
    void *w = array((size_t)m * 4);
    auto *mk = (uint8_t *)array((size_t)m);
    auto *lb = (int32_t *)array((size_t)n * 4);
    auto *tt = (double *)array(nv.size() * 8);
    call = [=]() {
      return msf_compute_batched((int32_t)vo.size() - 1, vo.data(), eo.data(), s, d, w, MSF_F32, mk, lb, tt, nullptr);
    };
  };
  auto outputs = [&](int64_t n, int64_t m) {
    auto *mk = (uint8_t *)array((size_t)m);
    auto *lb = (int32_t *)array((size_t)n * 4);
    auto *tt = (double *)array(8);
    return [=](msf_graph *g) { return msf_compute(g, mk, lb, tt, nullptr); };
  };
  const std::string what = name.substr(0, name.find(' '));
  if (what == "build_one") graph(100, 300, false, nullptr);
  else if (what == "build") graph(20000, 60000, false, nullptr);
  else if (what == "build_sampled") graph(20000, 1 << 20, false, nullptr);
  else if (what == "build_csr") graph(20000, 60000, true, nullptr);
  else if (what == "build_csr_large") graph(20000, 13 << 20, true, nullptr);
  else if (what == "build_radix" || what == "build_bucket") {
    msf::options().build_mode = what == "build_radix" ? 2 : 3;
    graph(20000, 60000, false, nullptr);
  } else if (what == "compute_small") graph(100, 300, false, outputs(100, 300));
  else if (what == "compute_loop") {
    graph(20000, 60000, false, outputs(20000, 60000));
    auto build = call;
    call = [=]() {  // (the build with its default options)
      return build();
    };
    msf::options().exec_mode = 0;
    msf::options().tau = 0.25;
  } else if (what == "compute") graph(20000, 60000, false, outputs(20000, 60000));
  else if (what == "components") {
    auto *lb = (int32_t *)array(20000 * 4);
    graph(20000, 60000, false, [=](msf_graph *g) { return msf_connected_components(g, lb, nullptr); });
  } else if (what == "min_edge") {
    auto *p = (int32_t *)array(20000 * 4);
    auto *r = (uint64_t *)array(20000 * 8);
    graph(20000, 60000, false, [=](msf_graph *g) {
      const int rc = msf_min_edge(g, p, r, nullptr);
      return rc ? rc : msf_min_edge_part(g, p, 1, 3, r, nullptr);
    });
  } else if (what == "one_small") batch({100}, {300});
  else if (what == "one") batch({50000}, {200000});
  else if (what == "batch_small") batch({100, 300, 5000}, {300, 900, 20000});
  else if (what == "batch") batch({100, 70000, 300, 80000}, {300, 100000, 0, 90000});
  else if (what == "backward") {
    auto *mk = (uint8_t *)array(1000);
    auto *gt = (double *)array(8 * 3);
    auto *gw = (float *)array(4000);
    static const int64_t eo[4] = {0, 10, 500, 1000};
    call = [=]() { return msf_weight_backward(1000, 3, eo, mk, gt, gw, nullptr); };
  } else {
    std::printf("no scenario %s\n", name.c_str());
    return 2;
  }
  const size_t live = blocks.size();
  auto once = [&](const char *how, long k) {
    found.clear();
    const size_t before = blocks.size();
    allocs = calls = 0;
    const int rc = call();
    if (blocks.size() != before) found.push_back(std::to_string(blocks.size() - before) + " blocks not given back");
    for (const auto &f : found) std::printf("%s %ld (result %d): %s\n", how, k, rc, f.c_str());
    cudaStreamSynchronize(nullptr);
    for (auto &b : blocks) b.second.busy.clear();
    while (blocks.size() > live) {  // (lost blocks are reported once)
      bool any = false;
      for (auto &b : blocks)
        if (b.second.kind == 0) {
          used -= b.second.bytes;
          blocks.erase(b.first);
          any = true;
          break;
        }
      if (!any) break;
    }
    return rc;
  };
  if (argc > 2) {
    auto least = [&]() {
      size_t lo = 0, hi = (size_t)1 << 32;
      while (hi - lo > 1) {
        budget = (lo + hi) / 2;
        (once("budget", (long)budget) == MSF_ERR_OOM ? lo : hi) = budget;
      }
      return hi;
    };
    const size_t a = least();
    refused = (size_t)std::atol(argv[2]);
    std::printf("%zu %zu\n", a, least());
    return 0;
  }
  const int rc = once("plain", 0);
  const long na = allocs, nc = calls;
  for (long k = 0; k < na; ++k) {
    fail_alloc = k;
    once("allocation", k);
  }
  fail_alloc = -1;
  for (long k = 0; k < nc; ++k) {
    fail_call = k;
    once("call", k);
  }
  std::printf("done: result %d, %ld allocations, %ld calls\n", rc, na, nc);
  return 0;
}
