// fake_cudart.cpp -- a stand-in for the CUDA runtime, preloaded before the
// library in a child process (test_host_launches_cpu.py): the host code plans,
// allocates and launches as on a device of 152 SMs with 227 KB of shared memory
// a block, and nothing runs.  Device pointers are host addresses of known
// extent; every copy, clear and kernel argument is checked against them, and a
// violation or a launch is a line of the log.
#include <dlfcn.h>
#include <sys/mman.h>
#include <unistd.h>

#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

#include <cuda_runtime.h>

#include "../paper_2402_13259_gb300/csrc/internal.h"

using namespace eulernet;

namespace {

std::map<uintptr_t, size_t>& blocks() {
  static auto* m = new std::map<uintptr_t, size_t>();
  return *m;
}
std::map<const void*, std::string>& kernels() {
  static auto* m = new std::map<const void*, std::string>();
  return *m;
}
std::string& text() {
  static auto* s = new std::string();
  return *s;
}
std::map<const void*, int>& smem_limit() {
  static auto* m = new std::map<const void*, int>();
  return *m;
}
std::recursive_mutex all;  // several threads may call
#define LOCKED std::lock_guard<std::recursive_mutex> lock_(all)
thread_local cudaError_t last_error = cudaSuccess;  // kept until it is asked for
cudaError_t failed(cudaError_t e) { return last_error = e; }
long long fail_from = 0, allocs = 0;  // allocations numbered from fail_from on fail (0: none)

void line(const char* fmt, const char* what, long long a, long long b) {
  char buf[256];
  std::snprintf(buf, sizeof buf, fmt, what, a, b);
  text() += buf;
}

// [p, p + bytes) lies inside one allocation.
void within(const void* p, int64_t bytes, const char* what) {
  if (bytes <= 0) return;
  const uintptr_t a = (uintptr_t)p;
  auto it = blocks().upper_bound(a);
  if (it != blocks().begin()) {
    --it;
    if (a - it->first <= it->second && (uint64_t)bytes <= it->second - (a - it->first)) return;
    line("VIOLATION %s: %lld bytes, %lld there\n", what, bytes,
         a - it->first < it->second ? (long long)(it->second - (a - it->first)) : 0);
    return;
  }
  line("VIOLATION %s: %lld bytes, %lld there\n", what, bytes, 0);
}

void check_hbm(const NetTables* t, const RunParams& p, const HbmState& hs, const char* who, bool scores, bool soj) {
  const std::string w = std::string(who) + " ";
  if (hs.ld < p.R) line("VIOLATION %s: ld %lld below R %lld\n", who, hs.ld, p.R);
  if (t) {
    within(hs.N, 4 * (int64_t)t->n * hs.ld, (w + "N").c_str());
    within(hs.Redge, 4 * (int64_t)(hs.depth > 2 ? hs.depth : 2) * t->E * hs.ld, (w + "Redge").c_str());
    within(hs.racc, 32 * p.R, (w + "racc").c_str());
    if (scores) {
      within(hs.mu_acc, 8 * (int64_t)t->n * hs.ld, (w + "mu_acc").c_str());
      within(hs.th_acc, 24 * (int64_t)t->n_ex * hs.ld, (w + "th_acc").c_str());
    }
  }
  if (soj) {
    within(hs.cloc, 8 * (int64_t)hs.S * hs.ld, (w + "cloc").c_str());
    within(hs.cpos, 4 * (int64_t)hs.S * hs.ld, (w + "cpos").c_str());
    within(hs.csteps, 4 * (int64_t)hs.S * hs.ld, (w + "csteps").c_str());
  }
}

cudaError_t launched(const void* fn, dim3 grid, dim3 block, void** a, size_t smem) {
  LOCKED;
  if (smem > 48 * 1024 && (int)smem > smem_limit()[fn]) return failed(cudaErrorInvalidValue);
  const std::string name = kernels()[fn];
  auto is = [&](const char* s) { return name.find(s) != std::string::npos; };
  auto net = [&](int k) { return static_cast<const NetTables*>(a[k]); };
  auto run = [&](int k) -> const RunParams& { return *static_cast<const RunParams*>(a[k]); };
  auto hbm = [&](int k) -> const HbmState& { return *static_cast<const HbmState*>(a[k]); };
  if (is("persistent_kernel")) {
    const RunParams& p = run(1);
    within(p.acc, 8 * p.acc_stride * (int64_t)grid.x, "persistent_kernel acc");
    line("persistent_kernel %s tile_reps=%lld tiles=%lld", "", p.tile_reps, p.num_tiles - p.tile0);
    line("%s block=%lld smem=%lld\n", "", (long long)block.x, (long long)smem);
  } else if (is("batch_kernel")) {
    const int64_t slot = *static_cast<int64_t*>(a[6]);
    within(*static_cast<void**>(a[5]), 8 * slot * (int64_t)grid.x, "batch_kernel sums");
    within(*static_cast<void**>(a[2]), 8 * (int64_t)*static_cast<int*>(a[3]), "batch_kernel items");
    line("batch_kernel %s items=%lld block=%lld\n", "", *static_cast<int*>(a[3]), (long long)block.x);
  } else if (is("hbm_phase_kernel")) {
    const HbmState& hs = hbm(2);
    check_hbm(net(0), run(1), hs, "hbm_phase_kernel", hs.mu_acc != nullptr, hs.cloc != nullptr);
    line("hbm_phase_kernel %s R=%lld block=%lld\n", "", run(1).R, (long long)block.x);
  } else if (is("hbm_init_kernel") || is("hbm_finish_kernel")) {
    check_hbm(net(0), run(1), hbm(2), "hbm_init/finish", false, false);
  } else if (is("hbm_scores_kernel")) {
    check_hbm(net(0), run(1), hbm(2), "hbm_scores_kernel", true, false);
  } else if (is("hbm_sojourn_init") || is("hbm_sojourn_finish")) {
    check_hbm(nullptr, run(0), hbm(1), "hbm_sojourn", false, true);
  }
  return cudaSuccess;
}

}  // namespace

extern "C" {

const char* fake_log() { return text().c_str(); }
void fake_clear() { text().clear(); }
// The n-th allocation from now on and all that follow it fail (0: none).
void fake_fail_malloc(long long n) {
  allocs = 0;
  fail_from = n;
}
long long fake_live_bytes() {
  long long s = 0;
  for (auto& b : blocks()) s += (long long)b.second;
  return s;
}

void __cudaRegisterFunction(void** h, const char* host, char* dev, const char* name, int lim, uint3* tid, uint3* bid,
                            dim3* bd, dim3* gd, int* ws) {
  kernels()[host] = name;
  using Fn = void (*)(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*);
  static Fn real = (Fn)dlsym(RTLD_NEXT, "__cudaRegisterFunction");
  if (real) real(h, host, dev, name, lim, tid, bid, bd, gd, ws);
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fn) {
  *k = (cudaKernel_t)fn;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** a, size_t smem, cudaStream_t) {
  return launched((const void*)k, g, b, a, smem);
}
cudaError_t cudaLaunchKernel(const void* fn, dim3 g, dim3 b, void** a, size_t smem, cudaStream_t) {
  return launched(fn, g, b, a, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void** a) {
  return launched(fn, c->gridDim, c->blockDim, a, c->dynamicSmemBytes);
}

cudaError_t cudaMalloc(void** p, size_t n) {
  LOCKED;
  *p = nullptr;
  if (fail_from > 0 && ++allocs >= fail_from) return failed(cudaErrorMemoryAllocation);
  void* q = mmap(nullptr, n ? n : 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (q == MAP_FAILED) return failed(cudaErrorMemoryAllocation);
  blocks()[(uintptr_t)q] = n;
  *p = q;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  LOCKED;
  if (!p) return cudaSuccess;
  auto it = blocks().find((uintptr_t)p);
  if (it == blocks().end()) {
    line("VIOLATION %s: %lld %lld\n", "free of an address not allocated", 0, 0);
    return failed(cudaErrorInvalidValue);
  }
  munmap(p, it->second ? it->second : 1);
  blocks().erase(it);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) {
  LOCKED;
  within(p, (int64_t)n, "memset");
  if (n <= 4096 && blocks().count((uintptr_t)p)) std::memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) {
  LOCKED;
  within(k == cudaMemcpyDeviceToHost ? s : d, (int64_t)n, "memcpy");
  if (k == cudaMemcpyDeviceToHost) std::memset(d, 0, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  return cudaMemcpy(d, s, n, k);
}

cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr at, int) {
  *v = at == cudaDevAttrMultiProcessorCount ? 152 : at == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 227 * 1024 : 0;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* v, const void*, int block, size_t smem) {
  const int by_regs = 65536 / (64 * block), by_smem = (int)(228 * 1024 / (smem + 1024));
  *v = by_regs < by_smem ? by_regs : by_smem;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* fn, cudaFuncAttribute, int bytes) {
  usleep(20);  // another thread's call may come between this one and the launch
  LOCKED;
  // what a function's static memory leaves (batch_kernel: its work item's tables)
  const int most = 227 * 1024 - (kernels()[fn].find("batch_kernel") != std::string::npos ? 448 : 0);
  if (bytes > most) return failed(cudaErrorInvalidValue);
  smem_limit()[fn] = bytes;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = last_error;
  last_error = cudaSuccess;
  return e;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = (cudaStream_t)0x10;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  *g = (cudaGraph_t)0x20;
  return cudaSuccess;
}
bool capturing = false;
void fake_capturing(int on) { capturing = on != 0; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* st) {
  *st = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = (cudaGraphExec_t)0x30;
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  *e = (cudaEvent_t)0x40;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  static int k = 0;
  *ms = (float)(++k * 37 % 101 + 1);  // some order among an autotuner's trials
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }

}  // extern "C"
