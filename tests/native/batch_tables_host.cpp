// The batch's tables on the host, against a fake of the CUDA runtime: this program defines the runtime calls
// that the library's batch code makes, ahead of the real ones, over host memory.  Prints "ok" or what went
// wrong.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <string>
#include <vector>

#include "../../include/lbm_d2q37.h"

static std::map<void*, size_t> g_blocks;     // allocations alive
static std::vector<void*> g_launched;        // tables that a launch was given
static bool g_destroying = false;
static int g_fail_malloc = 0;                // fail the n-th next allocation
static size_t g_new_limit = 0;               // refuse larger host allocations (0: none)
static std::string g_wrong;

static void wrong(const char* what) {
  if (g_wrong.empty()) g_wrong = what;
}

void* operator new(size_t n) {
  if (g_new_limit && n > g_new_limit) throw std::bad_alloc();
  if (void* p = std::malloc(n)) return p;
  throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }

extern "C" {
#undef cudaGetDeviceProperties
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  std::memset(p, 0, sizeof(*p));
  p->multiProcessorCount = 152;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) {
  if (g_fail_malloc && --g_fail_malloc == 0) return cudaErrorMemoryAllocation;
  *p = std::malloc(n);
  g_blocks[*p] = n;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  if (!g_blocks.erase(p)) wrong("freed twice");
  for (void* t : g_launched)
    if (t == p && !g_destroying) wrong("a table in use was freed");
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* dst, const void* src, size_t n, cudaMemcpyKind) {
  for (void* t : g_launched)
    if (t == dst) wrong("a table in use was written");
  const auto b = g_blocks.find(dst);
  if (b == g_blocks.end() || b->second < n) return wrong("copy out of bounds"), cudaErrorInvalidValue;
  std::memcpy(dst, src, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  return *n = 2, cudaSuccess;
}
// a step of a batch: arguments (lattices, tiles, number of tiles, ...) of either mode
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* cfg, const void*, void** args) {
  void* tiles = *(void**)args[1];
  const long long total = *(long long*)args[2];
  const auto b = g_blocks.find(tiles);
  if (b == g_blocks.end() || b->second < (size_t)total * 16) return wrong("launched without its table"), cudaSuccess;
  const int* t = (const int*)tiles;  // lattice, x0, y0, pad: lattice 0 is 20 x 70
  long long n = 0;
  for (; n < total && t[4 * n] == 0; ++n)
    if (t[4 * n + 1] >= 20 || t[4 * n + 1] % (int)cfg->blockDim.y || t[4 * n + 2] >= 70) wrong("a tile out of its lattice");
  const long long w = cfg->blockDim.y;
  if (n != (20 + w - 1) / w * 3) wrong("tiles missing");
  g_launched.push_back(tiles);
  return cudaSuccess;
}
}

static void expect(int32_t got, int32_t want, const char* what) {
  if (got != want) wrong(what);
}

int main(int argc, char** argv) {
  const std::string what = argc > 1 ? argv[1] : "";
  lbm_params p[2] = {};
  for (int j = 0; j < 2; ++j) p[j] = {j ? 9 : 20, j ? 33 : 70, LBM_FP64, LBM_BC_WALLS, 0.8, 0.0, -1e-4, 1.15, 0.85, 1.0};
  void *fa[2] = {(void*)0x10000000, (void*)0x20000000}, *fb[2] = {(void*)0x30000000, (void*)0x40000000};
  lbm_batch* b = nullptr;
  if (what == "in_flight") {  // the tables of runs that may still be in flight stay as they are
    expect(lbm_batch_plan(p, fa, fb, 2, &b), LBM_OK, "plan");
    for (int tx : {4, 1, 8, 2, 4, 8, 1})
      for (int mode : {LBM_BATCH_PER_STEP, LBM_BATCH_PERSISTENT}) {
        expect(lbm_batch_configure(b, mode, tx, 0), LBM_OK, "configure");
        expect(lbm_batch_run(b, 2, nullptr), LBM_OK, "run");
      }
  } else if (what == "no_device_memory") {  // the configuration before stays, and runs
    expect(lbm_batch_plan(p, fa, fb, 2, &b), LBM_OK, "plan");
    expect(lbm_batch_configure(b, LBM_BATCH_PER_STEP, 8, 0), LBM_OK, "configure");
    g_fail_malloc = 1;
    expect(lbm_batch_configure(b, LBM_BATCH_PERSISTENT, 1, 3), LBM_ENOMEM, "no device memory");
    int32_t mode = 0, tx = 0;
    lbm_batch_config(b, &mode, &tx, nullptr);
    if (mode != LBM_BATCH_PER_STEP || tx != 8) wrong("the configuration changed");
    expect(lbm_batch_run(b, 1, nullptr), LBM_OK, "run");
    expect(lbm_batch_configure(b, LBM_BATCH_PERSISTENT, 1, 0), LBM_OK, "configure again");
    expect(lbm_batch_run(b, 1, nullptr), LBM_OK, "run");
  } else if (what == "no_host_memory") {  // an error, not an exception
    try {
      expect(lbm_batch_plan(p, fa, fb, 2, &b), LBM_OK, "plan");
      g_new_limit = 256;
      expect(lbm_batch_configure(b, LBM_BATCH_PER_STEP, 1, 0), LBM_ENOMEM, "no host memory");
      lbm_batch* other = nullptr;
      expect(lbm_batch_plan(p, fa, fb, 2, &other), LBM_ENOMEM, "no host memory for a plan");
      if (other) wrong("a batch without memory");
      g_new_limit = 0;
      expect(lbm_batch_run(b, 1, nullptr), LBM_OK, "run");
    } catch (...) {
      wrong("an exception left the library");
    }
  } else if (what == "plan") {  // every allocation of a plan failing in turn: nothing is left behind
    for (int n = 1; n <= 3; ++n) {
      g_fail_malloc = n;
      if (lbm_batch_plan(p, fa, fb, 2, &b) == LBM_OK || b) wrong("a plan without memory");
      if (!g_blocks.empty()) wrong("memory left behind");
    }
    g_fail_malloc = 0;
    expect(lbm_batch_plan(p, fa, fb, 2, &b), LBM_OK, "plan");
  } else {
    wrong("which test?");
  }
  g_destroying = true;
  lbm_batch_destroy(b);
  if (!g_blocks.empty()) wrong("memory left behind");
  std::printf("%s\n", g_wrong.empty() ? "ok" : g_wrong.c_str());
  return 0;
}
