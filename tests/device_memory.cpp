// Host harness of test_device_memory.py: the context management of apip.cu against a
// fake CUDA runtime (no GPU, no CUDA library) whose device has a given number of bytes.
// For a float64 context and a box it finds the bytes that the context cannot do without
// (the most it holds when only that fits), then gives the device that much and more, up
// to the pair terms' size beyond, and creates the context and sets the box each time.
// Prints "<lam_mode> <needed> <kept pair terms on a large device> <refusals> <budgets>".
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <map>
#include <vector>

#include "apip.h"
#include "apip_internal.h"

static size_t g_budget, g_used, g_most;
static std::map<void*, size_t> g_live;

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) {
  if (g_used + n > g_budget) return cudaErrorMemoryAllocation;
  *p = std::malloc(1);
  g_live[*p] = n;
  g_used += n;
  g_most = g_used > g_most ? g_used : g_most;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  g_used -= g_live[p];
  g_live.erase(p);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = g_budget - g_used; *t = g_budget; return cudaSuccess; }
cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "out of memory"; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
// (what a translation unit of nvcc calls at start and exit)
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
}

namespace apip {   // (as declared in kernels.h)
template <typename T> int ace_stream_occupancy(const AceDev<T>&);
template <typename T> cudaError_t ace_stream_set_consts(const double*, int, const double*);
template <> int ace_stream_occupancy<double>(const AceDev<double>&) { return 2; }
template <> cudaError_t ace_stream_set_consts<double>(const double*, int, const double*) { return cudaSuccess; }
cudaError_t exp_table_set() { return cudaSuccess; }
}  // namespace apip

// creates the context and gives it a box; true if neither is refused
static bool run(const apip_params& p, size_t budget) {
  g_budget = budget;
  g_most = 0;
  apip_ctx* c = nullptr;
  const double box[3] = {300, 300, 300};
  bool ok = apip_create(&p, 20000, &c) == APIP_OK;
  ok = ok && apip_build_neighbors(c, nullptr, box, nullptr, 0, nullptr) == APIP_OK;
  if (c) apip_destroy(c);
  if (g_used) std::abort();
  return ok;
}

int main() {
  for (int mode : {APIP_LAM_PAPER, APIP_LAM_LEARNED}) {
    apip_params p = {};
    p.precision = APIP_FP64;
    p.lam_mode = mode;
    p.eam_rc = 4.4; p.eam_rc_width = 0.5;
    p.ace_n_max = 2; p.ace_l_max = 1; p.ace_nu_max = 2; p.ace_rc = 5; p.ace_rc_width = 1; p.ace_eps = 0.01;
    p.ace_n_basis = apip_ace_basis_size(2, 1, 2);
    std::vector<double> c(p.ace_n_basis, 0.1);
    p.ace_c1 = p.ace_c2 = c.data();
    p.sw_r_w = 5; p.sw_r_w_width = 1; p.sw_d_hi = 1; p.csp_rcut = 4.5; p.csp_nnb = 8;
    p.skin = 0.5; p.max_nb = 80; p.cell_cap = 48;
    const size_t keep = (size_t)16 * 20000 * 40;
    run(p, (size_t)1 << 40);
    const size_t most = g_most;
    // the least budget that is accepted, by bisection
    size_t lo = 0, hi = most;
    while (hi - lo > 1) {
      const size_t mid = lo + (hi - lo) / 2;
      (run(p, mid) ? hi : lo) = mid;
    }
    int refused = 0, tried = 0;
    for (size_t b = hi; b <= hi + 2 * keep; b += keep / 64) {
      ++tried;
      refused += run(p, b) ? 0 : 1;
    }
    std::printf("%d %zu %d %d %d\n", mode, hi, most - hi == keep ? 1 : 0, refused, tried);
  }
  return 0;
}
