// The quadratic ACE kernel (ace_quad.cuh): body order 4 in float32.
#include <type_traits>
#include <vector>

#include "apip_internal.h"
#include "gaunt_layout.h"

namespace apip {
namespace {
__constant__ float c_norm[(kLmaxCap + 1) * (kLmaxCap + 1)];
__constant__ float c_gaunt[kGaunt4Total];
struct Consts {
  static __device__ __forceinline__ float ynorm(int k) { return c_norm[k]; }
  static __device__ __forceinline__ float gaunt(int e) { return c_gaunt[e]; }
};
}  // namespace
}  // namespace apip

#include "ace_quad.cuh"

namespace apip {

cudaError_t ace_quad_set_consts(const double* norms, int count) {
  std::vector<double> gd(kGaunt4Total);
  gaunt4_fill(gd.data());
  std::vector<float> f(norms, norms + count), gv(gd.begin(), gd.end());
  const cudaError_t e = cudaMemcpyToSymbol(c_norm, f.data(), sizeof(float) * count);
  if (e != cudaSuccess) return e;
  return cudaMemcpyToSymbol(c_gaunt, gv.data(), sizeof(float) * kGaunt4Total);
}

void launch_ace_quad(const Args<float>& a, const AceDev<float>& t, int blocks, cudaStream_t s) {
  quad_dispatch<Consts>(&a, t, blocks, s, false);
}

int ace_quad_occupancy(const AceDev<float>& t) { return quad_dispatch<Consts>(nullptr, t, 0, nullptr, true); }

}  // namespace apip
