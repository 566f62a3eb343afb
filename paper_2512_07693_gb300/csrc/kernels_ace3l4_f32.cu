// float instantiation of the body-order <= 3 ACE kernel (ace_stream.cuh), l_max = 4: half
// of these kernels' compile time, in a translation unit of its own.
#include <vector>

#include "apip_internal.h"
#include "gaunt_layout.h"

namespace apip {
namespace {
__constant__ float c_norm[(kLmaxCap + 1) * (kLmaxCap + 1)];
__constant__ float c_gaunt[kGauntTotal];
struct Consts {
  static __device__ __forceinline__ float ynorm(int k) { return c_norm[k]; }
  static __device__ __forceinline__ float gaunt(int e) { return c_gaunt[e]; }
};
}  // namespace
}  // namespace apip

#include "ace_stream.cuh"

namespace apip {

template <> cudaError_t ace_stream_l4_set_consts<float>(const double* norms, int count, const double* gaunt) {
  std::vector<float> f(norms, norms + count), gv(gaunt, gaunt + kGauntTotal);
  const cudaError_t e = cudaMemcpyToSymbol(c_norm, f.data(), sizeof(float) * count);
  if (e != cudaSuccess) return e;
  return cudaMemcpyToSymbol(c_gaunt, gv.data(), sizeof(float) * kGauntTotal);
}

template <> int ace_stream_l4<float>(const Args<float>* a, const AceDev<float>& t, int group, int blocks, cudaStream_t s,
                                      bool query) {
  return stream_g<float, Consts, 4>(a, t, group, blocks, s, query);
}

}  // namespace apip
