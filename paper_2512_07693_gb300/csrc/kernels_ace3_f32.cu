// float instantiation of the body-order <= 3 ACE kernel (ace_stream.cuh), l_max <= 3.
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

template <> cudaError_t ace_stream_set_consts<float>(const double* norms, int count, const double* gaunt) {
  std::vector<float> f(norms, norms + count), gv(gaunt, gaunt + kGauntTotal);
  const cudaError_t e = cudaMemcpyToSymbol(c_norm, f.data(), sizeof(float) * count);
  if (e != cudaSuccess) return e;
  const cudaError_t e2 = cudaMemcpyToSymbol(c_gaunt, gv.data(), sizeof(float) * kGauntTotal);
  return e2 != cudaSuccess ? e2 : ace_stream_l4_set_consts<float>(norms, count, gaunt);
}

template <> void launch_ace_stream<float>(const Args<float>& a, const AceDev<float>& t, cudaStream_t s) {
  stream_launch<float, Consts>(a, t, s);
}

template <> int ace_stream_occupancy<float>(const AceDev<float>& t) {
  return stream_dispatch<float, Consts>(nullptr, t, t.group, 0, nullptr, true);
}

}  // namespace apip
