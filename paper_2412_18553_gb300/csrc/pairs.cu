// The epilogue inputs of the exact-slice adjoint and projected energy as FP32
// pairs (adjoint_tc.cuh).
#include <algorithm>

#include "adjoint_tc.cuh"

namespace te {

namespace {

__global__ void __launch_bounds__(256) k_pair_inputs(const double* __restrict__ ovov, const double* __restrict__ t1,
                                                     const double* __restrict__ eps_o, const double* __restrict__ eps_v,
                                                     int o, int v, PairBuffers b) {
  const int eo = exp_of_high(b.hi[0]), et = exp_of_high(b.hi[1]);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    reinterpret_cast<int*>(b.hi)[2] = eo;
    reinterpret_cast<int*>(b.hi)[3] = et;
  }
  const double fo = ldexp(0.5, -eo), ft = ldexp(1.0, -et);
  const int64_t n = (int64_t)o * v * o * v, n1 = (int64_t)o * v, ne = o + v;
  for (int64_t e = blockIdx.x * 256LL + threadIdx.x; e < n + n1 + ne; e += gridDim.x * 256LL) {
    if (e < n) {
      const int64_t row = e / v;  // (i v + a) o + j
      const int y = (int)(e - row * v), j = (int)(row % o);
      const int64_t ia = row / o;
      const int a = (int)(ia % v), i = (int)(ia / v);
      b.ovs[e] = pr_of(fo * (ovov[e] + ovov[(((int64_t)j * v + y) * o + i) * v + a]));
    } else if (e < n + n1) {
      b.t1[e - n] = pr_of(ft * t1[e - n]);
    } else {
      const int64_t q = e - n - n1;
      b.eps[q] = pr_of(q < o ? eps_o[q] : eps_v[q - o]);
    }
  }
}

}  // namespace

cudaError_t launch_pair_inputs(const te_cluster* c, const PairBuffers& b, cudaStream_t s) {
  const int64_t o = c->nocc, v = c->nvir, n = o * v * o * v + o * v + o + v;
  k_pair_inputs<<<(unsigned)std::min<int64_t>((n + 255) / 256, 16384), 256, 0, s>>>(c->ovov, c->t1, c->eps_o, c->eps_v,
                                                                                    (int)o, (int)v, b);
  return cudaGetLastError();
}

}  // namespace te
