// Host-side failure of the MP2 step's tensor-core product, without a GPU: links
// the product's own object (mp2.cu) against fakes of everything it calls, the
// product failing, and counts what the call allocates and gives back.
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <new>

#include "te_internal.h"

struct __nv_bfloat16;
namespace te {
struct GemmView;
}

static long live = 0;
void* operator new(std::size_t n) {
  ++live;
  return std::malloc(n);
}
void* operator new(std::size_t n, const std::nothrow_t&) noexcept {
  ++live;
  return std::malloc(n);
}
void operator delete(void* p) noexcept {
  if (p) --live;
  std::free(p);
}
void operator delete(void* p, std::size_t) noexcept { operator delete(p); }

namespace te {
te_status fail(te_status st, const char*, ...) { return st; }
te_status ensure_workspace_public(Handle* h, size_t bytes) {
  h->ws_bytes = bytes;
  return TE_OK;
}
int64_t splitk_cap(int64_t, int64_t) { return 0; }
cudaError_t launch_check_mp2(const double*, int64_t, const double*, int64_t, const double*, int64_t, int64_t,
                             unsigned int*, int, cudaStream_t, unsigned int*) {
  return cudaSuccess;
}
cudaError_t slice_rows(const double*, int64_t, int64_t, int64_t, int, const unsigned int*, int*, __nv_bfloat16*,
                       cudaStream_t, int64_t*) {
  return cudaSuccess;
}
cudaError_t gemm_strided(const GemmView&, int, double*, int64_t, cudaStream_t, int64_t*) { return cudaSuccess; }
te_status vt_product(Handle*, const void*, int64_t, int64_t, const void*, int64_t, int64_t, int64_t, int64_t, int,
                     const int*, const int*, double*, cudaStream_t) {
  return TE_EUNSUPPORTED;  // the failure under test
}
}  // namespace te

extern "C" {
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return ""; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t __cudaGetKernel(void**, const void*) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
char __cudaInitModule(void**) { return 0; }
}

int main() {
  te::Handle h;
  h.cc_major = 10;
  h.num_sms = 152;
  double x = 0.0;
  const te_mp2_cluster c{2, 3, 4, &x, &x, &x};
  te_mp2_out o{};
  o.pop_o = &x;
  const long before = live;
  const te_status st = t_mp2_bno_batched(reinterpret_cast<te_handle>(&h), &c, &o, 1, TE_OZAKI, nullptr);
  std::printf("%d %ld\n", (int)st, live - before);
  return 0;
}
