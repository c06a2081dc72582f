// CUDA runtime calls that plan configuration makes, faked for a host without a
// GPU: every kernel reports g_fake_registers registers a thread, and tensor maps
// encode without a driver.  Linked before the shared runtime library.
#include <cuda.h>
#include <cuda_runtime_api.h>

int g_fake_registers = 64;

static CUresult fake_encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                            const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                            CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}

extern "C" {
cudaError_t CUDARTAPI cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  *a = cudaFuncAttributes{};
  a->numRegs = g_fake_registers;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 228 * 1024;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                                       cudaDriverEntryPointQueryResult* q) {
  *f = reinterpret_cast<void*>(fake_encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
}
