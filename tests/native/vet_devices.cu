// sas_vet.cu over a fake of the runtime's device calls, for tests without a GPU:
// which kernels were given their shared-memory limit on which device.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <vector>

namespace fake {
int device = 0;
std::map<int, std::set<const void*>> limits;
template <typename F>
cudaError_t set_attribute(F f, cudaFuncAttribute, int) {
  limits[device].insert((const void*)f);
  return cudaSuccess;
}
inline cudaError_t get_device(int* d) {
  *d = device;
  return cudaSuccess;
}
inline cudaError_t set_device(int d) {
  device = d;
  return cudaSuccess;
}
inline cudaError_t device_attribute(int* v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
inline cudaError_t allocate(void** p, size_t) {
  *p = std::malloc(1);
  return cudaSuccess;
}
inline cudaError_t release(void* p) {
  std::free(p);
  return cudaSuccess;
}
}  // namespace fake

#define cudaFuncSetAttribute fake::set_attribute
#define cudaGetDevice fake::get_device
#define cudaSetDevice fake::set_device
#define cudaDeviceGetAttribute fake::device_attribute
#define cudaMalloc fake::allocate
#define cudaFree fake::release
#define cudaMemset(p, v, n) cudaSuccess
#define cudaDeviceSynchronize() cudaSuccess
#include "../../paper_2509_26279_gb300/csrc/sas_vet.cu"

// Creates a vetter on `device`; returns the number of kernels with a limit there, -1 on an error.
extern "C" int limits_after_create(int device) {
  sas_vet* vt = nullptr;
  if (sas_vet_create(device, 16, &vt) != SAS_OK) return -1;
  free_vet(vt);
  return (int)fake::limits[device].size();
}
