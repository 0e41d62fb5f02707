// Host-only harness of the network context's set-up (kp_mlp.cu), for CPU
// tests: the CUDA runtime's calls on the way are replaced by fakes that record
// what was asked of which device.  No device code runs: the first copy to the
// device reports an error, and kp_mlp_create returns it before any launch.
#include <cuda_runtime.h>

#include <vector>

namespace fake {
struct Limit {
  int device;
  const void* kernel;
  int bytes;
};
int device = 0;
std::vector<Limit> limits;

cudaError_t get_device(int* d) {
  *d = device;
  return cudaSuccess;
}
cudaError_t get_attribute(int* v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
template <class T>
cudaError_t set_attribute(T* kernel, cudaFuncAttribute a, int bytes) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize)
    limits.push_back({device, reinterpret_cast<const void*>(kernel), bytes});
  return cudaSuccess;
}
cudaError_t copy(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t last_error() { return cudaSuccess; }
}  // namespace fake

#define cudaGetDevice fake::get_device
#define cudaDeviceGetAttribute fake::get_attribute
#define cudaFuncSetAttribute fake::set_attribute
#define cudaMemcpyAsync fake::copy
#define cudaGetLastError fake::last_error
#include "../../paper_2409_06807_gb300/csrc/kp_mlp.cu"

extern "C" {

// Creates (as far as the first copy) a network on the device numbered
// 'device'; returns kp_mlp_create's status.
int kpt_mlp_create_on(int device) {
  fake::device = device;
  std::vector<float> params((size_t)kp_mlp_num_params(), 0.0f);
  kp_mlp* n = nullptr;
  return kp_mlp_create(reinterpret_cast<void*>(4096), kp_mlp_required_bytes(64), 64, params.data(),
                       nullptr, &n);
}

// The shared memory limit that the device has for the inference (0) or the
// training (1) kernel, 0 when none was set there.
int kpt_mlp_limit(int device, int training) {
  const void* k = training ? (const void*)kp::tc::kp_mlp_train_kernel
                           : (const void*)kp::tc::kp_mlp_forward_tc_kernel;
  int bytes = 0;
  for (const auto& l : fake::limits)
    if (l.device == device && l.kernel == k) bytes = l.bytes;
  return bytes;
}
int kpt_mlp_needs(int training) { return training ? kp::tc::ST_SMEM : kp::tc::FT_SMEM; }

}  // extern "C"
