// kp_mlp.cu -- the learned proposal's network: the kp_mlp_* entry points of
// include/kp.h.  Inference and training (forward, backward, Adam) are one
// kernel each on the tcgen05 tensor cores (kp_mlp_tc.cuh: BF16 operands, FP32
// accumulation in tensor memory); FP32 master weights and Adam moments.
// Like the planner, the network context allocates no device memory: it
// lives in a caller-owned arena.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <new>

#include "../../include/kp.h"
#include "kp_mlp.cuh"
#include "kp_mlp_tc.cuh"
#include "kp_tc.cuh"

namespace kp {

using bf16 = __nv_bfloat16;

using tc::N_PARAMS;
using tc::OFF_B1;
using tc::OFF_B2;
using tc::OFF_B3;
constexpr int N_WEIGHTS_BF16 = MLP_H * MLP_IN + MLP_H * MLP_H + MLP_OUT * MLP_H;

// ---------------------------------------------------------------------------
// Adam on the FP32 master vector; refreshes the BF16 weight copies
// ---------------------------------------------------------------------------

// One Adam step; the loss to *loss.
__global__ void kp_mlp_adam_kernel(tc::AdamArgs a, float c1, float c2, float* loss) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N_PARAMS / 4)
    tc::adam_update(a, i, c1, c2);
  else if (i == N_PARAMS / 4)
    *loss = tc::slot_sum(a.slots, a.n_slots, i).x;
}

// The gradient and, after it, the loss: the sums over the slots.
__global__ void kp_mlp_gradient_kernel(const float* slots, int n, float* g) {
  const int gr = blockIdx.x * blockDim.x + threadIdx.x;
  if (gr < tc::SLOT / 4)
    *reinterpret_cast<float4*>(g + tc::slot_param(gr)) = tc::slot_sum(slots, n, gr);
}

__global__ void kp_mlp_round_kernel(const float* p, bf16* w3, bf16* wf, bf16* wt) {
  const int i = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (i < N_PARAMS) tc::store_weights(i, *reinterpret_cast<const float4*>(p + i), w3, wf, wt);
}

}  // namespace kp

using namespace kp;

// ---------------------------------------------------------------------------
// context
// ---------------------------------------------------------------------------

struct kp_mlp {
  char* arena;
  size_t bytes;
  cudaStream_t stream;
  int max_batch;
  int step;
  int num_sms;
  float *p, *m, *v, *g;
  float* loss;      // right after the gradient
  float* slots;     // a CTA's share of the gradient each
  uint32_t* bar;    // an epoch's barrier word and loss sum, cleared together
  float* loss_sum;
  bf16* w3;     // output layer, BF16 row-major
  bf16* wf;     // W1 | W2 | W3 in BF16, fragment order (planner loop)
  bf16* wt;     // W2 | W1 in BF16, tensor-core operand order
  int* err;     // nonzero: a tensor-core kernel's bounded wait expired
  unsigned long long wait_ns;  // limit of those waits
  int hold;                    // test hook: launches hold their products back
};

namespace {

struct MlpLayout {
  size_t p, m, v, g, w3, wf, wt, err, epoch, slots, total;
};

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

// CTAs that work on a mini-batch of B rows, each with a gradient slot.
int tile_ctas(int B) {
  const int tiles = (B + 127) / 128;
  return tiles < tc::ST_MAX_SLOTS ? tiles : tc::ST_MAX_SLOTS;
}

// The parameters, their moments, gradient and loss, the BF16 copies and the
// gradient slots: the kernels keep nothing per row in global memory.
MlpLayout mlp_layout(int B) {
  MlpLayout L{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = a256(off + bytes);
    return o;
  };
  L.p = take((size_t)N_PARAMS * 4);
  L.m = take((size_t)N_PARAMS * 4);
  L.v = take((size_t)N_PARAMS * 4);
  L.g = take((size_t)tc::SLOT * 4);  // gradient, loss
  L.w3 = take((size_t)MLP_OUT * MLP_H * 2);
  L.wf = take((size_t)N_WEIGHTS_BF16 * 2);
  L.wt = take((size_t)tc::WT_ELEMS * 2);
  L.err = take(16);
  L.epoch = take(16);
  L.slots = take((size_t)tile_ctas(B) * tc::SLOT * 4);
  L.total = off;
  return L;
}

#define MLP_CUDA(call)                            \
  do {                                            \
    if ((call) != cudaSuccess) {                  \
      cudaGetLastError();                         \
      return KP_ERR_CUDA;                         \
    }                                             \
  } while (0)

// Raises the dynamic shared memory limit of the tensor-core kernels on the
// current device (outside any stream capture): with every network, since the
// limit is a device's own and a process may have networks on several.
kp_status tc_configure() {
  MLP_CUDA(cudaFuncSetAttribute(tc::kp_mlp_forward_tc_kernel,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, tc::FT_SMEM));
  MLP_CUDA(cudaFuncSetAttribute(tc::kp_mlp_train_kernel,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, tc::ST_SMEM));
  return KP_OK;
}

// KP_ERR_TIMEOUT once a tensor-core kernel's bounded wait has expired (the
// word is sticky until the parameters are set again).  Stream synchronised.
kp_status device_error(const kp_mlp* n) {
  int e = 0;
  MLP_CUDA(cudaMemcpy(&e, n->err, 4, cudaMemcpyDeviceToHost));
  return e ? KP_ERR_TIMEOUT : KP_OK;
}

constexpr unsigned long long kWaitNs = 2000000000ull;

// CTAs that work on tiles (one gradient slot each).
int slots_used(const kp_mlp* n, int M) {
  const int c = tile_ctas(M);
  return c < n->num_sms ? c : n->num_sms;
}

tc::AdamArgs adam_args(const kp_mlp* n, int M, float lr) {
  tc::AdamArgs a{};
  a.p = n->p;
  a.m = n->m;
  a.v = n->v;
  a.w3 = n->w3;
  a.wf = n->wf;
  a.wt = n->wt;
  a.lr = lr;
  a.slots = n->slots;
  a.n_slots = slots_used(n, M);
  return a;
}

tc::StepArgs step_args(const kp_mlp* n, const float* x, const float* t, int M, float lr) {
  tc::StepArgs a{};
  a.x = x;
  a.t = t;
  a.M = M;
  a.steps = 1;
  a.adam = adam_args(n, M, lr);
  a.slots = n->slots;
  a.err = n->err;
  a.wait_ns = n->wait_ns;
  a.hold = n->hold;
  return a;
}

// Forward, loss and backward of one mini-batch into the slots.
kp_status forward_backward(kp_mlp* n, const float* x, const float* t, int M) {
  tc::kp_mlp_train_kernel<<<slots_used(n, M), tc::ST_THREADS, tc::ST_SMEM, n->stream>>>(
      step_args(n, x, t, M, 0.0f));
  MLP_CUDA(cudaGetLastError());
  return KP_OK;
}

}  // namespace

extern "C" {

size_t kp_mlp_required_bytes(int32_t max_batch) {
  if (max_batch < 1 || max_batch > (1 << 24)) return 0;
  return mlp_layout(max_batch).total;
}

kp_status kp_mlp_create(void* dev_arena, size_t arena_bytes, int32_t max_batch,
                        const float* host_params, void* cuda_stream, kp_mlp** out) {
  if (!out || !dev_arena || ((uintptr_t)dev_arena & 255u) || !host_params) return KP_ERR_ARG;
  *out = nullptr;
  if (max_batch < 1 || max_batch > (1 << 24)) return KP_ERR_ARG;
  const MlpLayout L = mlp_layout(max_batch);
  if (arena_bytes < L.total) return KP_ERR_OOM;
  kp_mlp* n = new (std::nothrow) kp_mlp();
  if (!n) return KP_ERR_OOM;
  n->arena = static_cast<char*>(dev_arena);
  n->bytes = arena_bytes;
  n->stream = static_cast<cudaStream_t>(cuda_stream);
  n->max_batch = max_batch;
  n->wait_ns = kWaitNs;
  n->hold = 0;
  char* A = n->arena;
  n->p = reinterpret_cast<float*>(A + L.p);
  n->m = reinterpret_cast<float*>(A + L.m);
  n->v = reinterpret_cast<float*>(A + L.v);
  n->g = reinterpret_cast<float*>(A + L.g);
  n->loss = n->g + N_PARAMS;
  n->slots = reinterpret_cast<float*>(A + L.slots);
  n->bar = reinterpret_cast<uint32_t*>(A + L.epoch);
  n->loss_sum = reinterpret_cast<float*>(A + L.epoch) + 1;
  n->w3 = reinterpret_cast<bf16*>(A + L.w3);
  n->wf = reinterpret_cast<bf16*>(A + L.wf);
  n->wt = reinterpret_cast<bf16*>(A + L.wt);
  n->err = reinterpret_cast<int*>(A + L.err);
  int dev = 0;
  kp_status s = KP_OK;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&n->num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    s = KP_ERR_CUDA;
  }
  if (s == KP_OK) s = tc_configure();
  if (s == KP_OK) s = kp_mlp_set_params(n, host_params);
  if (s != KP_OK) {
    delete n;
    return s;
  }
  *out = n;
  return KP_OK;
}

kp_status kp_mlp_set_params(kp_mlp* n, const float* host_params) {
  if (!n || !host_params) return KP_ERR_ARG;
  for (int i = 0; i < N_PARAMS; ++i)
    if (!std::isfinite(host_params[i])) return KP_ERR_ARG;
  MLP_CUDA(cudaMemcpyAsync(n->p, host_params, (size_t)N_PARAMS * 4, cudaMemcpyHostToDevice,
                           n->stream));
  MLP_CUDA(cudaMemsetAsync(n->m, 0, (size_t)N_PARAMS * 4, n->stream));
  MLP_CUDA(cudaMemsetAsync(n->v, 0, (size_t)N_PARAMS * 4, n->stream));
  MLP_CUDA(cudaMemsetAsync(n->err, 0, 16, n->stream));
  kp_mlp_round_kernel<<<(N_PARAMS / 4 + 255) / 256, 256, 0, n->stream>>>(n->p, n->w3, n->wf, n->wt);
  MLP_CUDA(cudaGetLastError());
  MLP_CUDA(cudaStreamSynchronize(n->stream));
  n->step = 0;
  return KP_OK;
}

kp_status kp_mlp_get_params(kp_mlp* n, float* host_params) {
  if (!n || !host_params) return KP_ERR_ARG;
  MLP_CUDA(cudaMemcpyAsync(host_params, n->p, (size_t)N_PARAMS * 4, cudaMemcpyDeviceToHost,
                           n->stream));
  MLP_CUDA(cudaStreamSynchronize(n->stream));
  return KP_OK;
}

int32_t kp_mlp_num_params(void) { return N_PARAMS; }

kp_status kp_mlp_selftest_hold(kp_mlp* n, uint64_t limit_ns) {
  if (!n || limit_ns > kWaitNs) return KP_ERR_ARG;
  n->hold = limit_ns > 0 ? 1 : 0;
  n->wait_ns = limit_ns > 0 ? limit_ns : kWaitNs;
  return KP_OK;
}

kp_status kp_mlp_forward(kp_mlp* n, const float* dev_x, int32_t M, float* dev_out) {
  if (!n || !dev_x || !dev_out || M < 0 || M > n->max_batch) return KP_ERR_ARG;
  if (M == 0) return KP_OK;
  tc::FtArgs a{};
  a.wt = n->wt;
  a.W3 = n->w3;
  a.b1 = n->p + OFF_B1;
  a.b2 = n->p + OFF_B2;
  a.b3 = n->p + OFF_B3;
  a.x = dev_x;
  a.out = dev_out;
  a.M = M;
  a.vec = ((uintptr_t)dev_x & 15u) == 0 && ((uintptr_t)dev_out & 7u) == 0;
  a.err = n->err;
  a.wait_ns = n->wait_ns;
  a.hold = n->hold;
  const int tiles = (M + tc::FT_ROWS - 1) / tc::FT_ROWS;
  tc::kp_mlp_forward_tc_kernel<<<tiles < n->num_sms ? tiles : n->num_sms, tc::FT_THREADS,
                                 tc::FT_SMEM, n->stream>>>(a);
  MLP_CUDA(cudaGetLastError());
  return KP_OK;
}

kp_status kp_mlp_gradients(kp_mlp* n, const float* dev_x, const float* dev_t, int32_t M,
                           float* host_grad, float* host_loss) {
  if (!n || !dev_x || !dev_t || M < 1 || M > n->max_batch) return KP_ERR_ARG;
  kp_status s = forward_backward(n, dev_x, dev_t, M);
  if (s != KP_OK) return s;
  kp_mlp_gradient_kernel<<<(tc::SLOT / 4 + 255) / 256, 256, 0, n->stream>>>(
      n->slots, slots_used(n, M), n->g);
  MLP_CUDA(cudaGetLastError());
  if (host_grad)
    MLP_CUDA(cudaMemcpyAsync(host_grad, n->g, (size_t)N_PARAMS * 4, cudaMemcpyDeviceToHost,
                             n->stream));
  if (host_loss)
    MLP_CUDA(cudaMemcpyAsync(host_loss, n->loss, 4, cudaMemcpyDeviceToHost, n->stream));
  MLP_CUDA(cudaStreamSynchronize(n->stream));
  return device_error(n);
}

kp_status kp_mlp_train_step(kp_mlp* n, const float* dev_x, const float* dev_t, int32_t M,
                            float lr, float* host_loss) {
  if (!n || !dev_x || !dev_t || M < 1 || M > n->max_batch || !(lr > 0.0f)) return KP_ERR_ARG;
  kp_status s = forward_backward(n, dev_x, dev_t, M);
  if (s != KP_OK) return s;
  n->step += 1;
  kp_mlp_adam_kernel<<<(N_PARAMS / 4 + 256) / 256, 256, 0, n->stream>>>(
      adam_args(n, M, lr), 1.0f - powf(0.9f, (float)n->step), 1.0f - powf(0.999f, (float)n->step),
      n->loss);
  MLP_CUDA(cudaGetLastError());
  if (host_loss) {
    MLP_CUDA(cudaMemcpyAsync(host_loss, n->loss, 4, cudaMemcpyDeviceToHost, n->stream));
    MLP_CUDA(cudaStreamSynchronize(n->stream));
    return device_error(n);
  }
  return KP_OK;
}

kp_status kp_mlp_train_epoch(kp_mlp* n, const float* dev_x, const float* dev_t,
                             const int32_t* dev_perm, int64_t rows, float lr, float* host_loss) {
  if (!n || !dev_x || !dev_t || !dev_perm || rows < 0 || !(lr > 0.0f)) return KP_ERR_ARG;
  const int B = n->max_batch;
  const int64_t nb = rows / B;
  if (host_loss) *host_loss = 0.0f;
  if (nb == 0) return KP_OK;
  if (nb > (1 << 30)) return KP_ERR_ARG;
  MLP_CUDA(cudaMemsetAsync(n->bar, 0, 8, n->stream));  // and the epoch's loss
  tc::StepArgs a = step_args(n, dev_x, dev_t, B, lr);
  a.perm = dev_perm;
  a.steps = nb;
  a.epoch = 1;
  a.step0 = n->step;
  a.loss_sum = n->loss_sum;
  a.bar = n->bar;
  // a CTA a tile; the others up to 128 share the optimiser's step
  int grid = a.adam.n_slots > 128 ? a.adam.n_slots : 128;
  if (grid > n->num_sms) grid = n->num_sms;
  void* args[] = {&a};
  MLP_CUDA(cudaLaunchCooperativeKernel((const void*)tc::kp_mlp_train_kernel, dim3(grid),
                                       dim3(tc::ST_THREADS), args, tc::ST_SMEM, n->stream));
  n->step += (int)nb;
  float sum = 0.0f;
  MLP_CUDA(cudaMemcpyAsync(&sum, n->loss_sum, 4, cudaMemcpyDeviceToHost, n->stream));
  MLP_CUDA(cudaStreamSynchronize(n->stream));
  if (host_loss) *host_loss = sum / (float)nb;
  return device_error(n);
}

void kp_mlp_destroy(kp_mlp* n) {
  delete n;
}

}  // extern "C"

namespace kp {
// Device pointers of the network's weights for the planner's loop kernel:
// BF16 weights in fragment order (frag_index_hidden / frag_index_out), FP32
// biases.
void mlp_device_weights(const kp_mlp* n, const void** W1, const float** b1, const void** W2,
                        const float** b2, const void** W3, const float** b3) {
  *W1 = n->wf;
  *b1 = n->p + OFF_B1;
  *W2 = n->wf + MLP_H * MLP_IN;
  *b2 = n->p + OFF_B2;
  *W3 = n->wf + MLP_H * MLP_IN + MLP_H * MLP_H;
  *b3 = n->p + OFF_B3;
}
}  // namespace kp
