// kp_mlp.cu -- the learned proposal's network: optimiser kernels and the
// kp_mlp_* entry points of include/kp.h.  Inference and the forward and backward
// pass of a training step are one kernel each on the tcgen05 tensor cores
// (kp_mlp_tc.cuh: BF16 operands, FP32 accumulation in tensor memory); FP32
// master weights and Adam moments.
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

// flat parameter vector (FP32), row-major: W1 b1 W2 b2 W3 b3
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + MLP_H * MLP_IN, OFF_W2 = OFF_B1 + MLP_H,
              OFF_B2 = OFF_W2 + MLP_H * MLP_H, OFF_W3 = OFF_B2 + MLP_H,
              OFF_B3 = OFF_W3 + MLP_OUT * MLP_H, N_PARAMS = OFF_B3 + MLP_OUT;
constexpr int N_WEIGHTS_BF16 = MLP_H * MLP_IN + MLP_H * MLP_H + MLP_OUT * MLP_H;

// ---------------------------------------------------------------------------
// Adam on the FP32 master vector; refreshes the BF16 weight copies
// ---------------------------------------------------------------------------

// Parameter i rounded to BF16 into the copies the kernels read: the hidden
// layers' weights in tensor-core operand order (wt) and in the fragment order
// of the planner's loop kernel (wf); the output layer's row-major (w3) and in
// fragment order.
__device__ __forceinline__ void store_weight(int i, float pi, bf16* w3, bf16* wf, bf16* wt) {
  const bf16 b = __float2bfloat16_rn(pi);
  if (i < OFF_B1) {
    wt[tc::wt_index_w1(i / MLP_IN, i % MLP_IN)] = b;
    wf[frag_index_hidden(i / MLP_IN, i % MLP_IN, MLP_IN)] = b;
  } else if (i >= OFF_W2 && i < OFF_B2) {
    const int j = i - OFF_W2;
    wt[tc::wt_index_w2(j / MLP_H, j % MLP_H)] = b;
    wf[MLP_H * MLP_IN + frag_index_hidden(j / MLP_H, j % MLP_H, MLP_H)] = b;
  } else if (i >= OFF_W3 && i < OFF_B3) {
    const int j = i - OFF_W3;
    w3[j] = b;
    wf[MLP_H * MLP_IN + MLP_H * MLP_H + frag_index_out(j / MLP_H, j % MLP_H)] = b;
  }
}

struct AdamArgs {
  float *p, *g, *m, *v;
  bf16 *w3, *wf, *wt;
  float lr, c1, c2;      // c1, c2: 1 - beta^step (epoch null)
  tc::EpochCtl* epoch;   // learning rate and step from here; the gradient and
  float* loss;           // the loss are cleared for the next mini-batch
};

// One Adam step (beta 0.9 / 0.999, eps 1e-8), one thread a parameter.  In a
// device-driven epoch it also closes the mini-batch: the gradient it has used
// is cleared for the next one's additions, the loss is added to the epoch's,
// and the batch index moves on.
__global__ void kp_mlp_adam_kernel(AdamArgs a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N_PARAMS) return;
  const float beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
  float lr = a.lr, c1 = a.c1, c2 = a.c2;
  if (a.epoch) {
    const float step = (float)a.epoch->step;
    lr = a.epoch->lr;
    c1 = 1.0f - powf(beta1, step);
    c2 = 1.0f - powf(beta2, step);
  }
  const float gi = a.g[i];
  const float mi = beta1 * a.m[i] + (1.0f - beta1) * gi;
  const float vi = beta2 * a.v[i] + (1.0f - beta2) * gi * gi;
  a.m[i] = mi;
  a.v[i] = vi;
  const float pi = a.p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  a.p[i] = pi;
  store_weight(i, pi, a.w3, a.wf, a.wt);
  if (a.epoch) {
    a.g[i] = 0.0f;
    if (i == 0) {
      a.epoch->loss_sum += *a.loss;
      *a.loss = 0.0f;
      a.epoch->batch += 1;
    }
  }
}

__global__ void kp_mlp_round_kernel(const float* p, bf16* w3, bf16* wf, bf16* wt) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N_PARAMS) return;
  store_weight(i, p[i], w3, wf, wt);
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
  float* loss;  // right after g: cleared with it
  bf16* w3;     // output layer, BF16 row-major
  bf16* wf;     // W1 | W2 | W3 in BF16, fragment order (planner loop)
  bf16* wt;     // W2 | W1 in BF16, tensor-core operand order
  int* err;     // nonzero: a tensor-core kernel's bounded wait expired
  tc::EpochCtl* ec;
  cudaGraph_t graph = nullptr;     // one mini-batch: step kernel, Adam
  cudaGraphExec_t graph_exec = nullptr;
  cudaStream_t gstream = nullptr;  // the graph's own stream (capture needs a
  cudaEvent_t gev = nullptr;       // non-default stream), ordered by an event
};

namespace {

struct MlpLayout {
  size_t p, m, v, g, w3, wf, wt, err, ec, total;
};

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

// The parameters, their moments, gradient and loss, and the BF16 copies.  The
// kernels keep nothing per row in global memory; 16 bytes a row stay reserved,
// so that the size asked for still grows with the batch.
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
  L.g = take((size_t)(N_PARAMS + 1) * 4);
  L.w3 = take((size_t)MLP_OUT * MLP_H * 2);
  L.wf = take((size_t)N_WEIGHTS_BF16 * 2);
  L.wt = take((size_t)tc::WT_ELEMS * 2);
  L.err = take(16);
  L.ec = take(sizeof(tc::EpochCtl));
  take((size_t)B * 16);
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


// Raises the dynamic shared memory limit of the tensor-core kernels (once,
// outside any stream capture).
kp_status tc_configure() {
  static bool done = false;
  if (!done) {
    MLP_CUDA(cudaFuncSetAttribute(tc::kp_mlp_forward_tc_kernel,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, tc::FT_SMEM));
    MLP_CUDA(cudaFuncSetAttribute(tc::kp_mlp_step_kernel,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, tc::ST_SMEM));
    done = true;
  }
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

// The gradient and the loss cleared (they are added to by every tile).
cudaError_t clear_gradient(kp_mlp* n, cudaStream_t stream) {
  return cudaMemsetAsync(n->g, 0, (size_t)(N_PARAMS + 1) * 4, stream);
}

// Forward, loss and backward of one mini-batch, added to n->g and n->loss.
kp_status forward_backward(kp_mlp* n, const float* x, const float* t, tc::EpochCtl* epoch, int M,
                           cudaStream_t stream) {
  tc::StepArgs a{};
  a.wt = n->wt;
  a.W3 = n->w3;
  a.b1 = n->p + OFF_B1;
  a.b2 = n->p + OFF_B2;
  a.b3 = n->p + OFF_B3;
  a.x = x;
  a.t = t;
  a.epoch = epoch;
  a.M = M;
  a.g_W1 = n->g + OFF_W1;
  a.g_b1 = n->g + OFF_B1;
  a.g_W2 = n->g + OFF_W2;
  a.g_b2 = n->g + OFF_B2;
  a.g_W3 = n->g + OFF_W3;
  a.g_b3 = n->g + OFF_B3;
  a.loss = n->loss;
  a.err = n->err;
  a.wait_ns = kWaitNs;
  tc::kp_mlp_step_kernel<<<(M + 127) / 128, tc::ST_THREADS, tc::ST_SMEM, stream>>>(a);
  MLP_CUDA(cudaGetLastError());
  return KP_OK;
}

// One Adam step on n->g.  epoch null: c1, c2 of n->step.
kp_status adam(kp_mlp* n, float lr, tc::EpochCtl* epoch, cudaStream_t stream) {
  AdamArgs a{};
  a.p = n->p;
  a.g = n->g;
  a.m = n->m;
  a.v = n->v;
  a.w3 = n->w3;
  a.wf = n->wf;
  a.wt = n->wt;
  a.lr = lr;
  a.c1 = 1.0f - powf(0.9f, (float)n->step);
  a.c2 = 1.0f - powf(0.999f, (float)n->step);
  a.epoch = epoch;
  a.loss = n->loss;
  kp_mlp_adam_kernel<<<(N_PARAMS + 255) / 256, 256, 0, stream>>>(a);
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
  char* A = n->arena;
  n->p = reinterpret_cast<float*>(A + L.p);
  n->m = reinterpret_cast<float*>(A + L.m);
  n->v = reinterpret_cast<float*>(A + L.v);
  n->g = reinterpret_cast<float*>(A + L.g);
  n->loss = n->g + N_PARAMS;
  n->w3 = reinterpret_cast<bf16*>(A + L.w3);
  n->wf = reinterpret_cast<bf16*>(A + L.wf);
  n->wt = reinterpret_cast<bf16*>(A + L.wt);
  n->err = reinterpret_cast<int*>(A + L.err);
  n->ec = reinterpret_cast<tc::EpochCtl*>(A + L.ec);
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
  kp_mlp_round_kernel<<<(N_PARAMS + 255) / 256, 256, 0, n->stream>>>(n->p, n->w3, n->wf, n->wt);
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
  a.wait_ns = kWaitNs;
  const int tiles = (M + tc::FT_ROWS - 1) / tc::FT_ROWS;
  tc::kp_mlp_forward_tc_kernel<<<tiles < n->num_sms ? tiles : n->num_sms, tc::FT_THREADS,
                                 tc::FT_SMEM, n->stream>>>(a);
  MLP_CUDA(cudaGetLastError());
  return KP_OK;
}

kp_status kp_mlp_gradients(kp_mlp* n, const float* dev_x, const float* dev_t, int32_t M,
                           float* host_grad, float* host_loss) {
  if (!n || !dev_x || !dev_t || M < 1 || M > n->max_batch) return KP_ERR_ARG;
  MLP_CUDA(clear_gradient(n, n->stream));
  kp_status s = forward_backward(n, dev_x, dev_t, nullptr, M, n->stream);
  if (s != KP_OK) return s;
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
  MLP_CUDA(clear_gradient(n, n->stream));
  kp_status s = forward_backward(n, dev_x, dev_t, nullptr, M, n->stream);
  if (s != KP_OK) return s;
  n->step += 1;
  s = adam(n, lr, nullptr, n->stream);
  if (s != KP_OK) return s;
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
  if (!n->gstream) {
    MLP_CUDA(cudaStreamCreateWithFlags(&n->gstream, cudaStreamNonBlocking));
    MLP_CUDA(cudaEventCreateWithFlags(&n->gev, cudaEventDisableTiming));
  }
  // the epoch runs after the work already queued on the caller's stream
  MLP_CUDA(cudaEventRecord(n->gev, n->stream));
  MLP_CUDA(cudaStreamWaitEvent(n->gstream, n->gev, 0));
  tc::EpochCtl h{dev_x, dev_t, dev_perm, 0, n->step, lr, 0.0f};
  MLP_CUDA(cudaMemcpyAsync(n->ec, &h, sizeof(h), cudaMemcpyHostToDevice, n->gstream));
  MLP_CUDA(clear_gradient(n, n->gstream));  // each step's Adam launch clears it again
  if (!n->graph_exec) {
    // one mini-batch: rows by the permutation, forward, backward; Adam
    if (cudaStreamBeginCapture(n->gstream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      cudaGetLastError();
      return KP_ERR_CUDA;
    }
    kp_status s = forward_backward(n, nullptr, nullptr, n->ec, B, n->gstream);
    if (s == KP_OK) s = adam(n, 0.0f, n->ec, n->gstream);
    cudaGraph_t g = nullptr;
    const cudaError_t e = cudaStreamEndCapture(n->gstream, &g);
    if (s != KP_OK || e != cudaSuccess) {
      if (g) cudaGraphDestroy(g);
      cudaGetLastError();
      return s != KP_OK ? s : KP_ERR_CUDA;
    }
    if (cudaGraphInstantiate(&n->graph_exec, g, 0) != cudaSuccess) {
      cudaGraphDestroy(g);
      n->graph_exec = nullptr;
      cudaGetLastError();
      return KP_ERR_CUDA;
    }
    n->graph = g;
  }
  for (int64_t b = 0; b < nb; ++b) MLP_CUDA(cudaGraphLaunch(n->graph_exec, n->gstream));
  n->step += (int)nb;
  tc::EpochCtl out{};
  MLP_CUDA(cudaMemcpyAsync(&out, n->ec, sizeof(out), cudaMemcpyDeviceToHost, n->gstream));
  MLP_CUDA(cudaStreamSynchronize(n->gstream));
  if (host_loss) *host_loss = out.loss_sum / (float)nb;
  return device_error(n);
}

void kp_mlp_destroy(kp_mlp* n) {
  if (!n) return;
  if (n->graph_exec) cudaGraphExecDestroy(n->graph_exec);
  if (n->graph) cudaGraphDestroy(n->graph);
  if (n->gev) cudaEventDestroy(n->gev);
  if (n->gstream) cudaStreamDestroy(n->gstream);
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
