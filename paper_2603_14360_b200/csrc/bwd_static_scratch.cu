// m2rnn_bwd for callers that cannot allocate device memory: the scratch the backward pass needs
// lives in a fixed array that is part of the library's device image.
#include <cuda_runtime.h>

#include <mutex>

#include "internal.h"
#include "m2rnn.h"

namespace {

// Every GPU that loads the library holds this array until the process exits.  All calls share it.
static __device__ __align__(256) unsigned char g_static_scratch[M2RNN_STATIC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
struct Known { void *addr; uint64_t context; };
Known g_scratch[kMaxDevices];   // device address of g_static_scratch, per device, and the context it belongs to; null = not looked up yet
std::mutex g_scratch_mutex;

// In host code `g_static_scratch` only names the symbol; the device address has to be asked for,
// with that device current: once per device, and again when the device has another context than then (after a
// reset the array may lie elsewhere).
int scratch_address(void **out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return M2RNN_ERR_CUDA;
  uint64_t context = 0;
  const bool told = m2rnn::current_context(&context);
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  Known &k = g_scratch[dev];
  if (!k.addr || !told || k.context != context) {
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) {
      (void)cudaGetLastError();
      return M2RNN_ERR_CUDA;
    }
    if (!told) (void)m2rnn::current_context(&context);   // (the lookup makes a context current where there was none)
    k = Known{p, context};
  }
  *out = k.addr;
  return M2RNN_OK;
}

}  // namespace

extern "C" int m2rnn_bwd_static_scratch(const m2rnn_params *params, const void *q, const void *k,
                                        const void *v, const float *gate, const void *W,
                                        const float *h0, const float *alpha, const float *beta,
                                        const void *w_r, const float *ckpt, const void *dy,
                                        const float *d_hT, void *dq, void *dk, void *dv,
                                        float *dgate, float *dW, float *dh0, int32_t *dev_status,
                                        void *stream) {
  if (!params) return M2RNN_ERR_NULL;
  // size check first: a problem that does not fit is refused before the device is touched
  constexpr size_t kHave = M2RNN_STATIC_SCRATCH_BYTES;
  // An fp32 problem whose shares of dv and dW (one per group of rows) do not fit is taken one group after the other, which
  // needs none: B 2, T 512, N 8, K = V = 64 with checkpoints 4.3 MiB instead of 36.5.
  const bool lean = m2rnn::bwd_workspace_bytes(params, ckpt != nullptr, false) > kHave;
  if (lean && m2rnn::bwd_workspace_bytes(params, ckpt != nullptr, true) > kHave) return M2RNN_ERR_WORKSPACE;
  void *scratch = nullptr;
  const int rc = scratch_address(&scratch);
  if (rc != M2RNN_OK) return rc;
  // every word of the scratch that the backward kernels read is written earlier in the same call,
  // so what an earlier call left behind never needs clearing
  return m2rnn::bwd_call(params, q, k, v, gate, W, h0, alpha, beta, w_r, ckpt, dy, d_hT, dq, dk, dv, dgate,
                         dW, dh0, scratch, kHave, lean, dev_status, stream);
}
