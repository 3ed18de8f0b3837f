// C ABI of the M2RNN scan library: argument checks, workspace layout, dispatch.
// No allocation, no synchronisation.  Kept between calls: constants of the device (its SM count) and which
// kernels have had their limit of shared memory raised (smem_limit.h), both asked for once.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cstring>

#include "internal.h"
#include "m2rnn.h"
#include "smem_limit.h"

namespace m2rnn {

namespace {
constexpr int kMaxDevices = 64;
int current_device() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) { (void)cudaGetLastError(); return -1; }
  return dev;
}
}  // namespace

// SMs of the current device (the plans size their grids by it); 148, a B200's count, when no device
// can be asked -- the size queries of the ABI also run on hosts without a GPU.
int sm_count() {
  static std::atomic<int> known[kMaxDevices];   // a constant of the device: asked for once
  const int dev = current_device();
  if (dev < 0) return 148;
  if (dev < kMaxDevices)
    if (const int n = known[dev].load(std::memory_order_relaxed)) return n;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) {
    (void)cudaGetLastError();
    return 148;
  }
  if (dev < kMaxDevices) known[dev].store(sms, std::memory_order_relaxed);
  return sms;
}

// cuCtxGetId through the runtime's driver entry point (no link against libcuda)
bool current_context(uint64_t *id) {
  using GetId = CUresult (*)(CUcontext, unsigned long long *);
  static const GetId get = [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuCtxGetId", &p, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) {
      (void)cudaGetLastError();
      p = nullptr;
    }
    return reinterpret_cast<GetId>(p);
  }();
  unsigned long long n = 0;
  if (!get || get(nullptr, &n) != CUDA_SUCCESS) return false;   // (null: the current context)
  *id = n;
  return true;
}

namespace {
struct CudaSmem {
  bool context(uint64_t *id) const { return current_context(id); }
  int most(const void *kernel, int *n) const {
    int dev = 0, optin = 0;
    cudaFuncAttributes at;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, kernel);
    if (e == cudaSuccess) *n = optin - (int)at.sharedSizeBytes;
    return e;
  }
  int set(const void *kernel, int n) const { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, n); }
};
}  // namespace

// Lets `kernel` be launched with `bytes` of dynamic shared memory in the current context.  (Asking the runtime on
// every launch cost a small call a tenth of its host time.)
cudaError_t allow_smem(const void *kernel, size_t bytes) {
  if (bytes <= 40 * 1024) return cudaSuccess;   // with up to 8 KB of static shared memory: what every kernel may use unasked
  static SmemLimits<CudaSmem> limits(cudaErrorInvalidValue);
  CudaSmem api;
  return static_cast<cudaError_t>(limits.allow(api, kernel, bytes));
}

bool bwd_use_tc(int B, int N, int K, int V, int io_dtype) {
  if (io_dtype != M2RNN_BF16 || V != 128 || K % bwd_tc_rows_per_cta()) return false;   // 32-row CTAs
  const char *variant = getenv("M2RNN_BWD_VARIANT");
  if (variant && !strcmp(variant, "mma")) return false;
  (void)B; (void)N;
  return true;
}

size_t tokens_of(const m2rnn_params *p) { return p->cu_seqlens ? (size_t)p->total_tokens : (size_t)p->B * p->T; }

BwdPlan plan_bwd(const m2rnn_params *p, bool lean, bool have_ckpt) {
  const int B = p->B, N = p->N, K = p->K, V = p->V;
  BwdPlan pl{};
  if (p->io_dtype == M2RNN_F32) {
    pl.KC = lean ? K : bwd_f32_rows(B, N, K, V, p->T > 0 ? tokens_of(p) * N * V * sizeof(float) : 0); pl.C = pl.interval = bwd_f32_piece(); pl.C_max = 64;
    return pl;
  }
  // V = 16: scan_bwd_v16.cu, except where every slab of 16 rows has an SM to itself: there a slab's step is quicker spread over
  // the specialised warps of scan_bwd_bf16.cu (1 024 steps, us: 16 slabs 232 against 245, 64 of heads of their own 208 / 232;
  // 160 slabs 296 / 249).  The latter keeps two chunks on chip, 16 rows of them up to any supported interval.
  if (V == 16 && (long)(B > 0 ? B : 1) * N * (K / 16) > sm_count()) {
    BwdPlan fast = plan_bwd_v16(B, N, p->Nq, p->Nk, K, p->T, p->ckpt_interval, false);
    if (!have_ckpt && !p->ckpt_interval) fast.interval = fast.C;      // (the call's own checkpoints: a chunk's first is enough)
    return lean ? plan_bwd_v16(B, N, p->Nq, p->Nk, K, p->T, p->ckpt_interval || have_ckpt ? fast.interval : 16, true) : fast;
  }
  if (bwd_use_tc(B, N, K, V, p->io_dtype)) {   // 32-row CTAs, chunks of four steps
    pl.KC = bwd_tc_rows_per_cta(); pl.C = pl.interval = pl.C_max = bwd_tc_chunk();
    return pl;
  }
  // Rows per CTA: the largest slab that still spreads the problem over the SMs (rows are independent
  // recurrences; a smaller slab only shortens the work per step).  V = 128 keeps the slab at 32 rows
  // for the sake of registers.
  const int kSMs = sm_count();
  const long units = (long)(B > 0 ? B : 1) * N;
  const int cap = V > 64 ? 32 : 64;
  int KC = 16;
  for (int cand = 32; cand <= cap; cand *= 2)
    if (K % cand == 0) KC = cand;
  while (KC > 16 && units * (K / KC) < kSMs && units * (K / (KC / 2)) <= kSMs) KC /= 2;
  pl.KC = KC;
  // Checkpoint interval: as many steps as two chunk buffers fit in shared memory (even, <= 16)
  constexpr size_t kSmemLimit = 227 * 1024;
  int c = 16;
  while (c > 2 && bwd_bf16_smem_bytes(KC, V, c) > kSmemLimit) c -= 2;
  pl.C = pl.interval = pl.C_max = c;
  return pl;
}

bool fwd_use_tc(int B, int N, int K, int V, int io_dtype) {
  if (io_dtype != M2RNN_BF16) return false;
  const char *variant = getenv("M2RNN_FWD_VARIANT");
  if (variant && !strcmp(variant, "tc")) return true;
  if (variant && !strcmp(variant, "mma")) return false;
  // Measured (B200): the round trip of a tcgen05 step (operand store, proxy fence, barrier, eight
  // MMAs at ~30 cycles of issue each, commit, mbarrier, tcgen05.ld) is ~400 cycles before any
  // arithmetic, against ~30 for mma.sync on registers.  It pays only where the register kernels
  // are bound by the legacy tensor path and there are rows to amortise it over: V = 128, 64-row CTAs, and so many of
  // them that 32-row CTAs no longer fit one to an SM (1024 steps of K = V = 128, us: 37 units 442 against 809, 40
  // units 861 against 816; with checkpoints 995 against 926).
  // Below V = 128 it stays slower at every number of units (1024 steps, us, register kernels / this one): K = V = 64, 128 units
  // 302 / 448, 192 599 / 694, 256 600 / 696 (with checkpoints 660 / 813), 384 896 / 1375; K = 128, V = 64, 128 units 618 / 741;
  // K = V = 32, 256 units 169 / 453; K = 64, V = 16, 256 units 137 / 831.
  return V == 128 && K % 64 == 0 && (long)(B > 0 ? B : 1) * N * (K / 32) > sm_count();
}

int plan_fwd_rows(int B, int N, int K, int V, int io_dtype, size_t tokens, bool lean) {
  if (io_dtype == M2RNN_F32) return lean ? K : fwd_f32_rows(B, N, K, V, tokens * N * V * sizeof(float));
  if (fwd_use_tc(B, N, K, V, io_dtype)) return fwd_tc_rows_per_cta(B, N, K, V);
  // The smallest slab (a multiple of 16 rows that divides K) that still gives every CTA an SM of its own; with more
  // units than SMs the largest that the column-split kernel has: 32 rows at V = 128 for the sake of
  // registers, 64 below.  Up to 128 rows in one CTA of the one-warp-per-slab kernel only where a K that 48 and
  // 64 do not divide would make V = 32 slabs of 16 rows (440 units, K = 112: 1029 against 1226 us for 1024 steps; K = 96,
  // V = 64, 192 units: 1682 against 759), or the slabs' shares of y (fp32, added afterwards) take more than 4 GB or
  // there is no room for them at all (lean).
  const int kSMs = sm_count();
  const long units = (long)(B > 0 ? B : 1) * N;
  int cap = V > 64 ? 32 : 128;
  if (V > 16 && V <= 64 && K > 64 && !lean) {
    int kc = 64;
    while (K % kc) kc -= 16;
    if ((V == 64 || kc > 16) && tokens * N * V * sizeof(float) * (K / kc) <= ((size_t)4 << 30)) cap = kc;
  }
  int best = 0;
  for (int kc = 16; kc <= K && kc <= cap; kc += 16) {
    if (K % kc) continue;
    best = kc;                                   // largest admissible slab so far
    if (units * (K / kc) <= kSMs) break;         // first (smallest) slab that fits one wave
  }
  return best;
}

namespace {

// A refused launch, attribute or copy: the runtime's last-error slot is cleared here, so that the
// caller's own next cudaGetLastError() does not report this library's failure a second time.
int cuda_failed() {
  (void)cudaGetLastError();
  return M2RNN_ERR_CUDA;
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// The longest checkpoint interval, by a plan that has not seen the caller's: that one is still to be checked.
int longest_interval(const m2rnn_params *p) {
  m2rnn_params unset = *p;
  unset.ckpt_interval = 0;
  return plan_bwd(&unset).C_max;
}

int check_params(const m2rnn_params *p, bool need_T) {
  if (!p) return M2RNN_ERR_NULL;
  if (p->B < 0 || p->N <= 0 || p->K <= 0 || p->V <= 0 || (need_T && p->T < 0)) return M2RNN_ERR_SHAPE;
  if (p->Nq <= 0 || p->Nk <= 0 || p->Nq > p->N || p->Nk > p->N || p->N % p->Nq || p->N % p->Nk)
    return M2RNN_ERR_SHAPE;
  if (p->io_dtype != M2RNN_F32 && p->io_dtype != M2RNN_BF16) return M2RNN_ERR_UNSUPPORTED;
  if (p->gate_kind < M2RNN_GATE_VALUE || p->gate_kind > M2RNN_GATE_PSI) return M2RNN_ERR_UNSUPPORTED;
  if (p->K % 16 || p->K < 16 || p->K > 128) return M2RNN_ERR_UNSUPPORTED;
  if (p->V != 16 && p->V != 32 && p->V != 64 && p->V != 128) return M2RNN_ERR_UNSUPPORTED;
  if (p->ckpt_interval < 0 || (p->ckpt_interval > 0 && p->ckpt_interval > longest_interval(p))) return M2RNN_ERR_UNSUPPORTED;
  // the bf16 kernels take steps in pairs and checkpoint between pairs
  if (p->io_dtype == M2RNN_BF16 && (p->ckpt_interval & 1)) return M2RNN_ERR_UNSUPPORTED;
  // token strides: at least a token's heads, in 16-byte units
  const int64_t unit16 = p->io_dtype == M2RNN_BF16 ? 8 : 4;
  const int64_t dense[3] = {(int64_t)p->Nq * p->K, (int64_t)p->Nk * p->K, (int64_t)p->N * p->V};
  const int64_t given[3] = {p->q_stride, p->k_stride, p->v_stride};
  for (int x = 0; x < 3; ++x)
    if (given[x] != 0 && (given[x] < dense[x] || given[x] % unit16)) return M2RNN_ERR_SHAPE;
  if (p->total_tokens < 0 || (!p->cu_seqlens && p->total_tokens != 0)) return M2RNN_ERR_SHAPE;
  if (p->cu_seqlens && (need_T && p->total_tokens > (int64_t)p->B * p->T)) return M2RNN_ERR_SHAPE;
  return M2RNN_OK;
}

int interval_of(const m2rnn_params *p) { return p->ckpt_interval ? p->ckpt_interval : plan_bwd(p).interval; }

struct Workspace {
  size_t ckpt, dW_part, dq_part, dk_part, chunk_states, dv_part, dgate_part, total;
};

Workspace layout(const m2rnn_params *p, const BwdPlan &pl, bool have_ckpt) {
  Workspace w{};
  const int C = p->ckpt_interval ? p->ckpt_interval : pl.interval;
  const size_t nch = p->T > 0 ? (size_t)(p->T + C - 1) / C : 0;
  const size_t BN = (size_t)p->B * p->N, KV = (size_t)p->K * p->V;
  size_t off = 0;
  w.ckpt = off;
  if (!have_ckpt) off += align_up(BN * nch * KV * sizeof(float));
  const int RS = p->K / pl.KC;   // row slabs per state
  w.dW_part = off;
  off += align_up(BN * RS * p->V * p->V * sizeof(float));
  const size_t TT = tokens_of(p);
  const int shares = pl.groups ? pl.groups : p->N;   // of a shared head's dq or dk
  w.dq_part = off;
  if (p->Nq < shares) off += align_up(TT * shares * p->K * sizeof(float));
  w.dk_part = off;
  if (p->Nk < shares) off += align_up(TT * shares * p->K * sizeof(float));
  w.chunk_states = off;
  if (p->io_dtype == M2RNN_F32 && C > bwd_f32_piece()) off += align_up(BN * ((C + bwd_f32_piece() - 1) / bwd_f32_piece()) * KV * sizeof(float));
  w.dv_part = off;
  if (RS > 1) off += align_up((size_t)RS * TT * p->N * p->V * sizeof(float));
  w.dgate_part = off;
  if (RS > 1) off += align_up((size_t)RS * TT * p->N * sizeof(float));
  w.total = off;
  return w;
}

ScanArgs base_args(const m2rnn_params *p) {
  ScanArgs a{};
  a.B = p->B; a.T = p->T; a.N = p->N; a.Nq = p->Nq; a.Nk = p->Nk; a.K = p->K; a.V = p->V;
  a.gate_kind = p->gate_kind;
  a.dh_clip = p->dh_clip;
  a.qs = p->q_stride ? p->q_stride : (long long)p->Nq * p->K;
  a.ks = p->k_stride ? p->k_stride : (long long)p->Nk * p->K;
  a.vs = p->v_stride ? p->v_stride : (long long)p->N * p->V;
  a.TT = (long long)tokens_of(p);
  a.cu = p->cu_seqlens;
  return a;
}
// (plans only where a call uses them: they are a part of a small call's host time)
void plan_forward(ScanArgs &a, const m2rnn_params *p) { a.KCf = plan_fwd_rows(p->B, p->N, p->K, p->V, p->io_dtype, tokens_of(p)); }
void plan_backward(ScanArgs &a, const m2rnn_params *p, const BwdPlan &pl) {
  a.KC = pl.KC; a.hg = pl.hg; a.groups = pl.groups; a.set = pl.set;
  a.C = p->ckpt_interval ? p->ckpt_interval : pl.C;
  const int interval = p->ckpt_interval ? p->ckpt_interval : pl.interval;
  a.per = a.C / interval;
  a.nchunks = p->T > 0 ? (p->T + interval - 1) / interval : 0;
}

}  // namespace

size_t bwd_workspace_bytes(const m2rnn_params *params, bool have_ckpt, bool lean) {
  if (check_params(params, true) != M2RNN_OK) return 0;
  return layout(params, plan_bwd(params, lean, have_ckpt), have_ckpt).total;
}

int bwd_call(const m2rnn_params *params, const void *q, const void *k, const void *v, const float *gate, const void *W,
             const float *h0, const float *alpha, const float *beta, const void *w_r, const float *ckpt, const void *dy,
             const float *d_hT, void *dq, void *dk, void *dv, float *dgate, float *dW, float *dh0, void *workspace,
             size_t workspace_bytes, bool lean, int32_t *dev_status, void *stream) {
  int rc = check_params(params, true);
  if (rc != M2RNN_OK) return rc;
  if (!dW) return M2RNN_ERR_NULL;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (params->B == 0 || params->T == 0 || tokens_of(params) == 0) {
    // empty scan: the only defined outputs are dW = 0 and dh0 = d_hT (or 0)
    if (!aligned16(dW) || !aligned16(dh0) || !aligned16(d_hT)) return M2RNN_ERR_ALIGN;
    cudaError_t e = cudaMemsetAsync(dW, 0, sizeof(float) * params->N * params->V * params->V, s);
    if (e == cudaSuccess && dh0 && params->B > 0) {
      const size_t bytes = sizeof(float) * (size_t)params->B * params->N * params->K * params->V;
      e = d_hT ? cudaMemcpyAsync(dh0, d_hT, bytes, cudaMemcpyDeviceToDevice, s) : cudaMemsetAsync(dh0, 0, bytes, s);
    }
    return e == cudaSuccess ? M2RNN_OK : cuda_failed();
  }
  if (!q || !k || !v || !gate || !W || !dy || !dq || !dk || !dv || !dgate) return M2RNN_ERR_NULL;
  if (params->gate_kind == M2RNN_GATE_PSI && (!alpha || !beta)) return M2RNN_ERR_NULL;
  const void *ptrs[] = {q, k, v, gate, W, h0, w_r, ckpt, dy, d_hT, dq, dk, dv, dgate, dW, dh0};
  for (const void *p : ptrs)
    if (!aligned16(p)) return M2RNN_ERR_ALIGN;
  const BwdPlan pl = plan_bwd(params, lean, ckpt != nullptr);
  const Workspace w = layout(params, pl, ckpt != nullptr);
  if (w.total > 0 && (!workspace || workspace_bytes < w.total)) return M2RNN_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(workspace) % kAlign) return M2RNN_ERR_ALIGN;
  char *ws = static_cast<char *>(workspace);

  ScanArgs a = base_args(params);
  plan_backward(a, params, pl);
  a.q = q; a.k = k; a.v = v; a.gate = gate; a.W = W; a.h0 = h0; a.w_r = w_r;
  a.alpha = params->gate_kind == M2RNN_GATE_PSI ? alpha : nullptr;
  a.beta = params->gate_kind == M2RNN_GATE_PSI ? beta : nullptr;
  a.dev_status = dev_status;
  const bool f32 = params->io_dtype == M2RNN_F32;
  cudaError_t e = cudaSuccess;
  if (!ckpt) {
    // pass 1 of Algorithm 2, thinned: save the state every C steps only
    ScanArgs f = a;
    plan_forward(f, params);
    f.C = a.C / a.per;
    f.y = nullptr; f.hT = nullptr;
    f.ckpt = reinterpret_cast<float *>(ws + w.ckpt);
    e = f32 ? launch_fwd_f32(f, s) : launch_fwd_bf16(f, s);
    if (e != cudaSuccess) return cuda_failed();
    a.ckpt = f.ckpt;
  } else {
    a.ckpt = const_cast<float *>(ckpt);
  }
  a.dy = dy; a.d_hT = d_hT; a.dq = dq; a.dk = dk; a.dv = dv; a.dgate = dgate; a.dh0 = dh0;
  a.dW_part = reinterpret_cast<float *>(ws + w.dW_part);
  const int shares = a.groups ? a.groups : params->N;
  a.dq_part = params->Nq < shares ? reinterpret_cast<float *>(ws + w.dq_part) : nullptr;
  a.dk_part = params->Nk < shares ? reinterpret_cast<float *>(ws + w.dk_part) : nullptr;
  a.chunk_states = f32 ? reinterpret_cast<float *>(ws + w.chunk_states) : nullptr;
  const int RS = params->K / a.KC;
  a.dv_part = RS > 1 ? reinterpret_cast<float *>(ws + w.dv_part) : nullptr;
  a.dgate_part = RS > 1 ? reinterpret_cast<float *>(ws + w.dgate_part) : nullptr;
  e = f32 ? launch_bwd_f32(a, s)
      : a.hg ? launch_bwd_v16(a, s)
          : (bwd_use_tc(params->B, params->N, params->K, params->V, params->io_dtype) ? launch_bwd_bf16_tc(a, s) : launch_bwd_bf16(a, s));
  if (e != cudaSuccess) return cuda_failed();
  e = launch_reduce_dW(a.dW_part, dW, params->B * RS, params->N, params->V, s);
  if (e != cudaSuccess) return cuda_failed();
  const size_t BT = tokens_of(params);
  if (RS > 1) {
    e = launch_reduce_slabs(a.dv_part, dv, params->io_dtype, RS, BT * params->N * params->V, s);
    if (e != cudaSuccess) return cuda_failed();
    e = launch_reduce_slabs(a.dgate_part, dgate, M2RNN_F32, RS, BT * params->N, s);
    if (e != cudaSuccess) return cuda_failed();
  }
  if (a.dq_part) {
    e = launch_reduce_heads(a.dq_part, dq, params->io_dtype, BT, shares, params->Nq, params->K, s);
    if (e != cudaSuccess) return cuda_failed();
  }
  if (a.dk_part) {
    e = launch_reduce_heads(a.dk_part, dk, params->io_dtype, BT, shares, params->Nk, params->K, s);
    if (e != cudaSuccess) return cuda_failed();
  }
  return M2RNN_OK;
}

}  // namespace m2rnn

using namespace m2rnn;

extern "C" {

int m2rnn_version(void) { return 100; }

const char *m2rnn_status_string(int status) {
  switch (status) {
    case M2RNN_OK: return "ok";
    case M2RNN_ERR_NULL: return "a required pointer is NULL";
    case M2RNN_ERR_SHAPE: return "bad size: non-positive, or a head count that does not divide N";
    case M2RNN_ERR_UNSUPPORTED: return "unsupported K, V, dtype, gate kind or checkpoint interval";
    case M2RNN_ERR_ALIGN: return "a pointer is not 16-byte aligned (workspace: 256-byte)";
    case M2RNN_ERR_WORKSPACE: return "workspace missing or too small";
    case M2RNN_ERR_CUDA: return "the CUDA runtime refused the launch";
    case M2RNN_ERR_TIMEOUT: return "a bounded device-side wait ran out";
    default: return "unknown status";
  }
}

int m2rnn_ckpt_interval(const m2rnn_params *params) {
  int rc = check_params(params, false);
  if (rc != M2RNN_OK) return rc;
  return interval_of(params);
}

int m2rnn_bwd_row_slab(const m2rnn_params *params) {
  int rc = check_params(params, false);
  if (rc != M2RNN_OK) return rc;
  return plan_bwd(params).KC;
}

size_t m2rnn_ckpt_bytes(const m2rnn_params *params) {
  if (check_params(params, true) != M2RNN_OK || params->T == 0) return 0;
  const int C = interval_of(params);
  return (size_t)params->B * params->N * ((params->T + C - 1) / C) * params->K * params->V * sizeof(float);
}

size_t m2rnn_fwd_workspace_bytes(const m2rnn_params *params) {
  if (check_params(params, true) != M2RNN_OK) return 0;
  const int kcf = plan_fwd_rows(params->B, params->N, params->K, params->V, params->io_dtype, tokens_of(params));
  const int RS = (params->K + kcf - 1) / kcf;
  if (RS <= 1) return 0;
  return align_up((size_t)RS * tokens_of(params) * params->N * params->V * sizeof(float));
}

int m2rnn_fwd(const m2rnn_params *params, const void *q, const void *k, const void *v,
              const float *gate, const void *W, const float *h0, const float *alpha,
              const float *beta, const void *w_r, void *y, float *hT, float *ckpt,
              void *workspace, size_t workspace_bytes, int32_t *dev_status, void *stream) {
  int rc = check_params(params, true);
  if (rc != M2RNN_OK) return rc;
  if (params->B == 0 || params->T == 0 || tokens_of(params) == 0) return M2RNN_OK;
  if (!q || !k || !v || !gate || !W || !y) return M2RNN_ERR_NULL;
  if (params->gate_kind == M2RNN_GATE_PSI && (!alpha || !beta)) return M2RNN_ERR_NULL;
  const void *ptrs[] = {q, k, v, gate, W, h0, w_r, y, hT, ckpt};
  for (const void *p : ptrs)
    if (!aligned16(p)) return M2RNN_ERR_ALIGN;
  ScanArgs a = base_args(params);
  a.q = q; a.k = k; a.v = v; a.gate = gate; a.W = W; a.h0 = h0; a.w_r = w_r;
  a.alpha = params->gate_kind == M2RNN_GATE_PSI ? alpha : nullptr;
  a.beta = params->gate_kind == M2RNN_GATE_PSI ? beta : nullptr;
  plan_forward(a, params);
  if (ckpt) {
    plan_backward(a, params, plan_bwd(params));
    a.C /= a.per;                                       // (the checkpoints' interval)
  }
  a.y = y; a.hT = hT; a.ckpt = ckpt; a.dev_status = dev_status;
  size_t need = m2rnn_fwd_workspace_bytes(params);
  if (need > 0 && !workspace && workspace_bytes == 0) {   // without shares of y, where the kernels can
    const int rows = plan_fwd_rows(params->B, params->N, params->K, params->V, params->io_dtype, tokens_of(params), true);
    if (rows == params->K) { a.KCf = rows; need = 0; }
  }
  if (need > 0) {
    if (!workspace || workspace_bytes < need) return M2RNN_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(workspace) % kAlign) return M2RNN_ERR_ALIGN;
    a.y_part = static_cast<float *>(workspace);
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = params->io_dtype == M2RNN_F32 ? launch_fwd_f32(a, s) : launch_fwd_bf16(a, s);
  if (e == cudaSuccess && a.y_part)
    e = launch_reduce_slabs(a.y_part, y, params->io_dtype, (params->K + a.KCf - 1) / a.KCf,
                            tokens_of(params) * params->N * params->V, s);
  return e == cudaSuccess ? M2RNN_OK : cuda_failed();
}

size_t m2rnn_bwd_workspace_bytes(const m2rnn_params *params, int have_ckpt) {
  if (check_params(params, true) != M2RNN_OK) return 0;
  const BwdPlan pl = plan_bwd(params, false, have_ckpt != 0);
  size_t most = layout(params, pl, have_ckpt != 0).total;
  if (pl.T_from > 1 && pl.T_from <= params->T) {
    // What the shorter sequences of this size take that have another plan: a workspace for the longest does for all
    m2rnn_params p = *params;
    p.T = pl.T_from - 1;
    if (p.total_tokens > (int64_t)p.B * p.T) p.total_tokens = (int64_t)p.B * p.T;
    most = std::max(most, layout(&p, plan_bwd(&p, false, have_ckpt != 0), have_ckpt != 0).total);
  }
  return most;
}

int m2rnn_bwd(const m2rnn_params *params, const void *q, const void *k, const void *v,
              const float *gate, const void *W, const float *h0, const float *alpha,
              const float *beta, const void *w_r, const float *ckpt, const void *dy,
              const float *d_hT, void *dq, void *dk, void *dv, float *dgate, float *dW,
              float *dh0, void *workspace, size_t workspace_bytes, int32_t *dev_status,
              void *stream) {
  return bwd_call(params, q, k, v, gate, W, h0, alpha, beta, w_r, ckpt, dy, d_hT, dq, dk, dv, dgate, dW, dh0, workspace, workspace_bytes,
                  false, dev_status, stream);
}

int m2rnn_decode_step(const m2rnn_params *params, const void *q, const void *k, const void *v,
                      const float *gate, const void *W, const float *alpha, const float *beta,
                      const void *w_r, float *state, void *y, int32_t *dev_status, void *stream) {
  int rc = check_params(params, false);
  if (rc != M2RNN_OK) return rc;
  if (params->B == 0) return M2RNN_OK;
  if (!q || !k || !v || !gate || !W || !state || !y) return M2RNN_ERR_NULL;
  if (params->gate_kind == M2RNN_GATE_PSI && (!alpha || !beta)) return M2RNN_ERR_NULL;
  const void *ptrs[] = {q, k, v, gate, W, w_r, state, y};
  for (const void *p : ptrs)
    if (!aligned16(p)) return M2RNN_ERR_ALIGN;
  ScanArgs a = base_args(params);
  a.T = 1; a.nchunks = 1;
  a.q = q; a.k = k; a.v = v; a.gate = gate; a.W = W; a.w_r = w_r;
  a.alpha = params->gate_kind == M2RNN_GATE_PSI ? alpha : nullptr;
  a.beta = params->gate_kind == M2RNN_GATE_PSI ? beta : nullptr;
  a.h0 = state; a.hT = state; a.y = y; a.ckpt = nullptr; a.dev_status = dev_status;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // one step of Eq. 1-3, the state read and written in place
  cudaError_t e = params->io_dtype == M2RNN_F32 ? launch_decode_f32(a, s) : launch_decode_bf16(a, s);
  return e == cudaSuccess ? M2RNN_OK : cuda_failed();
}

}  // extern "C"
