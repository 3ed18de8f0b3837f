// Internal declarations shared by the host API and the kernel translation units.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "m2rnn.h"

namespace m2rnn {

// Everything a kernel needs, by value.  Pointers are device pointers.
struct ScanArgs {
  int B, T, N, Nq, Nk, K, V;
  int gate_kind;
  int KC;         // backward: state rows per CTA (a divisor of K)
  int KCf;        // forward: state rows per CTA (a divisor of K)
  int C;          // checkpoint interval (steps); backward: steps of a chunk, `per` intervals
  int nchunks;    // checkpoints of a unit: ceil(T / interval)
  float dh_clip;
  const void *q, *k, *v, *W, *w_r;
  const float *gate, *h0, *alpha, *beta;
  void *y;
  float *y_part;  // forward, K/KCf > 1: [K/KCf][B,T,N,V] fp32 per-row-slab y, else null
  float *hT;
  float *ckpt;    // fwd: written (may be null); bwd: read
  // backward only
  const void *dy;
  const float *d_hT;
  void *dq, *dk, *dv;  // dq/dk: final tensors when the head is not shared, else see dq_part
  float *dgate, *dh0;
  float *dW_part;      // [B*K/KC,N,V,V] per-CTA partial sums of dW
  float *dv_part;      // [K/KC][B,T,N,V] fp32 per-row-slab dv when K/KC > 1, else null
  float *dgate_part;   // [K/KC][B,T,N] fp32 per-row-slab dgate when K/KC > 1, else null
  float *dq_part;      // [B,T,shares,K] fp32 shares of dq when Nq < N (a share per head; V = 16: per CTA's heads), else null
  float *dk_part;      // likewise dk, when Nk < N
  float *chunk_states; // fp32 path, C > 16: [B*N, ceil(C/16), K, V] states between the pieces of a chunk
  int32_t *dev_status;
  // token addressing: elements between consecutive tokens of q, k, v (dense: Nq K, Nk K, N V; larger
  // when they alias one fused projection output), the tokens in the batch (B T, or the packed total)
  // and, for packed variable-length batches, the device array of B + 1 token offsets
  long long qs, ks, vs;
  long long TT;
  const int32_t *cu;
  int hg, groups, set;   // backward, V = 16: heads per CTA, CTAs per token's heads (= shares of dq and dk), heads that a CTA's are taken from
  int per;        // backward, V = 16: checkpoints to a chunk (else 1)
  int rank;       // B where the sequences of a packed batch are taken longest first, else 0
};

// First token and length of batch entry b: a slice [cu[b], cu[b+1]) of a packed batch, else b T .. b T + T
struct UnitSpan { size_t tok0; int T; };
#ifdef __CUDACC__
__device__ __forceinline__ UnitSpan unit_span(const ScanArgs &a, int b) {
  if (a.cu) {   // lengths outside 0 .. T are cut to that range: nothing is addressed beyond what T sized
    const int s = a.cu[b], len = a.cu[b + 1] - s;
    return UnitSpan{(size_t)s, len < 0 ? 0 : (len > a.T ? a.T : len)};
  }
  return UnitSpan{(size_t)b * a.T, a.T};
}
// The batch entry that the CTAs at place `pos` of the grid's order take.  Sequences of a packed batch are
// taken longest first (a.rank > 0, see in_order): CTAs are handed out in order, and a long one that starts last leaves the
// other SMs idle (12 sequences of up to 4 000 tokens, K = V = 128, forward + backward: 20.4 -> 18.6 ms).
// Every thread of the CTA calls it, before it uses `scratch` (shared memory) otherwise.
// (Not inlined, and the condition no simpler than it is: the kernels' inner loops are sensitive to what the compiler
// schedules around them.  `a.rank` alone costs every scan at V = 128 1.2 %, packed or not, `a.cu && a.rank` four slabs of
// V = 64 0.5 %; a ranking on keys staged in shared memory, four times as fast, the V = 128 backward 0.7 %.)
static __device__ __noinline__ int longest_first(const int32_t *cu, int B, int pos, int *scratch);
__device__ __forceinline__ int batch_entry(const ScanArgs &a, int pos, void *scratch) {
  // (through a shuffle: known to be the same in all lanes, so that what derives from it stays in uniform
  // registers -- 5 to 9 % of a step in the tcgen05 kernel)
  return __shfl_sync(0xffffffffu, a.cu && a.rank > 1 && a.rank <= 1024 ? longest_first(a.cu, a.B, pos, static_cast<int *>(scratch)) : pos, 0);
}
static __device__ __noinline__ int longest_first(const int32_t *cu, int B, int pos, int *scratch) {
  for (int b = threadIdx.x; b < B; b += blockDim.x) {
    const int len = cu[b + 1] - cu[b];
    int rank = 0;
    for (int o = 0; o < B; ++o) {
      const int other = cu[o + 1] - cu[o];
      rank += other > len || (other == len && o < b);
    }
    if (rank == pos) *scratch = b;
  }
  __syncthreads();
  const int b = *static_cast<volatile int *>(scratch);
  __syncthreads();
  return b;
}
// A launch whose set-up overlaps the end of the kernel before it in the stream (programmatic dependent launch): its CTAs come as
// that one's last end, and wait in begin_dependent, every thread's first statement that is not address arithmetic, until that one
// is done and its writes are seen.  For the kernels of 2 to 100 us, whose gaps count: a decoding step (B=48, N=84, K=64, V=16, steps
// back to back) 8.2 -> 6.0 us, conv forward + backward [8, 2048, 3072] 100.3 -> 93.9, [1, 927, 3920] 20.6 -> 14.9, the gated norm's
// pair (16 384 rows of 1 344) 70.4 -> 64.6, 1 001 rows 14.4 -> 10.0.  No kernel asks for its dependents before it ends
// (launch_dependents): waiting CTAs then land where the running ones happen to leave room, not one on each SM, and a grid of one
// or two rounds is bound by its fullest SM: [1, 927, 3920] 21.4 us so, conv forward in fp32 [1, 2000, 3072] 16.7 against 11.1 (plain
// 12.4).  Of the scans those of short steps take it: 1 001 tokens through conv, scan and norm (N=84, K=64, V=16) 99.7 -> 98.0, one
// sequence of 433 tokens forward + backward (30 heads of K=V=32) 196.5 -> 192.2; the V = 128 kernels on the tensor memory gain nothing.
template <typename... P, typename... A>
inline cudaError_t launch_early(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cfg.attrs = &at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
__device__ __forceinline__ void begin_dependent() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// The arguments of a scan kernel's launch of `ctas` CTAs of `threads`, with the order of a packed batch decided.
// `pace`: the kernel's time per step, in 0.1 us.
// Every CTA ranks the batch for itself, B comparisons for each sequence that a thread takes, some 0.02 us each.
// Waves of CTAs times that has to stay below what the order can give, a part of the longest scan, which counts once.
// Forward, two heads of K = V = 64, us in the grid's order / ranked: 256 sequences of up to 256 tokens 164 / 136, 512 of
// 2048 2050 / 1810 -- ranked by the rule; 512 of 256 286 / 357, 1000 of 32 113 / 922 -- not.  16 heads of K = 64,
// V = 16: 256 of 2048 1490 / 1392 ranked, of 256 201 / 277 not.
inline ScanArgs in_order(const ScanArgs &args, long ctas, int threads, int pace) {
  ScanArgs a = args;
  const double waves = (double)ctas * threads / 75776.;   // (512 threads on each of 148 SMs)
  a.rank = a.cu && a.B > 1 && waves * a.B * ((a.B + threads - 1) / threads) <= 2.7 * pace * a.T ? a.B : 0;
  return a;
}
#endif

constexpr size_t kAlign = 256;
inline size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

// How the backward pass splits a problem: state rows per CTA and the checkpoint interval (bounded
// by shared memory in the bf16 backward kernel, which keeps two chunks of recomputed states on chip).
struct BwdPlan {
  int KC;     // rows per CTA (fp32 path: 4 or 8, or K for one launch per group of eight)
  int C;      // steps of a chunk where the caller gives no interval
  int interval;   // steps between checkpoints: C, or half of it (V = 16, bf16)
  int C_max;  // largest supported checkpoint interval
  int T_from; // the plan is that of T >= T_from, another one below
  int hg, groups, set;   // V = 16 (bf16): see ScanArgs
};
int sm_count();   // SMs of the current device (148 when there is none to ask)
bool current_context(uint64_t *id);   // the current context's number, unique for the life of the process
cudaError_t allow_smem(const void *kernel, size_t bytes);   // dynamic shared memory a launch may use
template <typename... A> cudaError_t allow_smem(void (*kernel)(A...), size_t bytes) {
  return allow_smem(reinterpret_cast<const void *>(kernel), bytes);
}
// (lean: as little scratch as there can be: an fp32 problem's groups of rows one after the other, without shares of
// dv and dW; have_ckpt false: the interval is the call's own business)
BwdPlan plan_bwd(const m2rnn_params *p, bool lean = false, bool have_ckpt = true);
BwdPlan plan_bwd_v16(int B, int N, int Nq, int Nk, int K, int T, int interval, bool lean);   // scan_bwd_v16.cu: V = 16, bf16
size_t tokens_of(const m2rnn_params *p);
// m2rnn_bwd and its workspace query; lean: see plan_bwd
size_t bwd_workspace_bytes(const m2rnn_params *params, bool have_ckpt, bool lean);
int bwd_call(const m2rnn_params *params, const void *q, const void *k, const void *v, const float *gate, const void *W,
             const float *h0, const float *alpha, const float *beta, const void *w_r, const float *ckpt, const void *dy,
             const float *d_hT, void *dq, void *dk, void *dv, float *dgate, float *dW, float *dh0, void *workspace,
             size_t workspace_bytes, bool lean, int32_t *dev_status, void *stream);
int plan_fwd_rows(int B, int N, int K, int V, int io_dtype, size_t tokens = 0, bool lean = false);   // state rows per CTA of the forward kernel
// Which bf16 forward kernel takes a problem: the tcgen05 kernel (scan_fwd_tc.cu) or the mma.sync
// kernels (scan_fwd_bf16*.cu).  The environment variable M2RNN_FWD_VARIANT = tc | mma
// overrides the choice (benchmarking only).
bool fwd_use_tc(int B, int N, int K, int V, int io_dtype);
int fwd_tc_rows_per_cta(int B, int N, int K, int V);                 // scan_fwd_tc.cu: 32 or 64
cudaError_t launch_fwd_bf16_tc(const ScanArgs &a, cudaStream_t s);  // scan_fwd_tc.cu
size_t bwd_bf16_smem_bytes(int KC, int V, int C);  // scan_bwd_bf16.cu

// fp32 FMA path (scan_f32.cu)
cudaError_t launch_fwd_f32(const ScanArgs &a, cudaStream_t s);
cudaError_t launch_bwd_f32(const ScanArgs &a, cudaStream_t s);      // KC = 4, 8: every group of that many rows at once, KC = K: groups of eight one after the other
cudaError_t launch_decode_f32(const ScanArgs &a, cudaStream_t s);
int fwd_f32_rows(int B, int N, int K, int V, size_t share_bytes);
int bwd_f32_rows(int B, int N, int K, int V, size_t share_bytes);
int bwd_f32_piece();   // steps whose states the backward kernel keeps on chip

// bf16 tensor-core path
cudaError_t launch_fwd_bf16(const ScanArgs &a, cudaStream_t s);     // scan_fwd_bf16.cu: picks a variant
cudaError_t launch_fwd_v16(const ScanArgs &a, cudaStream_t s);      // scan_fwd_v16.cu: V = 16
bool fwd_cs_supported(const ScanArgs &a);                            // scan_fwd_bf16_cs.cu
cudaError_t launch_fwd_bf16_cs(const ScanArgs &a, cudaStream_t s);  // scan_fwd_bf16_cs.cu: two or four warps per 16-row slab
cudaError_t launch_bwd_bf16(const ScanArgs &a, cudaStream_t s);     // scan_bwd_bf16.cu: 32 <= V
cudaError_t launch_bwd_v16(const ScanArgs &a, cudaStream_t s);      // scan_bwd_v16.cu: V = 16
// The tcgen05 backward kernel (scan_bwd_tc.cu) takes V = 128; M2RNN_BWD_VARIANT = tc | mma overrides
// the choice (benchmarking only).
bool bwd_use_tc(int B, int N, int K, int V, int io_dtype);
int bwd_tc_rows_per_cta();
int bwd_tc_chunk();
cudaError_t launch_bwd_bf16_tc(const ScanArgs &a, cudaStream_t s);  // scan_bwd_tc.cu
cudaError_t launch_decode_bf16(const ScanArgs &a, cudaStream_t s);  // decode_bf16.cu: picks a kernel
cudaError_t launch_decode_tc_bf16(const ScanArgs &a, cudaStream_t s);  // decode_tc_bf16.cu: tcgen05 path

// reductions shared by both paths (reduce.cu)
cudaError_t launch_reduce_dW(const float *dW_part, float *dW, int B, int N, int V, cudaStream_t s);
cudaError_t launch_reduce_slabs(const float *part, void *out, int io_dtype, int R, size_t n, cudaStream_t s);
cudaError_t launch_reduce_heads(const float *part, void *out, int io_dtype, size_t BT, int N,
                                int Ng, int K, cudaStream_t s);

}  // namespace m2rnn
