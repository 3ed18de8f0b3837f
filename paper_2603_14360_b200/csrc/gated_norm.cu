// Output path of the layer after the scan ("M2RNN block" equations: y_gt = RMSNorm(y_t (.) g_t),
// g_t = SiLU of the gate projection; RMSNorm appendix for the formulas and their backward), fused
// into one pass each way: y and g are read once, the normalised product is written once, the
// product y (.) g never goes to memory.  Per token over the d = N V features of all heads:
//     x = y (.) g,   s = 1 / sqrt(mean x^2 + eps),   out = w (.) x s            (s is cached)
//     p = w (.) dout, r = sum p x, dx = s p - r s^3 x / d, dy = dx (.) g, dg = dx (.) y (SiLU'),
//     dw = sum over tokens of dout (.) x s.
// HBM-bound.  One to eight warps share a row so that a lane holds at most three chunks of eight features (four of a row
// of 1 024, see split_of):
// that keeps its share of the row, its columns' dw sums and the next row on the way (16-byte cp.async
// into a ring) within two (backward) to four CTAs per SM, whatever the row length.  One partial of dw per
// persistent CTA, added by a fixed-order second stage.  16 384 rows: of 1 344 features (84 heads x 16)
// forward 26 us (5.1 TB/s), backward 39 us (5.6 TB/s); of 1 888, 42 and 69 us (6.0 TB/s).  (Launches apart; one after the
// other, each started while the one before it ends, the pair of 1 344 takes 65 us and took 70.)  (A warp per row,
// rows of other lengths than 256 times a power of two walked twice: 31 and 80, 64 and 141 us.  A CTA
// per row or four rows at a time, a chunk per thread: 31-42 and 60 us, the barriers show.)
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "internal.h"
#include "m2rnn.h"

namespace m2rnn {
namespace {

constexpr int kMaxCtas = 592;   // 4 per SM on 148 SMs: the number of dw partials at most
constexpr int kMaxD = 8192;
constexpr int kThreads = 256, kWarps = kThreads / 32;

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t *>(&v);
}
__device__ __forceinline__ void store8(__nv_bfloat16 *p, const float (&f)[8]) {
  *reinterpret_cast<uint4 *>(p) = make_uint4(pack2(f[0], f[1]), pack2(f[2], f[3]), pack2(f[4], f[5]), pack2(f[6], f[7]));
}
__device__ __forceinline__ void store8(float *p, const float (&f)[8]) {
  *reinterpret_cast<float4 *>(p) = make_float4(f[0], f[1], f[2], f[3]);
  *reinterpret_cast<float4 *>(p + 4) = make_float4(f[4], f[5], f[6], f[7]);
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Sigmoid of a pair.  fp32 I/O: through ex2.approx + rcp.approx (~1e-6 relative); bf16 I/O: through
// tanh.approx (~2^-11, below the rounding of the bf16 result), half the work of the special-function unit.
// The arithmetic below is in packed fp32 pairs: the backward kernel is bound by instruction issue as
// much as by HBM.
template <typename T>
__device__ __forceinline__ float2 sigmoid2(float2 x) {
  if constexpr (sizeof(T) == 2) {
    const float2 h = __fmul2_rn(x, make_float2(0.5f, 0.5f));
    float2 th;
    asm("tanh.approx.f32 %0, %1;" : "=f"(th.x) : "f"(h.x));
    asm("tanh.approx.f32 %0, %1;" : "=f"(th.y) : "f"(h.y));
    return __ffma2_rn(th, make_float2(0.5f, 0.5f), make_float2(0.5f, 0.5f));
  } else {
    return make_float2(__fdividef(1.f, 1.f + __expf(-x.x)), __fdividef(1.f, 1.f + __expf(-x.y)));
  }
}

// eight elements of a row: one (bf16) or two (fp32) pieces of 16 bytes
template <typename T> struct Raw8 { static constexpr int kPieces = sizeof(T) / 2; uint4 v[kPieces]; };
__device__ __forceinline__ float2 pair_of(const Raw8<__nv_bfloat16> &r, int i) {
  const uint32_t u[4] = {r.v[0].x, r.v[0].y, r.v[0].z, r.v[0].w};
  return make_float2(__uint_as_float(u[i] << 16), __uint_as_float(u[i] & 0xffff0000u));
}
__device__ __forceinline__ float2 pair_of(const Raw8<float> &r, int i) {
  const uint4 q = r.v[i >> 1];
  return (i & 1) ? make_float2(__uint_as_float(q.z), __uint_as_float(q.w)) : make_float2(__uint_as_float(q.x), __uint_as_float(q.y));
}
template <typename T>
__device__ __forceinline__ Raw8<T> load_raw(const T *p) {
  Raw8<T> r;
#pragma unroll
  for (int i = 0; i < Raw8<T>::kPieces; ++i) r.v[i] = reinterpret_cast<const uint4 *>(p)[i];
  return r;
}

// Whether rows go through the ring (below) or straight to registers: bf16 only.  (fp32 moves twice the bytes
// per lane, its ring leaves room for one CTA per SM: 4 096 x 1 344 forward 22 us with it, 16 without.)
__host__ __device__ constexpr bool uses_ring(int elem) { return elem == 2; }
// CTAs per SM a variant is compiled for and launched with: what its registers and its ring allow.
// chunks: of a lane at a time (CPL R); full: see Walk
__host__ __device__ constexpr int resident(bool bwd, int elem, int chunks, bool full) {
  if (full) return bwd ? (chunks == 1 ? 3 : (chunks == 2 ? 2 : 1)) : (chunks == 1 ? 8 : (chunks == 2 && elem == 2 ? 5 : 3));
  return bwd ? (elem == 4 && chunks > 3 ? 1 : 2) : (chunks <= 2 ? 4 : 3);
}

// The way of a CTA's warps over the rows.  G warps share a row, a lane takes CPL chunks of eight features of it;
// the CTA holds 8/G such groups, each with R rows at a time (short rows only).  Rows travel through a
// ring of two stages in shared memory of which a lane copies (cp.async) and reads its own 16-byte
// pieces only: the next rows are on their way while these are worked on, a second pass over a row
// reads them again, and no barrier is needed.
// FULL: a row is exactly the lanes' chunks, which then are loaded without a look at the row's end, all of them
// before the first is used, and need no ring.
template <typename T, int CPL, int R, int G, int NTENS, bool FULL>
struct Walk {
  static constexpr int NP = Raw8<T>::kPieces, kGroups = kWarps / G;
  static constexpr bool kRing = uses_ring(sizeof(T)) && !FULL;
  static constexpr int kSmem = kRing ? 2 * NTENS * R * CPL * NP * kThreads * 16 : 0;
  uint4 *ring;
  int lane, group, gw;               // gw: warp of the group
  long t, step, tokens;
  int d, col;                        // the lane's first column; chunk j is 256 G columns further
  __device__ __forceinline__ Walk(unsigned char *smem, long tokens_, int d_) {
    const int tid = threadIdx.x, warp = tid >> 5;
    lane = tid & 31;
    group = warp / G; gw = warp % G;
    ring = reinterpret_cast<uint4 *>(smem) + tid;
    tokens = tokens_; d = d_;
    t = ((long)blockIdx.x * kGroups + group) * R;
    step = (long)gridDim.x * kGroups * R;
    col = 8 * (32 * gw + lane);
  }
  __device__ __forceinline__ bool on(int j) const { return FULL || col + 256 * G * j < d; }
  __device__ __forceinline__ uint4 *piece(int stage, int x, int r, int j, int p) const {
    return ring + ((((stage * NTENS + x) * R + r) * CPL + j) * NP + p) * kThreads;
  }
  __device__ __forceinline__ void fetch(int stage, long t0, const T *const (&src)[NTENS]) const {   // always one group, possibly empty
    if constexpr (!kRing) return;
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (t0 + r < tokens) {
#pragma unroll
        for (int x = 0; x < NTENS; ++x) {
          const T *p = src[x] + (t0 + r) * d + col;
#pragma unroll
          for (int j = 0; j < CPL; ++j)
            if (on(j))
#pragma unroll
              for (int q = 0; q < NP; ++q)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(piece(stage, x, r, j, q))),
                             "l"(reinterpret_cast<const uint4 *>(p + 256 * G * j) + q) : "memory");
        }
      }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  __device__ __forceinline__ Raw8<T> get(const T *const (&src)[NTENS], int stage, int x, int r, int j) const {
    Raw8<T> v;
    if constexpr (!kRing) return t + r < tokens ? load_raw(src[x] + (t + r) * d + col + 256 * G * j) : Raw8<T>{};
#pragma unroll
    for (int q = 0; q < NP; ++q) v.v[q] = *piece(stage, x, r, j, q);
    return v;
  }
  // the lane's chunks of this row (FULL)
  template <int N> __device__ __forceinline__ void get_row(const T *const (&src)[NTENS], Raw8<T> (&row)[N][CPL]) const {
    static_assert(FULL && R == 1 && N == NTENS);
#pragma unroll
    for (int j = 0; j < CPL; ++j)
#pragma unroll
      for (int x = 0; x < N; ++x) row[x][j] = load_raw(src[x] + t * d + col + 256 * G * j);
  }
  // v[r] summed over the group.  red: [2][kWarps][R] floats, used in turn so that one barrier a call is enough
  __device__ __forceinline__ void row_sums(float (&v)[R], float *red, int buf) const {
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = warp_sum(v[r]);
    if constexpr (G > 1) {
      red += (buf * kWarps + group * G) * R;
      if (lane == 0) {
#pragma unroll
        for (int r = 0; r < R; ++r) red[gw * R + r] = v[r];
      }
      asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(32 * G) : "memory");
#pragma unroll
      for (int r = 0; r < R; ++r) {
        v[r] = red[r];
#pragma unroll
        for (int w = 1; w < G; ++w) v[r] += red[w * R + r];
      }
    }
  }
};

template <typename T, int CPL, int R, int G, bool FULL>
__global__ void __launch_bounds__(kThreads, resident(false, sizeof(T), CPL * R, FULL)) gated_norm_fwd_kernel(
    long tokens, int d, const T *__restrict__ y, const T *__restrict__ g_in, const T *__restrict__ w, float eps, int use_silu,
    T *__restrict__ out, float *__restrict__ rstd) {
  extern __shared__ __align__(16) unsigned char smem[];
  begin_dependent();
  __shared__ float red[2 * kWarps * R];
  Walk<T, CPL, R, G, 2, FULL> wk(smem, tokens, d);
  const T *const src[2] = {y, g_in};
  wk.fetch(0, wk.t, src);
  const float inv_d = 1.f / (float)d;
  int st = 0;
  for (; wk.t < tokens; wk.t += wk.step, st ^= 1) {
    wk.fetch(st ^ 1, wk.t + wk.step, src);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    float2 x[R][CPL][4];
    float ss[R];
    Raw8<T> row[2][FULL ? CPL : 1];
    if constexpr (FULL) wk.get_row(src, row);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float2 s2 = make_float2(0.f, 0.f);
#pragma unroll
      for (int j = 0; j < CPL; ++j)
        if (wk.on(j)) {
          const Raw8<T> a = FULL ? row[0][FULL ? j : 0] : wk.get(src, st, 0, r, j), b = FULL ? row[1][FULL ? j : 0] : wk.get(src, st, 1, r, j);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float2 g = pair_of(b, i);
            if (use_silu) g = __fmul2_rn(g, sigmoid2<T>(g));
            x[r][j][i] = __fmul2_rn(pair_of(a, i), g);
            s2 = __ffma2_rn(x[r][j][i], x[r][j][i], s2);
          }
        }
      ss[r] = s2.x + s2.y;
    }
    wk.row_sums(ss, red, st);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (wk.t + r >= tokens) break;   // (a row past the end: arithmetic on stale shared memory, nothing stored)
      const float s = 1.f / sqrtf(ss[r] * inv_d + eps);
#pragma unroll
      for (int j = 0; j < CPL; ++j)
        if (wk.on(j)) {
          const Raw8<T> wv = load_raw(w + wk.col + 256 * G * j);
          float o[8];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float2 p = __fmul2_rn(__fmul2_rn(pair_of(wv, i), x[r][j][i]), make_float2(s, s));
            o[2 * i] = p.x; o[2 * i + 1] = p.y;
          }
          store8(out + (wk.t + r) * d + wk.col + 256 * G * j, o);
        }
      if (rstd && wk.col == 0) rstd[wk.t + r] = s;
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

template <typename T, int CPL, int R, int G, bool FULL>
__global__ void __launch_bounds__(kThreads, resident(true, sizeof(T), CPL * R, FULL)) gated_norm_bwd_kernel(
    long tokens, int d, const T *__restrict__ y, const T *__restrict__ g_in, const T *__restrict__ w, const float *__restrict__ rstd,
    int use_silu, const T *__restrict__ dout, T *__restrict__ dy, T *__restrict__ dg_in, float *__restrict__ dw_part) {
  extern __shared__ __align__(16) unsigned char smem[];
  begin_dependent();
  __shared__ float red[2 * kWarps * R];
  Walk<T, CPL, R, G, 3, FULL> wk(smem, tokens, d);
  const T *const src[3] = {y, g_in, dout};
  wk.fetch(0, wk.t, src);
  Raw8<T> wr[CPL];
  float2 acc[CPL][4];
#pragma unroll
  for (int j = 0; j < CPL; ++j) {
    if (wk.on(j)) wr[j] = load_raw(w + wk.col + 256 * G * j);
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[j][i] = make_float2(0.f, 0.f);
  }
  const float inv_d = 1.f / (float)d;
  const float2 one = make_float2(1.f, 1.f), mone = make_float2(-1.f, -1.f);
  int st = 0;
  for (; wk.t < tokens; wk.t += wk.step, st ^= 1) {
    float s[R], rs[R];
#pragma unroll
    for (int r = 0; r < R; ++r) s[r] = wk.t + r < tokens ? rstd[wk.t + r] : 0.f;
    wk.fetch(st ^ 1, wk.t + wk.step, src);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    float2 sg[R][CPL][4];
    Raw8<T> row[3][FULL ? CPL : 1];
    if constexpr (FULL) wk.get_row(src, row);
    auto piece = [&](int x, int r, int j) { return FULL ? row[x][FULL ? j : 0] : wk.get(src, st, x, r, j); };
#pragma unroll
    for (int r = 0; r < R; ++r) {   // r = sum_j w_j dout_j x_j
      float2 r2 = make_float2(0.f, 0.f);
#pragma unroll
      for (int j = 0; j < CPL; ++j)
        if (wk.on(j)) {
          const Raw8<T> a = piece(0, r, j), b = piece(1, r, j), dv = piece(2, r, j);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float2 g = pair_of(b, i);
            sg[r][j][i] = one;
            if (use_silu) { sg[r][j][i] = sigmoid2<T>(g); g = __fmul2_rn(g, sg[r][j][i]); }
            r2 = __ffma2_rn(__fmul2_rn(pair_of(wr[j], i), pair_of(dv, i)), __fmul2_rn(pair_of(a, i), g), r2);
          }
        }
      rs[r] = r2.x + r2.y;
    }
    wk.row_sums(rs, red, st);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (wk.t + r >= tokens) break;
      const float k3 = rs[r] * s[r] * s[r] * s[r] * inv_d;
      const float2 mk = make_float2(-k3, -k3), s2 = make_float2(s[r], s[r]);
#pragma unroll
      for (int j = 0; j < CPL; ++j)
        if (wk.on(j)) {
          const Raw8<T> a = piece(0, r, j), b = piece(1, r, j), dv = piece(2, r, j);
          float o1[8], o2[8];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float2 av = pair_of(a, i), bv = pair_of(b, i), sd = __fmul2_rn(s2, pair_of(dv, i)), q = sg[r][j][i];
            const float2 g = use_silu ? __fmul2_rn(bv, q) : bv;
            const float2 x = __fmul2_rn(av, g);
            const float2 dx = __ffma2_rn(pair_of(wr[j], i), sd, __fmul2_rn(mk, x));           // s w dout - k3 x
            const float2 p1 = __fmul2_rn(dx, g);
            float2 p2 = __fmul2_rn(dx, av);
            if (use_silu) p2 = __fmul2_rn(p2, __ffma2_rn(g, __ffma2_rn(q, mone, one), q));      // SiLU' = sg + g (1 - sg)
            acc[j][i] = __ffma2_rn(sd, x, acc[j][i]);
            o1[2 * i] = p1.x; o1[2 * i + 1] = p1.y;
            o2[2 * i] = p2.x; o2[2 * i + 1] = p2.y;
          }
          store8(dy + (wk.t + r) * d + wk.col + 256 * G * j, o1);
          store8(dg_in + (wk.t + r) * d + wk.col + 256 * G * j, o2);
        }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  // this CTA's partial of dw: the groups' sums in a fixed order, through shared memory (kGroups x d floats)
  float *sh = reinterpret_cast<float *>(smem);
  __syncthreads();
#pragma unroll
  for (int j = 0; j < CPL; ++j)
    if (wk.on(j))
#pragma unroll
      for (int i = 0; i < 4; ++i) *reinterpret_cast<float2 *>(sh + wk.group * d + wk.col + 256 * G * j + 2 * i) = acc[j][i];
  __syncthreads();
  for (int c = threadIdx.x; c < d; c += kThreads) {
    float v = 0.f;
#pragma unroll
    for (int k = 0; k < kWarps / G; ++k) v += sh[k * d + c];
    dw_part[(size_t)blockIdx.x * d + c] = v;
  }
}

// dw[j] = sum over the R per-CTA partials, in a fixed order: 32 interleaved running sums per column (one
// per warp of the CTA), then their sum in warp order
__global__ void __launch_bounds__(1024) reduce_partials_kernel(const float *__restrict__ part, float *__restrict__ out, int R, int n) {
  begin_dependent();
  __shared__ float sm[32][33];
  const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
  const int j = blockIdx.x * 32 + lane;
  float v = 0.f;
  if (j < n) {
#pragma unroll 4
    for (int r = grp; r < R; r += 32) v += part[(size_t)r * n + j];
  }
  sm[grp][lane] = v;
  __syncthreads();
  v = warp_sum(sm[lane][grp]);   // warp grp adds column grp's 32 sums
  if (lane == 0 && blockIdx.x * 32 + grp < n) out[blockIdx.x * 32 + grp] = v;
}

// How a call is split: warps per row (a lane holds at most three chunks: with four the backward kernel spills at
// two CTAs per SM; d > 6 144 has no choice), chunks per lane, rows at a time (short rows: as many
// bytes on their way as four chunks) and persistent CTAs, as many as are resident.
// Rows of exactly 256, 512 or 1 024 features: a warp each, its whole row loaded at once and without a ring, forward
// in as many CTAs as there are rows for, up to eight an SM.  The general form costs such rows 2 to 35 % (16 384
// rows, us: bf16 forward 7.7, 12.3, 19.7 -> 6.2, 10.3, 18.0; fp32 forward of 256 and 512 15.4, 22.9 -> 11.2, 18.4,
// backward 27, 46, 65 -> 20, 33, 59).  Not where it is no better: the bf16 backward (14.4, 20.9, 31.3, ring) and the fp32 forward
// of 1 024 (33.1, two warps a row; one 33 to 37).
struct Split { int g, cpl, r, grid; bool full; };
Split split_of(long tokens, int d, bool bwd, int io_dtype) {
  Split s;
  const int chunks = d / 8;
  const int sms = sm_count();
  const bool f32 = io_dtype == M2RNN_F32;
  s.full = bwd ? f32 && (chunks == 32 || chunks == 64 || chunks == 128) : chunks == 32 || chunks == 64 || (chunks == 128 && !f32);
  if (s.full) {
    s.g = 1; s.cpl = chunks / 32; s.r = 1;
    const long need = (tokens + kWarps - 1) / kWarps, slots = (long)sms * (bwd ? resident(true, 4, s.cpl, true) : 8);
    s.grid = (int)(need < slots ? need : slots);
    if (bwd && s.grid > kMaxCtas) s.grid = kMaxCtas;
    return s;
  }
  const int most = f32 ? 64 : 96;   // chunks of a warp
  s.g = chunks <= most ? 1 : (chunks <= 2 * most ? 2 : (chunks <= 4 * most ? 4 : 8));
  s.cpl = (chunks + 32 * s.g - 1) / (32 * s.g);
  s.r = s.g > 1 || s.cpl > 2 ? 1 : (s.cpl == 1 ? 4 : 2);
  const int per = kWarps / s.g;
  if (tokens < 8L * sms * per) s.r = 1;
  const long need = (tokens + per * s.r - 1) / (per * s.r);
  const long slots = (long)sms * resident(bwd, f32 ? 4 : 2, s.cpl * s.r, false);
  s.grid = (int)(need < slots ? need : slots);
  if (s.grid > kMaxCtas) s.grid = kMaxCtas;
  return s;
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int check(long tokens, int d, int io_dtype) {
  if (tokens < 0 || d <= 0) return M2RNN_ERR_SHAPE;
  if (io_dtype != M2RNN_F32 && io_dtype != M2RNN_BF16) return M2RNN_ERR_UNSUPPORTED;
  if (d % 8 || d > kMaxD) return M2RNN_ERR_UNSUPPORTED;
  return M2RNN_OK;
}

// f(CPL, R, G, FULL) as compile-time constants; kFull: the most chunks a lane of a FULL form takes (0: there is none)
template <int kFull, typename F>
cudaError_t with_split(const Split &s, F f) {
  using No = std::false_type;
  using One = std::integral_constant<int, 1>;
  if constexpr (kFull >= 2) {
    if (s.full && s.cpl == 1) return f(One{}, One{}, One{}, std::true_type{});
    if (s.full && s.cpl == 2) return f(std::integral_constant<int, 2>{}, One{}, One{}, std::true_type{});
  }
  if constexpr (kFull >= 4)
    if (s.full && s.cpl == 4) return f(std::integral_constant<int, 4>{}, One{}, One{}, std::true_type{});
#define M2RNN_CASE(C, R_, G_) \
  if (s.cpl == C && s.r == R_ && s.g == G_) \
    return f(std::integral_constant<int, C>{}, std::integral_constant<int, R_>{}, std::integral_constant<int, G_>{}, No{})
  M2RNN_CASE(1, 4, 1); M2RNN_CASE(1, 1, 1); M2RNN_CASE(2, 2, 1); M2RNN_CASE(2, 1, 1); M2RNN_CASE(3, 1, 1);
  M2RNN_CASE(2, 1, 2); M2RNN_CASE(3, 1, 2); M2RNN_CASE(2, 1, 4); M2RNN_CASE(3, 1, 4); M2RNN_CASE(2, 1, 8); M2RNN_CASE(3, 1, 8); M2RNN_CASE(4, 1, 8);
#undef M2RNN_CASE
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_fwd(long tokens, int d, const void *y, const void *g, const void *w, float eps, int silu_on, void *out,
                       float *rstd, cudaStream_t s) {
  const Split sp = split_of(tokens, d, false, sizeof(T) == 2 ? M2RNN_BF16 : M2RNN_F32);
  return with_split<sizeof(T) == 4 ? 2 : 4>(sp, [&](auto C, auto R, auto G, auto FULL) {
    auto kern = gated_norm_fwd_kernel<T, C(), R(), G(), FULL()>;
    constexpr int smem = Walk<T, C(), R(), G(), 2, FULL()>::kSmem;
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    (void)launch_early(kern, sp.grid, kThreads, smem, s, tokens, d, static_cast<const T *>(y), static_cast<const T *>(g), static_cast<const T *>(w), eps, silu_on,
                                         static_cast<T *>(out), rstd);
    return cudaGetLastError();
  });
}

template <typename T>
cudaError_t launch_bwd(long tokens, int d, const void *y, const void *g, const void *w, const float *rstd, int silu_on,
                       const void *dout, void *dy, void *dg, float *dw_part, cudaStream_t s) {
  const Split sp = split_of(tokens, d, true, sizeof(T) == 2 ? M2RNN_BF16 : M2RNN_F32);
  return with_split<sizeof(T) == 4 ? 4 : 0>(sp, [&](auto C, auto R, auto G, auto FULL) {
    auto kern = gated_norm_bwd_kernel<T, C(), R(), G(), FULL()>;
    constexpr int sums = 256 * C() * kWarps * 4;    // groups x the columns they can hold, at the end
    constexpr int smem = Walk<T, C(), R(), G(), 3, FULL()>::kSmem > sums ? Walk<T, C(), R(), G(), 3, FULL()>::kSmem : sums;
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    (void)launch_early(kern, sp.grid, kThreads, smem, s, tokens, d, static_cast<const T *>(y), static_cast<const T *>(g), static_cast<const T *>(w), rstd, silu_on,
                                         static_cast<const T *>(dout), static_cast<T *>(dy), static_cast<T *>(dg), dw_part);
    return cudaGetLastError();
  });
}

}  // namespace
}  // namespace m2rnn

using namespace m2rnn;

extern "C" {

int m2rnn_gated_norm_fwd(int64_t tokens, int32_t d, int32_t io_dtype, const void *y, const void *g_in, const void *w,
                         float eps, int32_t silu_on, void *out, float *rstd, void *stream) {
  const int rc = check((long)tokens, d, io_dtype);
  if (rc != M2RNN_OK) return rc;
  if (tokens == 0) return M2RNN_OK;   // nothing to read or write
  if (!y || !g_in || !w || !out) return M2RNN_ERR_NULL;
  if (!aligned16(y) || !aligned16(g_in) || !aligned16(w) || !aligned16(out)) return M2RNN_ERR_ALIGN;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const cudaError_t e = io_dtype == M2RNN_BF16 ? launch_fwd<__nv_bfloat16>((long)tokens, d, y, g_in, w, eps, silu_on, out, rstd, s)
                                               : launch_fwd<float>((long)tokens, d, y, g_in, w, eps, silu_on, out, rstd, s);
  if (e != cudaSuccess) (void)cudaGetLastError();   // leave the runtime's last-error slot clear
  return e == cudaSuccess ? M2RNN_OK : M2RNN_ERR_CUDA;
}

size_t m2rnn_gated_norm_bwd_workspace_bytes(int64_t tokens, int32_t d) {
  if (tokens <= 0 || d <= 0) return 0;
  return (size_t)kMaxCtas * (size_t)d * sizeof(float);   // an upper bound that does not depend on the dtype
}

int m2rnn_gated_norm_bwd(int64_t tokens, int32_t d, int32_t io_dtype, const void *y, const void *g_in, const void *w,
                         const float *rstd, int32_t silu_on, const void *dout, void *dy, void *dg_in, float *dw,
                         void *workspace, size_t workspace_bytes, void *stream) {
  const int rc = check((long)tokens, d, io_dtype);
  if (rc != M2RNN_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (tokens == 0) {   // an empty sum
    if (!dw) return M2RNN_ERR_NULL;
    return cudaMemsetAsync(dw, 0, (size_t)d * sizeof(float), s) == cudaSuccess ? M2RNN_OK : M2RNN_ERR_CUDA;
  }
  if (!y || !g_in || !w || !rstd || !dout || !dy || !dg_in || !dw) return M2RNN_ERR_NULL;
  if (!aligned16(y) || !aligned16(g_in) || !aligned16(w) || !aligned16(dout) || !aligned16(dy) || !aligned16(dg_in) || !aligned16(dw))
    return M2RNN_ERR_ALIGN;
  if (!workspace || workspace_bytes < m2rnn_gated_norm_bwd_workspace_bytes(tokens, d)) return M2RNN_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(workspace) & 255u) return M2RNN_ERR_ALIGN;
  float *part = static_cast<float *>(workspace);
  cudaError_t e = io_dtype == M2RNN_BF16 ? launch_bwd<__nv_bfloat16>((long)tokens, d, y, g_in, w, rstd, silu_on, dout, dy, dg_in, part, s)
                                         : launch_bwd<float>((long)tokens, d, y, g_in, w, rstd, silu_on, dout, dy, dg_in, part, s);
  if (e != cudaSuccess) { (void)cudaGetLastError(); return M2RNN_ERR_CUDA; }
  (void)launch_early(reduce_partials_kernel, (d + 31) / 32, 1024, 0, s, part, dw, split_of((long)tokens, d, true, io_dtype).grid, d);
  return cudaGetLastError() == cudaSuccess ? M2RNN_OK : M2RNN_ERR_CUDA;
}

}  // extern "C"
