// fp32 FMA path of the M2RNN scan (forward, decoding step, backward through time): the accuracy path
// (<= 1e-4).  Everything is fp32 FMA with tanhf / expf.
//
// The rows of a state are independent recurrences, so the unit of work is a group of eight rows, and
// the product of a step, [8 x V] times the V x V transition matrix, is laid out to keep the matrix in
// registers: lane (p, cg) of warp w holds the V/8 rows l of W that belong to part p for the two columns
// 8w + 2cg, +1.  Per state row it reads its V/8 entries of the row from shared memory (the four lanes of
// a part share them: one wavefront for a warp), multiplies, and leaves a partial sum per row and column;
// three rounds of recursive halving over p then leave every lane with the finished sums of ONE row, p,
// for its two columns -- the elements it owns for the element-wise part of the step.  One CTA barrier a
// step makes the new rows visible.  Sums over l pair even and odd entries (packed fp32x2 FMA).
// (Until then a CTA held a whole state and read W from shared memory for every product: 1 MB of
// shared-memory traffic a step and a sixteenth of the SMs at 16 units.  K = V = 64, 16 units, T = 512:
// forward 3.19 -> 0.37 ms, backward 18.6 -> 0.63 ms.  Since then the forward from V = 32 on and the backward of V = 64 have a cut of
// the product with fewer lanes to a column, below: 0.21 and 0.56 ms.)
#include "device_common.cuh"
#include "internal.h"

namespace m2rnn {
namespace {

constexpr int kRows = 8;      // rows of a group (forward and backward: or four, see rows_per_group)
constexpr int kSteps = 16;    // steps staged at a time, and steps of state the backward kernel keeps on chip

template <int V>
struct Geom {
  static constexpr int NW = V / 8;             // warps of a CTA
  static constexpr int kThreads = 32 * NW;
  static constexpr int HP = V + 8;             // row pitch: the eight rows of a group start 32 bytes apart
                                               // in the banks, so their 32-byte pieces are conflict-free
  static constexpr int NP = V / 16;            // pairs of l per thread
  static constexpr int kTile = kRows * HP;     // floats of a group of eight rows
};

// first l of pair i of part p: parts interleave in 16-byte (V = 16: 8-byte) pieces
template <int V>
__device__ __forceinline__ int pair_l(int i, int p) {
  return V == 16 ? 2 * p : 32 * (i >> 1) + 4 * p + 2 * (i & 1);
}

// this thread's part of W for the product rows x W: columns c0, c0 + 1
template <int V>
__device__ __forceinline__ void load_w(const float *__restrict__ W, int p, int c0, float2 (&w)[Geom<V>::NP][2]) {
#pragma unroll
  for (int i = 0; i < Geom<V>::NP; ++i) {
    const int l = pair_l<V>(i, p);
    const float2 a = *reinterpret_cast<const float2 *>(W + (size_t)l * V + c0), b = *reinterpret_cast<const float2 *>(W + (size_t)(l + 1) * V + c0);
    w[i][0] = make_float2(a.x, b.x);
    w[i][1] = make_float2(a.y, b.y);
  }
}
// ... for rows x W^T
template <int V>
__device__ __forceinline__ void load_wt(const float *__restrict__ W, int p, int c0, float2 (&w)[Geom<V>::NP][2]) {
#pragma unroll
  for (int i = 0; i < Geom<V>::NP; ++i) {
    const int j = pair_l<V>(i, p);
    w[i][0] = *reinterpret_cast<const float2 *>(W + (size_t)c0 * V + j);
    w[i][1] = *reinterpret_cast<const float2 *>(W + (size_t)(c0 + 1) * V + j);
  }
}

// What a lane owns of a group of R rows: E = R/4 adjacent columns of one row -- of eight rows row p, both
// columns; of four, row p/2, column p%2.
template <int R>
struct Own {
  static constexpr int E = R / 4;
  __device__ static int row(int p) { return R == 8 ? p : p >> 1; }
  __device__ static int col(int p, int c0) { return R == 8 ? c0 : c0 + (p & 1); }
};
template <int E> struct Vec { float x[E]; };
template <int E>
__device__ __forceinline__ Vec<E> get(const float *p) {
  Vec<E> v;
  if constexpr (E == 2) { const float2 t = *reinterpret_cast<const float2 *>(p); v.x[0] = t.x; v.x[1] = t.y; }
  else v.x[0] = *p;
  return v;
}
template <int E>
__device__ __forceinline__ void put(float *p, const Vec<E> &v) {
  if constexpr (E == 2) *reinterpret_cast<float2 *>(p) = make_float2(v.x[0], v.x[1]);
  else *p = v.x[0];
}

// R rows (pitch HP, shared memory) times the matrix held in w -> the lane's own elements
template <int V, int R>
__device__ __forceinline__ Vec<R / 4> product(const float *rows, const float2 (&w)[Geom<V>::NP][2], int p, int lane) {
  using G = Geom<V>;
  float s[R][2];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    float2 a0 = make_float2(0.f, 0.f), a1 = a0;
    const float *row = rows + r * G::HP;
    if constexpr (V == 16) {
      const float2 h = *reinterpret_cast<const float2 *>(row + 2 * p);
      a0 = __fmul2_rn(h, w[0][0]);
      a1 = __fmul2_rn(h, w[0][1]);
    } else {
#pragma unroll
      for (int i = 0; i < V / 32; ++i) {
        const float4 h = *reinterpret_cast<const float4 *>(row + 32 * i + 4 * p);
        a0 = __ffma2_rn(make_float2(h.x, h.y), w[2 * i][0], a0);
        a1 = __ffma2_rn(make_float2(h.x, h.y), w[2 * i][1], a1);
        a0 = __ffma2_rn(make_float2(h.z, h.w), w[2 * i + 1][0], a0);
        a1 = __ffma2_rn(make_float2(h.z, h.w), w[2 * i + 1][1], a1);
      }
    }
    s[r][0] = a0.x + a0.y;
    s[r][1] = a1.x + a1.y;
  }
  // recursive halving over the parts (lane bits 4, 3, 2), rows first, then (four rows) columns
#pragma unroll
  for (int m = R / 2, bit = 16; m >= 1; m >>= 1, bit >>= 1) {
    const bool up = lane & bit;
#pragma unroll
    for (int r = 0; r < m; ++r)
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const float send = up ? s[r][x] : s[r + m][x], keep = up ? s[r + m][x] : s[r][x];
        s[r][x] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
      }
  }
  Vec<R / 4> o;
  if constexpr (R == 8) {
    o.x[0] = s[0][0]; o.x[1] = s[0][1];
  } else {
    const bool up = lane & 4;
    o.x[0] = (up ? s[0][1] : s[0][0]) + __shfl_xor_sync(0xffffffffu, up ? s[0][0] : s[0][1], 4);
  }
  return o;
}

__device__ __forceinline__ void cp16(float *dst, const float *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp4(float *dst, const float *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// [len][width] floats (width a multiple of 4) from rows `stride` apart, into dense rows, by the CTA
__device__ __forceinline__ void stage_rows(float *dst, const float *src, long long stride, int len, int width, int tid, int nthreads) {
  const int w4 = width >> 2;
  for (int x = tid; x < len * w4; x += nthreads) {
    const int t = x / w4, j = (x - t * w4) * 4;
    cp16(dst + t * width + j, src + t * stride + j);
  }
}

// The readout (Eq. 3) adds shares of four rows, in the order of the rows, whatever the group size: a scan in
// groups of four, one in groups of eight and a decoding step agree bit for bit.  Column of y that a lane holds:
template <int R> __device__ __forceinline__ int y_col(int lane, int c0) { return R == 8 ? c0 + ((lane >> 3) & 1) : c0 + ((lane >> 2) & 1); }
template <int R> __device__ __forceinline__ bool y_owner(int lane) { return R == 8 ? (lane & 20) == 0 : (lane & 24) == 0; }
// y (of this lane's column) plus the group's shares; first: y is wr v of that column, to be added to the first share
template <int R>
__device__ __forceinline__ float readout(float y, bool first, float wr, float v, float q, const Vec<R / 4> &h, int lane) {
  float t;
  if constexpr (R == 8) {   // rows p: bits 8 and 4 of the lane inside a half, bit 16 the half
    const bool up = lane & 8;
    const float a = __fmul_rn(q, h.x[0]), b = __fmul_rn(q, h.x[1]);
    t = (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, 8);
    t += __shfl_xor_sync(0xffffffffu, t, 4);
  } else {                  // rows p / 2: bits 16 and 8
    t = __fmul_rn(q, h.x[0]);
    t += __shfl_xor_sync(0xffffffffu, t, 16);
    t += __shfl_xor_sync(0xffffffffu, t, 8);
  }
  y = first ? fmaf(wr, v, t) : y + t;
  if constexpr (R == 8) y += __shfl_xor_sync(0xffffffffu, t, 16);   // (lanes of the first half, which own y)
  return y;
}

// Eq. 1 and 2 for the lane's elements of a row (roundings spelled out: a decoding step repeats a step of the
// scan bit for bit)
template <int E>
__device__ __forceinline__ Vec<E> update(const Vec<E> &o, float k, const Vec<E> &v, float f, const Vec<E> &h, Vec<E> &z) {
  Vec<E> r;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    z.x[e] = tanhf(fmaf(k, v.x[e], o.x[e]));
    r.x[e] = fmaf(1.f - f, z.x[e], __fmul_rn(f, h.x[e]));
  }
  return r;
}

// ------------------------------------------------------------------ forward (Algorithm 1)
// One CTA per (b, n, slab of R = 8 ng rows); the groups of a slab take turns inside a step.
template <int V>
__host__ __device__ constexpr int fwd_stage_floats(int R) { return kSteps * (2 * R + V + 1); }
template <int V>
__host__ size_t fwd_f32_smem(int R) { return sizeof(float) * (2 * (size_t)R * Geom<V>::HP + 2 * (size_t)fwd_stage_floats<V>(R) + 2 * kSteps); }

// GR: rows of a group
template <int V, int GR>
__global__ void __launch_bounds__(Geom<V>::kThreads) fwd_f32_kernel(ScanArgs a) {
  using G = Geom<V>;
  constexpr int E = GR / 4;
  constexpr int kTile = GR * G::HP;
  extern __shared__ __align__(16) float smem[];
  begin_dependent();
  const int K = a.K, N = a.N, R = a.KCf, RS = K / R, ng = R / GR;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, p = lane >> 2, c0 = 8 * warp + 2 * (lane & 3);
  const int orow = Own<GR>::row(p), ocol = Own<GR>::col(p, c0), ycol = y_col<GR>(lane, c0);
  const int place = blockIdx.x / RS, rs = blockIdx.x % RS, rbase = rs * R;
  const int b = batch_entry(a, place / N, smem), n = place % N, bn = b * N + n;
  const UnitSpan span = unit_span(a, b);   // this batch entry's tokens (a slice of a packed batch, or b T ..)
  const int T = span.T;
  const size_t tok0 = span.tok0, KV = (size_t)K * V;
  const int hq = n / (N / a.Nq), hk = n / (N / a.Nk);

  float *H0 = smem, *H1 = H0 + R * G::HP;                    // the state before and after a step
  float *stages = H1 + R * G::HP;                             // two stages: q, k [16][R], v [16][V], gate [16]
  float *fS = stages + 2 * fwd_stage_floats<V>(R);            // [2][16] evaluated gates

  float2 w[G::NP][2];
  load_w<V>(static_cast<const float *>(a.W) + (size_t)n * V * V, p, c0, w);
  for (int g = 0; g < ng; ++g) {
    const int row = GR * g + orow;
    put<E>(H0 + row * G::HP + ocol, a.h0 ? get<E>(a.h0 + bn * KV + (size_t)(rbase + row) * V + ocol) : Vec<E>{});
  }
  const float al = a.alpha ? a.alpha[n] : 1.f, be = a.beta ? a.beta[n] : 0.f;
  const float *qg = static_cast<const float *>(a.q), *kg = static_cast<const float *>(a.k);
  const float *vg = static_cast<const float *>(a.v), *wr = static_cast<const float *>(a.w_r);
  const bool want_y = a.y != nullptr;
  float *yg = a.y_part ? a.y_part + (size_t)rs * a.TT * N * V : static_cast<float *>(a.y);
  const float wre = wr && rs == 0 ? wr[(size_t)n * V + ycol] : 0.f;

  auto stage = [&](int x) { return stages + (x & 1) * fwd_stage_floats<V>(R); };
  auto fetch = [&](int ch) {
    float *st = stage(ch);
    const int t0 = ch * kSteps, len = min(kSteps, T - t0);
    const size_t bt = tok0 + t0;
    if (want_y) stage_rows(st, qg + bt * a.qs + hq * K + rbase, a.qs, len, R, tid, G::kThreads);
    stage_rows(st + kSteps * R, kg + bt * a.ks + hk * K + rbase, a.ks, len, R, tid, G::kThreads);
    stage_rows(st + 2 * kSteps * R, vg + bt * a.vs + n * V, a.vs, len, V, tid, G::kThreads);
    if (tid < len) cp4(st + kSteps * (2 * R + V) + tid, a.gate + (bt + tid) * N + n);
    cp_commit();
  };
  auto gates = [&](int ch) {   // the thread that copied a gate evaluates it
    if (tid < min(kSteps, T - ch * kSteps)) fS[(ch & 1) * kSteps + tid] = gate_value(a.gate_kind, stage(ch)[kSteps * (2 * R + V) + tid], al, be, nullptr);
  };
  const int nst = (T + kSteps - 1) / kSteps;
  if (nst > 0) {
    fetch(0);
    cp_wait<0>();
    gates(0);
  }
  __syncthreads();
  int ck_left = 0, ck_idx = 0;
  for (int ch = 0; ch < nst; ++ch) {
    if (ch + 1 < nst) fetch(ch + 1);
    const float *qS = stage(ch), *kS = qS + kSteps * R, *vS = kS + kSteps * R, *fs = fS + (ch & 1) * kSteps;
    const int len = min(kSteps, T - ch * kSteps);
    for (int s = 0; s < len; ++s) {
      if (a.ckpt) {
        if (ck_left == 0) {
          float *dst = a.ckpt + ((size_t)bn * a.nchunks + ck_idx) * KV + (size_t)rbase * V;
          for (int g = 0; g < ng; ++g)
            put<E>(dst + (size_t)(GR * g + orow) * V + ocol, get<E>(H0 + (GR * g + orow) * G::HP + ocol));
          ++ck_idx;
          ck_left = a.C;
        }
        --ck_left;
      }
      const float f = fs[s];
      const Vec<E> v = get<E>(vS + s * V + ocol);
      const float vy = vS[s * V + ycol];
      float y = 0.f;     // Eq. 3, group by group (the order in which the shares of single groups are added too)
      for (int g = 0; g < ng; ++g) {
        const Vec<E> o = product<V, GR>(H0 + g * kTile, w, p, lane);
        const int row = GR * g + orow;
        Vec<E> z;
        const Vec<E> h = update<E>(o, kS[s * R + row], v, f, get<E>(H0 + row * G::HP + ocol), z);
        put<E>(H1 + row * G::HP + ocol, h);
        if (want_y) y = readout<GR>(y, g == 0, wre, vy, qS[s * R + row], h, lane);
      }
      __syncthreads();   // H_t is complete, H_{t-1} is free
      if (want_y && y_owner<GR>(lane)) yg[((tok0 + ch * kSteps + s) * N + n) * V + ycol] = y;
      float *t = H0; H0 = H1; H1 = t;
    }
    if (ch + 1 < nst) {
      cp_wait<0>();
      gates(ch + 1);
      __syncthreads();
    }
  }
  if (a.hT)
    for (int g = 0; g < ng; ++g)
      put<E>(a.hT + bn * KV + (size_t)(rbase + GR * g + orow) * V + ocol, get<E>(H0 + (GR * g + orow) * G::HP + ocol));
}

// ------------------------------------------------------------------ forward, V >= 32, few rows at a time
// The same step with the product cut the other way: a warp takes R rows of a group of four and, up to V = 64, all of their
// columns (V = 128: a quarter), so that up to V = 64 nothing but the warp itself waits for a step.  Lane (q, cg) holds 8 / P of
// the eight parts of l for CP columns, V CP / P entries of W, 128 registers at V >= 64.  What held the kernel above were
// the shuffles that add eight lanes' shares of every product (345 us for 512 steps of 16 units, K = V = 64; 218 without
// them) and the shared memory's bandwidth; here seven eighths of that sum are inside the lane, in the order of the shuffles, so that the
// two kernels and the decoding step agree bit for bit.
template <int V>
struct Wide {
  static constexpr int CP = V == 32 ? 2 : 4, P = V == 128 ? 4 : 2;      // columns of a lane; lanes that share a column
  static constexpr int CW = 32 / P * CP, NWR = V / CW;                  // columns of a warp; warps of a row
  static constexpr int E = CP / P, M = 8 / P, NB = V / 32;              // columns that a lane owns; its parts of l; pieces of a part
  static constexpr int HP = V + 4;
  // the l of piece x of part m of lane part q: 4 from 32 x + 4 (q + P m)
  __device__ static int l_of(int q, int m, int x) { return 32 * x + 4 * (q + P * m); }
};
template <int V>
__device__ __forceinline__ void wide_load_w(const float *__restrict__ W, int q, int c0, float2 (&w)[Wide<V>::M][2 * Wide<V>::NB][Wide<V>::CP]) {
  using G = Wide<V>;
#pragma unroll
  for (int m = 0; m < G::M; ++m)
#pragma unroll
    for (int x = 0; x < 2 * G::NB; ++x) {
      const float *src = W + (size_t)(G::l_of(q, m, x >> 1) + 2 * (x & 1)) * V + c0;
#pragma unroll
      for (int e = 0; e < G::CP; ++e) w[m][x][e] = make_float2(src[e], src[V + e]);
    }
}
template <int V>
__device__ __forceinline__ void wide_load_wt(const float *__restrict__ W, int q, int c0, float2 (&w)[Wide<V>::M][2 * Wide<V>::NB][Wide<V>::CP]) {
  using G = Wide<V>;
#pragma unroll
  for (int m = 0; m < G::M; ++m)
#pragma unroll
    for (int x = 0; x < 2 * G::NB; ++x)
#pragma unroll
      for (int e = 0; e < G::CP; ++e) w[m][x][e] = *reinterpret_cast<const float2 *>(W + (size_t)(c0 + e) * V + G::l_of(q, m, x >> 1) + 2 * (x & 1));
}
// a warp's fragments to shared memory and back: 16 bytes a lane at a time
template <int V>
__device__ __forceinline__ void frags_out(float *dst, int lane, const float2 (&w)[Wide<V>::M][2 * Wide<V>::NB][Wide<V>::CP]) {
  using G = Wide<V>;
#pragma unroll
  for (int m = 0; m < G::M; ++m)
#pragma unroll
    for (int x = 0; x < 2 * G::NB; ++x)
#pragma unroll
      for (int e = 0; e < G::CP; e += 2)
        *reinterpret_cast<float4 *>(dst + (((m * 2 * G::NB + x) * (G::CP / 2) + e / 2) * 32 + lane) * 4) = make_float4(w[m][x][e].x, w[m][x][e].y, w[m][x][e + 1].x, w[m][x][e + 1].y);
}
template <int V>
__device__ __forceinline__ void frags_in(const float *src, int lane, float2 (&w)[Wide<V>::M][2 * Wide<V>::NB][Wide<V>::CP]) {
  using G = Wide<V>;
#pragma unroll
  for (int m = 0; m < G::M; ++m)
#pragma unroll
    for (int x = 0; x < 2 * G::NB; ++x)
#pragma unroll
      for (int e = 0; e < G::CP; e += 2) {
        const float4 t = *reinterpret_cast<const float4 *>(src + (((m * 2 * G::NB + x) * (G::CP / 2) + e / 2) * 32 + lane) * 4);
        w[m][x][e] = make_float2(t.x, t.y); w[m][x][e + 1] = make_float2(t.z, t.w);
      }
}
// R rows, `pitch` floats apart, times the matrix held in w: o[r][e], column c0 + E q + e of row r
template <int V, int R>
__device__ __forceinline__ void wide_product(const float *rows, int pitch, const float2 (&w)[Wide<V>::M][2 * Wide<V>::NB][Wide<V>::CP], int q, int lane,
                                             float (&o)[R][Wide<V>::E]) {
  using G = Wide<V>;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    float u[G::M][G::CP];
#pragma unroll
    for (int m = 0; m < G::M; ++m) {
      float2 acc[G::CP];
#pragma unroll
      for (int e = 0; e < G::CP; ++e) acc[e] = make_float2(0.f, 0.f);
#pragma unroll
      for (int x = 0; x < G::NB; ++x) {
        const float4 h = *reinterpret_cast<const float4 *>(rows + r * pitch + G::l_of(q, m, x));
#pragma unroll
        for (int e = 0; e < G::CP; ++e) {
          acc[e] = __ffma2_rn(make_float2(h.x, h.y), w[m][2 * x][e], acc[e]);
          acc[e] = __ffma2_rn(make_float2(h.z, h.w), w[m][2 * x + 1][e], acc[e]);
        }
      }
#pragma unroll
      for (int e = 0; e < G::CP; ++e) u[m][e] = acc[e].x + acc[e].y;
    }
    // parts p and p ^ 4, then p ^ 2, then p ^ 1: those of a lane are q + P m
#pragma unroll
    for (int h = G::M / 2; h >= 1; h >>= 1)
#pragma unroll
      for (int m = 0; m < h; ++m)
#pragma unroll
        for (int e = 0; e < G::CP; ++e) u[m][e] += u[m + h][e];
    float t[G::CP];
#pragma unroll
    for (int e = 0; e < G::CP; ++e) t[e] = u[0][e];
#pragma unroll
    for (int n = G::CP / 2, bit = 16, qb = G::P / 2; qb >= 1; n >>= 1, bit >>= 1, qb >>= 1) {      // (lane bit 16: the higher bit of q)
      const bool up = lane & bit;
#pragma unroll
      for (int e = 0; e < n; ++e) {
        const float send = up ? t[e] : t[e + n], keep = up ? t[e + n] : t[e];
        t[e] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
      }
    }
#pragma unroll
    for (int e = 0; e < G::E; ++e) o[r][e] = t[e];
  }
}

// One CTA per (b, n, group of four rows): 4 / R row sets of NWR warps; set i takes rows i, i + 4 / R, ..
template <int V, int R>
struct WideFwd {
  using G = Wide<V>;
  static constexpr int kSets = 4 / R, kThreads = 32 * G::NWR * kSets;
  static constexpr int kStage = kSteps * (2 * 4 + V + 1 + 3);      // q, k [16][4], v [16][V], gate [16] (+ alignment)
  static constexpr int kFloats = 2 * 4 * G::HP + 2 * kStage + 2 * kSteps + kSteps * kSets * V;
};
template <int V, int R>
__global__ void __launch_bounds__(WideFwd<V, R>::kThreads) fwd_f32_wide_kernel(ScanArgs a) {
  using G = Wide<V>;
  using WF = WideFwd<V, R>;
  constexpr int kSets = WF::kSets, E = G::E;
  extern __shared__ __align__(16) float smem[];
  begin_dependent();
  const int K = a.K, N = a.N, RS = K / 4;
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), set = warp / G::NWR;
  const int q = lane / (32 / G::P), c0 = (warp % G::NWR) * G::CW + G::CP * (lane % (32 / G::P)), col = c0 + E * q;
  const int place = blockIdx.x / RS, rs = blockIdx.x % RS, rbase = rs * 4;
  const int b = batch_entry(a, place / N, smem), n = place % N, bn = b * N + n;
  const UnitSpan span = unit_span(a, b);   // this batch entry's tokens (a slice of a packed batch, or b T ..)
  const int T = span.T;
  const size_t tok0 = span.tok0, KV = (size_t)K * V;
  const int hq = n / (N / a.Nq), hk = n / (N / a.Nk);

  float *H0 = smem + set * G::HP, *H1 = H0 + 4 * G::HP;       // this set's rows before and after a step, kSets HP apart
  float *stages = smem + 8 * G::HP, *fS = stages + 2 * WF::kStage, *yS = fS + 2 * kSteps;      // [16][sets][V] shares of y

  float2 w[G::M][2 * G::NB][G::CP];
  wide_load_w<V>(static_cast<const float *>(a.W) + (size_t)n * V * V, q, c0, w);
  const size_t own = (size_t)(rbase + set) * V + col;      // (row i of the set: i kSets V further)
  float H[R][E];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const Vec<E> h = a.h0 ? get<E>(a.h0 + bn * KV + own + (size_t)r * kSets * V) : Vec<E>{};
#pragma unroll
    for (int e = 0; e < E; ++e) H[r][e] = h.x[e];
    put<E>(H0 + r * kSets * G::HP + col, h);
  }
  auto store_state = [&](float *dst) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      Vec<E> h;
#pragma unroll
      for (int e = 0; e < E; ++e) h.x[e] = H[r][e];
      put<E>(dst + own + (size_t)r * kSets * V, h);
    }
  };
  const float al = a.alpha ? a.alpha[n] : 1.f, be = a.beta ? a.beta[n] : 0.f;
  const float *qg = static_cast<const float *>(a.q), *kg = static_cast<const float *>(a.k);
  const float *vg = static_cast<const float *>(a.v), *wr = rs == 0 ? static_cast<const float *>(a.w_r) : nullptr;
  const bool want_y = a.y != nullptr;
  float *yg = a.y_part ? a.y_part + (size_t)rs * a.TT * N * V : static_cast<float *>(a.y);

  auto stage = [&](int x) { return stages + (x & 1) * WF::kStage; };
  constexpr int oK = 4 * kSteps, oV = 8 * kSteps, oG = oV + kSteps * V;
  auto fetch = [&](int ch) {
    float *st = stage(ch);
    const int t0 = ch * kSteps, len = min(kSteps, T - t0);
    const size_t bt = tok0 + t0;
    if (want_y) stage_rows(st, qg + bt * a.qs + hq * K + rbase, a.qs, len, 4, tid, WF::kThreads);
    stage_rows(st + oK, kg + bt * a.ks + hk * K + rbase, a.ks, len, 4, tid, WF::kThreads);
    stage_rows(st + oV, vg + bt * a.vs + n * V, a.vs, len, V, tid, WF::kThreads);
    if (tid < len) cp4(st + oG + tid, a.gate + (bt + tid) * N + n);
    cp_commit();
  };
  auto gates = [&](int ch) {   // the thread that copied a gate evaluates it
    if (tid < min(kSteps, T - ch * kSteps)) fS[(ch & 1) * kSteps + tid] = gate_value(a.gate_kind, stage(ch)[oG + tid], al, be, nullptr);
  };
  auto row_sync = [&]() {      // the warps of a set have left their columns
    if constexpr (G::NWR == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + set), "n"(32 * G::NWR) : "memory");
  };
  const int nst = (T + kSteps - 1) / kSteps;
  if (nst > 0) {
    fetch(0);
    cp_wait<0>();
    gates(0);
  }
  __syncthreads();
  int ck_left = 0;
  float *ck = a.ckpt ? a.ckpt + (size_t)bn * a.nchunks * KV : nullptr;
  for (int ch = 0; ch < nst; ++ch) {
    if (ch + 1 < nst) fetch(ch + 1);
    const float *st = stage(ch), *fs = fS + (ch & 1) * kSteps;
    const int len = min(kSteps, T - ch * kSteps);
    for (int s = 0; s < len; ++s) {
      if (ck) {
        if (ck_left == 0) { store_state(ck); ck += KV; ck_left = a.C; }
        --ck_left;
      }
      float o[R][E], kk[R], qq[R];
      const float f = fs[s];
      const Vec<E> v = get<E>(st + oV + s * V + col);
#pragma unroll
      for (int r = 0; r < R; ++r) { kk[r] = st[oK + 4 * s + set + r * kSets]; qq[r] = st[4 * s + set + r * kSets]; }
      wide_product<V, R>(H0, kSets * G::HP, w, q, lane, o);
      Vec<E> qh[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        Vec<E> ov, hv, z;
#pragma unroll
        for (int e = 0; e < E; ++e) { ov.x[e] = o[r][e]; hv.x[e] = H[r][e]; }
        const Vec<E> h = update<E>(ov, kk[r], v, f, hv, z);
        put<E>(H1 + r * kSets * G::HP + col, h);
#pragma unroll
        for (int e = 0; e < E; ++e) {
          H[r][e] = h.x[e];
          qh[r].x[e] = __fmul_rn(qq[r], h.x[e]);
        }
      }
      // (rows 0 and 2, 1 and 3, then both; R = 1: all of that when the stage is done)
#pragma unroll
      for (int h = R / 2; h >= 1; h >>= 1)
#pragma unroll
        for (int r = 0; r < h; ++r)
#pragma unroll
          for (int e = 0; e < E; ++e) qh[r].x[e] += qh[r + h].x[e];
      put<E>(yS + (s * kSets + set) * V + col, qh[0]);
      row_sync();
      float *x = H0; H0 = H1; H1 = x;
    }
    if (ch + 1 < nst) { cp_wait<0>(); gates(ch + 1); }
    __syncthreads();          // the next stage is in, this one's shares of y are
    // Eq. 3: the sets' shares, in the same order
    if (want_y)
      for (int x = tid; x < len * (V / 4); x += WF::kThreads) {
        const int s = x / (V / 4), j = 4 * (x % (V / 4));
        float4 y4 = *reinterpret_cast<const float4 *>(yS + s * kSets * V + j);
        auto add = [](float4 &p, const float4 &r) { p.x += r.x; p.y += r.y; p.z += r.z; p.w += r.w; };
        if constexpr (kSets == 2) add(y4, *reinterpret_cast<const float4 *>(yS + (s * kSets + 1) * V + j));
        if constexpr (kSets == 4) {
          float4 o4 = *reinterpret_cast<const float4 *>(yS + (s * kSets + 1) * V + j);
          add(y4, *reinterpret_cast<const float4 *>(yS + (s * kSets + 2) * V + j));
          add(o4, *reinterpret_cast<const float4 *>(yS + (s * kSets + 3) * V + j));
          add(y4, o4);
        }
        float4 w4 = make_float4(0.f, 0.f, 0.f, 0.f), v4 = w4;
        if (wr) { w4 = *reinterpret_cast<const float4 *>(wr + (size_t)n * V + j); v4 = *reinterpret_cast<const float4 *>(st + oV + s * V + j); }
        y4.x = fmaf(w4.x, v4.x, y4.x); y4.y = fmaf(w4.y, v4.y, y4.y); y4.z = fmaf(w4.z, v4.z, y4.z); y4.w = fmaf(w4.w, v4.w, y4.w);
        *reinterpret_cast<float4 *>(yg + ((tok0 + ch * kSteps + s) * N + n) * V + j) = y4;
      }
    __syncthreads();          // (the shares' place, and this stage's, are taken again)
  }
  if (a.hT) store_state(a.hT + bn * KV);
}

// ------------------------------------------------------------------ backward (Algorithm 2)
// One CTA per (b, n, group of eight rows).  Time goes backwards in pieces of up to 16 steps; of a piece
// the CTA (A) redoes the forward steps, keeping H_{t-1} and Z_t of every step in shared memory,
// (B) walks them backwards -- G = C + q dy^T, dX, C <- f G + dX W^T, dX in Z's place --, and (C) takes
// everything that is a sum over steps or rows from those two arrays at once: dW += H_{t-1}^T dX as a
// register-tiled product over the piece's 8 x 16 rows, dq, dk, dv, dgate.  Only (A) and (B) are serial,
// with one barrier a step.  A checkpoint interval above 16 first walks the chunk forward once and
// leaves the states between pieces in the scratch tensor.
// slab0 / nslab: the groups of rows this launch takes.  All of them (nslab = K/8), each leaving its
// shares of dv, dgate and dW as partials; or one after the other (nslab = 1), the later ones
// adding to what the earlier ones wrote.
// WIDE (V = 64, groups of four): the products as in the kernel above, a row a warp; the fragments of W and W^T, 128 registers each,
// lie in shared memory and are taken from there once per piece and direction.
template <int V, int GR, bool WIDE>
struct BwdGeom {
  using G = Geom<V>;
  static constexpr int kThreads = WIDE ? 32 * GR : G::kThreads;
  static constexpr int kWideFloats = WIDE ? 2 * V * V : 0;
  static_assert(!WIDE || (V == 64 && GR == 4), "the fragments of a warp that has all columns of a row");
  static constexpr int kTile = GR * G::HP;
  static constexpr int kStage = kSteps * (2 * GR + 2 * V + 1);        // q, k [16][GR], v, dy [16][V], gate [16]
  // dW tiles: 4 x JT elements per thread; with fewer tiles than threads, SP threads share a tile and
  // take every SP-th step
  static constexpr int JT = V == 128 || WIDE ? 8 : 4;
  static constexpr int kTiles = (V / 4) * (V / JT), SP = kThreads / kTiles;
  static_assert(SP >= 1, "a tile a thread");
  static constexpr int kFloats = (2 * kSteps + 1) * kTile + 2 * kStage + 4 * kSteps + kSteps * kThreads + kWideFloats;
  // W and W^T both stay in registers where they fit beside the dW tile; at V = 128 (32 + 32 + 32 of 128
  // registers) each phase reloads its own from L2 once per piece
  static constexpr bool kReload = V == 128;
};

template <int V, int GR, bool WIDE>
__global__ void __launch_bounds__(BwdGeom<V, GR, WIDE>::kThreads, WIDE ? 2 : 512 / Geom<V>::kThreads) bwd_f32_kernel(ScanArgs a, int slab0, int nslab) {
  using G = Geom<V>;
  using BG = BwdGeom<V, GR, WIDE>;
  using WG = Wide<64>;      // (of the wide form)
  constexpr int E = WIDE ? WG::E : GR / 4, kThreads = BG::kThreads;
  extern __shared__ __align__(16) float smem[];
  begin_dependent();
  const int K = a.K, N = a.N;
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int p = WIDE ? lane / (32 / WG::P) : lane >> 2, c0 = WIDE ? WG::CP * (lane % (32 / WG::P)) : 8 * warp + 2 * (lane & 3);
  const int place = blockIdx.x / nslab, rs = slab0 + blockIdx.x % nslab, rbase = rs * GR;
  const int b = batch_entry(a, place / N, smem), n = place % N, bn = b * N + n;
  const bool add = nslab == 1 && rs > 0;   // earlier launches have written dv, dgate and dW
  const UnitSpan span = unit_span(a, b);
  const int T = span.T;
  const size_t tok0 = span.tok0, KV = (size_t)K * V;
  const int hq = n / (N / a.Nq), hk = n / (N / a.Nk);

  float *Hc = smem;                               // [17][GR][HP]: H before step s of the piece; [len] the last H_t
  float *Xc = Hc + (kSteps + 1) * BG::kTile;       // [16][GR][HP]: Z_t, then dX_t
  float *stages = Xc + kSteps * BG::kTile;
  float *fS = stages + 2 * BG::kStage, *dfS = fS + 2 * kSteps;   // [2][16] gates and their slopes
  float *dfp = dfS + 2 * kSteps;                  // [16][threads] shares of df

  const float *Wn = static_cast<const float *>(a.W) + (size_t)n * V * V;
  float *wS = dfp + kSteps * kThreads;            // the fragments of W and W^T, 16 bytes a lane at a time
  float2 w[WIDE ? 1 : G::NP][2], wt[WIDE || BG::kReload ? 1 : G::NP][2];
  float2 ww[WIDE ? WG::M : 1][2 * WG::NB][WG::CP];
  if constexpr (WIDE) {
    wide_load_w<V>(Wn, p, c0, ww);
    if (warp == 0) frags_out<V>(wS, lane, ww);
    wide_load_wt<V>(Wn, p, c0, ww);
    if (warp == 0) frags_out<V>(wS + V * V, lane, ww);
  } else if constexpr (!BG::kReload) {
    load_w<V>(Wn, p, c0, w);
    load_wt<V>(Wn, p, c0, wt);
  }
  const float al = a.alpha ? a.alpha[n] : 1.f, be = a.beta ? a.beta[n] : 0.f;
  const float *qg = static_cast<const float *>(a.q), *kg = static_cast<const float *>(a.k);
  const float *vg = static_cast<const float *>(a.v), *wr = static_cast<const float *>(a.w_r);
  const float *dyg = static_cast<const float *>(a.dy);
  const int orow = WIDE ? warp : Own<GR>::row(p), ocol = WIDE ? c0 + E * p : Own<GR>::col(p, c0);
  const int own = orow * G::HP + ocol;            // this thread's elements inside a group of rows
  const size_t own_g = (size_t)(rbase + orow) * V + ocol;   // ... inside a state in memory

  // pieces: chunk ch (the checkpoint interval) holds ceil(len / 16) of them
  const int ppc = (a.C + kSteps - 1) / kSteps, nch = (T + a.C - 1) / a.C;
  struct Piece { int t0, len; };
  auto piece = [&](int ch, int i) {
    const int t0 = ch * a.C + i * kSteps;
    return Piece{t0, max(0, min(min(kSteps, a.C - i * kSteps), T - t0))};
  };
  auto stage = [&](int x) { return stages + (x & 1) * BG::kStage; };
  constexpr int oK = kSteps * GR, oV = 2 * oK, oDY = oV + kSteps * V, oG = oDY + kSteps * V;
  auto fetch = [&](int x, Piece pc) {
    float *st = stage(x);
    const size_t bt = tok0 + pc.t0;
    stage_rows(st, qg + bt * a.qs + hq * K + rbase, a.qs, pc.len, GR, tid, kThreads);
    stage_rows(st + oK, kg + bt * a.ks + hk * K + rbase, a.ks, pc.len, GR, tid, kThreads);
    stage_rows(st + oV, vg + bt * a.vs + n * V, a.vs, pc.len, V, tid, kThreads);
    stage_rows(st + oDY, dyg + (bt * N + n) * V, (long long)N * V, pc.len, V, tid, kThreads);
    if (tid < pc.len) cp4(st + oG + tid, a.gate + (bt + tid) * N + n);
    cp_commit();
  };
  auto gates = [&](int x, Piece pc) {
    if (tid < pc.len) fS[(x & 1) * kSteps + tid] = gate_value(a.gate_kind, stage(x)[oG + tid], al, be, &dfS[(x & 1) * kSteps + tid]);
  };
  float *scratch = a.chunk_states + (size_t)bn * ppc * KV;   // states at the start of a chunk's pieces

  Vec<E> C = a.d_hT ? get<E>(a.d_hT + (size_t)bn * KV + own_g) : Vec<E>{};   // carried dL/dH_t
  // the group's rows at `rows` times W or W^T, this thread's elements of it
  auto mul = [&](const float *rows, bool transposed) {
    if constexpr (WIDE) {
      float t[1][E];
      Vec<E> o;
      wide_product<V, 1>(rows + warp * G::HP, 0, ww, p, lane, t);
#pragma unroll
      for (int e = 0; e < E; ++e) o.x[e] = t[0][e];
      return o;
    } else if constexpr (BG::kReload) {
      return product<V, GR>(rows, w, p, lane);
    } else {
      return transposed ? product<V, GR>(rows, wt, p, lane) : product<V, GR>(rows, w, p, lane);
    }
  };
  // the rows of a step are written (wide: the warp's own is all that its next product needs)
  auto row_sync = [&]() {
    if constexpr (WIDE) __syncwarp();
    else __syncthreads();
  };
  float2 dW[4][BG::JT / 2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < BG::JT / 2; ++j) dW[i][j] = make_float2(0.f, 0.f);
  // (a warp's tiles are four by eight, so that its loads of H and dX are one wavefront each)
  constexpr int WJ = V > 32 ? (BG::JT == 8 ? V / 2 : V) / 32 : 1;
  const int tile = tid % BG::kTiles, tsp = tid / BG::kTiles, tw = tile >> 5;
  const int tl = 4 * (V == 16 ? (tile >> 2) : 4 * (tw / WJ) + (lane >> 3)), tj = 4 * (V == 16 ? (tile & 3) : 8 * (tw % WJ) + (lane & 7));

  // forward steps of a piece from the state in Hc[0]
  auto forward = [&](int x, int len) {
    const float *st = stage(x), *fs = fS + (x & 1) * kSteps;
    for (int s = 0; s < len; ++s) {
      float *hs = Hc + s * BG::kTile;
      const Vec<E> o = mul(hs, false);
      Vec<E> z;
      const Vec<E> h = update<E>(o, st[oK + s * GR + orow], get<E>(st + oV + s * V + ocol), fs[s], get<E>(hs + own), z);
      put<E>(hs + BG::kTile + own, h);
      put<E>(Xc + s * BG::kTile + own, z);
      row_sync();
    }
  };

  int x = 0;   // piece counter: picks the stage
  bool fetched = false;
  for (int ch = nch - 1; ch >= 0; --ch) {
    int np = (min(a.C, T - ch * a.C) + kSteps - 1) / kSteps;
    const float *ck = a.ckpt + ((size_t)bn * a.nchunks + ch) * KV + own_g;
    if (np > 1) {   // walk the chunk forward once, leaving the states between its pieces
      if constexpr (BG::kReload) load_w<V>(Wn, p, c0, w);
      __syncthreads();   // the piece before is done with every array
      if constexpr (WIDE) frags_in<V>(wS, lane, ww);
      Vec<E> h = get<E>(ck);
      for (int i = 0; i + 1 < np; ++i, ++x) {
        const Piece pc = piece(ch, i);
        put<E>(Hc + own, h);
        fetch(x, pc);
        cp_wait<0>();
        gates(x, pc);
        __syncthreads();
        forward(x, pc.len);
        h = get<E>(Hc + pc.len * BG::kTile + own);
        put<E>(scratch + (size_t)(i + 1) * KV + own_g, h);
        __syncthreads();
      }
      fetched = false;
    }
    for (int i = np - 1; i >= 0; --i, ++x) {
      const Piece pc = piece(ch, i);
      if (!fetched) fetch(x, pc);
      const Vec<E> h0 = get<E>(i > 0 ? scratch + (size_t)i * KV + own_g : ck);
      if constexpr (BG::kReload) load_w<V>(Wn, p, c0, w);
      cp_wait<0>();
      gates(x, pc);
      __syncthreads();   // inputs are in; the piece before is done with every array
      put<E>(Hc + own, h0);
      if constexpr (WIDE) frags_in<V>(wS, lane, ww);
      __syncthreads();
      // the next piece's inputs, unless a pass over its chunk comes first
      fetched = i > 0 || (ch > 0 && a.C <= kSteps);
      if (fetched) fetch(x + 1, i > 0 ? piece(ch, i - 1) : piece(ch - 1, 0));
      // (A)
      forward(x, pc.len);
      // (B)
      const float *st = stage(x), *fs = fS + (x & 1) * kSteps;
      if constexpr (BG::kReload) load_wt<V>(Wn, p, c0, w);
      if constexpr (WIDE) frags_in<V>(wS + V * V, lane, ww);
      for (int s = pc.len - 1; s >= 0; --s) {
        const float f = fs[s], q = st[s * GR + orow];
        const Vec<E> dy = get<E>(st + oDY + s * V + ocol), hp = get<E>(Hc + s * BG::kTile + own);
        float *xs = Xc + s * BG::kTile;
        const Vec<E> z = get<E>(xs + own);
        Vec<E> Gv, dX;
        float df = 0.f;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          Gv.x[e] = fmaf(q, dy.x[e], C.x[e]);                        // G = C + q dy^T
          df = fmaf(Gv.x[e], hp.x[e] - z.x[e], df);                  // df = sum G (.) (H_{t-1} - Z)
          dX.x[e] = (1.f - f) * Gv.x[e] * (1.f - z.x[e] * z.x[e]);   // through the gate and tanh
        }
        dfp[s * kThreads + tid] = df;
        put<E>(xs + own, dX);
        row_sync();
        const Vec<E> o = mul(xs, true);                              // C_{t-1} = f G + dX W^T
#pragma unroll
        for (int e = 0; e < E; ++e) {
          C.x[e] = fmaf(f, Gv.x[e], o.x[e]);
          if (a.dh_clip > 0.f) C.x[e] = fminf(fmaxf(C.x[e], -a.dh_clip), a.dh_clip);
        }
      }
      if constexpr (WIDE) __syncthreads();      // all rows of the piece are in
      // (C) dW += H_{t-1}^T dX over the piece's steps and rows
      for (int s = tsp; s < pc.len; s += BG::SP) {
        const float *hs = Hc + s * BG::kTile + tl, *xs = Xc + s * BG::kTile + tj;
#pragma unroll
        for (int r = 0; r < GR; ++r) {
          const float4 h4 = *reinterpret_cast<const float4 *>(hs + r * G::HP);
          const float hv[4] = {h4.x, h4.y, h4.z, h4.w};
#pragma unroll
          for (int jj = 0; jj < BG::JT / 4; ++jj) {
            const float4 x4 = *reinterpret_cast<const float4 *>(xs + r * G::HP + jj * (V / 2));
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              dW[e][2 * jj] = __ffma2_rn(make_float2(hv[e], hv[e]), make_float2(x4.x, x4.y), dW[e][2 * jj]);
              dW[e][2 * jj + 1] = __ffma2_rn(make_float2(hv[e], hv[e]), make_float2(x4.z, x4.w), dW[e][2 * jj + 1]);
            }
          }
        }
      }
      // dq = H_t dy, dk = dX v: eight lanes per (step, row)
      const size_t bt0 = tok0 + pc.t0;
      for (int it = tid >> 3; it < pc.len * GR; it += kThreads / 8) {
        const int s = it / GR, r = it % GR, e = tid & 7;
        const float *hs = Hc + (s + 1) * BG::kTile + r * G::HP, *xs = Xc + s * BG::kTile + r * G::HP;
        const float *dys = st + oDY + s * V, *vs = st + oV + s * V;
        float dq = 0.f, dk = 0.f;
#pragma unroll
        for (int j = 0; j < V / 16; ++j) {
          const int c = 16 * j + 2 * e;
          const float2 h2 = *reinterpret_cast<const float2 *>(hs + c), d2 = *reinterpret_cast<const float2 *>(dys + c);
          const float2 x2 = *reinterpret_cast<const float2 *>(xs + c), v2 = *reinterpret_cast<const float2 *>(vs + c);
          dq = fmaf(h2.x, d2.x, fmaf(h2.y, d2.y, dq));
          dk = fmaf(x2.x, v2.x, fmaf(x2.y, v2.y, dk));
        }
        // (all lanes of a warp take the same number of turns: len x GR items are whole groups of four)
#pragma unroll
        for (int off = 1; off < 8; off <<= 1) { dq += __shfl_xor_sync(0xffffffffu, dq, off); dk += __shfl_xor_sync(0xffffffffu, dk, off); }
        if (e == 0) {
          const size_t bt = bt0 + s;
          if (a.dq_part) a.dq_part[(bt * N + n) * K + rbase + r] = dq;
          else static_cast<float *>(a.dq)[(bt * a.Nq + hq) * K + rbase + r] = dq;
          if (a.dk_part) a.dk_part[(bt * N + n) * K + rbase + r] = dk;
          else static_cast<float *>(a.dk)[(bt * a.Nk + hk) * K + rbase + r] = dk;
        }
      }
      // dv = dX^T k over these rows (+ w_r (.) dy from Eq. 3, added with the first group)
      for (int it = tid; it < pc.len * (V / 4); it += kThreads) {
        const int s = it / (V / 4), j = 4 * (it % (V / 4));
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int r = 0; r < GR; ++r) {
          const float k = st[oK + s * GR + r];
          const float4 x4 = *reinterpret_cast<const float4 *>(Xc + s * BG::kTile + r * G::HP + j);
          o.x = fmaf(k, x4.x, o.x); o.y = fmaf(k, x4.y, o.y); o.z = fmaf(k, x4.z, o.z); o.w = fmaf(k, x4.w, o.w);
        }
        if (wr && rs == 0) {
          const float4 w4 = *reinterpret_cast<const float4 *>(wr + (size_t)n * V + j), d4 = *reinterpret_cast<const float4 *>(st + oDY + s * V + j);
          o.x = fmaf(w4.x, d4.x, o.x); o.y = fmaf(w4.y, d4.y, o.y); o.z = fmaf(w4.z, d4.z, o.z); o.w = fmaf(w4.w, d4.w, o.w);
        }
        const size_t at = ((bt0 + s) * N + n) * V + j;
        float4 *dst = reinterpret_cast<float4 *>((a.dv_part ? a.dv_part + (size_t)rs * a.TT * N * V : static_cast<float *>(a.dv)) + at);
        if (add) { const float4 old = *dst; o.x += old.x; o.y += old.y; o.z += old.z; o.w += old.w; }
        *dst = o;
      }
      // dgate: a warp sums the threads' shares of a step, then the gate's slope
      for (int s = warp; s < pc.len; s += kThreads / 32) {
        float df = 0.f;
#pragma unroll
        for (int i2 = 0; i2 < kThreads / 32; ++i2) df += dfp[s * kThreads + 32 * i2 + lane];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) df += __shfl_xor_sync(0xffffffffu, df, off);
        if (lane == 0) {
          float *dst = (a.dgate_part ? a.dgate_part + (size_t)rs * a.TT * N : a.dgate) + (bt0 + s) * N + n;
          df *= dfS[(x & 1) * kSteps + s];
          *dst = add ? *dst + df : df;
        }
      }
    }
  }
  if (a.dh0) put<E>(a.dh0 + (size_t)bn * KV + own_g, C);
  // dW: the threads that share a tile are added in a fixed order
  float *dWp = a.dW_part + (nslab == 1 ? (size_t)bn : ((size_t)b * nslab + rs) * N + n) * V * V;
  if constexpr (BG::SP > 1) {
    float *sh = Hc;   // [SP - 1][tiles][16]
    __syncthreads();
    if (tsp > 0)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        *reinterpret_cast<float4 *>(sh + ((size_t)(tsp - 1) * BG::kTiles + tile) * 16 + 4 * e) = make_float4(dW[e][0].x, dW[e][0].y, dW[e][1].x, dW[e][1].y);
    __syncthreads();
    if (tsp > 0) return;
    for (int k = 0; k < BG::SP - 1; ++k)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float4 o = *reinterpret_cast<const float4 *>(sh + ((size_t)k * BG::kTiles + tile) * 16 + 4 * e);
        dW[e][0].x += o.x; dW[e][0].y += o.y; dW[e][1].x += o.z; dW[e][1].y += o.w;
      }
  }
#pragma unroll
  for (int e = 0; e < 4; ++e)
#pragma unroll
    for (int jj = 0; jj < BG::JT / 4; ++jj) {
      float4 *dst = reinterpret_cast<float4 *>(dWp + (size_t)(tl + e) * V + tj + jj * (V / 2));
      float4 o = make_float4(dW[e][2 * jj].x, dW[e][2 * jj].y, dW[e][2 * jj + 1].x, dW[e][2 * jj + 1].y);
      if (add) { const float4 old = *dst; o.x += old.x; o.y += old.y; o.z += old.z; o.w += old.w; }
      *dst = o;
    }
}

// ------------------------------------------------------------------ decoding step (Eq. 1-3 once)
// Persistent CTAs over (head, batch entry) in head-major order, W reloaded only when the head changes;
// the groups of eight rows of a state stream through a ring of kRing stages (cp.async), are
// multiplied, updated and written back in place.  The readout is complete inside the CTA.
// Bound by FMA at V >= 64 (V/8 FMA per byte of state against 6 at the chip's rates), by HBM below.
constexpr int kRing = 4;

template <int V>
struct DecGeom {
  static constexpr int kOcc = V == 128 ? 1 : 768 / Geom<V>::kThreads;   // CTAs per SM: 24 warps (V = 128: 16) at 85 registers or more
  static constexpr int kStage = Geom<V>::kTile + 2 * kRows + V;   // rows, then k [8], q [8], v [V]
};

template <int V>
__global__ void __launch_bounds__(Geom<V>::kThreads, DecGeom<V>::kOcc) decode_f32_kernel(ScanArgs a) {
  using G = Geom<V>;
  constexpr int kStage = DecGeom<V>::kStage;
  extern __shared__ __align__(16) float smem[];
  begin_dependent();
  const int K = a.K, N = a.N, B = a.B, ng = K / kRows;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, p = lane >> 2, c0 = 8 * warp + 2 * (lane & 3), ycol = y_col<kRows>(lane, c0);
  const size_t KV = (size_t)K * V;
  const float *qg = static_cast<const float *>(a.q), *kg = static_cast<const float *>(a.k);
  const float *vg = static_cast<const float *>(a.v), *wr = static_cast<const float *>(a.w_r);
  float *state = a.hT, *yg = static_cast<float *>(a.y);   // state == a.h0: updated in place
  const long units = (long)N * B, u0 = units * blockIdx.x / gridDim.x, u1 = units * (blockIdx.x + 1) / gridDim.x;

  long uf = u0;   // next group to fetch: unit and group
  int gf = 0;
  auto fetch = [&](int slot) {   // always one commit group, possibly empty
    if (uf < u1) {
      const int n = (int)(uf / B), b = (int)(uf % B), r0 = gf * kRows;
      const size_t bn = (size_t)b * N + n;
      float *st = smem + slot * kStage;
      const float *src = state + bn * KV + (size_t)r0 * V;
      for (int i = tid; i < kRows * (V / 4); i += G::kThreads) cp16(st + (i / (V / 4)) * G::HP + 4 * (i % (V / 4)), src + 4 * i);
      if (tid < 2) cp16(st + G::kTile + 4 * tid, kg + ((size_t)b * a.Nk + n / (N / a.Nk)) * K + r0 + 4 * tid);
      else if (tid < 4) cp16(st + G::kTile + 4 * tid, qg + ((size_t)b * a.Nq + n / (N / a.Nq)) * K + r0 + 4 * (tid - 2));
      else if (tid < 4 + V / 4) cp16(st + G::kTile + 4 * tid, vg + bn * V + 4 * (tid - 4));
      if (++gf == ng) { gf = 0; ++uf; }
    }
    cp_commit();
  };
#pragma unroll
  for (int i = 0; i < kRing - 1; ++i) fetch(i);
  float2 w[G::NP][2];
  int head = -1, slot = 0;
  for (long u = u0; u < u1; ++u) {
    const int n = (int)(u / B), b = (int)(u % B);
    const size_t bn = (size_t)b * N + n;
    const float graw = a.gate[bn];
    if (n != head) { load_w<V>(static_cast<const float *>(a.W) + (size_t)n * V * V, p, c0, w); head = n; }
    const float f = gate_value(a.gate_kind, graw, a.alpha ? a.alpha[n] : 1.f, a.beta ? a.beta[n] : 0.f, nullptr);
    float y = 0.f;
    const float wrv = wr ? wr[(size_t)n * V + ycol] : 0.f;
    for (int g = 0; g < ng; ++g) {
      cp_wait<kRing - 2>();
      __syncthreads();                                   // this group is in for everybody; the one before is used up
      const float *st = smem + slot * kStage, *vec = st + G::kTile;
      fetch(slot == 0 ? kRing - 1 : slot - 1);           // into the slot just freed
      const Vec<2> o = product<V, kRows>(st, w, p, lane);
      Vec<2> z;
      const Vec<2> h = update<2>(o, vec[p], get<2>(vec + 2 * kRows + c0), f, get<2>(st + p * G::HP + c0), z);
      put<2>(state + bn * KV + (size_t)(g * kRows + p) * V + c0, h);
      y = readout<kRows>(y, g == 0, wrv, vec[2 * kRows + ycol], vec[kRows + p], h, lane);
      slot = slot + 1 == kRing ? 0 : slot + 1;
    }
    if (y_owner<kRows>(lane)) yg[bn * V + ycol] = y;
  }
  cp_wait<0>();
}

template <int V, int GR>
cudaError_t launch_fwd_g(const ScanArgs &a, cudaStream_t s) {
  const size_t smem = fwd_f32_smem<V>(a.KCf);
  const cudaError_t e = allow_smem(fwd_f32_kernel<V, GR>, smem);
  if (e != cudaSuccess) return e;
  const int ctas = a.B * a.N * (a.K / a.KCf);
  return launch_early(fwd_f32_kernel<V, GR>, ctas, Geom<V>::kThreads, smem, s, in_order(a, ctas, Geom<V>::kThreads, 7));
}
template <int V, int R>
cudaError_t launch_fwd_w(const ScanArgs &a, cudaStream_t s) {
  constexpr size_t smem = sizeof(float) * (size_t)WideFwd<V, R>::kFloats;
  constexpr int kThreads = WideFwd<V, R>::kThreads;
  const cudaError_t e = allow_smem(fwd_f32_wide_kernel<V, R>, smem);
  if (e != cudaSuccess) return e;
  const int ctas = a.B * a.N * (a.K / 4);
  return launch_early(fwd_f32_wide_kernel<V, R>, ctas, kThreads, smem, s, in_order(a, ctas, kThreads, 4));
}
template <int V>
cudaError_t launch_fwd_v(const ScanArgs &a, cudaStream_t s) {
  if constexpr (V >= 32) {
    if (a.KCf == kRows / 2) {
      // One row a warp while that makes no more than 11 warps an SM, then two, then four: a warp's step is a chain, as long as its rows
      // are many (256 steps of K = V = 64, us, one / two / four rows: 1 024 rows in all 108 / 118 / 189, 2 048 204 / 185 / 192, 6 144
      // 538 / 517 / 476; V = 128, two and four: 512 rows 157 / 179, 2 048 585 / 548).
      const long warps = (long)a.B * a.N * a.K * Wide<V>::NWR, most = 11L * sm_count();
      if constexpr (V <= 64)
        if (warps <= most) return launch_fwd_w<V, 1>(a, s);
      return warps <= 2 * most ? launch_fwd_w<V, 2>(a, s) : launch_fwd_w<V, 4>(a, s);
    }
    return launch_fwd_g<V, kRows>(a, s);
  } else {
    return a.KCf == kRows / 2 ? launch_fwd_g<V, kRows / 2>(a, s) : launch_fwd_g<V, kRows>(a, s);
  }
}

template <int V, int GR, bool WIDE>
cudaError_t launch_bwd_g(const ScanArgs &a, cudaStream_t s) {
  using BG = BwdGeom<V, GR, WIDE>;
  const size_t smem = sizeof(float) * (size_t)BG::kFloats;
  cudaError_t e = allow_smem(bwd_f32_kernel<V, GR, WIDE>, smem);
  const int slabs = a.K / GR, nslab = a.KC == GR ? slabs : 1;
  for (int s0 = 0; s0 < slabs && e == cudaSuccess; s0 += nslab) {
    e = launch_early(bwd_f32_kernel<V, GR, WIDE>, a.B * a.N * nslab, BG::kThreads, smem, s, in_order(a, (long)a.B * a.N * nslab, BG::kThreads, 12), s0, nslab);
  }
  return e;
}
template <int V>
cudaError_t launch_bwd_v(const ScanArgs &a, cudaStream_t s) {
  // (wide, 512 steps of K = V = 64, us: 16 units 630 -> 564, 64 units against groups of eight 2 133 -> 1 949, 256 units 3 677 -> 3 793; K = V =
  // 32, 16 units 306 -> 329)
  return a.KC == kRows / 2 ? launch_bwd_g<V, kRows / 2, V == 64>(a, s) : launch_bwd_g<V, kRows, false>(a, s);
}

template <int V>
cudaError_t launch_decode_v(const ScanArgs &a, cudaStream_t s) {
  const size_t smem = sizeof(float) * (size_t)kRing * DecGeom<V>::kStage;
  const cudaError_t e = allow_smem(decode_f32_kernel<V>, smem);
  if (e != cudaSuccess) return e;
  const long units = (long)a.B * a.N, room = (long)sm_count() * DecGeom<V>::kOcc;
  return launch_early(decode_f32_kernel<V>, (unsigned)(units < room ? units : room), Geom<V>::kThreads, smem, s, a);
}

}  // namespace

// Rows per CTA.  The step of a warp is a chain of dependent instructions, so a problem wants its rows spread over many warps.
// Forward, V >= 32: groups of four rows (fwd_f32_wide_kernel), at any number of units that their shares of y leave room for.  256
// steps, us, groups of four / of eight / whole states: K = V = 64, 16 units 106 / 194 / 1 097, 128 625 / 836 / 1 098, 512 2 137 / 3 183 / 3 153, 2 048
// 8 443 / 12 486 / 10 372; K = V = 32, 2 048 units 1 631 / 2 422 / 2 002; K = V = 128, 16 units 548 / 759 / 4 539, 256 7 355 / 10 580 / 9 073.  The shares
// are memory bought for that 18 to 50 %, 4 GiB of the GPU's 180 at most.  Where groups of four would need more, groups of eight while
// the units alone leave an SM fewer than 16 warps and their shares fit (four sequences of 32 768 tokens, ten heads of K = V = 64, ms: 34 by
// groups of four in 5 GiB, 46 in 2.5, whole states 139); whole states beyond.  Where groups of eight would leave an SM fewer than 16 warps
// it is groups of four up to 8 GiB (one of 70 000, 16 heads: 27 against 51 and 298).
// V = 16 and the backward: groups of four rows while groups of eight would leave an SM fewer than 16 warps (V = 64: 32), else of eight,
// which need fewer instructions in all.  Whole states forward (V = 16) where that gives every SM 16 warps -- the groups take turns
// behind one barrier a step and y needs no shares in memory.  Backward: K stands for one launch per group of eight, each adding to
// the results of the one before, where the units alone give every SM 64 warps.  `share_bytes`: one group's share of y or dv; whole
// states (one group after the other) too where the shares of all groups would exceed kMaxShares.
constexpr size_t kMaxShares = (size_t)4 << 30;
int fwd_f32_rows(int B, int N, int K, int V, size_t share_bytes) {
  const long warps = (long)(B > 0 ? B : 1) * N * (V / 8), most = 16L * sm_count();   // of whole states
  if (V >= 32 && share_bytes * (K / (kRows / 2)) <= kMaxShares) return kRows / 2;
  if (warps >= most || share_bytes * (K / kRows) > kMaxShares) return K;
  return warps * (K / kRows) >= most ? kRows : kRows / 2;
}
int bwd_f32_rows(int B, int N, int K, int V, size_t share_bytes) {
  const long warps = (long)(B > 0 ? B : 1) * N * (V / 8), most = 16L * sm_count();
  if (warps >= 4 * most || share_bytes * (K / kRows) > kMaxShares) return K;
  return warps * (K / kRows) >= (V == 64 ? 2 : 1) * most ? kRows : kRows / 2;
}
int bwd_f32_piece() { return kSteps; }

cudaError_t launch_fwd_f32(const ScanArgs &a, cudaStream_t s) {
  switch (a.V) {
    case 16: return launch_fwd_v<16>(a, s);
    case 32: return launch_fwd_v<32>(a, s);
    case 64: return launch_fwd_v<64>(a, s);
    default: return launch_fwd_v<128>(a, s);
  }
}
cudaError_t launch_bwd_f32(const ScanArgs &a, cudaStream_t s) {
  switch (a.V) {
    case 16: return launch_bwd_v<16>(a, s);
    case 32: return launch_bwd_v<32>(a, s);
    case 64: return launch_bwd_v<64>(a, s);
    default: return launch_bwd_v<128>(a, s);
  }
}
cudaError_t launch_decode_f32(const ScanArgs &a, cudaStream_t s) {
  switch (a.V) {
    case 16: return launch_decode_v<16>(a, s);
    case 32: return launch_decode_v<32>(a, s);
    case 64: return launch_decode_v<64>(a, s);
    default: return launch_decode_v<128>(a, s);
  }
}

}  // namespace m2rnn
