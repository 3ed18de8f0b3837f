// bf16 decoding step (Eq. 1-3 once on a cached fp32 state) for sm_100a, V <= 64.
//
// The step streams every state through the chip once (fp32, read and write), so the kernel is laid out
// around HBM: warps that need nothing from one another.  A warp takes a contiguous range of (head,
// batch) units in head-major order, keeps the head's transition matrix as MMA fragments in registers,
// and walks its units in slabs of 16 rows (16 V contiguous floats).  Slabs are copied (cp.async) several
// ahead into a ring in shared memory whose every 16 bytes are read by the lane that copied them: no
// barrier of any kind.  A slab goes through mma.sync (bf16 operands, fp32 accumulate), outer product,
// tanh and gate in registers and is stored straight back.  The readout is summed over a unit's slabs
// in registers.
// The code a warp runs once is kept short: the first pass through an instruction comes from the L2
// (the slab loop unrolled by four cost a small batch 4 us, 64-bit divisions another 1.5).
// A CTA that takes eight slabs at a time behind barriers, two stages ahead, spends 1.9 us of latency on
// them whatever their size.  The paper's layer (N = 84, K = 64, V = 16) at batch 48: 25.6 -> 8.2 us, 6.0
// where steps follow one another on a stream (the early launch hides the gap between them; a step after which the GPU is waited for,
// host and all, 17.2 -> 16.1); at batch 400: 200 -> 50 us (5.5 TB/s).
#include "device_common.cuh"
#include "internal.h"
#include "mma_tile.cuh"
#include "pipeline.cuh"

namespace m2rnn {
namespace {

template <int V>
struct DecCfg {
  static constexpr int kWarps = V == 64 ? 8 : (V == 32 ? 16 : 32);  // one CTA per SM (its warps share nothing but the launch)
  static constexpr int kStages = V == 64 ? 6 : (V == 32 ? 5 : 4);   // slabs on their way per warp: 6 x 4, 5 x 2, 4 x 1 KB
  static constexpr bool kSplit = V >= 64;   // the state enters the product as the sum of two bf16 operands
  static constexpr int kSlabBytes = 16 * V * 4;
  static constexpr int kSmem = kWarps * kStages * kSlabBytes;
};

// Memory column of MMA column m = 8nt + 2c + e: a thread's registers of the tile pair
// (2x, 2x+1) are the four adjacent columns 16x + 4c .. 16x + 4c + 3, so the four lanes of a row
// group touch 64 contiguous bytes of a row.
__host__ __device__ constexpr int dec_col(int m) { return 16 * (m >> 4) + 4 * ((m & 7) >> 1) + 2 * ((m >> 3) & 1) + (m & 1); }

__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t a) {
  uint32_t d;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
  return d;
}
// A operand of k-tile kt from the state in accumulator layout: the bf16 rounding, and what it leaves out
// as a second operand (used where kSplit: the product then sees the state with 16 bits of mantissa)
template <int NT>
__device__ __forceinline__ void a_fragment(const float (&H)[NT][4], int kt, uint32_t (&hi)[4], uint32_t (&lo)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float x = H[2 * kt + (i >> 1)][2 * (i & 1)], y = H[2 * kt + (i >> 1)][2 * (i & 1) + 1];
    hi[i] = pack_bf16(x, y);
    lo[i] = pack_bf16(x - __uint_as_float(hi[i] << 16), y - __uint_as_float(hi[i] & 0xffff0000u));
  }
}

template <int V>
__global__ void __launch_bounds__(32 * DecCfg<V>::kWarps, 1) decode_bf16_kernel(ScanArgs a, int per, int extra) {
  using Cfg = DecCfg<V>;
  constexpr int NT = V / 8, KT = V / 16, SEG = V / 4, NX = V / 16, kStages = Cfg::kStages, kWarps = Cfg::kWarps;
  extern __shared__ __align__(128) unsigned char smem[];
  begin_dependent();
  const int K = a.K, N = a.N, B = a.B, slabs = K / 16;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  const int dq = N / a.Nq, dk = N / a.Nk;
  const size_t KV = (size_t)K * V;
  const uint16_t *qg = static_cast<const uint16_t *>(a.q), *kg = static_cast<const uint16_t *>(a.k), *Wg = static_cast<const uint16_t *>(a.W);
  const __nv_bfloat16 *vg = static_cast<const __nv_bfloat16 *>(a.v), *wr = static_cast<const __nv_bfloat16 *>(a.w_r);
  __nv_bfloat16 *yg = static_cast<__nv_bfloat16 *>(a.y);
  float *state = a.hT;   // == a.h0: updated in place

  // this warp's units (the first `extra` warps take per + 1); neighbouring ranges go to different SMs
  const int wid = warp * (int)gridDim.x + (int)blockIdx.x;
  int left = per + (wid < extra);           // units to go, and to request
  if (left == 0) return;
  const unsigned u0 = (unsigned)wid * per + min(wid, extra);

  // a stage of the ring: [2 V/16 chunks][32 lanes] x 16 bytes
  const uint32_t ring_sa = smem_u32(smem) + (uint32_t)warp * kStages * Cfg::kSlabBytes + 16u * lane;
  const int lane_off = g * V + 4 * c;   // this lane's first element of a slab

  int n = (int)(u0 / (unsigned)B), b = (int)(u0 - (unsigned)n * B);
  // the next slab to request
  const size_t unit_step = (size_t)N * KV;
  const float *pf = state + ((size_t)b * N + n) * KV + lane_off;
  int nf = n, bf = b, sf = 0;
  int todo = left;
  auto request = [&](int st) {   // always one group, possibly empty
    if (todo > 0) {
      const uint32_t dst = ring_sa + (uint32_t)st * Cfg::kSlabBytes;
#pragma unroll
      for (int x = 0; x < NX; ++x) {
        cp16(dst + 1024u * x, pf + 16 * x);
        cp16(dst + 1024u * x + 512u, pf + 16 * x + 8 * V);
      }
      pf += 16 * V;
      if (++sf == slabs) {
        sf = 0; --todo; ++bf;
        pf += unit_step - KV;
        if (bf == B) { bf = 0; ++nf; pf = state + (size_t)nf * KV + lane_off; }
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int s = 0; s < kStages; ++s) request(s);

  // A unit's vectors, fetched one unit ahead.  k and q: lane (g, c) holds the entries of rows g and g + 8 of
  // slabs c and c + 4 as one word each; slab s takes its pair from lane (g, s % 4).
  struct Vecs { uint32_t k[2], q[2]; uint2 v[NX]; float gate; };
  auto fetch = [&](int n, int b, int hk, int hq, Vecs &o) {
    const uint16_t *kp = kg + ((size_t)b * a.Nk + hk) * K, *qp = qg + ((size_t)b * a.Nq + hq) * K;
    const size_t bn = (size_t)b * N + n;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      o.k[h] = o.q[h] = 0u;
      if (c + 4 * h < slabs) {
        const int r = 16 * (c + 4 * h) + g;
        o.k[h] = (uint32_t)kp[r] | ((uint32_t)kp[r + 8] << 16);
        o.q[h] = (uint32_t)qp[r] | ((uint32_t)qp[r + 8] << 16);
      }
    }
#pragma unroll
    for (int x = 0; x < NX; ++x) o.v[x] = *reinterpret_cast<const uint2 *>(vg + bn * V + 16 * x + 4 * c);
    o.gate = a.gate[bn];
  };
  Vecs next;
  int hk = n / dk, hq = n / dq;
  fetch(n, b, hk, hq, next);

  uint32_t W[KT][NT][2];
  int head = -1, st = 0;
  for (; left > 0; --left) {
    const Vecs cur = next;
    const size_t bn = (size_t)b * N + n;
    int n1 = n, b1 = b + 1;
    if (b1 == B) { b1 = 0; ++n1; hk = n1 / dk; hq = n1 / dq; }
    if (left > 1) fetch(n1, b1, hk, hq, next);
    if (n != head) {
      // B fragments: a word of W holds two adjacent columns of a row, the fragment wants two adjacent rows
      // of a column: one 8 x 8 transpose per register
      const uint16_t *w = Wg + (size_t)n * V * V;
#pragma unroll
      for (int kt = 0; kt < KT; ++kt)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            W[kt][nt][h] = movmatrix_trans(*reinterpret_cast<const uint32_t *>(w + dec_col(16 * kt + 8 * h + g) * V + dec_col(8 * nt + 2 * c)));
      head = n;
    }
    const float f = gate_value(a.gate_kind, cur.gate, a.alpha ? a.alpha[n] : 1.f, a.beta ? a.beta[n] : 0.f, nullptr);
    float part[SEG];
#pragma unroll
    for (int e = 0; e < SEG; ++e) part[e] = 0.f;
#pragma unroll 1
    for (int s = 0; s < slabs; ++s) {
      const uint32_t kk = __shfl_sync(0xffffffffu, s < 4 ? cur.k[0] : cur.k[1], 4 * g + (s & 3));
      const uint32_t qq = __shfl_sync(0xffffffffu, s < 4 ? cur.q[0] : cur.q[1], 4 * g + (s & 3));
      const float k0 = __uint_as_float(kk << 16), k1 = __uint_as_float(kk & 0xffff0000u);
      const float q0 = __uint_as_float(qq << 16), q1 = __uint_as_float(qq & 0xffff0000u);
      asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 1) : "memory");
      // rows g and g + 8 of the slab in accumulator layout
      float H[NT][4];
      const uint32_t src = ring_sa + (uint32_t)st * Cfg::kSlabBytes;
#pragma unroll
      for (int x = 0; x < NX; ++x) {
        const float4 t0 = lds128(src + 1024u * x), t1 = lds128(src + 1024u * x + 512u);
        H[2 * x][0] = t0.x; H[2 * x][1] = t0.y; H[2 * x + 1][0] = t0.z; H[2 * x + 1][1] = t0.w;
        H[2 * x][2] = t1.x; H[2 * x][3] = t1.y; H[2 * x + 1][2] = t1.z; H[2 * x + 1][3] = t1.w;
      }
      request(st);   // the stage is read (by this lane, which alone uses its part of it)
      if (++st == kStages) st = 0;
      // P = k v^T + H W   (Eq. 1 before the non-linearity)
      float P[NT][4];
#pragma unroll
      for (int x = 0; x < NX; ++x) {
        const float2 va = make_float2(__uint_as_float(cur.v[x].x << 16), __uint_as_float(cur.v[x].x & 0xffff0000u));
        const float2 vb = make_float2(__uint_as_float(cur.v[x].y << 16), __uint_as_float(cur.v[x].y & 0xffff0000u));
        P[2 * x][0] = k0 * va.x; P[2 * x][1] = k0 * va.y; P[2 * x][2] = k1 * va.x; P[2 * x][3] = k1 * va.y;
        P[2 * x + 1][0] = k0 * vb.x; P[2 * x + 1][1] = k0 * vb.y; P[2 * x + 1][2] = k1 * vb.x; P[2 * x + 1][3] = k1 * vb.y;
      }
#pragma unroll
      for (int kt = 0; kt < KT; ++kt) {
        uint32_t hi[4], lo[4];
        a_fragment<NT>(H, kt, hi, lo);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          mma_bf16_16816(P[nt], hi, W[kt][nt][0], W[kt][nt][1]);
          if constexpr (Cfg::kSplit) mma_bf16_16816(P[nt], lo, W[kt][nt][0], W[kt][nt][1]);
        }
      }
      float *dst = state + bn * KV + (size_t)(16 * s + g) * V + 4 * c;
#pragma unroll
      for (int x = 0; x < NX; ++x) {
#pragma unroll
        for (int nt = 2 * x; nt < 2 * x + 2; ++nt)
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const float z = tanh_approx(P[nt][r]);        // Eq. 1
            H[nt][r] = fmaf(f, H[nt][r] - z, z);          // Eq. 2
          }
        *reinterpret_cast<float4 *>(dst + 16 * x) = make_float4(H[2 * x][0], H[2 * x][1], H[2 * x + 1][0], H[2 * x + 1][1]);
        *reinterpret_cast<float4 *>(dst + 16 * x + 8 * V) = make_float4(H[2 * x][2], H[2 * x][3], H[2 * x + 1][2], H[2 * x + 1][3]);
#pragma unroll
        for (int nt = 2 * x; nt < 2 * x + 2; ++nt)
#pragma unroll
          for (int e = 0; e < 2; ++e) part[2 * nt + e] = fmaf(q0, H[nt][e], fmaf(q1, H[nt][2 + e], part[2 * nt + e]));   // Eq. 3, this thread's two rows
      }
    }
    // column sums over the unit's rows; idx = 2nt+e of a thread <-> memory column 16(idx>>2)+4c+(idx&3)
    reduce_over_rows<SEG>(part, lane);
    using RO = RowReduceOut<V>;
    if (RO::owner(lane)) {
      const int idx0 = (g >> (3 - RO::R)) * RO::CNT, col = 16 * (idx0 >> 2) + 4 * c + (idx0 & 3);
      if (wr) {
#pragma unroll
        for (int j = 0; j < RO::CNT; ++j)
          part[j] = fmaf(__bfloat162float(wr[(size_t)n * V + col + j]), __bfloat162float(vg[bn * V + col + j]), part[j]);
      }
      if constexpr (RO::CNT == 2) *reinterpret_cast<uint32_t *>(yg + bn * V + col) = pack_bf16(part[0], part[1]);
      else yg[bn * V + col] = __float2bfloat16_rn(part[0]);
    }
    n = n1; b = b1;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

template <int V>
cudaError_t launch_decode_v(const ScanArgs &a, cudaStream_t s) {
  const cudaError_t e = allow_smem(decode_bf16_kernel<V>, DecCfg<V>::kSmem);
  if (e != cudaSuccess) return e;
  const long units = (long)a.B * a.N, room = sm_count(), grid = units < room ? units : room, warps = grid * DecCfg<V>::kWarps;
  return launch_early(decode_bf16_kernel<V>, (unsigned)grid, 32 * DecCfg<V>::kWarps, DecCfg<V>::kSmem, s, a, (int)(units / warps), (int)(units % warps));
}

}  // namespace

// V = 128 goes to the tcgen05 kernel: there a slab's 256 mma.sync take longer than its bytes need (2.1 GB of
// state: 622 us with W shared through shared memory, 395 there).  At V = 64 they do not (210 MB: 44 us
// here, 61 there).
cudaError_t launch_decode_bf16(const ScanArgs &a, cudaStream_t s) {
  switch (a.V) {
    case 16: return launch_decode_v<16>(a, s);
    case 32: return launch_decode_v<32>(a, s);
    case 64: return launch_decode_v<64>(a, s);
    default: return launch_decode_tc_bf16(a, s);
  }
}

}  // namespace m2rnn
