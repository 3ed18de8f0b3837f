// bf16 tensor-core backward through time for V = 16, the state size of the paper's own layers.
//
// A CTA takes hg value heads of one batch entry and R slabs of 16 state rows each; a slab warp owns one (head, slab)
// pair for all T steps and does all of its arithmetic.  Time is walked in chunks of C steps (the checkpoint interval),
// last chunk first: the forward steps of chunk j + 1 (from its checkpoint) and the reverse steps of chunk j are
// interleaved one by one in the same instruction stream.  They do not depend on each other, so each covers the other's
// latency.  The forward steps leave H_{t-1} (bf16, the A fragment they need anyway) and Z_t (fp16) in the warp's own piece of
// shared memory, each in the place that the reverse step before it has left; no other warp reads them.  dq = H_t dy,
// dk = dX v and dv = dX^T k are small MMAs on fragments at hand; for dW += H_{t-1}^T dX the fragments are transposed in
// registers (movmatrix).
//   loader warp   k, q, v, dy of coming chunks as they are (cp.async), gates evaluated, a lane each;
//   writer warp   adds the heads' shares of dq and dk (heads that share them), the slabs' shares of dv and dgate, and
//                 writes a finished chunk out.
// Hand-over is by mbarriers between these two and the slab warps only; every wait is bounded and reports through dev_status.
//
// What bounds it: instruction issue, and with it how many slab warps the busiest scheduler has (three on the paper's layer
// shape: 84 heads, K = 64, batch 4, one wave of ten slabs an SM, 442 ns a step; a warp with a scheduler to itself 240).  A step is
// some 165 instructions of a slab warp, 57 of them on the FMA pipe, whose packed fp32 pairs take two cycles like two single ones:
// products and sums of 16-bit operands are taken without unpacking instead (fma.f32.bf16, add.f32.f16, one cycle each).
// Backward call of that shape, 1 024 steps: 799 us with four kinds of warps that handed states over through shared memory, two waves,
// and a share of dq and dk per head; 473 now, 452 of them this kernel.  Tried and slower: states of a chunk in registers (eight steps unrolled twice:
// the instruction cache), fp32 copies of k, v, q, dy (shared-memory bandwidth), stmatrix and ldmatrix for the transposition.
#include <algorithm>
#include <climits>
#include <numeric>

#include "device_common.cuh"
#include "internal.h"
#include "mma_tile.cuh"
#include "pipeline.cuh"
#include "tile.cuh"

namespace m2rnn {
namespace {

constexpr int kV = 16;
constexpr int kRing = 4;         // chunks of staged inputs
constexpr int kBarBytes = 128;

// Byte offsets; CC: the most steps of a chunk.  A ring slot: per head v, dy [CC][16] bf16, gates [CC] x four times {f, f - 1}, df/dgate [CC];
// then per slab q and k [CC][16] bf16.
template <int CC>
struct Lay {
  static constexpr uint32_t kDy = 32 * CC, kF = 64 * CC, kDf = 96 * CC, kHead = 100 * CC, kRows = 32 * CC;
  // results of a slab and chunk: dq, dk [CC][16 rows], dv [CC][16] (in the order of the fragments), dgate's share [CC]
  static constexpr uint32_t kDk = 64 * CC, kDv = 128 * CC, kOutDf = 192 * CC, kOut = 196 * CC;
  // a slab warp's own: two checkpoints, the lanes' shares of df, H_{t-1} and Z of a chunk's steps and one more
  static constexpr uint32_t kShare = 2 * 1024, kKept = kShare + 128 * CC, kWarp = kKept + 1024 * (CC + 1);
  // (qb, kb: slabs of q and k that the CTA stages)
  __host__ __device__ static uint32_t slot(int hg, int qb, int kb) { return (uint32_t)hg * kHead + (uint32_t)(qb + kb) * kRows; }
  __host__ __device__ static uint32_t out(int hg, int qb, int kb) { return kBarBytes + kRing * slot(hg, qb, kb); }
  __host__ __device__ static uint32_t warp(int hg, int qb, int kb, int slabs) { return out(hg, qb, kb) + 2u * (uint32_t)slabs * kOut; }
  __host__ __device__ static uint32_t total(int hg, int qb, int kb, int slabs) { return warp(hg, qb, kb, slabs) + (uint32_t)slabs * kWarp; }
};
constexpr int kMostSlabs = 10;   // slab warps of a CTA
constexpr int kRoomWarps = 14;   // warps of an SM with the kernel's registers

__device__ __forceinline__ uint32_t ldsu32(uint32_t addr) {
  uint32_t x;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(x) : "r"(addr));
  return x;
}
__device__ __forceinline__ uint2 ldsu64(uint32_t addr) {
  uint2 x;
  asm volatile("ld.shared.v2.b32 {%0,%1}, [%2];" : "=r"(x.x), "=r"(x.y) : "r"(addr));
  return x;
}
__device__ __forceinline__ uint4 get128(uint32_t addr) {
  uint4 x;
  asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w) : "r"(addr) : "memory");
  return x;
}
__device__ __forceinline__ void put128(uint32_t addr, const uint4 x) {
  asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(x.x), "r"(x.y), "r"(x.z), "r"(x.w) : "memory");
}
__device__ __forceinline__ uint32_t transposed(uint32_t x) {   // an 8 x 8 matrix, two entries of a row a thread
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}
// (bounds for two warps more than a CTA has: 144 registers, which the plan counts with)
// PER: checkpoints to a chunk, which starts from the first of them.  A template's argument, and the pointer worked out anew where it is
// not 1: one that walks by a runtime step costs the short chunks up to 9 % (B 10, 36 heads of their own, K = 64, T 40: 36.9 -> 40.4 us),
// one that walks two checkpoints 0 to 4 % (the same, T 1 024: 666 -> 699).
template <int CC, bool CLIP, int PER>
__global__ void __launch_bounds__(kRoomWarps * 32, 1) bwd_v16_kernel(ScanArgs a) {
  using L = Lay<CC>;
  extern __shared__ __align__(128) unsigned char smem[];
  begin_dependent();
  const int K = a.K, N = a.N, C = a.C;
  const int R = a.KC / 16, RS = K / a.KC, hg = a.hg;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31, g = lane >> 2, c = lane & 3;
  const int rs = blockIdx.x % RS, place = blockIdx.x / RS;
  const int b = batch_entry(a, place / a.groups, smem), grp = place % a.groups;
  // heads n0 .. n0 + nh - 1: sets of a.set heads (that share a q and a k head, where any do) in pieces of hg
  const int per = (a.set + hg - 1) / hg, n0 = grp / per * a.set + grp % per * hg, nh = min(hg, a.set - grp % per * hg);
  const bool one_q = a.Nq < N, one_k = a.Nk < N;      // shared heads: the CTA's heads have one q (k) between them
  const int qb = one_q ? R : hg * R, kb = one_k ? R : hg * R, slabs = nh * R;
  const UnitSpan span = unit_span(a, b);
  const int T = span.T, nch = (T + C - 1) / C;
  const size_t tok0 = span.tok0;
  const int rbase = rs * a.KC;
  const size_t KV = (size_t)K * kV;

  uint64_t *bars = reinterpret_cast<uint64_t *>(smem);
  uint64_t *in_full = bars, *slot_free = bars + kRing, *out_full = bars + 2 * kRing, *out_free = out_full + 2, *dw_full = out_free + 2;
  static_assert((2 * kRing + 5) * 8 <= kBarBytes, "barrier area");
  if (tid == 0) {
    for (int s = 0; s < kRing; ++s) { mbar_init(&in_full[s], 33); mbar_init(&slot_free[s], 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(&out_full[s], slabs); mbar_init(&out_free[s], 1); }
    mbar_init(dw_full, slabs);
    fence_mbar_init();
  }
  __syncthreads();

  const uint32_t sm0 = smem_u32(smem), slot_bytes = L::slot(hg, qb, kb), out0 = sm0 + L::out(hg, qb, kb);
  const uint32_t qrow = (uint32_t)hg * L::kHead, krow = qrow + (uint32_t)qb * L::kRows;
  auto slot_sa = [&](int j) { return sm0 + kBarBytes + (uint32_t)(j % kRing) * slot_bytes; };
  // chunk j of the sweep covers steps [t0, t0 + len) of time chunk nch-1-j
  auto chunk_t0 = [&](int j) { return (nch - 1 - j) * C; };
  auto chunk_len = [&](int j) { return min(C, T - chunk_t0(j)); };

  if (warp < hg * R) {
    // ================================================================= slab warps
    if (warp >= slabs) return;          // (the last piece of a set may have fewer heads)
    const int h = warp / R, r = warp % R, n = n0 + h;
    const int row0 = rbase + 16 * r + 2 * g;           // memory rows row0, row0 + 1 <-> MMA rows g, g + 8; columns 4c .. 4c + 3
    const size_t unit = (size_t)b * N + n, own = (size_t)row0 * kV + 4 * c;
    const __nv_bfloat16 *Wn = static_cast<const __nv_bfloat16 *>(a.W) + (size_t)n * kV * kV;
    uint32_t Wr[2][2], WTr[2][2];
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      load_w_fragment<kV>(Wn, 0, nt, lane, Wr[nt][0], Wr[nt][1]);
      load_wt_fragment<kV>(Wn, 0, nt, lane, WTr[nt][0], WTr[nt][1]);
    }
    const uint32_t v_off = (uint32_t)h * L::kHead + 8u * c;                                  // this thread's four columns of v, dy; the gate
    const uint32_t q_off = qrow + (uint32_t)((one_q ? 0 : h * R) + r) * L::kRows + 4u * g;   // its two rows
    const uint32_t k_blk = krow + (uint32_t)((one_k ? 0 : h * R) + r) * L::kRows, k_off = k_blk + 4u * g, k4_off = k_blk + 8u * c;
    const uint32_t mine = sm0 + L::warp(hg, qb, kb, hg * R) + (uint32_t)warp * L::kWarp, kept = mine + L::kKept + 16u * lane;

    float H[2][4], Cg[2][4], acc[2][4];    // state of the recomputation, carried dL/dH, dW
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int x = 0; x < 4; ++x) acc[nt][x] = Cg[nt][x] = 0.f;
    if (a.d_hT) {
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const float4 t4 = *reinterpret_cast<const float4 *>(a.d_hT + unit * KV + own + x * kV);
        Cg[0][2 * x] = t4.x; Cg[0][2 * x + 1] = t4.y; Cg[1][2 * x] = t4.z; Cg[1][2 * x + 1] = t4.w;
      }
    }
    const float clip = a.dh_clip;
    uint32_t ha[4], hb[4];      // H_t of the step at hand = H_{t-1} of the one done before, and that one's, in turn

    // checkpoints come by cp.async into the warp's own memory, a chunk ahead; each thread reads back what it fetched
    const float *ck = a.ckpt + (unit * a.nchunks + (nch > 0 ? nch - 1 : 0)) * KV + own;
    const uint32_t ck_sa = mine + 16u * lane;
    auto fetch_ckpt = [&](int j) {
      if constexpr (PER > 1) ck = a.ckpt + (unit * a.nchunks + PER * (nch - 1 - j)) * KV + own;
      cp16(ck_sa + 1024u * (j & 1), ck);
      cp16(ck_sa + 1024u * (j & 1) + 512u, ck + kV);
      if constexpr (PER == 1) ck -= KV;
    };
    auto take_ckpt = [&](int j) {
      asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const float4 t4 = lds128(ck_sa + 1024u * (j & 1) + 512u * x);
        H[0][2 * x] = t4.x; H[0][2 * x + 1] = t4.y; H[1][2 * x] = t4.z; H[1][2 * x + 1] = t4.w;
      }
    };

    // What a forward and a reverse step take from shared memory: `v`, `k`, `q` the thread's place in the step's rows
    struct RecIn { uint32_t k; uint2 v; float f; };
    struct RevIn { uint32_t q; uint2 dy, v; float2 f; uint4 h, z; };
    auto rec_in = [&](uint32_t k, uint32_t v) { return RecIn{ldsu32(k), ldsu64(v), lds32(v + L::kF)}; };
    auto rev_in = [&](uint32_t q, uint32_t v, uint32_t place) {
      return RevIn{ldsu32(q), ldsu64(v + L::kDy), ldsu64(v), lds64(v + L::kF), get128(place), get128(place + 512u)};
    };
    // One forward step of the recomputation in two halves (Eq. 1 up to the product; tanh and Eq. 2); leaves H_{t-1} and -Z_t at `place`
    auto rec_mma = [&](const RecIn &in, uint32_t place, float (&P)[2][4]) {
      uint32_t p[4];
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        p[2 * nt] = pack_bf16(H[nt][0], H[nt][1]); p[2 * nt + 1] = pack_bf16(H[nt][2], H[nt][3]);
        const uint32_t v = nt ? in.v.y : in.v.x;
        P[nt][0] = fma_bf16<0, 0>(in.k, v, 0.f); P[nt][1] = fma_bf16<0, 1>(in.k, v, 0.f);
        P[nt][2] = fma_bf16<1, 0>(in.k, v, 0.f); P[nt][3] = fma_bf16<1, 1>(in.k, v, 0.f);
      }
      mma_bf16_16816(P[0], p, Wr[0][0], Wr[0][1]);
      mma_bf16_16816(P[1], p, Wr[1][0], Wr[1][1]);
      put128(place, make_uint4(p[0], p[1], p[2], p[3]));
    };
    auto rec_gate = [&](const float (&P)[2][4], float f, uint32_t place) {
      const float2 f2 = make_float2(f, f), m1 = make_float2(-1.f, -1.f);
      uint32_t z[4];
#pragma unroll
      for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const float2 z2 = make_float2(tanh_approx(P[nt][2 * x]), tanh_approx(P[nt][2 * x + 1]));
          const float2 d2 = __ffma2_rn(z2, m1, make_float2(H[nt][2 * x], H[nt][2 * x + 1]));
          const float2 h2 = __ffma2_rn(f2, d2, z2);
          z[2 * nt + x] = pack_f16(-z2.x, -z2.y);
          H[nt][2 * x] = h2.x; H[nt][2 * x + 1] = h2.y;
        }
      put128(place + 512u, make_uint4(z[0], z[1], z[2], z[3]));
    };
    // A reverse step's chain: dX and the carried gradient; returns this thread's share of df.  hp: H_{t-1} as it was packed.
    auto rev_chain = [&](const RevIn &in, uint32_t (&hp)[4], uint32_t (&xp)[4]) -> float {
      const float2 f2 = make_float2(in.f.x, in.f.x), nomf2 = make_float2(in.f.y, in.f.y);
      const uint32_t z[4] = {in.z.x, in.z.y, in.z.z, in.z.w};
      hp[0] = in.h.x; hp[1] = in.h.y; hp[2] = in.h.z; hp[3] = in.h.w;
      float2 df2 = make_float2(0.f, 0.f);
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        const uint32_t dy = nt ? in.dy.y : in.dy.x;
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const float2 G2 = x ? make_float2(fma_bf16<1, 0>(in.q, dy, Cg[nt][2]), fma_bf16<1, 1>(in.q, dy, Cg[nt][3]))
                              : make_float2(fma_bf16<0, 0>(in.q, dy, Cg[nt][0]), fma_bf16<0, 1>(in.q, dy, Cg[nt][1]));   // G = C + q dy^T
          df2 = __ffma2_rn(G2, add_f16x2(z[2 * nt + x], unpack_bf16(hp[2 * nt + x])), df2);                              // df = sum G (.) (H_{t-1} - Z)
          const float2 x2 = __fmul2_rn(__fmul2_rn(nomf2, G2), square_f16x2(z[2 * nt + x], -1.f));                        // dX = (1-f) G (1 - Z^2)
          const float2 c2 = __fmul2_rn(f2, G2);                                                                          // gated path into H_{t-1}
          Cg[nt][2 * x] = c2.x; Cg[nt][2 * x + 1] = c2.y;
          xp[2 * nt + x] = pack_bf16(x2.x, x2.y);
        }
      }
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) mma_bf16_16816(Cg[nt], xp, WTr[nt][0], WTr[nt][1]);     // C_{t-1} = f G + dX W^T
      if constexpr (CLIP) {
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
          for (int x = 0; x < 4; ++x) Cg[nt][x] = fminf(fmaxf(Cg[nt][x], -clip), clip);
      }
      return df2.x + df2.y;
    };
    // What hangs on a reverse step: every column of dq and dk is the product
    struct Sums { float dq[4], dk[4], dv[4]; };
    auto rev_rest = [&](const RevIn &in, const uint32_t (&hn)[4], const uint32_t (&hp)[4], const uint32_t (&xp)[4], uint32_t k4, Sums &o) {
      mma_bf16_16816_zero(o.dk, xp, in.v.x, in.v.y);         // dk = dX v
      mma_bf16_16816_zero(o.dq, hn, in.dy.x, in.dy.y);       // dq = H_t dy
      const uint2 kw = ldsu64(k4);                           // rows 4c .. 4c + 3: MMA rows 2c, 8 + 2c, 2c + 1, 9 + 2c
      const uint32_t xt[4] = {transposed(xp[0]), transposed(xp[2]), transposed(xp[1]), transposed(xp[3])};
      const uint32_t ht[4] = {transposed(hp[0]), transposed(hp[1]), transposed(hp[2]), transposed(hp[3])};
      mma_bf16_16816_zero(o.dv, xt, __byte_perm(kw.x, kw.y, 0x5410), __byte_perm(kw.x, kw.y, 0x7632));   // dv = dX^T k
      mma_bf16_16816(acc[0], xt, ht[0], ht[1]);              // dW^T += dX^T H_{t-1}
      mma_bf16_16816(acc[1], xt, ht[2], ht[3]);
    };
    auto put_sums = [&](uint32_t o, const Sums &x) {
      if (c == 0) {
        sts64(o, make_float2(x.dq[0], x.dq[2]));
        sts64(o + L::kDk, make_float2(x.dk[0], x.dk[2]));
        sts64(o + L::kDv, make_float2(x.dv[0], x.dv[2]));
      }
    };

    if (nch > 0) {
      fetch_ckpt(0);
      if (!mbar_wait(&in_full[0], 0)) { report_timeout(a.dev_status); return; }
      take_ckpt(0);
      if (nch > 1) fetch_ckpt(1);
      const uint32_t sl = slot_sa(0);
      const int len = chunk_len(0);
#pragma unroll 1
      for (int s = 0; s < len; ++s) {
        float P[2][4];
        const RecIn in = rec_in(sl + k_off + 32u * s, sl + v_off + 32u * s);
        rec_mma(in, kept + 1024u * s, P);
        rec_gate(P, in.f, kept + 1024u * s);
      }
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) { hb[2 * nt] = pack_bf16(H[nt][0], H[nt][1]); hb[2 * nt + 1] = pack_bf16(H[nt][2], H[nt][3]); }
    }
    for (int j = 0; j < nch; ++j) {
      const bool more = j + 1 < nch;
      if (more && !mbar_wait(&in_full[(j + 1) % kRing], ((j + 1) / kRing) & 1)) { report_timeout(a.dev_status); return; }
      if (j >= 2 && !mbar_wait(&out_free[j & 1], ((j >> 1) - 1) & 1)) { report_timeout(a.dev_status); return; }
      const uint32_t sa = slot_sa(j), sb = slot_sa(j + 1);
      const uint32_t out = out0 + (uint32_t)((j & 1) * hg * R + warp) * L::kOut;
      const int len = chunk_len(j);
      if (more) {
        take_ckpt(j + 1);
        if (j + 2 < nch) fetch_ckpt(j + 2);
      }
      // Step s of an even chunk is kept at place s, of an odd one at C - s: the place that a forward step takes is the one that the
      // reverse step before it has left.
      const uint32_t dir = j & 1 ? 1024u : -1024u;             // from a reverse step's place to the next
      uint32_t pr = kept + 1024u * (j & 1 ? C - len + 1 : len - 1), pw = kept + 1024u * (j & 1 ? 0 : C);
      uint32_t rk = sb + k_off, rv = sb + v_off;               // the forward step's rows
      const uint32_t back = 32u * (len - 1);
      uint32_t eq = sa + q_off + back, ev = sa + v_off + back, ek = sa + k4_off + back;      // the reverse step's
      uint32_t eo = out + 8u * g + 64u * (len - 1), ed = mine + L::kShare + 4u * lane + 128u * (len - 1);
      if (more && len == C) {
        // A step's results are stored a step later, the forward step's loads are requested a step ahead, and each chain's
        // arithmetic covers the latency of the other's products.
        Sums sum;
        auto step = [&](const uint32_t (&hn)[4], uint32_t (&hp)[4], uint32_t u) {
          float P[2][4];
          uint32_t xp[4];
          const RevIn vi = rev_in(eq - 32u * u, ev - 32u * u, pr);
          const RecIn ri = rec_in(rk + 32u * u, rv + 32u * u);
          rec_mma(ri, pw, P);
          sts32(ed - 128u * u, rev_chain(vi, hp, xp));
          rev_rest(vi, hn, hp, xp, ek - 32u * u, sum);
          rec_gate(P, ri.f, pw);
          put_sums(eo - 64u * u, sum);
          pr += dir; pw += dir;
        };
#pragma unroll 1
        for (int i = 0; i < C; i += 2) {
          step(hb, ha, 0);
          step(ha, hb, 1);
          rk += 64u; rv += 64u; eq -= 64u; ev -= 64u; ek -= 64u; eo -= 128u; ed -= 256u;
        }
      } else {      // a ragged chunk or the last one
#pragma unroll 1
        for (int s = 0; s < len; ++s) {
          uint32_t xp[4];
          Sums sum;
          const RevIn vi = rev_in(eq, ev, pr);
          sts32(ed, rev_chain(vi, ha, xp));
          rev_rest(vi, hb, ha, xp, ek, sum);
          put_sums(eo, sum);
#pragma unroll
          for (int x = 0; x < 4; ++x) hb[x] = ha[x];
          pr += dir; eq -= 32u; ev -= 32u; ek -= 32u; eo -= 64u; ed -= 128u;
        }
        if (more) {
#pragma unroll 1
          for (int s = 0; s < C; ++s) {
            float P[2][4];
            const RecIn in = rec_in(rk, rv);
            rec_mma(in, pw, P);
            rec_gate(P, in.f, pw);
            rk += 32u; rv += 32u; pw += dir;
          }
        }
      }
      __syncwarp();
      for (int t = g; t < len; t += 8) {      // df: the lanes' shares, four lanes a step
        const float4 p = lds128(mine + L::kShare + 128u * t + 32u * c), p1 = lds128(mine + L::kShare + 128u * t + 32u * c + 16u);
        float d = ((p.x + p.y) + (p.z + p.w)) + ((p1.x + p1.y) + (p1.z + p1.w));
        const uint32_t who = 0xfu << (4 * g);
        d += __shfl_xor_sync(who, d, 1);
        d += __shfl_xor_sync(who, d, 2);
        if (c == 0) sts32(out + L::kOutDf + 4u * t, d);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&out_full[j & 1]);
    }
    if (a.dh0) {
#pragma unroll
      for (int x = 0; x < 2; ++x)
        *reinterpret_cast<float4 *>(a.dh0 + unit * KV + own + x * kV) = make_float4(Cg[0][2 * x], Cg[0][2 * x + 1], Cg[1][2 * x], Cg[1][2 * x + 1]);
    }
    // dW of the CTA's slabs of a head: through the warps' own memory, added by the head's first warp
    const uint32_t part = mine + 16u * lane;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) sts128(part + 512u * nt, make_float4(acc[nt][0], acc[nt][1], acc[nt][2], acc[nt][3]));
    __syncwarp();
    if (lane == 0) mbar_arrive(dw_full);
    if (r == 0 && R > 1 && !mbar_wait(dw_full, 0)) { report_timeout(a.dev_status); return; }
    if (r == 0) {
      float *dst = a.dW_part + ((size_t)(b * RS + rs) * N + n) * kV * kV;
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        float4 s4 = make_float4(acc[nt][0], acc[nt][1], acc[nt][2], acc[nt][3]);
        for (int x = 1; x < R; ++x) {
          const float4 o = lds128(part + (uint32_t)x * L::kWarp + 512u * nt);
          s4.x += o.x; s4.y += o.y; s4.z += o.z; s4.w += o.w;
        }
        // (the product's rows g, g + 8 are state columns j, its columns 8 nt + 2c, + 1 state columns l)
        using G = TileGeom<kV>;
        const int l = G::mem_col(8 * nt + 2 * c), j0 = G::mem_col(g), j1 = G::mem_col(g + 8);
        dst[l * kV + j0] = s4.x; dst[(l + 1) * kV + j0] = s4.y; dst[l * kV + j1] = s4.z; dst[(l + 1) * kV + j1] = s4.w;
      }
    }
    return;
  }

  const int hq = n0 / (N / a.Nq), hk = n0 / (N / a.Nk);      // the first head's q and k heads
  if (warp == hg * R) {
    // ================================================================= loader warp
    // A lane's requests: 16-byte half lane % 2 of head or slab 2 i + lane / 2 % 2 at step lane / 4 (+ 8).
    constexpr int kPairs = kMostSlabs / 2, kGates = (kMostSlabs + 3) / 4, kOct = CC / 8;
    const int half = lane & 1, sub = (lane >> 1) & 1, t4 = lane >> 2;
    const uint32_t dst0 = 32u * t4 + 16u * half;
    const __nv_bfloat16 *vg = static_cast<const __nv_bfloat16 *>(a.v) + tok0 * a.vs + (n0 + sub) * kV + 8 * half;
    const __nv_bfloat16 *dyg = static_cast<const __nv_bfloat16 *>(a.dy) + (tok0 * N + n0 + sub) * kV + 8 * half;
    const __nv_bfloat16 *qg = static_cast<const __nv_bfloat16 *>(a.q) + tok0 * a.qs + hq * K + rbase + 8 * half;
    const __nv_bfloat16 *kg = static_cast<const __nv_bfloat16 *>(a.k) + tok0 * a.ks + hk * K + rbase + 8 * half;
    const int qblocks = one_q ? R : slabs, kblocks = one_k ? R : slabs;
    int blk_at[kPairs];       // where slab 2 i + sub's rows begin among a token's q (k)
#pragma unroll
    for (int i = 0; i < kPairs; ++i) blk_at[i] = (2 * i + sub) / R * K + (2 * i + sub) % R * 16;
    // gates: step lane % 8 (+ 8) of head lane / 8 + 4 i
    const int t8 = lane & 7, h8 = lane >> 3;
    float graw[kOct][kGates], al[kGates], be[kGates];
#pragma unroll
    for (int i = 0; i < kGates; ++i) {
      const int h = h8 + 4 * i;
      al[i] = a.alpha && h < nh ? a.alpha[n0 + h] : 1.f;
      be[i] = a.beta && h < nh ? a.beta[n0 + h] : 0.f;
    }
    auto fetch_gates = [&](int j) {
      const int t0 = chunk_t0(j), len = chunk_len(j);
#pragma unroll
      for (int u = 0; u < kOct; ++u)
#pragma unroll
        for (int i = 0; i < kGates; ++i)
          graw[u][i] = t8 + 8 * u < len && h8 + 4 * i < nh ? a.gate[(tok0 + t0 + t8 + 8 * u) * N + n0 + h8 + 4 * i] : 0.f;
    };
    if (nch > 0) fetch_gates(0);
    for (int j = 0; j < nch; ++j) {
      if (j >= kRing && !mbar_wait<200>(&slot_free[j % kRing], ((j / kRing) - 1) & 1)) { report_timeout(a.dev_status); return; }
      const uint32_t sl = slot_sa(j);
      const int t0 = chunk_t0(j), len = chunk_len(j);
#pragma unroll
      for (int u = 0; u < kOct; ++u) {
        const int t = t4 + 8 * u;
        if (t < len) {
          const size_t at = (size_t)(t0 + t);
          const __nv_bfloat16 *vs = vg + at * a.vs, *ds = dyg + at * N * kV, *qs = qg + at * a.qs, *ks = kg + at * a.ks;
          const uint32_t dst = sl + dst0 + 256u * u;
#pragma unroll
          for (int i = 0; i < kPairs; ++i) {
            if (2 * i + sub < nh) {
              cp16(dst + (2u * i + sub) * L::kHead, vs + 2 * i * kV);
              cp16(dst + (2u * i + sub) * L::kHead + L::kDy, ds + 2 * i * kV);
            }
            if (2 * i + sub < qblocks) cp16(dst + qrow + (2u * i + sub) * L::kRows, qs + blk_at[i]);
            if (2 * i + sub < kblocks) cp16(dst + krow + (2u * i + sub) * L::kRows, ks + blk_at[i]);
          }
        }
      }
      cp_arrive(&in_full[j % kRing]);
#pragma unroll
      for (int u = 0; u < kOct; ++u)
#pragma unroll
        for (int i = 0; i < kGates; ++i) {
          if (h8 + 4 * i >= nh || t8 + 8 * u >= len) continue;
          float dfdx;
          const float f = gate_value(a.gate_kind, graw[u][i], al[i], be[i], &dfdx);
          const int t = t8 + 8 * u;
          const uint32_t hd = sl + (uint32_t)(h8 + 4 * i) * L::kHead;
          const float4 f4 = make_float4(f, f - 1.f, f, f - 1.f);
          sts128(hd + L::kF + 32u * t, f4);
          sts128(hd + L::kF + 32u * t + 16u, f4);
          sts32(hd + L::kDf + 4u * t, dfdx);
        }
      if (j + 1 < nch) fetch_gates(j + 1);
      __syncwarp();
      if (lane == 0) mbar_arrive(&in_full[j % kRing]);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    return;
  }

  // =================================================================== writer warp
  // A round of the warp is a slab's 16 rows or a head's 16 columns at eight steps: four entries a lane.
  const int quad = lane & 3, t4 = lane >> 2, t8 = lane & 7, h8 = lane >> 3;
  const __nv_bfloat16 *wr = rs == 0 ? static_cast<const __nv_bfloat16 *>(a.w_r) : nullptr;
  const size_t BT = (size_t)a.TT;
  for (int j = 0; j < nch; ++j) {
    if (!mbar_wait<200>(&out_full[j & 1], (j >> 1) & 1)) { report_timeout(a.dev_status); return; }
    const uint32_t out = out0 + (uint32_t)((j & 1) * hg * R) * L::kOut, sl = slot_sa(j);
    const int t0 = chunk_t0(j), len = chunk_len(j);
    for (int u = 0; 8 * u < len; ++u) {
      const int t = t4 + 8 * u;
      const size_t tok = tok0 + t0 + t;
      if (t < len) {
        const uint32_t src = out + 64u * t + 16u * quad;
        // (four blocks at a time: their loads travel together)
        auto add = [](float4 &x, const float4 &y) { x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w; };
        // dq, dk, summed over the CTA's heads where they share them
        auto rows_out = [&](uint32_t off, bool one, float *part, void *whole, int heads, int h0) {
          const int blocks = one ? R : slabs;      // (head, slab)
          for (int x0 = 0; x0 < blocks; x0 += 4) {
            float4 s4[4];
#pragma unroll
            for (int y = 0; y < 4; ++y) s4[y] = lds128(src + off + (uint32_t)min(x0 + y, blocks - 1) * L::kOut);
            if (one)
              for (int h = 1; h < nh; ++h)
#pragma unroll
                for (int y = 0; y < 4; ++y) add(s4[y], lds128(src + off + (uint32_t)(h * R + min(x0 + y, R - 1)) * L::kOut));
#pragma unroll
            for (int y = 0; y < 4; ++y) {
              if (x0 + y >= blocks) break;
              const int h = one ? 0 : (x0 + y) / R, i = rbase + 16 * (x0 + y - h * R) + 4 * quad;
              if (part) *reinterpret_cast<float4 *>(part + (tok * a.groups + grp) * K + i) = s4[y];
              else *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(whole) + (tok * heads + h0 + h) * K + i) = make_uint2(pack_bf16(s4[y].x, s4[y].y), pack_bf16(s4[y].z, s4[y].w));
            }
          }
        };
        rows_out(0, one_q, a.dq_part, a.dq, a.Nq, hq);
        rows_out(L::kDk, one_k, a.dk_part, a.dk, a.Nk, hk);
        // dv (+ w_r (.) dy from Eq. 3, added by the first row slab only)
        for (int x0 = 0; x0 < nh; x0 += 4) {
          float4 f4[4];
#pragma unroll
          for (int y = 0; y < 4; ++y) f4[y] = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int r = 0; r < R; ++r)
#pragma unroll
            for (int y = 0; y < 4; ++y) add(f4[y], lds128(src + L::kDv + (uint32_t)(min(x0 + y, nh - 1) * R + r) * L::kOut));
#pragma unroll
          for (int y = 0; y < 4; ++y) {
            const int h = x0 + y;
            if (h >= nh) break;
            float4 s4 = make_float4(f4[y].x, f4[y].z, f4[y].y, f4[y].w);     // (the fragments' order: columns 0, 2, 1, 3 of a quad)
            if (wr) {
              const uint2 w4 = *reinterpret_cast<const uint2 *>(wr + (size_t)(n0 + h) * kV + 4 * quad);
              const uint2 d4 = ldsu64(sl + (uint32_t)h * L::kHead + L::kDy + 32u * t + 8u * quad);
              const float2 w0 = unpack_bf16(w4.x), w1 = unpack_bf16(w4.y), d0 = unpack_bf16(d4.x), d1 = unpack_bf16(d4.y);
              s4.x = fmaf(w0.x, d0.x, s4.x); s4.y = fmaf(w0.y, d0.y, s4.y); s4.z = fmaf(w1.x, d1.x, s4.z); s4.w = fmaf(w1.y, d1.y, s4.w);
            }
            const size_t o = (tok * N + n0 + h) * kV + 4 * quad;
            if (a.dv_part) *reinterpret_cast<float4 *>(a.dv_part + (size_t)rs * BT * N * kV + o) = s4;
            else *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(a.dv) + o) = make_uint2(pack_bf16(s4.x, s4.y), pack_bf16(s4.z, s4.w));
          }
        }
      }
      const int td = t8 + 8 * u;
      if (td < len)
        for (int h = h8; h < nh; h += 4) {
          float s = 0.f;
          for (int r = 0; r < R; ++r) s += lds32(out + (uint32_t)(h * R + r) * L::kOut + L::kOutDf + 4u * td);
          s *= lds32(sl + (uint32_t)h * L::kHead + L::kDf + 4u * td);
          const size_t o = (tok0 + t0 + td) * N + n0 + h;
          if (a.dgate_part) a.dgate_part[(size_t)rs * BT * N + o] = s;
          else a.dgate[o] = s;
        }
    }
    __syncwarp();
    if (lane == 0) { mbar_arrive(&out_free[j & 1]); mbar_arrive(&slot_free[j % kRing]); }
  }
}

template <int CC, bool CLIP, int PER>
cudaError_t launch_t(const ScanArgs &a, cudaStream_t s) {
  const int R = a.KC / 16, qb = a.Nq < a.N ? R : a.hg * R, kb = a.Nk < a.N ? R : a.hg * R;
  const size_t smem = Lay<CC>::total(a.hg, qb, kb, a.hg * R);
  const cudaError_t e = allow_smem(bwd_v16_kernel<CC, CLIP, PER>, smem);
  if (e != cudaSuccess) return e;
  const int ctas = a.B * a.groups * (a.K / a.KC), threads = (a.hg * R + 2) * 32;
  return launch_early(bwd_v16_kernel<CC, CLIP, PER>, ctas, threads, smem, s, in_order(a, ctas, threads, 2));
}

}  // namespace

// What a chunk of a V = 16 problem's backward looks like: slabs and heads of a CTA, steps of a chunk.
//
// A step costs what its busiest scheduler's slab warps cost (ns; one CTA with the SM to itself, 2 048 steps): one slab 239, four
// 259, six 355, eight 382, ten 424, with chunks of 16 steps some 20 less; where heads do not share q and k the service warps have
// a head's rows for each slab: eight 494.  Fewer CTAs than SMs want small ones, more want ten slabs each: 336 units of K = 64
// run as 136 CTAs of 5 heads and two slabs in one wave (1 024 steps 452 us; 336 CTAs of four slabs 644, 1 344 of one slab 687).
// Heads of a CTA that share q and k leave one share of dq and dk, slabs of a CTA one of dv and dgate: the shares' way through
// memory counts too, and the two launches that add the slabs' shares.
// Two plans are looked for, of whole states (a CTA has all slabs of its heads) and of split ones, and T decides between them: the two
// launches that add the slabs' shares count 5 us of a call.  That keeps the short calls whole and is late for some (backward, us, whole /
// split: B 6, 8 heads, K = 64, T 32 17.9 / 19.0, 128 42.8 / 40.1, 512 144 / 128, split from 322 on; B 1, 57 heads with k of their own, T 64
// 29.2 / 30.5, 256 76.1 / 74.4, 512 140.5 / 133.8, split from 341 on).  The checkpoints' interval must not
// follow T -- a buffer for the longest sequence has to do for every shorter one, and the interval is asked for without a T --, so it is
// eight steps where either plan has chunks of eight, and a chunk of sixteen then begins at every second checkpoint (B 2, 84
// heads sharing q and k, K = 64, 768 steps: forward 102 -> 105, backward 262; in chunks of eight 307).
BwdPlan plan_bwd_v16(int B, int N, int Nq, int Nk, int K, int T, int interval, bool lean) {
  const int sms = sm_count();
  // heads that a CTA's are taken from: those that share a q and a k head (where heads share at all)
  const int set = std::gcd(Nq < N ? N / Nq : N, Nk < N ? N / Nk : N);
  const bool own_rows = Nq == N || Nk == N;
  BwdPlan whole{}, split{};
  double whole_cost = 0., split_cost = 0.;
  const int choices[2] = {interval ? interval : 8, 16};
  for (int x = 0; x < (interval ? 1 : 2); ++x)
    for (int R = 1; R <= K / 16 && R <= kMostSlabs; ++R)
      for (int hg = 1; K / 16 % R == 0 && hg * R <= kMostSlabs && hg <= set; ++hg) {
        const int C = choices[x], groups = N / set * ((set + hg - 1) / hg), slabs = hg * R, qb = Nq < N ? R : slabs, kb = Nk < N ? R : slabs;
        const long ctas = (long)(B > 0 ? B : 1) * groups * (K / (16 * R));
        const size_t smem = (C <= 8 ? Lay<8>::total(hg, qb, kb, slabs) : Lay<16>::total(hg, qb, kb, slabs)) + 1024;
        constexpr size_t kSm = 228 * 1024;
        const long by_regs = kRoomWarps / (slabs + 2), by_smem = (long)(kSm / smem), room = by_regs < by_smem ? by_regs : by_smem;
        if (room < 1 || smem - 1024 > 227 * 1024) continue;
        auto step = [&](long n) {     // of an SM with n CTAs
          const long s = n * slabs;
          return n ? 155. + 100. * ((s + 3) / 4) + 4. * s + (C <= 8 ? 20. : 0.) + (own_rows ? 12. * (s > 4 ? s - 4 : 0) + 4. * (slabs - 1) : 0.) : 0.;
        };
        const long waves = ctas / (sms * room), left = ctas % (sms * room);
        const int RS = K / (16 * R);
        double cost = waves * step(room) + step((left + sms - 1) / sms);
        cost += ((Nq < groups ? 1 : 0) + (Nk < groups ? 1 : 0)) * 8. * B * groups * K / 5500. + (RS > 1 ? 128. * B * N * RS / 5500. : 0.);
        BwdPlan &best = RS > 1 ? split : whole;
        double &best_cost = RS > 1 ? split_cost : whole_cost;
        const bool better = !best.KC || (lean ? 16 * R > best.KC || (16 * R == best.KC && hg > best.hg) : cost < best_cost);
        if (!better) continue;
        best_cost = cost;
        best.KC = 16 * R; best.C = C; best.hg = hg; best.groups = groups; best.set = set;
      }
  whole.T_from = 1;
  if (split.KC) {
    const double gain = whole_cost - split_cost, from = gain > 0. ? 5000. / gain : 1e9;    // (ns a step)
    split.T_from = lean || from > 1e9 - 1. ? INT_MAX : (int)from + 1;
    if (!whole.KC) split.T_from = 1;
  }
  const bool take_split = split.KC && (T > 0 ? T : 1) >= split.T_from;
  BwdPlan best = take_split ? split : whole;
  best.interval = interval ? interval : whole.KC && split.KC && !lean ? std::min(whole.C, split.C) : best.C;
  best.C_max = 16;
  return best;
}

cudaError_t launch_bwd_v16(const ScanArgs &a, cudaStream_t s) {
  const bool clip = a.dh_clip > 0.f;
  if (a.C <= 8) return clip ? launch_t<8, true, 1>(a, s) : launch_t<8, false, 1>(a, s);
  if (a.per == 2) return clip ? launch_t<16, true, 2>(a, s) : launch_t<16, false, 2>(a, s);
  return clip ? launch_t<16, true, 1>(a, s) : launch_t<16, false, 1>(a, s);
}

}  // namespace m2rnn
