// bf16 tensor-core forward scan (Algorithm 1) for V = 16, the state size of the paper's own layers.
//
// One CTA per (b, n, row slab group); below, K is the group's row count.  A chain warp owns 16 state rows for
// all T steps: Eq. 1's product is two mma.sync.m16n8k16 whose A operand is the state as packed at the end of
// the step before and whose accumulators start as the outer product.  With so little arithmetic per
// step the scan is the latency of that chain (MMA, tanh, gate, pack), so nothing else may sit in it:
//   - the readout (Eq. 3) is the service warps' work: a chain warp leaves its packed H_t as a tile in the stage,
//     and the service warps form y_t = H_t^T q_t for a finished stage on the tensor cores (ldmatrix.trans
//     turns the tiles into B operands, q is row 0 of A, all slabs of a step add into one accumulator);
//   - k, v and q travel from memory to the stage as they are (cp.async, no registers and no waiting in
//     between); gates are evaluated for 8 or 16 stages at a time, a lane each.
// Stages of kTC steps are handed over by mbarriers; every wait is bounded and reports through
// dev_status.
// (One service warp that fetched and widened a stage when it was free, readout in the chain warps: 84 heads,
// K = 64, batch 1, 2 and 4 took 120, 161 and 191 ns per step; then 99, 133 and 179; now, with seeds straight from bf16
// (fma.f32.bf16: no unpacking) and half slabs where a CTA has its SM to itself, 94, 126 and 174.  What counted, in order: the
// service warps' time per stage, which was longer than the chain's; with three CTAs per SM the
// shared-memory traffic -- k and v as fp32, f per row, cost 10 %.)
#include "device_common.cuh"
#include "internal.h"
#include "mma_tile.cuh"
#include "pipeline.cuh"
#include "tile.cuh"

namespace m2rnn {
namespace {

constexpr int kV = 16;
constexpr int kTC = 8;          // steps of a stage
constexpr int kStages = 3;
constexpr int kBarBytes = 64;

struct Lay16 {                  // byte offsets inside a stage: H_t tiles [8][K/16] x 512, then k, q [8][K] and v [8][16] as they are, f [8]
  __host__ __device__ static constexpr uint32_t a() { return 0; }
  __host__ __device__ static constexpr uint32_t k(int K) { return kTC * K * 32; }
  __host__ __device__ static constexpr uint32_t q(int K) { return k(K) + kTC * K * 2; }
  __host__ __device__ static constexpr uint32_t v(int K) { return q(K) + kTC * K * 2; }
  __host__ __device__ static constexpr uint32_t f(int K) { return v(K) + kTC * kV * 2; }
  __host__ __device__ static constexpr uint32_t bytes(int K) { return f(K) + kTC * 4; }
};

__device__ __forceinline__ float lds_bf16(uint32_t addr) {
  uint16_t x;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(x) : "r"(addr));
  return __uint_as_float((uint32_t)x << 16);
}

// byte offset of eight-column chunk `chunk` of row `row` of a slab's H_t tile, [16 rows][16 columns] bf16:
// chunks swapped in every other group of four rows, so that the eight rows of an ldmatrix cover all banks
__device__ __forceinline__ uint32_t tile16_off(int row, int chunk) { return (uint32_t)(row * 32 + ((chunk ^ ((row >> 2) & 1)) << 4)); }

// NW: slabs of the CTA, a chain warp each, or two of eight rows (HALF).  kSvc service warps: four (one per scheduler, two steps of a stage each)
// where a CTA has the SM to itself and their latency counts, two (four steps each) where several CTAs
// share it and their instructions do.
template <int NW, bool CKPT, int OCC, int kSvc, bool HALF>
__global__ void __launch_bounds__(((HALF ? 2 : 1) * NW + kSvc) * 32, OCC) fwd_v16_kernel(ScanArgs a) {
  constexpr int CW = HALF ? 2 * NW : NW, NH = HALF ? 1 : 2;      // chain warps; rows of a thread
  constexpr int K = 16 * NW, kMine = kTC / kSvc, kBlk = 32 / kMine;   // steps of a stage per service warp; stages of a block of gates
  static_assert(kMine * K / 8 <= 32, "a lane stages eight entries of k");
  extern __shared__ __align__(16) unsigned char smem[];
  begin_dependent();
  const int Kf = a.K, N = a.N, RS = Kf / K;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31, g = lane >> 2, c = lane & 3;
  const int place = blockIdx.x / RS, rs = blockIdx.x % RS, rbase = rs * K;
  const int b = batch_entry(a, place / N, smem), n = place % N, bn = b * N + n;
  const UnitSpan span = unit_span(a, b);
  const int T = span.T, nst = (T + kTC - 1) / kTC;
  const size_t tok0 = span.tok0, KV = (size_t)Kf * kV;
  uint64_t *full = reinterpret_cast<uint64_t *>(smem), *done = full + kStages;
  const uint32_t st0 = smem_u32(smem) + kBarBytes;
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(&full[s], 33 * kSvc); mbar_init(&done[s], CW); }
    fence_mbar_init();
  }
  __syncthreads();

  if (warp >= CW) {
    // ------------------------------------------------------------------ service warps
    // Warp sw takes steps sw, sw + kSvc, .. of every stage, for staging and readout alike: it overwrites only q and
    // v that it alone reads (the chain warps are through with a stage when it is done, and write
    // fragments into it only when all service warps have filled it).
    const int sw = warp - CW;
    const int hq = n / (N / a.Nq), hk = n / (N / a.Nk);
    const float al = a.alpha ? a.alpha[n] : 1.f, be = a.beta ? a.beta[n] : 0.f;
    const bool want_y = a.y != nullptr;
    // this lane's share of a stage: eight entries of k and of q of one step, eight of v; all addresses walk
    const bool has_k = lane < kMine * K / 8, has_v = lane < 2 * kMine;
    const int kt = sw + kSvc * (lane / (K / 8)), kj = (lane % (K / 8)) * 8, vt = sw + kSvc * (lane >> 1), vj = (lane & 1) * 8;
    const __nv_bfloat16 *kp = static_cast<const __nv_bfloat16 *>(a.k) + (tok0 + kt) * a.ks + hk * Kf + rbase + kj;
    const __nv_bfloat16 *qp = static_cast<const __nv_bfloat16 *>(a.q) + (tok0 + kt) * a.qs + hq * Kf + rbase + kj;
    const __nv_bfloat16 *vp = static_cast<const __nv_bfloat16 *>(a.v) + (tok0 + vt) * a.vs + n * kV + vj;
    int tk = kt, tv = vt;          // the steps that the pointers are at
    // The gates of this warp's steps of kBlk stages at a time, a lane each.  Raw values of the next block are
    // fetched a block ahead.
    int tg = sw + kSvc * (lane % kMine) + kTC * (lane / kMine);
    const float *gp = a.gate + (tok0 + tg) * N + n;
    float graw = tg < T ? *gp : 0.f, fblk = 0.f;
    auto next_gates = [&]() {
      fblk = gate_value(a.gate_kind, graw, al, be, nullptr);
      gp += (size_t)kBlk * kTC * N; tg += kBlk * kTC;
      if (tg < T) graw = *gp;
    };
    const uint32_t kdst = Lay16::k(K) + 2u * (uint32_t)(kt * K + kj), vdst = Lay16::v(K) + 2u * (uint32_t)(vt * kV + vj);
    // requests stage st into slot s; the slot is full when every lane's copies have landed and the gates are in
    auto fill = [&](int st, int s) {
      const uint32_t sa = st0 + (uint32_t)s * Lay16::bytes(K);
      if (has_k && tk < T) {
        cp16(sa + kdst, kp);
        if (want_y) cp16(sa + kdst + (Lay16::q(K) - Lay16::k(K)), qp);
      }
      if (has_v && tv < T) cp16(sa + vdst, vp);
      cp_arrive(&full[s]);
      kp += kTC * a.ks; qp += kTC * a.qs; vp += kTC * a.vs;
      tk += kTC; tv += kTC;
      if (st % kBlk == 0) next_gates();
      const float f = __shfl_sync(0xffffffffu, fblk, kMine * (st % kBlk) + lane % kMine);
      if (lane < kMine) sts32(sa + Lay16::f(K) + 4u * (uint32_t)(sw + kSvc * lane), f);
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[s]);
    };
    const bool has_wr = a.w_r && rs == 0;
    float wr0 = 0.f, wr1 = 0.f;    // of columns g and g + 8
    if (has_wr) {
      const __nv_bfloat16 *wr = static_cast<const __nv_bfloat16 *>(a.w_r) + (size_t)n * kV + g;
      wr0 = __bfloat162float(wr[0]); wr1 = __bfloat162float(wr[8]);
    }
    // ldmatrix: lane supplies row lane % 8 of matrix lane / 8: (rows 0-7, columns 0-7), (0-7, 8-15), (8-15, 0-7), (8-15, 8-15)
    const uint32_t ld_off = Lay16::a() + tile16_off((lane & 7) + 8 * (lane >> 4), (lane >> 3) & 1);
    const uint32_t lq_off = Lay16::q(K) + 16u * (lane >> 3);     // q: matrix m = entries 8m .. 8m+7, the same in all rows
    // y of this warp's steps goes out in pieces of eight columns, one per lane, through shared memory
    const uint32_t ybuf = st0 + kStages * Lay16::bytes(K) + 64u * kMine * sw;
    const size_t ystep = (size_t)N * kV;    // elements between tokens of y
    const bool has_y = lane < 2 * kMine;
    int ty = sw + kSvc * (lane >> 1);
    const size_t yat = (tok0 + ty) * ystep + n * kV + 8 * (lane & 1);
    __nv_bfloat16 *yg = static_cast<__nv_bfloat16 *>(a.y) + yat;
    float *yp = a.y_part ? a.y_part + (size_t)rs * a.TT * ystep + yat : nullptr;
    for (int st = 0; st < kStages && st < nst; ++st) fill(st, st);
#pragma unroll 1
    for (int st = 0, s = 0, par = 0; st < nst; ++st) {
      if (!mbar_wait(&done[s], par)) { report_timeout(a.dev_status); return; }
      if (want_y) {
        const uint32_t sa = st0 + (uint32_t)s * Lay16::bytes(K);
        // y^T = H_t^T q: the slab's tile, read transposed, is A (its rows the state's columns), q every column
        // of B, so that every column of the product is y
        float Y[kMine][4];
#pragma unroll
        for (int i = 0; i < kMine; ++i) Y[i][0] = Y[i][1] = Y[i][2] = Y[i][3] = 0.f;
#pragma unroll
        for (int w = 0; w < NW; w += 2)
#pragma unroll
          for (int i = 0; i < kMine; ++i) {
            const int t = sw + kSvc * i;
            uint32_t A[4], Q[4];
            ldmatrix_x4(sa + lq_off + 2u * (uint32_t)(t * K + 16 * w), Q);      // q of slabs w and w + 1 (past the last: unused)
            ldmatrix_x4_trans(sa + ld_off + 512u * (uint32_t)(t * NW + w), A[0], A[1], A[2], A[3]);
            mma_bf16_16816(Y[i], A, Q[0], Q[1]);
            if (w + 1 < NW) {
              ldmatrix_x4_trans(sa + ld_off + 512u * (uint32_t)(t * NW + w + 1), A[0], A[1], A[2], A[3]);
              mma_bf16_16816(Y[i], A, Q[2], Q[3]);
            }
          }
        if (c == 0) {   // columns g and g + 8 of y
#pragma unroll
          for (int i = 0; i < kMine; ++i) {
            if (has_wr) {
              const uint32_t vs = sa + Lay16::v(K) + 2u * (uint32_t)((sw + kSvc * i) * kV + g);
              Y[i][0] = fmaf(wr0, lds_bf16(vs), Y[i][0]);
              Y[i][2] = fmaf(wr1, lds_bf16(vs + 16u), Y[i][2]);
            }
            sts32(ybuf + 4u * (uint32_t)(16 * i + g), Y[i][0]);
            sts32(ybuf + 4u * (uint32_t)(16 * i + g + 8), Y[i][2]);
          }
        }
        __syncwarp();
        if (has_y && ty < T) {
          const float4 lo = lds128(ybuf + 32u * lane), hi = lds128(ybuf + 32u * lane + 16u);
          if (yp) {
            *reinterpret_cast<float4 *>(yp) = lo;
            *reinterpret_cast<float4 *>(yp + 4) = hi;
          } else {
            *reinterpret_cast<uint4 *>(yg) = make_uint4(pack_bf16(lo.x, lo.y), pack_bf16(lo.z, lo.w), pack_bf16(hi.x, hi.y), pack_bf16(hi.z, hi.w));
          }
        }
        ty += kTC;
        yg += kTC * ystep;
        if (yp) yp += kTC * ystep;
      }
      if (st + kStages < nst) {
        __syncwarp();
        fill(st + kStages, s);
      }
      if (++s == kStages) { s = 0; par ^= 1; }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    return;
  }

  // -------------------------------------------------------------------- chain warps
  // rows of this thread: row0 and row0 + 1 are MMA rows g and g + 8, or (HALF) row0 is MMA row g of a product whose other eight rows are
  // zero; columns 4c .. 4c+3
  const int row0 = HALF ? 8 * warp + g : 16 * warp + 2 * g;
  uint32_t Wr[2][2];
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
    load_w_fragment<kV>(static_cast<const __nv_bfloat16 *>(a.W) + (size_t)n * kV * kV, 0, nt, lane, Wr[nt][0], Wr[nt][1]);
  float H[2][4];   // H[nt] = {row0: columns 2nt, 2nt+1 of the four | row0 + 1: same}
  const size_t own = (size_t)(rbase + row0) * kV + 4 * c;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float4 t4 = h < NH && a.h0 ? *reinterpret_cast<const float4 *>(a.h0 + bn * KV + own + h * kV) : make_float4(0.f, 0.f, 0.f, 0.f);
    H[0][2 * h] = t4.x; H[0][2 * h + 1] = t4.y; H[1][2 * h] = t4.z; H[1][2 * h + 1] = t4.w;
  }
  auto store_state = [&](float *dst) {
#pragma unroll
    for (int h = 0; h < NH; ++h)
      *reinterpret_cast<float4 *>(dst + own + h * kV) = make_float4(H[0][2 * h], H[0][2 * h + 1], H[1][2 * h], H[1][2 * h + 1]);
  };
  // this lane's eight bytes of its rows in a slab's tile
  const int slab = HALF ? warp >> 1 : warp, trow = HALF ? row0 & 15 : 2 * g;
  const uint32_t hoff0 = tile16_off(trow, c >> 1) + 8u * (c & 1), hoff1 = tile16_off((trow + 1) & 15, c >> 1) + 8u * (c & 1);
  auto pack = [&](uint32_t (&A)[4]) {
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) { A[2 * nt] = pack_bf16(H[nt][0], H[nt][1]); A[2 * nt + 1] = HALF ? 0u : pack_bf16(H[nt][2], H[nt][3]); }
  };
  // P <- k v^T (the accumulators of a step), straight from bf16
  auto seed = [&](float (&P)[2][4], uint32_t kp, uint32_t vp) {
    uint32_t kk, v0, v1;
    if constexpr (HALF) { uint16_t x; asm volatile("ld.shared.u16 %0, [%1];" : "=h"(x) : "r"(kp)); kk = x; }
    else asm volatile("ld.shared.b32 %0, [%1];" : "=r"(kk) : "r"(kp));
    asm volatile("ld.shared.v2.b32 {%0,%1}, [%2];" : "=r"(v0), "=r"(v1) : "r"(vp));
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      const uint32_t v = nt ? v1 : v0;
      P[nt][0] = fma_bf16<0, 0>(kk, v, 0.f); P[nt][1] = fma_bf16<0, 1>(kk, v, 0.f);
      if constexpr (HALF) { P[nt][2] = P[nt][3] = 0.f; }
      else { P[nt][2] = fma_bf16<1, 0>(kk, v, 0.f); P[nt][3] = fma_bf16<1, 1>(kk, v, 0.f); }
    }
  };
  // One step.  Pc: H_{t-1} W + k_t v_t^T; Pn: k_{t+1} v_{t+1}^T on entry, that plus H_t W on exit.
  auto step = [&](float (&Pc)[2][4], float (&Pn)[2][4], float f, uint32_t adst) {
    const float2 f2 = make_float2(f, f), m1 = make_float2(-1.f, -1.f);
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        const float2 z = make_float2(tanh_approx(Pc[nt][2 * h]), tanh_approx(Pc[nt][2 * h + 1]));   // Eq. 1
        const float2 d = __ffma2_rn(z, m1, make_float2(H[nt][2 * h], H[nt][2 * h + 1]));            // H - Z
        const float2 hh = __ffma2_rn(f2, d, z);                                                     // Eq. 2
        H[nt][2 * h] = hh.x; H[nt][2 * h + 1] = hh.y;
      }
    uint32_t A[4];
    pack(A);
    mma_bf16_16816(Pn[0], A, Wr[0][0], Wr[0][1]);
    mma_bf16_16816(Pn[1], A, Wr[1][0], Wr[1][1]);
    asm volatile("st.shared.v2.b32 [%0], {%1,%2};" ::"r"(adst + hoff0), "r"(A[0]), "r"(A[2]) : "memory");
    if constexpr (!HALF) asm volatile("st.shared.v2.b32 [%0], {%1,%2};" ::"r"(adst + hoff1), "r"(A[1]), "r"(A[3]) : "memory");
  };

  float P0[2][4], P1[2][4];
  int ck_left = 0;   // steps until the next checkpoint
  float *ck_ptr = CKPT ? a.ckpt + (size_t)bn * a.nchunks * KV : nullptr;
  auto maybe_checkpoint = [&](int steps) {   // called before an even-numbered step
    if constexpr (CKPT) {
      if (ck_left == 0) {
        store_state(ck_ptr);
        ck_ptr += KV;
        ck_left = a.C;
      }
      ck_left -= steps;
    }
  };
  const uint32_t ok = Lay16::k(K) + 2u * (uint32_t)row0, ov = Lay16::v(K) + 8u * c, oa = Lay16::a() + 512u * (uint32_t)slab;
  constexpr uint32_t dk = 2u * K, dv = 2u * kV, da = 512u * NW;   // per step
  if (T > 0) {
    if (!mbar_wait(&full[0], 0)) { report_timeout(a.dev_status); return; }
    seed(P0, st0 + ok, st0 + ov);
    uint32_t A[4];
    pack(A);
    mma_bf16_16816(P0[0], A, Wr[0][0], Wr[0][1]);
    mma_bf16_16816(P0[1], A, Wr[1][0], Wr[1][1]);
  }
#pragma unroll 1
  for (int st = 0, s = 0; st < nst; ++st) {
    const uint32_t sa = st0 + (uint32_t)s * Lay16::bytes(K);
    const int sn = s + 1 == kStages ? 0 : s + 1;
    const int len = min(kTC, T - st * kTC);
    // what the stage's last step seeds: the next stage's first (after the last step: any valid row)
    uint32_t nx = sa;
    if (st + 1 < nst) {
      if (!mbar_wait(&full[sn], ((st + 1) / kStages) & 1)) { report_timeout(a.dev_status); return; }
      nx = st0 + (uint32_t)sn * Lay16::bytes(K);
    }
    if (len == kTC) {
      float f[kTC];
#pragma unroll
      for (int i = 0; i < kTC; i += 4) {
        const float4 f4 = lds128(sa + Lay16::f(K) + 4u * i);
        f[i] = f4.x; f[i + 1] = f4.y; f[i + 2] = f4.z; f[i + 3] = f4.w;
      }
#pragma unroll
      for (int t = 0; t < kTC; t += 2) {
        maybe_checkpoint(2);
        seed(P1, sa + ok + (t + 1) * dk, sa + ov + (t + 1) * dv);
        step(P0, P1, f[t], sa + oa + t * da);
        if (t + 2 < kTC) seed(P0, sa + ok + (t + 2) * dk, sa + ov + (t + 2) * dv);
        else seed(P0, nx + ok, nx + ov);
        step(P1, P0, f[t + 1], sa + oa + (t + 1) * da);
      }
    } else {   // ragged last stage
      for (int t = 0; t < len; ++t) {
        if ((t & 1) == 0) maybe_checkpoint(min(2, len - t));
        const int tn = min(t + 1, len - 1);
        seed(P1, sa + ok + tn * dk, sa + ov + tn * dv);
        step(P0, P1, lds32(sa + Lay16::f(K) + 4u * t), sa + oa + t * da);
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
          for (int r = 0; r < 4; ++r) P0[nt][r] = P1[nt][r];
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&done[s]);
    s = sn;
  }
  if (a.hT) store_state(a.hT + bn * KV);
}

template <int NW, bool CKPT, int OCC, bool HALF>
cudaError_t launch_t(const ScanArgs &a, cudaStream_t s) {
  constexpr int kSvc = OCC > 1 ? 2 : 4;
  constexpr size_t smem = kBarBytes + (size_t)kStages * Lay16::bytes(16 * NW) + kTC * kV * 4;
  const cudaError_t e = allow_smem(fwd_v16_kernel<NW, CKPT, OCC, kSvc, HALF>, smem);
  if (e != cudaSuccess) return e;
  const int ctas = a.B * a.N * (a.K / (16 * NW)), threads = ((HALF ? 2 : 1) * NW + kSvc) * 32;
  return launch_early(fwd_v16_kernel<NW, CKPT, OCC, kSvc, HALF>, ctas, threads, smem, s, in_order(a, ctas, threads, 1));
}

template <int NW, bool CKPT>
cudaError_t launch_o(const ScanArgs &a, cudaStream_t s) {
  // as many CTAs per SM as there are for each, up to three: the state is small, and e.g. the 336 units of
  // the paper's layer shape (84 heads x batch 4) then take one wave instead of two
  const long ctas = (long)a.B * a.N * (a.K / (16 * NW)), sms = sm_count();
  if constexpr (NW <= 4) {
    if (ctas > 2 * sms) return launch_t<NW, CKPT, 3, false>(a, s);
    if (ctas > sms) return launch_t<NW, CKPT, 2, false>(a, s);
  }
  // Alone on an SM, up to four slabs run as twice as many warps of eight rows each: half of a step's MMAs is zeros, but a warp's step
  // is its chain, and that is shorter by four tanh (1 024 steps, us: 16 heads of K = 64, a slab to an SM 94.9 -> 77.0, 84 heads, four
  // to an SM 98 -> 94; two CTAs of 168 heads to an SM 129 -> 145).
  return launch_t<NW, CKPT, 1, (NW <= 4)>(a, s);
}

}  // namespace

cudaError_t launch_fwd_v16(const ScanArgs &a, cudaStream_t s) {
  switch (a.KCf / 16) {
#define M2RNN_CASE(NW) case NW: return a.ckpt ? launch_o<NW, true>(a, s) : launch_o<NW, false>(a, s)
    M2RNN_CASE(1); M2RNN_CASE(2); M2RNN_CASE(3); M2RNN_CASE(4); M2RNN_CASE(5); M2RNN_CASE(6); M2RNN_CASE(7); M2RNN_CASE(8);
#undef M2RNN_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace m2rnn
