// bf16 tensor-core forward scan (Algorithm 1), column-split variant, for sm_100a.
//
// One CTA per (b, n, row slab group).  Every 16-row slab of the state is shared by SP = 2 or 4 chain
// warps, each owning V/SP of the columns, for all T steps.  A warp's step needs the whole slab as the A
// operand of H W: it has its own columns in registers, issues the MMAs of those at once, and gets the other
// warps' from the fragments of H_t that they all leave, one named barrier per slab and step.  A warp's part of W
// (V x V/SP) stays in registers.
// The scan is the latency of that chain, so nothing else sits in it: the fragments of a stage of TC steps stay in
// shared memory, and up to four service warps (one per scheduler) form y_t = H_t^T q_t (Eq. 3) of a finished
// stage from them on the tensor cores, bring q, k and v in with cp.async, and evaluate the gates
// of several stages at a time, a lane each.  Stages are handed over by mbarriers; every wait is bounded and
// reports through dev_status.
// (With the readout in the chain warps, as eight movmatrix and four MMAs of a step, 128 units of K = V = 64 took 658 us for
// 2048 steps, now 595; 64 units of K = V = 32 and 64 for 8192 steps 1036 and 1945, now 965 and 1726; 192
// of K = 16, V = 128 for 1024 steps 586, now 529.  Tried and slower: H_t as row-major tiles, read back by ldmatrix, whose
// stores are twice as many; k and v as bf16 up to the chain warps, which then widen them, 5 %.)
// The slab count NW is a template parameter and four steps form one loop iteration, so that
// every shared-memory offset of a step is an immediate.
//
// Accumulator element map of warp (slab s, part hf), lane (g = lane/4, c = lane%4):
//   MMA rows g and g+8  <->  memory rows 16s+2g and 16s+2g+1; MMA column m of the part  <->  memory column
//   hf*V/SP + SEG*c' + 2*(m>>3) + (m&1) with SEG = V/(4 SP) and c' = (m&7)>>1, i.e. a thread holds SEG adjacent
//   columns of two adjacent rows.
#include "device_common.cuh"
#include "internal.h"
#include "mma_tile.cuh"
#include "pipeline.cuh"
#include "tile.cuh"

namespace m2rnn {
namespace {

constexpr int kBarrierBytes = 128;

// Byte offsets inside a stage of TC steps: H_t fragments [TC][K/16][V/16][512], then k [TC][K], v [TC][V] and f [TC] as
// fp32 and q [TC][K] as it is.
// The hand-over of a stage costs the chain warps some 50 ns, so a stage is 16 steps where three of that size fit into
// shared memory or else two do (their chain warps then look for the next stage only when they need its first
// row, which leaves the service warps the time between), and three of 8 steps for the largest groups.
template <int V, int K, int OCC>
struct CsStage {
  static constexpr size_t kSmemMax = (OCC == 1 ? 227 : 228 / OCC - 1) * 1024;
  static constexpr size_t total_of(int tc, int stages) {
    return kBarrierBytes + (size_t)stages * tc * (K * V * 2 + K * 4 + V * 4 + 4 + K * 2 + (K + V) * 2) + (size_t)tc * 2 * V * 4;
  }
  static constexpr bool k16 = OCC == 1 || K <= 32;      // (two service warps stage no more than that)
  static constexpr bool kThree = k16 && total_of(16, 3) <= kSmemMax, kTwo = k16 && total_of(16, 2) <= kSmemMax;
  static constexpr int TC = kThree || kTwo ? 16 : 8, kStages = kThree || (!kTwo && total_of(8, 3) <= kSmemMax) ? 3 : 2;
  static constexpr bool kFits = total_of(TC, kStages) <= kSmemMax;
  static constexpr bool kLate = kStages == 2 || V == 128;
  static constexpr uint32_t k = TC * K * V * 2;
  static constexpr uint32_t v = k + TC * K * 4;
  static constexpr uint32_t f = v + TC * V * 4;
  static constexpr uint32_t q = f + TC * 4;
  static constexpr uint32_t bytes = q + TC * K * 2;
  // the ring in which k and v arrive as they are
  static constexpr uint32_t raw = TC * (K + V) * 2;
  // both halves of the sums of a stage's y
  static constexpr uint32_t ybytes = TC * 2 * V * 4;
  static constexpr uint32_t total = kBarrierBytes + kStages * (bytes + raw) + ybytes;
  static_assert(total == total_of(TC, kStages), "a block's shared memory");
};

// Where lane (g, c) of a chain warp keeps the 16 bytes of an A fragment inside the fragment's 512: for the warps of the slab
// it is the same place (any permutation would do); a service warp's ldmatrix takes the lanes of one c as the rows of a
// matrix, and this order spreads those eight over all banks.
__device__ __forceinline__ uint32_t frag_off(int g, int c) {
  const int rev = ((g & 1) << 2) | (g & 2) | (g >> 2);
  return (uint32_t)((g >> 1) * 128 + ((rev ^ c) << 4));
}

// memory column (inside a part of VP columns) of MMA column m of that part
template <int VP>
__host__ __device__ constexpr int part_col(int m) { return (VP / 4) * ((m & 7) >> 1) + 2 * (m >> 3) + (m & 1); }

// service warps of a CTA: one per scheduler that also hosts chain warps, so that their work does not
// weigh on a single scheduler (the chain warps of a slab advance in lockstep with the slowest); two where CTAs share
// an SM
__host__ __device__ constexpr int cs_service_warps(int chain_warps, int occ) { return occ > 1 ? 2 : chain_warps < 4 ? chain_warps : 4; }
__host__ __device__ constexpr int cs_threads(int chain_warps, int occ) { return (chain_warps + cs_service_warps(chain_warps, occ)) * 32; }
// registers a thread can have
__host__ __device__ constexpr int cs_regs(int chain_warps, int occ) { return 65536 / (occ * cs_threads(chain_warps, occ)); }

__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void lds_b128(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// eight bf16 from one place in shared memory to another, as fp32
__device__ __forceinline__ void widen8(uint32_t src_sa, uint32_t dst_sa) {
  uint32_t r[4];
  lds_b128(src_sa, r);
#pragma unroll
  for (int x = 0; x < 2; ++x)
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(dst_sa + 16u * x), "r"(r[2 * x] << 16), "r"(r[2 * x] & 0xffff0000u), "r"(r[2 * x + 1] << 16),
                 "r"(r[2 * x + 1] & 0xffff0000u) : "memory");
}
__device__ __forceinline__ float2 widen(uint32_t x) { return make_float2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u)); }

template <int V, int SP, int NW, bool CKPT, int OCC>
__global__ void __launch_bounds__(cs_threads(SP * NW, OCC), OCC) fwd_bf16_cs_kernel(ScanArgs a) {
  constexpr int K = 16 * NW;         // rows of this CTA's slab group (NW slabs of 16 rows): a.KCf
  using S = CsStage<V, K, OCC>;
  constexpr int kSvc = cs_service_warps(SP * NW, OCC);
  constexpr int VH = V / SP;         // columns of a part
  constexpr int NTH = VH / 8;        // accumulator tiles of a warp
  constexpr int KT = V / 16;         // k-tiles of the product
  constexpr int KTH = KT / SP;       // k-tiles a warp produces itself
  constexpr int KTP = KT - KTH;      // k-tiles it receives
  constexpr int SEGH = VH / 4;       // adjacent memory columns per thread
  constexpr int TC = S::TC, kStages = S::kStages;
  constexpr int kMine = TC / kSvc, kBlk = 32 / kMine;   // steps of a stage per service warp; stages of a block of gates
  constexpr int PV = kMine * V / 8 > 32 ? kMine * V / 8 / 32 : 1, kNextV = kSvc * 256 / V;   // pieces of v per lane, kNextV steps apart
  static_assert(kMine * K / 8 <= 32, "a lane stages eight entries of k");
  static_assert(kMine % 2 == 0, "the readout of one slab takes two steps at a time");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  begin_dependent();

  const int Kf = a.K, N = a.N;            // rows of the whole state
  const int RS = Kf / K;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31, g = lane >> 2, c = lane & 3;
  const int place = blockIdx.x / RS, rs = blockIdx.x % RS;
  const int b = batch_entry(a, place / N, smem_raw), n = place % N, bn = b * N + n;
  const UnitSpan span = unit_span(a, b);   // this batch entry's tokens (a slice of a packed batch, or b T ..)
  const int T = span.T, nst = (T + TC - 1) / TC;
  const size_t tok0 = span.tok0;
  const int rbase = rs * K;
  uint64_t *full = reinterpret_cast<uint64_t *>(smem_raw), *done = full + kStages;   // [kStages] each
  const uint32_t st0 = smem_u32(smem_raw) + kBarrierBytes;

  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], kSvc);
      mbar_init(&done[s], SP * NW);
    }
    fence_mbar_init();
  }
  __syncthreads();

  if (warp >= SP * NW) {
    // ------------------------------------------------------------------ service warps
    // Warp sw takes steps sw, sw + kSvc, .. of every stage, for staging and readout alike: it overwrites only q and
    // v that it alone reads (the chain warps are through with a stage when it is done, and write
    // fragments into it only when all service warps have filled it).
    const int sw = warp - SP * NW;
    const int hq = n / (N / a.Nq), hk = n / (N / a.Nk);
    const float al = a.alpha ? a.alpha[n] : 1.f, be = a.beta ? a.beta[n] : 0.f;
    const bool want_y = a.y != nullptr;
    // this lane's share of a stage: eight entries of k and of q of one step, eight of v; all addresses walk
    const bool has_k = lane < kMine * K / 8, has_v = lane < kMine * V / 8;
    const int kt = sw + kSvc * (lane / (K / 8)), kj = (lane % (K / 8)) * 8, vt = sw + kSvc * (lane / (V / 8)), vj = (lane % (V / 8)) * 8;
    const __nv_bfloat16 *kp = static_cast<const __nv_bfloat16 *>(a.k) + (tok0 + kt) * a.ks + hk * Kf + rbase + kj;
    const __nv_bfloat16 *qp = static_cast<const __nv_bfloat16 *>(a.q) + (tok0 + kt) * a.qs + hq * Kf + rbase + kj;
    const __nv_bfloat16 *vp = static_cast<const __nv_bfloat16 *>(a.v) + (tok0 + vt) * a.vs + n * V + vj;
    int tk = kt, tq = kt, tv = vt;          // the steps that the pointers are at
    // The gates of this warp's steps of kBlk stages at a time, a lane each.  Raw values of the next block are
    // fetched a block ahead.
    int tg = sw + kSvc * (lane % kMine) + TC * (lane / kMine);
    const float *gp = a.gate + (tok0 + tg) * N + n;
    float graw = tg < T ? *gp : 0.f, fblk = 0.f;
    auto next_gates = [&]() {
      fblk = gate_value(a.gate_kind, graw, al, be, nullptr);
      gp += (size_t)kBlk * TC * N; tg += kBlk * TC;
      if (tg < T) graw = *gp;
    };
    const uint32_t klane = (uint32_t)(kt * K + kj), vlane = (uint32_t)(vt * V + vj);
    const uint32_t raw0 = st0 + kStages * S::bytes;
    // k and v of stage st arrive as they are in its slot of a ring of their own, two more stages ahead, and are
    // widened into the stage's slot when that is free; q goes to the slot itself
    auto request_kv = [&](int s) {
      const uint32_t sa = raw0 + (uint32_t)s * S::raw;
      if (has_k && tk < T) cp16(sa + 2u * klane, kp);
#pragma unroll
      for (int x = 0; x < PV; ++x)
        if (has_v && tv + x * kNextV < T) cp16(sa + 2u * (TC * K + vlane + x * kNextV * V), vp + x * kNextV * a.vs);
      kp += TC * a.ks; vp += TC * a.vs;
      tk += TC; tv += TC;
    };
    auto request_q = [&](int s) {
      if (want_y && has_k && tq < T) cp16(st0 + (uint32_t)s * S::bytes + S::q + 2u * klane, qp);
      qp += TC * a.qs; tq += TC;
    };
    auto widen_kv = [&](int st, int s) {
      const uint32_t sa = st0 + (uint32_t)s * S::bytes, ra = raw0 + (uint32_t)s * S::raw;
      if (has_k) widen8(ra + 2u * klane, sa + S::k + 4u * klane);
#pragma unroll
      for (int x = 0; x < PV; ++x)
        if (has_v) widen8(ra + 2u * (TC * K + vlane + x * kNextV * V), sa + S::v + 4u * (vlane + x * kNextV * V));
      if (st % kBlk == 0) next_gates();
      const float f = __shfl_sync(0xffffffffu, fblk, kMine * (st % kBlk) + lane % kMine);
      if (lane < kMine) sts32(sa + S::f + 4u * (uint32_t)(sw + kSvc * lane), f);
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[s]);
    };
    // y of this warp's steps goes out through shared memory, as two halves of the sum, in pieces of eight columns: those
    // of vt and vj
    const uint32_t ybuf = raw0 + kStages * S::raw + 4u * (uint32_t)(kMine * 2 * V * sw);
    const uint32_t yout = ybuf + 4u * (uint32_t)((lane / (V / 8)) * 2 * V + vj);
    uint4 wr8 = make_uint4(0u, 0u, 0u, 0u);
    const bool has_wr = a.w_r && rs == 0;
    if (has_wr && has_v) wr8 = *reinterpret_cast<const uint4 *>(static_cast<const __nv_bfloat16 *>(a.w_r) + (size_t)n * V + vj);
    const size_t ystep = (size_t)N * V;     // elements between tokens of y
    int ty = vt;
    const size_t yat = (tok0 + ty) * ystep + n * V + vj;
    __nv_bfloat16 *yg = static_cast<__nv_bfloat16 *>(a.y) + yat;
    float *yp = a.y_part ? a.y_part + (size_t)rs * a.TT * ystep + yat : nullptr;
    // Readout.  A lane's 16 bytes of a fragment are {two columns of row g, of row g + 8, two more of row g, of row g + 8}.
    // Taken as the rows of ldmatrix matrices (the lanes of one c: g = 0 .. 7) and transposed they are eight rows of
    // an A operand whose k runs over g: its rows 0, 1, 4, 5 belong to the state rows of MMA rows 0-7 and 2, 3, 6, 7 to those
    // of 8-15.  B holds q of the first in its even columns and of the second in the odd ones, each
    // row of the product is taken from the column that fits it, and the two halves of y are added at the
    // end.  A matrix quarter: (c = 2 cp, slab w), (2 cp + 1, w), (2 cp, w + 1), (2 cp + 1, w + 1).
    const uint32_t ld0 = frag_off(lane & 7, (lane >> 3) & 1);                   // cp = 1: 32 bytes away in the line, by XOR
    const int w_of = lane >> 4;
    const uint32_t qsel = (g & 1) ? 0x7632u : 0x5410u;
    // With one slab the other half of k takes another step of this warp, whose y are columns 2 and 3 (and 6, 7).
    constexpr bool kPair = NW == 1;
    // One k-tile at a time where the chain warps' own loads would wait behind a burst of the readout's: with one slab (K = 16,
    // V = 128: 307 -> 297 ns a step) and with four (600 -> 594 us below); with two or three the burst ends sooner.
    constexpr int G = NW == 1 || NW == 4 ? 1 : KT;
    const uint32_t yin = ybuf + 4u * (uint32_t)((kPair ? (c & 1) * 2 * V + SEGH * (c >> 1) : SEGH * c) + ((g >> 1) & 1) * V + 2 * (g >> 2) + (g & 1));
    for (int st = 0; st < kStages && st < nst; ++st) { request_kv(st); request_q(st); }
    cp_commit();
    cp_wait<0>();
    for (int st = 0; st < kStages && st < nst; ++st) widen_kv(st, st);
    for (int st = 0; st < kStages; ++st) { request_kv(st); cp_commit(); }
#pragma unroll 1
    for (int st = 0, s = 0, par = 0; st < nst; ++st) {
      if (!mbar_wait(&done[s], par)) { report_timeout(a.dev_status); return; }
      cp_wait<kStages - 1>();   // this thread's part of q of stage st and of k and v of stage st + kStages
      __syncwarp();
      if (want_y) {
        const uint32_t sa = st0 + (uint32_t)s * S::bytes;
#pragma unroll 1
        for (int i = 0; i < kMine; i += kPair ? 2 : 1) {
          const int t = sw + kSvc * i;
          // (past the end there are no fragments, and what stands in their place may be no number: zeros of B do not undo that)
          const int t_of = w_of && st * TC + t + kSvc < T ? t + kSvc : t;
#pragma unroll 1
          for (int kb = 0; kb < KT; kb += G) {   // k-tiles of y
            float Y[G][2][4];
#pragma unroll
            for (int kt = 0; kt < G; ++kt)
#pragma unroll
              for (int cp = 0; cp < 2; ++cp) Y[kt][cp][0] = Y[kt][cp][1] = Y[kt][cp][2] = Y[kt][cp][3] = 0.f;
#pragma unroll
            for (int w = 0; w < NW; w += 2) {
              constexpr bool kOdd = NW & 1;
              const bool single = kOdd && !kPair && w + 1 == NW;       // no second slab: its q is zero
              uint32_t b[2];
#pragma unroll
              for (int x = 0; x < 2; ++x) {
                uint32_t q0 = 0u, q1 = 0u;
                if (!(single && x)) asm volatile("ld.shared.v2.b32 {%0,%1}, [%2];" : "=r"(q0), "=r"(q1) : "r"(sa + S::q + 2u * (uint32_t)((kPair ? t + kSvc * x : t) * K + 16 * (kPair ? w : w + x) + 4 * c)));
                b[x] = kPair && ((g >> 1) & 1) != x ? 0u : __byte_perm(q0, q1, qsel);
              }
              const uint32_t fr = sa + (uint32_t)((kPair ? t_of : t * NW + w + (single ? 0 : w_of)) * (KT * 512));
#pragma unroll
              for (int kt = 0; kt < G; ++kt)
#pragma unroll
                for (int cp = 0; cp < 2; ++cp) {
                  uint32_t A[4];
                  ldmatrix_x4_trans(fr + 512u * (kb + kt) + (ld0 ^ (32u * cp)), A[0], A[1], A[2], A[3]);
                  mma_bf16_16816(Y[kt][cp], A, b[0], b[1]);
                }
            }
            // row e of quarter c: columns 2 (2 kth + (e >> 2)) + (e & 1) of the part's segment c, from the even column
            // or the odd one by bit 1 of e; all lanes of a row hold the same, lane c keeps quarter c
#pragma unroll
            for (int kt = 0; kt < G; ++kt) {
              float v[4];
#pragma unroll
              for (int cp = 0; cp < 2; ++cp) {
                v[2 * cp] = (g & 2) ? Y[kt][cp][1] : Y[kt][cp][0];
                v[2 * cp + 1] = (g & 2) ? Y[kt][cp][3] : Y[kt][cp][2];
              }
              const uint32_t at = yin + 4u * (uint32_t)(i * 2 * V + ((kb + kt) / KTH) * VH + 4 * ((kb + kt) % KTH));
              if constexpr (kPair) {   // of step c % 2, quarters c / 2 and c / 2 + 2
                sts32(at, (c & 2) ? v[1] : v[0]);
                sts32(at + 8u * SEGH, (c & 2) ? v[3] : v[2]);
                continue;
              }
              const float m = (c & 2) ? ((c & 1) ? v[3] : v[2]) : ((c & 1) ? v[1] : v[0]);
              sts32(at, m);
            }
          }
        }
        __syncwarp();
#pragma unroll
        for (int x = 0; x < PV; ++x) {
          if (!has_v || ty + x * kNextV >= T) continue;
          const uint32_t yo = yout + 4u * (uint32_t)(x * (32 * 8 / V) * 2 * V);
          float4 lo = lds128(yo), hi = lds128(yo + 16u);
          const float4 lo2 = lds128(yo + 4u * V), hi2 = lds128(yo + 4u * V + 16u);
          lo.x += lo2.x; lo.y += lo2.y; lo.z += lo2.z; lo.w += lo2.w;
          hi.x += hi2.x; hi.y += hi2.y; hi.z += hi2.z; hi.w += hi2.w;
          if (has_wr) {   // + w_r (.) v
            const float4 v0 = lds128(sa + S::v + 4u * (vlane + x * kNextV * V)), v1 = lds128(sa + S::v + 4u * (vlane + x * kNextV * V) + 16u);
            const float2 a0 = __ffma2_rn(widen(wr8.x), make_float2(v0.x, v0.y), make_float2(lo.x, lo.y)), a1 = __ffma2_rn(widen(wr8.y), make_float2(v0.z, v0.w), make_float2(lo.z, lo.w));
            const float2 a2 = __ffma2_rn(widen(wr8.z), make_float2(v1.x, v1.y), make_float2(hi.x, hi.y)), a3 = __ffma2_rn(widen(wr8.w), make_float2(v1.z, v1.w), make_float2(hi.z, hi.w));
            lo = make_float4(a0.x, a0.y, a1.x, a1.y);
            hi = make_float4(a2.x, a2.y, a3.x, a3.y);
          }
          if (yp) {   // this slab group's share of y, fp32; the shares are added by a second kernel
            *reinterpret_cast<float4 *>(yp + x * kNextV * ystep) = lo;
            *reinterpret_cast<float4 *>(yp + x * kNextV * ystep + 4) = hi;
          } else {
            *reinterpret_cast<uint4 *>(yg + x * kNextV * ystep) = make_uint4(pack_bf16(lo.x, lo.y), pack_bf16(lo.z, lo.w), pack_bf16(hi.x, hi.y), pack_bf16(hi.z, hi.w));
          }
        }
        ty += TC;
        yg += TC * ystep;
        if (yp) yp += TC * ystep;
      }
      __syncwarp();
      if (st + kStages < nst) {
        request_q(s);
        widen_kv(st + kStages, s);
        request_kv(s);          // of the stage that follows it in this slot
      }
      cp_commit();
      if (++s == kStages) { s = 0; par ^= 1; }
    }
    cp_wait<0>();
    return;
  }

  // -------------------------------------------------------------------- chain warps
  const int slab = warp / SP, hf = warp % SP;
  const int row0 = 16 * slab + 2 * g;    // memory rows row0, row0 + 1  <->  MMA rows g, g + 8
  const int col0 = hf * VH + SEGH * c;   // first of this thread's SEGH adjacent memory columns
  const size_t KV = (size_t)Kf * V;

  // B fragments of this warp's part of W: all KT k-tiles x NTH column tiles, kept in the order the
  // warp uses them (its own k-tiles first, then the others') so that every index is static
  uint32_t Wr[KT][NTH][2];
  {
    const uint16_t *w = reinterpret_cast<const uint16_t *>(a.W) + (size_t)n * V * V;
#pragma unroll
    for (int kt = 0; kt < KT; ++kt) {
      const int hk = (hf + kt / KTH) % SP, kth = kt % KTH;   // the k-tile's part (own part first, then round the ring) and its index inside it
      auto row = [&](int m) { return hk * VH + part_col<VH>(16 * kth + m); };
      const int l0 = row(2 * c), l1 = row(2 * c + 1), l2 = row(2 * c + 8), l3 = row(2 * c + 9);
#pragma unroll
      for (int nt = 0; nt < NTH; ++nt) {
        const int j = hf * VH + part_col<VH>(8 * nt + g);
        Wr[kt][nt][0] = (uint32_t)w[l0 * V + j] | ((uint32_t)w[l1 * V + j] << 16);
        Wr[kt][nt][1] = (uint32_t)w[l2 * V + j] | ((uint32_t)w[l3 * V + j] << 16);
      }
    }
  }

  // H[nt] = {row0: cols 2nt, 2nt+1 of the thread's segment | row0 + 1: same}
  float H[NTH][4];
  const size_t own = (size_t)(rbase + row0) * V + col0;
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int x = 0; x < KTH; ++x) {
      const float4 t4 = a.h0 ? *reinterpret_cast<const float4 *>(a.h0 + bn * KV + own + h * V + 4 * x) : make_float4(0.f, 0.f, 0.f, 0.f);
      H[2 * x][2 * h] = t4.x; H[2 * x][2 * h + 1] = t4.y; H[2 * x + 1][2 * h] = t4.z; H[2 * x + 1][2 * h + 1] = t4.w;
    }
  auto store_state = [&](float *dst) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int x = 0; x < KTH; ++x)
        *reinterpret_cast<float4 *>(dst + own + h * V + 4 * x) =
            make_float4(H[2 * x][2 * h], H[2 * x][2 * h + 1], H[2 * x + 1][2 * h], H[2 * x + 1][2 * h + 1]);
  };

  // A fragment of the thread's own k-tile kth = accumulator tiles 2kth, 2kth+1, into registers and the slab's fragments
  const uint32_t foff = frag_off(g, c);
  auto pack_put = [&](uint32_t (&A)[4], int kth, uint32_t tile) {
    A[0] = pack_bf16(H[2 * kth][0], H[2 * kth][1]);
    A[1] = pack_bf16(H[2 * kth][2], H[2 * kth][3]);
    A[2] = pack_bf16(H[2 * kth + 1][0], H[2 * kth + 1][1]);
    A[3] = pack_bf16(H[2 * kth + 1][2], H[2 * kth + 1][3]);
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(tile + (uint32_t)(512 * (KTH * hf + kth))), "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]) : "memory");
  };
  auto slab_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + slab), "n"(32 * SP) : "memory"); };

  // P <- k v^T, then the own k-tiles, then the others'
  auto seed = [&](float (&P)[NTH][4], uint32_t kp, uint32_t vp) {
    const float2 k2 = lds64(kp);
#pragma unroll
    for (int x = 0; x < SEGH / 4; ++x) {
      const float4 v4 = lds128(vp + 16u * x);
      const float2 a0 = __fmul2_rn(make_float2(k2.x, k2.x), make_float2(v4.x, v4.y)), a1 = __fmul2_rn(make_float2(k2.y, k2.y), make_float2(v4.x, v4.y));
      const float2 b0 = __fmul2_rn(make_float2(k2.x, k2.x), make_float2(v4.z, v4.w)), b1 = __fmul2_rn(make_float2(k2.y, k2.y), make_float2(v4.z, v4.w));
      P[2 * x][0] = a0.x; P[2 * x][1] = a0.y; P[2 * x][2] = a1.x; P[2 * x][3] = a1.y;
      P[2 * x + 1][0] = b0.x; P[2 * x + 1][1] = b0.y; P[2 * x + 1][2] = b1.x; P[2 * x + 1][3] = b1.y;
    }
  };
  auto mma_partner = [&](float (&P)[NTH][4], uint32_t tile) {
    uint32_t A[KTP][4];
#pragma unroll
    for (int i = 0; i < KTP; ++i) lds_b128(tile + (uint32_t)(512 * (KTH * ((hf + 1 + i / KTH) % SP) + i % KTH)), A[i]);   // same ring order as Wr
#pragma unroll
    for (int i = 0; i < KTP; ++i)
#pragma unroll
      for (int nt = 0; nt < NTH; ++nt) mma_bf16_16816(P[nt], A[i], Wr[KTH + i][nt][0], Wr[KTH + i][nt][1]);
  };

  // One step.  Pc: H_{t-1} W + k_t v_t^T, complete or in flight on entry.
  // Pn receives the same for step t+1 (after the last step: fed a valid but meaningless row).
  auto step = [&](float (&Pc)[NTH][4], float (&Pn)[NTH][4], float f, uint32_t tile, uint32_t kn, uint32_t vn) {
    seed(Pn, kn, vn);
    const float2 f2 = make_float2(f, f), m1 = make_float2(-1.f, -1.f);
    // Unit u = (accumulator tile u/2, row half u%2): Eq. 1 and 2 for two elements.
    auto unit = [&](int u) {
      const int nt = u >> 1, h = u & 1;
      const float2 z = make_float2(tanh_approx(Pc[nt][2 * h]), tanh_approx(Pc[nt][2 * h + 1]));   // Eq. 1
      const float2 d = __ffma2_rn(z, m1, make_float2(H[nt][2 * h], H[nt][2 * h + 1]));            // H - Z
      const float2 hh = __ffma2_rn(f2, d, z);                                                     // Eq. 2
      H[nt][2 * h] = hh.x; H[nt][2 * h + 1] = hh.y;
    };
    uint32_t A[KTH][4];
    // The MMAs of own k-tile kth are issued between the units of the next k-tile's two
    // accumulator tiles, so that the tensor pipe and the tanh unit work at the same time
    // inside one in-order warp.
#pragma unroll
    for (int u = 0; u < 4; ++u) unit(u);
    pack_put(A[0], 0, tile);
    if constexpr (KTH == 2) {
#pragma unroll
      for (int nt = 0; nt < NTH; ++nt) {
        mma_bf16_16816(Pn[nt], A[0], Wr[0][nt][0], Wr[0][nt][1]);
#pragma unroll
        for (int u = 4 * nt / NTH; u < 4 * (nt + 1) / NTH; ++u) unit(4 + u);
      }
      pack_put(A[1], 1, tile);
    }
#pragma unroll
    for (int nt = 0; nt < NTH; ++nt) mma_bf16_16816(Pn[nt], A[KTH - 1], Wr[KTH - 1][nt][0], Wr[KTH - 1][nt][1]);
    slab_sync();
    mma_partner(Pn, tile);
  };

  float P0[NTH][4], P1[NTH][4];
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
  const uint32_t ok = S::k + 4u * (uint32_t)row0, ov = S::v + 4u * (uint32_t)col0, ot = (uint32_t)(slab * 32 * V) + foff;
  constexpr uint32_t dk = 4u * K, dv = 4u * V, dt = 2u * K * V;   // per step
  if (T > 0) {
    if (!mbar_wait(&full[0], 0)) { report_timeout(a.dev_status); return; }
    // prologue: the first step's product from the initial state, through the tile of the first stage's last step
    // (written again only behind the barriers of the steps between)
    uint32_t A[KTH][4];
    const uint32_t tile = st0 + ot + (TC - 1) * dt;
#pragma unroll
    for (int kth = 0; kth < KTH; ++kth) pack_put(A[kth], kth, tile);
    seed(P0, st0 + ok, st0 + ov);
#pragma unroll
    for (int kth = 0; kth < KTH; ++kth)
#pragma unroll
      for (int nt = 0; nt < NTH; ++nt) mma_bf16_16816(P0[nt], A[kth], Wr[kth][nt][0], Wr[kth][nt][1]);
    slab_sync();
    mma_partner(P0, tile);
  }
#pragma unroll 1
  for (int st = 0, s = 0; st < nst; ++st) {
    const uint32_t sa = st0 + (uint32_t)s * S::bytes;
    const int sn = s + 1 == kStages ? 0 : s + 1;
    const int len = min(TC, T - st * TC);
    uint32_t nx = sa;
    auto next_stage = [&]() -> bool {   // what the stage's last step seeds: the next stage's first (after the last step: any valid row)
      if (st + 1 < nst) {
        if (!mbar_wait(&full[sn], ((st + 1) / kStages) & 1)) { report_timeout(a.dev_status); return false; }
        nx = st0 + (uint32_t)sn * S::bytes;
      }
      return true;
    };
    if (!S::kLate && !next_stage()) return;
    if (len == TC) {
      uint32_t tile = sa + ot, kp = sa + ok, vp = sa + ov;
#pragma unroll 1
      for (int t0 = 0; t0 < TC; t0 += 4, tile += 4 * dt, kp += 4 * dk, vp += 4 * dv) {
        const float4 f = lds128(sa + S::f + 4u * (uint32_t)t0);
        const bool last = t0 + 4 == TC;
        if (S::kLate && last && !next_stage()) return;
        const uint32_t kn = last ? nx + ok : kp + 4 * dk, vn = last ? nx + ov : vp + 4 * dv;
        maybe_checkpoint(2);
        step(P0, P1, f.x, tile, kp + dk, vp + dv);
        step(P1, P0, f.y, tile + dt, kp + 2 * dk, vp + 2 * dv);
        maybe_checkpoint(2);
        step(P0, P1, f.z, tile + 2 * dt, kp + 3 * dk, vp + 3 * dv);
        step(P1, P0, f.w, tile + 3 * dt, kn, vn);
      }
    } else {   // ragged last stage
      for (int t = 0; t < len; ++t) {
        if ((t & 1) == 0) maybe_checkpoint(min(2, len - t));
        const int tn = min(t + 1, len - 1);
        step(P0, P1, lds32(sa + S::f + 4u * t), sa + ot + t * dt, sa + ok + tn * dk, sa + ov + tn * dv);
#pragma unroll
        for (int nt = 0; nt < NTH; ++nt)
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

template <int V, int SP, int NW, bool CKPT, int OCC>
cudaError_t launch_cs(const ScanArgs &a, cudaStream_t s) {
  constexpr size_t smem = CsStage<V, 16 * NW, OCC>::total;
  static_assert(CsStage<V, 16 * NW, OCC>::kFits, "a block's shared memory");
  cudaError_t e = allow_smem(fwd_bf16_cs_kernel<V, SP, NW, CKPT, OCC>, smem);
  if (e != cudaSuccess) return e;
  const int ctas = a.B * a.N * (a.K / (16 * NW)), threads = cs_threads(SP * NW, OCC);
  return launch_early(fwd_bf16_cs_kernel<V, SP, NW, CKPT, OCC>, ctas, threads, smem, s, in_order(a, ctas, threads, 3));
}

template <int V, int SP, int NW, bool CKPT>
cudaError_t launch_cs_o(const ScanArgs &a, cudaStream_t s) {
  // With more CTAs than SMs two, or of the smaller groups three, share an SM, whose tensor pipe and tanh unit one
  // CTA's chain leaves idle most of the time (1024 steps of 192 units, us: K = V = 32 258 -> 168, K = 48, V = 64
  // 564 -> 481; of 440, three to an SM: K = V = 32 385 -> 223).  Where a round of pairs takes 1.8 times one of single CTAs,
  // only if the rounds come out fewer for it; four slabs of V = 64 have no registers to share.
  constexpr bool kHeavy = NW == 4;
  const long ctas = (long)a.B * a.N * (a.K / (16 * NW)), sms = sm_count(), alone = (ctas + sms - 1) / sms, pairs = (ctas + 2 * sms - 1) / (2 * sms);
  if constexpr (CsStage<V, 16 * NW, 3>::kFits && cs_regs(SP * NW, 3) >= 88)
    if (ctas > 2 * sms) return launch_cs<V, SP, NW, CKPT, 3>(a, s);
  if constexpr (CsStage<V, 16 * NW, 2>::kFits && cs_regs(SP * NW, 2) >= 88)
    if (ctas > sms && (!kHeavy || 9 * pairs <= 5 * alone)) return launch_cs<V, SP, NW, CKPT, 2>(a, s);
  return launch_cs<V, SP, NW, CKPT, 1>(a, s);
}

template <int V, int SP, int NW>
cudaError_t launch_cs_v(const ScanArgs &a, cudaStream_t s) {
  return a.ckpt ? launch_cs_o<V, SP, NW, true>(a, s) : launch_cs_o<V, SP, NW, false>(a, s);
}

}  // namespace

// slabs per CTA this variant supports for a V: the register file holds (parts * slabs + 1) warps
bool fwd_cs_supported(const ScanArgs &a) {
  if (a.V == 128) return a.KCf <= 32;
  return (a.V == 32 || a.V == 64) && a.KCf <= 64;
}

// The slab count is a template parameter so that every shared-memory offset of a step is a
// compile-time constant.  Four warps per slab where the CTA would otherwise leave schedulers idle
// (one slab) and at V = 128 (a quarter of W per warp fits in registers), two elsewhere.
cudaError_t launch_fwd_bf16_cs(const ScanArgs &a, cudaStream_t s) {
  const int nw = a.KCf / 16;
  switch (a.V) {
    case 32:
      switch (nw) {
        case 1: return launch_cs_v<32, 2, 1>(a, s);
        case 2: return launch_cs_v<32, 2, 2>(a, s);
        case 3: return launch_cs_v<32, 2, 3>(a, s);
        case 4: return launch_cs_v<32, 2, 4>(a, s);
      }
      break;
    case 64:
      switch (nw) {
        case 1: return launch_cs_v<64, 4, 1>(a, s);
        case 2: return launch_cs_v<64, 2, 2>(a, s);
        case 3: return launch_cs_v<64, 2, 3>(a, s);
        case 4: return launch_cs_v<64, 2, 4>(a, s);
      }
      break;
    case 128:
      switch (nw) {
        case 1: return launch_cs_v<128, 4, 1>(a, s);
        case 2: return launch_cs_v<128, 4, 2>(a, s);
      }
      break;
  }
  return cudaErrorInvalidValue;
}

}  // namespace m2rnn
