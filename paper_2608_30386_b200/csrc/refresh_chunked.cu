// Suffix refresh, chunked form, on the Blackwell tensor cores (tcgen05 + TMEM), warp-specialised:
// 32-token chunks, two CTAs resident per SM (or one with more warps, where a launch has no more), several units (request, layer, value
// head) per CTA one after another.
//
// Eq. 1 (transposed orientation) over a chunk of C = 32 tokens starting from S_0, with
// G_t the running sum of the log-decay inside the chunk and m the chunk midpoint:
//   Kt_t = k_t * exp(G_t - G_m),  Kh_t = k_t * exp(G_m - G_t),  Qt_t = q_t * exp(G_t - G_m)
//   S'   = Diag(exp(G_m)) S_0                                   (state decayed to the midpoint)
//   A    = strict_lower(Kt Kh^T) * beta,   P = lower_incl_diag(Qt Kh^T)
//   U    = (I + A)^-1 * beta * (V - Kt S')                      (the deltas written at each token)
//   O    = Qt S' + P U
//   S_C  = Diag(exp(G_C - G_m)) (S' + Kh^T U)
//
// Roles.  The operand tiles Kt, Qt, Kh depend on the token inputs only, not on the state, so they
// are built by four PRODUCER warps while the chunk before is in flight; their inputs come by TMA into the
// tiles they become.  One TRIANGULAR warp forms T = (I + A)^-1, also state-independent.  Eight CHAIN warps
// carry the state-dependent sequence: state rescale -> right-hand side -> deltas -> outputs.  One warp
// issues all tensor-core work.  The groups meet only at mbarriers.  GDN (one scalar log-decay per token)
// keeps the decay out of the products: MMA1 and MMA2 run on the raw k, q and the per-token factors are
// applied where A, P, k S' and the outputs leave tensor memory.
//   MMA1  [Kt;Qt] Kh^T            -> A (first two TMEM quadrants, 16 rows each), P (last two)   smem x smem, M = 64
//   MMA2  S'^T [Kt;Qt]^T          -> R^T | (Qt S')^T                            tmem x smem
//   MMA3  RHS^T T^T               -> U^T      (RHS as a tf32 high/low pair)     tmem x smem
//   MMA4  (Qt S')^T += U^T P^T    -> O^T                                         tmem x smem
//   MMA5  S'^T      += U^T Kh     -> state    (U as a tf32 high/low pair)       tmem x smem
// Buffers: the Kt/Qt tile of chunk n+1 may be written once MMA2 of chunk n has completed, the Kh tile once its
// MMA1 has; MMA5 contracts over the tokens and reads Kh as an MN-major operand from a second tile (tf32
// MN-major operands have a swizzle of their own), which, read last, is double-buffered by chunk parity.
//
// Bound, measured (B200, 64 requests x 256 tokens x 4 layers x 32 heads): KDA 1064 us = 1.97 G token-heads/s = 62 % of the
// rate at which HBM could bring its bytes (657 us), GDN 825 us = 2.54 G (50 %; 849 with the inverse by columns), in single passes 0.1 s apart, which
// the power limit leaves alone; 1685 and 1630 us in the form this one grew from, 1090 and 885 with a CTA per unit.  What is nearest its limit is the SM's shared-memory data pipe (load/store units and the tensor core's operand
// reads together): per chunk and SM (two CTAs) KDA takes 4.1 k cycles, of which that pipe is busy 83 %, the issue slots 51 %, the tensor
// pipe 38 %; GDN 3.1 k, 97 %, 48 %, 46 %; the state-only form 3.4 k at 2 to 4 chunks per unit, 76 %, 53 %, 33 %.  A CTA alone
// on its SM is bound by its chain of hand-offs: a chunk every 3.7 k cycles (GDN 3.3 k) in the form made for it (see alone_for), 5.0 k
// (3.8 k) in the other.
// What it was before, in the order in which it was found: 103 cycles of issue per tensor-core instruction (behind
// `lane == 0` instead of an elected lane), 119 KB of code in the instruction caches (half of that now), and 85 % of the
// shared-memory pipe (8-byte accesses in 16-byte places, A padded to 128 rows, V and O value by value).
// Under sustained load the part is at its 1000 W limit and runs this kernel at 1.7 instead of 1.965 GHz.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "dasc_internal.h"
#include "launch.cuh"
#include "tcgen05_util.cuh"

namespace {

using namespace tc5;

constexpr int C = 32;          // chunk length
constexpr int D = 128;         // d_k = d_v
constexpr int NCH = 256;       // chain threads (warps 0-7)
// Two forms.  SHARED: two CTAs per SM.  ALONE (see alone_for): one, with more warps and second buffers, so that the tiles, MMA1 and T of
// the next chunk are made while the chain is in this one, and the outputs leave meanwhile.
template <bool ALONE>
struct Form {
  static constexpr int NP = ALONE ? 256 : 128;           // producer threads (from warp 8 on)
  static constexpr int WARP_T = 8 + NP / 32;             // the warp that inverts the triangular system (in TMEM quadrant 0)
  // ALONE: MMA1, rows 16-31 of A and the copies of the inputs are a warp's own (in quadrant 1), P and the outputs those of four more
  // (one per quadrant), so that the issuing warp and the chain warps do the chain's work only.
  static constexpr int WARP_MMA1 = WARP_T + 1;
  static constexpr int WARP_O = WARP_T + 2;
  static constexpr int WARP_MMA = ALONE ? WARP_O + 4 : WARP_T + 1;  // the warp that issues tensor-core work (SHARED: in quadrant 1)
  static constexpr int NT = (WARP_MMA + 1) * 32;
  static constexpr int BUF = ALONE ? 2 : 1;              // buffers of what SHARED has one of: Kt/Qt, K-major Kh (GDN: raw k, q), T, A|P, R|O
  static constexpr int RING = ALONE ? 8 : 4;             // per-token scalars, by chunk index mod RING
  static constexpr int FAC = ALONE ? 4 : 2;              // state factors, by chunk index mod FAC
  static constexpr uint32_t TMEM_COLS = ALONE ? 512 : 256;
};
// row pitches (floats) of the fp32 triangular work matrices: A^T (KDA) and X; -A (GDN)
constexpr int LDX = 36, LDL = 40;

// TMEM columns; RO: R^T 32 columns | (Qt S')^T 32; RL: the right-hand side's low part (SHARED: over the consumed A|P)
constexpr uint32_t COL_S = 0, COL_AP = 128;
template <bool ALONE>
constexpr uint32_t COL_RO = ALONE ? 192 : 160;  // ALONE: AP 128-191, RO 192-383 (three), U 384-415, RL 416-447
template <bool ALONE>
constexpr uint32_t COL_U = ALONE ? 384 : 224;

// shared memory map (bytes)
constexpr uint32_t OFF_KQ = 0;                          // [4][64 rows][128 B]  rows 0-31 Kt, 32-63 Qt
constexpr uint32_t OFF_KHT = OFF_KQ + 4 * 64 * 128;     // [2][4][32 rows][128 B] Kh[t][c] once more, as the MN-major operand of MMA5, by chunk parity
constexpr uint32_t OFF_KH = OFF_KHT + 2 * 128 * 128;    // [4][32 rows][128 B]  Kh[t][c]
constexpr uint32_t OFF_TM = OFF_KH + 4 * 32 * 128;      // [1][32 rows][128 B]  T[t][i]; TM|PM later the bf16 O tile
constexpr uint32_t OFF_PM = OFF_TM + 32 * 128;          // [1][32 rows][128 B]  P[t][i]
constexpr uint32_t OFF_V = OFF_PM + 32 * 128;           // [2][32 rows][128 B] V[t][v] bf16
constexpr uint32_t OFF_L = OFF_V + C * D * 2;           // fp32 A^T [32][LDX], GDN -A [32][LDL] (entries on and above A's diagonal are not used)
constexpr uint32_t OFF_X = OFF_L + C * LDL * 4;         // [32][LDX] fp32 X = (I + A)^-1
constexpr uint32_t OFF_FAC = OFF_X + C * LDX * 4;       // [2][128] fp32 state factor per channel, by chunk parity
constexpr uint32_t OFF_POST = OFF_FAC + 2 * D * 4;      // log-factor owed after a chunk: KDA [2][128] fp32 by chunk parity, GDN [4] by chunk index mod 4
constexpr uint32_t OFF_BETA = OFF_POST + 2 * D * 4;     // [4][32] fp32, by chunk index mod 4 (written well ahead)
// GDN only, same ring as beta: per-token factors of the scalar decay, e1 = exp(G_t - G_m), e2 = exp(G_m - G_t)
constexpr uint32_t OFF_E1C = OFF_BETA + 4 * C * 4;      // [4][32] fp32 e1 * (truncation compensation)
constexpr uint32_t OFF_E2 = OFF_E1C + 4 * C * 4;        // [4][32] fp32 e2
constexpr uint32_t OFF_BTE1 = OFF_E2 + 4 * C * 4;       // [4][32] fp32 beta * e1
constexpr uint32_t OFF_FIN = OFF_BTE1 + 4 * C * 4;      // [128] fp32 state factor per channel behind the last chunk of a unit
constexpr uint32_t OFF_UNIT = OFF_FIN + D * 4;          // the CTA's units
constexpr uint32_t OFF_MISC = OFF_UNIT + 16 * 48;       // barriers, tmem base, flags
// (GDN: the K-major Kh tile's place holds raw k (rows 0-31) and q (rows 32-63) as bf16, [2][64 rows][128 B])
constexpr uint32_t SMEM_BYTES = OFF_MISC + 320;
static_assert(SMEM_BYTES <= 113 * 1024, "two CTAs per SM");
// ALONE: the second buffers and longer rings, behind the map above
constexpr uint32_t OFF_KQ_2 = (SMEM_BYTES + 1023) / 1024 * 1024;
constexpr uint32_t OFF_KH_2 = OFF_KQ_2 + 4 * 64 * 128;     // (GDN: raw k, q)
constexpr uint32_t OFF_TM_2 = OFF_KH_2 + 4 * 32 * 128;
constexpr uint32_t OFF_OUT_2 = OFF_TM_2 + 32 * 128;        // the bf16 O tile
constexpr uint32_t OFF_KHT_2 = OFF_OUT_2 + C * D * 2;      // third and fourth MN-major Kh tile
constexpr uint32_t OFF_RING_2 = OFF_KHT_2 + 2 * 128 * 128;     // beta, e1c, e2, bte1: [8][32] fp32 each
constexpr uint32_t OFF_FAC_2 = OFF_RING_2 + 4 * 8 * C * 4;     // [4][128] fp32 state factors
constexpr uint32_t SMEM_ALONE = OFF_FAC_2 + 4 * D * 4;
static_assert(SMEM_ALONE <= 227 * 1024, "one CTA per SM");

constexpr uint32_t kMaxPolls = 1u << 22;

// Largest |sum of the log-decay over half a chunk| per channel for which every factor formed relative to the chunk
// midpoint stays a normal fp32 number with room for the products that follow.
constexpr float kMaxHalfDecay = 80.f;

// The tensor core reads the fp32 state as tf32 by dropping its low 13 mantissa bits, i.e. rounding
// towards zero: on average the operand is 2^-11 * E[1/m] = 3.52e-4 too small in magnitude (m the
// significand, log-uniform in [1, 2)).  The rows of Kt and Qt, the only partners of that operand,
// are scaled up by this factor to cancel the bias; A and P, which also come from those rows, are
// scaled back down when they are taken out of TMEM.
constexpr float kTruncComp = 1.000352f;
constexpr float kInvTruncComp = 1.0f / kTruncComp;
constexpr float kLog2TruncComp = 5.0774e-4f;  // log2(kTruncComp)

struct Misc {
  // Each barrier completes one phase per chunk.  Where the arrivals are "per warp", a warp's first lane arrives for it.
  // tensor core -> chain warps (one tcgen05.commit each); bar_ap also releases the triangular and the issuing warp and the
  // next log-decay (KDA) or k, q (GDN), bar_ro the Kt/Qt tile, bar_s the Kh tile of its parity (KDA)
  // (two of each, by chunk parity, where a phase could complete before all have waited for the one before: all three in ALONE; bar_s in
  // both forms, since the KDA producers wait for chunk n - 1's after they have handed over chunk n's tiles, which its products 5 need)
  uint64_t bar_ap[2], bar_ro[2], bar_s[2], bar_u, bar_o;
  // producer -> issuing warp: the tiles of a chunk are ready (per warp: 4 arrivals; KDA one more from the triangular warp, for beta)
  uint64_t rdy_prep[2];  // (ALONE: by chunk parity)
  // producer -> chain warps: the state factors of a chunk are ready (KDA per warp: 4 arrivals; GDN the first warp only: 1)
  // One barrier per chunk parity (ALONE: by chunk index mod 4): the producer may hand over the factors of chunk n+1 (n+3) before the chain
  // warps have waited for those of chunk n, and a single barrier cannot tell phases two apart.
  uint64_t rdy_fac[4];
  // chain warps -> issuing warp (per warp: 8 arrivals each)
  uint64_t rdy_state, rdy_half, rdy_rhs, rdy_u;  // (rdy_half, ALONE: the first half of the state's channels)
  // triangular warp -> chain warps (A has left TMEM: 1 arrival) and -> issuing warp (T tile ready: 1 arrival)
  uint64_t a_taken, rdy_t;
  // chain warps -> triangular warp and one another: the T|P tile region is free again (per warp: 8 arrivals)
  uint64_t tp_free;
  // issuing thread, only after a wait has run out: arrives once every tensor-core product issued so far has completed
  uint64_t drain, drain_1;
  // TMA -> producer warps: the log-decay of a chunk has landed in the Kh tile (KDA: 4 copies, one arrival with each); its raw
  // k, q have landed (4 copies, 2 without outputs)
  uint64_t g_full[2], kq_full[2];
  // TMA -> chain warps: V of a chunk has landed (2 copies, started by the triangular warp)
  uint64_t v_full;
  uint32_t tmem_base;
  volatile uint32_t abort_flag;   // a bounded wait ran out: every later wait of this CTA returns at once
  int32_t n_units, n_replayed, all_chunks;  // this CTA's units, those of them that have tokens (listed first), the chunks of all
  volatile uint32_t domain_flag[4];  // a half-chunk decay sum left the range the midpoint factors can carry; by unit index mod 4
};
static_assert(sizeof(Misc) <= 320, "Misc outgrew its shared-memory slot");

// One of a CTA's units, as all roles read it from shared memory.
constexpr int kMaxWalk = 16;
struct alignas(16) Unit {
  int64_t state;  // offset of its state, in floats
  int64_t tok0;   // its first token in the streams of the call
  int32_t n_tok, head, k_head, index, keep_row;
};

__device__ __forceinline__ float ex2f(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// One arrival for the whole warp, behind whatever its lanes did before.
__device__ __forceinline__ void arrive_warp(uint64_t *bar, int lane) {
  __syncwarp();
  if (lane == 0) mbar_arrive(bar);
}

// Barrier among the 256 chain threads: does the predicate hold for any of them?
__device__ __forceinline__ bool any_chain(bool p) {
  uint32_t any;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.or.pred.aligned q, 1, 256, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(any)
      : "r"(static_cast<uint32_t>(p))
      : "memory");
  return any != 0;
}

// What comes out of a broadcast shuffle the compiler may keep in uniform registers.
__device__ __forceinline__ int uni(int x) { return __shfl_sync(0xffffffffu, x, 0); }

// Bounded wait; after one time-out no wait of this CTA lasts longer than one poll (which itself waits for a while).  Inlined at some
// thirty places, so it is written as the smallest loop there is: the roles' code together has to stay within reach of the
// instruction caches.
__device__ __forceinline__ void wait_bar(uint64_t *bar, uint32_t parity, Misc *misc) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .b32 n, f;\n\t"
      "mov.b32 n, 0;\n"
      "POLL:\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%0], %1;\n\t"
      "@p bra DONE;\n\t"
      "ld.volatile.shared.b32 f, [%2];\n\t"
      "add.u32 n, n, 1;\n\t"
      "setp.ne.b32 q, n, %3;\n\t"
      "setp.eq.and.b32 p, f, 0, q;\n\t"
      "@p bra POLL;\n\t"
      "st.volatile.shared.b32 [%2], 1;\n"
      "DONE:\n\t}" ::"r"(smem_u32(bar)),
      "r"(parity), "r"(smem_u32(const_cast<uint32_t *>(&misc->abort_flag))), "n"(kMaxPolls)
      : "memory");
}

// The test hook's wait: `max_polls` non-blocking looks at the barrier, so that a short limit runs out
// whatever the time slice of a blocking poll is.
__device__ __forceinline__ void wait_bar_short(uint64_t *bar, uint32_t parity, Misc *misc, uint32_t max_polls) {
  bool done = false;
  for (uint32_t i = 0; i < max_polls && !done; ++i) done = mbar_test_wait(bar, parity);
  if (!done) misc->abort_flag = 1;
}

// This CTA does not (or could not) replay its unit: put the unit on the list that the token-by-token kernel walks
// next on the same stream.  Without a list, or when it is full, or when the caller asked for this kernel alone, an
// out-of-range unit is an error (word 1).
__device__ __forceinline__ void hand_over(const DascRefreshArgs &a, int unit, bool out_of_range) {
  uint32_t *ws = static_cast<uint32_t *>(a.workspace);
  const uint32_t idx = atomicAdd(ws + 2, 1u);
  const bool listed = a.unit_list && idx < static_cast<uint32_t>(a.unit_list_cap);
  if (listed) a.unit_list[idx] = unit;
  if (!listed || (out_of_range && a.domain_is_error)) atomicExch(ws + 1, 1u);
}

__device__ __forceinline__ void mma_tf32_16x8x8(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// One warp: acc (16x16) += A (16x16) * B (16x16), blocks in shared memory with pitch LDX; A row-major or its transpose.
template <bool A_TRANSPOSED>
__device__ __forceinline__ void warp_mm_acc(float (&acc)[2][4], const float *A, const float *B, int lane) {
  const int g = lane >> 2, tig = lane & 3;
#pragma unroll
  for (int kh = 0; kh < 2; ++kh) {
    uint32_t af[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = g + (i & 1) * 8, k = 8 * kh + tig + (i >> 1) * 4;
      af[i] = tf32_pre(A_TRANSPOSED ? A[k * LDX + r] : A[r * LDX + k]);
    }
#pragma unroll
    for (int nh = 0; nh < 2; ++nh) {
      uint32_t bf[2];
      bf[0] = tf32_pre(B[(8 * kh + tig) * LDX + 8 * nh + g]);
      bf[1] = tf32_pre(B[(8 * kh + tig + 4) * LDX + 8 * nh + g]);
      mma_tf32_16x8x8(acc[nh], af, bf);
    }
  }
}
__device__ __forceinline__ void warp_mm_store(float *Cb, const float (&acc)[2][4], float sign, int lane) {
  const int g = lane >> 2, tig = lane & 3;
#pragma unroll
  for (int nh = 0; nh < 2; ++nh) {
    *reinterpret_cast<float2 *>(Cb + g * LDX + 8 * nh + 2 * tig) = make_float2(sign * acc[nh][0], sign * acc[nh][1]);
    *reinterpret_cast<float2 *>(Cb + (g + 8) * LDX + 8 * nh + 2 * tig) = make_float2(sign * acc[nh][2], sign * acc[nh][3]);
  }
}

__device__ __forceinline__ float bf16lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// packed pairs of fp32 (one instruction per pair)
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// 8 x 8 blocks of 16-bit values, transposed on the way: lane's row address; register m of the result belongs to block m.
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr) : "memory");
}
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(r0), "r"(r1), "r"(r2), "r"(r3)
               : "memory");
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  uint32_t w;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w) : "f"(hi), "f"(lo));
  return w;
}

// Rows row0 .. row0 + 15 of A = strict_lower(Kt Kh^T) * beta out of tensor memory (`taddr`: first lane of the warp's quadrant).
// KDA: transposed into L; the decay is inside the product, whose Kt rows carry the truncation compensation; `rowf` = beta.
// GDN: -A into L; the product is the raw k_t . k_j and the decay exp(G_t - G_j) = e1_t e2_j is applied here; `rowf` = beta e1, `colf` = e2.
template <bool KDA>
__device__ __forceinline__ void take_a_rows(uint32_t taddr, int row0, const float *rowf, const float *colf, float *L, int lane) {
  const int g = lane >> 2, tig = lane & 3;
  uint32_t x[16];
  tmem_ld_16x256b(taddr, x);
  const float f0 = rowf[row0 + g] * (KDA ? kInvTruncComp : -1.f), f1 = rowf[row0 + g + 8] * (KDA ? kInvTruncComp : -1.f);
  tmem_ld_wait();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if constexpr (KDA) {
      float *d = L + (8 * i + 2 * tig) * LDX + row0 + g;
      d[0] = __uint_as_float(x[4 * i]) * f0;
      d[LDX] = __uint_as_float(x[4 * i + 1]) * f0;
      d[8] = __uint_as_float(x[4 * i + 2]) * f1;
      d[LDX + 8] = __uint_as_float(x[4 * i + 3]) * f1;
    } else {
      const uint64_t e = *reinterpret_cast<const uint64_t *>(colf + 8 * i + 2 * tig);
      uint64_t *const d = reinterpret_cast<uint64_t *>(L + (row0 + g) * LDL + 8 * i + 2 * tig);
      d[0] = mul2(pack2(__uint_as_float(x[4 * i]), __uint_as_float(x[4 * i + 1])), mul2(pack2(f0, f0), e));
      d[4 * LDL] = mul2(pack2(__uint_as_float(x[4 * i + 2]), __uint_as_float(x[4 * i + 3])), mul2(pack2(f1, f1), e));
    }
  }
}

// (a, b) *= f on fp32 bit patterns
__device__ __forceinline__ void scale2(uint32_t &a, uint32_t &b, uint64_t f) {
  float x, y;
  unpack2(mul2(pack2(__uint_as_float(a), __uint_as_float(b)), f), x, y);
  a = __float_as_uint(x);
  b = __float_as_uint(y);
}

// WITH_O = false is the state-only variant (no outputs wanted): q is never read, the Qt rows, P and the
// output product are left out.
// WALK = false: one unit per CTA, known at compile time (grid_for left the grid at that; always so where ALONE): the bookkeeping between
// units costs 1 to 4 % of a chunk where there is none to do.
// ZERO: the merge mode, whose units start from zero.  Their first chunk, one of about three in a window of 128 tokens, needs no state pass and no
// product 2, and its product 5 replaces what the accumulator holds.  32 requests of 1 .. 128 tokens x 4 layers x 32 heads, KDA: 212.0 -> 205.8 us.  For calls without outputs, the load policy's, and at compile time: as flags in the issuing warp's loop it cost
// every other call 1 to 3 %.  Calls without outputs and without ZERO are of the continue mode only, and still look at a.mode: with the merge mode's
// branches out at compile time GDN took 1 % less (296 units of 300 tokens 33.5 / 33.0 us), but KDA alone on an SM 2 % more (32 of 509 34.5 / 35.3, 148 of
// 256 22.7 / 23.1), for no reason that the source shows; with a flag for both worked out once, KDA 2 % more and GDN the same.
template <bool KDA, typename OT, bool WITH_O, bool ALONE, bool WALK, bool ZERO>
__global__ void __launch_bounds__(Form<ALONE>::NT, ALONE ? 1 : 2) refresh_chunked_kernel(const __grid_constant__ DascRefreshArgs a, const __grid_constant__ CUtensorMap tmap_q,
                                                                const __grid_constant__ CUtensorMap tmap_k,
                                                                const __grid_constant__ CUtensorMap tmap_v,
                                                                const __grid_constant__ CUtensorMap tmap_g) {
  // The base is a link-time constant (there is no static shared memory), so every operand descriptor is an immediate.
  extern __shared__ __align__(1024) unsigned char smem[];
  const uint32_t sbase = smem_u32(smem);
  using F = Form<ALONE>;
  constexpr int NP = F::NP, WARP_T = F::WARP_T, WARP_MMA = F::WARP_MMA, WARP_O = F::WARP_O, WARP_MMA1 = F::WARP_MMA1, RING = F::RING, FAC = F::FAC;
  // where chunk n's buffer is, and the barrier and the parity that stand for it
  auto buf = [](int n) { return static_cast<uint32_t>(ALONE ? n & 1 : 0); };
  auto phase2 = [](int n) { return static_cast<uint32_t>((n >> 1) & 1); };  // of what there are two of
  auto phase = [&](int n) { return ALONE ? phase2(n) : static_cast<uint32_t>(n & 1); };
  auto off_kq = [&](int n) { return OFF_KQ + buf(n) * (OFF_KQ_2 - OFF_KQ); };
  auto off_kh = [&](int n) { return OFF_KH + buf(n) * (OFF_KH_2 - OFF_KH); };  // GDN: raw k, q
  auto off_kht = [&](int n) { return OFF_KHT + (n & 1) * (128 * 128) + (ALONE && (n & 2) ? OFF_KHT_2 - OFF_KHT : 0u); };
  auto off_t = [&](int n) { return OFF_TM + buf(n) * (OFF_TM_2 - OFF_TM); };
  auto col_ap = [&](int n) { return COL_AP + buf(n) * 32; };
  auto col_ro = [&](int n) { return COL_RO<ALONE> + (ALONE ? static_cast<uint32_t>(n) % 3u * 64 : 0u); };
  constexpr uint32_t COL_RL = ALONE ? 416 : COL_AP, OFF_O = ALONE ? OFF_OUT_2 : OFF_TM;
  float *Lm = reinterpret_cast<float *>(smem + OFF_L);
  float *Xm = reinterpret_cast<float *>(smem + OFF_X);
  float *fac_s = reinterpret_cast<float *>(smem + (ALONE ? OFF_FAC_2 : OFF_FAC));
  float *post_s = reinterpret_cast<float *>(smem + OFF_POST);
  float *beta_s = reinterpret_cast<float *>(smem + (ALONE ? OFF_RING_2 + 0 * 8 * C * 4 : OFF_BETA));
  float *e1c_s = reinterpret_cast<float *>(smem + (ALONE ? OFF_RING_2 + 1 * 8 * C * 4 : OFF_E1C));
  float *e2_s = reinterpret_cast<float *>(smem + (ALONE ? OFF_RING_2 + 2 * 8 * C * 4 : OFF_E2));
  float *bte1_s = reinterpret_cast<float *>(smem + (ALONE ? OFF_RING_2 + 3 * 8 * C * 4 : OFF_BTE1));
  float *fin_s = reinterpret_cast<float *>(smem + OFF_FIN);
  Unit *const units = reinterpret_cast<Unit *>(smem + OFF_UNIT);
  Misc *misc = reinterpret_cast<Misc *>(smem + OFF_MISC);

  const int tid = threadIdx.x, warp = uni(tid >> 5), lane = tid & 31;
  const int64_t v_stride = static_cast<int64_t>(a.H_v) * D;

  // ---- set-up: barriers and tensor memory ----
  if (tid == 0) {
    for (int i = 0; i < F::BUF; ++i) {
      mbar_init(&misc->rdy_prep[i], NP / 32 + (KDA && !ALONE ? 1 : 0));
      mbar_init(&misc->bar_ap[i], 1);
      mbar_init(&misc->bar_ro[i], 1);
      mbar_init(&misc->g_full[i], 4);
      mbar_init(&misc->kq_full[i], WITH_O ? 4 : 2);
    }
    for (int i = 0; i < 2; ++i) mbar_init(&misc->bar_s[i], 1);
    for (int i = 0; i < FAC; ++i) mbar_init(&misc->rdy_fac[i], KDA ? 4 : 1);
    mbar_init(&misc->bar_u, 1);
    mbar_init(&misc->bar_o, 1);
    mbar_init(&misc->rdy_state, NCH / 32);
    mbar_init(&misc->rdy_half, NCH / 32);
    mbar_init(&misc->rdy_rhs, NCH / 32 + (ALONE ? (WITH_O ? 5 : 1) : 0));
    mbar_init(&misc->rdy_u, NCH / 32);
    mbar_init(&misc->a_taken, 1);
    mbar_init(&misc->rdy_t, 1);
    mbar_init(&misc->tp_free, NCH / 32);
    mbar_init(&misc->drain, 1);
    mbar_init(&misc->drain_1, 1);

    mbar_init(&misc->v_full, 2);
    misc->abort_flag = 0;
    for (int i = 0; i < 4; ++i) misc->domain_flag[i] = 0;
    fence_mbar_init();
  }
  if (warp == WARP_MMA) {
    tmem_alloc(&misc->tmem_base, F::TMEM_COLS);
    tmem_relinquish();
  }
  // This CTA's units, a lane of one warp each: every gridDim.x-th, there and back (see grid_for; one where WALK is false).  Which they are is worked out
  // before the wait for earlier work, their tokens and state are looked up behind it.
  if (warp == WARP_T) {
    const int64_t idx = static_cast<int64_t>(lane) * gridDim.x + ((lane & 1) ? gridDim.x - 1u - blockIdx.x : blockIdx.x);
    bool here = lane < (WALK ? kMaxWalk : 1) && idx < static_cast<int64_t>(a.n_req) * a.n_layers_in_call * a.H_v;
    const uint32_t row = static_cast<uint32_t>(idx) / a.H_v;  // (the host sees to it that units fit 31 bits)
    Unit x;
    x.head = static_cast<int32_t>(static_cast<uint32_t>(idx) - row * a.H_v);
    x.k_head = KDA && a.H_k == a.H_v ? x.head : x.head / (a.H_v / a.H_k);
    int r = static_cast<int>(row / a.n_layers_in_call);
    const int lc = static_cast<int>(row) - r * a.n_layers_in_call;
    x.keep_row = (a.layer_begin + lc) * static_cast<int32_t>(a.rows_per_layer) + x.head * D;
    x.n_tok = 0;
    stream_order_wait();
    if (here) {
      if (a.ordered) r = static_cast<const uint8_t *>(a.workspace)[kRefreshWsOrder + r];
      const int t_begin = a.tok_begin ? a.tok_begin[r] : a.cu_seqlens[r];
      x.n_tok = max(a.cu_seqlens[r + 1] - t_begin, 0);
      x.tok0 = static_cast<int64_t>(lc) * a.total_tokens + t_begin;
      x.state = a.req_idx[r] * a.req_stride + (a.layer_begin + lc) * a.layer_stride + x.head * (D * D);
      x.index = (r * a.n_layers_in_call + lc) * a.H_v + x.head;
      if (x.n_tok == 0 && a.mode == DASC_REFRESH_CONTINUE) {
        here = false;
      } else if (x.n_tok <= a.short_thr) {  // left to the exact kernel (short_thr = -1: never)
        hand_over(a, x.index, false);
        here = false;
      }
    }
    const uint32_t with = __ballot_sync(0xffffffffu, here && x.n_tok > 0), without = __ballot_sync(0xffffffffu, here && x.n_tok == 0);
    const uint32_t before = (1u << lane) - 1u;
    if (here) units[x.n_tok > 0 ? __popc(with & before) : __popc(with) + __popc(without & before)] = x;  // those without tokens last
    const int chunks = __reduce_add_sync(0xffffffffu, here ? (x.n_tok + C - 1) / C : 0);
    if (lane == 0) {
      misc->n_units = __popc(with | without);
      misc->n_replayed = __popc(with);
      misc->all_chunks = chunks;
    }
  } else {
    stream_order_wait();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tm = static_cast<uint32_t>(uni(static_cast<int>(misc->tmem_base)));
  const int all_chunks = uni(misc->all_chunks);  // of all the CTA's units: buffers and barrier phases go by the index among these
  constexpr float LOG2E = 1.4426950408889634f;

  constexpr uint32_t ID_N32 = idesc_tf32(128, 32, false, false);
  constexpr uint32_t ID_M64 = idesc_tf32(64, 32, false, false), ID_BF16_M64 = idesc_bf16(64, 32);
  constexpr uint32_t ID_N64 = idesc_tf32(128, 64, false, false);
  constexpr uint32_t ID_N128_MN = idesc_tf32(128, 128, false, true);  // B = Kh[t][c]: the channel index N is the contiguous one

  auto mma1 = [&](int n) {
    // MMA1: [Kt;Qt] Kh^T, M = 64: 16 rows in each TMEM quadrant, A's in the first two, P's in the last two.
    wait_bar(&misc->rdy_prep[buf(n)], phase(n), misc);
    tc_fence_after_sync();
    if (elect_one()) {
      if constexpr (KDA) {
#pragma unroll
        for (int kk = 0; kk < 16; ++kk)  // K = 128 in slices of 8: block kk / 4, 32 bytes per slice inside a block
          mma_ss(tm + col_ap(n), desc_kmajor(sbase + off_kq(n) + (kk >> 2) * (64 * 128) + (kk & 3) * 32),
                 desc_kmajor(sbase + off_kh(n) + (kk >> 2) * (32 * 128) + (kk & 3) * 32), ID_M64, kk != 0);
      } else {
        // GDN: the decay is one scalar per token, so it is applied to A and P after the product, and the product
        // itself is [k; q] k^T on the raw bf16 inputs: exact operands, K = 16 per instruction.  A and B come from
        // the same tile (B = its first 32 rows).
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const uint64_t d = desc_kmajor(sbase + off_kh(n) + (kk >> 2) * (64 * 128) + (kk & 3) * 32);
          mma_ss_bf16(tm + col_ap(n), d, d, ID_BF16_M64, kk != 0);
        }
      }
      mma_commit(&misc->bar_ap[buf(n)]);
    }
    __syncwarp();
  };
  // Test hook: a first, short wait for the tiles of the first chunk, by the warp that issues MMA1, as soon as nothing but copies that have
  // just been started can have gone into them.
  auto first_wait = [&]() {
    if (a.poll_limit_first_wait && all_chunks > 0) wait_bar_short(&misc->rdy_prep[0], 0, misc, a.poll_limit_first_wait);
  };
  auto take_a = [&](int n) {
    // rows 16-31 of A are in this warp's quadrant: hand them to the triangular warp
    wait_bar(&misc->bar_ap[buf(n)], phase(n), misc);
    if (ALONE && n > 0) wait_bar(&misc->rdy_rhs, (n - 1) & 1, misc);  // the triangular warp has read the chunk before's
    tc_fence_after_sync();
    take_a_rows<KDA>(tm + (32u << 16) + col_ap(n), 16, (KDA ? beta_s : bte1_s) + (n % RING) * C, e2_s + (n % RING) * C, Lm, lane);
    // A full barrier on both sides: after a time-out no wait below keeps this warp from the next chunk, and a second bare arrival of its own
    // would complete the barrier without the triangular warp, which would later wait for an arrival that never comes.
    asm volatile("bar.sync 3, 64;" ::: "memory");
  };
  // where a chunk's raw k, q lie: rows of a 64-channel block, and q behind k
  constexpr uint32_t RAW_ROWS = KDA ? 32 : 64, OFF_RAW_Q = KDA ? 2 * 32 * 128 : 32 * 128;
  // ---- the two steps that the chain warps take, or warps of their own ----
  // P = lower_incl_diag(Qt Kh^T) of chunk n out of TMEM (rows 0-15, 16-31 are in the third and fourth quadrant) straight to its operand
  // tile, 16 columns.  GDN: the raw q_t . k_j gets its column factor e2_j here, the row factor e1_t is applied to the outputs.
  const int quad = warp & 3;                                             // TMEM lane quadrant
  const uint32_t tlane = tm + (static_cast<uint32_t>(quad * 32) << 16);  // this warp's TMEM lanes
  const int g = lane >> 2, tig = lane & 3;
  auto take_p = [&](int n, int colh) {
    wait_bar(&misc->bar_ap[buf(n)], phase(n), misc);
    tc_fence_after_sync();
    uint32_t x[8];
    tmem_ld_16x256b(tlane + col_ap(n) + colh * 16, x);
    if (!ALONE && n > 0) wait_bar(&misc->tp_free, (n - 1) & 1, misc);  // the previous chunk's outputs have left this storage
    tmem_ld_wait();
    const int t = (quad - 2) * 16 + g;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int j = colh * 16 + 8 * i + 2 * tig;
      float2 e = make_float2(kInvTruncComp, kInvTruncComp);
      if constexpr (!KDA) {
        const float2 e2 = *reinterpret_cast<const float2 *>(e2_s + (n % RING) * C + j);
        e.x *= e2.x;
        e.y *= e2.y;
      }
      unsigned char *const p = smem + OFF_PM + sw128_offset(32, t, j);
      *reinterpret_cast<uint2 *>(p) = make_uint2(j <= t ? tf32_pre(__uint_as_float(x[4 * i]) * e.x) : 0u,
                                                 j + 1 <= t ? tf32_pre(__uint_as_float(x[4 * i + 1]) * e.y) : 0u);
      *reinterpret_cast<uint2 *>(p + 1024) = make_uint2(j <= t + 8 ? tf32_pre(__uint_as_float(x[4 * i + 2]) * e.x) : 0u,
                                                        j + 1 <= t + 8 ? tf32_pre(__uint_as_float(x[4 * i + 3]) * e.y) : 0u);
    }
    fence_smem_to_async();
  };
  // Outputs of chunk n, of which `ntok` tokens are the request's: one token half (SHARED: the warp's) or both
  // by this warp, thread ti of those that take them.  The caller has waited for bar_o; no second wait for it here, since in the ALONE form
  // product 4 of the next chunk is on its way by then and could turn the parity first.
  auto outputs = [&](int n, int ntok, OT *go, int half_0, int ti) {
    constexpr int NTH = ALONE ? 128 : NCH;
    tc_fence_after_sync();
    if (WITH_O) {
#pragma unroll
      for (int k = 0; k < F::BUF; ++k) {
        const int tb = (half_0 + k) * 16;
        const int ot = tb + (lane >> 4) * 8 + (lane & 7);  // blocks of one stmatrix: as for V
        uint32_t xx[2][8];
        tmem_ld_16x256b(tlane + col_ro(n) + 32 + tb, xx[0]);
        tmem_ld_16x256b(tlane + (1u << 20) + col_ro(n) + 32 + tb, xx[1]);
        tmem_ld_wait();
#pragma unroll
        for (uint32_t hh = 0; hh < 2; ++hh) {
          uint32_t(&x)[8] = xx[hh];
          if constexpr (!KDA) {
            // GDN: the accumulated q_t (S' + sum_j e2_j k_j u_j^T) still lacks its row factor e1_t, the query scale and
            // the truncation compensation
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const float2 e = *reinterpret_cast<const float2 *>(e1c_s + (n % RING) * C + tb + 8 * i + 2 * tig);
              x[4 * i + 0] = __float_as_uint(__uint_as_float(x[4 * i + 0]) * (e.x * a.q_scale));
              x[4 * i + 1] = __float_as_uint(__uint_as_float(x[4 * i + 1]) * (e.y * a.q_scale));
              x[4 * i + 2] = __float_as_uint(__uint_as_float(x[4 * i + 2]) * (e.x * a.q_scale));
              x[4 * i + 3] = __float_as_uint(__uint_as_float(x[4 * i + 3]) * (e.y * a.q_scale));
            }
          }
          if constexpr (sizeof(OT) == 2) {
            uint32_t w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) w[i] = pack_bf16x2(__uint_as_float(x[2 * i]), __uint_as_float(x[2 * i + 1]));
            stmatrix_x4_trans(sbase + OFF_O + ot * 256 + (((quad * 4 + hh * 2 + ((lane >> 3) & 1)) ^ (ot & 7)) << 4), w[0], w[1], w[2], w[3]);
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int t = tb + (i >> 1) * 8 + 2 * tig, v = quad * 32 + hh * 16 + (i & 1) * 8 + g;
              if (t < ntok) go[t * v_stride + v] = __uint_as_float(x[2 * i]);
              if (t + 1 < ntok) go[(t + 1) * v_stride + v] = __uint_as_float(x[2 * i + 1]);
            }
          }
        }
      }
      if constexpr (sizeof(OT) == 2) {
        // through shared memory (SHARED: where the T and P tiles were, which are free now) so that global stores are 16 bytes wide
        asm volatile("bar.sync %0, %1;" ::"n"(ALONE ? 6 : 1), "n"(NTH) : "memory");
        const int j = ti & 15;
#pragma unroll
        for (int i = 0; i < C / (NTH / 16); ++i) {
          const int t = (ti >> 4) + NTH / 16 * i;
          if (t < ntok)
            *reinterpret_cast<uint4 *>(go + i * (NTH / 16) * v_stride) =
                *reinterpret_cast<const uint4 *>(smem + OFF_O + t * 256 + ((j ^ (t & 7)) << 4));
        }
      }
    }
  };

  if (warp == WARP_MMA) {
    // =========================== tensor-core issue warp ===========================
    // The whole warp walks the chunks and waits; an elected lane issues.
    if (!ALONE) first_wait();
    int left = 0, next_u = 0;  // ZERO: chunks left of the unit; the unit behind it
    for (int n = 0; n < all_chunks; ++n) {
      const uint32_t par = n & 1;
      bool zero = false;  // this chunk's start state is zero, and nothing has been written where it would be
      if (ZERO) {
        zero = left == 0;
        if (zero) left = (uni(units[next_u++].n_tok) + C - 1) / C;
        --left;
      }
      if (!ALONE) {
        mma1(n);
        take_a(n);
      }
      // MMA2: S'^T [Kt;Qt]^T, the fp32 state read as a tf32 operand
      // (GDN in ALONE unrolled by two: 4 units of 2000 tokens 115.2 -> 112.5 us, 32 of 509 35.1 -> 34.3, 148 of 512 41.1 -> 40.9.  KDA by four: 4 of 2000
      // 126.4 -> 124.5, but 148 of 512 48.3 -> 49.1.  SHARED keeps its code small.)
      auto mma2 = [&](int kb_0, int kb_n) {
#pragma unroll ALONE && !KDA ? 2 : 1
        for (int kb = kb_0; kb < kb_n; ++kb) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            mma_ts(tm + col_ro(n), tm + COL_S + kb * 32 + kk * 8, desc_kmajor(sbase + off_kq(n) + kk * 32) + kb * (64 * 128 / 16),
                   WITH_O ? ID_N64 : ID_N32, (kb | kk) != 0);  // without outputs only the Kt rows are needed
        }
      };
      if (ALONE) {
        wait_bar(&misc->bar_ap[buf(n)], phase(n), misc);  // the tiles of this chunk are there: the warp that issued MMA1 has waited for them
        wait_bar(&misc->rdy_half, par, misc);
        tc_fence_after_sync();
        if (!zero && elect_one()) mma2(0, 2);
        __syncwarp();
      }
      wait_bar(&misc->rdy_state, par, misc);
      tc_fence_after_sync();
      if (elect_one()) {
        if (!zero) mma2(ALONE ? 2 : 0, 4);
        mma_commit(&misc->bar_ro[buf(n)]);
      }
      __syncwarp();
      // MMA3: U^T = RHS^T T^T; RHS^T is a tf32 pair (high part over R^T, low part in the A|P columns)
      if (!ALONE) wait_bar(&misc->rdy_t, par, misc);  // (ALONE: the triangular and the output warps arrive on rdy_rhs)
      wait_bar(&misc->rdy_rhs, par, misc);
      tc_fence_after_sync();
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)
          mma_ts(tm + COL_U<ALONE>, tm + (kk < 4 ? col_ro(n) : COL_RL) + (kk & 3) * 8, desc_kmajor(sbase + off_t(n) + (kk & 3) * 32),
                 ID_N32, kk != 0);
        mma_commit(&misc->bar_u);
      }
      __syncwarp();
      // U^T stays where MMA3 leaves it: read as an operand, each fp32 value gives its high (truncated) part, and
      // the chain warps supply the exact remainder afterwards (U = U_hi + U_lo).  The high-part products go out
      // without a round trip through the chain warps:
      // MMA4 (high): O^T += U_hi^T P^T;  MMA5 (high): S'^T += U_hi^T Kh
      // U must have arrived in tensor memory before another product reads it as its A operand: the tensor pipe's issue
      // order does not see to that (it orders accumulators only).
      // ALONE: the state's product first, it is what the chain waits for; SHARED: the chain warps take the outputs next.
      auto mma4 = [&](uint32_t u_t) {
        if (WITH_O) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            mma_ts(tm + col_ro(n) + 32, tm + u_t + kk * 8, desc_kmajor(sbase + OFF_PM + kk * 32), ID_N32, true);
        }
      };
      auto mma5 = [&](uint32_t u_t, bool add) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_ts(tm + COL_S, tm + u_t + kk * 8, desc_mn32(sbase + off_kht(n) + kk * 1024, 32 * 128), ID_N128_MN, add || kk != 0);
      };
      wait_bar(&misc->bar_u, par, misc);
      tc_fence_after_sync();
      if (elect_one()) {
        if (!ALONE) mma4(COL_U<ALONE>);
        mma5(COL_U<ALONE>, !zero);
      }
      __syncwarp();
      // MMA4 (low), MMA5 (low): the same with U_lo^T, which the chain warps wrote over the consumed RHS^T
      wait_bar(&misc->rdy_u, par, misc);
      tc_fence_after_sync();
      if (elect_one()) {
        if (ALONE) {
          mma5(col_ro(n), true);
          mma_commit(&misc->bar_s[par]);
          mma4(COL_U<ALONE>);
        }
        mma4(col_ro(n));
        if (WITH_O || !ALONE) mma_commit(&misc->bar_o);  // (only where someone waits for it: an arrival must not outlive the CTA)
        if (!ALONE) {
          mma5(col_ro(n), true);
          mma_commit(&misc->bar_s[par]);
        }
      }
      __syncwarp();
    }
    // After a time-out the other roles no longer wait for the products: make sure none is still in flight when the
    // tensor memory is given back (a real wait, bounded like the others).
    if (misc->abort_flag) {
      if (elect_one()) mma_commit(&misc->drain);
      __syncwarp();
      mbar_wait_bounded(&misc->drain, 0, kMaxPolls);
    }
    __syncwarp();
  } else if (warp == WARP_T) {
    // ================================ triangular warp ================================
    // T = (I + A)^-1 depends on the token inputs only, so it is formed off the chain: rows 0-15 of A out of TMEM (this
    // warp's quadrant; the issuing warp brings rows 16-31), 16x16 diagonal blocks by fp32 substitution, the off-diagonal
    // block by mma.sync products.  (GDN: by rows of the inverse and from -A, KDA by its columns and from A^T: see below.)
    // This warp also starts the copies of V, a chunk ahead: two boxes of 32 tokens x 64 values with the 128-byte swizzle (no bank
    // conflicts for the 8 x 8 blocks it is read in).  Started by two of the chain warps they held those up for 280 cycles of every
    // chunk; here they fall into the wait for the next A (0.3 to 1 % of a launch).
    // HELD: the next copy's unit in registers.  GDN looks it up where the copy is started in a walk, whose inverse by rows left no room for
    // it (16 bytes spilled, 4 without outputs; 592 units of 1 .. 1199 tokens 143 us both ways); with a unit per CTA it is kept, since looked up it
    // cost 1 % (296 units of 300 tokens 39.1 / 39.7 us).
    constexpr bool HELD = KDA || !WALK;
    int v_issued = 0, v_unit = 0, v_tok = 0;  // copies started; the next one's unit, its first token in that,
    int v_n = 0, v_row = 0, v_head = 0;       // of how many, and its coordinates
    auto next_v = [&]() {
      v_tok = 0;
      if (HELD) {
        v_n = units[v_unit].n_tok;
        v_row = static_cast<int32_t>(units[v_unit].tok0);
        v_head = units[v_unit].head;
      }
    };
    if (all_chunks > 0) next_v();
    auto stage_v = [&]() {  // (the copies by the first lane)
      if (lane == 0 && !misc->abort_flag) {
        const Unit &x = units[v_unit];
        const int head = HELD ? v_head : x.head, row = HELD ? v_row : static_cast<int32_t>(x.tok0) + v_tok;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          mbar_expect_tx(&misc->v_full, C * 128);
          tma_load_3d(sbase + OFF_V + i * (C * 128), &tmap_v, i * 64, head, row, &misc->v_full);
        }
        // the state that the unit starts from, 64 KB in one piece, is brought into L2 meanwhile
        if (WALK && v_tok == 0 && v_issued > 0 && a.mode == DASC_REFRESH_CONTINUE)
          asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a.state + units[v_unit].state), "n"(D * D * 4) : "memory");
        ++v_issued;
      }
      v_tok += C;
      if (HELD) v_row += C;
      if (WALK && v_tok >= (HELD ? v_n : units[v_unit].n_tok) && ++v_unit < misc->n_replayed) next_v();
    };
    // KDA: it also brings in beta, a chunk ahead, and arrives on rdy_prep (ALONE: the MMA1 warp; GDN: the producer warps, whose per-token
    // factors contain it).
    auto fetch_beta = [&]() {  // of the chunk whose copy comes next, lane = token
      return lane < v_n - v_tok ? a.beta[static_cast<int64_t>(v_row + lane) * a.H_v + v_head] : 0.f;
    };
    if (all_chunks > 0) {
      if (KDA && !ALONE) {
        beta_s[lane] = fetch_beta();
        arrive_warp(&misc->rdy_prep[0], lane);
      }
      stage_v();
    }
    for (int n = 0; n < all_chunks; ++n) {
      const uint32_t par = n & 1;
      float beta_next = 0.f;
      if (KDA && !ALONE && n + 1 < all_chunks) beta_next = fetch_beta();
      wait_bar(&misc->bar_ap[buf(n)], phase(n), misc);
      tc_fence_after_sync();
      take_a_rows<KDA>(tm + col_ap(n), 0, (KDA ? beta_s : bte1_s) + (n % RING) * C, e2_s + (n % RING) * C, Lm, lane);
      tc_fence_before_sync();
      asm volatile("bar.sync 3, 64;" ::: "memory");
      arrive_warp(&misc->a_taken, lane);  // the chain warps may reuse the A|P columns
      // X = (I + A)^-1, then T, to its tf32 operand tile straight from the registers.  The tile's storage (shared with the P tile and the chain
      // warps' output tile) is free once the chain warps have copied the previous chunk's outputs out.
      auto storage_free = [&]() {
        if (!ALONE && n > 0) wait_bar(&misc->tp_free, par ^ 1, misc);
      };
      // Where two CTAs share an SM T is the last operand of MMA3 to be ready, and how long it takes is this warp's count of instructions.  GDN
      // by rows of X, a chunk's 6195 warp instructions become 6037 (us, by columns / by rows: 152 units of 256 tokens 32.4 / 31.4, 296 of 300 40.5 / 39.1, 424 of
      // 300 74.6 / 65.5, 296 of 1 .. 1999 157 / 152; ALONE: 148 of 512 43.2 / 41.2, 4 of 2000 116.8 / 115.5).  KDA by columns: by rows SHARED
      // gained at most 2 %, and 148 units of 512 tokens went from 48.9 to 43.7, but calls of few units got slower, 4 of 2000 125.5 -> 131.1, 32 of
      // 509 38.7 -> 39.6, wherever in the chunk this step was put (why is not known); and all forms have to give the same bits, so SHARED alone cannot have it.  In between, 8x8
      // diagonal blocks and products of hi / lo pairs: KDA 4 of 2000 128.4, but GDN 152 of 256 33.2, 424 of 300 75.7.
      if constexpr (KDA) {
        // diagonal 16x16 blocks: lane (block b, column cc) solves (I + L_bb) x = e_cc, column by column: every row that a new
        // entry of x acts on is updated at once, so the serial chain is one multiply-add per row
        {
          const int b = lane >> 4, cc = lane & 15;
          const float *Lb = Lm + (b * 16) * LDX + b * 16;
          float xs[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) xs[i] = i == cc ? 1.f : 0.f;
#pragma unroll
          for (int j = 0; j < 15; ++j) {
#pragma unroll
            for (int r4 = (j + 1) / 4 * 4; r4 < 16; r4 += 4) {
              const float4 l4 = *reinterpret_cast<const float4 *>(Lb + j * LDX + r4);
              if (r4 + 0 > j) xs[r4 + 0] = fmaf(-l4.x, xs[j], xs[r4 + 0]);
              if (r4 + 1 > j) xs[r4 + 1] = fmaf(-l4.y, xs[j], xs[r4 + 1]);
              if (r4 + 2 > j) xs[r4 + 2] = fmaf(-l4.z, xs[j], xs[r4 + 2]);
              if (r4 + 3 > j) xs[r4 + 3] = fmaf(-l4.w, xs[j], xs[r4 + 3]);
            }
          }
#pragma unroll
          for (int rr = 0; rr < 16; ++rr) Xm[(b * 16 + rr) * LDX + b * 16 + cc] = xs[rr];
          __syncwarp();
          // off-diagonal block: X_10 = -X_11 (L_10 X_00); the product L_10 X_00 is parked in the unused block (0,1)
          float acc[2][4] = {};
          warp_mm_acc<true>(acc, Lm + 16, Xm, lane);
          warp_mm_store(Xm + 16, acc, 1.f, lane);
          storage_free();
#pragma unroll
          for (int rr = 0; rr < 16; ++rr)
            *reinterpret_cast<uint32_t *>(smem + off_t(n) + sw128_offset(32, b * 16 + rr, b * 16 + cc)) = tf32_pre(xs[rr]);
#pragma unroll
          for (int i = 0; i < 2; ++i)
            *reinterpret_cast<uint4 *>(smem + off_t(n) + sw128_offset(32, i * 8 + (lane >> 2), 16 + (lane & 3) * 4)) = make_uint4(0u, 0u, 0u, 0u);
        }
        __syncwarp();
        {
          float acc2[2][4] = {};
          warp_mm_acc<false>(acc2, Xm + 16 * LDX + 16, Xm + 16, lane);
          const int g = lane >> 2, tig = lane & 3;
#pragma unroll
          for (int nh = 0; nh < 2; ++nh) {
            unsigned char *const p = smem + off_t(n) + sw128_offset(32, 16 + g, 8 * nh + 2 * tig);
            *reinterpret_cast<uint2 *>(p) = make_uint2(tf32_pre(-acc2[nh][0]), tf32_pre(-acc2[nh][1]));
            *reinterpret_cast<uint2 *>(p + 1024) = make_uint2(tf32_pre(-acc2[nh][2]), tf32_pre(-acc2[nh][3]));
          }
        }
      } else {
        // By rows: lane (block b, row i) solves x (I + A_bb) = e_i, from the diagonal down: all entries that a new one acts on are updated at
        // once, in pairs, so the serial chain is one multiply-add per entry, and a lane's entries leave 16 bytes at a time.
        const int g = lane >> 2, tig = lane & 3;
        {
          const int b = lane >> 4, row = lane & 15;
          const float *const Lb = Lm + (b * 16) * LDL + b * 16;
          uint64_t x[8];
#pragma unroll
          for (int p = 0; p < 8; ++p) x[p] = pack2(2 * p == row ? 1.f : 0.f, 2 * p + 1 == row ? 1.f : 0.f);
#pragma unroll
          for (int k = 15; k > 0; --k) {
            float lo, hi;
            unpack2(x[k >> 1], lo, hi);
            const float f = k & 1 ? hi : lo;
            const uint64_t f2 = pack2(f, f);
#pragma unroll
            for (int j4 = 0; j4 < k; j4 += 4) {
              const ulonglong2 l = *reinterpret_cast<const ulonglong2 *>(Lb + k * LDL + j4);
#pragma unroll
              for (int p = 0; p < 2; ++p) {
                const int j = j4 + 2 * p;
                const uint64_t l2 = p ? l.y : l.x;
                if (j + 1 < k) {
                  x[j >> 1] = fma2(f2, l2, x[j >> 1]);
                } else if (j < k) {  // the pair of entry k itself: its first entry only
                  float l0, l1;
                  unpack2(l2, l0, l1);
                  x[j >> 1] = pack2(fmaf(f, l0, lo), hi);
                }
              }
            }
          }
          float xs[16];
#pragma unroll
          for (int p = 0; p < 8; ++p) unpack2(x[p], xs[2 * p], xs[2 * p + 1]);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            *reinterpret_cast<float4 *>(Xm + lane * LDX + b * 16 + 4 * q) = make_float4(xs[4 * q], xs[4 * q + 1], xs[4 * q + 2], xs[4 * q + 3]);
          storage_free();
          const uint32_t t0 = sw128_offset(32, lane, b * 16);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            *reinterpret_cast<uint4 *>(smem + off_t(n) + (t0 ^ (q << 4))) =
                make_uint4(tf32_pre(xs[4 * q]), tf32_pre(xs[4 * q + 1]), tf32_pre(xs[4 * q + 2]), tf32_pre(xs[4 * q + 3]));
#pragma unroll
          for (int i = 0; i < 2; ++i)
            *reinterpret_cast<uint4 *>(smem + off_t(n) + sw128_offset(32, i * 8 + (lane >> 2), 16 + (lane & 3) * 4)) = make_uint4(0u, 0u, 0u, 0u);
        }
        __syncwarp();
        // off-diagonal block: X_10 = X_11 (-A_10 X_00).  The inner product transposed, and the contraction index of a slice of 8 taken as
        // 2 tig, 2 tig + 1: its accumulators are then the outer product's second operand as they are.
        {
          float m[2][4] = {}, acc[2][4] = {};  // m[half of A_10's rows]: rows = columns of X_00, columns = rows of A_10
#pragma unroll
          for (int kh = 0; kh < 2; ++kh) {
            const float *const x0 = Xm + (8 * kh + 2 * tig) * LDX + g;
            const uint32_t af[4] = {tf32_pre(x0[0]), tf32_pre(x0[8]), tf32_pre(x0[LDX]), tf32_pre(x0[LDX + 8])};
#pragma unroll
            for (int rh = 0; rh < 2; ++rh) {
              const float2 l10 = *reinterpret_cast<const float2 *>(Lm + (16 + 8 * rh + g) * LDL + 8 * kh + 2 * tig);
              const uint32_t bf[2] = {tf32_pre(l10.x), tf32_pre(l10.y)};
              mma_tf32_16x8x8(m[rh], af, bf);
            }
          }
#pragma unroll
          for (int kh = 0; kh < 2; ++kh) {
            const float *const x1 = Xm + (16 + g) * LDX + 16 + 8 * kh + 2 * tig;
            const float2 r0 = *reinterpret_cast<const float2 *>(x1), r1 = *reinterpret_cast<const float2 *>(x1 + 8 * LDX);
            const uint32_t af[4] = {tf32_pre(r0.x), tf32_pre(r1.x), tf32_pre(r0.y), tf32_pre(r1.y)};
#pragma unroll
            for (int ch = 0; ch < 2; ++ch) {
              const uint32_t bf[2] = {tf32_pre(m[kh][2 * ch]), tf32_pre(m[kh][2 * ch + 1])};
              mma_tf32_16x8x8(acc[ch], af, bf);
            }
          }
#pragma unroll
          for (int ch = 0; ch < 2; ++ch) {
            unsigned char *const p = smem + off_t(n) + sw128_offset(32, 16 + g, 8 * ch + 2 * tig);
            *reinterpret_cast<uint2 *>(p) = make_uint2(tf32_pre(acc[ch][0]), tf32_pre(acc[ch][1]));
            *reinterpret_cast<uint2 *>(p + 1024) = make_uint2(tf32_pre(acc[ch][2]), tf32_pre(acc[ch][3]));
          }
        }
      }
      fence_smem_to_async();
      arrive_warp(ALONE ? &misc->rdy_rhs : &misc->rdy_t, lane);  // -> MMA3
      if (n + 1 < all_chunks) {  // once V has been read by every chain warp the next chunk's may land
        if (KDA && !ALONE) {
          beta_s[((n + 1) % RING) * C + lane] = beta_next;
          arrive_warp(&misc->rdy_prep[0], lane);
        }
        wait_bar(&misc->rdy_rhs, par, misc);
        stage_v();
      }
      __syncwarp();
    }
    // after a time-out the last copies of V may not have been waited for: they must have landed before the CTA leaves
    if (lane == 0 && misc->abort_flag && v_issued > 0) mbar_wait_bounded(&misc->v_full, (v_issued - 1) & 1, kMaxPolls);
  } else if (ALONE && warp == WARP_MMA1) {
    // ================================= MMA1, input copies (ALONE) =================================
    // MMA1 goes out behind MMA2 of the chunk before, i.e. while the chain warps form its right-hand side.  By then A and P of two chunks
    // ago, whose columns are written again, have been read.  Copies are two chunks ahead, a box per lane: KDA the log-decay by lanes 0-3;
    // k by lanes 4, 5; q by lanes 6, 7.
    const Unit &x = units[0];
    const bool copies_g = KDA && lane < 4, copies_kq = lane >= 4 && lane < (WITH_O ? 8 : 6);
    int issued = 0;
    auto copy = [&](int n) {
      if ((copies_g || copies_kq) && !misc->abort_flag) {
        const int32_t z = static_cast<int32_t>(x.tok0 + n * C);
        uint64_t *const full = copies_g ? &misc->g_full[buf(n)] : &misc->kq_full[buf(n)];
        const uint32_t raw = sbase + (KDA ? off_kht(n) : off_kh(n)) + (lane & 1) * (RAW_ROWS * 128);
        mbar_expect_tx(full, C * 128);
        if (copies_g)
          tma_load_3d(sbase + off_kh(n) + lane * (C * 128), &tmap_g, lane * 32, x.head, z, full);
        else if (lane < 6)
          tma_load_3d(raw, &tmap_k, (lane & 1) * 64, x.k_head, z, full);
        else
          tma_load_3d(raw + OFF_RAW_Q, &tmap_q, (lane & 1) * 64, x.k_head, z, full);
        issued = n + 1;
      }
      __syncwarp();
    };
    for (int n = 0; n < 2 && n < all_chunks; ++n) copy(n);
    first_wait();
    // KDA: beta as well, lane = token, into its ring before MMA1 goes out (its readers wait for that product)
    auto fetch_beta = [&](int n) { return lane < x.n_tok - n * C ? a.beta[(x.tok0 + n * C + lane) * a.H_v + x.head] : 0.f; };
    float beta = KDA && all_chunks > 0 ? fetch_beta(0) : 0.f;
    for (int n = 0; n < all_chunks; ++n) {
      if (KDA) {
        beta_s[(n % RING) * C + lane] = beta;
        __syncwarp();
        beta = fetch_beta(n + 1);
      }
      if (n > 0) wait_bar(&misc->bar_ro[buf(n - 1)], phase(n - 1), misc);
      mma1(n);
      take_a(n);
      // MMA1 has read what the copies land on (KDA: the K-major Kh; GDN: raw k, q).  KDA, raw k, q: the MN-major tile, of which there are
      // four, was read by MMA5 of two chunks ago, which the chain warps had seen complete before MMA2 of the chunk before.
      if (n + 2 < all_chunks) copy(n + 2);
    }
    // after a time-out the last copies, those of two chunks, may not have been waited for: they must have landed before the CTA leaves
    if (misc->abort_flag)
      for (int n = max(issued - 2, 0); n < issued; ++n)
        mbar_wait_bounded(copies_g ? &misc->g_full[buf(n)] : &misc->kq_full[buf(n)], phase(n), kMaxPolls);
    __syncwarp();
    // (after a time-out: as for the issuing warp)
    if (misc->abort_flag) {
      if (elect_one()) mma_commit(&misc->drain_1);
      __syncwarp();
      mbar_wait_bounded(&misc->drain_1, 0, kMaxPolls);
    }
    __syncwarp();
  } else if (ALONE && warp >= WARP_O) {
    // ================================= output warps (ALONE) =================================
    // P and the outputs off the chain: P of the next chunk as soon as the products that read this one's have completed.
    if (WITH_O && all_chunks > 0) {
      const int ti = tid - WARP_O * 32;
      OT *go = static_cast<OT *>(a.o) + (units[0].tok0 * a.H_v + units[0].head) * D;
      if (sizeof(OT) == 2) go += (ti >> 4) * v_stride + (ti & 15) * 8;
      auto next_p = [&](int n) {
        if (quad >= 2) {
          take_p(n, 0);
          take_p(n, 1);
        }
        // -> MMA3, whose issue also says that the outputs up to chunk n - 2 have left tensor memory (there are three buffers)
        arrive_warp(&misc->rdy_rhs, lane);
      };
      next_p(0);
      const int n_tok = uni(units[0].n_tok);
      for (int n = 0; n < all_chunks; ++n) {
        wait_bar(&misc->bar_o, n & 1, misc);
        if (n + 1 < all_chunks) next_p(n + 1);
        asm volatile("bar.sync 6, 128;" ::: "memory");  // all have copied the previous chunk's out of the O tile
        outputs(n, min(C, n_tok - n * C), go, 0, ti);
        go += C * v_stride;
        tc_fence_before_sync();
      }
    }
  } else if (warp >= 8) {
    // =============================== producer warps ===============================
    // warp = block of 32 channels; per half of the chunk, lane = (4 adjacent channels, 4 consecutive tokens), a 4 x 4
    // tile.  The midpoint is the end of the first half: first-half exponents are (local sum - the half's total),
    // second-half exponents the local sums themselves, so the halves are independent of one another.
    const int pw = ALONE ? (warp & 3) : warp - 8;  // ALONE: warps 8-11 take the first half of the tokens, 12-15 the second
    const int half_0 = ALONE ? (warp - 8) >> 2 : 0, half_n = ALONE ? half_0 + 1 : 2;
    const int cq = lane & 7, tg = lane >> 3;
    const int c0 = pw * 32 + cq * 4;
    // Inputs come by TMA a chunk ahead into tiles they will be overwritten with (KDA) or that are
    // operands as they are (GDN): shared memory holds no staging buffers, and no load or store instruction moves them.
    //   log-decay (KDA, the largest stream): four boxes of 32 tokens x 32 channels with the 128-byte swizzle, i.e. exactly
    //   the layout of the Kh tile, so that a lane finds the decay of its vectors where its Kh vectors go;
    //   raw k, q: two boxes each of 32 tokens x 64 channels.  KDA: into the MN-major Kh tile of the chunk's parity, written
    //   half by half once all producers have read that half (both layouts keep 16 tokens in 2 KB of every 4 KB).  GDN:
    //   the operand tile of MMA1 itself.
    int g_issued = 0, kq_issued = 0;
    // Each warp's first lane starts one box of each stream: a copy takes its issuing thread 200 to 300 cycles, and the warp that
    // issued all of them arrived 800 cycles behind the others.
    // token coordinate, head and key head of a chunk's copies, read ahead of the waits that the copies stand behind
    int32_t cp_tok = 0, cp_head = 0, cp_k_head = 0;
    auto next_copies = [&](const Unit &x, int t0) {
      cp_tok = static_cast<int32_t>(x.tok0 + t0);
      cp_head = x.head;
      cp_k_head = x.k_head;
    };
    auto stage_kq = [&](int n) {
      if (!WITH_O && pw >= 2) return;
      const uint32_t dst = sbase + (KDA ? off_kht(n) : off_kh(n)) + (pw & 1) * (RAW_ROWS * 128);
      uint64_t *const full = &misc->kq_full[0];
      mbar_expect_tx(full, C * 128);
      if (pw < 2)
        tma_load_3d(dst, &tmap_k, pw * 64, cp_k_head, cp_tok, full);
      else
        tma_load_3d(dst + OFF_RAW_Q, &tmap_q, (pw & 1) * 64, cp_k_head, cp_tok, full);
      ++kq_issued;
    };
    auto stage_g = [&](int n) {
      uint64_t *const full = &misc->g_full[0];
      mbar_expect_tx(full, C * 128);
      tma_load_3d(sbase + off_kh(n) + pw * (C * 128), &tmap_g, pw * 32, cp_head, cp_tok, full);
      ++g_issued;
    };
    if (!ALONE && lane == 0 && all_chunks > 0) {
      next_copies(units[0], 0);
      if (KDA) stage_g(0);
      stage_kq(0);
    }
    // GDN, per-token scalars, by the first warp (lane = token): a chunk's go to their ring slots (the chain warps are at most two
    // chunks behind) while MMA1 of the chunk before runs; the next chunk's are fetched then and stored one chunk later.
    float beta_next = 0.f, gsc_next = 0.f;
    auto fetch_scalars = [&](const Unit &x, int t0) {
      const bool here = lane < x.n_tok - t0;
      const int64_t off = (x.tok0 + t0 + lane) * a.H_v + x.head;
      beta_next = here ? a.beta[off] : 0.f;
      gsc_next = here ? a.g[off] : 0.f;
    };
    float post_prev = 0.f;  // the factor owed by the previous chunk
    // One scalar log-decay per token: the running sums and the per-token factors are formed here; nothing per
    // channel needs an exponential, and k, q stay exactly their bf16 values:
    //   e1_t = exp(G_t - G_m), e2_t = exp(G_m - G_t) with m the end of the first half;
    //   MMA1 works on raw k, q (bf16 tile), MMA2 on raw k, q widened to tf32 containers, MMA5 on k_t e2_t;
    //   e1_t goes onto the rows of A, R and the outputs where they leave tensor memory, e2_j onto the columns of A, P.
    auto scalars = [&](int n, int u, int t0) {  // chunk n of the CTA: the tokens of unit u from t0 on
      const int slot = (n % RING) * C + lane;
      const float beta = beta_next;
      beta_s[slot] = beta;
      float incl = gsc_next;
#pragma unroll
      for (int dlt = 1; dlt < 32; dlt <<= 1) {
        const float x = __shfl_up_sync(0xffffffffu, incl, dlt);
        if (lane >= dlt) incl += x;
      }
      const float tot0 = __shfl_sync(0xffffffffu, incl, 15);          // G_m: the first half's total
      const float tot1 = __shfl_sync(0xffffffffu, incl, 31) - tot0;   // G_C - G_m
      const float d2 = (incl - tot0) * LOG2E;
      const float e1 = ex2f(d2), e2 = ex2f(-d2);
      e1c_s[slot] = e1 * kTruncComp;
      e2_s[slot] = e2;
      bte1_s[slot] = beta * e1;
      if (lane == 0 && (!(fabsf(tot0) <= kMaxHalfDecay) || !(fabsf(tot1) <= kMaxHalfDecay))) misc->domain_flag[u & 3] = 1;  // also true for NaN
      // state factor from where the previous chunk left the state to this chunk's midpoint, and the factor owed after
      // it; scalars here, written for every channel so that the chain warps read them as they do for KDA
      if (t0 == 0) post_prev = 0.f;
      const float f = ex2f((post_prev + tot0) * LOG2E);
      post_prev = tot1;
      *reinterpret_cast<float4 *>(fac_s + (n % FAC) * D + lane * 4) = make_float4(f, f, f, f);
      if (lane == 0) post_s[n & 3] = tot1;
      arrive_warp(&misc->rdy_fac[n % FAC], lane);
      t0 += C;
      if (WALK && t0 >= units[u].n_tok) {
        t0 = 0;
        ++u;
      }
      if (n + 1 < all_chunks) fetch_scalars(units[u], t0);
    };
    if (!KDA && warp == 8 && all_chunks > 0) {
      fetch_scalars(units[0], 0);
      scalars(0, 0, 0);
    }
    int n_tok = units[0].n_tok;
    for (int n = 0, u = 0, t0 = 0; n < all_chunks; ++n) {
      const uint32_t par = n & 1;
      const int ntok = min(C, n_tok - t0);
      unsigned char *kht_tile = smem + off_kht(n);
      unsigned char *raw = KDA ? kht_tile : smem + off_kh(n);
      unsigned char *const kq_tile = smem + off_kq(n), *const kh_tile = smem + off_kh(n);
      // GDN: the per-token factors are visible to all producer warps.  ALONE: so is what the chunk before owes, and all have read that
      // chunk's raw inputs
      if (!KDA || ALONE) asm volatile("bar.sync 2, %0;" ::"n"(NP) : "memory");
      bool out_of_range = false;
      wait_bar(&misc->kq_full[buf(n)], phase(n), misc);
      if (KDA) wait_bar(&misc->g_full[buf(n)], phase(n), misc);
      if (ALONE && n > 1) wait_bar(&misc->bar_ro[buf(n)], phase(n - 2), misc);  // Kt/Qt of two chunks ago have been read
      const uint64_t l2e2 = pack2(LOG2E, LOG2E), comp2 = pack2(kLog2TruncComp, kLog2TruncComp);
      const uint64_t qs2 = pack2(a.q_scale, a.q_scale);
#pragma unroll 1
      for (int half = half_0; half < half_n; ++half) {
        const int tr = half * 16 + tg * 4;
        // This lane's vectors (token tr + j): tr is a multiple of 4, so the row's part of a swizzle is an exclusive or with j.
        const uint32_t or0 = sw128_offset_bf16(RAW_ROWS, tr, c0), ok0 = sw128_offset(64, tr, c0), oh0 = sw128_offset(32, tr, c0),
                       om0 = mn32_offset(32, tr, c0);
        const int left = ntok - tr;  // tokens of this request from this lane's first on
        uint2 kw[4], qw[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          unsigned char *p = raw + (or0 ^ (j << 4)) + j * 128;
          kw[j] = *reinterpret_cast<const uint2 *>(p);
          if (WITH_O) qw[j] = *reinterpret_cast<const uint2 *>(p + OFF_RAW_Q);
        }
        if (left < 4) {
          // the boxes reached past the request's last token and brought in other tokens' values (zeros past the end of
          // the stream): those keys are cleared, so that what they hold cannot matter
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j >= left) {
              kw[j] = make_uint2(0u, 0u);
              if (!KDA) *reinterpret_cast<uint2 *>(raw + (or0 ^ (j << 4)) + j * 128) = kw[j];
            }
        }
        if constexpr (KDA) {
          float4 g4[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) g4[j] = *reinterpret_cast<const float4 *>(kh_tile + (oh0 ^ (j << 4)) + j * 128);
          if (left < 4) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (j >= left) g4[j] = make_float4(0.f, 0.f, 0.f, 0.f);
          }
          // sums: this lane's total, the prefix over the four token groups of the warp (lanes 8 apart), the half's total
          float run0[4], tot[4];
          const float own[4] = {(g4[0].x + g4[1].x) + (g4[2].x + g4[3].x), (g4[0].y + g4[1].y) + (g4[2].y + g4[3].y),
                                (g4[0].z + g4[1].z) + (g4[2].z + g4[3].z), (g4[0].w + g4[1].w) + (g4[2].w + g4[3].w)};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float incl = own[i];
            float x = __shfl_up_sync(0xffffffffu, incl, 8);
            if (tg >= 1) incl += x;
            x = __shfl_up_sync(0xffffffffu, incl, 16);
            if (tg >= 2) incl += x;
            run0[i] = incl - own[i];                            // accumulated before this lane's first token
            tot[i] = __shfl_sync(0xffffffffu, incl, cq + 24);    // the half's total
            out_of_range |= !(fabsf(tot[i]) <= kMaxHalfDecay);   // also true for NaN
          }
          uint64_t ref01 = 0ull, ref23 = 0ull;  // minus the midpoint reference, in log2 units
          if (half == 0) {
            // The factor that takes the state from where the previous chunk left it to this chunk's midpoint needs
            // the first half's sums only: it is handed to the chain warps before the tiles are built.
            if (tg == 0) {
              const float4 pp = t0 > 0 ? *reinterpret_cast<const float4 *>(post_s + (par ^ 1) * D + c0) : make_float4(0.f, 0.f, 0.f, 0.f);
              *reinterpret_cast<float4 *>(fac_s + (n % FAC) * D + c0) =
                  make_float4(ex2f((pp.x + tot[0]) * LOG2E), ex2f((pp.y + tot[1]) * LOG2E), ex2f((pp.z + tot[2]) * LOG2E),
                              ex2f((pp.w + tot[3]) * LOG2E));
            }
            arrive_warp(&misc->rdy_fac[n % FAC], lane);
            ref01 = pack2(-tot[0] * LOG2E, -tot[1] * LOG2E);
            ref23 = pack2(-tot[2] * LOG2E, -tot[3] * LOG2E);
          } else if (tg == 0) {
            *reinterpret_cast<float4 *>(post_s + par * D + c0) = make_float4(tot[0], tot[1], tot[2], tot[3]);  // G_C - G_m
          }
          asm volatile("bar.sync %0, 128;" ::"r"(ALONE ? 4 + half : 2) : "memory");  // this half's raw k, q have been read: Kh may take their place
          // the Kt/Qt tile is free once MMA2 of the previous chunk has completed
          if (!ALONE && n > 0 && half == 0) wait_bar(&misc->bar_ro[0], par ^ 1, misc);
          uint64_t run01 = pack2(run0[0], run0[1]), run23 = pack2(run0[2], run0[3]);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint64_t k01 = pack2(bf16lo(kw[j].x), bf16hi(kw[j].x)), k23 = pack2(bf16lo(kw[j].y), bf16hi(kw[j].y));
            run01 = add2(run01, pack2(g4[j].x, g4[j].y));
            run23 = add2(run23, pack2(g4[j].z, g4[j].w));
            const uint64_t d01 = fma2(run01, l2e2, ref01), d23 = fma2(run23, l2e2, ref23);  // (G_t - G_m) log2(e)
            float d[4], dc[4];
            unpack2(d01, d[0], d[1]);
            unpack2(d23, d[2], d[3]);
            unpack2(add2(d01, comp2), dc[0], dc[1]);
            unpack2(add2(d23, comp2), dc[2], dc[3]);
            const uint64_t e1_01 = pack2(ex2f(dc[0]), ex2f(dc[1])), e1_23 = pack2(ex2f(dc[2]), ex2f(dc[3]));
            const uint64_t e2_01 = pack2(ex2f(-d[0]), ex2f(-d[1])), e2_23 = pack2(ex2f(-d[2]), ex2f(-d[3]));
            float kt[4], kh[4];
            unpack2(mul2(k01, e1_01), kt[0], kt[1]);
            unpack2(mul2(k23, e1_23), kt[2], kt[3]);
            unpack2(mul2(k01, e2_01), kh[0], kh[1]);
            unpack2(mul2(k23, e2_23), kh[2], kh[3]);
            unsigned char *pk = kq_tile + (ok0 ^ (j << 4)) + j * 128;
            if (WITH_O) {
              const uint64_t q01 = pack2(bf16lo(qw[j].x), bf16hi(qw[j].x)), q23 = pack2(bf16lo(qw[j].y), bf16hi(qw[j].y));
              float qt[4];
              unpack2(mul2(q01, mul2(e1_01, qs2)), qt[0], qt[1]);
              unpack2(mul2(q23, mul2(e1_23, qs2)), qt[2], qt[3]);
              *reinterpret_cast<uint4 *>(pk + 32 * 128) = make_uint4(tf32_pre(qt[0]), tf32_pre(qt[1]), tf32_pre(qt[2]), tf32_pre(qt[3]));
            }
            *reinterpret_cast<uint4 *>(pk) = make_uint4(tf32_pre(kt[0]), tf32_pre(kt[1]), tf32_pre(kt[2]), tf32_pre(kt[3]));
            // Kh goes out twice, the same four values in both places: K-major (MMA1 contracts over the channels) and
            // MN-major (MMA5 contracts over the tokens).  A tf32 MN-major operand has a swizzle of its own, so the two
            // tiles differ in where a vector lands, not in what it holds.
            const uint4 khv = make_uint4(tf32_pre(kh[0]), tf32_pre(kh[1]), tf32_pre(kh[2]), tf32_pre(kh[3]));
            *reinterpret_cast<uint4 *>(kh_tile + (oh0 ^ (j << 4)) + j * 128) = khv;
            *reinterpret_cast<uint4 *>(kht_tile + (om0 ^ (j << 5)) + j * 128) = khv;
          }
        } else {
          if (!ALONE && n > 0 && half == 0) wait_bar(&misc->bar_ro[0], par ^ 1, misc);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            unsigned char *pk = kq_tile + (ok0 ^ (j << 4)) + j * 128;
            const uint4 kf = make_uint4(kw[j].x << 16, kw[j].x & 0xFFFF0000u, kw[j].y << 16, kw[j].y & 0xFFFF0000u);  // exact
            *reinterpret_cast<uint4 *>(pk) = kf;
            if (WITH_O)
              *reinterpret_cast<uint4 *>(pk + 32 * 128) = make_uint4(qw[j].x << 16, qw[j].x & 0xFFFF0000u, qw[j].y << 16, qw[j].y & 0xFFFF0000u);
            const float e2 = e2_s[(n % RING) * C + tr + j];
            *reinterpret_cast<uint4 *>(kht_tile + (om0 ^ (j << 5)) + j * 128) =
                make_uint4(tf32_pre(__uint_as_float(kf.x) * e2), tf32_pre(__uint_as_float(kf.y) * e2),
                           tf32_pre(__uint_as_float(kf.z) * e2), tf32_pre(__uint_as_float(kf.w) * e2));
          }
        }
      }
      // the exponents of this chunk may have overflowed: the unit will not be written back
      if (KDA && out_of_range && tg == 0) misc->domain_flag[u & 3] = 1;
      fence_smem_to_async();
      arrive_warp(&misc->rdy_prep[buf(n)], lane);  // -> MMA1
      t0 += C;
      cp_tok += C;
      if (WALK && t0 >= n_tok && n + 1 < all_chunks) {
        t0 = 0;
        ++u;
        next_copies(units[u], 0);
        n_tok = units[u].n_tok;
      }
      if (n + 1 < all_chunks) {
        if (!KDA && warp == 8) scalars(n + 1, u, t0);
        // The next raw k, q (KDA) land once MMA5 of the previous chunk has read the Kh tile of that parity; the next
        // log-decay (KDA) or k, q (GDN) once MMA1 of this chunk has read the tile they go to.
        if (KDA && !ALONE) {
          if (n > 0) wait_bar(&misc->bar_s[par ^ 1], phase2(n - 1), misc);
          if (lane == 0 && !misc->abort_flag) stage_kq(n + 1);
        }
        if (!ALONE) {
          wait_bar(&misc->bar_ap[0], par, misc);
          if (lane == 0 && !misc->abort_flag) {
            if (KDA) stage_g(n + 1); else stage_kq(n + 1);
          }
        }
      }
    }
    // after a time-out the last copies may not have been waited for: they must have landed before the CTA leaves
    if (lane == 0 && misc->abort_flag) {
      if (g_issued > 0) mbar_wait_bounded(&misc->g_full[0], (g_issued - 1) & 1, kMaxPolls);
      if (kq_issued > 0) mbar_wait_bounded(&misc->kq_full[0], (kq_issued - 1) & 1, kMaxPolls);
    }
  } else {
    // ================================= chain warps =================================
    const int colh = warp >> 2;            // column half
    const int vrow = quad * 32 + lane;     // the TMEM lane this thread owns

    auto col_block = [&](int i) { return ALONE ? i * 64 + colh * 32 : colh * 64 + i * 32; };  // this warp's two blocks of 32 state columns
    int n = 0;  // index among the CTA's chunks
#pragma unroll 1
    for (int u = 0; u < (WALK ? uni(misc->n_units) : min(uni(misc->n_units), 1)); ++u) {
      const Unit &x = units[u];
      // where this thread's part of the outputs of a chunk starts (bf16: 16 bytes of every 16th token; fp32: see below)
      OT *go = WITH_O ? static_cast<OT *>(a.o) + (x.tok0 * a.H_v + x.head) * D : nullptr;
      if (WITH_O && sizeof(OT) == 2) go += (tid >> 4) * v_stride + (tid & 15) * 8;
      const int n_tok = uni(x.n_tok), n_chunks = (n_tok + C - 1) / C;
      if (!ZERO && n_chunks > 0) {
        // the start state goes into TMEM as it is; the first chunk's state pass scales it like any other.  (The state of the unit
        // before has been read out by the same threads.)
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
          const int c0 = col_block(i);
          const float *const st_c = a.state + x.state + (c0 * D + vrow);
          uint32_t s[32];
          if (a.mode == DASC_REFRESH_CONTINUE) {
#pragma unroll
            for (int j = 0; j < 32; ++j) s[j] = __float_as_uint(st_c[j * D]);
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) s[j] = 0u;
          }
          tmem_st32(tlane + COL_S + c0, s);
        }
        tmem_st_wait();
      }
      for (int ch = 0; ch < n_chunks; ++ch, ++n) {
        const uint32_t par = n & 1;
        const int ntok = min(C, n_tok - ch * C);
        const float *beta_c = beta_s + (n % RING) * C;
        const float *fac_c = fac_s + (n % FAC) * D;
        if (n + 1 == all_chunks && tid == 0) stream_order_release();  // one chunk (2.5 us) before the end: see launch.cuh

        // ---- (1) the previous chunk's state update is complete; this chunk's factors and tiles are ready ----
        wait_bar(&misc->rdy_fac[n % FAC], (n / FAC) & 1, misc);
        if (ch > 0) wait_bar(&misc->bar_s[(n - 1) & 1], phase2(n - 1), misc);
        tc_fence_after_sync();

        // ---- (2) state pass (columns = channels, half of them per warp): scale the state to this chunk's midpoint ----
        if (ZERO && ch == 0) {
          if (ALONE) {
            tc_fence_before_sync();
            arrive_warp(&misc->rdy_half, lane);
          }
        } else {
          if constexpr (ALONE) {
            // channels 0-63 first: MMA2 starts on them while 64-127 are scaled
            uint32_t s[2][2][16];
#pragma unroll
            for (uint32_t part = 0; part < 2; ++part)
#pragma unroll
              for (uint32_t hh = 0; hh < 2; ++hh) tmem_ld_16x256b(tlane + (hh << 20) + COL_S + part * 64 + colh * 32, s[part][hh]);
            tmem_ld_wait();
#pragma unroll
            for (uint32_t part = 0; part < 2; ++part) {
              const int c = part * 64 + colh * 32;
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const uint64_t f = *reinterpret_cast<const uint64_t *>(fac_c + c + 8 * i + 2 * tig);
#pragma unroll
                for (uint32_t hh = 0; hh < 2; ++hh) {
                  scale2(s[part][hh][4 * i + 0], s[part][hh][4 * i + 1], f);
                  scale2(s[part][hh][4 * i + 2], s[part][hh][4 * i + 3], f);
                }
              }
              if (part == 1) {  // the first part's stores have had the time of this scaling
                tmem_st_wait();
                tc_fence_before_sync();
                arrive_warp(&misc->rdy_half, lane);  // -> MMA2's first half
              }
#pragma unroll
              for (uint32_t hh = 0; hh < 2; ++hh) tmem_st_16x256b(tlane + (hh << 20) + COL_S + c, s[part][hh]);
            }
          } else {
            uint64_t f[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) f[i] = *reinterpret_cast<const uint64_t *>(fac_c + colh * 64 + 8 * i + 2 * tig);
#pragma unroll 1
            for (uint32_t hh = 0; hh < 2; ++hh) {  // lanes 0-15, 16-31 of the quadrant
              const uint32_t addr = tlane + (hh << 20) + COL_S + colh * 64;
              uint32_t s[32];
              tmem_ld_16x256b(addr, s);
              tmem_ld_wait();
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                scale2(s[4 * i + 0], s[4 * i + 1], f[i]);
                scale2(s[4 * i + 2], s[4 * i + 3], f[i]);
              }
              tmem_st_16x256b(addr, s);
            }
          }
          tmem_st_wait();
        }
        tc_fence_before_sync();
        arrive_warp(&misc->rdy_state, lane);  // -> MMA2

        // ---- (3) P ----
        if (!ALONE && WITH_O && quad >= 2) take_p(n, colh);

        // ---- (4) RHS^T = beta (V - R)^T as a tf32 pair: high over R^T, low in the consumed A|P columns ----
        // A's and P's columns are about to be overwritten: A's by warps that wait for its readers (the issuing warp read its rows
        // before it issued MMA2), P's by the warps that read them.  (The wait that comes last in time is the last one.)
        wait_bar(&misc->a_taken, par, misc);
        wait_bar(&misc->v_full, par, misc);
        {
          const int tb = colh * 16;
          // V and the per-token factors are fetched before the last wait.  Blocks of one ldmatrix: tokens 0-7 of the half with values
          // 0-7, 8-15, tokens 8-15 with the same
          const int vt = tb + (lane >> 4) * 8 + (lane & 7);
          uint32_t xx[2][8], vvv[2][4];
          uint64_t beta2[2], e1c2[2];
#pragma unroll
          for (uint32_t hh = 0; hh < 2; ++hh)
            ldmatrix_x4_trans(vvv[hh], sbase + OFF_V + (quad >> 1) * (C * 128) + vt * 128 +
                                           ((((quad & 1) * 4 + hh * 2 + ((lane >> 3) & 1)) ^ (vt & 7)) << 4));
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            beta2[i] = *reinterpret_cast<const uint64_t *>(beta_c + tb + i * 8 + 2 * tig);
            if (!KDA) e1c2[i] = *reinterpret_cast<const uint64_t *>(e1c_s + (n % RING) * C + tb + i * 8 + 2 * tig);
          }
          wait_bar(&misc->bar_ro[buf(n)], phase(n), misc);
          tc_fence_after_sync();
#pragma unroll
          for (uint32_t hh = 0; hh < 2; ++hh) tmem_ld_16x256b(tlane + (hh << 20) + col_ro(n) + tb, xx[hh]);
          tmem_ld_wait();
          if (ZERO && ch == 0) {
#pragma unroll
            for (int i = 0; i < 8; ++i) xx[0][i] = xx[1][i] = 0u;  // no product 2
          }
#pragma unroll
          for (uint32_t hh = 0; hh < 2; ++hh) {
            uint32_t(&x)[8] = xx[hh], (&vv)[4] = vvv[hh], lo[8];
            if (ntok < C) {
              // the boxes reached past the request's last token: those values are other tokens' (zeros past the end of the stream)
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const int t = tb + (i >> 1) * 8 + 2 * tig;
                if (t >= ntok) vv[i] = 0u;
                else if (t + 1 >= ntok) vv[i] &= 0xFFFFu;
              }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              uint64_t r = pack2(__uint_as_float(x[2 * i]), __uint_as_float(x[2 * i + 1]));
              // GDN: the product is k_t S' on the raw keys; its row factor e1_t (with the truncation compensation) comes here
              if constexpr (!KDA) r = mul2(e1c2[i >> 1], r);
              r = mul2(beta2[i >> 1], sub2(pack2(bf16lo(vv[i]), bf16hi(vv[i])), r));
              // the high part is the value itself, which the tensor core truncates on reading; the low part the exact rest
              float r0, r1;
              unpack2(r, r0, r1);
              x[2 * i] = __float_as_uint(r0);
              x[2 * i + 1] = __float_as_uint(r1);
              unpack2(sub2(r, pack2(__uint_as_float(x[2 * i] & 0xFFFFE000u), __uint_as_float(x[2 * i + 1] & 0xFFFFE000u))), r0, r1);
              lo[2 * i] = tf32_pre(r0);
              lo[2 * i + 1] = tf32_pre(r1);
            }
            tmem_st_16x256b(tlane + (hh << 20) + col_ro(n) + tb, x);
            tmem_st_16x256b(tlane + (hh << 20) + COL_RL + tb, lo);
          }
          tmem_st_wait();
        }
        tc_fence_before_sync();
        arrive_warp(&misc->rdy_rhs, lane);  // -> MMA3 (T tile and RHS^T are ready)

        // ---- (5) the part of U^T the tensor core drops when it reads it (the low 13 mantissa bits), written over
        //          the consumed RHS^T: U = U_hi + U_lo exactly ----
        wait_bar(&misc->bar_u, par, misc);
        tc_fence_after_sync();
        {
          const int tb = colh * 16;
          uint32_t x[16];
          tmem_ld16(tlane + COL_U<ALONE> + tb, x);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 16; ++j)
            x[j] = tf32_pre(__uint_as_float(x[j]) - __uint_as_float(x[j] & 0xFFFFE000u));
          tmem_st16(tlane + col_ro(n) + tb, x);
          tmem_st_wait();
        }
        tc_fence_before_sync();
        arrive_warp(&misc->rdy_u, lane);  // -> MMA4, MMA5

        // ---- (6) outputs of this chunk (without outputs MMA5 is waited for here as well) ----
        if (!ALONE) {
          wait_bar(&misc->bar_o, par, misc);
          outputs(n, ntok, go, colh, tid);
          if (WITH_O) go += C * v_stride;
          tc_fence_before_sync();
          arrive_warp(&misc->tp_free, lane);  // this thread is done with the T|P|O tile region
        }
      }
      // ---- final state: the factor still owed, then write back ----
      // Which of this warp's rows are written, a bit each, fetched before the waits: looked up row by row beside the stores, the
      // 64 loads came one behind the other and the write-back of a unit in the merge mode took 7.1 k cycles (2.6 k where all rows
      // are written); 32 requests of 1 .. 128 tokens x 4 layers x 32 heads, state only: 277 -> 262 us.
      uint32_t rows[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const uint8_t *keep = a.row_keep + x.keep_row;
        rows[i] = __ballot_sync(0xffffffffu, a.mode == DASC_REFRESH_CONTINUE || !keep[col_block(i) + lane]);
      }
      // post_s of the last chunk is visible: its writers arrived on rdy_prep, which the issuing warp waited for before it met the
      // triangular warp, which arrived on a_taken, which these warps have waited for.  (Waiting for rdy_prep itself here could wait for
      // the wrong phase: the next unit's tiles can be complete by now.)
      if (n_chunks > 0) wait_bar(&misc->bar_s[(n - 1) & 1], phase2(n - 1), misc);
      // A unit without tokens has no factor and must not touch fin_s: it meets no wait on the way here, so the slower chain warps can
      // still be scaling the unit before.  (One with tokens has been through rdy_state, which all of them arrive on behind that.)
      if (n_chunks > 0 && tid < D) fin_s[tid] = ex2f(post_s[KDA ? ((n - 1) & 1) * D + tid : (n - 1) & 3] * LOG2E);
      // In a walk other roles are in the next unit and can run out of a wait there at any time, so what the barrier answers, not a look at
      // the flag by each thread, says whether this unit is written: all of it or nothing.
      const bool gave_up = any_chain(misc->abort_flag != 0);
      tc_fence_after_sync();
      // A unit whose decay left the range, or whose CTA gave up on a wait, is NOT written back: its stored state keeps
      // the bits it had before the call, so that it can be replayed by the exact kernel (or by the caller).
      const bool bad = gave_up || misc->domain_flag[u & 3] != 0;
      // The flag of unit u - 1, which everyone has looked at, becomes that of unit u + 3, which the producer warps cannot have reached.
      if (tid == 0) misc->domain_flag[(u + 3) & 3] = 0;
      if (bad) {
        if (tid == 0 && !gave_up) hand_over(a, x.index, true);
      } else {
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
          const int c0 = col_block(i);
          const uint32_t write = i == 0 ? rows[0] : rows[1];
          float *const st_c = a.state + x.state + (c0 * D + vrow);
          const float *const fin_c = fin_s + c0;
          if (n_chunks > 0) {
            uint32_t s[32];
            tmem_ld32(tlane + COL_S + c0, s);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (write >> j & 1u) st_c[j * D] = __uint_as_float(s[j]) * fin_c[j];
          } else {  // scratch mode with an empty suffix
#pragma unroll 1
            for (int j = 0; j < 32; ++j)
              if (write >> j & 1u) st_c[j * D] = 0.f;
          }
        }
      }
      if (!WALK) break;
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == WARP_MMA) tmem_dealloc(tm, F::TMEM_COLS);
  if (tid == 0 && misc->abort_flag) atomicExch(static_cast<uint32_t *>(a.workspace), 1u);  // a wait ran out
}

// Blocks are placed in index order, so the requests are taken longest first: a long one started last would run on while
// the rest of the GPU is idle.  Requests of 1 .. 1023 tokens on B200 (296 units resident): 64 x 32 heads 618 -> 528 us, 240 x 4 heads
// 335 -> 264 us.  Ties keep their order.  The limit of 240 requests is what fits the spare bytes of the workspace header, not
// where the order stops to pay: 241 x 4 heads take 354 us, and 265 us where the caller lists them longest first.
bool ordered(const DascRefreshArgs &a) { return a.n_req > 1 && a.n_req <= kRefreshOrderMax; }

constexpr int kPrepThreads = 256;
static_assert(kPrepThreads >= kRefreshOrderMax);
// One thread per request; block 0 also clears the header words and ranks the requests.
__global__ void __launch_bounds__(kPrepThreads) refresh_prep_kernel(uint32_t *ws, const int32_t *cu, int32_t n_req, int32_t window,
                                                                    int32_t *tok_begin, bool order) {
  stream_order_begin();
  const int r = blockIdx.x * kPrepThreads + threadIdx.x;
  if (ws && r < 4) ws[r] = 0;
  int len = -1;
  if (r < n_req && (tok_begin || order)) {
    const int lo = cu[r], hi = cu[r + 1];
    len = hi - lo;
    if (tok_begin) {
      const int64_t b = static_cast<int64_t>(hi) - window;
      const int first = b > lo ? static_cast<int>(b) : lo;
      tok_begin[r] = first;
      len = hi - first;
    }
  }
  if (!order) return;  // (one block when there is an order)
  __shared__ __align__(16) int lens[kPrepThreads];
  lens[threadIdx.x] = len;
  __syncthreads();
  if (r < n_req) {
    int rank = 0;
    for (int j = 0; j < n_req; j += 4) {
      const int4 l4 = *reinterpret_cast<const int4 *>(lens + j);  // entries past n_req are -1: they rank below
      const int l[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) rank += l[i] > len || (l[i] == len && j + i < r);
    }
    reinterpret_cast<uint8_t *>(ws)[kRefreshWsOrder + rank] = static_cast<uint8_t>(r);
  }
}

// cuTensorMapEncodeTiled is a driver entry point.  It is looked up through the runtime at first use, so that the library
// has no link-time dependency on libcuda and still loads (plan building, accessors) on a machine without a driver.
using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled_fn() {
  static EncodeTiledFn fn = [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

// CTAs of a launch.  A CTA replays its units one behind the other, and the roles that need no state (tiles, A, T) run into the next
// unit's first chunk while the chain warps write the last one's state back: a unit of its own costs a CTA about 16 k cycles
// of start and end beside 7.5 k per chunk.  With a grid of G, CTA b takes units b, 2G - 1 - b, 2G + b, ... (there and back): as
// requests come longest first, each gets long and short ones, and adjacent heads still run side by side.  The grid is a
// multiple of the CTAs that are resident at once, so that no last wave is nearly empty.
// Measured, us, a CTA per unit / this rule (KDA unless GDN): 4096 units of 1 .. 128 tokens, state only 253 / 223; 8192 of 64 tokens, state
// only 379 / 309; 7680 of 16 tokens, state only 255 / 182; 8192 of 256 tokens 1128 / 1090 (GDN 879 / 829), 4096 of 64 GDN 209 / 160.
// Where the lines lie:
//  - kWalkChunks chunks per CTA on average, by the estimate of Load (a quarter of a millisecond; lengths just above a multiple of a chunk, or
//    uneven ones, can give a CTA half as many more): work of other streams is placed when CTAs end.  One grid of
//    resident CTAs, whatever they have to do, gains nothing more where there are more chunks than that (1365, GDN 1101).
//  - no request longer than half of a CTA's share by the caller's bound, since here a CTA's units are fixed beforehand, while blocks of
//    a unit each go to whichever CTA ends first: 2048 units of 1 .. 1023 tokens take 669 / 658 walked, 1600 of 1 .. 1199 596 / 601: little
//    to gain where units are long.
//  - requests that are not in order of length (more than kRefreshOrderMax): only if they are about equally long.
//  - up to two units per CTA, taken there and back, are what blocks of a unit each would come to as well (the shortest of the first G
//    with the longest of the rest), whatever the lengths, so only the start of the second one is saved; but the CTAs that have one
//    unit pay 1 to 4 % for the walk.  Hence from 1.5 units per CTA on (1.3 with short requests), where lengths differ.  us, a CTA per unit /
//    walked, requests of 1 .. 2 n - 1 tokens, KDA: 424 units, n = 56 40.7 / 37.8, 480 units, n = 128 63.9 / 59.6, n = 600 195 /
//    170, 592 units, n = 128 75.8 / 68.8, n = 1000 361 / 322; 392 units, n = 56 39.9 / 35.8 but n = 1000 233 / 247; 344 units 2 % more.  GDN: 392 units, n = 56 35.2 / 32.3, n = 128
//    45.9 / 40.1, n = 1000 170 / 173.5; 424, n = 56 37.1 / 34.6; 480, n = 128 50.7 / 47.5, n = 600 141 / 125; 592, n = 1000 262 / 233.
//    By the bound alone lengths may differ where they are equal, and with 1.4 units per CTA equal long ones lose: bounds of twice the
//    length, 424 units of 700 tokens 170 / 190 (GDN 126 / 144), 424 of 300 96.9 / 95.3 (65.0 / 71.6), 448 of 700 192.5 / 193.5 (144.6 / 144.0), 464 of 300
//    99.2 / 98.2 (75.3 / 73.9); short ones at most 5 %: 388 units of 95 tokens 35.1 / 35.1 (28.3 / 29.5), 412 of 40 27.8 / 26.7 (23.5 / 23.8).  What that
//    costs uneven lengths below 1.5 units per CTA: GDN, n = 300, 392 units 69.8 / 66.2, 424 73.8 / 67.2 (KDA 98.6 / 90.0).
constexpr int64_t kSms = 148, kResident = 2 * kSms, kWalkChunks = 64;

// What the host knows of a launch: the longest request (by the caller's bound) and all units together, in chunks (about: half a one
// more per request).
struct Load {
  int64_t n_units, longest, per_head, chunks;
  bool in_order;  // requests come longest first
};
Load load_of(const DascRefreshArgs &a) {
  const int64_t tokens = a.window > 0 ? std::min<int64_t>(a.total_tokens, static_cast<int64_t>(a.n_req) * a.window) : a.total_tokens;
  Load l;
  l.n_units = static_cast<int64_t>(a.n_req) * a.n_layers_in_call * a.H_v;
  l.longest = (std::max<int64_t>(std::min<int64_t>(a.max_seqlen, tokens), 1) + C - 1) / C;  // (any int32 is a legal bound)
  l.per_head = tokens / C + a.n_req / 2;
  l.chunks = l.per_head * a.n_layers_in_call * a.H_v;
  l.in_order = a.ordered || a.n_req == 1;
  return l;
}

int64_t grid_for(const DascRefreshArgs &a) {
  const Load l = load_of(a);
  const int64_t g = kResident * std::max<int64_t>((l.chunks + kResident * kWalkChunks - 1) / (kResident * kWalkChunks),
                                                  (l.n_units + kResident * kMaxWalk - 1) / (kResident * kMaxWalk));
  const bool even = l.in_order ? l.longest * 2 * g <= l.chunks : l.longest * a.n_req * 9 <= l.per_head * 10;
  const bool two = l.in_order && l.n_units <= 2 * kResident && l.n_units * 10 >= kResident * (l.longest * 4 <= kWalkChunks ? 13 : 15) &&
                   l.longest <= kWalkChunks && l.longest * a.n_req * 2 >= l.per_head * 3;
  return (even || two) && g < l.n_units ? g : l.n_units;
}

// With at most a CTA per SM the time is the chain of one CTA: hand-offs, not any unit of the SM, bound it.  The ALONE form takes off
// the chain what need not be on it: producers with twice the warps, running up to two chunks ahead of the chain into second (MN-major Kh:
// fourth) buffers; MMA1, the copies of the inputs, P and the outputs in warps of their own (one warp that issued all products was busy all of
// the time: 100 to 120 cycles per barrier, 40 per product); MMA2 started on the first half of the scaled state; the state's product ahead of
// the outputs'.  A chunk takes 3.7 k cycles instead of 5.0 k (GDN 3.3 k, 3.8 k; from the times of 512 and 2048 tokens), KDA from cold inputs 5.6 k in SHARED.
// Measured, us, SHARED / ALONE, 256 tokens (GDN): 8 units 27.3 / 23.4 (22.5 / 20.5), 80 units 27.7 / 23.4 (22.8 / 21.1), 148 units 33.3 / 27.0
// (24.6 / 24.5), state only 29.8 / 22.6 (21.4 / 20.4); 148 units of 1 .. 599 tokens 68.3 / 57.6 (50.2 / 48.9), of 1000 tokens 116.0 / 87.2
// (91.3 / 75.0); 152 units 37.9 / 43.5 (31.4 / 39.5): the line is where a second CTA per SM begins to be needed.
// Between 148 and 296 units ALONE would still be the better one where one request is longer than an SM's share of all (192 units of
// 1 .. 1199 tokens 123 / 95 (GDN 87 / 81), 256 of 1 .. 799 98.5 / 80.7 (63.4 / 62.5)), but the host knows only a bound on that length, and where the
// bound is loose and the lengths are even ALONE loses: 152 units of 40 tokens 16.0 / 20.4 (14.2 / 18.8), 296 of 300 tokens 53.0 / 65.3 (38.9 / 54.0),
// windows of 512 tokens over 256 prefixes of 100 20.9 / 27.2 (17.8 / 24.4).
// Its 58,880 registers leave no room for a block of the copy kernels beside it (one CTA of SHARED leaves 33,280), so a Store on another stream
// has the SMs without a unit, and where there are few waits for the refresh to end.  Hence ALONE for long requests only on half of
// the SMs, else up to kWalkChunks chunks: like the CTAs of a walk they are gone after an eighth of a millisecond.  A Store of 16
// checkpoints (85 us by itself) / the refresh it started with, us until each has ended, SHARED and ALONE:
//   64 units of 4096 tokens 133 / 424, 155 / 290;   128 units 175 / 431, 335 / 332;   148 units 201 / 535, 420 / 420;   148 units of
//   2048 tokens 199 / 250, 269 / 266 (GDN 193 / 203, 244 / 242), of 1024 tokens 175 / 174, 190 / 193 (GDN 156 / 154, 179 / 176).
// With registers capped at 72 (one block fits) the Store still ended at 435 beside 148 units and the refresh by itself took 1 to 6 % longer;
// at 64, spilling, 382 and 50 %.  Two launches on two streams share the SMs as well in SHARED: 2 x 148 units of 256 tokens 50 / 57
// (2048 tokens 336 / 303), but 2 x 100 units 41 / 37, 2 x 72 39 / 29.
bool alone_for(const DascRefreshArgs &a) {
  const Load l = load_of(a);
  return l.n_units <= kSms / 2 || (l.n_units <= kSms && l.longest <= kWalkChunks);
}

template <bool KDA, typename OT, bool WITH_O, bool ZERO = false>
int launch(DascRefreshArgs a, void *stream) {
  const int64_t n_units = static_cast<int64_t>(a.n_req) * a.n_layers_in_call * a.H_v;
  a.ordered = ordered(a);
  const bool alone = alone_for(a);
  const int64_t grid = alone ? n_units : grid_for(a);  // (dasc_debug_refresh_form answers the same)
  auto kern = alone ? refresh_chunked_kernel<KDA, OT, WITH_O, true, false, ZERO>
              : grid < n_units ? refresh_chunked_kernel<KDA, OT, WITH_O, false, true, ZERO>
                               : refresh_chunked_kernel<KDA, OT, WITH_O, false, false, ZERO>;
  const uint32_t smem = alone ? SMEM_ALONE : SMEM_BYTES;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return static_cast<int>(e);
  if (n_units == 0) return cudaSuccess;
  if (n_units > 2147483647LL) return static_cast<int>(cudaErrorInvalidConfiguration);
  const int prep = dasc_launch_refresh_prep(a, stream);
  if (prep != 0) return prep;
  // tensor maps of the token streams [Lc*T tokens][heads][128]: boxes of 32 tokens x one head x 128 bytes of channels with
  // the 128-byte swizzle, which is the layout of one block of an operand tile
  CUtensorMap tmap_q{}, tmap_k{}, tmap_v{}, tmap_g{};
  const EncodeTiledFn encode = encode_tiled_fn();
  if (!encode) return static_cast<int>(cudaErrorNotSupported);
  auto make_map = [&](CUtensorMap *m, CUtensorMapDataType type, const void *base, int heads, cuuint64_t esz) {
    const cuuint64_t dims[3] = {static_cast<cuuint64_t>(D), static_cast<cuuint64_t>(heads),
                                static_cast<cuuint64_t>(a.n_layers_in_call) * static_cast<cuuint64_t>(a.total_tokens)};
    const cuuint64_t strides[2] = {D * esz, static_cast<cuuint64_t>(heads) * D * esz};
    const cuuint32_t box[3] = {static_cast<cuuint32_t>(128 / esz), 1, static_cast<cuuint32_t>(C)};
    const cuuint32_t ones[3] = {1, 1, 1};
    return encode(m, type, 3, const_cast<void *>(base), dims, strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  };
  if (!make_map(&tmap_k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, a.k, a.H_k, 2) || !make_map(&tmap_v, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, a.v, a.H_v, 2) ||
      (WITH_O && !make_map(&tmap_q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, a.q, a.H_k, 2)) ||
      (KDA && !make_map(&tmap_g, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, a.g, a.H_v, 4)))
    return static_cast<int>(cudaErrorInvalidValue);
  return static_cast<int>(launch_in_order(kern, dim3(static_cast<unsigned>(grid)),
                                          dim3(alone ? Form<true>::NT : Form<false>::NT), smem, stream, a, tmap_q, tmap_k, tmap_v, tmap_g));
}

}  // namespace

int dasc_launch_refresh_prep(const DascRefreshArgs &a, void *stream) {
  const int blocks = a.window > 0 || a.tok_begin ? (a.n_req + kPrepThreads - 1) / kPrepThreads : 1;
  return static_cast<int>(launch_in_order(refresh_prep_kernel, dim3(static_cast<unsigned>(blocks)), dim3(kPrepThreads), 0, stream,
                                          static_cast<uint32_t *>(a.workspace), a.cu_seqlens, a.n_req, a.window, a.tok_begin,
                                          a.ordered != 0));
}

// Scratch the chunked kernel needs: the 256-byte header (flags and counters) and one list entry per unit of the call.
size_t dasc_refresh_chunked_workspace_bytes(int32_t n_req, int32_t n_layers_in_call, int32_t H_v) {
  const size_t units = static_cast<size_t>(n_req) * static_cast<size_t>(n_layers_in_call) * static_cast<size_t>(H_v);
  return kRefreshWsHeader + (units * sizeof(int32_t) + 255) / 256 * 256;
}

uint32_t g_dasc_debug_poll_limit = 0;

int32_t dasc_debug_refresh_form(int32_t n_req, int32_t units_per_req, int64_t total_tokens, int32_t window, int32_t max_seqlen,
                                int64_t *n_blocks) {
  DascRefreshArgs a{};
  a.n_req = n_req;
  a.n_layers_in_call = 1;
  a.H_v = units_per_req;
  a.total_tokens = total_tokens;
  a.window = window;
  a.max_seqlen = max_seqlen;
  a.ordered = ordered(a);
  const int64_t n_units = static_cast<int64_t>(n_req) * units_per_req;
  const bool alone = alone_for(a);
  const int64_t grid = alone ? n_units : grid_for(a);
  if (n_blocks) *n_blocks = grid;
  return alone ? 2 : grid < n_units ? 1 : 0;
}

// Returns a cudaError_t as int, or -1 if this kernel does not take the request
// (it needs d_k = d_v = 128 and bf16 token streams).
int dasc_launch_refresh_chunked(const DascRefreshArgs &a_in, void *stream) {
  if (a_in.d_k != D || a_in.d_v != D || !a_in.io_bf16) return -1;
  DascRefreshArgs a = a_in;
  a.poll_limit_first_wait = __atomic_load_n(&g_dasc_debug_poll_limit, __ATOMIC_RELAXED);
  const bool kda = a.kind == DASC_KDA;
  if (!a.o && a.mode == DASC_REFRESH_SCRATCH_MERGE_LOCAL)
    return kda ? launch<true, __nv_bfloat16, false, true>(a, stream) : launch<false, __nv_bfloat16, false, true>(a, stream);
  if (!a.o) return kda ? launch<true, __nv_bfloat16, false>(a, stream) : launch<false, __nv_bfloat16, false>(a, stream);
  if (a.o_bf16) return kda ? launch<true, __nv_bfloat16, true>(a, stream) : launch<false, __nv_bfloat16, true>(a, stream);
  return kda ? launch<true, float, true>(a, stream) : launch<false, float, true>(a, stream);
}

// ---------------------------------------------------------------------------------------------
// dasc_refresh_static: the chunked refresh without any caller-provided workspace.
// ---------------------------------------------------------------------------------------------
namespace {

// Scratch of the static variant.  It lives in the library image: every GPU that loads libdasc
// holds these bytes until the process exits.  In host code the name below is only a handle; the
// device address is obtained once per device with cudaGetSymbolAddress.
constexpr size_t kStaticScratchBytes = 4096;
static __device__ __align__(256) unsigned char g_refresh_static_scratch[kStaticScratchBytes];

constexpr int kMaxDevices = 64;
void *g_static_scratch_addr[kMaxDevices] = {};  // device address per CUDA device, filled on first use

// Device address of the static scratch on device `dev`, which must be the CURRENT device; resolves it on the
// first call.
cudaError_t static_scratch_address(int dev, void **out) {
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  void *p = __atomic_load_n(&g_static_scratch_addr[dev], __ATOMIC_ACQUIRE);
  if (!p) {
    const cudaError_t e = cudaGetSymbolAddress(&p, g_refresh_static_scratch);
    if (e != cudaSuccess) return e;
    __atomic_store_n(&g_static_scratch_addr[dev], p, __ATOMIC_RELEASE);  // racing first calls store the same value
  }
  *out = p;
  return cudaSuccess;
}

}  // namespace

extern "C" dasc_status_t dasc_refresh_static(const dasc_plan_t *plan, float *state_base, int64_t layer_stride,
                                             int64_t req_stride, const int32_t *req_idx, const void *q, const void *k,
                                             const void *v, const float *g, const float *beta,
                                             const int32_t *cu_seqlens, int32_t n_req, int64_t total_tokens,
                                             int32_t max_seqlen, int32_t layer_begin, int32_t layer_end, float q_scale,
                                             void *o, int32_t o_dtype, int32_t mode, void **scratch_out,
                                             void *cuda_stream) {
  if (scratch_out) *scratch_out = nullptr;
  if (!plan || plan->info.device < 0) return DASC_ERR_INVALID_ARG;
  if (n_req < 0 || total_tokens < 0 || max_seqlen < 0) return DASC_ERR_INVALID_ARG;
  if (layer_begin < 0 || layer_end < layer_begin || layer_end > plan->info.n_layers) return DASC_ERR_INVALID_ARG;
  if (o && o_dtype != DASC_IO_BF16 && o_dtype != DASC_IO_FP32) return DASC_ERR_INVALID_ARG;
  if (mode != DASC_REFRESH_CONTINUE && mode != DASC_REFRESH_SCRATCH_MERGE_LOCAL) return DASC_ERR_INVALID_ARG;
  if (plan->info.d_k != D || plan->info.d_v != D) return DASC_ERR_SHAPE;  // the chunked kernel's shape
  // The plan's tables, the caller's buffers and the scratch all have to be on the device the kernel runs on.
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return DASC_ERR_CUDA;
  if (dev != plan->info.device) return DASC_ERR_INVALID_ARG;
  // The scratch this kernel cannot do without (the header words) must fit the static array; the list of units left
  // unwritten is as long as the rest of the array allows (a longer list is cut, the error word is set all the same).
  const size_t need = kRefreshWsHeader;
  if (need > kStaticScratchBytes) return DASC_ERR_WORKSPACE;
  void *scratch = nullptr;
  if (static_scratch_address(dev, &scratch) != cudaSuccess) return DASC_ERR_CUDA;
  if (scratch_out) *scratch_out = scratch;
  if (n_req == 0 || layer_end == layer_begin || total_tokens == 0) return DASC_OK;
  if (!state_base || !req_idx || !q || !k || !v || !g || !beta || !cu_seqlens) return DASC_ERR_INVALID_ARG;
  auto misaligned = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) != 0; };
  if (misaligned(state_base) || misaligned(q) || misaligned(k) || misaligned(v) || misaligned(g) || (o && misaligned(o)))
    return DASC_ERR_INVALID_ARG;
  if (layer_stride < 0 || req_stride < 0 || layer_stride % 4 || req_stride % 4) return DASC_ERR_INVALID_ARG;

  DascRefreshArgs a{};
  a.kind = plan->info.kind;
  a.H_v = plan->info.n_v_heads;
  a.H_k = plan->info.n_k_heads;
  a.d_k = plan->info.d_k;
  a.d_v = plan->info.d_v;
  a.state = state_base;
  a.layer_stride = layer_stride;
  a.req_stride = req_stride;
  a.req_idx = req_idx;
  a.q = q;
  a.k = k;
  a.v = v;
  a.io_bf16 = 1;
  a.g = g;
  a.beta = beta;
  a.cu_seqlens = cu_seqlens;
  a.n_req = n_req;
  a.total_tokens = total_tokens;
  a.max_seqlen = max_seqlen;
  a.layer_begin = layer_begin;
  a.n_layers_in_call = layer_end - layer_begin;
  a.q_scale = q_scale;
  a.o = o;
  a.o_bf16 = o_dtype == DASC_IO_BF16;
  a.mode = mode;
  a.row_keep = plan->d_row_keep;
  a.rows_per_layer = plan->rows_per_layer;
  a.workspace = scratch;  // the launcher clears the header words on the stream
  a.workspace_bytes = kStaticScratchBytes;
  // units outside the chunked kernel's log-decay range are listed behind the header, left unwritten, and replayed by
  // the exact kernel right after (it needs no scratch of its own); units that do not fit the list are an error
  a.unit_list = reinterpret_cast<int32_t *>(static_cast<unsigned char *>(scratch) + kRefreshWsHeader);
  a.unit_list_cap = static_cast<int32_t>((kStaticScratchBytes - kRefreshWsHeader) / sizeof(int32_t));
  a.short_thr = -1;
  a.domain_is_error = 0;
  int e = dasc_launch_refresh_chunked(a, cuda_stream);
  if (e == -1) return DASC_ERR_SHAPE;
  if (e == 0) {
    a.from_list = 1;
    e = dasc_launch_refresh_seq(a, cuda_stream);
  }
  return e == 0 ? DASC_OK : DASC_ERR_CUDA;
}
