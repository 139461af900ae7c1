// Suffix refresh, sequential form: the gated delta rule (Eq. 1, transposed
// orientation) replayed token by token in fp32 on the CUDA cores.  Exact for any
// log-decay g <= 0; it is the reference point for the chunked tensor-core kernel
// and the path for shapes that kernel does not take.
//
// One CTA per (request, layer, value head), or per part of its columns when units are few (second half of the file).  Columns of the
// state do not interact, so there is no barrier between tokens: a column's d_k entries live in the registers of SL adjacent lanes, and
// S^T k, S^T q are shuffles.
// Per token
//   S   <- Diag(alpha_t) S                       (decay on the key-channel index)
//   r   <- S^T k_t
//   u   <- beta_t (v_t - r)
//   S   <- S + k_t u^T
//   o_t <- q_scale * S^T q_t
// A lane holds rows 4 (i SL + slice) ... + 3, i = 0, 1, ..., of COLS columns: the SL lanes of a column read one contiguous
// stretch of k, q, alpha, and row pairs are the operand pairs of the packed fp32 instructions.  Bound: when units are few the
// serial chain (a dot product and its shuffles per token; the next token's is started before this token's update, see
// below), else instruction issue and the registers' share of the shared-memory bandwidth (128 bytes per cycle whatever is
// broadcast, hence 4 columns per lane).
// Measured on B200, fp32 (the form before: one column per thread and row half, a block barrier per token): 256 units of 128 x 128, 256
// tokens 407 -> 345 us; 8192 of them 11.2 -> 9.6 ms.
// Token inputs are staged TB tokens at a time: raw rows by cp.async into a double
// buffer, then converted once (bf16 -> fp32, alpha = exp(g)); outputs leave a group later, 16 bytes per store.  With NHELP > 0
// that many extra threads do both, a group ahead of and a group behind the tokens being replayed.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "dasc_internal.h"
#include "launch.cuh"

namespace {

constexpr int TB = 16;  // tokens staged per group

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
  const uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
  const uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all committed groups, or all but the last one
__device__ __forceinline__ void cp_async_wait_but(bool one) {
  if (one)
    asm volatile("cp.async.wait_group 1;" ::: "memory");
  else
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <typename IO>
__device__ __forceinline__ float io_to_float(IO x);
template <>
__device__ __forceinline__ float io_to_float<float>(float x) { return x; }
template <>
__device__ __forceinline__ float io_to_float<__nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }

template <typename IO>
__device__ __forceinline__ IO float_to_io(float x);
template <>
__device__ __forceinline__ float float_to_io<float>(float x) { return x; }
template <>
__device__ __forceinline__ __nv_bfloat16 float_to_io<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

// packed pairs of fp32 (one instruction per pair)
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float sum2(uint64_t v) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
  return lo + hi;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
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

template <int DK, int DV, int NOP, bool AHEAD, typename IO, bool KDA>
struct SeqSmem {
  // raw staging, double buffered
  alignas(16) IO q[2][TB][DK];
  alignas(16) IO k[2][TB][DK];
  alignas(16) IO v[2][TB][DV];
  alignas(16) float g[2][TB][KDA ? DK : 4];
  alignas(16) float beta[2][TB];
  // converted; two groups when extra warps convert the next one meanwhile
  struct Group {
    alignas(16) float kf[TB][DK];
    alignas(16) float qf[TB][DK];
    alignas(16) float af[TB][KDA ? DK : 4];
    alignas(16) float vf[TB][DV];
    alignas(16) float of[TB][DV][NOP];  // NOP shares of each of the group's outputs
    float bf[TB], cf[TB];                     // beta;  c_t = (alpha_t k_t) . k_{t-1}
  } grp[AHEAD ? 2 : 1];
};

template <int COLS>
__device__ __forceinline__ void load_cols(float (&x)[COLS], const float *p) {
  if constexpr (COLS == 4) {
    const float4 v = *reinterpret_cast<const float4 *>(p);
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
  } else {
    const float2 v = *reinterpret_cast<const float2 *>(p);
    x[0] = v.x; x[1] = v.y;
  }
}
template <int COLS>
__device__ __forceinline__ void store_cols(float *p, const float (&x)[COLS]) {
  if constexpr (COLS == 4)
    *reinterpret_cast<float4 *>(p) = make_float4(x[0], x[1], x[2], x[3]);
  else if constexpr (COLS == 1)
    *p = x[0];
  else
    *reinterpret_cast<float2 *>(p) = make_float2(x[0], x[1]);
}

// One (request, layer, value head) unit, replayed token by token by the whole CTA; COLS columns per lane, SL lanes per column.
template <int DK, int DV, int COLS, int SL, int NHELP, typename IO, typename OT, bool KDA>
__device__ __forceinline__ void seq_unit(const DascRefreshArgs &a, int unit, unsigned char *smem_raw) {
  constexpr int NC = DV / COLS * SL;      // threads that replay tokens
  constexpr int NT = NHELP > 0 ? NHELP : NC;  // threads that bring the tokens in and the outputs out
  constexpr int NV = DK / SL / 4;  // groups of four rows held by one lane
  constexpr int NOP = SL / COLS;
  constexpr bool AHEAD = NHELP > 0;
  using Smem = SeqSmem<DK, DV, NOP, AHEAD, IO, KDA>;
  Smem &sm = *reinterpret_cast<Smem *>(smem_raw);

  const int tid = threadIdx.x;
  const bool helper = AHEAD && tid >= NC;
  const int ht = AHEAD ? tid - NC : tid;  // index among the latter (negative: none of them)
  const int slice = tid % SL;
  const int col0 = tid / SL * COLS;
  const int own = slice % COLS;  // the one of this lane's columns whose sums it ends up with

  const int h = unit % a.H_v;
  const int lc = (unit / a.H_v) % a.n_layers_in_call;
  const int r = unit / (a.H_v * a.n_layers_in_call);
  const int hk = h / (a.H_v / a.H_k);
  const int layer = a.layer_begin + lc;
  const int64_t t_begin = a.tok_begin ? a.tok_begin[r] : a.cu_seqlens[r];
  const int n_tok = static_cast<int>(a.cu_seqlens[r + 1] - t_begin);
  // An empty suffix continues nothing; in the scratch mode it still replaces the omitted
  // units by the (all-zero) scratch state, as the definition says.
  if (n_tok <= 0 && a.mode == DASC_REFRESH_CONTINUE) return;

  float *st = a.state + static_cast<int64_t>(a.req_idx[r]) * a.req_stride + static_cast<int64_t>(layer) * a.layer_stride +
              static_cast<int64_t>(h) * DK * DV;
  const int64_t tok0 = static_cast<int64_t>(lc) * a.total_tokens + t_begin;
  const IO *gq = static_cast<const IO *>(a.q) + (tok0 * a.H_k + hk) * DK;
  const IO *gk = static_cast<const IO *>(a.k) + (tok0 * a.H_k + hk) * DK;
  const IO *gv = static_cast<const IO *>(a.v) + (tok0 * a.H_v + h) * DV;
  const float *gg = a.g + (tok0 * a.H_v + h) * (KDA ? DK : 1);
  const float *gb = a.beta + tok0 * a.H_v + h;
  OT *go = a.o ? static_cast<OT *>(a.o) + (tok0 * a.H_v + h) * DV : nullptr;
  const int64_t qk_stride = static_cast<int64_t>(a.H_k) * DK, v_stride = static_cast<int64_t>(a.H_v) * DV;
  const int64_t g_stride = static_cast<int64_t>(a.H_v) * (KDA ? DK : 1), b_stride = a.H_v;

  // raw rows of a group -> shared memory; consecutive threads take 16-byte vectors of all streams
  auto stage = [&](int grp) {
    const int t_lo = grp * TB, buf = grp & 1;
    const int cnt = min(TB, n_tok - t_lo);
    constexpr int QV = DK * sizeof(IO) / 16, VV = DV * sizeof(IO) / 16, GV = KDA ? DK * 4 / 16 : 1;
    for (int i = ht; i < cnt * QV; i += NT) {
      const int t = i / QV, j = i % QV;
      cp_async16(reinterpret_cast<char *>(&sm.q[buf][t][0]) + j * 16,
                 reinterpret_cast<const char *>(gq + (t_lo + t) * qk_stride) + j * 16);
      cp_async16(reinterpret_cast<char *>(&sm.k[buf][t][0]) + j * 16,
                 reinterpret_cast<const char *>(gk + (t_lo + t) * qk_stride) + j * 16);
    }
    for (int i = ht; i < cnt * VV; i += NT) {
      const int t = i / VV, j = i % VV;
      cp_async16(reinterpret_cast<char *>(&sm.v[buf][t][0]) + j * 16,
                 reinterpret_cast<const char *>(gv + (t_lo + t) * v_stride) + j * 16);
    }
    if constexpr (KDA) {
      for (int i = ht; i < cnt * GV; i += NT) {
        const int t = i / GV, j = i % GV;
        cp_async16(reinterpret_cast<char *>(&sm.g[buf][t][0]) + j * 16,
                   reinterpret_cast<const char *>(gg + (t_lo + t) * g_stride) + j * 16);
      }
    } else {
      for (int t = ht; t < cnt; t += NT) cp_async4(&sm.g[buf][t][0], gg + (t_lo + t) * g_stride);
    }
    for (int t = ht; t < cnt; t += NT) cp_async4(&sm.beta[buf][t], gb + (t_lo + t) * b_stride);
    cp_async_commit();
  };

  const int n_grp = n_tok > 0 ? (n_tok + TB - 1) / TB : 0;

  // row pairs (4 (i SL + slice) + 2p, + 1) of column col0 + c
  uint64_t S[NV][2][COLS];
#pragma unroll
  for (int i = 0; i < NV; ++i)
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const float *row = st + (4 * (i * SL + slice) + 2 * p) * DV + col0;
      float x[COLS] = {}, y[COLS] = {};
      if (a.mode == DASC_REFRESH_CONTINUE && !helper) {
        load_cols<COLS>(x, row);
        load_cols<COLS>(y, row + DV);
      }
#pragma unroll
      for (int c = 0; c < COLS; ++c) S[i][p][c] = pack2(x[c], y[c]);
    }

  // x[c] summed over the COLS lanes around this one, column `own` of it: COLS - 1 shuffles
  auto scatter = [&](float (&x)[COLS]) {
#pragma unroll
    for (int w = COLS / 2; w > 0; w >>= 1) {
      const bool up = (slice & w) != 0;
#pragma unroll
      for (int c = 0; c < w; ++c) {
        const float give = up ? x[c] : x[c + w];
        x[c] = (up ? x[c + w] : x[c]) + __shfl_xor_sync(0xffffffffu, give, w);
      }
    }
    return x[0];
  };
  // column sums over the whole column's lanes, of column `own`
  auto reduce = [&](const uint64_t (&acc)[COLS][2]) {
    float x[COLS];
#pragma unroll
    for (int c = 0; c < COLS; ++c) x[c] = sum2(add2(acc[c][0], acc[c][1]));
    float r = scatter(x);
#pragma unroll
    for (int d = COLS; d < SL; d <<= 1) r += __shfl_xor_sync(0xffffffffu, r, d);
    return r;
  };
  // raw -> converted
  auto convert = [&](int grp) {
    const int buf = grp & 1, cnt = min(TB, n_tok - grp * TB);
    typename Smem::Group &G = sm.grp[AHEAD ? buf : 0];
#pragma unroll 4
    for (int i = ht; i < cnt * DK; i += NT) {
      const int t = i / DK, c = i % DK;
      G.kf[t][c] = io_to_float<IO>(sm.k[buf][t][c]);
      if (go) G.qf[t][c] = io_to_float<IO>(sm.q[buf][t][c]) * a.q_scale;
      if constexpr (KDA) G.af[t][c] = expf(sm.g[buf][t][c]);
    }
    for (int i = ht; i < cnt * DV; i += NT) G.vf[i / DV][i % DV] = io_to_float<IO>(sm.v[buf][i / DV][i % DV]);
    for (int t = ht; t < cnt; t += NT) {
      G.bf[t] = sm.beta[buf][t];
      if constexpr (!KDA) G.af[t][0] = expf(sm.g[buf][t][0]);
    }
    for (int t = ht / 32 + 1; t < cnt; t += NT / 32) {  // a warp per token
      float c = 0.f;
#pragma unroll
      for (int i = ht % 32; i < DK; i += 32)
        c = fmaf(io_to_float<IO>(sm.k[buf][t][i]) * (KDA ? expf(sm.g[buf][t][i]) : 1.f), io_to_float<IO>(sm.k[buf][t - 1][i]), c);
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) c += __shfl_xor_sync(0xffffffffu, c, d);
      if constexpr (!KDA) c *= expf(sm.g[buf][t][0]);
      if (ht % 32 == 0) G.cf[t] = c;
    }
  };
  // the outputs of a group, 16 bytes of `OT` per store
  auto flush = [&](int grp) {
    if (!go) return;
    constexpr int OV = 16 / sizeof(OT);
    const int t_lo = grp * TB, cnt = min(TB, n_tok - t_lo);
    const typename Smem::Group &G = sm.grp[AHEAD ? grp & 1 : 0];
    for (int i = ht; i < cnt * (DV / OV); i += NT) {
      const int t = i / (DV / OV), j = i % (DV / OV) * OV;
      alignas(16) OT w[OV];
#pragma unroll
      for (int e = 0; e < OV; ++e) {
        const float2 *p = reinterpret_cast<const float2 *>(G.of[t][j + e]);
        float x = 0.f, y = 0.f;
#pragma unroll
        for (int sl = 0; sl < NOP / 2; ++sl) {
          x += p[sl].x;
          y += p[sl].y;
        }
        w[e] = float_to_io<OT>(x + y);
      }
      *reinterpret_cast<uint4 *>(go + (t_lo + t) * v_stride + j) = *reinterpret_cast<const uint4 *>(w);
    }
  };
  auto sync_helpers = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); };

  // Group 0 is converted by the helpers (or by everyone) before the loop.
  if (n_grp > 0 && ht >= 0) {
    stage(0);
    if (AHEAD) {
      cp_async_wait_all();
      sync_helpers();
      if (n_grp > 1) stage(1);
      convert(0);
    }
  }
  if (AHEAD) __syncthreads();
  for (int grp = 0; grp < n_grp; ++grp) {
    const int cnt = min(TB, n_tok - grp * TB);
    // one token group (about 2 us) before the end: see launch.cuh; a list has more units to come
    if (grp + 1 == n_grp && !a.from_list) stream_order_release();
    if constexpr (AHEAD) {
      // extra warps: the group before goes out, the next one is converted, the one after that is fetched
      if (helper) {
        if (grp + 1 < n_grp) {
          if (grp + 2 < n_grp) stage(grp + 2);
          cp_async_wait_but(grp + 2 < n_grp);
          sync_helpers();
          convert(grp + 1);
        }
        if (grp > 0) flush(grp - 1);
        __syncthreads();
        continue;
      }
    } else {
      cp_async_wait_all();
      __syncthreads();  // the raw rows have landed; everyone is past the previous group's converted rows
      if (grp + 1 < n_grp) stage(grp + 1);
      if (grp > 0) flush(grp - 1);
      convert(grp);
      __syncthreads();
    }
    const typename Smem::Group &G = sm.grp[AHEAD ? grp & 1 : 0];

    // (alpha_t k_t)^T x over this lane's rows, x = the state before or behind the decay of the token before
    uint64_t al2[NV][2];
    auto dot = [&](int t, uint64_t (&acc)[COLS][2]) {
      uint64_t as = 0ull;
      if constexpr (!KDA) as = pack2(G.af[t][0], G.af[t][0]);
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const ulonglong2 kk = (reinterpret_cast<const ulonglong2 *>(G.kf[t]) + slice)[i * SL];
        ulonglong2 al = make_ulonglong2(as, as);
        if constexpr (KDA) al = (reinterpret_cast<const ulonglong2 *>(G.af[t]) + slice)[i * SL];
        al2[i][0] = al.x;
        al2[i][1] = al.y;
        const uint64_t k0 = mul2(kk.x, al.x), k1 = mul2(kk.y, al.y);
#pragma unroll
        for (int c = 0; c < COLS; ++c) {
          acc[c][0] = i == 0 ? mul2(k0, S[i][0][c]) : fma2(k0, S[i][0][c], acc[c][0]);
          acc[c][1] = i == 0 ? mul2(k1, S[i][1][c]) : fma2(k1, S[i][1][c], acc[c][1]);
        }
      }
    };
    // u of one column in every lane that holds it; S <- alpha S (the decay of the token whose dot() came last)
    auto decay = [&]() {
#pragma unroll
      for (int i = 0; i < NV; ++i)
#pragma unroll
        for (int c = 0; c < COLS; ++c) {
          S[i][0][c] = mul2(S[i][0][c], al2[i][0]);
          S[i][1][c] = mul2(S[i][1][c], al2[i][1]);
        }
    };
    uint64_t acc[COLS][2];
    dot(0, acc);
    decay();
    float u = G.bf[0] * (G.vf[0][col0 + own] - reduce(acc));
    auto token = [&](int t, auto has_next) {
      // S = Diag(alpha_t) S_{t-1} here.  The next token's r is split, r_{t+1} = (alpha k)_{t+1}^T Diag(alpha_t) S_{t-1} + c_{t+1} u_t,
      // so that its dot product and shuffles run beside this token's update instead of behind it.
      constexpr bool next = decltype(has_next)::value;
      if constexpr (next) dot(t + 1, acc);
      uint64_t uu[COLS];
#pragma unroll
      for (int c = 0; c < COLS; ++c) {
        const float x = __shfl_sync(0xffffffffu, u, (threadIdx.x & 31 & ~(COLS - 1)) + c);
        uu[c] = pack2(x, x);
      }
      float p = 0.f;
      if constexpr (next) p = reduce(acc);
      uint64_t oa[COLS][2];
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const ulonglong2 kk = (reinterpret_cast<const ulonglong2 *>(G.kf[t]) + slice)[i * SL];
        const ulonglong2 qq = (reinterpret_cast<const ulonglong2 *>(G.qf[t]) + slice)[i * SL];
#pragma unroll
        for (int c = 0; c < COLS; ++c) {
          S[i][0][c] = fma2(kk.x, uu[c], S[i][0][c]);
          S[i][1][c] = fma2(kk.y, uu[c], S[i][1][c]);
          oa[c][0] = i == 0 ? mul2(qq.x, S[i][0][c]) : fma2(qq.x, S[i][0][c], oa[c][0]);
          oa[c][1] = i == 0 ? mul2(qq.y, S[i][1][c]) : fma2(qq.y, S[i][1][c], oa[c][1]);
        }
      }
      if constexpr (next) {
        decay();
        u = G.bf[t + 1] * (G.vf[t + 1][col0 + own] - fmaf(G.cf[t + 1], u, p));
      }
      if (go) {
        float x[COLS];
#pragma unroll
        for (int c = 0; c < COLS; ++c) x[c] = sum2(add2(oa[c][0], oa[c][1]));
        const float o = scatter(x);
        // no "memory" clobber: the loads of the next token may be moved above this store
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(&G.of[t][col0 + own][slice / COLS]))), "f"(o));
      }
    };
    // one straight block per token, so that the scheduler can interleave the two halves
#pragma unroll 2
    for (int t = 0; t + 1 < cnt; ++t) token(t, std::true_type{});
    token(cnt - 1, std::false_type{});
    if (AHEAD) __syncthreads();
  }
  __syncthreads();
  if (n_grp > 0 && (!AHEAD || helper)) flush(n_grp - 1);
  if (helper) return;

  const uint8_t *keep = a.row_keep + static_cast<int64_t>(layer) * a.rows_per_layer + static_cast<int64_t>(h) * DK;
  const bool all_rows = a.mode == DASC_REFRESH_CONTINUE;
#pragma unroll
  for (int i = 0; i < NV; ++i)
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int row = 4 * (i * SL + slice) + 2 * p;
      float lo[COLS], hi[COLS];
#pragma unroll
      for (int c = 0; c < COLS; ++c) asm("mov.b64 {%0, %1}, %2;" : "=f"(lo[c]), "=f"(hi[c]) : "l"(S[i][p][c]));
      float *d = st + row * DV + col0;
      if (all_rows || !keep[row]) store_cols<COLS>(d, lo);
      if (all_rows || !keep[row + 1]) store_cols<COLS>(d + DV, hi);
    }
}

// grid = one CTA per unit (from_list == 0), or a fixed grid whose CTAs walk the list of units that the
// chunked kernel handed over (from_list == 1; the list and its length are in the workspace, written earlier on the same stream).
template <int DK, int DV, int COLS, int SL, int NHELP, typename IO, typename OT, bool KDA>
__global__ void __launch_bounds__(DV / COLS *SL + NHELP) refresh_seq_kernel(DascRefreshArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  stream_order_wait();
  if (!a.from_list) {
    seq_unit<DK, DV, COLS, SL, NHELP, IO, OT, KDA>(a, static_cast<int>(blockIdx.x), smem_raw);
    return;
  }
  uint32_t *ws = static_cast<uint32_t *>(a.workspace);
  const uint32_t listed = ws[2];
  const int n_list = static_cast<int>(listed < static_cast<uint32_t>(a.unit_list_cap) ? listed : a.unit_list_cap);
  for (int i = blockIdx.x; i < n_list; i += gridDim.x) {
    seq_unit<DK, DV, COLS, SL, NHELP, IO, OT, KDA>(a, a.unit_list[i], smem_raw);
    if (threadIdx.x == 0) atomicAdd(ws + 3, 1u);
    __syncthreads();  // the next unit reuses the staging buffers
  }
}

template <int DK, int DV, int COLS, int SL, int NHELP, typename IO, typename OT, bool KDA>
int launch(const DascRefreshArgs &a, void *stream) {
  constexpr size_t smem = sizeof(SeqSmem<DK, DV, SL / COLS, (NHELP > 0), IO, KDA>);
  auto kern = refresh_seq_kernel<DK, DV, COLS, SL, NHELP, IO, OT, KDA>;
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return static_cast<int>(e);
  }
  const int64_t n_ctas = static_cast<int64_t>(a.n_req) * a.n_layers_in_call * a.H_v;
  if (n_ctas == 0) return cudaSuccess;
  if (n_ctas > 2147483647LL) return static_cast<int>(cudaErrorInvalidConfiguration);
  // a handed-over list is short (units outside the chunked kernel's range or below its length threshold): a grid
  // of a CTA per SM walks it, and costs next to nothing when the list is empty
  const int64_t grid = a.from_list ? (n_ctas < 148 ? n_ctas : 148) : n_ctas;
  return static_cast<int>(launch_in_order(kern, dim3(static_cast<unsigned>(grid)), dim3(DV / COLS * SL + NHELP), smem, stream, a));
}

// ---------------------------------------------------------------------------------------------
// Four tokens at a time, where no SM has more than one unit or part of one (d = 32: two): there the serial chain is all there is.
// With D_t the product of the decays of the block's tokens up to t, and everything else over the block's tokens j < t or j <= t,
//   r_t = (D_t k_t)^T S_0 + sum_j c_tj u_j        c_tj = k_t^T Diag(alpha_{j+1} ... alpha_t) k_j
//   o_t = (D_t q_t)^T S_0 + sum_j p_tj u_j        p_tj = q_t^T Diag(alpha_{j+1} ... alpha_t) k_j
//   S_4 = Diag(D_3) S_0 + sum_j w_j u_j^T         w_j = Diag(alpha_{j+1} ... alpha_3) k_j
// so that the four dot products of a lane and their shuffles run side by side and one chain of multiply-adds per block is left.  All
// factors are products of at most two exponentials, of sums of the log-decay: no division, and half of the token-by-token form's error
// against fp64 (4 units of 64 x 64, 64 tokens: state 6.2e-7 -> 3.0e-7, outputs 3.5e-7 -> 2.0e-7), whose decays multiply up one token at
// a time.  The helper warps form D k, D q, w and the 16 coefficients of a block, a group of tokens ahead.  Narrow parts take 95 ns per token at
// d = 64 (135 before), 750 cycles per block.  No unit of the SM is at its limit then (4 units of 1024 tokens: issue slots 41 % busy, of the SM's
// busiest quarter 53 %, the shared-memory pipe 62 %): what is left is the chain of a block and the hand-over of groups, whose shares have not been
// told apart.  Wide parts are bound by the replaying lanes' operand reads.  More helper warps, or copies and outputs in warps of their own, gained nothing.
// ---------------------------------------------------------------------------------------------
constexpr int NB = TB / 4;  // blocks of a group

template <int DK, int NCOL, int SL, typename IO, bool KDA>
struct BlockSmem {
  // raw staging, NRAW - 1 groups ahead of the one that is being converted: a group takes less than a trip to memory
  static constexpr int NRAW = DK * NCOL <= 128 * 32 ? 4 : 3;
  alignas(16) IO q[NRAW][TB][DK];
  alignas(16) IO k[NRAW][TB][DK];
  alignas(16) IO v[NRAW][TB][NCOL];
  alignas(16) float g[NRAW][TB][KDA ? DK : 4];
  alignas(16) float beta[NRAW][TB];
  struct Group {
    alignas(16) float kf[TB][DK];  // D k
    alignas(16) float qf[TB][DK];  // D q
    alignas(16) float wf[TB][DK];
    alignas(16) float df[NB][DK];  // D_3
    alignas(16) float cf[NB][2][16];  // two shares of c_10, c_20, c_21, c_30, c_31, c_32, p_00, p_10, p_11, p_20 ... p_33
    alignas(16) float vf[TB][NCOL];
    alignas(16) float bf[TB];
    alignas(16) float of[TB][NCOL][SL];  // SL shares of each output
  } grp[2];
};

template <int DK, int DV, int NCOL, int COLS, int SL, int NHELP, typename IO, typename OT, bool KDA>
__device__ __forceinline__ void seq_unit_blocks(const DascRefreshArgs &a, int unit, int part, unsigned char *smem_raw) {
  constexpr int NC = NCOL / COLS * SL;  // threads that replay tokens, COLS columns per SL lanes
  constexpr int NV = DK / SL / 4;  // groups of four rows held by one lane
  // Looks at whether any tokens are left, ahead of so many of a group's later blocks: a call of a few tokens does not replay blocks of
  // nothing.  128 tokens' worth of wide parts does not notice them, narrow ones lose the overlap of a block with the next
  // (4 units of 64 x 64, 250 tokens 26.7 us without, 27.6 with all three; of 128 x 128 38.2 without, 38.2 with one, 38.7 with two).
  // us for one token, without / with: 148 units of 64 x 64 7.0 / 4.4, 74 of 128 x 128 9.3 / 5.8 (5.3 with two columns per load and store of
  // the state), 4 of them 4.8 / 4.0.
  constexpr int CHECKS = DK * NCOL >= 2048 ? NB - 1 : DK * NCOL < 1024 ? 0 : DK == 32 ? 1 : 2;
  using Smem = BlockSmem<DK, NCOL, SL, IO, KDA>;
  constexpr int NRAW = Smem::NRAW;
  Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
  const int tid = threadIdx.x;
  const bool helper = tid >= NC;
  const int ht = tid - NC;  // index among the helpers
  const int slice = tid % SL, col = tid / SL * COLS;

  const int h = unit % a.H_v;
  const int lc = (unit / a.H_v) % a.n_layers_in_call;
  const int r = unit / (a.H_v * a.n_layers_in_call);
  const int hk = h / (a.H_v / a.H_k);
  const int layer = a.layer_begin + lc;
  const int64_t t_begin = a.tok_begin ? a.tok_begin[r] : a.cu_seqlens[r];
  const int n_tok = static_cast<int>(a.cu_seqlens[r + 1] - t_begin);
  if (n_tok <= 0 && a.mode == DASC_REFRESH_CONTINUE) return;

  float *st = a.state + static_cast<int64_t>(a.req_idx[r]) * a.req_stride + static_cast<int64_t>(layer) * a.layer_stride +
              static_cast<int64_t>(h) * DK * DV + part * NCOL;
  const int64_t tok0 = static_cast<int64_t>(lc) * a.total_tokens + t_begin;
  const IO *gq = static_cast<const IO *>(a.q) + (tok0 * a.H_k + hk) * DK;
  const IO *gk = static_cast<const IO *>(a.k) + (tok0 * a.H_k + hk) * DK;
  const IO *gv = static_cast<const IO *>(a.v) + (tok0 * a.H_v + h) * DV + part * NCOL;
  const float *gg = a.g + (tok0 * a.H_v + h) * (KDA ? DK : 1);
  const float *gb = a.beta + tok0 * a.H_v + h;
  OT *go = a.o ? static_cast<OT *>(a.o) + (tok0 * a.H_v + h) * DV + part * NCOL : nullptr;
  const int64_t qk_stride = static_cast<int64_t>(a.H_k) * DK, v_stride = static_cast<int64_t>(a.H_v) * DV;
  const int64_t g_stride = static_cast<int64_t>(a.H_v) * (KDA ? DK : 1), b_stride = a.H_v;
  const int n_grp = n_tok > 0 ? (n_tok + TB - 1) / TB : 0;

  // raw rows of a group -> shared memory; consecutive threads take 16-byte vectors of all streams
  auto stage = [&](int grp) {
    const int t_lo = grp * TB, buf = grp % NRAW;
    const int cnt = min(TB, n_tok - t_lo);  // (none past the end: an empty group is committed)
    constexpr int QV = DK * sizeof(IO) / 16, VV = NCOL * sizeof(IO) / 16, GV = KDA ? DK * 4 / 16 : 1;
    for (int i = ht; i < cnt * QV; i += NHELP) {
      const int t = i / QV, j = i % QV;
      if (go)
        cp_async16(reinterpret_cast<char *>(&sm.q[buf][t][0]) + j * 16, reinterpret_cast<const char *>(gq + (t_lo + t) * qk_stride) + j * 16);
      cp_async16(reinterpret_cast<char *>(&sm.k[buf][t][0]) + j * 16, reinterpret_cast<const char *>(gk + (t_lo + t) * qk_stride) + j * 16);
    }
    for (int i = ht; i < cnt * VV; i += NHELP) {
      const int t = i / VV, j = i % VV;
      cp_async16(reinterpret_cast<char *>(&sm.v[buf][t][0]) + j * 16, reinterpret_cast<const char *>(gv + (t_lo + t) * v_stride) + j * 16);
    }
    if constexpr (KDA) {
      for (int i = ht; i < cnt * GV; i += NHELP) {
        const int t = i / GV, j = i % GV;
        cp_async16(reinterpret_cast<char *>(&sm.g[buf][t][0]) + j * 16, reinterpret_cast<const char *>(gg + (t_lo + t) * g_stride) + j * 16);
      }
    } else {
      for (int t = ht; t < cnt; t += NHELP) cp_async4(&sm.g[buf][t][0], gg + (t_lo + t) * g_stride);
    }
    for (int t = ht; t < cnt; t += NHELP) cp_async4(&sm.beta[buf][t], gb + (t_lo + t) * b_stride);
    cp_async_commit();
  };
  // raw -> what the replaying lanes read.  Tokens past the end of the request: k = q = v = beta = 0, alpha = 1.
  auto convert = [&](int grp) {
    const int buf = grp % NRAW, cnt = min(TB, n_tok - grp * TB);
    typename Smem::Group &G = sm.grp[grp & 1];
    constexpr int PER = DK < NHELP / NB ? DK : NHELP / NB;  // threads of a block
    static_assert(PER % 32 == 0 && PER <= 64 && DK % PER == 0);
    if (const int b = ht / PER; b < NB && (CHECKS == 0 || min(b, CHECKS) * 4 < cnt)) {  // (what will be replayed; a warp's threads are in one block)
      float x[16] = {};
      // products of decays, mostly as exponentials of sums: at most two of them multiplied instead of four
      float dd[4], a1, a2, a3, a12, a23, a13;
      auto decays = [&](int c) {
        float g[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) g[t] = b * 4 + t < cnt ? sm.g[buf][b * 4 + t][c] : 0.f;
        const float g23 = g[2] + g[3];
        a1 = expf(g[1]), a2 = expf(g[2]), a3 = expf(g[3]), a12 = expf(g[1] + g[2]), a23 = expf(g23), a13 = expf(g[1] + g23);
        dd[0] = expf(g[0]), dd[1] = dd[0] * a1, dd[2] = dd[0] * a12, dd[3] = dd[0] * a13;
      };
      if constexpr (!KDA) decays(0);
#pragma unroll
      for (int c = ht % PER; c < DK; c += PER) {
        if constexpr (KDA) decays(c);
        float k[4], q[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int tt = b * 4 + t;
          const bool in = tt < cnt;
          k[t] = in ? io_to_float<IO>(sm.k[buf][tt][c]) : 0.f;
          q[t] = in && go ? io_to_float<IO>(sm.q[buf][tt][c]) * a.q_scale : 0.f;
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          G.kf[b * 4 + t][c] = k[t] * dd[t];
          if (go) G.qf[b * 4 + t][c] = q[t] * dd[t];
        }
        // from[t][j]: k_j carried from token j to token t
        const float k01 = k[0] * a1, k02 = k[0] * a12, k03 = k[0] * a13, k12 = k[1] * a2, k13 = k[1] * a23, k23 = k[2] * a3;
        G.wf[b * 4 + 0][c] = k03;
        G.wf[b * 4 + 1][c] = k13;
        G.wf[b * 4 + 2][c] = k23;
        G.wf[b * 4 + 3][c] = k[3];
        G.df[b][c] = dd[3];
        x[0] = fmaf(k[1], k01, x[0]);
        x[1] = fmaf(k[2], k02, x[1]);
        x[2] = fmaf(k[2], k12, x[2]);
        x[3] = fmaf(k[3], k03, x[3]);
        x[4] = fmaf(k[3], k13, x[4]);
        x[5] = fmaf(k[3], k23, x[5]);
        x[6] = fmaf(q[0], k[0], x[6]);
        x[7] = fmaf(q[1], k01, x[7]);
        x[8] = fmaf(q[1], k[1], x[8]);
        x[9] = fmaf(q[2], k02, x[9]);
        x[10] = fmaf(q[2], k12, x[10]);
        x[11] = fmaf(q[2], k[2], x[11]);
        x[12] = fmaf(q[3], k03, x[12]);
        x[13] = fmaf(q[3], k13, x[13]);
        x[14] = fmaf(q[3], k23, x[14]);
        x[15] = fmaf(q[3], k[3], x[15]);
      }
      // the warp's sums, number i in lanes 2i and 2i + 1
      const int lane = ht & 31;
#pragma unroll
      for (int w = 8; w > 0; w >>= 1) {
        const bool up = (lane & (2 * w)) != 0;
#pragma unroll
        for (int i = 0; i < w; ++i) {
          const float give = up ? x[i] : x[i + w];
          x[i] = (up ? x[i + w] : x[i]) + __shfl_xor_sync(0xffffffffu, give, 2 * w);
        }
      }
      x[0] += __shfl_xor_sync(0xffffffffu, x[0], 1);
      if ((lane & 1) == 0) G.cf[b][ht % PER / 32][lane / 2] = x[0];
      if (PER == 32 && (lane & 1) == 1) G.cf[b][1][lane / 2] = 0.f;
    }
    for (int i = ht; i < TB * NCOL; i += NHELP) {
      const int t = i / NCOL, c = i % NCOL;
      G.vf[t][c] = t < cnt ? io_to_float<IO>(sm.v[buf][t][c]) : 0.f;
    }
    for (int t = ht; t < TB; t += NHELP) G.bf[t] = t < cnt ? sm.beta[buf][t] : 0.f;
  };
  // the outputs of a group, 16 bytes of `OT` per store
  auto flush = [&](int grp) {
    if (!go) return;
    constexpr int OV = 16 / sizeof(OT);
    const int t_lo = grp * TB, cnt = min(TB, n_tok - t_lo);
    const typename Smem::Group &G = sm.grp[grp & 1];
    for (int i = ht; i < cnt * (NCOL / OV); i += NHELP) {
      const int t = i / (NCOL / OV), j = i % (NCOL / OV) * OV;
      alignas(16) OT w[OV];
#pragma unroll
      for (int e = 0; e < OV; ++e) {
        const float4 *p = reinterpret_cast<const float4 *>(G.of[t][j + e]);
        float4 s = p[0];
#pragma unroll
        for (int sl = 1; sl < SL / 4; ++sl) s = make_float4(s.x + p[sl].x, s.y + p[sl].y, s.z + p[sl].z, s.w + p[sl].w);
        w[e] = float_to_io<OT>((s.x + s.y) + (s.z + s.w));
      }
      *reinterpret_cast<uint4 *>(go + (t_lo + t) * v_stride + j) = *reinterpret_cast<const uint4 *>(w);
    }
  };
  // the oldest group but NRAW - 2 has landed, for all helpers (who are past the conversion whose raw rows are overwritten next)
  auto landed = [&]() {
    asm volatile("cp.async.wait_group %0;\n\tbar.sync 1, %1;" ::"n"(NRAW - 2), "n"(NHELP) : "memory");
  };

  if (helper) {
    if (n_grp > 0) {
#pragma unroll
      for (int i = 0; i < NRAW - 1; ++i) stage(i);
      landed();
      convert(0);
    }
    __syncthreads();
    for (int grp = 0; grp < n_grp; ++grp) {
      // the group before goes out, the next one is converted, the one after that is fetched
      if (grp + 1 < n_grp) {
        stage(grp + NRAW - 1);
        landed();
        convert(grp + 1);
      }
      if (grp > 0) flush(grp - 1);
      __syncthreads();
    }
    if (n_grp > 0) flush(n_grp - 1);
    return;
  }

  // row pairs (4 (i SL + slice) + 2p, + 1) of this lane's columns
  uint64_t S[COLS][NV][2];
#pragma unroll
  for (int i = 0; i < NV; ++i)
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const float *row = st + (4 * (i * SL + slice) + 2 * p) * DV + col;
      if constexpr (COLS == 1) {  // (as below it took 0.07 us of the 8.7 us of 4 units of 64 x 64, 64 tokens)
        S[0][i][p] = a.mode == DASC_REFRESH_CONTINUE ? pack2(row[0], row[DV]) : 0ull;
      } else {
        float x[COLS] = {}, y[COLS] = {};
        if (a.mode == DASC_REFRESH_CONTINUE) {
          load_cols<COLS>(x, row);
          load_cols<COLS>(y, row + DV);
        }
#pragma unroll
        for (int e = 0; e < COLS; ++e) S[e][i][p] = pack2(x[e], y[e]);
      }
    }
  __syncthreads();
  for (int grp = 0; grp < n_grp; ++grp) {
    const int cnt = min(TB, n_tok - grp * TB);
    // one token group before the end: see launch.cuh
    if (grp + 1 == n_grp) stream_order_release();
    typename Smem::Group &G = sm.grp[grp & 1];
    // straight code for the whole group but for CHECKS (tokens past its end are zeros), so that the outputs of a block fill the waits of the
    // next one
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      if (b > 0 && b <= CHECKS && b * 4 >= cnt) break;
      ulonglong2 k[4][NV], w[4][NV], d[NV];
      auto load = [&](ulonglong2(&x)[NV], const float *row) {
#pragma unroll
        for (int i = 0; i < NV; ++i) x[i] = (reinterpret_cast<const ulonglong2 *>(row) + slice)[i * SL];
      };
#pragma unroll
      for (int t = 0; t < 4; ++t) load(k[t], G.kf[b * 4 + t]);
      float v[COLS][4], cf[16];
#pragma unroll
      for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int e = 0; e < COLS; ++e) v[e][t] = G.vf[b * 4 + t][col + e];
      const float4 be4 = *reinterpret_cast<const float4 *>(&G.bf[b * 4]);
      const float be[4] = {be4.x, be4.y, be4.z, be4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 x = reinterpret_cast<const float4 *>(G.cf[b][0])[i], y = reinterpret_cast<const float4 *>(G.cf[b][1])[i];
        cf[4 * i] = x.x + y.x;
        cf[4 * i + 1] = x.y + y.y;
        cf[4 * i + 2] = x.z + y.z;
        cf[4 * i + 3] = x.w + y.w;
      }
      load(d, G.df[b]);
#pragma unroll
      for (int t = 0; t < 4; ++t) load(w[t], G.wf[b * 4 + t]);
      auto dot = [&](const ulonglong2(&x)[NV], int e) {
        uint64_t acc0 = mul2(x[0].x, S[e][0][0]), acc1 = mul2(x[0].y, S[e][0][1]);
#pragma unroll
        for (int i = 1; i < NV; ++i) {
          acc0 = fma2(x[i].x, S[e][i][0], acc0);
          acc1 = fma2(x[i].y, S[e][i][1], acc1);
        }
        return sum2(add2(acc0, acc1));
      };
      float p[COLS][4], o[COLS][4];
#pragma unroll
      for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int e = 0; e < COLS; ++e) p[e][t] = dot(k[t], e);
      if (go) {  // this lane's shares of the outputs, from the state before the block
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          load(k[t], G.qf[b * 4 + t]);
#pragma unroll
          for (int e = 0; e < COLS; ++e) o[e][t] = dot(k[t], e);
        }
      }
#pragma unroll
      for (int e = 0; e < COLS; ++e)
#pragma unroll
        for (int i = 0; i < NV; ++i) {
          S[e][i][0] = mul2(S[e][i][0], d[i].x);
          S[e][i][1] = mul2(S[e][i][1], d[i].y);
        }
#pragma unroll
      for (int dd = 1; dd < SL; dd <<= 1)
#pragma unroll
        for (int t = 0; t < 4; ++t)
#pragma unroll
          for (int e = 0; e < COLS; ++e) p[e][t] += __shfl_xor_sync(0xffffffffu, p[e][t], dd);
      // tokens past the end write nothing, whatever the state holds
      float u[COLS][4];
#pragma unroll
      for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int e = 0; e < COLS; ++e) {
          float x = v[e][t] - p[e][t];
#pragma unroll
          for (int j = 0; j < t; ++j) x = fmaf(-cf[t * (t - 1) / 2 + j], u[e][j], x);
          u[e][t] = b * 4 + t < cnt ? be[t] * x : 0.f;
        }
#pragma unroll
      for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int e = 0; e < COLS; ++e) {
          const uint64_t uu = pack2(u[e][t], u[e][t]);
#pragma unroll
          for (int i = 0; i < NV; ++i) {
            S[e][i][0] = fma2(w[t][i].x, uu, S[e][i][0]);
            S[e][i][1] = fma2(w[t][i].y, uu, S[e][i][1]);
          }
        }
      if (go) {
        // the part of the block's own tokens goes into the first lane's share
#pragma unroll
        for (int t = 0; t < 4; ++t)
#pragma unroll
          for (int e = 0; e < COLS; ++e) {
            float x = 0.f;
#pragma unroll
            for (int j = 0; j <= t; ++j) x = fmaf(cf[6 + t * (t + 1) / 2 + j], u[e][j], x);
            if (slice == 0) o[e][t] += x;
            // no "memory" clobber: the loads of the next block may be moved above these stores
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(&G.of[b * 4 + t][col + e][slice]))),
                         "f"(o[e][t]));
          }
      }
    }
    __syncthreads();
  }

  const uint8_t *keep = a.row_keep + static_cast<int64_t>(layer) * a.rows_per_layer + static_cast<int64_t>(h) * DK;
  const bool all_rows = a.mode == DASC_REFRESH_CONTINUE;
#pragma unroll
  for (int i = 0; i < NV; ++i)
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int row = 4 * (i * SL + slice) + 2 * p;
      float lo[COLS], hi[COLS];
#pragma unroll
      for (int e = 0; e < COLS; ++e) asm("mov.b64 {%0, %1}, %2;" : "=f"(lo[e]), "=f"(hi[e]) : "l"(S[e][i][p]));
      float *d = st + row * DV + col;
      if (all_rows || !keep[row]) store_cols<COLS>(d, lo);
      if (all_rows || !keep[row + 1]) store_cols<COLS>(d + DV, hi);
    }
}

template <int DK, int DV, int NCOL, int COLS, int SL, int NHELP, typename IO, typename OT, bool KDA>
__global__ void __launch_bounds__(NCOL / COLS *SL + NHELP) refresh_seq_blocks_kernel(DascRefreshArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  stream_order_wait();
  constexpr int PARTS = DV / NCOL;
  seq_unit_blocks<DK, DV, NCOL, COLS, SL, NHELP, IO, OT, KDA>(a, static_cast<int>(blockIdx.x) / PARTS, static_cast<int>(blockIdx.x) % PARTS, smem_raw);
}

template <int DK, int DV, int NCOL, int COLS, int SL, int NHELP, typename IO, typename OT, bool KDA>
int launch_blocks(const DascRefreshArgs &a, void *stream) {
  constexpr size_t smem = sizeof(BlockSmem<DK, NCOL, SL, IO, KDA>);
  static_assert(smem <= 227 * 1024);
  auto kern = refresh_seq_blocks_kernel<DK, DV, NCOL, COLS, SL, NHELP, IO, OT, KDA>;
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return static_cast<int>(e);
  }
  const int64_t n_ctas = static_cast<int64_t>(a.n_req) * a.n_layers_in_call * a.H_v * (DV / NCOL);
  if (n_ctas == 0) return cudaSuccess;
  if (n_ctas > 2147483647LL) return static_cast<int>(cudaErrorInvalidConfiguration);
  return static_cast<int>(launch_in_order(kern, dim3(static_cast<unsigned>(n_ctas)), dim3(NCOL / COLS * SL + NHELP), smem, stream, a));
}

// Columns do not interact, so units that leave SMs idle are split by columns: the widest parts that still have an SM each, down to 8
// columns (16 at d = 32), replayed four tokens at a time.  Beyond a CTA per SM the conversions, which every part repeats, cost more
// than the shorter chain saves.  From 32 columns on a part is bound by the operand reads of its replaying lanes (a warp's read costs its
// registers' share, whatever is broadcast), so that two columns per lane and few lanes per column pay there; narrow
// parts want the short dot products of 8 lanes.  d = 32 has operands small enough for two CTAs per SM.
// B200, 128 fp32 tokens, microseconds, KDA / GDN; "before" is the token-by-token form, split where the line before lay:
//   d = 32    4 units  16 columns 12.5 / 12.2, whole in blocks 15.6 / 15.5
//           148        16 columns 17.6 / 17.0, whole in blocks 15.8 / 15.7
//           152        16 columns 28.2 / 27.5, whole in blocks 30.4 / 30.1, before 35.7 / 36.0; 296 units 33.5, 30.8, 35.5; 304: 43.6, 45.2, 45.0
//   d = 64   18        8 columns 15.2 / 14.7, 16: 18.5 / 18.1
//            36        8 columns 26.9 / 26.4, 16: 18.5 / 18.0 (8 lanes 19.1 / 18.6), before 29.1
//            74        16 columns 36.1 / 35.1, 32: 24.2 / 23.8 (2 columns per lane, 8 lanes 25.0 / 24.4), before 41.9 / 40.5
//           148        32 columns 47.4 / 46.6, 64: 31.2 / 30.3 (1 per lane 41.6 / 41.3), before 42.2 / 41.0
//           152        64 columns 56.9 / 55.7, before 57.5 / 55.2; 296 units 60.8 / 59.0, 57.6 / 55.4
//   d = 128   8        8 columns 21.5 / 20.7, 16: 27.4 / 26.6
//            18        8 columns 41.7 / 39.5, 16: 27.7 / 26.8, before 59.5 / 36.3
//            36        16 columns 54.1 / 52.5, 32: 35.4 / 34.6 (1 per lane, 4 lanes 39.6 / 39.2), before 59.3 / 58.3
//            74        32 columns 69.1 / 67.2, 64: 48.4 / 46.8 (8 lanes 56.1 / 55.1), before 59.4 / 58.5
//            76        64 columns 87.9 / 86.4, whole in blocks 96.5 / 92.2, before 91.3 / 84.4; 148 units 95.2 / 92.3, 97.1 / 91.6, 89.6 / 83.0
constexpr int64_t kSms = 148;

template <int D, typename IO, typename OT, bool KDA>
int dispatch_split(const DascRefreshArgs &a, void *stream) {
  const int64_t n_units = static_cast<int64_t>(a.n_req) * a.n_layers_in_call * a.H_v;
  const auto fits = [&](int parts, int64_t ctas) { return !a.from_list && n_units * parts <= ctas; };
  if constexpr (D == 32) {
    // A few tokens end sooner without helper warps and groups of 16: us for 1 / 5 / 16 / 24 tokens, 296 units 7.3 / 7.5 / 7.8 / 10.9 in blocks,
    // 3.9 / 4.7 / 6.9 / 9.1 token by token (64: 17.6, 19.1); 148 units 4.0 / 4.1 / 4.2 / 5.9 and 3.8 / 3.9 / 6.0 / 7.8.
    const bool few = a.max_seqlen <= (n_units > kSms ? 24 : 5);
    if (!few && fits(2, kSms)) return launch_blocks<32, 32, 16, 1, 4, 256, IO, OT, KDA>(a, stream);
    if (!few && fits(1, 2 * kSms)) return launch_blocks<32, 32, 32, 1, 4, 256, IO, OT, KDA>(a, stream);
    return launch<32, 32, 2, 8, 0, IO, OT, KDA>(a, stream);
  } else if constexpr (D == 64) {
    if (fits(8, kSms)) return launch_blocks<64, 64, 8, 1, 8, 256, IO, OT, KDA>(a, stream);
    if (fits(4, kSms)) return launch_blocks<64, 64, 16, 1, 4, 256, IO, OT, KDA>(a, stream);
    if (fits(2, kSms)) return launch_blocks<64, 64, 32, 1, 4, 256, IO, OT, KDA>(a, stream);
    if (fits(1, kSms)) return launch_blocks<64, 64, 64, 2, 4, 256, IO, OT, KDA>(a, stream);
    return launch<64, 64, 4, 8, 128, IO, OT, KDA>(a, stream);
  } else {
    if (fits(16, kSms)) return launch_blocks<128, 128, 8, 1, 8, 256, IO, OT, KDA>(a, stream);
    if (fits(8, kSms)) return launch_blocks<128, 128, 16, 1, 8, 256, IO, OT, KDA>(a, stream);
    if (fits(4, kSms)) return launch_blocks<128, 128, 32, 2, 8, 256, IO, OT, KDA>(a, stream);
    if (fits(2, kSms)) return launch_blocks<128, 128, 64, 2, 4, 256, IO, OT, KDA>(a, stream);
    return launch<128, 128, 4, 16, 0, IO, OT, KDA>(a, stream);
  }
}

template <int D, typename IO, typename OT>
int dispatch_kind(const DascRefreshArgs &a, void *stream) {
  return a.kind == DASC_KDA ? dispatch_split<D, IO, OT, true>(a, stream) : dispatch_split<D, IO, OT, false>(a, stream);
}

}  // namespace

// Compiled once per head dimension (DASC_SEQ_DIM), each in a translation unit of its own, side by side: 30 s for the longest
// (128) against 70 s for all in one.  The type of the outputs stays a template parameter: looked at at run time it halves the
// kernels and leaves fewer that spill (5 instead of 12, at most 60 bytes), but at d = 128 those are 1 to 14 % slower.
template <int D>
int dasc_launch_refresh_seq_dim(const DascRefreshArgs &a, void *stream) {
  const bool o_bf16 = a.o ? a.o_bf16 != 0 : a.io_bf16 != 0;  // no output: any instantiation will do
  if (a.io_bf16)
    return o_bf16 ? dispatch_kind<D, __nv_bfloat16, __nv_bfloat16>(a, stream) : dispatch_kind<D, __nv_bfloat16, float>(a, stream);
  return o_bf16 ? dispatch_kind<D, float, __nv_bfloat16>(a, stream) : dispatch_kind<D, float, float>(a, stream);
}

template int dasc_launch_refresh_seq_dim<DASC_SEQ_DIM>(const DascRefreshArgs &, void *);
