// Decode step of ONE row (M = 1) under the complete-graph law with q equal groups, in ONE launch: a projection
// y = act(x *_q W + b), the FFN  y = act(x *_q W_up + b_up) *_q W_down + b_down, or the gated FFN
// y = (silu(x * W_gate) .* (x * W_up)) * W_down  (the M = 1 rows of the paper's kernel tables, appendix "Kernel
// Benchmark Details").
//
// A row of type i needs, for the output group j, the block W_ij of its row panel and the diagonal block W_jj
// (Eqs. typed-diag / typed-off): 2 s of the q s weight rows above every output column.  The step is a pair of
// matrix-vector products bound by memory LATENCY, so it runs on plain FMAs and is organised around the dependent
// round trips.  A warp owns a piece of 8 or 16 output columns (and, while there are more warps than pieces, a
// share of the weight rows); its lanes split the rows, every lane keeps all its loads of 16 bytes in flight and
// reads the activations it needs straight from global memory -- no staging, one CTA barrier per phase at most.
// The first weight loads are issued before the launch's dependency resolves (weights do not depend on the previous
// kernel), those of W_down before the second phase of an FFN.  Phase 1 of an FFN writes the hidden row h (bf16) to the
// handle's exchange buffer; phase 2 is the same routine on h and W_down, and a lane waits (bounded) for the values of h
// it needs -- the two groups its columns take -- not for the whole grid (exchange.cuh).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "exchange.cuh"
#include "tc_common.cuh"
#include "trace.cuh"

namespace algproj {
ALG_TRACE_DEFINE(row_decode)
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kPieceCols = 16;   // columns of a piece where the group width allows (32 and 64 measured the same or slower)

// 16-byte weight loads a lane keeps in flight: RC rows of two segments, for the gate and the up columns.  RC (2, 4, 8 or,
// projections only, 16) is what the shape needs: code for more rows is code the one pass has to fetch around, and up to
// four rows leave registers for two CTAs per SM, so that the next launch's loads go out while this one computes.  Gated
// 2048 -> 6144 -> 2048 at q = 32, one row, per layer of a graph of layers: 8.3 us with 8 rows for every shape, 6.6 with
// RC = 2, 6.0 with the sums halved across the lanes and one lane per column at the end.  Shapes that need 8 rows are
// better off with all of them in flight than with two passes of 4 (4096 -> 12288: 13.2 against 13.8 us).
template <bool GATED, int RC>
constexpr int kLoads = RC * (GATED ? 4 : 2);

// One matrix-vector phase as the kernel sees it.
struct Phase {
  const __nv_bfloat16 *W;   // weight bank, `ldw` elements per row
  int64_t ldw;
  int s;                    // rows of one input group
  int group_w;              // columns of one output group
  float inv_group_w;
  int n_cols;               // output columns (GATED: the up columns sit n_cols further in the bank)
  int pc;                   // columns of a piece: 8 or 16
  int ks;                   // warps that share the rows of a piece: 1, 2, 4 or 8
};

// Where a lane stands in a piece: `sub` = which 8 columns, `lr` = which share of the rows.
struct Lane {
  int piece, part, sub, lr, rl, col, j;
  bool on;
};
// (ks and pc / 8 are powers of two: shifts, and the group of a column by a reciprocal -- the step is bound by latency,
// and a handful of integer divisions on the way to the first load are a few hundred cycles of it)
__device__ __forceinline__ Lane lane_of(const Phase &p, int unit) {
  Lane l;
  const int lane = threadIdx.x & 31, po = p.pc >> 3, po_sh = __ffs(po) - 1, ks_sh = __ffs(p.ks) - 1;
  l.piece = unit >> ks_sh, l.part = unit & (p.ks - 1);
  l.sub = lane & (po - 1), l.lr = lane >> po_sh, l.rl = 32 >> po_sh;
  l.col = l.piece * p.pc + 8 * l.sub;
  l.on = l.col < p.n_cols;
  int j = (int)(((float)l.col + 0.5f) * p.inv_group_w);   // exact below 2^22 columns up to one step, corrected here
  if (j * p.group_w > l.col) --j;
  if ((j + 1) * p.group_w <= l.col) ++j;
  l.j = l.on ? j : 0;
  return l;
}

// Unit (piece x share of its rows) of this warp in round rd.  The warps that share a piece sit in one CTA; the pieces
// go round-robin over the CTAs, so that every SM carries the same number of busy warps (768 pieces on 148 SMs: five or
// six warps each, not eight on 96 of them; measured equal to the blocked order -- the step is bound by the chain of
// round trips, not by any one SM).
__device__ __forceinline__ int unit_of(int rd, int ks) {
  const int warp = threadIdx.x >> 5, ks_sh = __ffs(ks) - 1, slot = warp >> ks_sh, part = warp & (ks - 1);
  const int piece = (rd * (kWarps >> ks_sh) + slot) * gridDim.x + blockIdx.x;
  return piece * ks + part;
}

// Loads of one chunk: rows r0 .. of both segments (the diagonal block of group j, then -- unless the row's own type is
// j -- its panel block), for the gate and, GATED, the up columns.  RC rows per segment and chunk.
template <bool GATED, int RC>
__device__ __forceinline__ void load_chunk(uint4 (&w)[kLoads<GATED, RC>], const Phase &p, const Lane &l, int type, int c0) {
  const int step = p.ks * l.rl, first = l.part * l.rl + l.lr;
  const int nr = ((p.s + step - 1) >> (__ffs(step) - 1)) - c0;   // rows of this chunk some lane has (the same in every lane)
#pragma unroll
  for (int sg = 0; sg < 2; ++sg) {
    const int g = sg == 0 ? l.j : type;
    const bool seg_on = l.on && (sg == 0 || type != l.j);
    const __nv_bfloat16 *base = p.W + (int64_t)g * p.s * p.ldw + l.col;
#pragma unroll
    for (int u = 0; u < RC; ++u) {
      if (u >= nr) break;
      const int kk = first + (c0 + u) * step;
      const bool ok = seg_on && kk < p.s;
      const __nv_bfloat16 *src = base + (int64_t)kk * p.ldw;
      w[(sg * RC + u) * (GATED ? 2 : 1)] = ok ? __ldg((const uint4 *)src) : make_uint4(0, 0, 0, 0);
      if (GATED) w[(sg * RC + u) * 2 + 1] = ok ? __ldg((const uint4 *)(src + p.n_cols)) : make_uint4(0, 0, 0, 0);
    }
  }
}

// Asks L2 for the weights of this warp's first unit of a phase (a 16- or 8-column piece of a row is one sector).  Sent
// before the launch's dependency resolves, so that W_down, which is loaded when phase 1 is over, comes from L2 and not from
// HBM.  (A wrong type costs nothing but the hint.)
__device__ __forceinline__ void prefetch_unit(const Phase &p, int n_units, int type) {
  const int unit = unit_of(0, p.ks);
  const Lane l = lane_of(p, unit);
  if (unit >= n_units || !l.on || type < 0 || l.sub != 0) return;
  for (int sg = 0; sg < (type == l.j ? 1 : 2); ++sg) {
    const __nv_bfloat16 *base = p.W + (int64_t)(sg == 0 ? l.j : type) * p.s * p.ldw + l.col;
    for (int kk = l.part * l.rl + l.lr; kk < p.s; kk += p.ks * l.rl)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(base + (int64_t)kk * p.ldw));
  }
}

// Bound of the waits for hidden values.
struct Wait {
  long long t0, limit;
  volatile int *abort_flag;   // shared memory: one wait that ran out ends the others
  int *status;
};

// acc[0..8) (gate or plain) and acc[8..16) (up) += x[kk] * w[kk][...] for one chunk.  x is read from global memory
// (HIDDEN: from the exchange buffer, where it may yet have to arrive).
template <bool GATED, bool HIDDEN, int RC>
__device__ __forceinline__ void fma_chunk(const uint4 (&w)[kLoads<GATED, RC>], const Phase &p, const Lane &l, int type, int c0,
                                          const __nv_bfloat16 *x, uint64_t (&acc)[GATED ? 8 : 4], const Wait &wait) {
  const int step = p.ks * l.rl, first = l.part * l.rl + l.lr;
  const int nr = ((p.s + step - 1) >> (__ffs(step) - 1)) - c0;   // rows of this chunk some lane has (the same in every lane)
  float xv[2 * RC];
#pragma unroll
  for (int sg = 0; sg < 2; ++sg) {
    const int g = sg == 0 ? l.j : type;
    const bool seg_on = l.on && (sg == 0 || type != l.j);
#pragma unroll
    for (int u = 0; u < RC; ++u) {
      if (u >= nr) break;
      const int kk = first + (c0 + u) * step;
      unsigned short raw = 0;
      if (seg_on && kk < p.s) {
        const unsigned short *src = (const unsigned short *)(x + (int64_t)g * p.s + kk);
        raw = HIDDEN ? exch_load(src) : __ldg(src);
      }
      xv[sg * RC + u] = __uint_as_float((uint32_t)raw << 16);
    }
  }
  if (HIDDEN) {   // what had not arrived is loaded again
    uint32_t spins = 0;
    bool missing = true;
    while (missing) {
      missing = false;
#pragma unroll
      for (int sg = 0; sg < 2; ++sg) {
        const int g = sg == 0 ? l.j : type;
#pragma unroll
        for (int u = 0; u < RC; ++u) {
          if (u >= nr) break;
          if (__float_as_uint(xv[sg * RC + u]) == 0xFFFF0000u) {
            missing = true;
            xv[sg * RC + u] = __uint_as_float((uint32_t)exch_load((const unsigned short *)(x + (int64_t)g * p.s + first + (c0 + u) * step)) << 16);
          }
        }
      }
      if (missing && (++spins & 63u) == 0) {
        if (*wait.abort_flag) break;
        if (clock64() - wait.t0 > wait.limit) {
          *wait.abort_flag = 1;
          atomicExch(wait.status, (int)ALG_ERR_DEVICE_TIMEOUT);
        }
      }
    }
  }
#pragma unroll
  for (int e = 0; e < 2 * RC; ++e) {
    if ((e % RC) >= nr) continue;
    const uint64_t xx = tc::pack2(xv[e], xv[e]);
#pragma unroll
    for (int h = 0; h < (GATED ? 2 : 1); ++h) {
      const uint4 &v = w[e * (GATED ? 2 : 1) + h];
      const uint32_t p[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int c = 0; c < 4; ++c)
        acc[h * 4 + c] = tc::fma2(xx, tc::pack2(__uint_as_float(p[c] << 16), __uint_as_float(p[c] & 0xFFFF0000u)), acc[h * 4 + c]);
    }
  }
}

// The sums of a piece: NV values of every lane over the lanes that share its columns, halved step by step (a lane ends
// with one value), then over the warps that share the piece, through shared memory.  One lane per column calls emit(column
// of the piece, gate or plain value, up value).  `meet` is the barrier of those warps.
template <bool GATED, typename Meet, typename Emit>
__device__ __forceinline__ void finish_piece(const uint64_t (&acc)[GATED ? 8 : 4], const Phase &p, const Lane &l, float *partial, Meet meet,
                                             Emit emit) {
  constexpr int NV = GATED ? 16 : 8;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, po = p.pc >> 3;
  float v[NV];
#pragma unroll
  for (int i = 0; i < NV / 2; ++i) v[2 * i] = __uint_as_float((uint32_t)acc[i]), v[2 * i + 1] = __uint_as_float((uint32_t)(acc[i] >> 32));
  int n = NV;
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) {
    if (n > 1) {   // (16 or 8 lanes away at least: never a lane with other columns)
      n >>= 1;
      const bool hi = lane & d;
#pragma unroll
      for (int i = 0; i < NV / 2; ++i)
        if (i < n) {
          const float send = hi ? v[i] : v[i + n], keep = hi ? v[i + n] : v[i];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, d);
        }
    } else if (d >= po) {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], d);
    }
  }
  // lane: value lane / (32 / NV) of the columns l.sub
  partial[(warp * 2 + l.sub) * 16 + lane / (32 / NV)] = v[0];
  if (p.ks > 1) meet(); else __syncwarp();
  if (l.part == 0 && lane < p.pc) {
    const float *src = partial + (warp * 2 + (lane >> 3)) * 16 + (lane & 7);
    float g = 0.f, u = 0.f;
    for (int o = 0; o < p.ks; ++o) {
      g += src[o * 32];
      if (GATED) u += src[o * 32 + 8];
    }
    emit(lane, g, u);
  }
  if (p.ks > 1) meet(); else __syncwarp();
}

// One phase for the units of this warp.  `w` holds the first chunk of the first unit when have_first.  Results:
// emit(column, gate or plain value, up value), one lane per column.
template <bool GATED, bool HIDDEN, int RC, typename Emit>
__device__ __forceinline__ void run_phase(const Phase &p, int type, const __nv_bfloat16 *x, uint4 (&w)[kLoads<GATED, RC>], bool have_first,
                                          int n_units, float *partial, const Wait &wait, Emit emit) {
  const int total_warps = gridDim.x * kWarps;
  const int rounds = (n_units + total_warps - 1) / total_warps;
  for (int rd = 0; rd < rounds; ++rd) {
    const int unit = unit_of(rd, p.ks);
    Lane l = lane_of(p, unit);
    if (unit >= n_units) l.on = false;
    uint64_t acc[GATED ? 8 : 4] = {};
    const int rows_per_lane = (p.s + p.ks * l.rl - 1) >> (__ffs(p.ks * l.rl) - 1);
    for (int c0 = 0; c0 < rows_per_lane; c0 += RC) {
      if (!(have_first && rd == 0 && c0 == 0)) load_chunk<GATED, RC>(w, p, l, type, c0);
      fma_chunk<GATED, HIDDEN, RC>(w, p, l, type, c0, x, acc, wait);
    }
    const int col0 = l.piece * p.pc;
    finish_piece<GATED>(acc, p, l, partial, [] { __syncthreads(); }, [&](int c, float g, float u) {
      if (unit < n_units && col0 + c < p.n_cols) emit(col0 + c, g, u);
    });
  }
}

// (row types are read twice, early and after the wait for the kernel that may write them: from L2, never a stale L1 line)
__device__ __forceinline__ int read_type(const RowDecodeArgs &a) {
  const int t = a.types ? __ldcg(a.types) : 0;
  return t < 0 || t >= a.q ? -1 : t;
}

__device__ __forceinline__ float activate(float z, int act) {
  if (act == ALG_ACT_GELU_ERF) return 0.5f * z * (1.f + erff(z * 0.70710678118654752f));
  if (act == ALG_ACT_GELU_TANH) return 0.5f * z * (1.f + tanhf(0.79788456080286536f * (z + 0.044715f * z * z * z)));
  return z;
}

// one result: + bias, activation
__device__ __forceinline__ float finish1(float z, int col, const void *bias, int act) {
  if (bias) z += __bfloat162float(__ldg((const __nv_bfloat16 *)bias + col));
  return act == ALG_ACT_NONE ? z : activate(z, act);
}
__device__ __forceinline__ void store1(void *out, int64_t at, bool out_bf16, float z) {
  if (out_bf16) ((__nv_bfloat16 *)out)[at] = __float2bfloat16_rn(z);
  else ((float *)out)[at] = z;
}
__device__ __forceinline__ float gated1(float g, float u) { return g / (1.f + __expf(-g)) * u; }   // silu(g) * u

// Y lies over X (an FFN in place): a CTA says when it has used its X, and stores Y once every CTA of the grid has.  The
// hidden values a CTA waits for tell it nothing about the CTAs whose values it does not need, and those may start late.
__device__ __forceinline__ void used_x(const RowDecodeArgs &a, const ExchTurn &turn) {
  __syncthreads();
  if (threadIdx.x == 0) exch_hint(a.exch, turn);
}
__device__ __forceinline__ void all_used_x(const RowDecodeArgs &a, const ExchTurn &turn, const Wait &wait) {
  if (threadIdx.x == 0) {
    while (!exch_hinted(a.exch, turn, gridDim.x))
      if (clock64() - wait.t0 > wait.limit) {
        *wait.abort_flag = 1;
        atomicExch(wait.status, (int)ALG_ERR_DEVICE_TIMEOUT);
        break;
      }
  }
  __syncthreads();
}

// MODE 0: gated FFN, 1: FFN, 2: projection (W1 only)
template <int MODE, int RC>
__global__ void __launch_bounds__(kThreads, RC <= 4 ? 2 : 1) row_decode_kernel(const RowDecodeArgs a) {
  constexpr bool GATED = MODE == 0, FFN = MODE != 2;
  __shared__ float partial[kWarps * 2 * 16];   // a piece has at most 2 x 8 columns
  __shared__ int s_abort, s_early;
  ALG_TRACE_VARS;
  if (threadIdx.x == 0) ALG_TRACE(0, 1);
  // phase 1 maps the D (projection: K) inputs to F (N) columns of W1; phase 2 maps F back to D through W2
  Phase p1, p2;
  p1.W = (const __nv_bfloat16 *)a.W1, p1.ldw = a.ldw1, p1.s = a.gs, p1.group_w = a.gr, p1.inv_group_w = a.inv_gr, p1.n_cols = a.F;
  p1.pc = a.pc1, p1.ks = a.ks1;
  p2.W = (const __nv_bfloat16 *)a.W2, p2.ldw = a.ldw2, p2.s = a.gr, p2.group_w = a.gs, p2.inv_group_w = a.inv_gs, p2.n_cols = a.D;
  p2.pc = a.pc2, p2.ks = a.ks2;
  const __nv_bfloat16 *X = (const __nv_bfloat16 *)a.X;
  __nv_bfloat16 *H = nullptr;   // hidden rows in the exchange buffer
  const int warp = threadIdx.x >> 5;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // ---- before the dependency resolves: the row type as it stands now and the first W1 loads it asks for (the type
  // is read again after the wait).  One thread reads it for the CTA: the previous kernel may be writing it, and warps
  // that share a piece have to agree on what they compute and on the barriers they meet at ----
  if (threadIdx.x == 0) s_abort = 0, s_early = read_type(a);
  __syncthreads();
  const int t_early = s_early;
  uint4 w[kLoads<GATED, RC>];
  {
    const int unit = unit_of(0, p1.ks);
    Lane l = lane_of(p1, unit);
    if (unit >= a.units1 || t_early < 0) l.on = false;
    load_chunk<GATED, RC>(w, p1, l, max(t_early, 0), 0);
  }
  if (FFN && a.warm2) prefetch_unit(p2, a.units2, t_early);
  if (threadIdx.x == 0) ALG_TRACE(0, 2);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (threadIdx.x == 0) ALG_TRACE(0, 3);
  const int type = read_type(a);   // (in flight while phase 1 runs on the early value)
  const Wait wait = {clock64(), a.wait_limit, &s_abort, a.status};
  ExchTurn turn = {0u, 0};
  if (FFN) {
    turn = exch_turn(a.exch);
    H = (__nv_bfloat16 *)(a.exch + kExchHeader + turn.parity * (unsigned)a.exch_bytes);
  }
  const bool keep = FFN && a.test_withhold && blockIdx.x == 0;

  // ---- phase 1 on the type read early, again if the type has changed since.  Gated: h = silu(x * W_gate) .*
  // (x * W_up); FFN: h = act(x * W_up + b_up); projection: y = act(x * W + b) ----
  for (int pass = 0; pass < 2; ++pass) {
    const int t = pass == 0 ? t_early : type;
    if (pass == 1 && type == t_early) break;
    if (t < 0) continue;
    run_phase<GATED, false, RC>(p1, t, X, w, pass == 0, a.units1, partial, wait, [&](int col, float g, float u) {
      if (t != type || keep) return;   // (hidden values are taken as soon as they are there: only the right ones are stored)
      if (GATED) exch_store1(H + col, gated1(g, u));
      else if (FFN) exch_store1(H + col, finish1(g, col, a.b1, a.act));
      else store1(a.Y, col, a.y_bf16 != 0, finish1(g, col, a.b1, a.act));
    });
  }
  if (type < 0 && threadIdx.x == 0 && blockIdx.x == 0) atomicExch(a.status, (int)ALG_ERR_BAD_TYPE);   // y = 0
  if (threadIdx.x == 0) ALG_TRACE(0, 6);
  if (!FFN) {
    if (type < 0) {   // a row type outside [0, q): the row of Y is zero
      for (int c = blockIdx.x * kThreads + threadIdx.x; c < a.F; c += gridDim.x * kThreads) {
        if (a.y_bf16) ((__nv_bfloat16 *)a.Y)[c] = __float2bfloat16_rn(0.f);
        else ((float *)a.Y)[c] = 0.f;
      }
    }
    return;
  }

  if (a.in_place) used_x(a, turn);
  // ---- the first W_down loads go out before the hidden values are waited for ----
  uint4 w2[kLoads<false, RC>];
  {
    const int unit = unit_of(0, p2.ks);
    Lane l = lane_of(p2, unit);
    if (unit >= a.units2 || type < 0) l.on = false;
    load_chunk<false, RC>(w2, p2, l, max(type, 0), 0);
  }

  exch_clear(a.exch, a.exch_bytes, turn, a.F * 2, 1);
  if (threadIdx.x == 0) ALG_TRACE(0, 9);
  if (a.in_place) all_used_x(a, turn, wait);

  // ---- phase 2: y = h * W_down (+ b_down) ----
  if (type >= 0) {
    run_phase<false, true, RC>(p2, type, H, w2, true, a.units2, partial, wait,
                                [&](int col, float z, float) { store1(a.Y, col, a.y_bf16 != 0, finish1(z, col, a.b2, ALG_ACT_NONE)); });
  } else {   // a row type outside [0, q): the row of Y is zero
    for (int c = blockIdx.x * kThreads + threadIdx.x; c < a.D; c += gridDim.x * kThreads) {
      if (a.y_bf16) ((__nv_bfloat16 *)a.Y)[c] = __float2bfloat16_rn(0.f);
      else ((float *)a.Y)[c] = 0.f;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    ALG_TRACE(0, 12);
    exch_leave(a.exch);
  }
}

__device__ __forceinline__ int read_row_type(const RowDecodeArgs &a, int m) {
  const int t = a.types ? __ldcg(a.types + m) : m % a.q;
  return t < 0 || t >= a.q ? -1 : t;
}

// The same phase for several rows: unit = (row, piece, share of the piece's weight rows), rows outermost.  `w` holds
// the first chunk of the first unit when have_first, fetched for row type t_first; the other units read their row's
// type themselves.  Results: emit(row, column, gate or plain value, up value), one lane per column.
// Barrier of the warps that share a piece (2, 4 or 8 of them: at most four groups per CTA).  The ids are literals so
// that the kernel reserves five hardware barriers, not all sixteen -- with sixteen a second CTA (the next launch's,
// which starts early to request its weights) could not become resident beside this one.
__device__ __forceinline__ void group_barrier(int id, int threads) {
  switch (id) {
    case 1: asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory"); break;
    case 2: asm volatile("bar.sync 2, %0;" ::"r"(threads) : "memory"); break;
    case 3: asm volatile("bar.sync 3, %0;" ::"r"(threads) : "memory"); break;
    default: asm volatile("bar.sync 4, %0;" ::"r"(threads) : "memory"); break;
  }
}

// A row whose type lies outside [0, q) reads nothing; with LAST (the phase that writes Y) its pieces are stored as zeros
// and the status word says so.
template <bool GATED, bool HIDDEN, bool LAST, int RC, typename Emit>
__device__ __forceinline__ void run_rows_phase(const RowDecodeArgs &a, const Phase &p, const __nv_bfloat16 *x, int64_t ldx,
                                          uint4 (&w)[kLoads<GATED, RC>], bool have_first, int t_first, int n_units, float *partial, const Wait &wait, Emit emit) {
  const int warp = threadIdx.x >> 5;
  const int total_warps = gridDim.x * kWarps;
  const int rounds = (n_units + total_warps - 1) / total_warps;
  const int per_row = a.M == 1 ? n_units : n_units / a.M;   // (one row: no division on the way to the first load)
  for (int rd = 0; rd < rounds; ++rd) {
    const int unit = unit_of(rd, p.ks);
    const int m = a.M == 1 ? 0 : min(unit / per_row, a.M - 1);
    const int real = read_row_type(a, m);   // (on its way while the first attempt below runs on the type read early)
    int type = have_first && rd == 0 ? t_first : real;
    const __nv_bfloat16 *xm = x + (int64_t)m * ldx;
    // the first unit runs on the type read before the launch's dependency resolved; if the type has changed since, the
    // warps of the piece (they share the row) do it again -- they meet at a barrier of their own, not the CTA's
    for (int attempt = 0; attempt < 2; ++attempt) {
      Lane l = lane_of(p, unit - m * per_row);
      if (unit >= n_units || type < 0) l.on = false;
      uint64_t acc[GATED ? 8 : 4] = {};
      const int rows_per_lane = (p.s + p.ks * l.rl - 1) >> (__ffs(p.ks * l.rl) - 1);
      for (int c0 = 0; c0 < rows_per_lane; c0 += RC) {
        if (!(have_first && rd == 0 && attempt == 0 && c0 == 0)) load_chunk<GATED, RC>(w, p, l, max(type, 0), c0);
        fma_chunk<GATED, HIDDEN, RC>(w, p, l, max(type, 0), c0, xm, acc, wait);
      }
      const int col0 = l.piece * p.pc;
      const bool again = attempt == 0 && type != real;
      finish_piece<GATED>(acc, p, l, partial, [&] { group_barrier(1 + warp / p.ks, 32 * p.ks); }, [&](int c, float g, float u) {
        if (again || unit >= n_units || col0 + c >= p.n_cols) return;
        if (type >= 0) {
          emit(m, col0 + c, g, u);
        } else if (LAST) {
          store1(a.Y, (int64_t)m * a.ldy + col0 + c, a.y_bf16 != 0, 0.f);
          if (c == 0) atomicExch(a.status, (int)ALG_ERR_BAD_TYPE);
        }
      });
      if (!again) break;
      type = real;
    }
  }
}

// Several rows (2 .. kRowDecodeMaxM): the row is the outermost dimension of the units; every warp reads the type of the
// rows it works on.  (A kernel of its own: the index arithmetic of the general form costs the one-row step 0.4-1 us.)
// MODE 0: gated FFN, 1: FFN, 2: projection (W1 only)
template <int MODE, int RC>
__global__ void __launch_bounds__(kThreads, RC <= 4 ? 2 : 1) rows_decode_kernel(const RowDecodeArgs a) {
  constexpr bool GATED = MODE == 0, FFN = MODE != 2;
  __shared__ float partial[kWarps * 2 * 16];   // a piece has at most 2 x 8 columns
  __shared__ int s_abort, s_early[kRowDecodeMaxM];
  ALG_TRACE_VARS;
  if (threadIdx.x == 0) ALG_TRACE(0, 1);
  // phase 1 maps the D (projection: K) inputs to F (N) columns of W1; phase 2 maps F back to D through W2
  Phase p1, p2;
  p1.W = (const __nv_bfloat16 *)a.W1, p1.ldw = a.ldw1, p1.s = a.gs, p1.group_w = a.gr, p1.inv_group_w = a.inv_gr, p1.n_cols = a.F;
  p1.pc = a.pc1, p1.ks = a.ks1;
  p2.W = (const __nv_bfloat16 *)a.W2, p2.ldw = a.ldw2, p2.s = a.gr, p2.group_w = a.gs, p2.inv_group_w = a.inv_gs, p2.n_cols = a.D;
  p2.pc = a.pc2, p2.ks = a.ks2;
  const __nv_bfloat16 *X = (const __nv_bfloat16 *)a.X;
  __nv_bfloat16 *H = nullptr;   // hidden rows in the exchange buffer
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (threadIdx.x == 0) s_abort = 0;

  // ---- before the dependency resolves: the type of this warp's first row as it stands now and the first W1 loads it
  // asks for (the type is read again after the wait).  A thread per row reads it for the CTA, as above ----
  if ((int)threadIdx.x < a.M) s_early[threadIdx.x] = read_row_type(a, threadIdx.x);
  __syncthreads();
  const int per_row1 = a.M == 1 ? a.units1 : a.units1 / a.M;
  const int unit1 = unit_of(0, p1.ks), m1 = a.M == 1 ? 0 : min(unit1 / per_row1, a.M - 1);
  const int t_early = s_early[m1];
  uint4 w[kLoads<GATED, RC>];
  {
    Lane l = lane_of(p1, unit1 - m1 * per_row1);
    if (unit1 >= a.units1 || t_early < 0) l.on = false;
    load_chunk<GATED, RC>(w, p1, l, max(t_early, 0), 0);
  }
  if (threadIdx.x == 0) ALG_TRACE(0, 2);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (threadIdx.x == 0) ALG_TRACE(0, 3);
  const Wait wait = {clock64(), a.wait_limit, &s_abort, a.status};
  ExchTurn turn = {0u, 0};
  if (FFN) {
    turn = exch_turn(a.exch);
    H = (__nv_bfloat16 *)(a.exch + kExchHeader + turn.parity * (unsigned)a.exch_bytes);
  }
  const bool keep = FFN && a.test_withhold && blockIdx.x == 0;

  // ---- phase 1 (its first unit on the type read early).  Gated: h = silu(x * W_gate) .* (x * W_up); FFN:
  // h = act(x * W_up + b_up); projection: y = act(x * W + b) ----
  {
    run_rows_phase<GATED, false, !FFN, RC>(a, p1, X, a.ldx, w, true, t_early, a.units1, partial, wait, [&](int m, int col, float g, float u) {
      if (keep) return;
      if (GATED) exch_store1(H + (int64_t)m * a.F + col, gated1(g, u));
      else if (FFN) exch_store1(H + (int64_t)m * a.F + col, finish1(g, col, a.b1, a.act));
      else store1(a.Y, (int64_t)m * a.ldy + col, a.y_bf16 != 0, finish1(g, col, a.b1, a.act));
    });
  }
  if (threadIdx.x == 0) ALG_TRACE(0, 6);

  if (FFN) {
    // the phases share the barriers of the pieces' warps: where those are groups of different sizes, no warp may come to a
    // barrier of phase 2 while others still meet at the one of that number in phase 1
    if (p1.ks != p2.ks && p1.ks > 1 && p2.ks > 1) __syncthreads();
    if (a.in_place) used_x(a, turn);
    // ---- the first W_down loads go out before the hidden values are waited for ----
    uint4 w2[kLoads<false, RC>];
    const int per_row2 = a.M == 1 ? a.units2 : a.units2 / a.M;
    const int unit2 = unit_of(0, p2.ks), m2 = a.M == 1 ? 0 : min(unit2 / per_row2, a.M - 1);
    const int type2 = read_row_type(a, m2);
    {
      Lane l = lane_of(p2, unit2 - m2 * per_row2);
      if (unit2 >= a.units2 || type2 < 0) l.on = false;
      load_chunk<false, RC>(w2, p2, l, max(type2, 0), 0);
    }

    exch_clear(a.exch, a.exch_bytes, turn, a.F * 2, a.M);
    if (threadIdx.x == 0) ALG_TRACE(0, 9);
    if (a.in_place) all_used_x(a, turn, wait);

    // ---- phase 2: y = h * W_down (+ b_down) ----
    run_rows_phase<false, true, true, RC>(a, p2, H, a.F, w2, true, type2, a.units2, partial, wait, [&](int m, int col, float z, float) {
      store1(a.Y, (int64_t)m * a.ldy + col, a.y_bf16 != 0, finish1(z, col, a.b2, ALG_ACT_NONE));
    });
    __syncthreads();
    if (threadIdx.x == 0) {
      ALG_TRACE(0, 12);
      exch_leave(a.exch);
    }
  }
}

// warps per piece: as many (a power of two, at most the warps of a CTA) as the grid has warps for
int pick_ks(int pieces, int grid) {
  int ks = 1;
  while (ks < kWarps && pieces * ks * 2 <= grid * kWarps) ks *= 2;
  return ks;
}

template <int MODE, int RC>
cudaError_t launch_rc(const RowDecodeArgs &a, int grid, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaError_t e = a.M == 1 ? cudaLaunchKernelEx(&cfg, row_decode_kernel<MODE, RC>, a) : cudaLaunchKernelEx(&cfg, rows_decode_kernel<MODE, RC>, a);
  count_launch(1);
  return e;
}

template <int MODE>
cudaError_t launch_mode(const RowDecodeArgs &a, int grid, cudaStream_t st) {
  // rows of a segment per lane in the wider of the two phases
  auto rows = [](int s, int pc, int ks) { return ceil_div(s, ks * (32 / (pc / 8))); };
  const int need = std::max(rows(a.gs, a.pc1, a.ks1), a.units2 ? rows(a.gr, a.pc2, a.ks2) : 0);
  if (need <= 2) return launch_rc<MODE, 2>(a, grid, st);
  if (need <= 4) return launch_rc<MODE, 4>(a, grid, st);
  if constexpr (MODE == 2) {
    if (need > 8) return launch_rc<MODE, 16>(a, grid, st);
  }
  return launch_rc<MODE, 8>(a, grid, st);
}

}  // namespace

bool row_decode_fits(int q, int D, int F) {
  if (q < 1 || D % q || F % q) return false;
  return (D / q) % 8 == 0 && (F / q) % 8 == 0;
}

cudaError_t launch_row_decode(const RowDecodeArgs &in, int num_sms, cudaStream_t st) {
  RowDecodeArgs a = in;
  if (a.mode < 0 || a.mode > 2 || a.M < 1 || a.M > kRowDecodeMaxM || !row_decode_fits(a.q, a.D, a.F)) return cudaErrorInvalidValue;
  const int s = a.D / a.q, r = a.F / a.q;
  a.gs = s, a.gr = r, a.inv_gs = 1.f / (float)s, a.inv_gr = 1.f / (float)r;
  auto piece = [](int group_w) { return group_w % kPieceCols == 0 ? kPieceCols : group_w % 16 == 0 ? 16 : 8; };
  a.pc1 = piece(r);
  a.pc2 = piece(s);
  const int pieces1 = a.F / a.pc1, pieces2 = a.mode == 2 ? 0 : a.D / a.pc2;
  a.ks1 = pick_ks(pieces1 * a.M, num_sms);
  a.ks2 = pieces2 ? pick_ks(pieces2 * a.M, num_sms) : 1;
  a.units1 = a.M * pieces1 * a.ks1;
  a.units2 = a.M * pieces2 * a.ks2;
  // every CTA of an FFN must be resident for the wait between the phases: one CTA per SM at most
  const int grid = std::min(num_sms, std::max(a.units1 / a.ks1, a.units2 / a.ks2));   // at most one piece group per CTA and slot
  // The hint pays where phase 2 has a piece for every CTA to itself (ks2 = all warps) up to 5 MB of W2 (a row's share, two
  // segments), elsewhere up to 2.5 MB: with more, the hints stand in the way of the previous layer's loads.  Without / with,
  // 10 layers in a graph, gated unless said, us.  ks2 = 8: 2048 -> 6144 at q = 32 (1.6 MB) 61.5 / 61.3, 12 layers 74.5 / 73.6; q = 16, plain:
  // 2048 -> 6144 (3.1) 80.6 / 79.2, 2048 -> 8192 (4.2) 88.2 / 86.4; 1024 -> 4096 at q = 8 (2.1) 80.7 / 78.7; 768 -> 3072 at q = 2 (4.7)
  // 157.6 / 153.6; 512 -> 2048 at q = 4 (1.0) 72.5 / 71.8, but 512 -> 1024 at q = 2 (1.0) 67.7 / 68.0; 2048 -> 8192 at q = 8 (8.4) 148.2 / 149.5.
  // ks2 < 8: 7168 -> 2048 at q = 32 (1.8) 65.8 / 64.3; 4096 -> 4096, plain (2.1) 63.3 / 62.0; 3072 -> 3072 at q = 16 (2.4) 81.4 / 80.5; 2560 ->
  // 9728 (3.1) 103.3 / 103.6; 5120 -> 5120 (3.3) even; 4096 -> 8192 (4.2) 95.1 / 95.5; 4096 -> 12288 (6.3) 133.4 / 135.2.  Not for next to
  // nothing: 2048 -> 768 (0.2) 47.1 / 47.3.  Several rows, 2560 -> 9728, three of them: 209.9 / 217.9.
  const double share = 4.0 * a.D * (double)a.F / a.q;
  a.warm2 = a.mode != 2 && share >= 0.5e6 && share <= (a.ks2 == kWarps ? 5e6 : 2.5e6);
  if (a.mode == 0) return launch_mode<0>(a, grid, st);
  if (a.mode == 1) return launch_mode<1>(a, grid, st);
  return launch_mode<2>(a, grid, st);
}

}  // namespace algproj
