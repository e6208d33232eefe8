// The one-launch decode FFN of ffn_decode.cu for 1 or 2 rows, on plain FMAs.  Included there: same decomposition (CTA c
// owns `su` columns of the hidden state and `sd` of the output, both weight slices in shared memory, requested before
// the launch's dependency resolves), same arguments.
//
// With this few rows the step is a chain of latencies: after the previous kernel, X and the row types (one round trip),
// the up products, the hidden values' way through L2, the down products.  The matrix path spends 0.8 + 1.1 us of it on
// loops of fragment loads for 24 + 96 matrix instructions per warp and another 1.5 us on staging activations behind
// barriers.  Here a thread owns row PAIRS 2 t, 2 t + 512, ... of both banks: it loads the activations of its rows
// straight into registers (all of them in flight at once; hidden values as they arrive, exchange.cuh), multiplies them
// with the 16-byte weight pieces of its rows out of shared memory, 8 columns at a time, and the partial sums are
// halved across the lanes (a lane keeps the columns it will own) and added over the 8 warps in order.  Two CTA barriers
// in all.  Row types, needed input groups and the row rule are registers of every thread.
// 768 -> 3072 -> 768, q = 2, per layer of a graph of layers: one row 7.5 (matrix path) -> 5.5 us, two rows 8.4 -> 7.1 us.
// The products of 4 rows take longer here than there (9.4 against 7.8 us a layer).  The 16 CTAs of 128 that a row's
// reader has yet to wait for when it starts (three quarters of the hints) save 0.1 us; with two rows waiting for all
// hints is 0.3 us better, loads that come too early cost more there.  Where Y lies over X a CTA with one row waits for all
// hints too: the values it needs (those of the row's type, for the group of its type) do not say that the CTAs of the
// other hidden groups have used X.
#pragma once

constexpr int kRowsMax = 2;          // rows of ffn_rows_kernel
constexpr int kRowsUp = 4, kRowsDn = 8;   // row pairs per thread and phase: D <= 2048, F <= 4096

struct RowsCtl {
  uint64_t bar_up, bar_dn, bar_miss[2];
  uint32_t spec_up, spec_dn;   // input groups requested for the row types as they stood early
  volatile int abort_flag;
};

// NV values per lane -> one (lane l: the sum over the lanes of value l / (32 / NV))
template <int NV>
__device__ __forceinline__ float halve(float (&v)[NV]) {
  const int lane = threadIdx.x & 31;
  int n = NV;
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) {
    if (n > 1) {
      n >>= 1;
      const bool hi = lane & d;
#pragma unroll
      for (int i = 0; i < NV / 2; ++i)
        if (i < n) {
          const float send = hi ? v[i] : v[i + n], keep = hi ? v[i + n] : v[i];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, d);
        }
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], d);
    }
  }
  return v[0];
}

// Byte offset of 16-byte piece o of row r of a slice of NT pieces per row.  The copies swizzle rows of 2 or 4 pieces
// (32- and 64-byte swizzle); together with the lane's choice of which of its two rows comes first the eight lanes of a
// shared-memory phase touch all 32 banks for every NT.
template <int NT>
__device__ __forceinline__ uint32_t piece_at(int r, int o) {
  const int x = NT == 2 ? (r >> 2) & 1 : NT == 4 ? (r >> 1) & 3 : 0;
  return (uint32_t)(r * (NT * 16) + ((o ^ x) << 4));
}
// x[it][m] = activations (2 t + 512 it, + 1) of row m, 0 where the row does not use them; w = this CTA's weight slice,
// [K][8 NT] bf16.  Partial sums of every warp to part[warp][NT][MR][8].
template <int NT, int MR, int U>
__device__ __forceinline__ void rows_product(const uint32_t (&x)[U][MR], uint32_t live, uint32_t w, float *part) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int NV = 8 * MR;
  const int first = (lane >> 2) & 1;   // which row of a pair this lane takes first
#pragma unroll(MR == 1 ? NT : 1)
  for (int o = 0; o < NT; ++o) {
    uint64_t acc[NV / 2];
#pragma unroll
    for (int i = 0; i < NV / 2; ++i) acc[i] = 0;
#pragma unroll
    for (int it = 0; it < U; ++it) {
      if ((live >> it) & 1u) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int second = h ^ first;
          uint32_t p[4];
          asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(p[0]), "=r"(p[1]), "=r"(p[2]), "=r"(p[3]) : "r"(w + piece_at<NT>(2 * tid + 512 * it + second, o)));
#pragma unroll
          for (int m = 0; m < MR; ++m) {
            const float xv = __uint_as_float(second ? x[it][m] & 0xFFFF0000u : x[it][m] << 16);
            const uint64_t xx = pack2(xv, xv);
#pragma unroll
            for (int e = 0; e < 4; ++e)
              acc[m * 4 + e] = fma2(xx, pack2(__uint_as_float(p[e] << 16), __uint_as_float(p[e] & 0xFFFF0000u)), acc[m * 4 + e]);
          }
        }
      }
    }
    float v[NV];
#pragma unroll
    for (int i = 0; i < NV / 2; ++i) v[2 * i] = __uint_as_float((uint32_t)acc[i]), v[2 * i + 1] = __uint_as_float((uint32_t)(acc[i] >> 32));
    const float s = halve<NV>(v);
    if ((lane & (32 / NV - 1)) == 0) part[(warp * NT + o) * NV + lane / (32 / NV)] = s;
  }
}
// value (row m, column c) of the CTA's strip: the warps' partial sums in order
template <int NT, int MR>
__device__ __forceinline__ float rows_sum(const float *part, int m, int c) {
  float z = 0.f;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) z += part[((w * NT + (c >> 3)) * MR + m) * 8 + (c & 7)];
  return z;
}

template <int NTU, int NTD, int MR>
__global__ void __launch_bounds__(kThreads, 2) ffn_rows_kernel(const __grid_constant__ CUtensorMap tm_up, const __grid_constant__ CUtensorMap tm_dn, const FfnDecodeArgs a) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 511) & ~(uintptr_t)511);
  const uint32_t wd = smem_u32(smem), wu = smem_u32(smem + a.off_wu);
  float *part_up = (float *)(smem + a.off_p), *part_dn = part_up + kWarps * NTU * 8 * MR;
  RowsCtl *ctl = (RowsCtl *)(smem + a.off_ctl);
  const int tid = threadIdx.x, c = blockIdx.x, q = a.q, M = a.M;
  const int c_dn = a.apart ? c - a.n_up : c;
  const bool has_up = c < a.n_up, has_dn = c_dn >= 0 && c_dn < a.n_dn;
  const int col_u = c * (8 * NTU), col_d = c_dn * (8 * NTD), D = a.D, F = a.F;
  const uint32_t bar_up = smem_u32(&ctl->bar_up), bar_dn = smem_u32(&ctl->bar_dn), bar_miss = smem_u32(&ctl->bar_miss[0]);
  if (tid == 0) {
    mbar_init(bar_up, 1);
    mbar_init(bar_dn, 1);
    mbar_init(bar_miss, 1);
    mbar_init(bar_miss + 8, 1);
    ctl->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  auto read_type = [&](int m) {
    const int t = m >= M ? -1 : a.types ? __ldcg(a.types + m) : m % q;
    return t < 0 || t >= q ? -1 : t;
  };
  // output groups of the two strips (a strip never straddles groups)
  int ju = 0, jd = 0;
  while (ju + 1 < q && a.so_f[ju + 1] <= col_u) ++ju;
  while (jd + 1 < q && a.so_d[jd + 1] <= col_d) ++jd;
  // kept input groups of every row type for the two strips, 8 bits a type
  uint64_t keeps_up = 0, keeps_dn = 0;
  for (int t = 0; t < q; ++t) keeps_up |= (uint64_t)a.keep[t * q + ju] << (8 * t), keeps_dn |= (uint64_t)a.keep[t * q + jd] << (8 * t);
  if (tid == 0) {
    // speculative: the previous kernel may still be writing the types, so one thread reads them for all -- read by every
    // thread for itself, a warp could miss the late copies another one had asked for
    uint32_t up = 0, dn = 0;
#pragma unroll
    for (int m = 0; m < MR; ++m) {
      const int t = read_type(m);
      if (t >= 0) up |= (uint32_t)(keeps_up >> (8 * t)) & 0xFFu, dn |= (uint32_t)(keeps_dn >> (8 * t)) & 0xFFu;
    }
    if (!has_up) up = 0;
    if (!has_dn) dn = 0;
    ctl->spec_up = up, ctl->spec_dn = dn;
    request_slice(&tm_up, bar_up, wu, a.so_d, up, q, col_u, NTU * 16, a.box_up, a.extra_expect_bytes);
    request_slice(&tm_dn, bar_dn, wd, a.so_f, dn, q, col_d, NTD * 16, a.box_dn, a.extra_expect_bytes);
  }
  __syncthreads();   // the barriers are ready, what was requested is known
  const uint32_t spec_up = ctl->spec_up, spec_dn = ctl->spec_dn;
  // input group of this thread's row pairs, 4 bits each (15: past the end)
  uint32_t gid_up = 0, gid_dn = 0;
#pragma unroll
  for (int it = 0; it < kRowsDn; ++it) {
    const int r = 2 * tid + 512 * it;
    if (it < kRowsUp) {
      int g = 0;
      while (g + 1 < q && a.so_d[g + 1] <= r) ++g;
      gid_up |= (uint32_t)(r < D ? g : 15) << (4 * it);
    }
    int g = 0;
    while (g + 1 < q && a.so_f[g + 1] <= r) ++g;
    gid_dn |= (uint32_t)(r < F ? g : 15) << (4 * it);
  }
  // ---- everything below may depend on the previous kernel of the stream ----
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const ExchTurn turn = exch_turn(a.exch);
  uint32_t xu[kRowsUp][MR];
#pragma unroll
  for (int it = 0; it < kRowsUp; ++it)
#pragma unroll
    for (int m = 0; m < MR; ++m) {
      const int r = 2 * tid + 512 * it;
      xu[it][m] = has_up && m < M && r < D ? __ldcg((const uint32_t *)((const __nv_bfloat16 *)a.X + (int64_t)m * D + r)) : 0u;
    }
  // the row types as the previous kernel left them: the ones that count
  uint32_t keep_up[MR], keep_dn[MR], need_up = 0, need_dn = 0, bad = 0;
#pragma unroll
  for (int m = 0; m < MR; ++m) {
    const int t = read_type(m);
    keep_up[m] = t >= 0 ? (uint32_t)(keeps_up >> (8 * t)) & 0xFFu : 0u, keep_dn[m] = t >= 0 ? (uint32_t)(keeps_dn >> (8 * t)) & 0xFFu : 0u;
    need_up |= keep_up[m], need_dn |= keep_dn[m];
    if (t < 0 && m < M) bad |= 1u << m;
  }
  if (bad && c == 0 && tid == 0) atomicExch(a.status, (int)ALG_ERR_BAD_TYPE);
  if (!has_up) need_up = 0;
  if (!has_dn) need_dn = 0;
  const uint32_t miss_up = need_up & ~spec_up, miss_dn = need_dn & ~spec_dn;
  const bool missed = (miss_up | miss_dn) != 0u;   // rare: blocks the final types need and the early request did not cover
  if (missed && tid == 0) {
    if (miss_up) request_slice(&tm_up, bar_miss, wu, a.so_d, miss_up, q, col_u, NTU * 16, a.box_up, 0);
    if (miss_dn) request_slice(&tm_dn, bar_miss + 8, wd, a.so_f, miss_dn, q, col_d, NTD * 16, a.box_dn, 0);
  }
  const long long t0 = clock64();
  // bounded wait; false once any wait of the CTA has run out
  auto give_up = [&](uint32_t &spins) {
    if ((++spins & 63u) != 0) return false;
    if (ctl->abort_flag) return true;
    if (clock64() - t0 <= a.wait_limit) return false;
    ctl->abort_flag = 1;
    atomicExch(a.status, (int)ALG_ERR_DEVICE_TIMEOUT);
    return true;
  };
  auto landed = [&](uint32_t bar) {
    uint32_t spins = 0;
    while (!mbar_try_wait(bar, 0))
      if (give_up(spins)) return;
  };
  __nv_bfloat16 *const hidden = (__nv_bfloat16 *)(a.exch + kExchHeader + turn.parity * (unsigned)a.exch_bytes);

  // ---------------- up phase: H[:, strip] = act(X *_q W_up + b_up) ----------------
  if (has_up) {
    uint32_t live = 0;
#pragma unroll
    for (int it = 0; it < kRowsUp; ++it) {
      const uint32_t g = (gid_up >> (4 * it)) & 15u;
      if ((need_up >> g) & 1u) live |= 1u << it;
#pragma unroll
      for (int m = 0; m < MR; ++m)
        if (!((keep_up[m] >> g) & 1u)) xu[it][m] = 0u;
    }
    landed(bar_up);
    if (miss_up) landed(bar_miss);
    rows_product<NTU, MR, kRowsUp>(xu, live, wu, part_up);
    __syncthreads();
    if (tid < M * (8 * NTU) && !ctl->abort_flag) {
      const int m = MR == 1 ? 0 : tid / (8 * NTU), cc = tid - m * (8 * NTU);
      float z = rows_sum<NTU, MR>(part_up, m, cc);
      if (a.b_up) z += __bfloat162float(((const __nv_bfloat16 *)a.b_up)[col_u + cc]);
      z = act_f(z, a.act);
      if ((bad >> m) & 1u) z = 0.f;
      exch_store1(hidden + (int64_t)m * F + col_u + cc, z);
    }
    if (tid == 0 && !ctl->abort_flag) exch_hint(a.exch, turn);
  } else {
    __syncthreads();   // every thread has asked for the turn
  }
  if (tid == 96) exch_leave(a.exch);   // (not the thread that waits for the hints)
  exch_clear(a.exch, a.exch_bytes, turn, F * 2, M);

  // ---------------- down phase: Y[:, strip] = H *_q W_down + b_down ----------------
  if (has_dn) {
    uint32_t spins = 0;
    if (tid == 0)
      while (!exch_hinted(a.exch, turn, MR == 1 && !a.in_place ? a.n_up - (a.n_up >> 2) : a.n_up))
        if (give_up(spins)) break;
    __syncthreads();
    uint32_t xd[kRowsDn][MR], live = 0;
#pragma unroll
    for (int it = 0; it < kRowsDn; ++it) {
      const uint32_t g = (gid_dn >> (4 * it)) & 15u;
      if ((need_dn >> g) & 1u) live |= 1u << it;
#pragma unroll
      for (int m = 0; m < MR; ++m)
        xd[it][m] = ((keep_dn[m] >> g) & 1u) ? exch_load2(hidden + (int64_t)m * F + 2 * tid + 512 * it) : 0u;
    }
    landed(bar_dn);
    if (miss_dn) landed(bar_miss + 8);
    for (bool missing = true; missing;) {   // what had not arrived is loaded again
      missing = false;
#pragma unroll
      for (int it = 0; it < kRowsDn; ++it)
#pragma unroll
        for (int m = 0; m < MR; ++m)
          if (!exch_ready2(xd[it][m])) {
            missing = true;
            xd[it][m] = exch_load2(hidden + (int64_t)m * F + 2 * tid + 512 * it);
          }
      if (missing && give_up(spins)) break;
    }
    rows_product<NTD, MR, kRowsDn>(xd, live, wd, part_dn);
    __syncthreads();
    if (tid < M * (8 * NTD) && !ctl->abort_flag) {
      const int m = MR == 1 ? 0 : tid / (8 * NTD), cc = tid - m * (8 * NTD), col = col_d + cc;
      float z = rows_sum<NTD, MR>(part_dn, m, cc);
      if (a.b_down) z += __bfloat162float(((const __nv_bfloat16 *)a.b_down)[col]);
      if ((bad >> m) & 1u) z = 0.f;   // out-of-range type: the row's output is defined to be zero
      if (a.y_bf16) ((__nv_bfloat16 *)a.Y)[(int64_t)m * D + col] = __float2bfloat16_rn(z);
      else ((float *)a.Y)[(int64_t)m * D + col] = z;
    }
  }
  if (ctl->abort_flag) {  // copies that are still in flight get time to land before shared memory is released
    while (clock64() - t0 < a.wait_limit + 2000000LL) {
    }
  }
}
