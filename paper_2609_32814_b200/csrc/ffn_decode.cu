// Decode step of the whole two-map FFN in ONE launch:  Y = act(X *_q W_up + b_up) *_q W_down + b_down
// for M <= 16 new rows (Section "One-Token Inference": one new row per sequence, typed by its
// absolute position; the regime is bound by weight traffic and by latency, not by arithmetic).
//
// Why one launch.  A 768 -> 3072 -> 768 layer streams 9.4 MB of weights, 1.4 us of HBM time, while a
// chain of dependent kernels pays several microseconds of serial latency per kernel.  Here every
// CTA requests its slice of BOTH banks the moment it starts -- before it waits for the previous
// kernel of the stream (programmatic dependent launch) -- and a CTA needs less than half of an SM's
// shared memory, so the CTAs of the next layer's launch sit beside the ones of the running layer
// and their weight stream overlaps its arithmetic.
//
// Decomposition.  No reduction across CTAs anywhere: CTA c owns `su` columns of the hidden state
// (all D input rows of W_up for them) and `sd` columns of the output (all F rows of W_down).
//   before the wait : row types read speculatively -> input groups some row needs (blocks W_kj that
//                     no present row type uses are never fetched) -> both slices requested by one
//                     thread with tiled copies (request_slice).
//   after the wait  : X staged in shared memory (all groups, unmasked) while the row types are read
//                     again; if they differ, the blocks that are missing are requested now.
//   up phase        : 8 warps split the K steps; mma.sync m16n8k16 (bf16 x bf16 -> fp32); the rule
//                     "row b uses block k only if k in B(t_b, j)" is applied by clearing the A
//                     fragment rows that do not use the block; the 8 partial tiles are summed in a
//                     fixed order through shared memory; bias, activation, bf16 -> H.
//   exchange        : H goes through the handle's exchange buffer: no fence, no barrier over the grid
//                     (exchange.cuh).
//   down phase      : H staged from L2 over the shared memory the W_up slice no longer needs; same
//                     MMA / reduction; bias; Y stored.
// Up to kRowsMax rows take a kernel on plain FMAs of the same decomposition (ffn_rows.cuh).
// Every wait (mbarriers the copies arrive on, values of H) is bounded by the handle's wait limit; on expiry the CTA
// raises ALG_ERR_DEVICE_TIMEOUT, skips its arithmetic, gives copies in flight time to land and
// returns.
#include <algorithm>

#include "exchange.cuh"
#include "tc_common.cuh"

namespace algproj {

using namespace tc;

ALG_TRACE_DEFINE(ffn_decode)

namespace {

constexpr int kThreads = 256, kWarps = 8;
// Two CTAs (this launch and the next layer's) per SM.  Where both weight slices of a CTA do not fit that, a CTA has one of
// them (`apart`), still in one launch (1024 -> 4096 -> 1024, q = 2, per layer of a graph, two launches / both strips in a CTA
// that fills an SM / apart: M = 1 18.8 / 8.1 / 6.8 us, M = 2 25.2 / 10.0 / 8.5, M = 8 16.2 / 11.3 / 11.7, M = 16 15.0 / 12.9 / 15.1).
// A CTA waits for values of others of its launch, so a launch ends only if those get a place.  The CTAs of a launch take
// their places in the order of their indexes: apart, the CTAs with up strips come first, wait for nobody but their own
// copies and the previous kernel, and leave; the others find every CTA they wait for placed before them, whatever else runs
// on the GPU.  With one CTA per SM for both strips (and all of its shared memory) two such launches of two streams could
// hold half of the GPU each and wait for the other's half until the limit.
constexpr int kSmemBudget = 112 * 1024, kSmemBudgetOne = 220 * 1024;

constexpr int kStagers = 128;   // warps 4-7 stage the activations

struct Ctl {
  uint64_t bar_up, bar_dn, bar_miss, bar_x;
  int so_d[kMaxQ + 1], so_f[kMaxQ + 1];   // input-group offsets of the up (D) / down (F) projection
  uint32_t need_up, need_dn;              // input groups some present row needs for this CTA's strips
  uint32_t miss_up, miss_dn;              // needed by the final types, not requested for the speculative ones
  uint32_t rows_up[kMaxQ], rows_dn[kMaxQ];  // bit m: row m uses input group k
  uint32_t bad_rows;
  volatile int abort_flag;
};

__device__ __forceinline__ void cp_async_16_zfill(uint32_t dst, const void *src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
// arrives on the barrier once every copy this thread has issued so far has landed
__device__ __forceinline__ void cp_async_arrive(uint32_t bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x2(uint32_t addr, uint32_t &r0, uint32_t &r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x2_trans(uint32_t addr, uint32_t &r0, uint32_t &r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float act_f(float z, int act) {
  if (act == ALG_ACT_GELU_ERF) return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f));
  if (act == ALG_ACT_GELU_TANH) {
    float u = 0.7978845608028654f * (z + 0.044715f * z * z * z);
    return 0.5f * z * (1.0f + tanhf(u));
  }
  return z;
}
// staged activations: [m_pad][kc] bf16, 16-byte pieces XOR-swizzled by the row (conflict-free ldmatrix)
__device__ __forceinline__ uint32_t x_off(int m, int chunk, int pitch_bytes) {
  return (uint32_t)(m * pitch_bytes + ((chunk ^ (m & 7)) << 4));
}

// One thread requests the rows of the input groups in `mask` of a weight slice (tiled copies; `so` = group offsets) and
// tells the barrier how many bytes will come.  (16-byte asynchronous copies by 128 threads cost the SM's load path
// about 5 k cycles per layer -- a slice is 16 to 64 bytes wide, a warp's copies touch 32 lines -- beside the CTA of
// the running layer: one row of 768 -> 3072 -> 768 at q = 2 took 7.0 us a layer with them and 5.7 with tiled copies.)
__device__ __forceinline__ void request_slice(const CUtensorMap *map, uint32_t bar, uint32_t dst, const int *so, uint32_t mask, int q,
                                              int col0, int pitch, int box, int extra) {
  uint32_t bytes = (uint32_t)extra;   // (test aid: bytes that never come)
  for (int k = 0; k < q; ++k)
    if ((mask >> k) & 1u) bytes += (uint32_t)((so[k + 1] - so[k]) * pitch);
  mbar_expect_tx(bar, bytes);
  for (int k = 0; k < q; ++k)
    if ((mask >> k) & 1u)
      for (int r = so[k]; r < so[k + 1]; r += box) tma_load_2d(dst + (uint32_t)(r * pitch), map, bar, col0, r);
}

// Warp 0: from the types of the M rows (lane m holds the type of row m, -1 = out of range) to the
// input groups this CTA's strips need and, per group, the rows that use it.
__device__ __forceinline__ void derive_masks(Ctl *ctl, const FfnDecodeArgs &a, int my_type, int M, int q, int ju, int jd,
                                             int lane) {
  const bool live = lane < M && my_type >= 0;
  const uint32_t *keep = a.small_q ? a.keep : a.tab_up->keep;   // by value in the kernel parameters when the table is small
  const uint32_t ku = (live && ju >= 0) ? keep[my_type * q + ju] : 0u;
  const uint32_t kd = (live && jd >= 0) ? keep[my_type * q + jd] : 0u;
  const uint32_t nu = __reduce_or_sync(0xffffffffu, ku), nd = __reduce_or_sync(0xffffffffu, kd);
  const uint32_t bad = __ballot_sync(0xffffffffu, lane < M && my_type < 0);
  for (int k = 0; k < q; ++k) {
    const uint32_t vu = __ballot_sync(0xffffffffu, (ku >> k) & 1u), vd = __ballot_sync(0xffffffffu, (kd >> k) & 1u);
    if (lane == 0) ctl->rows_up[k] = vu, ctl->rows_dn[k] = vd;
  }
  if (lane == 0) ctl->need_up = nu, ctl->need_dn = nd, ctl->bad_rows = bad;
}

// What one projection phase (up or down) of a CTA works on.
struct Phase {
  const __nv_bfloat16 *src;   // activations in global memory: X, or H written by the up phase of all CTAs
  int ld, K;                  // their leading dimension; the reduction length (D or F)
  int kc, pitch_bytes;        // staged K chunk and its row pitch
  uint32_t stage_base;        // shared memory of the staged chunk [m_pad][kc], 16-byte pieces XOR-swizzled by row
  uint32_t w_base;            // weight slice [K][cols] in shared memory
  int cols, col0;             // strip width, first column
  const int *so;              // input-group offsets
  const uint32_t *rows_k;     // per input group: rows that use it
  uint32_t need;              // input groups some row needs
  const void *bias;
  int act;
  void *out;                  // H (bf16) or Y
  int out_ld, out_bf16;
};
struct Shared {
  Ctl *ctl;
  float *p_sm;
  uint32_t bar_x;
  int M, m_pad, q;
  long long wait_limit;
  int *status;
};

// bounded wait on an mbarrier (all threads)
__device__ __forceinline__ bool wait_bar(const Shared &sh, uint32_t bar, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (sh.ctl->abort_flag) return false;
    if (clock64() - t0 > sh.wait_limit) {
      sh.ctl->abort_flag = 1;
      atomicExch(sh.status, (int)ALG_ERR_DEVICE_TIMEOUT);
      return false;
    }
  }
  return true;
}

// Warps 4-7 stage one K chunk of an activation matrix (rows >= M are zero) and arrive on bar_x.
__device__ __forceinline__ void stage_chunk(const Shared &sh, const Phase &ph, int kc0, int len) {
  const int tid = threadIdx.x;
  if (tid < kThreads - kStagers) return;
  const bool half_tile = sh.m_pad == 8;
  const int cpr = len >> 3;   // 16-byte pieces per row
  // 128 stagers over m_pad rows: 16 (or 8) neighbouring threads walk along one row
  const int t = tid - (kThreads - kStagers);
  const int tpr = half_tile ? kStagers / 8 : kStagers / 16;
  const int m = half_tile ? (t >> 4) : (t >> 3);
  const bool valid = m < sh.M;
  const __nv_bfloat16 *row = ph.src + (int64_t)(valid ? m : 0) * ph.ld + kc0;
  const uint32_t dst_row = ph.stage_base + (uint32_t)(m * ph.pitch_bytes);
  for (int ch = t & (tpr - 1); ch < cpr; ch += tpr)
    cp_async_16_zfill(dst_row + (uint32_t)((ch ^ (m & 7)) << 4), row + ch * 8, valid);
  cp_async_arrive(sh.bar_x);
}

// All threads: rows < M of one K chunk of the hidden state out of the exchange buffer, copied like any activation; what
// a copy found missing (exchange.cuh) is loaded again.  (The other staged rows keep whatever is there: the row rule
// clears their A fragments.)
template <int MP>
__device__ __forceinline__ void stage_hidden(const Shared &sh, const Phase &ph, int kc0, int len) {
  constexpr int TPR = kThreads / MP;   // threads that walk along a row
  const int cpr = len >> 3, m = threadIdx.x / TPR, ch0 = threadIdx.x % TPR;
  if (m >= sh.M) return;
  const __nv_bfloat16 *row = ph.src + (int64_t)m * ph.ld + kc0;
  for (int ch = ch0; ch < cpr; ch += TPR) cp_async_16_zfill(ph.stage_base + x_off(m, ch, ph.pitch_bytes), row + ch * 8, true);
  asm volatile("cp.async.wait_all;" ::: "memory");
  const long long t0 = clock64();
  uint32_t spins = 0;
  for (int ch = ch0; ch < cpr; ch += TPR) {
    const uint32_t dst = ph.stage_base + x_off(m, ch, ph.pitch_bytes);
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(dst) : "memory");
    if (exch_ready(v)) continue;
    while (!exch_ready(v)) {
      if ((++spins & 63u) == 0) {
        if (sh.ctl->abort_flag) return;
        if (clock64() - t0 > sh.wait_limit) {
          sh.ctl->abort_flag = 1;
          atomicExch(sh.status, (int)ALG_ERR_DEVICE_TIMEOUT);
          return;
        }
      }
      v = exch_load4(row + ch * 8);
    }
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
  }
}

// One projection phase of a CTA:  out[:, strip] = act(src *_q W[:, strip] + bias).
// The K range is staged chunk by chunk (one chunk for M <= 8 at the benchmark shape).  Warp w takes
// the 16-deep K steps w, w+8, ... of every needed input group, in batches of SETS steps: all
// fragments of a batch are loaded first, then its MMAs go to SETS independent accumulator sets, so
// neither the shared-memory latency nor the chain of dependent MMAs is paid per step.  The rule
// "row b uses block k only if k in B(t_b, j)" is applied by clearing the rows of the A fragment that
// do not use the block.  The 8 warps' partial tiles are then summed in warp order through shared
// memory (deterministic), bias and activation applied, rows < M stored.
// NT = 8-column tiles of the strip, MP = staged rows (8 or 16).  HIDDEN: the phase reads the hidden state (down); else
// it writes it (up).  Returns false when a wait ran out.
template <int NT, bool HIDDEN, int MP>
__device__ __forceinline__ bool run_phase_t(const Shared &sh, const Phase &ph, uint32_t &x_parity) {
  constexpr int SETS = NT <= 2 ? 4 : (NT <= 4 ? 2 : 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr bool HALF = MP == 8;
  const int g = lane >> 2, t4 = lane & 3;
  const int frag_row = (lane & 7) + ((lane >> 3) & 1) * 8;
  const int a_row = HALF ? (lane & 7) : frag_row;
  const int a_sel = HALF ? ((lane >> 3) & 1) : (lane >> 4);
  const uint32_t a_lane = ph.stage_base + (uint32_t)(a_row * ph.pitch_bytes);
  const int a_x = a_row & 7;
  const int w_pitch_bytes = ph.cols * 2;
  const uint32_t w_lane = ph.w_base + (uint32_t)(frag_row * w_pitch_bytes);
  float d[SETS][NT][4];
#pragma unroll
  for (int s = 0; s < SETS; ++s)
#pragma unroll
    for (int o = 0; o < NT; ++o) d[s][o][0] = d[s][o][1] = d[s][o][2] = d[s][o][3] = 0.f;
  bool ok = true;
  for (int kc0 = 0; kc0 < ph.K && ok; kc0 += ph.kc) {
    const int len = min(ph.kc, ph.K - kc0);
    if (HIDDEN) {
      if (kc0) __syncthreads();   // the previous chunk has been consumed
      stage_hidden<MP>(sh, ph, kc0, len);
      __syncthreads();
      ok = !sh.ctl->abort_flag;
    } else {
      if (kc0) {   // (the caller has requested the first one)
        __syncthreads();   // the previous chunk has been consumed
        stage_chunk(sh, ph, kc0, len);
      }
      ok = wait_bar(sh, sh.bar_x, x_parity);
      x_parity ^= 1u;
    }
    if (!ok) break;
    for (int k = 0; k < sh.q; ++k) {
      if (!((ph.need >> k) & 1u)) continue;
      const int b = max(ph.so[k], kc0), e = min(ph.so[k + 1], kc0 + len);
      if (b >= e) continue;
      const uint32_t rk = ph.rows_k[k];
      const uint32_t mlo = ((rk >> g) & 1u) ? 0xffffffffu : 0u, mhi = ((rk >> (g + 8)) & 1u) ? 0xffffffffu : 0u;
      for (int kk = b + 16 * warp; kk < e; kk += SETS * 16 * kWarps) {
        uint32_t af[SETS][4], bf[SETS][NT][2];
#pragma unroll
        for (int s = 0; s < SETS; ++s) {
          const int ks = kk + s * 16 * kWarps;
          if (ks < e) {
            const uint32_t a_addr = a_lane + (uint32_t)(((((ks - kc0) >> 3) + a_sel) ^ a_x) << 4);
            if (HALF) {
              ldmatrix_x2(a_addr, af[s][0], af[s][2]);
              af[s][1] = af[s][3] = 0u;
            } else {
              ldmatrix_x4(a_addr, af[s]);
            }
            const uint32_t wrow = w_lane + (uint32_t)(ks * w_pitch_bytes);
#pragma unroll
            for (int o = 0; o < NT; ++o) ldmatrix_x2_trans(wrow + (uint32_t)(o << 4), bf[s][o][0], bf[s][o][1]);
          }
        }
#pragma unroll
        for (int s = 0; s < SETS; ++s) {
          if (kk + s * 16 * kWarps < e) {
            af[s][0] &= mlo, af[s][2] &= mlo, af[s][1] &= mhi, af[s][3] &= mhi;
#pragma unroll
            for (int o = 0; o < NT; ++o) mma_bf16(d[s][o], af[s], bf[s][o][0], bf[s][o][1]);
          }
        }
      }
    }
  }
  __syncthreads();
  if (sh.ctl->abort_flag) return false;
  // ---- the 8 warps' partial tiles -> shared memory -> ordered sum, bias, activation, store ----
  const int cols = ph.cols;
#pragma unroll
  for (int o = 0; o < NT; ++o) {
    float v[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      v[x] = d[0][o][x];
#pragma unroll
      for (int s = 1; s < SETS; ++s) v[x] += d[s][o][x];
    }
    float *p = sh.p_sm + ((warp * sh.m_pad + g) * cols + o * 8 + t4 * 2);
    *(float2 *)p = make_float2(v[0], v[1]);
    if (!HALF) *(float2 *)(p + 8 * cols) = make_float2(v[2], v[3]);
  }
  __syncthreads();
  const int pairs = cols >> 1;
  const int m = tid >> 4;   // 16 rows x 16 threads that walk along the row's column pairs
  for (int pr = tid & 15; pr < pairs && m < sh.M; pr += 16) {
    const int cp = pr * 2;
    float z0 = 0.f, z1 = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const float2 v = *(const float2 *)(sh.p_sm + ((w * sh.m_pad + m) * cols + cp));
      z0 += v.x, z1 += v.y;
    }
    const int col = ph.col0 + cp;
    if (ph.bias) {
      z0 += __bfloat162float(((const __nv_bfloat16 *)ph.bias)[col]);
      z1 += __bfloat162float(((const __nv_bfloat16 *)ph.bias)[col + 1]);
    }
    z0 = act_f(z0, ph.act), z1 = act_f(z1, ph.act);
    if ((sh.ctl->bad_rows >> m) & 1u) z0 = z1 = 0.f;   // out-of-range type: the row's output is defined to be zero
    if (!HIDDEN) {
      __nv_bfloat162 v = __floats2bfloat162_rn(z0, z1);
      exch_store((__nv_bfloat16 *)ph.out + (int64_t)m * ph.out_ld + col, *(uint32_t *)&v);
    } else if (ph.out_bf16) {
      __nv_bfloat162 v = __floats2bfloat162_rn(z0, z1);
      *(uint32_t *)((__nv_bfloat16 *)ph.out + (int64_t)m * ph.out_ld + col) = *(uint32_t *)&v;
    } else {
      *(float2 *)((float *)ph.out + (int64_t)m * ph.out_ld + col) = make_float2(z0, z1);
    }
  }
  return true;
}
// NTU / NTD: 8-column tiles of the up / down strip (compile-time, so that every kernel gets the
// registers its own shape needs).
template <int NTU, int NTD, int MP>
__global__ void __launch_bounds__(kThreads, 2) ffn_decode_kernel(const __grid_constant__ CUtensorMap tm_up, const __grid_constant__ CUtensorMap tm_dn, const FfnDecodeArgs a) {
  // the next launch of the stream may start now: it only requests its own weights before it waits
  // (triggering later -- after the up phase or after the exchange -- was measured no faster)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
  uint8_t *wd_sm = smem;                        // W_down slice  [F][sd]
  uint8_t *wu_sm = smem + a.off_wu;             // W_up slice    [D][su]; later part of the H stage
  uint8_t *st_sm = smem + a.off_stage;          // X stage; the H stage (off_hidden) starts at wu_sm and runs through here
  Ctl *ctl = (Ctl *)(smem + a.off_ctl);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int c = blockIdx.x, q = a.q, M = a.M;
  const int c_dn = a.apart ? c - a.n_up : c;
  const bool has_up = c < a.n_up, has_dn = c_dn >= 0 && c_dn < a.n_dn;
  const int col_u = c * a.su, col_d = c_dn * a.sd;
  const int D = a.D, F = a.F;
  ALG_TRACE_VARS;
#define TR(tag) do { if (tid == 0) ALG_TRACE(0, tag); ALG_TRACE_SEQ(tag); } while (0)
  TR(1);

  // ---- tables, barriers ----
  if (a.small_q) {
    for (int e = tid; e <= q; e += kThreads) ctl->so_d[e] = a.so_d[e], ctl->so_f[e] = a.so_f[e];
  } else {
    for (int e = tid; e <= q; e += kThreads) ctl->so_d[e] = a.tab_up->so[e], ctl->so_f[e] = a.tab_dn->so[e];
  }
  const uint32_t bar_up = smem_u32(&ctl->bar_up), bar_dn = smem_u32(&ctl->bar_dn);
  const uint32_t bar_miss = smem_u32(&ctl->bar_miss), bar_x = smem_u32(&ctl->bar_x);
  if (tid == 0) {
    mbar_init(bar_up, 1);
    mbar_init(bar_dn, 1);
    mbar_init(bar_miss, 2);   // both slices
    mbar_init(bar_x, kStagers);
    ctl->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  int spec_type = -1;
  if (tid < M) {   // speculative: the previous kernel may still be writing the types
    spec_type = a.types ? __ldcg(a.types + tid) : (tid % q);
    if (spec_type < 0 || spec_type >= q) spec_type = -1;
  }
  __syncthreads();
  // output groups of the two strips (a strip never straddles groups: su | every f width, sd | every d width)
  int ju = -1, jd = -1;
  if (has_up) {
    ju = 0;
    while (ju + 1 < q && ctl->so_f[ju + 1] <= col_u) ++ju;   // hidden columns are the outputs of up = the inputs of down
  }
  if (has_dn) {
    jd = 0;
    while (jd + 1 < q && ctl->so_d[jd + 1] <= col_d) ++jd;
  }
  if (warp == 0) derive_masks(ctl, a, spec_type, M, q, ju, jd, lane);
  __syncthreads();
  const uint32_t spec_up = ctl->need_up, spec_dn = ctl->need_dn;

  // ---- both weight slices, requested before anything else is waited for ----
  if (tid == 0) {
    request_slice(&tm_up, bar_up, smem_u32(wu_sm), ctl->so_d, has_up ? spec_up : 0u, q, col_u, a.su * 2, a.box_up, a.extra_expect_bytes);
    request_slice(&tm_dn, bar_dn, smem_u32(wd_sm), ctl->so_f, has_dn ? spec_dn : 0u, q, col_d, a.sd * 2, a.box_dn, a.extra_expect_bytes);
  }
  TR(2);
  // ---- everything below may depend on the previous kernel of the stream ----
  asm volatile("griddepcontrol.wait;" ::: "memory");
  TR(3);

  const ExchTurn turn = exch_turn(a.exch);   // (on its way while the activations are staged)
  Shared sh;
  sh.ctl = ctl, sh.p_sm = (float *)(smem + a.off_p), sh.bar_x = bar_x;
  sh.M = M, sh.m_pad = a.m_pad, sh.q = q, sh.wait_limit = a.wait_limit, sh.status = a.status;
  Phase up;
  up.src = (const __nv_bfloat16 *)a.X, up.ld = D, up.K = D, up.kc = a.kc_up, up.pitch_bytes = a.kc_up * 2;
  up.stage_base = smem_u32(st_sm), up.w_base = smem_u32(wu_sm), up.cols = a.su, up.col0 = col_u;
  up.so = ctl->so_d, up.rows_k = ctl->rows_up, up.bias = a.b_up, up.act = a.act;
  up.out_ld = F, up.out_bf16 = 1;
  uint32_t x_parity = 0;
  if (has_up) stage_chunk(sh, up, 0, min(a.kc_up, D));
  // the row types as the previous kernel left them: the ones that count
  int my_type = -1;
  if (tid < M) {
    my_type = a.types ? __ldcg(a.types + tid) : (tid % q);
    if (my_type < 0 || my_type >= q) {
      atomicExch(a.status, (int)ALG_ERR_BAD_TYPE);
      my_type = -1;
    }
  }
  if (warp == 0) {
    if (__any_sync(0xffffffffu, my_type != spec_type)) derive_masks(ctl, a, my_type, M, q, ju, jd, lane);
    __syncwarp();
    if (lane == 0) ctl->miss_up = ctl->need_up & ~spec_up, ctl->miss_dn = ctl->need_dn & ~spec_dn;
  }
  __syncthreads();   // final masks visible
  const bool missed = (ctl->miss_up | ctl->miss_dn) != 0u;
  if (missed && tid == 0) {   // rare: blocks the final types need and the early request did not cover
    request_slice(&tm_up, bar_miss, smem_u32(wu_sm), ctl->so_d, has_up ? ctl->miss_up : 0u, q, col_u, a.su * 2, a.box_up, 0);
    request_slice(&tm_dn, bar_miss, smem_u32(wd_sm), ctl->so_f, has_dn ? ctl->miss_dn : 0u, q, col_d, a.sd * 2, a.box_dn, 0);
  }
  TR(4);
  bool ok = true;
  void *const hidden = a.exch + kExchHeader + turn.parity * (unsigned)a.exch_bytes;

  // ---------------- up phase: H[:, strip] = act(X *_q W_up + b_up) ----------------
  if (has_up) {
    ok = wait_bar(sh, bar_up, 0);
    if (ok && missed) ok = wait_bar(sh, bar_miss, 0);
    TR(5);
    up.need = ctl->need_up;
    up.out = hidden;
    if (ok) ok = run_phase_t<NTU, false, MP>(sh, up, x_parity);
    TR(6);
    if (tid == 0 && ok) exch_hint(a.exch, turn);
  } else {
    __syncthreads();   // every thread has asked for the turn
  }
  if (tid == 96) exch_leave(a.exch);   // (not the thread that waits for the hints)
  exch_clear(a.exch, a.exch_bytes, turn, F * 2, M);
  if (has_dn) {
    // ---------------- exchange: most of H is on its way ----------------
    if (tid == 0) {
      const long long t0 = clock64();
      while (!ctl->abort_flag && !exch_hinted(a.exch, turn, a.n_up - (a.n_up >> 2)))
        if (clock64() - t0 > a.wait_limit) {
          atomicExch(a.status, (int)ALG_ERR_DEVICE_TIMEOUT);
          ctl->abort_flag = 1;
        }
    }
    __syncthreads();   // also: every warp is done with the W_up slice and the partial-sum buffer
    ok = !ctl->abort_flag;
    TR(7);
    // ---------------- down phase: Y[:, strip] = H *_q W_down + b_down ----------------
    if (ok) {
      Phase dn;
      dn.src = (const __nv_bfloat16 *)hidden, dn.ld = F, dn.K = F, dn.kc = a.kc_dn, dn.pitch_bytes = a.kc_dn * 2;
      dn.stage_base = smem_u32(smem + a.off_hidden), dn.w_base = smem_u32(wd_sm), dn.cols = a.sd, dn.col0 = col_d;
      dn.so = ctl->so_f, dn.rows_k = ctl->rows_dn, dn.need = ctl->need_dn, dn.bias = a.b_down, dn.act = ALG_ACT_NONE;
      dn.out = a.Y, dn.out_ld = D, dn.out_bf16 = a.y_bf16;
      ok = wait_bar(sh, bar_dn, 0);
      if (ok && missed && !has_up) ok = wait_bar(sh, bar_miss, 0);
      TR(8);
      if (ok) ok = run_phase_t<NTD, true, MP>(sh, dn, x_parity);
    }
  }
  TR(9);
  if (ctl->abort_flag) {  // copies that are still in flight get time to land before shared memory is released
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000LL) {
    }
  }
#undef TR
}

#include "ffn_rows.cuh"

int gcd_i(int x, int y) {
  while (y) {
    const int t = x % y;
    x = y, y = t;
  }
  return x;
}

// smallest strip width (multiple of 8 that divides every group width) that needs at most num_sms CTAs
int pick_strip(int q, const int *w, int total, int num_sms) {
  int g = 0;
  for (int k = 0; k < q; ++k) g = gcd_i(g, w[k]);
  for (int s = 8; s <= 64; s += 8)
    if (g % s == 0 && total / s <= num_sms) return s;
  return 0;
}
// the instantiated strip widths: up to 32 hidden columns and 16 output columns per CTA
using Kernel = void (*)(const CUtensorMap, const CUtensorMap, const FfnDecodeArgs);
template <int NTU, int NTD>
Kernel pick_rows(bool fma, int M) {
  if (fma) return M == 1 ? ffn_rows_kernel<NTU, NTD, 1> : ffn_rows_kernel<NTU, NTD, 2>;
  return M <= 8 ? ffn_decode_kernel<NTU, NTD, 8> : ffn_decode_kernel<NTU, NTD, 16>;
}
template <int NTD>
Kernel pick_up(int ntu, bool fma, int M) {
  return ntu == 1   ? pick_rows<1, NTD>(fma, M)
         : ntu == 2 ? pick_rows<2, NTD>(fma, M)
         : ntu == 3 ? pick_rows<3, NTD>(fma, M)
         : ntu == 4 ? pick_rows<4, NTD>(fma, M)
                    : nullptr;
}
Kernel pick_kernel(int ntu, int ntd, bool fma, int M) {
  return ntd == 1 ? pick_up<1>(ntu, fma, M) : ntd == 2 ? pick_up<2>(ntu, fma, M) : nullptr;
}

}  // namespace

bool ffn_decode_plan(int q, const int *dw, const int *fw, int D, int F, int num_sms, FfnDecodePlan *plan) {
  for (int k = 0; k < q; ++k)
    if (dw[k] % 16 || fw[k] % 16) return false;
  FfnDecodePlan p = {};
  p.su = pick_strip(q, fw, F, num_sms);
  p.sd = pick_strip(q, dw, D, num_sms);
  if (!p.su || !p.sd || !pick_kernel(p.su >> 3, p.sd >> 3, false, 1)) return false;
  p.n_up = F / p.su, p.n_dn = D / p.sd;
  auto box = [&](const int *w) {   // widths are multiples of 16
    int g = 0;
    for (int k = 0; k < q; ++k) g = gcd_i(g, w[k]);
    int b = 16;
    for (int v = 16; v <= 256; v += 16)
      if (g % v == 0) b = v;
    return b;
  };
  p.box_up = box(dw), p.box_dn = box(fw);
  p.wd_bytes = F * p.sd * 2;
  p.wu_bytes = D * p.su * 2;
  p.p_bytes = kWarps * 16 * (p.su > p.sd ? p.su : p.sd) * 4;   // for 16 staged rows; half of it for 8
  p.ctl_bytes = ((int)sizeof(Ctl) + 127) & ~127;
  for (bool apart : {false, true}) {
    p.apart = apart;
    p.w_bytes = apart ? std::max(p.wd_bytes, p.wu_bytes) : p.wd_bytes + p.wu_bytes;
    p.stage_bytes = (kSmemBudget - 128 - p.w_bytes - p.p_bytes - p.ctl_bytes) & ~127;
    if (p.stage_bytes >= 16 * 64 * 2) break;
  }
  if (p.stage_bytes < 16 * 64 * 2) return false;   // at least one 64-deep chunk of 16 rows
  *plan = p;
  return true;
}

cudaError_t launch_ffn_decode(const FfnDecodeArgs &args, const FfnDecodePlan &p, cudaStream_t st) {
  FfnDecodeArgs a = args;
  a.apart = p.apart;
  a.su = p.su, a.sd = p.sd, a.n_up = p.n_up, a.n_dn = p.n_dn, a.box_up = p.box_up, a.box_dn = p.box_dn;
  // up to kRowsMax rows on plain FMAs (tables in the kernel parameters only)
  const bool rows = a.M <= kRowsMax && a.small_q && a.D <= 512 * kRowsUp && a.F <= 512 * kRowsDn;
  const Kernel kernel = pick_kernel(p.su >> 3, p.sd >> 3, rows, a.M);
  if (!kernel) return cudaErrorInvalidConfiguration;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudgetOne);
  if (e != cudaSuccess) return e;
  int ctl_bytes = p.ctl_bytes;
  a.off_wu = p.apart ? 0 : p.wd_bytes;
  if (rows) {
    a.off_p = p.w_bytes;
    a.off_ctl = (a.off_p + kWarps * (p.su + p.sd) * a.M * 4 + 127) & ~127;
    ctl_bytes = (int)sizeof(RowsCtl);
  } else {
    a.m_pad = a.M <= 8 ? 8 : 16;
    // the partial-sum buffer shrinks with the staged rows; what it gives up goes to the activation stage
    const int p_bytes = p.p_bytes * a.m_pad / 16;
    int stage_bytes = p.stage_bytes + (p.p_bytes - p_bytes);
    // apart, hidden rows in more than three chunks: one CTA per SM (1024 -> 4096 at M = 9 14.7 us, two per SM 16.6)
    if (p.apart && stage_bytes / (a.m_pad * 2) < a.F / 3) stage_bytes += kSmemBudgetOne - kSmemBudget;
    a.off_stage = p.w_bytes;
    a.off_hidden = p.apart ? a.off_stage : a.off_wu;   // (over the slice of W_up, which the CTA has used up by then)
    a.off_p = a.off_stage + stage_bytes;
    a.off_ctl = a.off_p + p_bytes;
    auto round64 = [](int v) { return (v + 63) & ~63; };
    a.kc_up = std::min(round64(a.D), (stage_bytes / (a.m_pad * 2)) & ~63);
    a.kc_dn = std::min(round64(a.F), ((a.off_p - a.off_hidden) / (a.m_pad * 2)) & ~63);
    if (a.kc_up < 64 || a.kc_dn < 64) return cudaErrorInvalidConfiguration;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.apart ? a.n_up + a.n_dn : std::max(a.n_up, a.n_dn), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = a.off_ctl + ctl_bytes + (rows ? 512 : 128);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  CUtensorMap up, dn;
  auto swizzle = [&](int strip) { return rows && (strip == 16 || strip == 32) ? strip * 2 : 0; };
  e = make_map_2d_sw(&up, a.W_up, (uint64_t)a.F, (uint64_t)a.D, (uint64_t)a.F * 2, (uint32_t)a.su, (uint32_t)a.box_up, swizzle(a.su));
  if (e == cudaSuccess)
    e = make_map_2d_sw(&dn, a.W_down, (uint64_t)a.D, (uint64_t)a.F, (uint64_t)a.D * 2, (uint32_t)a.sd, (uint32_t)a.box_dn, swizzle(a.sd));
  if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, kernel, up, dn, a);
  count_launch(1);
  return e;
}

}  // namespace algproj
