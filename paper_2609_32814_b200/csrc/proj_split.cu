// Grouped bf16 GEMM for launches with few output tiles (sm_100a): a cluster of S = 2, 4 or 8 CTAs shares ONE tile and
// splits its reduction.
//
// The persistent kernel (proj_tc.cu) gives a tile to one SM.  A small batch, or the weight gradient of a small bank, has
// fewer tiles than the GPU has SMs and long reductions: 1777 rows of 3072 -> 768 are 56 tiles of 192 columns with 24 or
// 48 stages of 64, 13 us of stages on a third of the SMs.  Here CTA r of a cluster takes the stages
// [n r / S, n (r + 1) / S) of the tile's reduction into its own tensor memory; then every CTA owns TILE_N / S columns of
// the result: it sends its partial sums of the other columns into the owners' shared memory (asynchronous stores that
// count their bytes on the owner's mbarrier), adds what it receives to its own in rank order -- one owner per element,
// bitwise repeatable --, applies bias and activation and stores.
//
// One tile per cluster, no persistence, so the prologue is short: the tile is found by one warp from the bucket offsets
// with a scan over the tile classes.  3072 -> 768 at q = 2 and 1777 rows: 19.8 us on the persistent kernel, 15 here; dW of
// 768 x 3072 over 8003 rows (72 tiles of 256 columns, 126 stages): 43 us on 128-wide tiles, 37.6 here.
//
// Warp roles (320 threads): warp 0 = TMA producer, warp 1 = TMEM allocator + MMA issuer, warps 2..9 = epilogue (two per
// TMEM lane quadrant, half of every column slice each); warp 2 also finds the tile.
// Every wait on an mbarrier is bounded (ALG_ERR_DEVICE_TIMEOUT); the CTAs of a cluster leave together, so nobody sends
// into the shared memory of a CTA that is gone.
#include "tc_common.cuh"

namespace algproj {

using namespace tc;

namespace {

constexpr int kThreads = 320;
constexpr int kMaxStages = 6;
constexpr int kABytes = 128 * 64 * 2, kBChunkBytes = 64 * 64 * 2;

struct CtlS {
  uint64_t full[kMaxStages], empty[kMaxStages];
  uint64_t acc_full, ready, recv;   // own sums complete; everybody's; partial sums received
  uint32_t tmem_base;
  volatile int abort_flag;
  int row0, rows, pair, n0, n_kb;   // the tile; row0 < 0: none
  int whole;                        // the blocks (k, k) of a weight gradient take X and G as they lie
  int so[kMaxQ + 1];
  uint32_t keep[kMaxPairs];
};

template <int TILE_N, int S>
struct CfgS {
  static constexpr int kSlice = TILE_N / S;                   // columns of the result a CTA owns
  static constexpr int kHalf = kSlice / 2;                    // an epilogue warp's share of a slice
  static constexpr int kChunk = kHalf % 32 == 0 ? 32 : kHalf % 16 == 0 ? 16 : 8;   // columns per TMEM load
  static constexpr int kTmemCols = TILE_N == 128 ? 128 : 256;
  static constexpr int kStageBytes = kABytes + kBChunkBytes * (TILE_N / 64);
  static constexpr int kRecvBytes = (S - 1) * kSlice * 128 * 4;
  static constexpr int kStages = 208 * 1024 / kStageBytes > kMaxStages ? kMaxStages : 208 * 1024 / kStageBytes;
  static constexpr int kSmemBytes = kStages * kStageBytes + (int)sizeof(CtlS) + 1024;
  static_assert(kRecvBytes <= kStages * kStageBytes, "the partial sums lie over the stages");
  static constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(TILE_N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
  static_assert(kHalf % 8 == 0 && kStages >= 2, "slice width, pipeline depth");
};

__device__ __noinline__ bool wait_s(uint32_t bar, uint32_t parity, CtlS *ctl, long long limit, int *status) {
  const long long t0 = clock64();
  uint32_t spins = 0;
  while (!mbar_try_wait(bar, parity)) {
    if ((++spins & 63u) != 0) continue;
    if (ctl->abort_flag) return false;
    if (clock64() - t0 > limit) {
      ctl->abort_flag = 1;
      atomicExch(status, (int)ALG_ERR_DEVICE_TIMEOUT);
      return false;
    }
  }
  return true;
}

template <int N>
__device__ __forceinline__ void tc_ld_n(uint32_t taddr, uint32_t (&v)[N]) {
  static_assert(N == 8 || N == 16 || N == 32, "columns per load");
  if constexpr (N == 32) {
    tc_ld_32x32(taddr, v);
  } else if constexpr (N == 16) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
                   "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                 : "r"(taddr)
                 : "memory");
  } else {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr)
                 : "memory");
  }
}

// sixteen bytes to the same place in the shared memory of CTA `rank`, counted on its barrier
__device__ __forceinline__ void send16(uint32_t addr, uint32_t bar, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr), "r"(a), "r"(b),
               "r"(c), "r"(d), "r"(bar)
               : "memory");
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

// WHOLE: weight gradient whose blocks (k, k) are reduced over X and G as they lie (ProjArgs::whole_rows): their maps.
template <bool WHOLE>
struct MoreMaps {};
template <>
struct MoreMaps<true> {
  CUtensorMap A, B;
};

// ROWS: rows of A one behind the other and the canonical bank, known at compile time (as OPS = 1 in proj_tc.cu).
template <int TILE_N, int S, bool WHOLE, bool ROWS>
__global__ void __launch_bounds__(kThreads, 1)
proj_split_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const ProjArgs a,
                  const __grid_constant__ MoreMaps<WHOLE> more) {
  using C = CfgS<TILE_N, S>;
  const bool a_mn = WHOLE ? true : ROWS ? false : a.a_mn != 0;
  const bool w_kmajor = WHOLE || ROWS ? false : a.w_kmajor != 0;
  const bool b_3d = ROWS ? true : a.b_3d != 0, a_cyclic = ROWS ? false : a.a_cyclic_rows != 0;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  // partial sums arrive over the stages: nobody sends before every CTA of the cluster has used its operands up (the bytes
  // in flight are what a CTA's operand fill hangs on; with room of their own they left three stages of a 256-wide tile)
  uint8_t *recv = smem;
  CtlS *ctl = (CtlS *)(smem + C::kStages * C::kStageBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = a.q;
  const int rank = (int)(blockIdx.x % S), tile = (int)(blockIdx.x / S);
  const DevTable *__restrict__ tab = a.tab;

  // ---- what does not depend on the previous kernel ----
  ClassRec cls = {};
  if (warp == 0) {
    if (lane < C::kStages) {
      mbar_init(smem_u32(&ctl->full[lane]), 1);
      mbar_init(smem_u32(&ctl->empty[lane]), 1);
    } else if (lane == C::kStages) {
      mbar_init(smem_u32(&ctl->acc_full), 1);
      mbar_init(smem_u32(&ctl->ready), S);
      mbar_init(smem_u32(&ctl->recv), 1);
      ctl->abort_flag = 0;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB) : "memory");
    }
  } else if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)), "r"((uint32_t)C::kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  } else if (warp == 2) {
    if (lane < a.n_classes) cls = tab->cls[lane];
  } else if (warp == 3) {
    for (int e = lane; e < q * q; e += 32) ctl->keep[e] = tab->keep[e];
  } else if (warp == 4 && !a.dyn_so) {
    for (int e = lane; e <= q; e += 32) ctl->so[e] = a.seg_rows ? e * a.seg_rows : tab->so[e];
  }
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // this CTA's barriers are ready for its peers
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (warp == 4 && a.dyn_so) {
    for (int e = lane; e <= q; e += 32) ctl->so[e] = __ldcg(a.dyn_so + e);
    if (WHOLE && lane == 0) ctl->whole = __ldcg(a.whole_valid) == a.whole_rows;
  } else if (warp == 2) {
    // tile -> (class, m-tile, n-tile): tiles are enumerated class by class, the n-tile fastest
    int before = 0, row0 = -1;
    for (int c0 = 0; c0 < a.n_classes; c0 += 32) {
      if (c0) cls = c0 + lane < a.n_classes ? tab->cls[c0 + lane] : ClassRec{};
      const bool live = c0 + lane < a.n_classes;
      int lo = 0, hi = 0;
      if (live) lo = a.offsets ? __ldcg(a.offsets + cls.i) : (int)cls.i * a.cyclic_rows, hi = a.offsets ? __ldcg(a.offsets + cls.i + 1) : lo + a.cyclic_rows;
      const int count = ((hi - lo + 127) >> 7) * (int)cls.n_tiles;
      int incl = count;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += n;
      }
      const unsigned hit = __ballot_sync(0xffffffffu, live && tile < before + incl);
      if (hit) {
        if (lane == __ffs(hit) - 1) {
          const int loc = tile - (before + incl - count), nt_n = (int)cls.n_tiles, mt = loc / nt_n, nt = loc - mt * nt_n;
          ctl->rows = min(128, hi - lo - (mt << 7));
          ctl->pair = (int)cls.i * q + (int)cls.j;
          ctl->n0 = cls.col0 + nt * (int)cls.cols;
          ctl->row0 = lo + (mt << 7);
        }
        row0 = 0;
        break;
      }
      before += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (row0 < 0 && lane == 0) ctl->row0 = -1;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  const uint32_t tmem = ctl->tmem_base;

  if (ctl->row0 >= 0) {
    const int row0 = ctl->row0, rows = ctl->rows, pair = ctl->pair, n0 = ctl->n0, type_i = pair / q;
    const uint32_t mask = ctl->keep[pair];
    const bool whole = WHOLE && ctl->whole && pair % (q + 1) == 0;   // a block (k, k): one segment, all rows
    int n_kb = whole ? (a.whole_rows + 63) >> 6 : 0;
    for (int k = 0; k < q && !whole; ++k)
      if ((mask >> k) & 1u) n_kb += (ctl->so[k + 1] - ctl->so[k]) >> 6;
    const int b0 = n_kb * rank / S, b1 = n_kb * (rank + 1) / S;   // this CTA's stages of the reduction
    if (warp == 0) {
      // ---------------- TMA producer (warp-uniform loops, one elected lane issues) ----------------
      const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]), smem0 = smem_u32(smem);
      const int a_row = a.a_cyclic_rows ? row0 - type_i * a.a_cyclic_rows : row0;
      int stage = 0, blk = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int k = 0; k < (whole ? 1 : q) && ok; ++k) {
        if (!whole && !((mask >> k) & 1u)) continue;
        const int k_begin = whole ? 0 : ctl->so[k], n = whole ? n_kb : (ctl->so[k + 1] - k_begin) >> 6;
        for (int i = max(0, b0 - blk); i < min(n, b1 - blk); ++i) {
          ok = __all_sync(0xffffffffu, mbar_try_wait(empty0 + 8u * stage, phase ^ 1u) || wait_s(empty0 + 8u * stage, phase ^ 1u, ctl, a.wait_limit, a.status));
          if (!ok) break;
          const uint32_t bar = full0 + 8u * stage, sa = smem0 + (uint32_t)(stage * C::kStageBytes);
          const int k0 = k_begin + (i << 6);
          if (elect_one()) {
            mbar_expect_tx(bar, (uint32_t)C::kStageBytes);
            if (a_mn) {   // weight gradient: rows of X and G as they lie, features / columns contiguous
              const int pos0 = a.seg_rows ? i << 6 : k0, seg = a.seg_rows ? k : 0;
              const CUtensorMap *map_a = &tmA, *map_b = &tmB;
              if constexpr (WHOLE) {
                if (whole) map_a = &more.A, map_b = &more.B;
              }
#pragma unroll
              for (int c = 0; c < 2; ++c) tma_load_3d(sa + c * kBChunkBytes, map_a, bar, row0 + c * 64, seg, pos0);
#pragma unroll
              for (int c = 0; c < TILE_N / 64; ++c) tma_load_3d(sa + kABytes + c * kBChunkBytes, map_b, bar, n0 + c * 64, seg, pos0);
            } else {
              if (a_cyclic) tma_load_3d(sa, &tmA, bar, k0, type_i, a_row);
              else tma_load_2d(sa, &tmA, bar, k0, a_row);
              if (w_kmajor) {
                tma_load_2d(sa + kABytes, &tmB, bar, k0, n0);
              } else if (b_3d) {
                tma_load_3d(sa + kABytes, &tmB, bar, 0, k0, n0 >> 6);
              } else {
#pragma unroll
                for (int c = 0; c < TILE_N / 64; ++c) tma_load_2d(sa + kABytes + c * kBChunkBytes, &tmB, bar, n0 + c * 64, k0);
              }
            }
          }
          __syncwarp();
          if (++stage == C::kStages) stage = 0, phase ^= 1u;
        }
        blk += n;
      }
    } else if (warp == 1) {
      // ---------------- MMA issuer (operand layouts as in proj_tc.cu) ----------------
      const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
      const uint64_t da0 = a_mn ? make_smem_desc(smem_u32(smem), 64 * 64 * 2, 1024) : make_smem_desc(smem_u32(smem), 16, 1024);
      const uint64_t da_step = a_mn ? 128 : 2;
      const uint64_t db0 = w_kmajor ? make_smem_desc(smem_u32(smem) + kABytes, 16, 1024) : make_smem_desc(smem_u32(smem) + kABytes, kBChunkBytes, 1024);
      const uint64_t db_step = w_kmajor ? 2 : 128;
      const uint32_t idesc = (w_kmajor ? (C::kIdesc & ~(1u << 16)) : C::kIdesc) | (a_mn ? (1u << 15) : 0u);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int kb = b0; kb < b1; ++kb) {
        ok = __all_sync(0xffffffffu, mbar_try_wait(full0 + 8u * stage, phase) || wait_s(full0 + 8u * stage, phase, ctl, a.wait_limit, a.status));
        if (!ok) break;
        tc_fence_after();
        const uint64_t at = (uint64_t)(stage * (C::kStageBytes >> 4));
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            tc_mma_bf16(tmem, da0 + at + (uint64_t)kk * da_step, db0 + at + (uint64_t)kk * db_step, idesc, (kb > b0 || kk) ? 1u : 0u);
          tc_commit(empty0 + 8u * stage);
        }
        __syncwarp();
        if (++stage == C::kStages) stage = 0, phase ^= 1u;
      }
      if (ok && b1 > b0) {
        if (elect_one()) tc_commit(smem_u32(&ctl->acc_full));
        __syncwarp();
      }
    } else {
      // ---------------- epilogue ----------------
      const int quad = warp & 3, half = (warp - 2) >> 2, r = quad * 32 + lane;
      const int groups = (rows + 31) >> 5;   // 32-row groups that hold rows of the tile
      const uint32_t recv_bar = smem_u32(&ctl->recv);
      if (warp == 2 && lane == 0) mbar_expect_tx(recv_bar, (uint32_t)((S - 1) * C::kSlice * groups * 32 * 4));
      if (quad < groups) {
        const bool mine = b1 > b0;   // (more CTAs than stages: this one has nothing to add)
        bool ok = !mine || mbar_try_wait(smem_u32(&ctl->acc_full), 0) || wait_s(smem_u32(&ctl->acc_full), 0, ctl, a.wait_limit, a.status);
        ok = __all_sync(0xffffffffu, ok);
        tc_fence_after();
        if (warp == 4 && ok && lane < S)   // (quadrant 0: never without rows)
          asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(map_rank(smem_u32(&ctl->ready), (uint32_t)lane)) : "memory");
        if (ok) ok = mbar_try_wait(smem_u32(&ctl->ready), 0) || wait_s(smem_u32(&ctl->ready), 0, ctl, a.wait_limit, a.status);
        ok = __all_sync(0xffffffffu, ok);
        const uint32_t t_row = tmem + ((uint32_t)(quad * 32) << 16);
        constexpr int kHalf = C::kHalf;
        auto slot_at = [&](int slot, int col) { return smem_u32(recv) + (uint32_t)(((slot * (C::kSlice / 4) + (col >> 2)) * 128 + r) * 16); };
        if (ok) {
#pragma unroll 1
          for (int d = 1; d < S; ++d) {
            const int owner = (rank + d) % S, slot = rank < owner ? rank : rank - 1;
            const uint32_t bar = map_rank(recv_bar, (uint32_t)owner);
#pragma unroll 1
            for (int c = half * kHalf; c < (half + 1) * kHalf; c += C::kChunk) {
              uint32_t v[C::kChunk];
              if (mine) {
                tc_ld_n(t_row + (uint32_t)(owner * C::kSlice + c), v);
                tc_wait_ld();
              } else {
#pragma unroll
                for (int x = 0; x < C::kChunk; ++x) v[x] = 0u;
              }
              const uint32_t at = map_rank(slot_at(slot, c), (uint32_t)owner);
#pragma unroll
              for (int x = 0; x < C::kChunk; x += 4) send16(at + (uint32_t)(x >> 2) * 2048u, bar, v[x], v[x + 1], v[x + 2], v[x + 3]);
            }
          }
          int64_t out_row = -1;
          if (r < rows) {
            if (a.out_cyclic_rows) out_row = (int64_t)(row0 + r - type_i * a.out_cyclic_rows) * q + type_i;
            else out_row = a.perm ? __ldg(a.perm + row0 + r) : (row0 + r);
            if (out_row >= a.M) out_row = -1;   // never store outside Y, whatever the tile says
          }
          ok = mbar_try_wait(recv_bar, 0) || wait_s(recv_bar, 0, ctl, a.wait_limit, a.status);
          ok = __all_sync(0xffffffffu, ok);
          if (ok) {
#pragma unroll 1
            for (int c = half * kHalf; c < (half + 1) * kHalf; c += C::kChunk) {
              float f[C::kChunk];
              uint32_t v[C::kChunk];
              if (mine) {
                tc_ld_n(t_row + (uint32_t)(rank * C::kSlice + c), v);
                tc_wait_ld();
              } else {
#pragma unroll
                for (int x = 0; x < C::kChunk; ++x) v[x] = 0u;
              }
#pragma unroll
              for (int x = 0; x < C::kChunk; ++x) f[x] = 0.f;
#pragma unroll
              for (int s = 0; s < S; ++s) {   // in rank order
                if (s == rank) {
#pragma unroll
                  for (int x = 0; x < C::kChunk; ++x) f[x] += __uint_as_float(v[x]);
                } else {
                  const uint32_t at = slot_at(s < rank ? s : s - 1, c);
#pragma unroll
                  for (int x = 0; x < C::kChunk; x += 4) {
                    float4 p;
                    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(p.x), "=f"(p.y), "=f"(p.z), "=f"(p.w) : "r"(at + (uint32_t)(x >> 2) * 2048u));
                    f[x] += p.x, f[x + 1] += p.y, f[x + 2] += p.z, f[x + 3] += p.w;
                  }
                }
              }
              const int col = n0 + rank * C::kSlice + c;
              if (a.bias) {
#pragma unroll
                for (int x = 0; x < C::kChunk; ++x) f[x] += __bfloat162float(__ldg((const __nv_bfloat16 *)a.bias + col + x));
              }
              if (a.act == ALG_ACT_GELU_ERF) {
#pragma unroll
                for (int x = 0; x < C::kChunk; x += 2) gelu_erf2(f[x], f[x + 1]);
              } else if (a.act == ALG_ACT_GELU_TANH) {
#pragma unroll
                for (int x = 0; x < C::kChunk; ++x) f[x] = gelu_tanh(f[x]);
              }
              if (out_row >= 0) {
                if (a.y_bf16) {
                  uint4 *dst = (uint4 *)((__nv_bfloat16 *)a.Y + out_row * a.ldy + col);
#pragma unroll
                  for (int x = 0; x < C::kChunk; x += 8) {
                    uint32_t w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                      __nv_bfloat162 p = __floats2bfloat162_rn(f[x + 2 * e], f[x + 2 * e + 1]);
                      w[e] = *(uint32_t *)&p;
                    }
                    dst[x >> 3] = make_uint4(w[0], w[1], w[2], w[3]);
                  }
                } else {
                  float4 *dst = (float4 *)((float *)a.Y + out_row * a.ldy + col);
#pragma unroll
                  for (int x = 0; x < C::kChunk; x += 4) dst[x >> 2] = make_float4(f[x], f[x + 1], f[x + 2], f[x + 3]);
                }
              }
            }
          }
        }
      }
    }
  }

  // ---------------- teardown ----------------
  __syncwarp();
  if (ctl->abort_flag) {
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000LL) {   // copies still in flight land before shared memory is released
    }
  }
  tc_fence_before();
  __syncthreads();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)C::kTmemCols) : "memory");
  }
}

template <int TILE_N, int S, bool WHOLE, bool ROWS>
cudaError_t launch_w(const ProjArgs &a, int tiles, cudaStream_t st) {
  using C = CfgS<TILE_N, S>;
  static_assert(C::kSmemBytes <= 227 * 1024, "shared memory budget");
  cudaError_t e = cudaFuncSetAttribute(proj_split_kernel<TILE_N, S, WHOLE, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
  if (e != cudaSuccess) return e;
  CUtensorMap tmA, tmB;
  ProjArgs b = a;
  e = make_tc_maps(&tmA, &tmB, &b, TILE_N, 128, false, 64);
  if (e != cudaSuccess) return e;
  if constexpr (ROWS) {
    if (!b.b_3d) return launch_w<TILE_N, S, WHOLE, false>(a, tiles, st);
  }
  MoreMaps<WHOLE> more;
  if constexpr (WHOLE) {
    e = make_grad_maps(&more.A, &more.B, a.whole_x, a.whole_ldx, a.M, a.whole_g, a.whole_ldg, a.N, 1, a.whole_rows);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(tiles * S), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = C::kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = S, at[1].val.clusterDim.y = 1, at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  count_launch(1);
  return cudaLaunchKernelEx(&cfg, proj_split_kernel<TILE_N, S, WHOLE, ROWS>, tmA, tmB, b, more);
}
template <int TILE_N, int S>
cudaError_t launch_s(const ProjArgs &a, int tiles, cudaStream_t st) {
  if (a.whole_rows) return launch_w<TILE_N, S, true, false>(a, tiles, st);
  return a.a_mn || a.w_kmajor || a.a_cyclic_rows ? launch_w<TILE_N, S, false, false>(a, tiles, st) : launch_w<TILE_N, S, false, true>(a, tiles, st);
}

}  // namespace

cudaError_t launch_proj_split(const ProjArgs &a, int tile_n, int splits, int tiles, cudaStream_t st) {
  cudaError_t e = tc_init();
  if (e != cudaSuccess) return e;
  if (a.geom.tile_m != 128 || a.block_k != 64 || a.gated_f || a.run_rows || a.in_perm || tiles < 1 || (a.whole_rows && !a.a_mn)) return cudaErrorInvalidValue;
  if (tile_n == 256) {
    if (splits == 2) return launch_s<256, 2>(a, tiles, st);
    if (splits == 4) return launch_s<256, 4>(a, tiles, st);
    if (splits == 8) return launch_s<256, 8>(a, tiles, st);
  } else if (tile_n == 192) {
    if (splits == 2) return launch_s<192, 2>(a, tiles, st);
    if (splits == 4) return launch_s<192, 4>(a, tiles, st);
  } else if (tile_n == 128) {
    if (splits == 2) return launch_s<128, 2>(a, tiles, st);
    if (splits == 4) return launch_s<128, 4>(a, tiles, st);
    if (splits == 8) return launch_s<128, 8>(a, tiles, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace algproj
