// SIMT grouped projections: true fp32 FMAs, any group widths.  One CTA computes an output tile of one
// (row type i, output group j) pair and sums every kept product x_k W_kj (k in B(i,j),
// Eq. recursive-row-action) in registers before the single store.
//   proj_f32_kernel   fp32 operands: asynchronous copies into a three-stage ring, register tiles.
//   proj_simt_kernel  bf16 operands of the shapes the tensor-core paths do not cover (and their input gradient).
#include <algorithm>

#include "tile_map.cuh"

namespace algproj {

namespace {

constexpr int TM = 64, TN = 64, TK = 16;

__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }

__device__ __forceinline__ float apply_act(float z, int act) {
  if (act == ALG_ACT_GELU_ERF) return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f));
  if (act == ALG_ACT_GELU_TANH) {
    float u = 0.7978845608028654f * (z + 0.044715f * z * z * z);
    return 0.5f * z * (1.0f + tanhf(u));
  }
  return z;
}

template <typename T>
__global__ void __launch_bounds__(256) proj_simt_kernel(const ProjArgs a) {
  __shared__ float As[TK][TM + 1];
  __shared__ float Bs[TK][TN];
  __shared__ int s_rows[TM];
  extern __shared__ __align__(16) unsigned char s_map[];  // tile_map_bytes(n_classes)
  TileMap *tm = reinterpret_cast<TileMap *>(s_map);
  const DevTable *__restrict__ tab = a.tab;
  const int q = a.q;
  tile_map_classes(tm, tab, a.st, q, a.n_classes, threadIdx.x, 256);
  tile_map_build(tm, q, a.n_classes, a.offsets, a.cyclic_rows, a.M, a.geom);
  const int n_tiles = tm->total;
  const T *__restrict__ X = (const T *)a.X;
  const T *__restrict__ W = (const T *)a.W;
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;  // 16 x 16 threads, 4 x 4 outputs each

  for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    TileRec rec = tile_map_decode(tm, a.geom, tile);
    rec.pair &= 0xFFFF;
    const int j = rec.pair % q;
    const int n_valid = min(TN, tab->ro[j + 1] - rec.n0);
    __syncthreads();
    if (tid < TM) {
      int r = rec.row0 + tid;
      s_rows[tid] = (tid < rec.rows) ? (a.in_perm ? a.in_perm[r] : r) : -1;
    }
    __syncthreads();
    float acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) acc[u][v] = 0.f;

    const uint32_t mask = tab->keep[rec.pair];
    for (int k = 0; k < q; ++k) {
      if (!((mask >> k) & 1u)) continue;
      const int k_begin = tab->so[k], k_end = tab->so[k + 1];
      for (int k0 = k_begin; k0 < k_end; k0 += TK) {
        // A tile: 64 rows x 16 k  (4 elements per thread), B tile: 16 k x 64 cols
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          int idx = tid + e * 256;
          int r = idx >> 4, kk = idx & 15;
          int src = s_rows[r];
          float v = 0.f;
          if (src >= 0 && k0 + kk < k_end) v = to_f32(X[(int64_t)src * a.ldx + k0 + kk]);
          As[kk][r] = v;
          int kb = idx >> 6, c = idx & 63;
          float w = 0.f;
          if (k0 + kb < k_end && c < n_valid)
            w = to_f32(a.w_kmajor ? W[(int64_t)(rec.n0 + c) * a.ldw + k0 + kb] : W[(int64_t)(k0 + kb) * a.ldw + rec.n0 + c]);
          Bs[kb][c] = w;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < TK; ++kk) {
          float av[4], bv[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) av[u] = As[kk][ty * 4 + u];
#pragma unroll
          for (int v = 0; v < 4; ++v) bv[v] = Bs[kk][tx * 4 + v];
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(av[u], bv[v], acc[u][v]);
        }
        __syncthreads();
      }
    }
    // epilogue: bias, activation, scatter to the original row order
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      int r = ty * 4 + u;
      if (r >= rec.rows) continue;
      int out_row = a.perm ? a.perm[rec.row0 + r] : rec.row0 + r;
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        int c = tx * 4 + v;
        if (c >= n_valid) continue;
        int col = rec.n0 + c;
        float z = acc[u][v];
        if (a.bias) z += to_f32(((const T *)a.bias)[col]);
        z = apply_act(z, a.act);
        if (a.y_bf16) ((__nv_bfloat16 *)a.Y)[(int64_t)out_row * a.ldy + col] = __float2bfloat16_rn(z);
        else ((float *)a.Y)[(int64_t)out_row * a.ldy + col] = z;
      }
    }
  }
}

// ---- fp32 operands ----
//
// TM x 64 tile, 256 threads in kGroups groups that share out the k of every chunk (four at a time, round robin) and
// are summed through shared memory in a fixed order at the end.  A thread of a group owns 8 x 8 outputs: rows
// ty + (TM / 8) u, columns 4 tx .. and 32 + 4 tx ..  Both operands arrive in shared memory as they lie in global memory
// (A: rows along k, B: rows along n), by 16-byte asynchronous copies with zero fill at the edges (4-byte ones when a
// width, a leading dimension or a base is no multiple of 16 bytes), in a ring of kF32Stages chunks of 64 k.  Four k at
// a time a thread reads a float4 of each of its rows and eight of B for 256 FMAs, so FP32 issue is the limit once
// there are enough tiles; the register tile of 8 x 8 and the split of k give a single tile the instruction-level
// parallelism it needs when there is only one per SM.
// Measured against the kernel this one replaced (16-deep chunks loaded, waited for and used by 4 x 4 register tiles, and
// a bucketing launch before it): 256 -> 1024 at q = 2, M = 512 41.0 -> 14.1 us a call, M = 4096 118 -> 68; 640 -> 2560
// at q = 4, M = 4096 380 -> 215 (17.6 FP32 TFLOP/s of the kept products).
constexpr int kCountQ = kParamQ;    // most types of a batch whose buckets the CTAs count themselves
static_assert(kCountQ == 8 && kCountRows <= 256 * 16 && kCountRows < (1 << 16), "sixteen rows of 4 bits per thread, counts of 16 bits");
constexpr int kF32Sms = 148;
constexpr int F_TN = 64, F_TK = 64, kF32Stages = 3;
constexpr int kAPitch = F_TK + 4;   // floats: the four rows a warp reads at once sit on other banks
template <int TM_>
struct F32Cfg {
  static constexpr int kGroupThreads = TM_ * F_TN / 64, kGroups = 256 / kGroupThreads;
  static constexpr int kABytes = TM_ * kAPitch * 4;
  static constexpr int kStageBytes = kABytes + F_TK * F_TN * 4;
  static constexpr int kRingBytes = kF32Stages * kStageBytes;
  static_assert(kRingBytes >= kGroups * TM_ * F_TN * 4, "the partial tiles of the groups reuse the ring");
};

template <int BYTES>
__device__ __forceinline__ void cp_async_zfill(uint32_t dst, const void *src, int src_bytes) {
  if (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}

// The buckets of a small batch, found by every CTA for itself instead of by a launch of their own: thread t looks at rows
// [t n, (t + 1) n), n = M / 256 rounded up, and keeps their types in 4 bits each; counts of four types share one 64-bit
// word (16 bits each), so a scan over the threads is a scan of two words.  (In shared memory: the main loop has no
// registers to spare for it.)
struct RowCount {
  uint64_t types[256];         // 4 bits per row; kCountQ = outside [0, q)
  uint64_t before[2][256];     // rows of types 0..3 / 4..7 in the threads before this one
  uint64_t warp_sum[8][2];
  int off[kCountQ + 2];
};
__device__ __forceinline__ void count_rows(const ProjArgs &a, RowCount &rc) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = (a.M + 255) >> 8, row0 = tid * per, n = max(0, min(per, a.M - row0));
  uint64_t types = 0, lo = 0, hi = 0;
#pragma unroll 4
  for (int e = 0; e < n; ++e) {
    int t = a.types ? __ldg(a.types + row0 + e) : (row0 + e) % a.q;
    if (t < 0 || t >= a.q) {
      t = kCountQ;
      if ((row0 + e) % (int)gridDim.x == (int)blockIdx.x) {   // out-of-range type: the row's output is defined to be zero
        atomicExch(a.status, (int)ALG_ERR_BAD_TYPE);
        char *y = (char *)a.Y + (int64_t)(row0 + e) * a.ldy * (a.y_bf16 ? 2 : 4);
        for (int b = 0; b < a.N * (a.y_bf16 ? 2 : 4); ++b) y[b] = 0;
      }
    }
    types |= (uint64_t)t << (4 * e);
    if (t < 4) lo += 1ull << (16 * t);
    else if (t < kCountQ) hi += 1ull << (16 * (t - 4));
  }
  const uint64_t own_lo = lo, own_hi = hi;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint64_t l = __shfl_up_sync(0xffffffffu, lo, d), h = __shfl_up_sync(0xffffffffu, hi, d);
    if (lane >= d) lo += l, hi += h;
  }
  if (lane == 31) rc.warp_sum[warp][0] = lo, rc.warp_sum[warp][1] = hi;
  __syncthreads();
  uint64_t all_lo = 0, all_hi = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    if (w == warp) lo += all_lo, hi += all_hi;
    all_lo += rc.warp_sum[w][0], all_hi += rc.warp_sum[w][1];
  }
  rc.types[tid] = types, rc.before[0][tid] = lo - own_lo, rc.before[1][tid] = hi - own_hi;
  if (tid == 0) {
    int at = 0;
    for (int t = 0; t < a.q; ++t) {
      rc.off[t] = at;
      at += (int)(((t < 4 ? all_lo : all_hi) >> (16 * (t & 3))) & 0xFFFFu);
    }
    rc.off[a.q] = at, rc.off[a.q + 1] = a.M;
  }
  __syncthreads();
}
// rows[0 .. n): the rows of type i with ranks first .. first + n - 1 among the rows of their type
__device__ __forceinline__ void rows_of_type(const RowCount &rc, int M, int i, int first, int n, int *rows) {
  const int tid = threadIdx.x, per = (M + 255) >> 8;
  uint64_t types = rc.types[tid];
  int rank = (int)((rc.before[i >> 2][tid] >> (16 * (i & 3))) & 0xFFFFu) - first;
  for (int e = 0; e < per && tid * per + e < M; ++e, types >>= 4)
    if ((int)(types & 15u) == i) {
      if (rank >= 0 && rank < n) rows[rank] = tid * per + e;
      ++rank;
    }
}

template <int TM_, int VEC>
__global__ void __launch_bounds__(256, TM_ == 64 ? 2 : 1) proj_f32_kernel(const ProjArgs a) {
  using C = F32Cfg<TM_>;
  extern __shared__ __align__(16) unsigned char smem[];   // ring, then tile_map_bytes(n_classes)
  __shared__ int s_rows[TM_];
  __shared__ int s_len[kF32Stages];   // k of the chunks in the ring (the last chunk of a group may be short)
  __shared__ RowCount s_count;
  TileMap *tm = reinterpret_cast<TileMap *>(smem + C::kRingBytes);
  const DevTable *__restrict__ tab = a.tab;
  const int q = a.q, tid = threadIdx.x;
  const int grp = tid / C::kGroupThreads, tx = tid & 7, ty = (tid % C::kGroupThreads) >> 3;
  tile_map_classes(tm, tab, a.st, q, a.n_classes, tid, 256);
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the bucket offsets come from the previous kernel
  if (a.count_rows) count_rows(a, s_count);
  tile_map_build(tm, q, a.n_classes, a.count_rows ? s_count.off : a.offsets, a.cyclic_rows, a.M, a.geom);
  const int n_tiles = tm->total;
  const float *__restrict__ X = (const float *)a.X;
  const float *__restrict__ W = (const float *)a.W;
  const uint32_t ring = (uint32_t)__cvta_generic_to_shared(smem);

  for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    TileRec rec = tile_map_decode(tm, a.geom, tile);
    rec.pair &= 0xFFFF;
    const int j = rec.pair % q;
    const int n_valid = min(F_TN, (a.st.valid ? a.st.ro[j + 1] : tab->ro[j + 1]) - rec.n0);
    const uint32_t mask = a.st.valid ? a.st.keep[rec.pair] : tab->keep[rec.pair];
    __syncthreads();   // the previous tile is done with s_rows and the ring
    if (tid < TM_) {
      const int r = rec.row0 + tid;
      s_rows[tid] = tid < rec.rows && !a.count_rows ? (a.in_perm ? a.in_perm[r] : r) : -1;
    }
    if (a.count_rows) {
      __syncthreads();
      const int i = rec.pair / q;
      rows_of_type(s_count, a.M, i, rec.row0 - s_count.off[i], rec.rows, s_rows);
    }
    __syncthreads();

    // walk over the chunks of the kept groups, ascending: (k_at, k_end) = next chunk to request
    uint32_t left = mask;
    int k_at = 0, k_end = 0, n_req = 0;
    auto so = [&](int k) { return a.st.valid ? a.st.so[k] : tab->so[k]; };
    auto advance = [&]() {   // true if there is a chunk to request
      if (k_at < k_end) return true;
      if (!left) return false;
      const int k = __ffs(left) - 1;
      left &= left - 1;
      k_at = so(k), k_end = so(k + 1);
      return true;
    };
    auto request = [&]() {
      if (advance()) {
        const uint32_t sa = ring + (uint32_t)(n_req % kF32Stages) * C::kStageBytes, sb = sa + C::kABytes;
        constexpr int PA = F_TK / VEC, PB = F_TN / VEC;   // pieces per row
#pragma unroll
        for (int e = 0; e < TM_ * PA / 256; ++e) {
          const int idx = tid + e * 256, r = idx / PA, kk = (idx % PA) * VEC;
          const int src = s_rows[r], n = min(VEC, k_end - k_at - kk);
          const bool ok = src >= 0 && n > 0;
          cp_async_zfill<4 * VEC>(sa + (uint32_t)(r * kAPitch + kk) * 4u, ok ? X + (int64_t)src * a.ldx + k_at + kk : X, ok ? 4 * n : 0);
        }
#pragma unroll
        for (int e = 0; e < F_TK * PB / 256; ++e) {
          const int idx = tid + e * 256, kb = idx / PB, c = (idx % PB) * VEC;
          const int n = min(VEC, n_valid - c);
          const bool ok = k_at + kb < k_end && n > 0;
          cp_async_zfill<4 * VEC>(sb + (uint32_t)(kb * F_TN + c) * 4u, ok ? W + (int64_t)(k_at + kb) * a.ldw + rec.n0 + c : W, ok ? 4 * n : 0);
        }
        if (tid == 0) s_len[n_req % kF32Stages] = min(F_TK, k_end - k_at);
        k_at += F_TK;
        ++n_req;
      }
      asm volatile("cp.async.commit_group;" ::: "memory");   // (an empty group keeps the count of groups in step)
    };
    float acc[8][8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
      for (int v = 0; v < 8; ++v) acc[u][v] = 0.f;
#pragma unroll
    for (int s = 0; s < kF32Stages - 1; ++s) request();
    for (int n = 0; n < n_req; ++n) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kF32Stages - 2) : "memory");
      __syncthreads();   // chunk n has landed for every thread; chunk n - 1 is used up
      request();
      const int len = s_len[n % kF32Stages];
      const float *As = (const float *)(smem + (n % kF32Stages) * C::kStageBytes) + ty * kAPitch;
      const float *Bs = (const float *)(smem + (n % kF32Stages) * C::kStageBytes + C::kABytes) + tx * 4;
#pragma unroll
      for (int k4 = 0; k4 < F_TK / 4 / C::kGroups; ++k4) {
        const int kk = (k4 * C::kGroups + grp) * 4;
        if (kk >= len) break;   // (the same for a whole group; the rest of the chunk is zeros)
        float4 av[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) av[u] = *(const float4 *)(As + (TM_ / 8) * u * kAPitch + kk);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float4 b0 = *(const float4 *)(Bs + (kk + e) * F_TN), b1 = *(const float4 *)(Bs + (kk + e) * F_TN + 32);
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const float x = e == 0 ? av[u].x : e == 1 ? av[u].y : e == 2 ? av[u].z : av[u].w;
            acc[u][0] = fmaf(x, b0.x, acc[u][0]), acc[u][1] = fmaf(x, b0.y, acc[u][1]);
            acc[u][2] = fmaf(x, b0.z, acc[u][2]), acc[u][3] = fmaf(x, b0.w, acc[u][3]);
            acc[u][4] = fmaf(x, b1.x, acc[u][4]), acc[u][5] = fmaf(x, b1.y, acc[u][5]);
            acc[u][6] = fmaf(x, b1.z, acc[u][6]), acc[u][7] = fmaf(x, b1.w, acc[u][7]);
          }
        }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    // The next launch may start here and not earlier: its CTAs would be placed wherever a slot is free while most SMs
    // are busy, two of them on one SM and none on another (256 -> 1024, M = 512: 22.2 us a call with the trigger at the
    // top, 16.6 here, 14.1 with one CTA per SM as well, see launch_f32)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __syncthreads();
    // the groups' partial tiles go over the ring, their sum (in group order) leaves: bias, activation, scatter to the
    // original row order
    float *part = (float *)smem;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      float *dst = part + (grp * TM_ + ty + (TM_ / 8) * u) * F_TN + tx * 4;
      *(float4 *)dst = make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
      *(float4 *)(dst + 32) = make_float4(acc[u][4], acc[u][5], acc[u][6], acc[u][7]);
    }
    __syncthreads();
    const int cx = (tid & 15) * 4, col = rec.n0 + cx;
    const bool vec_store = (rec.n0 & 3) == 0 && cx + 4 <= n_valid;
    for (int r = tid >> 4; r < rec.rows; r += 16) {
      float4 s = *(const float4 *)(part + r * F_TN + cx);
#pragma unroll
      for (int g = 1; g < C::kGroups; ++g) {
        const float4 p = *(const float4 *)(part + (g * TM_ + r) * F_TN + cx);
        s.x += p.x, s.y += p.y, s.z += p.z, s.w += p.w;
      }
      float z[4] = {s.x, s.y, s.z, s.w};
      const int64_t at = (int64_t)(a.count_rows ? s_rows[r] : a.perm ? a.perm[rec.row0 + r] : rec.row0 + r) * a.ldy + col;
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        if (a.bias && cx + v < n_valid) z[v] += ((const float *)a.bias)[col + v];
        z[v] = apply_act(z[v], a.act);
      }
      if (vec_store && !a.y_bf16) {
        *(float4 *)((float *)a.Y + at) = make_float4(z[0], z[1], z[2], z[3]);
      } else {
#pragma unroll
        for (int v = 0; v < 4; ++v)
          if (cx + v < n_valid) {
            if (a.y_bf16) ((__nv_bfloat16 *)a.Y)[at + v] = __float2bfloat16_rn(z[v]);
            else ((float *)a.Y)[at + v] = z[v];
          }
      }
    }
  }
}

template <int TM_, int VEC>
cudaError_t launch_f32(const ProjArgs &a, int grid, cudaStream_t st) {
  const size_t smem = F32Cfg<TM_>::kRingBytes + tile_map_bytes(a.n_classes);
  static OncePerDevice limit;
  const cudaError_t e = limit([] {
    return cudaFuncSetAttribute(proj_f32_kernel<TM_, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                F32Cfg<TM_>::kRingBytes + (int)tile_map_bytes(kMaxClasses));
  });
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(256, 1, 1);
  // at most one tile per SM: one CTA per SM (more than half of its shared memory), so that no two share one while
  // another idles
  constexpr size_t kHalfSm = 116 * 1024;
  cfg.dynamicSmemBytes = (int64_t)ceil_div(a.M, TM_) * ceil_div(a.N, F_TN) <= kF32Sms ? std::max(smem, kHalfSm) : smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  count_launch(1);
  return cudaLaunchKernelEx(&cfg, proj_f32_kernel<TM_, VEC>, a);
}

}  // namespace

int simt_tile_m(bool in_bf16, int M, int N) {
  if (in_bf16) return TM;
  // fp32: 128-row tiles read less shared memory per FMA and are about 10 % faster per row, 64-row tiles leave less of a
  // last round empty; compare the rounds over the SMs.  Measured, 64 / 128 rows: 256 -> 1024 at M = 512 14.1 / 21.7 us,
  // M = 2048 34.8 / 33.8; 640 -> 2560 at M = 600 51.2 / 61.6, M = 1500 89.5 / 86.7; 320 -> 640 at M = 4096 56.4 / 65.6
  const int64_t n = ceil_div(N, F_TN), r64 = (ceil_div(M, 64) * n + kF32Sms - 1) / kF32Sms,
                r128 = 2 * ((ceil_div(M, 128) * n + kF32Sms - 1) / kF32Sms);
  return 9 * r128 <= 10 * r64 ? 128 : 64;
}

// widths4: every group width of both sides is a multiple of 4
cudaError_t launch_proj_simt(const ProjArgs &a, bool in_bf16, bool widths4, cudaStream_t st) {
  // (upper bound of the tiles: every type may end in a ragged one, every output group in a narrow one)
  const int64_t tiles = (int64_t)(a.M / a.geom.tile_m + a.q) * (a.N / F_TN + a.q);
  if (!in_bf16) {
    if (a.w_kmajor || (a.count_rows && (a.q > kCountQ || a.M > kCountRows))) return cudaErrorInvalidValue;
    const bool vec = widths4 && ((uintptr_t)a.X & 15) == 0 && ((uintptr_t)a.W & 15) == 0 && a.ldx % 4 == 0 && a.ldw % 4 == 0;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(tiles, kF32Sms * (a.geom.tile_m == 128 ? 1 : 2)));
    if (a.geom.tile_m == 128) return vec ? launch_f32<128, 4>(a, grid, st) : launch_f32<128, 1>(a, grid, st);
    return vec ? launch_f32<64, 4>(a, grid, st) : launch_f32<64, 1>(a, grid, st);
  }
  const int grid = 148 * 4;
  const size_t map_bytes = tile_map_bytes(a.n_classes);
  static OncePerDevice limit;
  const cudaError_t e = limit([] { return cudaFuncSetAttribute(proj_simt_kernel<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 1024); });
  if (e != cudaSuccess) return e;
  proj_simt_kernel<__nv_bfloat16><<<grid, 256, map_bytes, st>>>(a);
  count_launch(1);
  return cudaGetLastError();
}

}  // namespace algproj
