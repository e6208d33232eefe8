// Row-type bucketing: the index sets I_i of Algorithm 1 (all rows of type i), built as one stable
// permutation.  No host synchronisation anywhere: the row counts per type never leave the device
// (the GEMM kernels turn the bucket offsets into their tile enumeration themselves).
//
//   M <= 65536: one kernel of M/1024 CTAs: each histograms its own 1024 rows, publishes the counts,
//               meets the others at a counter (bounded wait) and places its rows.
//   larger M:
//   kernel 1 (count):   per-chunk histograms (at most 256 chunks).
//   kernel 2 (scatter): each CTA scans the histograms for the bucket offsets and its own bases,
//                       then perm[offset[t] + base[t] + rank_in_chunk] = row  (stable); CTA 0
//                       publishes the bucket offsets.
//   kernel 3 (gather):  Xb[d,:] = X[perm[d],:]  -- every type becomes a contiguous M-slab.
//   M <= 8192 with a copy of X to write: one kernel for all of it (bucket_copy_kernel).
#include <algorithm>

#include "common.cuh"
#include "trace.cuh"

namespace algproj {
ALG_TRACE_DEFINE(bucket)

namespace {

__device__ __forceinline__ int row_type(const BucketArgs &a, int row) {
  int t = a.types ? a.types[row] : (row % a.q);
  return (t < 0 || t >= a.q) ? a.q : t;  // pseudo-type q collects out-of-range rows
}

// offsets of the same buckets when each is padded to a multiple of 64 rows
__device__ __forceinline__ void write_pad_offsets(WsHeader *hdr, const int *offset, int q) {
  int run = 0;
  for (int t = 0; t < q; ++t) {
    hdr->pad_offsets[t] = run;
    run += (offset[t + 1] - offset[t] + 63) & ~63;
  }
  hdr->pad_offsets[q] = run;
}

// Kernel 1: per-chunk histograms of the row types (pseudo-type q = out of range).  CAP = largest q + 1
// the instantiation serves: kMaxQ + 1 for table-driven handles, kBigMaxQ + 1 for the large-algebra path.
template <int CAP>
__global__ void __launch_bounds__(256) bucket_count_kernel(const BucketArgs a) {
  __shared__ int s_cnt[CAP];
  const int tid = threadIdx.x;
  const int nt = a.q + 1;
  for (int t = tid; t < nt; t += 256) s_cnt[t] = 0;
  __syncthreads();
  const int row_begin = blockIdx.x * a.chunk_rows;
  const int row_end = min(a.M, row_begin + a.chunk_rows);
  for (int row = row_begin + tid; row < row_end; row += 256) {
    int t = row_type(a, row);
    if (t == a.q) atomicExch(a.status, (int)ALG_ERR_BAD_TYPE);
    atomicAdd(&s_cnt[t], 1);
  }
  __syncthreads();
  for (int t = tid; t < nt; t += 256) a.chunk_counts[blockIdx.x * nt + t] = s_cnt[t];
}

// Kernel 2: every CTA scans the (at most 256) chunk histograms to find the bucket offsets and
// its own base inside each bucket, then places its rows (stable inside a type).  CTA 0 also
// publishes the offsets.
template <int CAP>
__global__ void __launch_bounds__(256) bucket_scatter_kernel(const BucketArgs a) {
  __shared__ int s_wcnt[8][CAP];
  __shared__ int s_total[CAP];
  __shared__ int s_base[CAP];     // rows of this type in earlier chunks (+ earlier sub-blocks)
  __shared__ int s_offset[CAP + 1];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nt = a.q + 1;
  const int n_chunks = gridDim.x;
  for (int t = warp; t < nt; t += 8) {
    int before = 0, total = 0;
    for (int c = lane; c < n_chunks; c += 32) {
      int v = a.chunk_counts[c * nt + t];
      total += v;
      if (c < (int)blockIdx.x) before += v;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      before += __shfl_xor_sync(0xffffffffu, before, d);
      total += __shfl_xor_sync(0xffffffffu, total, d);
    }
    if (lane == 0) {
      s_total[t] = total;
      s_base[t] = before;
    }
  }
  __syncthreads();
  if (tid == 0) {
    int run = 0;
    for (int t = 0; t < nt; ++t) {
      s_offset[t] = run;
      run += s_total[t];
    }
    s_offset[nt] = run;  // == M
  }
  __syncthreads();

  const int row_begin = blockIdx.x * a.chunk_rows;
  const int row_end = min(a.M, row_begin + a.chunk_rows);
  for (int r0 = row_begin; r0 < row_end; r0 += 256) {
    for (int e = tid; e < 8 * CAP; e += 256) (&s_wcnt[0][0])[e] = 0;
    __syncthreads();
    const int row = r0 + tid;
    const bool live = row < row_end;
    const int t = live ? row_type(a, row) : -1 - lane;  // dead lanes never match each other
    const unsigned peers = __match_any_sync(0xffffffffu, t);
    const int rank_in_warp = __popc(peers & ((1u << lane) - 1u));
    if (live && rank_in_warp == 0) s_wcnt[warp][t] = __popc(peers);
    __syncthreads();
    if (live) {
      int before = 0;
      for (int w = 0; w < warp; ++w) before += s_wcnt[w][t];
      a.perm[s_offset[t] + s_base[t] + before + rank_in_warp] = row;
      if (t == a.q && a.Y) {  // out-of-range type: the row's output is defined to be zero
        char *y = (char *)a.Y + (size_t)row * a.ldy * a.y_elem_bytes;
        for (int e = 0; e < a.N * a.y_elem_bytes; ++e) y[e] = 0;
      }
    }
    __syncthreads();
    for (int t2 = tid; t2 < nt; t2 += 256) {
      int add = 0;
      for (int w = 0; w < 8; ++w) add += s_wcnt[w][t2];
      s_base[t2] += add;
    }
    __syncthreads();
  }

  if (blockIdx.x == 0) {
    // more than kMaxQ types: the offsets go to the caller's array (the fixed header has no room for them)
    int *offsets = a.big_offsets ? a.big_offsets : a.hdr->offsets;
    for (int t = tid; t <= nt; t += 256) offsets[t] = s_offset[t];
    if (tid == 0 && !a.big_offsets) write_pad_offsets(a.hdr, s_offset, a.q);
  }
}

// One-pass variant for M <= 65536 (at most 64 CTAs of 1024 threads, one row per thread): every row
// type is read exactly once.  A CTA ranks its rows inside their type (warp match + per-warp counts),
// publishes its per-type counts, arrives on a counter and waits (bounded) until every CTA has;
// then it sums the counts of all chunks (bucket offsets) and of the chunks before it (its base)
// and writes perm.  All CTAs are resident together: the grid is far smaller than the machine, and
// the kernel launched after it starts only once every CTA of this one has.  The last CTA past the
// wait clears the counter for the next launch.
//
// CLUSTER (M <= 8192, M <= 16384 where the device takes clusters of 16): the CTAs form one thread-block cluster; the per-type counts stay in shared memory, the
// cluster's hardware barrier replaces the counter and every CTA reads its peers' counts through the cluster's
// shared-memory window -- no round trip to L2 between the ranking and the write of perm.
constexpr int kFusedThreads = 1024;
constexpr int kClusterRows = 8 * kFusedThreads;
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
template <bool CLUSTER>
__global__ void __launch_bounds__(kFusedThreads) bucket_onepass_kernel(const BucketArgs a) {
  __shared__ int s_wcnt[32][kMaxQ + 1];   // rows of type t in warp w; then exclusive prefix over the warps
  __shared__ int s_base[kMaxQ + 1], s_offset[kMaxQ + 2];
  __shared__ int s_tot[kMaxQ + 1];        // CLUSTER: rows of type t in this CTA, read by the peers
  __shared__ int s_go;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nt = a.q + 1;
  const int n_chunks = gridDim.x;
  ALG_TRACE_VARS;
  if (tid == 0) ALG_TRACE(0, 1);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the row types may come from the previous kernel
  if (tid == 0) ALG_TRACE(0, 2);
  for (int e = tid; e < 32 * (kMaxQ + 1); e += kFusedThreads) (&s_wcnt[0][0])[e] = 0;
  const int row = blockIdx.x * kFusedThreads + tid;
  const bool live = row < a.M;
  const int t = live ? row_type(a, row) : -1 - lane;  // dead lanes never match each other
  if (live && t == a.q) atomicExch(a.status, (int)ALG_ERR_BAD_TYPE);
  const unsigned peers = __match_any_sync(0xffffffffu, t);
  const int rank_in_warp = __popc(peers & ((1u << lane) - 1u));
  if (tid == 0) ALG_TRACE(0, 3);
  __syncthreads();
  if (live && rank_in_warp == 0) s_wcnt[warp][t] = __popc(peers);
  __syncthreads();
  for (int ty = warp; ty < nt; ty += kFusedThreads / 32) {   // exclusive prefix over the warps (lane = warp); the total goes to global memory
    const int v = s_wcnt[lane][ty];
    int incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += o;
    }
    s_wcnt[lane][ty] = incl - v;
    if (lane == 31) {
      if (CLUSTER) {
        s_tot[ty] = incl;
      } else {
        a.chunk_counts[blockIdx.x * nt + ty] = incl;
        __threadfence();
      }
    }
  }
  if (CLUSTER) {
    cluster_sync_all();   // (also orders the shared-memory writes above for this CTA's own threads)
    for (int ty = warp; ty < nt; ty += kFusedThreads / 32) {   // lanes over the CTAs of the cluster (at most 16)
      int v = 0;
      if (lane < n_chunks) {
        uint32_t remote;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"((uint32_t)__cvta_generic_to_shared(&s_tot[ty])), "r"(lane));
        asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(remote) : "memory");
      }
      int before = lane < (int)blockIdx.x ? v : 0, total = v;
#pragma unroll
      for (int d = 8; d > 0; d >>= 1) {
        before += __shfl_xor_sync(0xffffffffu, before, d);
        total += __shfl_xor_sync(0xffffffffu, total, d);
      }
      if (lane == 0) s_base[ty] = before, s_offset[ty] = total;
    }
    cluster_sync_all();   // no CTA leaves (or overwrites s_tot) while a peer may still read its counts
  } else {
  __syncthreads();
  if (tid == 0) {
    ALG_TRACE(0, 4);
    atomicAdd(a.sync, 1u);
    const long long t0 = clock64();
    int go = 1;
    unsigned v;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.sync) : "memory");
      if (v < (unsigned)n_chunks && clock64() - t0 > a.wait_limit) {
        atomicExch(a.status, (int)ALG_ERR_DEVICE_TIMEOUT);
        go = 0;
        break;
      }
    } while (v < (unsigned)n_chunks);
    s_go = go;
    ALG_TRACE(0, 5);
  }
  __syncthreads();
  if (!s_go) return;
  if (tid == 0 && atomicAdd(a.sync + 1, 1u) == (unsigned)(n_chunks - 1)) a.sync[0] = 0u, a.sync[1] = 0u;
  {   // lanes over the chunks (at most 64); the warps share the types, so that their round trips to L2 overlap
    for (int ty = warp; ty < nt; ty += kFusedThreads / 32) {
      int before = 0, total = 0;
      for (int c = lane; c < n_chunks; c += 32) {
        const int v = __ldcg(a.chunk_counts + c * nt + ty);
        total += v;
        if (c < (int)blockIdx.x) before += v;
      }
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) {
        before += __shfl_xor_sync(0xffffffffu, before, d);
        total += __shfl_xor_sync(0xffffffffu, total, d);
      }
      if (lane == 0) s_base[ty] = before, s_offset[ty] = total;
    }
  }
  __syncthreads();
  }
  if (tid == 0) ALG_TRACE(0, 6);
  if (warp == 0) {   // bucket offsets: exclusive prefix of the totals over the types (nt <= 33: lane 0 takes two)
    const int v0 = lane < nt ? s_offset[lane] : 0, v1 = lane == 0 && nt > 32 ? s_offset[32] : 0;
    int incl = v0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += o;
    }
    const int total32 = __shfl_sync(0xffffffffu, incl, 31);
    if (lane < nt) s_offset[lane] = incl - v0;
    if (lane == 0) {
      if (nt > 32) s_offset[32] = total32, s_offset[33] = total32 + v1;
      else s_offset[nt] = total32;   // == M
    }
  }
  __syncthreads();
  if (live) {
    a.perm[s_offset[t] + s_base[t] + s_wcnt[warp][t] + rank_in_warp] = row;
    if (t == a.q && a.Y) {  // out-of-range type: the row's output is defined to be zero
      char *y = (char *)a.Y + (size_t)row * a.ldy * a.y_elem_bytes;
      for (int e = 0; e < a.N * a.y_elem_bytes; ++e) y[e] = 0;
    }
  }
  if (tid == 0) ALG_TRACE(0, 7);
  if (blockIdx.x == 0) {
    for (int t2 = tid; t2 <= nt; t2 += kFusedThreads) a.hdr->offsets[t2] = s_offset[t2];
    if (warp == 1) {   // offsets of the buckets padded to multiples of 64 rows (q <= 32: one lane per type)
      const int v = lane < a.q ? (s_offset[lane + 1] - s_offset[lane] + 63) & ~63 : 0;
      int incl = v;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
      }
      if (lane < a.q) a.hdr->pad_offsets[lane] = incl - v;
      if (lane == 31) a.hdr->pad_offsets[a.q] = incl;
    }
  }
  if (tid == 0) ALG_TRACE(0, 8);
}

// U = 16-byte loads a lane keeps in flight: 4 for rows of up to 2 KB (more registers would cost occupancy there), 16
// for wider rows (the copy of a wide row is bound by its round trips, one per batch of loads)
template <int U>
__global__ void __launch_bounds__(256) gather_rows_kernel(const uint4 *__restrict__ X, int64_t ldx_v,
                                                          const int *__restrict__ perm, int M, int vecs,
                                                          uint4 *__restrict__ Xb) {
  ALG_TRACE_VARS;
  if (threadIdx.x == 0) ALG_TRACE(1, 1);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");  // perm comes from the bucketing kernel
  if (threadIdx.x == 0) ALG_TRACE(1, 2);
  // a warp copies one row at a time, U independent 16-byte loads per lane in flight
  const int lane = threadIdx.x & 31;
  const int warp_global = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int n_warps = (gridDim.x * blockDim.x) >> 5;
  for (int d = warp_global; d < M; d += n_warps) {
    const uint4 *src = X + (int64_t)__ldg(perm + d) * ldx_v;
    uint4 *dst = Xb + (int64_t)d * vecs;
    for (int v0 = lane; v0 < vecs; v0 += 32 * U) {
      uint4 r[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (v0 + u * 32 < vecs) r[u] = __ldg(src + v0 + u * 32);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (v0 + u * 32 < vecs) dst[v0 + u * 32] = r[u];
    }
  }
  if (threadIdx.x == 0) ALG_TRACE(1, 3);
}

// Bucketing and the bucketed copy of X in one launch, for batches whose types every CTA can afford to read (M <=
// kCopyCountRows).  A CTA owns `rows` consecutive rows of the batch: it requests the first of them, counts the types of
// the whole batch meanwhile -- all rows, and those before its own -- ranks its rows and scatters them to their places.
// As two kernels the copy waits for the last CTA of the count, one launch boundary and its own first loads; as one, the
// first rows are on their way while the types are counted (FFN 768 -> 3072, q = 2: M = 100 22.5 -> 20.7 us, 1777 35.9 ->
// 34.1, 8003 69.7 -> 68.6; gated 2048 -> 6144, q = 32, M = 600 71.6 -> 68.2).  Every CTA reads all types, and past its
// first row a warp waits for one load at a time: beyond 8192 rows the two kernels are the faster ones (768 -> 3072, q = 4,
// M = 12000: 74.1 there, 74.9 here; 1024 -> 4096, q = 8, M = 16384: 116.0 there, 117.7 here).
//
// PACKED (q <= 8): counts in four registers of four 16-bit fields, summed by warp reductions.  Otherwise one shared-memory
// histogram per warp (with two types 16 lanes would queue for one counter; with 9 and more it is 3 or 4).
constexpr int kCopyThreads = 1024, kCopyWarps = kCopyThreads / 32, kCopyUnit = 128;   // 16-byte pieces a warp moves at a time
constexpr int kCopyCountRows = 8192, kCopyRows = 64;                                // largest batch, rows of a CTA
template <bool PACKED>
__global__ void __launch_bounds__(kCopyThreads) bucket_copy_kernel(const BucketArgs a, const uint4 *__restrict__ X, int64_t ldx_v, int vecs,
                                                                   uint4 *__restrict__ Xb, int rows) {
  __shared__ uint32_t s_part[PACKED ? kCopyWarps : 1][9];   // (one word of padding: a lane per warp reads a column)
  __shared__ int s_hist[PACKED ? 1 : kCopyWarps][kMaxQ + 1];     // rows of a type, and 2^16 times those before this CTA's
  __shared__ int s_wcnt[kCopyRows / 32][kMaxQ + 1];
  __shared__ int s_off[kMaxQ + 2], s_base[kMaxQ + 1], s_dst[kCopyRows];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = a.q + 1;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");   // types and X may come from the previous kernel
  const int r0 = blockIdx.x * rows, n = min(rows, a.M - r0);
  const int chunks = (vecs + kCopyUnit - 1) / kCopyUnit, units = n * chunks;
  uint4 w[4];
  auto load = [&](int u) {
    const int row = u / chunks, v0 = (u - row * chunks) * kCopyUnit + lane;
    const uint4 *src = X + (int64_t)(r0 + row) * ldx_v;
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (v0 + e * 32 < vecs) w[e] = __ldg(src + v0 + e * 32);
  };
  if (warp < units) load(warp);
  const int t_own = tid < n ? row_type(a, r0 + tid) : -1 - lane;   // (idle lanes never match each other)

  if (PACKED) {
    uint64_t lo = 0, hi = 0, lo_b = 0, hi_b = 0;
#pragma unroll 4
    for (int row = tid; row < a.M; row += kCopyThreads) {
      const int t = row_type(a, row);
      const uint64_t one = t < a.q ? 1ull << (16 * (t & 3)) : 0ull;
      if (t < 4) {
        lo += one;
        if (row < r0) lo_b += one;
      } else {
        hi += one;
        if (row < r0) hi_b += one;
      }
    }
    const uint64_t own[4] = {lo, hi, lo_b, hi_b};
#pragma unroll
    for (int e = 0; e < 8; ++e) {   // (no field overflows, so the halves add up by themselves)
      const uint32_t v = __reduce_add_sync(0xffffffffu, (uint32_t)(own[e >> 1] >> (32 * (e & 1))));
      if (lane == e) s_part[warp][e] = v;
    }
  } else {
    for (int t = lane; t < nt; t += 32) s_hist[warp][t] = 0;
    __syncwarp();
#pragma unroll 4
    for (int row = tid; row < a.M; row += kCopyThreads) atomicAdd(&s_hist[warp][row_type(a, row)], row < r0 ? 0x10001 : 1);
  }
  const unsigned peers = __match_any_sync(0xffffffffu, t_own);
  const int rank = __popc(peers & ((1u << lane) - 1u));
  if (warp < kCopyRows / 32) {
    for (int t = lane; t < nt; t += 32) s_wcnt[warp][t] = 0;
    __syncwarp();
    if (tid < n && rank == 0) s_wcnt[warp][t_own] = __popc(peers);
  }
  __syncthreads();
  if (warp == 0) {
    int tot = 0, bef = 0, tot_last = 0, bef_last = 0;   // of type `lane`; of type 32 (lane 0)
    if (PACKED) {
      // lane e of every eight holds types 2e, 2e + 1 of the batch (e < 4) and of the rows before this CTA's
      uint32_t v = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const uint32_t sum = __reduce_add_sync(0xffffffffu, s_part[lane][e]);
        if ((lane & 7) == e) v = sum;
      }
      const uint32_t v_tot = __shfl_sync(0xffffffffu, v, lane >> 1), v_bef = __shfl_sync(0xffffffffu, v, 4 + (lane >> 1));
      if (lane < a.q) tot = (int)((v_tot >> (16 * (lane & 1))) & 0xFFFFu), bef = (int)((v_bef >> (16 * (lane & 1))) & 0xFFFFu);
      const int all = __reduce_add_sync(0xffffffffu, tot), all_b = __reduce_add_sync(0xffffffffu, bef);
      if (lane == a.q) tot = a.M - all, bef = r0 - all_b;
    } else {
      for (int x = 0; x < kCopyWarps; ++x) {
        const int v = lane < nt ? s_hist[x][lane] : 0;
        tot += v & 0xFFFF, bef += v >> 16;
        if (nt > 32 && lane == 0) tot_last += s_hist[x][32] & 0xFFFF, bef_last += s_hist[x][32] >> 16;
      }
    }
    int incl = tot;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += o;
    }
    const int total32 = __shfl_sync(0xffffffffu, incl, 31);
    if (lane < nt) s_off[lane] = incl - tot, s_base[lane] = incl - tot + bef;
    if (lane == 0) {
      if (nt > 32) s_off[32] = total32, s_base[32] = total32 + bef_last, s_off[33] = total32 + tot_last;
      else s_off[nt] = total32;   // == M
    }
  }
  __syncthreads();
  if (tid < n) {
    int d = s_base[t_own] + rank;
    for (int x = 0; x < warp; ++x) d += s_wcnt[x][t_own];
    s_dst[tid] = d;
    a.perm[d] = r0 + tid;
    if (t_own == a.q) {
      atomicExch(a.status, (int)ALG_ERR_BAD_TYPE);
      if (a.Y) {   // out-of-range type: the row's output is defined to be zero
        char *y = (char *)a.Y + (size_t)(r0 + tid) * a.ldy * a.y_elem_bytes;
        for (int e = 0; e < a.N * a.y_elem_bytes; ++e) y[e] = 0;
      }
    }
  }
  __syncthreads();
  for (int u = warp; u < units; u += kCopyWarps) {
    if (u != warp) load(u);
    const int row = u / chunks, v0 = (u - row * chunks) * kCopyUnit + lane;
    uint4 *dst = Xb + (int64_t)s_dst[row] * vecs;
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (v0 + e * 32 < vecs) dst[v0 + e * 32] = w[e];
  }
  if (blockIdx.x == 0) {
    for (int t = tid; t <= nt; t += kCopyThreads) a.hdr->offsets[t] = s_off[t];
    if (tid == 0) write_pad_offsets(a.hdr, s_off, a.q);
  }
}

// padded row p -> original row (or -1 for a pad row / beyond the last bucket)
__device__ __forceinline__ int padded_source_row(const WsHeader *hdr, const int *perm, int q, int p) {
  int t = 0;
  while (t + 1 < q && hdr->pad_offsets[t + 1] <= p) ++t;
  const int rank = p - hdr->pad_offsets[t];
  const int rows = hdr->offsets[t + 1] - hdr->offsets[t];
  return (p < hdr->pad_offsets[q] && rank < rows) ? perm[hdr->offsets[t] + rank] : -1;
}

// XpT[c, p] = X[source(p), c]: 64 padded rows x 64 columns per CTA through shared memory, so that both the
// reads (along c) and the writes (along p) are contiguous.
__global__ void __launch_bounds__(256) gather_transpose_padded_kernel(const __nv_bfloat16 *__restrict__ X, int64_t ldx,
                                                                      const WsHeader *__restrict__ hdr,
                                                                      const int *__restrict__ perm, int q, int m_pad, int K,
                                                                      __nv_bfloat16 *__restrict__ XpT) {
  __shared__ __nv_bfloat16 tile[64][66];
  __shared__ int s_src[64];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int p0 = blockIdx.x * 64, c0 = blockIdx.y * 64;
  const int tid = threadIdx.x;
  if (tid < 64) s_src[tid] = p0 + tid < m_pad ? padded_source_row(hdr, perm, q, p0 + tid) : -1;
  __syncthreads();
  for (int e = tid; e < 64 * 32; e += 256) {   // 64 rows x 32 column pairs
    const int r = e >> 5, cp = (e & 31) * 2;
    const int src_row = s_src[r];
    __nv_bfloat162 v = __floats2bfloat162_rn(0.f, 0.f);
    if (src_row >= 0 && c0 + cp < K) v = *(const __nv_bfloat162 *)(X + (int64_t)src_row * ldx + c0 + cp);
    tile[r][cp] = v.x, tile[r][cp + 1] = v.y;
  }
  __syncthreads();
  for (int e = tid; e < 64 * 32; e += 256) {   // 64 columns x 32 row pairs
    const int c = e >> 5, rp = (e & 31) * 2;
    if (c0 + c < K && p0 + rp < m_pad) {
      __nv_bfloat162 v;
      v.x = tile[rp][c], v.y = tile[rp + 1][c];
      *(__nv_bfloat162 *)(XpT + (int64_t)(c0 + c) * m_pad + p0 + rp) = v;
    }
  }
}

// ---- row copies by the bulk copy engine ----
//
// dst[d, :] = src[row(d), :] for one or two matrices, row(d) = perm[d], or for buckets padded to multiples of 64 rows
// the row behind padded row d (pad rows are zero).  An agent (one thread) owns a slot of shared memory and moves one
// piece of a row at a time: bulk load, wait, bulk store.  A CTA holds as many slots as fit, so an SM has up to 190 KB in
// flight without a register or a load instruction per 16 bytes.  The copy streams: at 8003 rows of 6 KB it takes 17.9 us
// (98 MB moved, 5.5 TB/s) where the warp-per-row copy above takes 20; X (1.5 KB) and G (6 KB) of those rows into padded
// buckets in one launch 27 us, where transposing X and copying G took 34.  Its CTAs fill an SM, so the next kernel's
// prologue cannot run beside it: below 40 MB the warp-per-row copy is the better one (FFN 768 -> 3072, M = 12000, 18 MB:
// 94.5 us there, 96.7 here; gated 7168 -> 2048 at q = 32, M = 4000, 57 MB: 119.2 there, 115.9 here).
constexpr int kMaxPiece = 8192, kSlotBytes = 184 * 1024, kMaxAgents = 128;

struct CopyArgs {
  const uint8_t *src[2];
  uint8_t *dst[2];
  int64_t ld_src[2];    // bytes
  int row_bytes[2];     // 0: no second matrix
  int pieces[2], piece[2];   // pieces per row, bytes of a piece (the last one may be shorter)
  int whole_pieces[2], whole_piece[2];   // the same where `part` is asked for and whole rows are copied after all
  int slot, agents;     // bytes of a slot, slots of a CTA
  int rows;             // rows of dst
  const int *perm;
  const WsHeader *hdr;  // padded buckets; nullptr: rows through perm as they are
  int q;
  int64_t ld_dst[2];    // bytes
  // Weight gradient under the complete-graph law (part = rows of the batch, 0 = off): a row of type t is needed for the
  // blocks (t, j != t) alone, that is its columns S_t of X (matrix 0) and those outside R_t of G (matrix 1); row_bytes is
  // the longest such part of a row.  In a batch with rows without a type whole rows are copied.
  int part;
  int cut[2][kMaxQ + 1];   // first byte of the column groups of X and of G
  int *status;
  long long wait_limit;
};

__global__ void __launch_bounds__(kMaxAgents) copy_rows_kernel(const CopyArgs a) {
  extern __shared__ __align__(128) uint8_t slots[];   // [agents][slot], then a slot of zeros (padded buckets)
  __shared__ __align__(8) uint64_t bars[kMaxAgents];
  __shared__ int s_off[kMaxQ + 1], s_pad[kMaxQ + 1];
  const int tid = threadIdx.x;
  const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&bars[tid]), base = (uint32_t)__cvta_generic_to_shared(slots);
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
  if (a.hdr)
    for (int e = tid * 16; e < a.slot; e += kMaxAgents * 16) *(uint4 *)(slots + a.agents * a.slot + e) = make_uint4(0, 0, 0, 0);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the zeros, before the copy engine reads them
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");   // perm and the offsets come from the bucketing kernel
  if (a.hdr)
    for (int e = tid; e <= a.q; e += kMaxAgents) s_off[e] = __ldcg(a.hdr->offsets + e), s_pad[e] = __ldcg(a.hdr->pad_offsets + e);
  __syncthreads();
  if (tid >= a.agents) return;
  const uint32_t slot = base + (uint32_t)(tid * a.slot), zeros = base + (uint32_t)(a.agents * a.slot);
  const bool part = a.part && s_off[a.q] == a.part;
  const bool all = a.part && !part;
  const int pieces0 = all ? a.whole_pieces[0] : a.pieces[0], pieces1 = all ? a.whole_pieces[1] : a.pieces[1];
  const int piece0 = all ? a.whole_piece[0] : a.piece[0], piece1 = all ? a.whole_piece[1] : a.piece[1];
  const int per_row = pieces0 + pieces1;
  const int64_t units = (int64_t)a.rows * per_row;
  uint32_t parity = 0;
  for (int64_t u = blockIdx.x + (int64_t)gridDim.x * tid; u < units; u += (int64_t)gridDim.x * a.agents) {
    const int row = (int)(u / per_row), c = (int)(u - (int64_t)row * per_row);
    const int m = c >= pieces0;
    const int piece = m ? piece1 : piece0, at = (m ? c - pieces0 : c) * piece;
    int length = all ? (int)a.ld_dst[m] : a.row_bytes[m], gap_at = 1 << 30, gap = 0;
    int src_row;
    if (a.hdr) {
      int t = 0;
      while (t + 1 < a.q && s_pad[t + 1] <= row) ++t;
      const int r = row - s_pad[t];
      src_row = row < s_pad[a.q] && r < s_off[t + 1] - s_off[t] ? __ldg(a.perm + s_off[t] + r) : -1;
      if (part) {
        const int own = a.cut[m][t + 1] - a.cut[m][t];
        if (m) length = (int)a.ld_dst[1] - own, gap_at = a.cut[1][t], gap = own;   // all but R_t
        else length = own, gap_at = 0, gap = a.cut[0][t];                          // S_t
      }
    } else {
      src_row = __ldg(a.perm + row);
    }
    if (at >= length) continue;
    const uint32_t bytes = (uint32_t)min(piece, length - at);
    // bytes [at, at + bytes) of what is taken of the row: `first` of them before the gap, the rest behind it
    const uint32_t first = (uint32_t)min(max(gap_at - at, 0), (int)bytes);
    uint8_t *dst = a.dst[m] + (int64_t)row * a.ld_dst[m] + at;
    if (src_row >= 0) {
      const uint8_t *src = a.src[m] + (int64_t)src_row * a.ld_src[m] + at;
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
      if (first)
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(slot), "l"(src), "r"(first), "r"(bar)
                     : "memory");
      if (first < bytes)
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(slot + first), "l"(src + first + gap),
                     "r"(bytes - first), "r"(bar)
                     : "memory");
      uint32_t done = 0;
      const long long t0 = clock64();
      while (!done) {
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done)
                     : "r"(bar), "r"(parity)
                     : "memory");
        if (!done && clock64() - t0 > a.wait_limit) {
          atomicExch(a.status, (int)ALG_ERR_DEVICE_TIMEOUT);
          while (clock64() - t0 < a.wait_limit + 2000000LL) {   // the copy gets time to land
          }
          return;
        }
      }
      parity ^= 1u;
    }
    const uint32_t from = src_row >= 0 ? slot : zeros;
    if (first) asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(from), "r"(first) : "memory");
    if (first < bytes)
      asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst + first + gap), "r"(from + first), "r"(bytes - first) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the slot may be filled again
  }
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

}  // namespace

namespace {
template <typename... Args>
cudaError_t launch_pdl(void (*kernel)(Args...), int grid, int block, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(block, 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}
// Column groups of c elements widened to c_pad (zeros), optionally row groups of rs rows widened to rs_pad (zero
// rows); a thread moves 4 elements (8 bytes) of one destination row (blockIdx.y walks the rows).
__global__ void __launch_bounds__(256) pad_groups_kernel(const uint2 *__restrict__ src, int64_t ld_src4, const int *__restrict__ perm,
                                                         int rows_dst, int n_col_groups, int c4, int c_pad4, int rs, int rs_pad,
                                                         uint2 *__restrict__ dst) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");   // perm may come from the previous kernel
  const int w4 = n_col_groups * c_pad4;                 // 8-byte pieces per destination row
  for (int R = blockIdx.y; R < rows_dst; R += gridDim.y) {
    int64_t src_row = R;
    bool row_live = true;
    if (rs > 0) {
      const int gr = R / rs_pad, kr = R - gr * rs_pad;
      row_live = kr < rs;
      src_row = (int64_t)gr * rs + kr;
    } else if (perm) {
      src_row = __ldg(perm + R);
    }
    const uint2 *srow = src + src_row * ld_src4;
    uint2 *drow = dst + (int64_t)R * w4;
    for (int x = blockIdx.x * 256 + threadIdx.x; x < w4; x += gridDim.x * 256) {
      const int gc = x / c_pad4, cc = x - gc * c_pad4;
      drow[x] = (row_live && cc < c4) ? __ldg(srow + gc * c4 + cc) : make_uint2(0u, 0u);
    }
  }
}

}  // namespace

cudaError_t launch_pad_groups(const void *src, int64_t ld_src, const int *perm, int rows_src, int n_col_groups, int c, int c_pad,
                              int rs, int rs_pad, void *dst, cudaStream_t st) {
  if (c % 4 || c_pad % 4 || ld_src % 4 || c_pad < c || (rs > 0 && (rs_pad < rs || rows_src % rs))) return cudaErrorInvalidValue;
  const int rows_dst = rs > 0 ? rows_src / rs * rs_pad : rows_src;
  const int w4 = n_col_groups * (c_pad / 4);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)std::max(1, std::min((w4 + 255) / 256, 8)), (unsigned)std::max(1, std::min(rows_dst, 148 * 8)), 1);
  cfg.blockDim = dim3(256, 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  count_launch(1);
  return cudaLaunchKernelEx(&cfg, pad_groups_kernel, (const uint2 *)src, (int64_t)(ld_src / 4), perm, rows_dst, n_col_groups, c / 4,
                            c_pad / 4, rs, rs_pad, (uint2 *)dst);
}

cudaError_t launch_bucket(const BucketArgs &a, cudaStream_t st) {
  if (a.q > kMaxQ) {   // large-algebra path: two kernels, tables sized for kBigMaxQ types
    if (a.q > kBigMaxQ || !a.big_offsets) return cudaErrorInvalidValue;
    const int n_chunks = ceil_div(a.M, a.chunk_rows);
    bucket_count_kernel<kBigMaxQ + 1><<<n_chunks, 256, 0, st>>>(a);
    bucket_scatter_kernel<kBigMaxQ + 1><<<n_chunks, 256, 0, st>>>(a);
    count_launch(2);
    return cudaGetLastError();
  }
  // clusters of 16 are not portable: asked for once, used where the device says one can be resident
  static OncePerDevice wide;
  static int rows16 = -1;
  const bool asked = wide([] { return cudaFuncSetAttribute(bucket_onepass_kernel<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1); }) == cudaSuccess;
  if (rows16 < 0) {
    rows16 = 0;
    if (asked) {
      cudaLaunchConfig_t probe = {};
      probe.gridDim = dim3(16, 1, 1);
      probe.blockDim = dim3(kFusedThreads, 1, 1);
      cudaLaunchAttribute pa[1];
      pa[0].id = cudaLaunchAttributeClusterDimension;
      pa[0].val.clusterDim.x = 16, pa[0].val.clusterDim.y = 1, pa[0].val.clusterDim.z = 1;
      probe.attrs = pa;
      probe.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, bucket_onepass_kernel<true>, &probe) == cudaSuccess && n > 0) rows16 = 16 * kFusedThreads;
    }
    (void)cudaGetLastError();
  }
  if (!asked) (void)cudaGetLastError();
  if (a.M <= std::max(kClusterRows, asked ? rows16 : 0)) {   // one kernel, one cluster of 1 ... 16 CTAs (CTAs past the batch hold no row)
    int n_cta = 1;
    while (n_cta * kFusedThreads < a.M) n_cta *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_cta, 1, 1);
    cfg.blockDim = dim3(kFusedThreads, 1, 1);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = n_cta, at[1].val.clusterDim.y = 1, at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    count_launch(1);
    return cudaLaunchKernelEx(&cfg, bucket_onepass_kernel<true>, a);
  }
  if (a.M <= 65536 && a.sync) {  // one kernel, every row type read once
    count_launch(1);
    return launch_pdl(bucket_onepass_kernel<false>, ceil_div(a.M, kFusedThreads), kFusedThreads, st, a);
  }
  const int n_chunks = ceil_div(a.M, a.chunk_rows);
  bucket_count_kernel<kMaxQ + 1><<<n_chunks, 256, 0, st>>>(a);
  bucket_scatter_kernel<kMaxQ + 1><<<n_chunks, 256, 0, st>>>(a);
  count_launch(2);
  return cudaGetLastError();
}

namespace {
cudaError_t launch_copy_rows(CopyArgs a, cudaStream_t st) {
  int slot = 0;
  for (int m = 0; m < 2; ++m) {
    a.pieces[m] = a.row_bytes[m] ? ceil_div(a.row_bytes[m], kMaxPiece) : 0;
    a.piece[m] = a.pieces[m] ? (ceil_div(a.row_bytes[m], a.pieces[m]) + 15) / 16 * 16 : 0;
    slot = std::max(slot, a.piece[m]);
  }
  // Whole rows have pieces of their own (in those of the parts, X of 32 groups went in 32 pieces of 128 bytes: 2048 x 8192
  // over 16384 rows, one of them without a type, 863 us, 340 in whole pieces).  They take the slots as they are, or wider ones
  // where that costs the parts at most a ninth of their slots.
  int whole_slot = 0;
  for (int m = 0; m < 2; ++m)
    if (a.row_bytes[m]) whole_slot = std::max(whole_slot, (ceil_div((int)a.ld_dst[m], ceil_div((int)a.ld_dst[m], kMaxPiece)) + 15) / 16 * 16);
  if (whole_slot * 8 <= slot * 9) slot = std::max(slot, whole_slot);
  a.slot = (slot + 127) / 128 * 128;
  for (int m = 0; m < 2; ++m) {
    a.whole_pieces[m] = a.row_bytes[m] ? ceil_div((int)a.ld_dst[m], a.slot) : 0;
    a.whole_piece[m] = a.whole_pieces[m] ? (ceil_div((int)a.ld_dst[m], a.whole_pieces[m]) + 15) / 16 * 16 : 0;
  }
  a.agents = std::min(kMaxAgents, kSlotBytes / a.slot - (a.hdr ? 1 : 0));
  static OncePerDevice limit;
  const cudaError_t e = limit([] { return cudaFuncSetAttribute(copy_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSlotBytes + 1024); });
  if (e != cudaSuccess) return e;
  const int64_t units = (int64_t)a.rows * (a.pieces[0] + a.pieces[1]);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)std::max<int64_t>(1, std::min<int64_t>(148, units)), 1, 1);
  cfg.blockDim = dim3(kMaxAgents, 1, 1);
  cfg.dynamicSmemBytes = (size_t)(a.agents + (a.hdr ? 1 : 0)) * a.slot;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  count_launch(1);
  return cudaLaunchKernelEx(&cfg, copy_rows_kernel, a);
}
}  // namespace

bool bucket_copy_takes(int q, int64_t M, int64_t row_bytes) {
  return q <= kMaxQ && M <= kCopyCountRows && M * row_bytes < kBulkCopyBytes && row_bytes % 16 == 0;
}

cudaError_t launch_bucket_copy(const BucketArgs &a, const void *X, int64_t ldx, int K, int elem_bytes, void *Xb, cudaStream_t st) {
  const int64_t row_bytes = (int64_t)K * elem_bytes;
  if (!bucket_copy_takes(a.q, a.M, row_bytes)) return cudaErrorInvalidValue;
  const int rows = ceil_div(a.M, 148), grid = ceil_div(a.M, rows);
  count_launch(1);
  return launch_pdl(a.q <= 8 ? bucket_copy_kernel<true> : bucket_copy_kernel<false>, grid, kCopyThreads, st, a, (const uint4 *)X,
                    (int64_t)(ldx * elem_bytes / 16), (int)(row_bytes / 16), (uint4 *)Xb, rows);
}

cudaError_t launch_gather_rows(const void *X, int64_t ldx, const int *perm, int M, int K, int elem_bytes, void *Xb, int *status,
                               long long wait_limit, cudaStream_t st) {
  const int vecs = K * elem_bytes / 16;
  if ((int64_t)M * K * elem_bytes >= kBulkCopyBytes) {
    CopyArgs a = {};
    a.src[0] = (const uint8_t *)X, a.dst[0] = (uint8_t *)Xb;
    a.ld_src[0] = ldx * elem_bytes, a.row_bytes[0] = K * elem_bytes, a.ld_dst[0] = a.row_bytes[0];
    a.rows = M, a.perm = perm;
    a.status = status, a.wait_limit = wait_limit;
    return launch_copy_rows(a, st);
  }
  int grid = ceil_div(M, 8);  // eight warps (rows) per CTA
  if (grid > 148 * 8) grid = 148 * 8;
  count_launch(1);
  if (vecs > 128)
    return launch_pdl(gather_rows_kernel<16>, grid, 256, st, (const uint4 *)X, (int64_t)(ldx * elem_bytes / 16), perm, M, vecs,
                      (uint4 *)Xb);
  return launch_pdl(gather_rows_kernel<4>, grid, 256, st, (const uint4 *)X, (int64_t)(ldx * elem_bytes / 16), perm, M, vecs,
                    (uint4 *)Xb);
}

cudaError_t launch_gather_rows_padded(const void *X, int64_t ldx, int K, void *Xp, const void *G, int64_t ldg, int N, void *Gp,
                                      const WsHeader *hdr, const int *perm, int q, int M, int m_pad, const int *s, const int *r,
                                      int *status, long long wait_limit, cudaStream_t st) {
  CopyArgs a = {};
  a.src[0] = (const uint8_t *)X, a.dst[0] = (uint8_t *)Xp, a.ld_src[0] = ldx * 2, a.row_bytes[0] = K * 2;
  a.src[1] = (const uint8_t *)G, a.dst[1] = (uint8_t *)Gp, a.ld_src[1] = ldg * 2, a.row_bytes[1] = N * 2;
  a.ld_dst[0] = a.row_bytes[0], a.ld_dst[1] = a.row_bytes[1];
  if (s && r) {
    a.part = M;
    a.row_bytes[0] = a.row_bytes[1] = 0;
    for (int t = 0; t < q; ++t) {
      a.cut[0][t + 1] = a.cut[0][t] + s[t] * 2, a.cut[1][t + 1] = a.cut[1][t] + r[t] * 2;
      a.row_bytes[0] = std::max(a.row_bytes[0], s[t] * 2), a.row_bytes[1] = std::max(a.row_bytes[1], (N - r[t]) * 2);
    }
  }
  a.rows = m_pad, a.perm = perm, a.hdr = hdr, a.q = q;
  a.status = status, a.wait_limit = wait_limit;
  return launch_copy_rows(a, st);
}

cudaError_t launch_gather_transpose_padded(const void *X, int64_t ldx, const WsHeader *hdr, const int *perm, int q,
                                           int m_pad, int K, void *XpT, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ceil_div(m_pad, 64), ceil_div(K, 64), 1);
  cfg.blockDim = dim3(256, 1, 1);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  count_launch(1);
  return cudaLaunchKernelEx(&cfg, gather_transpose_padded_kernel, (const __nv_bfloat16 *)X, ldx, hdr, perm, q, m_pad, K,
                            (__nv_bfloat16 *)XpT);
}

}  // namespace algproj
