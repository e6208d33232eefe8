// How the hidden rows of a one-launch FFN get from the CTAs that compute them to the CTAs that need them: the data is
// its own flag.
//
// The handle owns two buffers of bf16 hidden rows and a turn count.  A launch writes its hidden values into the buffer
// of its turn's parity, where every 16-bit half reads 0xFFFF beforehand; a consumer loads what it needs and loads again
// whatever still reads 0xFFFF (a NaN pattern a stored value never has: conversions give the canonical 0x7FFF, and
// `exch_value` makes sure).  So a value travels in one store and one load, and a CTA waits for the values it needs
// only -- no fence, no arrival counter to add to and poll, no wait for the slowest CTA of the grid.
// Per layer in a graph of layers: 768 -> 3072 -> 768 at q = 2, one row, 9.2 -> 7.5 us; gated 2048 -> 6144 at q = 32, one
// row, 9.8 -> 8.3 us, four rows 17.8 -> 16.7 us.
// Where every CTA reads the whole hidden state (ffn_decode.cu) loading it over and over would get in the way of the
// values themselves (96 CTAs, 8 rows of 3072: 12.1 us a layer): there one thread of a CTA waits for a hint first, a count
// of the CTAs whose values are on their way.  The hint is not ordered behind the values, so it costs no fence; it says
// when to look, the values say what is there.
//
// Meanwhile every launch fills the OTHER buffer (the rows its predecessor used) with 0xFFFF for its successor.  All of it
// happens behind griddepcontrol.wait, so the predecessor is done with that buffer, and the successor starts reading only
// after this launch is complete.  The turn count grows by exactly 2^20 per launch -- every CTA adds its share once all
// its threads have asked for the turn -- so count >> 20 is the launch's turn whenever a CTA of it asks, whatever the
// grid.  A launch that gave up leaves behind the same state as any other.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace algproj {

constexpr int kExchHeader = 256;         // ExchHead, then the two buffers
constexpr unsigned kExchTurn = 1u << 20;

struct ExchHead {
  unsigned long long turns;   // turn << 20
  int rows[2];                // rows the last launch that used a buffer wrote there
  unsigned hints[2];          // CTAs of the turn whose values are on their way
};

struct ExchTurn {
  unsigned parity;
  int stale_rows;   // rows of the other buffer to clear
};
__device__ __forceinline__ ExchTurn exch_turn(const uint8_t *exch) {
  uint4 h;   // (the turn's parity is in the low word of the count; everything of the head in one round trip)
  asm volatile("ld.relaxed.gpu.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(h.x), "=r"(h.y), "=r"(h.z), "=r"(h.w) : "l"(exch) : "memory");
  const unsigned parity = (h.x >> 20) & 1u;
  return {parity, (int)(parity ? h.z : h.w)};
}
// One thread of the CTA, after a CTA barrier behind exch_turn.
__device__ __forceinline__ void exch_leave(uint8_t *exch) {
  const unsigned share = kExchTurn / gridDim.x;
  const unsigned long long add = blockIdx.x ? share : kExchTurn - share * (gridDim.x - 1);
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(exch), "l"(add) : "memory");
}
// This CTA's part of the buffer the next launch will use, and a note of the rows this launch writes.
__device__ __forceinline__ void exch_clear(uint8_t *exch, int exch_bytes, const ExchTurn &turn, int row_bytes, int rows) {
  const int bytes = min(turn.stale_rows * row_bytes, exch_bytes);
  uint8_t *buf = exch + kExchHeader + (turn.parity ^ 1u) * (unsigned)exch_bytes;
  for (int e = (blockIdx.x + threadIdx.x * gridDim.x) * 16; e < bytes; e += gridDim.x * blockDim.x * 16)
    *(uint4 *)(buf + e) = make_uint4(~0u, ~0u, ~0u, ~0u);
  if (blockIdx.x == 0 && threadIdx.x == 0) ((ExchHead *)exch)->rows[turn.parity] = rows, ((ExchHead *)exch)->hints[turn.parity ^ 1u] = 0u;
}
// "My values are on their way": not ordered behind them, so that it costs no fence, and no proof that they are there.
__device__ __forceinline__ void exch_hint(uint8_t *exch, const ExchTurn &turn) {
  asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(&((ExchHead *)exch)->hints[turn.parity]) : "memory");
}
__device__ __forceinline__ bool exch_hinted(const uint8_t *exch, const ExchTurn &turn, int ctas) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&((const ExchHead *)exch)->hints[turn.parity]) : "memory");
  return v >= (unsigned)ctas;
}
// Two bf16 values on their way into the buffer.
__device__ __forceinline__ uint32_t exch_value(uint32_t v) {
  if ((v & 0xFFFFu) == 0xFFFFu) v ^= 0x8000u;
  if ((v >> 16) == 0xFFFFu) v ^= 0x80000000u;
  return v;
}
__device__ __forceinline__ void exch_store(void *dst, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(dst), "r"(exch_value(v)) : "memory");
}
__device__ __forceinline__ void exch_store4(void *dst, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(dst), "r"(exch_value(a)), "r"(exch_value(b)),
               "r"(exch_value(c)), "r"(exch_value(d))
               : "memory");
}
__device__ __forceinline__ uint4 exch_load4(const void *src) {
  uint4 v;
  asm volatile("ld.relaxed.gpu.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(src) : "memory");
  return v;
}
__device__ __forceinline__ unsigned short exch_load(const void *src) {
  unsigned short v;
  asm volatile("ld.relaxed.gpu.global.u16 %0, [%1];" : "=h"(v) : "l"(src) : "memory");
  return v;
}
// Single values, and pairs of them.
__device__ __forceinline__ void exch_store1(void *dst, float z) {
  unsigned short v = __bfloat16_as_ushort(__float2bfloat16_rn(z));
  if (v == 0xFFFFu) v = 0x7FFFu;
  asm volatile("st.relaxed.gpu.global.u16 [%0], %1;" ::"l"(dst), "h"(v) : "memory");
}
__device__ __forceinline__ uint32_t exch_load2(const void *src) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(src) : "memory");
  return v;
}
__device__ __forceinline__ bool exch_ready2(uint32_t v) { return (v & 0xFFFFu) != 0xFFFFu && v < 0xFFFF0000u; }
// (a producer stores whole 32-bit words, so a word is there or not)
__device__ __forceinline__ bool exch_ready(const uint4 &v) { return v.x != ~0u && v.y != ~0u && v.z != ~0u && v.w != ~0u; }

}  // namespace algproj
