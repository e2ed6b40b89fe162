// Two-word keys (k from 33 to 64): the slot, its hash and claim, and keys cut
// from the packed stream, shared by the direct and the binned insert.
#pragma once

#include "dbg_internal.cuh"

namespace dbg {

struct WideSlot {
  unsigned long long w0;  // key bits 64..127 (kEmpty: empty slot)
  unsigned long long w1;  // key bits 0..63
  uint32_t cnt[4];
};
static_assert(sizeof(WideSlot) == 32, "one sector per slot");

constexpr int kWideTile = 128;        // reads per tile
constexpr int kWideWinBytes = 16384;  // staged bytes per tile (wider tiles read global memory)

// A multilinear hash (Dietzfelbinger's multiply-add-shift with fixed odd
// multipliers): its leading bits choose the home slot.
__device__ __forceinline__ uint64_t wide_hash(uint64_t hi, uint64_t lo) {
  return hi * 0x9E3779B97F4A7C15ull + lo * 0xD1B54A32D192ED03ull;
}
__device__ __forceinline__ uint64_t wide_home(uint64_t hi, uint64_t lo, uint64_t n_slots) {
  return __umul64hi(wide_hash(hi, lo), n_slots);
}

// Atomic 128-bit compare-and-swap of a slot's key words; returns the old pair.
__device__ __forceinline__ void cas128(WideSlot *s, uint64_t c0, uint64_t c1, uint64_t v0,
                                       uint64_t v1, uint64_t &o0, uint64_t &o1) {
  asm volatile(
      "{\n"
      ".reg .b128 c, v, d;\n"
      "mov.b128 c, {%2, %3};\n"
      "mov.b128 v, {%4, %5};\n"
      "atom.relaxed.gpu.global.cas.b128 d, [%6], c, v;\n"
      "mov.b128 {%0, %1}, d;\n"
      "}\n"
      : "=l"(o0), "=l"(o1)
      : "l"(c0), "l"(c1), "l"(v0), "l"(v1), "l"(&s->w0)
      : "memory");
}

// Both key words of a slot in one single-copy atomic load.
__device__ __forceinline__ void load128(const WideSlot *s, uint64_t &w0, uint64_t &w1) {
  asm volatile(
      "{\n"
      ".reg .b128 d;\n"
      "ld.relaxed.gpu.global.b128 d, [%2];\n"
      "mov.b128 {%0, %1}, d;\n"
      "}\n"
      : "=l"(w0), "=l"(w1)
      : "l"(&s->w0)
      : "memory");
}

// Slot of key (hi, lo), claimed if absent; false after max_probes slots.
__device__ __forceinline__ bool wide_find_or_claim(WideSlot *t, uint64_t n_slots,
                                                   uint32_t max_probes, uint64_t hi, uint64_t lo,
                                                   uint64_t &slot,
                                                   bool *claimed = nullptr) {
  uint64_t s = wide_home(hi, lo, n_slots);
  for (uint32_t i = 0; i < max_probes; ++i) {
    uint64_t w0, w1;
    load128(&t[s], w0, w1);
    if (w0 == kEmpty) {
      cas128(&t[s], kEmpty, 0ull, hi, lo, w0, w1);
      if (w0 == kEmpty) {
        if (claimed) *claimed = true;
        w0 = hi;
        w1 = lo;
      }
    }
    if (w0 == hi && w1 == lo) {
      slot = s;
      return true;
    }
    if (++s == n_slots) s = 0;
  }
  return false;
}

__device__ __forceinline__ uint64_t rev_pairs(uint64_t x) {
  x = __brevll(x);
  return ((x >> 1) & 0x5555555555555555ull) | ((x & 0x5555555555555555ull) << 1);
}

// Key (hi, lo) of m bases (32 <= m <= 63) whose little-endian 2-bit stream
// starts at bit `sh` (< 64) of the words w0, w1, w2.
__device__ __forceinline__ void wide_key(uint64_t w0, uint64_t w1, uint64_t w2, uint32_t sh,
                                         int m, uint64_t &hi, uint64_t &lo) {
  const uint64_t x_lo = sh ? (w0 >> sh) | (w1 << (64u - sh)) : w0;  // bases 0..31
  const uint64_t x_hi = sh ? (w1 >> sh) | (w2 << (64u - sh)) : w1;  // bases 32..63
  const uint64_t a = rev_pairs(x_lo), b = rev_pairs(x_hi);          // base 0 on top of a
  const int s = 128 - 2 * m;                                        // 2 .. 64
  if (s == 64) {
    hi = 0;
    lo = a;
  } else {
    hi = a >> s;
    lo = (b >> s) | (a << (64 - s));
  }
}

// Little-endian 64-bit word of the stream at byte `at`, bytes past nbytes as 0.
__device__ __forceinline__ uint64_t word_at(const uint8_t *packed, uint64_t nbytes, uint64_t at) {
  uint64_t w = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (at + i < nbytes) w |= (uint64_t)__ldg(packed + at + i) << (8 * i);
  return w;
}

}  // namespace dbg
