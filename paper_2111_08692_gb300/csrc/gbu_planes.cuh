// gbu_planes.cuh -- UTF-8 validation of a lane's 32 consecutive bytes on bit planes.
//
// Paper Section 3's rules 1-6, with one 32-bit register per bit of a byte: bit i of plane b is bit
// b of byte i.  A test that the byte-wise form (gbu_chunk.cuh) makes for four bytes at a time is
// then one operation for 32, and the shifts between neighbouring bytes are register shifts.  The
// transposition costs 16 PRMT (bytes i, i + 8, i + 16, i + 24 into one register) and 48 operations
// (three stages of an 8 x 8 bit transposition), 12 of them left shifts that the multiply pipe can
// do; the rules cost about 35.  The byte-wise form took 80 (two-byte text), 139 (three-byte) and 163
// (four-byte) warp instructions per 16 bytes and lane.
#pragma once

#include <stdint.h>

#include "gbu_device.cuh"

namespace gbu {

// Swaps the bits outside m of a with the bits inside m of b, S places apart (one step of a bit
// transposition).
template <int S>
__device__ __forceinline__ void swap_bits(uint32_t &a, uint32_t &b, uint32_t m) {
  const uint32_t x = (a & m) | ((b << S) & ~m);
  const uint32_t y = ((a >> S) & m) | (b & ~m);
  a = x;
  b = y;
}

// b[k], k = 0..7: the planes of the 32 bytes W.
__device__ __forceinline__ void bit_planes(const uint32_t (&W)[8], uint32_t (&b)[8]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {  // register k: bytes k, k + 8, k + 16, k + 24
    const uint32_t p = __byte_perm(W[h], W[h + 2], 0x5140), q = __byte_perm(W[h], W[h + 2], 0x7362);
    const uint32_t r = __byte_perm(W[h + 4], W[h + 6], 0x5140), s = __byte_perm(W[h + 4], W[h + 6], 0x7362);
    b[4 * h] = __byte_perm(p, r, 0x5410);
    b[4 * h + 1] = __byte_perm(p, r, 0x7632);
    b[4 * h + 2] = __byte_perm(q, s, 0x5410);
    b[4 * h + 3] = __byte_perm(q, s, 0x7632);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) swap_bits<4>(b[k], b[k + 4], 0x0F0F0F0Fu);
#pragma unroll
  for (int k = 0; k < 8; k += 4) {
    swap_bits<2>(b[k], b[k + 2], 0x33333333u);
    swap_bits<2>(b[k + 1], b[k + 3], 0x33333333u);
  }
#pragma unroll
  for (int k = 0; k < 8; k += 2) swap_bits<1>(b[k], b[k + 1], 0x55555555u);
}

// The continuation bytes that leading bytes in the last three bytes of w want after it: bit i: the
// i-th byte after w.
__device__ __forceinline__ uint32_t wanted_after(uint32_t w) {
  const uint32_t g = w & (w << 1) & 0x80808080u, gE = g & (w << 2), gF = gE & (w << 3);
  return (g >> 31) | (gE >> 31 << 1) | ((gE >> 23) & 1u) | (gF >> 31 << 2) | ((gF >> 23) & 1u) << 1 | ((gF >> 15) & 1u);
}

// Nonzero where the 32 bytes W break a rule.  exchange: takes the continuation bytes that W's leading
// bytes want after it (as wanted_after) and gives those that leading bytes before W want in it;
// next: the word after W (its first byte is looked at).  A sequence cut by the end is flagged by
// the lane that holds the byte after it.  high: the lane has a byte >= E0.  All lanes of a warp.
template <class Exchange>
__device__ __forceinline__ uint32_t utf8_plane_errors(const uint32_t (&W)[8], Exchange exchange, uint32_t next,
                                                      bool &high) {
  uint32_t b[8];
  bit_planes(W, b);
  const uint32_t g2 = b[7] & b[6], g3 = g2 & b[5];  // bytes >= C0, >= E0
  const uint32_t g4 = g3 & b[4];                    // >= F0
  high = g3 != 0;
  // rules 1-3: a byte is a continuation byte exactly when a leading byte 1, 2 or 3 back wants it
  const uint32_t wanted = exchange((g2 >> 31) | (g3 >> 30) | (g4 >> 29));
  uint32_t err = (wanted | g2 << 1 | g3 << 2 | g4 << 3) ^ (b[7] & ~b[6]);
  // rules 4-6 (and 1 for F8-FF): with the structure right, only these leading bytes and second
  // bytes can be out of range: C0, C1; E0 then 80-9F; ED then A0-BF; F0 then 80-8F; F4 then 90-BF;
  // F5-FF
  const uint32_t zero = ~(b[3] | b[2] | b[1]);                          // low nibble 0 or 1
  const uint32_t n5 = b[5] >> 1 | ((next << 26) & 0x80000000u);         // bit 5 of the byte after
  const uint32_t e = g3 & ~b[4];                                        // E0-EF
  err |= g2 & ~b[5] & ~b[4] & zero;                                     // C0, C1
  err |= e & zero & ~b[0] & ~n5;                                        // E0
  err |= e & (b[3] & b[2] & ~b[1]) & b[0] & n5;                         // ED
  if (__any_sync(0xffffffffu, g4 != 0)) {
    const uint32_t n54 = n5 | b[4] >> 1 | ((next << 27) & 0x80000000u);  // the byte after is >= 90
    err |= g4 & zero & ~b[0] & ~n54;                                     // F0
    err |= g4 & (~b[3] & b[2] & ~b[1]) & ~b[0] & n54;                    // F4
    err |= g4 & (b[3] | (b[2] & (b[1] | b[0])));                         // F5-FF
  }
  return err;
}

// The same for a region without a byte >= E0, four bytes at a time and without the transposition:
// false (for the whole warp) if it has one, else err as above.  76 operations per lane against the
// planes' 110, and no word after W.
template <class Exchange>
__device__ __forceinline__ bool utf8_two_byte_errors(const uint32_t (&W)[8], Exchange exchange, uint32_t &err) {
  uint32_t prev = 0, e0 = 0, first = 0, wrong = 0, low = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const uint32_t w = W[k], t = w << 1, lead = w & t;  // bit 7 of a byte: >= C0
    e0 |= lead & (w << 2);
    const uint32_t wanted = __funnelshift_l(prev, lead, 8);
    if (k == 0) first = wanted;
    else wrong |= wanted ^ (w & ~t);
    low |= lead & ~((w & 0x1E1E1E1Eu) + 0x7E7E7E7Eu);  // C0, C1 (bit 5 is clear)
    prev = lead;
  }
  if (__any_sync(0xffffffffu, (e0 & 0x80808080u) != 0)) return false;
  // continuation bytes wanted from before the lane, one bit each, to bit 7 of the first bytes
  const uint32_t before = (exchange(prev >> 31) * 0x00204080u) & 0x00808080u;
  wrong |= ((first & 0x80808080u) | before) ^ (W[0] & ~(W[0] << 1));
  err = (wrong | low) & 0x80808080u;
  return true;
}

}  // namespace gbu
