// gbu_wide_utf8.cuh -- the UTF-8 -> UTF-16LE codec (validating) of the wide partition loop
// (gbu_wide.cuh): a lane validates and converts 32 consecutive bytes.
//
// Paper Section 3 defines both formats; Section 5 states that transcoding validates.  A lane
// treats its 32 bytes as eight 32-bit words and works on four byte positions at a time:
//   * classification and rules 1-6 as in gbu_chunk.cuh (lead and continuation flags in bit 7
//     of each byte; structure by funnel-shifted lead flags; values by word-level byte tests of
//     the special leading bytes);
//   * decoding keeps the output word of every position as two byte planes, its high byte H and
//     low byte L, each computed for four positions per operation from the position's byte and
//     the one or two bytes after it (S1, S2 = the byte stream moved by one and two positions):
//       two bytes   110abcde 10fghijk      -> H = 00000abc,  L = de fghijk
//       three bytes 1110abcd 10efghij 10k.. -> H = abcd efgh, L = ij k.....
//     and for a four-byte sequence the two surrogates: the leading byte gives the first (D7C0 +
//     the code point's bits 20-10), the byte after it the second (DC00 + bits 9-0), which seen
//     from there is the three-byte form's expression with other upper bits, so that a position
//     never gives more than one word (with both at the leading byte and the second one stored
//     under its own predicate: 512 MiB of emoji text 569 us, now 525; of mixed text 769, now 721);
//   * PRMT interleaves H and L into 16-bit words, which go to consecutive places of the staging
//     buffer, through 32-bit shared-memory addresses.  Every position stores its word, whether it
//     is a leading byte's or not, at the place the next leading byte's word takes: what a
//     continuation byte writes is overwritten by the lane's next leading byte.  Only the lane's
//     last positions, which no leading byte may follow, store under a predicate.  The places of a word's four positions are byte dot products of its leading
//     flags with one to four ones, added to the running address: the multiply pipe makes them,
//     and of the test, store and add that every position cost before, on the integer pipe that
//     bounds the kernel, only the store is left (CJK: 756 to 723 warp instructions per KiB; 1 GiB
//     of Latin 809 to 789 us, 100 MB of CJK 118 to 115 us).  Past the first error a lane can
//     overwrite the next lane's first word: that word lies past the valid prefix.
// A lane that breaks a rule reports its start; the last CTA turns the smallest one into the
// exact offset and kind (resolve_utf8_error).
#pragma once

#include <stdint.h>

#include "gbu_codec_utf8.cuh"
#include "gbu_wide.cuh"

namespace gbu {

// Byte mask (0xFF where bit 7 of the byte of x is set).
__device__ __forceinline__ uint32_t byte_mask(uint32_t x) { return prmt(x, 0u, 0xBA98u); }

// Bits 4k .. 4k + 3 of m as bit 7 of each byte: bit j of the nibble times 1 << (7 + 7j) lands at bit
// 8j + 7, and no two terms of the product meet.
__device__ __forceinline__ uint32_t nibble_flags(uint32_t m, int k) {
  return (((m >> (4 * k)) & 0xFu) * 0x10204080u) & 0x80808080u;
}

// The 16-bit word of position j (0..3) from the byte planes L and H.
__device__ __forceinline__ uint32_t plane_word(uint32_t L, uint32_t H, int j) {
  return __byte_perm(L, H, (uint32_t)(j | ((4 + j) << 4)));
}

struct Utf8ToUtf16Wide {
  using Out = uint16_t;
  using Narrow = Utf8ToUtf16;
  // A region yields at most 1024 words (one per position), plus 7 words of alignment offset and the
  // place after the last word, which continuation bytes may write to after an error.
  static constexpr uint32_t WSTAGE = 1024 + 48;
  static_assert(1024 + 7 + 1 <= WSTAGE, "staging buffer too small");
  static constexpr bool CARRY = true;  // a lane's last byte can give a word to the next lane
  __device__ __forceinline__ static bool gives_word(uint32_t w) { return w >= 0xF0000000u; }

  static constexpr uint32_t F_NONASCII = Narrow::F_NONASCII;
  static constexpr uint32_t F_C2 = Narrow::F_C2;
  static constexpr uint32_t F_C3 = Narrow::F_C3;
  static constexpr uint32_t F_C4 = Narrow::F_C4;

  static constexpr uint32_t ASCII_MASK = 0x80808080u;  // nonzero in a word: a byte >= 0x80
  static constexpr uint32_t LANE_UNITS = 32;            // words out of 32 ASCII bytes
  static constexpr uint32_t WREGION_UNITS = 1024;       // words out of an all-ASCII region
  static constexpr uint32_t WDIRECT_ALIGN = 8;          // its lanes store 32 words (64 bytes) each

  __device__ __forceinline__ static bool wascii_region(uint32_t, uint32_t rflags) { return rflags == 0; }

  // Rule 2 across the region's start: a leading byte in the word before it that wants
  // continuation bytes inside it (the region's bytes are all ASCII).  Lane 0 only.
  __device__ __forceinline__ static void check_prev_lead(uint32_t prev, long long c, unsigned long long &err_pos) {
    const Flags8 fp = classify8(prev);
    const uint32_t req = __funnelshift_l(fp.geC0, 0u, 8) | __funnelshift_l(fp.geE0, 0u, 16) |
                         __funnelshift_l(fp.geF0, 0u, 24);
    if (req && (unsigned long long)c < err_pos) err_pos = (unsigned long long)c;
  }

  // An all-ASCII region inside the buffer whose output starts at dst, 16-byte aligned: each
  // lane widens its 32 bytes and stores them with two 32-byte stores (or four 16-byte ones)
  // (Section 4's ASCII path).  The 32-byte stores carry an evict-first L2 policy: the output,
  // twice the input, would otherwise push out of L2 the input lines the count pass has read
  // for the conversion to read again.
  __device__ __forceinline__ static void wascii_direct(uint16_t *dst, const uint32_t W[8], uint32_t prev, long long c,
                                                       unsigned long long &err_pos) {
    const int lane = threadIdx.x & 31;
    if (lane == 0) check_prev_lead(prev, c, err_pos);
    uint4 q[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      q[i] = make_uint4(__byte_perm(W[2 * i], 0, 0x4140), __byte_perm(W[2 * i], 0, 0x4342),
                        __byte_perm(W[2 * i + 1], 0, 0x4140), __byte_perm(W[2 * i + 1], 0, 0x4342));
    uint4 *d = reinterpret_cast<uint4 *>(dst) + 4 * lane;
    if (((uintptr_t)dst & 31) == 0) {
      const uint64_t pol = l2_policy_last_use();
      st_global_32B_hint(d, q[0], q[1], pol);
      st_global_32B_hint(d + 2, q[2], q[3], pol);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) d[i] = q[i];
    }
  }

  // UTF-16 words of the lane's 32 bytes (one per byte that is not a continuation byte, one
  // more per byte F0-FF: the length formula) and the leading-byte classes present.
  __device__ __forceinline__ static uint32_t wcount(const Params &p, const uint32_t W[8], long long c, bool edge,
                                                    uint32_t &flags) {
    uint32_t any = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) any |= W[k];
    if (!edge && (any & 0x80808080u) == 0) {  // all ASCII
      flags = 0;
      return 32;
    }
    // per byte, as bit 7: not a continuation byte (10xxxxxx), >= C0, >= E0 and >= F0.  Byte dot
    // products with 0x01 weights (FMA pipe) add 0x80 per flag; the leading-byte classes follow
    // from the sums (C0-DF present when there are more bytes >= C0 than >= E0, and so on), so
    // the integer ALU does four logic operations per word
    uint32_t an = 0, aG = 0, aE = 0, aF = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint32_t w = W[k], s1 = w * 2u, s2 = w * 4u, s3 = w * 8u;
      const uint32_t vm = edge ? byte_range_mask(c + 4 * k, p.off0, (long long)p.vbytes) : 0x80808080u;
      const uint32_t ge = w & s1 & vm;  // >= C0
      const uint32_t gE = ge & s2;      // >= E0
      const uint32_t f0 = gE & s3;      // >= F0
      an = __dp4a((~w | s1) & vm, 0x01010101u, an);
      aG = __dp4a(ge, 0x01010101u, aG);
      aE = __dp4a(gE, 0x01010101u, aE);
      aF = __dp4a(f0, 0x01010101u, aF);
    }
    flags = F_NONASCII | (aG > aE ? F_C2 : 0u) | (aE > aF ? F_C3 : 0u) | (aF ? F_C4 : 0u);
    return (an + aF) >> 7;
  }

  // Validates the lane's 32 bytes W[1..8] (W[0] the word before, W[9] the word after) of a
  // region that lies inside the buffer and whose output fits the staging buffer, and stages
  // their words from shared address sa on; returns nonzero when a rule is broken.  H2 / H3 /
  // H4: leading bytes C0-DF / E0-EF / F0-FF occur in the region or in bytes 1-3 of the word
  // before it (the code for an absent class is left out).  Each non-continuation byte and each byte
  // after a leading byte F0-FF takes the place of one word, the count the count pass gave the lane.
  // NW: the words of the lane (W[1..NW]).  EXACT: the lane may hold bytes outside its string (m: one
  // bit per byte inside) and other strings' words lie next to the lane's, so every word is stored
  // under its predicate and a lane never writes past the words it counts.  U32: one 32-bit unit (the
  // code point) per leading byte instead, its third byte in a plane of its own.
  template <bool H2, bool H3, bool H4, int NW = 8, bool EXACT = false, bool U32 = false>
  __device__ __forceinline__ static uint32_t wconvert_fast(const uint32_t (&W)[NW + 2], uint32_t sa, uint32_t m = 0) {
    // with a single class present, every byte >= C0 is a leading byte of that class; without
    // H4 there is no byte >= F0
    constexpr bool ONE = (int)H2 + (int)H3 + (int)H4 == 1;
    uint32_t bad = 0;
    // lead flags of the word before (bytes 1-3 reach into the lane's bytes)
    uint32_t pg, pE = 0, pF = 0;
    {
      const uint32_t w = W[0];
      pg = w & (w << 1) & 0x80808080u;
      if (H3 || H4) pE = ONE ? pg : pg & (w << 2);
      if (H4) pF = ONE ? pg : pE & (w << 3);
    }
#pragma unroll
    for (int k = 1; k <= NW; ++k) {
      const uint32_t w = W[k], wn = W[k + 1];
      const uint32_t s1 = w << 1;
      const uint32_t g = w & s1 & 0x80808080u;     // >= C0
      const uint32_t n = (~w | s1) & 0x80808080u;  // not a continuation byte
      uint32_t gE = 0, gF = 0;
      if (H3 || H4) gE = ONE ? g : g & (w << 2);   // >= E0
      if (H4) gF = ONE ? g : gE & (w << 3);        // >= F0
      // rules 1-3: a byte is a continuation exactly when a leading byte 1, 2 or 3 back wants it
      uint32_t req = __funnelshift_l(pg, g, 8);
      const uint32_t F1 = H4 ? __funnelshift_l(pF, gF, 8) : 0u;  // the byte after a leading byte F0-FF
      if (H3 || H4) req |= __funnelshift_l(pE, gE, 16);
      if (H4) req |= __funnelshift_l(pF, gF, 24);
      bad |= (req ^ n) ^ 0x80808080u;
      pg = g;
      pE = gE;
      pF = gF;

      const uint32_t S1 = __funnelshift_r(w, wn, 8);  // byte j: the byte after byte j
      const uint32_t wF = w & 0x0F0F0F0Fu;
      // rules 4-6 for the special leading bytes (see utf8_special_errors)
      if (H2) bad |= g & ~((w & 0x3E3E3E3Eu) + 0x7F7F7F7Fu);  // C0, C1
      if (H3) {
        const uint32_t y = (S1 >> 5) & 0x01010101u;
        const uint32_t q = wF ^ (y * 0x0Du);
        bad |= (ONE ? g : gE & ~gF) & ~(q + 0x7F7F7F7Fu);  // E0 + 80..9F, ED + A0..BF
      }
      if (H4) {
        const uint32_t y4 = ((S1 >> 2) | (S1 >> 3)) & 0x04040404u;
        bad |= gF & (~((wF ^ y4) + 0x7F7F7F7Fu) | (wF + 0x7B7B7B7Bu));  // F0 + 80..8F, F4 + 90..BF, F5..FF
      }

      // byte planes of the output words
      uint32_t L = w, H = 0, U = 0;
      uint32_t S2 = 0;
      if (H3 || H4) S2 = __funnelshift_r(w, wn, 16);
      if (H2) {
        const uint32_t L2 = (w & 0x03030303u) * 64u + (S1 & 0x3F3F3F3Fu);
        const uint32_t H2v = (w >> 2) & 0x07070707u;
        const uint32_t M2 = byte_mask(ONE ? g : g & ~gE);
        L = (L2 & M2) | (L & ~M2);
        H = H2v & M2;
      }
      uint32_t L3 = 0, H3v = 0;
      if (H3 || (H4 && !U32)) {
        L3 = (S1 & 0x03030303u) * 64u + (S2 & 0x3F3F3F3Fu);
        H3v = (S1 >> 2) & 0x0F0F0F0Fu;
      }
      if (H3) {
        const uint32_t M3 = byte_mask(ONE ? g : (H4 ? gE & ~gF : gE));
        L = (L3 & M3) | (L & ~M3);
        H = ((wF * 16u + H3v) & M3) | (H & ~M3);
      }
      if (H4 && U32) {
        // 11110abc 10defghi 10jk.... 10......: U = abc de, H = fghi jk.., L = the last eight bits
        const uint32_t S3 = __funnelshift_r(w, wn, 24), M4 = byte_mask(gF);
        L = (((S2 & 0x03030303u) * 64u + (S3 & 0x3F3F3F3Fu)) & M4) | (L & ~M4);
        H = (((S1 & 0x0F0F0F0Fu) * 16u + ((S2 >> 2) & 0x0F0F0F0Fu)) & M4) | (H & ~M4);
        U = ((w & 0x07070707u) * 4u + ((S1 >> 4) & 0x03030303u)) & M4;
      } else if (H4) {
        const uint32_t M4 = byte_mask(gF), M1 = byte_mask(F1);
        // second surrogate: DC00 | (third byte & 0F) << 6 | (fourth byte & 3F)
        L = (L3 & M1) | (L & ~M1);
        H = (((H3v & 0x03030303u) | 0xDCDCDCDCu) & M1) | (H & ~M1);
        // first surrogate: D7C0 + ((lead & 7) << 8 | Y), Y = (second & 3F) << 2 | (third >> 4) & 3;
        // Y is cleared outside F0-FF positions, so the per-byte sums below carry at most into
        // the byte after a leading byte, where M4 drops them
        const uint32_t Y = ((S1 & 0x3F3F3F3Fu) * 4u + ((S2 >> 4) & 0x03030303u)) & M4;
        const uint32_t cy = ((Y | (Y << 1)) >> 7) & 0x01010101u;  // Y >= 0x40: the low byte wraps
        L = ((Y + 0xC0C0C0C0u) & M4) | (L & ~M4);
        H = (((w & 0x07070707u) + cy + 0xD7D7D7D7u) & M4) | (H & ~M4);
      }
      // stage the words
      const uint32_t all = U32 ? n : n | F1;  // the positions that give one
      const uint32_t lead = EXACT ? all & nibble_flags(m, k - 1) : all;
      if (U32) {
        const uint32_t step = lead >> 5;
        // two positions' low halves, then each with its third byte (below 20: its sign gives the zero)
        const uint32_t P[2] = {__byte_perm(L, H, 0x5140), __byte_perm(L, H, 0x7362)};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t bit = 0x80u << (8 * j), ones = 0x01010101u >> (32 - 8 * j - (j == 0 ? 8 : 0));
          const uint32_t at = j == 0 ? sa : __dp4a(step, ones, sa);
          const uint32_t lo = (j & 1) ? 0x32u : 0x10u, u = 4u + (uint32_t)j;
          const uint32_t unit = prmt(P[j >> 1], U, lo | u << 8 | (8u + u) << 12);
          if (!EXACT && (k < NW || j < 1)) sts_u32(at, unit);
          else sts_u32_if(at, unit, lead, bit);
        }
        if (k < NW) sa = __dp4a(step, 0x01010101u, sa);
        continue;
      }
      const uint32_t step = lead >> 6;
      constexpr int FREE = 2;  // the last word's positions that another word of the lane always follows
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t bit = 0x80u << (8 * j), ones = 0x01010101u >> (32 - 8 * j - (j == 0 ? 8 : 0));
        const uint32_t at = j == 0 ? sa : __dp4a(step, ones, sa);
        if (!EXACT && (k < NW || j < FREE)) sts_u16(at, plane_word(L, H, j));
        else sts_u16_if(at, plane_word(L, H, j), lead, bit);
      }
      if (k < NW) sa = __dp4a(step, 0x01010101u, sa);
    }
    return bad;
  }

  // Validates the lane's 32 bytes and stages their UTF-16 words.  x0 (the lane's offset in
  // the region), rtot and rflags come from the count pass.
  __device__ __forceinline__ static Region wconvert(const Params &p, const uint32_t W[8], uint32_t prev,
                                                    uint32_t next, long long c, bool edge, bool inside, uint16_t *st,
                                                    uint32_t base, uint32_t x0, uint32_t rtot, uint32_t rflags,
                                                    unsigned long long &err_pos) {
    const int lane = threadIdx.x & 31;
    const uint32_t sbase = smem_addr(st);
    if (rflags == 0) {
      // an all-ASCII region: one word per byte; the only possible error is a leading byte
      // just before the region that wants continuation bytes inside it (lane 0's bytes)
      if (lane == 0) check_prev_lead(prev, c, err_pos);
      const uint32_t x = base + 32 * lane;
      const uint32_t a = sbase + 2 * x;
      if ((x & 7) == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          sts_v4(a + 16 * i, __byte_perm(W[2 * i], 0, 0x4140), __byte_perm(W[2 * i], 0, 0x4342),
                 __byte_perm(W[2 * i + 1], 0, 0x4140), __byte_perm(W[2 * i + 1], 0, 0x4342));
      } else if ((x & 1) == 0) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          sts_u32(a + 8 * k, __byte_perm(W[k], 0, 0x4140));
          sts_u32(a + 8 * k + 4, __byte_perm(W[k], 0, 0x4342));
        }
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k)
#pragma unroll
          for (int j = 0; j < 4; ++j) sts_u16(a + 8 * k + 2 * j, (W[k] >> (8 * j)) & 0xFFu);
      }
      return Region{1024u, 0u, 0u, 1024u};
    }
    const uint32_t Wx[10] = {prev, W[0], W[1], W[2], W[3], W[4], W[5], W[6], W[7], next};
    const uint32_t sa = sbase + 2 * (base + x0);
    uint32_t bad;
    if (inside) {
      // the leading-byte classes: the region's own (from the count pass) and those of bytes
      // 1-3 of the word before it (a sequence starting there reaches into the region, and the
      // structure test reads those bytes)
      const uint32_t pc = lane == 0 ? Narrow::lead_classes(prev, 0x80808000u) : 0u;
      const uint32_t cls = rflags | __shfl_sync(0xffffffffu, pc, 0);
      const bool h2 = cls & F_C2, h3 = cls & F_C3, h4 = cls & F_C4;
      if (h4) {
        bad = (h2 || h3) ? wconvert_fast<true, true, true>(Wx, sa) : wconvert_fast<false, false, true>(Wx, sa);
      } else if (h3) {
        bad = h2 ? wconvert_fast<true, true, false>(Wx, sa) : wconvert_fast<false, true, false>(Wx, sa);
      } else {
        bad = h2 ? wconvert_fast<true, false, false>(Wx, sa) : wconvert_fast<true, true, true>(Wx, sa);
      }
    } else {
      // a region at a buffer end: all classes, the bytes outside masked off (with the 16-byte
      // general path inlined here, 512 MiB of ASCII took 292 us instead of 273, 100 MB of CJK 114
      // instead of 100: its code and registers weighed on the paths that run)
      const long long a = (long long)p.off0 - c, b = (long long)p.vbytes - c;
      const uint32_t from = a <= 0 ? 0u : (a >= 32 ? 32u : (uint32_t)a), to = b <= 0 ? 0u : (b >= 32 ? 32u : (uint32_t)b);
      const uint32_t below = to == 32 ? 0xFFFFFFFFu : (1u << to) - 1u;
      bad = wconvert_fast<true, true, true, 8, true>(Wx, sa, from == 32 ? 0u : below & (0xFFFFFFFFu << from));
    }
    if (bad && (unsigned long long)c < err_pos) err_pos = (unsigned long long)c;
    return Region{rtot, 0u, 0u, rtot};
  }
};

}  // namespace gbu
