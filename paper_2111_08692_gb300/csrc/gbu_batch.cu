// gbu_batch.cu -- batched forms of the six operations: many strings in one launch, and the
// exclusive scan that turns batched output lengths into output offsets.
//
// The strings come in CSR form (one buffer holding them back to back and B+1 offsets in
// code units) or as an array of descriptors (pointer and length of each input and output).
// In a persistent grid of CTAs (NWARPS warps each)
//   * every warp claims groups of up to 32 consecutive strings (a counter in the workspace) and
//     packs them: the strings' 16-byte chunks are numbered back to back, a lane takes one chunk,
//     and a warp step handles 32 of them, whatever strings they belong to.  Segmented scans give each string its
//     length, its first error and its place in the output.  A warp step on one string at a time
//     left most lanes idle (half of a log-normal column's strings have under 64 bytes, four
//     lanes' worth): 522 to 1427 warp instructions per string of 197 bytes on average, now 109
//     to 393.  A million such strings, lengths, scan and conversion in both directions: 4,421 us
//     before, 1,088 us now (GB300);
//   * a string of at least long_bytes input bytes is set aside and handled by the whole CTA once
//     its warps find no more groups (or its list of them fills up): NWARPS 512-byte regions per
//     step (one 16-byte chunk per lane); for a transcoding each warp counts its region first and the
//     CTA scans the counts, so every region knows where its output starts.
// The chunks' analysis is that of the single-buffer kernels, so each string's result is the one a
// single-buffer call on it gives.
// A batch of no more strings than resident CTAs gives each a CTA of its own (gbu_batch_plan.h).
// Strings never wait on one another, so nothing spins.  Output offsets of a transcoding come
// from the caller's dst_off (for example the exclusive scan of the batched lengths).
// What bounds it: instruction issue on the integer pipe (63-65% busy in the conversions), then the
// latency of a step's loads, which are issued a step ahead.
// The launch geometry (warps per CTA, strings per claim, long-string threshold) is the library's, the
// caller's or the autotuner's, which times candidates.
#include <stdint.h>

#include "gbu_batch_plan.h"
#include "gbu_chunk.cuh"
#include "gbu_codec_utf16.cuh"
#include "gbu_codec_utf8.cuh"
#include "gbu_device.cuh"
#include "gbu_kernels.h"
#include "gbu_wide_utf16.cuh"
#include "gbu_wide_utf8.cuh"

namespace gbu {

constexpr uint32_t BATCH_LONGS = 512;  // long strings a CTA can set aside
// A string of this many input bytes goes to the whole CTA whatever the threshold (positions inside
// a packed string are kept in 32 bits).
constexpr uint32_t PACK_LIMIT = 1u << 28;

template <int MODE>
struct BatchTraits {
  static constexpr bool UTF8_IN = MODE == B_V8 || MODE == B_L16 || MODE == B_C8;
  static constexpr uint32_t IN_UNIT = UTF8_IN ? 1u : 2u;
  static constexpr bool CONVERT = MODE == B_C8 || MODE == B_C16;
  static constexpr bool LENGTH = MODE == B_L16 || MODE == B_L8;
  // UTF-8 validation (also inside a transcoding) judges the three positions past the end
  static constexpr uint32_t TAIL = (MODE == B_V8 || MODE == B_C8) ? 3u : 0u;
};

template <int MODE>
struct BatchCodec {
  using C = Utf8ToUtf16;
};
template <>
struct BatchCodec<B_C16> {
  using C = Utf16ToUtf8;
};

// The strings of a warp's group (at most G) that hold at least one chunk, in order.
template <int G>
struct PackedStrings {
  uint64_t src[G];    // address of the first byte (its low four bits: the offset in its 16-byte block)
  uint64_t dst[G];    // transcoders: address of the first output unit
  uint32_t first[G];  // number of its first chunk in the group
  uint32_t end[G];    // bytes from its first 16-byte block on
  uint32_t cap[G];    // transcoders: output units (clamped to 32 bits)
  uint32_t index[G];  // its index in the group
};

template <int MODE, int NWARPS>
struct __align__(128) BatchSmem {
  using Out = typename BatchCodec<MODE>::C::Out;
  static constexpr int SW = BatchTraits<MODE>::CONVERT ? NWARPS : 1;
  static constexpr uint32_t SU = BatchTraits<MODE>::CONVERT ? BatchCodec<MODE>::C::STAGE : 8u;
  Out staging[SW][2][SU];
  static constexpr int GROUP = (int)batch_group_max(NWARPS);
  PackedStrings<GROUP> packed[NWARPS];
  uint32_t rcount[2][NWARPS];        // long strings: units of each warp's region in a step
  unsigned long long red[NWARPS];    // long strings: per-warp error position or count
  uint64_t longs[BATCH_LONGS];       // long strings set aside
  uint32_t nlong;
  uint32_t more;                     // a warp stopped for the list's sake: groups are left
};

// The single-buffer parameters of string i (base, off0, vbytes, n; destination and cap for a
// transcoding).
template <int MODE>
__device__ __forceinline__ Params string_params(const BatchParams &bp, uint64_t i) {
  using T = BatchTraits<MODE>;
  constexpr uint32_t OUT_UNIT = MODE == B_C8 ? 2u : 1u;
  Params sp;
  uintptr_t a, da = 0;
  uint64_t n, cap = 0;
  if (bp.desc) {
    const StringDesc d = bp.desc[i];
    a = (uintptr_t)d.src;
    n = d.n;
    if (T::CONVERT) {
      da = (uintptr_t)d.dst;
      cap = d.cap;
    }
  } else {
    const uint64_t start = bp.off[i], end = bp.off[i + 1];
    n = end > start ? end - start : 0;
    a = (uintptr_t)(bp.src + start * T::IN_UNIT);
    if (T::CONVERT) {
      const uint64_t d0 = bp.dst_off[i], d1 = bp.dst_off[i + 1];
      da = (uintptr_t)(bp.dst + d0 * OUT_UNIT);
      cap = d1 > d0 ? d1 - d0 : 0;
    }
  }
  sp.base = (const uint8_t *)(a & ~(uintptr_t)15);
  sp.off0 = (uint32_t)(a & 15);
  sp.n = n;
  sp.vbytes = sp.off0 + n * T::IN_UNIT;
  sp.dbase = (uint8_t *)(da & ~(uintptr_t)15);
  sp.dshift = (uint32_t)((da & 15) / OUT_UNIT);
  sp.cap = cap;
  return sp;
}

// Input code units of string i.
__device__ __forceinline__ uint64_t string_units(const BatchParams &bp, uint64_t i) {
  if (bp.desc) return bp.desc[i].n;
  const uint64_t s = bp.off[i], e = bp.off[i + 1];
  return e > s ? e - s : 0;
}

// Virtual end of the positions to judge (0 for an empty string).
template <int MODE>
__device__ __forceinline__ long long string_span(const Params &sp) {
  return sp.n == 0 ? 0 : (long long)sp.vbytes + BatchTraits<MODE>::TAIL;
}

// The chunk at virtual position c (lane's chunk of a region) and the words just before and
// after it (one warp, all lanes).
__device__ __forceinline__ void region_load(const Params &sp, long long c, uint4 &v, uint32_t &prev,
                                            uint32_t &next) {
  const int lane = threadIdx.x & 31;
  const long long lo = sp.off0, hi = (long long)sp.vbytes;
  const bool inside = c - 4 >= lo && c + 20 <= hi;
  v = load_chunk(sp, c, inside);
  prev = __shfl_up_sync(0xffffffffu, v.w, 1);
  next = __shfl_down_sync(0xffffffffu, v.x, 1);
  if (lane == 0) prev = inside ? ldg_word(sp.base + c - 4) : load_word_checked(sp, c - 4);
  if (lane == 31) next = inside ? ldg_word(sp.base + c + 16) : load_word_checked(sp, c + 16);
}

// Read-only analysis of one chunk: the smallest erroring chunk start goes to err_pos
// (validation), the units to total (lengths).
template <int MODE>
__device__ __forceinline__ void region_read(const Params &sp, long long c, uint4 v, uint32_t prev,
                                            uint32_t next, unsigned long long &err_pos,
                                            unsigned long long &total) {
  const long long lo = sp.off0, hi = (long long)sp.vbytes;
  const bool edge = c < lo || c + 16 > hi;
  if (MODE == B_V8 || MODE == B_L16) {
    const uint32_t W[6] = {prev, v.x, v.y, v.z, v.w, next};
    Flags8 f[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) f[k] = classify8(W[k]);
    if (MODE == B_L16) {
      total += utf8_count_units(f, c, edge, lo, hi);
    } else {
      uint32_t err = utf8_structure_errors(f);
      uint32_t c2 = 0, c3 = 0, c4 = 0;
#pragma unroll
      for (int k = 1; k <= 4; ++k) {
        c2 |= f[k].geC0 & ~f[k].geE0;
        c3 |= f[k].geE0 & ~f[k].geF0;
        c4 |= f[k].geF0;
      }
      err |= utf8_special_errors(W, f, __any_sync(0xffffffffu, c2 != 0), __any_sync(0xffffffffu, c3 != 0),
                                 __any_sync(0xffffffffu, c4 != 0));
      if (err && (unsigned long long)c < err_pos) err_pos = (unsigned long long)c;
    }
  } else {
    const uint32_t Wd[4] = {v.x, v.y, v.z, v.w};
    if (MODE == B_L8) {
      uint32_t cnt = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t w = (Wd[j >> 1] >> (16 * (j & 1))) & 0xFFFFu;
        const bool valid = !edge || (c + 2 * j >= lo && c + 2 * j < hi);
        cnt += valid ? len8_of_word(w) : 0u;
      }
      total += cnt;
    } else if (utf16_chunk_errors(Wd, prev, next, c, edge, lo, hi)) {
      if ((unsigned long long)c < err_pos) err_pos = (unsigned long long)c;
    }
  }
}

// Converts one region whose output starts at unit S of the string's destination (one warp).
template <int MODE, int NWARPS>
__device__ __forceinline__ uint32_t region_convert(const Params &sp, long long c, uint4 v, uint32_t prev,
                                                   uint32_t next, uint64_t S, BatchSmem<MODE, NWARPS> &sm,
                                                   uint32_t &use, unsigned long long &err_pos) {
  using C = typename BatchCodec<MODE>::C;
  constexpr uint32_t V = 16 / sizeof(typename C::Out);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long lo = sp.off0, hi = (long long)sp.vbytes;
  const bool edge = c < lo || c + 16 > hi;
  typename C::Out *st = sm.staging[warp][use & 1];
  ++use;
  const uint32_t h = (uint32_t)((sp.dshift + S) & (V - 1));
  if (lane == 0) bulk_wait_read<1>();  // the store of two regions ago has read this buffer
  __syncwarp();
  const long long r0 = c - (long long)CHUNK * lane;  // the region's start
  const bool inside = r0 >= (long long)sp.off0 && r0 + (long long)REGION_BYTES <= (long long)sp.vbytes;
  const Region g = convert_counted<C>(sp, v, prev, next, c, edge, inside, st, h, err_pos);
  fence_proxy_async_smem();
  __syncwarp();
  store_region(sp, st, S, g.skip, g.total, g.extra);
  return g.units;
}

// Writes string i's result (lane 0 / thread 0).
template <int MODE>
__device__ __forceinline__ void string_result(const BatchParams &bp, uint64_t i, const Params &sp,
                                              unsigned long long err_pos, unsigned long long total,
                                              uint64_t units) {
  using T = BatchTraits<MODE>;
  if (T::LENGTH) {
    bp.lens[i] = total;
  } else if (err_pos != NO_ERROR) {
    int32_t kind = GBU_SURROGATE;
    uint64_t off;
    if (T::UTF8_IN)
      resolve_utf8_error(sp.base + sp.off0, sp.n, (long long)err_pos - (long long)sp.off0, &kind, &off);
    else
      resolve_utf16_error(reinterpret_cast<const uint16_t *>(sp.base + sp.off0), sp.n,
                          ((long long)err_pos - (long long)sp.off0) / 2, &off);
    write_result(&bp.results[i], kind, off);
  } else if (T::CONVERT) {
    write_result(&bp.results[i], units > sp.cap ? GBU_OUTPUT_TOO_SMALL : GBU_OK, units);
  } else {
    write_result(&bp.results[i], GBU_OK, sp.n);
  }
}

// ---- packed strings --------------------------------------------------------------------------------

// Bit i: byte i of the 16 bytes at position c lies inside [lo, hi).
__device__ __forceinline__ uint32_t chunk_valid_bits(uint32_t c, uint32_t lo, uint32_t hi) {
  const uint32_t from = c == 0 ? lo : 0u, left = hi > c ? hi - c : 0u;
  const uint32_t upto = left >= 16 ? 0xFFFFu : (1u << left) - 1u;
  return upto & (0xFFFFu << from);
}

// Bits 0-3 of m as byte masks.
__device__ __forceinline__ uint32_t nibble_bytes(uint32_t m) { return byte_mask(nibble_flags(m, 0)); }

// The classes of leading bytes in w: 1: C0-DF, 2: E0-EF, 4: F0-FF.
__device__ __forceinline__ uint32_t lead_classes_of(uint32_t w) {
  const uint32_t g = w & (w << 1) & 0x80808080u, gE = g & (w << 2), gF = gE & (w << 3);
  return ((g & ~gE) ? 1u : 0u) | ((gE & ~gF) ? 2u : 0u) | (gF ? 4u : 0u);
}

// Stores the bytes of a register's two UTF-16 words from staging address o on and advances o; v,
// two, three: words inside the string, of at least two bytes, of three (bit 15 of each lane).
__device__ __forceinline__ void put_words(uint32_t &o, uint32_t v, uint32_t two, uint32_t three, uint32_t B0,
                                          uint32_t B1, uint32_t B2) {
  const uint32_t size = (v >> 15) + (two >> 15) + (three >> 15);
  const uint32_t o1 = __dp2a_lo(size, 0x0001u, o);
  sts_u8_if_set<0>(o, B0, v, 0x8000u);
  sts_u8_if_set<1>(o, B1, two, 0x8000u);
  sts_u8_if_set<2>(o, B2, three, 0x8000u);
  sts_u8_if_set<0>(o1, B0 >> 16, v, 0x80000000u);
  sts_u8_if_set<1>(o1, B1 >> 16, two, 0x80000000u);
  sts_u8_if_set<2>(o1, B2 >> 16, three, 0x80000000u);
  o = __dp2a_lo(size, 0x0101u, o);
}

// The UTF-8 bytes of a lane's eight UTF-16 words (W[1..4]; W[0], W[5]: the words before and after),
// staged from address o on.  Each surrogate writes the two bytes of its own slots (see
// gbu_wide_utf16.cuh), so a lane never writes outside the bytes it counts.  SUR, WIDE, THREE:
// surrogates, other words >= 0x80, three-byte words may occur.  Nonzero: an unpaired surrogate.
template <bool SUR, bool WIDE, bool THREE>
__device__ __forceinline__ uint32_t words_to_utf8(const uint32_t (&W)[6], uint32_t o, uint32_t m) {
  uint32_t Hp = SUR ? lanes16_sur(W[0]) & ~(W[0] << 5) : 0u;  // first-surrogate flags of the register before
  uint32_t err = 0;
#pragma unroll
  for (int k = 1; k <= 4; ++k) {
    const uint32_t X = W[k], A6 = X >> 6;
    const uint32_t v = ((m >> (4 * k - 4)) & 1u) << 15 | ((m >> (4 * k - 2)) & 1u) << 31;
    const uint32_t last = (X & 0x003F003Fu) | 0x00800080u;
    uint32_t B0 = X, B1 = last, two = 0, three = 0;
    const uint32_t S = SUR ? lanes16_sur(X) : 0u;
    if (WIDE) {
      two = lanes16_ge80(X);
      const uint32_t G1 = prmt(two, 0u, 0xBB99u);
      B0 = (((A6 & 0x001F001Fu) | 0x00C000C0u) & G1) | (X & ~G1);
    } else if (SUR) {
      two = S;
    }
    if (THREE) {
      three = lanes16_ge800(X) & ~S;
      const uint32_t G2 = prmt(three, 0u, 0xBB99u);
      B0 = ((((X >> 12) & 0x000F000Fu) | 0x00E000E0u) & G2) | (B0 & ~G2);
      B1 = (((A6 & 0x003F003Fu) | 0x00800080u) & G2) | (last & ~G2);
    }
    if (SUR) {
      // a word is a second surrogate exactly when the one before it is a first one
      const uint32_t b10 = X << 5, H = S & ~b10, L = S & b10;
      err |= L ^ __funnelshift_l(Hp, H, 16);
      Hp = H;
      const uint32_t T = (X & 0x03FF03FFu) + 0x00400040u;
      const uint32_t Xp = __funnelshift_l(W[k - 1], X, 16);  // each lane's word before
      const uint32_t h0 = ((T >> 8) & 0x00070007u) | 0x00F000F0u, h1 = ((T >> 2) & 0x003F003Fu) | 0x00800080u;
      const uint32_t l0 = (Xp & 0x00030003u) * 16u + ((A6 & 0x000F000Fu) | 0x00800080u);
      const uint32_t HM = prmt(H, 0u, 0xBB99u), LM = prmt(L, 0u, 0xBB99u);
      B0 = (h0 & HM) | (B0 & ~HM);
      B0 = (l0 & LM) | (B0 & ~LM);
      B1 = (h1 & HM) | (B1 & ~HM);
    }
    put_words(o, v, two, three, B0, B1, last);
  }
  if (SUR) {
    const uint32_t Ln = lanes16_sur(W[5]) & (W[5] << 5);
    err |= (Hp >> 31) ^ ((Ln >> 15) & 1u);
  }
  return err;
}

// A lane's chunk of UTF-8 (W[1..4]): its UTF-16 words, and the leading-byte classes present.
// convert: the words as the conversion stores them (the second surrogate of a four-byte sequence at
// the byte after its leading byte), else the length formula.
__device__ __forceinline__ uint32_t chunk_units8(const uint32_t (&W)[6], uint32_t m, bool convert, uint32_t &flags) {
  uint32_t n = 0, c2 = 0, c3 = 0, c4 = 0;
  uint32_t pF = W[0] & (W[0] * 2u) & (W[0] * 4u) & (W[0] * 8u) & 0x80808080u;
#pragma unroll
  for (int k = 1; k <= 4; ++k) {
    const uint32_t w = W[k], s1 = w * 2u;
    const uint32_t g = w & s1 & 0x80808080u, gE = g & (w * 4u), gF = gE & (w * 8u);
    if (convert) {
      n = __dp4a((~w | s1 | __funnelshift_l(pF, gF, 8)) & nibble_flags(m, k - 1), 0x01010101u, n);
      pF = gF;
    } else {
      n = __dp4a((~w | s1) & nibble_flags(m, k - 1), 0x01010101u, n);
      n = __dp4a(gF, 0x01010101u, n);
    }
    if (convert) {
      c2 |= g & ~gE;
      c3 |= gE & ~gF;
      c4 |= gF;
    }
  }
  flags = (c2 ? 1u : 0u) | (c3 ? 2u : 0u) | (c4 ? 4u : 0u);
  return n >> 7;
}

// A lane's chunk of UTF-16: its UTF-8 bytes, and whether surrogates (1), three-byte words (2) and
// other words >= 0x80 (4) occur.  Words outside the string read as zero.
__device__ __forceinline__ uint32_t chunk_units16(const uint32_t (&W)[6], uint32_t m, uint32_t &flags) {
  uint32_t n80 = 0, n800 = 0, sur = 0;
#pragma unroll
  for (int k = 1; k <= 4; k += 2) {
    const uint32_t hb = __byte_perm(W[k], W[k + 1], 0x7531), lb = __byte_perm(W[k], W[k + 1], 0x6420);
    n80 = __dp4a((((hb & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | hb | lb) & 0x80808080u, 0x01010101u, n80);
    n800 = __dp4a((((hb & 0x78787878u) + 0x78787878u) | hb) & 0x80808080u, 0x01010101u, n800);
    sur = __dp4a(bytes_sur(hb), 0x01010101u, sur);
  }
  flags = (sur ? 1u : 0u) | (n800 != sur ? 2u : 0u) | (n80 != sur ? 4u : 0u);
  return (uint32_t)__popc(m) / 2u + ((n80 + n800 - sur) >> 7);
}

// Handles strings g0 .. g0 + count - 1 (count <= GROUP), except the long ones, which are noted for
// the whole CTA (one warp, all lanes).
template <int MODE, int NWARPS>
__device__ __forceinline__ void packed_strings(const BatchParams &bp, uint64_t g0, uint32_t count,
                                               BatchSmem<MODE, NWARPS> &sm) {
  using T = BatchTraits<MODE>;
  using Out = typename BatchCodec<MODE>::C::Out;
  constexpr uint32_t V = 16 / sizeof(Out);
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t le = 0xFFFFFFFFu >> (31 - lane);  // lanes up to this one
  auto &ps = sm.packed[warp];
  // the group's strings, one per lane
  uint32_t chunks = 0, end = 0;
  Params sp;
  if (lane < count) {
    sp = string_params<MODE>(bp, g0 + lane);
    const uint64_t bytes = sp.n * T::IN_UNIT;
    if (bytes >= bp.long_bytes || bytes >= PACK_LIMIT) {
      sm.longs[atomicAdd(&sm.nlong, 1u)] = g0 + lane;
    } else if (sp.n == 0) {
      string_result<MODE>(bp, g0 + lane, sp, NO_ERROR, 0, 0);
    } else {
      end = (uint32_t)sp.vbytes;
      chunks = (end + T::TAIL + CHUNK - 1) / CHUNK;
    }
  }
  uint32_t first = chunks;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, first, d);
    if (lane >= d) first += y;
  }
  const uint32_t total = __shfl_sync(0xffffffffu, first, 31);
  first -= chunks;
  const uint32_t some = __ballot_sync(0xffffffffu, chunks != 0);
  if (chunks) {
    const uint32_t e = __popc(some & le) - 1;
    ps.src[e] = (uint64_t)(sp.base + sp.off0);
    ps.first[e] = first;
    ps.end[e] = end;
    ps.index[e] = lane;
    if (T::CONVERT) {
      ps.dst[e] = (uint64_t)sp.dbase + (uint64_t)sp.dshift * sizeof(Out);
      ps.cap[e] = sp.cap < 0xFFFFFFFFull ? (uint32_t)sp.cap : 0xFFFFFFFFu;
    }
  }
  __syncwarp();

  Out *const st = &sm.staging[T::CONVERT ? warp : 0][0][0];
  // A step's chunks, loaded a step ahead (raw: blocks that hold a data byte are read whole -- an
  // aligned block cannot cross a page -- and cleared outside the string when the step comes).
  struct Step {
    uint32_t starts;      // lanes at which a string starts
    uint32_t e;           // the lane's string
    uint32_t c, hi, m;    // the chunk's position and the string's end in it; its bytes inside
    uint64_t src;         // the string's first 16-byte block | the offset of its first byte in it
    uint4 q;
    uint32_t after;       // lane 31: the word after the chunk
  };
  uint32_t entry = 0xFFFFFFFFu;  // the string that the last step loaded ends in
  auto load_step = [&](uint32_t v0) {
    Step t;
    const uint32_t rel = first - v0;
    t.starts = __reduce_or_sync(0xffffffffu, chunks && rel < 32u ? 1u << rel : 0u);
    // the string of each lane's chunk: one more than the lane before's where a string starts
    t.e = entry + __popc(t.starts & le);
    entry += __popc(t.starts);
    t.c = t.hi = t.m = 0;
    t.src = 0;
    t.q = make_uint4(0u, 0u, 0u, 0u);
    t.after = 0;
    if (v0 + lane < total) {
      t.src = ps.src[t.e];
      t.c = (v0 + lane - ps.first[t.e]) * CHUNK;
      t.hi = ps.end[t.e];
      const uint32_t lo = (uint32_t)t.src & 15u;
      const uint8_t *const at = reinterpret_cast<const uint8_t *>(t.src - lo) + t.c;
      t.m = chunk_valid_bits(t.c, lo, t.hi);
      if (t.m) t.q = ldg_stream(at);
      if (!T::LENGTH && lane == 31 && t.c + CHUNK < t.hi) t.after = ldg_word(at + CHUNK);
    }
    return t;
  };
  uint32_t carry = 0, carry_word = 0;       // its units so far; its last word in that step
  uint32_t carry_err = 0xFFFFFFFFu;         // its first flagged chunk
  Step ahead;
  if (total) ahead = load_step(0);
  for (uint32_t v0 = 0; v0 < total; v0 += 32) {
    const Step t = ahead;
    if (v0 + 32 < total) ahead = load_step(v0 + 32);
    const uint32_t starts = t.starts, mine = starts & le, e = t.e, c = t.c, hi = t.hi, m = t.m;
    const uint32_t lo = (uint32_t)t.src & 15u;
    const uint64_t src = t.src;
    const bool active = v0 + lane < total;
    const uint32_t seg = mine ? 31u - __clz(mine) : 0u;  // the first lane of the string in this step
    uint4 q = t.q;
    if (m != 0xFFFFu) {
      q.x &= nibble_bytes(m);
      q.y &= nibble_bytes(m >> 4);
      q.z &= nibble_bytes(m >> 8);
      q.w &= nibble_bytes(m >> 12);
    }
    uint32_t W[6] = {0u, q.x, q.y, q.z, q.w, 0u};
    const bool ends = active && c + CHUNK >= hi + T::TAIL;  // the string's last chunk
    if (!T::LENGTH) {
      const uint32_t up = __shfl_up_sync(0xffffffffu, q.w, 1);
      const uint32_t down = __shfl_down_sync(0xffffffffu, q.x, 1);
      W[0] = c == 0 ? 0u : (lane == 0 ? carry_word : up);
      W[5] = ends ? 0u : down;
      if (lane == 31) {
        const uint32_t left = hi > c + CHUNK ? hi - c - CHUNK : 0u;
        W[5] = left >= 4 ? t.after : t.after & ((1u << (8 * left)) - 1u);
      }
      carry_word = __shfl_sync(0xffffffffu, q.w, 31);
    }
    // units of the chunk; the lanes' places in the step and in their strings
    uint32_t units = 0, flags = 0, at = 0, x0 = 0;
    if (T::LENGTH || T::CONVERT) {
      if (T::UTF8_IN) units = chunk_units8(W, m, T::CONVERT, flags);
      else units = chunk_units16(W, m, flags);
      uint32_t incl = units;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
      }
      at = incl - units;
      x0 = at - __shfl_sync(0xffffffffu, at, seg) + (mine ? 0u : carry);
      carry = __shfl_sync(0xffffffffu, x0 + units, 31);
    }
    // analysis and conversion
    uint32_t bad = 0;
    if (MODE == B_V8) {
      Flags8 f[5];
      uint32_t c2 = 0, c3 = 0, c4 = 0;
#pragma unroll
      for (int k = 0; k < 5; ++k) f[k] = classify8(W[k]);
#pragma unroll
      for (int k = 1; k <= 4; ++k) {
        c2 |= f[k].geC0 & ~f[k].geE0;
        c3 |= f[k].geE0 & ~f[k].geF0;
        c4 |= f[k].geF0;
      }
      bad = utf8_structure_errors(f) |
            utf8_special_errors(W, f, __any_sync(0xffffffffu, c2 != 0), __any_sync(0xffffffffu, c3 != 0),
                                __any_sync(0xffffffffu, c4 != 0));
    } else if (MODE == B_V16) {
      // words outside the string read as zero, which is no surrogate
      const uint32_t Wd[4] = {W[1], W[2], W[3], W[4]};
      uint32_t P0, P1;
      utf16_high_bytes(Wd, P0, P1);
      const uint32_t S0 = bytes_sur(P0), S1 = bytes_sur(P1);
      bad = (S0 | S1) != 0 && utf16_pair_errors_bytes(P0, P1, S0, S1, W[0], W[5]);
    } else if (T::CONVERT) {
      const uint32_t step_units = __shfl_sync(0xffffffffu, at + units, 31);
      const uint64_t dst = active ? ps.dst[e] : 0;
      // The step's output is one piece where the strings' outputs lie back to back and fit: then it
      // goes out as in the single-buffer transcoders, else string by string.
      const uint64_t origin = dst + (uint64_t)x0 * sizeof(Out) - (uint64_t)at * sizeof(Out);
      const uint64_t origin0 = __shfl_sync(0xffffffffu, origin, 0);
      const bool one = __all_sync(0xffffffffu, !active || (origin == origin0 && x0 + units <= ps.cap[e]));
      const uint32_t h = one ? (uint32_t)(origin0 / sizeof(Out)) & (V - 1) : 0u;
      if (lane == 0) bulk_wait_read<0>();  // the last step's store has read the buffer
      __syncwarp();
      const uint32_t sa = smem_addr(st) + (h + at) * (uint32_t)sizeof(Out);
      if (T::UTF8_IN) {
        // Routes by the classes in the step, which is often one string's or one script's (a million
        // strings, both directions: 1118 us with three routes here and three below, 1089 so); bytes
        // 1-3 of the word before a chunk may hold leading bytes of another class.
        if (lane == 0) flags |= lead_classes_of(W[0] & 0xFFFFFF00u);
        const uint32_t cls = __reduce_or_sync(0xffffffffu, flags);
        if (cls == 4u) bad = Utf8ToUtf16Wide::wconvert_fast<false, false, true, 4, true>(W, sa, m);
        else if (cls == 2u) bad = Utf8ToUtf16Wide::wconvert_fast<false, true, false, 4, true>(W, sa, m);
        else if (cls & 4u) bad = Utf8ToUtf16Wide::wconvert_fast<true, true, true, 4, true>(W, sa, m);
        else if (cls & 2u) bad = Utf8ToUtf16Wide::wconvert_fast<true, true, false, 4, true>(W, sa, m);
        else bad = Utf8ToUtf16Wide::wconvert_fast<true, false, false, 4, true>(W, sa, m);
      } else {
        // the pair rule reaches from the step before into lane 0's words
        if (lane == 0 && is_high16(W[0] >> 16)) flags |= 1u;
        const uint32_t cls = __reduce_or_sync(0xffffffffu, flags);
        if (cls == 0) bad = words_to_utf8<false, false, false>(W, sa, m);
        else if (cls == 4u) bad = words_to_utf8<false, true, false>(W, sa, m);
        else if (cls == 1u) bad = words_to_utf8<true, false, false>(W, sa, m);
        else if (!(cls & 1u)) bad = words_to_utf8<false, true, true>(W, sa, m);
        else bad = words_to_utf8<true, true, true>(W, sa, m);
      }
      if (one) {
        fence_proxy_async_smem();
        __syncwarp();
        store_staged(reinterpret_cast<Out *>(origin0) - h, st, h, 0xFFFFFFFFu, 0, step_units, 0);
      } else {
        __syncwarp();
        // each string's piece, coalesced
        uint32_t left = starts | 1u;  // first lanes of the strings in this step
        while (left) {
          const uint32_t a = __ffs(left) - 1;
          left &= left - 1;
          const uint32_t b = left ? __ffs(left) - 1 : 32u;  // the next string's first lane
          const uint32_t s0 = __shfl_sync(0xffffffffu, at, a), y0 = __shfl_sync(0xffffffffu, x0, a);
          const uint32_t s1 = b < 32 ? __shfl_sync(0xffffffffu, at, b & 31) : step_units;
          const uint64_t d = __shfl_sync(0xffffffffu, dst, a);
          const uint32_t cap = __shfl_sync(0xffffffffu, active ? ps.cap[e] : 0u, a);
          const uint32_t n = min(s1 - s0, cap > y0 ? cap - y0 : 0u);
          for (uint32_t i = lane; i < n; i += 32) reinterpret_cast<Out *>(d)[y0 + i] = st[s0 + i];
        }
        __syncwarp();
      }
    }
    // results of the strings that end in this step
    uint32_t err = 0xFFFFFFFFu;
    if (!T::LENGTH) {
      const uint32_t flagged = __ballot_sync(0xffffffffu, active && bad != 0) & le & (0xFFFFFFFFu << seg);
      if (!mine) err = carry_err;
      if (err == 0xFFFFFFFFu && flagged) err = c - (lane - (uint32_t)(__ffs(flagged) - 1)) * CHUNK;
      carry_err = __shfl_sync(0xffffffffu, err, 31);
    }
    if (ends) {
      Params rp;
      rp.base = reinterpret_cast<const uint8_t *>(src - lo);
      rp.off0 = lo;
      rp.n = (hi - lo) / T::IN_UNIT;
      rp.cap = T::CONVERT ? ps.cap[e] : 0u;
      string_result<MODE>(bp, g0 + ps.index[e], rp, err == 0xFFFFFFFFu ? NO_ERROR : err, x0 + units, x0 + units);
    }
  }
  __syncwarp();  // ps is rewritten by the next group
  if (T::CONVERT) {
    if (lane == 0) bulk_wait_read<0>();  // the staging buffer is free for the CTA's long strings
    __syncwarp();
  }
}

// A string handled by the whole CTA, NWARPS regions per step (all threads).
template <int MODE, int NWARPS>
__device__ __forceinline__ void cta_string(const BatchParams &bp, uint64_t i, BatchSmem<MODE, NWARPS> &sm,
                                           uint32_t &use) {
  using T = BatchTraits<MODE>;
  using C = typename BatchCodec<MODE>::C;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const Params sp = string_params<MODE>(bp, i);
  const long long span = string_span<MODE>(sp);
  const long long lo = sp.off0, hi = (long long)sp.vbytes;
  unsigned long long err_pos = NO_ERROR, total = 0;
  uint64_t running = 0;
  int buf = 0;
  for (long long s0 = 0; s0 < span; s0 += (long long)NWARPS * REGION_BYTES, buf ^= 1) {
    const long long c = s0 + (long long)warp * REGION_BYTES + CHUNK * lane;
    uint4 v;
    uint32_t prev, next;
    region_load(sp, c, v, prev, next);
    if (T::CONVERT) {
      // region offsets inside the step: count first, then scan the NWARPS region counts
      const bool edge = c < lo || c + 16 > hi;
      uint32_t cf;
      uint32_t cnt = C::count(sp, v, c, edge, cf);
#pragma unroll
      for (int d = 16; d >= 1; d >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, d);
      if (lane == 0) sm.rcount[buf][warp] = cnt;
      __syncthreads();  // also: rcount[buf ^ 1] of the step before is no longer read
      uint32_t before = 0, step_total = 0;
#pragma unroll
      for (int w = 0; w < NWARPS; ++w) {
        const uint32_t x = sm.rcount[buf][w];
        before += w < warp ? x : 0u;
        step_total += x;
      }
      region_convert<MODE, NWARPS>(sp, c, v, prev, next, running + before, sm, use, err_pos);
      running += step_total;
    } else {
      region_read<MODE>(sp, c, v, prev, next, err_pos, total);
    }
  }
  unsigned long long x = T::LENGTH ? warp_sum_u64(total) : warp_min_u64(err_pos);
  if (lane == 0) sm.red[warp] = x;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long a = T::LENGTH ? 0ull : NO_ERROR;
    for (int w = 0; w < NWARPS; ++w) a = T::LENGTH ? a + sm.red[w] : (sm.red[w] < a ? sm.red[w] : a);
    string_result<MODE>(bp, i, sp, T::LENGTH ? NO_ERROR : a, T::LENGTH ? a : 0ull, running);
  }
  __syncthreads();  // sm.red and sm.rcount are reused by the next long string
}

// Resident warps per SM the register budget is held to: 32 (64 registers a thread), 24 for the
// UTF-8 -> UTF-16 transcoder (80); its CTAs of 16 warps do not share an SM then, so they get up to 128
// registers for 16 resident warps (a million strings: 395 us, with 8 warps 377).  FEW: CTA i handles string i and nothing else, together or with its
// first warp (an instance of its own: the same test inside the claim loop spilled more registers there,
// and a million strings took 1,090 us instead of 1,084).
template <int MODE, int NWARPS, bool FEW>
__global__ void __launch_bounds__(NWARPS * 32, (MODE == B_C8 ? 24 : 32) / NWARPS) batch_kernel(const BatchParams bp) {
  using T = BatchTraits<MODE>;
  using Smem = BatchSmem<MODE, NWARPS>;
  __shared__ Smem sm;
  const int lane = threadIdx.x & 31;
  uint32_t use = 0;  // regions staged by this warp (picks its staging buffer)
  if (FEW) {
    const uint64_t bytes = string_units(bp, blockIdx.x) * T::IN_UNIT;
    if (bytes >= bp.long_bytes || bytes >= PACK_LIMIT) cta_string<MODE, NWARPS>(bp, blockIdx.x, sm, use);
    else if (threadIdx.x < 32) packed_strings<MODE, NWARPS>(bp, blockIdx.x, 1, sm);
    if (T::CONVERT && lane == 0) bulk_wait_all<0>();
    return;
  }
  constexpr uint32_t FULL = Smem::GROUP;
  static_assert(BATCH_LONGS >= 2 * FULL * NWARPS, "room for every warp's group past the stop mark");
  const uint32_t group = bp.group;  // at most FULL
  if (threadIdx.x == 0) sm.nlong = sm.more = 0;
  __syncthreads();
  while (true) {
    while (true) {
      uint64_t g0 = 0;
      uint32_t full = 0;
      if (lane == 0) {
        full = *(volatile uint32_t *)&sm.nlong > BATCH_LONGS - FULL * NWARPS;
        if (full) sm.more = 1;
        else g0 = (uint64_t)atomicAdd(&bp.ws->ticket, 1u) * group;
      }
      g0 = __shfl_sync(0xffffffffu, g0, 0);
      if (__shfl_sync(0xffffffffu, full, 0) || g0 >= bp.B) break;
      packed_strings<MODE, NWARPS>(bp, g0, bp.B - g0 < group ? (uint32_t)(bp.B - g0) : group, sm);
    }
    __syncthreads();
    const uint32_t nl = sm.nlong, more = sm.more;
    for (uint32_t k = 0; k < nl; ++k) cta_string<MODE, NWARPS>(bp, sm.longs[k], sm, use);
    if (!more) break;
    __syncthreads();
    if (threadIdx.x == 0) sm.nlong = sm.more = 0;
    __syncthreads();
  }
  if (T::CONVERT && lane == 0) bulk_wait_all<0>();
  // the last CTA to finish resets the claim counter for the next launch
  if (threadIdx.x == 0) {
    __threadfence();
    const uint32_t prev = atomicAdd(&bp.ws->done, 1u);
    if (prev == gridDim.x - 1) {
      __threadfence();
      bp.ws->ticket = 0;
      bp.ws->done = 0;
      __threadfence();
    }
  }
}

// ---- exclusive scan of uint64 values (output offsets from batched lengths) -----------------

constexpr int SCAN_THREADS = 512;
constexpr int SCAN_ITEMS = 8;
constexpr uint32_t SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

// out[k] = in[0] + ... + in[k-1] for k = 0 .. count (out has count + 1 entries; out[count] is
// the total).  Tiles of SCAN_TILE values are claimed by ticket and chained by the decoupled
// look-back; the last CTA writes the result {status, total} and resets the workspace.
__global__ void __launch_bounds__(SCAN_THREADS) scan_u64_kernel(const ScanParams sp) {
  __shared__ unsigned long long warp_tot[SCAN_THREADS / 32 + 1];
  __shared__ LookbackSmem<SCAN_THREADS> lb;
  __shared__ uint32_t ticket;
  __shared__ int is_last;
  const Params &p = sp.lb;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t epoch = p.ws->epoch;
  while (true) {
    if (threadIdx.x == 0) ticket = atomicAdd(&p.ws->ticket, 1u);
    __syncthreads();
    const uint32_t t = ticket;
    if (t >= p.ntiles) break;
    const uint64_t b0 = (uint64_t)t * SCAN_TILE + (uint64_t)threadIdx.x * SCAN_ITEMS;
    uint64_t x[SCAN_ITEMS], s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
      x[k] = b0 + k < sp.count ? sp.in[b0 + k] : 0ull;
      s += x[k];
    }
    uint64_t incl = s;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += y;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      const uint64_t w = lane < SCAN_THREADS / 32 ? warp_tot[lane] : 0ull;
      uint64_t wi = w;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, wi, d);
        if (lane >= d) wi += y;
      }
      if (lane < SCAN_THREADS / 32) warp_tot[lane] = wi - w;
      if (lane == SCAN_THREADS / 32 - 1) warp_tot[SCAN_THREADS / 32] = wi;
    }
    __syncthreads();
    const uint64_t tile_total = warp_tot[SCAN_THREADS / 32];
    uint64_t run = warp_tot[warp] + incl - s;
    if (threadIdx.x == 0) {
      publish_aggregate(p, t, tile_total, epoch);
      atomicAdd(&p.ws->total, (unsigned long long)tile_total);
    }
    run += lookback_cta<SCAN_THREADS>(p, t, tile_total, epoch, lb);
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
      if (b0 + k <= sp.count) sp.out[b0 + k] = run;
      run += x[k];
    }
    __syncthreads();  // warp_tot and ticket are rewritten by the next tile
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const uint32_t prev = atomicAdd(&p.ws->done, 1u);
    is_last = prev == gridDim.x - 1;
    if (is_last) {
      __threadfence();
      const uint32_t status = *(volatile uint32_t *)&p.ws->status;
      const unsigned long long tot = *(volatile unsigned long long *)&p.ws->total;
      // look-back values carry 44 bits: a larger total cannot be chained
      write_result(sp.result, status ? GBU_TIMEOUT : (tot > ST_VALUE_MASK ? GBU_BAD_ARGUMENT : GBU_OK), tot);
    }
  }
  __syncthreads();
  if (is_last) reset_workspace(p, epoch);
}

// ---- host-side handles -------------------------------------------------------------------

template <int MODE>
static const void *batch_ptr_for(int nwarps, bool few) {
  switch (nwarps) {
    case 4: return few ? (const void *)batch_kernel<MODE, 4, true> : (const void *)batch_kernel<MODE, 4, false>;
    case 16: return few ? (const void *)batch_kernel<MODE, 16, true> : (const void *)batch_kernel<MODE, 16, false>;
    default: return few ? (const void *)batch_kernel<MODE, 8, true> : (const void *)batch_kernel<MODE, 8, false>;
  }
}

const void *batch_kernel_ptr(int mode, int nwarps, bool few) {
  switch (mode) {
    case B_V8: return batch_ptr_for<B_V8>(nwarps, few);
    case B_L16: return batch_ptr_for<B_L16>(nwarps, few);
    case B_C8: return batch_ptr_for<B_C8>(nwarps, few);
    case B_V16: return batch_ptr_for<B_V16>(nwarps, few);
    case B_L8: return batch_ptr_for<B_L8>(nwarps, few);
    default: return batch_ptr_for<B_C16>(nwarps, few);
  }
}

const void *scan_kernel_ptr() { return (const void *)scan_u64_kernel; }
uint32_t scan_tile_items() { return SCAN_TILE; }
int scan_threads() { return SCAN_THREADS; }

}  // namespace gbu
