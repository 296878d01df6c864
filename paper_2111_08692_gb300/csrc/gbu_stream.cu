// gbu_stream.cu -- read-only kernels: validate_utf8, utf16_length_from_utf8,
// validate_utf16le, utf8_length_from_utf16le.
//
// UTF-8 validation has a kernel of its own (validate8_kernel: bit planes, 32 bytes per lane); the
// others are modes of stream_kernel.
// These never wait on another CTA, so they stream straight from global memory: each warp
// owns 4 KB warp tiles (round-robin over all warps of the grid), issues all eight 16-byte
// loads of a lane before using any (ld.global.nc, no L1 allocation), and takes each chunk's
// neighbouring words from the adjacent lanes with shuffles (the warp tile's outer
// neighbours with two extra 4-byte loads).  Only the warp tiles that straddle the ends of
// the buffer read byte by byte with bounds checks.  Per-thread results (smallest erroring
// chunk start, or unit count) are folded over the CTA and into the workspace; the last CTA
// writes the result.
#include <stdint.h>

#include "gbu_chunk.cuh"
#include "gbu_device.cuh"
#include "gbu_kernels.h"
#include "gbu_planes.cuh"

namespace gbu {

enum StreamMode { S_V8 = 0, S_L16 = 1, S_V16 = 2, S_L8 = 3, S_V16BE = 4, S_L8BE = 5 };

// A UTF-16BE mode runs its UTF-16LE mode on words whose two bytes it exchanges after loading.
template <int MODE>
__host__ __device__ constexpr int base_mode() { return MODE == S_V16BE ? S_V16 : (MODE == S_L8BE ? S_L8 : MODE); }
template <int MODE>
__host__ __device__ constexpr bool big_endian() { return MODE == S_V16BE || MODE == S_L8BE; }
__device__ __forceinline__ uint32_t swap16x2(uint32_t w) { return __byte_perm(w, 0, 0x2301); }

constexpr int ST_WARPS = STREAM_THREADS / 32;
constexpr int ST_ROUNDS = 8;                              // 16-byte chunks per lane per tile
constexpr uint32_t WT_BYTES = 32u * 16u * ST_ROUNDS;      // 4096 bytes per warp tile

// Resident CTAs per SM the register budget is held to: three for the validations (at most 80
// registers), four for the lengths (64).
template <int MODE>
__host__ __device__ constexpr int stream_min_blocks() {
  return (base_mode<MODE>() == S_L16 || base_mode<MODE>() == S_L8) ? 4 : 3;
}

// What a read-only launch has changed in the header (last CTA, thread 0); it uses no scan states, so
// their epoch stays.
__device__ __forceinline__ void reset_read_only(WsHeader *ws) {
  ws->total = 0;
  ws->errkey = NO_ERROR;
  ws->stop_tile = 0xFFFFFFFFu;
}

template <int KMODE>
__global__ void __launch_bounds__(STREAM_THREADS, stream_min_blocks<KMODE>()) stream_kernel(const Params p) {
  constexpr int MODE = base_mode<KMODE>();
  constexpr bool BE = big_endian<KMODE>();
  __shared__ unsigned long long red[ST_WARPS];
  __shared__ int is_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long gw = (long long)blockIdx.x * ST_WARPS + warp;
  const long long nw = (long long)gridDim.x * ST_WARPS;
  const long long lo = p.off0, hi = (long long)p.vbytes;
  unsigned long long err_pos = NO_ERROR, total = 0;
  // Early exit (validation): a warp's tiles lie at increasing positions, so once a warp has
  // flagged a chunk it stops, and no warp starts a tile past the smallest tile flagged so far
  // (the workspace's stop tile, published at once; a snapshot is refreshed every 8th tile of
  // the warp -- all warps read that one word, so reading it every tile would queue them on one
  // L2 slice -- by a load that overlaps the tile's own loads).  The smallest flagged chunk is
  // never skipped.
  const bool early = MODE == S_V16 && p.early_exit != 0;
  uint32_t known = 0xFFFFFFFFu;
  // after a tile: publish a flagged tile and stop, or take the refreshed snapshot
  uint32_t it = 0;  // tiles this warp has started
  auto stop_after_tile = [&](long long wt, uint32_t snap) -> bool {
    if (__any_sync(0xffffffffu, err_pos != NO_ERROR)) {
      if (lane == 0) atomicMin(&p.ws->stop_tile, (uint32_t)wt);
      return true;
    }
    if ((it & 7u) == 1u) known = __shfl_sync(0xffffffffu, snap, 0);
    return false;
  };

  for (long long wt = gw; wt < (long long)p.ntiles; wt += nw) {
    const long long t0 = wt * WT_BYTES;
    if (early && (uint32_t)wt > known) break;  // uniform over the warp
    uint32_t snap = 0xFFFFFFFFu;
    if (early && lane == 0 && (it & 7u) == 0) snap = ld_relaxed_u32(&p.ws->stop_tile);
    ++it;
    const bool fast = t0 - 4 >= lo && t0 + (long long)WT_BYTES + 4 <= hi;
    uint4 v[ST_ROUNDS];
    uint32_t pre, post;
#pragma unroll
    for (int r = 0; r < ST_ROUNDS; ++r) v[r] = load_chunk(p, t0 + 512 * r + 16 * lane, fast);
    if (fast) {
      pre = ldg_word(p.base + t0 - 4);
      post = ldg_word(p.base + t0 + WT_BYTES);
    } else {
      pre = load_word_checked(p, t0 - 4);
      post = load_word_checked(p, t0 + WT_BYTES);
    }
    if (BE) {
#pragma unroll
      for (int r = 0; r < ST_ROUNDS; ++r)
        v[r] = make_uint4(swap16x2(v[r].x), swap16x2(v[r].y), swap16x2(v[r].z), swap16x2(v[r].w));
      pre = swap16x2(pre);
      post = swap16x2(post);
    }
    if ((MODE == S_L16 || MODE == S_L8) && fast) {
      // a warp tile inside the buffer: no neighbouring words and no bounds (1 GiB of CJK, UTF-16
      // length: 208 us with the shuffles of the general loop below, 156 without)
      constexpr uint32_t UNITS = MODE == S_L16 ? 16u : 8u;  // units of an ASCII chunk
      uint32_t any = 0;
#pragma unroll
      for (int r = 0; r < ST_ROUNDS; ++r) any |= v[r].x | v[r].y | v[r].z | v[r].w;
      if (__all_sync(0xffffffffu, (any & (MODE == S_L16 ? 0x80808080u : 0xFF80FF80u)) == 0)) {
        total += UNITS * ST_ROUNDS;
        continue;
      }
      // flags in bit 7 of each byte, summed by byte dot products (0x80 per flag)
      uint32_t add = 0, sub = 0;
#pragma unroll
      for (int r = 0; r < ST_ROUNDS; ++r) {
        const uint32_t Wd[4] = {v[r].x, v[r].y, v[r].z, v[r].w};
        if (MODE == S_L16) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint32_t w = Wd[k], s1 = w * 2u;
            add = __dp4a((~w | s1) & 0x80808080u, 0x01010101u, add);                          // not a continuation
            add = __dp4a(w & s1 & (w * 4u) & (w * 8u) & 0x80808080u, 0x01010101u, add);       // >= F0
          }
        } else {
#pragma unroll
          for (int k = 0; k < 4; k += 2) {  // the high and the low bytes of four words
            const uint32_t hb = __byte_perm(Wd[k], Wd[k + 1], 0x7531), lb = __byte_perm(Wd[k], Wd[k + 1], 0x6420);
            add = __dp4a((((hb & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | hb | lb) & 0x80808080u, 0x01010101u, add);  // >= 80
            add = __dp4a((((hb & 0x78787878u) + 0x78787878u) | hb) & 0x80808080u, 0x01010101u, add);       // >= 800
            sub = __dp4a(bytes_sur(hb), 0x01010101u, sub);
          }
        }
      }
      total += (MODE == S_L8 ? UNITS * ST_ROUNDS : 0u) + ((add - sub) >> 7);
      continue;
    }
    if (MODE == S_V16 && fast) {
      // A warp tile inside the buffer: surrogate flags of every word's high byte first; a tile
      // without a surrogate word has no error and needs no neighbouring words, and in any
      // other tile every chunk is judged, its neighbours taken from the adjacent lanes.
      uint32_t anys = 0;
#pragma unroll
      for (int r = 0; r < ST_ROUNDS; ++r) {
        const uint32_t Wd[4] = {v[r].x, v[r].y, v[r].z, v[r].w};
        uint32_t P0, P1;
        utf16_high_bytes(Wd, P0, P1);
        anys |= bytes_sur(P0) | bytes_sur(P1);
      }
      if (__any_sync(0xffffffffu, anys != 0)) {
#pragma unroll
        for (int r = 0; r < ST_ROUNDS; ++r) {
          const uint32_t Wd[4] = {v[r].x, v[r].y, v[r].z, v[r].w};
          const uint32_t up = __shfl_up_sync(0xffffffffu, v[r].w, 1);
          const uint32_t down = __shfl_down_sync(0xffffffffu, v[r].x, 1);
          const uint32_t before = r == 0 ? pre : __shfl_sync(0xffffffffu, v[r > 0 ? r - 1 : 0].w, 31);
          const uint32_t after =
              r == ST_ROUNDS - 1 ? post : __shfl_sync(0xffffffffu, v[r < ST_ROUNDS - 1 ? r + 1 : r].x, 0);
          uint32_t P0, P1;
          utf16_high_bytes(Wd, P0, P1);
          const uint32_t S0 = bytes_sur(P0), S1 = bytes_sur(P1);
          const bool bad = ((S0 | S1) != 0) & utf16_pair_errors_bytes(P0, P1, S0, S1, lane == 0 ? before : up,
                                                                    lane == 31 ? after : down);
          const long long c = t0 + 512 * r + 16 * lane;
          if (bad && (unsigned long long)c < err_pos) err_pos = (unsigned long long)c;
        }
      }
      if (early && stop_after_tile(wt, snap)) break;
      continue;
    }
#pragma unroll
    for (int r = 0; r < ST_ROUNDS; ++r) {
      const long long c = t0 + 512 * r + 16 * lane;
      const bool edge = !fast && (c < lo || c + 16 > hi);
      uint32_t W[6];
      W[1] = v[r].x; W[2] = v[r].y; W[3] = v[r].z; W[4] = v[r].w;
      const uint32_t up = __shfl_up_sync(0xffffffffu, v[r].w, 1);
      const uint32_t down = __shfl_down_sync(0xffffffffu, v[r].x, 1);
      const uint32_t before = r == 0 ? pre : __shfl_sync(0xffffffffu, v[r > 0 ? r - 1 : 0].w, 31);
      const uint32_t after =
          r == ST_ROUNDS - 1 ? post : __shfl_sync(0xffffffffu, v[r < ST_ROUNDS - 1 ? r + 1 : r].x, 0);
      W[0] = lane == 0 ? before : up;
      W[5] = lane == 31 ? after : down;

      if (MODE == S_L16) {
        Flags8 f[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) f[k] = classify8(W[k]);
        total += utf8_count_units(f, c, edge, lo, hi);
      } else if (MODE == S_V16) {
        const uint32_t Wd[4] = {W[1], W[2], W[3], W[4]};
        if (utf16_chunk_errors(Wd, W[0], W[5], c, edge, lo, hi) && (unsigned long long)c < err_pos)
          err_pos = (unsigned long long)c;
      } else if (MODE == S_L8) {
        const uint32_t Wd[4] = {W[1], W[2], W[3], W[4]};
        uint32_t cnt = 0;
        if (!edge) {
          cnt = utf16_len8_inside(Wd);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint32_t w = (Wd[j >> 1] >> (16 * (j & 1))) & 0xFFFFu;
            const bool valid = c + 2 * j >= lo && c + 2 * j < hi;
            cnt += valid ? len8_of_word(w) : 0u;
          }
        }
        total += cnt;
      }
    }
    if (early && stop_after_tile(wt, snap)) break;
  }

  unsigned long long cta = 0;
  if (MODE == S_L16 || MODE == S_L8) {
    total = warp_sum_u64(total);
    if (lane == 0) red[warp] = total;
    __syncthreads();
    if (threadIdx.x == 0)
      for (int w = 0; w < ST_WARPS; ++w) cta += red[w];
  }
  unsigned long long tot;
  bool errors;
  if (!finish_packed<STREAM_THREADS>(p, err_pos, cta, red, &is_last, &tot, &errors)) return;
  if (threadIdx.x == 0) {
    if (MODE == S_L16 || MODE == S_L8) {
      *p.len_out = tot;
    } else if (!errors) {
      write_result(p.result, GBU_OK, p.n);
    } else {
      const unsigned long long key = *(volatile unsigned long long *)&p.ws->errkey;
      uint64_t off;
      resolve_utf16_error<BE>(reinterpret_cast<const uint16_t *>(p.base + p.off0), p.n,
                              ((long long)key - (long long)p.off0) / 2, &off);
      write_result(p.result, GBU_SURROGATE, off);
    }
    reset_read_only(p.ws);
  }
}

// UTF-8 validation: a warp streams 4 KiB warp tiles, four regions of 1 KiB, a lane 32 consecutive
// bytes of each (the source base is rounded to 32 bytes), judged on bit planes (gbu_planes.cuh).  A
// region without a byte >= 80 takes one vote; one without a byte >= E0 is judged four bytes at a
// time, tried only while the warp's last region was such a one.  Bound by HBM for ASCII, by the
// integer pipe else.  1 GiB, us (GB300, one sitting): ASCII / Latin / CJK / emoji 150 / 254 / 441 /
// 531 by the byte-wise kernel before the planes, 150 / 271 / 271 / 289 on the planes alone,
// 148 / 216 / 278 / 296 with the two-byte route.  The warp's next tile is loaded when all four regions
// are judged, two 16-byte loads for a lane's 32 bytes: with one 256-bit load as soon as each region
// was judged, 152 / 218 / 281 / 300, and ASCII right after a kernel that left L2 full of its output
// 183 instead of 171.
constexpr int V8_REGIONS = (int)(WT_BYTES / 1024u);

// The lane's 32 bytes at virtual position c (bytes outside the input read as zero).
__device__ __forceinline__ void load_lane32(const Params &p, long long c, bool inside, uint32_t (&w)[8]) {
  uint4 a, b;
  if (inside) {
    a = ldg_stream(p.base + c);
    b = ldg_stream(p.base + c + 16);
  } else {
    a = load_chunk(p, c, false);
    b = load_chunk(p, c + 16, false);
  }
  w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
  w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
}

__global__ void __launch_bounds__(STREAM_THREADS, 3) validate8_kernel(const Params p) {
  __shared__ unsigned long long red[ST_WARPS];
  __shared__ int is_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long nw = (long long)gridDim.x * ST_WARPS;
  const long long lo = p.off0, hi = (long long)p.vbytes;
  auto inside = [&](long long t0) { return t0 - 4 >= lo && t0 + (long long)WT_BYTES + 4 <= hi; };
  auto edge_word = [&](long long v, bool in) { return in ? ldg_word(p.base + v) : load_word_checked(p, v); };
  unsigned long long err_pos = NO_ERROR;
  // early exit as in stream_kernel
  const bool early = p.early_exit != 0;
  uint32_t known = 0xFFFFFFFFu, it = 0;
  long long wt = (long long)blockIdx.x * ST_WARPS + warp;
  bool high = false;  // the warp's last judged region had a byte >= E0: go to the planes at once
  uint32_t W[V8_REGIONS][8], pre = 0, post = 0;
  if (wt < (long long)p.ntiles) {
    const long long t0 = wt * WT_BYTES;
    const bool in = inside(t0);
#pragma unroll
    for (int r = 0; r < V8_REGIONS; ++r) load_lane32(p, t0 + 1024 * r + 32 * lane, in, W[r]);
    pre = edge_word(t0 - 4, in);
    post = edge_word(t0 + WT_BYTES, in);
  }
  for (; wt < (long long)p.ntiles; wt += nw) {
    const long long t0 = wt * WT_BYTES, t1 = t0 + nw * WT_BYTES;  // this tile, the warp's next one
    if (early && (uint32_t)wt > known) break;  // uniform over the warp
    uint32_t snap = 0xFFFFFFFFu;
    if (early && lane == 0 && (it & 7u) == 0) snap = ld_relaxed_u32(&p.ws->stop_tile);
    ++it;
    const bool more = wt + nw < (long long)p.ntiles, in = inside(t1);
    uint32_t em = 0;  // the regions whose bytes of this lane hold an error
    // continuation bytes wanted in the lane's bytes of the next region by those of this one (used
    // from lane 31, for lane 0), at first those wanted by the word before the tile
    uint32_t pending = wanted_after(pre);
#pragma unroll
    for (int r = 0; r < V8_REGIONS; ++r) {
      uint32_t any = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) any |= W[r][k];
      if (__any_sync(0xffffffffu, (any & 0x80808080u) != 0 || (lane == 31 && pending != 0))) {
        auto exchange = [&](uint32_t out) {
          const uint32_t wanted = __shfl_sync(0xffffffffu, lane == 31 ? pending : out, (lane + 31) & 31);
          pending = out;
          return wanted;
        };
        uint32_t err;
        if (high || !utf8_two_byte_errors(W[r], exchange, err)) {
          const uint32_t after = r + 1 < V8_REGIONS ? W[r + 1 < V8_REGIONS ? r + 1 : r][0] : post;
          const uint32_t next = __shfl_sync(0xffffffffu, lane == 0 ? after : W[r][0], (lane + 1) & 31);
          bool any3;
          err = utf8_plane_errors(W[r], exchange, next, any3);
          high = __any_sync(0xffffffffu, any3);
        }
        em |= err ? 1u << r : 0u;
      } else {
        pending = 0;
      }
    }
    if (more) {
#pragma unroll
      for (int r = 0; r < V8_REGIONS; ++r) load_lane32(p, t1 + 1024 * r + 32 * lane, in, W[r]);
      pre = edge_word(t1 - 4, in);
      post = edge_word(t1 + WT_BYTES, in);
    }
    if (em) {
      const unsigned long long c = (unsigned long long)(t0 + 1024 * (__ffs(em) - 1) + 32 * lane);
      if (c < err_pos) err_pos = c;
    }
    if (early) {
      if (__any_sync(0xffffffffu, err_pos != NO_ERROR)) {
        if (lane == 0) atomicMin(&p.ws->stop_tile, (uint32_t)wt);
        break;
      }
      if ((it & 7u) == 1u) known = __shfl_sync(0xffffffffu, snap, 0);
    }
  }
  unsigned long long tot;
  bool errors;
  if (!finish_packed<STREAM_THREADS>(p, err_pos, 0, red, &is_last, &tot, &errors)) return;
  if (threadIdx.x == 0) {
    if (!errors) {
      write_result(p.result, GBU_OK, p.n);
    } else {
      const unsigned long long key = *(volatile unsigned long long *)&p.ws->errkey;
      int32_t kind;
      uint64_t off;
      resolve_utf8_error(p.base + p.off0, p.n, (long long)key - (long long)p.off0, &kind, &off);
      write_result(p.result, kind, off);
    }
    reset_read_only(p.ws);
  }
}

const void *stream_kernel_ptr(int mode) {
  switch (mode) {
    case S_V8: return (const void *)validate8_kernel;
    case S_L16: return (const void *)stream_kernel<S_L16>;
    case S_V16: return (const void *)stream_kernel<S_V16>;
    case S_V16BE: return (const void *)stream_kernel<S_V16BE>;
    case S_L8BE: return (const void *)stream_kernel<S_L8BE>;
    default: return (const void *)stream_kernel<S_L8>;
  }
}

uint32_t stream_tile_bytes() { return WT_BYTES; }

}  // namespace gbu
