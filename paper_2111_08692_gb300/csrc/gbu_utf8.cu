// gbu_utf8.cu -- the UTF-8 -> UTF-16LE transcoders (validating): the single-buffer kernel (the
// wide partition loop of gbu_wide.cuh with the codec of gbu_wide_utf8.cuh) and the kernel over
// several strings (the partition loop of gbu_xcode.cuh with the codec of gbu_codec_utf8.cuh).
#include <stdint.h>

#include "gbu_codec_utf8.cuh"
#include "gbu_kernels.h"
#include "gbu_wide_utf8.cuh"

namespace gbu {

template <int R>
__global__ void __launch_bounds__(XT, XBLOCKS) utf8_to_utf16_kernel(const Params p) {
  extern __shared__ __align__(128) unsigned char smem_raw[];  // sizeof(WSmem), set at launch
  WSmem<Utf8ToUtf16Wide, R> &sm = *reinterpret_cast<WSmem<Utf8ToUtf16Wide, R> *>(smem_raw);
  wtranscode<Utf8ToUtf16Wide, R>(p, sm, [&](uint32_t status, unsigned long long key, unsigned long long tot) {
    if (status) {
      write_result(p.result, GBU_TIMEOUT, 0);
    } else if (key != NO_ERROR) {
      int32_t kind;
      uint64_t off;
      resolve_utf8_error(p.base + p.off0, p.n, (long long)key - (long long)p.off0, &kind, &off);
      write_result(p.result, kind, off);
    } else {
      write_result(p.result, tot > p.cap ? GBU_OUTPUT_TOO_SMALL : GBU_OK, tot);
    }
  });
}

// Several strings per launch (the serving loop's large requests): one result per string.
__global__ void __launch_bounds__(XT, XBLOCKS) utf8_to_utf16_segments_kernel(const SegParams q) {
  extern __shared__ __align__(128) unsigned char smem_raw[];  // sizeof(XSmem), set at launch
  XSmem<Utf8ToUtf16> &sm = *reinterpret_cast<XSmem<Utf8ToUtf16> *>(smem_raw);
  transcode_segments<Utf8ToUtf16>(q, sm, [&](const Params &p, const SegState &st, uint32_t) {
    const uint32_t status = *(volatile uint32_t *)&p.ws->status;
    const unsigned long long key = *(volatile const unsigned long long *)&st.errkey;
    const unsigned long long tot = *(volatile const unsigned long long *)&st.total;
    if (status) {
      write_result(p.result, GBU_TIMEOUT, 0);
    } else if (key != NO_ERROR) {
      int32_t kind;
      uint64_t off;
      resolve_utf8_error(p.base + p.off0, p.n, (long long)key - (long long)p.off0, &kind, &off);
      write_result(p.result, kind, off);
    } else {
      write_result(p.result, tot > p.cap ? GBU_OUTPUT_TOO_SMALL : GBU_OK, tot);
    }
  });
}

const void *utf8_to_utf16_kernel_ptr(bool small) {
  return small ? (const void *)utf8_to_utf16_kernel<1> : (const void *)utf8_to_utf16_kernel<WROUNDS>;
}
size_t utf8_to_utf16_smem_bytes(bool small) {
  return small ? sizeof(WSmem<Utf8ToUtf16Wide, 1>) : sizeof(WSmem<Utf8ToUtf16Wide, WROUNDS>);
}
size_t utf8_to_utf16_segments_smem_bytes() { return sizeof(XSmem<Utf8ToUtf16>); }

const void *utf8_to_utf16_segments_kernel_ptr() { return (const void *)utf8_to_utf16_segments_kernel; }

}  // namespace gbu
