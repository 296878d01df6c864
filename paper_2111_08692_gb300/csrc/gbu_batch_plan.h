// gbu_batch_plan.h -- the launch shape of a batched call: how many CTAs, how many strings a warp
// claims at a time, and from which length on a whole CTA takes a string (plain host code).
#pragma once

#include <stdint.h>

namespace gbu {

// Strings a warp packs at most: 32, or 16 where 16 warps' groups and staging buffers share 48 KB.
constexpr uint32_t batch_group_max(int warps_per_cta) { return warps_per_cta == 16 ? 16u : 32u; }

// Few strings: a string of this many input bytes is handled by its CTA's warps together.  One string,
// 8 -> 16 / 16 -> 8, us per launch (GB300), by a warp and by its CTA: 1016 bytes 4.2 / 4.2 and 4.8 / 5.6,
// 1500 bytes 5.4 / 5.1 and 4.8 / 5.8, 2040 bytes 6.4 / 6.1 and 4.7 / 5.4.
constexpr uint32_t BATCH_FEW_LONG_BYTES = 1536;

struct BatchPlan {
  uint32_t grid;        // CTAs
  uint32_t group;       // strings a warp claims and packs at a time
  bool per_cta;         // CTA i handles string i and nothing else (grid == B)
  uint32_t long_bytes;  // strings of at least this many input bytes go to a whole CTA
};

// B strings (B >= 1) on a device with `sms` SMs and `ctas_per_sm` resident CTAs of `warps` warps each.
// claim, long_bytes: the context's geometry; chosen: long_bytes was set by the caller, or by the tuner
// on few strings, and holds for few strings too.
inline BatchPlan batch_plan(uint64_t B, uint32_t sms, uint32_t ctas_per_sm, int warps, uint32_t claim,
                            uint32_t long_bytes, bool chosen) {
  const uint32_t full = batch_group_max(warps);
  const uint64_t resident = (uint64_t)sms * ctas_per_sm;
  BatchPlan p;
  // No more strings than CTAs that run at once: a CTA each, side by side, and its warps share even a
  // short string, as nothing else is waiting for them.  8 -> 16, us per launch: strings of 15,000 bytes,
  // 1 / 8 / 300 of them, packed by warps 37.1 / 47.1 / 49.1, so 11.9 / 12.0 / 15.8; of 2,040 bytes
  // 7.7 / 10.8 / 12.1, so 4.4 / 4.8 / 6.7; past the resident CTAs packing is the faster one (3,000 of
  // 15,000 bytes: 177, against 410 by whole CTAs).
  if (B <= resident) {
    p.grid = (uint32_t)B;
    p.group = 1;
    p.per_cta = true;
    p.long_bytes = chosen || long_bytes < BATCH_FEW_LONG_BYTES ? long_bytes : BATCH_FEW_LONG_BYTES;
    return p;
  }
  // A batch with fewer claims than SMs is cut finer, down to a string per warp; a warp takes its share
  // of a claim, and a full group where every warp gets several, whatever the claim: each claim is an
  // atomic on one address (a million strings, 8 -> 16 / 16 -> 8, us, by a warp's share: 1 string 1,058 /
  // 922, 4 489 / 507, 8 427 / 446, 16 385 / 416, 32 380 / 412).
  uint64_t grab = claim;
  const uint64_t fine = B / sms > (uint64_t)warps ? B / sms : (uint64_t)warps;
  if (fine < grab) grab = fine;
  const uint64_t claims = (B + grab - 1) / grab;
  p.grid = (uint32_t)(claims < resident ? claims : resident);
  p.group = (uint32_t)(grab / (uint64_t)warps);
  if (p.group < 1) p.group = 1;
  if (p.group > full || B >= resident * 4 * full * (uint64_t)warps) p.group = full;
  p.per_cta = false;
  p.long_bytes = long_bytes;
  return p;
}

struct BatchCandidate {
  int warps;
  uint32_t claim, long_bytes;
};
constexpr int BATCH_CANDIDATES = 60;

// The geometries that the tuner times on a batch of B strings, without those that come to the launch of
// an earlier one: warps 4, 8 and 16, a warp's share of a claim 32, 16, 4 and 1 strings (the largest
// first: of claims that are one launch here, the largest is the one to keep for other batches), and long
// strings from 2 to 32 KiB.  ctas_per_sm: resident CTAs per SM for 4, 8 and 16 warps.  Returns their number.
inline int batch_candidates(uint64_t B, uint32_t sms, const int (&ctas_per_sm)[3], BatchCandidate (&out)[BATCH_CANDIDATES]) {
  const int warps[3] = {4, 8, 16};
  const uint32_t shares[4] = {32, 16, 4, 1}, lines[5] = {2048, 4096, 8192, 16384, 32768};
  int n = 0;
  for (int w = 0; w < 3; ++w) {
    BatchPlan seen[20];
    int m = 0;
    for (uint32_t share : shares)
      for (uint32_t line : lines) {
        const BatchPlan p = batch_plan(B, sms, (uint32_t)ctas_per_sm[w], warps[w], share * (uint32_t)warps[w], line, true);
        bool dup = false;
        for (int i = 0; i < m; ++i)
          dup = dup || (seen[i].grid == p.grid && seen[i].group == p.group && seen[i].long_bytes == p.long_bytes);
        if (dup) continue;
        seen[m++] = p;
        out[n++] = BatchCandidate{warps[w], share * (uint32_t)warps[w], line};
      }
  }
  return n;
}

}  // namespace gbu
