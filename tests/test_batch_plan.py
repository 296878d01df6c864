"""The launch shape of a batched call (csrc/gbu_batch_plan.h), compiled alone and run on the CPU:
every plan covers its strings within the kernel's limits, and a batch of few strings gives each its
own CTA."""
import ctypes
import hashlib
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2111_08692_gb300", "csrc")
BUILD = os.path.join(ROOT, "tests", "_build")
SHIM = r"""
#include "gbu_batch_plan.h"
extern "C" void plan(uint64_t B, uint32_t sms, uint32_t per_sm, int warps, uint32_t claim, uint32_t long_bytes,
                     int chosen, uint32_t *out) {
  const gbu::BatchPlan p = gbu::batch_plan(B, sms, per_sm, warps, claim, long_bytes, chosen != 0);
  out[0] = p.grid; out[1] = p.group; out[2] = p.per_cta; out[3] = p.long_bytes;
}
extern "C" int candidates(uint64_t B, uint32_t sms, int p4, int p8, int p16, uint32_t *out) {
  gbu::BatchCandidate c[gbu::BATCH_CANDIDATES];
  const int per_sm[3] = {p4, p8, p16}, n = gbu::batch_candidates(B, sms, per_sm, c);
  for (int i = 0; i < n; ++i) { out[3 * i] = c[i].warps; out[3 * i + 1] = c[i].claim; out[3 * i + 2] = c[i].long_bytes; }
  return n;
}
"""
SMS = 152
PER_SM = {4: 8, 8: 4, 16: 2}


@pytest.fixture(scope="module")
def plan():
    os.makedirs(BUILD, exist_ok=True)
    header = open(os.path.join(CSRC, "gbu_batch_plan.h")).read()
    so = os.path.join(BUILD, "libplan_%s.so" % hashlib.sha1((SHIM + header).encode()).hexdigest()[:16])
    if not os.path.exists(so):
        src, tmp = so[:-3] + ".cpp", so + f".tmp{os.getpid()}"
        open(src, "w").write(SHIM)
        subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, src, "-o", tmp])
        os.replace(tmp, so)
    lib = ctypes.CDLL(so)
    lib.plan.argtypes = [ctypes.c_uint64, ctypes.c_uint32, ctypes.c_uint32, ctypes.c_int, ctypes.c_uint32,
                         ctypes.c_uint32, ctypes.c_int, ctypes.c_void_p]

    def call(B, warps=8, claim=64, long_bytes=16384, chosen=False):
        out = (ctypes.c_uint32 * 4)()
        lib.plan(B, SMS, PER_SM[warps], warps, claim, long_bytes, int(chosen), out)
        return dict(zip(("grid", "group", "per_cta", "long_bytes"), out))
    call.lib = lib
    return call


@pytest.mark.parametrize("warps", [4, 8, 16])
@pytest.mark.parametrize("chosen", [False, True])
def test_every_plan_is_within_the_kernels_limits(plan, warps, chosen):
    resident = SMS * PER_SM[warps]
    full = 16 if warps == 16 else 32
    for B in (1, 2, 7, 8, 9, 151, 152, resident - 1, resident, resident + 1, 5000, 10 ** 5, 10 ** 6, 10 ** 9, 1 << 40):
        for claim in (1, 8, 64, 512, 1024):
            p = plan(B, warps, claim, chosen=chosen)
            assert 1 <= p["grid"] <= resident and 1 <= p["group"] <= full, (B, claim, p)
            assert not p["per_cta"] or (p["grid"] == B and p["group"] == 1), (B, claim, p)


@pytest.mark.parametrize("warps", [4, 8, 16])
def test_few_strings_get_a_cta_each(plan, warps):
    """No more strings than resident CTAs: one string per CTA, and by the library's own choice a
    string's CTA works on it together from 1.5 KiB on; a threshold that was set stays."""
    resident = SMS * PER_SM[warps]
    for B in (1, 8, 64, 300):
        assert plan(B, warps) == {"grid": B, "group": 1, "per_cta": 1, "long_bytes": 1536}
        assert plan(B, warps, long_bytes=4096, chosen=True)["long_bytes"] == 4096
    p = plan(resident + 1, warps)
    assert not p["per_cta"] and p["long_bytes"] == 16384


@pytest.mark.parametrize("warps", [4, 8, 16])
@pytest.mark.parametrize("chosen", [False, True])
def test_a_warps_share(plan, warps, chosen):
    """The claim's share where no SM idles, less where one would, the largest in a large batch."""
    full = 16 if warps == 16 else 32
    for claim in (1, warps, 4 * warps, 10 * warps, 1024):
        assert plan(300_000, warps, claim, chosen=chosen)["group"] == max(1, min(full, claim // warps))
        assert plan(2000, warps, claim, chosen=chosen)["group"] <= max(1, 2000 // SMS // warps)
        assert plan(10 ** 6, warps, claim, chosen=chosen)["group"] == full


@pytest.mark.parametrize("B", [1, 300, 609, 5000, 20000, 10 ** 6])
def test_the_tuners_candidates_are_distinct_launches(plan, B):
    out = (ctypes.c_uint32 * 180)()
    n = plan.lib.candidates(ctypes.c_uint64(B), SMS, PER_SM[4], PER_SM[8], PER_SM[16], out)
    seen = set()
    for i in range(n):
        warps, claim, line = out[3 * i:3 * i + 3]
        p = plan(B, warps, claim, line, chosen=True)
        seen.add((warps, p["grid"], p["group"], p["long_bytes"]))
        assert 1 <= claim <= 1024 and line >= 512
    assert len(seen) == n
    if B in (1, 300, 10 ** 6):  # every claim comes to the same launch: the largest is kept
        assert n == 15 and all(out[3 * i + 1] == 32 * out[3 * i] for i in range(n))
    assert {w for w, *_ in seen} == {4, 8, 16} and {s[3] for s in seen} == {2048, 4096, 8192, 16384, 32768}
