"""The number of CTAs of a single-buffer launch (csrc/gbu_grid.h), compiled alone and run on the CPU: it
fits the completion word's counters whatever the device holds."""
import ctypes
import hashlib
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2111_08692_gb300", "csrc")
BUILD = os.path.join(ROOT, "tests", "_build")
SHIM = r"""
#include "gbu_grid.h"
extern "C" uint32_t grid(uint64_t resident, uint64_t useful) { return gbu::launch_grid(resident, useful); }
extern "C" uint32_t counter_max() { return (uint32_t)((1ull << gbu::FIN_CTA_BITS) - 1); }
"""


def test_a_grid_fits_the_completion_counters():
    os.makedirs(BUILD, exist_ok=True)
    header = open(os.path.join(CSRC, "gbu_grid.h")).read()
    so = os.path.join(BUILD, "libgrid_%s.so" % hashlib.sha1((SHIM + header).encode()).hexdigest()[:16])
    if not os.path.exists(so):
        src, tmp = so[:-3] + ".cpp", so + f".tmp{os.getpid()}"
        open(src, "w").write(SHIM)
        subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, src, "-o", tmp])
        os.replace(tmp, so)
    lib = ctypes.CDLL(so)
    lib.grid.argtypes = [ctypes.c_uint64, ctypes.c_uint64]
    lib.grid.restype = lib.counter_max.restype = ctypes.c_uint32
    for resident, useful, want in ((1216, 0, 1), (1216, 1, 1), (1216, 100, 100), (1216, 1 << 32, 1216),
                                   (4095, 1 << 32, 4095), (4096, 1 << 32, 4095), (100000, 5000, 4095)):
        got = lib.grid(resident, useful)
        assert got == want and got <= lib.counter_max(), (resident, useful, got)
    # every launch whose kernel ends in the packed completion goes through it
    for name, call in (("gbu_api.cu", "launch_grid((uint64_t)c->num_sms"), ("gbu_noalloc.cu", "launch_grid((uint64_t)s.grid")):
        assert call in open(os.path.join(CSRC, name)).read(), name
