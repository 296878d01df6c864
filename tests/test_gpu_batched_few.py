"""Batched calls on few strings, by the library's own geometry: each string has a CTA of its own up to
the number of CTAs that run at once, and is packed by a warp past it.  Expected values come from oracle/
only (exact: bytes, counts and kinds)."""
import numpy as np
import pytest

import workloads as W
from test_gpu_batched import _check_all

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


@pytest.mark.parametrize("B", [1, 2, 9, 300, 455, 457, 609])
@pytest.mark.parametrize("median", [40, 1500, 6000])
def test_few_strings(torch, B, median):
    from paper_2111_08692_gb300 import Codec
    codec = Codec(0, max_units=1 << 26)
    try:
        _check_all(torch, codec, W.batched_strings(B, 3000 + B + median, median=median, max_len=65536,
                                                   error_fraction=0.1, cache=False))
        _check_all(torch, codec, W.batched_strings(B, 4000 + B + median, median=median, max_len=65536,
                                                   error_fraction=0.1, cache=False), tight_seed=B)
    finally:
        codec.close()


@pytest.mark.parametrize("size", [1008, 1533, 1536, 1539, 4093, 4096, 4100, 16384])
def test_one_string_around_the_lines(torch, size):
    """One string whose length lies at a line between the two routes or at a CTA step's end, whole and cut
    inside a character, at two alignments."""
    import oracle
    from paper_2111_08692_gb300 import Codec, result_tuple
    u8, _ = W.profile_buffers("mixed", 1 << 15, 0, 91, cache=False)
    codec = Codec(0, max_units=1 << 16)
    try:
        for shift in (0, 5):
            data = np.array(u8[:size])
            src = torch.from_numpy(np.concatenate([np.full(shift, 0x41, np.uint8), data, np.full(9, 0x80, np.uint8)])).cuda()
            off = torch.tensor([shift, shift + size], dtype=torch.int64, device="cuda")
            want, units = oracle.convert_utf8_to_utf16le(data)
            cap = max(units.size, 1)
            dst = torch.full((cap + 8,), 0x5A5A, dtype=torch.int16, device="cuda")
            res = codec.convert_utf8_to_utf16le_batched(src, off, dst, torch.tensor([0, cap], device="cuda"))
            assert result_tuple(res[0]) == want
            ok = want[1] if want[0] == "OK" else oracle.utf16_length_from_utf8(data[:want[1]])
            host = dst.cpu().numpy().view(np.uint16)
            assert np.array_equal(host[:ok], units[:ok]) and (host[cap:] == 0x5A5A).all()
            assert result_tuple(codec.validate_utf8_batched(src, off)[0]) == oracle.validate_utf8(data)
            assert int(codec.utf16_length_from_utf8_batched(src, off)[0]) == oracle.utf16_length_from_utf8(data)
    finally:
        codec.close()


def _cost(torch, B, geometry=None, tune=False):
    """Time of 20 launches on B strings of 15000 bytes, 8 -> 16 (the best of 12)."""
    from paper_2111_08692_gb300 import Codec
    u8, _ = W.profile_buffers("mixed", 1 << 20, 0, 92, cache=False)
    starts = np.flatnonzero((u8 & 0xC0) != 0x80)
    one = np.array(u8[:starts[np.searchsorted(starts, 15000)]])
    side = torch.cuda.Stream()
    op = "convert_utf8_to_utf16le"
    codec = Codec(0, max_units=1 << 20)
    try:
        if geometry:
            codec.set_batch_config(op, *geometry)
        if tune:
            many = torch.from_numpy(np.tile(one[:200], 20000)).cuda()
            off = torch.arange(20001, dtype=torch.int64, device="cuda") * 200
            codec.tune_batched(op, many, off, codec.new_results(20000),
                               torch.empty(many.numel(), dtype=torch.int16, device="cuda"), off, reps=1)
        src = torch.from_numpy(np.tile(one, B)).cuda()
        off = torch.arange(B + 1, dtype=torch.int64, device="cuda") * one.size
        dst = torch.empty(B * one.size, dtype=torch.int16, device="cuda")
        res = codec.new_results(B)
        torch.cuda.synchronize()

        def body():
            for _ in range(20):
                codec.convert_utf8_to_utf16le_batched(src, off, dst, off, res, stream=side)
        graph = codec.capture(body, side)
        times = []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(side)
            graph.launch(side)
            b.record(side)
            side.synchronize()
            times.append(a.elapsed_time(b))
        graph.close()
        return min(times)
    finally:
        codec.close()


def test_few_long_strings_run_side_by_side(torch):
    """A string of 15000 bytes alone, and eight of them, cost by the library's own geometry at most twice
    what one costs when its CTA works on it together (a warp alone takes three times as long), also after
    the geometry was tuned on a large batch."""
    together = _cost(torch, 1, (8, 64, 512))
    assert _cost(torch, 1) < 2 * together
    assert _cost(torch, 8) < 2 * together
    assert _cost(torch, 1, tune=True) < 2 * together
