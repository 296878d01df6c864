"""The transcoders' two partition sizes (4 KiB for small inputs, 16 KiB past a line that depends on
the device): sizes around one partition of each kind and around the line, in both directions and
byte orders, valid and with an error near the end, and the reuse of one context across the line.
Expected values come from oracle/ only (exact)."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def _line():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count * 8 * 4096 * 3 // 2


@pytest.mark.parametrize("profile", ["mixed", "ascii"])
def test_both_sides_of_the_line(profile):
    import torch
    from paper_2111_08692_gb300 import Codec, result_tuple
    line = _line()
    sizes = [1, 4095, 4096, 4097, 16384, 16389, line - 70, line - 3, line - 2, line + 33, line + 4096]
    u8, u16 = W.profile_buffers(profile, max(sizes), max(sizes) // 2, 77, cache=False)
    codec = Codec(0, max_units=max(sizes))
    try:
        for n in sizes:
            for bad in (False, True):
                a, w = np.array(u8[:n]), np.array(u16[:max(n // 2, 1)])
                if bad:
                    a[-1], w[-1] = 0xFF, 0xDC00
                src8, src16 = torch.from_numpy(a).cuda(), torch.from_numpy(w.view(np.int16)).cuda()
                be = torch.from_numpy(w.byteswap().view(np.int16)).cuda()
                want, units = oracle.convert_utf8_to_utf16le(a)
                dst = torch.zeros(max(units.size, 1), dtype=torch.int16, device="cuda")
                ok = units.size if want[0] == "OK" else oracle.utf16_length_from_utf8(a[:want[1]])
                for call, order in ((codec.convert_utf8_to_utf16le, lambda x: x), (codec.convert_utf8_to_utf16be, np.ndarray.byteswap)):
                    assert result_tuple(call(src8, dst, cap=units.size)) == want, (n, bad)
                    assert np.array_equal(order(dst.cpu().numpy().view(np.uint16)[:ok]), units[:ok]), (n, bad)
                want, units = oracle.convert_utf16le_to_utf8(w)
                dst = torch.zeros(max(units.size, 1), dtype=torch.uint8, device="cuda")
                ok = units.size if want[0] == "OK" else oracle.utf8_length_from_utf16le(w[:want[1]])
                for call, src in ((codec.convert_utf16le_to_utf8, src16), (codec.convert_utf16be_to_utf8, be)):
                    assert result_tuple(call(src, dst, cap=units.size)) == want, (n, bad)
                    assert np.array_equal(dst.cpu().numpy()[:ok], units[:ok]), (n, bad)
    finally:
        codec.close()


def test_stop_past_an_error():
    """Errors early, midway and late in a buffer of many partitions: CTAs stop claiming past a known
    error; the result and the valid prefix are the oracle's, and the next call is complete."""
    import torch
    from paper_2111_08692_gb300 import Codec, result_tuple
    n = 48 << 20
    u8, _ = W.profile_buffers("cyrillic", n, 0, 78, cache=False)
    starts = np.flatnonzero((u8 & 0xC0) != 0x80)
    codec = Codec(0, max_units=n)
    try:
        clean, units = oracle.convert_utf8_to_utf16le(u8)
        dst = torch.zeros(units.size, dtype=torch.int16, device="cuda")
        for share in (0.0, 0.01, 0.5, 0.99):
            at = int(starts[int(share * (starts.size - 1))])
            a = np.array(u8)
            a[at] = 0xFF
            assert result_tuple(codec.convert_utf8_to_utf16le(torch.from_numpy(a).cuda(), dst)) == ("HEADER_BITS", at)
            ok = oracle.utf16_length_from_utf8(a[:at])
            assert np.array_equal(dst.cpu().numpy().view(np.uint16)[:ok], units[:ok])
            assert result_tuple(codec.convert_utf8_to_utf16le(torch.from_numpy(np.array(u8)).cuda(), dst)) == clean
            assert np.array_equal(dst.cpu().numpy().view(np.uint16), units)
    finally:
        codec.close()
