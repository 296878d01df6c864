"""UTF-32 -> UTF-8 at a buffer's ends, whose regions take a body of their own by the largest unit in them:
units on both sides of 0x800 in the first, the last or the only region, at every alignment, and short
capacities.  Expected values come from oracle/ only (exact)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("high", [0x7F, 0x7FF, 0x800, 0x10FFFF])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 63, 64, 127, 128, 129, 255, 4096, 4100])
def test_ends(n, high):
    import torch
    from paper_2111_08692_gb300 import Codec, result_tuple
    rng = np.random.default_rng(n + high)
    codec = Codec(0, max_units=1 << 16)
    try:
        for shift in range(4):
            units = rng.choice(np.array([0x41, 0x7F, 0x80, 0x7FF], np.uint32), size=n)
            if high < 0x80:
                units &= 0x7F
            units[int(rng.integers(0, n))] = high
            for bad in (None, 0, n - 1):
                u = units.copy()
                if bad is not None:
                    u[bad] = 0xD800
                buf = torch.full((n + shift + 8,), 0x10FFFF, dtype=torch.int32, device="cuda")
                buf[shift:shift + n] = torch.from_numpy(u.view(np.int32).copy())
                want, out = oracle.convert_utf32_to_utf8(u)
                for cap in {out.size, max(out.size - 1, 0)} if bad is None else {out.size}:
                    dst = torch.full((cap + 24,), 0x5A, dtype=torch.uint8, device="cuda")
                    got = result_tuple(codec.convert_utf32_to_utf8(buf[shift:shift + n], dst[shift:], cap=cap))
                    assert got == (want if bad is not None or cap == out.size else ("OUTPUT_TOO_SMALL", out.size))
                    ok = min(cap, oracle.utf8_length_from_utf32(u[:want[1]]) if bad is not None else cap)
                    host = dst.cpu().numpy()
                    assert np.array_equal(host[shift:shift + ok], out[:ok]), (shift, bad, cap)
                    assert (host[:shift] == 0x5A).all() and (host[shift + cap:] == 0x5A).all(), (shift, bad, cap)
    finally:
        codec.close()
