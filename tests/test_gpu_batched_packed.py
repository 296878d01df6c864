"""Batched calls on short strings: a warp step packs the 16-byte chunks of many strings, so what
can go wrong sits at the strings' ends: a string's words next to another string's, strings of a
few bytes at every alignment, empty ones between them, an ill-formed one whose neighbours must
not change, and outputs that do not lie back to back.  Expected values come from oracle/ only
(exact: bytes, counts and kinds)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

TEXT = ("a", "é", "中", "\U0001F600", "￿", "퟿", "ࠀ", "߿")
BAD8 = (b"\x80", b"\xc1\xbf", b"\xe0\x9f\xbf", b"\xed\xa0\x80", b"\xf4\x90\x80\x80", b"\xff", b"\xf0", b"\xf0" * 20,
        b"\xe4\xb8", b"\x80" * 33)
BAD16 = ([0xD800], [0xDC00], [0xDBFF, 0x41], [0xDC00] * 17, [0xD800] * 17)


def _strings(longest, count, seed, wide):
    """Strings of 0..longest units over characters of every size, one in five ill-formed."""
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(count):
        n = int(rng.integers(0, longest + 1))
        s = "".join(TEXT[int(k)] for k in rng.integers(0, len(TEXT) if rng.random() < 0.7 else 1, size=n))
        if wide:
            u = np.frombuffer(s.encode("utf-16-le"), np.uint16)[:n]
            if rng.random() < 0.2:
                u = np.concatenate([u, np.array(BAD16[int(rng.integers(0, len(BAD16)))], np.uint16)])
        else:
            u = np.frombuffer(s.encode("utf-8"), np.uint8)[:n]  # may cut a character: ill-formed too
            if rng.random() < 0.2:
                u = np.concatenate([u, np.frombuffer(BAD8[int(rng.integers(0, len(BAD8)))], np.uint8)])
        out.append(u)
    return out


@pytest.mark.parametrize("gap", [0, 3])
@pytest.mark.parametrize("longest,count", [(3, 900), (17, 700), (40, 2500), (600, 300)])
@pytest.mark.parametrize("wide", [False, True])
def test_short_strings(wide, longest, count, gap):
    import torch
    from paper_2111_08692_gb300 import STATUS, Codec
    strings = _strings(longest, count, 100 * longest + gap + wide, wide)
    src = np.concatenate(strings) if count else np.zeros(0, np.uint8)
    off = np.concatenate([[0], np.cumsum([s.size for s in strings])]).astype(np.int64)
    length = oracle.utf8_length_from_utf16le if wide else oracle.utf16_length_from_utf8
    convert = oracle.convert_utf16le_to_utf8 if wide else oracle.convert_utf8_to_utf16le
    validate = oracle.validate_utf16le if wide else oracle.validate_utf8
    lens = np.array([length(s) for s in strings], np.int64)
    # outputs back to back, or in slots with canaries between them
    dst_off = np.concatenate([[0], np.cumsum(lens + gap)]).astype(np.int64)
    codec = Codec(0, max_units=1 << 20)
    try:
        d_src = torch.from_numpy(src.view(np.int16) if wide else src).cuda()
        d_off, d_dst_off = torch.from_numpy(off).cuda(), torch.from_numpy(dst_off).cuda()
        canary = 0x5A if wide else 0x5A5A
        total = int(dst_off[-1])
        dst = torch.full((total + 64,), canary, dtype=torch.uint8 if wide else torch.int16, device="cuda")
        got_len = (codec.utf8_length_from_utf16le_batched if wide else codec.utf16_length_from_utf8_batched)(d_src, d_off)
        assert np.array_equal(got_len.cpu().numpy(), lens)
        check = (codec.validate_utf16le_batched if wide else codec.validate_utf8_batched)(d_src, d_off).cpu().numpy()
        res = (codec.convert_utf16le_to_utf8_batched if wide else codec.convert_utf8_to_utf16le_batched)(
            d_src, d_off, dst[:total], d_dst_off).cpu().numpy()
        out = dst.cpu().numpy().view(np.uint8 if wide else np.uint16)
        for i, s in enumerate(strings):
            want = validate(s)
            assert (STATUS[int(check[i, 0]) & 0xFFFFFFFF], int(check[i, 1])) == want, (i, s)
            kind, units = convert(s, int(lens[i]))
            assert (STATUS[int(res[i, 0]) & 0xFFFFFFFF], int(res[i, 1])) == kind, (i, s)
            valid = int(lens[i]) if want[0] == "OK" else int(length(s[:want[1]]))
            a = int(dst_off[i])
            assert np.array_equal(out[a:a + valid], units[:valid]), (i, s)
            assert (out[a + int(lens[i]):int(dst_off[i + 1])] == canary).all() or want[0] != "OK", (i, s)
        assert (out[total:] == canary).all()
    finally:
        codec.close()


@pytest.mark.parametrize("wide", [False, True])
def test_small_capacities(wide):
    """Slots a few units too small: the defined prefix of the slot, the required length, no neighbour touched."""
    import torch
    from paper_2111_08692_gb300 import STATUS, Codec
    strings = [s for s in _strings(40, 600, 9 + wide, wide) if (oracle.validate_utf16le if wide else oracle.validate_utf8)(s)[0] == "OK"]
    src = np.concatenate(strings)
    off = np.concatenate([[0], np.cumsum([s.size for s in strings])]).astype(np.int64)
    convert = oracle.convert_utf16le_to_utf8 if wide else oracle.convert_utf8_to_utf16le
    lens = np.array([(oracle.utf8_length_from_utf16le if wide else oracle.utf16_length_from_utf8)(s) for s in strings], np.int64)
    caps = np.maximum(lens - np.arange(lens.size) % 3, 0)
    dst_off = np.concatenate([[0], np.cumsum(caps)]).astype(np.int64)
    codec = Codec(0, max_units=1 << 20)
    try:
        d_src = torch.from_numpy(src.view(np.int16) if wide else src).cuda()
        dst = torch.zeros(int(dst_off[-1]), dtype=torch.uint8 if wide else torch.int16, device="cuda")
        res = (codec.convert_utf16le_to_utf8_batched if wide else codec.convert_utf8_to_utf16le_batched)(
            d_src, torch.from_numpy(off).cuda(), dst, torch.from_numpy(dst_off).cuda()).cpu().numpy()
        out = dst.cpu().numpy().view(np.uint8 if wide else np.uint16)
        for i, s in enumerate(strings):
            kind, units = convert(s, int(caps[i]))
            assert (STATUS[int(res[i, 0]) & 0xFFFFFFFF], int(res[i, 1])) == kind, (i, s)
            assert np.array_equal(out[int(dst_off[i]):int(dst_off[i + 1])], units[:int(caps[i])]), (i, s)
    finally:
        codec.close()
