"""A batch in which every string is a long one, and of more of them than all CTAs' lists hold at once: the
lists fill to their stop mark, are worked off and filled again.  Every string is one of a few kinds, so the
expected results are the oracle's on each kind, repeated (exact)."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

LISTED = 512  # long strings a CTA sets aside at most (csrc/gbu_batch.cu)


@pytest.mark.parametrize("wide", [False, True])
def test_lists_of_long_strings_fill_up(wide):
    import torch
    from paper_2111_08692_gb300 import STATUS_CODE, Codec
    B = torch.cuda.get_device_properties(0).multi_processor_count * 5 * LISTED
    u8, u16 = W.profile_buffers("mixed", 1 << 16, 1 << 15, 95, cache=False)
    text = u16 if wide else u8
    starts = np.flatnonzero((text & 0xFC00) != 0xDC00 if wide else (text & 0xC0) != 0x80)
    shortest = 256 if wide else 512  # units of 512 bytes
    kinds = []
    for k in range(24):
        a = int(starts[np.searchsorted(starts, 900 * k)])
        s = np.array(text[a:int(starts[np.searchsorted(starts, a + shortest + k % 5)])])
        if k % 6 == 5:
            s[int(10 * k)] = 0xDC00 if wide else 0xFF
        kinds.append(s)
    validate = oracle.validate_utf16le if wide else oracle.validate_utf8
    length = oracle.utf8_length_from_utf16le if wide else oracle.utf16_length_from_utf8
    convert = oracle.convert_utf16le_to_utf8 if wide else oracle.convert_utf8_to_utf16le
    reps = B // len(kinds) + 1
    n = len(kinds) * reps
    sizes, lens = [np.tile([f(s) for s in kinds], reps) for f in (len, length)]
    off, dst_off = [torch.from_numpy(np.concatenate([[0], np.cumsum(x)]).astype(np.int64)).cuda() for x in (sizes, lens)]
    one = np.concatenate(kinds)
    src = torch.from_numpy(one.view(np.int16) if wide else one).cuda().repeat(reps)
    outs = [convert(s)[1] for s in kinds]
    want_out = np.concatenate([np.resize(o, int(length(s))) for o, s in zip(outs, kinds)])
    defined = np.concatenate([np.arange(int(length(s))) < (int(length(s)) if validate(s)[0] == "OK" else
                                                           int(length(s[:validate(s)[1]]))) for s in kinds])
    codec = Codec(0, max_units=1 << 20)
    try:
        for op in ("validate", "length", "convert"):
            name = {"validate": ("validate_utf8", "validate_utf16le"),
                    "length": ("utf16_length_from_utf8", "utf8_length_from_utf16le"),
                    "convert": ("convert_utf8_to_utf16le", "convert_utf16le_to_utf8")}[op][wide]
            codec.set_batch_config(name, 8, 256, 512)
            call = getattr(codec, name + "_batched")
            if op == "length":
                assert torch.equal(call(src, off), dst_off[1:] - dst_off[:-1])
                continue
            if op == "convert":
                dst = torch.zeros(int(dst_off[-1]), dtype=torch.uint8 if wide else torch.int16, device="cuda")
                res = call(src, off, dst, dst_off)
                want = [convert(s, int(length(s)))[0] for s in kinds]
                mask = torch.from_numpy(defined).cuda()
                exp = torch.from_numpy(want_out if wide else want_out.view(np.int16)).cuda()
                rows = dst.view(reps, -1)
                assert bool(((rows == exp) | ~mask).all())
            else:
                res = call(src, off)
                want = [validate(s) for s in kinds]
            rows = torch.tensor([[STATUS_CODE[k], c] for k, c in want], dtype=torch.int64, device="cuda").repeat(reps, 1)
            got = res.clone()
            got[:, 0] &= 0xFFFFFFFF
            assert torch.equal(got, rows) and n == got.shape[0]
    finally:
        codec.close()
