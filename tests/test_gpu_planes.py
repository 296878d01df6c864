"""UTF-8 validation on bit planes (32 bytes per lane, 1 KiB regions, 4 KiB tiles): every special
leading byte with second bytes on both sides of its bound, at the positions where a sequence
crosses a lane, a region or a tile, at several source alignments; and the lengths around the tiles
that are counted without neighbouring words.  Expected values come from oracle/ only (exact)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SEQUENCES = [bytes([a, b]) + t
             for a, bs in ((0xC1, (0xBF,)), (0xC2, (0x7F, 0x80)), (0xE0, (0x9F, 0xA0)), (0xED, (0x9F, 0xA0)),
                           (0xEF, (0xBF, 0xC0)), (0xF0, (0x8F, 0x90)), (0xF4, (0x8F, 0x90)), (0xF5, (0x80,)), (0xFF, (0x80,)))
             for b in bs for t in (b"", b"\x80", b"\x80\x80", b"\x80\x80\x80")]


@pytest.mark.parametrize("edge", [32, 1024, 4096, 3 * 4096])
@pytest.mark.parametrize("shift", [0, 1, 17])
def test_sequences_at_edges(edge, shift):
    import torch
    from paper_2111_08692_gb300 import Codec, result_tuple
    codec = Codec(0, max_units=1 << 20)
    try:
        for lead in range(edge - 4, edge + 1):
            for cut in (False, True):  # text after the sequence, or the buffer's end
                for seq in SEQUENCES:
                    at = lead - shift
                    data = np.frombuffer(b"a" * at + seq + (b"" if cut else b"bcd" * 1500), np.uint8)
                    buf = torch.zeros(data.size + shift, dtype=torch.uint8, device="cuda")
                    buf[shift:] = torch.from_numpy(data.copy())
                    got = result_tuple(codec.validate_utf8(buf[shift:]))
                    assert got == oracle.validate_utf8(data), (lead, cut, seq.hex())
    finally:
        codec.close()


@pytest.mark.parametrize("n", [4095, 4096, 4104, 8192, 3 * 4096 + 5])
@pytest.mark.parametrize("shift", [0, 3])
def test_lengths_around_tiles(n, shift):
    """Arbitrary bytes and words (the length formulas are defined for any input)."""
    import torch
    from paper_2111_08692_gb300 import Codec
    rng = np.random.default_rng(n + shift)
    u8 = rng.integers(0, 256, size=n, dtype=np.uint8)
    u16 = np.where(rng.random(n) < 0.5, rng.integers(0, 0x900, size=n), rng.integers(0xD700, 0xE100, size=n)).astype(np.uint16)
    codec = Codec(0, max_units=1 << 20)
    try:
        b8 = torch.zeros(n + shift, dtype=torch.uint8, device="cuda")
        b8[shift:] = torch.from_numpy(u8)
        b16 = torch.zeros(n + shift, dtype=torch.int16, device="cuda")
        b16[shift:] = torch.from_numpy(u16.view(np.int16))
        assert int(codec.utf16_length_from_utf8(b8[shift:]).item()) == oracle.utf16_length_from_utf8(u8)
        assert int(codec.utf8_length_from_utf16le(b16[shift:]).item()) == oracle.utf8_length_from_utf16le(u16)
        be = torch.zeros(n + shift, dtype=torch.int16, device="cuda")
        be[shift:] = torch.from_numpy(u16.byteswap().view(np.int16))
        assert int(codec.utf8_length_from_utf16be(be[shift:]).item()) == oracle.utf8_length_from_utf16le(u16)
    finally:
        codec.close()


@pytest.mark.parametrize("shift", [0, 5])
@pytest.mark.parametrize("at", [32, 1022, 1024, 2048, 4094, 4096, 8192])
def test_sequences_in_two_byte_text(at, shift):
    """Regions of two-byte characters are judged without the planes: every sequence inside them."""
    import torch
    from paper_2111_08692_gb300 import Codec, result_tuple
    codec = Codec(0, max_units=1 << 20)
    try:
        for lead in range(at, at + 4):
            for seq in SEQUENCES + ["\u0416".encode(), "\u6c34".encode(), "\U0001f600".encode()]:
                pairs = (lead - shift) // 2
                head = "\u044f".encode() * pairs + b"a" * (lead - shift - 2 * pairs)
                data = np.frombuffer(head + seq + "\u00e9".encode() * 6000, np.uint8)
                buf = torch.zeros(data.size + shift, dtype=torch.uint8, device="cuda")
                buf[shift:] = torch.from_numpy(data.copy())
                got = result_tuple(codec.validate_utf8(buf[shift:]))
                assert got == oracle.validate_utf8(data), (lead, seq.hex())
    finally:
        codec.close()
