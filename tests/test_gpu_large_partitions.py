"""The transcoders' 16 KiB instance, which inputs past a line that depends on the device take: errors,
cut characters, capacities, alignments, early exit, repeated runs and the timeout hook around its lanes
(32 bytes), regions (1 KiB), warp slices (4 KiB) and partitions, in all four directions.  A case is a short
head or tail around a fixed valid filler that carries the buffer past the line; expected values are the
oracle's on head, filler and tail, each of whole characters (exact)."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

PART = 16384
BAD8 = [bytes.fromhex(h) for h in ("80", "c1bf", "c3", "e09fbf", "eda080", "f08fbfbf", "f4908080", "f09f98", "ff")]
BAD16 = ([0xD800], [0xDC00], [0xDBFF, 0x41], [0xDFFF, 0xDFFF])


class Large:
    """One direction: wide: from UTF-16 (else from UTF-8); be: the UTF-16 side is big-endian."""

    def __init__(self, torch, codec, wide, be):
        self.torch, self.codec, self.wide, self.be = torch, codec, wide, be
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        line = sms * 8 * 4096 * 3 // 2
        u8, u16 = W.profile_buffers("mixed", line + 40000, (line + 40000) // 2, 83, cache=False)
        self.convert = oracle.convert_utf16le_to_utf8 if wide else oracle.convert_utf8_to_utf16le
        self.length = oracle.utf8_length_from_utf16le if wide else oracle.utf16_length_from_utf8
        self.unit = 2 if wide else 1
        self.filler = u16 if wide else u8
        assert self.filler.size * self.unit > line
        (kind, _), out = self.convert(self.filler)
        assert kind == "OK"
        starts = np.flatnonzero((self.filler & 0xFC00) != 0xDC00 if wide else (self.filler & 0xC0) != 0x80)
        self.lead = self.filler[:starts[4]]  # whole characters: what an error at a head's end runs into
        self.filler_out = self._out(out)
        self.filler_dev = self._dev(self.filler)
        call = {(False, False): "convert_utf8_to_utf16le", (False, True): "convert_utf8_to_utf16be",
                (True, False): "convert_utf16le_to_utf8", (True, True): "convert_utf16be_to_utf8"}[wide, be]
        self.call = getattr(codec, call)
        self.src = torch.zeros(self.filler.size + 8 * PART, dtype=self.filler_dev.dtype, device="cuda")
        self.dst = torch.zeros(self.filler_out.numel() + 24 * PART, dtype=self.filler_out.dtype, device="cuda")

    def _dev(self, a):
        a = np.ascontiguousarray(a)
        if self.wide:
            a = (a.byteswap() if self.be else a).view(np.int16)
        return self.torch.from_numpy(a.copy()).cuda()

    def _out(self, a):
        if not self.wide:
            a = (a.byteswap() if self.be else a).view(np.int16)
        return self.torch.from_numpy(np.ascontiguousarray(a).copy()).cuda()

    def check(self, head=None, tail=None, src_off=0, dst_off=0, cap=None, early=None):
        """head + filler + tail at the given alignments (units past a 256-byte boundary)."""
        from paper_2111_08692_gb300 import result_tuple
        torch = self.torch
        none = self.filler[:0]
        head, tail = none if head is None else head, none if tail is None else tail
        (hk, hc), hout = self.convert(np.concatenate([head, self.lead]))
        h_ok = hk == "OK"
        hout = self._out(hout)
        n_head = self.length(head)
        (tk, tc), tout = self.convert(tail)
        tout = self._out(tout)
        total = n_head + self.filler_out.numel() + self.length(tail)
        cap = total if cap is None else (cap if cap >= 0 else total + cap)
        if not h_ok:
            want, defined = (hk, hc), self.length(head[:hc])
        elif tk != "OK":
            want = (tk, head.size + self.filler.size + tc)
            defined = n_head + self.filler_out.numel() + self.length(tail[:tc])
        else:
            want, defined = ("OK" if total <= cap else "OUTPUT_TOO_SMALL", total), total
        defined = min(defined, cap)
        a, b = src_off + head.size, src_off + head.size + self.filler.size
        if head.size:
            self.src[src_off:a] = self._dev(head)
        self.src[a:b] = self.filler_dev
        if tail.size:
            self.src[b:b + tail.size] = self._dev(tail)
        canary = 0x5A
        self.dst.fill_(canary)
        n = head.size + self.filler.size + tail.size
        if early is not None:
            self.codec.set_early_exit(early)
        got = result_tuple(self.call(self.src[src_off:src_off + n], self.dst[dst_off:dst_off + cap], cap=cap))
        if early is not None:
            self.codec.set_early_exit(True)
        where = (head.size, tail.size, src_off, dst_off, cap, early)
        assert got == want, (got, want, where)
        out = self.dst[dst_off:dst_off + defined]
        pieces = [hout[:n_head], self.filler_out, tout]
        at = 0
        for p in pieces:
            m = min(p.numel(), defined - at)
            assert torch.equal(out[at:at + m], p[:m]), where
            at += m
        assert at == defined, where
        assert bool((self.dst[:dst_off] == canary).all()) and bool((self.dst[dst_off + cap:] == canary).all()), where


@pytest.fixture(scope="module")
def codec():
    import torch
    from paper_2111_08692_gb300 import Codec
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = Codec(0, max_units=1 << 24)
    yield c
    c.close()


@pytest.fixture(scope="module", params=[(False, False), (False, True), (True, False), (True, True)],
                ids=["8to16le", "8to16be", "16leto8", "16beto8"])
def large(request, codec):
    import torch
    return Large(torch, codec, *request.param)


def _text(large, size, profile="mixed", seed=84):
    """`size` units or a little fewer of whole characters, and where characters start."""
    u8, u16 = W.profile_buffers(profile, 4 * PART, 2 * PART, seed, cache=False)
    a = u16 if large.wide else u8
    starts = np.flatnonzero((a & 0xFC00) != 0xDC00 if large.wide else (a & 0xC0) != 0x80)
    return a[:starts[np.searchsorted(starts, size, side="right") - 1]], starts


def _bads(large):
    return [np.array(b, np.uint16) for b in BAD16] if large.wide else [np.frombuffer(b, np.uint8) for b in BAD8]


EDGES = (32, 1024, 3072, 4096, 12288, PART, PART + 1024, 2 * PART)  # bytes


def test_errors_at_the_start(large):
    """Each kind of error at characters around each edge of the first partitions."""
    text, starts = _text(large, 3 * PART // large.unit)
    for edge in EDGES:
        for k, bad in enumerate(_bads(large)):
            off = (0, 3, 13)[k % 3]
            e = edge // large.unit - off
            for i in sorted({int(starts[np.searchsorted(starts, max(e + d, 0))]) for d in range(-4, 3)}):
                large.check(np.concatenate([text[:i], bad, text[i:]]), src_off=off, dst_off=k, early=bool(k & 1))


def test_errors_at_the_end(large):
    """Errors and cut characters in the buffer's last regions, whose partition lies partly outside."""
    text, starts = _text(large, PART // large.unit)
    for n in (0, 1, 15, 16, 17, 500, 512, 700, 2048, 5000):
        j = int(starts[np.searchsorted(starts, n)])
        for k, bad in enumerate(_bads(large)):
            large.check(tail=np.concatenate([text[:j], bad]), src_off=k, dst_off=k, early=bool(k & 1))
            large.check(tail=np.concatenate([text[:j], bad, text[j:j + 900]]), src_off=8 - k if k < 8 else 0)


@pytest.mark.parametrize("profile", ["ascii", "latin", "cjk", "emoji"])
def test_characters_cut_by_edges(large, profile):
    """A character of every size across every edge, in text of one class, at several alignments."""
    text, starts = _text(large, 3 * PART // large.unit, profile)
    code = "utf-16-le" if large.wide else "utf-8"
    dtype = np.uint16 if large.wide else np.uint8
    for edge in EDGES:
        for k, ch in enumerate(("é", "中", "\U0001F600")):
            c = np.frombuffer(ch.encode(code), dtype)
            for d in range(1, max(c.size, 2)):
                off = (0, 1, 7)[k]
                at = edge // large.unit - d - off  # where the character starts
                j = int(starts[np.searchsorted(starts, max(at - 3, 0), side="right") - 1])
                pad = np.full(at - j, 0x41, dtype)
                large.check(np.concatenate([text[:j], pad, c, text[j:]]), src_off=off, dst_off=(k * 5) % 8)


def test_capacities(large):
    text, _ = _text(large, 2 * PART // large.unit)
    n = large.length(text)
    for k, cap in enumerate((0, 1, 7, 8, 9, 511, 512, 1024, 4095, n - 1, n, n + 1, -1, -17, -5000)):
        large.check(text, cap=cap, src_off=k % 4, dst_off=k % 16)
    # an error takes precedence over the capacity
    large.check(text, tail=_bads(large)[0], cap=100)


def test_alignments_and_repeated_runs(large):
    text, _ = _text(large, PART // large.unit)
    for off in range(16):
        large.check(text, src_off=off, dst_off=(5 * off) % 16)
    for _ in range(20):
        large.check(text, text)


def test_a_wait_that_runs_out(large):
    from paper_2111_08692_gb300 import result_tuple
    large.check()
    large.codec.set_wait_limit(2000)
    large.codec.debug_skip_publish(2)  # partition 3 must look back past it
    try:
        r = result_tuple(large.call(large.src[:large.filler.size], large.dst, cap=large.dst.numel()))
    finally:
        large.codec.debug_skip_publish(-1)
        large.codec.set_wait_limit(1 << 22)
    assert r[0] == "TIMEOUT"
    large.check()


@pytest.mark.parametrize("size", [3 * PART, None], ids=["4KiB", "16KiB"])
@pytest.mark.parametrize("be", [False, True])
def test_second_surrogate_first_in_a_partition(codec, size, be):
    """An unpaired second surrogate that is the first word of a partition, after a region with pairs: the
    last lane of that region flags it, in the partition before the one it lies in, so that with early exit
    the latter may be left out; the result is the same."""
    import torch
    from paper_2111_08692_gb300 import result_tuple
    large = Large(torch, codec, True, be)
    part = 4096 if size else PART
    for at in (part // 2, part, 4 * part // 2):
        pairs = np.tile(np.array([0xD83D, 0xDE00], np.uint16), at // 2)
        head = np.concatenate([pairs, np.array([0xDC00, 0x41], np.uint16), pairs[:600]])
        for early in (True, False):
            if size is None:
                large.check(head, early=early)
                continue
            codec.set_early_exit(early)
            src = large._dev(head)
            dst = torch.zeros(3 * head.size, dtype=torch.uint8, device="cuda")
            assert result_tuple(large.call(src, dst)) == ("SURROGATE", at)
            out = torch.from_numpy(oracle.convert_utf16le_to_utf8(pairs)[1].copy()).cuda()
            assert torch.equal(dst[:out.numel()], out)
            codec.set_early_exit(True)
