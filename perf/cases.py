"""Timed cases of the library: what a program that uses it has it do, call by call.

Every case draws its text on the GPU from a seed (the character mixtures of the test inputs:
mixed, ASCII, Latin, Cyrillic, CJK, emoji), keeps what such a program keeps (a context, the
input, an output buffer that holds the largest output, zeroed) and runs one pass of public calls.

Kinds:
  sync       one small text through the host-synchronising UTF-8 -> UTF-16LE call: latency
  six        the six calls (validate, length, convert, both directions) on one text
  check8     UTF-8 validation of one buffer and the length of its UTF-16 form
  to16, to8  UTF-8 -> UTF-16LE and UTF-16LE -> UTF-8 of one buffer
  dirty      validation and conversion of a UTF-8 buffer with an invalid byte part way
  batch      many strings: lengths, output offsets and conversion, both directions
  formats    the conversions between UTF-8 and UTF-16BE / UTF-32
  serve      a burst of requests of mixed sizes through the serving loop
"""
from __future__ import annotations

import math
import random
import time

import numpy as np
import torch

from paper_2111_08692_gb300 import Codec
from paper_2111_08692_gb300 import binding as B

MIB = 1 << 20
GIB = 1 << 30
CHUNK = 1 << 25  # characters drawn and encoded at a time

PROFILES = ("mixed", "ascii", "latin", "cyrillic", "cjk", "emoji")
# expected UTF-8 bytes and UTF-16 words per character
BYTES8 = {"mixed": 1.9, "ascii": 1.0, "latin": 1.05, "cyrillic": 1.7, "cjk": 2.7, "emoji": 1.9}
WORDS16 = {"mixed": 1.1, "ascii": 1.0, "latin": 1.0, "cyrillic": 1.0, "cjk": 1.0, "emoji": 1.3}
BATCH_MEDIAN, BATCH_SIGMA, BATCH_MAX = 64, 1.5, 65536
SERVE_MIN, SERVE_MAX = 16, 16 * MIB
SERVE_PROFILES = PROFILES[1:]


def listed() -> list[dict]:
    return [
        # a short document converted by a program that waits for it (one request, one field);
        # an odd size, smaller than one unit of the kernels' work
        {"name": "small_sync", "kind": "sync", "profile": "mixed", "n": 4099},
        # the 1 MiB mixed buffer: every call on a text that fits in L2
        {"name": "mixed_1mib", "kind": "six", "profile": "mixed", "n": MIB, "shift": 0},
        # plain ASCII (logs, markup, source code): every call on a text larger than L2
        {"name": "ascii_256mib", "kind": "six", "profile": "ascii", "n": 256 * MIB, "shift": 0},
        # checking a large CJK file on ingest and sizing its UTF-16 form
        {"name": "check_cjk_1gib", "kind": "check8", "profile": "cjk", "n": GIB, "shift": 0},
        # a large Western European file read into a UTF-16 program
        {"name": "to16_latin_1gib", "kind": "to16", "profile": "latin", "n": GIB, "shift": 0},
        # a CJK text inside a larger buffer: odd size, unaligned input and output
        {"name": "to16_cjk_odd", "kind": "to16", "profile": "cjk", "n": 100_000_003, "shift": 5},
        # writing a large Cyrillic UTF-16 text as UTF-8
        {"name": "to8_cyrillic_1gib", "kind": "to8", "profile": "cyrillic", "n": GIB // 2, "shift": 0},
        # chat text full of surrogate pairs: odd size, unaligned input and output
        {"name": "to8_emoji_odd", "kind": "to8", "profile": "emoji", "n": 20_000_001, "shift": 3},
        # a file with an invalid byte part way: the first error is what the caller wants
        {"name": "dirty_cyrillic", "kind": "dirty", "profile": "cyrillic", "words": 150_000_000, "at": 0.6},
        # a column of a million short strings, both directions into packed outputs
        {"name": "batch_1m", "kind": "batch", "strings": 1_000_000},
        # the other byte order and UTF-32
        {"name": "formats_64mib", "kind": "formats", "profile": "mixed", "n": 64 * MIB},
        # requests of 16 B to 16 MiB that arrive at once at a server
        {"name": "serve_burst", "kind": "serve", "requests": 64},
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random) -> dict:
    kind = rng.choice(("sync", "six", "check8", "to16", "to16", "to8", "to8", "dirty", "batch", "formats", "serve"))
    profile = rng.choice(PROFILES)
    if kind == "sync":
        return {"kind": kind, "profile": profile, "n": _log_int(rng, 64, 1 << 16)}
    if kind == "six":
        return {"kind": kind, "profile": profile, "n": _log_int(rng, 1 << 14, 256 * MIB), "shift": rng.choice((0, 0, 1, 7))}
    if kind in ("check8", "to16"):
        return {"kind": kind, "profile": profile, "n": _log_int(rng, 1 << 16, GIB), "shift": rng.choice((0, 1, 5, 15))}
    if kind == "to8":
        return {"kind": kind, "profile": profile, "n": _log_int(rng, 1 << 15, GIB // 2), "shift": rng.choice((0, 1, 3, 7))}
    if kind == "dirty":
        return {"kind": kind, "profile": profile, "words": _log_int(rng, MIB // 2, 128 * MIB), "at": round(rng.uniform(0.05, 0.95), 3)}
    if kind == "batch":
        return {"kind": kind, "strings": _log_int(rng, 1000, 1_000_000)}
    if kind == "formats":
        return {"kind": kind, "profile": profile, "n": _log_int(rng, 1 << 16, 64 * MIB)}
    return {"kind": kind, "requests": rng.randint(16, 64)}


# ---- text ---------------------------------------------------------------------------------

def _generator(seed: int) -> torch.Generator:
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(g, lo, hi, m):
    return torch.randint(lo, hi, (m,), generator=g, device="cuda", dtype=torch.int32)


def _codepoints(profile: str, m: int, g: torch.Generator) -> torch.Tensor:
    """m code points of a profile (int32)."""
    if profile == "ascii":
        return _uniform(g, 0x20, 0x7F, m)
    u = torch.rand(m, generator=g, device="cuda")
    if profile == "mixed":
        bmp = _uniform(g, 0x800, 0xF800, m)
        bmp = torch.where(bmp >= 0xD800, bmp + 0x800, bmp)
        out = torch.where(u < 0.9, bmp, _uniform(g, 0x10000, 0x110000, m))
        out = torch.where(u < 0.7, _uniform(g, 0x80, 0x800, m), out)
        return torch.where(u < 0.5, _uniform(g, 0, 0x80, m), out)
    if profile == "cyrillic":
        punct = torch.tensor([c for c in range(0x21, 0x7F) if not chr(c).isalnum()], dtype=torch.int32, device="cuda")
        out = torch.where(u < 0.85, 0x20, punct[_uniform(g, 0, punct.numel(), m).long()]).to(torch.int32)
        return torch.where(u < 0.7, _uniform(g, 0x400, 0x500, m), out)
    share, lo, hi = {"latin": (0.05, 0xC0, 0x180), "cjk": (0.85, 0x4E00, 0xA000), "emoji": (0.30, 0x1F300, 0x1FB00)}[profile]
    return torch.where(u < share, _uniform(g, lo, hi, m), _uniform(g, 0x20, 0x7F, m))


def _size8(c):
    return 1 + (c >= 0x80).to(torch.int32) + (c >= 0x800).to(torch.int32) + (c >= 0x10000).to(torch.int32)


def _size16(c):
    return 1 + (c >= 0x10000).to(torch.int32)


def _put8(out, at, c):
    """Writes the UTF-8 bytes of code points c at positions at."""
    size = _size8(c)
    lead = torch.where(size == 1, c, torch.where(size == 2, 0xC0 | (c >> 6), torch.where(size == 3, 0xE0 | (c >> 12), 0xF0 | (c >> 18))))
    out[at] = lead.to(torch.uint8)
    for k in (1, 2, 3):  # the k-th byte of the characters that have one
        sel = size > k
        cs, ps = c[sel], at[sel] + k
        out[ps] = (0x80 | ((cs >> (6 * (size[sel] - 1 - k))) & 0x3F)).to(torch.uint8)


def _put16(out, at, c):
    """Writes the UTF-16 words of code points c at positions at."""
    big = c >= 0x10000
    out[at] = torch.where(big, 0xD800 + ((c - 0x10000) >> 10), c).to(torch.int16)
    out[at[big] + 1] = (0xDC00 + (c[big] & 0x3FF)).to(torch.int16)


def _encode(text: list[torch.Tensor], size, put, dtype, shift: int = 0) -> torch.Tensor:
    """The text's units, as a view `shift` units into its buffer."""
    n = sum(int(size(c).sum()) for c in text)
    buf = torch.zeros(n + shift, dtype=dtype, device="cuda")
    out, base = buf[shift:], 0
    for c in text:
        end = torch.cumsum(size(c).long(), 0)
        put(out, end - size(c) + base, c)
        base += int(end[-1]) if c.numel() else 0
    return out


def _utf8(text, shift=0):
    return _encode(text, _size8, _put8, torch.uint8, shift)


def _utf16(text, shift=0):
    return _encode(text, _size16, _put16, torch.int16, shift)


def _text(profile: str, seed: int, n: int, size=_size8) -> list[torch.Tensor]:
    """Code points (in pieces) whose encoding has exactly n units, U+0020 at its end if need be."""
    g, left, parts = _generator(seed), n, []
    mean = BYTES8[profile] if size is _size8 else WORDS16[profile]
    while left > 0:
        c = _codepoints(profile, min(CHUNK, int(left / mean * 1.01) + 16), g)
        end = torch.cumsum(size(c).long(), 0)
        k = int((end <= left).sum())
        if k < c.numel():
            pad = left - (int(end[k - 1]) if k else 0)
            c = torch.cat((c[:k], torch.full((pad,), 0x20, dtype=torch.int32, device="cuda")))
            left = 0
        else:
            left -= int(end[-1])
        parts.append(c)
    return parts


def _batch_text(strings: int, seed: int):
    """Code points of all strings back to back and each string's first character (strings + 1):
    log-normal lengths (its quantiles, in random order), each string of a profile drawn uniformly."""
    g = _generator(seed)
    q = (torch.arange(strings, device="cuda", dtype=torch.float64) + 0.5) / strings
    length = torch.exp(math.log(BATCH_MEDIAN) + BATCH_SIGMA * torch.special.ndtri(q))
    length = length[torch.randperm(strings, generator=g, device="cuda")]
    kinds = PROFILES[1:]
    which = torch.randint(0, len(kinds), (strings,), generator=g, device="cuda")
    mean = torch.tensor([BYTES8[k] for k in kinds], device="cuda", dtype=torch.float64)[which]
    chars = (length.clamp(1, BATCH_MAX) / mean).round().clamp(min=1).long()
    start = torch.zeros(strings + 1, dtype=torch.int64, device="cuda")
    start[1:] = torch.cumsum(chars, 0)
    m = int(start[-1])
    of = torch.repeat_interleave(which, chars)
    c = torch.zeros(m, dtype=torch.int32, device="cuda")
    for k, profile in enumerate(kinds):
        c = torch.where(of == k, _codepoints(profile, m, g), c)
    return c, start


def _offsets(c, start, size):
    """Unit offsets of the strings that start at characters `start`."""
    end = torch.zeros(c.numel() + 1, dtype=torch.int64, device="cuda")
    end[1:] = torch.cumsum(size(c).long(), 0)
    return end[start]


def _batch_caps(strings: int) -> tuple[int, int]:
    """UTF-8 bytes and UTF-16 words that hold any batch of so many strings (twice the expected ones)."""
    n8 = strings * BATCH_MEDIAN * math.exp(BATCH_SIGMA ** 2 / 2)
    return int(2 * n8) + 4096, int(2 * n8) + 4096


def _serve_plan(case, seed):
    """(op, profile, units, seed) of each request: sizes log-uniform, one in ten validates only."""
    mix, rng = random.Random(case["requests"]), random.Random(seed)
    plan = []
    for k in range(case["requests"]):
        u = mix.random()
        op = "validate_utf8" if u < 0.05 else "validate_utf16le" if u < 0.10 else \
            "convert_utf8_to_utf16le" if u < 0.55 else "convert_utf16le_to_utf8"
        # sizes spread evenly over the range (not drawn), so that every burst is the same work
        size = SERVE_MIN * (SERVE_MAX / SERVE_MIN) ** ((k + 0.5) / case["requests"])
        wide = op in ("validate_utf16le", "convert_utf16le_to_utf8")
        plan.append((op, rng.choice(SERVE_PROFILES), max(1, int(size / (2 if wide else 1))), seed * 1009 + k))
    return plan


def _request_text(profile, n, seed, op):
    wide = op in ("validate_utf16le", "convert_utf16le_to_utf8")
    return _text(profile, seed, n, _size16 if wide else _size8), wide


# ---- the cases ------------------------------------------------------------------------------

def _result():
    return torch.empty(2, dtype=torch.int64, device="cuda")


def _swap(w: torch.Tensor) -> torch.Tensor:
    """The words with their two bytes exchanged."""
    return w.view(torch.uint8).view(-1, 2).flip(1).reshape(-1).view(torch.int16)


def _dst(units: int, dtype, shift: int = 0) -> torch.Tensor:
    return torch.zeros(units + shift, dtype=dtype, device="cuda")[shift:]


def _serve_dst(op: str, n: int):
    """The caller's own buffer for a request's output (None: a validation)."""
    if op.startswith("validate"):
        return None
    return _dst(n, torch.int16) if op == "convert_utf8_to_utf16le" else _dst(3 * n, torch.uint8)


def _in(dst: torch.Tensor, units: torch.Tensor) -> torch.Tensor:
    """A zeroed buffer with an output at its start."""
    dst[:units.numel()] = units
    return dst


def prepare(case: dict, seed: int) -> dict:
    kind = case["kind"]
    st = {"case": case}
    if kind == "serve":
        st["requests"] = []
        for op, profile, n, s in _serve_plan(case, seed):
            text, wide = _request_text(profile, n, s, op)
            st["requests"].append((op, _utf16(text) if wide else _utf8(text), _serve_dst(op, n)))
        st["server"] = B.Server(torch.cuda.current_device(), budget_bytes=2 * GIB, max_request_units=SERVE_MAX)
        torch.cuda.synchronize()
        return st
    if kind == "batch":
        c, start = _batch_text(case["strings"], seed)
        st["u8"], st["off8"] = _utf8([c]), _offsets(c, start, _size8)
        st["u16"], st["off16"] = _utf16([c]), _offsets(c, start, _size16)
        cap8, cap16 = _batch_caps(case["strings"])
        st["dst16"], st["dst8"] = _dst(cap16, torch.int16), _dst(cap8, torch.uint8)
        st["codec"] = Codec(max_units=max(st["u8"].numel(), case["strings"] + 1))
        return st
    if kind == "dirty":
        words = case["words"]
        text = _text(case["profile"], seed, words, _size16)
        st["u8"], _ = _dirty(text, words, case["at"])
        st["dst16"], st["codec"] = _dst(st["u8"].numel(), torch.int16), Codec(max_units=st["u8"].numel())
        return st
    shift, n = case.get("shift", 0), case["n"]
    text = _text(case["profile"], seed, n, _size16 if kind == "to8" else _size8)
    st["codec"] = Codec(max_units=n)
    if kind != "to8":
        st["u8"] = _utf8(text, shift)
    if kind in ("six", "to8"):
        st["u16"] = _utf16(text, shift)
    if kind in ("sync", "to16", "six"):
        st["dst16"] = _dst(n, torch.int16, shift)
    if kind in ("to8", "six"):
        st["dst8"] = _dst(3 * n if kind == "to8" else n, torch.uint8, shift)
    if kind == "formats":
        st["u32"] = torch.cat(text)
        st["be"] = _swap(_utf16(text))
        st["dst8"], st["dst8b"] = _dst(n, torch.uint8), _dst(n, torch.uint8)
        st["dstbe"], st["dst32"] = _dst(n, torch.int16), _dst(n, torch.int32)
    return st


def _dirty(text, words: int, at: float):
    """The text's UTF-8 with a byte FF over a character that starts at UTF-16 word int(at x words), or
    one word before where a pair covers that word; and the place of that byte."""
    want, seen, place = int(at * words), 0, 0
    u8 = _utf8(text)
    for c in text:
        end16 = torch.cumsum(_size16(c).long(), 0)
        k = int((end16 <= want - seen).sum())  # characters of this piece before the broken one
        place += int(_size8(c[:k]).sum())
        if k < c.numel():
            break
        seen += int(end16[-1])
    u8[place] = 0xFF
    return u8, place


class _DeviceView:
    """Device memory at an address, as torch.as_tensor takes it."""

    def __init__(self, address, units, typestr):
        self.__cuda_array_interface__ = {"data": (address, False), "shape": (units,), "typestr": typestr, "version": 2}


def _run_serve(st) -> list:
    server = st["server"]
    first = server.submit([(op, src, 0, k) for k, (op, src, _) in enumerate(st["requests"])])
    done = {}
    while len(done) < len(st["requests"]):
        got = server.poll()
        for c in got:
            done[c["id"] - first] = c
        if not got:
            time.sleep(0)
    out = [np.array([[B.STATUS_CODE[done[k]["status"]], done[k]["count"]] for k in range(len(done))], dtype=np.int64)]
    held = []
    for k, (op, _, dst) in enumerate(st["requests"]):
        c = done[k]
        if c["dst"]:
            view = _DeviceView(c["dst"], c["count"], "<i2" if op == "convert_utf8_to_utf16le" else "|u1")
            dst[:c["count"]].copy_(torch.as_tensor(view, device="cuda"))
            out.append(dst)
            held.append(c["id"])
    torch.cuda.current_stream().synchronize()  # the copies have read the server's outputs
    for rid in held:
        server.release(rid)
    return out


def run(st: dict):
    kind = st["case"]["kind"]
    if kind == "serve":
        return _run_serve(st)
    codec = st["codec"]
    if kind == "sync":
        status, count = codec.convert_utf8_to_utf16le_sync(st["u8"], st["dst16"])
        return [B.STATUS_CODE[status], count, st["dst16"]]
    if kind == "check8":
        return [codec.validate_utf8(st["u8"]), codec.utf16_length_from_utf8(st["u8"])]
    if kind == "to16":
        return [codec.convert_utf8_to_utf16le(st["u8"], st["dst16"]), st["dst16"]]
    if kind == "to8":
        return [codec.convert_utf16le_to_utf8(st["u16"], st["dst8"]), st["dst8"]]
    if kind == "six":
        return [codec.validate_utf8(st["u8"]), codec.utf16_length_from_utf8(st["u8"]),
                codec.convert_utf8_to_utf16le(st["u8"], st["dst16"]), st["dst16"],
                codec.validate_utf16le(st["u16"]), codec.utf8_length_from_utf16le(st["u16"]),
                codec.convert_utf16le_to_utf8(st["u16"], st["dst8"]), st["dst8"]]
    if kind == "dirty":
        return [codec.validate_utf8(st["u8"]), codec.convert_utf8_to_utf16le(st["u8"], st["dst16"]),
                st["dst16"][:int(st["case"]["at"] * st["case"]["words"]) - 1]]
    if kind == "formats":
        return [codec.convert_utf16be_to_utf8(st["be"], st["dst8"]), st["dst8"],
                codec.convert_utf8_to_utf16be(st["u8"], st["dstbe"]), st["dstbe"],
                codec.convert_utf32_to_utf8(st["u32"], st["dst8b"]), st["dst8b"],
                codec.convert_utf8_to_utf32(st["u8"], st["dst32"]), st["dst32"]]
    out = []  # batch
    for src, off, dst, length, convert in (
            (st["u8"], st["off8"], st["dst16"], codec.utf16_length_from_utf8_batched, codec.convert_utf8_to_utf16le_batched),
            (st["u16"], st["off16"], st["dst8"], codec.utf8_length_from_utf16le_batched, codec.convert_utf16le_to_utf8_batched)):
        lens = length(src, off)
        dst_off, total = codec.exclusive_scan_u64(lens)
        out += [lens, dst_off, total, convert(src, off, dst, dst_off), dst]
    return out


def work(case: dict) -> dict:
    """Bytes: every call's input once and its output once (results and offsets included)."""
    kind = case["kind"]
    if kind == "serve":
        total = 0
        for k in range(case["requests"]):
            size = SERVE_MIN * (SERVE_MAX / SERVE_MIN) ** ((k + 0.5) / case["requests"])
            total += size * (1 + 0.9 * (0.5 * 1.25 + 0.5 * 0.8))  # input, and the output of nine in ten
        return {"bytes": int(total), "flops": 0}
    if kind == "batch":
        s = case["strings"]
        mean = BATCH_MEDIAN * math.exp(BATCH_SIGMA ** 2 / 2)
        n8 = s * mean
        n16 = 2 * n8 * sum(WORDS16[p] / BYTES8[p] for p in PROFILES[1:]) / len(PROFILES[1:])
        # the lengths read an input and write 8 bytes a string, the scan reads and writes 8, the
        # conversion reads the input and two offsets and writes the output and 16 bytes a string
        return {"bytes": int(2 * n8 + n16 + 2 * n16 + n8 + 2 * s * (8 + 8 + 8 + 8 + 16 + 16)), "flops": 0}
    p = case["profile"]
    n = case["words"] if kind == "dirty" else case["n"]
    if kind in ("to8", "dirty"):
        n16 = 2 * n
        n8 = n * BYTES8[p] / WORDS16[p]
    else:
        n8 = n
        n16 = 2 * n * WORDS16[p] / BYTES8[p]
    n32 = 4 * n8 / BYTES8[p]
    total = {"sync": n8 + n16, "check8": 2 * n8, "to16": n8 + n16, "to8": n16 + n8, "six": 3 * n8 + n16 + 3 * n16 + n8,
             "dirty": (2 * n8 + n16) * case.get("at", 1.0), "formats": 2 * (n16 + n8) + 2 * (n32 + n8)}[kind]
    return {"bytes": int(total), "flops": 0}


def _pair(status: int, count: int) -> torch.Tensor:
    return torch.tensor([status, count], dtype=torch.int64)


def _lens(off):
    return off[1:] - off[:-1]


def exact(case: dict, seed: int):
    """The same outputs from the code points: every text here is valid but for the dirty one's byte."""
    kind = case["kind"]
    if kind == "serve":
        out = [np.zeros((case["requests"], 2), dtype=np.int64)]
        for k, (op, profile, n, s) in enumerate(_serve_plan(case, seed)):
            text, wide = _request_text(profile, n, s, op)
            if op.startswith("validate"):
                out[0][k] = (0, n)
            else:
                other = _utf8(text) if wide else _utf16(text)
                out[0][k] = (0, other.numel())
                out.append(_in(_serve_dst(op, n), other))
        return out
    if kind == "batch":
        c, start = _batch_text(case["strings"], seed)
        u8, u16 = _utf8([c]), _utf16([c])
        off8, off16 = _offsets(c, start, _size8), _offsets(c, start, _size16)
        out = []
        cap8, cap16 = _batch_caps(case["strings"])
        for units, off, cap in ((u16, off16, cap16), (u8, off8, cap8)):
            results = torch.stack((torch.zeros_like(off[1:]), _lens(off)), 1)
            out += [_lens(off), off, _pair(0, units.numel()), results, _in(_dst(cap, units.dtype), units)]
        return out
    if kind == "dirty":
        words = case["words"]
        text = _text(case["profile"], seed, words, _size16)
        _, place = _dirty(text, words, case["at"])
        return [_pair(1, place), _pair(1, place), _utf16(text)[:int(case["at"] * words) - 1]]
    n = case["n"]
    text = _text(case["profile"], seed, n, _size16 if kind == "to8" else _size8)
    if kind == "to8":
        u8 = _utf8(text)
        return [_pair(0, u8.numel()), _in(_dst(3 * n, torch.uint8), u8)]
    u16 = _utf16(text)
    words = u16.numel()
    if kind == "check8":
        return [_pair(0, n), torch.tensor([words])]
    if kind == "sync":
        return [0, words, _in(_dst(n, torch.int16), u16)]
    if kind == "to16":
        return [_pair(0, words), _in(_dst(n, torch.int16), u16)]
    u8 = _utf8(text)
    if kind == "six":
        return [_pair(0, n), torch.tensor([words]), _pair(0, words), _in(_dst(n, torch.int16), u16),
                _pair(0, words), torch.tensor([n]), _pair(0, n), u8]
    u32 = torch.cat(text)
    return [_pair(0, n), u8, _pair(0, words), _in(_dst(n, torch.int16), _swap(u16)), _pair(0, n), u8,
            _pair(0, u32.numel()), _in(_dst(n, torch.int32), u32)]
