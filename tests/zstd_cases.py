"""Zstandard pages of several blocks (golden/zstd_frames.json, made by libzstd)
and damaged copies of them that the CPU oracle rejects."""
import json
import os

import numpy as np

from oracle import zstd as Z

HERE = os.path.dirname(os.path.abspath(__file__))
PAGE = 2048


def frames():
    """{name: (frame bytes, decoded bytes)}"""
    with open(os.path.join(HERE, "golden", "zstd_frames.json")) as f:
        raw = {name: bytes.fromhex(h) for name, h in json.load(f).items()}
    return {name: (b, Z.decompress(b)) for name, b in raw.items()}


def block_kinds(frame):
    """What the blocks of a frame are made of: 'raw', 'rle', literals 0-3 as
    'lit0'.., streams 'four', and each sequence table's mode as 'll0'.. 'of0'.. 'ml0'.."""
    kinds, p = set(), 0
    while p < len(frame):
        if frame[p + 1:p + 4] == b"\x2a\x4d\x18":
            kinds.add("skippable")
            p += 8 + int.from_bytes(frame[p + 4:p + 8], "little")
            continue
        if p:
            kinds.add("second frame")
        fhd = frame[p + 4]
        single, fcs = (fhd >> 5) & 1, fhd >> 6
        p += 5 + (1 - single) + (0, 1, 2, 4)[fhd & 3] + (single if fcs == 0 else (0, 2, 4, 8)[fcs])
        last = 0
        while not last:
            h = int.from_bytes(frame[p:p + 3], "little")
            last, kind, size = h & 1, (h >> 1) & 3, h >> 3
            p += 3
            if kind < 2:
                kinds.add(("raw", "rle")[kind])
                p += size if kind == 0 else 1
                continue
            b = frame[p:p + size]
            p += size
            lit, sf = b[0] & 3, (b[0] >> 2) & 3
            kinds.add(f"lit{lit}")
            if lit < 2:
                n = (1, 2, 1, 3)[sf]
                used = n + ((int.from_bytes(b[:n], "little") >> (3 if n == 1 else 4)) if lit == 0 else 1)
            else:
                n, bits = (3, 3, 4, 5)[sf], (10, 10, 14, 18)[sf]
                used = n + ((int.from_bytes(b[:n], "little") >> (4 + bits)) & ((1 << bits) - 1))
                kinds |= {"four"} if sf else set()
            s = b[used:]
            if s[0]:
                m = s[1 if s[0] < 128 else 2 if s[0] < 255 else 3]
                kinds |= {f"ll{m >> 6}", f"of{(m >> 4) & 3}", f"ml{(m >> 2) & 3}"}
        p += 4 * ((fhd >> 2) & 1)
    return kinds


def _grown_block(frame):
    """The frame with a byte added to the end of its first compressed block (after
    the literals of a block without sequences, or before the last byte of its bits)."""
    fhd = frame[4]
    single, fcs = (fhd >> 5) & 1, fhd >> 6
    p = 5 + (1 - single) + (single if fcs == 0 else (0, 2, 4, 8)[fcs])
    while frame[:4] == b"\x28\xb5\x2f\xfd":
        h = int.from_bytes(frame[p:p + 3], "little")
        kind, size = (h >> 1) & 3, h >> 3
        if kind == 2:
            return frame[:p] + (h + 8).to_bytes(3, "little") + frame[p + 3:p + 3 + size] + b"\x01" + frame[p + 3 + size:]
        if h & 1:
            return None
        p += 3 + (1 if kind == 1 else size)
    return None


def damaged(count, seed=1):
    """`count` damaged 2 KiB pages that the oracle rejects, as (name, frame): each
    frame cut short and with a block grown by a byte, then with bytes changed."""
    good = {n: f for n, (f, d) in frames().items() if len(d) == PAGE}
    rng = np.random.default_rng(seed)
    out = []

    def add(name, frame):
        if frame is None:
            return
        try:
            if len(Z.decompress(frame)) == PAGE:
                return
        except (ValueError, IndexError):
            pass
        out.append((name, frame))
    for name, f in good.items():
        add(name + " grown", _grown_block(f))
        add(name + " cut", f[:int(rng.integers(4, len(f)))])
    names = sorted(good)
    while len(out) < count:
        name = names[int(rng.integers(len(names)))]
        f = bytearray(good[name])
        for _ in range(int(rng.integers(1, 4))):
            f[4 + int((len(f) - 4) * rng.random() ** 3)] = int(rng.integers(256))  # (headers and tables above all)
        add(name + " changed", bytes(f))
    return out[:count]
