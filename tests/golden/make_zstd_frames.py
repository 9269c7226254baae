"""Writes zstd_frames.json: Zstandard frames made by libzstd (through ctypes: run
it where the library is installed), of several blocks each, so that they hold
what one-block pages do not: treeless literals, RLE literals, repeated, RLE and
transmitted sequence tables, raw and RLE blocks, checksums, several frames and a
skippable one, blocks of 128 KiB.

Inputs only: expected values come from the CPU oracle.

    python tests/golden/make_zstd_frames.py
"""
import ctypes
import ctypes.util
import json
import os

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
PAGE = 2048    # bytes of every small page
LEVEL, WINDOW_LOG, CHECKSUM = 100, 101, 201  # ZSTD_cParameter
FLUSH, END = 1, 2                            # ZSTD_EndDirective


class _Buffer(ctypes.Structure):
    _fields_ = [("p", ctypes.c_void_p), ("size", ctypes.c_size_t), ("pos", ctypes.c_size_t)]


def _lib():
    z = ctypes.CDLL(ctypes.util.find_library("zstd"))
    z.ZSTD_createCCtx.restype = ctypes.c_void_p
    z.ZSTD_CCtx_setParameter.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int]
    z.ZSTD_CCtx_setParameter.restype = ctypes.c_size_t
    z.ZSTD_compressStream2.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    z.ZSTD_compressStream2.restype = ctypes.c_size_t
    z.ZSTD_isError.argtypes = [ctypes.c_size_t]
    z.ZSTD_freeCCtx.argtypes = [ctypes.c_void_p]
    return z


def compress(x, cuts=(), level=3, checksum=False):
    """x as one frame, with a block boundary at each of cuts."""
    z = _lib()
    c = z.ZSTD_createCCtx()
    for k, v in ((LEVEL, level), (CHECKSUM, int(checksum))):
        assert not z.ZSTD_isError(z.ZSTD_CCtx_setParameter(c, k, v))
    room = ctypes.create_string_buffer(2 * len(x) + 4096)
    out = _Buffer(ctypes.cast(room, ctypes.c_void_p), len(room), 0)
    at = 0
    for end in [*cuts, len(x)]:
        part = ctypes.create_string_buffer(bytes(x[at:end]), end - at + 1)
        src = _Buffer(ctypes.cast(part, ctypes.c_void_p), end - at, 0)
        left = 1
        while left or src.pos < src.size:
            left = z.ZSTD_compressStream2(c, ctypes.byref(out), ctypes.byref(src), END if end == len(x) else FLUSH)
            assert not z.ZSTD_isError(left)
        at = end
    z.ZSTD_freeCCtx(c)
    return room.raw[:out.pos]


def _text(rng, n, words, alphabet, sep):
    """n bytes of random words, some of them fresh, with separators between."""
    pool = [bytes(rng.integers(97, 97 + alphabet, int(rng.integers(3, 25)), dtype=np.uint8)) for _ in range(words)]
    out = bytearray()
    while len(out) < n:
        out += sep if rng.random() < 0.5 else b""
        out += pool[int(rng.integers(words))] if rng.random() < 0.7 else \
            bytes(rng.integers(97, 97 + alphabet, int(rng.integers(1, 12)), dtype=np.uint8))
    return bytes(out[:n])


def frames():
    rng = np.random.default_rng(20)
    out = {}
    for level in (1, 3, 9, 19, 22):
        for k in range(4):
            x = _text(rng, PAGE, int(rng.integers(2, 40)), int(rng.integers(3, 26)), b" ")
            cuts = sorted({int(c) for c in rng.integers(1, PAGE, 4 + 2 * k)})
            out[f"text_{level}_{k}"] = compress(x, cuts, level, checksum=k == 1)
    # literals of one value: a known word after each of its occurrences
    words = [bytes(rng.integers(97, 123, 16, dtype=np.uint8)) for _ in range(60)]
    x = b"".join(words) + b"".join(b"Z" + words[i] for i in rng.permutation(60))
    out["rle_literals"] = compress(x + b"Z" * (PAGE - len(x)), (960,), 22)
    # sequences that all have the same codes
    unit = bytes(rng.integers(0, 256, 24, dtype=np.uint8))
    x = unit + b"".join(bytes([int(v)]) + unit[:15] for v in rng.integers(0, 256, 200))
    out["rle_tables"] = compress(x[:PAGE], (24, 1000), 19)
    out["raw_and_rle_blocks"] = compress(bytes(rng.integers(0, 256, 700, dtype=np.uint8)) + b"q" * 900 +
                                         bytes(rng.integers(0, 256, 448, dtype=np.uint8)), (700, 1600), 3)
    a, b = _text(rng, 1000, 9, 12, b","), _text(rng, PAGE - 1000, 9, 12, b";")
    skip = (0x184D2A53).to_bytes(4, "little") + (5).to_bytes(4, "little") + b"skip!"
    out["two_frames"] = compress(a, (400,), 19) + skip + compress(b, (600,), 19, True)
    out["skippable_first"] = skip + compress(_text(rng, PAGE, 20, 20, b"-"), (), 3) + skip
    # blocks of the format's largest size
    words = _text(rng, 3000, 20, 20, b" ")
    x = b"".join(words[int(p):int(p) + int(n)] + bytes([int(c)]) for p, n, c in zip(
        rng.integers(0, 2900, 9000), rng.integers(20, 100, 9000), rng.integers(97, 117, 9000)))
    x = x[:344_064]
    out["three_blocks"] = compress(x, (), 3)
    out["three_blocks_19"] = compress(x, (), 19)
    return out


if __name__ == "__main__":
    path = os.path.join(HERE, "zstd_frames.json")
    with open(path, "w") as f:
        json.dump({name: frame.hex() for name, frame in frames().items()}, f, indent=0)
        f.write("\n")
    print(path, os.path.getsize(path))
