"""The transcode of DELTA_LENGTH_BYTE_ARRAY and DELTA_BYTE_ARRAY pages
(csrc/k_transcode.cu) run on the CPU, a thread block at a time (cuda_on_cpu.h),
under AddressSanitizer and UBSan: sound pages against the CPU oracle, damaged
ones rejected without an access outside the page and without threads of the
block parting at a barrier.  No GPU needed."""
import os
import pickle
import subprocess
import sys

import numpy as np
import pytest

from cuda_on_cpu import compile_kernels
from oracle import delta as D
from oracle import delta_strings as DS

LBA, BA = 6, 7

_RUN = r'''
import ctypes, pickle, sys
import numpy as np
lib = ctypes.CDLL(sys.argv[1])
ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
res = []
for pages, enc, rows, chars, seed in pickle.load(open(sys.argv[2], "rb")):
    at = np.cumsum([0] + [len(p) for p in pages]).astype(np.uint32)
    enc, rows, chars = np.array(enc, np.int32), np.array(rows, np.int32), np.array(chars, np.int64)
    values, lens = np.full(len(pages), -2, np.int32), np.zeros(int(rows.sum()) + 1, np.uint32)
    out, err = np.zeros(1 << 22, np.uint8), np.zeros(3, np.int32)
    text = ctypes.create_string_buffer(256)
    rc = lib.transcode_pages(b"".join(pages), ptr(at), ptr(enc), ptr(rows), ptr(chars), len(pages), seed, ptr(values),
                             ptr(lens), ptr(out), ptr(err), text)
    res.append((rc, text.value.decode(), err.tolist(), values.tolist(), lens.tolist(), out[:int(lens.sum())].tobytes()))
pickle.dump(res, open(sys.argv[3], "wb"))
'''


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    tmp = tmp_path_factory.mktemp("transcode_kernel")
    libs = [subprocess.run(["g++", f"-print-file-name=lib{s}.so"], capture_output=True, text=True).stdout.strip()
            for s in ("asan", "ubsan")]
    if not all(os.path.isabs(p) and os.path.exists(p) for p in libs):
        pytest.skip("no sanitizer runtime")
    lib = compile_kernels(tmp, "transcode_kernel_harness.cpp", sanitize=True)

    def go(cases):
        src, dst = str(tmp / "cases.pkl"), str(tmp / "results.pkl")
        with open(src, "wb") as f:
            pickle.dump(cases, f)
        env = dict(os.environ, LD_PRELOAD=":".join(libs), ASAN_OPTIONS="detect_leaks=0",
                   UBSAN_OPTIONS="halt_on_error=1:print_stacktrace=1")
        r = subprocess.run([sys.executable, "-c", _RUN, lib, src, dst], capture_output=True, text=True, env=env,
                           timeout=900)
        assert r.returncode == 0, r.stderr[-3000:]
        assert "AddressSanitizer" not in r.stderr and "runtime error" not in r.stderr, r.stderr[-3000:]
        with open(dst, "rb") as f:
            return pickle.load(f)
    return go


def _items(rng, n, kind):
    if kind == "empty":
        return [b""] * n
    if kind == "sorted":
        return sorted(b"%06d" % int(v) * int(rng.integers(1, 3)) for v in rng.integers(0, 2000, n))
    if kind == "long":
        return [bytes(rng.integers(97, 99, int(k), dtype=np.uint8)) for k in rng.integers(0, 6000, n)]
    return [bytes(rng.integers(97, 101, int(k), dtype=np.uint8)) for k in rng.integers(0, 12, n)]


def _encode(items, enc):
    return DS.encode_length_byte_array(items) if enc == LBA else DS.encode_byte_array(items)


def test_sound_pages(run):
    rng = np.random.default_rng(1)
    shapes = [(1, "short"), (2, "short"), (130, "short"), (700, "short"), (513, "sorted"), (2300, "sorted"), (60, "long"),
              (300, "empty")]
    pages = [(enc, _items(rng, n, kind)) for n, kind in shapes for enc in (LBA, BA)]
    got = run([([_encode(it, enc)], [enc], [len(it)], [sum(map(len, it))], seed)
               for seed, (enc, it) in enumerate(pages)])
    for (enc, it), (rc, fault, err, values, lens, out) in zip(pages, got):
        assert (rc, fault, err[0], values) == (0, "", 0, [len(it)])
        assert lens[:len(it)] == [len(x) for x in it] and out == b"".join(it)


def test_damaged_pages_are_rejected(run):
    rng = np.random.default_rng(2)
    items = _items(rng, 200, "sorted")
    n = len(items)
    lens = [len(x) for x in items]
    bad = [(LBA, D.encode([-1] + lens[1:], 32) + b"".join(items)),           # a negative length first
           (LBA, _encode(items, LBA)[:-1]),                                 # values longer than the page
           (LBA, _encode(items[:-1], LBA)), (BA, _encode(items[:-1], BA)),  # too few values
           (LBA, b""), (BA, b""), (LBA, b"\x80\x01\x04"),
           (BA, D.encode([0] * n, 32)),                                     # no suffixes
           (BA, D.encode([0] * n, 32) + b"\x80\x01\x04\xc8\x01"),           # a cut header of the second stream
           (BA, D.encode([0], 32)[:5] + b"\xff"),
           (BA, D.encode([-1] + [0] * (n - 1), 32) + DS.encode_length_byte_array(items)),
           (BA, D.encode([1] + [0] * (n - 1), 32) + DS.encode_length_byte_array(items)),
           (BA, D.encode([0] * n, 32) + D.encode([-5] + lens[1:], 32) + b"".join(items)),
           (BA, D.encode([0, 1000] + [0] * (n - 2), 32) + DS.encode_length_byte_array(items))]
    while len(bad) < 60:
        enc = (LBA, BA)[int(rng.integers(2))]
        f = bytearray(_encode(items, enc))
        for _ in range(int(rng.integers(1, 4))):
            f[int((len(f) - 1) * rng.random() ** 3)] = int(rng.integers(256))
        bad.append((enc, bytes(f)))
    good = _items(rng, 150, "short")
    rows = [1 if len(f) < 8 else n for _, f in bad]
    # warp 0 first in every phase, which is where a late note of an error shows, or shuffled;
    # (room in the pool for whatever a changed length adds up to)
    got = run([([f, _encode(good, BA)], [enc, BA], [r, len(good)], [1 << 20, 1 << 20], i if i % 3 == 2 else 0)
               for i, ((enc, f), r) in enumerate(zip(bad, rows))])
    rejected = 0
    for (enc, f), r, (rc, fault, err, values, _, out) in zip(bad, rows, got):
        assert (rc, fault) == (0, "")
        try:
            want = b"".join((DS.decode_length_byte_array if enc == LBA else DS.decode_byte_array)(f, 0, len(f), r)[0])
        except (ValueError, IndexError):
            want = None
        assert values[1] == len(good) and out.endswith(b"".join(good))
        if values[0] < 0:
            assert err[0] and err[1] == 0
            rejected += 1
        else:  # the change left a page of other values
            assert err[0] == 0 and want is not None and out == want + b"".join(good)
    assert rejected >= 40
