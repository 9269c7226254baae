"""The Zstandard kernel (csrc/k_zstd.cu) run on the CPU, a thread block at a time
(cuda_on_cpu.h), under AddressSanitizer and UBSan: pages of several blocks
against the CPU oracle, and damaged pages, which have to be rejected without an
access outside the page, without threads of the block parting at a barrier, and
without harm to the sound page that the same block decodes next.  No GPU needed."""
import os
import pickle
import subprocess
import sys

import pytest

import zstd_cases as C
from cuda_on_cpu import compile_kernels

_RUN = r'''
import ctypes, pickle, sys
import numpy as np
lib = ctypes.CDLL(sys.argv[1])
ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
res = []
for pages, sizes, seed in pickle.load(open(sys.argv[2], "rb")):
    at = np.cumsum([0] + [len(p) for p in pages]).astype(np.uint32)
    size = np.array(sizes, np.uint32)
    out, err = np.zeros(int(size.sum()) + 1, np.uint8), np.zeros(3, np.int32)
    text = ctypes.create_string_buffer(256)
    rc = lib.zstd_kernel_decode(b"".join(pages), ptr(at), ptr(size), len(pages), 1, seed, ptr(out), ptr(err), text)
    res.append((rc, text.value.decode(), int(err[0]), int(err[1]), int(err[2]), out[:-1].tobytes()))
pickle.dump(res, open(sys.argv[3], "wb"))
'''


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    """run([(pages, decoded sizes, seed of the warp order)]) -> [(return code,
    fault, error flags, first bad page, detail, output bytes)]"""
    tmp = tmp_path_factory.mktemp("zstd_kernel")
    libs = [subprocess.run(["g++", f"-print-file-name=lib{s}.so"], capture_output=True, text=True).stdout.strip()
            for s in ("asan", "ubsan")]
    if not all(os.path.isabs(p) and os.path.exists(p) for p in libs):
        pytest.skip("no sanitizer runtime")
    lib = compile_kernels(tmp, "zstd_kernel_harness.cpp", sanitize=True)

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


def test_frames_hold_every_kind_of_block():
    kinds = set().union(*(C.block_kinds(f) for f, _ in C.frames().values()))
    assert kinds >= {"raw", "rle", "lit0", "lit1", "lit2", "lit3", "four", "second frame", "skippable",
                     *(t + m for t in ("ll", "of", "ml") for m in "0123")}


def test_pages_of_several_blocks(run):
    cases = [(name, f, d) for name, (f, d) in C.frames().items() if len(d) == C.PAGE
             and (name.endswith("_0") or not name.startswith("text"))]
    got = run([([f], [len(d)], seed) for seed, (_, f, d) in enumerate(cases)])
    for (name, _, d), (rc, fault, flags, _, _, out) in zip(cases, got):
        assert (rc, fault, flags) == (0, "", 0), name
        assert out == d, name


def test_damaged_pages_are_rejected(run):
    bad = C.damaged(120)[::3]
    good, want = C.frames()["text_19_0"]
    # warp 0 first in every phase, which is where a late note of an error shows; the rest shuffled
    got = run([([f, good], [C.PAGE, C.PAGE], 0 if i % 3 else i) for i, (_, f) in enumerate(bad)])
    details = set()
    for (name, _), (rc, fault, flags, page, detail, out) in zip(bad, got):
        assert (rc, fault) == (0, ""), name
        assert flags != 0 and page == 0, name
        assert out[C.PAGE:] == want, name
        details.add(detail)
    assert len(details) >= 8, details  # kinds of error
