"""Planning and scan enqueueing (csrc/engine.cpp) compiled for the CPU with g++
over a CUDA runtime of the test's own: device memory is host memory and a kernel
is an entry in a log.  A launch that the runtime refuses has to come back as an
error from the scan, whichever it is.  No GPU needed."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import synth
from oracle import writer as W
from paper_2602_17335_gb300 import native as N

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(ROOT, "paper_2602_17335_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def scan(tmp_path_factory):
    """scan(file, flags, n_sms, fail_at) -> (status, {what: text})."""
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("no g++ or CUDA headers")
    out = str(tmp_path_factory.mktemp("scan_host") / "scan_host.so")
    # (-Bsymbolic: the runtime of this library, whatever else the process has loaded)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), "-I", CUDA_INC, os.path.join(HERE, "scan_host_harness.cpp"),
                    *(os.path.join(CSRC, f) for f in ("engine.cpp", "host_meta.cpp", "host_pages.cpp")), "-o", out],
                   check=True)
    lib = ctypes.CDLL(out)
    lib.scan_with_fake_cuda.argtypes = [ctypes.c_char_p, ctypes.c_uint64, ctypes.c_uint32, ctypes.c_int, ctypes.c_int,
                                        ctypes.c_int, ctypes.c_char_p, ctypes.c_uint64]

    def run(data, flags=0, n_sms=152, fail_at=-1, stale_error=0):
        text = ctypes.create_string_buffer(1 << 16)
        st = lib.scan_with_fake_cuda(data, len(data), flags, n_sms, fail_at, stale_error, text, len(text))
        return st, {k: v for k, _, v in (line.partition(" ") for line in text.value.decode().splitlines())}
    return run


def _eight(codec):
    spec = synth.config2_spec(2500, 4096, codec, 1)
    for c in spec.columns:
        c.compress_threshold = -1.0
    return W.write_file(synth.config2_table(6000, 2500, string_pool_size=200, zipf_k=300), spec)


def _split():
    """Snappy pages long enough to be decompressed by fragments."""
    from paper_2602_17335_gb300.tables import write_table
    from test_native_writer import _native
    _native()
    rng = np.random.default_rng(1)
    cols = [synth.ColumnData(f"x{k}", "INT64", rng.integers(0, 50_000, 60_000)) for k in range(3)]
    spec = synth.TableSpec(60_000, 1 << 20, [synth.ColumnSpec(e, "SNAPPY") for e in ("PLAIN", "RLE_DICTIONARY", "PLAIN")])
    for c in spec.columns:
        c.compress_threshold = -1.0
    return write_table(synth.Table(cols), spec).tobytes()


def _v2():
    return W.write_file(synth.v2_encodings_table(4000, 2000), synth.v2_encodings_spec(2000, 1500))


@pytest.mark.parametrize("flags", ["BATCHED", "PLAIN", "GRAPH", "TIMING"])
@pytest.mark.parametrize("n_sms", [1, 152])  # one: launched column by column, many: all columns together
@pytest.mark.parametrize("table", ["none", "snappy", "zstd", "split", "v2"])
def test_refused_launches_are_errors(scan, flags, n_sms, table):
    """Each launch of a scan refused in turn: the scan reports it, launches
    nothing after it, leaves no stream unjoined, records the plan's end (which
    freeing the plan waits for) and no error stays behind."""
    data = {"none": lambda: _eight("UNCOMPRESSED"), "snappy": lambda: _eight("SNAPPY"), "zstd": lambda: _eight("ZSTD"),
            "split": _split, "v2": _v2}[table]()
    fl = getattr(N, "PQ_SCAN_" + flags)
    st, good = scan(data, fl, n_sms)
    assert st == N.PQ_OK and good["done"] == "1" and good["last_error"] == "0"
    kernels = [k for k in good["launches"].split() if k != "graph"]
    assert "prepare" == kernels[0] and "copy_small" == kernels[-1]
    # (the count of kernels that a plan tells is the one that a scan launches)
    assert int(good["planned_kernels"]) == int(good["kernels"]) >= len(kernels)
    if table == "split" and flags != "PLAIN":
        assert "snappy_fragments" in kernels
    for k in range(len(kernels)):
        st, got = scan(data, fl, n_sms, k)
        assert st == N.PQ_ERR_CUDA, (k, kernels[k])
        assert got["launches"].split() == kernels[:k + 1], kernels[k]
        assert got["joins"] == good["joins"] and got["forks"] == good["forks"]
        assert got["last_error"] == "0"
        assert got["done"] == ("0" if flags == "GRAPH" else "1")  # (a graph that was not made has not run)


def test_plan_budget_covers_its_memory(scan):
    """What serving admits a request by is no less than what its plan takes (up to
    the allocator's rounding, less than 64 KiB an allocation): twelve columns of
    so few rows that they are cut into small work items."""
    from paper_2602_17335_gb300.tables import write_table
    from test_native_writer import _native
    _native()
    rows = 1_200_000
    v = np.random.default_rng(1).integers(0, 1000, rows).astype(np.int32)
    data = write_table(synth.Table([synth.ColumnData(f"x{k}", "INT32", v) for k in range(12)]),
                       synth.TableSpec(rows, 1 << 20, [synth.ColumnSpec("RLE_DICTIONARY") for _ in range(12)])).tobytes()
    st, got = scan(data)
    assert st == N.PQ_OK
    assert int(got["budget"]) >= int(got["plan_bytes"]) - 65536 * int(got["plan_mallocs"])


@pytest.mark.parametrize("flags", ["BATCHED", "GRAPH"])
@pytest.mark.parametrize("n_sms", [1, 152])
def test_unscanned_plan_after_a_graph(scan, flags, n_sms):
    """A plan that is freed without a scan waits for none of the events it was
    given, which an earlier plan may have recorded inside its graph."""
    st, got = scan(_eight("UNCOMPRESSED"), getattr(N, "PQ_SCAN_" + flags), n_sms)
    assert st == N.PQ_OK and got["last_error_unscanned"] == "0"


@pytest.mark.parametrize("flags", ["BATCHED", "GRAPH"])
def test_an_earlier_error_is_not_the_scans(scan, flags):
    st, got = scan(_eight("UNCOMPRESSED"), getattr(N, "PQ_SCAN_" + flags), stale_error=1)
    assert st == N.PQ_OK and got["kernels"] == got["planned_kernels"]


def test_a_reported_error_is_not_reported_again(scan):
    st, got = scan(_eight("UNCOMPRESSED"), fail_at=-2)
    assert st == N.PQ_ERR_CUDA and got["last_error"] == "0" and got["launches"] == ""


@pytest.mark.parametrize("flags,rows,rows_per_item", [
    ("BATCHED", 6000, 256), ("BATCHED", 40_000, 256),
    ("PLAIN", 6000, 256), ("PLAIN", 16 * 512 + 40, 512), ("PLAIN", 40_000, 2048)])
def test_items_of_few_rows(scan, flags, rows, rows_per_item):
    """Few rows are cut into small work items, so that there are some for every
    warp: of the GPU, or of a page's thread block where that takes a whole page."""
    col = synth.ColumnData("x", "INT32", np.arange(rows, dtype=np.int32) % 7)
    data = W.write_file(synth.Table([col]), synth.TableSpec(rows, 1 << 20, [synth.ColumnSpec("RLE_DICTIONARY")]))
    st, got = scan(data, getattr(N, "PQ_SCAN_" + flags))
    assert st == N.PQ_OK and int(got["items"]) == -(-rows // rows_per_item)


def test_wait_for_a_captured_scan_is_refused(scan):
    data = _eight("UNCOMPRESSED")
    st, got = scan(data, fail_at=-3)
    assert st == N.PQ_OK and int(got["wait"]) == N.PQ_ERR_CUDA and got["last_error_unscanned"] == "0"
    st, got = scan(data)
    assert st == N.PQ_OK and int(got["wait"]) == N.PQ_OK
