"""GPU decode where the launch follows the size of a page: thread blocks and
threads a page, and the work items that a batch of its runs covers.  Bit for bit
against the CPU oracle."""
import numpy as np
import pytest

import synth
from oracle import reader as R

from gpu_util import assert_columns_equal, engine, slice_result, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    e = engine()
    yield e
    e.close()


def _check(eng, columns, spec, ranges=()):
    from paper_2602_17335_gb300.tables import write_table
    data = write_table(synth.Table(columns), spec).tobytes()
    expect = R.read_file(data)
    dev = to_dev(data)
    assert_columns_equal(eng.read([dev]), expect)
    for lo, hi in ranges:
        assert_columns_equal(eng.read([dev], row_begin=lo, row_count=hi - lo), [slice_result(e, lo, hi) for e in expect])


@pytest.mark.parametrize("page", [64, 8 << 10, (8 << 10) + 64, 64 << 10, 248 << 10, 300_000, 1 << 20])
def test_byte_stream_split(eng, page):
    """Around a block's 8 KiB and the most blocks of a page, with a short last page."""
    rng = np.random.default_rng(page)
    rows = 90_001 if page > 64 else 5_003
    valid = rng.random(rows) > 0.2
    ints = rng.integers(-2**62, 2**62, rows)
    ints[~valid] = 0
    cols = [synth.ColumnData("d", "DOUBLE", rng.standard_normal(rows)),
            synth.ColumnData("i", "INT32", rng.integers(-2**31, 2**31, rows).astype(np.int32)),
            synth.ColumnData("o", "INT64", ints, valid)]
    _check(eng, cols, synth.TableSpec(70_000, page, [synth.ColumnSpec("BYTE_STREAM_SPLIT") for _ in cols]),
           [(1234, rows - 7)])


@pytest.mark.parametrize("kib", [2, 56, 64, 96, 256, 280, 600])
def test_regions_of_a_page(eng, kib):
    """DELTA pages and string dictionaries of a few regions (8 KiB, 4 KiB) up to
    more than the block that stitches them has warps."""
    rng = np.random.default_rng(kib)
    rows = 140 * kib + 77
    n = 60 * kib + 3
    lens = rng.integers(0, 24, n)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    strings = synth.StringData(off, rng.integers(33, 127, int(off[-1])).astype(np.uint8),
                               rng.integers(0, n, rows).astype(np.int32))
    cols = [synth.ColumnData("d", "INT64", rng.integers(-2**62, 2**62, rows)),
            synth.ColumnData("k", "INT32", np.cumsum(rng.integers(0, 8, rows)).astype(np.int32)),
            synth.ColumnData("s", "BYTE_ARRAY", strings)]
    spec = synth.TableSpec(rows, kib << 10, [synth.ColumnSpec(e) for e in ("DELTA_BINARY_PACKED", "DELTA_BINARY_PACKED",
                                                                         "RLE_DICTIONARY")])
    _check(eng, cols, spec, [(rows // 3, rows - 5)])


@pytest.mark.parametrize("nulls", ["random", "runs", "ends", "none"])
@pytest.mark.parametrize("mode", ["BATCHED", "PLAIN"])
def test_items_of_a_large_page(eng, nulls, mode):
    """One page of many items and many batches of runs: definition levels and
    dictionary indices, whole and from rows inside items on."""
    from paper_2602_17335_gb300 import native as N
    from paper_2602_17335_gb300.tables import write_table
    rng = np.random.default_rng(len(nulls))
    rows = 300_017
    valid = {"random": rng.random(rows) > 0.3, "none": np.ones(rows, bool),
             "runs": np.repeat(rng.random(rows // 700 + 1) > 0.5, 700)[:rows],
             "ends": (np.arange(rows) > 70_001) & (np.arange(rows) < 240_003)}[nulls]
    few, many = rng.integers(0, 5, rows), rng.integers(0, 3000, rows)
    runs = np.repeat(rng.integers(0, 9, rows // 50 + 1), 50)[:rows]
    cols = [synth.ColumnData(f"r{k}", "INT32", v.astype(np.int32)) for k, v in enumerate((few, many, runs))]
    for k, v in enumerate((few, many, runs)):
        v = v.copy()
        v[~valid] = 0
        cols.append(synth.ColumnData(f"o{k}", "INT64", v, valid))
    data = write_table(synth.Table(cols), synth.TableSpec(rows, 8 << 20, [synth.ColumnSpec("RLE_DICTIONARY") for _ in cols]))
    data = data.tobytes()
    expect, dev = R.read_file(data), to_dev(data)
    flags = getattr(N, "PQ_SCAN_" + mode)
    for lo, hi in ((0, rows), (1, rows), (127, 128), (70_000, 240_000), (299_001, rows)):
        outs = eng.read([dev], row_begin=lo, row_count=hi - lo, flags=flags)
        assert_columns_equal(outs, [slice_result(e, lo, hi) for e in expect])
