"""Columns of more pages, or dictionaries, than the y dimension of one launch
grid holds (65,535), bit for bit.  Kernels that take one page per grid row are
launched in slices there."""
import numpy as np
import pytest

import synth
from oracle import reader as R
from oracle.reader import ColumnResult

from gpu_util import assert_columns_equal, engine, to_dev

pytestmark = pytest.mark.gpu

PAGES = 65_535 + 5


@pytest.fixture(scope="module")
def eng():
    e = engine()
    yield e
    e.close()


def _read(eng, columns, spec):
    from paper_2602_17335_gb300 import native as N
    from paper_2602_17335_gb300.tables import write_table
    data = write_table(synth.Table(columns), spec).tobytes()
    dev = to_dev(data)
    idx = eng.index([dev])
    pages = N.pq_index_get_info(idx).n_data_pages
    N.pq_free_index(idx)
    assert pages == PAGES * len(columns)
    return data, eng.read([dev])


def test_byte_stream_split_pages(eng):
    v = np.random.default_rng(1).standard_normal(8 * PAGES)
    spec = synth.TableSpec(len(v), 64, [synth.ColumnSpec("BYTE_STREAM_SPLIT")])
    data, outs = _read(eng, [synth.ColumnData("x", "DOUBLE", v)], spec)
    assert_columns_equal(outs, R.read_file(data))


def test_delta_pages(eng):
    """Pages of one DELTA block each (compared with the column the file was
    written from: the oracle takes a minute to read them)."""
    v = np.random.default_rng(2).integers(-2**62, 2**62, 129 * PAGES)
    spec = synth.TableSpec(len(v), 64, [synth.ColumnSpec("DELTA_BINARY_PACKED")])
    _, outs = _read(eng, [synth.ColumnData("x", "INT64", v)], spec)
    assert_columns_equal(outs, [ColumnResult("x", "INT64", v, None)])


def test_dictionary_pages(eng):
    """A row group a row: as many dictionaries, of integers and of strings."""
    rng = np.random.default_rng(3)
    v = rng.integers(0, 1000, PAGES).astype(np.int32)
    lens = rng.integers(0, 30, 50)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    strings = synth.StringData(off, rng.integers(33, 127, int(off[-1])).astype(np.uint8),
                               rng.integers(0, 50, PAGES).astype(np.int32))
    o, chars = strings.materialize()
    spec = synth.TableSpec(1, 1 << 20, [synth.ColumnSpec("RLE_DICTIONARY") for _ in range(2)])
    _, outs = _read(eng, [synth.ColumnData("x", "INT32", v), synth.ColumnData("s", "BYTE_ARRAY", strings)], spec)
    assert_columns_equal(outs, [ColumnResult("x", "INT32", v, None),
                                ColumnResult("s", "BYTE_ARRAY", None, None, np.asarray(o), np.asarray(chars))])
