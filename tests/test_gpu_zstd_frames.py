"""Zstandard pages of several blocks on the GPU, bit for bit against the CPU
oracle: what libzstd writes into pages of more than 128 KiB (treeless literals,
repeated tables), RLE literals, several frames in a page; and damaged pages, an
error each, between sound ones that the same thread blocks go on to decode."""
import numpy as np
import pytest

import synth
from oracle import reader as R
from oracle import writer as W

import zstd_cases as C
from gpu_util import assert_columns_equal, engine, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    e = engine()
    yield e
    e.close()


def _file(monkeypatch, pages, n, damage=()):
    """A REQUIRED INT64 PLAIN column of pages of n decoded bytes, page i stored as
    pages[i][0] (or what `damage` has for i)."""
    stored = iter([damage[i] if i in damage else p[0] for i, p in enumerate(pages)])
    with monkeypatch.context() as m:
        m.setattr(W._zstd, "compress_stored", lambda b: next(stored))
        vals = np.frombuffer(b"".join(p[1] for p in pages), dtype=np.int64)
        spec = synth.TableSpec(n // 8, 1 << 24, [synth.ColumnSpec("PLAIN", "ZSTD")])
        spec.columns[0].compress_threshold = -1.0
        return W.write_file(synth.Table([synth.ColumnData("x", "INT64", vals)]), spec), vals


@pytest.mark.parametrize("n", sorted({len(d) for _, d in C.frames().values()}))
def test_pages_of_several_blocks(eng, monkeypatch, n):
    pages = [p for p in C.frames().values() if len(p[1]) == n]
    data, vals = _file(monkeypatch, pages, n)
    expect = R.read_file(data)
    assert np.array_equal(expect[0].values, vals)
    assert_columns_equal(eng.read([to_dev(data)]), expect)


def test_damaged_pages_between_sound_ones(eng, monkeypatch):
    """More pages than thread blocks run at a time, every fourth one damaged: the
    scan reports a corrupt page, and the sound pages' rows are right all the same."""
    from paper_2602_17335_gb300 import native as N
    from paper_2602_17335_gb300.scan import alloc_outputs
    good = [p for p in C.frames().values() if len(p[1]) == C.PAGE]
    bad = [f for _, f in C.damaged(400)]
    pages = [good[i % len(good)] for i in range(4 * len(bad))]
    damage = {4 * i + 1: f for i, f in enumerate(bad)}
    data, vals = _file(monkeypatch, pages, C.PAGE, damage)
    idx = eng.index([to_dev(data)])
    plan, sizes = eng.plan(idx, None, 0, -1, N.PQ_SCAN_BATCHED)
    for _ in range(2):
        outs = alloc_outputs(sizes)
        eng.scan(plan, outs)
        st, _ = eng.wait(plan, len(outs))
        assert st == N.PQ_ERR_CORRUPT
        got = outs[0].values.cpu().numpy().view(np.int64).reshape(len(pages), -1)
        want = vals.reshape(len(pages), -1)
        sound = [i for i in range(len(pages)) if i not in damage]
        assert np.array_equal(got[sound], want[sound])
    N.pq_free_plan(plan)
    N.pq_free_index(idx)


def test_each_damaged_page_is_an_error(eng, monkeypatch):
    from paper_2602_17335_gb300 import native as N
    good = C.frames()["text_19_0"]
    for name, f in C.damaged(60):
        data, _ = _file(monkeypatch, [good, good, good], C.PAGE, {1: f})
        with pytest.raises(N.PqError) as ei:
            eng.read([to_dev(data)])
        assert ei.value.status == N.PQ_ERR_CORRUPT, name
