"""GPU decode at the edges of the kernels' tiles, vs the CPU oracle, bit for
bit: windows, fragments and segments of Snappy pages with every element form
(and corrupt ones), Zstandard block counts and kinds, DELTA widths around the
32-bit paths, string lengths around the register copies, transcoded pages of
few values, and scans whose stages are launched for all columns together."""
import numpy as np
import pytest

import synth
from oracle import reader as R
from oracle import writer as W

from gpu_util import assert_columns_equal, engine, slice_result, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    e = engine()
    yield e
    e.close()


def _check(eng, data, columns=None, rb=0, rc=-1, **kw):
    expect = R.read_file(data)
    e0 = expect[0]
    rows = len(e0.values) if e0.values is not None else len(e0.offsets) - 1
    outs = eng.read([to_dev(data)], columns=columns, row_begin=rb, row_count=rc, **kw)
    hi = rows if rc < 0 else rb + rc
    assert_columns_equal(outs, [slice_result(expect[c], rb, hi) for c in (columns or range(len(expect)))])


# ------------------------------------------------------------------ Snappy elements

KINDS = {  # literal lengths, copy lengths, copy offsets, share of literals
    "short": ((1, 3), (1, 11), (1, 40), 0.4),
    "overlap": ((1, 9), (1, 64), (1, 7), 0.3),
    "mixed": ((1, 300), (1, 64), (1, 70_000), 0.5),
    "long": ((3_000, 66_000), (1, 64), (1, 3_000), 0.6),
}


def _uleb(v):
    out = bytearray()
    while v >= 128:
        out.append(v & 127 | 128)
        v >>= 7
    out.append(v)
    return bytes(out)


def _stream(n, kind, framed, rng):
    """(n output bytes, a Snappy stream of them): elements of one kind in every
    header form that can hold them; framed: none reaches across 64 KiB."""
    lits, lens, offs, p = KINDS[kind]
    out, s = bytearray(), bytearray(_uleb(n))
    while len(out) < n:
        at = len(out) % 65536 if framed else len(out)
        room = min(n - len(out), 65536 - at if framed else n)
        if at == 0 or rng.random() < p:
            ln = min(int(rng.integers(lits[0], lits[1] + 1)), room)
            need = 0 if ln <= 60 else ((ln - 1).bit_length() + 7) // 8
            nb = int(rng.integers(max(need, 0 if ln <= 60 else 1), 5)) if rng.random() < 0.2 or need else 0
            s += bytes([(ln - 1) << 2]) if nb == 0 else bytes([(59 + nb) << 2]) + (ln - 1).to_bytes(nb, "little")
            b = rng.integers(0, 256, ln, dtype=np.uint8).tobytes()
            s += b
            out += b
        else:
            off = min(int(rng.integers(offs[0], offs[1] + 1)), at)
            ln = min(int(rng.integers(lens[0], lens[1] + 1)), room)
            form = int(rng.integers(0, 3))
            if form == 0 and 4 <= ln <= 11 and off < 2048:
                s += bytes([1 | (ln - 4) << 2 | (off >> 8) << 5, off & 255])
            elif form <= 1 and off < 65536:
                s += bytes([2 | (ln - 1) << 2]) + off.to_bytes(2, "little")
            else:
                s += bytes([3 | (ln - 1) << 2]) + off.to_bytes(4, "little")
            out += (bytes(out[-off:]) * (ln // off + 1))[:ln]
    return bytes(out), bytes(s)


def _snappy_file(monkeypatch, n, pages, kind, framed, spoil=None):
    """A REQUIRED INT64 PLAIN column of `pages` pages of n bytes, each with a
    stream of its own."""
    rng = np.random.default_rng([n, pages, sorted(KINDS).index(kind), framed])
    made = [_stream(n, kind, framed, rng) for _ in range(pages)]
    table = dict(made)
    monkeypatch.setattr(W._snappy, "compress", lambda b: spoil(table[bytes(b)]) if spoil else table[bytes(b)])
    vals = np.frombuffer(b"".join(b for b, _ in made), dtype=np.int64)
    spec = synth.TableSpec(n // 8, 1 << 24, [synth.ColumnSpec("PLAIN", "SNAPPY")])
    spec.columns[0].compress_threshold = -1.0
    return W.write_file(synth.Table([synth.ColumnData("x", "INT64", vals)]), spec)


@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("n,pages,framed", [
    (8, 3, True), (2040, 400, True),                      # more pages than thread blocks of the wide shape
    (8184, 3, True), (8200, 3, False), (131072, 2, False),  # around a window; the largest page left whole
    (131080, 3, True), (131080, 2, False),                # the smallest split page, and one not framed
    (196608, 2, True), (393224, 2, True), (393216, 1, False)])
def test_snappy_elements(eng, monkeypatch, kind, n, pages, framed):
    _check(eng, _snappy_file(monkeypatch, n, pages, kind, framed))


@pytest.mark.parametrize("kind", ["short", "long"])
@pytest.mark.parametrize("n", [40_000, 393_224])
@pytest.mark.parametrize("spoil", ["cut", "offset", "length", "literal"])
def test_snappy_corrupt(eng, monkeypatch, kind, n, spoil):
    """A stream cut short, a copy from before the output, a length that is not
    the page's, a last literal longer than the input: an error, on pages
    decompressed whole and by fragments, with many elements and few."""
    from paper_2602_17335_gb300 import native as N
    change = {"cut": lambda s: s[:-1], "offset": lambda s: s[:len(_uleb(n))] + b"\x06\x01\x00" + s[len(_uleb(n)):],
              "length": lambda s: _uleb(n + 8) + s[len(_uleb(n)):], "literal": lambda s: s + b"\xf0\x09a"}[spoil]
    data = _snappy_file(monkeypatch, n, 2, kind, True, change)
    with pytest.raises(ValueError):
        R.read_file(data)
    with pytest.raises(N.PqError) as ei:
        eng.read([to_dev(data)])
    assert ei.value.status == N.PQ_ERR_CORRUPT


# ------------------------------------------------------------------ Zstandard blocks

@pytest.mark.parametrize("content", ["constant", "random", "words", "ramp"])
@pytest.mark.parametrize("rows", [1, 13, 16_383, 16_385, 40_000])  # 128 KiB is a block's most
def test_zstd_blocks(eng, content, rows):
    from paper_2602_17335_gb300.tables import write_table
    rng = np.random.default_rng(rows)
    vals = {"constant": np.full(rows, 0x0101010101010101, np.int64),
            "random": rng.integers(-2**63, 2**63 - 1, rows, dtype=np.int64),
            "words": rng.integers(0, 50, rows) ** 7,
            "ramp": np.arange(rows, dtype=np.int64) // 3}[content].astype(np.int64)
    spec = synth.TableSpec(rows, 1 << 24, [synth.ColumnSpec("PLAIN", "ZSTD")])
    spec.columns[0].compress_threshold = -1.0
    _check(eng, write_table(synth.Table([synth.ColumnData("x", "INT64", vals)]), spec).tobytes())


# ------------------------------------------------------------------ DELTA widths

@pytest.mark.parametrize("rows,page", [(1, 1 << 20), (2, 1 << 20), (129, 1 << 20), (130, 64), (4097, 1 << 20),
                                       (33_003, 8192)])
def test_delta_widths(eng, rows, page):
    """Steps of every width class (nothing stored, up to 24 bits, above, 32 bits
    and wider), REQUIRED and with nulls, both integer types; also from an odd row on."""
    rng = np.random.default_rng(rows)
    cols = []
    for w in (0, 1, 7, 16, 17, 24, 25, 31, 32, 33, 48, 64):
        steps = rng.integers(0, 2, rows).astype(np.uint64) if w == 1 else \
            rng.integers(0, 1 << w, rows, dtype=np.uint64, endpoint=False) if 0 < w < 64 else \
            rng.integers(0, 2**64 - 1, rows, dtype=np.uint64, endpoint=True) if w else np.full(rows, 3, np.uint64)
        x = np.cumsum(steps, dtype=np.uint64)
        for t, v in (("INT64", x.view(np.int64)), ("INT32", x.astype(np.uint32).view(np.int32))):
            if t == "INT32" and w > 32:
                continue
            for valid in (None, rng.random(rows) > 0.3):
                c = synth.ColumnData(f"{t}_{w}_{valid is None}", t, v.copy(), valid)
                if valid is not None:
                    c.values[~valid] = 0
                cols.append(c)
    spec = synth.TableSpec(rows, page, [synth.ColumnSpec("DELTA_BINARY_PACKED") for _ in cols])
    data = W.write_file(synth.Table(cols), spec)
    _check(eng, data)
    if rows > 2:
        _check(eng, data, rb=rows // 3, rc=rows // 2)


# ------------------------------------------------------------------ strings

def _strings(name, lens, rows, rng, valid=None):
    off = np.zeros(len(lens) + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    chars = rng.integers(33, 127, int(off[-1])).astype(np.uint8)
    return synth.ColumnData(name, "BYTE_ARRAY",
                            synth.StringData(off, chars, rng.integers(0, len(lens), rows).astype(np.int32)), valid)


@pytest.mark.parametrize("rows", [1, 31, 33, 2049, 20_000])
def test_dictionary_string_lengths(eng, rows):
    """Pools of one length each around the 16-byte steps of the register copy,
    pools mixed up to its limit and one string past it, and nulls."""
    rng = np.random.default_rng(rows)
    pools = [[ln] * 40 for ln in (0, 1, 3, 4, 15, 16, 17, 31, 32, 33, 47, 48, 49)]
    pools += [list(range(4)) * 20, list(range(33)), list(range(49)), list(range(50))]
    cols = [_strings(f"s{i}", np.array(p, np.int64), rows, rng, None if i % 2 else rng.random(rows) > 0.2)
            for i, p in enumerate(pools)]
    spec = synth.TableSpec(rows, 4096, [synth.ColumnSpec("RLE_DICTIONARY") for _ in cols])
    _check(eng, W.write_file(synth.Table(cols), spec))


@pytest.mark.parametrize("enc", ["DELTA_LENGTH_BYTE_ARRAY", "DELTA_BYTE_ARRAY"])
@pytest.mark.parametrize("rows", [1, 2, 129, 513, 1030])
def test_transcoded_string_counts(eng, enc, rows):
    rng = np.random.default_rng(rows)
    cols = [_strings("any", rng.integers(0, 30, 300), rows, rng),
            _strings("empty", np.zeros(3, np.int64), rows, rng),
            _strings("wide", rng.integers(100, 400, 50), rows, rng, rng.random(rows) > 0.5),
            _strings("null", np.array([5]), rows, rng, np.zeros(rows, bool))]
    for page, version in ((1 << 20, 1), (512, 2)):
        spec = synth.TableSpec(rows, page, [synth.ColumnSpec(enc, page_version=version) for _ in cols])
        _check(eng, W.write_file(synth.Table(cols), spec))


# ------------------------------------------------------------------ stages launched for all columns

@pytest.mark.parametrize("codec", ["UNCOMPRESSED", "SNAPPY", "ZSTD"])
@pytest.mark.parametrize("columns", [[5, 0], [5, 1, 4], list(range(8))])  # two: launched column by column
def test_merged_launches(eng, codec, columns):
    from paper_2602_17335_gb300 import native as N
    from paper_2602_17335_gb300.scan import alloc_outputs
    from paper_2602_17335_gb300.tables import write_table
    tab = synth.config2_table(40_000, 18_000, string_pool_size=9000, zipf_k=2000)
    spec = synth.config2_spec(18_000, 1 << 20, codec, 1)
    for c in spec.columns:
        c.compress_threshold = -1.0
    data = write_table(tab, spec).tobytes()
    _check(eng, data, columns)
    _check(eng, data, columns, 17_777, 3001)
    # one plan scanned again, replayed as a graph and launched anew
    expect = R.read_file(data)
    idx = eng.index([to_dev(data)])
    for flags in (N.PQ_SCAN_GRAPH, N.PQ_SCAN_BATCHED):
        plan, sizes = eng.plan(idx, columns, 0, -1, flags)
        for _ in range(3):
            outs = alloc_outputs(sizes)
            eng.scan(plan, outs)
            st, chars = eng.wait(plan, len(outs))
            assert st == N.PQ_OK, N.pq_last_error(eng.ctx)
            for o, c in zip(outs, chars):
                if o.chars is not None:
                    o.chars = o.chars[:c]
            assert_columns_equal(outs, [expect[c] for c in columns])
        N.pq_free_plan(plan)
    N.pq_free_index(idx)
