"""The scans this engine is used for, as cases to be timed and compared.

A case is a Parquet file (or a set of files) of seeded synthetic columns and
one call on it.  The files are written by the engine's own writer while a case
is prepared; what is timed is the reading: page index, plan, scan and wait
(``Engine.read``), one replay of a captured batch (``pq_batch_launch``), a scan
from pinned host memory to pinned host memory (``pq_scan_host``), or the
decoding of one DELTA stream (``pq_delta_decode_static``).

The columns are those of the repository's workloads: the eight-column table
(dictionary, DELTA, PLAIN, OPTIONAL and string columns), the six-column table
of the other V2 encodings, the single dictionary column, and the five kinds of
chunk of the batched workload.
"""
import math
import random

import numpy as np
import torch

from paper_2602_17335_gb300 import native as N
from paper_2602_17335_gb300.scan import Engine, alloc_outputs, stream_handle

KIB, MIB = 1 << 10, 1 << 20
I32, I64, F64, STR = N.PQ_TYPE_INT32, N.PQ_TYPE_INT64, N.PQ_TYPE_DOUBLE, N.PQ_TYPE_BYTE_ARRAY
PLAIN, DELTA, DLBA, DBA, DICT, BSS = 0, 5, 6, 7, 8, 9
CODEC = {"none": 0, "snappy": 1, "zstd": 6}

# What a row of a column costs at least: (type, OPTIONAL, encoding, encoded bits a row without the
# dictionary, most dictionary bytes a chunk, mean chars a row).
EIGHT = [(I32, False, DICT, 20, 4 << 20, 0), (I64, False, DELTA, 3.3, 0, 0), (F64, False, PLAIN, 64, 0, 0),
         (I32, False, DICT, 14, 40_000, 0), (I64, True, PLAIN, 58.8, 0, 0), (STR, False, DICT, 14, 240_000, 20),
         (I32, False, DICT, 4, 64, 0), (I32, False, DICT, 0.01, 20, 0)]
V2 = [(F64, False, BSS, 64, 0, 0), (I32, False, BSS, 32, 0, 0), (I64, True, BSS, 58.8, 0, 0),
      (STR, False, DLBA, 165, 0, 20), (STR, False, DBA, 12, 0, 18), (STR, True, DBA, 155, 0, 18)]
ONE = [(I32, False, DICT, 10, 4096, 0)]
DELTA_ONE = [(I64, False, DELTA, 3.3, 0, 0)]
KINDS = [(I32, False, DICT, 16, 4 << 16, 0), (STR, False, DICT, 10, 24_000, 20), (F64, False, PLAIN, 64, 0, 0),
         (I64, False, DELTA, 3.3, 0, 0), (I64, True, PLAIN, 58.8, 0, 0)]
TABLES = {"eight": EIGHT, "v2": V2, "one": ONE, "delta": DELTA_ONE, "kinds": KINDS}
# Compressed bytes of a column's pages, as a share of the encoded bytes above.
RATIO = {"none": 1.0, "snappy": 0.95, "zstd": 0.85}


def _case(name, call, table, rows, rg_rows, page_bytes, codec="none", version=1, columns="", row_begin=0, row_count=-1):
    return {"name": name, "call": call, "table": table, "rows": rows, "rg_rows": rg_rows, "page_bytes": page_bytes,
            "codec": codec, "version": version, "columns": columns, "row_begin": row_begin, "row_count": row_count}


def listed():
    return [
        # a small file of a partitioned data set, read whole: latency and launches
        _case("small_file", "read", "eight", 10_007, 10_007, MIB),
        # one dictionary column in a handful of pages: the fewest pages a large column comes in
        _case("one_dict_column", "read", "one", 1 << 20, 1 << 20, MIB),
        # the table scan the engine is quoted on: uncompressed, 1 MiB pages, the largest case
        _case("table_1mib", "read", "eight", 1 << 25, 1 << 22, MIB),
        # the same table as a CPU-oriented writer lays it out: thousands of 8 KiB pages
        _case("table_8kib", "read", "eight", 4_000_037, 1 << 20, 8 * KIB),
        # Snappy, the codec most files come with, in small and in large pages (V1 and V2)
        _case("table_snappy_64kib", "read", "eight", 1 << 23, 1 << 21, 64 * KIB, "snappy"),
        _case("table_snappy_1mib", "read", "eight", 1 << 23, 1 << 21, MIB, "snappy", 2),
        # Zstandard, the archival codec
        _case("table_zstd", "read", "eight", 1 << 20, 1 << 18, 64 * KIB, "zstd"),
        # byte streams split and delta-coded strings
        _case("table_v2_encodings", "read", "v2", 1 << 22, 1 << 20, MIB, "none", 2),
        # a query's projection and row range over a larger file, neither end on a page's edge
        _case("projected_range", "read", "eight", 6_000_011, 1 << 20, 64 * KIB, "none", 2, "1,4,5", 1_234_567, 3_333_333),
        # many uneven chunks of many files in one captured graph, half of them Snappy
        dict(_case("batch_of_files", "batch", "kinds", 1_000_000, 0, 0), files=120, layout=7),
        # file bytes in pinned host memory, columns back to pinned host memory
        _case("host_to_host", "host", "eight", 1 << 23, 1 << 20, MIB),
        # one DELTA stream without any allocation
        _case("delta_stream", "delta", "delta", 2_000_003, 2_000_003, 512 * KIB),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["read", "read", "read", "read", "read", "batch", "host", "delta"])
    if call == "batch":
        return dict(_pure(_case("", call, "kinds", _log(rng, 30_000, 1_000_000), 0, 0)), files=_log(rng, 8, 120),
                    layout=rng.randrange(1 << 20))
    if call == "delta":  # a stream of at most 1 MiB
        rows = _log(rng, 1_000, 2_000_000)
        return _pure(_case("", call, "delta", rows, rows, _log(rng, 8 * KIB, 768 * KIB)))
    page = _log(rng, 8 * KIB, 4 * MIB)
    version = rng.choice([1, 2])
    if call == "host":
        rows = _log(rng, 10_000, 1 << 23)
        return _pure(_case("", call, "eight", rows, _log(rng, max(rows // 12, 4096), rows), max(page, 32 * KIB),
                           rng.choice(["none", "snappy"]), version))
    table = rng.choice(["eight", "eight", "eight", "one", "v2"])
    codec = rng.choice(["none", "none", "snappy", "snappy", "zstd"])
    rows = _log(rng, 1_000, 1 << 23 if table != "v2" else 1 << 22)
    if codec == "zstd":
        rows, page = min(rows, 1 << 20), min(page, 128 * KIB)
    rg = _log(rng, max(rows // 16, 1_000), rows)
    if codec == "zstd":
        rg = min(rg, 1 << 18)
    c = _case("", call, table, rows, rg, page, codec, version)
    n = len(TABLES[table])
    if n > 1 and rng.random() < 0.4:
        c["columns"] = ",".join(map(str, sorted(rng.sample(range(n), rng.randint(1, n - 1)))))
    if rng.random() < 0.3:
        c["row_begin"] = rng.randrange(rows // 2 + 1)
        c["row_count"] = rng.randrange(1, rows - c["row_begin"] + 1)
    return _pure(c)


def _pure(c):
    return {k: v for k, v in c.items() if k != "name"}


def _columns(case):
    t = TABLES[case["table"]]
    return [int(k) for k in case["columns"].split(",")] if case["columns"] else list(range(len(t)))


def _range(case):
    a = case["row_begin"]
    return a, case["rows"] if case["row_count"] < 0 else a + case["row_count"]


# ------------------------------------------------------------------ the data

def _strings(g, n, lens, start, pool, index):
    """Row values of pool entries `index`: (int64 offsets, uint8 chars)."""
    ln = lens[index]
    off = torch.zeros(n + 1, dtype=torch.int64, device=g.device)
    torch.cumsum(ln, 0, out=off[1:])
    chars = torch.empty(int(off[-1]), dtype=torch.uint8, device=g.device)
    for a in range(0, n, 1 << 22):
        b = min(n, a + (1 << 22))
        src = torch.repeat_interleave(start[index[a:b]] - off[a:b], ln[a:b])
        lo, hi = int(off[a]), int(off[b])
        chars[lo:hi] = pool[src + torch.arange(lo, hi, device=g.device)]
    return off, chars


LETTERS = b"ABCDEFGHIJKLMNOPQRSTUVWXYZabcdefghijklmnopqrstuvwxyz0123456789"


def _random_strings(g, n, k, fixed, null_frac=0.0):
    """Rows uniform over about k random strings of 8-32 characters, as many of each length.  Which
    rows are null and how long each row is comes from `fixed`, so that every seed's outputs have
    the same shape; the strings, and which of its length a row takes, come from `g`."""
    per = k // 25
    length = torch.randint(8, 33, (n,), generator=fixed, device=g.device)
    valid = torch.rand(n, generator=fixed, device=g.device) >= null_frac if null_frac else None
    lens = torch.arange(8, 33, device=g.device).repeat_interleave(per)
    start = torch.cumsum(lens, 0) - lens
    letters = torch.tensor(list(LETTERS), dtype=torch.uint8, device=g.device)
    pool = letters[torch.randint(0, 62, (int(lens.sum()),), generator=g, device=g.device)]
    index = (length - 8) * per + torch.randint(0, per, (n,), generator=g, device=g.device)
    if valid is not None:  # a null row has no characters
        lens, start = torch.cat([lens, lens.new_zeros(1)]), torch.cat([start, start.new_zeros(1)])
        index = torch.where(valid, index, 25 * per)
    return (*_strings(g, n, lens, start, pool, index), valid)


def _stem_strings(g, n, rg_rows, seed, fixed, k=4096, stems=64):
    """Rows sorted in each row group over about k strings that share 64 stems of 4-12 characters, with tails of 0-20.
    The seed picks the letters, in their order: every seed's strings have the same lengths in the same rows."""
    r = random.Random(5)
    word = lambda m: bytes(r.choices(range(36), k=m))  # noqa: E731
    stem = [word(r.randint(4, 12)) for _ in range(stems)]
    pool = sorted({stem[r.randrange(stems)] + word(r.randint(0, 20)) for _ in range(k)})
    letters = sorted(random.Random(seed).sample(sorted(LETTERS), 36))
    lens = torch.tensor([len(p) for p in pool], device=g.device)
    chars = torch.tensor([letters[c] for c in b"".join(pool)], dtype=torch.uint8, device=g.device)
    index = _sorted_in_groups(torch.randint(0, len(pool), (n,), generator=fixed, device=g.device), rg_rows)
    return (*_strings(g, n, lens, torch.cumsum(lens, 0) - lens, chars, index), None)


def _sorted_in_groups(v, rg_rows):
    for a in range(0, v.numel(), rg_rows):
        v[a:a + rg_rows] = torch.sort(v[a:a + rg_rows])[0]
    return v


def _column(table, k, n, rg_rows, seed):
    """(values, chars, valid) of column k on the GPU; `values` are offsets for strings."""
    dev = torch.device("cuda")
    g = torch.Generator(dev)
    g.manual_seed((seed * 1000003 + k * 7919 + sorted(TABLES).index(table)) % (1 << 62))
    ints = lambda lo, hi, dt=torch.int32: torch.randint(lo, hi, (n,), generator=g, device=dev, dtype=dt)  # noqa: E731
    full = lambda: torch.randint(-(1 << 63), (1 << 63) - 1, (n,), generator=g, device=dev)  # noqa: E731
    kind = {"eight": ("u20", "keys", "normal", "zipf", "opt", "strings", "card16", "card5"),
            "v2": ("normal", "zipf", "opt", "strings", "stems", "optstrings"), "one": ("u10",), "delta": ("keys",),
            "kinds": ("u16", "strings1k", "normal", "keys", "opt")}[table][k]
    if kind in ("u20", "u16", "u10"):
        return ints(0, 1 << int(kind[1:])), None, None
    if kind == "keys":
        return torch.cumsum(ints(0, 8, torch.int64), 0) + 1, None, None
    if kind == "normal":
        return torch.randn(n, generator=g, device=dev, dtype=torch.float64), None, None
    if kind == "zipf":
        p = torch.arange(1, 10_001, device=dev, dtype=torch.float64) ** -1.1
        cdf = torch.cumsum(p, 0) / p.sum()
        rank = torch.searchsorted(cdf, torch.rand(n, generator=g, device=dev, dtype=torch.float64)).clamp_(max=9_999)
        value = torch.randperm(1 << 22, generator=g, device=dev)[:10_000] * 509 - (1 << 30)
        return value.to(torch.int32)[rank], None, None
    if kind == "opt":
        valid = torch.rand(n, generator=g, device=dev) >= 0.1
        return full() * valid, None, valid
    if kind in ("card16", "card5"):
        pool = torch.randperm(1 << 20, generator=g, device=dev)[:int(kind[4:])].to(torch.int32)
        v = pool[torch.randint(0, pool.numel(), (n,), generator=g, device=dev)]
        return (_sorted_in_groups(v, rg_rows) if kind == "card5" else v), None, None
    fixed = torch.Generator(dev)
    fixed.manual_seed(n + k)
    if kind == "stems":
        return _stem_strings(g, n, rg_rows, seed, fixed)
    return _random_strings(g, n, 1_000 if kind == "strings1k" else 10_000, fixed, 0.1 if kind == "optstrings" else 0.0)


def _write(columns, n, rg_rows, page_bytes, codec, version):
    """A file of [(spec, (values, chars, valid))], as a numpy array."""
    cols, keep = [], []
    for k, ((ptype, _, enc, *_), (values, chars, valid)) in enumerate(columns):
        host = [None if t is None else t.cpu().numpy() for t in (values, chars, valid)]
        w = N.pq_write_column()
        w.name, w.type, w.encoding, w.codec = b"c%d" % k, ptype, enc, CODEC[codec]
        w.page_version, w.compress_threshold = version, -1.0
        w.values = host[0].ctypes.data
        w.chars = host[1].ctypes.data if host[1] is not None and host[1].size else None
        if host[2] is not None:
            host[2] = np.ascontiguousarray(host[2], dtype=np.uint8)
            w.valid = host[2].ctypes.data
        keep.append(host)
        cols.append(w)
    return N.pq_write_table(cols, n, rg_rows, page_bytes)


def _table_file(case, seed):
    t = TABLES[case["table"]]
    cols = [(t[k], _column(case["table"], k, case["rows"], case["rg_rows"], seed)) for k in range(len(t))]
    data = _write(cols, case["rows"], case["rg_rows"], case["page_bytes"], case["codec"], case["version"])
    return torch.from_numpy(data), [0 if chars is None else chars.numel() for _, (_, chars, _) in cols]


def _batch_layout(case):
    """(kind, rows, page bytes, codec, version) of each file of a batch."""
    r = random.Random(case["layout"])
    return [(i % 5 if i < 5 else r.randrange(5), _log(r, 10_000, case["rows"]), _log(r, 4 * KIB, 2 * MIB),
             r.choice(["none", "snappy"]), r.choice([1, 2])) for i in range(case["files"])]


# ------------------------------------------------------------------ the calls

_ENGINE = []


def _engine():
    """The program's one engine."""
    if not _ENGINE:
        _ENGINE.append(Engine(0))
    return _ENGINE[0]


class _Batch:
    """The indexes, plans, outputs and captured graph of a set of files."""

    def __init__(self, case, seed):
        eng = _engine()
        files = [[] for _ in range(5)]
        for i, (kind, n, page, codec, version) in enumerate(_batch_layout(case)):
            col = _column("kinds", kind, n, n, seed * 4096 + i)
            files[kind].append(torch.from_numpy(_write([(KINDS[kind], col)], n, n, page, codec, version)).cuda())
        self.files = files
        self.indexes = [eng.index(f) for f in files]
        self.plans, self.outs = [], []
        for idx in self.indexes:
            plan, sizes = eng.plan(idx)
            self.plans.append(plan)
            self.outs.append(alloc_outputs(sizes))
        self.batch = N.pq_batch_create(eng.ctx, self.plans, [[o.desc() for o in outs] for outs in self.outs],
                                       N.PQ_SCAN_GRAPH)

    def __del__(self):
        if getattr(self, "batch", None):
            N.pq_batch_free(self.batch)
            for p in self.plans:
                N.pq_free_plan(p)
            for i in self.indexes:
                N.pq_free_index(i)


def _pinned(n, dtype):
    return torch.empty(max(int(n), 1), dtype=dtype, pin_memory=True)


def prepare(case, seed):
    s = {"call": case["call"], "columns": _columns(case)}
    if case["call"] == "batch":
        s["batch"] = _Batch(case, seed)
        return s
    data, chars_bytes = _table_file(case, seed)
    if case["call"] == "host":
        pinned = _pinned(data.numel(), torch.uint8).copy_(data)
        s["file"], s["outs"], s["descs"] = pinned, [], []
        n = case["rows"]
        for (ptype, optional, *_), total in zip(TABLES[case["table"]], chars_bytes):
            values = _pinned(n + 1 if ptype == STR else n, {I32: torch.int32, F64: torch.float64}.get(ptype, torch.int64))
            valid = _pinned((n + 31) // 32, torch.int32) if optional else None
            chars = _pinned(total, torch.uint8) if ptype == STR else None
            s["outs"].append((values, valid, chars))
            s["descs"].append(N.pq_column(values.data_ptr(), None if valid is None else valid.data_ptr(),
                                          None if chars is None else chars.data_ptr(),
                                          0 if chars is None else chars.numel()))
        return s
    s["file"] = data.cuda()
    if case["call"] == "delta":  # the value stream of the file's first data page
        idx = _engine().index([s["file"]])
        page = N.pq_index_copy_pages(idx)[0]
        N.pq_free_index(idx)
        s["at"], s["len"], s["n"] = page.header_offset + page.header_len, page.compressed_size, page.num_values
        s["out"] = torch.empty(s["n"], dtype=torch.int64, device="cuda")
        return s
    s["row_begin"], s["row_count"] = case["row_begin"], case["row_count"]
    return s


def _whole(outs):
    return [(o.values, o.validity, o.chars) for o in outs]


def run(state):
    eng = _engine()
    if state["call"] == "read":
        return _whole(eng.read([state["file"]], state["columns"], state["row_begin"], state["row_count"]))
    if state["call"] == "batch":
        b = state["batch"]
        N.pq_batch_launch(eng.ctx, b.batch, stream_handle())
        N.check(N.pq_batch_wait(b.batch), eng.ctx)
        return [_whole(outs) for outs in b.outs]
    if state["call"] == "host":
        f = state["file"]
        N.pq_scan_host(eng.ctx, [(f.data_ptr(), f.numel())], outs=state["descs"])
        return state["outs"]
    N.check(N.pq_delta_decode_static(eng.ctx, state["file"].data_ptr() + state["at"], state["len"], I64, state["n"],
                                     state["out"].data_ptr(), stream_handle()), eng.ctx)
    return state["out"]


# ------------------------------------------------------------------ what it costs, what it gives

def _bytes(spec, n, rg_rows, codec):
    """Stored bytes read and decoded bytes written for n rows of a column."""
    ptype, optional, _, bits, dictionary, chars = spec
    stored = n * bits / 8 + (n / 8 if optional else 0) + math.ceil(n / rg_rows) * min(dictionary, 4 * rg_rows)
    out = n * (4 if ptype == I32 else 8) + (n / 8 if optional else 0) + n * chars
    return stored * RATIO[codec] + out


def work(case):
    if case["call"] == "batch":
        total = sum(_bytes(KINDS[kind], n, n, codec) for kind, n, _, codec, _ in _batch_layout(case))
    elif case["call"] == "delta":  # the pages of a DELTA column hold 1 + 128 k values
        total = _bytes(DELTA_ONE[0], min(case["rows"], 8 * case["page_bytes"] / 3.3), case["rows"], "none")
    else:
        a, b = _range(case)
        total = sum(_bytes(TABLES[case["table"]][k], b - a, case["rg_rows"], case["codec"]) for k in _columns(case))
    return {"bytes": total, "flops": 0}


def exact(case, seed):
    """The columns the files were written from; the scan gives them back bit for bit."""
    if case["call"] == "batch":
        outs = [[] for _ in range(5)]
        for i, (kind, n, *_) in enumerate(_batch_layout(case)):
            outs[kind].append(_column("kinds", kind, n, n, seed * 4096 + i)[0])
        return [[(None if KINDS[k][0] == STR else torch.cat(o), None, None)] for k, o in enumerate(outs)]
    if case["call"] == "delta":
        return None  # whole numbers alone, which stay equal
    a, b = _range(case)
    cols = []
    for k in _columns(case):
        v = _column(case["table"], k, case["rows"], case["rg_rows"], seed)[0]
        cols.append((None if TABLES[case["table"]][k][0] == STR else v[a:b].clone(), None, None))
    return cols
