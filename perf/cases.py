"""Performance cases: the work a program has this library do, through its public entry points.

Every merge-like call returns its rows in an order of its own, so a program
that wants them in a fixed order puts them there.  A matched right row has one
left row here (unique left keys, the paper's benchmark tables), so `run` writes
each result row as one record, every column of it, to its right row's place in
a buffer the program keeps (an unmatched row of an outer join: to its own
place).  That step is part of each pass.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2101_08878_gb300 import mdj
from paper_2101_08878_gb300.datagen import log_uniform_sizes

DTYPES = {"i32": torch.int32, "i64": torch.int64, "f32": torch.float32, "f64": torch.float64}
NO_ROW = -1  # mdj.NO_ROW's bits as an int32


def listed():
    """The cases, smallest calls first."""
    return [
        # the smallest served request: 10K rows a side, where launches and allocations are all of the time
        {"name": "merge_10k", "kind": "merge", "nl": 10_007, "nr": 12_345, "P": 1, "frac": 0.3, "key": "i64",
         "pay": "f64"},
        # the plain single merge of two 1M-row tables
        {"name": "merge_1M", "kind": "merge", "nl": 1_000_000, "nr": 1_000_000, "P": 1, "frac": 0.3, "key": "i64",
         "pay": "f64"},
        # a served request with 4-byte keys and payloads, sides of unequal, ragged size
        {"name": "merge_i32_3M_7M", "kind": "merge", "nl": 3_000_017, "nr": 7_000_003, "P": 32, "frac": 0.3,
         "key": "i32", "pay": "f32"},
        # the paper's cuDF merge on one worker's tables (chunk size 1E8, 8 partitions, match fraction 0.3)
        {"name": "merge_100M", "kind": "merge", "nl": 100_000_000, "nr": 100_000_000, "P": 8, "frac": 0.3,
         "key": "i64", "pay": "f64"},
        # keys of two int32 columns (a composite key), 20M rows a side
        {"name": "multi_key_20M", "kind": "multi", "nl": 20_000_000, "nr": 20_000_000, "P": 8, "frac": 0.3,
         "key": "i32", "pay": "f64"},
        # 256 independent partition pairs of uneven sizes joined in one call
        {"name": "join_batch_256", "kind": "batch", "pairs": 256, "lo": 1_000, "hi": 4_000_000, "sizes": 3,
         "merge": False, "key": "i64", "pay": "f64"},
        # a group of queued merge requests of mixed sizes and partition counts, served together
        {"name": "served_group_12", "kind": "batch", "pairs": 12, "lo": 10_000, "hi": 20_000_000, "sizes": 44,
         "merge": True, "key": "i32", "pay": "f32"},
        # an outer join written window by window
        {"name": "stream_outer_20M", "kind": "stream", "nl": 20_000_000, "nr": 20_000_000, "P": 8, "frac": 0.3,
         "how": "outer", "windows": 4, "key": "i64", "pay": "f64"},
        # the skewed many-to-many merge (Zipf keys on both sides), counted and checksummed
        {"name": "zipf_count_50M_200M", "kind": "zipf", "nl": 50_000_000, "nr": 200_000_000, "P": 64,
         "values": 10_000_000, "s": 1.1},
        # the shuffle by itself: a table's rows to 8 workers' receive buffers
        {"name": "partition_50M", "kind": "partition", "n": 50_000_000, "P": 8, "cols": "i64,f64"},
        # host tables that fit the device, merged from pinned memory
        {"name": "host_merge_10M", "kind": "host", "nl": 10_000_000, "nr": 10_000_000, "P": 8, "frac": 0.3,
         "key": "i64", "pay": "f64"},
        # the sum of an array and its transpose at the paper's size
        {"name": "transpose_16384", "kind": "transpose", "n": 16_384, "dtype": "f64"},
    ]


def _size(rng, lo, hi):
    """A row count log-uniform in [lo, hi]."""
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    """One more case of the listed cases' ranges."""
    kind = rng.choice(["merge", "merge", "merge", "partition", "partition", "transpose", "multi", "stream", "batch",
                       "zipf", "host"])
    key, pay = rng.choice(["i32", "i64"]), rng.choice(["f32", "f64"])
    if kind in ("merge", "multi", "stream", "host"):
        top = {"merge": 40_000_000, "multi": 20_000_000, "stream": 20_000_000, "host": 10_000_000}[kind]
        c = {"kind": kind, "nl": _size(rng, 10_000, top), "nr": _size(rng, 10_000, top),
             "P": rng.choice([1, 7, 8, 32, 64]), "frac": round(rng.uniform(0.1, 0.9), 2), "key": key, "pay": pay}
        if kind == "stream":
            c |= {"how": rng.choice(["inner", "left", "right", "outer"]), "windows": rng.randint(1, 5)}
        return c
    if kind == "batch":
        merge = rng.random() < 0.5
        pairs = rng.randint(2, 16) if merge else rng.randint(16, 256)
        return {"kind": kind, "pairs": pairs, "lo": 10_000 if merge else 1_000,
                "hi": 20_000_000 // pairs if merge else 1_000_000, "sizes": rng.randrange(1 << 20), "merge": merge,
                "key": key, "pay": pay}
    if kind == "zipf":
        return {"kind": kind, "nl": _size(rng, 100_000, 20_000_000), "nr": _size(rng, 100_000, 50_000_000),
                "P": rng.choice([1, 8, 64]), "values": _size(rng, 10_000, 10_000_000), "s": 1.1}
    if kind == "partition":
        return {"kind": kind, "n": _size(rng, 1_000, 50_000_000), "P": rng.choice([1, 3, 8, 32, 100, 256, 1000, 4096]),
                "cols": rng.choice(["i64,f64", "i32,f32", "i64,f64,f32", "f64,i32,i64"])}
    return {"kind": "transpose", "n": _size(rng, 500, 16_384), "dtype": rng.choice(["f32", "f64", "i32", "i64"])}


# ------------------------------------------------------------------ inputs

def _payload(n, kind, g, dev):
    if kind.startswith("f"):
        return torch.rand(n, generator=g, device=dev, dtype=DTYPES[kind])
    return torch.randint(-(1 << 30), 1 << 30, (n,), generator=g, device=dev, dtype=DTYPES[kind])


def _match_keys(nl, nr, frac, dtype, g, dev):
    """Left keys a permutation of [0, nl); floor(frac * nr) right keys drawn from them, the rest from [nl, 2 nl)."""
    m = int(frac * nr)
    lk = torch.randperm(nl, generator=g, device=dev).to(dtype)
    rk = torch.cat([torch.randint(0, nl, (m,), generator=g, device=dev),
                    torch.randint(nl, 2 * nl, (nr - m,), generator=g, device=dev)])
    return lk, rk[torch.randperm(nr, generator=g, device=dev)].to(dtype)


def _zipf_keys(n, values, s, g, dev):
    """n keys in [0, values) with P(k) proportional to (k + 1)^-s, by inverse CDF."""
    cdf = np.cumsum(np.arange(1, values + 1, dtype=np.float64) ** -s)
    cdf = torch.from_numpy(cdf / cdf[-1]).to(dev)  # summed on the host: the same table every time
    u = torch.rand(n, generator=g, device=dev, dtype=torch.float64)
    return torch.searchsorted(cdf, u, right=True).clamp_(max=values - 1)


def _records(cols):
    """The rows of equally long columns as records of whole 16- or 8-byte words (an odd 4-byte column twice).  Two
    columns become one of twice the width as the parts of a complex number, whose bits are the columns' own."""
    narrow = [c.view(torch.float32) for c in cols if c.element_size() == 4]
    words = [c.view(torch.float64) for c in cols if c.element_size() == 8]
    if len(narrow) % 2:
        narrow.append(narrow[-1])
    words += [torch.complex(a, b).view(torch.float64) for a, b in zip(narrow[::2], narrow[1::2])]
    if len(words) % 2 == 0:
        words = [torch.complex(a, b) for a, b in zip(words[::2], words[1::2])]
    return torch.stack(words, 1)


def _place(buf, res, n_other=0):
    """The rows of `res` as records of every column at their right row's place of `buf`; a row without a right row
    goes to place n_other + its left row."""
    at = res.right_row.view(torch.int32)
    if n_other:
        lrow = res.left_row.view(torch.int32)
        at = torch.where(at == NO_ROW, lrow + n_other, at)
    if res.nrows:
        cols = [c for c in [res.key, res.left_row, res.right_row, *res.left_cols, *res.right_cols] if c.numel()]
        buf.index_copy_(0, at.long(), _records(cols))
    return buf.view(torch.float32).view(torch.int32)


def _batch_sizes(case):
    r = np.random.Generator(np.random.PCG64(case["sizes"]))
    nl = log_uniform_sizes(r, case["pairs"], case["lo"], case["hi"])
    nr = log_uniform_sizes(r, case["pairs"], case["lo"], case["hi"])
    return nl, nr, r.uniform(0.1, 0.9, case["pairs"]), r.choice([1, 8, 32], case["pairs"])


def prepare(case, seed):
    """The tables (or array) of one case, made from the seed, and the buffer that receives the ordered rows."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    kind = case["kind"]
    st = {"case": case}
    if kind == "transpose":
        st["x"] = _payload(case["n"] * case["n"], case["dtype"], g, dev).view(case["n"], case["n"])
        return st
    if kind == "partition":
        cols = [_payload(case["n"], c, g, dev) for c in case["cols"].split(",")]
        # a column of integers is the key: the benchmark's unique keys, shuffled
        ints = [j for j, c in enumerate(cols) if not c.is_floating_point()]
        st["key_col"] = ints[-1]
        cols[st["key_col"]] = torch.randperm(case["n"], generator=g, device=dev).to(cols[st["key_col"]].dtype)
        st["cols"] = cols
        return st
    if kind == "zipf":
        for side, n in (("left", case["nl"]), ("right", case["nr"])):
            st[side] = [_zipf_keys(n, case["values"], case["s"], g, dev), _payload(n, "f64", g, dev)]
        return st
    key = DTYPES[case["key"]]
    if kind == "batch":
        nl, nr, frac, P = _batch_sizes(case)
        pairs = [_match_keys(int(a), int(b), float(f), key, g, dev) for a, b, f in zip(nl, nr, frac)]
        lk, rk = torch.cat([p[0] for p in pairs]), torch.cat([p[1] for p in pairs])
        st["loff"] = [0] + [int(v) for v in np.cumsum(nl)]
        st["roff"] = [0] + [int(v) for v in np.cumsum(nr)]
        st["P"] = [int(p) for p in P]
    else:
        lk, rk = _match_keys(case["nl"], case["nr"], case["frac"], key, g, dev)
    left = [lk, _payload(lk.numel(), case["pay"], g, dev)]
    right = [rk, _payload(rk.numel(), case["pay"], g, dev)]
    if kind == "multi":
        # the key as two columns: its high and low part
        left = [lk // 4099, lk % 4099, left[1]]
        right = [rk // 4099, rk % 4099, right[1]]
    rows = torch.zeros(1, dtype=torch.int32, device=dev)
    one = _records([rows, rows, *[c[:1] for c in left], right[-1][:1]])  # a record of every result column
    places = rk.numel() + (lk.numel() if kind == "stream" else 0)
    st["buf"] = torch.zeros((places, one.shape[1]), dtype=one.dtype, device=dev)
    if kind == "host":
        left = [torch.empty(c.shape, dtype=c.dtype, pin_memory=True).copy_(c) for c in left]
        right = [torch.empty(c.shape, dtype=c.dtype, pin_memory=True).copy_(c) for c in right]
    st["left"], st["right"] = left, right
    return st


# -------------------------------------------------------------------- pass

def run(st):
    """One pass: the public call, and its rows put in order."""
    case = st["case"]
    kind = case["kind"]
    if kind == "transpose":
        return mdj.transpose_add(st["x"])
    if kind == "partition":
        offsets, row_ids, cols = mdj.mdj_partition(st["cols"], st["key_col"], case["P"])
        return [offsets, row_ids.view(torch.int32), cols]
    if kind == "zipf":
        count, checksum = mdj.mdj_count_checksum(st["left"], st["right"], case["P"])
        # the checksum is an unsigned 64-bit number: two halves
        return [count, checksum >> 32, checksum & 0xFFFFFFFF]
    if kind == "merge":
        return _place(st["buf"], mdj.mdj_merge(st["left"], st["right"], case["P"]))
    if kind == "multi":
        return _place(st["buf"], mdj.mdj_merge_multi(st["left"], st["right"], [0, 1], [0, 1], case["P"]))
    if kind == "batch":
        if case["merge"]:
            res, offs = mdj.mdj_merge_batch(st["left"], st["right"], st["loff"], st["roff"], st["P"])
        else:
            res, offs = mdj.mdj_join_batch(st["left"], st["right"], st["loff"], st["roff"])
        return [np.array(offs, dtype=np.int64), _place(st["buf"], res)]
    if kind == "stream":
        with mdj.MergeStream(st["left"], st["right"], case["P"], how=case["how"]) as ms:
            rows = max(1, -(-ms.total_rows // case["windows"]))
            for _, piece in ms.windows(rows):
                _place(st["buf"], piece, st["right"][0].numel())
        return st["buf"].view(torch.float32).view(torch.int32)
    # host tables: each window is put in order while it is on the device
    total, _ = mdj.merge_host_chunked(st["left"], st["right"], case["P"], 16 << 30,
                                      on_piece=lambda first, piece: _place(st["buf"], piece))
    return [total, st["buf"].view(torch.float32).view(torch.int32)]


def _width(name):
    return 4 if name.endswith("32") else 8


def work(case):
    """Bytes of one pass: each input read once, each output row written once."""
    kind = case["kind"]
    if kind == "transpose":
        n = case["n"]
        return {"bytes": 2 * n * n * _width(case["dtype"]), "flops": n * n if case["dtype"][0] == "f" else 0}
    if kind == "partition":
        w = sum(_width(c) for c in case["cols"].split(","))
        return {"bytes": case["n"] * (2 * w + 4) + 8 * (case["P"] + 1), "flops": 0}
    if kind == "zipf":
        return {"bytes": 16 * (case["nl"] + case["nr"]), "flops": 0}
    kw, pw = _width(case["key"]), _width(case["pay"])
    if kind == "batch":
        nl, nr, frac, _ = _batch_sizes(case)
        m = sum(int(f * b) for f, b in zip(frac, nr))
        return {"bytes": (kw + pw) * int(nl.sum() + nr.sum()) + (kw + 8 + 2 * pw) * m, "flops": 0}
    nl, nr = case["nl"], case["nr"]
    m = int(case["frac"] * nr)
    if kind == "multi":
        return {"bytes": (2 * kw + pw) * (nl + nr) + (2 * kw + 8 + 2 * pw) * m, "flops": 0}
    rows = m
    if kind == "stream":
        if case["how"] in ("right", "outer"):
            rows += nr - m
        if case["how"] in ("left", "outer"):  # left rows that no right row drew
            rows += int(nl * math.exp(-m / nl))
    return {"bytes": (kw + pw) * (nl + nr) + (kw + 8 + 2 * pw) * rows, "flops": 0}


def exact(case, seed):
    """The transpose-sum in 64 bits; every other output is whole numbers and copied bits."""
    if case["kind"] != "transpose" or case["dtype"][0] != "f":
        return None
    x = prepare(case, seed)["x"].double()
    return x + x.t()
