"""The merge's shuffle at the edges of its tiles: ragged sizes, columns that
start off a 16-byte boundary, several columns, and pass-2 tiles that touch
many pass-1 buckets.  Every result against the oracle, bit for bit."""
import numpy as np
import pytest

import oracle
from joinhelp import assert_same_result, gpu_result_np
from paper_2101_08878_gb300 import datagen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _shifted(cols, shift):
    """Device copies of `cols` that start `shift` elements into their allocations."""
    out = []
    for c in cols:
        t = torch.empty(c.size + shift, dtype=torch.from_numpy(c).dtype, device=DEV)
        t[shift:] = torch.from_numpy(c).to(DEV)
        out.append(t[shift:])
    return out


def _check(left, right, P, shift=0):
    from paper_2101_08878_gb300 import mdj
    res = mdj.mdj_merge(_shifted(left, shift), _shifted(right, shift), P)
    torch.cuda.synchronize()
    assert_same_result(gpu_result_np(res), oracle.merge_table(left, right, 0, 0))


def _tables(nl, nr, kd, pd, seed):
    rng = np.random.default_rng(seed)
    span = max(2, 2 * max(nl, nr))
    lk = rng.permutation(span)[:nl].astype(kd)
    rk = rng.integers(0, span, nr).astype(kd)
    return [lk, datagen.uniform_payload(rng, nl, pd)], [rk, datagen.uniform_payload(rng, nr, pd)]


@pytest.mark.parametrize("n", [1, 2, 15, 17, 5167, 5168, 5169, 5695, 5696, 5697, 6143, 6144, 6145, 12_289])
@pytest.mark.parametrize("kd,pd", [(np.int64, np.float64), (np.int32, np.float32)])
def test_tile_edges(n, kd, pd):
    left, right = _tables(n, n + 1, kd, pd, n)
    for P in (2, 128, 1000):
        _check(left, right, P)


@pytest.mark.parametrize("shift", [1, 2, 3])
@pytest.mark.parametrize("kd,pd", [(np.int64, np.float64), (np.int32, np.float32), (np.int64, np.float32),
                                   (np.int32, np.float64)])
def test_unaligned_columns(shift, kd, pd):
    left, right = _tables(40_003, 50_001, kd, pd, shift)
    _check(left, right, 8, shift)


@pytest.mark.parametrize("ncols", [0, 1, 2, 4])
def test_column_counts(ncols):
    rng = np.random.default_rng(ncols)
    left, right = _tables(30_011, 20_013, np.int64, np.float64, 9)
    kinds = [np.float32, np.float64, np.float32, np.float64]
    left = left[:1] + [datagen.uniform_payload(rng, 30_011, k) for k in kinds[:ncols]]
    right = right[:1] + [datagen.uniform_payload(rng, 20_013, k) for k in kinds[:ncols]]
    _check(left, right, 8, 1)


@pytest.mark.parametrize("nr", [3, 1000, 60_001, 400_003])
def test_two_level_plan_small_probe_side(nr):
    # the plan follows the 4M-row build side, so a small probe side's pass-1
    # buckets are shorter than a tile
    left, right = _tables(4_000_003, nr, np.int64, np.float64, 5)
    _check(left, right, 8, 1)


def test_two_level_plan_few_distinct_keys():
    # rows of a handful of pass-1 buckets far apart: tiles go direct
    rng = np.random.default_rng(6)
    left, _ = _tables(4_000_000, 1, np.int32, np.float32, 7)
    rk = rng.choice(left[0][:5], 30_000)
    _check(left, [rk, datagen.uniform_payload(rng, rk.size, np.float32)], 8)


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("kd,pd", [(np.int64, np.float64), (np.int32, np.float32)])
def test_batch_segments_of_ragged_sizes(kd, pd, shift):
    # segments start at any row, hold less than a tile or several, and differ in bucket counts
    from paper_2101_08878_gb300 import mdj
    nl = [1, 0, 5, 5183, 5184, 12_345, 3, 40_001, 700_001]
    nr = [2, 7, 0, 5185, 11_111, 1, 8192, 90_003, 50_001]
    P = [1, 8, 3, 32, 1, 1000, 8, 7, 1]
    pairs = [_tables(a, b, kd, pd, 100 + i) for i, (a, b) in enumerate(zip(nl, nr))]
    left = [np.concatenate([p[0][c] for p in pairs]) for c in (0, 1)]
    right = [np.concatenate([p[1][c] for p in pairs]) for c in (0, 1)]
    lo, ro = np.concatenate([[0], np.cumsum(nl)]), np.concatenate([[0], np.cumsum(nr)])
    res, offs = mdj.mdj_merge_batch(_shifted(left, shift), _shifted(right, shift), lo, ro, P)
    torch.cuda.synchronize()
    for i, (l, r) in enumerate(pairs):
        a, b = offs[i], offs[i + 1]
        part = mdj.JoinResult(b - a, res.key[a:b], res.left_row.view(torch.int32)[a:b] - int(lo[i]),
                              res.right_row.view(torch.int32)[a:b] - int(ro[i]), [c[a:b] for c in res.left_cols],
                              [c[a:b] for c in res.right_cols])
        assert_same_result(gpu_result_np(part), oracle.merge_table(l, r, 0, 0))


@pytest.mark.parametrize("nl,P", [(3481, 1), (3482, 1), (3482, 7), (3_564_544, 1), (3_564_545, 1), (3_564_545, 1000)])
def test_plan_boundaries(nl, P):
    # unpartitioned / one pass, and one pass / two passes, at the sizes where the plan changes
    left, right = _tables(nl, 12_289, np.int32, np.float32, nl % 1000)
    _check(left, right, P)


def test_one_pass_plan_with_many_items_per_bucket():
    # 20 build rows of each key against probe chunks of several items, empty buckets in between
    rng = np.random.default_rng(8)
    lk = np.repeat(rng.permutation(10_000)[:400], 20).astype(np.int64)
    rk = rng.choice(np.concatenate([lk[:40], rng.integers(0, 10_000, 300)]), 60_001)
    _check([lk, datagen.uniform_payload(rng, lk.size)], [rk, datagen.uniform_payload(rng, rk.size)], 16)


@pytest.mark.parametrize("P", [512, 513, 1024])
@pytest.mark.parametrize("nl,nr,shift", [(1, 2, 0), (70_001, 171_111, 1), (900_001, 1_800_003, 0), (10, 3_600_001, 1)])
@pytest.mark.parametrize("kd,pd", [(np.int64, np.float64), (np.int32, np.float32)])
def test_pass_in_wide_blocks(P, nl, nr, shift, kd, pd):
    # more than 512 buckets: one 1024-thread block per SM and tiles of up to 12288 rows
    left, right = _tables(nl, nr, kd, pd, nl + P)
    _check(left, right, P, shift)


@pytest.mark.parametrize("ncols", [0, 3])
def test_wide_blocks_column_counts(ncols):
    rng = np.random.default_rng(ncols)
    left, right = _tables(300_011, 2_000_013, np.int64, np.float64, 9)
    kinds = [np.float32, np.float64, np.float32]
    left = left[:1] + [datagen.uniform_payload(rng, 300_011, k) for k in kinds[:ncols]]
    right = right[:1] + [datagen.uniform_payload(rng, 2_000_013, k) for k in kinds[:ncols]]
    _check(left, right, 600, 1)


@pytest.mark.parametrize("P,short", [(299, 0), (300, 1), (300, 0), (512, 0)])
def test_wide_blocks_from_many_rows(P, short):
    # from 300 buckets on when both sides have 2^25 rows or more; row i of the
    # right side has key i, the left keys are a sample of them
    from paper_2101_08878_gb300 import mdj
    n_l = 5000
    n_r = 2**25 - n_l - short
    rng = np.random.default_rng(P)
    lk = rng.integers(-n_r // 3, n_r, n_l).astype(np.int32)
    lk[:2] = [0, n_r - 1]
    rp = torch.arange(n_r, dtype=torch.int32, device=DEV) * 3
    left = [torch.from_numpy(lk).to(DEV), torch.arange(n_l, dtype=torch.int32, device=DEV) * 7]
    res = mdj.mdj_merge(left, [torch.arange(n_r, dtype=torch.int32, device=DEV), rp], P)
    cols = (res.key, res.left_row.view(torch.int32), res.right_row.view(torch.int32), res.left_cols[0], res.right_cols[0])
    got = [t.cpu().numpy() for t in cols]
    lrow = np.flatnonzero(lk >= 0).astype(np.int32)
    want = [lk[lrow], lrow, lk[lrow], lrow * 7, lk[lrow] * 3]
    order = [np.lexsort((c[1], c[0])) for c in (got, want)]
    for g, w in zip(got, want):
        assert np.array_equal(g[order[0]], w[order[1]])


@pytest.mark.parametrize("env", ["MDJ_ORDERED_OUTPUT", "MDJ_STABLE_SHUFFLE"])
@pytest.mark.parametrize("nr", [3, 1000, 60_001])
def test_two_level_stable_plan_small_probe_side(monkeypatch, env, nr):
    # the stable passes' direct path: a tile of the small side touches most pass-1 buckets
    monkeypatch.setenv(env, "1")
    left, right = _tables(4_000_003, nr, np.int64, np.float32, nr)
    _check(left, right, 8, 1)
