"""mdj_count_checksum at the edges of its tables and plans, exact against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2101_08878_gb300 import datagen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _check(left, right, P, shift=0):
    from paper_2101_08878_gb300 import mdj

    def dev(cols):
        out = []
        for c in cols:
            t = torch.empty(c.size + shift, dtype=torch.from_numpy(c).dtype, device=DEV)
            t[shift:] = torch.from_numpy(c).to(DEV)
            out.append(t[shift:])
        return out

    pays = [c[1] if len(c) > 1 else np.zeros(c[0].size, np.uint64) for c in (left, right)]
    assert mdj.mdj_count_checksum(dev(left), dev(right), P) == oracle.count_checksum(left[0], pays[0], right[0], pays[1])


@pytest.mark.parametrize("P", [1, 8, 1000, 2000])
@pytest.mark.parametrize("hot", [4000, 4096, 4097, 8193, 30_000])
@pytest.mark.parametrize("kd,pd", [(np.int64, np.float64), (np.int32, np.float32)])
def test_hot_keys_around_one_table(P, hot, kd, pd):
    # one key with `hot` build rows (a table holds 4096), two with a few hundred, the rest spread; negative keys too
    rng = np.random.default_rng(hot + P)
    lk = np.concatenate([np.full(hot, -5), np.full(300, 7), np.full(700, 11), rng.integers(-3000, 3000, 9001)])
    rk = np.concatenate([np.full(9000, -5), np.full(50, 7), rng.integers(-6000, 6000, 12_007)])
    lk, rk = rng.permutation(lk).astype(kd), rng.permutation(rk).astype(kd)
    _check([lk, datagen.uniform_payload(rng, lk.size, pd)], [rk, datagen.uniform_payload(rng, rk.size, pd)], P, hot % 2)


@pytest.mark.parametrize("n_l,n_r,P", [(1, 1, 1), (3481, 70_000, 1), (3482, 131_073, 1), (100, 200_001, 4)])
def test_small_build_sides_and_many_probe_units(n_l, n_r, P):
    rng = np.random.default_rng(n_r)
    lk, rk = rng.integers(0, 500, n_l).astype(np.int64), rng.integers(0, 500, n_r).astype(np.int64)
    _check([lk, datagen.uniform_payload(rng, n_l)], [rk, datagen.uniform_payload(rng, n_r)], P, 1)


def test_two_level_plan_with_hot_keys_and_no_payload():
    rng = np.random.default_rng(3)
    lk = np.concatenate([rng.integers(0, 10**6, 4_000_000), np.full(50_000, 123), np.full(6000, 456)])
    rk = np.concatenate([rng.integers(0, 10**6, 500_000), np.full(100_000, 123)])
    _check([rng.permutation(lk)], [rng.permutation(rk)], 8)


def test_terms_under_the_stable_passes(monkeypatch):
    monkeypatch.setenv("MDJ_STABLE_SHUFFLE", "1")
    rng = np.random.default_rng(4)
    lk, rk = rng.integers(0, 5000, 60_000), rng.integers(0, 5000, 50_000)
    _check([lk, datagen.uniform_payload(rng, lk.size)], [rk, datagen.uniform_payload(rng, rk.size)], 8)


def test_largest_probe_side_of_an_unpartitioned_plan():
    # 2^32 - 1 probe rows, the most a table may have; row i's key is i's bits,
    # so a build key's one probe row is the key's own bits (-1 has none)
    from paper_2101_08878_gb300 import mdj
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info(DEV)[0] < 80 << 30:
        pytest.skip("needs 80 GB of device memory")
    n, step = 2**32 - 1, 1 << 27
    rk = torch.empty(n, dtype=torch.int32, device=DEV)
    for r0 in range(0, n, step):
        rk[r0:r0 + step] = torch.arange(r0, min(n, r0 + step), device=DEV)
    rng = np.random.default_rng(9)
    lk = np.concatenate([rng.integers(-2**31, 2**31, 3000), [-1, -2, 0, -1, 5, 5]]).astype(np.int32)
    hit = lk != -1
    rows = lk.view(np.uint32).astype(np.uint64)
    f, _ = oracle.checksum_terms(lk, np.zeros(lk.size, np.uint64), np.zeros(1, np.uint64))
    with np.errstate(over="ignore"):
        g = oracle.fmix64(np.uint64(0xC2B2AE3D27D4EB4F) * (rows + np.uint64(1)))
        want = int((f * g)[hit].sum(dtype=np.uint64))
    assert mdj.mdj_count_checksum([torch.from_numpy(lk).to(DEV)], [rk], 1) == (int(hit.sum()), want)
    del rk
    torch.cuda.empty_cache()


@pytest.mark.parametrize("n_l,hot", [(6_000_000, 0), (18_000_000, 0), (200_000, 16_384), (200_000, 16_385), (200_000, 17_000)])
def test_sub_buckets_around_four_tables(n_l, hot):
    # 1025 partitions have no sub-buckets: 5.9K and 17.6K build rows each,
    # mostly distinct keys (two tables, and the global one), or one partition
    # with a key of about four tables' rows
    rng = np.random.default_rng(n_l + hot)
    key_range = 2 * n_l
    lk = rng.integers(0, key_range, n_l).astype(np.int32)
    rk = rng.integers(0, key_range, 1_000_003).astype(np.int32)
    lk[:hot] = 77
    rk[:hot // 2] = 77
    lk, rk = rng.permutation(lk), rng.permutation(rk)
    lp, rp = datagen.uniform_payload(rng, lk.size, np.float32), datagen.uniform_payload(rng, rk.size, np.float32)
    from paper_2101_08878_gb300 import mdj
    left, right = [[torch.from_numpy(c).to(DEV) for c in t] for t in ((lk, lp), (rk, rp))]
    want = oracle.count_checksum_dense(lk, lp, rk, rp, key_range)
    assert mdj.mdj_count_checksum(left, right, 1025) == want
    assert mdj.mdj_count_checksum(left, right, 8) == want
