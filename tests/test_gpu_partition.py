"""mdj_partition (the shuffle) against the oracle's stable partition, bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2101_08878_gb300 import datagen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _mdj():
    from paper_2101_08878_gb300 import mdj
    return mdj


def _table(n, key_dtype, seed, key_range=None):
    rng = np.random.default_rng(seed)
    kr = key_range or max(4 * n, 16)
    key = rng.integers(-kr, kr, n).astype(key_dtype)
    f64 = datagen.uniform_payload(rng, n, np.float64)
    f32 = datagen.uniform_payload(rng, n, np.float32)
    i32 = rng.integers(-2**31, 2**31 - 1, n).astype(np.int32)
    return [key, f64, f32, i32]


def _check(cols_np, key_col, P):
    mdj = _mdj()
    dev = torch.device("cuda", 0)
    cols = [torch.from_numpy(c).to(dev) for c in cols_np]
    off, rid, outs = mdj.mdj_partition(cols, key_col, P)
    torch.cuda.synchronize()
    w_off, w_rid, w_cols = oracle.partition_table(cols_np, key_col, P)
    assert np.array_equal(off.cpu().numpy(), w_off)
    assert np.array_equal(rid.cpu().numpy().view(np.uint32), w_rid)
    for g, w in zip(outs, w_cols):
        g = g.cpu().numpy()
        assert g.dtype == w.dtype
        assert np.array_equal(g.view(np.uint8), w.view(np.uint8))


@pytest.mark.parametrize("n", [0, 1, 37, 8191, 8192, 8193, 100_003])
@pytest.mark.parametrize("P", [1, 8, 1024])
def test_partition_sizes(n, P):
    _check(_table(n, np.int64, seed=n + P), 0, P)


@pytest.mark.parametrize("P", [2, 3, 7, 64, 1000, 1023])
@pytest.mark.parametrize("key_dtype", [np.int32, np.int64])
def test_partition_fanouts(P, key_dtype):
    _check(_table(50_000, key_dtype, seed=P), 0, P)


@pytest.mark.parametrize("P", [1025, 4096, 65536])
def test_partition_lsd_large_P(P):
    # P above one pass's fan-out: two stable digit passes
    _check(_table(200_000, np.int64, seed=P), 0, P)


def test_partition_key_not_first_and_duplicates():
    cols = _table(60_000, np.int32, seed=5, key_range=40)  # heavy duplicates
    cols = [cols[1], cols[2], cols[0], cols[3]]
    _check(cols, 2, 16)


def test_partition_extreme_keys():
    rng = np.random.default_rng(11)
    ext = np.array([np.iinfo(np.int64).min, np.iinfo(np.int64).max, 0, -1], np.int64)
    key = rng.choice(ext, 20_000)
    _check([key, datagen.uniform_payload(rng, key.size)], 0, 8)


def test_partition_invalid_args():
    mdj = _mdj()
    dev = torch.device("cuda", 0)
    k = torch.arange(10, device=dev)
    for P in (0, 65537):
        with pytest.raises(mdj.MdjError) as e:
            mdj.mdj_partition([k], 0, P)
        assert e.value.status == -1
    with pytest.raises(mdj.MdjError) as e:
        mdj.mdj_partition([k.double()], 0, 4)  # float key
    assert e.value.status == -2


@pytest.mark.parametrize("P", [1, 63, 64, 65, 2000])
@pytest.mark.parametrize("n", [31, 511, 512, 4609, 5631, 5632, 5633, 6143, 6144, 6145, 30_001])
@pytest.mark.parametrize("layout", ["key", "wide", "narrow", "many"])
def test_partition_tile_edges_and_unaligned_columns(P, n, layout):
    # tiles of every size in use, columns that start one element off a 16-byte
    # boundary, both scatter kernels, and (P = 2000) a second pass that reads row ids
    mdj = _mdj()
    key, f64, f32, i32 = _table(n, np.int32 if layout == "narrow" else np.int64, seed=n + P)
    cols_np = {"key": [key], "wide": [f64, key], "narrow": [key, f32], "many": [f32, key, i32, f64]}[layout]
    key_col = next(j for j, c in enumerate(cols_np) if c is key)
    cols = []
    for c in cols_np:
        t = torch.empty(n + 1, dtype=torch.from_numpy(c).dtype, device="cuda:0")
        t[1:] = torch.from_numpy(c)
        cols.append(t[1:])
    w_off, w_rid, w_cols = oracle.partition_table(cols_np, key_col, P)
    for row_ids in (True, False):
        off, rid, outs = mdj.mdj_partition(cols, key_col, P, row_ids=row_ids)
        torch.cuda.synchronize()
        assert np.array_equal(off.cpu().numpy(), w_off)
        if row_ids:
            assert np.array_equal(rid.cpu().numpy().view(np.uint32), w_rid)
        for g, w in zip(outs, w_cols):
            assert np.array_equal(g.cpu().numpy().view(np.uint8), w.view(np.uint8))


def _fmix64(h):
    # MurmurHash3's 64-bit finalizer on an int64 tensor (wraparound multiplies, logical shifts)
    for mult in (0xff51afd7ed558ccd - 2**64, 0xc4ceb9fe1a85ec53 - 2**64):
        h = (h ^ ((h >> 33) & 0x7FFFFFFF)) * mult
    return h ^ ((h >> 33) & 0x7FFFFFFF)


@pytest.mark.parametrize("P", [8, 256])
def test_partition_of_the_largest_table(P):
    # 2^32 - 1 rows of one 4-byte key column, the most a table may have; row
    # i's key is i's bits, so the output checks itself: keys equal to the row
    # ids, ascending in every partition, each in its hash's partition, all there
    n = 2**32 - 1
    mdj = _mdj()
    dev = torch.device("cuda", 0)
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info(dev)[0] < 80 << 30:
        pytest.skip("needs 80 GB of device memory")
    step = 1 << 27
    keys = torch.empty(n, dtype=torch.int32, device=dev)
    for r0 in range(0, n, step):
        keys[r0:r0 + step] = torch.arange(r0, min(n, r0 + step), device=dev)
    off, rid, (out,) = mdj.mdj_partition([keys], 0, P)
    assert torch.equal(rid.view(torch.int32), out)
    del keys, rid
    off = off.cpu().tolist()
    assert off[0] == 0 and off[P] == n and sorted(off) == off
    bounds = torch.tensor(off[1:P], device=dev)
    starts = bounds[bounds < n]
    for r0 in range(0, n, step):
        k = out[r0:r0 + step].to(torch.int64)
        at = torch.arange(r0, r0 + k.numel(), device=dev)
        assert torch.equal(_fmix64(k) & (P - 1), torch.bucketize(at, bounds, right=True))
        row = k & 0xFFFFFFFF
        assert int(row.max()) < n
        last = out[r0 - 1:r0].to(torch.int64) & 0xFFFFFFFF if r0 else row[:0]
        up = torch.cat([last, row])
        down = torch.nonzero(up[1:] <= up[:-1]).view(-1) + r0 + (0 if r0 else 1)
        assert bool(torch.isin(down, starts).all())
    del out
    torch.cuda.empty_cache()


@pytest.mark.parametrize("shifts", [(1, 0, 0, 0), (0, 1, 1, 1), (1, 0, 2, 3), (0, 1, 3, 2)])
@pytest.mark.parametrize("n,P", [(1, 3), (5, 1), (6143, 8), (50_001, 64), (50_001, 65), (20_000, 5000)])
def test_partition_of_columns_off_16_bytes(n, P, shifts):
    # columns that start at any element of a 16-byte line (slices), 8 and 4 bytes wide
    mdj = _mdj()
    for key_col in (0, 3):
        cols_np = _table(n, np.int64, seed=n + P)
        cols = []
        for c, shift in zip(cols_np, shifts):
            t = torch.empty(n + shift, dtype=torch.from_numpy(c).dtype, device="cuda:0")
            t[shift:] = torch.from_numpy(c).to("cuda:0")
            cols.append(t[shift:])
        off, rid, outs = mdj.mdj_partition(cols, key_col, P)
        w_off, w_rid, w_cols = oracle.partition_table(cols_np, key_col, P)
        assert np.array_equal(off.cpu().numpy(), w_off)
        assert np.array_equal(rid.cpu().numpy().view(np.uint32), w_rid)
        for g, w in zip(outs, w_cols):
            assert np.array_equal(g.cpu().numpy().view(np.uint8), w.view(np.uint8))
