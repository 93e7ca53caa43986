"""The dense sum's two kernels meet at 912 tiles, and its offsets come from a
scatter or from searches: sizes on both sides, runs that fill a stage exactly,
spill into a second one or fill a whole tile, 1 to 33 workers, lists that are
not 16-byte aligned, and malformed lists, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2108_00951_gb300 as efs

pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import gpu_util as gu  # noqa: E402

TILE = efs.TILE


def _lists(d, counts, seed):
    """Ascending lists, entries drawn evenly; with whole dense tiles and runs of
    640 (a stage) and 641 pairs put into each."""
    rng = np.random.default_rng(seed)
    idx, val = [], []
    for w, c in enumerate(counts):
        j = rng.choice(d, c, replace=False)
        t = 3 + 2 * w  # tiles with runs of 4096, 640 and 641 pairs
        extra = [np.arange(t * TILE, (t + 1) * TILE),
                 (t + 1) * TILE + np.sort(rng.choice(TILE, 640 + w % 2, replace=False))]
        j = np.unique(np.concatenate([j] + (extra if c else [])))
        idx.append(j.astype(np.uint32))
        val.append((rng.standard_normal(j.size) * 10.0 ** rng.integers(-3, 3)).astype(np.float32))
    return idx, val


def _sum(idx, val, d, tiles, off=0):
    it = [gu.to_dev(i.view(np.int32), off) if i.size else
          torch.zeros(1, dtype=torch.int32, device=gu.DEV) for i in idx]
    vt = [gu.to_dev(v, off) if v.size else torch.zeros(1, device=gu.DEV) for v in val]
    counts = torch.tensor([i.size for i in idx], dtype=torch.int32, device=gu.DEV)
    tt = None
    if tiles:
        edges = np.arange(efs.tiles_for(d) - 1, dtype=np.int64) * TILE
        tt = [gu.to_dev(np.append(np.searchsorted(i.astype(np.int64), edges), i.size)
                        .astype(np.int32)) for i in idx]
    dense = torch.full((d,), float("nan"), device=gu.DEV)
    efs.sparse_aggregate(it, vt, counts, d, dense, tiles=tt)
    return dense.cpu().numpy()


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("tiles", [False, True])
@pytest.mark.parametrize("n", [1, 2, 16, 32, 33])
@pytest.mark.parametrize("d", [911 * TILE, 911 * TILE + 1, 1300 * TILE - 5])
def test_dense_sum_around_the_rule(d, n, tiles, off):
    counts = [0 if w % 5 == 4 else 40 * 10 ** (w % 4) for w in range(n)]
    idx, val = _lists(d, counts, n)
    gu.assert_bits(_sum(idx, val, d, tiles, off), oracle.sparse_aggregate(idx, val, d),
                   "d=%d n=%d tiles=%s off=%d" % (d, n, tiles, off))
    assert efs.ef_check_status() == efs.EF_OK


@pytest.mark.parametrize("n", [1, 31, 130, 256])
@pytest.mark.parametrize("tiles", [1, 2, 911])
def test_runs_searched_in_place(tiles, n):
    # up to 911 tiles the reduction searches its runs: empty lists, runs that
    # end with their list, lists that begin at a tile's edge, several hundred lists
    d = tiles * TILE - (3 if tiles < 911 else 0)
    rng = np.random.default_rng(n)
    idx = []
    for w in range(n):
        j = rng.choice(d, min(d, [0, 1, 7, 300][w % 4]), replace=False)
        if w % 4 == 2 and tiles > 1:
            j = np.concatenate([j, [TILE - 1, TILE, d - 1]])
        idx.append(np.unique(j).astype(np.uint32))
    val = [rng.standard_normal(j.size).astype(np.float32) for j in idx]
    gu.assert_bits(_sum(idx, val, d, False), oracle.sparse_aggregate(idx, val, d),
                   "tiles=%d n=%d" % (tiles, n))
    assert efs.ef_check_status() == efs.EF_OK


def test_more_entries_than_the_scatter_takes():
    d, n = 1300 * TILE - 5, 3
    idx, val = _lists(d, [3_000_000] * n, 9)  # over 8 M entries: searches
    gu.assert_bits(_sum(idx, val, d, False), oracle.sparse_aggregate(idx, val, d), "long lists")
    assert efs.ef_check_status() == efs.EF_OK


def test_many_lists_some_scattered_and_some_searched():
    # over 8 M entries together: lists of up to 64 a tile are scattered, the
    # longest and the shortest searched
    d = 1300 * TILE - 5
    two, twov = _lists(d, [75_000, 60_000], 5)
    other, otherv = _lists(d, [300_000, 30], 6)
    other[1], otherv[1] = other[1][:70], otherv[1][:70]
    idx, val = two * 60 + other, twov * 60 + otherv
    assert sum(i.size for i in idx) > 8 << 20
    gu.assert_bits(_sum(idx, val, d, False), oracle.sparse_aggregate(idx, val, d), "mixed lists")
    assert efs.ef_check_status() == efs.EF_OK


def test_one_list_of_more_entries_than_the_scatter_takes():
    # a step that sends 9.4 M pairs from a shifted error memory: its tile index
    # comes from the list, and so do the offsets of its exchange
    d = 9_400_003
    rng = np.random.default_rng(3)
    g, e = (rng.standard_normal(d).astype(np.float32) for _ in range(2))
    gd, ed = gu.to_dev(g), gu.to_dev(e, 1)
    idx = torch.empty(d, dtype=torch.int32, device=gu.DEV)
    val, dense = torch.empty(d, device=gu.DEV), torch.empty(d, device=gu.DEV)
    cnt = torch.empty(1, dtype=torch.int32, device=gu.DEV)
    tt = torch.full((efs.tiles_for(d),), -1, dtype=torch.int32, device=gu.DEV)
    efs.ef_hard_threshold(gd, ed, 0.1, 1e-6, idx, val, cnt, tiles_out=tt)
    ri, rv, _ = oracle.ef_hard_threshold(g, e, 0.1, 1e-6)
    assert int(cnt.item()) == ri.size > 8 << 20
    edges = np.arange(efs.tiles_for(d) - 1, dtype=np.int64) * TILE
    gu.assert_bits(tt.cpu().numpy(), np.append(np.searchsorted(ri.astype(np.int64), edges),
                                               ri.size).astype(np.int32), "tiles")
    efs.sparse_aggregate([idx], [val], cnt, d, dense)
    gu.assert_bits(dense.cpu().numpy(), oracle.sparse_aggregate([ri], [rv], d), "sum")
    assert efs.ef_check_status() == efs.EF_OK


def test_malformed_lists_many_tiles():
    # a tile index that sends a tile another tile's pairs, and an index past d:
    # skipped and latched, every other coordinate as if they were absent
    d = 1000 * TILE
    idx, val = _lists(d, [500, 500], 4)
    edges = np.arange(1000, dtype=np.int64) * TILE
    good = [np.append(np.searchsorted(i.astype(np.int64), edges), i.size) for i in idx]
    wrong = good[1].copy()
    wrong[10] = 0   # tile 10's run begins at the list's first pair
    idx[0][-1] = d + 7
    it = [gu.to_dev(i.view(np.int32)) for i in idx]
    vt = [gu.to_dev(v) for v in val]
    counts = torch.tensor([i.size for i in idx], dtype=torch.int32, device=gu.DEV)
    tt = [gu.to_dev(t.astype(np.int32)) for t in (good[0], wrong)]
    dense = torch.full((d,), float("nan"), device=gu.DEV)
    efs.sparse_aggregate(it, vt, counts, d, dense, tiles=tt)
    assert efs.ef_check_status() == efs.EF_ERR_BAD_INPUT
    got = dense.cpu().numpy()
    ref = oracle.sparse_aggregate([idx[0][:-1], idx[1]], [val[0][:-1], val[1]], d)
    mask = np.ones(d, bool)
    mask[9 * TILE:11 * TILE] = False   # tiles 9 and 10 got wrong runs
    gu.assert_bits(got[mask], ref[mask], "untouched tiles")
    assert np.all(np.isfinite(got))
