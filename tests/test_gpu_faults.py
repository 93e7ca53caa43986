"""Failure detection without faulting the GPU: bounded device waits that run
out latch EF_ERR_TIMEOUT and finish; malformed sparse input is skipped and
latched as EF_ERR_BAD_INPUT; in every case the context stays usable."""
import numpy as np
import pytest
import torch

import oracle
import paper_2108_00951_gb300 as efs

pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import gpu_util as gu  # noqa: E402


def _inputs(d):
    rng = np.random.default_rng(99)
    return (rng.standard_normal(d) * 1e-2).astype(np.float32), \
        (rng.standard_normal(d) * 1e-3).astype(np.float32)


def _healthy_call_matches_oracle(g, e):
    ri, rv, re_ = oracle.ef_hard_threshold(g, e, 0.1, 1e-3)
    gi, gv, ge = gu.ht(g, e, 0.1, 1e-3)
    gu.assert_bits(gi, ri, "idx")
    gu.assert_bits(gv, rv, "val")
    gu.assert_bits(ge, re_, "e'")
    assert efs.ef_check_status() == efs.EF_OK


@pytest.mark.usefixtures("stream_kernel")
@pytest.mark.parametrize("method", ["ht", "topk"])
def test_lookback_wait_runs_out_and_recovers(method):
    d = 40 * 4096 + 9
    g, e = _inputs(d)
    assert efs.ef_check_status() == efs.EF_OK
    efs.ef_test_set_lookback_fault(5, 2000)      # tile 5 never publishes; waits end after 2 ms
    try:
        if method == "ht":
            gu.ht(g, e, 0.1, 1e-3)
        else:
            gu.topk(g, e, 0.1, 1000)
        status = efs.ef_check_status()
    finally:
        efs.ef_test_set_lookback_fault(-1)
    assert status == efs.EF_ERR_TIMEOUT
    assert efs.ef_check_status() == efs.EF_OK     # cleared once reported
    _healthy_call_matches_oracle(g, e)


@pytest.mark.usefixtures("stream_kernel")
@pytest.mark.parametrize("e_off", [0, 1])
def test_count_after_a_wait_that_ran_out(e_off):
    # a failed call's count is 0 whatever the word held, so that nothing after
    # it (with a shifted e the kernel that finds the tile index) reads past the
    # lists
    d = 40 * 4096 + 9
    g, e = _inputs(d)
    gd, ed = gu.to_dev(g, e_off), gu.to_dev(e, e_off)
    idx = torch.zeros(d, dtype=torch.int32, device=gu.DEV)
    val = torch.empty(d, device=gu.DEV)
    cnt = torch.full((1,), 0x7fffffff, dtype=torch.int32, device=gu.DEV)
    tiles = torch.full((efs.tiles_for(d),), -1, dtype=torch.int32, device=gu.DEV)
    assert efs.ef_check_status() == efs.EF_OK
    efs.ef_test_set_lookback_fault(5, 2000)
    try:
        efs.ef_hard_threshold(gd, ed, 0.1, 1e-3, idx, val, cnt, tiles_out=tiles)
        status = efs.ef_check_status()
    finally:
        efs.ef_test_set_lookback_fault(-1)
    assert status == efs.EF_ERR_TIMEOUT
    assert int(cnt.item()) == 0
    if e_off:
        assert not tiles.any()
    _healthy_call_matches_oracle(g, e)


def test_aggregate_malformed_input_is_latched_not_faulting():
    d = 10_000
    good = np.array([1, 50, 9000], np.uint32)
    unsorted = np.array([9000, 5, 4097, 3], np.uint32)
    out_of_range = np.array([2, 9999, 10_000, 4_000_000_000], np.uint32)
    vals = [np.ones(3, np.float32), np.ones(4, np.float32), np.ones(4, np.float32)]
    out = gu.aggregate([good, unsorted, out_of_range], vals, d)
    assert np.all(np.isfinite(out))
    assert efs.ef_check_status() == efs.EF_ERR_BAD_INPUT
    assert efs.ef_check_status() == efs.EF_OK
    g, e = _inputs(5000)
    _healthy_call_matches_oracle(g, e)


def _long_run(at, fix):
    """1,500 ascending entries of tile 1, one of them replaced: position 1,024
    begins the second stage of the run."""
    j = np.arange(4096, 4096 + 3000, 2)
    j[at] = fix(j, at)
    return j


# every kind of malformed list in a call of its own, so that one kind's report
# cannot stand in for another's: (name, the list, the coordinates it may touch)
MALFORMED = [
    ("past the last tile", lambda d: [2, 9, 4_000_000_000]),
    ("at the last tile's end", lambda d: [2, -(-d // 4096) * 4096]),
    ("past d in the last tile", lambda d: [2, d + 1]),
    ("nothing but past d", lambda d: [4_000_000_000]),
    ("another tile's, before it", lambda d: [5000, 10]),
    ("descent within a tile", lambda d: [50, 40]),
    ("repeat within a tile", lambda d: [50, 50]),
    ("repeat across stages", lambda d: _long_run(1024, lambda j, a: j[a - 1])),
    ("descent across stages", lambda d: _long_run(1024, lambda j, a: j[a - 1] - 1)),
    ("repeat inside a stage", lambda d: _long_run(700, lambda j, a: j[a - 1])),
]


@pytest.mark.parametrize("update", [False, True])
@pytest.mark.parametrize("d", [10_000, 911 * 4096 - 3])
@pytest.mark.parametrize("bad", [m[1] for m in MALFORMED], ids=[m[0] for m in MALFORMED])
def test_each_malformed_list_is_latched(bad, d, update):
    good = np.array([1, 60, 9000], np.uint32)
    lists = [good, np.asarray(bad(d), np.int64).astype(np.uint32)]
    vals = [np.full(j.size, 2.0 + w, np.float32) for w, j in enumerate(lists)]
    idx = [gu.to_dev(j.view(np.int32)) for j in lists]
    val = [gu.to_dev(v) for v in vals]
    counts = torch.tensor([j.size for j in lists], dtype=torch.int32, device=gu.DEV)
    out = torch.zeros(d, device=gu.DEV)
    assert efs.ef_check_status() == efs.EF_OK
    if update:
        efs.sparse_aggregate_apply(idx, val, counts, d, 1.0, out)
    else:
        efs.sparse_aggregate(idx, val, counts, d, out)
    assert efs.ef_check_status() == efs.EF_ERR_BAD_INPUT
    assert efs.ef_check_status() == efs.EF_OK
    want = np.zeros(d, np.float32)
    want[good] = 2.0
    apart = np.ones(d, bool)               # coordinates the malformed list does not name
    apart[lists[1][lists[1] < d]] = False
    got = out.cpu().numpy() * (-1.0 if update else 1.0)
    gu.assert_bits((got + 0.0)[apart], want[apart], "the other coordinates")
    assert np.all(np.isfinite(got))


def test_invalid_arguments_launch_nothing():
    before = efs.ef_kernel_launches()
    x = torch.zeros(100, device=gu.DEV)
    i = torch.zeros(100, dtype=torch.int32, device=gu.DEV)
    with pytest.raises(efs.EfError) as err:
        efs.ef_hard_threshold(x, x.clone(), 0.1, -1.0, i, x.clone(), i[:1])
    assert err.value.status == efs.EF_ERR_INVALID_ARG
    i101 = torch.zeros(101, dtype=torch.int32, device=gu.DEV)
    with pytest.raises(efs.EfError) as err:        # k > d
        efs.ef_topk(x, x.clone(), 0.1, 101, i101, torch.zeros(101, device=gu.DEV), i[:1])
    assert err.value.status == efs.EF_ERR_INVALID_ARG
    with pytest.raises(efs.EfError):       # output aliases the error memory
        efs.ef_hard_threshold(x, x, 0.1, 1e-3, i, x[:100], i[:1])
    assert efs.ef_kernel_launches() == before
