"""Hard-threshold calls of 4.2 to 16.8 M coordinates change kernel with the
density of the calls before them (static chunks, or claimed groups once a call
sent at least 1/12): dense and sparse calls in a row on one stream, with and
without tile indexes and norm, each against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2108_00951_gb300 as efs

pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import gpu_util as gu  # noqa: E402


@pytest.mark.parametrize("d", [1024 * 4096 - 5, 1030 * 4096 + 1])
def test_dense_and_sparse_calls_in_a_row(d):
    rng = np.random.default_rng(d)
    g = rng.standard_normal(d).astype(np.float32)
    e0 = (rng.standard_normal(d) * 0.1).astype(np.float32)
    gd = gu.to_dev(g)
    idx = torch.empty(d, dtype=torch.int32, device=gu.DEV)
    val = torch.empty(d, device=gu.DEV)
    cnt = torch.empty(1, dtype=torch.int32, device=gu.DEV)
    tiles = torch.empty(efs.tiles_for(d), dtype=torch.int32, device=gu.DEV)
    err = torch.empty(1, dtype=torch.float64, device=gu.DEV)
    norms = {}
    want = {lam: oracle.ef_hard_threshold(g, e0, 0.1, lam) for lam in (0.1, 0.5)}  # 48 %, 0.04 %
    for n, lam in enumerate([0.1, 0.1, 0.1, 0.5, 0.5, 0.1, 0.5, 0.1]):
        ed = gu.to_dev(e0)
        with_norm = n % 3 == 2
        efs.ef_hard_threshold(gd, ed, 0.1, lam, idx, val, cnt,
                              err_sq_out=err if with_norm else None,
                              tiles_out=tiles if n % 2 else None)
        c = int(cnt.item())       # synchronises: the next call sees this one's density
        ri, rv, re_ = want[lam]
        what = "call %d lam=%g" % (n, lam)
        gu.assert_bits(idx[:c].cpu().numpy().view(np.uint32), ri, what + " idx")
        gu.assert_bits(val[:c].cpu().numpy(), rv, what + " val")
        gu.assert_bits(ed.cpu().numpy(), re_, what + " e'")
        if n % 2:
            edges = np.arange(efs.tiles_for(d) - 1, dtype=np.int64) * efs.TILE
            ref = np.append(np.searchsorted(ri.astype(np.int64), edges), ri.size)
            gu.assert_bits(tiles.cpu().numpy(), ref.astype(np.int32), what + " tiles")
        if with_norm:             # the same bits whatever ran before
            assert norms.setdefault(lam, err.item()) == err.item(), what
    assert efs.ef_check_status() == efs.EF_OK
