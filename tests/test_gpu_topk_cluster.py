"""Top-k of vectors that one thread-block cluster holds (up to 65,536
coordinates), in one launch: sizes around the slices and the rule's end, ragged
and misaligned, k from 0 to d, ties across slices cut in index order, zeros,
NaN and infinities, bf16 gradients and the norm, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2108_00951_gb300 as efs

pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import gpu_util as gu  # noqa: E402

MAX = 65_536


def _check(g, e, gamma, k, what, off=(0, 0)):
    gi, gv, ge = gu.topk(g, e, gamma, k, g_off=off[0], e_off=off[1])
    ri, rv, re_ = oracle.ef_topk(g, e, gamma, k)
    gu.assert_bits(gi, ri, what + " idx")
    gu.assert_bits(gv, rv, what + " val")
    gu.assert_bits(ge, re_, what + " e'")


@pytest.mark.parametrize("off", [(0, 0), (1, 3)])
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("d", [1, 2, 7, 31, 33, 4097, 30_001, MAX - 1, MAX, MAX + 1])
def test_sizes(d, bf16, off):
    rng = np.random.default_rng(d)
    g = (rng.standard_normal(d) * 1e-2).astype(np.float32)
    e = (rng.standard_normal(d) * 1e-3).astype(np.float32)
    if bf16:
        g = (g.view(np.uint32) >> 16).astype(np.uint16)
    for k in sorted({0, 1, max(1, d // 100), d // 2, d}):
        _check(g, e, 0.1, k, "d=%d k=%d" % (d, k), off)
    assert efs.ef_check_status() == efs.EF_OK


@pytest.mark.parametrize("kind", ["zeros", "one_value", "few_values", "special"])
def test_ties_and_special_values(kind):
    d = 60_001
    rng = np.random.default_rng(2)
    e = rng.standard_normal(d).astype(np.float32)
    if kind == "zeros":
        e[rng.random(d) < 0.95] = 0.0
        e[5::11] = -0.0
    elif kind == "one_value":
        e[:] = -0.25
    elif kind == "few_values":
        e = np.array([0.0, 0.5, -0.5, 1.0, -1.0], np.float32)[rng.integers(0, 5, d)]
    else:
        e[rng.integers(0, d, 50)] = np.nan
        e[rng.integers(0, d, 50)] = np.inf
        e[rng.integers(0, d, 50)] = 1e-42
    g = np.zeros(d, np.float32)
    for k in (1, 40, 777, 20_000, 45_000, d - 1):
        _check(g, e, 1.0, k, "%s k=%d" % (kind, k))
    assert efs.ef_check_status() == efs.EF_OK


@pytest.mark.parametrize("d,k", [(500, 1), (20_000, 1000), (MAX, 30_000), (3, 0)])
def test_norm(d, k):
    rng = np.random.default_rng(d)
    g, e = rng.standard_normal(d).astype(np.float32), rng.standard_normal(d).astype(np.float32)
    got = []
    for _ in range(2):
        gd, ed = gu.to_dev(g), gu.to_dev(e)
        idx = torch.empty(max(k, 1), dtype=torch.int32, device=gu.DEV)
        val = torch.empty(max(k, 1), device=gu.DEV)
        cnt = torch.empty(1, dtype=torch.int32, device=gu.DEV)
        err = torch.empty(1, dtype=torch.float64, device=gu.DEV)
        efs.ef_topk(gd, ed, 0.1, k, idx, val, cnt, err_sq_out=err)
        got.append(err.item())
    want = float(np.sum(oracle.ef_topk(g, e, 0.1, k)[2].astype(np.float64) ** 2))
    assert got[0] == got[1]                       # reproducible to the bit
    assert abs(got[0] - want) <= 1e-6 * want      # the header's bound


def test_between_calls_of_the_other_path():
    # the streaming calls keep per-call state blocks; a short call between
    # them leaves it alone
    rng = np.random.default_rng(8)
    for d in (MAX + 5, 1000, MAX + 5, MAX, 50_000, 2 * MAX + 1, 9):
        g, e = (rng.standard_normal(d).astype(np.float32) for _ in range(2))
        _check(g, e, 0.1, max(1, d // 50), "in a row d=%d" % d)
    assert efs.ef_check_status() == efs.EF_OK
