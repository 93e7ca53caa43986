"""Top-k with more candidates than one CTA holds: the on-chip select of the
grid (a window histogram, then the k-th one's window), and the inputs that make
it hand over to the radix select: a window with too many magnitudes, all of
them in one slice, and a k-th magnitude far above the bound; ties at the
threshold cut in position order. Pairs, residual and norm against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2108_00951_gb300 as efs

pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import gpu_util as gu  # noqa: E402

D = 2_000_003


def _values(kind):
    rng = np.random.default_rng(5)
    x = rng.standard_normal(D).astype(np.float32)
    if kind == "normal":
        return x
    if kind == "ties":        # about 100 equal magnitudes per step of 1/128
        return np.round(x * 128).astype(np.float32) / 128
    if kind == "one_value":   # a tenth of the vector has the threshold's magnitude
        x[rng.random(D) < 0.1] = -1.5
        return x
    if kind == "sorted":      # the threshold's window lies in one or two slices
        return np.sort(np.abs(x))[::-1].copy()
    if kind == "spread":      # magnitudes over 100 binades
        return (x * 2.0 ** rng.uniform(-50, 50, D)).astype(np.float32)
    x[rng.integers(0, D, 300)] = np.nan
    x[rng.integers(0, D, 300)] = -np.inf
    return x


@pytest.mark.usefixtures("stream_kernel")
@pytest.mark.parametrize("kind", ["normal", "ties", "one_value", "sorted", "spread", "special"])
@pytest.mark.parametrize("k", [40_001, 160_000, 500_000])
def test_long_candidate_lists(kind, k):
    e = _values(kind)
    g = np.zeros(D, np.float32)
    gi, gv, ge = gu.topk(g, e, 1.0, k)
    ri, rv, re_ = oracle.ef_topk(g, e, 1.0, k)
    gu.assert_bits(gi, ri, "idx")
    gu.assert_bits(gv, rv, "val")
    gu.assert_bits(ge, re_, "e'")
    assert efs.ef_check_status() == efs.EF_OK


@pytest.mark.parametrize("kind", ["normal", "one_value"])
def test_long_list_error_norm(kind):
    e = _values(kind)
    gd, ed = torch.zeros(D, device=gu.DEV), gu.to_dev(e)
    k = 160_000
    idx = torch.empty(k, dtype=torch.int32, device=gu.DEV)
    val = torch.empty(k, device=gu.DEV)
    cnt = torch.empty(1, dtype=torch.int32, device=gu.DEV)
    err = torch.empty(1, dtype=torch.float64, device=gu.DEV)
    efs.ef_topk(gd, ed, 1.0, k, idx, val, cnt, err_sq_out=err)
    want = float(np.sum(oracle.ef_topk(np.zeros(D, np.float32), e, 1.0, k)[2].astype(np.float64) ** 2))
    assert abs(err.item() - want) <= 1e-6 * want   # the header's bound
