"""The rounding step without an error norm runs in blocks of 2048 coordinates,
and the integer exchange in one thread per 4: sizes around both, arrays at odd
alignments, coordinates kept back at block edges, and calls of different sizes
in a row (the last CTA of each leaves the counters at zero)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2108_00951_gb300 as efs

pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import gpu_util as gu  # noqa: E402

SIZES = [1, 5, 2047, 2048, 2049, 3 * 2048, 100_003, 2048]


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("off", [0, 1, 2])
def test_blocks(off, bf16):
    for d in SIZES:
        rng = np.random.default_rng(d)
        g = rng.standard_normal(d).astype(np.float32)
        e = (rng.standard_normal(d) * 0.01).astype(np.float32)
        e[::2047] = 1e30          # does not fit an int32: kept back
        e[d // 2] = np.nan
        if bf16:
            g = (g.view(np.uint32) >> 16).astype(np.uint16)
        gd, ed = gu.g_device(g, off), gu.to_dev(e, off)
        q = torch.full((d + off,), 7, dtype=torch.int32, device=gu.DEV)[off:]
        unsent = torch.full((1,), -1, dtype=torch.int32, device=gu.DEV)
        efs.ef_scaled_round(gd, ed, 0.5, 12, q, unsent)
        rq, re_, ru = oracle.ef_scaled_round(g, e, 0.5, 12)
        what = "d=%d off=%d" % (d, off)
        gu.assert_bits(q.cpu().numpy().view(np.uint32), rq.view(np.uint32), what + " q")
        gu.assert_bits(ed.cpu().numpy(), re_, what + " e'")
        assert int(unsent.item()) == ru, what
        dense = torch.full((d + off,), float("nan"), device=gu.DEV)[off:]
        efs.int_aggregate([q, q, q], d, 12, dense)
        gu.assert_bits(dense.cpu().numpy(), oracle.int_aggregate([rq] * 3, d, 12), what + " sum")
    assert efs.ef_check_status() == efs.EF_OK
