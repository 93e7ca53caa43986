"""g and e at every element alignment: rows of an [n, d] matrix with an odd d,
or slices of flat buffers, stream through shifted tiles (stream_in.cuh). Every
residue of both bases modulo 16 bytes, with vectors that end before, at and
just after a tile boundary of the shifted positions, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2108_00951_gb300 as efs

pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import gpu_util as gu  # noqa: E402

SIZES = [1, 6, 9, 4096 - 3, 2 * 4096 + 1, 3 * 4096 - 2]


def _inputs(d, seed, bf16):
    rng = np.random.default_rng(seed)
    g = (rng.standard_normal(d) * 1e-2).astype(np.float32)
    e = (rng.standard_normal(d) * 1e-3).astype(np.float32)
    return ((g.view(np.uint32) >> 16).astype(np.uint16) if bf16 else g), e


def _same(got, want, what):
    for name, a, b in zip(("idx", "val", "e'"), got, want):
        gu.assert_bits(a, b, what + " " + name)


@pytest.mark.usefixtures("stream_kernel")
@pytest.mark.parametrize("e_off", [0, 1, 2, 3])
@pytest.mark.parametrize("g_off,bf16", [(o, False) for o in range(4)] +
                         [(o, True) for o in range(8)])
def test_every_alignment(g_off, bf16, e_off):
    for d in SIZES:
        g, e = _inputs(d, 1000 * g_off + e_off, bf16)
        what = "d=%d g+%d e+%d" % (d, g_off, e_off)
        _same(gu.ht(g, e, 0.1, 1.5e-3, g_off=g_off, e_off=e_off),
              oracle.ef_hard_threshold(g, e, 0.1, 1.5e-3), "ht " + what)
        k = max(1, d // 50)
        _same(gu.topk(g, e, 0.1, k, g_off=g_off, e_off=e_off), oracle.ef_topk(g, e, 0.1, k),
              "topk " + what)
    assert efs.ef_check_status() == efs.EF_OK


@pytest.mark.usefixtures("stream_kernel")
@pytest.mark.parametrize("g_off,e_off,bf16", [(1, 1, False), (2, 3, False), (5, 1, True),
                                              (7, 3, True), (3, 2, True)])
def test_layerwise_alignment(g_off, e_off, bf16):
    # segments that begin and end around the boundaries of shifted tiles, with
    # empty ones, ones of a few coordinates, and sampled ones (over 4096)
    sizes = [4096 - e_off, 0, 2, 5, 9000, 4096, 1, 3, 8192 + 7, 20_000, 4]
    ks = [40, 0, 1, 5, 90, 30, 1, 0, 81, 0, 2]
    g, e = _inputs(sum(sizes), 7, bf16)
    ends = np.cumsum(sizes)
    _same(gu.topk_layerwise(g, e, 0.1, ends, ks, g_off=g_off, e_off=e_off),
          oracle.ef_topk_layerwise(g, e, 0.1, ends, ks), "layerwise g+%d e+%d" % (g_off, e_off))
    assert efs.ef_check_status() == efs.EF_OK


@pytest.mark.parametrize("bf16", [False, True])
def test_rows_of_a_matrix(bf16):
    # the neighbouring rows keep every bit: no access past a row's coordinates writes
    n, d = 5, 3 * 4096 + 3
    g, e = _inputs(n * d, 3, bf16)
    gd, ed = gu.g_device(g).view(n, d), gu.to_dev(e).view(n, d)
    idx = torch.empty(d, dtype=torch.int32, device=gu.DEV)
    val = torch.empty(d, device=gu.DEV)
    cnt = torch.empty(1, dtype=torch.int32, device=gu.DEV)
    want = e.copy().reshape(n, d)
    for row in (1, 3, 4):
        ri, rv, want[row] = oracle.ef_hard_threshold(g.reshape(n, d)[row], want[row], 0.1, 1e-3)
        efs.ef_hard_threshold(gd[row], ed[row], 0.1, 1e-3, idx, val, cnt)
        c = int(cnt.item())
        gu.assert_bits(idx[:c].cpu().numpy().view(np.uint32), ri, "row %d idx" % row)
        gu.assert_bits(val[:c].cpu().numpy(), rv, "row %d val" % row)
        gu.assert_bits(ed.cpu().numpy(), want, "after row %d" % row)
