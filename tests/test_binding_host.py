"""Host-side behaviour of the Python binding (no GPU): it imports where torch
has no CUDA, and refuses an argument that is no number as a TypeError."""
import os
import subprocess
import sys

import pytest
import torch

import paper_2108_00951_gb300 as efs
from paper_2108_00951_gb300 import _binding

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_imports_on_a_torch_without_cuda():
    # such a build defines none of torch._C's CUDA functions
    script = ("import torch\n"
              "for name in [n for n in dir(torch._C) if n.startswith('_cuda_')]:\n"
              "    delattr(torch._C, name)\n"
              "import paper_2108_00951_gb300 as efs\n"
              "from paper_2108_00951_gb300 import ef_sgd, workloads\n"
              "assert efs.tiles_for(1) == 2\n"
              "try:\n"
              "    efs.ef_hard_threshold(torch.zeros(4), torch.zeros(4), 0.1, 0.1, None, None, None)\n"
              "except TypeError as err:\n"
              "    assert 'CUDA tensor' in str(err)\n"
              "    print('refused')\n")
    r = subprocess.run([sys.executable, "-c", script], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and "refused" in r.stdout, r.stdout + r.stderr


@pytest.fixture
def no_pointers(monkeypatch):
    """Arguments reach ctypes with fake addresses; every call below fails in
    their conversion, so none reaches the library."""
    monkeypatch.setattr(_binding, "_dev", lambda *a: 0x10000000)
    monkeypatch.setattr(_binding, "_stream", lambda s: 0)


@pytest.mark.usefixtures("no_pointers")
@pytest.mark.parametrize("bad", ["0.1", None, [0.1], 1j])
def test_scalars_that_are_no_numbers_are_type_errors(bad):
    x = torch.zeros(8)
    i = torch.zeros(8, dtype=torch.int32)
    lists = ([i], [x], i)
    calls = [lambda: efs.ef_hard_threshold(x, x, bad, 0.1, i, x, i),
             lambda: efs.ef_hard_threshold(x, x, 0.1, bad, i, x, i),
             lambda: efs.ef_topk(x, x, bad, 2, i, x, i),
             lambda: efs.ef_topk_layerwise(x, x, bad, [8], [2], i, x, i),
             lambda: efs.ef_scaled_round(x, x, bad, 4, i, i),
             lambda: efs.sparse_aggregate_apply(*lists, 8, bad, x),
             lambda: efs.sparse_aggregate_apply(*lists, 8, 0.5, x, m=x, momentum=bad),
             lambda: efs.sparse_aggregate_apply(*lists, 8, 0.5, x, m=x, lr=bad)]
    for call in calls:
        with pytest.raises(TypeError):
            call()
