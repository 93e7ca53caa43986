"""Host-side behaviour of the Python binding (no GPU): it imports where torch
has no CUDA."""
import os
import subprocess
import sys

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
