"""A hard-threshold call of the claimed-group kernel captured into a CUDA graph shares no hand-out counter
with the calls around it: calls before and after a capture that is never
replayed, and one replay between calls, each against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2108_00951_gb300 as efs

pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import gpu_util as gu  # noqa: E402


@pytest.fixture(params=[2, 3])
def group_kernel(request):
    efs.ef_test_set_stream_kernel(request.param)
    yield
    efs.ef_test_set_stream_kernel(0)


@pytest.mark.usefixtures("group_kernel")
@pytest.mark.parametrize("captures", [1, 2])
def test_calls_around_a_captured_one(captures):
    d = 40 * 4096 + 9
    rng = np.random.default_rng(6)
    g = (rng.standard_normal(d) * 1e-2).astype(np.float32)
    e = (rng.standard_normal(d) * 1e-3).astype(np.float32)
    want = oracle.ef_hard_threshold(g, e, 0.1, 1e-3)
    gd, e0 = gu.to_dev(g), gu.to_dev(e)
    ed = e0.clone()
    idx = torch.empty(d, dtype=torch.int32, device=gu.DEV)
    val = torch.empty(d, device=gu.DEV)
    cnt = torch.empty(1, dtype=torch.int32, device=gu.DEV)
    side = torch.cuda.Stream()

    def call():
        efs.ef_hard_threshold(gd, ed, 0.1, 1e-3, idx, val, cnt)

    def check(step, what):
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            ed.copy_(e0)
            cnt.fill_(-1)
            step()
        side.synchronize()
        c = int(cnt.item())
        gu.assert_bits(idx[:c].cpu().numpy().view(np.uint32), want[0], what + " idx")
        gu.assert_bits(val[:c].cpu().numpy(), want[1], what + " val")
        gu.assert_bits(ed.cpu().numpy(), want[2], what + " e'")
        assert efs.ef_check_status(side) == efs.EF_OK

    check(call, "before")
    graphs = []
    for _ in range(captures):
        graphs.append(torch.cuda.CUDAGraph())
        with torch.cuda.graph(graphs[-1], stream=side, capture_error_mode="thread_local"):
            call()
    for n in range(3):
        check(call, "call %d after the capture" % n)
    for n, graph in enumerate(graphs):
        check(graph.replay, "replay %d" % n)
        check(call, "call after replay %d" % n)
        check(call, "second call after replay %d" % n)
