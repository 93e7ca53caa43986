"""How the layer-wise select shares its CTAs (csrc/lw_share.h, compiled for the
host): teams and singles fit the budget, and no CTA is left with the short
tensors of a whole model, on the tensors of every workload and on drawn ones."""
import ctypes
import heapq
import os
import subprocess

import numpy as np
import pytest

from paper_2108_00951_gb300 import build, workloads

SOURCE = r"""
#include "lw_share.h"
extern "C" void share(uint32_t n, const uint64_t* candidates, const uint64_t* cost,
                      const uint32_t* least, uint32_t budget, int from_e, uint32_t* out) {
  std::vector<efs::LwWork> work(n);
  for (uint32_t i = 0; i < n; ++i) work[i] = {candidates[i], cost[i], least[i]};
  std::vector<uint32_t> team;
  efs::lw_share(work, budget, from_e != 0, team);
  std::copy(team.begin(), team.end(), out);
}
"""


@pytest.fixture(scope="module")
def share(tmp_path_factory):
    path = tmp_path_factory.mktemp("share")
    (path / "s.cpp").write_text(SOURCE)
    so = str(path / "s.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC,
                    str(path / "s.cpp"), "-o", so], check=True)
    fn = ctypes.CDLL(so).share

    def call(candidates, cost, least, budget, from_e=False):
        n = len(cost)
        out = (ctypes.c_uint32 * max(n, 1))()
        fn(n, (ctypes.c_uint64 * max(n, 1))(*candidates), (ctypes.c_uint64 * max(n, 1))(*cost),
           (ctypes.c_uint32 * max(n, 1))(*least), budget, int(from_e), out)
        return np.array(out[:n], np.int64)

    return call


def _loads(cost, team, ctas):
    """The loads of the singles' CTAs, dealt longest first to the least loaded."""
    single = sorted((c for c, t in zip(cost, team) if t == 1), reverse=True)
    loads = [0] * max(1, min(len(single), ctas))
    for c in single:
        heapq.heappush(loads, heapq.heappop(loads) + c)
    return loads


def _check(candidates, cost, least, budget, team, what):
    teams = int(team[team > 1].sum())
    assert teams + (1 if (team == 1).any() else 0) <= budget, what
    assert team.size == 0 or team.max() <= 32, what
    if max(least, default=1) > 1:
        return  # teams that lengths ask for come first
    # the singles have CTAs for 2 load positions each, or for the longest of them
    # (or all there are); dealing longest first leaves none with more than the
    # average and one single more. A rank holds at least half of load.
    rank = max((2 * -(-c // int(t)) for c, t in zip(candidates, team) if 1 < t < 32), default=0)
    longest = max((c for c, t in zip(cost, team) if t == 1), default=0)
    assert max(_loads(cost, team, budget - teams)) <= 2 * max(
        2 * rank, longest, 2 * 8192, sum(cost) // budget), what


# (sizes of the tensors): the workloads', and lengths drawn over four decades
MODELS = {w.name: list(w.segments) for w in workloads.WORKLOADS}
for _n, _d in ((60, 100_000_003), (100, 138_000_001), (200, 138_000_001), (200, 30_000_001)):
    _w = 10.0 ** np.random.default_rng(_n).uniform(0.0, 4.0, _n)
    MODELS["%d of %d" % (_n, _d)] = [max(1, int(x)) for x in _w / _w.sum() * _d]


@pytest.mark.parametrize("budget", [152, 16, 1])
@pytest.mark.parametrize("frac", [1e-3, 0.01, 0.03, 0.05, 0.1, 0.3])
@pytest.mark.parametrize("model", sorted(MODELS))
def test_no_cta_queues_the_singles(share, model, frac, budget):
    candidates, cost = [], []
    for ds in MODELS[model]:
        k = max(1, int(frac * ds))
        candidates.append(3 * k // 2 + ds // 512 if ds > 4096 else 0)
        cost.append(3 * k + 4096 if ds > 4096 else ds // 4 + 2048)
    for from_e in (False, True):
        team = share(candidates, cost, [1] * len(cost), budget, from_e)
        _check(candidates, cost, [1] * len(cost), budget, team, (model, frac, from_e))


def test_plenty_of_ctas_gives_ranks_of_8192(share):
    # an embedding of 281 K candidates among short tensors: as many ranks as its
    # load asks for, whatever the others are
    team = share([281_000] + [1000] * 13, [562_000] + [7000] * 13, [1] * 14, 152)
    assert team[0] == 32 and (team[1:] == 1).all()
    team = share([100_000] + [1000] * 13, [200_000] + [7000] * 13, [1] * 14, 152)
    assert team[0] == 13


@pytest.mark.parametrize("budget", [1, 2, 31, 152])
def test_lengths_that_ask_for_more_than_there_is(share, budget):
    rng = np.random.default_rng(budget)
    for n in (0, 1, 2, 9, 300):
        least = rng.integers(1, 257, n).tolist()
        candidates = rng.integers(0, 2_000_000, n).tolist()
        cost = [2 * c + 4096 for c in candidates]
        team = share(candidates, cost, least, budget)
        _check(candidates, cost, least, budget, team, (n, budget))
