"""Dealing out of histories: jobs of every size around a warp and a chunk in one
launch (a warp's refill then crosses chunks and jobs), and launches around the
sizes at which the chunk rule changes, against each job alone in the per-lane
kernel (gpet_options.kernel 1)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2603_07327_gb300 import build as B
    B.build()
    import paper_2603_07327_gb300 as G
    G.load()
    return G


def ordered(r):
    s = r.singles()
    o = np.lexsort((s["unit"], s["h"]))
    return {k: s[k][o] for k in s}


@pytest.mark.parametrize("sizes", [[1] * 70, [1, 31, 32, 33, 2, 255, 256, 257, 5], [7, 300_001, 3, 65, 1]],
                         ids=["ones", "edges", "uneven"])
@pytest.mark.parametrize("phantom", [False, True])
def test_jobs(G, sizes, phantom):
    sc = G.Scanner(W.config2_scanner("B"), W.hot_rod_phantom() if phantom else None)
    src = W.phantom_source() if phantom else W.point_source((1.0, 2.0, 3.0))
    jobs = [dict(scanner=sc, source=src, digitizer=W.digitizer(), n_decays=n, seed=40 + i) for i, n in enumerate(sizes)]
    for j, r in zip(jobs, G.simulate_batch(jobs)):
        one = sc.simulate(src, j["digitizer"], j["n_decays"], j["seed"], kernel=1)
        a, b = ordered(r), ordered(one)
        for k in a:
            assert np.array_equal(a[k], b[k]), (j["n_decays"], k)
        for k in ("hits", "singles", "coincidences"):
            assert r.counts()[k] == one.counts()[k]


@pytest.mark.parametrize("n", [2 * 4256 * 32 - 1, 2 * 4256 * 64 + 1, 2 * 4256 * 256 - 31, 8 * 4256 * 288 + 5])
def test_launch_sizes(G, n):
    """One job around the sizes at which a chunk grows, 4256 warps (2 CTAs of 14 warps on 152 multiprocessors)."""
    sc = G.Scanner(W.config1_scanner())
    a, b = (sc.simulate(W.point_source((0, 0, 0)), W.digitizer(), n, 9, kernel=k) for k in (3, 1))
    for k in ("hits", "singles", "coincidences", "det_steps", "flights"):
        assert a.counts()[k] == b.counts()[k]
    for x, y in zip(a.tallies(), b.tallies()):
        assert np.array_equal(x, y)
