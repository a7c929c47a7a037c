"""Launches of several geometries, around the numbers at which they stop fitting in
shared memory (where the transport takes another form of its kernel), with and
without a phantom: each job against the same job alone in the per-lane kernel
(gpet_options.kernel 1), value for value."""
import copy

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


@pytest.mark.parametrize("phantom", [False, True])
@pytest.mark.parametrize("count", [2, 3, 4, 7, 8, 16, 17])
def test_geometries(G, count, phantom):
    jobs = []
    for i in range(count):
        sc = copy.deepcopy(W.config2_scanner("AB"[i % 2]))
        sc["inner_radius"] = sc["inner_radius"] + i
        with_phantom = phantom and i % 3 == 0
        s = G.Scanner(sc, W.hot_rod_phantom() if with_phantom else None)
        src = W.phantom_source() if with_phantom else W.point_source((1.0, 2.0, float(i)))
        jobs.append(dict(scanner=s, source=src, digitizer=W.digitizer(), n_decays=3000 + 7 * i, seed=60 + i))
    for j, r in zip(jobs, G.simulate_batch(jobs)):
        one = j["scanner"].simulate(j["source"], j["digitizer"], j["n_decays"], j["seed"], kernel=1)
        a, b = ordered(r), ordered(one)
        for k in a:
            assert np.array_equal(a[k], b[k]), k
        for x, y in zip(r.tallies(), one.tallies()):
            assert np.array_equal(x, y)
