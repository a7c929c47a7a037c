"""Coincidences where clusters of singles run over many tiles of the sorter's one
pass, up to all singles of the run in one cluster or one window: the pairs of the
oracle's sorter, and a digitizer time that grows with the number of singles and
not with its square."""
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


def check(oracle, r, window_ns):
    s = r.singles()
    a, b = r.coincidences()
    st = np.zeros(len(s["h"]), [("t_ps", np.uint64), ("unit", np.int32), ("panel", np.int32), ("h", np.uint64)])
    for k in st.dtype.names:
        st[k] = s[k]
    _, oa, ob = oracle.coincidences(st, window_ns)
    lo, hi = np.minimum(oa, ob), np.maximum(oa, ob)
    o = np.argsort(lo)   # (the sorter may take singles of one time in another order)
    assert np.array_equal(a, lo[o]) and np.array_equal(b, hi[o])


# Mean gap of the singles 21 ns (activity 1e8): windows of half a gap to all of the run
@pytest.mark.parametrize("window_ns", [10.0, 20.0, 50.0, 100.0, 300.0, 5e3, 2.2e4, 1e6, 1e9])
@pytest.mark.parametrize("n", [2_000, 4_500, 700_001])
def test_pairs(G, oracle, n, window_ns):
    sc = G.Scanner(W.config2_scanner("A"))
    dg = W.digitizer(e_lo=50.0, window_ns=window_ns)
    check(oracle, sc.simulate(W.point_source((0.0, 0.0, 1.0), activity_bq=1e8), dg, n, 4), window_ns)
    sc.close()


def test_jobs_of_one_launch(G, oracle):
    """A job's cluster ends with the job, wherever in a tile that is."""
    sc = G.Scanner(W.config2_scanner("A"))
    dg = W.digitizer(e_lo=50.0, window_ns=1e9)
    jobs = [dict(scanner=sc, source=W.point_source((0.0, 0.0, float(j)), activity_bq=1e8), digitizer=dg, n_decays=n, seed=j)
            for j, n in enumerate([1, 30, 5_000, 200_000, 7, 40_000])]
    for r in G.simulate_batch(jobs):
        check(oracle, r, 1e9)
    sc.close()


def test_work_grows_with_the_singles(G):
    """Four times the singles, all in one cluster: a walk over them takes four times as long, and twice that is
    allowed for.  (With each tile walking from the cluster's start: 294 ms and 2.9 s, ten times as long.)"""
    sc = G.Scanner(W.config2_scanner("A"))
    dg = W.digitizer(e_lo=50.0, window_ns=1e9)
    ms = {}
    for n in (1_500_000, 6_000_000):
        for _ in range(2):   # (the first run's time includes the kernels' loading)
            r = sc.simulate(W.point_source((0.0, 0.0, 1.0), activity_bq=1e8), dg, n, 4)
            ms[n] = r.counts()["digitizer_ms"]
            r.free()
    assert ms[6_000_000] < 8.0 * ms[1_500_000], ms
    sc.close()
