"""The digitizer's time sort by buckets and its one-pass coincidence sorting.

The bucket sort serves runs whose decay times spread over buckets of at least
10 ns; the radix passes serve the rest.  Both are checked against numpy's order
of the same singles, and the coincidences against the oracle's sorter on them,
over activities that cross from one sort to the other and fill clusters across
many tiles, around the tile sizes, for a history range of a longer run, and for
jobs of very different sizes in one launch."""
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


def check(G, oracle, r, window_ns):
    s = r.singles()
    t = s["t_ps"].astype(np.int64)
    assert np.all(np.diff(t) >= 0)
    # one single per (history, unit); a history's singles of one time stamp keep their list's order
    assert len(np.unique(np.stack([s["h"].astype(np.int64), s["unit"].astype(np.int64)]), axis=1).T) == len(t)
    a, b = r.coincidences()
    assert np.array_equal(b, a + 1) and np.all(np.diff(a) > 0)
    st = np.zeros(len(t), [("t_ps", np.uint64), ("unit", np.int32), ("panel", np.int32), ("h", np.uint64)])
    for k in st.dtype.names:
        st[k] = s[k]
    _, oa, ob = oracle.coincidences(st, window_ns)
    o = np.argsort(np.minimum(oa, ob))   # (the sorter may take singles of one time in another order)
    assert np.array_equal(a, np.minimum(oa, ob)[o]) and np.array_equal(b, np.maximum(oa, ob)[o])
    return s


@pytest.mark.parametrize("activity", [1.7e4, 1e8, 3e9, 1e11, 1e13])
@pytest.mark.parametrize("n", [1, 40, 5_000, 300_001])
def test_activities(G, oracle, n, activity):
    """Same singles at every activity; the spans reach from 1 ps to 18 s."""
    sc = G.Scanner(W.config2_scanner("A"))
    dg = W.digitizer(e_lo=50.0)
    r = sc.simulate(W.point_source((0.0, 0.0, 1.0), activity_bq=activity), dg, n, 9)
    s = check(G, oracle, r, dg["window_ns"])
    ref = sc.simulate(W.point_source((0.0, 0.0, 1.0)), dg, n, 9).singles()
    for x, y in ((s, ref), (ref, s)):
        assert len(x["h"]) == len(y["h"])
    o, p = np.lexsort((s["unit"], s["h"])), np.lexsort((ref["unit"], ref["h"]))
    for k in ("h", "unit", "panel", "e", "e_raw", "doi"):
        assert np.array_equal(s[k][o], ref[k][p]), k
    sc.close()


def test_wide_window_clusters(G, oracle):
    """A coincidence window of many mean gaps: clusters run over several tiles."""
    sc = G.Scanner(W.config2_scanner("A"))
    for window_ns in (0.0, 50.0, 2e3, 2e5):
        dg = W.digitizer(e_lo=50.0, window_ns=window_ns)
        r = sc.simulate(W.point_source((0.0, 0.0, 1.0), activity_bq=1e8), dg, 100_000, 4)
        check(G, oracle, r, window_ns)
    sc.close()


def test_history_range_and_uneven_jobs(G, oracle):
    sc = G.Scanner(W.config2_scanner("B"))
    dg = W.digitizer()
    r = sc.simulate(W.point_source(), dg, 10**9, 3, h_begin=10**6, h_end=10**6 + 200_000)
    check(G, oracle, r, dg["window_ns"])
    jobs = [dict(scanner=sc, source=W.point_source((0.0, 0.0, float(j)), activity_bq=a), digitizer=dg, n_decays=n, seed=j)
            for j, (n, a) in enumerate([(1, 1.7e4), (900_000, 1e9), (33, 1e3), (50_000, 1.7e4), (2_000, 1e11)])]
    for job, r in zip(jobs, G.simulate_batch(jobs)):
        s = check(G, oracle, r, dg["window_ns"])
        alone = sc.simulate(job["source"], dg, job["n_decays"], job["seed"])
        for k, v in alone.singles().items():
            assert np.array_equal(np.sort(v), np.sort(s[k])), k
        for x, y in zip(alone.coincidences(), r.coincidences()):
            assert np.array_equal(x, y)
    sc.close()
