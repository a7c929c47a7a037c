"""Designs whose histories ask for more singles entries than a lane class of the
slot-pool kernel has (tests/test_slot_pool_on_cpu.py shows on the CPU that such
launches end, and that their classes run out): whatever a history finds, its
singles and tallies are those of the per-lane kernel, in a plain run, in a batch
and in a live launch."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# Compton and photoelectric coefficient (1/cm), depth, pitch, half-length (mm), cutoff (keV), pairs
DESIGNS = {"long_lyso": (0.5742, 0.2958, 20.0, 1.0, 150.0, 10.0, 1_000_003),
           "scatterer": (0.8, 0.07, 20.0, 1.0, 150.0, 10.0, 1_000_003),
           "compton_only": (1.5, 0.0, 25.0, 0.5, 150.0, 80.0, 300_007)}
COUNTS = ("hits", "singles", "coincidences", "det_steps", "flights", "compton_trials", "entered", "singles_formed")


@pytest.fixture(scope="module")
def G():
    from paper_2603_07327_gb300 import build as B
    B.build()
    import paper_2603_07327_gb300 as G
    G.load()
    return G


def job(G, design, readout=W.READOUT_CRYSTAL):
    compton, photo, depth, pitch, half_v, e_cut, n = DESIGNS[design]
    sc = W.scanner(12, 55.0, [W.layer(int(29.0 / pitch), int(2 * half_v / pitch), pitch, 0.0, depth)],
                   readout_level=readout)
    sc["materials"] = [W.AIR, dict(name="crystal", mu_total_511_cm=compton + photo,
                                   photo_frac_511=photo / (compton + photo), electron_density_cm3=0.0)]
    return dict(scanner=G.Scanner(sc), source=W.point_source((0.0, 0.0, 3.0)),
                digitizer=W.digitizer(e_lo=20.0, e_cut=e_cut), n_decays=n, seed=7)


def plain(j, kernel, seed=None):
    return j["scanner"].simulate(j["source"], j["digitizer"], j["n_decays"], seed or j["seed"], kernel=kernel)


def same(a, b, counts=COUNTS):
    ca, cb = a.counts(), b.counts()
    assert {k: ca[k] for k in counts} == {k: cb[k] for k in counts}
    sa, sb = a.singles(), b.singles()
    oa, ob = np.lexsort((sa["unit"], sa["h"])), np.lexsort((sb["unit"], sb["h"]))
    for k in sa:
        assert np.array_equal(sa[k][oa], sb[k][ob]), k
    for x, y in zip(a.tallies(), b.tallies()):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("readout", [W.READOUT_CRYSTAL, W.READOUT_MODULE])
@pytest.mark.parametrize("design", DESIGNS)
def test_plain_run(G, design, readout):
    j = job(G, design, readout)
    same(plain(j, 3), plain(j, 1))


def test_live_launch(G):
    jobs = [job(G, d) for d in DESIGNS]
    server = G.Server(hbm_budget_bytes=40 * 10**9)
    ids = [server.submit(j["scanner"], j["source"], j["digitizer"], j["n_decays"], j["seed"]) for j in jobs]
    for i, j in zip(ids, jobs):
        same(server.wait(i), plain(j, 1), ("hits", "singles", "coincidences"))
    server.close()


@pytest.mark.parametrize("n", range(3_420_000, 3_560_000, 20_000))
def test_batch_replays(G, n):
    """Which histories overflow depends on the schedule: sizes whose overflow list of one history in 16
    is just large enough, or just too small, for one run are replayed without an error all the same."""
    j = dict(job(G, "scatterer"), n_decays=n, digitizer=W.digitizer())
    b = G.Batch([j])
    first = b.result(0)
    c, t, ptr = first.counts(), first.tallies(), first.device_ptr(G.SINGLES_H)
    for _ in range(12):
        b.run()
    r = b.result(0)
    assert {k: r.counts()[k] for k in COUNTS} == {k: c[k] for k in COUNTS}
    assert all(np.array_equal(x, y) for x, y in zip(r.tallies(), t))
    # a view made before the replays shows them
    assert first.device_ptr(G.SINGLES_H) == ptr
    s, u = first.singles(), r.singles()
    assert all(np.array_equal(np.sort(s[k]), np.sort(u[k])) for k in s)
    b.close()
