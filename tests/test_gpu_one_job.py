"""A launch of one job (its tables come in the kernel's parameters) against the
same job among others, and against the per-lane kernel (gpet_options.kernel 1),
value for value: each form of the geometry, source and readout, and a kept graph
of one job."""
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


def equal(a, b):
    x, y = ordered(a), ordered(b)
    for k in x:
        assert np.array_equal(x[k], y[k]), k
    for k in ("hits", "singles", "coincidences"):
        assert a.counts()[k] == b.counts()[k]
    for x, y in zip(a.tallies(), b.tallies()):
        assert np.array_equal(x, y)


FORMS = ["ring", "four_layers", "split_module", "panel_readout", "phantom", "posed", "posed_phantom", "pencil"]


def form(name):
    sc = {"four_layers": lambda: W.four_layer_scanner(0), "split_module": lambda: W.h2rspet("split"),
          "posed": W.box_scanner, "posed_phantom": W.box_scanner}.get(name, lambda: W.config2_scanner("B"))()
    sc = copy.deepcopy(sc)
    if name == "split_module":
        sc["readout_level"] = 1
    if name == "panel_readout":
        sc["readout_level"] = 0
    phantom = W.hot_rod_phantom() if name.endswith("phantom") else None
    source = W.phantom_source() if phantom else W.point_source((3.0, 1.0, 5.0))
    if name == "pencil":
        source = W.pencil_source((0.0, 1.0, 0.5), (1.0, 0.2, 0.1))
    return sc, phantom, source


@pytest.mark.parametrize("name", FORMS)
def test_forms(G, name):
    sc, phantom, source = form(name)
    s = G.Scanner(sc, phantom)
    other = G.Scanner(W.config1_scanner())
    dg = W.digitizer(doi_fwhm_mm=2.0)
    n = 20_011
    one = s.simulate(source, dg, n, 5)
    equal(one, s.simulate(source, dg, n, 5, kernel=1))
    jobs = [dict(scanner=other, source=W.point_source((0, 0, 0)), digitizer=dg, n_decays=77, seed=4),
            dict(scanner=s, source=source, digitizer=dg, n_decays=n, seed=5)]
    equal(one, G.simulate_batch(jobs)[1])
    batch = G.Batch(jobs[1:])
    for _ in range(2):
        batch.run()
        equal(one, batch.result(0))
