"""The slot-pool transport kernel (gpet_options.kernel 3) in each of its forms
against the per-lane kernel (kernel 1), which runs the same events one history
per lane: the same histories, singles, tallies and event counts, value for
value, at sizes around a warp and around the pool, in rings of many shapes (a
photon that leaves through a panel's back ends without a flight there), with
panel poses, with a phantom, and with histories that touch more readout units
than a list or the pool's entries hold."""
import copy

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

COUNTS = ("hits", "singles", "coincidences", "det_steps", "flights", "compton_trials", "entered", "phantom_steps",
          "screened_flights", "singles_formed")


@pytest.fixture(scope="module")
def G():
    from paper_2603_07327_gb300 import build as B
    B.build()
    import paper_2603_07327_gb300 as G
    G.load()
    return G


def same(G, sc, src, dg, n, seed, phantom=None, **opts):
    s = G.Scanner(sc, phantom)
    a = s.simulate(src, dg, n, seed, kernel=3, keep_hits=True, **opts)
    b = s.simulate(src, dg, n, seed, kernel=1, keep_hits=True)
    ca, cb = a.counts(), b.counts()
    assert {k: ca[k] for k in COUNTS} == {k: cb[k] for k in COUNTS}
    ha, hb = a.hits(), b.hits()
    oa, ob = np.lexsort((ha["gstep"], ha["h"])), np.lexsort((hb["gstep"], hb["h"]))
    for k in ha:
        assert np.array_equal(ha[k][oa], hb[k][ob]), k
    sa, sb = a.singles(), b.singles()
    oa, ob = np.lexsort((sa["unit"], sa["h"])), np.lexsort((sb["unit"], sb["h"]))
    for k in sa:
        assert np.array_equal(sa[k][oa], sb[k][ob]), k
    for x, y in zip(a.tallies(), b.tallies()):
        assert np.array_equal(x, y)
    s.close()
    return ca


@pytest.mark.parametrize("block_size", [0, 128, 256, 512])
@pytest.mark.parametrize("n", [1, 31, 33, 1025, 60_001])
def test_sizes_and_shapes(G, n, block_size):
    same(G, W.config2_scanner("B"), W.point_source((2.0, 1.0, 5.0)), W.digitizer(doi_fwhm_mm=2.0), n, 11,
         block_size=block_size)


@pytest.mark.parametrize("block_size", [0, 128, 256, 512])
@pytest.mark.parametrize("case", ["phantom", "posed", "posed_phantom", "pencil"])
def test_forms(G, case, block_size):
    sc = W.box_scanner() if case.startswith("posed") else W.config3_scanner()
    ph = W.hot_rod_phantom() if case.endswith("phantom") else None
    src = W.phantom_source() if ph else W.pencil_source((0.0, 1.0, 0.5), (1.0, 0.2, 0.1)) if case == "pencil" \
        else W.point_source((1.0, -2.0, 0.5))
    same(G, sc, src, W.digitizer(), 40_000, 5, ph, block_size=block_size)


@pytest.mark.parametrize("panels,first_angle,depth", [(1, 0.0, 10.0), (2, 0.4, 10.0), (3, 0.1, 30.0), (4, 5.0, 2.0),
                                                      (5, -1.0, 20.0), (7, 3.0, 12.0), (17, 0.3, 25.0),
                                                      (36, 2.0, 8.0), (64, 0.0, 40.0)])
def test_rings(G, panels, first_angle, depth):
    """Exits through the back are ended without a flight where every other panel
    lies in front: rings of few, deep and many panels, source near a panel."""
    R = 60.0
    width = 0.96 * 2.0 * R * np.tan(np.pi / panels) if panels > 2 else 40.0
    n_u = max(1, int(min(width, 60.0) / 1.5))
    sc = W.scanner(panels, R, [W.layer(n_u, 16, 1.5, 0.1, depth / 2), W.layer(n_u, 16, 1.5, 0.1, depth / 2)],
                   modules_v=3, first_angle=first_angle)
    same(G, sc, W.point_source((0.8 * R, 3.0, 1.0)), W.digitizer(e_lo=100.0), 60_000, 7)


@pytest.mark.parametrize("readout", [W.READOUT_CRYSTAL, W.READOUT_MODULE, W.READOUT_PANEL])
def test_many_units(G, readout):
    """Compton-only crystals of 0.5 mm (cutoff 80 keV): many histories touch more units than a
    list holds, and a lane class's entries run out (both are simulated again)."""
    sc = copy.deepcopy(W.scanner(12, 55.0, [W.layer(50, 60, 0.5, 0.02, 25.0)], modules_v=3, readout_level=readout))
    sc["materials"] = [W.AIR, dict(name="scatterer", mu_total_511_cm=1.5, photo_frac_511=0.0, electron_density_cm3=0.0)]
    c = same(G, sc, W.point_source((0.0, 0.0, 3.0)), W.digitizer(e_lo=20.0, e_cut=80.0), 8_000, 3)
    assert c["hits"] > c["singles_formed"] or readout == W.READOUT_CRYSTAL
