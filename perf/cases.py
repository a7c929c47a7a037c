"""Performance cases: what users of this library have it do, through its public entry points.

Sizes come from the workloads, the tests and the benchmark: runs of 1e3 to 1e7 decays of one scanner (rings of one, two
and four layers, offset layers, posed heads; point and activity-map sources; crystal-, module- and panel-level readout),
launches of many designs and positions, the sensitivity map, a burst of served requests, and the time sort on its own.
Results are taken as a program takes them that keeps buffers from run to run, with room for one single and 0.3
coincidences per decay and zeros behind the last one: on the device, from the device pointers of the result's arrays, or
in page-locked host memory, by library copies of a result's or of the whole launch's arrays.  64-bit unsigned arrays are shown as int64
(time stamps and history ids below 2^63).
"""
import ctypes
import math

import numpy as np
import torch

import paper_2603_07327_gb300 as G
import workloads as W

SINGLES = (G.SINGLES_T_PS, G.SINGLES_H, G.SINGLES_UNIT, G.SINGLES_PANEL, G.SINGLES_E, G.SINGLES_E_RAW, G.SINGLES_DOI)
COINCIDENCES = (G.COINC_A, G.COINC_B)
TALLIES = (G.TALLY_COUNT, G.TALLY_EFX)
NAMES = {G.SINGLES_T_PS: "t_ps", G.SINGLES_H: "h", G.SINGLES_UNIT: "unit", G.SINGLES_PANEL: "panel", G.SINGLES_E: "e",
         G.SINGLES_E_RAW: "e_raw", G.SINGLES_DOI: "doi", G.COINC_A: "coinc_a", G.COINC_B: "coinc_b",
         G.TALLY_COUNT: "tally_count", G.TALLY_EFX: "tally_efx"}
DTYPES = {G.SINGLES_T_PS: "<i8", G.SINGLES_H: "<i8", G.SINGLES_E: "<f4", G.SINGLES_E_RAW: "<f4", G.SINGLES_DOI: "<f4",
          G.TALLY_COUNT: "<i8", G.TALLY_EFX: "<i8"}          # the rest are int32
COUNTS = ("n_decays", "hits", "singles", "coincidences", "n_crystals", "det_steps", "flights", "compton_trials",
          "entered", "phantom_steps", "screened_flights", "singles_formed")

# per decay, about: singles kept, and operations (integer and floating-point) of the events that a pair goes through,
# as the method needs them: one 10-round Philox block is ~100, a decay ~250, a flight ~250, a Woodcock step ~250, a
# Compton interaction ~500 and a single's blur ~200.
PER_DECAY = {"ring8": (0.03, 500), "ring12_a": (0.18, 1600), "ring12_b": (0.17, 1500), "ring12_offset": (0.17, 2600),
             "four_layer": (0.17, 1100), "box": (0.05, 1000), "h2r_1cl": (0.6, 2700), "h2r_split": (0.6, 2800),
             "h2r_2cl": (0.6, 2800), "designs": (0.2, 1600)}


def listed():
    return [
        # the smallest ordinary call: the tiny ring's quick look, results on the host; launches and latency are all there is
        dict(name="tiny_ring", kind="plain", scanner="ring8", n=20_000, activity=1.7e4, readout=3, host=True),
        # one position of a sensitivity sweep at a pilot's statistics, off the centre, an odd count
        dict(name="sweep_position", kind="plain", scanner="ring12_b", n=1_000_003, activity=1.7e4, readout=3, x=3.0, z=-30.0),
        # one position of the axial sweep at its full statistics, the paper's NEMA source
        dict(name="nema_position", kind="plain", scanner="ring12_a", n=10_000_000, activity=1.7e4, readout=3, z=4.0),
        # the hot-rod water phantom in the offset dual-layer ring: activity-map source and phantom scatter
        dict(name="hot_rods", kind="plain", scanner="ring12_offset", n=5_000_000, activity=1.7e4, readout=3, phantom=1.0),
        # a design that is no ring: four posed heads
        dict(name="posed_heads", kind="plain", scanner="box", n=2_000_000, activity=1.7e4, readout=3, x=1.0, z=-2.0),
        # a long ring with module-level readout and depth blur, source off the axis
        dict(name="module_readout", kind="plain", scanner="h2r_split", n=3_000_000, activity=1.7e4, readout=1, x=20.0,
             z=10.0, doi=2.0),
        # a stack of four layers at a few hundred thousand decays, panel-level readout
        dict(name="four_layer_panel", kind="plain", scanner="four_layer", n=300_000, activity=1.7e4, readout=0, y=2.0),
        # a batch kept and replayed: three source positions for each of two geometries
        dict(name="sweep_graph", kind="graph", n=10_000_000, positions=3, seed0=2),
        # a design study in one launch: random designs of 1e4 to 1e6 decays, results copied to the host
        dict(name="design_study", kind="designs", designs=24, scale=0.1, seed0=4),
        # the sensitivity study: two designs, profile positions, four energy windows, and their percent difference
        dict(name="sensitivity_map", kind="map", positions=16, n=200_000),
        # a burst of requests to a running server, point sources and phantoms mixed
        dict(name="served_burst", kind="served", requests=6, lo=1e5, hi=3e6, seed0=5),
        # the digitizer's time sort alone, for a program that owns its device memory
        dict(name="time_sort", kind="sort", n=300_007, span=1 << 46),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("plain", "plain", "plain", "plain", "graph", "designs", "map", "served", "sort"))
    if kind == "plain":
        scanner = rng.choice(("ring8", "ring12_a", "ring12_b", "ring12_offset", "four_layer", "box", "h2r_1cl",
                              "h2r_split", "h2r_2cl"))
        case = dict(kind=kind, scanner=scanner, n=log_int(1_000, 10_000_000), activity=rng.choice((1.7e4, 1e5)),
                    readout=rng.choice((3, 3, 1, 0)), x=round(rng.uniform(-12.0, 12.0), 2),
                    y=round(rng.uniform(-12.0, 12.0), 2), z=round(rng.uniform(-30.0, 30.0), 2),
                    doi=rng.choice((0.0, 0.0, 2.0)), host=rng.random() < 0.3)
        if scanner == "ring12_offset" and rng.random() < 0.6:
            case.update(n=log_int(1_000, 5_000_000), phantom=round(rng.uniform(0.5, 1.0), 2))
        return case
    if kind == "graph":
        return dict(kind=kind, n=log_int(20_000, 10_000_000), positions=rng.randint(1, 3), seed0=rng.randint(2, 900))
    if kind == "designs":
        return dict(kind=kind, designs=rng.randint(2, 48), scale=round(math.exp(rng.uniform(math.log(0.004), math.log(0.1))), 4),
                    seed0=rng.randint(2, 900))
    if kind == "map":
        return dict(kind=kind, positions=rng.randint(1, 24), n=log_int(2_000, 200_000))
    if kind == "served":
        return dict(kind=kind, requests=rng.randint(1, 6), lo=1e4, hi=float(log_int(1e5, 3e6)), seed0=rng.randint(2, 900))
    return dict(kind=kind, n=log_int(100, 1 << 20), span=1 << rng.randint(30, 60))


def _scanner(name, readout=3):
    if name == "box":
        return W.box_scanner(readout)
    if name == "four_layer":
        return W.four_layer_scanner(readout)
    sc = {"ring8": W.config1_scanner, "ring12_a": lambda: W.config2_scanner("A"), "ring12_b": lambda: W.config2_scanner("B"),
          "ring12_offset": W.config3_scanner, "h2r_1cl": lambda: W.h2rspet("1CL"), "h2r_split": lambda: W.h2rspet("split"),
          "h2r_2cl": lambda: W.h2rspet("2CL")}[name]()
    sc["readout_level"] = readout
    return sc


def _torch_dtype(which):
    return {"<i8": torch.int64, "<f4": torch.float32}.get(DTYPES.get(which), torch.int32)


def _room(n, crystals, host):
    """A program's own result buffers for runs of n decays."""
    sizes = {w: n + 1024 for w in SINGLES}
    sizes.update({w: int(0.3 * n) + 1024 for w in COINCIDENCES})
    sizes.update({w: crystals for w in TALLIES})
    return {w: torch.zeros(m, dtype=_torch_dtype(w), pin_memory=host, device="cpu" if host else "cuda")
            for w, m in sizes.items()}


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 26])
    key = int(rng.integers(1, 1 << 40))
    if kind == "plain":
        phantom = W.hot_rod_phantom(scale=case["phantom"]) if case.get("phantom") else None
        pos = (case.get("x", 0.0), case.get("y", 0.0), case.get("z", 0.0))
        source = W.phantom_source(case["activity"]) if phantom else W.point_source(pos, case["activity"])
        scanner = G.Scanner(_scanner(case["scanner"], case["readout"]), phantom)
        host = bool(case.get("host"))
        return dict(kind=kind, scanner=scanner, source=source, digitizer=W.digitizer(doi_fwhm_mm=case.get("doi", 0.0)),
                    n=case["n"], seed=key, host=host, room=_room(case["n"], scanner.n_crystals, host),
                    stream=torch.cuda.Stream() if host else None)
    if kind == "graph":
        scanners = [G.Scanner(_scanner("ring12_a")), G.Scanner(_scanner("ring12_b"))]
        zs = [float(z) for z in np.linspace(-30, 30, case["positions"] + 2)[1:-1]]
        jobs = [dict(scanner=sc, source=W.point_source((0.0, 0.0, z)), digitizer=W.digitizer(), n_decays=case["n"],
                     seed=key + case["seed0"] + i) for i, sc in enumerate(scanners) for z in zs]
        return dict(kind=kind, batch=G.Batch(jobs), room=[_room(case["n"], j["scanner"].n_crystals, False) for j in jobs])
    if kind == "designs":
        made = W.config4(n_designs=case["designs"], seed=case["seed0"], scale=case["scale"])
        jobs = [dict(scanner=G.Scanner(d["scanner"]), source=d["source"], digitizer=d["digitizer"], n_decays=d["n_decays"],
                     seed=key + i) for i, d in enumerate(made)]
        room = _room(sum(j["n_decays"] for j in jobs), sum(j["scanner"].n_crystals for j in jobs), True)
        return dict(kind=kind, jobs=jobs, room=room, stream=torch.cuda.Stream())
    if kind == "map":
        grid = W.sensitivity_positions()
        pick = np.linspace(0, len(grid) - 1, case["positions"]).astype(int)
        return dict(kind=kind, scanners=[G.Scanner(W.h2rspet("1CL")), G.Scanner(W.h2rspet("2CL"))],
                    positions=np.array(grid)[pick], digitizer=W.sensitivity_digitizer(), n=case["n"], seed=key)
    if kind == "served":
        design = np.random.default_rng(case["seed0"])
        sizes = np.exp(np.linspace(math.log(case["lo"]), math.log(case["hi"]), case["requests"])).astype(int)
        requests = []
        for i, n in enumerate(design.permutation(sizes)):
            desc, source, _ = W.random_design(design)
            phantom = None
            if i % 2:
                phantom, source = W.hot_rod_phantom(scale=float(design.uniform(0.5, 1.0))), W.phantom_source()
            requests.append((G.Scanner(desc, phantom), source, W.digitizer(), int(n), key + i))
        return dict(kind=kind, server=G.Server(hbm_budget_bytes=40 * 10**9), requests=requests,
                    room=[_room(r[3], r[0].n_crystals, True) for r in requests])
    keys = rng.integers(0, case["span"], size=case["n"], dtype=np.int64)
    keys = torch.from_numpy(keys).cuda()
    return dict(kind="sort", keys=keys, out=torch.empty_like(keys),
                perm=torch.empty(case["n"], dtype=torch.int32, device="cuda"))


class _DeviceArray:
    """A result array on the device, which keeps its result alive."""

    def __init__(self, result, which, n):
        self.result = result
        self.__cuda_array_interface__ = dict(shape=(n,), typestr=DTYPES.get(which, "<i4"), version=3, strides=None,
                                             data=(result.device_ptr(which), False))


def _keep(result, room):
    """Copy a result's arrays into the program's own device buffers."""
    c = result.counts()
    for w, buf in room.items():
        n = c["singles"] if w in SINGLES else c["coincidences"] if w in COINCIDENCES else c["n_crystals"]
        if n:
            buf[:n].copy_(torch.as_tensor(_DeviceArray(result, w, n), device="cuda"))
    return {NAMES[w]: buf for w, buf in room.items()}, c


def _to_host(result, room, stream):
    """Copy every array of a result's launch into the program's page-locked buffers."""
    for w, buf in room.items():
        result.copy_run_into_async(w, buf.data_ptr(), buf.numel() * buf.element_size(), stream.cuda_stream)
    stream.synchronize()
    return {NAMES[w]: buf for w, buf in room.items()}


def run(state):
    kind = state["kind"]
    if kind == "plain":
        result = state["scanner"].simulate(state["source"], state["digitizer"], state["n"], state["seed"])
        if state["host"]:
            out, c = _to_host(result, state["room"], state["stream"]), result.counts()
        else:
            out, c = _keep(result, state["room"])
        out["counts"] = np.array([c[k] for k in COUNTS], dtype=np.int64)
        return out
    if kind == "graph":
        state["batch"].run()
        total = state["batch"].counts()
        jobs = []
        for j, room in enumerate(state["room"]):
            out, _ = _keep(state["batch"].result(j), room)
            del out["panel"]                      # at most 64 outputs; the unit tells the panel
            jobs.append(out)
        return dict(jobs=jobs, counts=np.array([total[k] for k in COUNTS], dtype=np.int64))
    if kind == "designs":
        results = G.simulate_batch(state["jobs"])
        out = _to_host(results[0], state["room"], state["stream"])
        counts = [r.counts() for r in results]
        out["counts"] = np.array([[c[k] for k in ("hits", "singles", "coincidences", "n_crystals")] for c in counts], dtype=np.int64)
        return out
    if kind == "map":
        counts, sens, total = G.sensitivity_map(state["scanners"], state["positions"], state["digitizer"],
                                                W.SENS_WINDOWS_KEV, state["n"], state["seed"])
        return dict(counts=counts.view(np.int64), sens=sens, delta=np.nan_to_num(G.delta_sym(sens[0], sens[1])),
                    total=np.array([total[k] for k in COUNTS], dtype=np.int64))
    if kind == "served":
        server = state["server"]
        ids = [server.submit(*r) for r in state["requests"]]
        outs = []
        for i, room in zip(ids, state["room"]):
            result = server.wait(i)
            for w, buf in room.items():
                result.copy_into(w, buf.data_ptr(), buf.numel() * buf.element_size())
            # at most 64 outputs; the unit tells the panel
            outs.append({NAMES[w]: buf for w, buf in room.items() if w != G.SINGLES_PANEL})
        return outs
    keys, out, perm = state["keys"], state["out"], state["perm"]
    code = G.load().gpet_sort_times_noalloc(ctypes.c_void_p(keys.data_ptr()), keys.numel(), ctypes.c_void_p(out.data_ptr()),
                                            ctypes.c_void_p(perm.data_ptr()),
                                            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    if code != 0:
        raise RuntimeError(G.load().gpet_last_error().decode())
    return dict(t=out, perm=perm)


def exact(case, seed):
    """The sort has an exact answer.  A simulation has none that lines up value by value: a 64-bit run of the same
    histories takes another branch in about one of 1e5 of them, and every array that follows is then of another length."""
    if case["kind"] != "sort":
        return None
    keys = np.random.default_rng([int(seed) & 0x7FFFFFFF, 26])
    keys.integers(1, 1 << 40)
    t = keys.integers(0, case["span"], size=case["n"], dtype=np.int64)
    perm = np.argsort(t, kind="stable")
    return dict(t=t[perm], perm=perm.astype(np.int32))


def work(case):
    """Decays times what one decay needs: its kept singles written once in time order (44 bytes each), its share of the
    coincidences (8 bytes each) and of the tallies, and its operations."""
    kind = case["kind"]
    if kind == "sort":
        return dict(bytes=20 * case["n"], flops=0)
    crystals = 40_000
    if kind == "plain":
        n, (singles, ops) = case["n"], PER_DECAY[case["scanner"]]
    elif kind == "graph":
        n, (singles, ops) = 2 * case["positions"] * case["n"], PER_DECAY["ring12_a"]
    elif kind == "designs":
        n, (singles, ops) = int(case["designs"] * case["scale"] * 2.1e6), PER_DECAY["designs"]
    elif kind == "map":
        n, (singles, ops) = 2 * case["positions"] * case["n"], PER_DECAY["h2r_1cl"]
        return dict(bytes=2 * case["positions"] * 4 * 16, flops=n * ops)
    else:
        n = int(sum(np.exp(np.linspace(math.log(case["lo"]), math.log(case["hi"]), case["requests"]))))
        singles, ops = PER_DECAY["designs"]
    return dict(bytes=int(n * singles * 44 + n * singles * 0.1 * 8 + 16 * crystals), flops=n * ops)
