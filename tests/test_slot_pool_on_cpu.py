"""The slot-pool transport kernel's own source on the CPU, one CTA of it with
every lane a fiber (tests/pool_on_cpu), for designs from a tenth of a hit per
pair to thirty and for schedules in which the events take different times.

A history's singles are entries that the slots of a lane class share.  Whatever
a design asks of them, every launch ends within a bounded number of warp passes,
begins each history once, and gives the same tallies and the same singles under
any schedule; a history that found no entry is listed once for the
re-simulation and has no singles of its own.  A design of ordinary density
leaves fewer histories to the re-simulation than a run's first list holds."""
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_07327_gb300", "csrc")
HERE = os.path.join(ROOT, "tests", "pool_on_cpu")

# Compton and photoelectric coefficient (1/cm), depth, pitch, half-length (mm), cutoff (keV)
DESIGNS = {
    "short_lyso": (0.5742, 0.2958, 2.0, 1.0, 10.0, 10.0),       # 0.1 hits per pair
    "ring": (0.5742, 0.2958, 10.0, 1.0, 40.0, 10.0),            # 1.0
    "long_lyso": (0.5742, 0.2958, 20.0, 1.0, 150.0, 10.0),      # 2.6
    "scatterer": (0.8, 0.07, 20.0, 1.0, 150.0, 10.0),           # 3.8
    "long_scatterer": (0.8, 0.07, 20.0, 0.5, 400.0, 10.0),      # 4.2
    "compton_only": (1.5, 0.0, 25.0, 0.5, 400.0, 80.0),         # 11
    "thick_compton": (1.0, 0.0, 60.0, 0.5, 400.0, 20.0),        # 35
}


@pytest.fixture(scope="module")
def pool(tmp_path_factory):
    """The kernel's source as host code: shared memory is static, PTX one-liners are their values."""
    out = tmp_path_factory.mktemp("pool")
    texts = {}
    for name in ("device.cuh", "transport.cuh", "transport_cta.cu", "internal.h"):
        s = open(os.path.join(CSRC, name)).read()
        s = s.replace("extern __shared__ __align__(16) ", "extern ").replace("__shared__", "static")
        s = s.replace("__grid_constant__", "").replace("#include <cuda_runtime.h>", "").replace('#include "internal.h"', "")
        s = re.sub(r'asm\("mov\.u32 %0, %%lanemask_lt;"[^;]*;', "m = (1u << (threadIdx.x & 31)) - 1u;", s)
        texts[name] = re.sub(r'asm volatile\("mov\.u64 %0, %%globaltimer;"[^;]*;', "t = 0;", s)
    cta, header = texts["transport_cta.cu"], texts.pop("internal.h")
    counters = re.search(r"constexpr int kCtaCounters = .*;", header).group(0)
    kernel, rest = cta.split("// The launch shapes")
    totals = re.search(r"void cta_counters\(.*?\n}\n", rest, flags=re.S).group(0)
    texts["cta_kernel.inc"] = kernel.replace("namespace gpet {", "namespace gpet {\n" + counters, 1) + totals + "}\n"
    for name, s in texts.items():
        (out / name).write_text(s)
    exe = str(out / "pool")
    subprocess.run(["g++", "-std=c++20", "-O2", "-w", "-U_FORTIFY_SOURCE", "-ffp-contract=off", "-I", str(out), "-I", HERE,
                    "-I", "/usr/local/cuda/include", os.path.join(HERE, "pool.cpp"), "-o", exe], check=True)

    def run(shape, n, design, readout, seed, slow):
        # (a pair takes under ten passes per hit, even alone in its events; without progress there is no number)
        text = subprocess.run([exe, str(shape), str(n), *map(str, DESIGNS[design]), str(readout), str(seed), str(slow),
                               "1000"], check=True, capture_output=True, text=True, timeout=120).stdout.split("\n")
        rows = [list(map(int, r.split())) for r in text[:2] if len(r.split()) > 1]
        for end, status, begun, hits, *_ in rows:
            assert end == 0, "no end within the pass limit"
            assert status == 0 and begun == n
        assert len(rows) == 2 and int(text[2]) == 0
        return rows

    return run


@pytest.mark.parametrize("slow", [0.5, 1.0, 2.0])
@pytest.mark.parametrize("design", DESIGNS)
def test_every_launch_ends(pool, design, slow):
    for seed in (1, 3):
        rows = pool(14, 5_000, design, 3, seed, slow)
        # (and the last four of them do ask for more entries than there are)
        assert design not in list(DESIGNS)[3:] or min(r[5] for r in rows) > 0


@pytest.mark.parametrize("readout", [0, 1, 3])
@pytest.mark.parametrize("shape", [4, 8, 16, 114])
def test_shapes(pool, shape, readout):
    for design in ("ring", "scatterer", "compton_only"):
        pool(shape, 2_000, design, readout, 5, 1.0)


@pytest.mark.parametrize("n", [1, 33, 1025])
def test_few_histories(pool, n):
    pool(14, n, "thick_compton", 3, 1, 1.0)


@pytest.mark.parametrize("n", [3_300, 50_000])
def test_ordinary_designs_fit_the_first_overflow_list(pool, n):
    """A run's first list holds one history in 16: a run that fills it is simulated twice."""
    for design in ("ring", "long_lyso"):
        for row in pool(14, n, design, 3, 1, 1.0):
            assert row[5] <= n // 16
