"""The chain that a launch is fitted to (fit_launch in csrc/umi_plan.cu), on the host:
legal, within the planner's cap and the device's shared memory, at one position,
at both sides of G steps per resident warp, and for large bands; and a curve of
equal tiles gets at most 6 % more work on its busiest SM than at the rule's chain.
Without a GPU the library plans for a device of one SM."""
import os
import subprocess

import pytest

from paper_2604_06602_gb300 import build as libbuild
from tests.test_planner_host import chain_cap, sm_count

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WINDOWS = [1, 9, 17, 25, 33, 51, 73, 97, 121, 145, 217, 271, 361, 433, 543, 721, 895, 1089, 1441, 1793, 2161, 2521,
           2945, 3585, 4095]


@pytest.fixture(scope="module")
def fit(tmp_path_factory):
    lib = libbuild.build()
    exe = str(tmp_path_factory.mktemp("fit") / "fit")
    subprocess.run([libbuild.nvcc()] + libbuild.ARCH_FLAGS +
                   ["-std=c++17", os.path.join(ROOT, "tests", "launch_fit_driver.cu"), "-o", exe,
                    "-I" + libbuild.CSRC, "-I" + os.path.join(ROOT, "include"), lib,
                    "-Xlinker", "-rpath," + os.path.dirname(lib)], check=True)

    def run(launches):
        text = "".join("%d %d %d\n" % x for x in launches)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
        rows = [tuple(int(v) for v in line.split()) for line in out.splitlines()]
        assert len(rows) == len(launches)
        return rows

    return run


def resident_warps(G, R, minb):
    return 8 * (3 if G == 32 and R <= 12 else minb)      # per SM; pairs of windows run at 24


def sizes(G, R, minb):
    """Positions around G steps per resident warp, small and large."""
    edge = G * (32 // G) * resident_warps(G, R, minb) * sm_count()
    return [1, 31, 500, edge - 1, edge, edge + 1, 2 * edge, 7 * edge + 5, 100 * edge, 18_000_000]


def launches(fit):
    variants = fit([(W, 1, 1) for W in WINDOWS])
    return [(W, n, b) for W, v in zip(WINDOWS, variants) for n in sizes(*v[:3]) for b in (1, 3, 400) if n >= b]


def test_chains_are_legal(fit):
    todo = launches(fit)
    for (W, n, b), (G, R, minb, threads, rule, chain, smem) in zip(todo, fit(todo)):
        what = (W, n, b, G, R, chain)
        assert 1 <= chain <= chain_cap(G), what
        assert G == 32 or chain <= G or (chain % G == 0 and (chain // G) % 2 == 1), what
        assert smem <= 227 * 1024, what


def test_one_curve_keeps_its_busiest_sm_short(fit):
    todo = [x for x in launches(fit) if x[2] == 1]
    # 300,000 and 160,000 samples on 152 SMs, by SM.
    todo += [(W, n * sm_count(), 1) for W in WINDOWS for n in (1974, 1053)]

    def busiest(n, G, R, minb, threads, chain):
        """Steps of the busiest SM; CTAs that do not fill it run at its pace in
        proportion, and a tenth more, or at the full SM's with 8 warps per SM."""
        tiles = -(-n // (32 // G * chain))
        ctas = -(-(-(-tiles // (threads // 32))) // sm_count())
        full, rest = divmod(ctas, 8 * minb * 32 // threads)
        idle = 1.0 if minb == 1 else 0.1
        part = idle + (1 - idle) * rest * threads / 32 / (8 * minb) if rest else 0.0
        return (full + part) * (chain + (0.5 if G <= 2 else 0.75))

    for (W, n, _), (G, R, minb, threads, rule, chain, _) in zip(todo, fit(todo)):
        steps = -(-n // (32 // G * 8 * minb * sm_count()))
        if steps <= G or 2 < G < 32 or (G == 32 and R <= 12):
            continue                                     # one tile per warp; not held against the rule's
        got, ref = (busiest(n, G, R, minb, threads, c) for c in (chain, rule))
        assert got <= ref / 0.94 * 1.0001, (W, n, G, R, chain, rule, got, ref)
