"""The split position of the s = 1/2 block path for two-dimensional clusters, ladders and rings with far
neighbours: the smallest K from min(15, N / 2 + 2) to min(15, N - 2) whose slots hold the bonds
(csrc/blk_fit.h), against a count of the slots here."""
import os
import re
import shutil
import subprocess
from collections import Counter

import pytest

from lattices import LATTICES

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0706_3293_gb300", "csrc")
TEXT = open(os.path.join(CSRC, "blk_params.cuh")).read()
SL, SG, SX = (int(re.search(rf"HM_BLK_{k} = (\d+);", TEXT).group(1)) for k in ("SL", "SG", "SX"))


def fits(bonds, cls, K, own):
    low, cross, dist, seen = Counter(), Counter(), set(), Counter()
    for (p, q), c in zip(bonds, cls):
        if q < K:
            low[c, "low" if q < 8 else "second" if p >= 8 else "both"] += 1
            dist.add((c, q - p, 0 if own else seen[p, q, c]))        # a repeated bond takes a group of its own
            seen[p, q, c] += 1
        elif p < K:
            cross[c, p < 8] += 1
    return (K <= 15 and max(low.values(), default=0) <= SL and max(cross.values(), default=0) <= SX
            and max(Counter(d[0] for d in dist).values(), default=0) <= SG)


@pytest.fixture(scope="module")
def chosen(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("fit") / "blk_fit_check")
    subprocess.check_call([gxx, "-O1", "-std=c++17", "-I", CSRC, "-o", exe,
                           os.path.join(ROOT, "tests", "native", "blk_fit_check.cc")])

    def run(bonds, cls, own, k0, kmax):
        text = f"{len(bonds)} {int(own)} {k0} {kmax} {SL} {SX} {SG}\n" + "".join(f"{p} {q} {c}\n" for (p, q), c in zip(bonds, cls))
        return tuple(int(t) for t in subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split())
    return run


@pytest.mark.parametrize("name", LATTICES)
@pytest.mark.parametrize("every_own", [False, True], ids=["classes", "bonds"])
def test_split_of_lattices(chosen, name, every_own):
    (n, bonds, cls), K_classes = LATTICES[name]
    bonds = [(min(b), max(b)) for b in bonds]
    cls = [0] * len(bonds) if every_own else cls
    k0, kmax = min(max(8, min(15, n // 2 + 2)), n - 2), min(15, n - 2)
    want = [K for K in range(k0, kmax + 1) if fits(bonds, cls, K, every_own)]
    assert chosen(bonds, cls, every_own, k0, kmax) == ((want[0], 1) if want else (-1, 0))
    assert every_own or (want[0] if want else None) == K_classes
