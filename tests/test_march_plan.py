"""The rule that chooses lane width and segment length of the row march (host code, no GPU): the plan
of many grids from segment counts that are kept while grids come and go is the one that a pass
over all of them for every plan gives."""
import os
import random
import subprocess

import pytest

from paper_2007_07760_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="session")
def plan_main(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("plan") / "march_plan")
    flags = [f for f in _build._flags() if f != "-O3"]
    subprocess.run([_build.NVCC, "-O1"] + flags + [os.path.join(HERE, "march_plan_main.cu"), "-o", exe], check=True)
    return exe


def lines(precision):
    rng = random.Random(20070777 + precision)
    for variant in range(6):
        for count in (1, 1, 1, 2, 3, 7, 32, 100):
            lo, hi = rng.choice(((8, 64), (8, 600), (100, 4096), (300, 301)))
            sizes = [rng.randint(lo, hi) for _ in range(2 * count)]
            yield f"{precision} {variant} {rng.choice((152, 148, 20))} {count} " + " ".join(map(str, sizes))
    yield f"{precision} 4 152 0"


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_counted_segments_give_the_same_plan(plan_main, precision):
    text = list(lines(precision))
    out = subprocess.run([plan_main], input="\n".join(text), capture_output=True, text=True, check=True).stdout.splitlines()
    assert len(out) == len(text)
    for q, r in zip(text, out):
        v = r.split()
        assert v[:3] == v[3:], (q, r)
