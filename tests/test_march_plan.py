"""The rule that chooses lane width and segment length of the row march (host code, no GPU): the plan
of many grids from segment counts that are kept while grids come and go is the one that a pass
over all of them for every plan gives."""
import random

import pytest

import march_plans


def lines(precision):
    rng = random.Random(20070777 + precision)
    for kernel in (0, 1):
        for variant in range(6):
            for count in (1, 1, 1, 2, 3, 7, 32, 100):
                lo, hi = rng.choice(((8, 64), (8, 600), (100, 4096), (300, 301)))
                sizes = [rng.randint(lo, hi) for _ in range(2 * count)]
                yield f"{kernel} {precision} {variant} {rng.choice((152, 148, 20))} {count} " + " ".join(map(str, sizes))
    yield f"0 {precision} 4 152 0"


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_counted_segments_give_the_same_plan(precision):
    text = list(lines(precision))
    out = march_plans.run(text)
    assert len(out) == len(text)
    for q, r in zip(text, out):
        assert r[:3] == r[3:], (q, r)
