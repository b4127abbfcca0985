"""The rule that chooses lane width and segment length of the row march (host code, no GPU): the plan
of many grids from segment counts that are kept while grids come and go is the one that a pass
over all of them for every plan gives."""
import random

import pytest

import march_plans


def lines(precision):
    rng = random.Random(20070777 + precision)
    for kernel in ("2 0 0.8", "2 1 0.8", "3 0 0.3", "3 1 0.3", "1 0 0.3", "1 0 0.8", "1 0 1.0"):
        for variant in range(6):
            for count in (1, 1, 1, 2, 3, 7, 32, 100):
                lo, hi = rng.choice(((8, 64), (8, 600), (100, 4096), (300, 301)))
                sizes = [rng.randint(lo, hi) for _ in range(2 * count)]
                yield f"{kernel} {precision} {variant} {rng.choice((152, 148, 20))} {count} " + " ".join(map(str, sizes))
    yield f"2 0 0.8 {precision} 4 152 0"


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_counted_segments_give_the_same_plan(precision):
    text = list(lines(precision))
    out = march_plans.run(text)
    assert len(out) == len(text)
    for q, r in zip(text, out):
        assert r[:3] == r[3:], (q, r)


@pytest.mark.parametrize("kw,nx,ny,plans", [
    # columns and rows within 5 % of the best measured (us a step in a loop of n, and what the rule had taken there)
    (dict(flux=1), 230, 230, {(1, 2)}),            # 6.3; one row of pairs 7.1
    (dict(flux=1), 548, 548, {(1, 6), (1, 7)}),    # 14.1; five rows of pairs 15.4
    (dict(stages=3, cfl=0.3), 548, 548, {(1, 6), (1, 7)}),            # 34.5; five rows of pairs 37.0
    (dict(stages=3, flux=1, cfl=0.3), 230, 230, {(1, 2)}),            # 13.9; one row of pairs 17.1
    (dict(stages=1), 128, 128, {(1, 1)}),          # 4.9; two rows, the next kernel early, 6.5
    (dict(stages=1), 256, 256, {(1, 2), (1, 3)}),  # 7.2; one row 8.6
    (dict(stages=1, cfl=1.0), 312, 312, {(1, 2), (2, 1), (2, 2)}),    # 5.7; two rows, the next kernel early, 7.3
    (dict(), 1024, 1024, {(2, 16)}),               # as before
])
def test_plans_measured_best(kw, nx, ny, plans):
    got = march_plans.plan("fp32", [(nx, ny)], sms=152, **kw)
    assert got in plans


def test_autotuned_variants_differ():
    """No two variants that the autotuner times are the same plan at every size."""
    from paper_2007_07760_gb300 import autotune
    sizes = [(64, 64), (256, 256), (700, 700), (2048, 2048)]
    seen = {}
    for v in autotune.VARIANTS:
        key = tuple(march_plans.plan("fp32", [s], variant=v, sms=152) for s in sizes)
        assert key not in seen, (v, seen[key])
        seen[key] = v
