"""Sums of doubles as integers (the step's mass partials): the correctly rounded sum, on the host."""
import math
import os
import random
import subprocess

from paper_2007_07760_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


def sums(lists, folder):
    exe = os.path.join(folder, "sum")
    flags = [f for f in _build._flags() if f != "-O3"]
    subprocess.run([_build.NVCC, "-O1"] + flags + [os.path.join(HERE, "sum_main.cu"), "-o", exe], check=True)
    text = "\n".join(f"{len(v)} " + " ".join(x.hex() for x in v) for v in lists)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    return [(int(a), float.fromhex(b)) for a, b in (q.split() for q in out if q)]


def test_integer_sum_is_correctly_rounded(tmp_path):
    rng = random.Random(2007)
    lists = [[1.0], [0.0], [-0.0, 0.0], [1.0, -1.0], [1.0, 2.0 ** -53], [1.0, 2.0 ** -53, 2.0 ** -100], [-1.0, -2.0 ** -53],
             [2.0 ** 53, 1.0], [2.0 ** 53, 3.0], [1.0] * 2048, [-(2.0 - 2.0 ** -52)] * 2048, [1e300, 1e-300, 5e-324],
             [2.0 - 2.0 ** -52, 2.0 ** -53], [1e-200, 1e-200], [3.5, 2.0 ** -60, -3.5]]
    for n in (1, 2, 7, 100, 1152, 2048):
        for span in (0, 4, 30, 58):
            lists.append([rng.uniform(-1, 1) * 2.0 ** rng.randint(-span, 0) for _ in range(n)])
            lists.append([rng.uniform(0.9, 1.1) * 10.0 ** rng.uniform(0, span / 4) for _ in range(n)])
    for v, (ok, s) in zip(lists, sums(lists, str(tmp_path))):
        if max(map(abs, v)) in (0.0,):
            assert s == 0.0
            continue
        assert ok
        # (nothing lies below 2^-112 of the largest value, but in the list with a subnormal number)
        assert s == math.fsum(v), (v[:4], s, math.fsum(v))


def test_ranges_left_to_floating_point(tmp_path):
    assert [ok for ok, _ in sums([[1e308, 1.0], [1e-300], [float("inf"), 1.0], [float("nan")]], str(tmp_path))] == [0, 0, 0, 0]
