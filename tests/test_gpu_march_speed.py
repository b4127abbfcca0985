"""The marched kernels must not fall back to what they replaced: a step within about 1.25 times its measured
time (CUDA events, GB300 at 2070 MHz, calls of many steps), where the tile kernels before them took 1.24 to 3.8 times.
test_gpu_perf_guard.py bounds the same steps by twice the tile kernels' times.
"""
import numpy as np
import pytest

from paper_2007_07760_gb300 import native as N
from paper_2007_07760_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


def event_us(call, stream, steps):
    import torch
    call()
    times = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        call()
        b.record(stream)
        stream.synchronize()
        times.append(a.elapsed_time(b) * 1e3 / steps)
    return min(times)


# us a step: measured, the tile kernel's
@pytest.mark.parametrize("n,kw,measured,tiles", [
    (1024, dict(precision="fp32"), 35.2, 43.9),
    (2048, dict(precision="fp32"), 107.0, 159.0),
    (1024, dict(precision="fp16f"), 38.7, 52.6),
    (1024, dict(precision="fp32", order=2, flux=1), 33.8, 41.9),
    (512, dict(precision="fp32", stages=3, cfl=0.5), 29.1, 42.0),
    (850, dict(precision="fp32", stages=3, cfl=0.3), 64.0, 100.0),
    (548, dict(precision="fp16f", order=2, flux=1), 15.6, 20.0),
    (256, dict(precision="fp64"), 98.0, 143.0),
    (128, dict(precision="fp32", stages=1), 5.0, 14.4),
    (256, dict(precision="fp32", stages=1), 7.2, 14.5),
    (1024, dict(precision="fp32", stages=1), 25.1, 96.3),
    (1024, dict(precision="fp32", stages=1, cfl=1.0), 18.9, 72.8),
])
def test_step_time(n, kw, measured, tiles):
    import torch
    stream = torch.cuda.Stream()
    method = dict(W=4.0, M=0.02, cfl=0.8, order=3, flux=0, stages=2)
    method.update(kw)
    phi0 = WL.drops(n, n, [(0.4 * n, 0.6 * n)], [n / 5], 4.0)
    kind = "deformation" if method["stages"] == 3 else "vortex"
    with N.Solver(n, n, phi0, vel_kind=kind, vel=(float(n), 0.05, 2000.0), stream=stream.cuda_stream, **method) as s:
        us = event_us(lambda: N.dugks_step(s.ctx, 100), stream, 100)
        assert s.status() == 0
    assert us < min(1.25 * measured, 0.97 * tiles), (us, measured, tiles)


def test_batch_step_time():
    """32 grids of 64^2 to 512^2: 60.5 us a step, 84 over tiles."""
    import torch
    stream = torch.cuda.Stream()
    rng = np.random.default_rng(2007077603)
    sides = [int(round(np.exp(v))) for v in rng.uniform(np.log(64), np.log(512), 32)]
    with N.Batch(stream=stream.cuda_stream, precision="fp32", W=4.0, M=0.02, cfl=0.8, order=3, flux=0, stages=2) as b:
        for n in sides:
            b.add(WL.drops(n, n, [(0.4 * n, 0.6 * n)], [n / 5], 4.0), "uniform", (0.03, -0.02))
        us = event_us(lambda: b.step(80), stream, 80)
        assert b.status() == 0
    assert us < 72.0, us
