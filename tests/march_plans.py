"""Plans of the row march as the library chooses them, from a host program over its headers (march_plan_main.cu)."""
import functools
import os
import subprocess
import tempfile

from paper_2007_07760_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))
PRECISIONS = {"fp64": 0, "fp32": 1, "fp16f": 2}


@functools.lru_cache(maxsize=1)
def _program():
    folder = tempfile.TemporaryDirectory(prefix="march_plan_")
    exe = os.path.join(folder.name, "march_plan")
    flags = [f for f in _build._flags() if f != "-O3"]
    subprocess.run([_build.NVCC, "-O1"] + flags + [os.path.join(HERE, "march_plan_main.cu"), "-o", exe], check=True)
    return folder, exe


def run(lines):
    """The program's output lines, as lists of integers."""
    out = subprocess.run([_program()[1]], input="\n".join(lines), capture_output=True, text=True, check=True).stdout
    return [[int(v) for v in r.split()] for r in out.splitlines()]


def plan(precision, sizes, stages=2, flux=0, cfl=0.8, variant=4, sms=None):
    """(columns a lane, rows a segment) for grids of these (nx, ny) stepped together on this device."""
    if sms is None:
        import torch
        sms = torch.cuda.get_device_properties(0).multi_processor_count
    flat = " ".join(f"{x} {y}" for x, y in sizes)
    return tuple(run([f"{stages} {flux} {cfl} {PRECISIONS[precision]} {variant} {sms} {len(sizes)} {flat}"])[0][:2])
