"""The row march at the sizes where its strips and segments end, and the rule that gives some FP64
sizes to the tiles, against the generic kernel in FP64 (which test_gpu_parity.py holds to 1e-12 of the
CPU oracle).

Bounds: FP64 1e-12 of the largest |phi| (a dozen steps of sums of some fifty terms of size one: about
1e-14). FP32 5e-6: phi is of size one and a step adds about ten roundings of 6e-8 to a term of it, so
8e-6 would need every one of a dozen steps to round the same way. FP16 storage 2e-5: the values kept in
16 bits are deviations below 0.05 with weights up to 1/9, rounded to 2^-11, and a step takes
differences of them. Mass: 1e-13 (FP64) and 1e-6 of its value.
"""
import numpy as np
import pytest

from paper_2007_07760_gb300 import native as N
from paper_2007_07760_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 5e-6, "fp16f": 2e-5}
MASS = {"fp64": 1e-13, "fp32": 1e-6, "fp16f": 1e-6}


def velocity(kind, nx, ny):
    if kind == "field":
        X, Y = WL.centres(nx, ny)
        return dict(vel_kind="field", u=0.03 * np.sin(2 * np.pi * Y / ny), v=0.02 * np.cos(2 * np.pi * X / nx))
    par = {"uniform": (0.03, -0.02), "rotation": (nx / 2, ny / 2, 0.1 / max(nx, ny)),
           "vortex": (float(max(nx, ny)), 0.05, 20.0), "deformation": (float(max(nx, ny)), 0.05, 20.0)}[kind]
    return dict(vel_kind=kind, vel=par)


def solve(nx, ny, precision, variant, steps, kind="uniform", order=3, flux=0, stages=2, cfl=0.8):
    phi0 = WL.drops(nx, ny, [(0.4 * nx, 0.6 * ny), (0.02 * nx, 0.1 * ny)], [min(nx, ny) / 5, min(nx, ny) / 6], 4.0)
    with N.Solver(nx, ny, phi0, W=4.0, M=0.02, cfl=cfl, order=order, flux=flux, stages=stages, precision=precision,
                  **velocity(kind, nx, ny)) as s:
        if variant is not None:
            s.set_variant(variant)
        s.step(steps)
        assert s.status() == 0
        return s.phi(), s.mass()


def check(nx, ny, precision, variant=None, steps=12, **kw):
    ref, mref = solve(nx, ny, "fp64", -1, steps, **kw)
    phi, mass = solve(nx, ny, precision, variant, steps, **kw)
    assert np.abs(phi - ref).max() < TOL[precision] * np.abs(ref).max(), (nx, ny, precision, variant, kw)
    assert abs(mass - mref) < MASS[precision] * abs(mref)


# single columns: strips of 28 (FP64 also 26); pairs come with grids wider than a wave of single columns
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16f"])
@pytest.mark.parametrize("nx", [8, 26, 27, 28, 29, 53, 56, 57, 85])
def test_strip_edges(precision, nx):
    order, flux = (3, 0) if nx % 2 else (2, 1)
    check(nx, 21, precision, order=order, flux=flux, kind="rotation" if nx % 3 else "field")


@pytest.mark.parametrize("precision", ["fp32", "fp16f"])
@pytest.mark.parametrize("ny,flux,kind", [(64, 0, "vortex"), (64, 1, "uniform"), (128, 0, "field"), (128, 1, "field")])
@pytest.mark.parametrize("nx", [6418, 6419, 6420, 6421])
def test_pair_strip_edges(precision, nx, ny, flux, kind):
    """107 strips of 60 columns, 8-row segments: one wave (64 rows) and more than one (128)."""
    check(nx, ny, precision, variant=1, steps=6, flux=flux, kind=kind)


@pytest.mark.parametrize("variant", range(6))
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16f"])
def test_segment_edges(precision, variant):
    for ny in (8, 9, 17, 33, 65):
        check(30, ny, precision, variant=variant, kind="vortex")


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny", [(8, 8), (28, 9), (29, 66), (57, 33)])
def test_three_stage(precision, nx, ny):
    for order, flux in ((3, 0), (2, 1)):
        check(nx, ny, precision, order=order, flux=flux, stages=3, cfl=0.3, kind="deformation")


@pytest.mark.parametrize("nx", [6419, 6420])
def test_three_stage_pairs(nx):
    check(nx, 72, "fp32", steps=4, stages=3, cfl=0.3)


@pytest.mark.parametrize("order,flux", [(2, 0), (3, 1), (3, 0)])
@pytest.mark.parametrize("nx,ny", [(192, 192), (198, 198), (240, 240), (249, 211), (768, 64), (360, 360), (380, 380)])
def test_fp64_tiles_and_march(nx, ny, order, flux):
    """FP64 sizes on both sides of the line between the march and the tiles, and a change of path
    between the steps of one state."""
    check(nx, ny, "fp64", order=order, flux=flux, kind="rotation")
    ref, _ = solve(nx, ny, "fp64", -1, 9, order=order, flux=flux)
    phi0 = WL.drops(nx, ny, [(0.4 * nx, 0.6 * ny), (0.02 * nx, 0.1 * ny)], [min(nx, ny) / 5, min(nx, ny) / 6], 4.0)
    with N.Solver(nx, ny, phi0, W=4.0, M=0.02, cfl=0.8, order=order, flux=flux, precision="fp64",
                  **velocity("uniform", nx, ny)) as s:
        for variant in (2, 0, 2):
            s.set_variant(variant)
            s.step(3)
        assert np.abs(s.phi() - ref).max() < 1e-12 * np.abs(ref).max()
