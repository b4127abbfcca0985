"""Kernels that take two columns a lane, where the sizes of the other tests get one: the DVM in FP32, the
three-stage step over several waves, and the promise that a grid's result in a batch does not
depend on its company, which may turn the plan from single columns to pairs.

Bounds against FP64: FP32 5e-6, as in test_gpu_march.py (phi of size one, about ten roundings of 6e-8 a step
and a dozen steps).
"""
import numpy as np
import pytest

from march_plans import plan
from paper_2007_07760_gb300 import native as N
from paper_2007_07760_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


def field(nx, ny):
    return WL.drops(nx, ny, [(0.4 * nx, 0.6 * ny), (0.02 * nx, 0.1 * ny)], [min(nx, ny) / 5, min(nx, ny) / 6], 4.0)


def velocity(kind, nx, ny):
    if kind == "field":
        X, Y = WL.centres(nx, ny)
        return dict(vel_kind="field", u=0.03 * np.sin(2 * np.pi * Y / ny), v=0.02 * np.cos(2 * np.pi * X / nx))
    par = {"uniform": (0.03, -0.02), "rotation": (nx / 2, ny / 2, 0.1 / max(nx, ny)),
           "vortex": (float(max(nx, ny)), 0.05, 20.0), "deformation": (float(max(nx, ny)), 0.05, 20.0)}[kind]
    return dict(vel_kind=kind, vel=par)


def solve(nx, ny, precision, kind, steps, variant=None, calls=1, **kw):
    with N.Solver(nx, ny, field(nx, ny), W=4.0, M=0.02, precision=precision, **velocity(kind, nx, ny), **kw) as s:
        if variant is not None:
            s.set_variant(variant)
        for _ in range(calls):
            s.step(steps // calls)
        assert s.status() == 0
        return s.phi(), s.mass()


def agree(nx, ny, kind, steps, ref_variant=None, **kw):
    ref, mref = solve(nx, ny, "fp64", kind, steps, variant=ref_variant, **kw)
    phi, mass = solve(nx, ny, "fp32", kind, steps, **kw)
    assert np.abs(phi - ref).max() < 5e-6 * np.abs(ref).max(), (nx, ny, kind, kw)
    assert abs(mass - mref) < 1e-6 * abs(mref)


# (the FP64 DVM, single columns, is held to the oracle by test_gpu_dvm.py)
@pytest.mark.parametrize("cfl,order", [(1.0, 2), (0.8, 3), (0.8, 2), (0.3, 3), (0.3, 2)])
@pytest.mark.parametrize("nx,ny", [(5991, 40), (5992, 40), (5993, 48), (5994, 41)])
def test_dvm_pairs(nx, ny, cfl, order):
    """Strips of 56 columns from one before the grid: 107 of them, and one column, none or two in the last."""
    assert plan("fp32", [(nx, ny)], stages=1, cfl=cfl)[0] == 2
    for kind in ("field", "vortex") if nx % 2 else ("rotation", "deformation"):
        agree(nx, ny, kind, 8, cfl=cfl, order=order, stages=1)
        agree(nx, ny, kind, 4, cfl=cfl, order=order, stages=1, calls=4)   # every step with its mass partials


@pytest.mark.parametrize("cfl", [1.0, 0.8, 0.3])
@pytest.mark.parametrize("nx", [25, 26, 27, 52, 53])
def test_dvm_single_columns_at_strip_edges(oracle, nx, cfl):
    assert plan("fp32", [(nx, 19)], stages=1, cfl=cfl)[0] == 1
    p = oracle.Params(nx, 19, W=4.0, M=0.02, cfl=cfl, order=3, stages=1, vel_kind="uniform", vel=(0.03, -0.02))
    ref = oracle.State(p, field(nx, 19)).run(12)
    for precision, tol in (("fp64", 1e-12), ("fp32", 5e-6)):
        phi, mass = solve(nx, 19, precision, "uniform", 12, cfl=cfl, order=3, stages=1)
        assert np.abs(phi - ref.phi()).max() < tol * np.abs(ref.phi()).max()


@pytest.mark.parametrize("kind,flux,order", [("vortex", 0, 3), ("field", 0, 2), ("field", 1, 2), ("rotation", 1, 3)])
@pytest.mark.parametrize("nx,ny", [(6419, 512), (6420, 512), (6421, 72)])
def test_three_stage_pairs(nx, ny, kind, flux, order):
    """Several waves, and one."""
    assert plan("fp32", [(nx, ny)], stages=3, flux=flux, variant=2)[0] == 2
    agree(nx, ny, kind, 3, ref_variant=-1, cfl=0.3, order=order, flux=flux, stages=3)


COMPANY = (1024, 1024)


@pytest.mark.parametrize("precision", ["fp32", "fp16f"])
@pytest.mark.parametrize("order,flux", [(3, 0), (2, 1), (3, 1)])
def test_result_does_not_depend_on_the_lane_width(precision, order, flux):
    """Small grids alone, and beside a large one that comes after three steps and leaves after ten."""
    shapes, kinds = [(64, 64), (45, 27), (131, 90)], ["vortex", "uniform", "rotation"]
    assert plan(precision, shapes, flux=flux)[0] == 1 and plan(precision, shapes + [COMPANY], flux=flux)[0] == 2
    common = dict(W=4.0, M=0.02, cfl=0.8, order=order, flux=flux, stages=2, precision=precision)
    vel = [velocity(k, nx, ny)["vel"] for (nx, ny), k in zip(shapes, kinds)]
    alone = []
    for (nx, ny), k, v in zip(shapes, kinds, vel):
        with N.Batch(**common) as b:
            g = b.add(field(nx, ny), k, v)
            b.step(17)
            alone.append((b.phi(g), b.mass(g)))
    with N.Batch(**common) as b:
        ids = [b.add(field(nx, ny), k, v) for (nx, ny), k, v in zip(shapes, kinds, vel)]
        b.step(3)
        big = b.add(field(*COMPANY), "vortex", (1024.0, 0.05, 20.0))
        b.step(7)
        b.remove(big)
        b.step(7)
        assert b.status() == 0
        for g, (phi, mass) in zip(ids, alone):
            assert np.array_equal(b.phi(g), phi) and b.mass(g) == mass
