"""Obstacle cells among the initial classes are a solid like the cells of a fixed
body: the liquid and interface cells next to them are stepped the same, bit for
bit, in every storage, alone, in a batch, and with bodies elsewhere in the tank."""
import dataclasses

import numpy as np
import pytest

from paper_1201_0351_gb300 import inputs as I

pytestmark = pytest.mark.gpu

OBSTACLE = 8  # cell class


def _tank(periodic=0, wall_vel=None):
    """a tank with a surface and a seeded flow, and a box through the surface"""
    nx, ny, nz = 30, 22, 20
    flags, fill, rho = I.hydrostatic_tank(nx, ny, nz, lambda X, Y: 11.4, 1e-5, 1.0, periodic)
    vel = 0.01 * np.random.default_rng(7).standard_normal((nx * ny * nz, 3))
    vel[flags == I.GAS] = 0.0
    box = I.Box(center=(20.0, 11.0, 10.0), half=(4.0, 3.0, 3.5), mode=I.MODE_FIXED)
    return I.Scenario("tank", nx, ny, nz, periodic, 0.7, (0.0, 0.0, -1e-5), (0.0, 0.0, 0.0), 1.0, 1e-2, flags, fill,
                      rho, [box], 0, vel.reshape(-1), wall_vel=wall_vel)


def _solid_in_flags(sc):
    """the scenario with its last body's cells as obstacles of the initial classes"""
    b = sc.boxes[-1]
    z, y, x = np.meshgrid(np.arange(sc.nz) + 0.5, np.arange(sc.ny) + 0.5, np.arange(sc.nx) + 0.5, indexing="ij")
    ins = np.logical_and.reduce([np.abs(c - o) < h for c, o, h in zip((x, y, z), b.center, b.half)]).reshape(-1)
    return dataclasses.replace(sc, flags=np.where(ins, OBSTACLE, sc.flags).astype(np.uint8), boxes=list(sc.boxes[:-1]))


def _same(a, b):
    for key in ("flags", "f", "fill", "mass"):
        assert np.array_equal(a[0][key], b[0][key]), key
    assert a[1]["status"] == b[1]["status"] == 0
    assert a[1]["n_general"] == b[1]["n_general"] > 100


def _run(sc, storage, steps, use_graphs=True):
    from paper_1201_0351_gb300 import lbm_fs

    sim = lbm_fs.Simulation(sc, storage=storage, use_graphs=use_graphs)
    sim.step(steps)
    out = sim.fields(want_f=True), sim.stats()
    sim.close()
    return out


@pytest.mark.parametrize("storage", ["f64", "f32", "f16s"])
@pytest.mark.parametrize("periodic,wall", [(0, None), (1, None), (0, tuple(0.002 * k for k in range(18)))])
def test_obstacle_cells_equal_a_fixed_body(storage, periodic, wall):
    sc = _tank(periodic, wall)
    want = _run(sc, storage, 30)
    _same(_run(_solid_in_flags(sc), storage, 30), want)
    _same(_run(_solid_in_flags(sc), storage, 30, use_graphs=False), want)


@pytest.mark.parametrize("storage", ["f64", "f32", "f16s"])
def test_obstacle_cells_beside_other_bodies(storage):
    """two fixed bodies; the obstacle cells lie outside their ranges"""
    sc = _tank()
    other = [I.Box(center=(6.0, y, 9.0), half=(2.0, 2.0, 2.0), mode=I.MODE_FIXED) for y in (5.5, 15.5)]
    sc = sc.with_boxes(other + sc.boxes)
    _same(_run(_solid_in_flags(sc), storage, 30), _run(sc, storage, 30))


@pytest.mark.parametrize("storage", ["f64", "f32", "f16s"])
def test_obstacle_cells_in_a_batch(storage):
    from paper_1201_0351_gb300 import lbm_fs

    sc = _tank()
    bt = lbm_fs.Batch([_solid_in_flags(sc), sc], storage=storage)
    bt.step(30)
    res = [(t.fields(want_f=True), t.stats()) for t in bt.tanks]
    bt.close()
    want = _run(sc, storage, 30)
    for r in res:
        _same(r, want)
