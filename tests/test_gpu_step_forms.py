"""The forms a step can take by size, storage and parameters, at their edges.

Bit for bit: the bulk kernel of each storage (z-planes per block by grid size;
the FP16 ring of linear tiles, with rows shorter and longer than its patching
round and grids thinner than a tile) against the software-pipelined kernel, and
the cooperative-grid tail of a large tank against the batch's separate kernels.
Against the oracle (the FP64 parity bounds): the collision with and without an
acceleration across the gravity axis, and moving walls on thin grids."""
import dataclasses

import numpy as np
import pytest

from paper_1201_0351_gb300 import inputs as I

from parity import assert_f64_parity, run_both

pytestmark = pytest.mark.gpu


def _flow(nx, ny, nz, periodic, accel=(0.0, 0.0, 0.0), seed=3, eta=None):
    """A tank with a flat surface (none where eta is the height) and a seeded
    velocity field."""
    eta = max(1.0, 0.6 * nz) + 0.4 if eta is None else eta
    flags, fill, rho = I.hydrostatic_tank(nx, ny, nz, lambda X, Y: eta, 1e-5, 1.0, periodic)
    rng = np.random.default_rng(seed)
    vel = 0.01 * rng.standard_normal((nx * ny * nz, 3))
    vel[flags == I.GAS] = 0.0
    return I.Scenario("flow_%dx%dx%d" % (nx, ny, nz), nx, ny, nz, periodic, 0.7, (0.0, 0.0, -1e-5), accel, 1.0, 1e-2,
                      flags, fill, rho, [], 0, vel.reshape(-1))


def _run(sc, storage, steps):
    from paper_1201_0351_gb300 import lbm_fs

    sim = lbm_fs.Simulation(sc, storage=storage)
    sim.step(steps)
    g = sim.fields(want_f=True)
    sim.close()
    return g


@pytest.mark.parametrize("storage,dims,periodic", [
    ("f16s", (47, 9, 11), 0), ("f16s", (46, 9, 8), 0), ("f16s", (3, 7, 40), 0), ("f16s", (2, 6, 30), 3),
    ("f16s", (1, 5, 6), 0), ("f16s", (513, 3, 4), 0), ("f16s", (33, 17, 13), 1), ("f16s", (32, 16, 14), 2),
    ("f16s", (21, 19, 12), 7), ("f16s", (700, 1, 3), 0), ("f16s", (24, 22, 1), 0),
    ("f32", (45, 13, 9), 0), ("f32", (128, 128, 32), 0), ("f32", (512, 512, 24), 0)])
def test_bulk_forms_match_the_pipelined_kernel(storage, dims, periodic, monkeypatch):
    """all liquid in a closed or periodic box where it is one cell high"""
    sc = _flow(*dims, periodic, eta=float(dims[2]) if dims[2] == 1 or periodic & 4 else None)
    out = []
    for v in ("pipe", "plain"):
        monkeypatch.setenv("LBMFS_BULK", v)
        out.append(_run(sc, storage, 3))
    assert np.array_equal(out[0]["flags"], out[1]["flags"])
    assert np.array_equal(out[0]["f"], out[1]["f"])


@pytest.mark.parametrize("accel", [(0.0, 0.0, 0.0), (2e-5, -1e-5, 0.0)])
def test_double_collision_with_and_without_cross_acceleration(accel):
    g, o, gb, ob, gs, _ = run_both(_flow(13, 11, 12, 1, accel), 40)
    assert_f64_parity(g, o, gb, ob)


@pytest.mark.parametrize("dims", [(9, 5, 4), (7, 1, 9), (1, 6, 5)])
def test_moving_walls_on_thin_grids(dims):
    sc = dataclasses.replace(_flow(*dims, 0), wall_vel=tuple(0.003 * k for k in range(18)))
    g, o, gb, ob, gs, _ = run_both(sc, 30)
    assert_f64_parity(g, o, gb, ob)


@pytest.mark.parametrize("storage,steps", [("f64", 25), ("f16s", 25), ("f32", 90)])
def test_large_tank_tail_equals_the_batch(storage, steps):
    """400x340 cells per plane (above the cluster's limit): conversions, and
    cells covered and (in the longer run) uncovered by moving boxes, the same in
    the batch's kernels"""
    from paper_1201_0351_gb300 import lbm_fs

    sc = I.random_box_scene(400, 340, 18, seed=5, nboxes=2, speed=0.02)
    sim = lbm_fs.Simulation(sc, storage=storage)
    sim.step(steps)
    a, s = sim.fields(want_f=True), sim.stats()
    sim.close()
    bt = lbm_fs.Batch([sc], storage=storage)
    bt.step(steps)
    b, t = bt.tanks[0].fields(want_f=True), bt.tanks[0].stats()
    bt.close()
    assert s["covered"] > 0 and s["status"] == 0 and (s["uncovered"] > 0 or steps < 90)
    for key in ("flags", "f", "fill", "mass"):
        assert np.array_equal(a[key], b[key]), key
    for key in ("n_interface", "n_filled", "n_emptied", "n_new_from_gas", "n_new_from_liquid", "n_pending", "n_general"):
        assert s[key] == t[key], key
