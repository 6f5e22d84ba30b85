"""A splashing tank's conversion lists, and the cells that large bodies cover and
leave, are long: the tail kernel then works with all its blocks instead of one
cluster.  The results equal those of the batch's separate kernels bit for bit,
with and without graphs, and of the oracle."""
import dataclasses

import numpy as np
import pytest

from paper_1201_0351_gb300 import inputs as I

from parity import assert_f64_parity, macro_errors, run_both

pytestmark = pytest.mark.gpu

SHORT = 512  # entries up to which the cluster works alone


def splash(nx, ny, nz, drops, seed=1, speed=0.06):
    """a pool and liquid drops above it that move down and sideways"""
    rng = np.random.default_rng(seed)
    z, y, x = np.meshgrid(np.arange(nz) + 0.5, np.arange(ny) + 0.5, np.arange(nx) + 0.5, indexing="ij")
    depth = 0.35 * nz + 0.8 - z
    vel = np.zeros((nz, ny, nx, 3))
    for _ in range(drops):
        r = rng.uniform(3.0, 4.5)
        c = [rng.uniform(r + 2, n - r - 2) for n in (nx, ny)] + [rng.uniform(0.35 * nz + r + 1, nz - r - 2)]
        d = r + 0.5 - np.sqrt((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2)
        depth = np.maximum(depth, d)
        vel[d > 0] = (rng.uniform(-speed, speed), rng.uniform(-speed, speed), -rng.uniform(0, speed))
    fill = np.clip(depth, 0.0, 1.0)
    flags = np.where(depth >= 1.0, I.LIQUID, np.where(depth <= 0.0, I.GAS, I.INTERFACE)).astype(np.uint8)
    # closed interface layer along every link (nothing beyond the walls)
    pad = np.pad(flags, 1)
    near = np.zeros(flags.shape, bool)
    for dx, dy, dz in I._neighbour_offsets():
        near |= pad[1 + dz:nz + 1 + dz, 1 + dy:ny + 1 + dy, 1 + dx:nx + 1 + dx] == I.GAS
    flags[(flags == I.LIQUID) & near] = I.INTERFACE
    fill = np.where(flags == I.LIQUID, 1.0, np.where(flags == I.GAS, 0.0, np.clip(fill, 0.01, 1.0)))
    vel[flags == I.GAS] = 0.0
    return I.Scenario("splash", nx, ny, nz, 0, 0.7, (0.0, 0.0, -2e-5), (0.0, 0.0, 0.0), 1.0, 1e-2, flags.reshape(-1),
                      fill.reshape(-1), np.ones(nx * ny * nz), [], 0, vel.reshape(-1))


def large_moving_box(n):
    """all liquid, a heavy rotated box whose faces cross cells every step"""
    flags, fill, rho = I.uniform_state(n, n, n, I.LIQUID)
    box = I.Box(center=(n / 2 + 0.1, n / 2 + 0.2, n / 2), half=(0.31 * n, 0.27 * n, 0.23 * n), density_ratio=50.0,
                quat=I.heel_quat(17.0, (0.0, 0.6, 0.8)), vel=(0.12, 0.06, 0.0), mode=I.MODE_FREE)
    return I.Scenario("moving_box", n, n, n, 7, 0.8, (0.0, 0.0, 0.0), (0.0, 0.0, 0.0), 1.0, 1e-2, flags, fill, rho,
                      [box], 0)


def half_immersed_box(n):
    """a fast box through the surface of a half-full tank: cells that it leaves
    become liquid, interface and gas, about a hundred a step"""
    flags, fill, rho = I.hydrostatic_tank(n, n, n, lambda X, Y: 0.5 * n + 0.3, 1e-5, 1.0, 3)
    box = I.Box(center=(n / 2 + 0.1, n / 2 + 0.2, n / 2), half=(0.31 * n, 0.27 * n, 0.23 * n), density_ratio=50.0,
                quat=I.heel_quat(17.0, (0.0, 0.6, 0.8)), vel=(0.12, 0.06, 0.0), mode=I.MODE_FREE)
    return I.Scenario("half_immersed", n, n, n, 3, 0.8, (0.0, 0.0, -1e-5), (0.0, 0.0, 0.0), 1.0, 1e-2, flags, fill, rho,
                      [box], 0)


def _alone(sc, storage, steps, use_graphs=True):
    from paper_1201_0351_gb300 import lbm_fs

    sim = lbm_fs.Simulation(sc, storage=storage, use_graphs=use_graphs)
    entries = 0
    for _ in range(steps):
        sim.step(1)
        s = sim.stats()
        # (each uncovered cell of an all-liquid tank is pending and one is covered for it)
        entries = max(entries, s["n_filled"] + s["n_emptied"], s["n_pending"])
    out = sim.fields(want_f=True), s, entries
    sim.close()
    return out


def _batched(sc, storage, steps):
    from paper_1201_0351_gb300 import lbm_fs

    bt = lbm_fs.Batch([sc], storage=storage)
    bt.step(steps)
    out = bt.tanks[0].fields(want_f=True), bt.tanks[0].stats()
    bt.close()
    return out


@pytest.mark.parametrize("storage", ["f64", "f32", "f16s"])
@pytest.mark.parametrize("scene", ["splash", "box"])
def test_long_lists_equal_the_batch(scene, storage):
    sc = splash(100, 90, 80, 250) if scene == "splash" else large_moving_box(96)
    steps = 6
    a, s, entries = _alone(sc, storage, steps)
    assert entries > SHORT // (1 if scene == "splash" else 2) and s["status"] == 0, entries
    b, t = _batched(sc, storage, steps)
    c, u, _ = _alone(sc, storage, steps, use_graphs=False)
    for other, st in ((b, t), (c, u)):
        for key in ("flags", "f", "fill", "mass"):
            assert np.array_equal(a[key], other[key]), key
        for key in ("n_interface", "n_filled", "n_emptied", "n_new_from_gas", "n_new_from_liquid", "n_pending"):
            assert s[key] == st[key], key


PENDING_BY_WARPS = 36  # pending cells up to which each has a warp


@pytest.mark.parametrize("scene", ["half_immersed", "inside"])
def test_many_uncovered_cells_against_the_oracle(scene):
    """the remap's rule for long pending lists, a thread per cell"""
    sc = half_immersed_box(44) if scene == "half_immersed" else large_moving_box(40)
    g, o, gb, ob, gs, ref = run_both(sc, 6)
    assert gs["n_pending"] > PENDING_BY_WARPS
    assert_f64_parity(g, o, gb, ob)
    led = ref.ledger()
    for key in ("covered", "uncovered"):
        assert abs(gs[key] - led[key]) <= 1e-11 * led[key], key


@pytest.mark.parametrize("storage", ["f32", "f16s"])
def test_many_uncovered_cells_in_the_float_storages(storage):
    """alone and in a batch bit for bit; density within 2e-3 and classes of the
    oracle, the bounds of the parity tests"""
    import oracle

    sc = half_immersed_box(44)
    a, s, _ = _alone(sc, storage, 6)
    b, t = _batched(sc, storage, 6)
    assert s["n_pending"] > PENDING_BY_WARPS and s["status"] == 0
    for key in ("flags", "f", "fill", "mass"):
        assert np.array_equal(a[key], b[key]), key
    ref = oracle.OracleSim(sc)
    ref.step(6)
    e = macro_errors(a, ref.fields(want_f=True))
    assert e["flag_diff"] == 0 and e["rho"] <= 2e-3, e


@pytest.mark.parametrize("storage", ["f64", "f32", "f16s"])
def test_large_body_range(storage):
    """a body whose range takes more blocks than the force kernel's 64: the
    cells next to it and the remap's lists in a batch beside a small tank equal
    those alone, and (FP64) the oracle's"""
    from paper_1201_0351_gb300 import lbm_fs

    sc, small = half_immersed_box(72), half_immersed_box(30)
    a, s, _ = _alone(sc, storage, 4)
    bt = lbm_fs.Batch([small, sc], storage=storage)
    bt.step(4)
    b, t = bt.tanks[1].fields(want_f=True), bt.tanks[1].stats()
    bt.close()
    for key in ("flags", "f", "fill", "mass"):
        assert np.array_equal(a[key], b[key]), key
    assert s["n_general"] == t["n_general"] > 1000 and s["n_pending"] == t["n_pending"] > 0
    if storage == "f64":
        g, o, gb, ob, gs, ref = run_both(sc, 4)
        assert_f64_parity(g, o, gb, ob)


def test_long_lists_against_the_oracle():
    sc = splash(64, 60, 56, 90)
    g, o, gb, ob, gs, ref = run_both(sc, 4)
    assert gs["n_filled"] + gs["n_emptied"] > 0
    assert_f64_parity(g, o, gb, ob)
