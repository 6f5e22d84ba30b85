"""A cell that several bodies cover in the same step is booked once and belongs
to the first of them, as in the oracle: in the single tank and in a batch, in
every storage."""
import numpy as np
import pytest

from paper_1201_0351_gb300 import inputs as I

from parity import assert_f64_parity, run_both

pytestmark = pytest.mark.gpu

STEPS = 20


def _overlapping_boxes():
    """Two heavy boxes in a closed box of liquid that overlap in y and move
    along x with one velocity: their front faces lie in the same plane, which
    crosses the centres of a layer of cells in the second step."""
    nx, ny, nz = 24, 26, 18
    flags, fill, rho = I.uniform_state(nx, ny, nz, I.LIQUID)
    boxes = [I.Box(center=(10.45, y, 9.0), half=(3.0, 3.6, 2.6), density_ratio=1e4, vel=(0.03, 0.0, 0.0),
                   mode=I.MODE_FREE) for y in (11.0, 14.0)]
    return I.Scenario("overlapping_boxes", nx, ny, nz, 0, 0.8, (0.0, 0.0, 0.0), (0.0, 0.0, 0.0), 1.0, 1e-2, flags, fill,
                      rho, boxes, 0)


def _common_cells(sc):
    """cells of the layer that both boxes cover: both fronts move from below to
    above the centres x = 13.5"""
    y = np.arange(sc.ny) + 0.5
    z = np.arange(sc.nz) + 0.5
    iny = np.logical_and.reduce([np.abs(y - b.center[1]) < b.half[1] for b in sc.boxes])
    return int(iny.sum()) * int((np.abs(z - sc.boxes[0].center[2]) < sc.boxes[0].half[2]).sum())


def test_common_cells_match_the_oracle():
    sc = _overlapping_boxes()
    assert _common_cells(sc) == 30
    g, o, gb, ob, gs, ref = run_both(sc, STEPS)
    assert_f64_parity(g, o, gb, ob)
    led = ref.ledger()
    for key, mine in (("covered", gs["covered"]), ("uncovered", gs["uncovered"])):
        assert led[key] > 10.0 and abs(mine - led[key]) <= 1e-11 * led[key], key


@pytest.mark.parametrize("storage", ["f32", "f16s"])
def test_common_cells_in_the_float_storages(storage):
    """the covered mass is the oracle's to the storage's density error (2e-3, as
    in the parity tests); the common cells' mass is 30 of about 68"""
    from paper_1201_0351_gb300 import lbm_fs

    import oracle

    sc = _overlapping_boxes()
    ref = oracle.OracleSim(sc)
    ref.step(STEPS)
    led = ref.ledger()
    sim = lbm_fs.Simulation(sc, storage=storage)
    sim.step(STEPS)
    s = sim.stats()
    sim.close()
    assert s["status"] == 0
    for key in ("covered", "uncovered"):
        assert abs(s[key] - led[key]) <= 2e-3 * led[key], key


@pytest.mark.parametrize("storage", ["f64", "f32", "f16s"])
def test_common_cells_in_a_batch(storage):
    from paper_1201_0351_gb300 import lbm_fs

    sc = _overlapping_boxes()
    sim = lbm_fs.Simulation(sc, storage=storage)
    sim.step(STEPS)
    a, s, ab = sim.fields(want_f=True), sim.stats(), [sim.body(k) for k in (0, 1)]
    sim.close()
    bt = lbm_fs.Batch([sc, sc], storage=storage)
    bt.step(STEPS)
    for t in bt.tanks:
        g, u = t.fields(want_f=True), t.stats()
        for key in ("flags", "f", "mass"):
            assert np.array_equal(a[key], g[key]), key
        # (the ledger is summed by atomics in arrival order: to its rounding)
        assert abs(u["covered"] - s["covered"]) <= 1e-12 * s["covered"]
        for k in (0, 1):
            for key in ("F", "T", "vel"):
                assert np.array_equal(ab[k][key], t.body(k)[key]), key
    bt.close()
