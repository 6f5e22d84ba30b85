"""FP16 storage on both sides of the width below which the bulk step takes one
cell per thread instead of the ring: equal to the software-pipelined kernel bit
for bit, and in a batch of narrow and wide tanks to each tank alone."""
import numpy as np
import pytest

from paper_1201_0351_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _flow(nx, ny, nz, periodic, seed=3):
    flags, fill, rho = I.hydrostatic_tank(nx, ny, nz, lambda X, Y: 0.6 * nz + 0.4, 1e-5, 1.0, periodic)
    vel = 0.01 * np.random.default_rng(seed).standard_normal((nx * ny * nz, 3))
    vel[flags == I.GAS] = 0.0
    return I.Scenario("flow", nx, ny, nz, periodic, 0.7, (0.0, 0.0, -1e-5), (0.0, 0.0, 0.0), 1.0, 1e-2, flags, fill, rho,
                      [], 0, vel.reshape(-1))


def _alone(sc, steps):
    from paper_1201_0351_gb300 import lbm_fs

    sim = lbm_fs.Simulation(sc, storage="f16s")
    sim.step(steps)
    g, s = sim.fields(want_f=True), sim.stats()
    sim.close()
    assert s["status"] == 0
    return g


@pytest.mark.parametrize("dims,periodic", [((1, 300, 9), 1), ((2, 64, 40), 0), ((4, 40, 33), 1), ((5, 33, 30), 0),
                                           ((5, 31, 29), 3), ((6, 33, 30), 0), ((6, 31, 29), 1), ((7, 30, 31), 2)])
def test_narrow_grids_match_the_pipelined_kernel(dims, periodic, monkeypatch):
    sc = _flow(*dims, periodic)
    out = []
    for v in ("pipe", "plain"):
        monkeypatch.setenv("LBMFS_BULK", v)
        out.append(_alone(sc, 4))
    assert np.array_equal(out[0]["flags"], out[1]["flags"])
    assert np.array_equal(out[0]["f"], out[1]["f"])


@pytest.mark.parametrize("dims", [[(5, 33, 30), (40, 20, 18), (1, 90, 20), (6, 31, 29)], [(2, 40, 30), (5, 20, 20)]])
def test_narrow_tanks_in_a_batch(dims):
    from paper_1201_0351_gb300 import lbm_fs

    scenes = [_flow(*n, 1, seed=k) for k, n in enumerate(dims)]
    bt = lbm_fs.Batch(scenes, storage="f16s")
    bt.step(4)
    bt.autotune()
    bt.step(4)
    res = [t.fields(want_f=True) for t in bt.tanks]
    assert all(t.stats()["status"] == 0 for t in bt.tanks)
    bt.close()
    for sc, g in zip(scenes, res):
        a = _alone(sc, 8)
        for key in ("flags", "f", "fill", "mass"):
            assert np.array_equal(a[key], g[key]), (sc.nx, key)
