"""Several tanks stepped at the same time, each on a stream and from a thread of
its own, equal each tank alone bit for bit: the tail kernel of a splashing tank
lets those of its blocks work that have started, so their number differs from
step to step when other tanks hold the GPU.  And body states in any number: a
read that fits the pinned buffer (28 bodies) equals the larger one."""
import threading

import numpy as np
import pytest

from paper_1201_0351_gb300 import inputs as I

from test_gpu_long_lists import half_immersed_box, splash

pytestmark = pytest.mark.gpu

STEPS = 30


def _scenes():
    return [(splash(100, 90, 80, 250, seed=1), "f32"), (splash(96, 96, 84, 250, seed=2), "f16s"),
            (half_immersed_box(60), "f32"), (splash(64, 60, 56, 90, seed=3), "f64")]


def test_tanks_on_streams_and_threads_equal_each_alone():
    import torch

    from paper_1201_0351_gb300 import lbm_fs

    want, sims = [], []
    for sc, storage in _scenes():
        sim = lbm_fs.Simulation(sc, storage=storage)
        sim.step(STEPS)
        want.append((sim.fields(want_f=True), sim.stats()))
        sim.close()
        sims.append(lbm_fs.Simulation(sc, storage=storage, stream=torch.cuda.Stream()))

    failed = []

    def work(sim):
        try:
            for _ in range(STEPS // 5):
                sim.step(5)
            sim.sync()
        except Exception as e:  # reported by the test's thread
            failed.append(e)

    threads = [threading.Thread(target=work, args=(sim,)) for sim in sims]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for sim, (g, s) in zip(sims, want):
        h, u = sim.fields(want_f=True), sim.stats()
        sim.close()
        assert s["status"] == u["status"] == 0
        for key in ("flags", "f", "fill", "mass"):
            assert np.array_equal(g[key], h[key]), key
        for key in ("n_interface", "n_filled", "n_emptied", "n_pending"):
            assert s[key] == u[key], key


def test_body_states_of_many_bodies():
    from paper_1201_0351_gb300 import lbm_fs

    n = 72
    flags, fill, rho = I.hydrostatic_tank(n, n, n, lambda X, Y: 0.5 * n + 0.3, 1e-5, 1.0, 0)
    boxes = [I.Box(center=(6.0 + 11.0 * (k % 6), 6.0 + 11.0 * (k // 6), 0.5 * n), half=(3.2, 3.2, 3.2), density_ratio=0.5,
                   mode=I.MODE_FREE, shape=I.SHAPE_SPHERE, vel=(0.001 * k, 0.0, 0.0)) for k in range(36)]
    sc = I.Scenario("spheres", n, n, n, 0, 0.7, (0.0, 0.0, -1e-5), (0.0, 0.0, 0.0), 1.0, 1e-2, flags, fill, rho, boxes, 0)
    sim = lbm_fs.Simulation(sc, storage="f32")
    sim.step(3)
    one = [sim.body(k) for k in range(36)]
    assert any(np.abs(b["F"]).max() > 0 for b in one)
    for first, count in ((0, 36), (0, 28), (0, 29), (5, 31), (35, 1)):
        out = lbm_fs.lbm_fs_body_states(sim.h, first, count)
        for k in range(count):
            for key, field in (("F", "F"), ("T", "T"), ("center", "center"), ("quat", "quat"), ("vel", "vel"),
                               ("omega", "omega")):
                assert np.array_equal(np.array(getattr(out[k], field)), one[first + k][key]), (first, count, k, key)
    sim.close()
