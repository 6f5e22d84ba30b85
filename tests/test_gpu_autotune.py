"""Autotuning a batch changes its launch configuration only where a choice was
measured: an FP16 batch keeps its zb (its bulk kernels take none), and what the
statistics report is as before the call."""
import pytest

from paper_1201_0351_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f64", "f32", "f16s"])
def test_autotune_keeps_what_it_does_not_measure(storage):
    from paper_1201_0351_gb300 import lbm_fs

    scenes = [I.random_box_scene(40, 30, 22, seed=11, nboxes=2, speed=0.02),
              I.random_box_scene(24, 18, 18, seed=14, nboxes=1, periodic=1, speed=0.02)]
    bt = lbm_fs.Batch(scenes, storage=storage)
    cfg = bt.config()
    bt.set_config(3, cfg["bulk_blocks"], 700, 0)
    bt.step(5)
    before = [t.stats() for t in bt.tanks]
    new = bt.autotune()
    assert new["list_cells"] == 700 and new["lanes"] == cfg["lanes"] and new["bulk_ms"] > 0.0
    if storage == "f16s":
        assert new["zb"] == 3
    else:
        assert new["zb"] in (1, 2, 4, 8)
    for a, t in zip(before, bt.tanks):
        b = t.stats()
        for key in a:
            if key != "kernel_launches":
                assert a[key] == b[key], key
        assert a["n_interface"] > 0
    bt.close()
