"""Device memory that a tank takes per cell, counted through the caller's
allocator: the populations twice, two fill levels (double, and float for the
float storages), mass, worklists and class bytes -- no more than the 384 (FP64),
232 (FP32) and 160 (FP16) bytes that the largest grids of a memory budget are
chosen by."""
import pytest

from paper_1201_0351_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _bytes(nz, storage):
    import torch

    from paper_1201_0351_gb300 import lbm_fs

    total = [0]

    def alloc(n, ctx):
        total[0] += int(n)
        return int(torch.cuda.caching_allocator_alloc(int(n)))

    def free(p, ctx):
        torch.cuda.caching_allocator_delete(int(p))

    class Counting:
        c_alloc, c_free = lbm_fs.DEV_ALLOC(alloc), lbm_fs.DEV_FREE(free)

    n = 32
    flags, fill, rho = I.hydrostatic_tank(n, n, nz, lambda X, Y: 0.5 * nz + 0.3, 1e-6, 1.0, 0)
    sc = I.Scenario("t", n, n, nz, 0, 0.7, (0.0, 0.0, -1e-6), (0.0, 0.0, 0.0), 1.0, 1e-2, flags, fill, rho, [], 0)
    keep, c = [], Counting()
    h = lbm_fs.lbm_fs_create(lbm_fs.scenario_params(sc, storage, 0, True, c, keep))
    lbm_fs.lbm_fs_step(h, 2)
    lbm_fs.lbm_fs_sync(h)
    lbm_fs.lbm_fs_destroy(h)
    return total[0]


@pytest.mark.parametrize("storage,limit", [("f64", 384), ("f32", 232), ("f16s", 160)])
def test_bytes_per_cell(storage, limit):
    # two grids of one cross-section (guard bands and fixed buffers cancel)
    cells = 32 * 32 * (64 - 32)
    per_cell = (_bytes(64, storage) - _bytes(32, storage)) / cells
    assert per_cell <= limit, per_cell
