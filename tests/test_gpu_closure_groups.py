"""Which cells take the closure together: with the resident kernels the cells
of a block (up to block_floes floes of cells in decreasing order of size) do
so only if all of them qualify, whatever the size of the model or the GPU."""
import numpy as np
import pytest

from paper_2303_07819_gb300 import inputs as I
from tests.test_gpu_runs import crowd, join, soft

pytestmark = pytest.mark.gpu

NX, PER = 16, 16          # 256 cells of 16 floes: 16 cells to a block of 256 floes


@pytest.mark.parametrize("block,heavy,qualify", [(256, 16, 0), (256, 32, 128), (64, 16, 192), (32, 16, 224), (256, 0, 256)])
def test_a_block_keeps_its_closure_cells_only_together(block, heavy, qualify):
    """Every heavy-th cell holds ice of twice the thickness and lies outside
    the network's box: the cells of its block run their DEM with it."""
    from paper_2303_07819_gb300 import msdem as ms
    ms.load()
    side = 25e3
    parts = []
    for c in range(NX * NX):
        f = crowd(c, PER, side, 0.3)
        f["x"] += side * (c % NX)
        f["y"] += side * (c // NX)
        f["h"][:] = 2.0 if heavy and c % heavy == 0 else 1.0
        parts.append(f)
    f, p = join(parts), soft(NX, NX * side)
    m = ms.Model(p, f, ms.MS_FP32)
    m.set_resident(24.0, block)
    mass = m.moments()[:, 1] / side ** 2
    box = np.array([[-3e38] * 16, [3e38] * 16], dtype=np.float32)
    if heavy:
        out = np.arange(NX * NX) % heavy == 0
        assert mass[out].min() > 1.05 * mass[~out].max()
        box[1, 0] = 0.5 * (mass[out].min() + mass[~out].max())
    norm = {"mu_x": np.zeros(16), "sd_x": np.ones(16), "mu_y": np.zeros(4), "sd_y": np.ones(4)}
    m.closure_attach(ms.MLP(I.mlp_init(), norm, max_batch=256), 0, 1e30, box)
    m.step(10.0, p["N0"])                 # the first interval runs every cell's DEM
    assert m.closure_stats()["closure_cell_intervals"] == 0
    m.step(10.0, p["N0"])
    assert m.closure_stats()["closure_cell_intervals"] == qualify
