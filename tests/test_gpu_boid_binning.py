"""The boids' binning, in one launch for few boids and in five for many:
order by cell then id, and every cell's start, against numpy (needs a GB300)."""
import numpy as np
import pytest

from paper_2311_15088_gb300 import scenes
from paper_2311_15088_gb300.sph import Scene, sph_grid_dims

pytestmark = pytest.mark.gpu


# one launch up to 1,024 boids in fewer than 8,192 cells; ragged multiples of
# four and of the block; boids outside the tank; the cells beyond the limit
@pytest.mark.parametrize("nb,cell", [(1, 4.0), (3, 4.0), (129, 4.0), (1023, 4.0), (1024, 4.0), (1025, 4.0), (1000, 1.05)])
def test_boid_order_and_cell_starts(nb, cell):
    h = scenes.default_params()["h"]
    p = scenes.default_params(mass=0.012, boid_cell_size=scenes.f32(cell * h))
    rng = np.random.default_rng(nb)
    bp = np.zeros((nb, 4), np.float32)
    bp[:, :3] = rng.uniform(-0.1, 1.1, (nb, 3))
    bp[nb // 2:, :3] = rng.uniform(0.3, 0.4, (nb - nb // 2, 3))  # crowded cells
    bv = np.zeros((nb, 4), np.float32)
    fp = np.full((5, 4), 0.9, np.float32)
    s = Scene(p, 5, nb)
    s.set_state(fp, np.zeros_like(fp), bp, bv)
    s.step(1)
    dims = sph_grid_dims(p, 1)
    assert (np.prod(dims) < 8192) == (cell == 4.0)
    inv = np.float32(1.0) / np.float32(p["boid_cell_size"])
    c = np.clip(np.floor((bp[:, :3] - np.float32(0)) * inv), 0, np.array(dims) - 1).astype(np.int64)
    key = c[:, 0] + dims[0] * (c[:, 1] + dims[1] * c[:, 2])
    order = np.lexsort((np.arange(nb), key))
    assert np.array_equal(s.field("boid_perm").cpu().numpy(), order)
    starts = np.searchsorted(key[order], np.arange(np.prod(dims) + 1))
    assert np.array_equal(s.field("boid_cell_start").cpu().numpy(), starts)
