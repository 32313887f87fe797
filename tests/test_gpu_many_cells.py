"""A grid of just more and just less than 2^27 cells (a warp of the keys' field
per cell is then 2^32 threads): keys, order and cell starts of a step against
numpy (needs a GB300)."""
import numpy as np
import pytest

from paper_2311_15088_gb300 import scenes
from paper_2311_15088_gb300.sph import Scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [511, 514])
def test_keys_of_every_cell(side):
    cell = 0.03125  # exact in float32, so that a cell's corners are
    p = scenes.default_params(h=0.0625, cell_size=cell, box_max=(side * cell,) * 3, mass=0.001)
    rng = np.random.default_rng(side)
    c = rng.integers(0, side, size=(3000, 3))
    c[:64] = side - 1 - rng.integers(0, 2, size=(64, 3))  # the last cells
    c[64:128] = rng.integers(0, 2, size=(64, 3))          # the first ones
    pos = np.zeros((3000, 4), np.float32)
    pos[:, :3] = (c + rng.uniform(0.2, 0.8, size=(3000, 3))) * cell
    z = np.zeros((0, 4), np.float32)
    s = Scene(p, 3000, 0)
    assert s.ncells == side ** 3 and (s.ncells > 2 ** 27) == (side == 514)
    s.set_state(pos, np.zeros_like(pos), z, z)
    s.step(1)
    keys = s.field("keys").cpu().numpy().view(np.uint32)
    assert np.array_equal(keys, c[:, 0] + side * (c[:, 1] + side * c[:, 2]))
    order = np.argsort(keys, kind="stable")
    assert np.array_equal(s.field("perm").cpu().numpy(), order)
    start = s.field("cell_start").cpu().numpy().view(np.uint32)
    assert start[-1] == 3000 and np.array_equal(start[keys], np.searchsorted(keys[order], keys))
    assert s.status() == 0
