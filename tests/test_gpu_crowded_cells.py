"""The per-cell sort of crowded cells (more than 128 entries, ids compared 32 at
a time): sizes around 128 and multiples of 32, shifted starts, crowded and
small cells side by side in one warp; fluid particles and boids
against numpy's stable order (needs a GB300)."""
import numpy as np
import pytest

from paper_2311_15088_gb300 import scenes
from paper_2311_15088_gb300.sph import Scene, sph_grid_dims

pytestmark = pytest.mark.gpu

SIZES = {
    "edges": [127, 128, 129, 159, 160, 161, 1, 255, 256, 257, 2, 191, 192, 193, 129, 129],
    "one": [5000],
    "mixed": [130, 7, 140, 1, 1, 200, 31, 33, 129, 64, 1000],
}


def _points(sizes, cell, first):
    """sizes[k] points inside cell first + k (along x, then z), in a random order of ids."""
    rng = np.random.default_rng(sum(sizes))
    k = np.repeat(np.arange(len(sizes)), sizes)
    c = np.stack([first + k % 4, np.full(len(k), first), first + k // 4], 1)
    x = np.zeros((len(k), 4), np.float32)
    x[:, :3] = (c + rng.uniform(0.1, 0.9, size=(len(k), 3))) * cell
    return x[rng.permutation(len(k))]


def _check(keys, perm, start, ncells):
    order = np.argsort(keys, kind="stable")
    assert np.array_equal(perm, order)
    assert np.array_equal(start, np.searchsorted(keys[order], np.arange(ncells + 1)))


@pytest.mark.parametrize("name", SIZES)
@pytest.mark.parametrize("before", [0, 1, 2, 3])
def test_crowded_fluid_cells(name, before):
    p = scenes.default_params(mass=0.001)
    pos = _points(SIZES[name], p["cell_size"], 5)
    low = np.full((before, 4), 0.01, np.float32)  # particles in a cell before them shift their starts
    pos = np.concatenate([pos, low])
    z = np.zeros((0, 4), np.float32)
    s = Scene(p, len(pos), 0)
    s.set_state(pos, np.zeros_like(pos), z, z)
    s.step(1)
    keys = s.field("keys").cpu().numpy().view(np.uint32)
    start = s.field("cell_start").cpu().numpy().view(np.uint32)
    assert sorted(np.diff(start)[np.diff(start) > 0]) == sorted(SIZES[name] + [before] * (before > 0))
    _check(keys, s.field("perm").cpu().numpy(), start, s.ncells)


@pytest.mark.parametrize("name", SIZES)
def test_crowded_boid_cells(name):
    h = scenes.default_params()["h"]
    p = scenes.default_params(mass=0.012, boid_cell_size=scenes.f32(h))
    sizes = SIZES[name] + [1100]  # more boids than the one-launch binning takes
    bp = _points(sizes, h, 3)
    fp = np.full((5, 4), 0.9, np.float32)
    s = Scene(p, 5, len(bp))
    s.set_state(fp, np.zeros_like(fp), bp, np.zeros_like(bp))
    s.step(1)
    keys = s.field("boid_keys").cpu().numpy().view(np.uint32)
    start = s.field("boid_cell_start").cpu().numpy().view(np.uint32)
    assert sorted(np.diff(start)[np.diff(start) > 0]) == sorted(sizes)
    _check(keys, s.field("boid_perm").cpu().numpy(), start, int(np.prod(sph_grid_dims(p, 1))))
