"""Grids around 8,192 tiles, up to which the scan's (marching cubes') second
launch adds the tile totals itself; beyond, a launch of its own scans them
(needs a GB300)."""
import numpy as np
import pytest
import torch

from paper_2311_15088_gb300 import scenes, sph
from paper_2311_15088_gb300.sph import Scene

pytestmark = pytest.mark.gpu

SCAN_TILE, MC_TILE, TILES = 4096, 1024, 8192


@pytest.mark.parametrize("side,above", [(8.0, False), (8.4, True)])
def test_binning_of_many_cells(side, above):
    """Order and cell starts of two steps against numpy's stable order of the
    keys, whole numbers (the second step's counts start from the zeros that
    the first step's scan leaves)."""
    p = scenes.default_params(h=0.05, cell_size=0.025, box_max=(side, 8.0, 8.0), mass=0.001)
    n = 20000
    s = Scene(p, n, 0)
    assert (s.ncells > TILES * SCAN_TILE) == above and s.ncells > (TILES - 256) * SCAN_TILE
    rng = np.random.default_rng(3)
    pos = np.zeros((n, 4), np.float32)
    pos[:, :3] = rng.uniform(0.01, 7.99, size=(n, 3))
    pos[:500, :3] = 7.9 + rng.uniform(0, 0.02, size=(500, 3))  # crowded cells in the last tiles
    z = np.zeros((0, 4), np.float32)
    s.set_state(pos, np.zeros_like(pos), z, z)
    for _ in range(2):
        s.step(1)
        keys = s.field("keys").cpu().numpy().view(np.uint32)
        perm = s.field("perm").cpu().numpy()
        start = s.field("cell_start").cpu().numpy().view(np.uint32)
        order = np.argsort(keys, kind="stable")
        assert np.array_equal(perm, order)
        assert np.array_equal(start, np.searchsorted(keys[order], np.arange(s.ncells + 1)))
    assert s.status() == 0


@pytest.mark.parametrize("dims", [(204, 204, 204), (205, 205, 205)])
def test_marching_cubes_of_many_tiles(dims):
    """A grid's triangles are those of its two halves along z, one after the
    other, bit for bit (corner coordinates are exact: spacing 1/4)."""
    cubes = (dims[0] - 1) * (dims[1] - 1) * (dims[2] - 1)
    assert (cubes > TILES * MC_TILE) == (dims[0] == 205)
    x, y, z = (torch.arange(d, device="cuda", dtype=torch.float32) for d in dims)
    phi = (torch.sin(0.41 * x)[None, None, :] + torch.sin(0.37 * y)[None, :, None] + torch.sin(0.43 * z)[:, None, None])
    phi = phi.contiguous()
    tris, total = sph.marching_cubes(phi, dims, (0.0, 0.0, 0.0), 0.25, 0.3)
    assert total == len(tris) > 100000
    k = 97
    lo, n_lo = sph.marching_cubes(phi[:k + 1].contiguous(), (dims[0], dims[1], k + 1), (0.0, 0.0, 0.0), 0.25, 0.3)
    hi, n_hi = sph.marching_cubes(phi[k:].contiguous(), (dims[0], dims[1], dims[2] - k), (0.0, 0.0, 0.25 * k), 0.25, 0.3)
    assert n_lo + n_hi == total
    assert torch.equal(tris, torch.cat([lo, hi]))
