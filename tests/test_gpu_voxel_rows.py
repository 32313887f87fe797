"""The voxel density's walk by slot pairs: rows that start or end on either half
of a pair, its form for long rows and for short ones, attached particles and
positions that are not finite among the candidates, and an odd number of
particles over memory that held NaN before, against the surface oracle (needs
a GB300)."""
import numpy as np
import pytest
import torch

from oracle import surface as osurf
from paper_2311_15088_gb300 import scenes
from paper_2311_15088_gb300.sph import Scene

pytestmark = pytest.mark.gpu

H = scenes.default_params()["h"]
Z = np.zeros((0, 4), np.float32)


# neighbours within h: rows of 0 to 2 candidates, of a few, of some tens
@pytest.mark.parametrize("n,cell,cell_x", [(151, 0.5, 0.0), (150, 0.5, 0.0), (1501, 0.5, 0.125), (1500, 1.0, 0.0),
                                           (6001, 1.0, 0.0)])
@pytest.mark.parametrize("long_rows", [False, True])
def test_voxel_density_of_any_row(n, cell, cell_x, long_rows):
    """Counts bit-exact and phi within 1e-5 R of the oracle's; the particle
    mass decides the form alone."""
    side = 0.2
    p = scenes.default_params(box_max=(side,) * 3, cell_size=scenes.f32(cell * H), cell_size_x=scenes.f32(cell_x * H))
    # candidates a row: rho0 / mass * cell^2 * (4/3 R + cell_x) above or below 7
    p["mass"] = scenes.f32((1e-3 if long_rows else 1e3) * 1000.0 * H ** 3)
    rng = np.random.default_rng(n)
    fluid = np.zeros((n, 4), np.float32)
    fluid[:, :3] = rng.uniform(0, side, size=(n, 3))
    # binned beside the fluid at the two ends of the grid, none of it
    stray = np.zeros((6, 4), np.float32)
    stray[:, :3] = [[np.nan, 0.01, 0.01], [0.01, np.inf, 0.01], [0.01, 0.01, -np.inf], [0.19, 0.19, np.nan],
                    [3e38, 0.19, 0.19], [0.19, -3e38, 0.19]]
    boid = np.zeros((21, 4), np.float32)
    boid[:, :3] = rng.uniform(0, side, size=(21, 3))
    both = np.concatenate([fluid, stray])
    size = Scene(p, len(both), len(boid)).workspace.numel()
    torch.full((size,), 255, dtype=torch.uint8, device="cuda")  # bytes 255: NaN in every float
    s = Scene(p, len(both), len(boid))
    s.set_state(both, np.zeros_like(both), boid, np.zeros_like(boid))
    R = scenes.f32(H)
    phi, cnt, origin, dims = s.voxel_density(scenes.f32(0.4 * H), R, scenes.f32(0.25 * H))
    ophi, ocnt = osurf.voxel_density(fluid, origin, scenes.f32(0.4 * H), dims, R, scenes.f32(0.25 * H))
    assert np.array_equal(cnt.cpu().numpy(), ocnt) and (ocnt > 0).sum() > 100
    assert np.all(np.abs(phi.cpu().double().numpy() - ophi) <= 1e-5 * float(R))
