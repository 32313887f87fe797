"""The boid fields of a scene without boids: no entries, and cell starts of 0 over
memory that held other values before (needs a GB300)."""
import pytest
import torch

from paper_2311_15088_gb300 import scenes
from paper_2311_15088_gb300.sph import Scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [False, True])
def test_boid_fields_without_boids(batch):
    sc = scenes.scaled_block(500, 0, (1.0, 1.0, 1.0), (0.3, 0.3, 0.3), 3)
    p, n, b = ([sc["params"]] * 2, [250, 250], [0, 0]) if batch else (sc["params"], 500, 0)
    size = Scene(p, n, b).workspace.numel()
    torch.full((size,), 255, dtype=torch.uint8, device="cuda")
    s = Scene(p, n, b)
    s.set_state(sc["fluid_pos"], sc["fluid_vel"], sc["boid_pos"], sc["boid_vel"])
    s.step(1)
    start = s.field("boid_cell_start")
    assert len(start) == s.nbcells + 1 and not bool(start.any())
    assert s.field("boid_perm").numel() == s.field("boid_keys").numel() == 0 and s.status() == 0
