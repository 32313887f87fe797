"""The force pass with a warp per particle where a particle has more hit segments
than are stored (its candidates are tested again, side by side): a small scene
alone against the same scene inside a batch that takes a thread per particle,
bit for bit (needs a GB300)."""
import numpy as np
import pytest
import torch

from paper_2311_15088_gb300 import scenes
from paper_2311_15088_gb300.sph import Scene

pytestmark = pytest.mark.gpu

H = scenes.default_params()["h"]


# cells of h (9 rows a walk), h/2 and h/4 (more than 32 rows), narrow along x;
# clumps whose every particle overflows and one where some do
@pytest.mark.parametrize("n,side,cell,cell_x", [(5000, 0.9, 1.0, 0.0), (4500, 0.9, 0.5, 0.0), (4301, 0.8, 0.25, 0.125),
                                                (6000, 1.3, 0.5, 0.125)])
def test_overflowed_lists_by_warp_and_by_thread(n, side, cell, cell_x):
    nb = 40
    rng = np.random.default_rng(n)
    fp, bp = np.zeros((n, 4), np.float32), np.zeros((nb, 4), np.float32)
    fp[:, :3] = 0.4 + side * H * rng.random((n, 3))
    bp[:, :3] = 0.4 + side * H * rng.random((nb, 3))
    fp[7::50, :3] = fp[6::50, :3][:len(fp[7::50])]  # coincident pairs
    fp[-200:, :3] = 0.1 + 0.5 * rng.random((200, 3))  # and some with few neighbours
    fv, bv = 0.1 * rng.normal(size=(n, 4)).astype(np.float32), np.zeros((nb, 4), np.float32)
    fv[:, 3], bv[:, 0] = 0, 0.5
    p = scenes.default_params(mass=scenes.f32(1e-4), cell_size=scenes.f32(cell * H), cell_size_x=scenes.f32(cell_x * H))
    # the filler makes the batch too large for the warp forms
    many = torch.cuda.get_device_properties(0).multi_processor_count * 108 + 1
    fill = scenes.scaled_block(many, 3, (1.0, 1.0, 1.0), (0.9, 0.9, 0.9), 5)
    alone = Scene(p, n, nb, diagnostics=True)
    alone.set_state(fp, fv, bp, bv)
    both = Scene([fill["params"], p], [many, n], [3, nb], diagnostics=True)
    both.set_state(*[np.concatenate([fill[k], x]) for k, x in
                     zip(("fluid_pos", "fluid_vel", "boid_pos", "boid_vel"), (fp, fv, bp, bv))])
    for _ in range(2):
        alone.step(1)
        both.step(1)
        for field in ("rho", "nseg", "acc", "touched", "influence"):
            a, b = alone.field(field), both.field(field)
            # ids: every scene's boids first, then the fluids, scene by scene
            assert torch.equal(a, torch.cat([b[3:3 + nb], b[3 + nb + many:]])), field
    for a, b in zip(alone.get_state(), both.get_state()):
        assert torch.equal(a, b[len(b) - len(a):])
    over = alone.field("nseg") > 128
    assert int(over.sum()) > 500 and int((~over).sum()) > 100
    assert int(alone.field("touched").max()) > 0 and alone.status() == 0
