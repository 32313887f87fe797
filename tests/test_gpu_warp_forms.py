"""The density and force passes take a warp per particle in small launches and a
thread per particle in large ones: a small scene alone against the same scene
inside a batch too large for the warp form, bit for bit (needs a GB300)."""
import numpy as np
import pytest
import torch

from paper_2311_15088_gb300 import scenes
from paper_2311_15088_gb300.sph import Scene

pytestmark = pytest.mark.gpu

H = scenes.default_params()["h"]


def _scene(n, n_boid, region, cell, cell_x, seed):
    sc = scenes.scaled_block(n, n_boid, (1.0, 1.0, 1.0), region, seed)
    p = dict(sc["params"], cell_size=scenes.f32(cell * H), cell_size_x=scenes.f32(cell_x * H))
    return p, [sc["fluid_pos"], sc["fluid_vel"], sc["boid_pos"], sc["boid_vel"]]


# one particle; few neighbours; rows of the walk longer than 32 slots (several
# segments a row) with boids inside; more segments than a particle's list
# holds; fine cells (more than 32 rows a walk), narrow along x
CASES = {
    "single": (1, 0, (0.5, 0.5, 0.5), 0.5, 0.0),
    "sparse": (700, 9, (0.9, 0.9, 0.9), 0.5, 0.0),
    "long_rows": (3000, 60, (0.2, 0.2, 0.2), 1.0, 0.0),
    "many_segments": (6000, 5, (0.06, 0.06, 0.06), 0.5, 0.125),
    "fine_cells": (4000, 30, (0.3, 0.2, 0.2), 0.25, 0.125),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("diagnostics", [False, True])
def test_warp_and_thread_passes_agree(name, diagnostics):
    n, nb, region, cell, cell_x = CASES[name]
    p, state = _scene(n, nb, region, cell, cell_x, 77)
    # the filler makes the batch too large for the warp form
    per_sm = torch.cuda.get_device_properties(0).multi_processor_count * 108
    pf, fill = _scene(per_sm + 1, 3, (0.9, 0.9, 0.9), 0.5, 0.0, 5)
    alone = Scene(p, n, nb, diagnostics=diagnostics)
    alone.set_state(*state)
    both = Scene([pf, p], [per_sm + 1, n], [3, nb], diagnostics=diagnostics)
    both.set_state(*[np.concatenate([a, b]) for a, b in zip(fill, state)])
    for _ in range(2):
        alone.step(1)
        both.step(1)
        fields = ("rho", "pressure", "nbr_count", "nseg", "ncand")
        for field in fields + (("acc", "touched", "influence") if diagnostics else ()):
            a, b = alone.field(field).cpu().numpy(), both.field(field).cpu().numpy()
            # ids: every scene's boids first, then the fluids, scene by scene
            want = np.concatenate([b[3:3 + nb], b[3 + nb + per_sm + 1:]])
            assert np.array_equal(a, want), field
    for a, b in zip(alone.get_state(), both.get_state()):
        assert torch.equal(a, b[len(b) - len(a):])
    if name == "many_segments":
        assert int((alone.field("nseg") > 128).sum()) > 0
    if name == "long_rows":
        assert int((alone.field("nseg") > 9).sum()) > 0  # more segments than the nine rows of h cells
