"""With more boids than fit on the chip at once the force pass spreads their
blocks between the fluid particles' (every second to fourth block): the step
against the fused pipeline, which takes the boids from a queue of its own,
bit for bit (needs a GB300)."""
import pytest
import torch

from paper_2311_15088_gb300 import scenes
from paper_2311_15088_gb300.sph import Scene

pytestmark = pytest.mark.gpu


# fluid blocks per boid block below 1, 1 to 2 and above 3 at blocks of 256; at
# 128 and 512 a warp's place in its block differs
@pytest.mark.parametrize("n_fluid", [60_000, 200_003, 600_001])
@pytest.mark.parametrize("block", [128, 256, 512])
def test_spread_boid_blocks_agree_with_the_pipeline(n_fluid, block):
    nb = 33 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    sc = scenes.scaled_block(n_fluid, nb, (4.0, 1.0, 1.0), (4.0, 0.8, 0.8), 11)
    got = []
    for pipeline in (False, True):
        s = Scene(sc["params"], n_fluid, nb)
        s.set_state(sc["fluid_pos"], sc["fluid_vel"], sc["boid_pos"], sc["boid_vel"])
        if pipeline:
            s.set_pipeline(1024, 256)
        else:
            s.set_tuning(block, 1)
        s.step(2)
        got.append([t.clone() for t in s.get_state()] + [s.field("fb").clone(), s.field("att_vel").clone()])
        assert s.status() == 0
    assert all(torch.equal(a, b) for a, b in zip(*got))
    assert bool(got[0][-2].abs().sum() > 0)
