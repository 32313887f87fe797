"""The density and force passes with a thread per particle, which launches of
more than 108 and 80 particles per multiprocessor take: a first step against
the oracle, on the library and on its bounds-checked build, and the launch
shapes (block size, particles per thread, source of the pairs) bit for bit
(needs a GB300)."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_2311_15088_gb300 import build, scenes
from paper_2311_15088_gb300.sph import SPH_DEV_BOUNDS, Scene

from parity import compare_step, gpu_outputs, oracle_step

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def _above():
    """An odd number of particles, boids' included, just above both limits."""
    return torch.cuda.get_device_properties(0).multi_processor_count * 108 + 97


def _scene(n_boid, cell, cell_x, seed):
    sc = scenes.scaled_block(_above() - n_boid, n_boid, (1.0, 1.0, 1.0), (0.58, 0.58, 0.58), seed)
    sc["boid_pos"][:, :3] *= np.float32(0.58)  # among the fluid
    h = sc["params"]["h"]
    sc["params"].update(cell_size=scenes.f32(cell * h), cell_size_x=scenes.f32(cell_x * h))
    return sc


@pytest.mark.parametrize("cell,cell_x", [(0.5, 0.125), (1.0, 0.0)])
@pytest.mark.parametrize("use_segments", [1, 0])
def test_first_step_of_the_thread_forms(cell, cell_x, use_segments):
    sc = _scene(150, cell, cell_x, 31)
    p = sc["params"]
    s = Scene(p, len(sc["fluid_pos"]), 150, diagnostics=True)
    s.set_tuning(256, use_segments)
    s.set_state(sc["fluid_pos"], sc["fluid_vel"], sc["boid_pos"], sc["boid_vel"])
    s.step(1)
    compare_step(p, gpu_outputs(s), oracle_step(p, sc), 150)
    assert s.status() & SPH_DEV_BOUNDS == 0
    assert int(s.field("touched").sum()) > 0


def test_thread_forms_on_the_bounds_checked_build():
    """Every slot index of the walks and the hit segments is checked there."""
    lib = build.build(checked=True)
    env = dict(os.environ, SPH_GB300_LIB=lib)
    r = subprocess.run([sys.executable, "-m", "pytest", os.path.abspath(__file__), "-q", "-x", "-m", "gpu",
                        "-k", "first_step_of_the_thread_forms", "-p", "no:cacheprovider"],
                       env=env, capture_output=True, text=True, cwd=os.path.dirname(HERE), timeout=1200)
    tail = (r.stdout + r.stderr)[-3000:]
    assert r.returncode == 0, tail
    assert "4 passed" in r.stdout, tail


def _batch():
    """A scene above the limits between two small ones, one without boids."""
    big = _scene(40, 0.5, 0.0, 7)
    small = [scenes.scaled_block(900, 12, (1.0, 1.0, 1.0), (0.25, 0.2, 0.2), 8),
             scenes.scaled_block(333, 0, (1.0, 1.0, 1.0), (0.12, 0.2, 0.2), 9)]
    scs = [small[0], big, small[1]]
    s = Scene([c["params"] for c in scs], [len(c["fluid_pos"]) for c in scs], [len(c["boid_pos"]) for c in scs],
              diagnostics=True)
    return s, [np.concatenate([c[k] for c in scs]) for k in ("fluid_pos", "fluid_vel", "boid_pos", "boid_vel")]


@pytest.mark.parametrize("block,use_segments,ppt", [(64, 1, 1), (128, 1, 2), (256, 1, 4), (512, 1, 1), (512, 1, 4),
                                                    (64, 1, 2), (64, 0, 1), (256, 0, 2), (512, 0, 4)])
def test_launch_shape_of_the_thread_forms_changes_no_bit(block, use_segments, ppt):
    got = []
    for shape in (None, (block, use_segments, ppt)):
        s, state = _batch()
        if shape:
            s.set_tuning(block, use_segments)
            s.set_particles_per_thread(ppt)
        s.set_state(*state)
        s.step(3)
        got.append(s.get_state() + [s.field(f) for f in ("rho", "nbr_count", "ncand", "acc", "touched", "influence",
                                                         "fb")])
        assert s.status() == 0
    assert all(torch.equal(a, b) for a, b in zip(*got))
    assert int(got[0][-2].ne(0).sum()) > 0
