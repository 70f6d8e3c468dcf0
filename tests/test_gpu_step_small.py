"""Two FP32 A/B steps per launch on small lattices (csrc/step_small.cuh), the
default below 100,000 nodes where the plan finds it cheaper, against one step
per launch (variant 1): the intermediate state is kept as the FP32 values a
single step stores, so after any number of steps the populations must be the
same bits. Shapes: bricks that span axes (wrap inside the brick) and that end
ragged, walls on every axis, degenerate lattices, rows longer than a block (one
step per launch), each force mode and a decaying force; counts: odd, even, and
long enough for graph replays."""
import pytest
import torch

from gpu_common import dev, t
from paper_1801_04586_gb300 import Lattice, synthetic

pytestmark = pytest.mark.gpu

CASES = [
    # (nx, ny, nz), walls, force, decay
    ((16, 32, 32), 4, "uniform", 0.0),
    ((64, 20, 9), 0, "field", 1e-2),
    ((40, 33, 7), 6, "profile", 0.0),
    ((8, 70, 5), 7, "uniform", 0.0),
    ((33, 17, 9), 5, "field", 3e-3),
    ((150, 20, 12), 3, "field", 0.0),
    ((256, 1, 3), 0, "profile", 0.0),   # ny = 1, thin periodic z
    ((24, 50, 1), 4, "uniform", 0.0),   # nz = 1 between two z walls
    ((2, 3, 4), 1, "uniform", 0.0),
    ((1, 1, 40), 4, "uniform", 0.0),    # nx = 1: one step per launch
    ((1100, 3, 4), 2, "field", 0.0),    # rows split into bricks
    ((46, 46, 46), 7, "field", 0.0),
]


@pytest.mark.parametrize("shape_xyz,walls,force,decay", CASES)
def test_two_steps_per_launch_equal_single_steps(shape_xyz, walls, force, decay):
    nx, ny, nz = shape_xyz
    shape = (nz, ny, nx)
    rho = synthetic.density_perturbation(shape, 0.01, seed=801)
    u = synthetic.uniform_perturbation(shape, 0.03, seed=802)
    lats = []
    for variant in (0, 1):
        g = Lattice(nx, ny, nz, 0.02, walls=walls, s2b=1.2, s3=1.1, s4=0.9, variant=variant, device=dev())
        if force == "field":
            g.set_force_field(t(synthetic.gaussian_force(shape, 1e-4, seed=803)))
        elif force == "profile":
            g.set_force_profile_z(t(synthetic.kolmogorov_profile(nz, 1e-4)))
        else:
            g.set_force_uniform(1e-5, -2e-5, 3e-6)
        g.set_force_decay(decay)
        g.init_equilibrium(t(rho), t(u))
        lats.append(g)
    for n in (2, 1, 5, 37):
        for g in lats:
            g.step(n)
        assert torch.equal(lats[0].populations(deviation=True), lats[1].populations(deviation=True)), n
    lats[0].check()
    assert lats[0].steps_done == lats[1].steps_done == 45
