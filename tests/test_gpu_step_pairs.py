"""The FP32 A/B and in-place steps with two adjacent nodes per thread (csrc/step_pair.cuh),
the default of cascaded D3Q19 lattices of 100,000 nodes or more, against the
one-node step (variant 1): the pair rounds like the single node, so every
population must be the same bits. Shapes: rows of even and odd length (an odd
row's last pair holds one node), rows shorter than a warp of pairs and longer
than a block, planes that end inside a block, a single row or plane, walls on
every axis, each force mode, the smallest lattice that takes the kernel and one
below it (where both run the one-node step)."""
import pytest
import torch

from gpu_common import dev, t
from paper_1801_04586_gb300 import Lattice, synthetic

pytestmark = pytest.mark.gpu

CASES = [
    # (nx, ny, nz), walls, force
    ((250, 20, 20), 0, "field"),     # 100,000 nodes exactly
    ((249, 20, 20), 0, "field"),     # below: one node per thread
    ((257, 31, 13), 1, "profile"),   # odd rows between x walls
    ((151, 28, 24), 6, "uniform"),   # odd rows, ragged blocks, y and z walls
    ((6, 151, 113), 7, "field"),     # three pairs per row, walls on every axis
    ((3, 200, 167), 3, "uniform"),   # two pairs per row, the second of one node
    ((700, 1, 144), 0, "profile"),   # ny = 1: the y shift maps a row onto itself
    ((512, 200, 1), 4, "uniform"),   # nz = 1 between two z walls
    ((1000, 11, 10), 2, "field"),      # rows longer than a block
]
# in place too: even and odd kinds, and a lattice of an odd number of nodes (the even kind's last pair is one node)
IN_PLACE = CASES + [((75, 55, 27), 7, "field"), ((75, 55, 27), 0, "profile")]
ALL = [(*c, "ab") for c in CASES] + [(*c, "aa") for c in IN_PLACE]


@pytest.mark.parametrize("shape_xyz,walls,force,pattern", ALL)
def test_pair_step_equals_one_node_step(shape_xyz, walls, force, pattern):
    nx, ny, nz = shape_xyz
    shape = (nz, ny, nx)
    rho = synthetic.density_perturbation(shape, 0.01, seed=601)
    u = synthetic.uniform_perturbation(shape, 0.03, seed=602)
    out = []
    for variant in (0, 1):
        g = Lattice(nx, ny, nz, 0.02, walls=walls, s2b=1.2, s3=1.1, s4=0.9, variant=variant, pattern=pattern,
                    device=dev())
        if force == "field":
            g.set_force_field(t(synthetic.gaussian_force(shape, 1e-4, seed=603)))
        elif force == "profile":
            g.set_force_profile_z(t(synthetic.kolmogorov_profile(nz, 1e-4)))
        else:
            g.set_force_uniform(1e-5, -2e-5, 3e-6)
        g.init_equilibrium(t(rho), t(u))
        g.step(7)
        first = g.populations(deviation=True)
        g.step(1)
        g.check()
        out.append((first, g.populations(deviation=True)))
        g.close()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
