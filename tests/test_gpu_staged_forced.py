"""The staged steps (csrc/step_tma.cuh) at the tile shapes of
test_gpu_staged.py. By default lattices this small run the faster unstaged
forms; a context that bounds the staged waits (wait_cycles) runs staged at any
size, so here the staged kernels meet those shapes: the same bits as one node
per thread, and as the default form, which takes node pairs or single nodes."""
import pytest
import torch

from gpu_common import dev, t
from paper_1801_04586_gb300 import Lattice, synthetic
from test_gpu_staged import AA_CASES, CASES, CASES27, RATES

pytestmark = pytest.mark.gpu

WAIT = 4_000_000_000  # the default bound of a wait, named: runs staged at any size

ALL = ([(s, w, st, "field", dict(model=m)) for s, w, st, m in CASES]
       + [(s, w, st, "profile", dict(model=m, lattice=27)) for s, w, st, m in CASES27]
       + [(s, w, st, f, dict(pattern="aa")) for s, w, st, f in AA_CASES]
       + [((150, 96, 70), 2, "f16", "field", {}), ((152, 95, 71), 0, "bf16sr", "uniform", {}),  # node pairs by default
          ((151, 94, 72), 7, "f16sr", "profile", {})])                                          # ... of odd rows


@pytest.mark.parametrize("shape_xyz,walls,storage,force,kw", ALL)
def test_forms_agree(shape_xyz, walls, storage, force, kw):
    nx, ny, nz = shape_xyz
    shape = (nz, ny, nx)
    rho = synthetic.density_perturbation(shape, 0.01, seed=701)
    u = synthetic.uniform_perturbation(shape, 0.03, seed=702)
    out = []
    for form in (dict(variant=1), dict(variant=0, wait_cycles=WAIT), dict(variant=0)):
        g = Lattice(nx, ny, nz, 0.02, walls=walls, storage=storage, device=dev(), **RATES, **kw, **form)
        if force == "field":
            g.set_force_field(t(synthetic.gaussian_force(shape, 1e-4, seed=703)))
        elif force == "profile":
            g.set_force_profile_z(t(synthetic.kolmogorov_profile(nz, 1e-4)))
        else:
            g.set_force_uniform(1e-5, -2e-5, 3e-6)
        g.init_equilibrium(t(rho), t(u))
        g.step(1)
        first = g.populations(deviation=True)
        g.step(6)
        g.check()
        out.append((first, g.populations(deviation=True)))
        g.close()
    for other in out[1:]:
        assert torch.equal(out[0][0], other[0]) and torch.equal(out[0][1], other[1])
