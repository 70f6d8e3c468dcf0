"""Which kernel form a lattice's steps run in (clbm_get_step_form), and that a
lattice which reports the staged form computes the oracle's step: one staged
FP16 step with walls and a force field, at a size that only a bounded wait makes
run staged."""
import numpy as np
import pytest
import torch

import oracle
from gpu_common import W, dev, s2_of, t
from paper_1801_04586_gb300 import Lattice, synthetic
from test_gpu_staged import RATES, ulp16

pytestmark = pytest.mark.gpu

ONE, TWO, PAIRS, STAGED, STEPS = ("one node per thread", "two nodes per thread", "two adjacent nodes per thread",
                                  "staged in shared memory", "two steps per launch")
WAIT = 4_000_000_000


@pytest.mark.parametrize("shape,kw,form", [
    ((16, 32, 32), {}, STEPS),
    ((16, 32, 32), dict(pattern="aa"), ONE),
    ((64, 64, 64), {}, PAIRS),
    ((64, 64, 64), dict(pattern="aa"), PAIRS),
    ((64, 64, 64), dict(block=(64, 2)), ONE),
    ((64, 64, 64), dict(variant=1), ONE),
    ((64, 64, 64), dict(variant=2), TWO),
    ((64, 64, 64), dict(model="srt"), ONE),
    ((64, 64, 64), dict(lattice=27), ONE),
    ((24, 16, 16), dict(storage="f16"), ONE),
    ((24, 16, 16), dict(storage="f16", wait_cycles=WAIT), STAGED),
    ((24, 16, 16), dict(storage="bf16sr", wait_cycles=WAIT, pattern="aa"), STAGED),
    ((50, 50, 50), dict(storage="f16"), PAIRS),  # rows that are no multiple of 16 bytes
    ((50, 50, 50), dict(storage="f16", pattern="aa"), ONE),
    ((160, 160, 160), dict(storage="f16"), STAGED),
    ((160, 160, 160), dict(storage="f16", pattern="aa"), STAGED),
    ((24, 16, 16), dict(storage="f16", slab=3), STAGED),
    ((24, 16, 16), dict(slab=3), ONE),
])
def test_step_form(shape, kw, form):
    g = Lattice(*shape, 0.02, device=dev(), **kw)
    assert g.step_form() == form
    g.close()


@pytest.mark.parametrize("shape,kw,form", [
    # tiles of 520 nodes (one row each, half full) in two full rounds: rounds count, not nodes
    ((520, 20, 30), dict(storage="f16sr", lattice=27), STAGED),
    ((600, 25, 24), dict(storage="f16", lattice=27), STAGED),
    ((520, 80, 64), dict(storage="f16", pattern="aa"), ONE),
    ((520, 80, 64), dict(storage="f16"), PAIRS),
    # SRT and MRT below the node pairs' sizes; z walls make whole planes of slow tiles, x walls every tile
    ((80, 80, 80), dict(storage="f16", model="mrt"), STAGED),
    ((264, 60, 60), dict(storage="f16", model="mrt", walls=6), ONE),
    ((128, 128, 128), dict(storage="f16", model="srt", walls=1), ONE),
    ((128, 128, 100), dict(storage="f16", lattice=27), STAGED),
    ((128, 128, 100), dict(storage="f16", lattice=27, walls=1), ONE),
    ((64, 64, 64), dict(storage="f16sr", pattern="aa", walls=6), ONE),
    ((96, 96, 96), dict(storage="f16sr", pattern="aa", walls=6), STAGED),
])
def test_form_follows_the_tiles(shape, kw, form):
    g = Lattice(*shape, 0.02, device=dev(), **kw)
    assert g.step_form() == form
    g.close()


def test_step_form_follows_the_force():
    nx, ny, nz = 128, 128, 128
    g = Lattice(nx, ny, nz, 0.02, storage="f16", lattice=27, device=dev())
    assert g.step_form() == STAGED
    g.set_force_field(torch.zeros(3, nz, ny, nx, device=dev()))
    assert g.step_form() == ONE  # a tile's force rows do not fit beside 27 populations
    g.set_force_uniform(1e-6)
    assert g.step_form() == STAGED
    g.close()
    g = Lattice(24, 16, 16, 0.02, storage="f16", wait_cycles=WAIT, device=dev())
    odd = torch.zeros(3 * 24 * 16 * 16 + 1, device=dev())[1:].view(3, 16, 16, 24)  # 4-byte aligned only
    g.set_force_field(odd)
    assert g.step_form() == ONE
    g.close()


def test_staged_form_against_oracle():
    """Each stored deviation of one step from an FP16-representable state is the
    oracle's rounded to FP16: within half a unit in the last place plus the FP32
    arithmetic's error (the bound of the same test at the default form)."""
    nx, ny, nz, walls = 64, 24, 18, 6
    shape = (nz, ny, nx)
    g = Lattice(nx, ny, nz, 0.03, walls=walls, storage="f16", wait_cycles=WAIT, device=dev(), **RATES)
    o = oracle.Lattice(nx, ny, nz, walls=walls, s2=s2_of(0.03), **RATES)
    h0 = torch.from_numpy(synthetic.rng(511).uniform(-2e-3, 2e-3, (19,) + shape)).half().float().numpy()
    F = synthetic.gaussian_force(shape, 1e-4, seed=512)
    g.set_force_field(t(F))
    assert g.step_form() == STAGED
    g.set_populations(t(h0), deviation=True)
    g.step(1)
    ho = oracle.step(o, h0.astype(np.float64) + W, F, 1) - W
    hg = g.populations(deviation=True).double().cpu().numpy()
    err = np.abs(hg - ho) / ulp16(np.maximum(np.abs(hg), np.abs(ho)))
    assert err.max() <= 0.55
    g.check()
    g.close()
