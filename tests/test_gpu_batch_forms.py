"""The forms of the batched step (csrc/batch.cu, form_for): which one a batch's
size and tile select, and that every one of them stores the bits of each
lattice stepped alone. Small batches step one node per thread, larger ones
pairs of adjacent nodes, one block per tile up to a tile of 256 (FP32) or 128
(16-bit) threads and walked by resident blocks above it."""
import pytest
import torch

from gpu_common import dev
from paper_1801_04586_gb300 import Batch
from test_gpu_batch import DOMAINS, _single

pytestmark = pytest.mark.gpu

# 330,000 nodes: above the 280,000 from which every storage format takes pairs
# (152 SMs). Rows of odd and even length, walls on every axis, a domain of two
# nodes per row and one whose rows are longer than a tile.
LARGE = [
    dict(nx=61, ny=40, nz=37, walls=7, nu=0.05, fx=1e-5, fz=2e-6),
    dict(nx=64, ny=50, nz=41, walls=1, nu=0.02, s2b=1.2, s3=1.1, fy=1e-6),
    dict(nx=2, ny=90, nz=80, walls=3, nu=0.1, s4=0.8, fx=-2e-6, fz=4e-6),
    dict(nx=701, ny=9, nz=14, walls=6, nu=0.008, fx=5e-6),
    dict(nx=1, ny=70, nz=11, walls=4, nu=0.03, fx=2e-6),
]


def ntiles(doms, threads, pairs):
    rows = [((d["nx"] + 1) // 2 if pairs else d["nx"]) * d["ny"] * d["nz"] for d in doms]
    return sum(-(-r // threads) for r in rows)


@pytest.mark.parametrize("storage,pattern", [("f32", "ab"), ("f16", "ab"), ("bf16", "ab"), ("f16", "aa")])
def test_small_batches_step_one_node_per_thread_in_small_tiles(storage, pattern):
    b = Batch(DOMAINS, storage=storage, device=dev(), pattern=pattern)
    i = b.info()
    assert i["threads"] == 128 and i["ntiles"] == ntiles(DOMAINS, 128, False)
    b.close()


@pytest.mark.parametrize("storage,threads,pairs", [("f32", 32, True), ("f32", 128, True), ("f32", 160, True),
                                                   ("f32", 256, True), ("f32", 288, False), ("f32", 512, False)]
                         + [(s, n, True) for s in ("f16", "bf16") for n in (32, 96, 128, 160, 512)])
def test_forms_of_a_large_batch_equal_single_lattices(storage, threads, pairs):
    b = Batch(LARGE, storage=storage, device=dev())
    assert b.info()["threads"] == 128
    b.set_tile(threads)
    assert b.info()["ntiles"] == ntiles(LARGE, threads, pairs)
    b.init_equilibrium()
    b.step(19, Batch.GRAPH)
    b.check()
    for k, d in enumerate(LARGE):
        assert torch.equal(b.populations(k, deviation=True).cpu(), _single(d, 19, storage)), f"domain {k}"
    b.close()


@pytest.mark.parametrize("storage,pattern", [("f16", "ab"), ("f16", "aa")])
@pytest.mark.parametrize("threads", [64, 512])
def test_forms_of_a_small_batch_equal_single_lattices(storage, pattern, threads):
    b = Batch(DOMAINS, storage=storage, device=dev(), pattern=pattern)
    b.set_tile(threads)
    assert b.info()["ntiles"] == ntiles(DOMAINS, threads, False)
    b.init_equilibrium()
    b.step(19, Batch.GRAPH)
    b.check()
    for k, d in enumerate(DOMAINS):
        assert torch.equal(b.populations(k, deviation=True).cpu(), _single(d, 19, storage)), f"domain {k}"
    b.close()


def test_in_place_grid_follows_its_own_kernel():
    """The in-place FP16 even kind runs three blocks of 256 threads per SM (its
    registers), whatever the A/B kernel of the batch holds."""
    sms = torch.cuda.get_device_properties(dev()).multi_processor_count
    b = Batch([dict(nx=64, ny=64, nz=64, walls=4, nu=0.05)], storage="f16", device=dev(), pattern="aa")
    b.set_tile(256)
    i = b.info()
    assert i["ntiles"] == 1024 and i["grid"] == 3 * sms
    b.close()
