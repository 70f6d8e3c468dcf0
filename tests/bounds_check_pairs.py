"""Node pairs and batches against the bounds-checked build (libclbm_bc.so), as
bounds_check_cases.py: the FP32 pair kernels (A/B, in place), the 16-bit pairs
of rows that are not staged, and every form of the batched step, each at sizes
just above those that select it. Run as a script by
test_gpu_bounds_pairs.py."""
import json
import os
import sys
import traceback

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, HERE)
sys.path.insert(0, os.path.dirname(HERE))

import torch  # noqa: E402

from gpu_common import dev, t  # noqa: E402
from paper_1801_04586_gb300 import Batch, Lattice, _capi, synthetic  # noqa: E402
from test_gpu_batch import DOMAINS, _single  # noqa: E402
from test_gpu_batch_forms import LARGE  # noqa: E402

RATES = dict(s2b=1.2, s3=1.1, s4=0.9)
PAIRS = "two adjacent nodes per thread"


def pairs(shape_xyz, walls, storage, pattern):
    nx, ny, nz = shape_xyz
    shape = (nz, ny, nx)
    outs = []
    for variant in (0, 1):
        g = Lattice(nx, ny, nz, 0.03, walls=walls, storage=storage, pattern=pattern, variant=variant, device=dev(),
                    **RATES)
        assert (g.step_form() == PAIRS) == (variant == 0), g.step_form()
        g.set_force_field(t(synthetic.gaussian_force(shape, 1e-4, seed=61)))
        g.init_equilibrium(None, t(synthetic.divfree_velocity(shape, seed=62, umax=0.03)))
        g.step(5)
        g.check()
        outs.append(g.populations(deviation=True).cpu())
        g.close()
    assert torch.equal(outs[0], outs[1])


def batch(domains, storage, pattern, threads):
    b = Batch(domains, storage=storage, device=dev(), pattern=pattern)
    b.set_tile(threads)
    b.init_equilibrium()
    b.step(5, Batch.DIRECT)
    b.check()
    for k, d in enumerate(domains):
        assert torch.equal(b.populations(k, deviation=True).cpu(), _single(d, 5, storage)), f"domain {k}"
    b.close()


CASES = [(pairs, (s, w, st, p)) for s, w, st, p in [
    ((150, 28, 24), 0, "f32", "ab"),   # even rows: aligned pairs
    ((150, 28, 24), 7, "f32", "ab"),
    ((151, 28, 24), 0, "f32", "ab"),   # odd rows
    ((151, 28, 24), 7, "f32", "ab"),
    ((150, 28, 24), 0, "f32", "aa"),
    ((150, 28, 24), 7, "f32", "aa"),
    ((75, 55, 27), 0, "f32", "aa"),    # an odd number of nodes
    ((75, 55, 27), 7, "f32", "aa"),
    ((3, 200, 167), 3, "f32", "aa"),
    ((150, 28, 24), 7, "f16", "ab"),   # rows of no multiple of 16 bytes
    ((151, 28, 24), 0, "f16sr", "ab"),
    ((151, 28, 24), 7, "bf16sr", "ab"),
]] + [(batch, (d, st, p, n)) for d, st, p, n in [
    (LARGE, "f32", "ab", 128), (LARGE, "f32", "ab", 256), (LARGE, "f32", "ab", 512),
    (LARGE, "f16", "ab", 128), (LARGE, "bf16", "ab", 512), (LARGE, "f16", "aa", 128),
    (DOMAINS, "f32", "ab", 128), (DOMAINS, "f16", "ab", 96), (DOMAINS, "f32", "aa", 128),
]]


def main():
    assert os.environ.get("CLBM_LIBRARY") == "bounds_check"
    assert _capi.lib()._name.endswith("libclbm_bc.so")
    failed = 0
    for fn, args in CASES:
        name = {"case": fn.__name__, "args": str(args[-3:])}
        try:
            fn(*args)
            print(json.dumps({**name, "ok": True}), flush=True)
        except Exception:
            failed += 1
            print(json.dumps({**name, "ok": False, "error": traceback.format_exc()[-800:]}), flush=True)
    return 1 if failed else 0


if __name__ == "__main__":
    sys.exit(main())
