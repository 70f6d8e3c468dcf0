"""The in-place batch's grid (csrc/batch.cu)."""
import pytest
import torch

from gpu_common import dev
from paper_1801_04586_gb300 import Batch

pytestmark = pytest.mark.gpu


def test_in_place_grid_follows_its_own_kernel():
    """The in-place FP16 even kind runs three blocks of 256 threads per SM (its
    registers), whatever the A/B kernel of the batch holds."""
    sms = torch.cuda.get_device_properties(dev()).multi_processor_count
    b = Batch([dict(nx=64, ny=64, nz=64, walls=4, nu=0.05)], storage="f16", device=dev(), pattern="aa")
    b.set_tile(256)
    i = b.info()
    assert i["ntiles"] == 1024 and i["grid"] == 3 * sms
    b.close()
