"""The 3D build for many active regions per SM (five resident 32x8x4 regions)
on a grid sized for the GPU it runs on: both sides of the bound, the same
results as the generic kernel."""
import os
import re

import numpy as np
import pytest

from gen import grids
from helpers import gpu_solve, opts
from paper_1109_1146_gb300 import build

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _bound():
    with open(os.path.join(build.CSRC, "ard_discharge3d.cu")) as f:
        per_sm = int(re.search(r"constexpr int kMany3d = (\d+);", f.read()).group(1))
    return per_sm * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("above", [0, 1])
def test_both_sides_of_the_bound(above):
    # layers of 8 x 32 regions, the last row and the last layer of them ragged; every region starts active
    layers = _bound() // 256 + above
    inst = grids.random_grid((256, 250, 4 * layers - 2), 6, 12, cmax=9, tmax=120, p_zero=0.5)
    regions = 8 * 32 * layers
    assert (regions > _bound()) == bool(above)
    got, ref = gpu_solve(inst), gpu_solve(inst, opts=opts(kernel_variant=1))
    assert got["flow"] == ref["flow"]
    for k in ("smin", "smax", "res", "tres", "exc", "lab"):
        assert np.array_equal(got[k], ref[k]), k
    assert got["stats"].rounds == ref["stats"].rounds
