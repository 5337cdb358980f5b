"""The depth sort's paths around its bucket sort, bit-exact against the oracle's
lists: list lengths at its limits (128, 1,024), depths spread, all equal (every
key in one bucket: the chunk path decides by index), crowded at one depth with
a few far away, and at most / more than the crowding limit equal.
"""
import numpy as np
import pytest

from tests._scenes import ident_cam, make_scene
from tests.gpu_util import GpuRun
from tests.test_gpu_binning import _check_lists

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [31, 128, 129, 300, 1023, 1024, 1025])
@pytest.mark.parametrize("depths", ["spread", "equal", "crowd", "32 equal", "33 equal"])
def test_lists_of_one_tile(n, depths):
    rng = np.random.default_rng(n)
    z = rng.uniform(1.0, 4.0, n)
    if depths == "equal":
        z[:] = 2.0
    elif depths == "crowd":
        z[:] = 2.0 + rng.uniform(0, 1e-4, n)
        z[rng.integers(0, n, 3)] = 60.0
    elif depths.endswith("equal"):
        z[rng.permutation(n)[:int(depths[:2])]] = 2.0
    cam = ident_cam(W=16, H=16, f=16.0)
    means = np.stack([rng.uniform(-0.2, 0.2, n) * z, rng.uniform(-0.2, 0.2, n) * z, z], 1)
    sc = make_scene(means, np.full((n, 2), 0.02), rng.normal(size=(n, 4)), rng.uniform(0.2, 0.9, n))
    run = GpuRun(sc, [cam], K=4, cap=1 << 12, render=False)
    _check_lists(run, sc, [cam], 16, "accu")
