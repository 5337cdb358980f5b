"""GPU parity of the backward replay that also takes the feature gradients (few
channels, K > 8), against the oracle's FP64 analytic gradients: channels at and
beside the instances' 16 and 32, tile sizes, the persistent schedule, more
contributors than slots; the general path is the one K = 8 takes.  Tolerances as in
test_gpu_feat_grad_shapes.  And a pixel with an infinite dL/dF reaches only the
surfels that it selected.
"""
import numpy as np
import pytest
import torch

from paper_2604_10951_gb300 import scenes
from tests.gpu_util import GpuRun
from tests.test_gpu_backward import _gpu_backward
from tests.test_gpu_feat_grad_shapes import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,dtype,K,ts", [
    (4, torch.float32, 9, 16), (12, torch.float32, 16, 8), (16, torch.float32, 24, 16), (20, torch.float32, 10, 32),
    (32, torch.float32, 32, 16), (36, torch.float32, 9, 16), (8, torch.bfloat16, 9, 16), (16, torch.bfloat16, 17, 32),
    (24, torch.bfloat16, 12, 8), (32, torch.bfloat16, 24, 16), (16, torch.float32, 8, 16),
    (20, torch.float32, 9, 32), (36, torch.float32, 8, 32), (64, torch.float32, 16, 32), (68, torch.float32, 17, 32),
    (128, torch.float32, 32, 32), (40, torch.bfloat16, 32, 32), (64, torch.bfloat16, 24, 32), (64, torch.float32, 3, 32)])
def test_feature_gradients_in_the_replay(C, dtype, K, ts):
    sc, cam = scenes.tiny_scene(seed=51 + C, n=1200, C=C)
    sc.opacities *= np.float32(0.3)
    _check(sc, cam, K, dtype, tile_size=ts, seed=C + K)


@pytest.mark.parametrize("C,dtype,ts,W,H", [(12, torch.float32, 16, 605, 413), (16, torch.bfloat16, 8, 604, 415),
                                           (16, torch.float32, 32, 640, 410)])
def test_two_blocks_per_warp(C, dtype, ts, W, H):
    """Images large enough for the warps with two blocks; ragged below and to the right."""
    sc, cam = scenes.tiny_scene(seed=9, n=600, C=C)
    sc.opacities *= np.float32(0.4)
    s = W / cam.width
    big = scenes.Camera(cam.fx * s, cam.fy * s, W / 2, H / 2, W, H, cam.viewmat)
    assert -(-W // ts) * -(-H // ts) * (ts * ts // 32) >= 48 * torch.cuda.get_device_properties(0).multi_processor_count
    _check(sc, big, 12, dtype, tile_size=ts, seed=C)


@pytest.mark.parametrize("C", [16, 32, 64])
def test_an_infinite_gradient_stays_with_its_surfels(C):
    sc, cam = scenes.tiny_scene(seed=5, n=1200, C=C)
    run = GpuRun(sc, [cam], K=12, tile_size=32, feat_dtype=torch.float32)
    ids = np.asarray(run.view(0)["ids"])
    H, W = ids.shape[:2]
    gF = np.ones((H, W, C))
    y, x = np.argwhere((ids >= 0).any(-1))[0]
    gF[y, x] = np.inf
    g = _gpu_backward(run, gF, np.zeros((H, W, 3)), np.zeros((H, W)), feat_dtype=torch.float32)
    bad = ~np.isfinite(np.asarray(g["feat"])).all(-1)
    hit = np.unique(ids[y, x][ids[y, x] >= 0])
    assert np.array_equal(np.flatnonzero(bad), hit)
