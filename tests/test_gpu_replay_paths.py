"""The backward replays at the sizes where their dispatch takes them: products shared by
a warp's lanes with tiles of 8 and 16, in both types, on an image with enough blocks an SM (ragged to the
right and below); the feature rows written in the second stream after the replay; a
warp's two blocks, each with the surfels of its own warp mask; a dL/dF that is not finite; and the
feature kernel where its shared memory with the static part just exceeds 48 KB.
Gradients against the oracle's FP64 analytic ones, tolerances as in test_gpu_feat_grad_shapes.py;
the second stream against the same call captured on one stream, tolerance as in
test_gpu_autograd_graph.py (BF16 storage is not used).
"""
import numpy as np
import pytest
import torch

from paper_2604_10951_gb300 import _lib as L
from paper_2604_10951_gb300 import scenes
from paper_2604_10951_gb300.raster import Frame, make_params
from tests._scenes import ident_cam, make_scene
from tests.gpu_util import GpuRun, dev
from tests.test_gpu_backward import _gpu_backward
from tests.test_gpu_feat_grad_shapes import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,dtype,K,ts", [
    (64, torch.float32, 24, 8), (20, torch.float32, 16, 8), (64, torch.bfloat16, 24, 8), (40, torch.bfloat16, 32, 16),
    (64, torch.bfloat16, 18, 16), (128, torch.float32, 16, 16), (68, torch.float32, 20, 8), (64, torch.float32, 8, 16)])
def test_products_on_tiles_of_8_and_16(C, dtype, K, ts):
    W, H = 321, 243
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert -(-W // ts) * -(-H // ts) * (ts * ts // 32) >= 8 * sms  # the most that any of these asks for
    sc, cam = scenes.tiny_scene(seed=61 + C, n=800, C=C)
    sc.opacities *= np.float32(0.3)
    s = W / cam.width
    _check(sc, scenes.Camera(cam.fx * s, cam.fy * s, W / 2, H / 2, W, H, cam.viewmat), K, dtype, tile_size=ts, seed=C + K)


@pytest.mark.parametrize("N,C,K", [(200_000, 64, 0), (800_000, 16, 12), (400_000, 32, 10)])
def test_feature_rows_in_the_second_stream_after_the_replay(N, C, K):
    assert N * C * 4 >= 48 << 20  # where an eager call takes the second stream
    sc = scenes.room_scene(n=N, C=C, seed=4)
    cam = scenes.circle_poses(1, 320, 240, 262.5)[0]
    ins = [dev(x) for x in (sc.means, sc.scales, sc.quats, sc.opacities, sc.rgb, sc.feats)]
    fr = Frame([cam], sc.n, make_params(C=C, K=K), pair_capacity=1 << 21)
    fr.bin_and_sort(*ins[:4])
    F, rgb, T, ids = fr.new_outputs()
    fr.render_forward(ins[4], ins[5], F, rgb, T, ids)
    g = torch.Generator(device="cuda").manual_seed(1)
    dF, drgb = torch.randn(F.shape, generator=g, device="cuda"), torch.randn(rgb.shape, generator=g, device="cuda")
    grads = [torch.empty_like(x) for x in ins]

    def back():
        fr.render_backward(*ins, T, dF, drgb, None, *grads)

    back()
    eager = []
    for _ in range(3):
        for x in grads:
            x.fill_(7.0)
        back()
        eager.append([x.clone() for x in grads])  # read behind the call, on its stream
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        back()
    for x in grads:
        x.fill_(7.0)
    graph.replay()
    torch.cuda.synchronize()
    assert fr.read_status()[0] == 0
    for run in eager:
        for a, b in zip(run, grads):
            scale = b.abs().max().item()
            assert scale > 0 and (a - b).abs().max().item() <= 1e-5 * scale


def test_a_block_without_its_mask_bit_is_not_replayed():
    """Two blocks per warp: a surfel kept out of the upper block by the warp mask, as the
    forward leaves it out there, gets nothing from that block's pixels in the replay either."""
    W, H, K = 605, 413, 12
    means = np.array([[0.0, 0.0, 2.0], [0.0, 0.0, 3.0]])
    sc = make_scene(means, np.full((2, 2), 30.0), np.tile([1.0, 0.0, 0.0, 0.0], (2, 1)), np.array([0.5, 0.5]), C=8)
    run = GpuRun(sc, [ident_cam(W=W, H=H, f=500.0)], K=K, render=False)
    assert run.frame.region(L.REG_RANGES).numel() // 8 * 8 >= 48 * torch.cuda.get_device_properties(0).multi_processor_count
    assert run.ranges()[0].tolist() == [0, 2] and run.lists()[0] == 0
    masks = run.frame.region(L.REG_MASK).view(torch.int32)
    assert masks[0].item() == 0xff and masks[1].item() == 0xff
    masks[0] = 0xfe  # tile (0, 0), block 0: without the nearer surfel
    run.F, run.rgb_out, run.T, run.ids = run.frame.new_outputs()
    run.frame.render_forward(run.rgb, run.feats, run.F, run.rgb_out, run.T, run.ids)
    ids = run.view(0)["ids"]
    assert ids[0, 0].tolist() == [1] + [-1] * (K - 1) and ids[4, 0].tolist() == [0, 1] + [-1] * (K - 2)
    gT = np.zeros((H, W))
    gT[0, 0] = 1.0
    g = _gpu_backward(run, np.zeros((H, W, 8)), np.zeros((H, W, 3)), gT)
    assert g["opac"][1] != 0.0 and g["opac"][0] == 0.0
    gT[4, 0] = 1.0
    g = _gpu_backward(run, np.zeros((H, W, 8)), np.zeros((H, W, 3)), gT)
    assert g["opac"][0] != 0.0


@pytest.mark.parametrize("C,ts", [(16, 16), (64, 16), (64, 8), (128, 32)])
def test_an_infinite_gradient_without_a_selection(C, ts):
    """Full accumulation: a pixel with an infinite dL/dF reaches the surfels that it met and no others."""
    sc, cam = scenes.tiny_scene(seed=5, n=1200, C=C)
    run = GpuRun(sc, [cam], K=0, tile_size=ts)
    H, W = run.view(0)["T"].shape
    zero = np.zeros((H, W, C))
    y, x = np.argwhere(run.view(0)["T"] < 0.9)[0]
    gF, one = zero.copy(), zero.copy()
    gF[y, x] = np.inf
    one[y, x] = 1.0
    met = np.abs(_gpu_backward(run, one, zero[..., :3], zero[..., 0])["feat"]).max(-1) > 0
    g = _gpu_backward(run, gF, zero[..., :3], zero[..., 0])
    assert met.any() and np.array_equal(~np.isfinite(g["feat"]).all(-1), met)


@pytest.mark.parametrize("C,dtype,K,ts", [(12, torch.float32, 5, 16), (48, torch.float32, 4, 8)])
def test_feature_kernel_just_above_48_kb(C, dtype, K, ts):
    sc, cam = scenes.tiny_scene(seed=71 + C, n=600, C=C)
    _check(sc, cam, K, dtype, tile_size=ts, seed=C)


@pytest.mark.parametrize("C,dtype,ts", [(64, torch.float32, 8), (64, torch.bfloat16, 16), (128, torch.float32, 16)])
def test_an_infinite_gradient_with_products_on_small_tiles(C, dtype, ts):
    """Top-K: only the surfels that the pixel selected."""
    W, H, K = 321, 243, 24
    sc, cam = scenes.tiny_scene(seed=5, n=1200, C=C)
    s = W / cam.width
    run = GpuRun(sc, [scenes.Camera(cam.fx * s, cam.fy * s, W / 2, H / 2, W, H, cam.viewmat)], K=K, tile_size=ts, feat_dtype=dtype)
    ids = run.view(0)["ids"]
    gF = np.ones((H, W, C))
    y, x = np.argwhere((ids >= 0).any(-1))[0]
    gF[y, x] = np.inf
    g = _gpu_backward(run, gF, np.zeros((H, W, 3)), np.zeros((H, W)), feat_dtype=dtype)
    assert np.array_equal(np.flatnonzero(~np.isfinite(g["feat"]).all(-1)), np.unique(ids[y, x][ids[y, x] >= 0]))
