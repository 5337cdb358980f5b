"""GPU parity of the full accumulation (K = 0) whose products a warp's lanes
share: channels at and beside 16, 32, 64 and 128, tile sizes, the persistent
schedule, and numbers of contributors beside the eight rows of a product; sensor
outputs and the label argmax with many channels; and a feature that is not finite,
which reaches the pixels that met its surfel and no others.  Tolerances as in
test_gpu_feat_grad_shapes.py.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_10951_gb300 import scenes
from tests._scenes import ident_cam, make_scene
from tests.gpu_util import GpuRun, dev
from tests.outcomes import oracle_ref
from tests.test_gpu_backward import _assert_close, _gpu_backward, _resolved, _upstream
from tests.test_gpu_render import _compare
from tests.test_gpu_sensors import _aux_run, _check, _ref

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,dtype,ts,sched", [
    (4, torch.float32, 8, "grid"), (16, torch.float32, 32, "persistent"), (20, torch.float32, 16, "grid"),
    (32, torch.bfloat16, 8, "grid"), (36, torch.float32, 16, "persistent"), (40, torch.bfloat16, 32, "grid"),
    (64, torch.float32, 8, "grid"), (68, torch.float32, 32, "persistent"), (128, torch.bfloat16, 8, "grid"),
    (128, torch.float32, 32, "grid")])
def test_full_accumulation(C, dtype, ts, sched):
    sc, _ = scenes.tiny_scene(seed=C, n=1500, C=C)
    cam = ident_cam(W=75, H=50, f=70.0)
    cam.viewmat[2, 3] = 3.0
    run = GpuRun(sc, [cam], K=0, tile_size=ts, feat_dtype=dtype, schedule=sched)
    feats = torch.as_tensor(sc.feats).to(dtype).double().numpy()
    p = O.make_params(K=0, tile_size=ts)
    half = dtype == torch.bfloat16
    ref = _resolved(run, sc, cam, p, tol=2e-2 if half else 1e-4, feats=feats)
    got = run.view(0)
    ok = ~ref["unmatched"]
    tol = 1e-4 * np.abs(feats).max() + (np.abs(ref["F"]) * 2.0 ** -8 if half else 0.0)
    assert (np.abs(got["F"] - ref["F"]) <= tol)[ok].all()
    gF, grgb, gT = _upstream(ref, C, seed=C)
    gF = torch.as_tensor(gF).to(dtype).double().numpy()
    g_ref = O.render_backward(sc, cam, p, gF, grgb, gT, feats=feats, binned=ref["binned"], flip=ref["flip"])
    g = _gpu_backward(run, gF, grgb, gT, feat_dtype=dtype)
    _assert_close(g, g_ref, names=("means", "scales", "quats", "opac", "rgb"))
    if half:
        _assert_close(g, g_ref, rel=8e-3, floor=1e-4, names=("feat",))
    else:
        _assert_close(g, g_ref, names=("feat",))


def _stack(n, C, seed=0):
    """n faint surfels behind one another, each over the whole 32 x 32 image."""
    rng = np.random.default_rng(seed)
    z = np.linspace(2.0, 3.0, n)
    means = np.stack([np.zeros(n), np.zeros(n), z], axis=1)
    return make_scene(means, np.full((n, 2), 4.0), np.tile([1.0, 0.0, 0.0, 0.0], (n, 1)), rng.uniform(0.02, 0.05, n), C=C), ident_cam()


@pytest.mark.parametrize("n", [1, 7, 8, 9, 16, 17, 31, 32, 33, 65])
def test_numbers_of_contributors(n):
    sc, cam = _stack(n, 64)
    run = GpuRun(sc, [cam], K=0)
    ref, S = oracle_ref(sc, cam, O.make_params(K=0))
    assert (ref["ncontrib"] == n).all()
    _compare(run.view(0), ref, S, 1e-4, 0)


@pytest.mark.parametrize("C", [16, 64, 128])
def test_feature_that_is_not_finite(C):
    sc, cam = scenes.tiny_scene(seed=3, n=300, C=C)
    sc.feats[100, 3] = np.inf
    sc.feats[200, C - 1] = np.nan
    F = GpuRun(sc, [cam], K=0).view(0)["F"]
    sc2, _ = scenes.tiny_scene(seed=3, n=300, C=C)
    sc2.feats[100, 3] = sc2.feats[200, C - 1] = 0.0
    zero = GpuRun(sc2, [cam], K=0).view(0)["F"]
    sc2.feats[:] = 0.0
    sc2.feats[100, 3] = sc2.feats[200, C - 1] = 1.0
    met = GpuRun(sc2, [cam], K=0).view(0)["F"] != 0  # where those two values arrive
    assert met[..., 3].any() and met[..., C - 1].any()
    assert np.array_equal(~np.isfinite(F), met)
    assert np.array_equal(F[~met], zero[~met])


def test_sensor_outputs_and_labels_with_many_channels():
    C = 96
    sc, cam = scenes.tiny_scene(seed=8, n=1000, C=C)
    run = GpuRun(sc, [cam], K=0)
    _check(run, _aux_run(run), _ref(run, sc, cam, O.make_params(K=0)))
    fr, n = run.frame, run.frame.total_pix
    F, rgb, T, ids = fr.new_outputs()
    label = torch.full((n,), -7, device="cuda", dtype=torch.int32)
    fr.render_forward_aux(run.rgb, run.feats, F, rgb, T, ids, label=label)
    torch.cuda.synchronize()
    want = F.cpu().numpy().argmax(-1)
    want[(T == 1.0).cpu().numpy()] = -1
    assert np.array_equal(label.cpu().numpy(), want)
