"""Exact ties in the Top-K set: which of several equal smallest weights leaves depends
on K alone, not on the outputs that are asked for.  Up to 16 entries it is the one that
an insertion chain carries off the end (each larger weight moves the ones behind it on, an equal
one stays in its slot), beyond 16 the latest.  A plain frame, a frame with sensor outputs and one
with the low-pass filter select the same surfels, on a pixel whose weights are exact in
binary32 and mostly equal.
"""
import numpy as np
import pytest
import torch

from tests._scenes import ident_cam, make_scene
from tests.gpu_util import GpuRun

pytestmark = pytest.mark.gpu


def _tied(K, seed):
    """4 K surfels facing the camera, all centred on one pixel's ray, whose weights there are
    1 to 3 times c by what the binary32 recurrence T (1 - alpha) makes of them: the scene and the weights."""
    rng = np.random.default_rng(seed)
    n = 4 * K
    c = np.float32(1.0 / 256.0)
    o, w, T = [], [], np.float32(1.0)
    for m in rng.choice([1, 1, 1, 2, 2, 3], n):
        a = np.float32(c * np.float32(m) / T)
        o.append(a)
        w.append(np.float32(a * T))
        T = np.float32(T * np.float32(np.float32(1.0) - a))
    means = np.stack([np.zeros(n), np.zeros(n), 2.0 + 0.01 * np.arange(n)], 1)
    quats = np.tile([1.0, 0.0, 0.0, 0.0], (n, 1))
    sc = make_scene(means, np.full((n, 2), 0.2), quats, np.array(o), C=8)
    cam = ident_cam(W=32, H=32, f=32.0)
    cam.cx = cam.cy = 16.5
    return sc, cam, w


def _chain(w, K):
    sel = [(np.float32(-1.0), -1)] * K
    for x in zip(w, range(len(w))):
        if x[0] > sel[-1][0]:
            for k in range(K):
                if x[0] > sel[k][0]:
                    x, sel[k] = sel[k], x
    return sorted(i for _, i in sel)


def _latest(w, K):
    sel = list(zip(w[:K], range(K)))
    for x in zip(w[K:], range(K, len(w))):
        low = min(s[0] for s in sel)
        if x[0] > low:
            sel.remove(max(s for s in sel if s[0] == low))
            sel.append(x)
    return sorted(i for _, i in sel)


@pytest.mark.parametrize("seed", range(3))
@pytest.mark.parametrize("K", [8, 9, 12, 16, 17, 24, 32])
def test_the_same_surfel_leaves_whatever_the_outputs(K, seed):
    sc, cam, w = _tied(K, seed)
    chain, latest = _chain(w, K), _latest(w, K)
    if K >= 12:
        assert chain != latest  # the weights tell the two rules apart
    want = chain if K <= 16 else latest
    run = GpuRun(sc, [cam], K=K, alpha_min=1.0 / 1024.0, T_min=1e-6)
    np.testing.assert_array_equal(run.view(0)["ids"][16, 16], want)
    np.testing.assert_array_equal(run.view(0)["w"][16, 16], [w[i] for i in want])
    plain = run.view(0)["ids"]
    F, rgb, T, ids = run.frame.new_outputs()
    depth = torch.empty(run.frame.total_pix, device="cuda")
    run.frame.render_forward_aux(run.rgb, run.feats, F, rgb, T, ids, depth)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(ids.cpu().numpy().reshape(plain.shape), plain)
    soft = GpuRun(sc, [cam], K=K, alpha_min=1.0 / 1024.0, T_min=1e-6, lowpass=True)
    np.testing.assert_array_equal(soft.view(0)["ids"][16, 16], want)
