"""GPU parity of the Top-K forward for K > 8 (register sets to 16, then shared memory):
scenes of faint surfels, where most pixels meet more than K contributors and
slots are refilled, over K at and beside the slot groups of eight, the tile
sizes, a ragged image and the variants; and the tie rule (equal weights: the
earlier surfel stays), on a pixel whose weights are exact in binary32.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_10951_gb300 import scenes
from tests._scenes import ident_cam, make_scene
from tests.gpu_util import GpuRun
from tests.outcomes import oracle_ref
from tests.test_gpu_render import _compare

pytestmark = pytest.mark.gpu


def _faint(n, C, seed, scale=0.2):
    sc, cam = scenes.tiny_scene(seed=seed, n=n, C=C)
    sc.opacities *= np.float32(scale)
    return sc, cam


@pytest.mark.parametrize("K,ts,stop,kw", [
    (9, 16, "tmin", {}), (16, 8, "tmin", {}), (17, 16, "exact_topk", {}), (24, 32, "tmin", {}),
    (31, 16, "exact_topk", {}), (32, 32, "tmin", {}), (32, 8, "exact_topk", {"schedule": "persistent"}),
    (12, 16, "tmin", {"select": "front"}), (20, 16, "tmin", {"renorm": True})])
def test_more_contributors_than_slots(K, ts, stop, kw):
    sc, _ = _faint(6000, 12, seed=K)
    cam = ident_cam(W=100, H=75, f=90.0)
    cam.viewmat[2, 3] = 3.0
    run = GpuRun(sc, [cam], K=K, tile_size=ts, stop_rule=stop, cap=1 << 20, **kw)
    p = O.make_params(K=K, tile_size=ts, stop_rule=O.EXACT_TOPK if stop == "exact_topk" else O.TMIN,
                      select=1 if kw.get("select") == "front" else 0, renorm=int(kw.get("renorm", False)))
    ref, S = oracle_ref(sc, cam, p)
    assert (ref["ncontrib"] > K).mean() > 0.3
    _compare(run.view(0), ref, S, 1e-4, K)


@pytest.mark.parametrize("K", [17, 24, 32])
def test_equal_weights_keep_the_earlier_surfel(K):
    """Surfels facing the camera, all centred on one pixel's ray, so that alpha is the
    opacity itself there: the weights are what the binary32 recurrence T (1 - alpha)
    gives, with many equal ones, and later ones that push the latest equals out."""
    n = 3 * K
    c = np.float32(1.0 / 128.0)
    o, T = [], np.float32(1.0)
    for i in range(n):
        a = np.float32(c / T) if i % 7 != 6 else np.float32(2 * c / T)
        o.append(a)
        T = np.float32(T * np.float32(np.float32(1.0) - a))
    means = np.stack([np.zeros(n), np.zeros(n), 2.0 + 0.01 * np.arange(n)], 1)
    quats = np.tile([1.0, 0.0, 0.0, 0.0], (n, 1))
    sc = make_scene(means, np.full((n, 2), 0.2), quats, np.array(o), C=8)
    cam = ident_cam(W=32, H=32, f=32.0)
    cam.cx = cam.cy = 16.5
    run = GpuRun(sc, [cam], K=K)
    sel, T, equal = [], np.float32(1.0), 0
    for i, a in enumerate(np.asarray(sc.opacities, np.float32)):
        w = np.float32(a * T)
        T = np.float32(T * np.float32(np.float32(1.0) - a))
        if len(sel) < K:
            sel.append((w, i))
            continue
        low = min(s[0] for s in sel)
        if w > low:
            equal += sum(s[0] == low for s in sel) > 1
            sel.remove(max(s for s in sel if s[0] == low))
            sel.append((w, i))
    assert equal > 0
    v = run.view(0)
    np.testing.assert_array_equal(v["ids"][16, 16], sorted(i for _, i in sel))
    np.testing.assert_array_equal(v["w"][16, 16], [w for w, _ in sorted(sel, key=lambda s: s[1])])


@pytest.mark.parametrize("K", [4, 8, 9, 16])
def test_equal_weights_as_an_insertion_chain(K):
    """Surfels facing the camera, all centred on one pixel's ray, so that alpha is the
    opacity itself there: the weights are what the binary32 recurrence T (1 - alpha)
    gives, with many equal ones, and later ones that push one of the equals out: with the set in
    registers (K <= 16) the one that an insertion chain (each larger weight moves the ones behind it on, an equal one
    stays in its slot) carries off the end."""
    n = 3 * K
    c = np.float32(1.0 / 128.0)
    o, T = [], np.float32(1.0)
    for i in range(n):
        a = np.float32(c / T) if i % 7 != 6 else np.float32(2 * c / T)
        o.append(a)
        T = np.float32(T * np.float32(np.float32(1.0) - a))
    means = np.stack([np.zeros(n), np.zeros(n), 2.0 + 0.01 * np.arange(n)], 1)
    quats = np.tile([1.0, 0.0, 0.0, 0.0], (n, 1))
    sc = make_scene(means, np.full((n, 2), 0.2), quats, np.array(o), C=8)
    cam = ident_cam(W=32, H=32, f=32.0)
    cam.cx = cam.cy = 16.5
    run = GpuRun(sc, [cam], K=K)
    sel, T, equal = [], np.float32(1.0), 0
    for i, a in enumerate(np.asarray(sc.opacities, np.float32)):
        w = np.float32(a * T)
        T = np.float32(T * np.float32(np.float32(1.0) - a))
        if len(sel) == K and w > sel[-1][0]:
            equal += sel[-1][0] == sel[-2][0]
        x, sel = (w, i), sel + [(np.float32(-1.0), -1)] * (len(sel) < K)
        for k in range(len(sel)):
            if x[0] > sel[k][0]:
                x, sel[k] = sel[k], x
    assert equal > 0
    v = run.view(0)
    np.testing.assert_array_equal(v["ids"][16, 16], sorted(i for _, i in sel))
    np.testing.assert_array_equal(v["w"][16, 16], [w for w, _ in sorted(sel, key=lambda s: s[1])])
