"""The projection's cheap first cull drops only what the exact culls drop: tile
lists bit-exact against the oracle for surfels crowded at the frustum's edges,
of all sizes, nearly transparent and opaque, also with opacities above 1 (which
it must leave to the exact test), for off-centre and telephoto cameras, with
and without the low-pass filter, on both sides of its two launch shapes
(few items: 256 per CTA; many: 1024), and with the two and three times 1024
of still more.
"""
import numpy as np
import pytest

from paper_2604_10951_gb300 import scenes
from tests._scenes import ident_cam, make_scene
from tests.gpu_util import GpuRun
from tests.test_gpu_binning import _check_lists

pytestmark = pytest.mark.gpu


def _edge_scene(n, cam, seed):
    rng = np.random.default_rng(seed)
    z = np.exp(rng.uniform(np.log(0.05), np.log(50.0), n)) * rng.choice([1.0, 1.0, 1.0, -1.0], n)
    # image positions around the four edges, some far outside
    x = rng.choice([0.0, cam.width], n) + rng.normal(0, 0.1 * cam.width, n) * rng.choice([1.0, 10.0], n)
    y = rng.uniform(-0.2, 1.2, n) * cam.height
    swap = rng.random(n) < 0.5
    x, y = np.where(swap, rng.uniform(-0.2, 1.2, n) * cam.width, x), np.where(
        swap, rng.choice([0.0, cam.height], n) + rng.normal(0, 0.1 * cam.height, n), y)
    means = np.stack([(x - cam.cx) / cam.fx * z, (y - cam.cy) / cam.fy * z, z], 1)
    scales = np.exp(rng.normal(-3.0, 1.2, (n, 2)))
    opac = rng.choice([0.0039, 0.00393, 0.1, 0.9, 0.999999, 1.0, 1.5, 20.0], n)
    return make_scene(means, scales, rng.normal(size=(n, 4)), opac, C=4, seed=seed)


@pytest.mark.parametrize("lowpass", [0, 1])
@pytest.mark.parametrize("cam", [ident_cam(W=100, H=75, f=90.0), ident_cam(W=64, H=48, f=60.0, cx=900.0, cy=-300.0),
                                 ident_cam(W=33, H=17, f=4000.0), ident_cam(W=320, H=240, f=60.0, near=1.0)],
                         ids=["centred", "off-centre", "telephoto", "wide"])
def test_edge_surfels_binning_bit_exact(cam, lowpass):
    sc = _edge_scene(4000, cam, seed=lowpass + cam.width)
    run = GpuRun(sc, [cam], K=4, render=False, cap=1 << 21, lowpass=bool(lowpass))
    _check_lists(run, sc, [cam], 16, "accu", lowpass=lowpass)


def test_edge_surfels_many_items():
    cams = [ident_cam(W=48, H=48, f=50.0), ident_cam(W=64, H=32, f=40.0, cx=-20.0)]
    sc = _edge_scene(90_000, cams[0], seed=3)
    sc.scales *= np.float32(0.2)
    run = GpuRun(sc, cams, K=4, render=False, cap=1 << 23)
    _check_lists(run, sc, cams, 16, "accu")


@pytest.mark.parametrize("views", [8, 15])  # 672k and 1.26M items: two and three rounds per CTA
def test_edge_surfels_many_views(views):
    cams = [ident_cam(W=40 + v, H=30, f=40.0 + 2 * v, cx=20.0 * (v % 3), cy=15.0) for v in range(views)]
    sc = _edge_scene(84_001, cams[0], seed=4)
    sc.scales *= np.float32(0.05)
    run = GpuRun(sc, cams, K=4, render=False, cap=1 << 23)
    _check_lists(run, sc, cams, 16, "accu")
