"""The tile kernel's culling by 4x4 blocks and its grouped blend where they
can go wrong: needles at every angle (thin level sets between pixel centres,
chords of nearly flat conics), splats from far below a pixel to far above the
image, ragged image edges, list lengths around a group and a sub-batch, and
colours that are not finite."""
import numpy as np
import pytest

import oracle
import paper_2311_17089_gb300 as msgs
from paper_2311_17089_gb300 import inputs

from gpu_util import assert_image_close, gpu_frame, require_cuda

pytestmark = pytest.mark.gpu


def scene(n, seed, log_scale):
    sc = inputs.single_level_scene(n=n, seed=seed)
    sc.log_scale = np.asarray(log_scale, np.float32)
    return sc


def needle_scales(rng, n):
    ls = rng.uniform(-8.0, -6.0, (n, 3))
    ls[np.arange(n), rng.integers(0, 3, n)] = rng.uniform(-2.0, 2.5, n)
    return ls


SCALES = {
    "needles": needle_scales,
    "discs": lambda rng, n: np.where(rng.random((n, 3)) < 0.33, -8.0, rng.uniform(-3.0, 0.5, (n, 3))),
    "dots": lambda rng, n: rng.uniform(-9.0, -6.0, (n, 3)),
    "sheets": lambda rng, n: rng.uniform(0.5, 3.0, (n, 3)),
}


@pytest.mark.parametrize("kind", sorted(SCALES))
@pytest.mark.parametrize("wh", [(256, 192), (131, 77)])
def test_shapes(kind, wh):
    require_cuda()
    n = 300 if kind == "sheets" else 2500
    sc = scene(n, 7, SCALES[kind](np.random.default_rng(13), n))
    sc.opacity = np.random.default_rng(5).uniform(0.01, 0.6, n).astype(np.float32)
    cam = inputs.config1_camera(*wh)
    # against the group kernel, which evaluates every list entry at every
    # pixel with the same FP32 alpha; the transmittances are products of the
    # same factors in another order, so relatively within 2 L 2^-24 for lists
    # of L.  (Not the oracle: its FP64 power of a needle's FP32 conic is up to
    # 1e-3 in colour away from any FP32 evaluation.)
    g = gpu_frame(sc, cam, "all_levels", strategy="tile")
    r = gpu_frame(sc, cam, "all_levels", strategy="group8")
    longest = int((g["ranges"][:, 1] - g["ranges"][:, 0]).max())
    assert np.abs(g["image"] - r["image"]).max() <= 2 * longest * 2.0 ** -24
    assert np.abs(g["final_t"] - r["final_t"]).max() <= 2 * longest * 2.0 ** -24
    np.testing.assert_array_equal(g["n_contrib"], r["n_contrib"])
    np.testing.assert_array_equal(g["n_eval"], r["n_eval"])


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 8, 127, 128, 129, 131, 132, 133, 260])
def test_list_lengths(n):
    """One tile, every Gaussian over all of it: lists of n."""
    require_cuda()
    sc = scene(n, n, np.full((n, 3), 0.3))
    sc.opacity = np.full(n, 0.02, np.float32)
    cam = inputs.config1_camera(16, 16)
    assert_image_close(gpu_frame(sc, cam, "all_levels", strategy="tile"),
                       oracle.render(sc, cam, "all_levels"))


def test_colours_not_finite():
    require_cuda()
    n = 400
    sc = scene(n, 3, np.random.default_rng(1).uniform(-4.5, -2.5, (n, 3)))
    sc.color[5] = np.inf
    sc.color[77, 1] = np.nan
    cam = inputs.config1_camera(96, 80)
    g = gpu_frame(sc, cam, "all_levels", strategy="tile")
    clean = sc.copy()
    clean.color[5] = clean.color[77] = 0.5
    o = oracle.render(clean, cam, "all_levels")
    # which pixels blend one of the two, from frames in which they alone glow
    touched = np.zeros((cam.height, cam.width), bool)
    for i in (5, 77):
        lit = clean.copy()
        lit.color[i] = 1.5
        touched |= np.abs(oracle.render(lit, cam, "all_levels")["image"] - o["image"]).max(0) > 0
    finite = np.isfinite(g["image"]).all(0)
    assert touched.any() and not touched.all()
    sure = o["flags"] == 0
    np.testing.assert_array_equal(finite[sure], ~touched[sure])
    ok = sure & ~touched
    assert np.abs(g["image"] - o["image"])[:, ok].max() <= 2e-4
    np.testing.assert_array_equal(g["n_contrib"][sure], o["n_contrib"][sure])
