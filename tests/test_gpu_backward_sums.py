"""How exactly the raster backward forms its sums: the second moments of
splats smaller than a pixel, and the colour behind a record where almost
nothing is left behind it.  Scenes whose centres project exactly in FP32, so
that the gradients' own rounding is what is seen (u = 2^-24)."""
import numpy as np
import pytest

import oracle
from paper_2311_17089_gb300 import inputs

from test_gpu_backward import gpu_grads

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


def axis_camera(w, h, f):
    """At the origin, looking along +z; the principal point is the image's centre."""
    return inputs.Camera(np.eye(3, dtype=np.float32), np.zeros(3, np.float32),
                         np.zeros(3, np.float32), f, f, w / 2, h / 2, w, h)


def rgb_scene(mean, log_scale, opacity, color):
    n = len(mean)
    quat = np.tile(np.array([1, 0, 0, 0], np.float32), (n, 1))
    return inputs.Scene(np.asarray(mean, np.float32), np.asarray(log_scale, np.float32), quat,
                        np.asarray(opacity, np.float32), np.asarray(color, np.float32),
                        np.ones(n, np.uint8), 1, -1, np.zeros(n, np.float32),
                        np.full(n, np.inf, np.float32))


@pytest.mark.parametrize("sigma", [0.02, 0.1, 0.4])
@pytest.mark.parametrize("seed", [0, 1])
def test_splats_below_a_pixel(sigma, seed):
    """One splat per 8x8 pixels, none overlapping, with loss weights and
    colours above zero: a log-scale's gradient is a sum of second moments of
    one sign.  About 40 roundings of at most u/2 each lie between the alphas
    and it (exp2, the products, at most 9 sums, the chain to the log-scale):
    as a random walk 2 u rms, so below 16 u for every one of the 3072
    entries, relative to the larger of a splat's two."""
    rng = np.random.default_rng(seed)
    w, f, z = 128, 4096.0, 16.0
    g = np.arange(4, w, 8)
    gx, gy = (v.reshape(-1) for v in np.meshgrid(g, g))
    n = len(gx)
    at = np.stack([gx, gy], 1) + rng.integers(-512, 512, (n, 2)) / 256.0  # pixels, exact
    mean = np.concatenate([(at - w / 2) * (z / f), np.full((n, 1), z)], 1)
    ls = np.log(sigma * z / f) + rng.uniform(-0.3, 0.3, (n, 3))
    sc = rgb_scene(mean, ls, rng.uniform(0.3, 0.9, n), rng.uniform(0.2, 1.0, (n, 3)))
    cam = axis_camera(w, w, f)
    weight = rng.uniform(0.2, 1.0, (3, w, w)).astype(np.float32).astype(np.float64)
    gg, _ = gpu_grads(sc, cam, weight, strategy="tile")
    off, idx = oracle.tile_lists(oracle.footprints(sc, cam, "all_levels"), cam)
    go = oracle.grad64(sc, cam, off, idx, weight)
    got, ref = gg["log_scale"][:, :2], go["log_scale"][:, :2]
    assert (ref > 0).all()
    assert (np.abs(got - ref) / ref.max(1, keepdims=True)).max() <= 16 * U


@pytest.mark.parametrize("n", [2, 3])
@pytest.mark.parametrize("seed", range(8))
def test_last_record_of_a_dark_pixel(n, seed):
    """n splats centred exactly on one pixel, the loss on that pixel alone,
    where alpha is the opacity itself: behind the last one lies nothing, so
    its dL/dsigma is T sum_c dL/dC_c c, to the rounding of T (2 u per
    record before it), of the products and sums (7 u) and of the last
    weight (2 u): below 16 u."""
    rng = np.random.default_rng(seed)
    z = 4.0 + np.arange(n)
    mean = np.stack([np.zeros(n), np.zeros(n), z], 1)
    op = np.append(rng.uniform(0.7, 0.97, n - 1), rng.uniform(0.2, 0.5)).astype(np.float32)
    col = rng.uniform(0.2, 1.0, (n, 3)).astype(np.float32)
    sc = rgb_scene(mean, np.full((n, 3), -1.0), op, col)
    cam = axis_camera(17, 17, 32.0)
    weight = np.zeros((3, 17, 17), np.float32)
    weight[:, 8, 8] = rng.uniform(0.2, 1.0, 3)
    gg, _ = gpu_grads(sc, cam, weight, strategy="tile")
    T = np.prod(1.0 - op[:-1].astype(np.float64))
    ref = T * (weight[:, 8, 8].astype(np.float64) * col[-1].astype(np.float64)).sum()
    assert abs(gg["opacity"][-1] - ref) <= 16 * U * ref
