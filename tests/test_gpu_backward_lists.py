"""The backward's batches (96 records), slots (16 records summed at a time)
and 8x8 blocks at their edges: one tile with lists of n wide Gaussians, and
small ones that reach only some blocks, on whole and ragged tiles, against
the oracle's FP64 gradient (the tolerance of test_gpu_backward.compare)."""
import numpy as np
import pytest

import oracle
from paper_2311_17089_gb300 import inputs

from test_gpu_backward import compare, gpu_grads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wh", [(16, 16), (13, 9)])
@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 31, 32, 33, 95, 96, 97, 112, 191, 192, 193])
def test_list_lengths(n, wh):
    rng = np.random.default_rng(n)
    sc = inputs.tiny_scene(n=n, seed=n, sh_degree=-1, extent=0.5)
    wide = rng.random(n) < 0.5
    sc.log_scale[wide] = rng.uniform(-0.8, 0.2, (int(wide.sum()), 3)).astype(np.float32)
    sc.opacity = rng.uniform(0.02, 0.25, n).astype(np.float32)
    cam = inputs.config1_camera(*wh)
    w = rng.standard_normal((3, wh[1], wh[0]))
    gg, _ = gpu_grads(sc, cam, w, strategy="tile")
    off, idx = oracle.tile_lists(oracle.footprints(sc, cam, "all_levels"), cam)
    compare(gg, oracle.grad64(sc, cam, off, idx, w))
