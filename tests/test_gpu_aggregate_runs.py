"""ms_aggregate on voxels of chosen member counts (around the pooling
kernel's 32-member loads and across its 256-item blocks), every colour
width, and more cameras than one coverage launch takes, against the
oracle."""
import numpy as np
import pytest

import oracle
import paper_2311_17089_gb300 as msgs
from paper_2311_17089_gb300 import inputs

from gpu_util import require_cuda

pytestmark = pytest.mark.gpu
COUNTS = (1, 2, 7, 8, 9, 31, 32, 33, 63, 64, 65, 255, 256, 257, 600)


@pytest.mark.parametrize("deg", [-1, 0, 1, 2, 3])
def test_voxel_member_counts(deg):
    require_cuda()
    n = sum(COUNTS)
    sc = inputs.multiscale_scene(n=n, seed=20 + deg, split=(1.0, 0.0, 0.0, 0.0), box=1.0,
                                 cluster_sigma=0.1, n_clusters=4, sh_degree=max(deg, 0))
    sc.n_levels = 4
    rng = np.random.default_rng(deg + 50)
    if deg < 0:
        sc.color = rng.uniform(0, 1, (n, 3)).astype(np.float32)
        sc.sh_degree = -1
    # voxel v of the counts at its own place on a 200^3 grid over [-20, 20]
    # (extent 10), its members within a tenth of the voxel's 0.2 width;
    # member order shuffled over the scene
    place = np.repeat(np.arange(len(COUNTS)), COUNTS)[rng.permutation(n)]
    centre = np.stack([0.4 * place - 2.7, 0.1 + 0.0 * place, 0.1 + 0.0 * place], 1)
    sc.mean = (centre + rng.uniform(-0.02, 0.02, (n, 3))).astype(np.float32)
    sc.log_scale = np.minimum(sc.log_scale, -4.0).astype(np.float32)
    sc.opacity = np.maximum(sc.opacity, 0.05).astype(np.float32)
    cams = [inputs.downscale(c, 4) for c in
            inputs.orbit_cameras(9, seed=3, radius=10.0, width=256, height=192)]
    o, keys, _ = oracle.aggregate(sc, cams, 2, 10.0)
    assert len(keys) == len(COUNTS)
    g = msgs.aggregate_level(msgs.DeviceScene(sc), cams, 2, 10.0)
    assert g["mean"].shape[0] == len(keys)
    for f in ("mean", "log_scale", "quat", "opacity", "color"):
        got, ref = g[f].cpu().numpy(), o[f]
        # a sequential FP32 sum of c values is within c u sum |x| of the exact
        # one (u = 2^-24); the two sides may each be that far off, and the
        # log-scale's ln(2 / S_avg) adds the relative error of S_avg
        tol = 2 * (max(COUNTS) + 4) * 2.0 ** -24 * max(1.0, float(np.abs(ref).max()))
        np.testing.assert_allclose(got.reshape(ref.shape), ref, rtol=0, atol=tol, err_msg=f)
