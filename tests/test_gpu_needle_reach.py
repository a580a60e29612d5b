"""Needles of hundreds of pixels whose tips lie inside the image, one to a
frame: the record's FP32 conic and the rounding of its evaluated power put
accepted pixels beyond the covariance's half extents there.  The kernels that
leave records out by their reach (tile, list, backward) take the same pixels
as the group kernel, which evaluates every list entry at every pixel."""
import numpy as np
import pytest

import paper_2311_17089_gb300 as msgs
from paper_2311_17089_gb300 import autograd as ag
from paper_2311_17089_gb300 import inputs

from gpu_util import require_cuda

pytestmark = pytest.mark.gpu
W = H = 1200
F = 1200.0
N = 400


def needle(rng, lo, hi):
    """A needle of standard deviation lo..hi px, its tip inside the image."""
    z = 4.0
    sigma = np.exp(rng.uniform(np.log(lo), np.log(hi)))
    th = rng.uniform(0, 2 * np.pi)
    op = rng.uniform(0.05, 0.99)
    tip = rng.uniform(60, W - 60, 2)
    at = tip - np.sqrt(2 * np.log(255 * op)) * sigma * np.array([np.cos(th), np.sin(th)])
    mean = np.append((at - W / 2) * z / F, z)
    ls = np.log(np.array([sigma, rng.uniform(0.01, 1.0), 0.01]) * z / F)
    q = np.array([np.cos(th / 2), 0, 0, np.sin(th / 2)])
    f32 = lambda x: np.asarray([x], np.float32)
    return inputs.Scene(f32(mean), f32(ls), f32(q), f32(op), np.ones((1, 3), np.float32),
                        np.ones(1, np.uint8), 1, -1, np.zeros(1, np.float32),
                        np.full(1, np.inf, np.float32))


CAM = inputs.Camera(np.eye(3, dtype=np.float32), np.zeros(3, np.float32), np.zeros(3, np.float32),
                    F, F, W / 2, H / 2, W, H)


@pytest.mark.parametrize("lo,hi", [(20, 60), (60, 200), (200, 600), (600, 2000)])
def test_reach(lo, hi):
    torch = require_cuda()
    rng = np.random.default_rng(int(lo))
    dev = torch.device("cuda")
    r = msgs.Renderer(1, CAM.tiles_x * CAM.tiles_y, CAM.tiles_x * CAM.tiles_y)
    frame = ag.Frame(1, CAM, CAM.tiles_x * CAM.tiles_y, device=dev, strategy="group8")
    wrong = {"tile": [], "list": [], "backward": []}
    blended = 0
    for i in range(N):
        sc = needle(rng, lo, hi)
        ds = msgs.DeviceScene(sc)
        _, t0, n0 = r.render(ds, CAM, "all_levels", strategy="group8")
        blended += int(n0.sum())
        for strategy in ("tile", "list"):
            _, t, n = r.render(ds, CAM, "all_levels", strategy=strategy)
            if not (torch.equal(n, n0) and torch.equal(t, t0)):
                wrong[strategy].append((i, int((n != n0).sum())))
        # dL/dcolour of a loss on the faint pixels is the sum of their alphas:
        # a pixel left out is 1e-4 of it or more, below 4000 of them; the sum
        # in FP32 is within 1e-5
        alpha = 1.0 - t0
        faint = ((alpha > 0) & (alpha < 0.006) & (torch.rand_like(t0) < 0.5)).float()
        p = {k: torch.tensor(getattr(sc, k), device=dev, requires_grad=True)
             for k in ("mean", "log_scale", "quat", "opacity", "color")}
        img = ag.render(p, torch.tensor(sc.level, device=dev), torch.tensor(sc.s_max, device=dev),
                        torch.tensor(sc.s_min, device=dev), 1, -1, frame, "all_levels")
        (img[0] * faint).sum().backward()
        want = float((alpha.double() * faint.double()).sum())
        got = float(p["color"].grad[0, 0])
        assert int(faint.sum()) < 4000
        if abs(got - want) > 5e-5 * want:
            wrong["backward"].append((i, got, want))
    r.check()
    assert blended > 100 * N
    assert not any(wrong.values()), {k: (len(v), v[:5]) for k, v in wrong.items()}
