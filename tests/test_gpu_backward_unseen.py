"""The projection pass of the backward reads nothing of Gaussians that no
view blended but their 2D gradients: accumulating, their colour coefficients
and colour gradients (384 B each at SH degree 3) stay unread."""
import numpy as np
import pytest

import paper_2311_17089_gb300 as msgs
from paper_2311_17089_gb300 import inputs

from gpu_util import require_cuda

pytestmark = pytest.mark.gpu


def microseconds(torch, f, n=9):
    flush = torch.empty(64 << 20, dtype=torch.float32, device="cuda")
    best = []
    for _ in range(n):
        flush.zero_()
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        best.append(a.elapsed_time(b) * 1e3)
    return min(best)


def test_accumulating_costs_no_colour_rows():
    """2M Gaussians, none blended: 72 MB of 2D gradients are read, 768 MB of
    colour rows are not.  In less than half the time of a copy that moves as
    many bytes as the rows hold, which no pass that reads them can do."""
    torch = require_cuda()
    n = 2_000_000
    host = inputs.multiscale_scene(n=20000, seed=3, split=(0.7, 0.3))
    sc = host.subset(np.arange(n) % 20000)
    ds = msgs.DeviceScene(sc)
    cam = inputs.config1_camera(32, 32)
    r = msgs.Renderer(n, cam.tiles_x * cam.tiles_y, 4096, with_cover=False, with_mask=False)
    image, final_t, n_contrib = r.images(cam)
    dl = torch.ones_like(image)
    view = msgs.bwd_view(msgs.camera_struct(cam), r.proj, r.bins, image.data_ptr(),
                         n_contrib.data_ptr(), r.rws.data_ptr(), r.rws_bytes, dl.data_ptr())
    g = [torch.ones(s, device="cuda") for s in ((n, 3), (n, 3), (n, 4), (n,), (n, 48))]
    grads = msgs.ms_grads_t(*(x.data_ptr() for x in g))
    wsb = msgs.ms_raster_bwd_views_workspace_bytes(n, 1)
    ws = torch.zeros(wsb, dtype=torch.uint8, device="cuda")  # as a raster pass that blends nothing leaves it
    flags = msgs.MS_BWD_ACCUMULATE | msgs.MS_BWD_PROJECT_PASS
    took = microseconds(torch, lambda: msgs.ms_raster_bwd_views(ds.struct, [view], grads, flags,
                                                                ws.data_ptr(), wsb))
    rows = g[4].clone()
    copy = microseconds(torch, lambda: rows.copy_(g[4]))
    assert all(bool((x == 1).all()) for x in g)
    assert took < 0.5 * copy, (took, copy)
