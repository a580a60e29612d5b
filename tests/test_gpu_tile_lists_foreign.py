"""A projection binned with another camera's frame: tile counts or first
tiles that the frame does not have end in MS_ERR_TIMEOUT (the lists are not
valid), never in lists that silently miss a Gaussian or hold it in a wrong
tile."""
import numpy as np
import pytest

import paper_2311_17089_gb300 as msgs

from gpu_util import require_cuda
from test_gpu_tile_lists import Proj, binned, projection

pytestmark = pytest.mark.gpu


def one_foreign(n, tx, ty, x0, y0, w, h):
    """n ordinary Gaussians of a tx x ty frame, the middle one's rectangle
    replaced."""
    n_tiles, rect, depth = projection(n, tx, ty, "small", seed=n + tx)
    i = n // 2
    rect[i] = x0 | (y0 << 16), (x0 + w - 1) | ((y0 + h - 1) << 16)
    n_tiles[i] = w * h
    return n_tiles, rect, depth


@pytest.mark.parametrize("n", [1, 300, 6000])
@pytest.mark.parametrize("tx,ty,x0,y0,w,h", [
    (40, 26, 0, 0, 79, 52),      # every tile of a frame of twice the size
    (40, 26, 0, 0, 41, 26),      # one column more than the frame
    (20, 13, 0, 13, 1, 1),       # the first tile just past the frame
    (256, 256, 0, 300, 1, 1),    # a first tile past 65535
    (256, 256, 255, 511, 1, 1),  # one that is 65535 modulo 65536
    (1, 1, 0, 0, 2, 1),
])
def test_reported(n, tx, ty, x0, y0, w, h):
    torch = require_cuda()
    pr = Proj(torch, *one_foreign(n, tx, ty, x0, y0, w, h))
    with pytest.raises(msgs.MsError) as e:
        binned(torch, pr, n, tx, ty, 16 * n + 65536)
    assert e.value.code == msgs.MS_ERR_TIMEOUT
