"""ms_bin where the count pass's last CTA sums many rows of few tiles (a
thread per tile and run of rows): tile counts around the CTA's half, lists
and ranges against the host reference, and the time of a million entries in
one tile against the same entries spread over a thousand tiles."""
import numpy as np
import pytest

import paper_2311_17089_gb300 as msgs

from gpu_util import require_cuda
from test_gpu_backward_unseen import microseconds
from test_gpu_tile_lists import Proj, camera, check, projection

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tx,ty", [(1, 1), (2, 1), (3, 1), (4, 2), (9, 1), (15, 1), (8, 4), (33, 1),
                                   (9, 7), (64, 1), (13, 5), (127, 1), (16, 8), (43, 3)])
def test_lists(tx, ty):
    torch = require_cuda()
    n = 150000
    n_tiles, rect, depth = projection(n, tx, ty, "mixed", seed=tx + 7 * ty)
    check(torch, n_tiles, rect, depth, tx, ty, [1.0, 0.37])


def test_one_tile_takes_no_longer_than_many():
    """The depth sort is the same and one tile needs fewer launches and
    stores than a thousand: not above 1.1x."""
    torch = require_cuda()
    n = 1_000_000
    rng = np.random.default_rng(4)
    depth = rng.uniform(0.3, 60.0, n).astype(np.float32).view(np.uint32)
    took = []
    for tx, ty in ((1, 1), (33, 32)):
        x, y = rng.integers(0, tx, n), rng.integers(0, ty, n)
        at = (x | (y << 16)).astype(np.uint32)
        pr = Proj(torch, np.ones(n, np.uint32), np.stack([at, at], 1), depth)
        idx = torch.empty(n, dtype=torch.int32, device="cuda")
        ranges = torch.empty((tx * ty, 2), dtype=torch.int32, device="cuda")
        counts = torch.zeros(4, dtype=torch.int64, device="cuda")
        bins = msgs.ms_bins_t(idx.data_ptr(), ranges.data_ptr(), counts.data_ptr(), n)
        wsb = msgs.ms_bin_workspace_bytes(n, tx * ty, n)
        ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
        took.append(microseconds(torch, lambda: msgs.ms_bin(pr.struct, n, camera(tx, ty), bins,
                                                            ws.data_ptr(), wsb), n=25))
        assert msgs.ms_bin_counts(bins)[0] == msgs.MS_OK
    assert took[0] <= 1.1 * took[1], took
