"""ms_bin and ms_bin_ordered on made-up projections, so that every cut of the
tile stage (and the one-CTA depth sort) is met: one tile to 65536, empty to
full frames, Gaussians of one tile and of all of them, orders around a
block's 1024 positions and past 2048 blocks, capacities from one entry to more than needed.  The lists,
ranges and counts equal a host reference bit for bit: the listed Gaussians
by (depth bits, index), each one's tiles row by row, the first dup_capacity
of these entries, stably sorted by tile."""
import numpy as np
import pytest

import paper_2311_17089_gb300 as msgs

from gpu_util import require_cuda

pytestmark = pytest.mark.gpu


def projection(n, tx, ty, kind, seed):
    """n_tiles, rect and depth as ms_project lays them out, for a tx x ty
    tile frame."""
    rng = np.random.default_rng(seed)
    most = {"small": 3, "mixed": 3, "big": 1 << 20, "all": 1 << 20}[kind]
    x0 = rng.integers(0, tx, n)
    y0 = rng.integers(0, ty, n)
    w = rng.integers(1, np.minimum(tx - x0, most) + 1)
    h = rng.integers(1, np.minimum(ty - y0, most) + 1)
    if kind == "mixed":  # a few large ones first in depth, as near splats are
        big = rng.random(n) < 0.02
        x0[big], y0[big], w[big], h[big] = 0, 0, tx, ty
    if kind == "all":
        x0[:], y0[:], w[:], h[:] = 0, 0, tx, ty
    listed = rng.random(n) < (0.8 if n > 1 else 2.0)
    depth = rng.uniform(0.3, 60.0, n).astype(np.float32)
    depth[rng.random(n) < 0.3] = np.float32(7.0)  # ties
    if kind == "mixed":
        depth[big] = np.float32(0.25)
    rect = np.stack([x0 | (y0 << 16), (x0 + w - 1) | ((y0 + h - 1) << 16)], 1).astype(np.uint32)
    n_tiles = np.where(listed, w * h, 0).astype(np.uint32)
    return n_tiles, rect, depth.view(np.uint32)


def reference(n_tiles, rect, order, tx, tiles, cap):
    order = order[n_tiles[order] > 0]
    cnt = n_tiles[order].astype(np.int64)
    total = int(cnt.sum())
    keep = np.searchsorted(np.cumsum(cnt), cap) + 1  # enough items for cap entries
    order, cnt = order[:keep], cnt[:keep]
    idx = np.repeat(order, cnt)
    m = np.arange(len(idx)) - np.repeat(np.cumsum(cnt) - cnt, cnt)
    x0, y0 = (rect[idx, 0] & 0xffff).astype(np.int64), (rect[idx, 0] >> 16).astype(np.int64)
    w = (rect[idx, 1] & 0xffff).astype(np.int64) - x0 + 1
    tile = ((y0 + m // w) * tx + x0 + m % w)[:cap]
    idx = idx[:cap]
    s = np.argsort(tile, kind="stable")
    counts = np.bincount(tile, minlength=tiles)
    start = np.cumsum(counts) - counts
    ranges = np.stack([start, start + counts], 1)
    ranges[counts == 0] = 0
    return idx[s].astype(np.uint32), ranges.astype(np.uint32), total


class Proj:
    def __init__(self, torch, n_tiles, rect, depth):
        listed = n_tiles > 0
        stats = np.zeros(msgs.MS_STATS_WORDS, np.uint32)
        stats[0] = listed.sum()
        stats[2:4] = np.array([int(n_tiles.astype(np.int64).sum())], np.uint64).view(np.uint32)
        for p in range(4):
            stats[16 + 256 * p:16 + 256 * (p + 1)] = np.bincount((depth[listed] >> (8 * p)) & 255,
                                                                  minlength=256)
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()
        self.t = [dev(n_tiles), dev(rect), dev(depth), dev(stats)]
        nt, rc, de, st = (int(x.data_ptr()) for x in self.t)
        self.struct = msgs.ms_proj_t(0, rc, nt, de, 0, 0, st, len(n_tiles))


def camera(tx, ty):
    c = msgs.ms_camera_t()
    c.width, c.height, c.fx, c.fy, c.near_plane = 16 * tx, 16 * ty, 100.0, 100.0, 0.2
    return c


def binned(torch, pr, n, tx, ty, cap, order=None, order_stats=None):
    tiles = tx * ty
    g = torch.full((cap,), -1, dtype=torch.int32, device="cuda")
    r = torch.full((tiles, 2), -1, dtype=torch.int32, device="cuda")
    c = torch.zeros(4, dtype=torch.int64, device="cuda")
    bins = msgs.ms_bins_t(g.data_ptr(), r.data_ptr(), c.data_ptr(), cap)
    wsb = msgs.ms_bin_workspace_bytes(n, tiles, cap)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda").fill_(0xa5)
    if order is None:
        msgs.ms_bin(pr.struct, n, camera(tx, ty), bins, ws.data_ptr(), wsb)
    else:
        msgs.ms_bin_ordered(pr.struct, n, camera(tx, ty), bins, order.data_ptr(),
                            order_stats.data_ptr(), ws.data_ptr(), wsb)
    rc, d, s = msgs.ms_bin_counts(bins)
    torch.cuda.synchronize()
    return rc, d, s, g.cpu().numpy().view(np.uint32), r.cpu().numpy().view(np.uint32)


def check(torch, n_tiles, rect, depth, tx, ty, caps, order=None):
    n, tiles = len(n_tiles), tx * ty
    pr = Proj(torch, n_tiles, rect, depth)
    by_depth = np.lexsort((np.arange(n), depth))
    if order is None:
        host_order, dev_order, dev_stats = by_depth[n_tiles[by_depth] > 0], None, None
    else:
        host_order = order
        dev_order = torch.from_numpy(order.astype(np.int32)).cuda()
        st = np.zeros(msgs.MS_STATS_WORDS, np.uint32)
        st[0] = len(order)
        dev_stats = torch.from_numpy(st.view(np.int32)).cuda()
    total = int(n_tiles.astype(np.int64).sum())
    for cap in caps:
        cap = max(1, int(cap * total) if isinstance(cap, float) else cap)
        idx, ranges, _ = reference(n_tiles, rect, host_order, tx, tiles, cap)
        rc, d, s, got, got_r = binned(torch, pr, n, tx, ty, cap, dev_order, dev_stats)
        assert rc == (msgs.MS_OK if total <= cap else msgs.MS_ERR_CAPACITY), (cap, rc)
        assert d == total and s == int((n_tiles > 0).sum())
        np.testing.assert_array_equal(got_r, ranges, err_msg=f"ranges, cap {cap}")
        np.testing.assert_array_equal(got[:len(idx)], idx, err_msg=f"lists, cap {cap}")
        assert (got[len(idx):] == 0xffffffff).all()  # nothing written past the entries


CASES = [
    (1, 1, 1, "small"), (33, 1, 1, "small"), (5000, 1, 1, "small"), (300, 3, 1, "mixed"),
    (1023, 5, 4, "small"), (1024, 5, 4, "small"), (1025, 5, 4, "mixed"), (40000, 10, 7, "small"),
    (3000, 33, 31, "big"), (20000, 39, 27, "mixed"), (30000, 79, 52, "small"),
    (6000, 79, 52, "mixed"), (150, 79, 52, "all"), (2000, 96, 64, "small"), (2000, 97, 64, "small"),
    (1500, 128, 128, "mixed"), (1500, 129, 128, "mixed"), (700, 256, 256, "mixed"),
    (900, 2048, 32, "big"), (200000, 20, 13, "mixed"),
    # around the largest projection one CTA sorts
    (4095, 39, 27, "mixed"), (4096, 10, 7, "small"), (4096, 39, 27, "big"), (4097, 10, 7, "mixed"),
]


@pytest.mark.parametrize("n,tx,ty,kind", CASES)
def test_lists(n, tx, ty, kind):
    torch = require_cuda()
    n_tiles, rect, depth = projection(n, tx, ty, kind, seed=n + tx)
    check(torch, n_tiles, rect, depth, tx, ty, [1.05, 1.0, 0.6, 4 * n + 7, 40, 1])


def test_more_blocks_than_2048():
    torch = require_cuda()
    n = 2100003
    n_tiles, rect, depth = projection(n, 10, 7, "small", seed=5)
    check(torch, n_tiles, rect, depth, 10, 7, [1.0, 0.3])


@pytest.mark.parametrize("density", [1.0, 0.4, 0.02])
def test_order_of_a_superset(density):
    """A shared order may hold Gaussians this frame does not list, and be
    unaligned."""
    torch = require_cuda()
    n, tx, ty = 50001, 39, 27
    n_tiles, rect, depth = projection(n, tx, ty, "mixed", seed=11)
    drop = np.random.default_rng(3).random(n) >= density
    n_tiles[drop] = 0
    order = np.lexsort((np.arange(n), depth))
    check(torch, n_tiles, rect, depth, tx, ty, [1.05, 0.5], order)
