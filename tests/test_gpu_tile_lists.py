"""gs_bin_sort on hand-made records against the definition in numpy: the pairs
in a stable order by (depth bits, record), cut at the capacity, then stable by
tile.  Sizes sit where the list building changes: list lengths around a warp's
run, a group's and a block's share and beyond one chunk, rectangles with and
without a mask, equal depths, several views, small maps on many tiles, records
crowded into few tiles (the radix path), and capacities that cut the list inside
a record."""
import numpy as np
import pytest
import torch

import paper_2405_19614_gb300 as gs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2405_19614_gb300.build import build
    build()


def _records(rng, sizes, tile, n, drawn, side, z_values):
    """Random rectangles of up to side x side tiles and masks for n Gaussians a view."""
    V = len(sizes)
    rect = np.zeros((V * n, 4), np.int64)
    mask = np.zeros(V * n, np.uint64)
    tt = np.zeros(V * n, np.uint32)
    z = rng.choice(z_values, V * n).astype(np.float32)
    for v, (w, h) in enumerate(sizes):
        nx, ny = -(-w // tile[0]), -(-h // tile[1])
        for i in np.nonzero(rng.random(n) < drawn)[0]:
            r = v * n + i
            x0, y0 = rng.integers(0, nx), rng.integers(0, ny)
            x1, y1 = min(nx - 1, x0 + rng.integers(0, side)), min(ny - 1, y0 + rng.integers(0, side))
            rect[r] = x0, y0, x1, y1
            tiles = (x1 - x0 + 1) * (y1 - y0 + 1)
            if tiles <= 64:
                keep = rng.random(tiles) < 0.7
                mask[r] = sum(1 << int(k) for k in np.nonzero(keep)[0])
                tt[r] = keep.sum()
            else:
                tt[r] = tiles
    return rect, mask, tt, z


def _reference(sizes, tile, n, rect, mask, tt, z, cap):
    base, bases = 0, []
    for w, h in sizes:
        bases.append(base)
        base += -(-w // tile[0]) * -(-h // tile[1])
    tiles, ids = [], []
    for r in np.argsort(z.view(np.uint32), kind="stable"):
        if not tt[r]:
            continue
        v = r // n
        nx = -(-sizes[v][0] // tile[0])
        x0, y0, x1, y1 = rect[r]
        ys, xs = np.mgrid[y0:y1 + 1, x0:x1 + 1]
        t = (bases[v] + ys * nx + xs).ravel()
        if len(t) <= 64:
            t = t[[(int(mask[r]) >> k) & 1 == 1 for k in range(len(t))]]
        tiles.append(t)
        ids.append(np.full(len(t), r))
    tiles = np.concatenate(tiles) if tiles else np.zeros(0, np.int64)
    ids = np.concatenate(ids) if ids else np.zeros(0, np.int64)
    total = len(tiles)
    tiles, ids = tiles[:cap], ids[:cap]
    order = np.argsort(tiles, kind="stable")
    tiles, ids = tiles[order].astype(np.uint64), ids[order]
    keys = (tiles << np.uint64(32)) | z.view(np.uint32)[ids].astype(np.uint64)
    ranges = np.zeros((base, 2), np.uint32)
    for t in np.unique(tiles):
        at = np.nonzero(tiles == t)[0]
        ranges[int(t)] = at[0], at[-1] + 1
    return total, keys, (ids % n).astype(np.uint32), ranges


def _check(sizes, tile, n, rect, mask, tt, z, cap=None):
    V, dev = len(sizes), "cuda"
    total = int(tt.sum())
    cap = max(1, total) if cap is None else cap
    rast = gs.Rasterizer(n, 0, [[60.0, 60.0, w / 2, h / 2] for w, h in sizes], sizes, pair_capacity=cap, tile=tile)
    rec = np.zeros((V * n, 12), np.float32)
    rec[:, 2] = z
    packed = np.stack([rect[:, 0] | rect[:, 1] << 16, rect[:, 2] | rect[:, 3] << 16], 1).astype(np.uint32)
    put = lambda dst, a, dt: dst.view(-1).copy_(torch.from_numpy(np.ascontiguousarray(a).view(dt).ravel()).to(dev))
    put(rast.proj["rec"], rec, np.float32)
    put(rast.proj["rect"], packed, np.int32)
    put(rast.proj["tiles_touched"], tt, np.int32)
    put(rast.proj["tile_mask"], mask, np.int64)
    for k in ("keys", "vals", "ranges", "n_pairs"):
        rast.bins[k].fill_(-1)
    gs.gs_bin_sort(rast.proj, n, rast.views, rast.bins, rast.workspace)
    want, keys, vals, ranges = _reference(sizes, tile, n, rect, mask, tt, z, cap)
    assert rast.n_pairs() == want == total
    assert (rast.status() != 0) == (total > cap)
    K = min(total, cap)
    np.testing.assert_array_equal(rast.bins["ranges"].cpu().numpy().view(np.uint32), ranges)
    np.testing.assert_array_equal(rast.bins["keys"][:K].cpu().numpy().view(np.uint64), keys)
    np.testing.assert_array_equal(rast.bins["vals"][:K].cpu().numpy().view(np.uint32), vals)


@pytest.mark.parametrize("length", [1, 31, 32, 33, 64, 65, 128, 129, 256, 257, 512, 513, 1025, 2048, 2049, 4097, 8192,
                                    8193, 20000])
@pytest.mark.parametrize("depths", ["distinct", "few"])
def test_list_lengths(length, depths):
    """One tile of `length` words beside short ones; few depths: ties by index."""
    rng = np.random.default_rng(length)
    n = length + 200
    z_values = rng.uniform(0.3, 9.0, 4 * n) if depths == "distinct" else np.array([1.0, 1.5, 7.25])
    rect, mask, tt, z = _records(rng, [(64, 64)], (16, 16), n, 1.0, 3, z_values)
    on = rng.permutation(n)[:length]
    off = np.setdiff1d(np.arange(n), on)
    tt[off[100:]] = 0
    rect[on] = 2, 1, 2, 1
    mask[on] = 1
    tt[on] = 1
    tt[(tt > 0) & (mask == 0)] = 0
    _check([(64, 64)], (16, 16), n, rect, mask, tt, z)


@pytest.mark.parametrize("sizes,tile,n,drawn,side", [
    ([(321, 243), (283, 197), (97, 401)], (16, 16), 3001, 0.3, 4),    # uneven views
    ([(640, 480)], (8, 8), 1500, 0.5, 30),                            # rectangles beyond 64 tiles
    ([(1200, 680)], (16, 16), 300, 0.9, 6),                           # few records, many tiles
    ([(1288, 1280)], (8, 8), 2000, 0.8, 12),                          # more tiles than a block counts
    ([(64, 48)] * 5, (64, 32), 20000, 0.2, 2),                        # crowded: the radix path
    ([(64, 48), (33, 70)], (32, 32), 0, 1.0, 1),                      # no Gaussian
    ([(64, 48)], (16, 16), 700, 0.0, 1),                              # nothing drawn
    ([(64, 48)] * 64, (16, 16), 33, 0.7, 3),                          # the most views
])
def test_views_and_rectangles(sizes, tile, n, drawn, side):
    rng = np.random.default_rng(n + side)
    rect, mask, tt, z = _records(rng, sizes, tile, n, drawn, side, rng.uniform(0.3, 9.0, 5000))
    _check(sizes, tile, n, rect, mask, tt, z)


@pytest.mark.parametrize("n", [900, 30000])
@pytest.mark.parametrize("share", [0.0003, 0.31, 0.999])
def test_capacity_keeps_the_nearest(n, share):
    """30,000 records crowd the tiles onto the radix path; 900 do not."""
    rng = np.random.default_rng(n)
    sizes, tile = [(96, 80), (64, 33)], (32, 32) if n > 1000 else (16, 16)
    rect, mask, tt, z = _records(rng, sizes, tile, n, 0.6, 5, np.array([1.0, 2.0, 2.5, 3.0]))
    _check(sizes, tile, n, rect, mask, tt, z, cap=max(1, int(share * tt.sum())))
