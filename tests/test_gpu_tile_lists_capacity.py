"""gs_bin_sort over its pair capacity on the tile lists' path: exactly the pairs
of the nearest records that fit, in a stable order by (depth bits, record), are
binned, and finding them costs a fraction of the call.  Rectangles with masks and
beyond 64 tiles, lists of several sorted chunks, equal depths, both counting
grids, and maps below and above the records up to which the scan kernel cuts."""
import numpy as np
import pytest
import torch

import paper_2405_19614_gb300 as gs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2405_19614_gb300.build import build
    build()


def _records(rng, sizes, tile, n, drawn, side, depths):
    """Random rectangles of up to side x side tiles; masks on those of up to 64."""
    V = len(sizes)
    nx = np.repeat([-(-w // tile[0]) for w, _ in sizes], n)
    ny = np.repeat([-(-h // tile[1]) for _, h in sizes], n)
    x0, y0 = (rng.random(V * n) * nx).astype(np.int64), (rng.random(V * n) * ny).astype(np.int64)
    x1 = np.minimum(nx - 1, x0 + rng.integers(0, side, V * n))
    y1 = np.minimum(ny - 1, y0 + rng.integers(0, side, V * n))
    tiles = (x1 - x0 + 1) * (y1 - y0 + 1)
    full = np.where(tiles >= 64, np.uint64(0xFFFFFFFFFFFFFFFF),
                    (np.uint64(1) << np.minimum(tiles, 63).astype(np.uint64)) - np.uint64(1))
    mask = rng.integers(0, 1 << 63, V * n, dtype=np.uint64) * np.uint64(2) + rng.integers(0, 2, V * n, dtype=np.uint64)
    mask = np.where(tiles <= 64, mask & full, np.uint64(0))
    bits = np.unpackbits(mask.view(np.uint8).reshape(-1, 8), axis=1).sum(1)
    tt = np.where(tiles <= 64, bits, tiles)
    on = np.repeat(rng.random(V * n // 32 + 1) < drawn, 32)[:V * n]
    return np.stack([x0, y0, x1, y1], 1), mask, np.where(on, tt, 0).astype(np.uint32), depths(rng, V * n).astype(np.float32)


def _rasterizer(sizes, tile, n, rect, mask, tt, z, cap):
    r = gs.Rasterizer(n, 0, [[60.0, 60.0, w / 2, h / 2] for w, h in sizes], sizes, pair_capacity=cap, tile=tile)
    R = len(sizes) * n
    packed = np.stack([rect[:, 0] | rect[:, 1] << 16, rect[:, 2] | rect[:, 3] << 16], 1).astype(np.uint32)
    put = lambda dst, a, dt: dst.view(-1).copy_(torch.from_numpy(np.ascontiguousarray(a).view(dt).ravel()))
    r.proj["rec"].zero_()
    r.proj["rec"].view(R, 12)[:, 2] = torch.from_numpy(z).cuda()
    put(r.proj["rect"], packed, np.int32)
    put(r.proj["tiles_touched"], tt, np.int32)
    put(r.proj["tile_mask"], mask, np.int64)
    for k in ("keys", "vals", "ranges", "n_pairs"):
        r.bins[k].fill_(-1)
    return r


def _bin(r):
    gs.gs_bin_sort(r.proj, r.n, r.views, r.bins, r.workspace)


def _reference(sizes, tile, n, rect, mask, tt, z, cap):
    grid = [(-(-w // tile[0]), -(-h // tile[1])) for w, h in sizes]
    bases = np.cumsum([0] + [a * b for a, b in grid])
    order = np.argsort(z.view(np.uint32), kind="stable")
    order = order[tt[order] > 0]
    w = rect[order, 2] - rect[order, 0] + 1
    tiles = w * (rect[order, 3] - rect[order, 1] + 1)
    rec = np.repeat(np.arange(len(order)), tiles)  # one row a tile of the rectangle, then those of the mask
    i = np.arange(len(rec)) - np.repeat(np.cumsum(tiles) - tiles, tiles)
    keep = (tiles[rec] > 64) | ((mask[order][rec] >> np.minimum(i, 63).astype(np.uint64)) & np.uint64(1) == 1)
    rec, i = rec[keep], i[keep]
    assert len(rec) == int(tt.sum(dtype=np.int64))
    rec, i = rec[:cap], i[:cap]
    v = order[rec] // n
    nx = np.array([g[0] for g in grid])[v]
    t = bases[v] + (rect[order[rec], 1] + i // w[rec]) * nx + rect[order[rec], 0] + i % w[rec]
    by = np.argsort(t, kind="stable")
    first = np.searchsorted(t[by], np.arange(bases[-1] + 1))
    ranges = np.stack([first[:-1], first[1:]], 1)
    ranges[ranges[:, 0] == ranges[:, 1]] = 0
    g = order[rec][by]
    return (t[by].astype(np.uint64) << np.uint64(32)) | z.view(np.uint32)[g], (g % n).astype(np.uint32), ranges


SPREAD = lambda rng, n: rng.uniform(0.3, 9.0, n)
ONE = lambda rng, n: np.full(n, 1.5)
FEW = lambda rng, n: rng.choice([1.0, 2.0, 2.5, 3.0], n)
NEAR = lambda rng, n: 2.0 + 1e-6 * rng.random(n)  # a few neighbouring floats


@pytest.mark.parametrize("share", [0.0002, 0.4, 0.9999])
@pytest.mark.parametrize("depths", [SPREAD, ONE, FEW, NEAR], ids=["spread", "one", "few", "near"])
@pytest.mark.parametrize("sizes,tile,n,drawn,side", [
    ([(640, 480)], (16, 16), 9000, 0.5, 12),                      # rectangles beyond 64 tiles
    ([(96, 80), (64, 33)], (16, 16), 20000, 0.8, 3),              # lists of several thousand words
    ([(640, 480)], (8, 8), 1500, 0.7, 30),                        # counted in global words
    ([(64, 64)], (16, 16), 30000, 1.0, 2),                        # lists of several chunks
    ([(1200, 680)] * 3, (32, 16), 400_001, 0.05, 4),              # a launch a step
], ids=["wide", "long", "global", "chunks", "large"])
def test_the_nearest_pairs_that_fit(sizes, tile, n, drawn, side, depths, share):
    rng = np.random.default_rng(n + side)
    rect, mask, tt, z = _records(rng, sizes, tile, n, drawn, side, depths)
    total = int(tt.sum(dtype=np.int64))
    cap = max(1, int(share * total))
    r = _rasterizer(sizes, tile, n, rect, mask, tt, z, cap)
    keys, vals, ranges = _reference(sizes, tile, n, rect, mask, tt, z, cap)
    for _ in range(2):  # a second call in the same workspace
        _bin(r)
        assert r.n_pairs() == total and r.status() == 1 << 3
        np.testing.assert_array_equal(r.bins["ranges"].cpu().numpy(), ranges)
        np.testing.assert_array_equal(r.bins["keys"].cpu().numpy().view(np.uint64), keys)
        np.testing.assert_array_equal(r.bins["vals"].cpu().numpy().view(np.uint32), vals)


def _median_ms(r, calls=9):
    times = []
    for _ in range(calls + 3):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        _bin(r)
        e1.record()
        torch.cuda.synchronize()
        times.append(e0.elapsed_time(e1))
    return sorted(times[3:])[calls // 2]


@pytest.mark.parametrize("sizes,n", [([(1200, 680)], 300_000), ([(1200, 680)] * 4, 1_000_000)])
def test_a_cut_costs_a_few_binnings(sizes, n):
    """A cut by one block took 46 and 150 times the call without one."""
    rng = np.random.default_rng(5)
    rec = _records(rng, sizes, (32, 16), n, 0.3, 3, SPREAD)
    total = int(rec[2].sum(dtype=np.int64))
    fits = _rasterizer(sizes, (32, 16), n, *rec, total)
    cut = _rasterizer(sizes, (32, 16), n, *rec, 3 * total // 4)
    assert _median_ms(cut) <= 8 * _median_ms(fits)
