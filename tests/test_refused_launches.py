"""A call of several launches stops at the first that is refused and returns
GS_ERR_CUDA: a kernel behind it would take what the refused one did not write
(counts, places in a list) from uninitialised memory.  Shown without a GPU, on
the fake runtime, with each launch and clear of each call refused in turn."""
import ctypes

import pytest

import paper_2405_19614_gb300 as gs
from fake_runtime import FakeLib
from paper_2405_19614_gb300._lib import (GsBins, GsImage, GsOptions, GsParamGrads, GsParams, GsProjected)

GS_ERR_CUDA = 2
AT = 1 << 20  # a device address (nothing is read there)
ref = ctypes.byref


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return FakeLib(str(tmp_path_factory.mktemp("fake")))


def _views(size, count=1, tile=(16, 16)):
    return gs.make_views([[300.0, 300.0, size[0] / 2, size[1] / 2]] * count, [size] * count, tile)


PROJ, IMG, CAP = GsProjected(*[AT] * 5), GsImage(*[AT] * 5), 1 << 20
BINS, GRADS = GsBins(*[AT] * 5, CAP), GsParamGrads(*[AT] * 5)
FULL = _views((1200, 680), 8)


def _bin_sort(views, n):
    def call(lib):
        ws = lib.gs_bin_sort_workspace_size(n * len(views), CAP, 1)
        return lib.gs_bin_sort(ref(PROJ), n, views, len(views), ref(BINS), AT, ws, None)
    return call


def _params(degree):
    return GsParams(*[AT] * 5, 1000, degree)


def _render_bwd(views, degree):
    def call(lib):
        return lib.gs_render_bwd(ref(_params(degree)), views, AT, len(views), ref(GsOptions(0.2, 0.3, 1)), ref(PROJ),
                                 ref(BINS), ref(IMG), AT, AT, None, AT, ref(GRADS), AT, AT, None)
    return call


def _ssim(lib):
    return lib.gs_loss_ssim(AT, AT, FULL, len(FULL), 0.2, AT, AT, AT, lib.gs_ssim_workspace_size(8 * 1200 * 680), AT,
                            None)


def _densify(lib):
    ws = lib.gs_select_workspace_size(8 * 1200 * 680)
    return lib.gs_densify(AT, AT, AT, FULL, AT, len(FULL), 0.5, 0.0, ref(GRADS), 3, 1000, 100000, AT, AT, AT, ws, None)


def _prune(lib):
    return lib.gs_prune_select(AT, 100000, 0.1, AT, AT, AT, lib.gs_select_workspace_size(100000), None)


def _order(lib):
    return lib.gs_spatial_order(AT, 100000, AT, AT, lib.gs_spatial_order_workspace_size(100000), AT, None)


def _lookback(lib):
    return lib.gs_check_lookback_timeout(0, 0, AT, AT, lib.gs_check_lookback_timeout_workspace_size(), None)


CALLS = {
    "bins-private-counts": (_bin_sort(_views((1200, 680)), 300_000), 6),
    "bins-global-counts": (_bin_sort(_views((1280, 720), tile=(8, 8)), 20_000), 6),
    "bins-cut-launches": (_bin_sort(_views((1200, 680)), 2_000_000), 11),
    "bins-radix": (_bin_sort(_views((64, 48)), 100_000), 14),
    "render-fwd": (lambda lib: lib.gs_render_fwd(ref(PROJ), 1000, ref(BINS), FULL, len(FULL), ref(IMG), AT, None), 2),
    "render-bwd-0": (_render_bwd(FULL, 0), 4),
    "render-bwd-3": (_render_bwd(_views((64, 48)), 3), 3),
    "ssim": (_ssim, 2),
    "densify": (_densify, 3),
    "prune": (_prune, 3),
    "order": (_order, 9),
    "lookback": (_lookback, 3),
}


@pytest.mark.parametrize("name", CALLS)
def test_stops_at_the_first_refused_launch(fake, name):
    call, at_least = CALLS[name]
    status, total, events = fake.run(call)
    assert status == 0 and total >= at_least, events
    for k in range(1, total + 1):
        status, asked, events = fake.run(call, refuse=k)
        assert status == GS_ERR_CUDA, (k, events)
        assert asked == k, (k, events)
    assert fake.run(call)[:2] == (0, total)  # no error is left behind
