"""The shared memory that a kernel may be launched with belongs to the kernel,
for every host thread: once raised for a call it must not be lowered by another,
whose thread may run between the first one's limit and its launch.  Shown
without a GPU, on the fake runtime."""
import ctypes

import pytest

import paper_2405_19614_gb300 as gs
from fake_runtime import FakeLib
from paper_2405_19614_gb300._lib import GsBins, GsProjected


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return FakeLib(str(tmp_path_factory.mktemp("fake")))


def _bin_sort(size, n, cap=1 << 20):
    views = gs.make_views([[300.0, 300.0, 1.0, 1.0]], [size], (8, 8))
    proj, bins = GsProjected(*[4096] * 5), GsBins(*[4096] * 5, cap)

    def call(lib):
        ws = lib.gs_bin_sort_workspace_size(n, cap, 1)
        return lib.gs_bin_sort(ctypes.byref(proj), n, views, 1, ctypes.byref(bins), 1 << 20, ws, None)
    return call


def test_no_call_lowers_a_kernels_limit(fake):
    limits, large = {}, 0
    for size in [(1280, 720), (1200, 680), (1280, 800), (640, 480), (1200, 680)]:
        status, _, events = fake.run(_bin_sort(size, 400_000))
        assert status == 0, size
        for what, name, value in events:
            if what == "limit":
                assert int(value) >= limits.get(name, 0), (size, name)
                limits[name] = int(value)
            elif what == "launch":
                large += int(value) > 48 * 1024
    assert large >= 8  # the count and scatter of four views, beyond the default limit
