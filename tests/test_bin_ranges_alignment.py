"""The tile ranges are an array of uint32: on 4 bytes, not on 8, they are binned
by the kernels that access single words (seen on the fake runtime, no GPU)."""
import ctypes

import pytest

import paper_2405_19614_gb300 as gs
from fake_runtime import FakeLib
from paper_2405_19614_gb300._lib import GsBins, GsProjected


@pytest.mark.parametrize("offset,lists", [(0, True), (4, False), (8, True), (12, False)])
def test_the_path_follows_the_ranges_alignment(tmp_path_factory, offset, lists):
    fake = FakeLib(str(tmp_path_factory.mktemp("fake")))
    views = gs.make_views([[300.0, 300.0, 320.0, 240.0]], [(640, 480)])
    at = 1 << 20
    proj, bins = GsProjected(*[at] * 5), GsBins(at, at, at + offset, at, at, 1 << 20)
    status, _, events = fake.run(lambda lib: lib.gs_bin_sort(
        ctypes.byref(proj), 5000, views, 1, ctypes.byref(bins), at, lib.gs_bin_sort_workspace_size(5000, 1 << 20, 1200),
        None))
    names = " ".join(name for what, name, _ in events if what == "launch")
    assert status == 0 and ("tile_scan" in names) == lists and ("onesweep" in names) == (not lists)
