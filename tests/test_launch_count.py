"""The kernels that a mapping step reports for its binning are the ones that
gs_bin_sort launches, counted on the fake runtime (no GPU)."""
import ctypes

import pytest

import paper_2405_19614_gb300 as gs
from fake_runtime import FakeLib
from paper_2405_19614_gb300._lib import GsBins, GsProjected
from paper_2405_19614_gb300.pipeline import bin_kernels


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return FakeLib(str(tmp_path_factory.mktemp("fake")))


@pytest.mark.parametrize("size,count,n", [
    ((640, 480), 1, 8192), ((640, 480), 1, 8193),             # no list beyond one chunk; some may be
    ((1200, 680), 1, 1 << 20), ((1200, 680), 1, (1 << 20) + 1),  # cut in the scan kernel; by launches of its own
    ((1200, 680), 8, 1_000_000),
    ((64, 48), 1, 100_000), ((64, 48), 8, 100_000),           # crowded: the radix path
])
def test_binning(fake, size, count, n):
    views = gs.make_views([[300.0, 300.0, size[0] / 2, size[1] / 2]] * count, [size] * count)
    proj, bins = GsProjected(*[1 << 20] * 5), GsBins(*[1 << 20] * 5, 1 << 22)

    def call(lib):
        ws = lib.gs_bin_sort_workspace_size(n * count, 1 << 22, 1)
        return lib.gs_bin_sort(ctypes.byref(proj), n, views, count, ctypes.byref(bins), 1 << 20, ws, None)
    status, _, events = fake.run(call)
    launched = [name for what, name, _ in events if what == "launch" and "chain_clear" not in name]
    n_tiles = count * -(-size[0] // 16) * -(-size[1] // 16)
    assert status == 0 and len(launched) == bin_kernels(n, count, n_tiles), launched
