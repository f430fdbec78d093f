"""The library's own choice of compositing variants is a state of its own: what
gs_get_render_variants returns, given back to gs_set_render_variants, restores it.
Seen on the fake runtime by the kernels that are launched (no GPU)."""
import ctypes
import re

import pytest

import paper_2405_19614_gb300 as gs
from fake_runtime import FakeLib
from paper_2405_19614_gb300._lib import GsBins, GsImage, GsProjected

AT = 1 << 20
ref = ctypes.byref


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return FakeLib(str(tmp_path_factory.mktemp("fake")))


def _bands(fake, size):
    """(pixels a thread, band width) of the forward and backward kernels of a view."""
    views = gs.make_views([[300.0, 300.0, size[0] / 2, size[1] / 2]], [size])
    proj, bins, img = GsProjected(*[AT] * 5), GsBins(*[AT] * 5, 1 << 20), GsImage(*[AT] * 5)

    def call(lib):
        return (lib.gs_render_fwd(ref(proj), 1000, ref(bins), views, 1, ref(img), AT, None) or
                lib.gs_render_bwd_splats(ref(proj), 1000, ref(bins), views, 1, ref(img), AT, AT, None, AT, AT, None))
    status, _, events = fake.run(call)
    assert status == 0
    names = " ".join(name for what, name, _ in events if what == "launch")
    return tuple(tuple(int(x) for x in re.search(rf"render_{d}_kernelILi(\d+)ELi(\d+)E", names).groups())
                 for d in ("fwd", "bwd"))


def _get(fake):
    out = [ctypes.c_int32() for _ in range(4)]
    assert fake.lib.gs_get_render_variants(*[ref(o) for o in out]) == 0
    return tuple(o.value for o in out)


OWN = {(64, 48): ((1, 8), (1, 8)), (360, 300): ((2, 8), (2, 8)), (1200, 680): ((2, 8), (4, 8))}


def test_saved_variants_restore_the_own_choice(fake):
    assert {s: _bands(fake, s) for s in OWN} == OWN
    fwd, bwd, n_fwd, n_bwd = _get(fake)
    assert fake.lib.gs_set_render_variants(9, 7) == 0 and _get(fake)[:2] == (9, 7)
    assert all(_bands(fake, s) == ((4, 8), (2, 8)) for s in OWN)
    assert fake.lib.gs_set_render_variants(fwd, 7) == 0  # one pinned, the other the library's
    assert {s: _bands(fake, s)[0] for s in OWN} == {s: b[0] for s, b in OWN.items()}
    for bad in ((-2, 0), (0, -2), (n_fwd, 0), (0, n_bwd)):
        assert fake.lib.gs_set_render_variants(*bad) == 1
    assert fake.lib.gs_set_render_variants(fwd, bwd) == 0
    assert {s: _bands(fake, s) for s in OWN} == OWN


def test_the_backward_hands_out_items_where_they_outnumber_the_warps(fake):
    """Kernels of their own with and without the work counter (a branch inside one
    slowed the long walks by 2.4 %)."""
    def kernels(size, count):
        views = gs.make_views([[300.0, 300.0, size[0] / 2, size[1] / 2]] * count, [size] * count)
        proj, bins, img = GsProjected(*[AT] * 5), GsBins(*[AT] * 5, 1 << 20), GsImage(*[AT] * 5)
        status, _, events = fake.run(lambda lib: lib.gs_render_bwd_splats(
            ref(proj), 1000, ref(bins), views, count, ref(img), AT, AT, None, AT, AT, None))
        assert status == 0
        return [name for what, name, _ in events if what == "launch"]
    small, large = kernels((64, 48), 1), kernels((1200, 680), 8)
    assert len(small) == 1 and "render_bwd_kernelILi1ELi8ELi32ELb0ELb1ELb0EE" in small[0]
    assert len(large) == 2 and "render_bwd_kernelILi4ELi8ELi32ELb0ELb1ELb1EE" in large[1]
