"""gs_bin_sort from two host threads at once, on streams and buffers of their
own: views of more than 12,288 tiles, of different tile counts, need more shared
memory for the counting blocks than a kernel gets by default, and the limit that
is raised for them belongs to the kernel, not to the call.  Every call returns
GS_OK and every list equals the one a single thread made."""
import threading

import pytest
import torch

import paper_2405_19614_gb300 as gs

pytestmark = pytest.mark.gpu

N, CALLS = 400_000, 200


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2405_19614_gb300.build import build
    build()


def _rasterizer(w, h, seed):
    """N drawn one-tile records on a w x h view of 8x8 tiles."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    tx, ty = -(-w // 8), -(-h // 8)
    r = gs.Rasterizer(N, 0, [[300.0, 300.0, w / 2, h / 2]], [(w, h)], pair_capacity=N, tile=(8, 8))
    t = torch.randint(0, tx * ty, (N,), generator=g, device="cuda")
    corner = ((t % tx) | (t // tx) << 16).int()
    r.proj["rect"].view(-1)[:2 * N].view(N, 2).copy_(torch.stack([corner, corner], 1))
    r.proj["tile_mask"].view(-1)[:N].fill_(1)
    r.proj["tiles_touched"].view(-1)[:N].fill_(1)
    r.proj["rec"].view(-1)[:12 * N].view(N, 12)[:, 2] = 0.5 + 8 * torch.rand(N, generator=g, device="cuda")
    return r


def _bin(r, stream=None):
    gs.gs_bin_sort(r.proj, r.n, r.views, r.bins, r.workspace, stream)


def test_two_threads_with_different_shared_memory_sizes():
    rasts = [_rasterizer(1280, 720, 1), _rasterizer(1200, 680, 2)]  # 14,400 and 12,750 tiles
    want = []
    for r in rasts:
        _bin(r)
        want.append({k: r.bins[k].clone() for k in ("keys", "vals", "ranges", "n_pairs", "status")})
    torch.cuda.synchronize()
    faults, start = [], threading.Barrier(2)

    def work(r, w):
        try:
            s = torch.cuda.Stream()
            wrong = torch.zeros(1, dtype=torch.int64, device="cuda")
            torch.cuda.synchronize()
            start.wait()
            with torch.cuda.stream(s):
                for _ in range(CALLS):
                    for k in ("keys", "vals", "ranges"):
                        r.bins[k].fill_(-1)
                    _bin(r, s)
                    for k in w:
                        wrong += (r.bins[k] != w[k]).sum()
            s.synchronize()
            if int(wrong):
                faults.append(f"{int(wrong)} entries differ")
        except Exception as e:  # a refused call
            faults.append(repr(e))

    threads = [threading.Thread(target=work, args=a) for a in zip(rasts, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not faults, faults
