"""What a synchronous sort waits for, and what it leaves in flight."""
import time

import pytest
import torch

from paper_2501_12369_gb300 import darb, synth

from gpu_helpers import to_np

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2501_12369_gb300 import build
    build.build()


def _view(n=200000, width=640, height=360, tile=16):
    s = synth.cluster_scene(n, seed=2, sh_degree=0)
    cam = synth.fibonacci_cameras(16, 6.0, width, height, 500.0)[3]
    proj = darb.darb_preprocess(darb.splats_to_device(s), cam, darb.darb_kernel_defaults("half_cosine"), tile)

    def sort(capacity, sync, out=None, ws=None):
        if ws is None:
            ws = torch.empty(darb.darb_bin_sort_workspace_size(n, tile, cam, capacity), dtype=torch.uint8, device="cuda")
        return darb.darb_bin_sort(proj, n, tile, cam, ws, capacity, out, sync=sync), ws
    return sort


def test_synchronous_sort_does_not_wait_for_another_streams_sort():
    """An asynchronous sort is queued behind long work of another stream; the library's side stream then holds
    its tile counts.  A synchronous sort waits for its own count alone."""
    sort = _view()
    m = sort(1 << 21, True)[0].M
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        torch.cuda._sleep(int(1.0e9))  # half a second at most clock rates
        done = torch.cuda.Event()
        kept = sort(1 << 21, False)
        done.record()
    t = time.perf_counter()
    got = sort(1 << 21, True)[0].M
    t = time.perf_counter() - t
    pending = not done.query()
    torch.cuda.synchronize()
    assert got == m and pending, f"the synchronous sort returned after {t:.3f} s, with the other stream's"
    assert int(to_np(kept[0].num_instances)[0]) == m


@pytest.mark.parametrize("n,capacity", [(2000, 1 << 12), (200000, 1 << 18), (200000, 1)])
def test_overflow_leaves_nothing_in_flight(n, capacity):
    """After DARB_ERR_CAPACITY the buffers may be freed, or used on another stream at once.  The tile counts (and with
    them the rest of the sort) are held up by another stream's."""
    sort = _view(n)
    first, _ = sort(1 << 21, True)
    m = first.M
    assert m > capacity
    ref = to_np(first.values)[:m], to_np(first.ranges)
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        torch.cuda._sleep(int(2.0e8))  # a tenth of a second
        kept = sort(1 << 21, False)
    with pytest.raises(darb.DarbError) as e:
        sort(capacity, True)
    assert torch.cuda.current_stream().query()
    assert e.value.status == 3 and e.value.M == m
    with torch.cuda.stream(torch.cuda.Stream()):
        again, _ = sort(m, True)
    torch.cuda.synchronize()
    for b in (again, kept[0]):
        assert (to_np(b.values)[:m] == ref[0]).all() and (to_np(b.ranges) == ref[1]).all()
