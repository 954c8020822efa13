"""Layout on streams: memory that work on the current stream still reads, offsets built on another stream, capture, alignment."""
import numpy as np
import pytest
import torch

from oracle import nested_pair_oracle as orc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nt():
    from paper_2609_30379_b200 import binding
    return binding


def _same(L, lengths):
    want = orc.offsets_only(lengths)
    np.testing.assert_array_equal(L.tok_off.cpu().numpy(), want[0])
    np.testing.assert_array_equal(L.pair_off.cpu().numpy(), want[1])
    assert L.row_splits.cpu().numpy()[-1] == sum(n * n for n in lengths)
    np.testing.assert_array_equal(L.lengths_d.cpu().numpy(), lengths)
    assert L.device_status() == 0


@pytest.mark.parametrize("B", range(0, 10))
def test_every_array_is_aligned(nt, B):
    lengths = tuple(range(3, 3 + B))
    L = nt.Layout(lengths)
    assert all(t.data_ptr() % 16 == 0 for t in (L.status, L.lengths_d, L.tok_off, L.pair_off, L.row_splits) if t.numel())
    _same(L, lengths)


def test_side_stream_waits_for_the_memory_it_gets(nt):
    """A block of the allocator is freed while a copy from it is queued behind a long sleep; the Layout built on a side stream
    gets that block."""
    lengths = (5, 9, 30)
    side = torch.cuda.Stream()
    probe = nt.Layout(lengths, stream=side)
    torch.cuda.synchronize()
    n = probe.status.untyped_storage().nbytes() // 8
    del probe
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    old = torch.full((n,), 7, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    torch.cuda._sleep(200_000_000)
    seen = old.clone()
    where = old.data_ptr()
    del old
    L = nt.Layout(lengths, stream=side)
    assert L.status.data_ptr() == where      # or the test shows nothing
    torch.cuda.synchronize()
    assert bool((seen == 7).all())
    _same(L, lengths)


def test_rebuild_on_a_side_stream(nt):
    side = torch.cuda.Stream()
    L = nt.Layout((5, 9, 30), stream=side)
    torch.cuda._sleep(50_000_000)
    L.rebuild((30, 5, 9), stream=side)
    torch.cuda.synchronize()
    _same(L, (30, 5, 9))


def test_not_during_a_capture(nt):
    x = torch.zeros(4, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        x.add_(1)
        with pytest.raises(RuntimeError):
            nt.Layout((5, 9))
    g.replay()
    torch.cuda.synchronize()
    assert float(x[0]) == 1.0
    _same(nt.Layout((5, 9)), (5, 9))
