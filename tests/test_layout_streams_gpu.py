"""Layout: alignment of its arrays."""
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
