"""Input projections on either side of the tile count from which two CTAs share a tile (q | k and v | bias; a and b of the
triangle update), whole blocks against the CPU oracle: one tile, the last lengths below and the first above the line."""
import pytest

from paper_2609_30379_b200 import workloads as wl
from tests.test_parity_gpu import run_block_teacher_forced

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nt():
    from paper_2609_30379_b200 import binding
    return binding


@pytest.mark.parametrize("c,H,d", [(128, 4, 32), (64, 4, 16), (128, 2, 32)])
@pytest.mark.parametrize("lengths", [(3,), (96,), (97,), (98,), (64, 0, 72)])
def test_blocks_around_the_split(nt, lengths, c, H, d):
    cfg = wl.Config("split", "bf16", lengths, c_s=64, c_z=c, c_h=c, H=H, d=d, blocks=1, seed=911)
    run_block_teacher_forced(nt, cfg, wl.make_inputs(cfg), full_samples=range(cfg.B))
