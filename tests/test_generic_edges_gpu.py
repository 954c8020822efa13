"""Shape-generic reduction and accumulated projection at the edges of their loops: groups around multiples of the eight rows that
are in flight, outputs around multiples of the 64 columns of a tile, one row more or less than a block, against the CPU oracle."""
import numpy as np
import pytest
import torch

from oracle import nested_pair_oracle as orc
from paper_2609_30379_b200 import workloads as wl
from tests.parity_utils import check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nt():
    from paper_2609_30379_b200 import binding
    return binding


def _dev(a, dtype):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", torch.float32 if dtype == "f32" else torch.bfloat16)


def _host(t):
    return t.detach().to(torch.float32).cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("C", [256, 260, 300, 1030])
@pytest.mark.parametrize("op", ["mean", "sum"])
def test_wide_groups(nt, dtype, C, op):
    sizes = (0, 1, 7, 8, 9, 0, 15, 16, 17, 40)
    splits = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    v = np.random.default_rng(C).standard_normal((int(splits[-1]), C)).astype(np.float32)
    if dtype == "bf16":
        v = wl.round_to_bf16(v)
    out = torch.full((len(sizes), C), 3.0, dtype=torch.float32 if dtype == "f32" else torch.bfloat16, device="cuda")
    nt.nt_segment_reduce(nt.NT_REDUCE_MEAN if op == "mean" else nt.NT_REDUCE_SUM, torch.from_numpy(splits).cuda(), _dev(v, dtype), out)
    ref = orc.segment_reduce(v.astype(np.float64), splits, op)
    if dtype == "f32":
        check("f32", _host(out), ref, f"{op} C={C}")
    else:      # one rounding of a float sum
        assert (np.abs(_host(out) - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-5).all()


@pytest.mark.parametrize("rows", [1, 63, 64, 65, 200])
@pytest.mark.parametrize("c_z,c_s", [(16, 32), (19, 33), (64, 64), (96, 100), (5, 1), (130, 65)])
def test_accumulated_projection(nt, rows, c_z, c_s):
    rng = np.random.default_rng(rows + c_s)
    m, W, x = (rng.standard_normal(s).astype(np.float32) for s in ((rows, c_z), (c_s, c_z), (rows, c_s)))
    buf = torch.full((rows * c_s + 64,), 7.0, device="cuda")
    xd = buf[32:32 + rows * c_s].view(rows, c_s)
    xd.copy_(_dev(x, "f32"))
    nt.nt_token_update(_dev(m, "f32"), _dev(W, "f32"), xd)
    check("f32", _host(xd), orc.token_update(x.astype(np.float64), m.astype(np.float64), W), f"{rows} rows, {c_z} -> {c_s}")
    assert bool((buf[:32] == 7.0).all()) and bool((buf[32 + rows * c_s:] == 7.0).all())


@pytest.mark.parametrize("rows", [1, 65, 200])
@pytest.mark.parametrize("c_z,c_s", [(19, 33), (96, 100), (5, 1), (130, 65)])      # widths that the shape-generic kernel takes
def test_accumulated_projection_bf16(nt, rows, c_z, c_s):
    rng = np.random.default_rng(rows + c_s)
    m, W, x = (wl.round_to_bf16(rng.standard_normal(s).astype(np.float32)) for s in ((rows, c_z), (c_s, c_z), (rows, c_s)))
    xd = _dev(x, "bf16")
    nt.nt_token_update(_dev(m, "bf16"), _dev(W, "bf16"), xd)
    ref = orc.token_update(x.astype(np.float64), m.astype(np.float64), W)
    # float products and sums of bf16 values, rounded to bf16 once
    assert (np.abs(_host(xd) - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-4).all()
