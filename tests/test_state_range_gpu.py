"""The output stages meet the bf16 state itself, so their gates have to hold over its range: rows whose mean or spread lies
beyond the largest fp16 number, against the CPU oracle, and rows whose sum of squares lies beyond the largest float.

The bound: rounding the state to bf16 (2^-9 of the value; 2^-8 allows for a result that sits on the other side of a tie)
plus 4 % of the update's spread for the 16-bit intermediates of the update (each within 2^-9 of itself, a few of them in a
row, the worst of tens of thousands of elements)."""
import numpy as np
import pytest
import torch

from oracle import nested_pair_oracle as orc
from paper_2609_30379_b200 import workloads as wl

pytestmark = pytest.mark.gpu

LENGTHS = (70, 5, 131)


@pytest.fixture(scope="module")
def nt():
    from paper_2609_30379_b200 import binding
    return binding


def host(t):
    return t.detach().to(torch.float32).cpu().numpy().astype(np.float64)


def _run(nt, call, c, H, d, mean, spread):
    from paper_2609_30379_b200 import runner
    cfg = wl.Config("range", "bf16", LENGTHS, c_s=64, c_z=c, c_h=c, H=H, d=d, blocks=1, seed=313)
    inp = wl.make_inputs(cfg)
    rng = np.random.default_rng(17)
    tri = call.startswith("tri")
    W = inp["blocks"][0]["trimul" if tri else "attn"]
    # an update as large as the state, and LayerNorm offsets that its gate can feel
    W["W_o"] = wl.round_to_bf16((W["W_o"] * np.float32(min(spread, 1e6))).astype(np.float32))
    for k in ("ln_in_beta",) if tri else ("ln_beta",):
        W[k] = wl.round_to_bf16(rng.standard_normal(c).astype(np.float32))
    st = runner.PairStack(cfg, LENGTHS, inp["blocks"])
    z0 = wl.round_to_bf16((mean + spread * rng.standard_normal((st.L.T2, c))).astype(np.float32))
    z = runner.to_device(z0, torch.bfloat16)
    w = st.W[0]["trimul" if tri else "attn"]
    if tri:
        (nt.nt_tri_mul_out if call == "tri_out" else nt.nt_tri_mul_in)(st.L, w, 1e-5, z, st.workspace)
    elif call == "col":
        nt.nt_col_attn_pairbias(st.L, w, H, d, 1e-5, z, st.workspace)
    else:
        nt.nt_row_attn_pairbias(st.L, nt.NT_ORDER_PAIR_IJC, w, H, d, 1e-5, z, st.workspace)
    torch.cuda.synchronize()
    assert st.L.device_status() == 0
    return host(z), np.asarray(z0, dtype=np.float64), W


@pytest.mark.parametrize("call", ["row", "col", "tri_out", "tri_in"])
@pytest.mark.parametrize("c,H,d", [(128, 4, 32), (64, 4, 16)])
@pytest.mark.parametrize("mean,spread", [(1e5, 5e4), (0.0, 1e5), (-7e4, 2e4)])
def test_rows_beyond_fp16(nt, call, c, H, d, mean, spread):
    got, z0, W = _run(nt, call, c, H, d, mean, spread)
    if call.startswith("tri"):
        ref = (orc.tri_mul_out if call == "tri_out" else orc.tri_mul_in)(z0, LENGTHS, W)
    else:
        ref = (orc.col_attn_pairbias if call == "col" else orc.row_attn_pairbias)(z0, LENGTHS, W, H, d)
    assert np.isfinite(got).all()
    update = float(np.sqrt(np.mean((ref - z0) ** 2)))
    worst = float((np.abs(got - ref) - 2.0 ** -8 * np.abs(ref)).max()) / update
    assert worst <= 0.04, f"{call} c={c} mean={mean} spread={spread}: {worst:.4f} of the update's spread"


def test_rows_beyond_the_float_range_of_squares_stay_finite(nt):
    got, _, _ = _run(nt, "row", 128, 4, 32, 0.0, 1e19)
    assert np.isfinite(got).all()
