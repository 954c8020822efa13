"""GPU parity of the register-fragment attention core at its edges: chunks of 32 keys, blocks of 64, query quarters of 32,
query blocks of 128, row groups of two and three tiles, and rows whose scores jump by far more than the reference guess
allows (the exact path).  Every length goes to this core (nt_attn_core_mode(1)), rows and columns, with and without bias."""
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


def host(t):
    return t.detach().to(torch.float32).cpu().numpy().astype(np.float64)


def _run(nt, lengths, H, d, bias, col, z_scale=None):
    from paper_2609_30379_b200 import runner
    c = 64
    cfg = wl.Config("frag", "bf16", lengths, c_s=64, c_z=c, c_h=c, H=H, d=d, blocks=1, seed=611)
    inp = wl.make_inputs(cfg)
    W = inp["blocks"][0]["attn"]
    if not bias:
        W.pop("W_b")
    if z_scale is not None:        # larger queries and keys: neighbouring rows need references hundreds of binades apart
        W["W_q"] = wl.round_to_bf16((W["W_q"] * z_scale).astype(np.float32))
        W["W_k"] = wl.round_to_bf16((W["W_k"] * z_scale).astype(np.float32))
    st = runner.PairStack(cfg, lengths, inp["blocks"], prepare_weights=bias)
    x = runner.to_device(inp["x"], st.dtype)
    b = st.W[0]["broadcast"]
    nt.nt_pair_broadcast(st.L, x, b["W_a"], b["W_b"], b["ln_gamma"], b["ln_beta"], 1e-5, st.z, st.workspace)
    z0 = host(st.z)
    prev = nt.nt_attn_core_mode(1)
    try:
        if col:
            nt.nt_col_attn_pairbias(st.L, st.W[0]["attn"], H, d, 1e-5, st.z, st.workspace)
        else:
            nt.nt_row_attn_pairbias(st.L, nt.NT_ORDER_PAIR_IJC, st.W[0]["attn"], H, d, 1e-5, st.z, st.workspace)
        torch.cuda.synchronize()
    finally:
        nt.nt_attn_core_mode(prev)
    assert st.L.device_status() == 0
    ref = (orc.col_attn_pairbias if col else orc.row_attn_pairbias)(z0, lengths, W, H, d)
    return host(st.z), ref


@pytest.mark.parametrize("col", [False, True])
@pytest.mark.parametrize("bias", [False, True])
@pytest.mark.parametrize("H,d", [(4, 16), (2, 32), (1, 64)])
@pytest.mark.parametrize("lengths", [(1, 2, 3, 31, 32, 33), (63, 64, 65, 95, 96, 97), (127, 128, 129, 0, 161), (255, 257)])
def test_edges(nt, lengths, H, d, bias, col):
    got, ref = _run(nt, lengths, H, d, bias, col)
    check("bf16", got, ref, f"register-fragment core {lengths} {H}x{d} bias={bias} col={col}")


@pytest.mark.parametrize("col", [False, True])
@pytest.mark.parametrize("H,d", [(4, 16), (2, 32), (1, 64)])
def test_scores_beyond_the_reference_window_stay_finite(nt, H, d, col):
    """q and k x 40: scores of thousands, softmax nearly one-hot.  bf16 q, k, bias and the one-hot choice make the
    element-wise reference meaningless where two keys are close, so the result is compared in the mean: nearly one-hot
    rows that agree on their key agree to bf16 rounding, and the share that does not is bounded."""
    got, ref = _run(nt, (70, 130), H, d, True, col, z_scale=40.0)
    assert np.isfinite(got).all()
    far = np.abs(got - ref).max(axis=-1) > 0.1
    assert far.mean() < 0.2, far.mean()
