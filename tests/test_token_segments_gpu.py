"""Token projections with several segments in one launch (row and column tokens of a rectangular batch, on either side of the
row count from which a segment goes to the persistent tiles by itself), and outputs that are aligned to 16 bytes only
(32-byte stores need the other form), against the CPU oracle."""
import numpy as np
import pytest
import torch

from oracle import nested_pair_oracle as orc
from paper_2609_30379_b200 import workloads as wl
from tests.parity_utils import check
from tests.test_rect_gpu import _run_block, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nt():
    from paper_2609_30379_b200 import binding
    return binding


@pytest.mark.parametrize("ln,lm", [
    ((700, 700, 700), (3, 2, 1)), ((3, 2, 1), (700, 700, 700)),      # one segment alone is long enough
    ((65,), (63,)), ((1,), (129,)), ((64, 0), (65, 7)),              # tile edges, and a last tile one segment does not have
])
def test_segments_with_rows_of_their_own(nt, ln, lm):
    _run_block(nt, "bf16", ln, lm, c_s=128, c_z=128, seed=11)


@pytest.mark.parametrize("rows,offset", [(2100, 0), (2100, 8), (2048, 16), (2047, 8)])
def test_token_update_alignment(nt, rows, offset):
    rng = np.random.default_rng(rows + offset)
    c_s, c_z = 256, 128
    m, W, x = (wl.round_to_bf16(rng.standard_normal(s).astype(np.float32) * k) for s, k in (((rows, c_z), 1.0), ((c_s, c_z), 0.1), ((rows, c_s), 1.0)))
    dev = lambda a: torch.from_numpy(a).to("cuda", torch.bfloat16)
    buf = torch.zeros(rows * c_s + 32, dtype=torch.bfloat16, device="cuda")
    x_d = buf[offset:offset + rows * c_s].view(rows, c_s)
    x_d.copy_(dev(x))
    nt.nt_token_update(dev(m), dev(W), x_d)
    torch.cuda.synchronize()
    assert float(buf[:offset].abs().sum()) == 0 and float(buf[offset + rows * c_s:].abs().sum()) == 0
    check("bf16", host(x_d), orc.token_update(x.astype(np.float64), m.astype(np.float64), W), f"token update rows={rows} offset={offset}")


@pytest.mark.parametrize("shift", [0, 16])
def test_attention_workspace_alignment(nt, shift):
    from paper_2609_30379_b200 import runner
    cfg = wl.Config("al", "bf16", (37, 215, 130), c_s=64, c_z=128, c_h=128, H=4, d=32, blocks=1, seed=77)
    inp = wl.make_inputs(cfg)
    st = runner.PairStack(cfg, cfg.lengths, inp["blocks"][:1])
    x, b = runner.to_device(inp["x"], st.dtype), st.W[0]["broadcast"]
    nt.nt_pair_broadcast(st.L, x, b["W_a"], b["W_b"], b["ln_gamma"], b["ln_beta"], 1e-5, st.z, st.workspace)
    z0 = host(st.z)
    ws = torch.empty(st.workspace.numel() * st.workspace.element_size() + 64, dtype=torch.uint8, device="cuda")[shift:]
    nt.nt_row_attn_pairbias(st.L, nt.NT_ORDER_PAIR_IJC, st.W[0]["attn"], cfg.H, cfg.d, 1e-5, st.z, ws)
    torch.cuda.synchronize()
    assert st.L.device_status() == 0
    check("bf16", host(st.z), orc.row_attn_pairbias(z0, cfg.lengths, inp["blocks"][0]["attn"], cfg.H, cfg.d), f"row attention, workspace shifted by {shift}")
