"""Register-fragment attention core when a wait runs out: its producer stops after a few key blocks (nt_debug_attn_drop), the waits
for the next block end at their limit, and the call ends with NT_ERR_TIMEOUT in the status word, nothing written outside its
buffers and the context usable."""
import pytest
import torch

from paper_2609_30379_b200 import workloads as wl

pytestmark = pytest.mark.gpu

NT_ERR_TIMEOUT = 5


@pytest.fixture(scope="module")
def nt():
    from paper_2609_30379_b200 import binding
    return binding


@pytest.mark.parametrize("blocks", [0, 1, 4])
@pytest.mark.parametrize("H,d,col", [(4, 16, False), (2, 32, True), (1, 64, False)])
def test_missing_blocks_end_in_a_timeout_status(nt, H, d, col, blocks):
    from paper_2609_30379_b200 import runner
    cfg = wl.Config("drop", "bf16", (130, 260, 33), c_s=64, c_z=64, c_h=64, H=H, d=d, blocks=1, seed=3)
    inp = wl.make_inputs(cfg)
    st = runner.PairStack(cfg, cfg.lengths, inp["blocks"])
    n, guard = st.L.T2 * 64, 4096
    z_all = torch.full((n + 2 * guard,), 7.0, dtype=torch.bfloat16, device="cuda")
    z = z_all[guard:guard + n].view(st.L.T2, 64)
    size = st.workspace.numel() * st.workspace.element_size()
    ws_all = torch.full((size + 2 * guard,), 0x5A, dtype=torch.uint8, device="cuda")
    ws = ws_all[guard:guard + size]
    z0 = torch.randn((st.L.T2, 64), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda").to(torch.bfloat16)

    def call():
        z.copy_(z0)
        if col:
            nt.nt_col_attn_pairbias(st.L, st.W[0]["attn"], H, d, 1e-5, z, ws)
        else:
            nt.nt_row_attn_pairbias(st.L, nt.NT_ORDER_PAIR_IJC, st.W[0]["attn"], H, d, 1e-5, z, ws)
        torch.cuda.synchronize()
        return z.clone()

    prev = nt.nt_attn_core_mode(1)
    try:
        good = call()
        assert st.L.device_status() == 0
        off = nt.nt_debug_attn_drop(blocks)
        try:
            call()
        finally:
            assert nt.nt_debug_attn_drop(off) == blocks and off == -1
        assert st.L.device_status() == NT_ERR_TIMEOUT
        for buf, val, size_ in ((z_all, 7.0, n), (ws_all, 0x5A, size)):
            assert bool((buf[:guard] == val).all()) and bool((buf[guard + size_:] == val).all())
        st.L.status.zero_()
        assert torch.equal(call(), good)
        assert st.L.device_status() == 0
    finally:
        nt.nt_attn_core_mode(prev)
