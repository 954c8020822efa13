"""Register-fragment attention core where the reference guess fails: neighbouring rows whose log-sums lie more than a hundred nats
apart (the guess may be off by 42 downwards and 97 upwards), element by element against the CPU oracle.

The states are made for it: balanced +-1 codes, so that a query's own key wins by at least 16 nats (32 with heads of 16) over
every other and the weights are one-hot whatever the rounding of q and k; the amplitude changes from row to row.  The bound is that
of an ordinary row: the state's rounding to bf16 (2^-8 of the value) plus 4 % of the update's spread for the 16-bit
intermediates.  Taking another query's, key's or bias element's place would be off by the update itself."""
import numpy as np
import pytest
import torch

from oracle import nested_pair_oracle as orc
from paper_2609_30379_b200 import workloads as wl

pytestmark = pytest.mark.gpu

SHARPNESS = 8.0                       # of q and of k
AMPLITUDES = np.sqrt([0.5, 1.0, 1.9])


@pytest.fixture(scope="module")
def nt():
    from paper_2609_30379_b200 import binding
    return binding


def host(t):
    return t.detach().to(torch.float32).cpu().numpy().astype(np.float64)


def _codes(rng, n, d):
    """n balanced +-1 codes of d elements, distinct if there are enough of them"""
    seen, out = set(), []
    base = np.repeat([1.0, -1.0], d // 2)
    while len(out) < n:
        c = rng.permutation(base)
        if d > 16 or len(seen) > 12000 or c.tobytes() not in seen:
            seen.add(c.tobytes())
            out.append(c)
    return np.array(out)


def _position_codes(rng, n, H, d):
    """[n, n, H d]: no two positions of a row or of a column share a head's code"""
    heads = []
    for _ in range(H):
        table = _codes(rng, 4096, d)
        i, j = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
        heads.append(table[(i * 137 + j) % 4096])
    return np.concatenate(heads, axis=-1)


def _pair_state(rng, lengths, H, d, col):
    rows = []
    for n in lengths:
        if n == 0:
            continue
        a = AMPLITUDES[rng.integers(0, 3, n)]
        a = np.broadcast_to(a[None, :] if col else a[:, None], (n, n))[..., None]
        code = _position_codes(rng, n, H, d)
        fill = _codes(rng, n * n, 64).reshape(n, n, 64)
        rows.append(np.concatenate([a * code, np.sqrt(2.0 - a * a) * fill], axis=-1).reshape(n * n, 128))
    return wl.round_to_bf16(np.concatenate(rows).astype(np.float32))


def _weights(rng, W, bias):
    eye = np.concatenate([np.eye(64), np.zeros((64, 64))], axis=1).astype(np.float32)
    W["ln_gamma"], W["ln_beta"] = np.ones(128, np.float32), np.zeros(128, np.float32)
    W["W_q"] = W["W_k"] = eye * np.float32(SHARPNESS)
    W["W_v"] = eye[rng.permutation(64)] * rng.choice(np.array([-1, 1], np.float32), 64)[:, None]
    if not bias:
        W.pop("W_b")
    return W


def _check(got, z0, ref, what):
    assert np.isfinite(got).all(), what
    update = float(np.sqrt(np.mean((ref - z0) ** 2)))
    worst = float((np.abs(got - ref) - 2.0 ** -8 * np.abs(ref)).max()) / update
    assert worst <= 0.04, f"{what}: {worst:.4f} of the update's spread"


@pytest.mark.parametrize("col", [False, True])
@pytest.mark.parametrize("bias", [False, True])
@pytest.mark.parametrize("H,d", [(4, 16), (2, 32), (1, 64)])
def test_pair_rows_far_apart(nt, H, d, bias, col):
    from paper_2609_30379_b200 import runner
    lengths = (70, 130, 0, 33)
    rng = np.random.default_rng(d + 100 * col)
    cfg = wl.Config("window", "bf16", lengths, c_s=64, c_z=128, c_h=128, H=H, d=d, blocks=1, seed=19)
    inp = wl.make_inputs(cfg)
    W = _weights(rng, inp["blocks"][0]["attn"], bias)
    st = runner.PairStack(cfg, lengths, inp["blocks"], prepare_weights=bias)
    z0 = _pair_state(rng, lengths, H, d, col)
    z = runner.to_device(z0, torch.bfloat16)
    prev = nt.nt_attn_core_mode(1)
    try:
        if col:
            nt.nt_col_attn_pairbias(st.L, st.W[0]["attn"], H, d, 1e-5, z, st.workspace)
        else:
            nt.nt_row_attn_pairbias(st.L, nt.NT_ORDER_PAIR_IJC, st.W[0]["attn"], H, d, 1e-5, z, st.workspace)
    finally:
        nt.nt_attn_core_mode(prev)
    assert st.L.device_status() == 0
    z0 = np.asarray(z0, dtype=np.float64)
    ref = (orc.col_attn_pairbias if col else orc.row_attn_pairbias)(z0, lengths, W, H, d)
    _check(host(z), z0, ref, f"{H}x{d} bias={bias} col={col}")


@pytest.mark.parametrize("H,d", [(4, 16), (2, 32), (1, 64), (12, 64)])
def test_token_rows_far_apart(nt, H, d):
    """Token order without LayerNorm: the samples' amplitudes differ by powers of two, so q, k and v are exact."""
    lengths = (70, 130, 1, 45, 260, 64)
    c = H * d
    rng = np.random.default_rng(d)
    x0 = np.concatenate([s * np.concatenate([_codes(rng, n, d) for _ in range(H)], axis=1)
                         for n, s in zip(lengths, (1.0, 4.0, 0.5, 2.0, 0.5, 4.0))]).astype(np.float32)
    W = dict(W_q=np.eye(c, dtype=np.float32) * 8, W_k=np.eye(c, dtype=np.float32) * 8,
             W_v=np.eye(c, dtype=np.float32)[rng.permutation(c)],
             W_o=wl.round_to_bf16((rng.standard_normal((c, c)) * c ** -0.5).astype(np.float32)))
    L = nt.Layout(lengths)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", torch.bfloat16)  # noqa: E731
    x, Wd = dev(x0), {k: dev(v) for k, v in W.items()}
    ws = torch.empty(nt.nt_workspace_bytes(nt.NT_OP_ROW_ATTN, nt.NT_BF16, nt.NT_ORDER_TOKEN_NC, L.lengths_h, (c, c, 0, H, d)),
                     dtype=torch.uint8, device="cuda")
    nt.nt_row_attn_pairbias(L, nt.NT_ORDER_TOKEN_NC, Wd, H, d, 1e-5, x, ws)
    assert L.device_status() == 0
    x0 = x0.astype(np.float64)
    _check(host(x), x0, orc.row_attn_pairbias(x0, lengths, W, H, d, order="token"), f"token order {H}x{d}")


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("H,d", [(4, 16), (2, 32), (1, 64)])
def test_a_sample_without_finite_scores_leaves_the_others(nt, H, d, bad):
    """The references that a warp takes from such rows must not reach the rows after them: the other samples are computed as if
    alone, and in the ordinary way (a sample's rows on the exact path would take several times as long; the line is at three)."""
    from paper_2609_30379_b200 import runner
    lengths = (240, 300, 250)
    cfg = wl.Config("nan", "bf16", lengths, c_s=64, c_z=128, c_h=128, H=H, d=d, blocks=1, seed=29)
    inp = wl.make_inputs(cfg)
    st = runner.PairStack(cfg, lengths, inp["blocks"])
    first = lengths[0] ** 2
    z0 = torch.randn((st.L.T2, 128), generator=torch.Generator(device="cuda").manual_seed(2), device="cuda").to(torch.bfloat16)
    zbad = z0.clone()
    zbad[:first] = bad
    prev = nt.nt_attn_core_mode(1)
    try:
        outs, ms = [], []
        for start in (z0, z0, zbad):
            z = start.clone()
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            nt.nt_row_attn_pairbias(st.L, nt.NT_ORDER_PAIR_IJC, st.W[0]["attn"], H, d, 1e-5, z, st.workspace)
            e[1].record()
            torch.cuda.synchronize()
            outs.append(z)
            ms.append(e[0].elapsed_time(e[1]))
    finally:
        nt.nt_attn_core_mode(prev)
    assert st.L.device_status() == 0
    assert bool(torch.isnan(outs[2][:first].float()).any(dim=1).all())
    diff = (outs[2][first:].float() - outs[1][first:].float()).abs()
    assert bool(torch.isfinite(diff).all())
    # another reference moves a weight by a rounding of bf16: a few 2^-9 of an update below 2, and the state's own rounding
    assert float(diff.max()) <= 0.05
    assert ms[2] <= 3 * ms[1], ms
