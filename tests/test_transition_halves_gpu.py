"""Transition kernel where its split of the hidden width can go wrong: an odd number of 32-unit halves, one half alone, and
rows whose LayerNorm scale is at the ends of its range, against the CPU oracle."""
import numpy as np
import pytest
import torch

from oracle import nested_pair_oracle as orc
from paper_2609_30379_b200 import workloads as wl
from tests.parity_utils import check
from tests.test_transition_gpu import host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c,hidden,rows,scale,eps", [
    (64, 32, 40000, 1.0, 1e-5), (128, 32, 129, 1.0, 1e-5),          # the second half of the only chunk is not there
    (64, 96, 300, 1.0, 1e-5), (128, 160, 77000, 1.0, 1e-5),         # ... of the last chunk
    (128, 1024, 257, 1.0, 1e-5),                                    # the widest hidden layer
    (128, 512, 300, 0.0, 1e-5), (128, 512, 300, 0.0, 1e-10),        # zero rows: only the offset is left, 1 / rstd small
    (128, 512, 300, 4000.0, 1e-5),                                  # 1 / rstd large
])
def test_transition_halves(c, hidden, rows, scale, eps):
    from paper_2609_30379_b200 import binding as nt
    rng = np.random.default_rng(rows)
    W = {k: wl.round_to_bf16((rng.standard_normal(shape) * std + mean).astype(np.float32)) for k, shape, std, mean in (
        ("ln_gamma", (c,), 0.1, 1.0), ("ln_beta", (c,), 0.3, 0.0), ("W_a", (hidden, c), c ** -0.5, 0.0),
        ("W_b", (hidden, c), c ** -0.5, 0.0), ("W_2", (c, hidden), hidden ** -0.5, 0.0))}
    z = wl.round_to_bf16((rng.standard_normal((rows, c)) * scale + (0.5 if scale else 0.0)).astype(np.float32))
    z_d = torch.from_numpy(z).to("cuda", torch.bfloat16)
    W_d = {k: torch.from_numpy(np.ascontiguousarray(v)).to("cuda", torch.bfloat16) for k, v in W.items()}
    ws = torch.empty(nt.nt_transition_workspace_bytes(torch.bfloat16, c, hidden, rows), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    nt.nt_pair_transition(W_d, eps, z_d, ws, status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    check("bf16", host(z_d), orc.pair_transition(z, W, eps=eps), f"transition c={c} hidden={hidden} rows={rows}")
