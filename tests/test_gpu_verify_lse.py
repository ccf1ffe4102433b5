"""bd_verify_attn without an output (the block rows' normalisers only), which runs on the
window-LSE kernel, against the oracle: blocks that start on, before and after a 128-key tile
edge, fewer rows in the whole call than the kernel's 128-row operand tile, 128 rows per KV head,
a context shorter than a tile, and per-sequence lengths."""

import numpy as np
import pytest
import torch

import oracle
import paper_2606_00144_gb300 as bd
from paper_2606_00144_gb300 import workload as W
from tests.parity import f64

pytestmark = pytest.mark.gpu

# fp32 sums of at most 3000 terms, each off by a few 2^-24 from the tensor core's fp32 logits of
# |q.k|/sqrt(d) < 8 (absolute 8 * 2^-24 * sqrt(d)) and the exponential's 2 ulp
ATOL = 2e-5


@pytest.fixture(scope="module", autouse=True)
def built():
    bd.build()
    bd.library()


@pytest.mark.parametrize("b,h_q,h_kv,d,t,n_q", [
    (1, 2, 1, 64, 40, 3), (1, 1, 1, 128, 1, 1), (2, 8, 2, 128, 1408, 6), (2, 8, 2, 128, 1407, 2), (2, 8, 2, 64, 1403, 6),
    (1, 16, 2, 128, 2900, 16), (3, 4, 4, 128, 700, 128), (2, 32, 8, 128, (1500, 37), 32), (3, 6, 2, 64, (129, 128, 5), 7)])
def test_lse_only_block(b, h_q, h_kv, d, t, n_q):
    lens = list(t) if isinstance(t, tuple) else [t] * b
    t_max = max(lens)
    wl = W.tiny_workload(batch=b, h_q=h_q, h_kv=h_kv, head_dim=d, t_ctx=t_max, gamma=n_q, window=1, seed=5 + n_q)
    inp = W.make_layer(wl, 0, "cuda")
    g = torch.Generator(device="cuda").manual_seed(n_q)
    q = torch.randn(b, h_q, n_q, d, device="cuda", generator=g).to(torch.bfloat16)
    dl = torch.tensor(lens, dtype=torch.int32, device="cuda") if isinstance(t, tuple) else None
    shape = bd.make_shape(b, h_q, h_kv, d, t_max, wl.t_cap, dl)
    ws = bd.Workspace(bd.bd_workspace_size(shape, bd.BD_OP_VERIFY, 1, n_q))
    lse = torch.full((b, h_q, n_q), float("nan"), device="cuda")
    for _ in range(2):
        bd.bd_verify_attn(shape, q, n_q, inp.k_cache, None, None, lse, ws)
    torch.cuda.synchronize()
    assert ws.status() == 0
    for i, n in enumerate(lens):
        k, v = f64(inp.k_cache[i:i + 1, :, :n + n_q]), f64(inp.v_cache[i:i + 1, :, :n + n_q])
        _, ref = oracle.verify_attn(f64(q[i:i + 1]), k, v, n)
        err = np.abs(f64(lse[i:i + 1]) - ref).max()
        assert err <= ATOL, (i, err)
