"""bd_verify_attn without an output at the row counts where the kernel's operand holds four, two or
one copies of a unit's rows (32, 64 and 128 rows), each copy reducing its share of a tile's columns,
against the oracle; causal ends inside every share."""

import numpy as np
import pytest
import torch

import oracle
import paper_2606_00144_gb300 as bd
from paper_2606_00144_gb300 import workload as W
from tests.parity import f64

pytestmark = pytest.mark.gpu

ATOL = 2e-5       # as in test_gpu_verify_lse.py


@pytest.fixture(scope="module", autouse=True)
def built():
    bd.build()
    bd.library()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("group,n_q", [(4, 8), (3, 11), (1, 31), (16, 4), (5, 13), (9, 7), (8, 16)])
def test_row_counts_around_the_copies(group, n_q, ragged, d):
    lens = (2999, 5, 1300, 128 - n_q)
    b, h_kv, t_max = len(lens), 2, max(lens)
    if not ragged:
        lens = (t_max,) * b
    wl = W.tiny_workload(batch=b, h_q=group * h_kv, h_kv=h_kv, head_dim=d, t_ctx=t_max, gamma=n_q, window=1, seed=group)
    inp = W.make_layer(wl, 0, "cuda")
    g = torch.Generator(device="cuda").manual_seed(group)
    q = torch.randn(b, group * h_kv, n_q, d, device="cuda", generator=g).to(torch.bfloat16)
    dl = torch.tensor(lens, dtype=torch.int32, device="cuda") if ragged else None
    shape = bd.make_shape(b, group * h_kv, h_kv, d, t_max, wl.t_cap, dl)
    ws = bd.Workspace(bd.bd_workspace_size(shape, bd.BD_OP_VERIFY, 1, n_q))
    lse = torch.full((b, group * h_kv, n_q), float("nan"), device="cuda")
    bd.bd_verify_attn(shape, q, n_q, inp.k_cache, None, None, lse, ws)
    torch.cuda.synchronize()
    assert ws.status() == 0
    for i in range(b) if ragged else (0, b - 1):
        n = lens[i]
        k, v = f64(inp.k_cache[i:i + 1, :, :n + n_q]), f64(inp.v_cache[i:i + 1, :, :n + n_q])
        _, ref = oracle.verify_attn(f64(q[i:i + 1]), k, v, n)
        assert np.abs(f64(lse[i:i + 1]) - ref).max() <= ATOL, i
