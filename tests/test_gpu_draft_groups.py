"""Drafter passes of GQA groups of 8 and more over batches that fill the GPU, where rank 0's partials leave
room for fewer CTAs on an SM and the view is split over smaller clusters, against the oracle."""

import numpy as np
import pytest
import torch

import oracle
import paper_2606_00144_gb300 as bd
from paper_2606_00144_gb300 import workload as W
from tests.parity import check_attention, f64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    bd.build()
    bd.library()


@pytest.mark.parametrize("b,group,h_kv,d,budget", [
    (4, 8, 8, 128, 1024), (4, 8, 8, 128, 2048), (6, 16, 8, 128, 512), (4, 16, 8, 128, 1100), (2, 9, 8, 128, 900),
    (6, 16, 8, 64, 2048)])
def test_wide_groups(b, group, h_kv, d, budget):
    t, h_q, j = budget + 300, group * h_kv, 1
    wl = W.tiny_workload(batch=b, h_q=h_q, h_kv=h_kv, head_dim=d, t_ctx=t, budget=budget, gamma=2, window=1, seed=budget)
    inp = W.make_layer(wl, 0, "cuda")
    rng = np.random.default_rng(budget)
    idx = np.stack([np.sort(rng.permutation(t)[:budget]) for _ in range(b * h_kv)])
    idx = idx.astype(np.int32).reshape(b, h_kv, budget)
    cnt = np.full((b, h_kv), budget, np.int32)
    di, dc = torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda()
    shape = bd.make_shape(b, h_q, h_kv, d, t, wl.t_cap)
    ws = bd.Workspace(bd.bd_workspace_size(shape, bd.BD_OP_DRAFT, budget, 2))
    o = torch.full((b, h_q, d), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((b, h_q), float("nan"), device="cuda")
    bd.bd_draft_attn(shape, inp.q_draft[j], inp.k_cache, inp.v_cache, di, dc, budget, j, o, lse, ws)
    torch.cuda.synchronize()
    assert ws.status() == 0
    ro, rl = oracle.draft_attn(f64(inp.q_draft[j]), f64(inp.k_cache), f64(inp.v_cache), idx, cnt, t, j)
    check_attention(o, lse, ro, rl, f"draft G={group} units={b * h_kv} B={budget} d={d}")
