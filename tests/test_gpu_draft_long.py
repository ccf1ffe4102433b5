"""Drafter passes over views long enough for the draft kernel's wide instances (160-row tiles,
several thread-block clusters per unit), against the oracle: slices of one row more and less
than a tile, counts that leave CTAs and whole clusters without entries, every group instance, both
head sizes, per-sequence lengths, both orders of the dependency wait, a workspace without
room for the clusters' partials, and the allocation-free call."""

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


@pytest.mark.parametrize("b,h_q,h_kv,d,t,budget,counts", [
    (1, 8, 1, 128, 9000, 8192, (8192,)), (1, 2, 2, 64, 9000, 8192, (8192, 5)), (1, 8, 2, 128, 5200, 3835, (3835, 1)),
    (1, 16, 4, 64, 4000, 3841, (3841, 0, 160, 161)), (2, 16, 1, 128, 3000, 2560, (2560, 1279)),
    (2, 32, 8, 128, 4300, 4096, (4096,) * 16), (3, 32, 4, 128, (6000, 2500, 4100), 2400, (2400,) * 12)])
def test_long_views(b, h_q, h_kv, d, t, budget, counts):
    lens = list(t) if isinstance(t, tuple) else [t] * b
    wl = W.tiny_workload(batch=b, h_q=h_q, h_kv=h_kv, head_dim=d, t_ctx=max(lens), budget=budget, gamma=3, seed=budget)
    inp = W.make_layer(wl, 0, "cuda")
    rng = np.random.default_rng(budget)
    idx = np.full((b, h_kv, budget), -1, np.int32)
    cnt = np.array(counts, np.int32).reshape(b, h_kv)
    for i in range(b):
        for h in range(h_kv):
            idx[i, h, :cnt[i, h]] = np.sort(rng.permutation(lens[i])[:cnt[i, h]])
    di, dc = torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda()
    dl = torch.tensor(lens, dtype=torch.int32, device="cuda") if isinstance(t, tuple) else None
    shape = bd.make_shape(b, h_q, h_kv, d, max(lens), wl.t_cap, dl)
    full = bd.bd_workspace_size(shape, bd.BD_OP_DRAFT, budget, wl.gamma)
    small = 256 + -(-b * h_kv * 4 // 256) * 256      # the status word and the counters only
    o = torch.empty(b, h_q, d, dtype=torch.bfloat16, device="cuda")
    lse = torch.empty(b, h_q, device="cuda")
    for j, (size, flags) in enumerate([(full, 0), (full, bd.BD_DRAFT_VIEW_READY), (small, 0)]):
        ws = bd.Workspace(size)
        want = [oracle.draft_attn(f64(inp.q_draft[j][i:i + 1]), f64(inp.k_cache[i:i + 1]), f64(inp.v_cache[i:i + 1]),
                                  idx[i:i + 1], cnt[i:i + 1], lens[i], j) for i in range(b)]

        def check(what):
            torch.cuda.synchronize()
            for i, (ro, rl) in enumerate(want):
                check_attention(o[i:i + 1], lse[i:i + 1], ro, rl, f"draft long {what} B={budget} T={lens[i]} j={j}")

        for rep in range(2):
            o.fill_(float("nan"))
            bd.bd_draft_attn(shape, inp.q_draft[j], inp.k_cache, inp.v_cache, di, dc, budget, j, o, lse, ws, flags=flags)
            check(f"ws {size}")
        assert ws.status() == 0
        if flags == 0:
            o.fill_(float("nan"))
            bd.bd_draft_attn_static(shape, inp.q_draft[j], inp.k_cache, inp.v_cache, di, dc, budget, j, o, lse)
            check("static")
