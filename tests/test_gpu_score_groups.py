"""Selection with more window rows than four score accumulators hold (two, shared by the
kernel's four epilogue groups) over enough keys that every group takes several tiles of a CTA's
range: each tile's scores must come from its own accumulator phase."""

import numpy as np
import pytest
import torch

import oracle
import paper_2606_00144_gb300 as bd
from paper_2606_00144_gb300 import workload as W
from tests.parity import check_selection, f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,group,lens,ragged", [(128, 8, (16001,) * 4, False), (64, 8, (16001,) * 4, False),
                                                 (128, 5, (16001,) * 4, False), (128, 8, (20000, 9000, 15000, 20000), True)])
def test_two_accumulators_over_many_tiles(d, group, lens, ragged):
    bd.build()
    b, h_kv, window, budget, sink, recent, t = len(lens), 4, 32, 512, 4, 64, max(lens)
    wl = W.tiny_workload(batch=b, h_q=group * h_kv, h_kv=h_kv, head_dim=d, t_ctx=t, budget=budget, n_sink=sink,
                         n_recent=recent, window=window, gamma=1, seed=group + d)
    inp = W.make_layer(wl, 0, "cuda")
    lse = torch.empty(b, wl.h_q, window, device="cuda")
    for i, n in enumerate(lens):
        for h in range(h_kv):
            x = inp.q_win[i, h * group:(h + 1) * group].double() @ inp.k_cache[i, h, :n].double().T / d ** 0.5
            pos = n - window + torch.arange(window, device="cuda")
            x.masked_fill_(torch.arange(n, device="cuda")[None, None] > pos[None, :, None], -torch.inf)
            lse[i, h * group:(h + 1) * group] = torch.logsumexp(x, -1).float()
    dl = torch.tensor(lens, dtype=torch.int32, device="cuda") if ragged else None
    st = bd.SpecStep(b, wl.h_q, h_kv, d, t, wl.t_cap, budget, sink, recent, window, 1, 1, seq_lens=dl)
    for rep in range(2):
        st.idx.fill_(-7)
        st.select(inp.k_cache, inp.q_win, lse)
        torch.cuda.synchronize()
        assert st.ws.status() == 0
    for i in (0, b - 1):
        n = lens[i]
        score = oracle.window_scores(f64(inp.q_win[i:i + 1]), f64(inp.k_cache[i:i + 1, :, :n]), f64(lse[i:i + 1]), n)
        idx = np.stack([oracle.select_from_scores(score[0, h], n, budget, sink, recent, 1) for h in range(h_kv)])[None]
        cnt = np.full((1, h_kv), budget)
        check_selection(st.idx[i:i + 1], st.count[i:i + 1], idx, cnt, score, n, budget, sink, recent,
                        what=f"group {group} d{d} sequence {i}")
