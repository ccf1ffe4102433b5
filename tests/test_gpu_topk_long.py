"""Top-B over long middles (one thread-block cluster per unit, bd_topk_long.cu) against the
oracle, at the sizes where its route or its layout changes: one item past the register-resident
kernels, lengths that leave the last CTA of a cluster nearly or wholly empty, more items than the
cluster's registers hold (the items are then re-read in every pass), chunks with short first and
last members, sequences of unequal length (one of them within the budget) and a crowded boundary
(every middle score equal), which must keep the lowest positions."""

import numpy as np
import pytest
import torch

import oracle
import paper_2606_00144_gb300 as bd
from paper_2606_00144_gb300 import workload as W
from tests.parity import check_selection, f64

pytestmark = pytest.mark.gpu

SINK, RECENT, WINDOW = 4, 32, 8


@pytest.fixture(scope="module", autouse=True)
def built():
    bd.build()
    bd.library()


CASES = [
    # batch, h_kv, t_ctx (or lengths), budget, chunk, tied
    (1, 1, 16384 + 36 + 1, 300, 1, False),      # one item past the register-resident kernel
    (1, 2, 65536 + 36 + 1, 2048, 1, False),     # last CTA nearly empty
    (1, 1, 131072 + 36, 1024, 1, False),        # the registers of eight CTAs exactly full
    (1, 1, 131072 + 36 + 1, 1024, 1, False),    # one more: items re-read
    (40, 2, 16500, 200, 1, False),              # a batch that leaves no SMs: one CTA per unit
    (40, 2, 33000, 200, 1, False),              # the same beyond one CTA's shared memory
    (40, 2, 16500, 200, 8, False),
    (1, 1, 20000, 300, 1, True),                # all tied: exact fallback
    (1, 1, 150000, 300, 1, True),
    (1, 2, 16421, 300, 2, False),               # chunks, the first and the last short
    (1, 1, 36001, 1024, 8, False),
    (1, 1, 36001, 1024, 8, True),
    (1, 1, 140001, 500, 2, False),              # more chunks than registers: re-read
    (4, 1, (36001, 16500, 5000, 250), 300, 1, False),
    (4, 1, (36001, 16500, 5000, 250), 300, 8, False),
]


@pytest.mark.parametrize("case", CASES, ids=str)
def test_long_middle_matches_oracle(case):
    batch, h_kv, t, budget, chunk, tied = case
    lens = list(t) if isinstance(t, tuple) else [t] * batch
    t_max = max(lens)
    wl = W.tiny_workload(batch=batch, h_q=2 * h_kv, h_kv=h_kv, head_dim=64, t_ctx=t_max, budget=budget, n_sink=SINK,
                         n_recent=RECENT, window=WINDOW, gamma=1, seed=31 + t_max + chunk)
    inp = W.make_layer(wl, 0, "cuda")
    if tied:
        inp.k_cache[:, :, SINK: t_max - RECENT].zero_()
    seqs = range(batch) if batch <= 4 else (0, batch - 1)       # the oracle is slow: the outer sequences
    lse = torch.zeros(batch, wl.h_q, WINDOW, device="cuda")
    ref = {}
    for b in range(batch):
        tb = lens[b]
        k = inp.k_cache[b, :, :tb].double()
        for h in range(h_kv):                                   # carried LSE, fp64 on the device
            q = inp.q_win[b, 2 * h: 2 * h + 2].double()
            x = (q @ k[h].T) / 8.0
            pos = tb - WINDOW + torch.arange(WINDOW, device="cuda")
            x.masked_fill_(torch.arange(tb, device="cuda")[None, None] > pos[None, :, None], -torch.inf)
            lse[b, 2 * h: 2 * h + 2] = torch.logsumexp(x, -1).float()
        if b in seqs:
            K, QW = f64(inp.k_cache[b:b + 1, :, :tb]), f64(inp.q_win[b:b + 1])
            score = oracle.window_scores(QW, K, f64(lse[b:b + 1]), tb)
            idx = np.full((1, h_kv, budget), -1)
            cnt = np.zeros((1, h_kv), dtype=np.int64)
            for h in range(h_kv):
                keep = oracle.select_from_scores(score[0, h], tb, budget, SINK, RECENT, chunk)
                idx[0, h, :keep.size] = keep
                cnt[0, h] = keep.size
            ref[b] = (idx, cnt, score)
    dl = torch.tensor(lens, dtype=torch.int32, device="cuda") if isinstance(t, tuple) else None
    st = bd.SpecStep(batch, wl.h_q, h_kv, 64, t_max, wl.t_cap, budget, SINK, RECENT, WINDOW, 1, chunk, seq_lens=dl)
    for rep in range(2):                                        # the second call on a used workspace
        st.idx.fill_(-7)
        st.select(inp.k_cache, inp.q_win, lse)
        torch.cuda.synchronize()
        assert st.ws.status() == 0
        for b, (idx, cnt, score) in ref.items():
            check_selection(st.idx[b:b + 1], st.count[b:b + 1], idx, cnt, score, lens[b], budget, SINK, RECENT, chunk,
                            what=f"{case} sequence {b} rep {rep}")
            if tied:                                            # equal scores: exactly the oracle's (lowest) set
                assert np.array_equal(st.idx[b].cpu().numpy(), idx[0])
