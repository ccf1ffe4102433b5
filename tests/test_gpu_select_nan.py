"""Keys that hold NaN score 0: they are kept only where nothing else is left, no more positions than
the budget are written (the words past the output stay as they are), and the other keys are ranked
as without them.  Each top-B kernel: token and chunk level, one CTA and a cluster per unit."""

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


@pytest.mark.parametrize("batch,t,budget,chunk", [
    (1, 700, 100, 1), (1, 5000, 300, 1), (1, 16000, 300, 1), (1, 5000, 300, 8), (1, 16000, 300, 2),
    (40, 17000, 300, 1), (1, 40000, 300, 1), (1, 40000, 304, 8), (1, 140000, 300, 1)])
def test_nan_keys_are_never_ranked_above_others(batch, t, budget, chunk):
    wl = W.tiny_workload(batch=batch, h_q=2, h_kv=1, head_dim=64, t_ctx=t, budget=budget, n_sink=SINK,
                         n_recent=RECENT, window=WINDOW, gamma=1, seed=5 + t + chunk)
    inp = W.make_layer(wl, 0, "cuda")
    lse = torch.full((batch, 2, WINDOW), 9.0, device="cuda")
    bad = torch.arange(SINK + 3, t - RECENT, 97, device="cuda")
    clean = f64(inp.k_cache[:1, :, :t])
    inp.k_cache[:, :, bad] = float("nan")
    score = oracle.window_scores(f64(inp.q_win[:1]), clean, f64(lse[:1]), t)
    score[0, 0, bad.cpu().numpy()] = 0.0
    keep = oracle.select_from_scores(score[0, 0], t, budget, SINK, RECENT, chunk)
    idx = np.full((1, 1, budget), -1)
    idx[0, 0, :keep.size] = keep
    st = bd.SpecStep(batch, 2, 1, 64, t, wl.t_cap, budget, SINK, RECENT, WINDOW, 1, chunk)
    room = torch.full((batch * budget + 4096,), -7, dtype=torch.int32, device="cuda")
    st.idx = room[:batch * budget].view(batch, 1, budget)
    st.select(inp.k_cache, inp.q_win, lse)
    torch.cuda.synchronize()
    assert st.ws.status() == 0
    assert bool((room[batch * budget:] == -7).all())
    check_selection(st.idx[:1], st.count[:1], idx, np.array([[keep.size]]), score, t, budget, SINK, RECENT, chunk,
                    what=f"NaN keys T={t} chunk={chunk}")
    assert bool((st.count <= budget).all())
