"""bd_verify_attn without an output on batches of one long sequence and short ones: the long one's
units span more segments than the short ones have tiles, and every count of segments up to the
most is merged, against the oracle; twice from one workspace."""

import numpy as np
import pytest
import torch

import oracle
import paper_2606_00144_gb300 as bd
from paper_2606_00144_gb300 import workload as W
from tests.parity import f64

pytestmark = pytest.mark.gpu

# as in test_gpu_verify_lse.py, with up to 40000 terms in partial sums of 64 keys, segments and a merge
ATOL = 2e-5


@pytest.fixture(scope="module", autouse=True)
def built():
    bd.build()
    bd.library()


@pytest.mark.parametrize("h_q,h_kv,d,lens,n_q", [
    (4, 1, 128, (40000,), 5), (2, 2, 64, (30001, 100, 700), 16), (8, 1, 128, (8, 20000, 4000), 16), (1, 1, 64, (4223,), 1)])
def test_long_sequence_among_short_ones(h_q, h_kv, d, lens, n_q):
    b, t_max = len(lens), max(lens)
    wl = W.tiny_workload(batch=b, h_q=h_q, h_kv=h_kv, head_dim=d, t_ctx=t_max, gamma=n_q, window=1, seed=9 + n_q)
    inp = W.make_layer(wl, 0, "cuda")
    g = torch.Generator(device="cuda").manual_seed(n_q)
    q = torch.randn(b, h_q, n_q, d, device="cuda", generator=g).to(torch.bfloat16)
    dl = torch.tensor(lens, dtype=torch.int32, device="cuda")
    shape = bd.make_shape(b, h_q, h_kv, d, t_max, wl.t_cap, dl)
    ws = bd.Workspace(bd.bd_workspace_size(shape, bd.BD_OP_VERIFY, 1, n_q))
    for _ in range(2):
        lse = torch.full((b, h_q, n_q), float("nan"), device="cuda")
        bd.bd_verify_attn(shape, q, n_q, inp.k_cache, None, None, lse, ws)
        torch.cuda.synchronize()
        assert ws.status() == 0
        for i, n in enumerate(lens):
            k, v = f64(inp.k_cache[i:i + 1, :, :n + n_q]), f64(inp.v_cache[i:i + 1, :, :n + n_q])
            _, ref = oracle.verify_attn(f64(q[i:i + 1]), k, v, n)
            err = np.abs(f64(lse[i:i + 1]) - ref).max()
            assert err <= ATOL, (i, err)
