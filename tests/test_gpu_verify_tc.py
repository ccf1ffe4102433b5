"""Verify blocks with many query rows per KV head, which run on the tcgen05 kernel, against the
oracle: row counts around one and two 128-row operand tiles and their quarters, several chunks,
contexts of less than a tile and around tile ends (with the causal block across one), one job
per accumulator and none, per-sequence lengths, and scores that keep growing along the context
(the running maximum moves, and the accumulators are rescaled)."""

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


def block(b, h_q, h_kv, d, t, n_q, grow=0.0, repeat=2):
    lens = list(t) if isinstance(t, tuple) else [t] * b
    t_max = max(lens)
    wl = W.tiny_workload(batch=b, h_q=h_q, h_kv=h_kv, head_dim=d, t_ctx=t_max, gamma=n_q, window=1, seed=11 + n_q)
    inp = W.make_layer(wl, 0, "cuda")
    g = torch.Generator(device="cuda").manual_seed(n_q)
    q = torch.randn(b, h_q, n_q, d, device="cuda", generator=g).to(torch.bfloat16)
    if grow:
        # keys along the query direction, longer and longer: every tile beats the running max
        ramp = grow * torch.arange(inp.k_cache.shape[2], device="cuda") / t_max
        u = q.float().view(b, h_kv, -1, d).mean(2)
        inp.k_cache += (ramp[None, None, :, None] * (u / u.norm(dim=-1, keepdim=True))[:, :, None]).to(torch.bfloat16)
    dl = torch.tensor(lens, dtype=torch.int32, device="cuda") if isinstance(t, tuple) else None
    shape = bd.make_shape(b, h_q, h_kv, d, t_max, wl.t_cap, dl)
    ws = bd.Workspace(bd.bd_workspace_size(shape, bd.BD_OP_VERIFY, 1, n_q))
    for rep in range(repeat):
        o = torch.full((b, h_q, n_q, d), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((b, h_q, n_q), float("nan"), device="cuda")
        bd.bd_verify_attn(shape, q, n_q, inp.k_cache, inp.v_cache, o, lse, ws)
        torch.cuda.synchronize()
        assert ws.status() == 0
    for i, n in enumerate(lens):
        k, v = f64(inp.k_cache[i:i + 1, :, :n + n_q]), f64(inp.v_cache[i:i + 1, :, :n + n_q])
        ro, rl = oracle.verify_attn(f64(q[i:i + 1]), k, v, n)
        check_attention(o[i:i + 1], lse[i:i + 1], ro, rl, f"verify tc G={h_q // h_kv} n_q={n_q} T={n}")


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("h_q,h_kv,t,n_q", [
    (1, 1, 1, 25), (8, 2, 100, 7), (8, 1, 120, 8), (4, 2, 1000, 32), (8, 2, 1403, 16), (13, 1, 640, 5),
    (4, 1, 1407, 32), (3, 1, 1300, 43), (16, 2, 2900, 21), (32, 2, 511, 16), (1, 1, 255, 257), (32, 1, 300, 24),
    (8, 8, 5000, 100)])
def test_many_rows(h_q, h_kv, d, t, n_q):
    block(2, h_q, h_kv, d, t, n_q)


@pytest.mark.parametrize("h_q,h_kv,t,n_q", [(32, 8, (1500, 37, 896), 21), (16, 2, (129, 1, 5, 2000), 20)])
def test_many_rows_of_ragged_sequences(h_q, h_kv, t, n_q):
    block(len(t), h_q, h_kv, 128, t, n_q)


@pytest.mark.parametrize("n_q", [9, 20])
def test_growing_scores(n_q):
    block(1, 8, 1, 128, 30000, n_q, grow=40.0)


def test_many_units_per_cta():
    block(24, 64, 16, 64, 150, 8)


@pytest.mark.parametrize("rows", [16, 17, 24])
def test_few_rows_of_a_large_batch(rows):
    block(16, 8, 4, 128, 1100, rows // 2 if rows % 2 == 0 else 9, repeat=1)
    block(60, rows, 1, 128, 1100, 1, repeat=1)
