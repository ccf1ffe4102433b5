"""Verify blocks of per-sequence lengths over caches whose rows past each sequence's own block hold
NaN and infinities (memory that was never written): they must not reach the output.  Both verify
kernels, one and two M tiles, block ends inside, at and just past a tile's end, against the
oracle."""

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


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("h_q,h_kv,n_q", [(1, 1, 5), (8, 2, 6), (8, 2, 21), (8, 1, 32), (3, 1, 100)])
def test_rows_past_the_block_do_not_reach_the_output(h_q, h_kv, n_q, d):
    lens = (2000, 1, 128 - n_q, 129, 1700, 1024 - n_q, 1025, 640)
    b, t_max = len(lens), 2050                       # no sequence reaches the longest length
    wl = W.tiny_workload(batch=b, h_q=h_q, h_kv=h_kv, head_dim=d, t_ctx=t_max, gamma=n_q, window=1, seed=n_q)
    inp = W.make_layer(wl, 0, "cuda")
    g = torch.Generator(device="cuda").manual_seed(d + n_q)
    q = torch.randn(b, h_q, n_q, d, device="cuda", generator=g).to(torch.bfloat16)
    for i, n in enumerate(lens):
        for cache in (inp.k_cache, inp.v_cache):
            cache[i, :, n + n_q::2] = float("nan")
            cache[i, :, n + n_q + 1::2] = float("inf")
    dl = torch.tensor(lens, dtype=torch.int32, device="cuda")
    shape = bd.make_shape(b, h_q, h_kv, d, t_max, wl.t_cap, dl)
    ws = bd.Workspace(bd.bd_workspace_size(shape, bd.BD_OP_VERIFY, 1, n_q))
    o = torch.full((b, h_q, n_q, d), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((b, h_q, n_q), float("nan"), device="cuda")
    bd.bd_verify_attn(shape, q, n_q, inp.k_cache, inp.v_cache, o, lse, ws)
    torch.cuda.synchronize()
    assert ws.status() == 0
    for i, n in enumerate(lens):
        k, v = f64(inp.k_cache[i:i + 1, :, :n + n_q]), f64(inp.v_cache[i:i + 1, :, :n + n_q])
        ro, rl = oracle.verify_attn(f64(q[i:i + 1]), k, v, n)
        check_attention(o[i:i + 1], lse[i:i + 1], ro, rl, f"verify past end G={h_q // h_kv} n_q={n_q} T={n}")
