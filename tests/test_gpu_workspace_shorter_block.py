"""A workspace sized for the longest block of a shape serves every shorter one: its size does not
shrink as the block grows, and blocks on either side of a change of plan (24, 256 and 512 query
rows, a tile's end) run from one workspace, with and without an output."""

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


@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("b,h_q,h_kv,t", [(1, 64, 8, 4096), (4, 64, 8, 16384), (1, 8, 1, 128 * 152 - 2), (8, 32, 8, 1100),
                                          (1, 8, 8, 5000), (1, 2, 1, 128 * 151 + 127), (16, 4, 4, 300)])
def test_size_does_not_shrink_with_the_block(b, h_q, h_kv, t, ragged):
    lens = torch.full((b,), t, dtype=torch.int32, device="cuda") if ragged else None
    shape = bd.make_shape(b, h_q, h_kv, 128, t, t + 800, lens)
    sizes = [bd.bd_workspace_size(shape, bd.BD_OP_VERIFY, 1, n) for n in range(1, 768 // (h_q // h_kv) + 1)]
    assert all(x > 0 for x in sizes) and sizes == sorted(sizes)


@pytest.mark.parametrize("group,blocks", [(8, (33, 32, 3)), (8, (65, 64)), (4, (7, 6, 5, 4)), (1, (128, 2, 1))])
def test_shorter_blocks_run_from_the_longest_ones_workspace(group, blocks):
    b, h_kv, d, t = 1, 8, 128, 4096 - 1
    wl = W.tiny_workload(batch=b, h_q=group * h_kv, h_kv=h_kv, head_dim=d, t_ctx=t, gamma=blocks[0], window=1, seed=group)
    inp = W.make_layer(wl, 0, "cuda")
    # (a peaked softmax returns a row of V: halved, 4M normal draws stay below 4, where bf16 rounds by at
    # most 2^-7, inside the bar of 1e-2; at 5 it rounds by 2^-6, outside it)
    inp.v_cache.mul_(0.5)
    shape = bd.make_shape(b, wl.h_q, h_kv, d, t, wl.t_cap)
    ws = bd.Workspace(bd.bd_workspace_size(shape, bd.BD_OP_VERIFY, 1, blocks[0]))
    g = torch.Generator(device="cuda").manual_seed(group)
    for n_q in blocks:
        q = torch.randn(b, wl.h_q, n_q, d, device="cuda", generator=g).to(torch.bfloat16)
        o = torch.full((b, wl.h_q, n_q, d), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((b, wl.h_q, n_q), float("nan"), device="cuda")
        bd.bd_verify_attn(shape, q, n_q, inp.k_cache, inp.v_cache, o, lse, ws)
        k, v = f64(inp.k_cache[:, :, :t + n_q]), f64(inp.v_cache[:, :, :t + n_q])
        ro, rl = oracle.verify_attn(f64(q), k, v, t)
        check_attention(o, lse, ro, rl, f"shorter block G={group} n_q={n_q}")
        if group * n_q <= 128:
            lse.fill_(float("nan"))
            bd.bd_verify_attn(shape, q, n_q, inp.k_cache, None, None, lse, ws)
            assert float((lse.double().cpu() - torch.from_numpy(rl)).abs().max()) <= 1e-3
    assert ws.status() == 0
