"""SpecStep.window_lse on a stream of its own, while the caller's current stream is busy: its
workspace and its lengths are filled in the order of the stream that the call runs on."""

import pytest
import torch

import paper_2606_00144_gb300 as bd
from paper_2606_00144_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    bd.build()
    bd.library()


@pytest.mark.parametrize("as_int", [False, True])
@pytest.mark.parametrize("ragged", [False, True])
def test_the_call_waits_for_nothing_of_the_current_stream(ragged, as_int):
    wl = W.tiny_workload(batch=2, h_q=8, h_kv=2, head_dim=128, t_ctx=6000, budget=256, gamma=3, seed=3)
    inp = W.make_layer(wl, 0, "cuda")
    lens = torch.tensor([6000, 4100], dtype=torch.int32, device="cuda") if ragged else None
    st = bd.SpecStep(2, 8, 2, 128, 6000, wl.t_cap, 256, 4, 64, wl.window, 3, seq_lens=lens)
    want = st.window_lse(inp.k_cache, inp.q_win)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):
        # memory that is handed out again holds ones in every bit
        sizes = (1 << 25, 1 << 22, 1 << 19, 4096, 512)
        dirty = [torch.full((n,), 255, dtype=torch.uint8, device="cuda") for n in sizes]
        with torch.cuda.stream(side):
            dirty += [torch.full((n,), 255, dtype=torch.uint8, device="cuda") for n in sizes]
        torch.cuda.synchronize()
        del dirty
        torch.cuda._sleep(100_000_000)                          # tens of milliseconds
        got = st.window_lse(inp.k_cache, inp.q_win, stream=side.cuda_stream if as_int else side)
        side.synchronize()
        assert not torch.cuda.current_stream().query()          # the current stream is busy still
        torch.cuda.synchronize()
        assert torch.equal(got, want)
