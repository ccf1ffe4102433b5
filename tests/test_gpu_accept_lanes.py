"""bd_accept at the drafts where a sequence's lanes double (1, 2, 4, ... 32 of a warp), and batches that
leave the last warp and the last block partly empty."""

import pytest
import torch

import paper_2606_00144_gb300 as bd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    bd.build()
    bd.library()


@pytest.mark.parametrize("gamma", [0, 1, 2, 3, 4, 7, 8, 15, 16, 31, 32, 40])
@pytest.mark.parametrize("batch", [1, 3, 31, 130, 4097])
def test_lanes_per_sequence(batch, gamma):
    g = torch.Generator(device="cuda").manual_seed(batch + gamma)
    d = torch.randint(0, 3, (gamma, batch), generator=g, device="cuda", dtype=torch.int32)
    v = torch.randint(0, 3, (batch, gamma + 1), generator=g, device="cuda", dtype=torch.int32)
    full = torch.arange(batch, device="cuda") % 3 == 0                   # a third agree throughout
    v[full, :gamma] = d.T[full]
    n_acc = torch.full((batch + 64,), -7, dtype=torch.int32, device="cuda")
    emit = torch.full((batch + 64, gamma + 1), -7, dtype=torch.int32, device="cuda")
    bd.bd_accept(d, v, n_acc[:batch], emit[:batch])
    want = (d.T == v[:, :gamma]).int().cumprod(1).sum(1)
    keep = torch.arange(gamma + 1, device="cuda")[None] <= want[:, None]
    assert torch.equal(n_acc[:batch].long(), want.long())
    assert torch.equal(emit[:batch], torch.where(keep, v, -1))
    assert bool((n_acc[batch:] == -7).all()) and bool((emit[batch:] == -7).all())
