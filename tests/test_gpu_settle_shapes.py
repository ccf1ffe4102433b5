"""bd_argmax and bd_accept at the sizes where their splits change: rows of one vector, one vector
more and less than a CTA reads per round (one, two and four vectors a thread), unaligned rows,
maxima in the first and the last element and in the ragged ends, ties; drafts of 0, 31, 32, 33
and 64 tokens with the first disagreement everywhere around the 32-lane boundary."""

import pytest
import torch

import paper_2606_00144_gb300 as bd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    bd.build()
    bd.library()


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("rows,vocab", [(1, 1), (3, 7), (2, 4095), (2, 4097), (700, 8192), (700, 8200), (700, 4113), (5, 32771),
                                        (1300, 2049), (48, 32003), (9, 16385)])
def test_argmax_sizes(dtype, rows, vocab):
    g = torch.Generator(device="cuda").manual_seed(rows + vocab)
    x = torch.randn(rows, vocab, generator=g, device="cuda").to(dtype)
    ar = torch.arange(rows, device="cuda")
    x[ar, ar * 977 % vocab] = 50.0                        # a maximum anywhere in the row
    x[0, 0], x[rows - 1, vocab - 1] = 60.0, 60.0
    if rows > 2:                                          # equal maxima: the lowest id
        x[1, vocab // 2:] = 70.0
        x[2] = float("nan")
    ids = torch.full((rows,), -7, dtype=torch.int32, device="cuda")
    bd.bd_argmax(x, ids)
    want = torch.where(x.isnan().all(1), 0, x.float().nan_to_num(nan=float("-inf")).argmax(1))
    top = x.float().nan_to_num(nan=float("-inf")).max(1, keepdim=True).values
    first = torch.where(x.float() == top, torch.arange(vocab, device="cuda"), vocab).min(1).values
    want = torch.where(x.isnan().all(1), want, first)
    assert torch.equal(ids.long(), want.long())


@pytest.mark.parametrize("gamma", [0, 1, 31, 32, 33, 64])
def test_accept_prefixes(gamma):
    n = gamma + 1                                         # sequence i disagrees first at position i
    d = torch.randint(0, 1000, (max(gamma, 1), n), device="cuda", dtype=torch.int32)[:gamma]
    v = torch.randint(0, 1000, (n, gamma + 1), device="cuda", dtype=torch.int32)
    for i in range(n):
        v[i, :i] = d[:i, i]
        if i < gamma:
            v[i, i] = d[i, i] + 1
    n_acc = torch.empty(n, dtype=torch.int32, device="cuda")
    emit = torch.empty(n, gamma + 1, dtype=torch.int32, device="cuda")
    bd.bd_accept(d, v, n_acc, emit)
    assert n_acc.tolist() == list(range(n))
    for i in range(n):
        assert emit[i].tolist() == v[i, :i + 1].tolist() + [-1] * (gamma - i)
