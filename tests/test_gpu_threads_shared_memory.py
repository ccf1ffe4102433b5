"""Calls from two threads whose launches of one kernel need different amounts of shared memory: neither
takes the other's permission away between asking for it and launching."""

import threading

import pytest
import torch

import paper_2606_00144_gb300 as bd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    bd.build()
    bd.library()


def test_windows_of_two_sizes():
    shape = bd.make_shape(1, 1, 1, 128, 1000, 1010)
    errors = []
    start = threading.Barrier(6)

    def loop(window):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                n_acc = torch.zeros(1, dtype=torch.int32, device="cuda")
                q_win = torch.ones(1, 1, window, 128, dtype=torch.bfloat16, device="cuda")
                q_new = torch.ones(1, 1, 2, 128, dtype=torch.bfloat16, device="cuda")
                start.wait()
                for _ in range(12000):
                    bd.bd_advance(shape, window, 2, n_acc, q_new, None, q_win, None)
            stream.synchronize()
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=loop, args=(w,)) for w in (16, 700) * 3]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
