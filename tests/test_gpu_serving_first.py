"""A new server's first steps do no work that belongs to its creation: draining
a few requests takes a fresh server no longer than one that has run before."""

import time

import pytest
import torch

import paper_1302_6189_gb300 as md

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def test_the_first_drain_of_a_server_takes_no_longer_than_later_ones():
    xs = [torch.randn((64, 48, 96), dtype=torch.complex64, device=DEV) for _ in range(6)]
    ys = [torch.empty_like(x) for x in xs]
    first, later = [], []
    for rep in range(5):
        with md.Server(budget_bytes=1 << 30, max_inflight=16) as srv:
            srv.set_direct(0)  # batched steps: three per drain, eight tables in turn
            for k in range(8):
                ids = [srv.submit(x, y) for x, y in zip(xs, ys)]
                torch.cuda.synchronize()
                t = time.perf_counter()
                srv.drain()
                t = time.perf_counter() - t
                for i in ids:
                    srv.release(i)
                if rep > 0:  # (the first server of a process also loads the kernels)
                    (first if k < 3 else later).append(t)
    # the same steps on the same tables: a factor of 2 for noise (with the
    # graphs made in the steps the first three drains took 3 to 4 times as long)
    assert min(first) <= 2 * min(later), (first, later)
