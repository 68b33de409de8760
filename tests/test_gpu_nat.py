"""The layout-keeping line kernels (one axis of the natural array at a time,
in place after the first) against the pass kernels, which the counted
execution runs: the same butterflies in the same order, so the same bits, for
every line length as rows and as columns, at ragged edges of their tiles."""

import pytest
import torch

import paper_1302_6189_gb300 as md

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
LENGTHS = [n for n in range(2, 1025) if md.mdfft_supported_length(n, "c64")]


def _input(shape, seed, dtype="c64"):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    real = torch.float64 if dtype == "c128" else torch.float32
    return torch.view_as_complex(torch.rand(*shape, 2, generator=g, device=DEV, dtype=real) * 2 - 1)


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n", LENGTHS)
def test_every_length_as_rows_and_columns_equals_the_pass_kernels(n, dtype):
    # rows: 3 and 160 lines; columns: 3 and 160 neighbouring lines, one and two blocks of them
    for shape in ((3, n), (n, 3), (160, n), (2, n, 160)):
        x = _input(shape, n, dtype)
        keep = x.clone()
        with md.Plan(shape, 3, None, dtype) as pl:
            y = pl.exec(x)
            assert torch.equal(y, pl.exec_counted(x)[0]), shape
            z = pl.exec(x, dir=+1, normalize=True)
            assert torch.equal(z, pl.exec_counted(x, dir=+1, normalize=True)[0]), shape
            assert torch.equal(x, keep)


@pytest.mark.parametrize("shape,batch", [((1, 24, 1, 40), 1), ((16, 1, 60), 3), ((5, 6, 8, 10), 2), ((20, 12, 15, 3, 8), 1),
                                         ((48, 96, 160), 1), ((30, 240, 64), 2)])
def test_axes_of_length_one_batches_and_every_order_of_axes(shape, batch):
    full = shape if batch == 1 else (batch,) + shape
    x = _input(full, 11)
    M = len(shape)
    for first in range(M - 1):  # orders that transform the axes in different sequences
        rest = [a for a in range(M) if a != M - 1]
        rest = rest[first:] + rest[:first]
        layouts = [list(range(M))] + [[a for a in range(M) if a != f] + [f] for f in rest]
        order = "->".join("".join("abcde"[a] for a in lay) for lay in layouts)
        with md.Plan(shape, 4, order, batch=batch) as pl:
            want = pl.exec_counted(x)[0]
            assert torch.equal(pl.exec(x), want), order
            assert torch.equal(pl.exec(x, graph=True), want), order
        with md.Plan(shape, 4, order, flags=md.MDFFT_PLAN_INPLACE, batch=batch) as pl:
            buf = x.clone()
            assert torch.equal(pl.exec(buf, buf), want), order


def test_eight_byte_aligned_arrays_and_per_pass_times():
    shape = (24, 40, 32)
    data = _input(shape, 5)
    raw_in = torch.empty(data.numel() + 1, dtype=torch.complex64, device=DEV)
    raw_out = torch.empty_like(raw_in)
    x, y = raw_in[1:].view(shape), raw_out[1:].view(shape)
    x.copy_(data)
    with md.Plan(shape, 8) as pl:
        assert torch.equal(pl.exec(x, y), pl.exec_counted(data)[0])
        pl.set_timing(True)
        for _ in range(3):
            pl.exec(x, y)
        ms, n = pl.pass_times()
        assert n == 3 and all(t > 0 for t in ms)


# arrays of 96 MB and more: neighbouring axes of 64, 128 or 256 points run two to a launch
@pytest.mark.parametrize("shape,order,batch", [((15, 15, 15, 64, 64), None, 1),           # whole planes, a ragged last slab
                                               ((64, 64, 5, 640), None, 1),               # blocks of inner points
                                               ((64, 64, 60, 60), "abcd->abdc->acdb->bcda", 1),
                                               ((64, 64, 60, 60), "abcd->abdc->bcda->acdb", 1),  # the outer axis first
                                               ((64, 64, 64, 64), None, 1),               # two launches for four axes
                                               ((8, 128, 128, 128), None, 1), ((128, 128, 32, 24), "abcd->abdc->bcda->acdb", 1),
                                               ((192, 256, 256), None, 2), ((256, 256, 240), None, 1)])
def test_two_axes_in_one_launch_equal_the_pass_kernels(shape, order, batch):
    full = shape if batch == 1 else (batch,) + shape
    x = _input(full, 21)
    with md.Plan(shape, 16, order, batch=batch) as pl:
        assert pl.launches() < len(shape)
        want, want_inv = pl.exec_counted(x)[0], pl.exec_counted(x, dir=+1, normalize=True)[0]
        for _ in range(3):  # the counters of one launch are zero again for the next
            assert torch.equal(pl.exec(x), want)
        assert torch.equal(pl.exec(x, dir=+1, normalize=True), want_inv)
        pl.check()
    with md.Plan(shape, 16, order, flags=md.MDFFT_PLAN_INPLACE, batch=batch) as pl:
        buf = x.clone()
        assert torch.equal(pl.exec(buf, buf), want)


@pytest.mark.parametrize("shape", [(24, 40, 32), (64, 64, 64, 64)])  # axis launches; two-axis launches
def test_captured_by_the_callers_graph(shape):
    x, y = _input(shape, 31), None
    with md.Plan(shape, 16) as pl:
        want = pl.exec(x).clone()
        y = torch.empty_like(x)
        pl.exec(x, y)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            pl.exec(x, y)
        for _ in range(3):
            y.zero_()
            graph.replay()
            assert torch.equal(y, want)


@pytest.mark.parametrize("shape,batch", [((24, 24, 24, 24), 41), ((40, 240, 160), 9), ((12, 15, 16), 4400)])
def test_groups_of_a_batch_equal_the_pass_kernels(shape, batch):
    # batches of 96 MB and more run in groups of transforms that L2 holds, the last group smaller
    x = _input((batch,) + shape, 41)
    with md.Plan(shape, 16, batch=batch) as pl:
        assert pl.launches() > len(shape)
        assert torch.equal(pl.exec(x), pl.exec_counted(x)[0])
        assert torch.equal(pl.exec(x, dir=+1, normalize=True), pl.exec_counted(x, dir=+1, normalize=True)[0])
        pl.set_timing(True)
        pl.exec(x)
        assert len(pl.pass_times()[0]) == len(shape)
