"""mdfft_exec_graph on plans that replay captured graphs: spectra left in the
last layout, the tensor-core dtype, and plans whose tuning names the pass
kernels.  (Plans as made launch their axis kernels directly and capture
nothing.)  More (in, out) pairs and directions than the cache of 8 holds, and
a retune, which drops the captured graphs."""

import pytest
import torch

import paper_1302_6189_gb300 as md

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def _input(shape, seed, dtype):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    real = torch.float64 if dtype == "c128" else torch.float32
    return torch.view_as_complex(torch.rand(*shape, 2, generator=g, device=DEV, dtype=real) * 2 - 1)


@pytest.mark.parametrize("dtype,flags,passes", [("c64", md.MDFFT_PLAN_OUT_LAST_LAYOUT, False), ("c64_tc_fp16", 0, False),
                                                ("c64", 0, True), ("c128", 0, True)])
def test_replay_replacement_and_retuning(dtype, flags, passes):
    shape = (16, 24, 20)
    xs = [_input(shape, 80 + i, dtype) for i in range(6)]
    with md.Plan(shape, 8, None, dtype, flags) as pl:
        if passes:
            pl.set_tuning([dict(t, variant="passes") for t in pl.tuning()])
        assert pl.launches() == len(shape)
        ways = [dict(), dict(dir=+1, normalize=True)]
        want = [[pl.exec(x, **kw) for kw in ways] for x in xs]
        outs = [[torch.empty_like(w) for w in ws] for ws in want]

        def replay_all():
            for x, os, ws in zip(xs, outs, want):
                for o, w, kw in zip(os, ws, ways):
                    o.zero_()
                    pl.exec(x, o, graph=True, **kw)
                    assert torch.equal(o, w)

        for _ in range(2):  # 12 graphs through a cache of 8
            replay_all()
        for _ in range(3):  # the same one again: captured once, then replayed
            outs[0][0].zero_()
            pl.exec(xs[0], outs[0][0], graph=True)
            assert torch.equal(outs[0][0], want[0][0])
        tuning = pl.tuning()
        pl.autotune(xs[0], torch.empty_like(want[0][0]), reps=2)
        replay_all()
        pl.set_tuning(tuning)
        replay_all()
        # a replay changes with the input's values, not only with its address
        x, o = xs[1].clone(), outs[1][0]
        pl.exec(x, o, graph=True)
        x.mul_(0)
        pl.exec(x, o, graph=True)
        assert not bool(o.abs().max() > 0)
