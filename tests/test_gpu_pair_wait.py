"""The two-axis launches' bounded wait (fft_pair.cuh): with one tile of the
first axis left out the second axis's wait gives up after its limit, the plan
reports MDFFT_E_TIMEOUT, the counters are zero again, and the next executions
on the same plan give the bits of the pass kernels."""

import pytest
import torch

import paper_1302_6189_gb300 as md

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def _input(shape, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return torch.view_as_complex(torch.rand(*shape, 2, generator=g, device=DEV) * 2 - 1)


@pytest.mark.parametrize("shape,limit_us", [((64, 64, 5, 640), 200_000),  # blocks of inner points
                                            ((256, 256, 240), 100_000),   # the same with 256-point columns
                                            ((192, 256, 256), 1_000)])    # whole planes
def test_a_wait_that_gives_up_leaves_the_plan_usable(shape, limit_us):
    x = _input(shape, 51)
    y = torch.empty_like(x)
    with md.Plan(shape, 16) as pl:
        want = pl.exec_counted(x)[0]
        assert pl.launches() < len(shape)
        for _ in range(3):
            st, us = md.mdfft_selftest_pair_wait(pl.handle, x.data_ptr(), y.data_ptr(), limit_us)
            assert st == md.mdfft.MDFFT_E_TIMEOUT and limit_us <= us < limit_us + 2_000_000
            pl.check()  # the flag is reported once
            for _ in range(2):
                assert torch.equal(pl.exec(x, y), want)
            pl.check()


def test_arguments():
    x = _input((24, 40, 32), 52)
    y = torch.empty_like(x)
    with md.Plan((24, 40, 32), 8) as pl:
        assert md.mdfft_selftest_pair_wait(pl.handle, x.data_ptr(), y.data_ptr(), 1000)[0] == md.mdfft.MDFFT_E_UNSUPPORTED
        for limit in (0, 10**7 + 1):
            assert md.mdfft_selftest_pair_wait(pl.handle, x.data_ptr(), y.data_ptr(), limit)[0] == md.mdfft.MDFFT_E_ARG
        assert md.mdfft_selftest_pair_wait(pl.handle, x.data_ptr(), 0, 1000)[0] == md.mdfft.MDFFT_E_ARG
