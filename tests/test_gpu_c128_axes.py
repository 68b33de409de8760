"""complex128 axis launches: signs and scale of every direction bit for bit as
the pass kernels give them (signs of zeros too), and no slower than the passes
where the FP64 units bound both."""

import pytest
import torch

import paper_1302_6189_gb300 as md

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def _bits(x):
    return torch.view_as_real(x).view(torch.int64)


@pytest.mark.parametrize("shape", [(5, 12), (16, 48), (48, 20), (8, 60, 30), (2, 480), (1024, 3), (24, 1, 40)])
@pytest.mark.parametrize("zeros", [False, True])
def test_directions_and_scale_equal_the_pass_kernels(shape, zeros):
    g = torch.Generator(device=DEV)
    g.manual_seed(71)
    re = torch.rand(*shape, 2, generator=g, device=DEV, dtype=torch.float64) * 2 - 1
    if zeros:
        re = torch.copysign(torch.zeros_like(re), re)
    x = torch.view_as_complex(re)
    with md.Plan(shape, 2, None, "c128") as pl:
        for kw in (dict(), dict(dir=+1), dict(dir=+1, normalize=True)):
            assert torch.equal(_bits(pl.exec(x, **kw)), _bits(pl.exec_counted(x, **kw)[0])), kw


def _us(plan, x, y):
    best = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(10):
            plan.exec(x, y)
        b.record()
        torch.cuda.synchronize()
        best.append(a.elapsed_time(b) * 100)
    return min(best)


@pytest.mark.parametrize("shape,batch", [((48, 48, 48, 48), 1), ((48, 48, 48), 16), ((24, 48, 48), 4), ((80, 96, 48), 1)])
def test_48_point_axes_take_no_longer_than_the_passes(shape, batch):
    full = shape if batch == 1 else (batch,) + shape
    x = torch.randn(full, dtype=torch.complex128, device=DEV)
    y = torch.empty_like(x)
    with md.Plan(shape, 16, None, "c128", batch=batch) as pl:
        axes = _us(pl, x, y)
        pl.set_tuning([dict(t, variant="passes") for t in pl.tuning()])
        passes = _us(pl, x, y)
    assert axes <= 1.02 * passes, (axes, passes)
