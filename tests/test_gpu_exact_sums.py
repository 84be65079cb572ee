"""fp32 mode: channel sums without rounding between the blocks, the same bits from run to run."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2609_10632_b200 import workloads as wl

pytestmark = pytest.mark.gpu

VALUES = [  # what the nonzero rows of a channel hold: sums of which fp64 additions lose a part, which one depending on their order
    [1e30, 1.0, -1e30, 3e-20, 2.0**-149, -(2.0**-140)],
    [3.4e38, -3.4e38, 3.4e38, 1e-38, -3.4e38, 7.0],
    [2.0**-149, 2.0**-149, 2.0**-126, -(2.0**-149), 2.0**-127, 2.0**-130],
    [1.0, 2.0**60, 2.0**-60, -(2.0**60), 2.0**30, -(2.0**30)],
    [-1.5, 2.5, -3.5, 0.0, -0.0, 5.25],
    [2.0**104, -1.0, -(2.0**104), 2.0**-3, 0.0, 2.0**-25],
    [1e-10, 1e10, -1e10, 1e20, -1e20, 1e-30],
    [6.5, 2.0**127, 2.0**-100, 2.0**-149, -6.5, -(2.0**127)],
]


def _f32(v):
    return float(np.float32(v))


@pytest.mark.parametrize("h,w,c", [(24, 32, 8), (128, 160, 8), (24, 32, 264), (128, 160, 168)], ids=["", "two sets", "wide", "wide, two sets"])
def test_totals_are_the_sums_without_rounding(h, w, c):
    """A 1x1 convolution with the identity filter, whose output has one nonzero row in each of six tiles: every tile's sum is that
    row's value, and the mean is the exact sum of the six over M, rounded once to fp32.  Few and many adding blocks, and few and
    many channels (whose coefficients a kernel of its own derives); wide rows are also cut into k slices."""
    import torch

    from paper_2609_10632_b200 import binding as nb
    from paper_2609_10632_b200.block import CbsBlock

    shape = wl.ConvShape("exact", 1, h, w, c, c, 1, 1)
    blk = CbsBlock(shape, mode=nb.NB_MODE_F32_REF)
    blk.x.zero_()
    rows = blk.x.view(shape.m, c)
    for k, values in enumerate(VALUES):
        for t, v in enumerate(values):
            rows[t * 128 + 17, k::8] = v
    blk.w.copy_(torch.eye(c).view(c, 1, 1, c))
    blk.gamma.fill_(1.0)
    blk.beta.zero_()
    mean = None
    for _ in range(10):
        blk.forward()
        blk.poll()
        assert mean is None or np.array_equal(mean, blk.mean.cpu().numpy(), equal_nan=True)
        mean = blk.mean.cpu().numpy()
    for k in range(c):
        values = VALUES[k % 8]
        got, want = Fraction(float(mean[k])), sum((Fraction(_f32(v)) for v in values), Fraction(0)) / shape.m
        # one rounding to fp32, behind an fma per word and a product in fp64: a bit more than half a unit in the last place
        assert abs(got - want) <= abs(want) * Fraction(2) ** -23 + Fraction(2) ** -149, (k, float(got), float(want))


def test_infinities_and_nan_reach_the_statistics():
    import torch

    from paper_2609_10632_b200 import binding as nb
    from paper_2609_10632_b200.block import CbsBlock

    shape = wl.ConvShape("inf", 1, 24, 32, 8, 8, 1, 1)
    blk = CbsBlock(shape, mode=nb.NB_MODE_F32_REF)
    blk.w.copy_(torch.ones(8, 1, 1, 8))
    blk.gamma.fill_(1.0)
    blk.beta.zero_()
    for values, want in (([float("inf")], float("inf")), ([float("-inf")], float("-inf")), ([float("inf"), float("-inf")], float("nan")),
                         ([float("nan")], float("nan")), ([1.0], 8.0 / 768)):
        blk.x.zero_()
        for t, v in enumerate(values):
            blk.x.view(shape.m, 8)[t * 128] = v
        blk.forward()
        torch.cuda.synchronize()
        np.testing.assert_allclose(blk.mean.cpu().numpy(), want, rtol=1e-7)


@pytest.mark.parametrize("dims", [(2, 32, 32, 16, 32, 3, 1), (2, 40, 40, 64, 64, 3, 1), (3, 37, 29, 20, 1028, 1, 1), (4, 60, 60, 32, 48, 3, 2),
                                  (2, 40, 40, 64, 164, 3, 1), (4, 90, 80, 16, 192, 1, 1)], ids=str)
def test_default_steps_are_the_same_bits_from_run_to_run(dims):
    """Values whose block sums span 2^100, so that fp64 sums would depend on the order of the atomics."""
    import torch

    from paper_2609_10632_b200 import binding as nb
    from paper_2609_10632_b200.block import CbsBlock

    blk = CbsBlock(wl.ConvShape("bits", *dims), mode=nb.NB_MODE_F32_REF, running_stats=True)
    blk.fill_random(11)
    gen = torch.Generator(device="cuda").manual_seed(1)
    for t in (blk.x, blk.g):
        flat = t.view(-1, t.shape[-1])
        size = torch.randint(-50, 51, (flat.shape[0] // 32 + 1,), generator=gen, device="cuda").float().exp2()
        flat.mul_(size.repeat_interleave(32)[:flat.shape[0], None])
        half = flat.shape[0] // 2
        flat[half:2 * half] = -flat[:half]  # (large parts of the sums cancel)
    names = ("y", "a", "mean", "invstd", "running_mean", "running_var", "dgamma", "dbeta", "dy", "dx", "dw")
    first = None
    for _ in range(30):
        blk.running_mean.zero_()
        blk.running_var.fill_(1.0)
        blk.step()
        blk.poll()
        got = [getattr(blk, k).clone() for k in names]
        if first is not None:
            for k, a, b in zip(names, got, first):
                assert torch.equal(a.view(torch.int32), b.view(torch.int32)), k
        first = first or got
