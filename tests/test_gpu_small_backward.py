"""Small tensors: both backward passes in one launch (bn_silu_bwd_small_kernel) against the two launches it stands for."""
import pytest

from paper_2609_10632_b200 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [  # n, h, w, c_in, c_out, k, stride
    (1, 5, 3, 16, 16, 1, 1),       # fewer rows than one block has
    (1, 16, 16, 16, 32, 3, 1),
    (2, 20, 20, 288, 288, 3, 1),   # filter tiles to rearrange beside the rows
    (2, 10, 10, 64, 576, 1, 1),    # 72 vectors per row
    (3, 37, 29, 48, 48, 3, 1),     # a last row block that is nearly empty
    (1, 41, 23, 72, 136, 3, 1),    # 17 vectors per row
    (2, 40, 40, 32, 64, 3, 2),
    (2, 40, 40, 96, 96, 3, 1),
    (1, 8, 8, 16, 1024, 1, 1),     # a row as wide as a block
]


@pytest.mark.parametrize("mode", ["bf16", "f16"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_same_results_as_two_launches(shape, mode, monkeypatch):
    import torch

    from paper_2609_10632_b200 import binding as nb
    from paper_2609_10632_b200.block import CbsBlock

    modes = {"bf16": nb.NB_MODE_BF16_TC, "f16": nb.NB_MODE_F16_TC}
    got = []
    for slabs in ("1", "0"):
        monkeypatch.setenv("NB_EW_SLABS", slabs)
        blk = CbsBlock(wl.ConvShape("small", *shape), mode=modes[mode])
        blk.fill_random(7)
        wide = torch.randn(*blk.g.shape[:-1], blk.g.shape[-1] + 8, device="cuda", generator=torch.Generator("cuda").manual_seed(1)).to(blk.g.dtype)
        out = []
        for pitched in (False, True):  # the gradient dense and as a channel slice
            if pitched:
                blk.plan.set_pitches(ld_g=wide.stride(-2))
                blk.g = wide[..., 8:]
            blk.step()
            blk.poll()
            out += [t.clone() for t in (blk.dy, blk.dgamma, blk.dbeta, blk.dx)]
        got.append(out)
    for a, b in zip(*got):  # (the block sums reach the fp64 accumulators in any order)
        a, b = a.double(), b.double()
        assert (a - b).norm() <= 1e-3 * b.norm()
