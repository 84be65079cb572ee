"""Channel counts that are multiples of 8 but not of 16, counts without a wide divisor, and odd extents at stride 2: the
tensor-core kernels' padded last tile (zero-filled filter rows, clipped stores) at the places where it can go wrong."""
import pytest

from paper_2609_10632_b200 import workloads as wl
from tests import parity
from tests.test_gpu_parity import EPS, _compare, _oracle, _run_block

pytestmark = pytest.mark.gpu

SHAPES = [
    (2, 16, 8, 24, 24, 3, 1),     # 256 rows: the fewest that leave the CUDA cores; one padded tile of 32 columns
    (1, 19, 17, 40, 56, 3, 1),    # ragged rows; 56 = 48 + a half piece
    (2, 23, 21, 72, 136, 3, 1),   # 136 columns in one tile of 144: the second team's last piece is half padding
    (1, 18, 20, 136, 72, 1, 1),   # 1x1: tiled A map with a tail k-block of 8 channels
    (1, 17, 19, 104, 264, 1, 1),  # two tiles of 144 for 264 columns: the last 24 columns are padding, one piece whole
    (1, 16, 17, 64, 304, 1, 1),   # 304 = 16 x 19: no wide divisor, two tiles of 160
    (2, 33, 31, 32, 48, 3, 2),    # stride 2, odd height and width: the odd parity classes are one row / column short
    (1, 34, 47, 88, 104, 3, 2),   # stride 2, odd width, padded both ways
    (1, 48, 32, 40, 24, 3, 1),    # width a multiple of 16: the row-tile weight gradient with padded columns
]


@pytest.mark.parametrize("dims", SHAPES, ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("mode", ["bf16", "f16"])
def test_padded_tiles_match_oracle(dims, mode):
    import oracle
    import torch

    from paper_2609_10632_b200 import binding as nb

    shape = wl.ConvShape("padded", *dims)
    inp, blk, out = _run_block(shape, nb.NB_MODE_BF16_TC if mode == "bf16" else nb.NB_MODE_F16_TC, cfg_id=41, layer_id=SHAPES.index(dims), affine="random")
    assert blk.plan.paths == {"fprop": 1, "dgrad": 1, "wgrad": 1} and blk.plan.infer_fused
    _compare(out, _oracle(inp), 0)
    rm, rv, _ = wl.make_eval_stats(shape, 41, SHAPES.index(dims))
    up = lambda a: torch.from_numpy(a).to(blk.dev)
    o = torch.empty_like(blk.a)
    ws = torch.empty(max(blk.plan.infer_bytes, 256), dtype=torch.uint8, device=blk.dev)
    nb.nb_conv_bn_silu_infer(blk.plan, blk.x, blk.w, blk.gamma, blk.beta, up(rm), up(rv), o, ws)
    torch.cuda.synchronize()
    assert blk.poll() == ""  # nothing gave up, nothing counted as saturated
    parity.check("a_eval", o.double().cpu().numpy(), oracle.cbs_infer(inp.x, inp.w, inp.gamma, inp.beta, rm, rv, shape.stride, EPS), "bf16")
