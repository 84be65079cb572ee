"""The CUDA-core convolutions at the edges of their tiles and slices, in fp32 (1e-5 against the oracle) and as the 16-bit
fallback: ragged rows and columns, one and several slices, slices longer than 1024 products (flushed to fp64), three input
channels (no vector loads), every parity class of a stride-2 data gradient, a 1x1 stride-2 layer (pixels no tap reaches)."""
import pytest

from paper_2609_10632_b200 import workloads as wl
from tests import parity
from tests.test_gpu_parity import EPS, _compare, _oracle, _run_block

pytestmark = pytest.mark.gpu

SHAPES = [
    (1, 9, 7, 8, 12, 3, 1),        # less than one tile each way
    (2, 16, 16, 16, 32, 1, 1),     # one k step per tap, exact tiles
    (1, 31, 37, 68, 100, 3, 1),    # ragged rows and columns, several slices
    (1, 23, 26, 20, 36, 3, 2),     # stride 2, odd height
    (2, 13, 14, 24, 16, 1, 2),     # 1x1 stride 2
    (1, 24, 20, 3, 16, 3, 2),      # three channels
    (1, 160, 120, 128, 16, 3, 1),  # 300 tiles: one slice of 1152 products
]


@pytest.mark.parametrize("mode,dims", [(m, d) for m in ("f32", "bf16") for d in SHAPES if m == "f32" or d[4] % 8 == 0],
                         ids=lambda v: v if isinstance(v, str) else "x".join(map(str, v)))
def test_cuda_core_convolutions_match_oracle(mode, dims):
    from paper_2609_10632_b200 import binding as nb

    shape = wl.ConvShape("simt", *dims)
    f32 = mode == "f32"
    inp, blk, out = _run_block(shape, nb.NB_MODE_F32_REF if f32 else nb.NB_MODE_BF16_TC, cfg_id=42, layer_id=SHAPES.index(dims), affine="random",
                               flags=0 if f32 else nb.NB_CBS_FLAG_FORCE_SIMT)
    assert blk.plan.paths == {"fprop": 0, "dgrad": 0, "wgrad": 0}
    ref = _oracle(inp)
    if dims[5] == 1 and dims[6] == 2 and not f32:  # (the bar of a tensor of which three quarters are structural zeros)
        assert not out["dx"][:, 1::2].any() and not out["dx"][:, :, 1::2].any()
        out["dx"], ref.dx = out["dx"][:, ::2, ::2], ref.dx[:, ::2, ::2]
    _compare(out, ref, 1 if f32 else 0)


WIDE = [("f32", (1, 20, 20, 256, 1152, 3, 1)), ("f32", (1, 10, 11, 32, 1028, 3, 1)), ("bf16", (1, 12, 12, 40, 1280, 3, 1)), ("bf16", (1, 12, 12, 32, 2304, 3, 1))]


@pytest.mark.parametrize("mode,dims", WIDE, ids=lambda v: v if isinstance(v, str) else "x".join(map(str, v)))
def test_forward_slices_of_more_than_1024_channels(mode, dims):
    """Rows wider than 256 groups of four channels, up to the widest a plan may have: the pass that adds the slices of a split
    forward convolution has a thread for every group, in training (with the channel sums) and in evaluation mode."""
    import torch

    import oracle
    from paper_2609_10632_b200 import binding as nb

    shape = wl.ConvShape("wide", *dims)
    f32 = mode == "f32"
    inp, blk, out = _run_block(shape, nb.NB_MODE_F32_REF if f32 else nb.NB_MODE_BF16_TC, cfg_id=43, layer_id=WIDE.index((mode, dims)), affine="random",
                               flags=0 if f32 else nb.NB_CBS_FLAG_FORCE_SIMT)
    assert blk.plan.paths["fprop"] == 0
    _compare(out, _oracle(inp), 1 if f32 else 0)
    rm, rv, _ = wl.make_eval_stats(shape, 43, 0)
    up = lambda a: torch.from_numpy(a).to(blk.dev)
    a, ws = torch.empty_like(blk.a), torch.empty(blk.plan.infer_bytes, dtype=torch.uint8, device=blk.dev)
    nb.nb_conv_bn_silu_infer(blk.plan, blk.x, blk.w, blk.gamma, blk.beta, up(rm), up(rv), a, ws)
    parity.check("a_eval", a.double().cpu().numpy(), oracle.cbs_infer(inp.x, inp.w, inp.gamma, inp.beta, rm, rv, shape.stride, EPS), "f32" if f32 else "bf16")


def test_weight_gradient_of_more_pixels_than_the_grid_has_slices_for():
    """8 -> 8 1x1 in fp32 on 64 x 1024 x 1024 pixels: 65536 slices of 1024 pixels would be one more than a grid may have; the
    kernel takes longer slices (flushed to fp64).  The step against fp64 sums over the kernel's own dy."""
    import torch

    from paper_2609_10632_b200 import binding as nb
    from paper_2609_10632_b200.block import CbsBlock

    shape = wl.ConvShape("pixels", 64, 1024, 1024, 8, 8, 1, 1)
    blk = CbsBlock(shape, mode=nb.NB_MODE_F32_REF)
    blk.fill_random(5)
    blk.step()
    blk.poll()
    m = shape.m
    x, dy = blk.x.view(m, 8), blk.dy.view(m, 8)
    dw = sum(dy[i:i + m // 16].double().t() @ x[i:i + m // 16].double() for i in range(0, m, m // 16))
    # fp32 sums of up to 1024 products of random sign: 1024 roundings of 2^-24 of partial sums up to 32 products large are 6e-5
    # of a product's size together, in each of 65536 slices, 1.5e-2 in all; the sum is sqrt(m) = 8192 products large: 2e-6
    scale = float(dy[:m // 16].double().pow(2).mean().sqrt() * x[:m // 16].double().pow(2).mean().sqrt()) * m ** 0.5
    err = (blk.dw.view(8, 8).double() - dw).abs().max().item()
    assert err <= 1e-5 * scale, (err, scale)
