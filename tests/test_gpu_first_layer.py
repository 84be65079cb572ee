"""The first layer's own kernels (3 input channels, 3x3, stride 2) at the other channel counts they are built for."""
import pytest

from paper_2609_10632_b200 import workloads as wl
from tests import parity
from tests.test_gpu_parity import _compare, _oracle, _run_block

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c_out", [16, 32, 64, 80])
@pytest.mark.parametrize("n,h,w", [(2, 6, 46), (1, 34, 418), (1, 12, 656)])  # narrow strips, wide ones with a ragged end, more than one wide strip
@pytest.mark.parametrize("mode", ["bf16", "f16"])
def test_first_layer_matches_oracle(mode, n, h, w, c_out):
    import oracle
    import torch

    from paper_2609_10632_b200 import binding as nb

    shape = wl.ConvShape("first", n, h, w, 3, c_out, 3, 2, True)
    inp, blk, out = _run_block(shape, nb.NB_MODE_BF16_TC if mode == "bf16" else nb.NB_MODE_F16_TC, cfg_id=44, layer_id=c_out + w, affine="random")
    assert blk.plan.infer_fused
    _compare(out, _oracle(inp), 0)
    rm, rv, _ = wl.make_eval_stats(shape, 44, c_out + w)
    up = lambda a: torch.from_numpy(a).to(blk.dev)
    o = torch.empty_like(blk.a)
    ws = torch.empty(max(blk.plan.infer_bytes, 256), dtype=torch.uint8, device=blk.dev)
    nb.nb_conv_bn_silu_infer(blk.plan, blk.x, blk.w, blk.gamma, blk.beta, up(rm), up(rv), o, ws)
    torch.cuda.synchronize()
    parity.check("a_eval", o.double().cpu().numpy(), oracle.cbs_infer(inp.x, inp.w, inp.gamma, inp.beta, rm, rv, shape.stride, 1e-3), "bf16")
