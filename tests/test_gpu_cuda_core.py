"""The CUDA-core convolutions at the edges of their tiles and slices, in fp32 (1e-5 against the oracle) and as the 16-bit
fallback: ragged rows and columns, one and several slices, slices longer than 1024 products (flushed to fp64), three input
channels (no vector loads), every parity class of a stride-2 data gradient, a 1x1 stride-2 layer (pixels no tap reaches)."""
import pytest

from paper_2609_10632_b200 import workloads as wl
from tests.test_gpu_parity import _compare, _oracle, _run_block

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
