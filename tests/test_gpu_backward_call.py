"""nb_conv_bn_silu_bwd against the two calls it stands for, and the two calls with work of the caller's between them."""
import pytest

from paper_2609_10632_b200 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [  # mode, (n, h, w, c_in, c_out, k, stride)
    ("bf16", (2, 40, 40, 96, 96, 3, 1)),     # row-tile weight gradient
    ("bf16", (3, 37, 29, 72, 136, 3, 1)),    # padded channel counts
    ("f16", (2, 36, 36, 96, 192, 3, 2)),     # four parity classes
    ("bf16", (2, 20, 20, 384, 384, 1, 1)),
    ("bf16", (2, 64, 96, 3, 48, 3, 2)),      # first layer
    ("bf16", (2, 13, 9, 16, 16, 1, 2)),      # data gradient on the CUDA cores, weight gradient on the tensor cores
    ("f32", (2, 40, 40, 64, 64, 3, 1)),      # slices, and the pass that adds them, last in the data gradient
    ("f32", (1, 9, 7, 8, 12, 3, 1)),         # one slice each: nothing is added
    ("f32", (2, 32, 32, 16, 32, 3, 1)),      # slices of both, added in one launch
    ("f32", (4, 80, 80, 16, 16, 1, 1)),      # 200 slices of the weight gradient, one of the data gradient
    ("f32", (1, 24, 20, 3, 16, 3, 2)),       # element counts that are not multiples of four
]
IDS = ["-".join((m, "x".join(map(str, d)))) for m, d in SHAPES]


def _block(mode, dims, **kw):
    from paper_2609_10632_b200 import binding as nb
    from paper_2609_10632_b200.block import CbsBlock

    modes = {"bf16": nb.NB_MODE_BF16_TC, "f16": nb.NB_MODE_F16_TC, "f32": nb.NB_MODE_F32_REF}
    blk = CbsBlock(wl.ConvShape("bwd", *dims, image_input=dims[3] == 3), mode=modes[mode], flags=nb.NB_CBS_FLAG_SEPARATE_FINALIZE, **kw)
    blk.fill_random(5)
    blk.forward()
    return blk


@pytest.mark.parametrize("need_dx", [True, False], ids=["dx", "no dx"])
@pytest.mark.parametrize("mode,dims", SHAPES, ids=IDS)
def test_one_call_gives_the_bits_of_the_two(mode, dims, need_dx):
    import torch

    blk = _block(mode, dims, need_dx=need_dx)  # (statistics in a fixed order)
    names = [k for k in ("dy", "dx", "dw", "dgamma", "dbeta") if getattr(blk, k) is not None]
    blk.backward_data()
    torch.cuda.synchronize()
    blk.backward_weight()
    blk.poll()
    want = {k: getattr(blk, k).clone() for k in names}
    for _ in range(20):
        for k in names:
            getattr(blk, k).zero_()
        blk.ws.fill_(255)
        blk.backward()
        blk.poll()
        assert all(torch.equal(getattr(blk, k), want[k]) for k in names)


@pytest.mark.parametrize("mode,dims", SHAPES, ids=IDS)
def test_weight_gradient_sees_what_is_written_between_the_calls(mode, dims):
    """dy and x rewritten between the two calls, by kernels of the caller and by one that signals its dependents early (the
    glue addition), so that a weight gradient that did not wait would read the values before."""
    import torch

    from paper_2609_10632_b200 import binding as nb

    blk = _block(mode, dims)
    blk.backward_data()
    torch.cuda.synchronize()
    dy, x = blk.dy.clone(), blk.x.clone()
    x2 = torch.roll(x, 1, 0).flip(1).contiguous()
    blk.dy.copy_(dy * 4)
    blk.x.copy_(x2)
    blk.backward_weight()
    blk.poll()
    want = blk.dw.clone()
    dtype = {"bf16": nb.NB_DTYPE_BF16, "f16": nb.NB_DTYPE_F16, "f32": nb.NB_DTYPE_F32}[mode]
    for i in range(20):
        blk.x.copy_(x)
        blk.dw.zero_()
        blk.backward_data()
        if i % 2 and mode == "bf16":
            rows, c = blk.shape.m, blk.shape.c_out
            blk.x.copy_(x2)
            for _ in range(2):
                nb.nb_slice_add(dtype, rows, c, blk.dy, c, blk.dy, c, b=blk.dy, ld_b=c)
        else:
            blk.dy.mul_(4)
            blk.x.copy_(x2)
        blk.backward_weight()
        blk.poll()
        assert torch.equal(blk.dw, want)


@pytest.mark.parametrize("mode,dims", [c for c in SHAPES if c[0] == "f32"], ids=[i for i in IDS if i.startswith("f32")])
def test_profile_counts_the_launches_that_add_slices(mode, dims):
    """The one call reports as many launches at the site of the slices as it makes, in particular none where nothing is added."""
    from paper_2609_10632_b200 import binding as nb

    blk = _block(mode, dims)

    def sites(call):
        nb.nb_cbs_profile_enable(blk.plan, True)  # (clears the counts)
        before = nb.nb_cbs_launch_count()
        call()
        return nb.nb_cbs_launch_count() - before, nb.nb_cbs_profile_read(blk.plan)["wgrad_splitk_reduce"][1]

    launches2, two = sites(lambda: (blk.backward_data(), blk.backward_weight()))
    launches1, one = sites(blk.backward)
    assert launches2 - launches1 == two - one
    assert (one > 0) == (two > 0)
