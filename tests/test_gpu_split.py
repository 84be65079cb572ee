"""The split-K cluster form of the implicit GEMM (layers with few output tiles) with every cluster size forced: k-blocks that
do not divide evenly, a 32-channel tail k-block, ragged rows, padded columns, the parity classes of a stride-2 data gradient
with odd extents, and a data gradient added into a channel slice (the training calls use clusters of one alone).  Each test makes sure that its plans have this form."""
import re

import pytest

from paper_2609_10632_b200 import workloads as wl
from tests import parity
from tests.test_gpu_parity import EPS, _compare, _oracle, _run_block

pytestmark = pytest.mark.gpu

LINE = re.compile(r"split igemm( \(evaluation\))? M=(\d+) Ca=(\d+) rowsB=(\d+) .*BN=(\d+) S=(\d+) stages=(\d+)")


def _chosen(capfd):
    """The split launches that the plans created since the last look have chosen (their lines under NB_TC_VERBOSE):
    (evaluation call?, channels of the A operand, rows of the B operand, tile columns, cluster size, operand stages)."""
    found = LINE.findall(capfd.readouterr().err)
    return [(bool(ev), int(ca), int(rows), int(cols), int(size), int(stages)) for ev, _, ca, rows, cols, size, stages in found]


SHAPES = [
    (1, 20, 20, 192, 192, 3, 1),  # 27 k-blocks, four row tiles
    (2, 13, 11, 96, 80, 3, 1),    # 18 k-blocks of 64 and 32 channels, 286 rows
    (3, 11, 9, 72, 136, 3, 1),    # padded columns, tail of 8 channels
    (1, 17, 19, 128, 64, 3, 2),   # parity classes of 1, 2, 2 and 4 taps, odd height and width
    (2, 12, 14, 512, 48, 1, 1),   # tiled A map
]


@pytest.mark.parametrize("split", [1, 2, 4, 8])
@pytest.mark.parametrize("dims", SHAPES, ids=lambda d: "x".join(map(str, d)))
def test_split_launches_match_oracle(dims, split, monkeypatch, capfd):
    import oracle
    import torch

    from paper_2609_10632_b200 import binding as nb
    from paper_2609_10632_b200.block import CbsBlock

    monkeypatch.setenv("NB_TC_SPLIT_S", str(split))
    monkeypatch.setenv("NB_TC_VERBOSE", "1")
    shape = wl.ConvShape("split", *dims)
    mode = nb.NB_MODE_F16_TC if split == 2 else nb.NB_MODE_BF16_TC
    inp, blk, out = _run_block(shape, mode, cfg_id=43, layer_id=SHAPES.index(dims), affine="random")
    evaluation = (True, shape.c_in, shape.c_out, split)
    training = [(False, shape.c_in, shape.c_out, 1), (False, shape.c_out, shape.c_in, 1)]  # forward, data gradient
    chosen = [(ev, ca, rows, size) for ev, ca, rows, _, size, _ in _chosen(capfd)]
    assert sorted(chosen) == sorted([evaluation] + (training if split == 1 else []))
    _compare(out, _oracle(inp), 0)
    again = CbsBlock(shape, mode=mode, eps=EPS)
    again.upload(inp)
    again.step()
    assert torch.equal(again.y, blk.y) and torch.equal(again.dx, blk.dx)  # rank order: the same bits every run
    rm, rv, _ = wl.make_eval_stats(shape, 43, SHAPES.index(dims))
    up = lambda a: torch.from_numpy(a).to(blk.dev)
    o = torch.empty_like(blk.a)
    ws = torch.empty(max(blk.plan.infer_bytes, 256), dtype=torch.uint8, device=blk.dev)
    nb.nb_conv_bn_silu_infer(blk.plan, blk.x, blk.w, blk.gamma, blk.beta, up(rm), up(rv), o, ws)
    torch.cuda.synchronize()
    assert blk.poll() == ""
    parity.check("a_eval", o.double().cpu().numpy(), oracle.cbs_infer(inp.x, inp.w, inp.gamma, inp.beta, rm, rv, shape.stride, EPS), "bf16")
    if shape.stride == 1:  # round(old + dx) in a channel slice, nothing beside it
        wide = torch.randn(shape.n, shape.h, shape.w, shape.c_in + 24, device=blk.dev).to(blk.dx.dtype)
        want = wide.clone()
        want[..., 8:8 + shape.c_in] = (wide[..., 8:8 + shape.c_in].float() + blk.dx.float()).to(wide.dtype)
        blk.plan.set_dx_target(ld_dx=shape.c_in + 24, accumulate=True)
        blk.dx = wide[..., 8:8 + shape.c_in]
        blk.backward_data()
        torch.cuda.synchronize()
        assert torch.equal(wide, want)


WIDTHS = [16, 48, 80, 112, 128, 144, 208, 256]


def _evaluate(shape, seed):
    """One evaluation call of a fresh plan against the oracle."""
    import numpy as np
    import oracle
    import torch

    from paper_2609_10632_b200 import binding as nb

    inp = wl.make_inputs(shape, 47, seed, bf16=True, affine="random")
    rm, rv, _ = wl.make_eval_stats(shape, 47, seed)
    plan = nb.Plan.for_shape(shape, eps=EPS)
    dev = lambda a, dt=torch.float32: torch.from_numpy(np.ascontiguousarray(a)).to(dt).cuda()
    x, w = dev(inp.x, torch.bfloat16), dev(inp.w, torch.bfloat16)
    out = torch.full((shape.n, shape.ho, shape.wo, shape.c_out), 7.0, dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(max(plan.infer_bytes, 256), dtype=torch.uint8, device="cuda")
    nb.nb_conv_bn_silu_infer(plan, x, w, dev(inp.gamma), dev(inp.beta), dev(rm), dev(rv), out, ws)
    torch.cuda.synchronize()
    assert nb.nb_cbs_poll_status(plan) == ""
    parity.check("a_eval", out.double().cpu().numpy(), oracle.cbs_infer(inp.x, inp.w, inp.gamma, inp.beta, rm, rv, shape.stride, EPS), "bf16")


@pytest.mark.parametrize("cols,split", [(c, s) for c in WIDTHS for s in (1, 2, 8) if s == 1 or c <= 128])
def test_tile_widths_of_the_evaluation_call(cols, split, monkeypatch, capfd):
    """Every way in which the warps share a tile's columns: one 16-column piece to sixteen of them (clusters: to eight), a last
    tile with padding columns."""
    monkeypatch.setenv("NB_TC_SPLIT_S", str(split))
    monkeypatch.setenv("NB_TC_SPLIT_BN", str(cols))
    monkeypatch.setenv("NB_TC_VERBOSE", "1")
    shape = wl.ConvShape("width", 2, 9, 17, 128, 2 * cols - 8 if cols > 16 else 16, 3, 1)
    _evaluate(shape, cols)
    assert [c[3:5] for c in _chosen(capfd) if c[0]] == [(cols, split)]


@pytest.mark.parametrize("cols", [112, 128])
@pytest.mark.parametrize("per_rank", [1, 2])
@pytest.mark.parametrize("split", [2, 4, 8])
def test_short_k_ranges_of_a_cluster(split, per_rank, cols, monkeypatch, capfd):
    """One and two k-blocks a rank.  Two operand stages are the fewest; a rank lays its 128 x (columns + 8) sums over them before
    it hands them out, which fits exactly at 112 columns and takes a third stage at 128."""
    monkeypatch.setenv("NB_TC_SPLIT_S", str(split))
    monkeypatch.setenv("NB_TC_SPLIT_BN", str(cols))
    monkeypatch.setenv("NB_TC_VERBOSE", "1")
    shape = wl.ConvShape("short", 2, 9, 17, 64 * split * per_rank, cols, 1, 1)
    _evaluate(shape, 300 + cols)
    assert [c[3:] for c in _chosen(capfd) if c[0]] == [(cols, split, 2 if cols == 112 else 3)]


@pytest.mark.parametrize("dims,cols,calls", [  # the calls whose channel count has such a tile; the other one stays on the persistent kernel
    ((2, 20, 20, 288, 288, 3, 1), 144, "both"), ((1, 40, 40, 192, 192, 3, 1), 32, "both"), ((3, 11, 9, 96, 192, 3, 2), 48, "both"),
    ((1, 33, 31, 64, 144, 3, 1), 144, "forward"), ((4, 13, 9, 256, 176, 1, 1), 176, "forward"), ((2, 17, 19, 40, 256, 3, 1), 256, "forward"),
    ((1, 33, 31, 144, 64, 3, 1), 144, "data gradient"), ((2, 17, 19, 160, 40, 3, 1), 160, "data gradient")],
    ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_training_calls_have_the_bits_of_the_persistent_form(dims, cols, calls, monkeypatch, capfd):
    import torch

    from paper_2609_10632_b200.block import CbsBlock

    got = []
    monkeypatch.setenv("NB_TC_VERBOSE", "1")
    for split in ("0", "1"):
        monkeypatch.setenv("NB_TC_SPLIT", split)
        if split == "1":
            monkeypatch.setenv("NB_TC_SPLIT_BN", str(cols))
        blk = CbsBlock(wl.ConvShape("bits", *dims), eps=EPS)
        blk.fill_random(3)
        blk.step()
        blk.poll()
        got.append(blk)
        forward, data = (dims[3], dims[4], cols), (dims[4], dims[3], cols)
        expect = {"0": [], "1": {"both": [forward, data], "forward": [forward], "data gradient": [data]}[calls]}[split]
        assert sorted(c[1:4] for c in _chosen(capfd) if not c[0]) == sorted(expect)
    assert all(torch.equal(getattr(got[0], k), getattr(got[1], k)) for k in ("y", "mean", "invstd", "dx"))


@pytest.mark.parametrize("dims", [(1, 3, 11, 96, 96, 3, 1), (1, 7, 5, 96, 96, 3, 2), (1, 17, 17, 72, 80, 3, 1), (2, 9, 16, 40, 80, 3, 1)], ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("split", ["0", "1"])
def test_warps_of_which_some_rows_do_not_exist(split, dims, monkeypatch, capfd):
    """Accumulator rows past the last pixel, outside an odd parity class or past the last input channel of a tap, in a warp whose
    other rows are stored, with several pieces of columns a warp: the rows that exist are right in every piece."""
    monkeypatch.setenv("NB_TC_SPLIT", split)
    monkeypatch.setenv("NB_TC_SPLIT_S", "1")
    monkeypatch.setenv("NB_TC_SPLIT_BN", str((dims[4] + 15) // 16 * 16))
    monkeypatch.setenv("NB_TC_VERBOSE", "1")
    inp, blk, out = _run_block(wl.ConvShape("edge", *dims), 0, cfg_id=53, layer_id=dims[3], affine="random")
    assert blk.plan.paths == {"fprop": 1, "dgrad": 1, "wgrad": 1}
    assert any(not c[0] for c in _chosen(capfd)) == (split == "1")
    _compare(out, _oracle(inp), 0)
