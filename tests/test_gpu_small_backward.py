"""Small tensors: both backward passes in one launch (bn_silu_bwd_small_kernel) against the two launches it stands for, and both
against the formulas in fp64."""
import pytest

from paper_2609_10632_b200 import workloads as wl
from tests import parity

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
            out.append({k: getattr(blk, k).clone() for k in ("dy", "dgamma", "dbeta", "dx")})
            _against_fp64(blk)
        got.append(out)
    for one, two in zip(*got):  # one launch and two, dense and pitched
        # The block sums are the same fp32 values; the two launches add them to the fp64 accumulators in any order.  A total in
        # its last fp64 bit is an fp32 result in its last bit, and a coefficient in its last bit, of which dy has four, can
        # turn the rounding of a 16-bit value here and there.
        for k in ("dgamma", "dbeta"):
            a, b = one[k].double(), two[k].double()
            assert ((a - b).abs() <= 2.0**-22 * b.abs() + 2.0**-40 * b.abs().max()).all(), k
        a, b = one["dy"], two["dy"]
        apart = (a.view(torch.int16).int() - b.view(torch.int16).int()).abs()
        small = b.double().abs() <= 2.0**-12 * b.double().pow(2).mean().sqrt()  # (results of cancellation)
        assert (apart[~small] <= 1).all() and (apart[~small] > 0).double().mean() <= 1e-3
        dx = one["dx"].double() - two["dx"].double()
        assert dx.norm() <= 2e-4 * two["dx"].double().norm()


def _against_fp64(blk):
    import torch

    d = lambda t: t.detach().double()
    c, m = blk.shape.c_out, blk.shape.m
    mean, invstd, gamma, beta = d(blk.mean), d(blk.invstd), d(blk.gamma), d(blk.beta)
    y, g = d(blk.y).reshape(m, c), d(blk.g).reshape(m, c)
    xhat = (y - mean) * invstd
    z = gamma * xhat + beta
    s = torch.sigmoid(z)
    dz = g * s * (1 + z * (1 - s))
    dbeta, dgamma = dz.sum(0), (dz * xhat).sum(0)
    dy = gamma * invstd * (dz - dbeta / m - xhat * dgamma / m)
    for name, got, want in (("dbeta", blk.dbeta, dbeta), ("dgamma", blk.dgamma, dgamma), ("dy", blk.dy.reshape(m, c), dy)):
        parity.check(name, d(got).cpu().numpy(), want.cpu().numpy(), "bf16")


@pytest.mark.parametrize("blocks", [74, 75, 148, 149, 296, 297])
def test_reduction_at_its_block_counts(blocks):
    """All eight vectors of a thread at once up to two blocks an SM, a ring of three beyond; the last block one image row short."""
    from paper_2609_10632_b200 import binding as nb
    from paper_2609_10632_b200.block import CbsBlock

    blk = CbsBlock(wl.ConvShape("blocks", 1, 16 * blocks - 1, 16, 16, 64, 1, 1), mode=nb.NB_MODE_BF16_TC)  # 256 rows a block
    blk.fill_random(blocks)
    blk.step()
    blk.poll()
    _against_fp64(blk)


@pytest.mark.parametrize("blocks", [148, 149])
def test_reduction_of_rows_wider_than_256_threads(blocks):
    """2056 channels are a row of 257 threads: all vectors at once up to one block an SM."""
    from paper_2609_10632_b200.block import CbsBlock

    blk = CbsBlock(wl.ConvShape("wide", 1, blocks, 8, 16, 2056, 1, 1))  # eight rows a block
    blk.fill_random(blocks)
    blk.step()
    blk.poll()
    _against_fp64(blk)


def test_reduction_with_all_vectors_at_once_is_one_wave_of_blocks(tmp_path):
    """With all vectors of a thread in registers, the blocks of the backward reduction are on the device together: one an SM in the
    first form, two in the second.  Registers, shared memory and shape of every launch as the profiler reports them."""
    import json

    import torch
    from torch.profiler import ProfilerActivity, profile

    from paper_2609_10632_b200 import binding as nb
    from paper_2609_10632_b200.block import CbsBlock

    prop = torch.cuda.get_device_properties(0)
    sms, sm_smem = prop.multi_processor_count, prop.shared_memory_per_multiprocessor
    blks = []
    for mode, rows in ((nb.NB_MODE_BF16_TC, 256), (nb.NB_MODE_F16_TC, 256), (nb.NB_MODE_F32_REF, 128)):  # rows a block
        for blocks in (sms, sms + 1, 2 * sms):
            for pitched in (False, True):
                blk = CbsBlock(wl.ConvShape("wave", 1, rows // 16 * blocks - 1, 16, 16, 64, 1, 1), mode=mode)
                blk.fill_random(3)
                if pitched:
                    wide = torch.zeros(*blk.g.shape[:-1], 72, dtype=blk.g.dtype, device="cuda")
                    blk.plan.set_pitches(ld_g=72)
                    blk.g = wide[..., 8:]
                blk.step()
                blks.append((blocks, blk))
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        for _, blk in blks:
            blk.step()
        torch.cuda.synchronize()
    prof.export_chrome_trace(str(tmp_path / "trace.json"))
    events = json.loads((tmp_path / "trace.json").read_text())["traceEvents"]
    events = sorted((e for e in events if e.get("cat") == "kernel" and "bn_silu_bwd_reduce_kernel<" in e["name"]), key=lambda e: e["ts"])
    if not events:
        pytest.skip("the profiler delivers no launches here")
    assert len(events) == len(blks)
    for (blocks, _), e in zip(blks, events):
        a = e["args"]
        assert a["grid"][0] == blocks
        warps = -(-a["block"][0] // 32)
        registers = warps * 32 * (-(-a["registers per thread"] // 8) * 8)
        smem = a["shared memory"] + 1024  # (what the system keeps of each block)
        resident = min(65536 // registers, 64 // warps, sm_smem // smem)
        assert blocks <= resident * sms, (e["name"], a)
    forms = [e["name"].split(">(")[0].rsplit(", ", 1)[1] for e in events]
    assert forms == ["1" if blocks <= sms else "2" for blocks, _ in blks]
