"""Host-buffer steps in flight on several streams: a step waits for what its own stream holds and for no other step."""
import pytest

from paper_2609_10632_b200 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPE = wl.ConvShape("host", 2, 20, 20, 64, 96, 3, 1)
IN, OUT = ("x", "w", "gamma", "beta", "g"), ("a", "dx", "dw", "dgamma", "dbeta")


def _buffers(blk):
    import torch

    pinned = lambda t: torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    return {k: pinned(getattr(blk, k)).copy_(getattr(blk, k)) for k in IN}, {k: pinned(getattr(blk, k)) for k in OUT}


@pytest.mark.parametrize("separate", [True, False], ids=["calls of one plan", "calls of two default plans"])
def test_a_step_does_not_queue_behind_a_step_of_another_stream(separate):
    import torch

    from paper_2609_10632_b200 import binding as nb
    from paper_2609_10632_b200.block import CbsBlock

    flags = nb.NB_CBS_FLAG_SEPARATE_FINALIZE if separate else 0
    steps, want = [], []
    for seed in (1, 2):
        blk = CbsBlock(SHAPE, flags=flags)
        blk.fill_random(seed)
        plan = steps[0][0] if separate and steps else blk.plan
        host_in, host_out = _buffers(blk)
        scratch = torch.empty(plan.step_host_scratch_bytes(), dtype=torch.uint8, device="cuda")
        steps.append((plan, host_in, host_out, scratch, torch.cuda.Stream()))
        blk.step()
        blk.poll()
        want.append({k: getattr(blk, k).cpu() for k in OUT})

    def issue(plan, i, o, scratch, stream):
        nb.nb_conv_bn_silu_step_host(plan, *(i[k] for k in IN), *(o[k] for k in OUT), scratch, stream=stream)

    for s in steps:  # a first call each
        issue(*s)
    torch.cuda.synchronize()
    for s in steps:
        for t in s[2].values():
            t.zero_()
    behind, free = steps
    with torch.cuda.stream(behind[4]):
        torch.cuda._sleep(2_000_000_000)  # about a second
    issue(*behind)
    issue(*free)
    free[4].synchronize()
    assert not behind[4].query()
    torch.cuda.synchronize()
    for (plan, _, out, _, _), ref in zip(steps, want):
        nb.nb_cbs_poll_status(plan)
        for k in OUT:
            assert (out[k].double() - ref[k].double()).norm() <= 1e-3 * ref[k].double().norm(), k
            assert not separate or torch.equal(out[k], ref[k]), k  # (sums in a fixed order)


@pytest.mark.parametrize("asked", [True, False], ids=["copy streams", "caller's stream"])
def test_the_step_is_in_place_on_the_callers_stream(asked):
    """Overwriting the host inputs' device source before and reading the results behind the call needs no other ordering, with
    and without the plan's copy streams, and the same inside a graph that the caller records."""
    import torch

    from paper_2609_10632_b200 import binding as nb
    from paper_2609_10632_b200.block import CbsBlock

    blk = CbsBlock(SHAPE, flags=0)
    blk.fill_random(3)
    host_in, host_out = _buffers(blk)
    plan = nb.Plan.for_shape(SHAPE)
    size = (plan if asked else blk.plan).step_host_scratch_bytes()
    scratch = torch.empty(size, dtype=torch.uint8, device="cuda")
    src, stream = blk.x.clone(), torch.cuda.Stream()
    got = torch.empty_like(blk.a)
    host_in["x"].zero_()
    torch.cuda.synchronize()

    def issue():
        host_in["x"].copy_(src, non_blocking=True)
        nb.nb_conv_bn_silu_step_host(plan, *(host_in[k] for k in IN), *(host_out[k] for k in OUT), scratch, stream=stream)
        got.copy_(host_out["a"], non_blocking=True)

    blk.step()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        torch.cuda._sleep(100_000_000)
        issue()
    stream.synchronize()
    assert (got.double() - blk.a.double()).norm() <= 1e-3 * blk.a.double().norm()
    host_in["x"].zero_()
    got.zero_()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        issue()
    graph.replay()
    torch.cuda.synchronize()
    assert (got.double() - blk.a.double()).norm() <= 1e-3 * blk.a.double().norm()
