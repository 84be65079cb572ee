"""GraphRunner replays a recording of its passes from the second call with unchanged arguments on: the same bits as issuing
the calls, with new values in the same tensors, after a tensor or a plan option was replaced, on streams of the caller, and
inside a graph that the caller records."""
import pytest

from paper_2609_10632_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [False, True], ids=["one stream", "weight gradients on a second stream"])
def test_replayed_passes_give_the_issued_bits(side):
    import torch

    from paper_2609_10632_b200 import binding as nb
    from paper_2609_10632_b200.detector import GraphRunner

    ops, layers, outs, plain = wl.detector_graph(1, 64, plain_head=True)
    run = GraphRunner(ops, layers, outs, plain_layers=plain)
    run.fill_parameters(seed=3)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    for pl in run.plain:
        pl["w"].normal_(0.0, 0.05, generator=gen)
        pl["bias"].normal_(0.0, 0.5, generator=gen)
    second = torch.cuda.Stream() if side else None
    ws = torch.empty(max(b.plan.bwd_bytes for b in run.blocks), dtype=torch.uint8, device="cuda") if side else None

    def inputs(seed):
        gen.manual_seed(seed)
        run.buf["img"].uniform_(0.0, 1.0, generator=gen)
        for name in outs:
            run.grad[name].normal_(generator=gen)

    def results():
        torch.cuda.synchronize()
        run.poll()
        return [t.clone() for t in [run.buf[o] for o in outs] + [run.grad["img"]] + [b.dw for b in run.blocks] + [b.dgamma for b in run.blocks]]

    def step(stream=None):
        before = nb.nb_cbs_launch_count()
        run.forward(stream)
        run.backward(stream, wgrad_stream=second, wgrad_workspace=ws)
        return nb.nb_cbs_launch_count() - before

    def issued(seed):  # the calls themselves
        inputs(seed)
        run._forward(None)
        torch.cuda.synchronize()
        run._backward(None, second, ws)
        return results()

    def same(seed, stream=None):
        want = issued(seed)
        inputs(seed)
        torch.cuda.synchronize()
        n = step(stream)
        assert all(torch.equal(a, b) for a, b in zip(results(), want))
        return n

    counts = [same(seed) for seed in (1, 2, 3, 4)]  # issued, recorded and replayed, replayed, replayed
    assert len(set(counts)) == 1 and counts[0] > 400
    run.blocks[5].dw = torch.zeros_like(run.blocks[5].dw)  # another tensor: issued again, then recorded again
    assert [same(seed) for seed in (5, 6, 7)] == counts[:3]
    mine = torch.cuda.Stream()
    assert [same(seed, mine) for seed in (8, 9)] == counts[:2]
    want = issued(10)
    inputs(10)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        if side:
            second.wait_stream(torch.cuda.current_stream())
        step()
        if side:
            torch.cuda.current_stream().wait_stream(second)
    graph.replay()
    assert all(torch.equal(a, b) for a, b in zip(results(), want))


def _small_runner():
    import torch

    from paper_2609_10632_b200.detector import GraphRunner

    ops, layers, outs, plain = wl.detector_graph(1, 64, plain_head=True)
    run = GraphRunner(ops, layers, outs, plain_layers=plain)
    run.fill_parameters(seed=3)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    for pl in run.plain:
        pl["w"].normal_(0.0, 0.05, generator=gen)
        pl["bias"].normal_(0.0, 0.5, generator=gen)
    run.buf["img"].uniform_(0.0, 1.0, generator=gen)
    return run, outs


def test_a_plan_that_takes_the_place_of_another_is_issued_and_recorded():
    """Another plan of the same revision (every setter called as often), here with the statistics finished by kernels of their
    own: its launches are more.  The old plan stays alive until the end, so that a recording that was replayed by mistake
    would find its accumulators."""
    import torch

    from paper_2609_10632_b200 import binding as nb

    run, outs = _small_runner()

    def forward():
        before = nb.nb_cbs_launch_count()
        run.forward()
        torch.cuda.synchronize()
        return nb.nb_cbs_launch_count() - before, [run.buf[o].clone() for o in outs]

    n, first = forward()
    assert [forward()[0] for _ in range(2)] == [n, n]
    k = next(i for i, b in enumerate(run.blocks) if not hasattr(b, "res") and not hasattr(b, "gres"))
    blk = run.blocks[k]
    old, new = blk.plan, nb.Plan.for_shape(blk.shape, flags=nb.NB_CBS_FLAG_SEPARATE_FINALIZE)
    for _ in range(old.revision):
        new.set_pitches(ld_x=blk.x.stride(-2), ld_a=blk.a.stride(-2), ld_g=blk.g.stride(-2))
    assert new.revision == old.revision
    blk.plan = new
    more = [forward() for _ in range(3)]
    assert len({m for m, _ in more}) == 1 and more[0][0] > n
    assert all(torch.equal(a, b) for _, outputs in more[1:] for a, b in zip(outputs, more[0][1]))
    assert blk.plan is new and old.handle


@pytest.mark.parametrize("side", [False, True], ids=["one stream", "weight gradients on a second stream"])
def test_an_error_in_a_recorded_call_reaches_the_caller(side):
    """A call that refuses its arguments while the pass is being recorded, with branches open: the caller gets its error, and the
    runner records and replays again once the cause is gone."""
    import torch

    from paper_2609_10632_b200 import binding as nb

    run, outs = _small_runner()
    for name in outs:
        run.grad[name].normal_()
    second = torch.cuda.Stream() if side else None
    ws = torch.empty(max(b.plan.bwd_bytes for b in run.blocks), dtype=torch.uint8, device="cuda") if side else None

    def passes():
        run.forward()
        run.backward(wgrad_stream=second, wgrad_workspace=ws)

    passes()
    torch.cuda.synchronize()
    want = [run.grad["img"].clone()] + [b.dw.clone() for b in run.blocks]
    blk = run.blocks[20]
    good, blk.dy = blk.dy, blk.dy.view(-1)[1:]  # not on a 16-byte boundary
    for _ in range(3):
        with pytest.raises(nb.NbError) as ei:  # issued, recorded, recorded again
            passes()
        assert ei.value.status == nb.NB_ERR_ALIGNMENT
    blk.dy = good
    torch.cuda.synchronize()
    assert not torch.cuda.is_current_stream_capturing()
    for _ in range(3):
        run.grad["img"].zero_()
        passes()
        torch.cuda.synchronize()
        run.poll()
        assert all(torch.equal(a, b) for a, b in zip([run.grad["img"]] + [b.dw for b in run.blocks], want))


def test_garbage_of_others_does_not_end_a_recording(monkeypatch):
    """A CUDA graph that nobody holds any more but for a reference cycle, and enough new objects for a collection, in the middle of
    a recording: freeing the graph there would invalidate the capture."""
    import gc

    import torch

    run, outs = _small_runner()
    run.forward()
    torch.cuda.synchronize()
    want = [run.buf[o].clone() for o in outs]
    old, t = torch.cuda.CUDAGraph(), torch.zeros(16, device="cuda")
    with torch.cuda.graph(old):
        t.add_(1)
    old.replay()
    held, blk = [old], run.blocks[3]
    del old

    def forward(stream=None, call=blk.forward):
        cycle = [held.pop()] if held else []
        cycle.append(cycle)
        del cycle
        many = [[] for _ in range(100_000)]
        call(stream)
        assert len(many) == 100_000

    monkeypatch.setattr(blk, "forward", forward)
    assert gc.isenabled()
    run.forward()
    assert gc.isenabled() and not held
    torch.cuda.synchronize()
    assert all(torch.equal(run.buf[o], a) for o, a in zip(outs, want))
