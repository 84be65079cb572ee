"""The order of the host-buffer step (csrc/host_step.cuh) on stand-ins for its copies, calls and orderings, which fail at every
point in turn: what reads a tensor is ordered behind what wrote it, and however the call ends, the caller's stream is ordered
behind everything that was queued elsewhere."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include "host_step.cuh"
using namespace nbcbs;
struct Ops {
    int fail_at, n = 0;
    int op(const char* what, int a, int b) {
        const int s = n++ == fail_at ? 5 : 0;
        std::printf("%s %d %d %d\n", what, a, b, s);
        return s;
    }
    int copy(HostStepTensor t, HostStepStream st) { return op("copy", t, st); }
    int order(HostStepStream a, HostStepStream b) { return op("order", a, b); }
    int op(const char* what, int st) { return op(what, st, 0); }
    int forward() { return op("forward", HS_CALLER); }
    int backward_data() { return op("backward_data", HS_CALLER); }
    int backward_weight() { return op("backward_weight", HS_CALLER); }
};
int main(int, char** v) {
    Ops ops{std::atoi(v[3])};
    std::printf("end %d 0 0\n", host_step(ops, v[1][0] == '1', v[2][0] == '1'));
}
"""
CALLER, IN, OUT = range(3)
X, W, GAMMA, BETA, G, A, DX, DW, DGAMMA, DBETA = range(10)
NEEDS = {"forward": [X, W, GAMMA, BETA], "backward_data": [G, "forward"], "backward_weight": ["backward_data"],
         A: ["forward"], DX: ["backward_data"], DGAMMA: ["backward_data"], DBETA: ["backward_data"], DW: ["backward_weight"]}


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("host_step")
    (d / "harness.cc").write_text(HARNESS)
    subprocess.check_call([gxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_2609_10632_b200", "csrc"), "-x", "c++", str(d / "harness.cc"), "-o", str(d / "harness")])
    return str(d / "harness")


def _play(program, copy_streams, want_dx, fail_at):
    """(status, operations issued, what each stream is ordered behind at the end)"""
    out = subprocess.run([program, str(int(copy_streams)), str(int(want_dx)), str(fail_at)], capture_output=True, text=True, check=True).stdout
    behind, queued = {s: set() for s in (CALLER, IN, OUT)}, []
    for line in out.splitlines():
        what, a, b, failed = line.split()
        a, b, failed = int(a), int(b), int(failed)
        if what == "end":
            return a, queued, behind
        if what == "order":
            queued.append(what)
            if not failed:
                behind[b] |= behind[a]
            continue
        name, stream = (a, b) if what == "copy" else (what, a)
        queued.append(name)
        if not failed:
            assert all(n in behind[stream] for n in NEEDS.get(name, ())), (name, behind[stream])
            behind[stream].add(name)


@pytest.mark.parametrize("want_dx", [True, False], ids=["dx", "no dx"])
@pytest.mark.parametrize("copy_streams", [True, False], ids=["copy streams", "one stream"])
def test_order_and_every_way_to_fail(program, copy_streams, want_dx):
    status, whole, behind = _play(program, copy_streams, want_dx, -1)
    everything = {X, W, GAMMA, BETA, G, A, DW, DGAMMA, DBETA, "forward", "backward_data", "backward_weight"} | ({DX} if want_dx else set())
    assert status == 0 and behind[CALLER] == everything and set(whole) - {"order"} == everything
    assert copy_streams or "order" not in whole  # without streams of its own the step is issued on the caller's alone
    for fail_at in range(len(whole)):
        status, queued, behind = _play(program, copy_streams, want_dx, fail_at)
        assert status == 5, fail_at
        assert queued[:fail_at] == whole[:fail_at] and set(queued[fail_at + 1:]) <= {"order"}  # nothing more but the joins
        last = fail_at == len(whole) - 1 and copy_streams  # (the last join itself: nothing is left to try)
        assert last or behind[CALLER] >= behind[IN] | behind[OUT], fail_at
