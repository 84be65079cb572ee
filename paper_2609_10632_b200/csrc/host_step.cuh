// The order in which a training step from host buffers issues its copies and calls (nb_conv_bn_silu_step_host), apart from what
// issues them: plain C++ without CUDA types, so that a CPU test can run it on stand-ins that fail at any point.
#pragma once

namespace nbcbs {

enum HostStepStream { HS_CALLER, HS_IN, HS_OUT };
enum HostStepTensor { HT_X, HT_W, HT_GAMMA, HT_BETA, HT_G, HT_A, HT_DX, HT_DW, HT_DGAMMA, HT_DBETA };

// Ops: int copy(HostStepTensor, HostStepStream); int order(HostStepStream from, HostStepStream to) (`to` continues behind
// everything queued on `from` so far); int forward(), backward_data(), backward_weight(), all three on the caller's stream.
// Zero is success; the first failure is returned, with everything queued so far in front of what the caller queues next.
//
// PCIe moves data both ways at once.  With copy streams g travels in while a travels out, and dx goes out while the weight
// gradient is computed; on the caller's stream alone every byte of either direction waits for every other.  A caller that
// keeps several steps in flight on streams of its own has that overlap already, and there the additional streams and their
// event waits only hold the copies up: which of the two a plan does is the plan's (see copy_in in nb_cbs.cu).
template <class Ops> int host_step(Ops& ops, bool copy_streams, bool want_dx) {
    const HostStepStream in = copy_streams ? HS_IN : HS_CALLER, out = copy_streams ? HS_OUT : HS_CALLER;
    auto order = [&](HostStepStream from, HostStepStream to) { return from == to ? 0 : ops.order(from, to); };
    auto copy = [&](HostStepStream stream, auto... tensors) {
        int s = 0;
        ((s = s ? s : ops.copy(tensors, stream)), ...);
        return s;
    };
    auto issue = [&]() {
        int s = order(HS_CALLER, in);
        if (!s) s = copy(in, HT_W, HT_GAMMA, HT_BETA, HT_X);
        if (!s) s = order(in, HS_CALLER);
        if (!s) s = copy(in, HT_G);
        if (!s) s = ops.forward();
        if (!s && copy_streams) {
            s = order(HS_CALLER, out);
            if (!s) s = copy(out, HT_A);
            if (!s) s = order(in, HS_CALLER);
        }
        if (!s) s = ops.backward_data();
        if (!s && copy_streams) {
            s = order(HS_CALLER, out);
            if (!s && want_dx) s = copy(out, HT_DX);
            if (!s) s = copy(out, HT_DGAMMA, HT_DBETA);
        }
        if (!s) s = ops.backward_weight();
        if (!s && !copy_streams) {
            s = copy(out, HT_A);
            if (!s && want_dx) s = copy(out, HT_DX);
            if (!s) s = copy(out, HT_DGAMMA, HT_DBETA);
        }
        if (!s) s = copy(HS_CALLER, HT_DW);
        return s;
    };
    const int s = issue();
    if (!copy_streams) return s;
    const int i = s ? order(in, HS_CALLER) : 0;  // (after a whole step the caller's stream already waits for `in`)
    const int o = order(out, HS_CALLER);
    return s ? s : i ? i : o;
}

}  // namespace nbcbs
