// C ABI of the Conv -> BN(train) -> SiLU block library (see include/nb_cbs.h): plans, validation, workspace
// carving and kernel dispatch.  No device memory is allocated here except the plan's status block.
// (The optimiser step of include/nb_sgd.h lives in nb_sgd.cu, the glue calls of include/nb_glue.h in nb_glue.cu.)
#include "../../include/nb_cbs.h"

#include <algorithm>
#include <atomic>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "elementwise.cuh"
#include "host_step.cuh"
#include "simt_conv.cuh"
#include "stem_conv.cuh"
#include "tc_conv.cuh"
#include "api_common.cuh"

using namespace nbcbs;
using namespace nbapi;

namespace nbapi {  // shared with the other translation units of the library (api_common.cuh)

thread_local std::string g_err;

nb_status fail(nb_status code, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

std::atomic<unsigned long long> g_launches{0};  // kernels launched by this library in this process

}  // namespace nbapi

namespace {

enum Site { SITE_FPROP = 0, SITE_STATS, SITE_FINALIZE, SITE_APPLY, SITE_BWD_REDUCE, SITE_BWD_FINALIZE, SITE_BWD_DY,
            SITE_WTRANSFORM, SITE_DGRAD, SITE_WGRAD, SITE_SPLITK_REDUCE, SITE_INFER, SITE_EVAL_COEF, SITE_FOLD, SITE_COUNT };
const char* const kSiteNames[SITE_COUNT] = {"conv_fprop", "bn_stats", "bn_finalize", "bn_silu_apply", "bn_silu_bwd_reduce",
                                            "bn_bwd_finalize", "bn_silu_bwd_dy", "dgrad_weight_transform", "conv_dgrad",
                                            "conv_wgrad", "wgrad_splitk_reduce", "conv_infer_fused", "bn_eval_coef", "bn_fold"};

struct EwCfg {  // launch geometry of the [M][C] passes
    int vec, cgs, tpb;
    long long total_vecs;
    int blocks_reduce, blocks_map;  // stats / backward-reduce grids (they size the partial buffers) and apply / dy grids
    int blocks_stats, blocks_apply, blocks_dy;
    int wave_reduce;  // resident blocks of the backward-reduce kernel (ring form) on the whole device
    int wave_deep;  // the same of the form that asks for all vectors of a thread at once, at most two an SM
    int slabs, slab_ctas, slab_units, slab_threads;  // both backward passes in one launch: channel slabs (0: two launches), CTAs of a slab, row blocks and threads of a CTA
};

}  // namespace

struct SgCfg {  // launch of one CUDA-core convolution
    int bm, bn, splits;
    long long kchunk;
    dim3 grid;
    size_t partial_bytes;  // slices as fp32 (0: one slice)
};

constexpr size_t kStatusBytes = 256;  // ST_WORDS ints, padded so that what follows in the same allocation is 256-byte aligned
static_assert(ST_WORDS * sizeof(int) <= kStatusBytes, "status block");

struct nb_cbs_plan_s {
    nb_cbs_desc desc;
    Geom g;
    int device;
    int sm_count;
    int* status;  // device, ST_WORDS ints
    EwCfg ew;
    int nparts;      // rows of the partial-sum buffers
    SgCfg sg[3];     // CUDA-core convolutions: fprop, dgrad, wgrad
    TcPlan tc;       // tensor-core kernel choices (all disabled when unsupported or forced off)
    long long ld_a = 0, ld_g = 0;  // row pitch (elements) of a_out in the forward call and of g in the backward call (set by nb_cbs_plan_set_pitches; default c_out)
    const void* fwd_res = nullptr;  // residual added to the forward call's output (nb_cbs_plan_set_fwd_residual) and its row pitch
    long long ld_res = 0;
    void* bwd_gres = nullptr;       // tensor that the data-gradient call adds (or copies) its incoming gradient to (nb_cbs_plan_set_bwd_residual)
    long long ld_gres = 0;
    bool gres_add = true;
    long long ld_dx = 0;           // row pitch of dx in the data-gradient call and whether dx is added to (nb_cbs_plan_set_dx_target)
    bool dx_accumulate = false;
    bool pitched = false;
    // Channel sums go to accumulators that the consuming pass turns into coefficients itself (ChanAcc); off
    // (NB_CBS_FLAG_SEPARATE_FINALIZE): per-block partial sums and separate finalize kernels.
    bool fuse_finalize = true;
    double* acc = nullptr;      // device: [acc_copies_f][2][C] forward sums, then [acc_copies_b][2][C] backward sums (fp32 mode: 64-bit words); zero between calls
    int acc_copies_f = 0, acc_copies_b = 0;
    // fp32 mode, whose sums are ten words each: above 160 channels kernels of their own derive the coefficients, below every block
    // of the consuming pass does.  Measured (step; blocks / kernels, and what fp64 sums took that depended on the order of the
    // atomics), 2 x 40 x 40 pixels: 64 channels 58.5 / 62.0 us (57.3), 96 81.9 / 84.1 (77.9), 128 85.2 / 86.5 (81.5), 192 53.5 / 52.8
    // (51.0), 256 58.2 / 56.9 (54.9); 288 on 4 x 20 x 20 271.7 / 265.6 (262.3), 576 on 20 x 20 71.5 / 54.7 (53.5).
    bool exact_apart = false;
    bool stem = false;       // 3-channel 3x3 stride-2 first layer: dedicated direct kernels
    int stem_blocks = 0;     // blocks (= partial slices) of the stem wgrad kernel
    bool stem_wide = false;  // the stem forward kernel takes 320-pixel strips (wide images)
    int stem_fprop_blocks = 0;  // its grid (= its partial slices)
    int stem_wgrad_blocks = 0;  // grid (= partial slices) of the stem weight-gradient kernel (128-pixel strips on wide images)
    int stem_dgrad_blocks = 0;  // grid of the stem data-gradient kernel (at most one wave of five resident blocks per SM unless the bands alone are more)
    int stem_dgrad_rows = 0;    // output row pairs per block
    bool profiling = false;  // when set, every kernel site is bracketed by events and the call waits for it
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    // nb_conv_bn_silu_step_host: streams for its copies in either direction, one event per ordering of two of its streams.  A
    // default plan has them from its first nb_cbs_step_host_scratch_bytes on (its calls follow one another, so that a pair of its
    // own holds nothing up); an NB_CBS_FLAG_SEPARATE_FINALIZE plan never has, because calls of it may be in flight on several of
    // the caller's streams, which would all queue in that one pair.  Measured, the detector's 77 layers (3.6 GB in, 3.7 GB out)
    // with SEPARATE_FINALIZE plans on six streams: 96 ms with copy streams of the plans, 91 ms with one pair for all plans, 86.5 ms
    // with the copies on the caller's streams; on one stream 118, 118 and 146 ms (a default plan for every layer: 118 ms, on six
    // streams 90 ms).  One call at a time, default plan: 384 -> 384 1x1 on 16 x 40 x 40 pixels (40 MB each way) 1566 us on the
    // caller's stream, 1227 us with copy streams; 64 -> 64 3x3 on 2 x 20 x 20 (200 KB) 106 and 85 us.
    cudaStream_t copy_in = nullptr, copy_out = nullptr;
    cudaEvent_t copy_ev[3][3] = {};
    double prof_ms[SITE_COUNT] = {};
    long long prof_n[SITE_COUNT] = {};
    size_t fwd_bytes, bwd_bytes;
    size_t off_sgpart;           // slices of a split CUDA-core forward convolution
    size_t infer_bytes, off_iy, off_isg;  // evaluation-mode forward: scale and shift at the forward offsets, then the convolution output when not fused
    // workspace offsets
    size_t off_scale, off_shift, off_fpart;                  // forward
    size_t off_coef, off_bpart, off_wt, off_dgpart, off_wgpart;          // backward
};

namespace {

bool is_f32(const nb_cbs_plan_s* p) { return p->desc.mode == NB_MODE_F32_REF; }
bool is_f16(const nb_cbs_plan_s* p) { return p->desc.mode == NB_MODE_F16_TC; }
// Run an expression with AT = the plan's 16-bit activation type (bf16, or IEEE fp16 in NB_MODE_F16_TC).
#define NB_WITH_AT(p, ...) (is_f16(p) ? ([&]() { using AT = __half; return __VA_ARGS__; })() : ([&]() { using AT = __nv_bfloat16; return __VA_ARGS__; })())
// the evaluation-mode forward is one tensor-core kernel with the per-channel epilogue fused
bool infer_fused(const nb_cbs_plan_s* p) { return !is_f32(p) && (p->stem || p->tc.infer); }

nb_status check_ptr(const void* p, const char* name, bool nullable = false) {
    if (!p) return nullable ? NB_OK : fail(NB_ERR_INVALID_ARG, "%s is NULL", name);
    if (reinterpret_cast<uintptr_t>(p) & 15u) return fail(NB_ERR_ALIGNMENT, "%s is not 16-byte aligned", name);
    return NB_OK;
}
#define NB_CHECK_PTR(p, ...)                                   \
    do {                                                       \
        nb_status s__ = check_ptr((p), #p, ##__VA_ARGS__);     \
        if (s__ != NB_OK) return s__;                          \
    } while (0)


// Brackets one kernel site with events when the plan is in profiling mode (diagnostic; synchronises the stream).
struct SiteTimer {
    nb_cbs_plan_s* p;
    int site;
    cudaStream_t st;
    SiteTimer(nb_cbs_plan_s* plan, int s, cudaStream_t stream) : p(plan), site(s), st(stream) {
        if (p->profiling) cudaEventRecord(p->ev0, st);
    }
    ~SiteTimer() {
        if (!p->profiling) return;
        cudaEventRecord(p->ev1, st);
        float ms = 0.f;
        if (cudaEventSynchronize(p->ev1) == cudaSuccess && cudaEventElapsedTime(&ms, p->ev0, p->ev1) == cudaSuccess) {
            p->prof_ms[site] += ms;
            p->prof_n[site] += 1;
        }
    }
};


// The streams and events of nb_conv_bn_silu_step_host: all of them, or none when one cannot be had (the copies then take the
// caller's stream, as they do for a plan that nobody has asked for its scratch size).
void drop_copy_streams(nb_cbs_plan_s* p) {
    if (p->copy_in) cudaStreamDestroy(p->copy_in);  // (work still queued completes first)
    if (p->copy_out) cudaStreamDestroy(p->copy_out);
    p->copy_in = p->copy_out = nullptr;
    for (auto& row : p->copy_ev)
        for (cudaEvent_t& e : row) {
            if (e) cudaEventDestroy(e);
            e = nullptr;
        }
}
void make_copy_streams(nb_cbs_plan_s* p) {
    DeviceGuard on_device(p->device);
    bool ok = cudaStreamCreateWithFlags(&p->copy_in, cudaStreamNonBlocking) == cudaSuccess && cudaStreamCreateWithFlags(&p->copy_out, cudaStreamNonBlocking) == cudaSuccess;
    for (int copy = HS_IN; copy <= HS_OUT; ++copy)
        for (cudaEvent_t* e : {&p->copy_ev[HS_CALLER][copy], &p->copy_ev[copy][HS_CALLER]})
            ok = ok && cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess;
    if (ok) return;
    (void)cudaGetLastError();
    drop_copy_streams(p);
}

// ---------------------------------------------------------------- elementwise launch helpers
template <typename YT> nb_status run_stats_partial(nb_cbs_plan_s* p, const void* y, float* partials, cudaStream_t st) {
    const EwCfg& e = p->ew;
    SiteTimer tm(p, SITE_STATS, st);
    launch_k(bn_stats_partial_kernel<YT>, dim3(e.blocks_stats), dim3(e.tpb), (size_t)e.tpb * e.vec * sizeof(float), st, 1,
        static_cast<const YT*>(y), e.total_vecs, p->g.c_out, partials);
    return launch_ok("bn_stats_partial");
}

nb_status run_finalize(nb_cbs_plan_s* p, const float* partials, int nparts, const float* gamma, const float* beta, float* mean,
                       float* invstd, float* scale, float* shift, float* rmean, float* rvar, float* sum, float* sumsq,
                       cudaStream_t st) {
    const int C = p->g.c_out;
    SiteTimer tm(p, SITE_FINALIZE, st);
    launch_k(bn_finalize_kernel, dim3((C + 7) / 8), dim3(256), 0, st, 1, partials, nparts, C, (double)p->g.m, p->desc.eps, p->desc.momentum,
                                                              gamma, beta, mean, invstd, scale, shift, rmean, rvar, sum, sumsq);
    return launch_ok("bn_finalize");
}

// res != NULL (training forward with SiLU only): a = SiLU(...) + res, res with row pitch ld_res elements.
// fin != NULL (training forward with SiLU only): scale and shift are derived inside the kernel from the plan's forward accumulators.
template <typename YT, typename AT, bool FAST, bool ACT = true>
nb_status run_apply(nb_cbs_plan_s* p, const void* y, void* a, const float* scale, const float* shift, cudaStream_t st, long long ld_a = 0,
                    const void* res = nullptr, long long ld_res = 0, const FwdFin* fin = nullptr) {
    const EwCfg& e = p->ew;
    const int C = p->g.c_out;
    SiteTimer tm(p, SITE_APPLY, st);
    const ChanAcc none{nullptr, nullptr, 1};
    const FwdFin nofin{};
    auto go = [&](auto kernel, const ChanAcc& ca, const FwdFin& f, size_t smem) {
        launch_k(kernel, dim3(e.blocks_apply), dim3(e.tpb), smem, st, 1, static_cast<const YT*>(y), static_cast<AT*>(a), e.total_vecs, C, scale, shift,
                 ld_a ? ld_a : (long long)C, static_cast<const AT*>(res), ld_res ? ld_res : (long long)C, ca, f);
    };
    if constexpr (ACT) {
        if (fin) {
            const ChanAcc ca{p->acc, p->status + ST_READERS_FWD, p->acc_copies_f};
            const size_t smem = (size_t)2 * C * sizeof(float);
            const bool one = (long long)e.blocks_apply * e.tpb >= e.total_vecs;
            if (res) one ? go(bn_silu_apply_kernel<YT, AT, FAST, true, true, true, true, true>, ca, *fin, smem) : go(bn_silu_apply_kernel<YT, AT, FAST, true, true, true, true>, ca, *fin, smem);
            else if (ld_a) one ? go(bn_silu_apply_kernel<YT, AT, FAST, true, true, false, true, true>, ca, *fin, smem) : go(bn_silu_apply_kernel<YT, AT, FAST, true, true, false, true>, ca, *fin, smem);
            else one ? go(bn_silu_apply_kernel<YT, AT, FAST, true, false, false, true, true>, ca, *fin, smem) : go(bn_silu_apply_kernel<YT, AT, FAST, true, false, false, true>, ca, *fin, smem);
            return launch_ok("bn_silu_apply (statistics from the accumulators)");
        }
        if (res) {
            go(bn_silu_apply_kernel<YT, AT, FAST, true, true, true>, none, nofin, 0);
            return launch_ok("bn_silu_apply (+ residual)");
        }
    }
    if (ld_a) go(bn_silu_apply_kernel<YT, AT, FAST, ACT, true>, none, nofin, 0);
    else go(bn_silu_apply_kernel<YT, AT, FAST, ACT, false>, none, nofin, 0);
    return launch_ok("bn_silu_apply");
}

template <typename YT, typename AT, bool FAST>
nb_status run_bwd_elementwise(nb_cbs_plan_s* p, const void* g, const void* y, const float* mean, const float* invstd,
                              const float* gamma, const float* beta, float* dgamma, float* dbeta, void* dy, float* partials,
                              float* coef, cudaStream_t st, const void* w = nullptr, void* wt = nullptr, const WtParams* wtp = nullptr) {
    const EwCfg& e = p->ew;
    const int C = p->g.c_out;
    const bool fuse = p->fuse_finalize;
    WtParams none;
    if (!wtp) memset(&none, 0, sizeof none);
    const BwdFin bf{1.0 / (double)p->g.m, mean, invstd, gamma, beta, dgamma, dbeta};
    if constexpr (sizeof(AT) == 2) if (fuse && e.slabs) {  // both passes in one launch
        SiteTimer tm(p, SITE_BWD_DY, st);
        const int rows_grid = e.slabs * e.slab_ctas, tiles = wtp && wt ? wt_num_tiles(*wtp) : 0;
        const int wt_ctas = (std::min(tiles, 4 * p->sm_count) + e.slab_ctas - 1) / e.slab_ctas * e.slab_ctas;
        auto go = [&](auto kernel) {
            launch_k(kernel, dim3(rows_grid + wt_ctas), dim3(e.slab_threads), bwd_small_smem(C / e.slabs, e.slab_units, e.slab_threads, e.vec), st, e.slab_ctas, static_cast<const AT*>(g),
                     static_cast<const YT*>(y), static_cast<AT*>(dy), p->g.m, C, bf, static_cast<const __nv_bfloat16*>(w), static_cast<__nv_bfloat16*>(wt), wtp ? *wtp : none,
                     p->ld_g ? p->ld_g : (long long)C, static_cast<AT*>(p->bwd_gres), p->ld_gres ? p->ld_gres : (long long)C, p->gres_add ? 1 : 0,
                     e.slabs, e.slab_units, e.slab_ctas, e.blocks_reduce);
        };
        if (p->bwd_gres) p->ld_g ? go(bn_silu_bwd_small_kernel<YT, AT, FAST, true, true>) : go(bn_silu_bwd_small_kernel<YT, AT, FAST, false, true>);
        else p->ld_g ? go(bn_silu_bwd_small_kernel<YT, AT, FAST, true, false>) : go(bn_silu_bwd_small_kernel<YT, AT, FAST, false, false>);
        return launch_ok("bn_silu_bwd_small");
    }
    const ChanAcc ca{fuse ? p->acc + (size_t)p->acc_copies_f * 2 * C : nullptr, p->status + ST_READERS_BWD, p->acc_copies_b};
    {
        // sums of dz and dz*y per channel (into the accumulators, or as per-block partial sums); the blocks also rearrange the dgrad filter
        SiteTimer tm(p, SITE_BWD_REDUCE, st);
        BwdFused fb;
        memset(&fb, 0, sizeof fb);
        fb.acc = ca;
        if (fuse) {
            fb.w = static_cast<const __nv_bfloat16*>(w); fb.wt = wtp ? static_cast<__nv_bfloat16*>(wt) : nullptr;
        }
        // A small activation needs few blocks, a large filter many: every block takes two filter tiles, blocks without
        // rows of their own take nothing else (288 -> 288 3x3 on one 20 x 20 image has 405 tiles and 8 blocks of rows:
        // 61 us when those 8 rearranged the filter alone).  As many as three an SM, also where two blocks of rows fit one: with at most
        // two, 512 -> 512 3x3 on 16 x 20 x 20 takes 48.6 instead of 46.8 us (backward data call), on 4 x 20 x 20 29.7 instead of 28.5.
        int blocks = e.blocks_reduce;
        if (fb.wt) blocks = std::max(blocks, std::min(e.wave_reduce, (wt_num_tiles(*wtp) + 1) / 2));
        // All vectors of a thread at once where those are at most eight and the blocks of rows, at most two an SM, are resident together.
        // Measured (backward data call, us; blocks in brackets), ring / all at once: 288 -> 576 1x1 on 16 x 20 x 20 pixels (267)
        // 23.4 / 21.1, 576 -> 384 1x1 there (160) 23.0 / 22.0, 96 -> 96 1x1 on 21 x 40 x 40 (200) 20.5 / 18.8, on 222 x 224 (296)
        // 23.4 / 22.5, 64 -> 256 1x1 on 4 x 56 x 56 (196) 18.1 / 16.5, 288 -> 288 3x3 on 16 x 20 x 20 (115) 29.8 / 29.0.  With one register
        // too many for the second block on an SM the first five took 24.3, 23.8, 20.3, 23.7 and 18.5.  The form for one block an SM not
        // where filter tiles make more than two turns of them (512 -> 512 3x3 on 4 x 20 x 20, 50 + 394 blocks: 32.8 instead of 28.3).
        const bool deep = e.blocks_reduce <= e.wave_deep && (long long)e.blocks_reduce * e.tpb * 8 >= e.total_vecs;
        const bool deep1 = deep && e.blocks_reduce <= p->sm_count && blocks <= 2 * p->sm_count;
        const size_t red_smem = std::max((size_t)2 * e.tpb * e.vec * sizeof(float), deep ? (size_t)0 : (size_t)EW_RING * 2 * e.tpb * 16);
        auto go = [&](auto kernel, long long ld) {
            launch_k(kernel, dim3(blocks), dim3(e.tpb), red_smem, st, 1, static_cast<const AT*>(g), static_cast<const YT*>(y), e.total_vecs, C, mean, invstd,
                     gamma, beta, partials, fb, wtp ? *wtp : none, ld, e.blocks_reduce);
        };
        if (p->ld_g) deep1 ? go(bn_silu_bwd_reduce_kernel<YT, AT, FAST, true, 1>, p->ld_g) : deep ? go(bn_silu_bwd_reduce_kernel<YT, AT, FAST, true, 2>, p->ld_g) : go(bn_silu_bwd_reduce_kernel<YT, AT, FAST, true>, p->ld_g);
        else deep1 ? go(bn_silu_bwd_reduce_kernel<YT, AT, FAST, false, 1>, (long long)C) : deep ? go(bn_silu_bwd_reduce_kernel<YT, AT, FAST, false, 2>, (long long)C) : go(bn_silu_bwd_reduce_kernel<YT, AT, FAST, false>, (long long)C);
        NB_LAUNCH_OK("bn_silu_bwd_reduce");
    }
    if (!fuse) {
        SiteTimer tm(p, SITE_BWD_FINALIZE, st);
        const int fin_blocks = (C + 7) / 8;
        int wt_blocks = 0;
        if (wtp) {
            const size_t total = (size_t)wtp->c_in * wtp->k * wtp->k * wtp->c_out;
            wt_blocks = (int)std::min<size_t>((total + 255) / 256, (size_t)p->sm_count * 8);
        }
        launch_k(bn_bwd_finalize_kernel, dim3(fin_blocks + wt_blocks), dim3(256), 0, st, 1, partials, e.blocks_reduce, C, (double)p->g.m, mean, invstd, gamma, beta,
                 dgamma, dbeta, coef, fin_blocks, static_cast<const __nv_bfloat16*>(w), static_cast<__nv_bfloat16*>(wt), wtp ? *wtp : none);
        NB_LAUNCH_OK("bn_bwd_finalize");
    }
    if (p->exact_apart) {
        SiteTimer tm(p, SITE_BWD_FINALIZE, st);
        launch_k(bn_exact_bwd_finalize_kernel, dim3((unsigned)((2 * C + 127) / 128)), dim3(128), 0, st, 1, ca, C, bf, coef);
        NB_LAUNCH_OK("bn_exact_bwd_finalize");
    }
    SiteTimer tm(p, SITE_BWD_DY, st);
    auto go_dy = [&](auto kernel, size_t smem) {
        launch_k(kernel, dim3(e.blocks_dy), dim3(e.tpb), smem, st, 1, static_cast<const AT*>(g), static_cast<const YT*>(y), static_cast<AT*>(dy), e.total_vecs, C, coef,
                 p->ld_g ? p->ld_g : (long long)C, ca, bf, static_cast<AT*>(p->bwd_gres), p->ld_gres ? p->ld_gres : (long long)C, p->gres_add ? 1 : 0);
    };
    const size_t coef_smem = (size_t)4 * C * sizeof(float);
    const bool one = (long long)e.blocks_dy * e.tpb >= e.total_vecs;
    if (fuse && p->bwd_gres) {  // (the setter admits this only on plans that take this path)
        if (p->ld_g) one ? go_dy(bn_silu_bwd_dy_kernel<YT, AT, FAST, true, true, true, true>, coef_smem) : go_dy(bn_silu_bwd_dy_kernel<YT, AT, FAST, true, true, true>, coef_smem);
        else one ? go_dy(bn_silu_bwd_dy_kernel<YT, AT, FAST, false, true, true, true>, coef_smem) : go_dy(bn_silu_bwd_dy_kernel<YT, AT, FAST, false, true, true>, coef_smem);
    } else if (fuse && !p->exact_apart) {
        if (p->ld_g) one ? go_dy(bn_silu_bwd_dy_kernel<YT, AT, FAST, true, true, false, true>, coef_smem) : go_dy(bn_silu_bwd_dy_kernel<YT, AT, FAST, true, true>, coef_smem);
        else one ? go_dy(bn_silu_bwd_dy_kernel<YT, AT, FAST, false, true, false, true>, coef_smem) : go_dy(bn_silu_bwd_dy_kernel<YT, AT, FAST, false, true>, coef_smem);
    } else {
        if (p->ld_g) go_dy(bn_silu_bwd_dy_kernel<YT, AT, FAST, true, false>, 0);
        else go_dy(bn_silu_bwd_dy_kernel<YT, AT, FAST, false, false>, 0);
    }
    return launch_ok("bn_silu_bwd_dy");
}

// ---------------------------------------------------------------- first layer
// f(integral_constant) with the plan's output channel count (one of stem_cout_ok's)
template <class F> nb_status with_stem_cout(int c_out, F f) {
    switch (c_out) {
        case 16: return f(std::integral_constant<int, 16>{});
        case 32: return f(std::integral_constant<int, 32>{});
        case 48: return f(std::integral_constant<int, 48>{});
        case 64: return f(std::integral_constant<int, 64>{});
        default: return f(std::integral_constant<int, 80>{});
    }
}
template <typename OutT, typename AT, bool EPI>
nb_status run_stem_fprop(nb_cbs_plan_s* p, const void* x, const void* w, void* y, const StemEpi& ep, float* part, double* acc, cudaStream_t st) {
    return with_stem_cout(p->g.c_out, [&](auto co) {
        auto go = [&](auto kernel) {
            launch_k(kernel, dim3(p->stem_fprop_blocks), dim3(128), 0, st, 1, static_cast<const AT*>(x), static_cast<const AT*>(w), static_cast<OutT*>(y), p->g, ep, part, acc,
                     acc ? p->acc_copies_f : 1);
        };
        if (p->stem_wide) go(stem_fprop_mma_kernel<decltype(co)::value, OutT, EPI, AT, STEM_TQ_WIDE>);
        else go(stem_fprop_mma_kernel<decltype(co)::value, OutT, EPI, AT, STEM_TQ>);
        return launch_ok("stem_fprop");
    });
}
template <typename AT> nb_status run_stem_dgrad(nb_cbs_plan_s* p, const void* dy, const void* w, void* dx, cudaStream_t st) {
    return with_stem_cout(p->g.c_out, [&](auto co) {
        launch_k(stem_dgrad_mma_kernel<decltype(co)::value, AT>, dim3(p->stem_dgrad_blocks), dim3(128), 0, st, 1, static_cast<const AT*>(dy), static_cast<const AT*>(w),
                 static_cast<AT*>(dx), p->g, p->stem_dgrad_rows);
        return launch_ok("stem_dgrad");
    });
}
template <typename AT> nb_status run_stem_wgrad(nb_cbs_plan_s* p, const void* x, const void* dy, float* partial, bool overlap, cudaStream_t st) {
    return with_stem_cout(p->g.c_out, [&](auto co) {
        constexpr int CO = decltype(co)::value;
        auto go = [&](auto kernel, size_t smem) {
            launch_k(kernel, dim3(p->stem_wgrad_blocks), dim3(128), smem, st, 1, static_cast<const AT*>(x), static_cast<const AT*>(dy), partial, p->g, overlap ? 1 : 0);
        };
        if (p->stem_wide) go(stem_wgrad_mma_kernel<CO, AT, STEM_TQ_WGRAD>, stem_wgrad_smem_bytes<CO, AT, STEM_TQ_WGRAD>());
        else go(stem_wgrad_mma_kernel<CO, AT, STEM_TQ>, stem_wgrad_smem_bytes<CO, AT, STEM_TQ>());
        return launch_ok("stem_wgrad");
    });
}
// More dynamic shared memory than the 48 KB a kernel gets without asking (the weight gradient's ring), with the device current.
template <typename AT> cudaError_t stem_allow_smem(int c_out) {
    cudaError_t e = cudaSuccess;
    with_stem_cout(c_out, [&](auto co) {
        constexpr int CO = decltype(co)::value;
        e = cudaFuncSetAttribute(stem_wgrad_mma_kernel<CO, AT, STEM_TQ_WGRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)stem_wgrad_smem_bytes<CO, AT, STEM_TQ_WGRAD>());
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(stem_wgrad_mma_kernel<CO, AT, STEM_TQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)stem_wgrad_smem_bytes<CO, AT, STEM_TQ>());
        return NB_OK;
    });
    return e;
}

// ---------------------------------------------------------------- CUDA-core convolutions
// Tile and slices.  64 x 64; 32 x 64 where even eight-stage slices of such tiles would leave an SM fewer than two blocks;
// 64 x 32 for at most 32 columns and for the 16-bit fallback.  One block
// alone on an SM waits for its ring (0.5 us per 16-k stage, half of it latency), so where an SM has two tiles or fewer the k
// range is cut into slices of at least eight stages until it has up to six blocks (one more than fits a wave is worse than one fewer), and into slices
// of at most 1024 products where the slices fit 128 MB: such a slice needs no fp64 flush, whose shared memory leaves three
// blocks per SM, and evens out the last wave.  Slices cost a reduce launch and a trip through L2 (3 to 4 us), hence not
// below 16 stages.  Measured (step): 64 -> 64 3x3 at 2 x 40 x 40, one slice 75 us, five slices 59 us; 288 -> 288 3x3 at
// 4 x 20 x 20, 348 -> 262 us against at most four blocks per SM; 272 -> 304 stride 2 on 7 x 44 x 84, 1265 -> 982 us.
SgCfg sg_configure(const Geom& g, int kind, bool f32, int sm_count) {
    SgCfg c{};
    const int cols = kind == 0 ? g.c_out : kind == 1 ? g.c_in : g.kdim;
    const int taps = (g.k + g.stride - 1) / g.stride;  // data gradient: the most taps per axis that reach an input pixel
    const long long KK = kind == 2 ? g.m : kind == 0 ? (long long)g.kdim : (long long)taps * taps * g.c_out;
    c.bn = (!f32 || cols <= 32) ? 32 : 64;
    auto row_tiles = [&](int bm) {
        if (kind != 1) return ((kind == 0 ? g.m : (long long)g.c_out) + bm - 1) / bm;
        long long t = 0;
        for (int cls = 0; cls < g.stride * g.stride; ++cls) t += (sg_class(g, cls).rows + bm - 1) / bm;
        return t;
    };
    const long long col_tiles = (cols + c.bn - 1) / c.bn;
    const size_t out = kind == 0 ? (size_t)g.m * g.c_out : kind == 1 ? (size_t)g.n * g.h * g.w * g.c_in : (size_t)g.c_out * g.kdim;
    const long long most = std::max<long long>(1, KK / (8 * SG_BK));
    c.bm = 64;
    if (c.bn == 64 && row_tiles(64) * col_tiles * most < 2 * sm_count) c.bm = 32;
    const long long tiles = row_tiles(c.bm) * col_tiles;
    long long splits = 1;
    if (KK >= 16 * SG_BK) {
        if (tiles <= 2 * sm_count) splits = std::max<long long>(1, std::min<long long>(6LL * sm_count / tiles, most));
        const long long flush_free = (KK + 1023) / 1024;
        if (splits < flush_free && (size_t)flush_free * out * 4 <= (size_t)128 << 20) splits = flush_free;
        splits = std::min<long long>(splits, 65535);  // (slices are gridDim.z: 8 -> 8 1x1 has 65536 of 1024 pixels at 67.1 million)
    }
    c.kchunk = ((KK + splits - 1) / splits + SG_BK - 1) / SG_BK * SG_BK;
    c.splits = (int)((KK + c.kchunk - 1) / c.kchunk);
    c.grid = dim3((unsigned)row_tiles(c.bm), (unsigned)col_tiles, (unsigned)c.splits);
    c.partial_bytes = c.splits > 1 ? (size_t)c.splits * out * 4 : 0;
    return c;
}

template <int KIND, typename TIN, typename TO, int BM, int BN, int V>
nb_status launch_sg_tile(const nb_cbs_plan_s* p, const SgCfg& c, const void* a, const void* b, void* out, const SgArgs& args, cudaStream_t st) {
    using T = SgTile<KIND, BM, BN>;
    const size_t flush = (size_t)T::TM * 4 * SG_THREADS * sizeof(double);
    // Blocks become resident while the previous kernel still runs, wherever it leaves room: with room for five on an SM, 100
    // blocks of a small layer pile up on a few of them (measured: 28 us alone, 50 us behind the passes of the block).
    // Enough shared memory is asked for that an SM takes no more than its share.
    const long long blocks = (long long)c.grid.x * c.grid.y * c.grid.z;
    const long long share = (blocks + p->sm_count - 1) / p->sm_count;
    const size_t smem = std::max(T::stage_bytes(sizeof(TIN)) + (c.kchunk > 1024 ? flush : 0), share <= 4 ? (size_t)(233472 / (share + 1)) : (size_t)0);
    static std::atomic<unsigned long long> attr_set{0};  // one bit per device ordinal
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(attr_set.load(std::memory_order_acquire) & bit)) {
        NB_CUDA_CHECK(cudaFuncSetAttribute(simt_gemm_kernel<KIND, TIN, TO, BM, BN, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, 120 * 1024));
        attr_set.fetch_or(bit, std::memory_order_release);
    }
    launch_k(simt_gemm_kernel<KIND, TIN, TO, BM, BN, V>, c.grid, dim3(SG_THREADS), smem, st, 1, static_cast<const TIN*>(a), static_cast<const TIN*>(b), static_cast<TO*>(out), args);
    return launch_ok("simt convolution");
}
template <int KIND, typename TIN, typename TO>
nb_status launch_sg(const nb_cbs_plan_s* p, const void* a, const void* b, void* out, const SgArgs& args, cudaStream_t st) {
    const SgCfg& c = p->sg[KIND];
    const bool vec = p->g.c_in % 4 == 0;
    if constexpr (std::is_same<TIN, float>::value) {
        if (c.bn == 64 && c.bm == 64) return vec ? launch_sg_tile<KIND, TIN, TO, 64, 64, 4>(p, c, a, b, out, args, st) : launch_sg_tile<KIND, TIN, TO, 64, 64, 1>(p, c, a, b, out, args, st);
        if (c.bn == 64) return vec ? launch_sg_tile<KIND, TIN, TO, 32, 64, 4>(p, c, a, b, out, args, st) : launch_sg_tile<KIND, TIN, TO, 32, 64, 1>(p, c, a, b, out, args, st);
    }
    return vec ? launch_sg_tile<KIND, TIN, TO, 64, 32, 4>(p, c, a, b, out, args, st) : launch_sg_tile<KIND, TIN, TO, 64, 32, 1>(p, c, a, b, out, args, st);
}

// The pass that adds the slices of a split forward convolution: threads and blocks.
int fwd_reduce_threads(const Geom& g) {
    const int cgs = g.c_out / 4;
    return cgs >= 256 ? cgs : 256 / cgs * cgs;
}
int fwd_reduce_blocks(const Geom& g, int sm_count) {
    const int tpb = fwd_reduce_threads(g);
    return (int)std::min<long long>((g.m * (g.c_out / 4) + tpb - 1) / tpb, (long long)sm_count * 4);
}
// Blocks that add to the channel sums of a CUDA-core forward convolution: one per row tile, or those of that pass.
int simt_fwd_parts(const Geom& g, const SgCfg& c, int sm_count) { return c.splits == 1 ? (int)c.grid.x : fwd_reduce_blocks(g, sm_count); }

// `sums`: with a default plan the channel sums of y go to the plan's accumulators (false: y only, or separate statistics).
template <typename TIN, typename TOUT>
nb_status run_simt_fprop(nb_cbs_plan_s* p, const void* x, const void* w, void* y, void* partial, bool sums, cudaStream_t st) {
    const SgCfg& c = p->sg[0];
    const ChanAcc ca{sums ? p->acc : nullptr, nullptr, sums ? p->acc_copies_f : 1};
    const SgArgs args{p->g, c.kchunk, sums && c.splits == 1, ca, 0};
    {
        SiteTimer tm(p, SITE_FPROP, st);
        if (c.splits == 1) return launch_sg<0, TIN, TOUT>(p, x, w, y, args, st);
        NB_TRY((launch_sg<0, TIN, float>(p, x, w, partial, args, st)));
    }
    SiteTimer tm(p, SITE_SPLITK_REDUCE, st);
    const int tpb = fwd_reduce_threads(p->g);
    launch_k(splitk_fwd_reduce_kernel<TOUT>, dim3((unsigned)fwd_reduce_blocks(p->g, p->sm_count)), dim3(tpb), (size_t)tpb * 16, st, 1, static_cast<const float*>(partial),
             c.splits, p->g.m * (p->g.c_out / 4), p->g.c_out, static_cast<TOUT*>(y), ca);
    return launch_ok("splitk_fwd_reduce");
}

unsigned splitk_reduce_blocks(size_t elems, int sm_count) { return (unsigned)std::min<size_t>((elems / 4 + 255) / 256 + 1, (size_t)sm_count * 8); }
template <typename TIN> nb_status simt_dgrad_conv(nb_cbs_plan_s* p, const void* dy, const void* w, void* dx, void* partial, cudaStream_t st) {
    const SgCfg& c = p->sg[1];
    const SgArgs args{p->g, c.kchunk, false, ChanAcc{nullptr, nullptr, 1}, 0};
    SiteTimer tm(p, SITE_DGRAD, st);
    if (c.splits == 1) return launch_sg<1, TIN, TIN>(p, dy, w, dx, args, st);
    return launch_sg<1, TIN, float>(p, dy, w, partial, args, st);
}
template <typename TIN>
nb_status run_simt_dgrad(nb_cbs_plan_s* p, const void* dy, const void* w, void* dx, void* partial, cudaStream_t st) {
    NB_TRY(simt_dgrad_conv<TIN>(p, dy, w, dx, partial, st));
    const SgCfg& c = p->sg[1];
    if (c.splits == 1) return NB_OK;
    const size_t elems = (size_t)p->g.n * p->g.h * p->g.w * p->g.c_in;
    SiteTimer tm(p, SITE_SPLITK_REDUCE, st);
    launch_k(splitk_reduce_kernel<TIN, true>, dim3(splitk_reduce_blocks(elems, p->sm_count)), dim3(256), 0, st, 1, static_cast<const float*>(partial), c.splits, elems, static_cast<TIN*>(dx));
    return launch_ok("splitk_reduce");
}

template <typename TIN>
nb_status simt_wgrad_conv(nb_cbs_plan_s* p, const void* x, const void* dy, float* dw, float* partial, bool overlap, cudaStream_t st) {
    const SgCfg& c = p->sg[2];
    const SgArgs args{p->g, c.kchunk, false, ChanAcc{nullptr, nullptr, 1}, overlap ? 1 : 0};
    SiteTimer tm(p, SITE_WGRAD, st);
    return launch_sg<2, TIN, float>(p, dy, x, c.splits == 1 ? dw : partial, args, st);
}
template <typename TIN>
nb_status run_simt_wgrad(nb_cbs_plan_s* p, const void* x, const void* dy, float* dw, float* partial, bool overlap, cudaStream_t st) {
    NB_TRY(simt_wgrad_conv<TIN>(p, x, dy, dw, partial, overlap, st));
    const SgCfg& c = p->sg[2];
    if (c.splits == 1) return NB_OK;
    const size_t elems = (size_t)p->g.c_out * p->g.kdim;
    SiteTimer tm(p, SITE_SPLITK_REDUCE, st);
    if (c.splits >= 96) launch_k(splitk_reduce_tall_kernel, dim3((unsigned)((elems + 31) / 32)), dim3(1024), 0, st, 1, partial, c.splits, elems, dw);
    else launch_k(splitk_reduce_kernel<float>, dim3(splitk_reduce_blocks(elems, p->sm_count)), dim3(256), 0, st, 1, partial, c.splits, elems, dw);
    return launch_ok("splitk_reduce");
}

// Both gradients of a layer on the CUDA cores: the convolutions beside each other (the weight gradient is the very next launch
// behind the data gradient, see the end of common.cuh), then the slices of both in one launch.  With the data gradient's slices
// added in between, its convolution and the weight gradient followed one another, two launches more in a row.
template <typename TIN>
nb_status run_simt_grads(nb_cbs_plan_s* p, const void* x, const void* dy, const void* w, void* dx, float* dw, void* dgpart, float* wgpart, cudaStream_t st) {
    const SgCfg &d = p->sg[1], &c = p->sg[2];
    NB_TRY(simt_dgrad_conv<TIN>(p, dy, w, dx, dgpart, st));
    NB_TRY(simt_wgrad_conv<TIN>(p, x, dy, dw, wgpart, pdl_enabled(), st));
    const size_t elems1 = (size_t)p->g.n * p->g.h * p->g.w * p->g.c_in, elems2 = (size_t)p->g.c_out * p->g.kdim;
    if (d.splits > 1 && c.splits > 1 && c.splits < 96) {
        const unsigned b1 = splitk_reduce_blocks(elems1, p->sm_count), b2 = splitk_reduce_blocks(elems2, p->sm_count);
        SiteTimer tm(p, SITE_SPLITK_REDUCE, st);
        launch_k(splitk_reduce_both_kernel<TIN>, dim3(b1 + b2), dim3(256), 0, st, 1, static_cast<const float*>(dgpart), d.splits, elems1, static_cast<TIN*>(dx), (int)b1,
                 static_cast<const float*>(wgpart), c.splits, elems2, dw);
        return launch_ok("splitk_reduce_both");
    }
    if (d.splits > 1) {
        SiteTimer tm(p, SITE_SPLITK_REDUCE, st);
        launch_k(splitk_reduce_kernel<TIN>, dim3(splitk_reduce_blocks(elems1, p->sm_count)), dim3(256), 0, st, 1, static_cast<const float*>(dgpart), d.splits, elems1, static_cast<TIN*>(dx));
        NB_LAUNCH_OK("splitk_reduce");
    }
    if (c.splits == 1) return NB_OK;
    SiteTimer tm(p, SITE_SPLITK_REDUCE, st);
    if (c.splits >= 96) launch_k(splitk_reduce_tall_kernel, dim3((unsigned)((elems2 + 31) / 32)), dim3(1024), 0, st, 1, wgpart, c.splits, elems2, dw);
    else launch_k(splitk_reduce_kernel<float>, dim3(splitk_reduce_blocks(elems2, p->sm_count)), dim3(256), 0, st, 1, wgpart, c.splits, elems2, dw);
    return launch_ok("splitk_reduce");
}

}  // namespace

// ====================================================================================== exported functions
extern "C" {

uint32_t nb_abi_version(void) { return NB_CBS_ABI_VERSION; }

const char* nb_last_error(void) { return g_err.c_str(); }

nb_status nb_cbs_plan_create(const nb_cbs_desc* d, int device, nb_cbs_plan* out) {
    g_err.clear();
    if (!out) return fail(NB_ERR_INVALID_ARG, "out_plan is NULL");
    *out = nullptr;
    if (!d) return fail(NB_ERR_INVALID_ARG, "desc is NULL");
    if (d->struct_size != sizeof(nb_cbs_desc))
        return fail(NB_ERR_INVALID_ARG, "desc.struct_size is %u, this library expects %zu", d->struct_size, sizeof(nb_cbs_desc));
    if (d->n <= 0 || d->h <= 0 || d->w <= 0 || d->c_in <= 0 || d->c_out <= 0)
        return fail(NB_ERR_INVALID_ARG, "extents must be positive (n=%d h=%d w=%d c_in=%d c_out=%d)", d->n, d->h, d->w, d->c_in, d->c_out);
    if (d->ksize != 1 && d->ksize != 3) return fail(NB_ERR_INVALID_ARG, "ksize must be 1 or 3, got %d", d->ksize);
    if (d->stride != 1 && d->stride != 2) return fail(NB_ERR_INVALID_ARG, "stride must be 1 or 2, got %d", d->stride);
    if (d->mode != NB_MODE_BF16_TC && d->mode != NB_MODE_F32_REF && d->mode != NB_MODE_F16_TC) return fail(NB_ERR_INVALID_ARG, "unknown mode %d", d->mode);
    if (!(d->eps > 0.f)) return fail(NB_ERR_INVALID_ARG, "eps must be positive");
    if (!(d->momentum >= 0.f && d->momentum <= 1.f)) return fail(NB_ERR_INVALID_ARG, "momentum must be in [0,1]");
    const int vec = d->mode == NB_MODE_F32_REF ? 4 : 8;
    if (d->c_out % vec) return fail(NB_ERR_UNSUPPORTED, "c_out=%d must be a multiple of %d in this mode", d->c_out, vec);
    static_assert(288 * 8 <= SG_REDUCE_MAX * 4, "a block of splitk_fwd_reduce_kernel spans the channels of a row");
    if (d->c_out / vec > 288) return fail(NB_ERR_UNSUPPORTED, "c_out=%d is too large (at most %d channels in this mode)", d->c_out, 288 * vec);

    Geom g;
    g.n = d->n; g.h = d->h; g.w = d->w; g.c_in = d->c_in; g.c_out = d->c_out; g.k = d->ksize; g.stride = d->stride;
    g.pad = d->ksize / 2;
    g.ho = (g.h + 2 * g.pad - g.k) / g.stride + 1;
    g.wo = (g.w + 2 * g.pad - g.k) / g.stride + 1;
    g.m = (long long)g.n * g.ho * g.wo;
    g.kdim = g.k * g.k * g.c_in;
    if (g.m < 2) return fail(NB_ERR_INVALID_ARG, "batch statistics need at least 2 rows (N*Ho*Wo=%lld)", g.m);
    if ((double)g.m * g.c_out >= 9.0e18 || (long long)g.n * g.h * g.w * g.c_in < 0)
        return fail(NB_ERR_UNSUPPORTED, "tensor too large");

    int count = 0;
    NB_CUDA_CHECK(cudaGetDeviceCount(&count));
    if (device < 0 || device >= count) return fail(NB_ERR_INVALID_ARG, "device %d out of range (%d devices)", device, count);
    int major = 0, minor = 0, sms = 0;  // (attributes: cudaGetDeviceProperties takes 2.5 ms)
    NB_CUDA_CHECK(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device));
    NB_CUDA_CHECK(cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, device));
    NB_CUDA_CHECK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device));
    if (major != 10) return fail(NB_ERR_ARCH, "device %d is sm_%d%d; this library is built for sm_100a only", device, major, minor);

    nb_cbs_plan_s* p = new (std::nothrow) nb_cbs_plan_s();
    if (!p) return fail(NB_ERR_INTERNAL, "out of host memory");
    p->desc = *d;
    p->g = g;
    p->device = device;
    p->sm_count = sms;
    p->fuse_finalize = !(d->flags & NB_CBS_FLAG_SEPARATE_FINALIZE);

    EwCfg& e = p->ew;
    e.vec = vec;
    e.cgs = g.c_out / vec;
    const int R = e.cgs >= 256 ? 1 : 256 / e.cgs;
    e.tpb = e.cgs * R;
    e.total_vecs = g.m * e.cgs;
    const long long max_blocks = (e.total_vecs + e.tpb - 1) / e.tpb;
    // Grids are one wave of resident blocks (occupancy queried per kernel).  A tensor smaller than that gets as many blocks
    // as it has work for: eight vectors per thread in the backward reduction (a block also adds 2*C sums to the accumulators;
    // the grouping of the additions is part of the results' last bits, and stays), one in the maps, whose threads would
    // otherwise chain memory latencies: 16 -> 32 on 2 x 32 x 32 pixels, 36.3 -> 34.0 us for the step's kernels against four.
    {
        auto resident = [&](const void* fn, size_t dyn_smem) {
            int occ = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, e.tpb, dyn_smem) != cudaSuccess || occ < 1) {
                cudaGetLastError();
                occ = 1;
            }
            return p->sm_count * occ;
        };
        auto wave = [&](const void* fn, size_t dyn_smem, int min_vecs) {
            return (int)std::max<long long>(1, std::min<long long>((max_blocks + min_vecs - 1) / min_vecs, resident(fn, dyn_smem)));
        };
        const size_t red_smem = (size_t)e.tpb * vec * sizeof(float);
        auto reduce = [&](auto ring, auto deep, auto deep_pitched) {
            const size_t ring_smem = std::max(2 * red_smem, (size_t)EW_RING * 2 * e.tpb * 16);
            e.blocks_reduce = wave((const void*)ring, ring_smem, 8);
            e.wave_reduce = resident((const void*)ring, ring_smem);
            e.wave_deep = std::min({2 * p->sm_count, resident((const void*)deep, 2 * red_smem), resident((const void*)deep_pitched, 2 * red_smem)});
        };
        // the passes that derive their coefficients from the accumulators keep them in dynamic shared memory
        const size_t apply_smem = p->fuse_finalize ? (size_t)2 * g.c_out * sizeof(float) : 0, dy_smem = p->fuse_finalize ? (size_t)4 * g.c_out * sizeof(float) : 0;
        if (d->mode == NB_MODE_F32_REF) {
            e.blocks_stats = wave((const void*)bn_stats_partial_kernel<float>, red_smem, 4);
            reduce(bn_silu_bwd_reduce_kernel<float, float, false>, bn_silu_bwd_reduce_kernel<float, float, false, false, 2>, bn_silu_bwd_reduce_kernel<float, float, false, true, 2>);
            e.blocks_apply = wave((const void*)bn_silu_apply_kernel<float, float, false, true, false, false, true>, apply_smem, 1);
            e.blocks_dy = wave((const void*)bn_silu_bwd_dy_kernel<float, float, false, false, true>, dy_smem, 1);
        } else if (d->mode == NB_MODE_F16_TC) {
            e.blocks_stats = wave((const void*)bn_stats_partial_kernel<__half>, red_smem, 4);
            reduce(bn_silu_bwd_reduce_kernel<__half, __half, true>, bn_silu_bwd_reduce_kernel<__half, __half, true, false, 2>, bn_silu_bwd_reduce_kernel<__half, __half, true, true, 2>);
            e.blocks_apply = wave((const void*)bn_silu_apply_kernel<__half, __half, true, true, false, false, true>, apply_smem, 1);
            e.blocks_dy = wave((const void*)bn_silu_bwd_dy_kernel<__half, __half, true, false, true>, dy_smem, 1);
        } else {
            e.blocks_stats = wave((const void*)bn_stats_partial_kernel<__half>, red_smem, 4);
            reduce(bn_silu_bwd_reduce_kernel<__half, __nv_bfloat16, true>, bn_silu_bwd_reduce_kernel<__half, __nv_bfloat16, true, false, 2>, bn_silu_bwd_reduce_kernel<__half, __nv_bfloat16, true, true, 2>);
            e.blocks_apply = wave((const void*)bn_silu_apply_kernel<__half, __nv_bfloat16, true, true, false, false, true>, apply_smem, 1);
            e.blocks_dy = wave((const void*)bn_silu_bwd_dy_kernel<__half, __nv_bfloat16, true, false, true>, dy_smem, 1);
        }
        e.blocks_map = std::max(e.blocks_apply, e.blocks_dy);
        // Both backward passes in one launch (16-bit modes), where a thread of the reduction has at most eight vectors and its
        // blocks fit, by channel slabs, into clusters of eight CTAs (at most 48 KB of shared memory with the filter tile, which
        // needs no opt-in).  A CTA takes as few row blocks as eight CTAs allow, and as narrow a slab as leaves it 96 threads: the
        // work is a few row blocks of 256 threads with eight vectors each, and more SMs share it that way.  Above 24 row blocks the
        // eight vectors of a thread, one after the other, take as long as the launch saved: detector iteration at batch 2,
        // 320 x 320 with at most 0 / 8 / 16 / 24 / 40 row blocks 2282 / 2284 / 2268 / 2237 / 2245 us.  At least 256 / 128 / 96 / 64 /
        // 48 threads, the same iteration: 2117 / 2096 / 2049 / 2049 / 2081 us.  The fp32 mode, whose sigmoid is an exponential and
        // a division, loses 2 us (16 -> 32 on 2 x 32 x 32 pixels 38.1 -> 40.3).
        e.slabs = 0;
        const bool forbidden = getenv("NB_EW_SLABS") && atoi(getenv("NB_EW_SLABS")) == 0;
        if (p->fuse_finalize && !forbidden && d->mode != NB_MODE_F32_REF && e.blocks_reduce <= 24 && (long long)e.blocks_reduce * e.tpb * 8 >= e.total_vecs)
            for (int sl = 1; sl <= e.cgs; ++sl) {
                const int units = (e.blocks_reduce + 7) / 8, threads = e.tpb / sl * units;
                if (e.cgs % sl || units > sl || bwd_small_smem(g.c_out / sl, units, threads, vec) > 40 * 1024) continue;
                if (e.slabs && threads < 96) break;
                e.slabs = sl;
                e.slab_units = units;
                e.slab_threads = threads;
                e.slab_ctas = (e.blocks_reduce + units - 1) / units;
            }
    }

    for (int kind = 0; kind < 3; ++kind) p->sg[kind] = sg_configure(g, kind, d->mode == NB_MODE_F32_REF, p->sm_count);

    int cur = 0;
    NB_CUDA_CHECK(cudaGetDevice(&cur));
    cudaError_t ce = cudaSetDevice(device);
    // one allocation: the status words, then (256-byte aligned) the channel accumulators
    {
        auto copies = [](const char* name, int dflt) {
            const char* v = getenv(name);
            const int k = v ? atoi(v) : dflt;
            return k < 1 ? 1 : k > 16 ? 16 : k;
        };
        const bool exact = d->mode == NB_MODE_F32_REF;
        // (fp32: two sets from 256 adding blocks on: 96 channels on 2 x 40 x 40 81.8 -> 79.7 us, 32 -> 48 1x1 on 16 x 160 x 160
        // 335 -> 309; below, where they only add to what is read, 16 -> 32 on 2 x 32 x 32 37.7 -> 38.2; four are slower everywhere)
        const int sets = copies("NB_ACC_COPIES_FWD", simt_fwd_parts(g, p->sg[0], p->sm_count) < 256 ? 1 : 2);
        p->acc_copies_f = !p->fuse_finalize ? 0 : exact ? EXACT_WORDS * sets : copies("NB_ACC_COPIES_FWD", 2);
        p->acc_copies_b = !p->fuse_finalize ? 0 : exact ? EXACT_WORDS : copies("NB_ACC_COPIES_BWD", 4);
        p->exact_apart = p->fuse_finalize && exact && g.c_out > 160;
    }
    const size_t acc_bytes = (size_t)(p->acc_copies_f + p->acc_copies_b) * 2 * g.c_out * sizeof(double);
    if (ce == cudaSuccess) ce = cudaMalloc(&p->status, kStatusBytes + acc_bytes);
    if (ce == cudaSuccess) ce = cudaMemset(p->status, 0, kStatusBytes + acc_bytes);
    if (ce == cudaSuccess && acc_bytes) p->acc = reinterpret_cast<double*>(reinterpret_cast<char*>(p->status) + kStatusBytes);
    nb_status tcs = NB_OK;
    if (ce == cudaSuccess)
        tcs = tc_plan_init(&p->tc, g, d->mode != NB_MODE_F32_REF && !(d->flags & NB_CBS_FLAG_FORCE_SIMT), p->sm_count, d->mode == NB_MODE_F16_TC);
    cudaSetDevice(cur);
    if (ce != cudaSuccess || tcs != NB_OK) {
        if (p->status) cudaFree(p->status);
        delete p;
        if (tcs != NB_OK) return fail(tcs, "tensor-core plan setup failed: %s", tc_last_error());
        return fail(NB_ERR_CUDA, "status block allocation failed: %s", cudaGetErrorString(ce));
    }

    p->stem = d->mode != NB_MODE_F32_REF && !(d->flags & NB_CBS_FLAG_FORCE_SIMT) && g.c_in == 3 && g.k == 3 && g.stride == 2 &&
              stem_cout_ok(g.c_out) && g.h % 2 == 0 && g.w % 2 == 0 && g.m < (1LL << 31) && (long long)g.n * g.h * g.w * 3 < (1LL << 31);
    p->stem_blocks = (int)std::min<long long>(stem_num_strips(g), (long long)p->sm_count * stem_occ(g.c_out));  // grid of the first-layer kernels: one wave of resident blocks
    p->stem_dgrad_blocks = stem_dgrad_grid(g, p->sm_count * stem_dgrad_occ(g.c_out), &p->stem_dgrad_rows);
    p->stem_wide = g.wo >= STEM_TQ_WIDE / 2;  // (a strip of a narrower row would leave most of its tile slots empty)
    if (const char* e2 = getenv("NB_STEM_WIDE")) p->stem_wide = atoi(e2) != 0;
    p->stem_fprop_blocks = p->stem_wide ? (int)std::min<long long>(stem_num_strips(g, STEM_TQ_WIDE), (long long)p->sm_count * stem_occ(g.c_out)) : p->stem_blocks;
    p->stem_wgrad_blocks = p->stem_wide ? (int)std::min<long long>(stem_num_strips(g, STEM_TQ_WGRAD), (long long)p->sm_count * stem_occ(g.c_out)) : p->stem_blocks;
    if (p->stem) {
        DeviceGuard on_device(p->device);
        if (NB_WITH_AT(p, stem_allow_smem<AT>(g.c_out)) != cudaSuccess) {
            (void)cudaGetLastError();
            p->stem = false;  // the CUDA-core kernels take any shape
        }
    }
    p->nparts = std::max(std::max(std::max(e.blocks_reduce, e.blocks_stats), p->tc.fprop_parts), p->stem ? p->stem_blocks : 0);
    const size_t C = (size_t)g.c_out;
    size_t off = 0;
    p->off_scale = off; off = align_up(off + C * 4, 256);
    p->off_shift = off; off = align_up(off + C * 4, 256);
    p->off_fpart = off; off = align_up(off + (size_t)p->nparts * 2 * C * 4, 256);
    const bool simt_fwd = !p->stem && !p->tc.fprop, simt_dg = !p->stem && !p->tc.dgrad, simt_wg = !p->stem && !p->tc.wgrad;
    p->off_sgpart = off; off = align_up(off + (simt_fwd ? p->sg[0].partial_bytes : 0), 256);
    p->fwd_bytes = off;
    p->off_iy = p->off_fpart;
    p->off_isg = align_up(p->off_iy + (size_t)g.m * C * (is_f32(p) ? 4 : 2), 256);
    p->infer_bytes = infer_fused(p) ? p->off_fpart : align_up(p->off_isg + p->sg[0].partial_bytes, 256);
    off = 0;
    p->off_coef = off; off = align_up(off + 4 * C * 4, 256);
    p->off_bpart = off; off = align_up(off + (size_t)p->nparts * 2 * C * 4, 256);
    p->off_wt = off; off = align_up(off + p->tc.wt_bytes, 256);
    p->off_dgpart = off; off = align_up(off + (simt_dg ? p->sg[1].partial_bytes : 0), 256);  // (not shared with the weight gradient, which may run beside it)
    p->off_wgpart = off;
    {
        const size_t simt = simt_wg ? p->sg[2].partial_bytes : 0;
        size_t stem = p->stem ? (size_t)p->stem_blocks * C * g.kdim * 4 : 0;
        off = align_up(off + std::max(std::max(simt, stem), p->tc.wgrad_partial_bytes), 256);
    }
    p->bwd_bytes = off;
    *out = p;
    return NB_OK;
}

nb_status nb_cbs_plan_destroy(nb_cbs_plan p) {
    g_err.clear();
    if (!p) return NB_OK;
    if (p->status) {
        int cur = 0;
        cudaGetDevice(&cur);
        cudaSetDevice(p->device);
        cudaFree(p->status);
        if (p->ev0) cudaEventDestroy(p->ev0);
        if (p->ev1) cudaEventDestroy(p->ev1);
        drop_copy_streams(p);
        cudaSetDevice(cur);
    }
    delete p;
    return NB_OK;
}

nb_status nb_cbs_out_shape(nb_cbs_plan p, int32_t* ho, int32_t* wo) {
    g_err.clear();
    if (!p || !ho || !wo) return fail(NB_ERR_INVALID_ARG, "NULL argument");
    *ho = p->g.ho;
    *wo = p->g.wo;
    return NB_OK;
}

nb_status nb_cbs_workspace_bytes(nb_cbs_plan p, size_t* fwd, size_t* bwd) {
    g_err.clear();
    if (!p || !fwd || !bwd) return fail(NB_ERR_INVALID_ARG, "NULL argument");
    *fwd = p->fwd_bytes;
    *bwd = p->bwd_bytes;
    return NB_OK;
}

nb_status nb_cbs_plan_set_pitches(nb_cbs_plan p, int64_t ld_x, int64_t ld_a, int64_t ld_g) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    const int vec = is_f32(p) ? 4 : 8;
    auto bad = [&](int64_t ld, int channels) { return ld != 0 && ld != channels && (ld < channels || ld % vec != 0); };  // 0 or the channel count: dense
    if (bad(ld_x, p->g.c_in) || bad(ld_a, p->g.c_out) || bad(ld_g, p->g.c_out))
        return fail(NB_ERR_INVALID_ARG, "a pitch must be 0 (dense) or at least the channel count and a multiple of %d elements", vec);
    if (ld_x != 0 && ld_x != p->g.c_in && (is_f32(p) || p->stem || !p->tc.fprop || !p->tc.wgrad))
        return fail(NB_ERR_UNSUPPORTED, "an input pitch needs the tensor-core forward and weight-gradient kernels (this plan runs them elsewhere)");
    p->tc.ld_x = (ld_x == p->g.c_in) ? 0 : ld_x;
    p->ld_a = (ld_a == p->g.c_out) ? 0 : ld_a;
    p->ld_g = (ld_g == p->g.c_out) ? 0 : ld_g;
    p->pitched = p->tc.ld_x || p->ld_a || p->ld_g;
    // tensor maps cached for the previous layout are stale
    p->tc.fp.a_ptr = nullptr;
    p->tc.inf.a_ptr = nullptr;
    p->tc.fps.a_ptr = nullptr;
    p->tc.infs.a_ptr = nullptr;
    p->tc.wg_a_ptr = nullptr;
    return NB_OK;
}

nb_status nb_cbs_plan_set_fwd_residual(nb_cbs_plan p, const void* res, int64_t ld_res) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    NB_CHECK_PTR(res, true);
    const int vec = is_f32(p) ? 4 : 8;
    if (ld_res == p->g.c_out) ld_res = 0;
    if (res && ld_res != 0 && (ld_res < p->g.c_out || ld_res % vec != 0))
        return fail(NB_ERR_INVALID_ARG, "ld_res must be 0 (dense) or at least c_out and a multiple of %d elements", vec);
    p->fwd_res = res;
    p->ld_res = res ? ld_res : 0;
    return NB_OK;
}

nb_status nb_cbs_plan_set_bwd_residual(nb_cbs_plan p, void* gres, int64_t ld_gres, int32_t accumulate) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    NB_CHECK_PTR(gres, true);
    if (accumulate != 0 && accumulate != 1) return fail(NB_ERR_INVALID_ARG, "accumulate must be 0 or 1, got %d", accumulate);
    if (ld_gres == p->g.c_out) ld_gres = 0;
    if (gres && ld_gres != 0 && (ld_gres < p->g.c_out || ld_gres % 8 != 0))
        return fail(NB_ERR_INVALID_ARG, "ld_gres must be 0 (dense) or at least c_out and a multiple of 8 elements");
    if (gres && (!p->fuse_finalize || is_f32(p)))
        return fail(NB_ERR_UNSUPPORTED, "the shortcut's gradient rides in the dy pass of the default 16-bit plans only (not fp32 mode, not NB_CBS_FLAG_SEPARATE_FINALIZE)");
    p->bwd_gres = gres;
    p->ld_gres = gres ? ld_gres : 0;
    p->gres_add = accumulate != 0;
    return NB_OK;
}

nb_status nb_cbs_plan_set_dx_target(nb_cbs_plan p, int64_t ld_dx, int32_t accumulate) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    if (accumulate != 0 && accumulate != 1) return fail(NB_ERR_INVALID_ARG, "accumulate must be 0 or 1, got %d", accumulate);
    if (ld_dx == p->g.c_in) ld_dx = 0;
    if (ld_dx != 0 && (ld_dx < p->g.c_in || ld_dx % 8 != 0)) return fail(NB_ERR_INVALID_ARG, "ld_dx must be 0 (dense) or at least c_in and a multiple of 8 elements");
    if ((ld_dx != 0 || accumulate) && (is_f32(p) || p->stem || !p->tc.dgrad || p->g.stride != 1))
        return fail(NB_ERR_UNSUPPORTED, "a pitched or accumulating dx needs the tensor-core data gradient of a stride-1 layer (its epilogue stores through TMA)");
    p->ld_dx = ld_dx;
    p->dx_accumulate = accumulate != 0;
    return NB_OK;
}

nb_status nb_cbs_plan_paths(nb_cbs_plan p, int32_t* paths3) {
    g_err.clear();
    if (!p || !paths3) return fail(NB_ERR_INVALID_ARG, "NULL argument");
    paths3[0] = p->tc.fprop ? 1 : 0;
    paths3[1] = p->tc.dgrad ? 1 : 0;
    paths3[2] = p->tc.wgrad ? 1 : 0;
    return NB_OK;
}

unsigned long long nb_cbs_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

nb_status nb_cbs_profile_enable(nb_cbs_plan p, int32_t enable) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    if (enable && !p->ev0) {
        NB_CUDA_CHECK(cudaEventCreate(&p->ev0));
        NB_CUDA_CHECK(cudaEventCreate(&p->ev1));
    }
    p->profiling = enable != 0;
    for (int i = 0; i < SITE_COUNT; ++i) {
        p->prof_ms[i] = 0.0;
        p->prof_n[i] = 0;
    }
    return NB_OK;
}

const char* nb_cbs_profile_site_name(int32_t site) { return (site >= 0 && site < SITE_COUNT) ? kSiteNames[site] : nullptr; }

nb_status nb_cbs_profile_read(nb_cbs_plan p, int32_t site, double* total_ms, int64_t* launches) {
    g_err.clear();
    if (!p || !total_ms || !launches) return fail(NB_ERR_INVALID_ARG, "NULL argument");
    if (site < 0 || site >= SITE_COUNT) return fail(NB_ERR_INVALID_ARG, "site %d out of range", site);
    *total_ms = p->prof_ms[site];
    *launches = p->prof_n[site];
    return NB_OK;
}

nb_status nb_cbs_poll_status(nb_cbs_plan p, void* stream) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int host[ST_WORDS];
    NB_CUDA_CHECK(cudaStreamSynchronize(st));
    NB_CUDA_CHECK(cudaMemcpy(host, p->status, sizeof host, cudaMemcpyDeviceToHost));
    NB_CUDA_CHECK(cudaMemset(p->status, 0, sizeof host));
    if (host[ST_ERR] != 0 && p->acc)  // a kernel that gave up may have left sums behind: the next call must find zeros
        NB_CUDA_CHECK(cudaMemset(p->acc, 0, (size_t)(p->acc_copies_f + p->acc_copies_b) * 2 * p->g.c_out * sizeof(double)));
    if (host[ST_ERR] != 0)
        return fail((nb_status)host[ST_ERR], "device status: error %d at site %d (detail %d)", host[ST_ERR], host[ST_WHERE], host[ST_DETAIL]);
    if (host[ST_SAT] != 0) {
        char buf[96];
        snprintf(buf, sizeof buf, "%d fp16 stores of the saved convolution output saturated", host[ST_SAT]);
        g_err = buf;
    }
    return NB_OK;
}

nb_status nb_conv_bn_silu_fwd(nb_cbs_plan p, const void* x, const void* w, const float* gamma, const float* beta,
                              float* running_mean, float* running_var, void* y_saved, float* save_mean, float* save_invstd,
                              void* a_out, void* workspace, size_t workspace_bytes, void* stream) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    NB_CHECK_PTR(x); NB_CHECK_PTR(w); NB_CHECK_PTR(gamma); NB_CHECK_PTR(beta);
    NB_CHECK_PTR(y_saved); NB_CHECK_PTR(save_mean); NB_CHECK_PTR(save_invstd); NB_CHECK_PTR(a_out);
    if ((running_mean == nullptr) != (running_var == nullptr))
        return fail(NB_ERR_INVALID_ARG, "running_mean and running_var must both be given or both be NULL");
    NB_TRY(check_ws(workspace, workspace_bytes, p->fwd_bytes));
    DeviceGuard on_device(p->device);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    char* ws = static_cast<char*>(workspace);
    float* scale = reinterpret_cast<float*>(ws + p->off_scale);
    float* shift = reinterpret_cast<float*>(ws + p->off_shift);
    float* part = reinterpret_cast<float*>(ws + p->off_fpart);
    int nparts = p->ew.blocks_stats;
    bool finalized = false;
    if (is_f32(p)) {
        NB_TRY((run_simt_fprop<float, float>(p, x, w, y_saved, ws + p->off_sgpart, p->fuse_finalize, st)));
        finalized = p->fuse_finalize;
        if (!finalized) NB_TRY(run_stats_partial<float>(p, y_saved, part, st));
    } else if (p->stem) {
        // the first layer's kernel sums the statistics of the values it stores itself (one partial slice per block)
        SiteTimer tm(p, SITE_FPROP, st);
        const bool fuse = p->fuse_finalize;  // sums into the plan's accumulators; the normalise + SiLU pass finalizes
        NB_TRY(NB_WITH_AT(p, run_stem_fprop<__half, AT, false>(p, x, w, y_saved, StemEpi{}, fuse ? nullptr : part, fuse ? p->acc : nullptr, st)));
        nparts = p->stem_fprop_blocks;
        finalized = fuse;
    } else if (p->tc.fprop) {
        SiteTimer tm(p, SITE_FPROP, st);
        const long long l0 = p->tc.launches;
        // writes y (fp16) and adds its channel sums to the accumulators (or writes them as per-CTA partial sums)
        const bool fuse = p->fuse_finalize;
        const ChanAcc ca{fuse ? p->acc : nullptr, nullptr, fuse ? p->acc_copies_f : 1};
        const nb_status ts = tc_fprop(&p->tc, p->g, x, w, y_saved, part, p->status, st, ca);
        g_launches.fetch_add((unsigned long long)(p->tc.launches - l0), std::memory_order_relaxed);
        if (ts != NB_OK) return fail(ts, "%s", tc_last_error());
        nparts = p->tc.fprop_parts;
        finalized = fuse;
    } else {
        NB_TRY(NB_WITH_AT(p, run_simt_fprop<AT, __half>(p, x, w, y_saved, ws + p->off_sgpart, p->fuse_finalize, st)));
        finalized = p->fuse_finalize;
        if (!finalized) NB_TRY(run_stats_partial<__half>(p, y_saved, part, st));
    }
    if (!finalized)
        NB_TRY(run_finalize(p, part, nparts, gamma, beta, save_mean, save_invstd, scale, shift, running_mean, running_var, nullptr, nullptr, st));
    // when the convolution has left its sums in the accumulators the pass derives mean, invstd, scale and shift from them itself
    const double M = (double)p->g.m;
    const FwdFin fin{1.0 / M, M / (M - 1.0), p->desc.eps, p->desc.momentum, gamma, beta, save_mean, save_invstd, running_mean, running_var};
    if (p->exact_apart) {
        SiteTimer tm(p, SITE_FINALIZE, st);
        const ChanAcc ca{p->acc, nullptr, p->acc_copies_f};
        launch_k(bn_exact_finalize_kernel, dim3((unsigned)((2 * p->g.c_out + 127) / 128)), dim3(128), 0, st, 1, ca, p->g.c_out, fin, scale, shift);
        NB_LAUNCH_OK("bn_exact_finalize");
        finalized = false;  // (the pass reads scale and shift)
    }
    if (is_f32(p)) return run_apply<float, float, false>(p, y_saved, a_out, scale, shift, st, p->ld_a, p->fwd_res, p->ld_res, finalized ? &fin : nullptr);
    return NB_WITH_AT(p, run_apply<__half, AT, true>(p, y_saved, a_out, scale, shift, st, p->ld_a, p->fwd_res, p->ld_res, finalized ? &fin : nullptr));
}

namespace {
// conv -> out = act(conv*scale_c + shift_c) with (scale, shift) from evaluation-mode BN or a bias (see bn_eval_coef)
nb_status run_infer(nb_cbs_plan_s* p, const void* x, const void* w, const float* gamma, const float* beta, const float* rmean, const float* rvar,
                    int act, void* out, char* ws, cudaStream_t st) {
    if (infer_fused(p) && !p->stem) {
        SiteTimer tm(p, SITE_INFER, st);
        const long long l0 = p->tc.launches;
        const EpiAffine e{gamma, beta, rmean, rvar, p->desc.eps, act};
        const nb_status ts = tc_infer(&p->tc, p->g, x, w, out, e, p->status, st);
        g_launches.fetch_add((unsigned long long)(p->tc.launches - l0), std::memory_order_relaxed);
        if (ts != NB_OK) return fail(ts, "%s", tc_last_error());
        return NB_OK;
    }
    if (!is_f32(p) && p->stem) {  // the first layer's own kernel applies the coefficients and the activation itself
        SiteTimer tm(p, SITE_INFER, st);
        return NB_WITH_AT(p, run_stem_fprop<AT, AT, true>(p, x, w, out, StemEpi{gamma, beta, rmean, rvar, p->desc.eps, act}, nullptr, nullptr, st));
    }
    float* scale = reinterpret_cast<float*>(ws + p->off_scale);
    float* shift = reinterpret_cast<float*>(ws + p->off_shift);
    void* y = ws + p->off_iy;
    if (is_f32(p)) {
        NB_TRY((run_simt_fprop<float, float>(p, x, w, y, ws + p->off_isg, false, st)));
    } else {
        NB_TRY(NB_WITH_AT(p, run_simt_fprop<AT, __half>(p, x, w, y, ws + p->off_isg, false, st)));
    }
    {
        SiteTimer tm(p, SITE_EVAL_COEF, st);
        launch_k(bn_eval_coef_kernel, dim3((unsigned)((p->g.c_out + 255) / 256)), dim3(256), 0, st, 1, gamma, beta, rmean, rvar, p->desc.eps, p->g.c_out, scale, shift);
        NB_LAUNCH_OK("bn_eval_coef");
    }
    if (is_f32(p)) return act ? run_apply<float, float, false, true>(p, y, out, scale, shift, st) : run_apply<float, float, false, false>(p, y, out, scale, shift, st);
    return NB_WITH_AT(p, act ? run_apply<__half, AT, true, true>(p, y, out, scale, shift, st) : run_apply<__half, AT, true, false>(p, y, out, scale, shift, st));
}
}  // namespace

nb_status nb_cbs_infer_workspace_bytes(nb_cbs_plan p, size_t* bytes, int32_t* fused) {
    g_err.clear();
    if (!p || !bytes) return fail(NB_ERR_INVALID_ARG, "NULL argument");
    *bytes = p->infer_bytes;
    if (fused) *fused = infer_fused(p) ? 1 : 0;
    return NB_OK;
}

nb_status nb_conv_bn_silu_infer(nb_cbs_plan p, const void* x, const void* w, const float* gamma, const float* beta, const float* running_mean,
                                const float* running_var, void* a_out, void* workspace, size_t workspace_bytes, void* stream) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    NB_CHECK_PTR(x); NB_CHECK_PTR(w); NB_CHECK_PTR(gamma); NB_CHECK_PTR(beta); NB_CHECK_PTR(running_mean); NB_CHECK_PTR(running_var);
    NB_CHECK_PTR(a_out);
    if (p->pitched || p->fwd_res) return fail(NB_ERR_UNSUPPORTED, "the plan has row pitches or a residual set: only the training calls honour them");
    NB_TRY(check_ws(workspace, workspace_bytes, p->infer_bytes));
    DeviceGuard on_device(p->device);
    return run_infer(p, x, w, gamma, beta, running_mean, running_var, 1, a_out, static_cast<char*>(workspace), static_cast<cudaStream_t>(stream));
}

nb_status nb_conv_bias_act(nb_cbs_plan p, const void* x, const void* w, const float* bias, int32_t act, void* out, void* workspace,
                           size_t workspace_bytes, void* stream) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    NB_CHECK_PTR(x); NB_CHECK_PTR(w); NB_CHECK_PTR(bias, true); NB_CHECK_PTR(out);
    if (act != 0 && act != 1) return fail(NB_ERR_INVALID_ARG, "act must be 0 (none) or 1 (SiLU), got %d", act);
    if (p->pitched || p->fwd_res) return fail(NB_ERR_UNSUPPORTED, "the plan has row pitches or a residual set: only the training calls honour them");
    NB_TRY(check_ws(workspace, workspace_bytes, p->infer_bytes));
    DeviceGuard on_device(p->device);
    return run_infer(p, x, w, nullptr, bias, nullptr, nullptr, act, out, static_cast<char*>(workspace), static_cast<cudaStream_t>(stream));
}

nb_status nb_bn_fold(nb_cbs_plan p, const void* w, const float* gamma, const float* beta, const float* running_mean, const float* running_var,
                     void* w_folded, float* bias_folded, void* stream) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    NB_CHECK_PTR(w); NB_CHECK_PTR(gamma); NB_CHECK_PTR(beta); NB_CHECK_PTR(running_mean); NB_CHECK_PTR(running_var);
    NB_CHECK_PTR(w_folded); NB_CHECK_PTR(bias_folded);
    DeviceGuard on_device(p->device);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const long long K = p->g.kdim, total = K * p->g.c_out;
    const unsigned blocks = (unsigned)std::min<long long>((total + 255) / 256, (long long)p->sm_count * 8);
    SiteTimer tm(p, SITE_FOLD, st);
    if (is_f32(p))
        launch_k(bn_fold_kernel<float>, dim3(blocks), dim3(256), 0, st, 1, static_cast<const float*>(w), K, p->g.c_out, gamma, beta, running_mean, running_var,
                 p->desc.eps, static_cast<float*>(w_folded), bias_folded);
    else if (is_f16(p))
        launch_k(bn_fold_kernel<__half>, dim3(blocks), dim3(256), 0, st, 1, static_cast<const __half*>(w), K, p->g.c_out, gamma, beta, running_mean, running_var,
                 p->desc.eps, static_cast<__half*>(w_folded), bias_folded);
    else
        launch_k(bn_fold_kernel<__nv_bfloat16>, dim3(blocks), dim3(256), 0, st, 1, static_cast<const __nv_bfloat16*>(w), K, p->g.c_out, gamma, beta, running_mean,
                 running_var, p->desc.eps, static_cast<__nv_bfloat16*>(w_folded), bias_folded);
    return launch_ok("bn_fold");
}

nb_status nb_bn_stats(nb_cbs_plan p, const void* y, int32_t y_dtype, float* mean, float* invstd, float* sum, float* sumsq,
                      void* workspace, size_t workspace_bytes, void* stream) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    NB_CHECK_PTR(y); NB_CHECK_PTR(mean); NB_CHECK_PTR(invstd);
    NB_CHECK_PTR(sum, true); NB_CHECK_PTR(sumsq, true);
    const int want = is_f32(p) ? NB_DTYPE_F32 : NB_DTYPE_F16;
    if (y_dtype != want) return fail(NB_ERR_UNSUPPORTED, "y_dtype %d does not match the plan's mode (expected %d)", y_dtype, want);
    NB_TRY(check_ws(workspace, workspace_bytes, p->fwd_bytes));
    DeviceGuard on_device(p->device);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    float* part = reinterpret_cast<float*>(static_cast<char*>(workspace) + p->off_fpart);
    if (is_f32(p)) NB_TRY(run_stats_partial<float>(p, y, part, st));
    else NB_TRY(run_stats_partial<__half>(p, y, part, st));
    return run_finalize(p, part, p->ew.blocks_stats, nullptr, nullptr, mean, invstd, nullptr, nullptr, nullptr, nullptr, sum, sumsq, st);
}

namespace {
// dx from dy, the last step of a call or in front of the weight gradient.  rearranged: the pass that made dy has rearranged the
// filter for the tensor-core kernel; else that is done here.
nb_status run_dgrad(nb_cbs_plan_s* p, const void* dy, const void* w, void* dx, char* ws, bool rearranged, cudaStream_t st) {
    if (is_f32(p)) return run_simt_dgrad<float>(p, dy, w, dx, ws + p->off_dgpart, st);
    if (p->stem) {
        SiteTimer tm(p, SITE_DGRAD, st);
        return NB_WITH_AT(p, run_stem_dgrad<AT>(p, dy, w, dx, st));
    }
    if (p->tc.dgrad) {
        SiteTimer tm(p, SITE_DGRAD, st);
        const long long l0 = p->tc.launches;
        const nb_status ts = tc_dgrad(&p->tc, p->g, dy, w, dx, ws + p->off_wt, p->status, st, rearranged, p->ld_dx, p->dx_accumulate);
        g_launches.fetch_add((unsigned long long)(p->tc.launches - l0), std::memory_order_relaxed);
        return ts == NB_OK ? NB_OK : fail(ts, "%s", tc_last_error());
    }
    return NB_WITH_AT(p, run_simt_dgrad<AT>(p, dy, w, dx, ws + p->off_dgpart, st));
}

// overlap: the launch in front of this one on the stream is this layer's data gradient (see the end of common.cuh).  Only a
// caller that has just queued it itself, in the same call of the library, can say so.
nb_status run_wgrad(nb_cbs_plan_s* p, const void* x, const void* dy, float* dw, char* ws, bool overlap, cudaStream_t st) {
    float* partial = reinterpret_cast<float*>(ws + p->off_wgpart);
    overlap = overlap && pdl_enabled();
    if (is_f32(p)) return run_simt_wgrad<float>(p, x, dy, dw, partial, overlap, st);
    if (p->stem) {
        {
            SiteTimer tm(p, SITE_WGRAD, st);
            NB_TRY(NB_WITH_AT(p, run_stem_wgrad<AT>(p, x, dy, partial, overlap, st)));
        }
        const size_t elems = (size_t)p->g.c_out * p->g.kdim;
        SiteTimer tm(p, SITE_SPLITK_REDUCE, st);
        launch_k(splitk_reduce_tall_kernel, dim3((unsigned)((elems + 31) / 32)), dim3(1024), 0, st, 1, partial, p->stem_wgrad_blocks, elems, dw);
        return launch_ok("splitk_reduce");
    }
    if (p->tc.wgrad) {
        SiteTimer tm(p, SITE_WGRAD, st);
        const long long l0 = p->tc.launches;
        const nb_status ts = tc_wgrad(&p->tc, p->g, x, dy, dw, partial, p->status, st, overlap);
        g_launches.fetch_add((unsigned long long)(p->tc.launches - l0), std::memory_order_relaxed);
        return ts == NB_OK ? NB_OK : fail(ts, "%s", tc_last_error());
    }
    return NB_WITH_AT(p, run_simt_wgrad<AT>(p, x, dy, dw, partial, overlap, st));
}
}  // namespace

namespace {
// dgamma, dbeta and dy, and the checks of the data-gradient call; its convolution follows
nb_status run_bwd_head(nb_cbs_plan p, const void* g, const void* y_saved, const float* save_mean, const float* save_invstd, const float* gamma, const float* beta,
                       const void* w, void* dx, float* dgamma, float* dbeta, void* dy_out, void* workspace, size_t workspace_bytes, cudaStream_t st) {
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    NB_CHECK_PTR(g); NB_CHECK_PTR(y_saved); NB_CHECK_PTR(save_mean); NB_CHECK_PTR(save_invstd);
    NB_CHECK_PTR(gamma); NB_CHECK_PTR(beta); NB_CHECK_PTR(dgamma); NB_CHECK_PTR(dbeta); NB_CHECK_PTR(dy_out);
    NB_CHECK_PTR(dx, true);
    if (dx) NB_CHECK_PTR(w);
    NB_TRY(check_ws(workspace, workspace_bytes, p->bwd_bytes));
    char* ws = static_cast<char*>(workspace);
    float* coef = reinterpret_cast<float*>(ws + p->off_coef);
    float* part = reinterpret_cast<float*>(ws + p->off_bpart);
    if (is_f32(p)) {
        NB_TRY((run_bwd_elementwise<float, float, false>(p, g, y_saved, save_mean, save_invstd, gamma, beta, dgamma, dbeta, dy_out, part, coef, st)));
    } else {
        const bool tc_dg = dx && !p->stem && p->tc.dgrad;  // the finalize kernel also rearranges the filter for the tensor-core dgrad
        NB_TRY(NB_WITH_AT(p, run_bwd_elementwise<__half, AT, true>(p, g, y_saved, save_mean, save_invstd, gamma, beta, dgamma, dbeta, dy_out, part, coef, st,
                                                                   tc_dg ? w : nullptr, tc_dg ? ws + p->off_wt : nullptr, tc_dg ? &p->tc.wtp : nullptr)));
    }
    return NB_OK;
}
}  // namespace

nb_status nb_conv_bn_silu_bwd_data(nb_cbs_plan p, const void* g, const void* y_saved, const float* save_mean,
                                   const float* save_invstd, const float* gamma, const float* beta, const void* w, void* dx,
                                   float* dgamma, float* dbeta, void* dy_out, void* workspace, size_t workspace_bytes, void* stream) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    DeviceGuard on_device(p->device);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    NB_TRY(run_bwd_head(p, g, y_saved, save_mean, save_invstd, gamma, beta, w, dx, dgamma, dbeta, dy_out, workspace, workspace_bytes, st));
    return dx ? run_dgrad(p, dy_out, w, dx, static_cast<char*>(workspace), true, st) : NB_OK;
}

nb_status nb_conv_bn_silu_bwd_weight(nb_cbs_plan p, const void* x, const void* dy, float* dw, void* workspace,
                                     size_t workspace_bytes, void* stream) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    NB_CHECK_PTR(x); NB_CHECK_PTR(dy); NB_CHECK_PTR(dw);
    NB_TRY(check_ws(workspace, workspace_bytes, p->bwd_bytes));
    DeviceGuard on_device(p->device);
    return run_wgrad(p, x, dy, dw, static_cast<char*>(workspace), false, static_cast<cudaStream_t>(stream));
}

nb_status nb_conv_bn_silu_bwd(nb_cbs_plan p, const void* x, const void* g, const void* y_saved, const float* save_mean,
                              const float* save_invstd, const float* gamma, const float* beta, const void* w, void* dx, float* dw,
                              float* dgamma, float* dbeta, void* dy_out, void* workspace, size_t workspace_bytes, void* stream) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    NB_CHECK_PTR(x); NB_CHECK_PTR(dw);  // (the rest by the first of the two)
    DeviceGuard on_device(p->device);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    NB_TRY(run_bwd_head(p, g, y_saved, save_mean, save_invstd, gamma, beta, w, dx, dgamma, dbeta, dy_out, workspace, workspace_bytes, st));
    char* ws = static_cast<char*>(workspace);
    if (dx && !p->stem && !p->tc.dgrad && !p->tc.wgrad) {
        float* wgpart = reinterpret_cast<float*>(ws + p->off_wgpart);
        if (is_f32(p)) return run_simt_grads<float>(p, x, dy_out, w, dx, dw, ws + p->off_dgpart, wgpart, st);
        return NB_WITH_AT(p, run_simt_grads<AT>(p, x, dy_out, w, dx, dw, ws + p->off_dgpart, wgpart, st));
    }
    if (dx) NB_TRY(run_dgrad(p, dy_out, w, dx, ws, true, st));
    return run_wgrad(p, x, dy_out, dw, ws, dx != nullptr, st);
}

nb_status nb_conv_bias_bwd(nb_cbs_plan p, const void* x, const void* w, const void* dout, void* dx, float* dw, float* dbias, void* workspace,
                           size_t workspace_bytes, void* stream) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    NB_CHECK_PTR(x); NB_CHECK_PTR(dout); NB_CHECK_PTR(dw); NB_CHECK_PTR(dx, true); NB_CHECK_PTR(dbias, true);
    if (dx) NB_CHECK_PTR(w);
    if (p->pitched || p->ld_dx || p->dx_accumulate || p->fwd_res || p->bwd_gres) return fail(NB_ERR_UNSUPPORTED, "the plan has row pitches, a dx target or a residual set: only the training calls honour them");
    NB_TRY(check_ws(workspace, workspace_bytes, p->bwd_bytes));
    DeviceGuard on_device(p->device);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    char* ws = static_cast<char*>(workspace);
    if (dbias) {  // column sums of dout: the statistics kernels with only the raw sum requested
        float* part = reinterpret_cast<float*>(ws + p->off_bpart);
        if (is_f32(p)) NB_TRY(run_stats_partial<float>(p, dout, part, st));
        else NB_TRY(NB_WITH_AT(p, run_stats_partial<AT>(p, dout, part, st)));
        NB_TRY(run_finalize(p, part, p->ew.blocks_stats, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, dbias, nullptr, st));
    }
    if (dx) NB_TRY(run_dgrad(p, dout, w, dx, ws, false, st));
    return run_wgrad(p, x, dout, dw, ws, dx != nullptr, st);
}

}  // extern "C"

// ---------------------------------------------------------------- batch statistics without any allocation
// Scratch for nb_bn_stats_static: partial sums [kStaticParts][2][kStaticMaxC] floats = 2 MiB, resident on every
// GPU that loads this library until the process exits.  In host code the name `g_static_partials` is only a
// handle for the symbol, never a device address: the address comes from cudaGetSymbolAddress below.
namespace {
constexpr int kStaticParts = 256;
constexpr int kStaticMaxC = 1024;
constexpr int kStaticMaxDevices = 64;
}  // namespace
static __device__ __align__(256) float g_static_partials[(size_t)kStaticParts * 2 * kStaticMaxC];

namespace {
std::mutex g_static_mu;
float* g_static_ptr[kStaticMaxDevices] = {};
int g_static_sms[kStaticMaxDevices] = {};

// Once per device, with that device current: resolve the device address of the static scratch array.
nb_status static_scratch_for_current_device(float** out, int* sms) {
    int dev = -1;
    NB_CUDA_CHECK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kStaticMaxDevices) return fail(NB_ERR_UNSUPPORTED, "device ordinal %d is beyond %d", dev, kStaticMaxDevices);
    std::lock_guard<std::mutex> lock(g_static_mu);
    if (!g_static_ptr[dev]) {
        int major = 0, count = 0;
        NB_CUDA_CHECK(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev));
        if (major != 10) return fail(NB_ERR_ARCH, "device %d is not compute capability 10.x", dev);
        NB_CUDA_CHECK(cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev));
        void* ptr = nullptr;
        NB_CUDA_CHECK(cudaGetSymbolAddress(&ptr, g_static_partials));
        if (!ptr) return fail(NB_ERR_CUDA, "cudaGetSymbolAddress returned a null address");
        g_static_sms[dev] = count;
        g_static_ptr[dev] = static_cast<float*>(ptr);
    }
    *out = g_static_ptr[dev];
    *sms = g_static_sms[dev];
    return NB_OK;
}
}  // namespace

extern "C" nb_status nb_bn_stats_static(const void* y, int32_t y_dtype, int64_t m, int32_t c, float eps, float* mean, float* invstd,
                                        float* sum, float* sumsq, void* stream) {
    g_err.clear();
    NB_CHECK_PTR(y); NB_CHECK_PTR(mean); NB_CHECK_PTR(invstd);
    NB_CHECK_PTR(sum, true); NB_CHECK_PTR(sumsq, true);
    if (y_dtype != NB_DTYPE_F16 && y_dtype != NB_DTYPE_F32) return fail(NB_ERR_UNSUPPORTED, "y_dtype %d: only F16 and F32 are supported", y_dtype);
    if (m < 2 || c <= 0) return fail(NB_ERR_INVALID_ARG, "need m >= 2 rows and c > 0 channels (m=%lld c=%d)", (long long)m, c);
    if (!(eps > 0.f)) return fail(NB_ERR_INVALID_ARG, "eps must be positive");
    const int vec = y_dtype == NB_DTYPE_F32 ? 4 : 8;
    if (c % vec) return fail(NB_ERR_UNSUPPORTED, "c=%d must be a multiple of %d for this dtype", c, vec);
    if (c > kStaticMaxC)
        return fail(NB_ERR_UNSUPPORTED, "c=%d exceeds the %d channels the built-in scratch array holds; use nb_bn_stats with a workspace", c, kStaticMaxC);
    if ((double)m * c >= 9.0e18) return fail(NB_ERR_UNSUPPORTED, "tensor too large");
    float* part = nullptr;
    int sms = 0;
    NB_TRY(static_scratch_for_current_device(&part, &sms));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int cgs = c / vec;
    const int R = cgs >= 256 ? 1 : 256 / cgs;
    const int tpb = cgs * R;
    const long long total_vecs = (long long)m * cgs;
    const long long max_blocks = (total_vecs + tpb - 1) / tpb;
    const int blocks = (int)std::min<long long>(max_blocks, std::min(kStaticParts, std::max(1, sms)));
    // Every partial that the second kernel reads is written by the first one in this same call, so nothing in the
    // array has to start at zero and the previous call's contents do not matter.
    if (y_dtype == NB_DTYPE_F32)
        launch_k(bn_stats_partial_kernel<float>, dim3(blocks), dim3(tpb), (size_t)tpb * vec * sizeof(float), st, 1, static_cast<const float*>(y), total_vecs, c, part);
    else
        launch_k(bn_stats_partial_kernel<__half>, dim3(blocks), dim3(tpb), (size_t)tpb * vec * sizeof(float), st, 1, static_cast<const __half*>(y), total_vecs, c, part);
    NB_LAUNCH_OK("bn_stats_partial (static scratch)");
    launch_k(bn_finalize_kernel, dim3((c + 7) / 8), dim3(256), 0, st, 1, part, blocks, c, (double)m, eps, 0.f, nullptr, nullptr, mean, invstd, nullptr,
                                                              nullptr, nullptr, nullptr, sum, sumsq);
    return launch_ok("bn_finalize (static scratch)");
}

extern "C" {

// ---------------------------------------------------------------- host-buffer step
namespace {
struct StepLayout {
    size_t x, w, gamma, beta, g, y, mean, invstd, a, dy, dx, dw, dgamma, dbeta, ws_fwd, ws_bwd, total;
    size_t nx, nw, ny_act, ny_saved, ndw;  // byte counts
};
StepLayout step_layout(const nb_cbs_plan_s* p) {
    StepLayout L;
    const size_t act = is_f32(p) ? 4 : 2, ysz = is_f32(p) ? 4 : 2;
    const Geom& g = p->g;
    L.nx = (size_t)g.n * g.h * g.w * g.c_in * act;
    L.nw = (size_t)g.c_out * g.kdim * act;
    L.ny_act = (size_t)g.m * g.c_out * act;
    L.ny_saved = (size_t)g.m * g.c_out * ysz;
    L.ndw = (size_t)g.c_out * g.kdim * 4;
    const size_t cb = (size_t)g.c_out * 4;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 256); return o; };
    L.x = take(L.nx); L.w = take(L.nw); L.gamma = take(cb); L.beta = take(cb); L.g = take(L.ny_act);
    L.y = take(L.ny_saved); L.mean = take(cb); L.invstd = take(cb); L.a = take(L.ny_act); L.dy = take(L.ny_act);
    L.dx = take(L.nx); L.dw = take(L.ndw); L.dgamma = take(cb); L.dbeta = take(cb);
    L.ws_fwd = take(p->fwd_bytes); L.ws_bwd = take(p->bwd_bytes);
    L.total = off;
    return L;
}

// What host_step issues, and on what (host_step.cuh).
struct HostStepOps {
    nb_cbs_plan_s* p;
    const StepLayout& L;
    char* d;
    cudaStream_t st[3];  // by HostStepStream
    void* host[10] = {};  // by HostStepTensor
    float* f32(size_t off) const { return reinterpret_cast<float*>(d + off); }
    int order(HostStepStream from, HostStepStream to) {
        const cudaEvent_t ev = p->copy_ev[from][to];
        NB_CUDA_CHECK(cudaEventRecord(ev, st[from]));
        NB_CUDA_CHECK(cudaStreamWaitEvent(st[to], ev, 0));
        return NB_OK;
    }
    int copy(HostStepTensor t, HostStepStream stream) {
        const size_t off[10] = {L.x, L.w, L.gamma, L.beta, L.g, L.a, L.dx, L.dw, L.dgamma, L.dbeta};
        const size_t cb = (size_t)p->g.c_out * 4, bytes[10] = {L.nx, L.nw, cb, cb, L.ny_act, L.ny_act, L.nx, L.ndw, cb, cb};
        if (t < HT_A) NB_CUDA_CHECK(cudaMemcpyAsync(d + off[t], host[t], bytes[t], cudaMemcpyHostToDevice, st[stream]));
        else NB_CUDA_CHECK(cudaMemcpyAsync(host[t], d + off[t], bytes[t], cudaMemcpyDeviceToHost, st[stream]));
        return NB_OK;
    }
    int forward() {
        return nb_conv_bn_silu_fwd(p, d + L.x, d + L.w, f32(L.gamma), f32(L.beta), nullptr, nullptr, d + L.y, f32(L.mean), f32(L.invstd), d + L.a, d + L.ws_fwd,
                                   p->fwd_bytes, st[HS_CALLER]);
    }
    int backward_data() {
        return nb_conv_bn_silu_bwd_data(p, d + L.g, d + L.y, f32(L.mean), f32(L.invstd), f32(L.gamma), f32(L.beta), d + L.w, host[HT_DX] ? d + L.dx : nullptr,
                                        f32(L.dgamma), f32(L.dbeta), d + L.dy, d + L.ws_bwd, p->bwd_bytes, st[HS_CALLER]);
    }
    int backward_weight() {
        return nb_conv_bn_silu_bwd_weight(p, d + L.x, d + L.dy, f32(L.dw), d + L.ws_bwd, p->bwd_bytes, st[HS_CALLER]);
    }
};
}  // namespace

nb_status nb_cbs_step_host_scratch_bytes(nb_cbs_plan p, size_t* bytes) {
    g_err.clear();
    if (!p || !bytes) return fail(NB_ERR_INVALID_ARG, "NULL argument");
    *bytes = step_layout(p).total;
    if (p->fuse_finalize && !p->copy_in) make_copy_streams(p);
    return NB_OK;
}

nb_status nb_conv_bn_silu_step_host(nb_cbs_plan p, const void* host_x, const void* host_w, const float* host_gamma,
                                    const float* host_beta, const void* host_g, void* host_a, void* host_dx, float* host_dw,
                                    float* host_dgamma, float* host_dbeta, void* device_scratch, size_t scratch_bytes, void* stream) {
    g_err.clear();
    if (!p) return fail(NB_ERR_INVALID_ARG, "plan is NULL");
    if (!host_x || !host_w || !host_gamma || !host_beta || !host_g || !host_a || !host_dw || !host_dgamma || !host_dbeta)
        return fail(NB_ERR_INVALID_ARG, "a required host pointer is NULL");
    if (p->pitched || p->ld_dx || p->dx_accumulate || p->fwd_res || p->bwd_gres) return fail(NB_ERR_UNSUPPORTED, "the plan has row pitches, a dx target or a residual set: the host-buffer step works on dense tensors");
    const StepLayout L = step_layout(p);
    NB_TRY(check_ws(device_scratch, scratch_bytes, L.total));
    DeviceGuard on_device(p->device);
    HostStepOps ops{p, L, static_cast<char*>(device_scratch), {static_cast<cudaStream_t>(stream), p->copy_in, p->copy_out}};
    ops.host[HT_X] = const_cast<void*>(host_x); ops.host[HT_W] = const_cast<void*>(host_w); ops.host[HT_G] = const_cast<void*>(host_g);
    ops.host[HT_GAMMA] = const_cast<float*>(host_gamma); ops.host[HT_BETA] = const_cast<float*>(host_beta);
    ops.host[HT_A] = host_a; ops.host[HT_DX] = host_dx; ops.host[HT_DW] = host_dw;
    ops.host[HT_DGAMMA] = host_dgamma; ops.host[HT_DBETA] = host_dbeta;
    return host_step(ops, p->copy_in != nullptr, host_dx != nullptr);
}

}  // extern "C"

