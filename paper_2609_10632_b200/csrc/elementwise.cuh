// HBM-bound passes over [M][C] NHWC tensors: batch statistics, normalise+affine+SiLU, and their backward.
// All of them walk the tensor as a flat array of 16-byte vectors with a stride that is a multiple of the
// number of vectors per row, so a thread always sees the same channel group: per-channel parameters and
// accumulators live in registers, loads are fully coalesced, and the sums of a block have a fixed order; how block sums
// meet is at ChanAcc.
#pragma once
#include <type_traits>

#include "common.cuh"
#include "ptx_sm100.cuh"

namespace nbcbs {

// sigmoid(z).  The fast form is 0.5*tanh(z/2) + 0.5 with the hardware tanh approximation (one special-function
// instruction instead of an exponential and a reciprocal; absolute error about 2.5e-4, far below the bf16 rounding of
// the results it feeds); these passes issue enough instructions per byte that the special-function unit matters.
template <bool FAST> __device__ __forceinline__ float sigmoid_f(float z) {
    if (FAST) {
        float t;
        asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(0.5f * z));
        return fmaf(0.5f, t, 0.5f);
    } else {
        return 1.f / (1.f + expf(-z));
    }
}

// SiLU of two values given as halves: z * sigmoid(z) = h + h * tanh(h) with h = z / 2.
__device__ __forceinline__ float2 silu2_of_half(float2 h) {
    float2 t;
    asm("tanh.approx.f32 %0, %1;" : "=f"(t.x) : "f"(h.x));
    asm("tanh.approx.f32 %0, %1;" : "=f"(t.y) : "f"(h.y));
    return fma2(h, t, h);
}

// The same for two values at once, and dz = g * s * (1 + z*(1 - s)) with s = sigmoid(z) (the derivative of SiLU times g);
// the operations and their order are those of the scalar expressions the passes used to spell out, so the bits agree.
template <bool FAST> __device__ __forceinline__ float2 sigmoid2(float2 z) {
    if (FAST) {
        const float2 hz = mul2(splat2(0.5f), z);
        float2 t;
        asm("tanh.approx.f32 %0, %1;" : "=f"(t.x) : "f"(hz.x));
        asm("tanh.approx.f32 %0, %1;" : "=f"(t.y) : "f"(hz.y));
        return fma2(splat2(0.5f), t, splat2(0.5f));
    } else {
        return make_float2(sigmoid_f<false>(z.x), sigmoid_f<false>(z.y));
    }
}
template <bool FAST> __device__ __forceinline__ float2 silu_bwd_dz2(float2 z, float2 g) {
    const float2 s = sigmoid2<FAST>(z);
    const float2 oms = fma2(s, splat2(-1.f), splat2(1.f));  // 1 - s, exactly
    return mul2(mul2(g, s), fma2(z, oms, splat2(1.f)));
}

// A thread's next vectors of a long stream, in flight in shared memory: cp.async copies of 16 bytes into slots that only this
// thread reads (no barrier), EW_RING steps ahead.  Registers hold one step.  (Loads into registers had one step of each
// tensor in flight per thread, and an L2 prefetch two steps ahead.  Measured on the backward reduction, two / three / four
// steps against that: 67 MB tensors 41.4 -> 40.1 / 39.0 / 41.8 us, 41 MB 28.5 -> 24.9 / 23.7 / 24.1, 157 MB 70.0 -> 69.5 / 69.6 /
// 71.6.)
constexpr int EW_RING = 3;
__device__ __forceinline__ void ew_copy16(void* smem, const void* gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void ew_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void ew_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(EW_RING - 1) : "memory"); }

// ------------------------------------------------------------------ per-channel sum and sum of squares
// partials layout: [gridDim.x][2][C]; blockDim.x = (C/V) * R.
template <typename YT>
__global__ void __launch_bounds__(288, 3) bn_stats_partial_kernel(const YT* __restrict__ y, long long total_vecs, int C,
                                                                float* __restrict__ partials) {
    pdl_launch_dependents();
    pdl_wait();
    constexpr int V = Vec16<YT>::N;
    extern __shared__ float red[];  // [blockDim.x][V]
    const int tid = threadIdx.x;
    const int cgs = C / V;
    float s[V], ss[V];
#pragma unroll
    for (int i = 0; i < V; ++i) s[i] = ss[i] = 0.f;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long v = (long long)blockIdx.x * blockDim.x + tid; v < total_vecs; v += stride) {
        const Vec16<YT> q = ld16(y + v * V);
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const float f = to_f32(q.v[i]);
            s[i] += f;
            ss[i] = fmaf(f, f, ss[i]);
        }
    }
    const int R = blockDim.x / cgs;
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
        for (int i = 0; i < V; ++i) red[tid * V + i] = pass ? ss[i] : s[i];
        __syncthreads();
        for (int c = tid; c < C; c += blockDim.x) {
            const int g = c / V, e = c % V;
            float acc = 0.f;
            for (int r = 0; r < R; ++r) acc += red[(r * cgs + g) * V + e];
            partials[((size_t)blockIdx.x * 2 + pass) * C + c] = acc;
        }
        __syncthreads();
    }
}

// Both sums of channel c at once: s0 = sum over b of partials[b][0][c], s1 = the same for [b][1][c].  Lane l takes
// b = l, l+32, ... (all loads of a step are issued before any is used), then a butterfly over the 32 lanes, in fp64.
// The order is fixed, so the result is bitwise reproducible.
// L2 = read around L1 (the partials were written by other CTAs of the same launch).
// Sixteen loads (eight slices x two quantities) are issued before the first is used, so up to 256 slices cost one
// memory round trip; the fused finalize steps at the tail of other kernels sit on the critical path.
template <bool L2 = false>
__device__ __forceinline__ void warp_sum_partials2(const float* __restrict__ partials, int nparts, int C, int c, int lane, double& s0, double& s1) {
    double a0 = 0.0, a1 = 0.0, b0 = 0.0, b1 = 0.0;
    const float* base = partials + c;
    const size_t step = (size_t)2 * C;
    for (int b = lane; b < nparts; b += 256) {
        float u[8], v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int bk = b + 32 * k;
            const float* q = base + (size_t)bk * step;
            u[k] = bk < nparts ? (L2 ? __ldcg(q) : *q) : 0.f;
            v[k] = bk < nparts ? (L2 ? __ldcg(q + C) : q[C]) : 0.f;
        }
#pragma unroll
        for (int k = 0; k < 8; k += 2) {
            a0 += (double)u[k];
            b0 += (double)v[k];
            a1 += (double)u[k + 1];
            b1 += (double)v[k + 1];
        }
    }
    double s = a0 + a1, q = b0 + b1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        q += __shfl_xor_sync(0xffffffffu, q, o);
    }
    s0 = s;
    s1 = q;
}

// The finalize of one channel by one warp (also called from the tail of the tensor-core forward kernel).
template <bool L2>
__device__ __forceinline__ void bn_finalize_channel(const float* __restrict__ partials, int nparts, int C, int c, int lane, double M, float eps,
                                                    float momentum, const float* __restrict__ gamma, const float* __restrict__ beta, float* mean,
                                                    float* invstd, float* scale, float* shift, float* rmean, float* rvar, float* sum_out,
                                                    float* sumsq_out) {
    // the per-channel inputs of the last step are requested first so that they arrive while the partials are summed
    const float ga = scale ? gamma[c] : 0.f, be = scale ? beta[c] : 0.f;
    const float rm = rmean ? rmean[c] : 0.f, rv = rmean ? rvar[c] : 0.f;
    double s, q;
    warp_sum_partials2<L2>(partials, nparts, C, c, lane, s, q);
    if (lane == 0) {
        // (this chain sits on the critical path of the forward kernel's tail: one reciprocal serves all divisions by M,
        // and the inverse square root is the library's, accurate to within two units in the last place of fp64)
        const double inv_m = 1.0 / M;
        const double mu = s * inv_m;
        double var = q * inv_m - mu * mu;
        if (var < 0.0) var = 0.0;
        const double is = rsqrt(var + (double)eps);
        if (mean) mean[c] = (float)mu;
        if (invstd) invstd[c] = (float)is;
        if (scale) {
            const double sc = (double)ga * is;
            scale[c] = (float)sc;
            shift[c] = (float)((double)be - mu * sc);
        }
        if (sum_out) sum_out[c] = (float)s;
        if (sumsq_out) sumsq_out[c] = (float)q;
        if (rmean) {
            rmean[c] = (float)((1.0 - (double)momentum) * (double)rm + (double)momentum * mu);
            rvar[c] = (float)((1.0 - (double)momentum) * (double)rv + (double)momentum * var * M / (M - 1.0));
        }
    }
}

// Combine partials [nparts][2][C] and derive the per-channel quantities.  One warp per channel, 8 channels per block.
// Outputs (any may be NULL): mean, invstd, scale = gamma*invstd, shift = beta - mean*scale, raw sums,
// running statistics (in place; unbiased variance, momentum).
__global__ void __launch_bounds__(256) bn_finalize_kernel(const float* __restrict__ partials, int nparts, int C, double M, float eps,
                                                          float momentum, const float* __restrict__ gamma, const float* __restrict__ beta,
                                                          float* mean, float* invstd, float* scale, float* shift, float* rmean, float* rvar,
                                                          float* sum_out, float* sumsq_out) {
    pdl_launch_dependents();
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int c = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (c >= C) return;
    bn_finalize_channel<false>(partials, nparts, C, c, lane, M, eps, momentum, gamma, beta, mean, invstd, scale, shift, rmean, rvar, sum_out, sumsq_out);
}

// V consecutive per-channel floats (V = 4 or 8) with 16-byte loads.
template <int V> __device__ __forceinline__ void load_params(const float* __restrict__ p, int cg, float (&out)[V]) {
    const float4* q = reinterpret_cast<const float4*>(p + (size_t)cg * V);
#pragma unroll
    for (int i = 0; i < V / 4; ++i) {
        const float4 t = q[i];
        out[4 * i] = t.x;
        out[4 * i + 1] = t.y;
        out[4 * i + 2] = t.z;
        out[4 * i + 3] = t.w;
    }
}

template <int V> __device__ __forceinline__ void load_params(const float* __restrict__ p, int cg, float2 (&out)[V / 2]) {  // as pairs
    const float4* q = reinterpret_cast<const float4*>(p + (size_t)cg * V);
#pragma unroll
    for (int i = 0; i < V / 4; ++i) {
        const float4 t = q[i];
        out[2 * i] = make_float2(t.x, t.y);
        out[2 * i + 1] = make_float2(t.z, t.w);
    }
}

// ------------------------------------------------------------------ per-channel sums kept in fp64 accumulators
// The kernel that produces per-channel sums (the convolution's epilogue, the backward reduce pass) adds every block's
// fp32 partial sums to `acc` with fp64 atomics, and every block of the kernel that consumes them (the normalise + SiLU
// pass, the dy pass) reads the totals and derives its coefficients itself.  No block waits for another one: the
// producer needs neither a grid-wide barrier nor a resident grid, and the only ordering is the kernel boundary.
// acc holds `copies` sets of [2][C] doubles (block b adds to set b mod copies, so the cache lines of one set are not
// the target of every block at once).  The sets are zero when the producer starts: the last block of the consumer to
// have read them (counted in *readers) zeroes them again.  Adding a few hundred fp32 values in fp64 is exact unless
// their magnitudes differ by more than 2^20 or so; only then can a total depend on the order in which the atomics land.
// EXACT (the fp32 mode, whose results are the same bits from run to run): integers instead, see below.
struct ChanAcc {
    double* acc;   // NULL: the consumer reads coefficients that a finalize kernel has written
    int* readers;
    int copies;    // (EXACT: EXACT_WORDS for every set, the words of a sum lying where the sets of fp64 sums do)
};

// A sum of fp32 values as a fixed-point number of 64-bit words: word k counts units of 2^(32 k - 149), so that the 24 bits of
// a value fall into words k and k + 1, k its exponent / 32.  Integer additions commute: the words are the same whatever order
// the atomics land in, and the sum has no rounding at all (a word holds 2^31 values).  The last word has a
// bit for either infinity and for NaN.  Against fp64 sums: two atomics per value instead of one, ten words to read instead of
// two or four; measured at exact_apart in nb_cbs.cu (1 to 4 % of a step of up to 60 us, nothing on the smallest and the
// largest).
constexpr int EXACT_DIGITS = 9, EXACT_WORDS = EXACT_DIGITS + 1;
constexpr unsigned long long EXACT_POS_INF = 1, EXACT_NEG_INF = 2, EXACT_NAN = 4;
__device__ __forceinline__ void exact_add(unsigned long long* word, size_t pitch, float v) {
    const unsigned bits = __float_as_uint(v), e = (bits >> 23) & 255u, frac = bits & 0x7fffffu;
    if (e == 255u) {
        atomicOr(word + EXACT_DIGITS * pitch, frac ? EXACT_NAN : bits >> 31 ? EXACT_NEG_INF : EXACT_POS_INF);
        return;
    }
    const unsigned shift = e ? e - 1u : 0u;  // v = (24-bit integer) * 2^(shift - 149)
    const unsigned long long m = (unsigned long long)(e ? frac | 0x800000u : frac) << (shift & 31u);
    const unsigned long long lo = m & 0xffffffffull, hi = m >> 32, sign = bits >> 31 ? ~0ull : 0ull;
    unsigned long long* const w = word + (shift >> 5) * pitch;
    if (lo) atomicAdd(w, (lo ^ sign) - sign);
    if (hi) atomicAdd(w + pitch, (hi ^ sign) - sign);
}
__device__ __forceinline__ double exact_total(const unsigned long long (&w)[EXACT_WORDS]) {
    if (w[EXACT_DIGITS]) {
        const unsigned long long f = w[EXACT_DIGITS];
        return __longlong_as_double(f == EXACT_POS_INF ? 0x7ff0000000000000ll : f == EXACT_NEG_INF ? (long long)0xfff0000000000000ull : 0x7ff8000000000000ll);
    }
    double t = 0.0;
#pragma unroll
    for (int k = 0; k < EXACT_DIGITS; ++k)  // (lowest first; a word below 2^53 converts exactly; most words of a sum are zero)
        if (w[k]) t = fma((double)(long long)w[k], __longlong_as_double((long long)(1023 - 149 + 32 * k) << 52), t);
    return t;
}

template <bool EXACT> __device__ __forceinline__ void chan_acc_add(const ChanAcc& ca, int C, int which, int c, float v) {
    if (EXACT) {
        const size_t set = (size_t)((int)blockIdx.x % (ca.copies / EXACT_WORDS)) * EXACT_WORDS;
        exact_add(reinterpret_cast<unsigned long long*>(ca.acc) + (set * 2 + which) * C + c, (size_t)2 * C, v);
    }
    else atomicAdd(ca.acc + ((size_t)((int)blockIdx.x % ca.copies) * 2 + which) * C + c, (double)v);
}
// f(c, first total, second total, load(c)) for every channel (EXACT), by the threads of a block, or (CLEAR) of the grid, which
// then leave the words zero: two neighbouring lanes take a channel's two sums, whatever load reads and all words of a set
// requested before the first is used, and the even one calls f.
template <bool CLEAR, class Load, class F> __device__ __forceinline__ void exact_totals(const ChanAcc& ca, int C, Load load, F f) {
    const int threads = (int)blockDim.x & ~1;  // (whole pairs)
    if ((int)threadIdx.x >= threads) return;
#pragma unroll 1
    for (int i = (int)threadIdx.x + (CLEAR ? (int)blockIdx.x * threads : 0); i < 2 * C; i += threads * (CLEAR ? (int)gridDim.x : 1)) {
        const int c = i >> 1, which = i & 1;
        unsigned long long* const base = reinterpret_cast<unsigned long long*>(ca.acc) + (size_t)which * C + c;
        const auto prm = load(c);
        unsigned long long w[EXACT_WORDS];
#pragma unroll
        for (int k = 0; k < EXACT_WORDS; ++k) w[k] = __ldcg(base + (size_t)k * 2 * C);
        for (int set = EXACT_WORDS; set < ca.copies; set += EXACT_WORDS) {
#pragma unroll
            for (int k = 0; k < EXACT_WORDS; ++k) {
                const unsigned long long more = __ldcg(base + (size_t)(set + k) * 2 * C);
                w[k] = k == EXACT_DIGITS ? w[k] | more : w[k] + more;
            }
        }
        const double mine = exact_total(w), other = __shfl_xor_sync(3u << (threadIdx.x & 30u), mine, 1);
        if (!which) f(c, mine, other, prm);
        if (CLEAR)
            for (int k = 0; k < ca.copies; ++k) base[(size_t)k * 2 * C] = 0ull;
    }
}
// totals of channels c and c + 1 (c even) of both sums; read from L2, where the atomics were performed, with the loads
// of four sets in flight at a time (the consuming pass starts with this latency)
__device__ __forceinline__ void chan_acc_total2(const ChanAcc& ca, int C, int c, double2& t0, double2& t1) {
    t0 = t1 = make_double2(0.0, 0.0);
    const size_t set = (size_t)2 * C;
    const double* base = ca.acc + c;
    int k = 0;
    for (; k + 4 <= ca.copies; k += 4) {
        double2 a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            a[i] = __ldcg(reinterpret_cast<const double2*>(base + (k + i) * set));
            b[i] = __ldcg(reinterpret_cast<const double2*>(base + (k + i) * set + C));
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            t0.x += a[i].x; t0.y += a[i].y;
            t1.x += b[i].x; t1.y += b[i].y;
        }
    }
    for (; k < ca.copies; ++k) {
        const double2 a = __ldcg(reinterpret_cast<const double2*>(base + k * set)), b = __ldcg(reinterpret_cast<const double2*>(base + k * set + C));
        t0.x += a.x; t0.y += a.y;
        t1.x += b.x; t1.y += b.y;
    }
}
// One thread per block, after the block's reads of acc (and a block-level barrier): returns the number of blocks that
// had read before this one.  The value is needed only at the end of the kernel.  No fence: the block's reads have
// delivered their values (they were used before the barrier), and the zeroes are written only by the block that sees
// every other block's increment.
__device__ __forceinline__ int chan_acc_reader_arrive(const ChanAcc& ca) { return atomicAdd(ca.readers, 1); }
// All threads of the block, `last` block-uniform: the last reader leaves the sets and the counter zeroed.
__device__ __forceinline__ void chan_acc_reset_if(const ChanAcc& ca, int C, bool last) {
    if (!last) return;
    const int n = ca.copies * 2 * C;
    for (int i = threadIdx.x; i < n; i += blockDim.x) ca.acc[i] = 0.0;
    if (threadIdx.x == 0) *ca.readers = 0;
}

// 1/sqrt(v) for v well inside the fp32 range: the fp32 approximation refined by one Newton step in fp64 (relative error
// below 2^-44, i.e. exact once rounded to fp32 but for values within 2^-20 units in the last place of a rounding
// boundary).  The library's fp64 rsqrt is a chain three times as long, and every block of the consuming pass waits for it.
__device__ __forceinline__ double rsqrt_refined(double v) {
    const float vf = (float)v;
    if (!(vf > 1e-30f && vf < 1e30f)) return rsqrt(v);
    const double r = (double)rsqrtf(vf);
    const double e = fma(-(v * r), r, 1.0);
    return fma(0.5 * r, e, r);
}

// What a block of the normalise + SiLU pass needs to turn the totals (sum y, sum y^2) into scale and shift; block 0
// also writes the batch statistics and updates the running ones (the same fp64 chain as bn_finalize_channel).
struct FwdFin {
    double inv_m, unbias;  // 1/M and M/(M-1)
    float eps, momentum;
    const float *gamma, *beta;
    float *mean, *invstd, *rmean, *rvar;
};
__device__ __forceinline__ void fwd_coef_channel(const FwdFin& f, int c, double s, double q, float ga, float be, bool writer, float& scale, float& shift) {
    const double mu = s * f.inv_m;
    double var = q * f.inv_m - mu * mu;
    if (var < 0.0) var = 0.0;
    const double is = rsqrt_refined(var + (double)f.eps);
    const double sc = (double)ga * is;
    scale = (float)sc;
    shift = (float)((double)be - mu * sc);
    if (writer) {
        f.mean[c] = (float)mu;
        f.invstd[c] = (float)is;
        if (f.rmean) {
            f.rmean[c] = (float)((1.0 - (double)f.momentum) * (double)f.rmean[c] + (double)f.momentum * mu);
            f.rvar[c] = (float)((1.0 - (double)f.momentum) * (double)f.rvar[c] + (double)f.momentum * var * f.unbias);
        }
    }
}
template <bool EXACT> __device__ __forceinline__ void fwd_coef_from_acc(const ChanAcc& ca, const FwdFin& f, int C, float* s_coef /*[2][C] shared*/) {
    const bool writer = blockIdx.x == 0;
    auto channel = [&](int c, double s, double q, float ga, float be) { fwd_coef_channel(f, c, s, q, ga, be, writer, s_coef[c], s_coef[C + c]); };
    if constexpr (EXACT) {
        exact_totals<false>(ca, C, [&](int c) { return make_float2(f.gamma[c], f.beta[c]); },
                     [&](int c, double s, double q, float2 p) { channel(c, s, q, p.x, p.y); });
    } else {
        // two channels per thread and round (kept rolled: the fp64 chains must not crowd the registers of the streaming loop)
#pragma unroll 1
        for (int c = 2 * (int)threadIdx.x; c < C; c += 2 * (int)blockDim.x) {
            const float2 ga = *reinterpret_cast<const float2*>(f.gamma + c), be = *reinterpret_cast<const float2*>(f.beta + c);
            double2 s, q;
            chan_acc_total2(ca, C, c, s, q);
            channel(c, s.x, q.x, ga.x, be.x);
            channel(c + 1, s.y, q.y, ga.y, be.y);
        }
    }
}
template <int V> __device__ __forceinline__ void load_params_shared(const float* s, int cg, float2 (&out)[V / 2]) {
    const float4* q = reinterpret_cast<const float4*>(s + (size_t)cg * V);
#pragma unroll
    for (int i = 0; i < V / 4; ++i) {
        const float4 t = q[i];
        out[2 * i] = make_float2(t.x, t.y);
        out[2 * i + 1] = make_float2(t.z, t.w);
    }
}

// ------------------------------------------------------------------ a = SiLU(y*scale + shift)  (ACT = false: no SiLU)
// RES: a = SiLU(...) + res with res a (possibly pitched) tensor of the output's type -- the residual connection of a
// bottleneck performed by the block that feeds it; the sum is formed in fp32 and rounded once.
// FIN: scale and shift are derived here from the totals in `ca` (dynamic shared memory: 2*C floats); else they are read.
// ONE (with FIN): the grid has a thread for every vector.  The thread asks for its vector before the coefficients are
// derived, so that the two memory latencies of a small tensor's pass overlap (with more vectors per thread the registers
// that stay live across the fp64 arithmetic cost more than that).
template <typename YT, typename AT, bool FAST, bool ACT = true, bool PITCHED = false, bool RES = false, bool FIN = false, bool ONE = false>
__global__ void __launch_bounds__(288, 3) bn_silu_apply_kernel(const YT* __restrict__ y, AT* __restrict__ a,
                                                             long long total_vecs, int C, const float* __restrict__ scale,
                                                             const float* __restrict__ shift, long long ld_a, const AT* __restrict__ res, long long ld_r,
                                                             ChanAcc ca, FwdFin fin) {
    pdl_launch_dependents();
    pdl_wait();
    constexpr int V = Vec16<YT>::N;
    static_assert(V == Vec16<AT>::N, "y and a must have the same element size");
    const int cg = threadIdx.x % (C / V);
    float2 sc[V / 2], sh[V / 2];
    extern __shared__ __align__(16) float s_coef[];
    __shared__ int s_last;
    int readers_before = 0;
    Vec16<YT> q1;
    Vec16<AT> r1;
    if (ONE) {
        const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
        if (v < total_vecs) {
            q1 = ld16(y + v * V);
            if (RES) r1 = ld16(res + (v / (C / V)) * ld_r + (long long)cg * V);
        }
    }
    if (FIN) {
        fwd_coef_from_acc<std::is_same<YT, float>::value>(ca, fin, C, s_coef);
        __syncthreads();
        if (threadIdx.x == 0) readers_before = chan_acc_reader_arrive(ca);
        load_params_shared<V>(s_coef, cg, sc);
        load_params_shared<V>(s_coef + C, cg, sh);
    } else {
        load_params<V>(scale, cg, sc);
        load_params<V>(shift, cg, sh);
    }
    const long long stride = (long long)gridDim.x * blockDim.x;
    // a may be a channel slice of a wider tensor: row pitch ld_a elements (the stride is a whole number of rows, so the
    // output offset advances by a constant)
    const int cgs = C / V;
    const long long v0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long oa = PITCHED ? (v0 / cgs) * ld_a + (long long)cg * V : v0 * V;  // (dense: the flat offset, no division)
    const long long oa_step = PITCHED ? (stride / cgs) * ld_a : stride * V;
    long long orr = RES ? (v0 / cgs) * ld_r + (long long)cg * V : 0;
    const long long or_step = RES ? (stride / cgs) * ld_r : 0;
    // A thread's next vector is on its way while this one is worked on, and an L2 prefetch two steps ahead of that.  Measured (forward
    // call, without / with): 96 -> 96 1x1 on 16 x 160 x 160 pixels 70.5 / 67.1 us, 192 -> 192 on 16 x 80 x 80 38.5 / 36.8, 384 -> 384
    // on 16 x 40 x 40 25.9 / 25.0; 157 MB tensors the same.  (The dy pass has no registers left for it: 101 -> 125 us.)
    if (!ONE && v0 < total_vecs) q1 = ld16(y + v0 * V);
    for (long long v = v0; v < total_vecs; v += stride, oa += oa_step, orr += or_step) {
        const Vec16<YT> q = q1;
        if (!ONE && v + 3 * stride < total_vecs) asm volatile("prefetch.global.L2 [%0];" ::"l"(y + (v + 3 * stride) * V));
        if (!ONE && v + stride < total_vecs) q1 = ld16(y + (v + stride) * V);
        Vec16<AT> o, r;
        if (RES) r = ONE ? r1 : ld16(res + orr);
#pragma unroll
        for (int j = 0; j < V / 2; ++j) {
            const float2 z = fma2(pair_to_f32(q.v + 2 * j), sc[j], sh[j]);
            float2 out = ACT ? mul2(z, sigmoid2<FAST>(z)) : z;
            if (RES) out = add2(out, pair_to_f32(r.v + 2 * j));
            pair_from_f32(o.v + 2 * j, out);
        }
        st16(a + oa, o);
        if (ONE) break;
    }
    if (FIN) {
        if (threadIdx.x == 0) s_last = readers_before == (int)gridDim.x - 1;
        __syncthreads();
        chan_acc_reset_if(ca, C, s_last != 0);
    }
}

// ------------------------------------------------------------------ evaluation-mode coefficients and BN folding
// scale_c = gamma_c / sqrt(rvar_c + eps), shift_c = beta_c - rmean_c*scale_c (fp64 arithmetic, like the training-mode
// finalize).  gamma NULL: scale 1; rmean NULL: no normalisation (shift = beta, or 0 when beta is NULL too).
__device__ __forceinline__ void bn_eval_coef(const float* gamma, const float* beta, const float* rmean, const float* rvar, float eps, int c, double& sc,
                                             double& sh) {
    sc = gamma ? (double)gamma[c] : 1.0;
    sh = beta ? (double)beta[c] : 0.0;
    if (rmean) {
        sc /= sqrt((double)rvar[c] + (double)eps);
        sh -= (double)rmean[c] * sc;
    }
}
__global__ void __launch_bounds__(256) bn_eval_coef_kernel(const float* __restrict__ gamma, const float* __restrict__ beta, const float* __restrict__ rmean,
                                                           const float* __restrict__ rvar, float eps, int C, float* __restrict__ scale,
                                                           float* __restrict__ shift) {
    pdl_launch_dependents();
    pdl_wait();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    double sc, sh;
    bn_eval_coef(gamma, beta, rmean, rvar, eps, c, sc, sh);
    scale[c] = (float)sc;
    shift[c] = (float)sh;
}
// Folded filter w'[co][t] = scale_co * w[co][t] (rounded to WT once) and bias'[co] = shift_co; K = taps per output channel.
template <typename WT>
__global__ void __launch_bounds__(256) bn_fold_kernel(const WT* __restrict__ w, long long K, int C, const float* __restrict__ gamma,
                                                      const float* __restrict__ beta, const float* __restrict__ rmean, const float* __restrict__ rvar,
                                                      float eps, WT* __restrict__ w_folded, float* __restrict__ bias_folded) {
    pdl_launch_dependents();
    pdl_wait();
    const long long total = (long long)C * K;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int co = (int)(i / K);
        double sc, sh;
        bn_eval_coef(gamma, beta, rmean, rvar, eps, co, sc, sh);
        w_folded[i] = from_f32<WT>((float)((double)to_f32(w[i]) * sc));
        if (i - (long long)co * K == 0) bias_folded[co] = (float)sh;
    }
}

// partials [nparts][2][C] (sum dz, sum dz*y) -> dbeta, dgamma (fp32) and four per-channel coefficients for the dy pass:
//   coef[0] = a = gamma*invstd, coef[1] = b = beta - mean*a                      (z = y*a + b)
//   coef[2] = p1 = a*invstd*dgamma/M, coef[3] = p0 = p1*mean - a*dbeta/M        (dy = a*dz - p1*y + p0)
// which is dy = a*(dz - dbeta/M - xhat*dgamma/M) with xhat = (y - mean)*invstd written out in terms of y.
template <bool L2>
__device__ __forceinline__ void bn_bwd_finalize_channel(const float* __restrict__ partials, int nparts, int C, int c, int lane, double M,
                                                        const float* __restrict__ mean, const float* __restrict__ invstd,
                                                        const float* __restrict__ gamma, const float* __restrict__ beta, float* dgamma, float* dbeta,
                                                        float* coef /*[4][C]*/) {
    const float mu_f = mean[c], is_f = invstd[c], ga = gamma[c], be = beta[c];  // requested before the partials are summed
    double s0, s1;
    warp_sum_partials2<L2>(partials, nparts, C, c, lane, s0, s1);
    if (lane == 0) {
        const double mu = (double)mu_f, is = (double)is_f;
        const double inv_m = 1.0 / M;
        const double dg = is * (s1 - mu * s0);
        const double a = (double)ga * is;
        const double p1 = a * is * dg * inv_m;
        dbeta[c] = (float)s0;
        dgamma[c] = (float)dg;
        coef[c] = (float)a;
        coef[C + c] = (float)((double)be - mu * a);
        coef[2 * C + c] = (float)p1;
        coef[3 * C + c] = (float)(p1 * mu - a * s0 * inv_m);
    }
}

// ------------------------------------------------------------------ backward reductions: sum dz, sum dz*y
// z = y*a + b with a = gamma*invstd, b = beta - mean*a (recomputed here from the saved statistics).  The second
// sum is taken against y itself; sum dz*xhat = invstd*(sum dz*y - mean*sum dz) is formed in fp64 by the finalize
// kernel, so this pass needs only two per-channel values per element.
// Extras of the reduce kernel: with acc.acc != NULL the block sums go to the fp64 accumulators (and `partials` is not
// written); w / wt: filter and its rearranged copy for the data-gradient GEMM (wt = NULL: nothing to rearrange), work
// that the blocks of this kernel carry along because the memory latency of a few filter tiles costs them nothing.
struct BwdFused {
    ChanAcc acc;
    const __nv_bfloat16* w;
    __nv_bfloat16* wt;
};
// `row_blocks` blocks walk the tensor (the sums are grouped by them); blocks past those only rearrange filter tiles.
// DEEP: for tensors whose threads have at most eight vectors each and whose blocks are all resident: all vectors are on their way
// before the parameters are used (a small tensor's pass is one memory latency per step of this loop), with the registers that
// takes; the additions and their order are the same.  1: up to one block an SM.  2: up to two of at most 256 threads, so at most
// 128 registers: the bf16 form takes 129 with indices of 64 bits and 128 with indices of 32 (the tensor has fewer than 2^20 vectors).
// A launch bound that forces the count costs 0.2 to 0.3 us a call, since the compiler then asks for some of the vectors later.
// Up to one block an SM the second block's room does harm: blocks become resident while the pass before still runs, wherever it leaves
// room, and pile up two to an SM beside idle ones.  Form 1 / 2 in bf16, us a step: 72 -> 136 3x3 on 3 x 53 x 75 pixels (100 blocks)
// 55.1 / 57.6, 192 -> 192 3x3 on 4 x 40 x 40 (80) 43.5 / 45.4.  (Form 2 with half an SM's shared memory, one block an SM by that:
// 55.2 and 43.5, but then no block fits beside a weight gradient's: detector iteration at batch 2, 320 x 320 2036 -> 2044 us.)
template <typename YT, typename AT, bool FAST, bool PITCHED = false, int DEEP = 0>
__global__ void __launch_bounds__(288, DEEP ? 1 : 3) bn_silu_bwd_reduce_kernel(const AT* __restrict__ g, const YT* __restrict__ y,
                                                                  long long total_vecs, int C, const float* __restrict__ mean,
                                                                  const float* __restrict__ invstd, const float* __restrict__ gamma,
                                                                  const float* __restrict__ beta, float* __restrict__ partials, BwdFused fb,
                                                                  WtParams wtp, long long ld_g, int row_blocks) {
    pdl_launch_dependents();
    pdl_wait();
    constexpr int V = Vec16<YT>::N;
    static_assert(V == Vec16<AT>::N, "g and y must have the same element size");
    extern __shared__ __align__(16) float red[];
    const int tid = threadIdx.x;
    const int cgs = C / V;
    const int cg = tid % cgs;
    // The first two filter tiles of this block (for the data-gradient GEMM's rearranged filter) are requested now with
    // cp.async and written back after the streaming loop, so their memory latency costs nothing.
    __shared__ __align__(16) WtTileBuf wtile[2];
    const int wt_tiles = fb.wt ? wt_num_tiles(wtp) : 0;
    if (wt_tiles > 0) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int t = (int)blockIdx.x + k * (int)gridDim.x;
            if (t < wt_tiles) wt_tile_load_async(fb.w, wtp, wt_tile_decode(wtp, t), wtile[k]);
        }
    }
    const bool has_rows = (int)blockIdx.x < row_blocks;
    const long long stride = (long long)row_blocks * blockDim.x;
    // g may be a channel slice of a wider tensor (row pitch ld_g elements); the stride is a whole number of rows
    const long long v0 = (long long)blockIdx.x * blockDim.x + tid;
    long long og = PITCHED ? (v0 / cgs) * ld_g + (long long)cg * V : v0 * V;  // (dense: the flat offset)
    const long long og_step = PITCHED ? (stride / cgs) * ld_g : stride * V;
    constexpr int D = DEEP ? 8 : 1;
    Vec16<YT> qyd[D];
    Vec16<AT> qgd[D];
    using Index = std::conditional_t<DEEP == 2, int, long long>;
    const Index first = (Index)v0, step = (Index)stride, total = (Index)total_vecs;
    if (DEEP && has_rows) {
#pragma unroll
        for (int u = 0; u < D; ++u)
            if (first + u * step < total) {
                qyd[u] = ld16(y + (first + u * step) * V);
                qgd[u] = ld16(PITCHED || DEEP == 1 ? g + og + u * og_step : g + (first + u * step) * V);
            }
    }
    float2 a[V / 2], b[V / 2], sb[V / 2], sy[V / 2];
    {
        float mu[V], is[V], ga[V], be[V];
        load_params<V>(mean, cg, mu);
        load_params<V>(invstd, cg, is);
        load_params<V>(gamma, cg, ga);
        load_params<V>(beta, cg, be);
#pragma unroll
        for (int j = 0; j < V / 2; ++j) {
            a[j] = make_float2(ga[2 * j] * is[2 * j], ga[2 * j + 1] * is[2 * j + 1]);
            b[j] = make_float2(fmaf(-mu[2 * j], a[j].x, be[2 * j]), fmaf(-mu[2 * j + 1], a[j].y, be[2 * j + 1]));
            sb[j] = sy[j] = splat2(0.f);
        }
    }
    auto add_vec = [&](const Vec16<YT>& qy, const Vec16<AT>& qg) {
#pragma unroll
        for (int j = 0; j < V / 2; ++j) {
            const float2 yv = pair_to_f32(qy.v + 2 * j);
            const float2 dz = silu_bwd_dz2<FAST>(fma2(yv, a[j], b[j]), pair_to_f32(qg.v + 2 * j));
            sb[j] = add2(sb[j], dz);
            sy[j] = fma2(dz, yv, sy[j]);
        }
    };
    if (DEEP) {
        if (has_rows) {
#pragma unroll
            for (int u = 0; u < D; ++u)
                if (first + u * step < total) add_vec(qyd[u], qgd[u]);
        }
    } else {
        uint4* const ring = reinterpret_cast<uint4*>(red) + tid;  // [EW_RING][2][blockDim.x] vectors, in the space of the block's reduction below
        const int tpb = blockDim.x;
        long long vn = v0, ogn = og;  // the next vectors to request
        auto request = [&](int slot) {
            if (has_rows && vn < total_vecs) {
                ew_copy16(ring + (2 * slot) * tpb, y + vn * V);
                ew_copy16(ring + (2 * slot + 1) * tpb, g + ogn);
            }
            ew_commit();
            vn += stride;
            ogn += og_step;
        };
#pragma unroll
        for (int u = 0; u < EW_RING; ++u) request(u);
        int slot = 0;
        for (long long v = v0; has_rows && v < total_vecs; v += stride) {
            ew_wait();
            Vec16<YT> qy;
            Vec16<AT> qg;
            *reinterpret_cast<uint4*>(&qy) = ring[(2 * slot) * tpb];
            *reinterpret_cast<uint4*>(&qg) = ring[(2 * slot + 1) * tpb];
            request(slot);
            slot = slot + 1 == EW_RING ? 0 : slot + 1;
            add_vec(qy, qg);
        }
        __syncthreads();  // every thread is done with its slots
    }
    const int R = blockDim.x / cgs;
    if (has_rows) {  // both sums of every channel at once: red holds [2][blockDim.x][V]
        float* const red1 = red + (size_t)blockDim.x * V;
#pragma unroll
        for (int j = 0; j < V / 2; ++j) {
            *reinterpret_cast<float2*>(&red[tid * V + 2 * j]) = sb[j];
            *reinterpret_cast<float2*>(&red1[tid * V + 2 * j]) = sy[j];
        }
        __syncthreads();
        for (int e = tid; e < 2 * C; e += blockDim.x) {
            const int pass = e >= C ? 1 : 0, c = e - pass * C;  // pass 0: sum dz, pass 1: sum dz*y
            const float* const src = (pass ? red1 : red) + c;  // element c of row r: ((r * cgs + c / V) * V + c % V) = r * C + c
            float acc = 0.f;
            for (int r = 0; r < R; ++r) acc += src[r * C];
            if (fb.acc.acc) chan_acc_add<std::is_same<YT, float>::value>(fb.acc, C, pass, c, acc);
            else partials[((size_t)blockIdx.x * 2 + pass) * C + c] = acc;
        }
    }
    if (wt_tiles > 0) {
        wt_async_wait();
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int t = (int)blockIdx.x + k * (int)gridDim.x;
            if (t < wt_tiles) wt_tile_store(fb.wt, wtp, wt_tile_decode(wtp, t), wtile[k]);
        }
        if (wt_tiles > 2 * (int)gridDim.x) wt_transform_blocks(fb.w, fb.wt, wtp, (int)blockIdx.x, (int)gridDim.x, 2);  // rare: very large filters
    }
}

__global__ void __launch_bounds__(256) bn_bwd_finalize_kernel(const float* __restrict__ partials, int nparts, int C, double M,
                                                              const float* __restrict__ mean, const float* __restrict__ invstd,
                                                              const float* __restrict__ gamma, const float* __restrict__ beta,
                                                              float* dgamma, float* dbeta, float* coef /*[4][C]*/, int fin_blocks,
                                                              const __nv_bfloat16* __restrict__ w, __nv_bfloat16* __restrict__ wt, WtParams wtp) {
    pdl_launch_dependents();
    pdl_wait();
    // Blocks past the first `fin_blocks` rearrange the filter for the data-gradient GEMM that follows this call's dy pass
    // (independent work that fills the otherwise idle GPU while the short finalize chain runs).
    if ((int)blockIdx.x >= fin_blocks) {
        wt_transform_blocks(w, wt, wtp, (int)blockIdx.x - fin_blocks, (int)gridDim.x - fin_blocks);
        return;
    }
    const int lane = threadIdx.x & 31;
    const int c = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (c >= C) return;
    bn_bwd_finalize_channel<false>(partials, nparts, C, c, lane, M, mean, invstd, gamma, beta, dgamma, dbeta, coef);
}

// ------------------------------------------------------------------ dy = a*dz - p1*y + p0
// What a block of the dy pass needs to turn the totals (sum dz, sum dz*y) into its four coefficients; block 0 also
// writes dgamma and dbeta (the same fp64 chain as bn_bwd_finalize_channel).
struct BwdFin {
    double inv_m;
    const float *mean, *invstd, *gamma, *beta;
    float *dgamma, *dbeta;
};
struct BwdCoef {
    float a, b, p1, p0, dgamma;
};
__device__ __forceinline__ BwdCoef bwd_coef_channel(float mu_f, float is_f, float ga, float be, double s0, double s1, double inv_m) {
    const double mu = (double)mu_f, is = (double)is_f;
    const double dg = is * (s1 - mu * s0);
    const double a = (double)ga * is;
    const double p1 = a * is * dg * inv_m;
    return {(float)a, (float)((double)be - mu * a), (float)p1, (float)(p1 * mu - a * s0 * inv_m), (float)dg};
}
template <bool EXACT> __device__ __forceinline__ void bwd_coef_from_acc(const ChanAcc& ca, const BwdFin& f, int C, float* s_coef /*[4][C] shared*/) {
    const bool writer = blockIdx.x == 0;
    auto channel = [&](int c, double s0, double s1, float mu, float is, float ga, float be) {
        const BwdCoef k = bwd_coef_channel(mu, is, ga, be, s0, s1, f.inv_m);
        s_coef[c] = k.a;
        s_coef[C + c] = k.b;
        s_coef[2 * C + c] = k.p1;
        s_coef[3 * C + c] = k.p0;
        if (writer) {
            f.dbeta[c] = (float)s0;
            f.dgamma[c] = k.dgamma;
        }
    };
    if constexpr (EXACT) {
        exact_totals<false>(ca, C, [&](int c) { return make_float4(f.mean[c], f.invstd[c], f.gamma[c], f.beta[c]); },
                     [&](int c, double s0, double s1, float4 p) { channel(c, s0, s1, p.x, p.y, p.z, p.w); });
    } else {
#pragma unroll 1
        for (int c = 2 * (int)threadIdx.x; c < C; c += 2 * (int)blockDim.x) {  // two channels per thread and round, see fwd_coef_from_acc
            const float2 mu_f = *reinterpret_cast<const float2*>(f.mean + c), is_f = *reinterpret_cast<const float2*>(f.invstd + c);
            const float2 ga = *reinterpret_cast<const float2*>(f.gamma + c), be = *reinterpret_cast<const float2*>(f.beta + c);
            double2 t0, t1;
            chan_acc_total2(ca, C, c, t0, t1);
            channel(c, t0.x, t1.x, mu_f.x, is_f.x, ga.x, be.x);
            channel(c + 1, t0.y, t1.y, mu_f.y, is_f.y, ga.y, be.y);
        }
    }
}
// The coefficients of an EXACT plan whose words are too many for every block of the consuming pass to read (see exact_apart in
// nb_cbs.cu): by a kernel of their own, forward and backward, which leaves the words zero.
__global__ void __launch_bounds__(128) bn_exact_finalize_kernel(ChanAcc ca, int C, FwdFin f, float* __restrict__ scale, float* __restrict__ shift) {
    pdl_launch_dependents();
    pdl_wait();
    exact_totals<true>(ca, C, [&](int c) { return make_float2(f.gamma[c], f.beta[c]); },
                       [&](int c, double s, double q, float2 p) { fwd_coef_channel(f, c, s, q, p.x, p.y, true, scale[c], shift[c]); });
}
__global__ void __launch_bounds__(128) bn_exact_bwd_finalize_kernel(ChanAcc ca, int C, BwdFin f, float* __restrict__ coef /*[4][C]*/) {
    pdl_launch_dependents();
    pdl_wait();
    exact_totals<true>(ca, C, [&](int c) { return make_float4(f.mean[c], f.invstd[c], f.gamma[c], f.beta[c]); },
                       [&](int c, double s0, double s1, float4 p) {
                           const BwdCoef k = bwd_coef_channel(p.x, p.y, p.z, p.w, s0, s1, f.inv_m);
                           coef[c] = k.a;
                           coef[C + c] = k.b;
                           coef[2 * C + c] = k.p1;
                           coef[3 * C + c] = k.p0;
                           f.dbeta[c] = (float)s0;
                           f.dgamma[c] = k.dgamma;
                       });
}
// FIN: the coefficients are derived here from the totals in `ca` (dynamic shared memory: 4*C floats); else read from coef.
// GRES: the incoming gradient g is also the gradient of a residual connection's shortcut: the pass adds it to (or, with
// gres_add = 0, copies it into) `gres`, a tensor of g's shape with pixels ld_gres elements apart -- the backward
// counterpart of the RES form of the normalise + SiLU pass (fp32 sum, rounded once, like a separate accumulation pass).
// ONE (with FIN): a thread for every vector, asked for before the coefficients are derived (see the normalise + SiLU pass).
template <typename YT, typename AT, bool FAST, bool PITCHED = false, bool FIN = false, bool GRES = false, bool ONE = false>
__global__ void __launch_bounds__(288, 3) bn_silu_bwd_dy_kernel(const AT* __restrict__ g, const YT* __restrict__ y,
                                                              AT* __restrict__ dy, long long total_vecs, int C,
                                                              const float* __restrict__ coef, long long ld_g, ChanAcc ca, BwdFin fin,
                                                              AT* __restrict__ gres, long long ld_gres, int gres_add) {
    pdl_launch_dependents();
    pdl_wait();
    constexpr int V = Vec16<YT>::N;
    const int cg = threadIdx.x % (C / V);
    float2 a[V / 2], b[V / 2], np1[V / 2], p0[V / 2];
    extern __shared__ __align__(16) float s_coef[];
    __shared__ int s_last;
    int readers_before = 0;
    Vec16<YT> qy1;
    Vec16<AT> qg1;
    if (ONE) {
        const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
        if (v < total_vecs) {
            qy1 = ld16(y + v * V);
            qg1 = ld16(g + (PITCHED ? (v / (C / V)) * ld_g + (long long)cg * V : v * V));
        }
    }
    if (FIN) {
        bwd_coef_from_acc<std::is_same<YT, float>::value>(ca, fin, C, s_coef);
        __syncthreads();
        if (threadIdx.x == 0) readers_before = chan_acc_reader_arrive(ca);
        load_params_shared<V>(s_coef, cg, a);
        load_params_shared<V>(s_coef + C, cg, b);
        load_params_shared<V>(s_coef + 2 * C, cg, np1);
        load_params_shared<V>(s_coef + 3 * C, cg, p0);
    } else {
        load_params<V>(coef, cg, a);
        load_params<V>(coef + C, cg, b);
        load_params<V>(coef + 2 * C, cg, np1);
        load_params<V>(coef + 3 * C, cg, p0);
    }
#pragma unroll
    for (int j = 0; j < V / 2; ++j) np1[j] = make_float2(-np1[j].x, -np1[j].y);
    const long long stride = (long long)gridDim.x * blockDim.x;
    const int cgs = C / V;
    const long long v0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long og = PITCHED ? (v0 / cgs) * ld_g + (long long)cg * V : v0 * V;  // g may be a channel slice (row pitch ld_g), see the reduce kernel
    const long long og_step = PITCHED ? (stride / cgs) * ld_g : stride * V;
    long long ogr = GRES ? (v0 / cgs) * ld_gres + (long long)cg * V : 0;
    const long long ogr_step = GRES ? (stride / cgs) * ld_gres : 0;
    for (long long v = v0; v < total_vecs; v += stride, og += og_step, ogr += ogr_step) {
        if (!ONE && v + 2 * stride < total_vecs) {  // L2 prefetch two iterations ahead (see the reduce kernel)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(y + (v + 2 * stride) * V));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(g + og + 2 * og_step));
        }
        const Vec16<YT> qy = ONE ? qy1 : ld16(y + v * V);
        const Vec16<AT> qg = ONE ? qg1 : ld16(g + og);
        if (GRES) {
            Vec16<AT> r = qg;
            if (gres_add) {
                const Vec16<AT> old = ld16(gres + ogr);
#pragma unroll
                for (int j = 0; j < V / 2; ++j) pair_from_f32(r.v + 2 * j, add2(pair_to_f32(old.v + 2 * j), pair_to_f32(qg.v + 2 * j)));
            }
            st16(gres + ogr, r);
        }
        Vec16<AT> o;
#pragma unroll
        for (int j = 0; j < V / 2; ++j) {
            const float2 yv = pair_to_f32(qy.v + 2 * j);
            const float2 dz = silu_bwd_dz2<FAST>(fma2(yv, a[j], b[j]), pair_to_f32(qg.v + 2 * j));
            pair_from_f32(o.v + 2 * j, fma2(a[j], dz, fma2(np1[j], yv, p0[j])));
        }
        st16(dy + v * V, o);
        if (ONE) break;
    }
    if (FIN) {
        if (threadIdx.x == 0) s_last = readers_before == (int)gridDim.x - 1;
        __syncthreads();
        chan_acc_reset_if(ca, C, s_last != 0);
    }
}

// ------------------------------------------------------------------ both backward passes in one launch, for small tensors
// Where the reduction's threads have at most eight vectors each and few blocks, the two passes are two memory latencies, a
// launch and a trip of the sums through the fp64 accumulators, with nothing busy.  Here g and y stay in registers between
// them and the sums travel through distributed shared memory: the channels are cut into `slabs` (clusters of at most eight
// CTAs that need nothing from one another), and CTA q of a slab's cluster does the slab's share of the `units` row blocks
// from q * units on.  The additions and their grouping in fp32 are those of the reduce kernel, the block sums are added in
// fp64 as there, and dz is computed anew from the same coefficients as in the dy kernel, so the results are too.
// CTAs past the slabs rearrange filter tiles.
// Bound: latency (loads, two cluster barriers, the fp64 chain of a channel).  Measured (step): 336 -> 392 3x3 on 21 x 18 pixels
// 46.0 -> 43.5 us, 248 -> 208 3x3 on 60 x 19 48.1 -> 46.2, 16 -> 32 3x3 on 4 x 13 x 82 27.5 -> 26.7; more at e.slabs in nb_cbs.cu.
__device__ __forceinline__ double ld_dsmem_f64(uint32_t cluster_addr) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(cluster_addr) : "memory");
    return v;
}
// Dynamic shared memory: fp64 sums [2][wc], coefficients [4][wc], then red [2][threads * V] and part [2][units][wc].
// wc: channels of a slab, units: row blocks of a CTA, threads of a CTA
inline size_t bwd_small_smem(int wc, int units, int threads, int vec) { return (size_t)wc * 32 + ((size_t)2 * threads * vec + 2 * units * wc) * 4; }
template <typename YT, typename AT, bool FAST, bool PITCHED, bool GRES>
__global__ void __launch_bounds__(288, 1) bn_silu_bwd_small_kernel(const AT* __restrict__ g, const YT* __restrict__ y, AT* __restrict__ dy, long long rows,
                                                                   int C, BwdFin fin, const __nv_bfloat16* __restrict__ w, __nv_bfloat16* __restrict__ wt,
                                                                   WtParams wtp, long long ld_g, AT* __restrict__ gres, long long ld_gres, int gres_add,
                                                                   int slabs, int units, int cluster, int row_blocks) {
    pdl_launch_dependents();
    pdl_wait();
    const int slab = (int)blockIdx.x / cluster, q = (int)blockIdx.x % cluster;
    if (slab >= slabs) {
        wt_transform_blocks(w, wt, wtp, (int)blockIdx.x - slabs * cluster, (int)gridDim.x - slabs * cluster);
        return;
    }
    constexpr int V = Vec16<YT>::N, D = 8;
    static_assert(V == Vec16<AT>::N, "g and y must have the same element size");
    extern __shared__ __align__(16) float small_smem[];
    const int tid = threadIdx.x, tpb = blockDim.x;
    const int cgs = C / V, wv = cgs / slabs, wc = wv * V, R = tpb / (units * wv);  // vectors and channels of the slab, rows of a row block
    double* const s_tot = reinterpret_cast<double*>(small_smem);          // [2][wc]
    float* const s_coef = small_smem + 4 * wc;                            // [4][wc]
    float* const red = s_coef + 4 * wc;                                   // [2][tpb * V]
    float* const part = red + 2 * tpb * V;                                // [2][units][wc]
    const int jl = tid / (R * wv), rem = tid % (R * wv), cg = rem % wv;
    const int block = q * units + jl, uc = units * wc;                    // of the reduce kernel's grid
    const long long row0 = (long long)block * R + rem / wv, row_step = (long long)row_blocks * R;
    const int ch = (slab * wv + cg) * V;
    auto has = [&](int u) { return block < row_blocks && row0 + u * row_step < rows; };
    Vec16<YT> qy[D];
    Vec16<AT> qg[D];
#pragma unroll
    for (int u = 0; u < D; ++u)
        if (has(u)) {
            qy[u] = ld16(y + (row0 + u * row_step) * C + ch);
            qg[u] = ld16(g + (row0 + u * row_step) * (PITCHED ? ld_g : (long long)C) + ch);
        }
    float2 a[V / 2], b[V / 2];
    {
        float2 sb[V / 2], sy[V / 2];
        float mu[V], is[V], ga[V], be[V];
        load_params<V>(fin.mean, slab * wv + cg, mu);
        load_params<V>(fin.invstd, slab * wv + cg, is);
        load_params<V>(fin.gamma, slab * wv + cg, ga);
        load_params<V>(fin.beta, slab * wv + cg, be);
#pragma unroll
        for (int j = 0; j < V / 2; ++j) {
            a[j] = make_float2(ga[2 * j] * is[2 * j], ga[2 * j + 1] * is[2 * j + 1]);
            b[j] = make_float2(fmaf(-mu[2 * j], a[j].x, be[2 * j]), fmaf(-mu[2 * j + 1], a[j].y, be[2 * j + 1]));
            sb[j] = sy[j] = splat2(0.f);
        }
#pragma unroll
        for (int u = 0; u < D; ++u)
            if (has(u)) {
#pragma unroll
                for (int j = 0; j < V / 2; ++j) {
                    const float2 yv = pair_to_f32(qy[u].v + 2 * j);
                    const float2 dz = silu_bwd_dz2<FAST>(fma2(yv, a[j], b[j]), pair_to_f32(qg[u].v + 2 * j));
                    sb[j] = add2(sb[j], dz);
                    sy[j] = fma2(dz, yv, sy[j]);
                }
            }
#pragma unroll
        for (int j = 0; j < V / 2; ++j) {
            *reinterpret_cast<float2*>(&red[tid * V + 2 * j]) = sb[j];
            *reinterpret_cast<float2*>(&red[(tpb + tid) * V + 2 * j]) = sy[j];
        }
    }
    __syncthreads();
    for (int e = tid; e < 2 * uc; e += tpb) {  // the sums of every row block of this CTA (zero past the last)
        const int pass = e >= uc ? 1 : 0, k = e - pass * uc, bl = k / wc, c = k - bl * wc;
        const float* const src = red + (pass * tpb + bl * R * wv) * V + c;
        float acc = 0.f;
        for (int r = 0; r < R; ++r) acc += src[r * wc];
        part[e] = q * units + bl < row_blocks ? acc : 0.f;
    }
    __syncthreads();
    for (int e = tid; e < 2 * wc; e += tpb) {
        const int pass = e >= wc ? 1 : 0;
        const float* const src = part + pass * uc + (e - pass * wc);
        double t = 0.0;
        for (int bl = 0; bl < units; ++bl) t += (double)src[bl * wc];
        s_tot[e] = t;
    }
    __syncthreads();  // (the cluster barrier wants whole warps)
    if (cluster > 1) ptx::cluster_sync_all();
    const uint32_t tot = ptx::smem_u32(s_tot);
    for (int c = tid; c < wc; c += tpb) {
        double s0 = 0.0, s1 = 0.0;
        if (cluster > 1) {
            double t0[8], t1[8];  // (all peers asked before the first answer is used)
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (k < cluster) {
                    const uint32_t peer = ptx::mapa_u32(tot, (uint32_t)k);
                    t0[k] = ld_dsmem_f64(peer + 8u * (uint32_t)c);
                    t1[k] = ld_dsmem_f64(peer + 8u * (uint32_t)(wc + c));
                }
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (k < cluster) {
                    s0 += t0[k];
                    s1 += t1[k];
                }
        } else {
            s0 = s_tot[c];
            s1 = s_tot[wc + c];
        }
        const int cc = slab * wc + c;
        const BwdCoef k = bwd_coef_channel(fin.mean[cc], fin.invstd[cc], fin.gamma[cc], fin.beta[cc], s0, s1, fin.inv_m);
        s_coef[c] = k.a;
        s_coef[wc + c] = k.b;
        s_coef[2 * wc + c] = k.p1;
        s_coef[3 * wc + c] = k.p0;
        if (q == 0) {
            fin.dbeta[cc] = (float)s0;
            fin.dgamma[cc] = k.dgamma;
        }
    }
    __syncthreads();
    // behind its own reads a CTA tells its peers that they may leave
    if (cluster > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    float2 np1[V / 2], p0[V / 2];
    load_params_shared<V>(s_coef, cg, a);
    load_params_shared<V>(s_coef + wc, cg, b);
    load_params_shared<V>(s_coef + 2 * wc, cg, np1);
    load_params_shared<V>(s_coef + 3 * wc, cg, p0);
#pragma unroll
    for (int j = 0; j < V / 2; ++j) np1[j] = make_float2(-np1[j].x, -np1[j].y);
#pragma unroll
    for (int u = 0; u < D; ++u)
        if (has(u)) {
            const long long row = row0 + u * row_step;
            if (GRES) {
                Vec16<AT> r = qg[u];
                if (gres_add) {
                    const Vec16<AT> old = ld16(gres + row * ld_gres + ch);
#pragma unroll
                    for (int j = 0; j < V / 2; ++j) pair_from_f32(r.v + 2 * j, add2(pair_to_f32(old.v + 2 * j), pair_to_f32(qg[u].v + 2 * j)));
                }
                st16(gres + row * ld_gres + ch, r);
            }
            Vec16<AT> o;
#pragma unroll
            for (int j = 0; j < V / 2; ++j) {
                const float2 yv = pair_to_f32(qy[u].v + 2 * j);
                const float2 dz = silu_bwd_dz2<FAST>(fma2(yv, a[j], b[j]), pair_to_f32(qg[u].v + 2 * j));
                pair_from_f32(o.v + 2 * j, fma2(a[j], dz, fma2(np1[j], yv, p0[j])));
            }
            st16(dy + row * C + ch, o);
        }
    __syncwarp();
    if (cluster > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

}  // namespace nbcbs
