// CUDA-core implicit GEMMs for the three convolutions (fprop, dgrad, wgrad): any shape, fp32 or 16-bit inputs,
// fp32 accumulation flushed into fp64 every 1024 terms.  They carry the fp32 reference mode and every shape
// the tensor-core kernels do not take.
#pragma once
#include "common.cuh"
#include "elementwise.cuh"

namespace nbcbs {

// out[i][j] = sum_kk A(i,kk) * B(kk,j) on plain FMA units.  Bound: FMA issue on large problems (a thread's 8 x 4 tile takes
// 12 16-byte shared loads per 128 multiply-adds), memory latency on small ones.  A block is 128 threads on a
// [BM x BN] tile; both operand tiles travel global -> shared memory by cp.async through a ring of four stages of 16 k
// (element-wise loads into registers, two block barriers per 16 k and an index decode by 64-bit divisions per element
// are what the previous version spent its time on: 64 -> 64 channels 3x3 on 2 x 40 x 40 pixels, step 445 -> 59 us;
// 96 -> 96 at 2 x 80 x 80, 990 -> 275 us, 24 TFLOP/s in the convolutions; 31 with the idle columns of the second tile).
//   KIND 0 (fprop): rows = output pixels, cols = c_out, k = (tap, c_in).   A, B tiles [row][k], [col][k]
//   KIND 1 (dgrad): rows = input pixels, cols = c_in, k = (tap, c_out).    A tile [row][k], B tile [k][col]
//   KIND 2 (wgrad): rows = c_out, cols = (tap, c_in), k = output pixels.   A, B tiles [k][row], [k][col]
// A stride-2 data gradient walks the parity classes of the input pixels one after the other, each with the taps that
// reach it (a quarter of the products of the undivided sum).
// V = 4: channels come as vectors of four (c_in % 4 == 0); V = 1: element by element (c_in = 3).
constexpr int SG_BK = 16, SG_STAGES = 4, SG_THREADS = 128, SG_KPITCH = SG_BK + 4, SG_FLUSH = 1024 / SG_BK;

template <typename T> __device__ __forceinline__ float4 sg_ld4(const T* p);
template <> __device__ __forceinline__ float4 sg_ld4<float>(const float* p) { return *reinterpret_cast<const float4*>(p); }
template <> __device__ __forceinline__ float4 sg_ld4<__nv_bfloat16>(const __nv_bfloat16* p) {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x)), b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
template <> __device__ __forceinline__ float4 sg_ld4<__half>(const __half* p) {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x)), b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
// four elements global -> shared, zeros when !ok (src is then any valid address)
template <typename T> __device__ __forceinline__ void sg_copy4(T* dst, const T* src, bool ok) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if (sizeof(T) == 4) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(ok ? 8 : 0) : "memory");
}
template <typename T> __device__ __forceinline__ void sg_copy1(T* dst, const T* src, bool ok) {
    if (sizeof(T) == 4) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(ok ? 4 : 0) : "memory");
    } else {
        *dst = ok ? *src : from_f32<T>(0.f);  // (cp.async moves at least four bytes)
    }
}

template <int KIND, int BM, int BN> struct SgTile {
    static constexpr int A_ELEMS = KIND == 2 ? SG_BK * (BM + 4) : BM * SG_KPITCH;
    static constexpr int B_ELEMS = KIND == 0 ? BN * SG_KPITCH : SG_BK * (BN + 4);
    static constexpr int NTX = BN / 4, NTY = SG_THREADS / NTX, TM = BM / NTY;
    static __host__ __device__ constexpr size_t stage_bytes(size_t elem) { return SG_STAGES * (size_t)(A_ELEMS + B_ELEMS) * elem; }
};

struct SgArgs {
    Geom g;
    long long kchunk;  // k per slice (blockIdx.z), a multiple of SG_BK
    bool stats;        // KIND 0 with one slice: add the channel sums of the stored values to `acc`
    ChanAcc acc;
    int overlap;       // KIND 2: runs beside the data gradient in front of it (see the end of common.cuh)
};

// rows of parity class `cls` of a data gradient, and the grid that covers all classes (host and device)
struct SgClass {
    int pa, pb, hc, wc;  // parities, rows and columns of the class's pixel grid
    long long rows;
};
__host__ __device__ __forceinline__ SgClass sg_class(const Geom& g, int cls) {
    SgClass c;
    c.pa = cls / g.stride;
    c.pb = cls % g.stride;
    c.hc = (g.h - c.pa + g.stride - 1) / g.stride;
    c.wc = (g.w - c.pb + g.stride - 1) / g.stride;
    c.rows = (long long)g.n * c.hc * c.wc;
    return c;
}

// grid (row tiles, column tiles, slices).  With several slices `out` is a float buffer [slices][rows][cols].
template <int KIND, typename TIN, typename TO, int BM, int BN, int V>
__global__ void __launch_bounds__(SG_THREADS) simt_gemm_kernel(const TIN* __restrict__ asrc, const TIN* __restrict__ bsrc, TO* __restrict__ out, const SgArgs p) {
    if (KIND != 1) pdl_launch_dependents();
    using T = SgTile<KIND, BM, BN>;
    constexpr int TM = T::TM, NTX = T::NTX, NTY = T::NTY;
    extern __shared__ __align__(16) uint8_t sg_smem[];
    TIN* const sA = reinterpret_cast<TIN*>(sg_smem);
    TIN* const sB = sA + SG_STAGES * T::A_ELEMS;
    double* const flushed = reinterpret_cast<double*>(sg_smem + T::stage_bytes(sizeof(TIN)));  // [TM * 4][128 threads], slices longer than 1024 only
    const Geom& g = p.g;
    const int tid = threadIdx.x, tx = tid % NTX, ty = tid / NTX;
    const int j0 = blockIdx.y * BN;
    const int cols = KIND == 0 ? g.c_out : KIND == 1 ? g.c_in : g.kdim;

    // ---- the row tile: its class (data gradient), first row, taps
    long long i0 = (long long)blockIdx.x * BM, rows = KIND == 0 ? g.m : KIND == 1 ? 0 : g.c_out;
    SgClass cl{0, 0, g.h, g.w, 0};
    int r_first = 0, r_step = 1, nr = g.k, t_first = 0, nt = g.k;
    if (KIND == 1) {
        long long tile = blockIdx.x;
        int cls = 0;
        cl = sg_class(g, 0);
        while (tile >= (cl.rows + BM - 1) / BM) {
            tile -= (cl.rows + BM - 1) / BM;
            cl = sg_class(g, ++cls);
        }
        i0 = tile * BM;
        rows = cl.rows;
        r_step = g.stride;
        r_first = (cl.pa + g.pad) % g.stride;
        t_first = (cl.pb + g.pad) % g.stride;
        nr = (g.k - r_first + r_step - 1) / r_step;
        nt = (g.k - t_first + r_step - 1) / r_step;
    }
    const int ntd = nt > 0 ? nt : 1;  // (no tap reaches the odd pixels of a 1x1 stride-2 layer: K = 0, zeros are stored)
    const int kch = KIND == 1 ? g.c_out : g.c_in;  // channels per tap on the k side (KIND 0, 1)
    const long long KK = KIND == 2 ? g.m : (long long)nr * nt * kch;
    const long long kbeg = (long long)blockIdx.z * p.kchunk;
    const long long kend = kbeg + p.kchunk < KK ? kbeg + p.kchunk : KK;
    const int nsteps = kend > kbeg ? (int)((kend - kbeg + SG_BK - 1) / SG_BK) : 0;

    // ---- loader state (advanced by one stage per call)
    // [row][k] tiles: a thread copies four k (kv) of rows tid / 4 + 32 i
    constexpr int AP = KIND == 2 ? BM * SG_BK / 4 / SG_THREADS : BM / 32;  // copies of four per thread and stage
    constexpr int BP = KIND == 0 ? BN / 32 : BN * SG_BK / 4 / SG_THREADS;
    const int kv = (tid & 3) * 4;
    int a_h[AP > 0 ? AP : 1], a_w[AP > 0 ? AP : 1];
    long long a_base[AP > 0 ? AP : 1];
    bool a_ok[AP > 0 ? AP : 1];
    int tap_r = 0, tap_t = 0, ch = 0;  // tap and channel of this thread's four k (V = 4, or KIND 1)
    if (KIND != 2) {
#pragma unroll
        for (int i = 0; i < AP; ++i) {
            const long long row = i0 + (tid >> 2) + 32 * i;
            a_ok[i] = row < rows;
            const long long rr = a_ok[i] ? row : 0;
            if (KIND == 0) {
                const int q = (int)(rr % g.wo);
                const long long t1 = rr / g.wo;
                const int pp = (int)(t1 % g.ho);
                a_base[i] = (t1 / g.ho) * g.h * g.w;
                a_h[i] = pp * g.stride - g.pad;
                a_w[i] = q * g.stride - g.pad;
            } else {  // dy row and column of tap (r, t): (h + pad - r) / stride
                const int j = (int)(rr % cl.wc);
                const long long t1 = rr / cl.wc;
                const int ii = (int)(t1 % cl.hc);
                a_base[i] = (t1 / cl.hc) * g.ho * g.wo;
                a_h[i] = (ii * g.stride + cl.pa + g.pad - r_first) / g.stride;
                a_w[i] = (j * g.stride + cl.pb + g.pad - t_first) / g.stride;
            }
        }
        const long long k0 = kbeg + kv;
        const int tap = (int)(k0 / kch);
        ch = (int)(k0 - (long long)tap * kch);
        tap_r = tap / ntd;
        tap_t = tap - tap_r * ntd;
    }
    // [k][..] tiles: a thread copies four neighbouring rows / columns of k rows kr + i * step
    const int a_mv = (tid % (BM / 4)) * 4, a_kr = tid / (BM / 4);
    constexpr int A_KSTEP = SG_THREADS / (BM / 4), B_KSTEP = SG_THREADS / (BN / 4);
    const int b_nv = (tid % (BN / 4)) * 4, b_kr = tid / (BN / 4);
    int px_n[KIND == 2 ? BP : 1], px_p[KIND == 2 ? BP : 1], px_q[KIND == 2 ? BP : 1];  // pixel of each k row (weight gradient)
    int b_r[KIND == 2 ? 4 : 1], b_t[KIND == 2 ? 4 : 1], b_c[KIND == 2 ? 4 : 1];        // tap and channel of this thread's columns
    if (KIND == 2) {
#pragma unroll
        for (int i = 0; i < BP; ++i) {
            const long long px = kbeg + b_kr + i * B_KSTEP;
            const long long t1 = px / g.wo;
            px_q[i] = (int)(px - t1 * g.wo);
            px_n[i] = (int)(t1 / g.ho);
            px_p[i] = (int)(t1 - (long long)px_n[i] * g.ho);
        }
#pragma unroll
        for (int e = 0; e < (V == 4 ? 1 : 4); ++e) {
            const int j = j0 + b_nv + e < cols ? j0 + b_nv + e : 0;
            const int tap = j / g.c_in;
            b_c[e] = j - tap * g.c_in;
            b_r[e] = tap / g.k;
            b_t[e] = tap - b_r[e] * g.k;
        }
    }
    int f_co[KIND == 1 ? BP : 1], f_r[KIND == 1 ? BP : 1], f_t[KIND == 1 ? BP : 1];  // channel and tap of each k row of the filter tile (data gradient)
    if (KIND == 1) {
#pragma unroll
        for (int i = 0; i < BP; ++i) {
            const int kk = (int)kbeg + b_kr + i * B_KSTEP, tap = kk / kch;
            f_co[i] = kk - tap * kch;
            f_r[i] = tap / ntd;
            f_t[i] = tap - f_r[i] * ntd;
        }
    }
    long long kload = kbeg;  // first k of the next stage to load
    auto load_stage = [&](int s) {
        TIN* const a_s = sA + s * T::A_ELEMS;
        TIN* const b_s = sB + s * T::B_ELEMS;
        if (KIND == 0 && V == 1) {  // element by element, k decoded per element
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const long long kk = kload + kv + e;
                const int tap = (int)(kk / kch), c = (int)(kk - (long long)tap * kch), r = tap / g.k, t = tap - r * g.k;
#pragma unroll
                for (int i = 0; i < AP; ++i) {
                    const int h = a_h[i] + r, w = a_w[i] + t;
                    const bool ok = a_ok[i] && kk < kend && h >= 0 && h < g.h && w >= 0 && w < g.w;
                    sg_copy1(a_s + ((tid >> 2) + 32 * i) * SG_KPITCH + kv + e, ok ? asrc + (a_base[i] + (long long)h * g.w + w) * g.c_in + c : asrc, ok);
                }
#pragma unroll
                for (int i = 0; i < BP; ++i) {
                    const int col = j0 + (tid >> 2) + 32 * i;
                    const bool ok = col < cols && kk < kend;
                    sg_copy1(b_s + ((tid >> 2) + 32 * i) * SG_KPITCH + kv + e, ok ? bsrc + (long long)col * g.kdim + kk : bsrc, ok);
                }
            }
            kload += SG_BK;
            return;
        }
        if (KIND != 2) {
            const bool kok = kload + kv < kend;
#pragma unroll
            for (int i = 0; i < AP; ++i) {
                const int h = KIND == 0 ? a_h[i] + tap_r : a_h[i] - tap_r, w = KIND == 0 ? a_w[i] + tap_t : a_w[i] - tap_t;
                const int hh = KIND == 0 ? g.h : g.ho, ww = KIND == 0 ? g.w : g.wo;
                const bool ok = kok && a_ok[i] && h >= 0 && h < hh && w >= 0 && w < ww;
                sg_copy4(a_s + ((tid >> 2) + 32 * i) * SG_KPITCH + kv, ok ? asrc + (a_base[i] + (long long)h * ww + w) * kch + ch : asrc, ok);
            }
            if (KIND == 0) {
#pragma unroll
                for (int i = 0; i < BP; ++i) {
                    const int col = j0 + (tid >> 2) + 32 * i;
                    const bool ok = kok && col < cols;
                    sg_copy4(b_s + ((tid >> 2) + 32 * i) * SG_KPITCH + kv, ok ? bsrc + (long long)col * g.kdim + kload + kv : bsrc, ok);
                }
            } else {  // filter rows k = (tap, c_out), c_in contiguous
#pragma unroll
                for (int i = 0; i < BP; ++i) {
                    const int kr = b_kr + i * B_KSTEP;
                    const long long kk = kload + kr;
                    const TIN* src = bsrc + ((long long)f_co[i] * g.k * g.k + (r_first + f_r[i] * r_step) * g.k + t_first + f_t[i] * r_step) * g.c_in + j0 + b_nv;
                    f_co[i] += SG_BK;
                    while (f_co[i] >= kch) {
                        f_co[i] -= kch;
                        if (++f_t[i] == ntd) {
                            f_t[i] = 0;
                            ++f_r[i];
                        }
                    }
                    if (V == 4) {
                        const bool ok = kk < kend && j0 + b_nv < cols;
                        sg_copy4(b_s + kr * (BN + 4) + b_nv, ok ? src : bsrc, ok);
                    } else {
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const bool ok = kk < kend && j0 + b_nv + e < cols;
                            sg_copy1(b_s + kr * (BN + 4) + b_nv + e, ok ? src + e : bsrc, ok);
                        }
                    }
                }
            }
            ch += SG_BK;
            while (ch >= kch) {
                ch -= kch;
                if (++tap_t == nt) {
                    tap_t = 0;
                    ++tap_r;
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < AP; ++i) {
                const int kr = a_kr + i * A_KSTEP;
                const bool ok = kload + kr < kend && i0 + a_mv < rows;
                sg_copy4(a_s + kr * (BM + 4) + a_mv, ok ? asrc + (kload + kr) * g.c_out + i0 + a_mv : asrc, ok);
            }
#pragma unroll
            for (int i = 0; i < BP; ++i) {
                const int kr = b_kr + i * B_KSTEP;
                const bool kok = kload + kr < kend;
                const int hb = px_p[i] * g.stride - g.pad, wb = px_q[i] * g.stride - g.pad;
#pragma unroll
                for (int e = 0; e < (V == 4 ? 1 : 4); ++e) {
                    const int h = hb + b_r[e], w = wb + b_t[e];
                    const bool ok = kok && j0 + b_nv + e < cols && h >= 0 && h < g.h && w >= 0 && w < g.w;
                    const TIN* src = ok ? bsrc + (((long long)px_n[i] * g.h + h) * g.w + w) * g.c_in + b_c[e] : bsrc;
                    if (V == 4) sg_copy4(b_s + kr * (BN + 4) + b_nv, src, ok);
                    else sg_copy1(b_s + kr * (BN + 4) + b_nv + e, src, ok);
                }
                px_q[i] += SG_BK;
                while (px_q[i] >= g.wo) {
                    px_q[i] -= g.wo;
                    if (++px_p[i] == g.ho) {
                        px_p[i] = 0;
                        ++px_n[i];
                    }
                }
            }
        }
        kload += SG_BK;
    };

    float acc[TM][4];
#pragma unroll
    for (int u = 0; u < TM; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = 0.f;
    const bool flush = p.kchunk > 1024;
    if (flush) {
#pragma unroll
        for (int e = 0; e < TM * 4; ++e) flushed[e * SG_THREADS + tid] = 0.0;
    }
    if (KIND != 2 || !p.overlap) pdl_wait();
    if (KIND == 1) pdl_launch_dependents();  // (behind its own wait: see the end of common.cuh)
#pragma unroll
    for (int s = 0; s < SG_STAGES - 1; ++s) {
        if (s < nsteps) load_stage(s);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    int since = 0;
    for (int it = 0; it < nsteps; ++it) {
        asm volatile("cp.async.wait_group %0;" ::"n"(SG_STAGES - 2) : "memory");
        __syncthreads();
        if (it + SG_STAGES - 1 < nsteps) load_stage((it + SG_STAGES - 1) % SG_STAGES);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const TIN* const a_s = sA + (it % SG_STAGES) * T::A_ELEMS;
        const TIN* const b_s = sB + (it % SG_STAGES) * T::B_ELEMS;
        if (KIND != 2) {
#pragma unroll
            for (int kq = 0; kq < SG_BK; kq += 4) {
                float4 a[TM], b[4];
#pragma unroll
                for (int u = 0; u < TM; ++u) a[u] = sg_ld4(a_s + (ty + u * NTY) * SG_KPITCH + kq);
#pragma unroll
                for (int v = 0; v < 4; ++v) b[v] = KIND == 0 ? sg_ld4(b_s + (tx + v * NTX) * SG_KPITCH + kq) : sg_ld4(b_s + (kq + v) * (BN + 4) + tx * 4);
#pragma unroll
                for (int u = 0; u < TM; ++u) {
                    const float au[4] = {a[u].x, a[u].y, a[u].z, a[u].w};
#pragma unroll
                    for (int e = 0; e < 4; ++e)
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const float4 bb = KIND == 0 ? b[v] : b[e];  // KIND 0: column v at k e; KIND 1: k e at column v
                            const int at = KIND == 0 ? e : v;
                            acc[u][v] = fmaf(au[e], at == 0 ? bb.x : at == 1 ? bb.y : at == 2 ? bb.z : bb.w, acc[u][v]);
                        }
                }
            }
        } else {
#pragma unroll
            for (int k = 0; k < SG_BK; ++k) {
                float a[TM];
#pragma unroll
                for (int u = 0; u < TM; u += 4) {
                    const float4 t = sg_ld4(a_s + k * (BM + 4) + ty * TM + u);
                    a[u] = t.x; a[u + 1] = t.y; a[u + 2] = t.z; a[u + 3] = t.w;
                }
                const float4 b = sg_ld4(b_s + k * (BN + 4) + tx * 4);
#pragma unroll
                for (int u = 0; u < TM; ++u) {
                    acc[u][0] = fmaf(a[u], b.x, acc[u][0]);
                    acc[u][1] = fmaf(a[u], b.y, acc[u][1]);
                    acc[u][2] = fmaf(a[u], b.z, acc[u][2]);
                    acc[u][3] = fmaf(a[u], b.w, acc[u][3]);
                }
            }
        }
        if (flush && ++since == SG_FLUSH) {
            since = 0;
#pragma unroll
            for (int u = 0; u < TM; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    flushed[(u * 4 + v) * SG_THREADS + tid] += (double)acc[u][v];
                    acc[u][v] = 0.f;
                }
        }
    }

    // ---- store, and the channel sums of what is stored
    const long long out_rows = KIND == 0 ? g.m : KIND == 1 ? (long long)g.n * g.h * g.w : g.c_out;
    TO* const o = out + (size_t)blockIdx.z * (size_t)out_rows * (size_t)cols;
    float cs[4] = {0.f, 0.f, 0.f, 0.f}, cq[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int u = 0; u < TM; ++u) {
        const long long i = i0 + (KIND == 2 ? ty * TM + u : ty + u * NTY);
        if (i >= rows) continue;
        long long orow = i;
        if (KIND == 1 && g.stride > 1) {
            const int j = (int)(i % cl.wc);
            const long long t1 = i / cl.wc;
            orow = ((t1 / cl.hc) * g.h + (t1 % cl.hc) * g.stride + cl.pa) * g.w + (long long)j * g.stride + cl.pb;
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int j = j0 + (KIND == 0 ? tx + v * NTX : tx * 4 + v);
            if (j >= cols) continue;
            const float val = flush ? (float)(flushed[(u * 4 + v) * SG_THREADS + tid] + (double)acc[u][v]) : acc[u][v];
            const TO st = from_f32<TO>(val);
            o[(size_t)orow * cols + j] = st;
            if (KIND == 0) {
                const float f = to_f32(st);
                cs[v] += f;
                cq[v] = fmaf(f, f, cq[v]);
            }
        }
    }
    if (KIND == 0 && p.stats) {
        float* const red = reinterpret_cast<float*>(sg_smem);  // [NTY][2][BN]
        __syncthreads();
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            red[(ty * 2) * BN + tx + v * NTX] = cs[v];
            red[(ty * 2 + 1) * BN + tx + v * NTX] = cq[v];
        }
        __syncthreads();
        for (int e = tid; e < 2 * BN; e += SG_THREADS) {
            const int which = e / BN, c = e - which * BN;
            if (j0 + c >= cols) continue;
            float sum = 0.f;
            for (int r = 0; r < NTY; ++r) sum += red[(r * 2 + which) * BN + c];
            chan_acc_add<std::is_same<TIN, float>::value>(p.acc, g.c_out, which, j0 + c, sum);
        }
    }
    if (KIND == 2 && p.overlap) pdl_wait();
}

// out = sum over the slices of a split forward convolution (fp64, slice order), rounded to YT, and with acc.acc != NULL the
// channel sums of the stored values (a thread keeps one group of four channels, like the elementwise passes).
// A block is at least one row of channel groups: 288 at the 1152 channels that a plan may have in fp32, 576 at the 2304 of the
// 16-bit modes.
constexpr int SG_REDUCE_MAX = 576;
template <typename YT>
__global__ void __launch_bounds__(SG_REDUCE_MAX) splitk_fwd_reduce_kernel(const float* __restrict__ partial, int splits, long long vecs, int C, YT* __restrict__ out, ChanAcc acc) {
    pdl_launch_dependents();
    pdl_wait();
    extern __shared__ float red[];  // [blockDim.x][4]
    const int tid = threadIdx.x, cgs = C / 4;
    float s[4] = {0.f, 0.f, 0.f, 0.f}, q[4] = {0.f, 0.f, 0.f, 0.f};
    const float4* p4 = reinterpret_cast<const float4*>(partial);
    for (long long v = (long long)blockIdx.x * blockDim.x + tid; v < vecs; v += (long long)gridDim.x * blockDim.x) {
        double d[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
        for (int z = 0; z < splits; ++z) {
            const float4 a = p4[(size_t)z * vecs + v];
            d[0] += (double)a.x; d[1] += (double)a.y; d[2] += (double)a.z; d[3] += (double)a.w;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const YT y = from_f32<YT>((float)d[i]);
            out[v * 4 + i] = y;
            const float f = to_f32(y);
            s[i] += f;
            q[i] = fmaf(f, f, q[i]);
        }
    }
    if (!acc.acc) return;
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
        for (int i = 0; i < 4; ++i) red[tid * 4 + i] = pass ? q[i] : s[i];
        __syncthreads();
        for (int c = tid; c < C; c += blockDim.x) {
            float sum = 0.f;
            for (int r = c / 4; r < (int)blockDim.x; r += cgs) sum += red[r * 4 + (c & 3)];
            chan_acc_add<std::is_same<YT, float>::value>(acc, C, pass, c, sum);
        }
        __syncthreads();
    }
}

// out[e] = sum_z partial[z][e], summed in fp64 in slice order (four elements per thread when the count allows).
// Eight slices are loaded before any is added so that a thread keeps eight independent 16-byte loads in flight:
// the kernel is tiny and otherwise bound by one memory latency per slice.
// LATE: the last launch of a data gradient (it signals its dependents behind its own wait: see the end of common.cuh).
// (thread `at` of `stride` threads)
template <typename TO> __device__ __forceinline__ void splitk_reduce(const float* __restrict__ partial, int splits, size_t elems, TO* __restrict__ out, size_t at, size_t stride) {
    if ((elems & 3) == 0) {
        const size_t nv = elems >> 2;
        const float4* p4 = reinterpret_cast<const float4*>(partial);
        for (size_t v = at; v < nv; v += stride) {
            double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
            for (int z0 = 0; z0 < splits; z0 += 8) {
                float4 a[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (z0 + u < splits) a[u] = p4[(size_t)(z0 + u) * nv + v];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (z0 + u < splits) {
                        s0 += (double)a[u].x;
                        s1 += (double)a[u].y;
                        s2 += (double)a[u].z;
                        s3 += (double)a[u].w;
                    }
            }
            if constexpr (sizeof(TO) == 4) {
                reinterpret_cast<float4*>(out)[v] = make_float4((float)s0, (float)s1, (float)s2, (float)s3);
            } else {
                TO o[4] = {from_f32<TO>((float)s0), from_f32<TO>((float)s1), from_f32<TO>((float)s2), from_f32<TO>((float)s3)};
                reinterpret_cast<uint2*>(out)[v] = *reinterpret_cast<const uint2*>(o);
            }
        }
    } else {
        for (size_t e = at; e < elems; e += stride) {
            double s = 0.0;
            for (int z = 0; z < splits; ++z) s += (double)partial[(size_t)z * elems + e];
            out[e] = from_f32<TO>((float)s);
        }
    }
}
template <typename TO, bool LATE = false>
__global__ void __launch_bounds__(256) splitk_reduce_kernel(const float* __restrict__ partial, int splits, size_t elems, TO* __restrict__ out) {
    if (!LATE) pdl_launch_dependents();
    pdl_wait();
    if (LATE) pdl_launch_dependents();
    splitk_reduce(partial, splits, elems, out, (size_t)blockIdx.x * blockDim.x + threadIdx.x, (size_t)gridDim.x * blockDim.x);
}
// The slices of a data gradient (the first `blocks1` blocks) and of the weight gradient beside it, in one launch.
template <typename TO>
__global__ void __launch_bounds__(256) splitk_reduce_both_kernel(const float* __restrict__ partial1, int splits1, size_t elems1, TO* __restrict__ out1, int blocks1,
                                                                 const float* __restrict__ partial2, int splits2, size_t elems2, float* __restrict__ out2) {
    pdl_launch_dependents();
    pdl_wait();
    const int b = (int)blockIdx.x;
    if (b < blocks1) splitk_reduce(partial1, splits1, elems1, out1, (size_t)b * blockDim.x + threadIdx.x, (size_t)blocks1 * blockDim.x);
    else splitk_reduce(partial2, splits2, elems2, out2, (size_t)(b - blocks1) * blockDim.x + threadIdx.x, (size_t)((int)gridDim.x - blocks1) * blockDim.x);
}

// The same sum for many slices of few elements (the first layer's weight gradient: ~1200 slices of 1296 values): a block of
// 32 x 32 threads takes 32 consecutive elements; thread (e, zg) adds slices zg, zg + 32, ... in that order in fp64 (coalesced
// 128-byte rows, eight loads in flight), and the 32 partial sums of an element are combined in the order of zg.
__global__ void __launch_bounds__(1024) splitk_reduce_tall_kernel(const float* __restrict__ partial, int splits, size_t elems, float* __restrict__ out) {
    pdl_launch_dependents();
    pdl_wait();
    __shared__ double red[32][33];
    const int ex = threadIdx.x & 31, zg = threadIdx.x >> 5;
    const size_t e = (size_t)blockIdx.x * 32 + ex;
    double acc = 0.0;
    if (e < elems) {
        for (int z0 = zg; z0 < splits; z0 += 256) {
            float a[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) a[u] = z0 + 32 * u < splits ? partial[(size_t)(z0 + 32 * u) * elems + e] : 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u) acc += (double)a[u];
        }
    }
    red[zg][ex] = acc;
    __syncthreads();
    if (zg == 0 && e < elems) {
        double s = 0.0;
#pragma unroll 8
        for (int k = 0; k < 32; ++k) s += red[k][ex];
        out[e] = (float)s;
    }
}

}  // namespace nbcbs
