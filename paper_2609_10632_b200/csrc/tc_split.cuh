// Implicit GEMM for layers with few output tiles (one or two images at 40 x 40 and below), sm_100a.
// The persistent kernel of tc_conv.cuh gives such a layer a handful of CTAs, each of which walks the whole K range alone:
// 288 -> 288 3x3 on one 20 x 20 image is 8 tiles of 45 k-blocks on 148 SMs, 20 us of one CTA's operand fetches.  Here the
// K range of a tile is cut over a CLUSTER of 1, 2, 4 or 8 CTAs.  Every CTA accumulates its share in TMEM and sends the rows of
// every rank to that rank's shared memory by bulk copies; CTA r then sums rows [128 r / S, 128 (r + 1) / S) of all S shares in
// rank order (the same bits every run), applies the epilogue and stores.
// The training calls use clusters of one (tiles of up to 256 columns, 160 in the data gradient): the sum of an element then
// runs over the k-blocks in the order in which the persistent kernel would add them (the same starting k-block), and the
// channel sums are formed as there, so that the results of a training step do not depend on which of the two kernels a layer
// gets -- a deep network in training mode turns a difference in the last bit of one layer into percents a few dozen layers on.
// No block waits for a block outside its cluster.  Bound: latency.  192 -> 192 3x3 on one 40 x 40 image, us behind the end of the
// launch before: 0.8 until that has reached the CTA, 0.6 until the last CTA runs (an SM holds one), 1.1 to the first operands,
// 0.15 a k-block (its 128 + BN rows are written to and read from shared memory once each), 0.5 to 0.8 behind the last MMA.
// The narrow tiles (often 32 to 64 columns) are part of the same idea: more CTAs, and less to hand over.
// Measured against the persistent kernel: see split_configure below.
// Included by tc_conv.cuh (uses its parameter record and bounded-wait helpers).
#pragma once

namespace nbcbs {

constexpr int SP_THREADS = 256;
constexpr int SP_PARTS = SP_THREADS / 128;  // warps that share a quarter's columns (sixteen warps: evaluation of one image 551 -> 563 us)
// First column of a part's share (whole 16-column pieces) and the part of a column.
__device__ __forceinline__ int sp_part_lo(int part, int BN) { return part * (BN / 16) / SP_PARTS * 16; }
__device__ __forceinline__ int sp_part_of(int c, int BN) { return (c / 16 * SP_PARTS + SP_PARTS - 1) / (BN / 16); }

// `bytes` of this CTA's shared memory to the shared memory of a CTA of the cluster; counted on that CTA's barrier `bar`.
__device__ __forceinline__ void copy_to_peer(uint32_t dst_cluster, const void* src, uint32_t bytes, uint32_t bar_cluster) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst_cluster), "r"(ptx::smem_u32(src)), "r"(bytes),
                 "r"(bar_cluster)
                 : "memory");
}
// 32 bytes on a 32-byte boundary
__device__ __forceinline__ void st_global32(void* p, const uint2 (&v)[4]) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0].x), "r"(v[0].y), "r"(v[1].x), "r"(v[1].y), "r"(v[2].x), "r"(v[2].y), "r"(v[3].x),
                 "r"(v[3].y)
                 : "memory");
}
__device__ __forceinline__ void prefetch_tile_2d(const CUtensorMap* m, int c0, int c1) {
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(reinterpret_cast<uint64_t>(m)), "r"(c0), "r"(c1) : "memory");
}

// MODE 0: plain 16-bit output (data gradient; may be pitched, may be added to what the output holds).  MODE 1: training
// forward (fp16 output, channel sums of the rounded values to the accumulators).  MODE 2: per-channel scale and shift, SiLU.
// S: CTAs of a cluster (p.split).
template <typename OutT, int MODE, int S>
__global__ void __launch_bounds__(SP_THREADS, 1) tc_split_kernel(const __grid_constant__ IgemmParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* sA = smem;
    uint8_t* sB = sA + (size_t)p.stages * p.a_stage_bytes;
    // S > 1: one slot per rank with that rank's share of this CTA's 128 / S rows, for each part of the columns [rows][columns + 4],
    // written by the ranks themselves (behind the operand stages, which may still be in use when a peer's share arrives)
    float* const part = reinterpret_cast<float*>(sB + (size_t)p.stages * p.b_stage_bytes);
    constexpr int ROWS = TC_BM / S;
    const int slot = ROWS * (p.BN + 4 * SP_PARTS);
    float* red = part + (S > 1 ? S * slot : 0);  // MODE 2: scale, shift [2][BN]
    uint64_t* bars = reinterpret_cast<uint64_t*>(red + 2 * 256);
    uint64_t* full = bars;
    uint64_t* empty = bars + p.stages;
    uint64_t* tfull = empty + p.stages;
    uint64_t* drain = tfull + 1;
    uint64_t* shares = drain + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(shares + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    if (MODE != 0) pdl_launch_dependents();
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int rank = (int)blockIdx.x % S, tile = (int)blockIdx.x / S;
    const int cls = tile / p.tiles_per_class, lt = tile - cls * p.tiles_per_class;
    const int m_tile = lt / p.n_tiles, n_tile = lt - m_tile * p.n_tiles;
    const int kblocks = p.cls_ntaps[cls] * p.kc_per_tap;
    const int kb0 = kblocks * rank / S, kb1 = kblocks * (rank + 1) / S;  // this CTA's share of the K range
    // MODE 0, 1: first k-block of the tile of the persistent kernel that contains this one
    int rot = 0;
    if (MODE != 2) {
        int full_tile = (m_tile * TC_BM / p.full_rows) * p.full_n_tiles + n_tile * p.BN / p.full_bn;
        if (p.nclasses == 4) {  // igemm_tile_class, solved for the tile
            const int round = full_tile * 4 / p.full_workers;
            full_tile = full_tile * 4 + ((cls - ((p.full_workers & 1) ? 0 : round)) & 3);
        }
        rot = (int)(((unsigned)(full_tile % p.full_workers) * 7u) % (unsigned)kblocks);
    }

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            ptx::mbar_init(full + s, 2);
            ptx::mbar_init(empty + s, 1);
        }
        ptx::mbar_init(tfull, 1);
        ptx::mbar_init(drain, 1);
        if (S > 1) ptx::mbar_init(shares, 1);
        *abort_flag = 0;
        ptx::fence_mbar_init();
        if (S > 1) {
            int cols = 0;
            for (int k = 0; k < SP_PARTS; ++k)
                if (sp_part_lo(k + 1, p.BN) > sp_part_lo(k, p.BN)) cols += sp_part_lo(k + 1, p.BN) - sp_part_lo(k, p.BN) + 4;
            ptx::mbar_expect_tx(shares, (uint32_t)(TC_BM * cols * 4));
        }
    }
    if (warp == 2 && lane == 0) {
        ptx::prefetch_tmap(&p.tmB[cls]);
        // this CTA's filter tiles start for L2 while the previous kernel still runs (a hint: L2 stays coherent whoever
        // writes the filter in the meantime)
        for (int i = kb0; i < kb1 && i < kb0 + 16; ++i) {
            const int kb = i + rot < kblocks ? i + rot : i + rot - kblocks;
            const int tap = kb / p.kc_per_tap, kc = kb - tap * p.kc_per_tap;
            prefetch_tile_2d(&p.tmB[cls], tap * p.Ca + kc * p.KC, n_tile * p.BN);
        }
    }
    if (warp == 0 && lane == 0) ptx::prefetch_tmap(&p.tmA);
    if (warp == 1) {
        ptx::tmem_alloc(tmem_slot, (uint32_t)p.tmem_cols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (S > 1) ptx::cluster_arrive_relaxed();  // (this CTA runs and its barriers are set up: the others may write its shared memory)
    const uint32_t tmem_base = *tmem_slot;
    // (the producers wait right before their first load; for the others, whose turn comes later, the wait is over by then)
    if (warp != 0 && warp != 2) pdl_wait();

    if (warp == 0 || warp == 2) {
        // ------------------------------------------------------------------ TMA producers: warp 0 feeds A, warp 2 feeds B
        const uint32_t leader = ptx::elect_one() ? 1u : 0u;
        const bool isA = warp == 0;
        const int kc_tail = p.tail32 ? p.kc_per_tap - 1 : -1;
        const uint32_t kb_bytes = isA ? (uint32_t)(TC_BM * p.KC * 2) : (uint32_t)(p.BN * p.KC * 2);
        const uint32_t base_u32 = ptx::smem_u32(isA ? sA : sB), stage_bytes = isA ? p.a_stage_bytes : p.b_stage_bytes, full_u32 = ptx::smem_u32(full);
        const CUtensorMap* tm_full = isA ? &p.tmA : &p.tmB[cls];
        const CUtensorMap* tm_tail = isA ? &p.tmA_t : &p.tmB_t[cls];
        const int m0 = m_tile * TC_BM;
        int cw0 = 0, ch0 = 0, n0 = 0;
        if (isA && !p.a_tiled) {
            const int j0 = m0 % p.Wq, t1 = m0 / p.Wq;
            const int i0 = t1 % p.Hq;
            n0 = t1 / p.Hq;
            cw0 = p.lo_w + j0 * p.ts;
            ch0 = p.lo_h + i0 * p.ts;
        }
        const int first = (kb0 + rot) % kblocks, ntaps = p.cls_ntaps[cls];
        int tap = first / p.kc_per_tap, kc = first - tap * p.kc_per_tap, s = 0, issued = 0;
        uint32_t ph = 0;
        bool ok = true;
        pdl_wait();
        if (MODE == 0 && isA) pdl_launch_dependents();  // (behind its own wait: see the end of common.cuh)
        for (int kb = kb0; kb < kb1; ++kb) {
            if (!wait_bar_fast(empty + s, ph ^ 1u, abort_flag, p.status, isA ? 1 : 5)) {
                ok = false;
                break;
            }
            const uint32_t bar = full_u32 + 8u * (uint32_t)s, dst = base_u32 + (uint32_t)s * stage_bytes;
            const bool tail = kc == kc_tail;
            ptx::mbar_expect_tx_u32_if(leader, bar, tail ? kb_bytes >> 1 : kb_bytes);
            const CUtensorMap* tm = tail ? tm_tail : tm_full;
            if (!isA) ptx::tma_load_2d_u32_if(leader, dst, tm, bar, tap * p.Ca + kc * p.KC, n_tile * p.BN);
            else if (p.a_tiled) ptx::tma_load_2d_u32_if(leader, dst, tm, bar, kc * p.KC, m0);
            else ptx::tma_load_im2col_4d_u32_if(leader, dst, tm, bar, kc * p.KC, cw0, ch0, n0, p.off_w[cls][tap], p.off_h[cls][tap]);
            if (++kc == p.kc_per_tap) {
                kc = 0;
                if (++tap == ntaps) tap = 0;
            }
            ++issued;
            if (++s == p.stages) {
                s = 0;
                ph ^= 1u;
            }
        }
        if (!ok) {  // gave up: wait (bounded) for the loads still in flight so that nothing lands after the CTA has exited
            const int back = issued < p.stages ? issued : p.stages;
            for (int b = 0; b < back; ++b) {
                s = (s == 0) ? p.stages - 1 : s - 1;
                if (s == p.stages - 1) ph ^= 1u;
                for (int i = 0; i < 100000 && !ptx::mbar_try_wait(full + s, ph); ++i) {
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        const uint32_t leader = ptx::elect_one() ? 1u : 0u;
        const int kc_tail = p.tail32 ? p.kc_per_tap - 1 : -1;
        const uint64_t tail_flip = ptx::make_smem_desc(0u, 16, p.sbo, p.umma_swizzle) ^ ptx::make_smem_desc(0u, 16, p.sbo >> 1, (uint32_t)ptx::kSwizzle64);
        const uint64_t da0 = ptx::make_smem_desc(ptx::smem_u32(sA), 16, p.sbo, p.umma_swizzle), db0 = ptx::make_smem_desc(ptx::smem_u32(sB), 16, p.sbo, p.umma_swizzle);
        const uint64_t a_stage16 = (uint64_t)(p.a_stage_bytes >> 4), b_stage16 = (uint64_t)(p.b_stage_bytes >> 4);
        const uint32_t empty_u32 = ptx::smem_u32(empty);
        int kc = (kb0 + rot) % kblocks % p.kc_per_tap, s = 0;
        uint32_t ph = 0, accumulate = 0;
        bool ok = true;
        for (int kb = kb0; kb < kb1; ++kb) {
            if (!wait_bar_fast(full + s, ph, abort_flag, p.status, 3)) {
                ok = false;
                break;
            }
            ptx::tc_fence_after();
            uint64_t da = da0 + (uint64_t)s * a_stage16, db = db0 + (uint64_t)s * b_stage16;
            const bool tail = kc == kc_tail;
            if (++kc == p.kc_per_tap) kc = 0;
            if (tail) {
                da ^= tail_flip;
                db ^= tail_flip;
            }
            ptx::umma_f16_if(leader, tmem_base, da, db, p.idesc, accumulate);
            ptx::umma_f16_if(leader, tmem_base, da + 2, db + 2, p.idesc, 1u);
            if (!tail) {
                ptx::umma_f16_if(leader, tmem_base, da + 4, db + 4, p.idesc, 1u);
                ptx::umma_f16_if(leader, tmem_base, da + 6, db + 6, p.idesc, 1u);
            }
            accumulate = 1u;
            ptx::umma_commit_u32_if(leader, empty_u32 + 8u * (uint32_t)s);
            if (++s == p.stages) {
                s = 0;
                ph ^= 1u;
            }
        }
        if (ok) {
            ptx::umma_commit_u32_if(leader, ptx::smem_u32(tfull));
        } else {  // tfull is never signalled; the MMAs already issued must have retired before TMEM is released
            ptx::umma_commit_u32_if(leader, ptx::smem_u32(drain));
            for (int i = 0; i < 4000000 && !ptx::mbar_try_wait(drain, 0); ++i) {
            }
        }
    } else if (MODE == 2) {
        // the other warps meanwhile derive the coefficients of this tile's columns (fp64, like the training-mode finalize)
        for (int c = (int)threadIdx.x - 96; c < p.BN; c += SP_THREADS - 96) {
            double sc = 0.0, sh = 0.0;
            const int ch = n_tile * p.BN + c;
            if (ch < p.ldo) bn_eval_coef(p.fin_gamma, p.fin_beta, p.fin_rmean, p.fin_rvar, p.fin_eps, ch, sc, sh);
            const double half = p.epi_act ? 0.5 : 1.0;  // (exact; see finish)
            red[c] = (float)(sc * half);
            red[p.BN + c] = (float)(sh * half);
        }
    }
    __syncwarp();

    // ---------------------------------------------------------------------- all warps: accumulators -> rounding -> rows
    bool ok = true;
    if (lane == 0) ok = wait_bar(tfull, 0, abort_flag, p.status, 4);
    ok = __syncthreads_and((int)(__shfl_sync(0xffffffffu, (int)ok, 0) != 0)) != 0;
    const int q = warp & 3, share = warp >> 2, c_lo = sp_part_lo(share, p.BN), nc = sp_part_lo(share + 1, p.BN) - c_lo;  // its rows and columns
    int sat_bits = 0;
    // act(v * scale + shift) of four neighbouring columns from c on (MODE 2), rounded and packed.  (With SiLU the
    // coefficients are halved.)
    auto finish = [&](const float* v, int c) {
        float2 a = make_float2(v[0], v[1]), b = make_float2(v[2], v[3]);
        if (MODE == 2) {
            const float4 sc = *reinterpret_cast<const float4*>(red + c), sh = *reinterpret_cast<const float4*>(red + p.BN + c);
            a = fma2(a, make_float2(sc.x, sc.y), make_float2(sh.x, sh.y));
            b = fma2(b, make_float2(sc.z, sc.w), make_float2(sh.z, sh.w));
            if (p.epi_act) {
                a = silu2_of_half(a);
                b = silu2_of_half(b);
            }
        }
        return make_uint2(pack2<OutT>(a.x, a.y, &sat_bits), pack2<OutT>(b.x, b.y, &sat_bits));
    };
    ptx::tc_fence_after();
    if constexpr (S == 1) {
        // MODE 1: the rounded rows for the channel sums, [quarter][32 rows] of BN * 2 + 16 bytes over the consumed operand stages
        const int srow = p.BN * 2 + 16, squarter = 32 * srow + 32;  // (32 bytes between the quarters: other banks)
        // A lane stores its row's 32 bytes of a piece at once.  Fewer instructions count most here, since a warp runs this code once:
        // a [128 x 48] tile leaves 0.75 us behind its last MMA, 1.0 with the rows staged in shared memory for stores of whole
        // lines, 2.3 when all accumulators went through shared memory to threads of four columns; [128 x 96] 1.4, 1.6 and 4.1.
        if (ok) {
            const int grow = m_tile * TC_BM + q * 32 + lane;  // (row counts of the tensor-core path fit 31 bits)
            bool live = grow < (int)p.M;
            long long orow = grow;
            if (MODE == 0 && p.os != 1) {
                const unsigned t1 = (unsigned)grow / (unsigned)p.Wq, n = t1 / (unsigned)p.Hq;
                const int oi = (int)(t1 - n * (unsigned)p.Hq) * p.os + p.cls_oa[cls], oj = (grow - (int)t1 * p.Wq) * p.os + p.cls_ob[cls];
                live = live && oi < p.Hout && oj < p.Wout;  // (odd extents: the grid of an odd parity is longer than the image)
                orow = ((long long)n * p.Hout + oi) * p.Wout + oj;
            }
            OutT* const dst = static_cast<OutT*>(p.out) + orow * p.ld_out + n_tile * p.BN;
            const bool wide = ((reinterpret_cast<uintptr_t>(p.out) | (uintptr_t)p.ld_out * 2) & 31) == 0;  // (pieces start at multiples of 32 bytes)
            const int cols = p.ldo - n_tile * p.BN;  // columns of this tile that exist (a multiple of 8)
            uint8_t* const staged = smem + (size_t)q * squarter + (size_t)lane * srow;
#pragma unroll 1
            for (int c = c_lo; c < c_lo + nc; c += 16) {
                uint32_t r[16];
                __syncwarp();  // (lanes without a row have left the last iteration early)
                ptx::tmem_ld_32x32b_x16(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)c, r);
                ptx::tmem_ld_wait();
                const int before = sat_bits;
                uint2 o[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) o[j] = finish(reinterpret_cast<const float*>(r) + 4 * j, c + 4 * j);
                if (MODE == 1) {
                    *reinterpret_cast<uint4*>(staged + c * 2) = make_uint4(o[0].x, o[0].y, o[1].x, o[1].y);
                    *reinterpret_cast<uint4*>(staged + c * 2 + 16) = make_uint4(o[2].x, o[2].y, o[3].x, o[3].y);
                }
                if (!live) {
                    sat_bits = before;
                    continue;
                }
                if (MODE == 0 && p.out_accumulate) {  // the rounded tile is added, as a TMA reduction would
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (c + 4 * j >= cols) break;
                        const uint2 old = *reinterpret_cast<const uint2*>(dst + c + 4 * j);
                        const OutT *po = reinterpret_cast<const OutT*>(&old), *pn = reinterpret_cast<const OutT*>(&o[j]);
                        uint2 sum;
                        OutT* ps = reinterpret_cast<OutT*>(&sum);
                        pair_from_f32(ps, add2(pair_to_f32(po), pair_to_f32(pn)));
                        pair_from_f32(ps + 2, add2(pair_to_f32(po + 2), pair_to_f32(pn + 2)));
                        o[j] = sum;
                    }
                }
                if (wide && c + 16 <= cols) {
                    st_global32(dst + c, o);
                } else {
                    if (c < cols) *reinterpret_cast<uint4*>(dst + c) = make_uint4(o[0].x, o[0].y, o[1].x, o[1].y);
                    if (c + 8 < cols) *reinterpret_cast<uint4*>(dst + c + 8) = make_uint4(o[2].x, o[2].y, o[3].x, o[3].y);
                }
            }
        }
        ptx::tc_fence_before();
        __syncthreads();
        for (int piece = warp; MODE == 1 && ok && piece < p.BN / 16; piece += SP_THREADS / 32) {
            // channel sums of the rounded values: a lane takes two channels of one quarter's 32 rows, even and odd rows apart, then
            // the four quarters are added in order (the persistent kernel's grouping; rows past the last pixel are zeros)
            const int c2 = piece * 8 + (lane & 7), grp = lane >> 3;
            float2 sa = make_float2(0.f, 0.f), sb = sa, qa = sa, qb = sa;
            const uint8_t* src = smem + (size_t)grp * squarter + c2 * 4;
#pragma unroll
            for (int rr = 0; rr < 32; rr += 2) {
                const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(src + rr * srow));
                const float2 f1 = __half22float2(*reinterpret_cast<const __half2*>(src + (rr + 1) * srow));
                sa = add2(sa, f0);
                sb = add2(sb, f1);
                qa = fma2(f0, f0, qa);
                qb = fma2(f1, f1, qb);
            }
            float v[4] = {sa.x + sb.x, sa.y + sb.y, qa.x + qb.x, qa.y + qb.y};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float v1 = __shfl_down_sync(0xffffffffu, v[e], 8), v2 = __shfl_down_sync(0xffffffffu, v[e], 16), v3 = __shfl_down_sync(0xffffffffu, v[e], 24);
                v[e] = ((v[e] + v1) + v2) + v3;
            }
            const int ch = n_tile * p.BN + 2 * c2;
            if (grp == 0 && ch < p.ldo) {
#pragma unroll
                for (int e = 0; e < 4; ++e) chan_acc_add<false>(p.acc, p.ldo, e >> 1, ch + (e & 1), v[e]);
            }
        }
    } else {
        // Every CTA's share of the sums goes to the rank that owns the rows: into this CTA's own shared memory (over the consumed
        // stages), from there as bulk copies, which a rank counts on its barrier `shares`.  Then each rank adds in rank order.
        // (Loads of the shares from the peers behind a cluster barrier: 2.4 us for [32 x 96] of four ranks; stores into the peers'
        // memory, 16 bytes of 32 rows at a time: 1.8 us and a cluster barrier of 1 us.)
        ptx::cluster_wait();
        if (ok && nc) {
            float* const mine = reinterpret_cast<float*>(smem) + TC_BM * (c_lo + 4 * share) + q * 32 * (nc + 4);
#pragma unroll 1
            for (int c = 0; c < nc; c += 16) {
                uint32_t r[16];
                ptx::tmem_ld_32x32b_x16(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(c_lo + c), r);
                ptx::tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 16; j += 4) *reinterpret_cast<uint4*>(mine + lane * (nc + 4) + c + j) = make_uint4(r[j], r[j + 1], r[j + 2], r[j + 3]);
            }
            ptx::fence_async_smem();
            __syncwarp();
            constexpr int CHUNK = ROWS < 32 ? ROWS : 32;  // rows of this warp that go to one rank
            if (lane < 32 / CHUNK) {
                const int row = q * 32 + lane * CHUNK;
                const uint32_t to = (uint32_t)(row / ROWS);
                copy_to_peer(ptx::mapa_u32(ptx::smem_u32(part + (size_t)rank * slot + ROWS * (c_lo + 4 * share) + row % ROWS * (nc + 4)), to), mine + lane * CHUNK * (nc + 4),
                             (uint32_t)(CHUNK * (nc + 4) * 4), ptx::mapa_u32(ptx::smem_u32(shares), to));
            }
        }
        ptx::tc_fence_before();
        if (lane == 0 && ok) ok = wait_bar(shares, 0, abort_flag, p.status, 4);
        ok = __syncthreads_and((int)(__shfl_sync(0xffffffffu, (int)ok, 0) != 0)) != 0;
        ptx::cluster_arrive_relaxed();
        if (ok) {
            // a thread keeps a group of four columns
            const int groups = p.BN / 4, r0 = (int)threadIdx.x / groups, rp = SP_THREADS / groups, c = ((int)threadIdx.x - r0 * groups) * 4;
            const int from = sp_part_of(c, p.BN), from_lo = sp_part_lo(from, p.BN), from_pitch = sp_part_lo(from + 1, p.BN) - from_lo + 4;
            const float* const base = part + ROWS * (from_lo + 4 * from) + c - from_lo;
            const int row_end = r0 < rp && c < p.ldo - n_tile * p.BN ? min(ROWS, (int)p.M - m_tile * TC_BM - rank * ROWS) : 0;
            OutT* const dst = static_cast<OutT*>(p.out) + (long long)(m_tile * TC_BM + rank * ROWS) * p.ld_out + n_tile * p.BN + c;
#pragma unroll 1
            for (int row = r0; row < row_end; row += rp) {
                const float* const src = base + row * from_pitch;
                float4 v[S];
#pragma unroll
                for (int j = 0; j < S; ++j) v[j] = *reinterpret_cast<const float4*>(src + (size_t)j * slot);
#pragma unroll
                for (int j = 1; j < S; ++j) {
                    v[0].x += v[j].x;
                    v[0].y += v[j].y;
                    v[0].z += v[j].z;
                    v[0].w += v[j].w;
                }
                *reinterpret_cast<uint2*>(dst + (long long)row * p.ld_out) = finish(reinterpret_cast<const float*>(&v[0]), c);
            }
        }
    }
    if (sat_bits & (int)0x80008000u) atomicAdd(p.status + ST_SAT, 1);
    __syncwarp();  // (what follows wants whole warps)
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }
    if (S > 1) ptx::cluster_wait();  // every rank has its shares: nobody reads this CTA's shared memory any more
}

}  // namespace nbcbs
