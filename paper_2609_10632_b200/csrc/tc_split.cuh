// Implicit GEMM for layers with few output tiles (one or two images at 40 x 40 and below), sm_100a.
// The persistent kernel of tc_conv.cuh gives such a layer a handful of CTAs, each of which walks the whole K range alone:
// 288 -> 288 3x3 on one 20 x 20 image is 8 tiles of 45 k-blocks on 148 SMs, 20 us of one CTA's operand fetches.  Here the
// K range of a tile is cut over a CLUSTER of 1, 2, 4 or 8 CTAs.  Every CTA accumulates its share in TMEM, leaves it as fp32
// in its own shared memory, and after one cluster barrier CTA r sums rows [128 r / S, 128 (r + 1) / S) of all S partial
// tiles through distributed shared memory, in rank order (the same bits every run), applies the epilogue and stores.
// The training calls use clusters of one (narrow tiles only): the sum of an element then runs over the k-blocks in the order
// in which the persistent kernel would add them (the same starting k-block), and the channel sums are formed as there, so
// that the results of a training step do not depend on which of the two kernels a layer gets -- a deep network in training
// mode turns a difference in the last bit of one layer into percents a few dozen layers on.
// No block waits for a block outside its cluster.  Bound: latency -- operand fetch to first MMA, the k-blocks of one CTA
// (a k-block is (128 + BN) 128-byte rows through TMA), accumulator -> shared memory -> peers -> rounding -> store.
// The narrow tiles (BN <= 128, often 32 to 64) are part of the same idea: more CTAs, and less to hand over.
// Measured against the persistent kernel: see split_configure below.
// Included by tc_conv.cuh (uses its parameter record and bounded-wait helpers).
#pragma once

namespace nbcbs {

constexpr int SP_THREADS = 256;

__device__ __forceinline__ float4 ld_dsmem4(uint32_t cluster_addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(cluster_addr) : "memory");
    return v;
}
__device__ __forceinline__ void prefetch_tile_2d(const CUtensorMap* m, int c0, int c1) {
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(reinterpret_cast<uint64_t>(m)), "r"(c0), "r"(c1) : "memory");
}

// MODE 0: plain 16-bit output (data gradient; may be pitched, may be added to what the output holds).  MODE 1: training
// forward (fp16 output, channel sums of the rounded values to the accumulators).  MODE 2: per-channel scale and shift, SiLU.
template <typename OutT, int MODE>
__global__ void __launch_bounds__(SP_THREADS, 1) tc_split_kernel(const __grid_constant__ IgemmParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* sA = smem;
    uint8_t* sB = sA + (size_t)p.stages * p.a_stage_bytes;
    float* part = reinterpret_cast<float*>(smem);  // [128][BN + 4] this CTA's share, over the operand stages once they are consumed
    const int S = p.split, pitch = p.BN + 4;
    const size_t stage_total = (size_t)p.stages * (p.a_stage_bytes + p.b_stage_bytes), part_total = (size_t)TC_BM * pitch * 4;
    float* red = reinterpret_cast<float*>(smem + ((stage_total > part_total ? stage_total : part_total) + 15) / 16 * 16);  // MODE 1: channel sums [4][2][BN]; MODE 2: scale, shift [2][BN]
    uint64_t* bars = reinterpret_cast<uint64_t*>(red + 8 * 128);
    uint64_t* full = bars;
    uint64_t* empty = bars + p.stages;
    uint64_t* tfull = empty + p.stages;
    uint64_t* drain = tfull + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
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
        *abort_flag = 0;
        ptx::fence_mbar_init();
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
    const uint32_t tmem_base = *tmem_slot;

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
        // warps 3-7 meanwhile derive the coefficients of this tile's columns (fp64, like the training-mode finalize)
        pdl_wait();
        for (int c = (int)threadIdx.x - 96; c < p.BN; c += SP_THREADS - 96) {
            double sc = 0.0, sh = 0.0;
            const int ch = n_tile * p.BN + c;
            if (ch < p.ldo) bn_eval_coef(p.fin_gamma, p.fin_beta, p.fin_rmean, p.fin_rvar, p.fin_eps, ch, sc, sh);
            red[c] = (float)sc;
            red[p.BN + c] = (float)sh;
        }
    }
    __syncwarp();

    // ---------------------------------------------------------------------- all eight warps: TMEM -> own shared memory
    bool ok = true;
    if (lane == 0) ok = wait_bar(tfull, 0, abort_flag, p.status, 4);
    ok = __syncthreads_and((int)(__shfl_sync(0xffffffffu, (int)ok, 0) != 0)) != 0;
    if (ok) {
        ptx::tc_fence_after();
        const int q = warp & 3;  // TMEM lanes (rows) 32 q .. 32 q + 31; the two warps of a quarter take alternate 16-column pieces
        float* row = part + (size_t)(q * 32 + lane) * pitch;
        for (int c = (warp >> 2) * 16; c < p.BN; c += 32) {
            uint32_t r[16];
            ptx::tmem_ld_32x32b_x16(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)c, r);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 16; j += 4)
                *reinterpret_cast<float4*>(row + c + j) = make_float4(__uint_as_float(r[j]), __uint_as_float(r[j + 1]), __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]));
        }
        ptx::tc_fence_before();
    }
    if (S > 1) ptx::cluster_sync_all(); else __syncthreads();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }

    // ---------------------------------------------------------------------- sum this CTA's rows over the cluster, epilogue, store
    pdl_wait();
    if (ok) {
        const int ng = p.BN / 4, rows = TC_BM / S, rp = SP_THREADS / ng;  // a thread keeps one group of four columns
        const int gi = (int)threadIdx.x % ng, r0 = (int)threadIdx.x / ng;
        const int col = n_tile * p.BN + gi * 4;
        const bool live = r0 < rp && col < p.ldo;
        const uint32_t part_u32 = ptx::smem_u32(part);
        float4 sc = make_float4(0.f, 0.f, 0.f, 0.f), sh = sc;
        if (MODE == 2) {
            sc = *reinterpret_cast<const float4*>(red + gi * 4);
            sh = *reinterpret_cast<const float4*>(red + p.BN + gi * 4);
        }
        int sat_bits = 0;
        for (int row = r0; live && row < rows; row += rp) {
            const int grow = m_tile * TC_BM + rank * rows + row;  // (row counts of the tensor-core path fit 31 bits)
            if (grow >= (int)p.M) break;
            const uint32_t at = part_u32 + (uint32_t)(((rank * rows + row) * pitch + gi * 4) * 4);
            float4 v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (j < S) v[j] = S > 1 ? ld_dsmem4(ptx::mapa_u32(at, (uint32_t)j)) : *reinterpret_cast<const float4*>(part + (size_t)row * pitch + gi * 4);
            float4 a = v[0];
#pragma unroll
            for (int j = 1; j < 8; ++j)
                if (j < S) {
                    a.x += v[j].x;
                    a.y += v[j].y;
                    a.z += v[j].z;
                    a.w += v[j].w;
                }
            if (MODE == 2) {
                float2 z0 = fma2(make_float2(a.x, a.y), make_float2(sc.x, sc.y), make_float2(sh.x, sh.y));
                float2 z1 = fma2(make_float2(a.z, a.w), make_float2(sc.z, sc.w), make_float2(sh.z, sh.w));
                if (p.epi_act) {
                    z0 = mul2(z0, sigmoid2<true>(z0));
                    z1 = mul2(z1, sigmoid2<true>(z1));
                }
                a = make_float4(z0.x, z0.y, z1.x, z1.y);
            }
            uint2 o;
            o.x = pack2<OutT>(a.x, a.y, &sat_bits);
            o.y = pack2<OutT>(a.z, a.w, &sat_bits);
            long long orow = grow;
            if (p.os != 1) {
                const unsigned t1 = (unsigned)grow / (unsigned)p.Wq, n = t1 / (unsigned)p.Hq;
                const int oi = (int)(t1 - n * (unsigned)p.Hq) * p.os + p.cls_oa[cls], oj = (grow - (int)t1 * p.Wq) * p.os + p.cls_ob[cls];
                if (oi >= p.Hout || oj >= p.Wout) continue;  // (odd extents: the grid of an odd parity is longer than the image)
                orow = ((long long)n * p.Hout + oi) * p.Wout + oj;
            }
            OutT* dst = static_cast<OutT*>(p.out) + orow * p.ld_out + col;
            if (MODE == 0 && p.out_accumulate) {  // the rounded tile is added, as a TMA reduction would
                const uint2 old = *reinterpret_cast<const uint2*>(dst);
                const OutT *po = reinterpret_cast<const OutT*>(&old), *pn = reinterpret_cast<const OutT*>(&o);
                uint2 sum;
                OutT* ps = reinterpret_cast<OutT*>(&sum);
                pair_from_f32(ps, add2(pair_to_f32(po), pair_to_f32(pn)));
                pair_from_f32(ps + 2, add2(pair_to_f32(po + 2), pair_to_f32(pn + 2)));
                o = sum;
            }
            *reinterpret_cast<uint2*>(dst) = o;
        }
        int sat = sat_bits & (int)0x80008000u ? 1 : 0;
        if (MODE == 1) {
            // channel sums of the rounded values: a thread takes two channels of 32 rows, even and odd rows apart, then the
            // four row groups are added in order (the persistent kernel's grouping; rows past the last pixel are zeros)
            const int c2 = (int)threadIdx.x % (p.BN / 2), grp = (int)threadIdx.x / (p.BN / 2);
            if (grp < 4) {
                float2 sa = make_float2(0.f, 0.f), sb = sa, qa = sa, qb = sa;
                const float* src = part + (size_t)grp * 32 * pitch + 2 * c2;
#pragma unroll 8
                for (int rr = 0; rr < 32; rr += 2) {
                    const float2 a0 = *reinterpret_cast<const float2*>(src + (size_t)rr * pitch), a1 = *reinterpret_cast<const float2*>(src + (size_t)(rr + 1) * pitch);
                    const uint32_t h0 = pack2<__half>(a0.x, a0.y, nullptr), h1 = pack2<__half>(a1.x, a1.y, nullptr);
                    const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&h0)), f1 = __half22float2(*reinterpret_cast<const __half2*>(&h1));
                    sa = add2(sa, f0);
                    sb = add2(sb, f1);
                    qa = fma2(f0, f0, qa);
                    qb = fma2(f1, f1, qb);
                }
                const float qx = qa.x + qb.x, qy = qa.y + qb.y;
                float* dst = red + (size_t)grp * 2 * p.BN + 2 * c2;
                *reinterpret_cast<float2*>(dst) = make_float2(sa.x + sb.x, sa.y + sb.y);
                *reinterpret_cast<float2*>(dst + p.BN) = make_float2(qx, qy);
            }
            __syncthreads();
            for (int e = threadIdx.x; e < 2 * p.BN; e += SP_THREADS) {
                const int c = e >= p.BN ? e - p.BN : e;
                if (n_tile * p.BN + c >= p.ldo) continue;
                const float* b = red + e;
                chan_acc_add<false>(p.acc, p.ldo, e >= p.BN ? 1 : 0, n_tile * p.BN + c, ((b[0] + b[2 * p.BN]) + b[4 * p.BN]) + b[6 * p.BN]);
            }
        }
        if (sat) atomicAdd(p.status + ST_SAT, sat);
    }
    if (S > 1) ptx::cluster_sync_all();  // no CTA leaves while a peer may still read its rows
}

}  // namespace nbcbs
