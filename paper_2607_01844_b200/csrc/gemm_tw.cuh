// Weight gradients on CTA pairs: dW[e] = A_e^T B_e with the expert's rows as K, one 256 x 256 tile of fp32 per pair
// (tcgen05.mma.cta_group::2, M = 256, N = 256).  Each CTA fetches its own 128 columns of A and half of B's 256 columns, 32 KiB
// per 64 rows where the one-CTA kernel (TC_WD, TC_WGU in gemm_tc.cuh) fetches 48 for the same 128 x 256 outputs, so that five
// stages fit beside the store boxes instead of three.  That pays where an expert has many rows (the loads share the SM's path
// to L2 with the tile's 128 KiB of stores); with few rows the stores alone set the pace and the single CTAs keep them steadier.
//
// K tail: rows past the expert's end in the last group of 16 belong to the next expert and are cleared in both operands.  The
// block that holds them does not complete on the leader's barrier: each CTA waits for its own half on a barrier of its own,
// clears it, and then arrives on the leader's (which expects two arrivals: both the leader's producer's for an ordinary block;
// an arrival of the other CTA's producer per block, and a wait that acquires at cluster scope, cost a quarter of the kernel's time).
//
// Everything else (tile order, epilogue with TMA tile stores, bounded waits, experts without rows) is as in the one-CTA kernel.
#pragma once
#include "gemm_tc2.cuh"

namespace mop {

constexpr int TW_STAGES = 5;
constexpr int TW_OP_BYTES = 2 * TC_CHUNK_BYTES;      // 16 KiB: 128 columns of an operand x 64 rows
constexpr int TW_STAGE_BYTES = 2 * TW_OP_BYTES;
constexpr int TW_EPI_WARPS = 8;
constexpr int TW_THREADS = 64 + 32 * TW_EPI_WARPS;
constexpr int TW_SMEM_BYTES = TW_STAGES * TW_STAGE_BYTES + 1024 /*align*/ + TC_BAR_BYTES + 4 * 16384;

__device__ __forceinline__ void tma2_load_2d_hint(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], "
        "[%1, {%3, %4}], [%2], %5;" ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "l"(policy)
        : "memory");
}

template <int KIND>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TW_THREADS, 1)
tw_wgrad_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB0,
                const __grid_constant__ CUtensorMap tmB1, const __grid_constant__ CUtensorMap tmO0,
                const __grid_constant__ CUtensorMap tmO1, const TcArgs args) {
    static_assert(KIND == TC_WD || KIND == TC_WGU, "weight gradients");
    constexpr bool SEL_B = TcTraits<KIND>::SEL_B;
    constexpr int S = TW_STAGES;
    extern __shared__ uint8_t tc_smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S * TW_STAGE_BYTES);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 3 * S + 4);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = warp_index(), lane = threadIdx.x % 32;
    const uint32_t rank = cluster_ctarank();
    const bool leader = rank == 0;
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t bar_base = smem_u32(bars);
    auto full_bar = [&](int s) { return bar_base + 8u * s; };               // the leader's are used
    auto empty_bar = [&](int s) { return bar_base + 8u * (S + s); };
    auto tail_bar = [&](int s) { return bar_base + 8u * (2 * S + s); };     // each CTA its own
    auto tfull_bar = [&](int b) { return bar_base + 8u * (3 * S + b); };
    auto tempty_bar = [&](int b) { return bar_base + 8u * (3 * S + 2 + b); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(full_bar(s), 2); mbar_init(empty_bar(s), 1); mbar_init(tail_bar(s), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(tfull_bar(b), 1); mbar_init(tempty_bar(b), 2 * TW_EPI_WARPS); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tma_prefetch_desc(&tmA); tma_prefetch_desc(&tmB0); tma_prefetch_desc(&tmO0);
        if (SEL_B) { tma_prefetch_desc(&tmB1); tma_prefetch_desc(&tmO1); }
    }
    if (warp == 1) tmem2_alloc(smem_u32(tmem_slot), 512);
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    pdl_begin_gemm(args.gemm_follows, PdlNote{});

    const int per_e = args.tiles_m_fixed * args.tiles_n;      // tiles_m_fixed: 256-row blocks of the gradient
    const int total_tiles = args.E * per_e;
    const int cluster_id = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;
    auto decode = [&](int t) {
        TileInfo ti;
        ti.e = t / per_e;
        const int r = t - ti.e * per_e;
        ti.m0 = (r / args.tiles_n) * 256 + 128 * (int)rank;
        ti.nt = r % args.tiles_n;
        ti.sel = 0;
        if constexpr (SEL_B) {
            const int half_n = args.tiles_n >> 1;
            if (ti.nt >= half_n) { ti.nt -= half_n; ti.sel = 1; }
        }
        ti.row0 = __ldg(args.offsets + ti.e);
        ti.rows = __ldg(args.offsets + ti.e + 1) - ti.row0;
        ti.skip = ti.rows <= 0;
        return ti;
    };
    // clears the rows [valid, next multiple of 16) of this CTA's half of a stage
    auto clear_tail = [&](int stage, int valid) {
        uint8_t* b = smem + stage * TW_STAGE_BYTES;
        const int n16 = (((valid + 15) & ~15) - valid) * 8;
        for (int i = lane; i < n16; i += 32) {
            const int off = (valid + (i >> 3)) * 128 + (i & 7) * 16;
#pragma unroll
            for (int ch = 0; ch < TW_STAGE_BYTES / TC_CHUNK_BYTES; ++ch)
                *reinterpret_cast<uint4*>(b + ch * TC_CHUNK_BYTES + off) = make_uint4(0, 0, 0, 0);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
    };

    if (warp == 0) {
        // ===================================================================== TMA producer (both CTAs)
        const bool el = elect_one();
        int stage = 0; uint32_t phase = 0; bool alive = true;
        const uint64_t keep = l2_policy_evict_last();
        TileInfo nxt = decode(min(cluster_id, max(total_tiles - 1, 0)));
        int expert = -1, ahead = 0;
        const int rows_total = __ldg(args.offsets + args.E);
        for (int t = cluster_id; t < total_tiles && alive; t += n_clusters) {
            const TileInfo ti = nxt;
            if (t + n_clusters < total_tiles) nxt = decode(t + n_clusters);
            if (ti.skip) continue;
            if (ti.e != expert) { expert = ti.e; wgrad_prefetch(args, ti.row0 + ti.rows, rows_total, ahead); }
            const int nb = ti.nt * 256 + 128 * (int)rank;
            const int nkb = (ti.rows + TC_BK - 1) / TC_BK;
            const CUtensorMap* mb = (SEL_B && ti.sel) ? &tmB1 : &tmB0;
            for (int kb = 0; kb < nkb; ++kb) {
                if (!mbar_wait_all(empty_bar(stage), phase ^ 1u, abort_flag, args.status, STATUS_WAIT_EMPTY)) {
                    alive = false; break;
                }
                const uint32_t sA = smem_base + stage * TW_STAGE_BYTES;
                const uint32_t sB = sA + TW_OP_BYTES;
                const int krow = ti.row0 + kb * TC_BK;
                const bool tail = kb + 1 == nkb && (ti.rows & 15) != 0;
                const uint32_t bar = tail ? tail_bar(stage) : full_bar(stage) & T2_PEER_MASK;
                if (el) {
                    if (tail) mbar_expect_tx(tail_bar(stage), TW_STAGE_BYTES);
                    else if (leader) { mbar_expect_tx(full_bar(stage), 2 * TW_STAGE_BYTES); mbar_arrive(full_bar(stage)); }
                    if (!args.a_split) tma2_load_3d_hint(sA, &tmA, bar, 0, krow, ti.m0 >> 6, keep);
                    else {
                        tma2_load_2d_hint(sA, &tmA, bar, ti.m0, krow, keep);
                        tma2_load_2d_hint(sA + TC_CHUNK_BYTES, &tmA, bar, ti.m0 + 64, krow, keep);
                    }
                    if (!args.b_split) tma2_load_3d_hint(sB, mb, bar, 0, krow, nb >> 6, keep);
                    else {
                        tma2_load_2d_hint(sB, mb, bar, nb, krow, keep);
                        tma2_load_2d_hint(sB + TC_CHUNK_BYTES, mb, bar, nb + 64, krow, keep);
                    }
                }
                if (++stage == S) { stage = 0; phase ^= 1u; }
            }
        }
    } else if (warp == 1) {
        // ===================================================================== MMA issuer (leader), tails (both)
        const bool el = elect_one();
        constexpr uint32_t idesc = make_idesc2(true, true);
        const uint64_t desc = smem_desc(0, TC_CHUNK_BYTES, 1024);
        int stage = 0; uint32_t phase = 0, tail_phase = 0; int it = 0; bool alive = true;
        TileInfo nxt = decode(min(cluster_id, max(total_tiles - 1, 0)));
        for (int t = cluster_id; t < total_tiles && alive; t += n_clusters) {
            const TileInfo ti = nxt;
            if (t + n_clusters < total_tiles) nxt = decode(t + n_clusters);
            if (ti.skip) continue;
            const int nkb = (ti.rows + TC_BK - 1) / TC_BK;
            const int buf = it & 1;
            const uint32_t d_tmem = tmem_base + (uint32_t)buf * TC_BN;
            if (leader) {
                if (!mbar_wait_all(tempty_bar(buf), ((uint32_t)(it >> 1) & 1u) ^ 1u, abort_flag, args.status,
                                   STATUS_WAIT_TMEM_EMPTY)) break;
                tc_fence_after();
            }
            for (int kb = 0; kb < nkb; ++kb) {
                const int valid = ti.rows - kb * TC_BK;
                int n_k4 = TC_BK / 16;
                if (valid < TC_BK) {
                    n_k4 = (valid + 15) >> 4;
                    if (valid & 15) {
                        if (!mbar_wait_all(tail_bar(stage), (tail_phase >> stage) & 1u, abort_flag, args.status,
                                           STATUS_WAIT_FULL)) { alive = false; break; }
                        tail_phase ^= 1u << stage;
                        clear_tail(stage, valid);
                        if (el) mbar_arrive_cluster(full_bar(stage) & T2_PEER_MASK);
                    }
                }
                if (leader) {
                    // (a cleared tail was written by the other CTA's threads as well: that wait acquires at cluster scope)
                    const bool ok = valid < TC_BK ? mbar_wait_cluster(full_bar(stage), phase, abort_flag, args.status, STATUS_WAIT_FULL)
                                                  : mbar_wait(full_bar(stage), phase, abort_flag, args.status, STATUS_WAIT_FULL);
                    if (!__all_sync(0xffffffffu, ok)) { alive = false; break; }
                    tc_fence_after();
                    const uint32_t sA = smem_base + stage * TW_STAGE_BYTES;
                    const uint64_t da = desc | (uint64_t)((sA & 0x3ffffu) >> 4);
                    const uint64_t db = desc | (uint64_t)(((sA + TW_OP_BYTES) & 0x3ffffu) >> 4);
                    if (el) {
#pragma unroll
                        for (int k4 = 0; k4 < TC_BK / 16; ++k4)
                            if (k4 < n_k4) umma2_bf16(d_tmem, da + k4 * (2048 >> 4), db + k4 * (2048 >> 4), idesc, (kb | k4) != 0 ? 1u : 0u);
                        umma2_commit_both(empty_bar(stage));
                    }
                }
                if (++stage == S) { stage = 0; phase ^= 1u; }
            }
            if (!alive) break;
            if (leader && el) umma2_commit_both(tfull_bar(buf));
            ++it;
        }
    } else {
        // ===================================================================== epilogue (8 warps, both CTAs)
        const int quarter = warp & 3;            // TMEM lanes 32*quarter .. +31 belong to this warp
        const int half = (warp - 2) >> 2;        // columns [128*half, 128*half + 128) of the tile
        const int r = quarter * 32 + lane;
        const int gbar = 1 + half;               // named barrier of this half's 128 threads
        uint8_t* gbase = smem + S * TW_STAGE_BYTES + TC_BAR_BYTES + half * 32768;
        const bool issuer = (quarter == 0 && lane == 0);
        const uint64_t stream_out = l2_policy_evict_first();
        int sbuf = 0, it = 0;
        TileInfo nxt = decode(min(cluster_id, max(total_tiles - 1, 0)));
        for (int t = cluster_id; t < total_tiles; t += n_clusters) {
            const TileInfo ti = nxt;
            if (t + n_clusters < total_tiles) nxt = decode(t + n_clusters);
            const int n0 = ti.nt * 256;
            if (ti.skip) {
                // expert without rows: its gradient is zero (or unchanged when accumulating)
                if (!args.ep.accumulate && !args.keep_empty && half == 0 && ti.m0 + r < args.Mfix) {
                    const size_t ro = ((size_t)ti.e * args.Mfix + ti.m0 + r) * args.N;
                    float* dst = (SEL_B && ti.sel) ? args.outf1 : args.ep.outf;
                    for (int c = 0; c < TC_BN; c += 4)
                        if (n0 + c < args.N) *reinterpret_cast<float4*>(dst + ro + n0 + c) = make_float4(0, 0, 0, 0);
                }
                continue;
            }
            const int buf = it & 1;
            bool ready = mbar_wait_warp(tfull_bar(buf), (uint32_t)(it >> 1) & 1u, abort_flag, args.status, STATUS_WAIT_TMEM_FULL, lane);
            ready = bar_vote_all(gbar, 128, ready);    // the four warps of a half meet at barriers below: all or none
            if (!ready) break;
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)buf * TC_BN + half * 128;
            const CUtensorMap* mo = (SEL_B && ti.sel) ? &tmO1 : &tmO0;
            float a0[32], a1[32], a2[32], a3[32];
            tmem_ld32_nowait(taddr, a0);
            tmem_ld32_nowait(taddr + 32, a1);
            tmem_ld32_nowait(taddr + 64, a2);
            tmem_ld32_nowait(taddr + 96, a3);
            tmem_ld_wait4(a0, a1, a2, a3);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(tempty_bar(buf) & T2_PEER_MASK);
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) {
                uint8_t* box = gbase + (sbuf & 1) * 16384;
                uint8_t* rowp = box + r * 128;
                const float(&v)[32] = cc == 0 ? a0 : cc == 1 ? a1 : cc == 2 ? a2 : a3;
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    *reinterpret_cast<float4*>(rowp + ((j ^ (lane & 7)) << 4)) =
                        make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                if (issuer) tma_store_wait_read<0>();
                asm volatile("bar.sync %0, 128;" ::"r"(gbar) : "memory");
                if (issuer) {
                    const int gcol = n0 + half * 128 + 32 * cc;
                    if (gcol < args.N && ti.m0 < args.Mfix) {
                        if (args.ep.accumulate) tma_reduce_add_3d(mo, smem_u32(box), gcol, ti.m0, ti.e);
                        else tma_store_3d_hint(mo, smem_u32(box), gcol, ti.m0, ti.e, stream_out);
                    }
                    tma_store_commit();
                }
                ++sbuf;
            }
            ++it;
        }
        if (issuer) tma_store_wait_all();        // boxes read before the CTA exits
    }

    // ------------------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000ll) __nanosleep(1000);
        __syncthreads();
    }
    cluster_sync_all();
    if (warp == 1) {
        tc_fence_after();
        tmem2_dealloc(tmem_base, 512);
    }
}

// ------------------------------------------------------------------------------------------ host
inline mop_status tw_init() {
    return cudaFuncSetAttribute(tw_wgrad_kernel<TC_WD>, cudaFuncAttributeMaxDynamicSharedMemorySize, TW_SMEM_BYTES) == cudaSuccess &&
                   cudaFuncSetAttribute(tw_wgrad_kernel<TC_WGU>, cudaFuncAttributeMaxDynamicSharedMemorySize, TW_SMEM_BYTES) == cudaSuccess
               ? MOP_OK : MOP_ERR_CUDA;
}
template <int KIND>
inline mop_status tw_launch(const TcPlan* p, const char* name, const CUtensorMap& a, const CUtensorMap& b0, const CUtensorMap& b1,
                            const CUtensorMap& o0, const CUtensorMap& o1, const TcArgs& args, cudaStream_t st) {
    p->prof->begin(name, st);
    pdl_launch(tw_wgrad_kernel<KIND>, p->sm_count & ~1, TW_THREADS, TW_SMEM_BYTES, st, a, b0, b1, o0, o1, args);
    p->prof->end(st);
    return cudaGetLastError() == cudaSuccess ? MOP_OK : MOP_ERR_CUDA;
}

}  // namespace mop
