// Host-side orchestration of the tensor-core grouped GEMMs: tensor maps, tile tables, launches.
#pragma once
#include "gemm_tc.cuh"
#include "gemm_tc2.cuh"
#include "gemm_tn.cuh"
#include "gemm_tw.cuh"

namespace mop {

// Schedules of the token-row kinds (TcPlan::pairs): 0 = one-CTA kernel on 128-row tiles; 1 = two-CTA
// kernel on 256-row pairs (the last pair of an expert may be partly empty); 2 = mixed: full pairs on
// the two-CTA kernel, the remaining < 256 rows of each expert on the one-CTA kernel.
inline size_t tc_tables_bytes(int M, int E) { return 3 * tc_tile_table_bytes(M, E); }

inline mop_status tc_build_row_tiles(const TcPlan* p, const int32_t* offsets, int32_t* tiles, cudaStream_t st) {
    int32_t* tiles2 = tiles + tc_tile_table_bytes(p->s.T * p->s.k, p->s.E) / 4;
    if (p->pairs == 2) return tc2_build_mixed(p, offsets, tiles, tiles2, st);
    if (p->pairs == 1) return tc2_build_tiles(p, offsets, tiles, st);
    return tc_build_tiles(p, offsets, tiles, st);
}

// One token-row GEMM under the plan's schedule.  b0p/b1p are the B maps boxed for a pair CTA (128 N
// rows for K-major weights); b0/b1 those of the one-CTA kernel.
template <int KIND>
inline mop_status tc_rows_gemm(const TcPlan* p, const char* name, const char* name2, const CUtensorMap& a0,
                               const CUtensorMap& a1, const CUtensorMap& b0, const CUtensorMap& b1,
                               const CUtensorMap& b0p, const CUtensorMap& b1p, TcArgs g, int32_t* tiles,
                               cudaStream_t st, int* launches) {
    mop_status r;
    if (p->pairs >= 1) {
        if ((r = tc2_launch<KIND>(p, name2, a0, a1, b0p, b1p, g, st)) != MOP_OK) return r;
        ++*launches;
    }
    if (p->pairs != 1) {
        if (p->pairs == 2) {
            int32_t* tiles2 = tiles + tc_tile_table_bytes(p->s.T * p->s.k, p->s.E) / 4;
            g.n_mtiles = tiles2;
            g.mtiles = reinterpret_cast<const int4*>(tiles2 + 64);
        }
        if ((r = tc_launch<KIND>(p, name, a0, a1, b0, b1, a0, a0, g, st)) != MOP_OK) return r;
        ++*launches;
    }
    return MOP_OK;
}

// The table of token tiles that an earlier kernel of a call may write for the GEMMs (tiles_ready); null: none that they would read,
// or tiles of another kind are needed too.
inline int32_t* tn_shared_table(const TcPlan* p, int32_t* tiles) { return p->fwd_tn == 15 ? tn_table(p, tiles) : nullptr; }

inline mop_status tc_ffn_fwd_impl(TcPlan* p, const TcFwdArgs& a, int32_t* tiles, int32_t* status, cudaStream_t st,
                                  int* launches, bool with_down);

inline mop_status tc_ffn_fwd(TcPlan* p, const TcFwdArgs& a, int32_t* tiles, int32_t* status, cudaStream_t st,
                             int* launches) {
    return tc_ffn_fwd_impl(p, a, tiles, status, st, launches, true);
}
// Up-projection + SwiGLU alone (the backward's recomputation of G, U, H).
inline mop_status tc_up_only(TcPlan* p, const TcFwdArgs& a, int32_t* tiles, int32_t* status, cudaStream_t st,
                             int* launches) {
    return tc_ffn_fwd_impl(p, a, tiles, status, st, launches, false);
}

inline mop_status tc_ffn_fwd_impl(TcPlan* p, const TcFwdArgs& a, int32_t* tiles, int32_t* status, cudaStream_t st,
                                  int* launches, bool with_down) {
    const mop_moe_shape& s = p->s;
    const uint64_t M = tc_rows(p);
    mop_status r;
    // Tokens-on-N kernels: fwd_tn bit 0 = up-projection, bit 1 = down-projection (set in mop_create)
    const bool gather = a.x_gather != nullptr;
    const bool tn_f1 = gather || (p->fwd_tn & 1), tn_f2 = p->fwd_tn & 2;
    if ((tn_f1 || tn_f2) && !a.tiles_ready) {
        if ((r = tn_build_tiles(p, a.offsets, tiles, !(tn_f1 && tn_f2) && p->pairs == 0, st)) != MOP_OK) return r;
        ++*launches;
    }
    if (!(tn_f1 && tn_f2) && !((tn_f1 || tn_f2) && p->pairs == 0)) {
        if ((r = tc_build_row_tiles(p, a.offsets, tiles, st)) != MOP_OK) return r;
        ++*launches;
    }
    // N-major weights as chunked maps: one-CTA tiles take 2 chunks per tensor (gate | up) or 4 (down);
    // a pair CTA takes 2 chunks
    CUtensorMap mXp, mWg, mWu, mH, mWd, mWdp;
    if (!tn_f1 && (!tc_map_2d(p, &mXp, a.Xp, M, s.d, 128) || !tc_map_chunked_3d(p, &mWg, a.W_gate, s.E, s.d, s.f, 2) ||
                   !tc_map_chunked_3d(p, &mWu, a.W_up, s.E, s.d, s.f, 2)))
        return MOP_ERR_CUDA;
    if (with_down && !tn_f2 && (!tc_map_2d(p, &mH, a.H, M, s.f, 128) || !tc_map_chunked_3d(p, &mWd, a.W_down, s.E, s.f, s.d, 4) ||
                                !tc_map_chunked_3d(p, &mWdp, a.W_down, s.E, s.f, s.d, 2)))
        return MOP_ERR_CUDA;
    if (gather) {
        if ((r = tn_up_swiglu_gather(p, a.x_gather, a, tiles, status, st)) != MOP_OK) return r;
        ++*launches;
    } else if (tn_f1) {
        if ((r = tn_up_swiglu(p, a, tiles, status, with_down && tn_f2, st)) != MOP_OK) return r;
        ++*launches;
    } else {   // F1: [G|U] = Xp [W_gate | W_up], SwiGLU epilogue
        TcArgs g = tc_base_args(p, a.offsets, tiles, status);
        g.tiles_n = ceil_div(s.f, 128); g.kblocks = ceil_div(s.d, TC_BK); g.N = s.f;
        g.ep.out0 = a.H; g.ep.out1 = a.G_save; g.ep.out2 = a.U_save; g.ep.ldo = s.f; g.ep.M_total = (int)M;
        if ((r = tc_rows_gemm<TC_F1>(p, "gemm_up_swiglu", "gemm_up_swiglu_2cta", mXp, mXp, mWg, mWu, mWg, mWu, g, tiles, st, launches)) != MOP_OK)
            return r;
    }
    if (!with_down) return MOP_OK;
    if (tn_f2) {
        if ((r = tn_down_gate(p, a, tiles, status, st)) != MOP_OK) return r;
        ++*launches;
    } else {   // F2: Yp = gate * (H W_down)
        TcArgs g = tc_base_args(p, a.offsets, tiles, status);
        g.tiles_n = ceil_div(s.d, 256); g.kblocks = ceil_div(s.f, TC_BK); g.N = s.d;
        g.ep.out0 = a.Yp; g.ep.gate = a.gate; g.ep.row_src = a.row_src; g.ep.ldo = s.d; g.ep.M_total = (int)M;
        if ((r = tc_rows_gemm<TC_F2>(p, "gemm_down_gate", "gemm_down_gate_2cta", mH, mH, mWd, mWd, mWdp, mWdp, g, tiles, st, launches)) != MOP_OK)
            return r;
    }
    return MOP_OK;
}

// Weight gradients on CTA pairs from 448 rows per expert on (average).  dW_down + (dW_gate, dW_up), us, single CTAs and pairs, both
// with the operands brought to L2 ahead: d = 2048, f = 1408, 64 experts of 256 rows 160 + 328 and 200 + 355, 384 rows 217 + 392 and
// 230 + 402, 448 rows 241 + 427 and 242 + 424, 512 rows 261 + 469 and 257 + 451, 1024 rows 408 + 770 and 400 + 725; d = 7168,
// f = 2048, 16 experts of 256 rows 205 + 396 and 286 + 560, 384 rows 254 + 494 and 256 + 486, 448 rows 286 + 555 and 276 + 522,
// 512 rows 312 + 608 and 294 + 562, 2048 rows 886 + 1695 and 802 + 1518.
inline bool tw_wanted(const TcPlan* p) { return p->fwd_tn == 15 && (uint64_t)p->s.T * p->s.k >= 448ull * p->s.E; }

inline mop_status tc_ffn_bwd(TcPlan* p, const TcBwdArgs& a, int32_t* tiles, int32_t* status, cudaStream_t st,
                             int* launches, int* ntile_part) {
    const mop_moe_shape& s = p->s;
    const uint64_t M = tc_rows(p);
    *ntile_part = ceil_div(s.f, 256);
    if (M == 0) {
        // no rows at all: gradients are zero unless accumulating
        if (!a.accumulate && !a.keep_empty) {
            const size_t n = (size_t)s.E * s.d * s.f * 4;
            if (cudaMemsetAsync(a.dW_gate, 0, n, st) != cudaSuccess || cudaMemsetAsync(a.dW_up, 0, n, st) != cudaSuccess ||
                cudaMemsetAsync(a.dW_down, 0, n, st) != cudaSuccess)
                return MOP_ERR_CUDA;
        }
        return MOP_OK;
    }
    mop_status r;
    if ((p->fwd_tn & 12) != 12) {   // row tiles of the tokens-on-M data gradients (the weight gradients need none)
        if ((r = tc_build_row_tiles(p, a.offsets, tiles, st)) != MOP_OK) return r;
        ++*launches;
    }
    const bool wpair = tw_wanted(p);
    const int bch = wpair ? 2 : 4;     // 64-wide chunks of B per copy: half of a tile per CTA of a pair
    CUtensorMap mgH, mdYpB, mXpA, mdGB, mdUB, moWd, moWg, moWu;   // weight gradients
    if (!tc_map_out_f32(p, &moWd, a.dW_down, s.E, s.f, s.d) || !tc_map_out_f32(p, &moWg, a.dW_gate, s.E, s.d, s.f) ||
        !tc_map_out_f32(p, &moWu, a.dW_up, s.E, s.d, s.f) || !tc_map_mn(p, &mgH, a.gH, M, s.f, 2) ||
        !tc_map_mn(p, &mdYpB, a.dYp, M, s.d, bch) || !tc_map_mn(p, &mXpA, a.Xp, M, s.d, 2) ||
        !tc_map_mn(p, &mdGB, a.dG, M, s.f, bch) || !tc_map_mn(p, &mdUB, a.dU, M, s.f, bch))
        return MOP_ERR_CUDA;
    // tokens-on-M data gradients: K-major weight maps boxed for one CTA (256 N rows) and for a pair CTA (128)
    CUtensorMap mdYpA, mWdK, mWdKp, mdG, mdU, mWgK, mWuK, mWgKp, mWuKp;
    if (!(p->fwd_tn & 8) && (!tc_map_2d(p, &mdYpA, a.dYp, M, s.d, 128) || !tc_map_3d(p, &mWdK, a.W_down, s.E, s.f, s.d, 256) ||
                             !tc_map_3d(p, &mWdKp, a.W_down, s.E, s.f, s.d, 128)))
        return MOP_ERR_CUDA;
    if (!(p->fwd_tn & 4) && (!tc_map_2d(p, &mdG, a.dG, M, s.f, 128) || !tc_map_2d(p, &mdU, a.dU, M, s.f, 128) ||
                             !tc_map_3d(p, &mWgK, a.W_gate, s.E, s.d, s.f, 256) || !tc_map_3d(p, &mWuK, a.W_up, s.E, s.d, s.f, 256) ||
                             !tc_map_3d(p, &mWgKp, a.W_gate, s.E, s.d, s.f, 128) || !tc_map_3d(p, &mWuKp, a.W_up, s.E, s.d, s.f, 128)))
        return MOP_ERR_CUDA;
    if ((p->fwd_tn & 12) && !a.tiles_ready) {
        if ((r = tn_build_tiles(p, a.offsets, tiles, false, st)) != MOP_OK) return r;
        ++*launches;
    }
    if (p->fwd_tn & 8) {   // B2 on the tokens-on-N kernel: one dgate partial per 32 columns of f
        *ntile_part = ceil_div(s.f, 32);
        if ((r = tn_dgrad_down(p, a, tiles, status, st)) != MOP_OK) return r;
        ++*launches;
    } else {   // B2: dHu = dYp W_down^T, SwiGLU backward epilogue
        TcArgs g = tc_base_args(p, a.offsets, tiles, status);
        g.tiles_n = ceil_div(s.f, 256); g.kblocks = ceil_div(s.d, TC_BK); g.N = s.f;
        g.ep.out0 = a.dG; g.ep.out1 = a.dU; g.ep.out2 = a.gH; g.ep.in0 = a.G_save; g.ep.in1 = a.U_save; g.ep.in2 = a.H;
        g.ep.gate = a.gate; g.ep.row_src = a.row_src; g.ep.part = a.part; g.ep.ldo = s.f; g.ep.M_total = (int)M;
        if ((r = tc_rows_gemm<TC_B2>(p, "gemm_dgrad_down_dswiglu", "gemm_dgrad_down_dswiglu_2cta", mdYpA, mdYpA, mWdK, mWdK, mWdKp,
                                     mWdKp, g, tiles, st, launches)) != MOP_OK)
            return r;
    }
    if (p->fwd_tn & 4) {   // B4 on the tokens-on-N kernel
        if ((r = tn_dgrad_gate_up(p, a, tiles, status, st)) != MOP_OK) return r;
        ++*launches;
    } else {   // B4: dXp = dG W_gate^T + dU W_up^T
        TcArgs g = tc_base_args(p, a.offsets, tiles, status);
        g.tiles_n = ceil_div(s.d, 256); g.kblocks = ceil_div(s.f, TC_BK); g.N = s.d;
        g.ep.out0 = a.dXp; g.ep.ldo = s.d; g.ep.M_total = (int)M;
        if ((r = tc_rows_gemm<TC_B4>(p, "gemm_dgrad_gate_up", "gemm_dgrad_gate_up_2cta", mdG, mdU, mWgK, mWuK, mWgKp, mWuKp, g, tiles, st,
                                     launches)) != MOP_OK)
            return r;
    }
    // Operands an expert ahead to L2 from 224 rows per expert on (average): with fewer the gradient stores alone set the pace
    // (d = 7168, 171 rows: 1094 + 2155 us without, 1137 + 2240 with; 256 rows in chunks of 16 experts: 1025 + 1907 and 1022 + 1834;
    // d = 2048, f = 1408, 384 rows: 225 + 429 and 220 + 395).
    const bool prefetch = (uint64_t)s.T * s.k >= 224ull * s.E;
    {   // WD: dW_down[e] = (gate H)_e^T dYp_e
        TcArgs g = tc_base_args(p, a.offsets, tiles, status);
        g.tiles_n = ceil_div(s.d, 256); g.tiles_m_fixed = ceil_div(s.f, wpair ? 256 : TC_BM); g.Mfix = s.f; g.N = s.d;
        g.a_split = s.f % 64 != 0; g.b_split = s.d % 64 != 0;
        g.ep.outf = a.dW_down; g.ep.accumulate = a.accumulate; g.keep_empty = a.keep_empty;
        g.gemm_follows = true;
        if (prefetch) { g.pf[0] = a.gH; g.pf_bytes[0] = s.f * 2; g.pf[1] = a.dYp; g.pf_bytes[1] = s.d * 2; }
        r = wpair ? tw_launch<TC_WD>(p, "gemm_wgrad_down", mgH, mdYpB, mdYpB, moWd, moWd, g, st)
                  : tc_launch<TC_WD>(p, "gemm_wgrad_down", mgH, mgH, mdYpB, mdYpB, moWd, moWd, g, st);
        if (r != MOP_OK) return r;
        ++*launches;
    }
    {   // WGU: dW_gate[e] = Xp_e^T dG_e and dW_up[e] = Xp_e^T dU_e: per m-block the n-tiles of dW_gate, then those of dW_up
        TcArgs g = tc_base_args(p, a.offsets, tiles, status);
        g.tiles_n = 2 * ceil_div(s.f, 256); g.tiles_m_fixed = ceil_div(s.d, wpair ? 256 : TC_BM); g.Mfix = s.d; g.N = s.f;
        g.a_split = s.d % 64 != 0; g.b_split = s.f % 64 != 0;
        g.ep.outf = a.dW_gate; g.outf1 = a.dW_up; g.ep.accumulate = a.accumulate; g.keep_empty = a.keep_empty;
        if (prefetch) {
            g.pf[0] = a.Xp; g.pf[1] = a.dG; g.pf[2] = a.dU;
            g.pf_bytes[0] = s.d * 2; g.pf_bytes[1] = g.pf_bytes[2] = s.f * 2;
        }
        r = wpair ? tw_launch<TC_WGU>(p, "gemm_wgrad_gate_up", mXpA, mdGB, mdUB, moWg, moWu, g, st)
                  : tc_launch<TC_WGU>(p, "gemm_wgrad_gate_up", mXpA, mXpA, mdGB, mdUB, moWg, moWu, g, st);
        if (r != MOP_OK) return r;
        ++*launches;
    }
    return MOP_OK;
}

}  // namespace mop
