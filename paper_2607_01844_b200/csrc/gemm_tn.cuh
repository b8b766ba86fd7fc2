// "Tokens on N" two-CTA grouped GEMMs: the MMA computes the TRANSPOSED product
//     D^T [weight rows (M = 256 across the CTA pair) x tokens (N <= 256)] = W^T-tile * Xp^T
// so that the ragged dimension (an expert's token count) sits on the MMA's N, whose granularity is
// 16, instead of on M, whose granularity is 128: an expert with 171 rows costs one N = 176 tile
// instead of two 128-row tiles (the tensor core takes N / 2 cycles per K = 16: 88 for N = 176, 128 for
// N = 256, 56 at the least, whatever the majors of A and B).  The weights are the "A" operand (each CTA of
// the pair holds its own 128 weight rows), the tokens the "B" operand (each CTA loads half of the tile's
// token rows), tcgen05.mma.cta_group::2 multiplies, and each CTA's TMEM receives [its 128 weight rows x N].
//
//   TN_F1  G^T|U^T: a CTA's 128 weight rows are 64 gate columns followed by the 64 matching up
//          columns of W_gate / W_up, so G and U of one (f, token) land in the same CTA (TMEM lanes
//          l and l + 64); the epilogue exchanges halves through shared memory, applies SwiGLU and
//          writes H (+ G, U stash) back in token-major layout.
//   TN_F2  O^T = W_down^T-tile * H^T, gate applied per token column, Yp written token-major.
//   TN_F1G as TN_F1, but the token operand is gathered straight from the unpermuted x [T, d]: every
//          lane of the producer warp owns four token rows of the tile and fetches them per K block
//          with one TMA gather4 copy, so the expert-contiguous copy Xp never exists (the
//          single-GPU form of keeping only a fraction of the routed inputs live, Section 3.3).
//          The TMA unit retires these 4-row copies far more slowly than one box (about
//          60 ns each on B200), so this form trades time for memory and is opt-in.
//   TN_B4  dXp^T = W_gate[e] dG^T + W_up[e] dU^T: the weights are read K-major ([E, d, f] as it
//          lies in memory, rows of d on M), two K phases into one accumulator, dXp token-major.
//   TN_B2  dHu^T = W_down[e] dYp^T (weights K-major, rows of f on M); the epilogue runs the SwiGLU
//          backward in the accumulator's layout: dG, dU, gate*H out, and one dgate partial per 32 columns of f.
//   TN_B2S the same where K is short: the epilogue's six tensors travel by TMA, with two pipeline stages less.
//
// Epilogues: the accumulator is read with tcgen05.ld.16x256b, whose layout is that of an mma fragment (a thread holds two
// neighbouring tokens of a feature), packed to bf16 pairs and turned token-major by stmatrix.trans: a block of 32 features x 32
// tokens costs 4 stmatrix, 4 16-byte shared loads and 4 16-byte global stores per lane where element-wise transposition took
// 32 two-byte stores and as many conversions.  Eight warps: four per accumulator, so that both drain at the same time.
//
// Barrier protocol, bounded waits and teardown as in the pair kernel (gemm_tc2.cuh).
#pragma once
#include "gemm_tc2.cuh"
#include "tiles.cuh"

namespace mop {

enum : int { TN_F1 = 0, TN_F2 = 1, TN_F1G = 2, TN_B4 = 3, TN_B2 = 4, TN_B2S = 5 };
__host__ __device__ constexpr bool tn_is_b2(int kind) { return kind == TN_B2 || kind == TN_B2S; }

constexpr int TN_STAGES = 6;
constexpr int TN_BK = 64;                            // K per stage
constexpr int TN_SUB_BYTES = 128 * TN_BK * 2;        // 16 KiB: this CTA's 128 weight rows, or up to 128 token rows
constexpr int TN_CHUNK_BYTES = 64 * TN_BK * 2;       // one 64-wide chunk of an M-major operand
constexpr int TN_STAGE_BYTES = 2 * TN_SUB_BYTES;
constexpr int TN_EPI_WARPS = 8;
constexpr int TN_EPI_BYTES = 4096;                   // per epilogue warp
constexpr int TN_SMEM_BYTES = TN_STAGES * TN_STAGE_BYTES + 1024 /*align*/ + TC_BAR_BYTES + TN_EPI_WARPS * TN_EPI_BYTES;
// The SwiGLU backward has two forms of its epilogue.  TN_B2 stages by warps like the others.  TN_B2S, where K is short and the epilogue
// the longer part, has three buffers per pair of warps of the stash's three tensors (16 tokens x 64 features) beside the gates of a
// tile, and two stages less.
constexpr int TN_STASH_BYTES = 16 * 128;             // of one tensor
constexpr int TN_STASH_BUFS = 3;
constexpr int TN_STASH_PAIR_BYTES = TN_STASH_BUFS * 3 * TN_STASH_BYTES;
__host__ __device__ constexpr int tn_stages(int kind) { return kind == TN_B2S ? 4 : TN_STAGES; }
static_assert(tn_stages(TN_B2S) * TN_STAGE_BYTES + 1024 + TC_BAR_BYTES + 4 * TN_STASH_PAIR_BYTES + TN_EPI_WARPS * 1024 <= TN_SMEM_BYTES,
              "shared memory");
constexpr int TN_THREADS = 64 + 32 * TN_EPI_WARPS;
constexpr int TN_RING = 16;                          // work items announced to the roles of a cluster
constexpr int TN_SIGNALS = 4;                        // requests for further items
constexpr int TN_BOXES = 8;                          // token boxes of 16, 32, .. 128 rows

struct TnMaps {
    CUtensorMap a0, a1;                // weights (F1: gate, up; B4: gate, up)
    CUtensorMap b[TN_BOXES];           // token rows, box of 16 (i + 1) rows
    CUtensorMap b1[TN_BOXES];          // B4: the second phase's token rows; B2S: [0..2] the stash G, U, H, [3..5] dG, dU, gH (16 rows)
};

// A tile's columns of the MMA, and the box (index into TnMaps) that holds one CTA's half of them.
__host__ __device__ constexpr int tn_nmma(int rows) { return (rows + 15) & ~15; }
__host__ __device__ constexpr int tn_box(int rows) { return ((tn_nmma(rows) >> 1) + 15) / 16 - 1; }

struct TnArgs {
    const int4* ttiles;       // {expert, first row, rows (1..256), position | number of tiles << 16} per token tile
    const int32_t* n_ttiles;  // device scalar
    int tiles_m;              // weight-row tiles per token tile (each 256 rows; F1: 128 columns of f)
    int kblocks;              // K / 64 rounded up
    int Mw;                   // weight rows in total (F1: f; F2: d)
    int a_split;              // F2: the two 64-wide weight chunks as one copy each (columns not a multiple of 64)
    const int32_t* row_src;   // F1G: assignment index t*k + j of every expert-contiguous row
    int topk;                 // F1G: k (token of a row = row_src / k)
    int32_t* next;            // work items handed out so far (zero when the kernel starts)
    int32_t* status;
    EpiArgs ep;
    bool gemm_follows;        // the next launch on the stream is a GEMM of this layer
};

// The tile tables of the token-row GEMMs in one launch: block 0 the token tiles, block 1 the 128-row tiles of the
// tokens-on-M kernels (where a forward or backward uses both).
__global__ void __launch_bounds__(1024) tn_build_ttiles_kernel(const int32_t* __restrict__ offsets, int E, int32_t* __restrict__ ttiles,
                                                               int32_t* __restrict__ mtiles) {
    pdl_begin();
    __shared__ int32_t scan[1025];
    if (blockIdx.x == 0) write_token_tiles<1024>(offsets, E, ttiles, scan);
    else tc_build_mtiles_body(offsets, E, reinterpret_cast<int4*>(mtiles + 64), mtiles, scan);
}

// Four rows of a [rows, cols] bf16 tensor (map box {64, 1}) -> 4 x 128 bytes at dst, swizzled like a tile box.
__device__ __forceinline__ void tma2_gather4(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int r0, int r1,
                                             int r2, int r3) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cta.global.tile::gather4.mbarrier::complete_tx::bytes.cta_group::2 [%0], "
        "[%1, {%3, %4, %5, %6, %7}], [%2];" ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(r0), "r"(r1), "r"(r2), "r"(r3)
        : "memory");
}

__device__ __forceinline__ void bar_pair_sync(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }

// ------------------------------------------------------------------------------------------ fragments
// 16 TMEM lanes x 8 R fp32 columns as an mma fragment: v[4 j + 0, 1] = lane t / 4, columns 8 j + 2 (t % 4), + 1; v[4 j + 2, 3] =
// lane t / 4 + 8, the same columns (t = the thread's lane).  The 16 lanes start at the lane field of taddr.  No wait.
__device__ __forceinline__ void tmem_frag4(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_frag2(uint32_t taddr, float (&v)[8]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
template <int N>
__device__ __forceinline__ void tmem_frag_wait(float (&a)[N], float (&b)[N]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < N; ++i) asm volatile("" : "+f"(a[i]), "+f"(b[i]));
}
__device__ __forceinline__ void stmatrix4_trans(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(r0), "r"(r1),
                 "r"(r2), "r"(r3)
                 : "memory");
}
__device__ __forceinline__ void ldmatrix4_trans(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts128(uint32_t addr, uint4 v) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ float2 lds64f(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
    return v;
}

// 16 bytes into the shared memory of CTA `rank` of the cluster (at this CTA's address `addr`), then one arrival on its barrier
__device__ __forceinline__ void publish16(uint32_t addr, uint32_t bar, uint32_t rank, int4 v) {
    asm volatile(
        "{\n.reg .b32 a, b;\nmapa.shared::cluster.u32 a, %0, %2;\nmapa.shared::cluster.u32 b, %1, %2;\n"
        "st.shared::cluster.v4.b32 [a], {%3, %4, %5, %6};\n"
        "mbarrier.arrive.release.cluster.shared::cluster.b64 _, [b];\n}" ::"r"(addr),
        "r"(bar), "r"(rank), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
        : "memory");
}

// Staging of a block token-major: 64-byte rows of 32 features, the four 16-byte pieces of a row XOR-swizzled by bits 1..2 of
// the token, so that the eight rows of a matrix and the 32 pieces of a row-wise access each touch every bank once.
// frag_off: this lane's row address for stmatrix / ldmatrix .x4 (matrix m = lane / 8 holds features 8 m .. 8 m + 7 of tokens
// 8 j + lane % 8; + 512 j).  piece_off: token lane / 4, features 8 (lane % 4) .. + 7 (+ 512 i for token 8 i + lane / 4).
__device__ __forceinline__ uint32_t frag_off(int lane) {
    return (uint32_t)((lane & 7) * 64 + ((((lane >> 3) ^ (lane >> 1)) & 3) << 4));
}
__device__ __forceinline__ uint32_t piece_off(int lane) {
    return (uint32_t)((lane >> 2) * 64 + (((lane ^ (lane >> 3)) & 3) << 4));
}

// 8 J tokens x 32 features staged at `st` -> global rows (16-byte pieces); features at and past Mw are not stored.
template <int J>
__device__ __forceinline__ void tn_write_rows(bf16* __restrict__ dst, int ldo, uint32_t st, int row0, int rows_left,
                                              int col0, int Mw, int lane) {
    const int col = col0 + (lane & 3) * 8;
#pragma unroll
    for (int i = 0; i < J; ++i) {
        const int tok = 8 * i + (lane >> 2);
        const uint4 v = lds128(st + 512 * i + piece_off(lane));
        if (tok < rows_left && col < Mw) *reinterpret_cast<uint4*>(dst + (size_t)(row0 + tok) * ldo + col) = v;
    }
}

// SwiGLU backward of 16 tokens x 32 features in the accumulator's fragments: frag holds G, U, H and becomes dG, dU, gate * H; dot are
// this lane's shares of <dHu, H> of its tokens.  gates: shared memory, of the step's first token on.
__device__ __forceinline__ void tn_swiglu_backward(uint32_t (&frag)[3][2][4], const float (&v0)[8], const float (&v1)[8], uint32_t gates,
                                                   int tpair, float (&dot)[2][2]) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        dot[j][0] = dot[j][1] = 0.0f;
        const float2 gt = lds64f(gates + 4u * (8 * j + tpair));
#pragma unroll
        for (int m = 0; m < 4; ++m) {          // features 8 m + lane / 4
            float dG[2], dU[2], gH[2];
#pragma unroll
            for (int p = 0; p < 2; ++p) {      // tokens tpair, tpair + 1
                const float G = p ? bf16_hi(frag[0][j][m]) : bf16_lo(frag[0][j][m]);
                const float U = p ? bf16_hi(frag[1][j][m]) : bf16_lo(frag[1][j][m]);
                const float H = p ? bf16_hi(frag[2][j][m]) : bf16_lo(frag[2][j][m]);
                const float gate = p ? gt.y : gt.x;
                const float dhu = m < 2 ? v0[4 * j + 2 * m + p] : v1[4 * j + 2 * (m - 2) + p];
                dot[j][p] = fmaf(dhu, H, dot[j][p]);
                const float dh = gate * dhu;
                const float sg = sigmoidf_fast(G);
                dG[p] = dh * U * sg * (1.0f + G * (1.0f - sg));
                dU[p] = dh * (G * sg);
                gH[p] = gate * H;
            }
            frag[0][j][m] = pack_bf16x2(dG[0], dG[1]);
            frag[1][j][m] = pack_bf16x2(dU[0], dU[1]);
            frag[2][j][m] = pack_bf16x2(gH[0], gH[1]);
        }
    }
}
// The 32 features' dot products: the 8 lanes with the same lane % 4 hold the shares of the same tokens.
__device__ __forceinline__ void tn_write_dots(const EpiArgs& ep, float (&dot)[2][2], int row0, int rows_left, int tpair, int fcol, int Mw,
                                              int lane) {
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int p = 0; p < 2; ++p) {
#pragma unroll
            for (int off = 4; off < 32; off <<= 1) dot[j][p] += __shfl_xor_sync(0xffffffffu, dot[j][p], off);
            const int tok = 8 * j + tpair + p;
            if (lane < 4 && tok < rows_left && fcol < Mw) ep.part[(size_t)(fcol >> 5) * ep.M_total + row0 + tok] = dot[j][p];
        }
}

// An epilogue warp's walk over the cluster's items: items n with n % 2 == group are drained, the others passed over.
// next(n): item n is there; false: none is left, or the wait for it gave up.  wait(n): its accumulator is ready, or the wait gave up.
// PAIRED: drain(n) meets a partner warp at barriers.  Two warps may see the CTA give up at different items, or one of them while
// the other sees the end, so neither leaves by itself: vote(ok), a barrier of the two that ANDs their outcomes, is taken once per
// drained item and once on leaving, and a warp that finds its partner leaving leaves too.
#pragma nv_exec_check_disable
template <bool PAIRED, class Next, class Wait, class Vote, class Drain>
__host__ __device__ __forceinline__ void tn_walk_items(int group, Next next, Wait wait, Vote vote, Drain drain) {
    for (int n = 0;; ++n) {
        if (!next(n)) {
            if constexpr (PAIRED) vote(false);
            return;
        }
        if ((n & 1) != group) continue;
        bool ready = wait(n);
        if constexpr (PAIRED) ready = vote(ready);
        if (!ready) return;
        drain(n);
    }
}

// ONCE: weights pass through L2 as evict-first (tn_stream_weights); a kernel of its own, since copies with a policy, or a choice
// at each, take 1 to 2 % more where the copies set the pace.
template <int KIND, bool ONCE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TN_THREADS, 1)
tn_gemm_kernel(const __grid_constant__ TnMaps maps, const TnArgs args) {
    constexpr int S = tn_stages(KIND), STAGE_BYTES = TN_STAGE_BYTES;
    constexpr int BUFS = TN_STASH_BUFS;
    extern __shared__ uint8_t tc_smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S * STAGE_BYTES);
    constexpr int STASH_BARS = KIND == TN_B2S ? 4 * BUFS : 0;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 4 + TN_RING + TN_SIGNALS + STASH_BARS);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = warp_index(), lane = threadIdx.x % 32;
    const uint32_t rank = cluster_ctarank();
    const bool leader = rank == 0;
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t bar_base = smem_u32(bars);
    const uint32_t epi_base = bar_base + TC_BAR_BYTES;
    auto full_bar = [&](int s) { return bar_base + 8u * s; };
    auto empty_bar = [&](int s) { return bar_base + 8u * (S + s); };
    auto tfull_bar = [&](int b) { return bar_base + 8u * (2 * S + b); };
    auto tempty_bar = [&](int b) { return bar_base + 8u * (2 * S + 2 + b); };
    // announced item n = 1, 2, .. is entry n - 1 of the ring (item 0 is never announced)
    auto item_bar = [&](int n) { return bar_base + 8u * (2 * S + 4 + ((n - 1) & (TN_RING - 1))); };
    auto item_slot = [&](int n) { return bar_base + 512u + 16u * ((n - 1) & (TN_RING - 1)); };
    auto signal_bar = [&](int n) { return bar_base + 8u * (2 * S + 4 + TN_RING + (n & (TN_SIGNALS - 1))); };
    auto stash_bar = [&](int pair, int b) { return bar_base + 8u * (2 * S + 4 + TN_RING + TN_SIGNALS + pair * BUFS + b); };
    (void)stash_bar;
    static_assert(8 * (2 * S + 4 + TN_RING + TN_SIGNALS + STASH_BARS) + 8 <= 512 && 512 + 16 * TN_RING <= TC_BAR_BYTES, "barrier block");

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(tfull_bar(b), 1); mbar_init(tempty_bar(b), 8); }
        for (int n = 0; n < TN_RING; ++n) mbar_init(item_bar(n), 1);
        for (int n = 0; n < TN_SIGNALS; ++n) mbar_init(signal_bar(n), 1);
        for (int n = 0; n < STASH_BARS; ++n) mbar_init(stash_bar(n / BUFS, n % BUFS), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tma_prefetch_desc(&maps.a0);
        if (KIND != TN_F2 && !tn_is_b2(KIND)) tma_prefetch_desc(&maps.a1);
        if (KIND == TN_B2S)
            for (int i = 0; i < 6; ++i) tma_prefetch_desc(&maps.b1[i]);
    }
    if (warp == 1) tmem2_alloc(smem_u32(tmem_slot), 512);
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    pdl_begin_gemm(args.gemm_follows, PdlNote{});

    const int total_tiles = (*args.n_ttiles) * args.tiles_m;
    const int nkb = (KIND == TN_B4 ? 2 : 1) * args.kblocks;   // K blocks per tile (B4: two phases)
    const int cluster_id = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;
    // Work items are handed out in order as the clusters go along (one atomic addition per item): the items of one expert that
    // share a weight tile start together and read it from L2 together, whatever the sizes of the items before them, and the
    // last items spread evenly.  With a fixed round-robin the clusters drifted apart by whole items and the weights were fetched
    // again: at d = 7168, f = 2048, 256 experts of 512 rows the up-projection took 7.3 ms under the power cap, 6.2 this way.
    // Item t -> token tile t / tiles_m (its expert, first row, rows) and weight-row tile t % tiles_m.
    // Item 0 of a cluster is its own number; the others are taken, decoded and written into the rings of both CTAs by the
    // second CTA's MMA warp, which has nothing else to do, when the second CTA's producer asks (`ahead` items early where K is
    // short: taking and announcing one takes about 2000 cycles).  No slot is written before it was read: the MMA is at most S
    // K blocks behind the producer and the epilogue two items behind the MMA; TN_RING is more than S + 2 + ahead + 1.
    struct Tile { int e, row0, rows, mt; };
    const bool handout = total_tiles > n_clusters;
    const int ahead = nkb >= 24 ? 0 : nkb >= 8 ? 1 : 3;
    const int ask_at = ahead ? 0 : nkb - 10;
    static_assert(TN_RING > S + 2 + 3 + 1 && TN_SIGNALS >= 3 + 1, "see above");
    // Within an expert the token tiles vary fastest.  e < 0: no item left.
    auto decode = [&](int t) {
        if (t >= total_tiles) return make_int4(-1, 0, 0, 0);
        const int q = t / args.tiles_m;
        int4 m = __ldg(args.ttiles + q);
        const int nt = m.w >> 16;
        int mt = t - q * args.tiles_m;
        if (nt > 1) {
            const int first = q - (m.w & 0xffff);                 // first token tile of this expert
            const int l = t - first * args.tiles_m;               // position among the expert's work items
            mt = l / nt;
            m = __ldg(args.ttiles + first + (l - mt * nt));
        }
        return make_int4(m.x, m.y, m.z, mt);
    };
    // The n-th item of this cluster; false: none left (or the CTA is giving up).
    auto next_item = [&](int n, Tile& ti) {
        int4 v;
        if (n == 0) v = decode(cluster_id);
        else {
            if (!handout) return false;
            if (!mbar_wait_cluster(item_bar(n), (uint32_t)((n - 1) / TN_RING) & 1u, abort_flag, args.status, STATUS_WAIT_FULL)) return false;
            const uint4 u = lds128(item_slot(n));
            v = make_int4((int)u.x, (int)u.y, (int)u.z, (int)u.w);
        }
        ti.e = v.x; ti.row0 = v.y; ti.rows = v.z; ti.mt = v.w;
        return ti.e >= 0;
    };

    if (warp == 0 && KIND == TN_F1G) {
        // ============================================ TMA producer with row gather (both CTAs, whole warp)
        int stage = 0; uint32_t phase = 0; bool alive = true;
        Tile ti;
        for (int n = 0; alive && __all_sync(0xffffffffu, next_item(n, ti)); ++n) {
            const int half = tn_nmma(ti.rows) >> 1;                    // token rows per CTA (multiple of 8)
            const int ngroups = half >> 2;                             // gather4 copies per K block (<= 32)
            const int brow0 = ti.row0 + (int)rank * half;
            const int last = ti.row0 + ti.rows - 1;                    // padding rows repeat the last valid one
            int tok[4] = {0, 0, 0, 0};
            if (lane < ngroups) {
#pragma unroll
                for (int j = 0; j < 4; ++j) tok[j] = __ldg(args.row_src + min(brow0 + 4 * lane + j, last)) / args.topk;
            }
            const uint32_t tx = 2u * (TN_SUB_BYTES + (uint32_t)half * 128u);
            for (int kb = 0; kb < args.kblocks; ++kb) {
                if (!mbar_wait_warp(empty_bar(stage), phase ^ 1u, abort_flag, args.status, STATUS_WAIT_EMPTY, lane)) {
                    alive = false; break;
                }
                const uint32_t fb = full_bar(stage) & T2_PEER_MASK;
                const uint32_t sA = smem_base + stage * STAGE_BYTES;
                const uint32_t sB = sA + TN_SUB_BYTES;
                const int k0 = kb * TN_BK;
                if (lane == 0) {
                    if (!leader && handout && kb == ask_at) mbar_arrive(signal_bar(n));
                    if (leader) mbar_expect_tx(full_bar(stage), tx);
                    const int f0 = ti.mt * 128 + 64 * (int)rank;
                    tma2_load_3d(sA, &maps.a0, fb, f0, k0, ti.e);
                    tma2_load_3d(sA + TN_CHUNK_BYTES, &maps.a1, fb, f0, k0, ti.e);
                }
                if (lane < ngroups) tma2_gather4(sB + lane * 512, &maps.b[0], fb, k0, tok[0], tok[1], tok[2], tok[3]);
                __syncwarp();
                if (++stage == S) { stage = 0; phase ^= 1u; }
            }
        }
    } else if (warp == 0) {
        // ===================================================================== TMA producer (both CTAs)
        const bool el = elect_one();
        const uint64_t once = ONCE ? l2_policy_evict_first() : 0;
        (void)once;
        auto load_w3 = [&](uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z) {
            if constexpr (ONCE) tma2_load_3d_hint(dst, map, bar, x, y, z, once);
            else tma2_load_3d(dst, map, bar, x, y, z);
        };
        int stage = 0; uint32_t phase = 0; bool alive = true;
        Tile ti;
        for (int n = 0; alive && __all_sync(0xffffffffu, next_item(n, ti)); ++n) {
            // this CTA's half of the token rows, in the smallest box that holds it (what a box fetches past the half belongs
            // to nobody: the MMA reads the half only)
            const int half = tn_nmma(ti.rows) >> 1, box = tn_box(ti.rows);
            const int brow0 = ti.row0 + (int)rank * half;
            const uint32_t tx = 2u * (TN_SUB_BYTES + (uint32_t)(box + 1) * 2048u);
            const CUtensorMap* mb = &maps.b[box];
            // first weight row of this CTA (F1: 64 gate columns, then the 64 matching up columns)
            const int m0 = KIND == TN_F1 ? ti.mt * 128 + 64 * (int)rank : ti.mt * 256 + 128 * (int)rank;
            for (int kb = 0; kb < nkb; ++kb) {
                if (!mbar_wait_all(empty_bar(stage), phase ^ 1u, abort_flag, args.status, STATUS_WAIT_EMPTY)) {
                    alive = false; break;
                }
                const uint32_t fb = full_bar(stage) & T2_PEER_MASK;
                const uint32_t sA = smem_base + stage * STAGE_BYTES;
                const uint32_t sB = sA + TN_SUB_BYTES;
                const int ph = (KIND == TN_B4 && kb >= args.kblocks) ? 1 : 0;   // B4: gate phase, then up phase
                const int k0 = (kb - ph * args.kblocks) * TN_BK;
                if (KIND == TN_B4 && kb == args.kblocks) mb = &maps.b1[box];
                if (el) {
                    if (!leader && handout && kb == ask_at) mbar_arrive(signal_bar(n));
                    if (leader) mbar_expect_tx(full_bar(stage), tx);
                    if constexpr (KIND == TN_B4 || tn_is_b2(KIND)) {
                        load_w3(sA, ph ? &maps.a1 : &maps.a0, fb, k0, m0, ti.e);   // K-major weights
                    } else if constexpr (KIND == TN_F1) {                               // N-major weights [E, d, f]
                        load_w3(sA, &maps.a0, fb, m0, k0, ti.e);
                        load_w3(sA + TN_CHUNK_BYTES, &maps.a1, fb, m0, k0, ti.e);
                    } else if (args.a_split) {
                        load_w3(sA, &maps.a0, fb, m0, k0, ti.e);
                        load_w3(sA + TN_CHUNK_BYTES, &maps.a0, fb, m0 + 64, k0, ti.e);
                    } else if constexpr (ONCE) {
                        tma2_load_4d_hint(sA, &maps.a0, fb, 0, k0, m0 >> 6, ti.e, once);   // two chunks in one copy
                    } else {
                        tma2_load_4d(sA, &maps.a0, fb, 0, k0, m0 >> 6, ti.e);
                    }
                    tma2_load_2d(sB, mb, fb, k0, brow0);
                }
                if (++stage == S) { stage = 0; phase ^= 1u; }
            }
        }
    } else if (warp == 1) {
        // ===================================================================== MMA issuer (leader CTA)
        if (leader) {
            const bool el = elect_one();
            constexpr bool A_KMAJOR = (KIND == TN_B4 || tn_is_b2(KIND));
            // descriptors without the start address: A is M-major (N-major weights) or K-major, B is K-major.
            // A M-major: the two 64-wide chunks are TN_CHUNK_BYTES apart, 2 KiB per K = 16; K-major: 32 bytes per K = 16
            const uint64_t desc_a = smem_desc(0, A_KMAJOR ? 0 : TN_CHUNK_BYTES, 1024);
            const uint64_t desc_b = smem_desc(0, 0, 1024);
            // M = 256 over the pair, N = the tile's tokens
            constexpr uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((A_KMAJOR ? 0u : 1u) << 15) | ((uint32_t)(256 >> 4) << 24);
            int stage = 0; uint32_t phase = 0; int it = 0; bool alive = true;
            Tile ti;
            for (int n = 0; alive && __all_sync(0xffffffffu, next_item(n, ti)); ++n) {
                const uint32_t idesc = idesc0 | ((uint32_t)(tn_nmma(ti.rows) >> 3) << 17);
                const int buf = it & 1;
                const uint32_t d_tmem = tmem_base + (uint32_t)buf * 256;
                if (!mbar_wait_all(tempty_bar(buf), ((uint32_t)(it >> 1) & 1u) ^ 1u, abort_flag, args.status, STATUS_WAIT_TMEM_EMPTY)) break;
                tc_fence_after();
                for (int kb = 0; kb < nkb; ++kb) {
                    if (!mbar_wait_all(full_bar(stage), phase, abort_flag, args.status, STATUS_WAIT_FULL)) { alive = false; break; }
                    tc_fence_after();
                    const uint32_t sA = smem_base + stage * STAGE_BYTES;
                    const uint64_t da = desc_a | (uint64_t)((sA & 0x3ffffu) >> 4);
                    const uint64_t db = desc_b | (uint64_t)(((sA + TN_SUB_BYTES) & 0x3ffffu) >> 4);
                    if (el) {
#pragma unroll
                        for (int k4 = 0; k4 < TN_BK / 16; ++k4)
                            umma2_bf16(d_tmem, da + k4 * (A_KMAJOR ? 2 : 2048 >> 4), db + k4 * 2, idesc, (kb | k4) != 0 ? 1u : 0u);
                        umma2_commit_both(empty_bar(stage));
                    }
                    if (++stage == S) { stage = 0; phase ^= 1u; }
                }
                if (!alive) break;
                if (el) umma2_commit_both(tfull_bar(buf));
                ++it;
            }
        } else if (handout && lane == 0) {
            // ================================================================= hands out work items (second CTA)
            for (int m = 1;; ++m) {
                const int r = m - 1 - ahead;             // announced when item r asks
                if (r >= 0 && !mbar_wait(signal_bar(r), (uint32_t)(r / TN_SIGNALS) & 1u, abort_flag, args.status, STATUS_WAIT_EMPTY)) break;
                const int4 v = decode(n_clusters + atomicAdd(args.next, 1));
                publish16(item_slot(m), item_bar(m), 0, v);
                publish16(item_slot(m), item_bar(m), 1, v);
                if (v.x < 0) break;
            }
        }
    } else {
        // ===================================================================== epilogue (8 warps, both CTAs)
        const int quarter = warp & 3;                 // TMEM lanes 32*quarter .. +31
        const int group = (warp - 2) >> 2;            // the accumulator these four warps drain
        const uint32_t wb = epi_base + (uint32_t)(warp - 2) * TN_EPI_BYTES;   // this warp's staging
        const uint32_t fo = frag_off(lane);
        const int tpair = 2 * (lane & 3);             // this thread's tokens within a run of 8: tpair, tpair + 1
        // F1: a gate warp and its up warp; B2S: two warps that share 128-byte lines of the stash
        constexpr bool PAIRED = KIND == TN_F1 || KIND == TN_F1G || KIND == TN_B2S;
        const int pair_bar = 1 + 2 * group + (KIND == TN_B2S ? quarter >> 1 : quarter & 1);
        const int buf = group;
        const uint32_t gbuf = KIND == TN_B2S ? epi_base + 4 * TN_STASH_PAIR_BYTES + (uint32_t)(warp - 2) * 1024 : wb + 3072;
        Tile ti = {0, 0, 0, 0};
        // B2S: the pair's buffers, its steps so far (16 tokens each; the buffers and their barriers' phases alternate) and the warp
        // that copies for both
        const int stash_pair = (warp - 2) >> 1;
        const uint32_t stash = epi_base + (uint32_t)stash_pair * TN_STASH_PAIR_BYTES;
        const bool el = elect_one();
        const bool copies = (quarter & 1) == 0 && el;
        int steps = 0;
        bool gone = false;
        (void)stash; (void)copies; (void)steps; (void)gone;
        auto fetch_stash = [&](int step, int row) {
            const int b = step % BUFS;
            const int f0 = ti.mt * 256 + 128 * (int)rank + 64 * (quarter >> 1);
            mbar_expect_tx(stash_bar(stash_pair, b), 3 * TN_STASH_BYTES);
#pragma unroll
            for (int a = 0; a < 3; ++a)
                tma_load_2d(stash + (b * 3 + a) * TN_STASH_BYTES, &maps.b1[a], stash_bar(stash_pair, b), f0, row);
        };
        // (the lanes give up together: a lane that left alone would be missed at the shuffles below)
        auto next = [&](int n) { return !gone && __all_sync(0xffffffffu, next_item(n, ti)) != 0; };
        auto wait = [&](int n) {
            if constexpr (KIND == TN_B2S) {       // the stash of the tile's first steps as well
                if (copies) {
                    tma_store_wait_read<0>();
#pragma unroll
                    for (int i = 0; i < BUFS; ++i)
                        if (16 * i < ti.rows) fetch_stash(steps + i, ti.row0 + 16 * i);
                }
            }
            // F2, B2: the gates of the tile's tokens (two dependent loads each) are fetched before the wait for the
            // accumulator, so that their latency is hidden behind the main loop
            if constexpr (KIND == TN_F2 || tn_is_b2(KIND)) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int tk = 32 * j + lane;
                    const float g = tk < ti.rows ? args.ep.gate[args.ep.row_src[ti.row0 + tk]] : 0.0f;
                    asm volatile("st.shared.f32 [%0], %1;" ::"r"(gbuf + 4u * tk), "f"(g) : "memory");
                }
                __syncwarp();
            }
            return mbar_wait_warp(tfull_bar(buf), (uint32_t)(n >> 1) & 1u, abort_flag, args.status, STATUS_WAIT_TMEM_FULL, lane);
        };
        auto vote = [&](bool ok) { return bar_vote_all(pair_bar, 64, ok); };
        tn_walk_items<PAIRED>(group, next, wait, vote, [&](int) {
            const int row0 = ti.row0, rows = ti.rows;
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)buf * 256;
            const int nmma = tn_nmma(rows);

            if constexpr (KIND == TN_F1 || KIND == TN_F1G) {
                // Lanes 0..63 of the CTA hold gate rows, lanes 64..127 the matching up rows: warp q (gate)
                // and warp q + 2 (up) own the same 32 f columns.  Per chunk of 32 tokens they swap halves
                // through shared memory (the gate warp hands over G of tokens 16..31, the up warp U of
                // tokens 0..15), so each evaluates SwiGLU for 16 tokens and writes 16 rows of H.
                const bool is_up = quarter >= 2;
                const int fcol = ti.mt * 128 + 64 * (int)rank + 32 * (quarter & 1);   // first f of this warp
                const uint32_t peer = epi_base + (uint32_t)(((warp - 2) & 4) + (((warp - 2) ^ 2) & 3)) * TN_EPI_BYTES;
                const uint32_t sb = wb + 2048;                                         // staged rows
                bf16* stash_out = is_up ? args.ep.out2 : args.ep.out1;
                const int t_own = is_up ? 16 : 0;
#pragma unroll 1
                for (int c = 0; c < nmma; c += 32) {
                    float v0[16], v1[16];
                    tmem_frag4(taddr + c, v0);
                    tmem_frag4(taddr + (16u << 16) + c, v1);
                    tmem_frag_wait(v0, v1);
                    const int rows_left = rows - c;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {      // the partner's half: 16 fp32 values, 16 bytes per lane and store
                        const int i = 4 * (q & 1);
                        float x[4];
#pragma unroll
                        for (int r = 0; r < 4; ++r)
                            x[r] = q < 2 ? (is_up ? v0[i + r] : v0[8 + i + r]) : (is_up ? v1[i + r] : v1[8 + i + r]);
                        sts128(wb + 512 * q + 16 * lane, make_uint4(__float_as_uint(x[0]), __float_as_uint(x[1]),
                                                                    __float_as_uint(x[2]), __float_as_uint(x[3])));
                    }
                    if (stash_out) {                   // own 32 tokens of G or U, in two halves of 1 KiB
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
#pragma unroll
                            for (int j = 2 * h; j < 2 * h + 2; ++j)
                                stmatrix4_trans(sb + 512 * (j & 1) + fo, pack_bf16x2(v0[4 * j], v0[4 * j + 1]),
                                                pack_bf16x2(v0[4 * j + 2], v0[4 * j + 3]), pack_bf16x2(v1[4 * j], v1[4 * j + 1]),
                                                pack_bf16x2(v1[4 * j + 2], v1[4 * j + 3]));
                            __syncwarp();
                            tn_write_rows<2>(stash_out, args.ep.ldo, sb, row0 + c + 16 * h, rows_left - 16 * h, fcol, args.Mw, lane);
                            __syncwarp();
                        }
                    }
                    bar_pair_sync(pair_bar);     // both halves are in shared memory
                    float h0[8], h1[8];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const uint4 o = lds128(peer + 512 * q + 16 * lane);
                        const float other[4] = {__uint_as_float(o.x), __uint_as_float(o.y), __uint_as_float(o.z), __uint_as_float(o.w)};
                        const int i = 4 * (q & 1);
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const float mine = q < 2 ? (is_up ? v0[8 + i + r] : v0[i + r]) : (is_up ? v1[8 + i + r] : v1[i + r]);
                            const float g = is_up ? other[r] : mine, u = is_up ? mine : other[r];
                            const float h = g * sigmoidf_fast(g) * u;
                            if (q < 2) h0[i + r] = h; else h1[i + r] = h;
                        }
                    }
#pragma unroll
                    for (int j = 0; j < 2; ++j)
                        stmatrix4_trans(sb + 512 * j + fo, pack_bf16x2(h0[4 * j], h0[4 * j + 1]), pack_bf16x2(h0[4 * j + 2], h0[4 * j + 3]),
                                        pack_bf16x2(h1[4 * j], h1[4 * j + 1]), pack_bf16x2(h1[4 * j + 2], h1[4 * j + 3]));
                    __syncwarp();
                    tn_write_rows<2>(args.ep.out0, args.ep.ldo, sb, row0 + c + t_own, rows_left - t_own, fcol, args.Mw, lane);
                    bar_pair_sync(pair_bar);     // the partner has read this warp's half
                }
            } else if constexpr (KIND == TN_B2) {
                // 16 tokens at a time: the stash (G, U, H) comes in as 16-byte pieces of token rows one step ahead, is staged and
                // read back as fragments (ldmatrix.trans) that match the accumulator's; the results leave the same way.
                const int fcol = ti.mt * 256 + 128 * (int)rank + 32 * quarter;      // first f column of this warp
                const int col = fcol + (lane & 3) * 8;
                const bf16* const src[3] = {args.ep.in0, args.ep.in1, args.ep.in2};
                bf16* const dst[3] = {args.ep.out0, args.ep.out1, args.ep.out2};
                uint4 pre[3][2];
                auto fetch = [&](int c) {
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const int tok = c + 8 * i + (lane >> 2);
                        const bool okk = tok < rows && col < args.Mw;
                        const size_t o = (size_t)(row0 + tok) * args.ep.ldo + col;
#pragma unroll
                        for (int a = 0; a < 3; ++a)
                            pre[a][i] = okk ? *reinterpret_cast<const uint4*>(src[a] + o) : make_uint4(0, 0, 0, 0);
                    }
                };
                fetch(0);
#pragma unroll 1
                for (int c = 0; c < nmma; c += 16) {
                    float v0[8], v1[8];
                    tmem_frag2(taddr + c, v0);
                    tmem_frag2(taddr + (16u << 16) + c, v1);
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int i = 0; i < 2; ++i) sts128(wb + 1024 * a + 512 * i + piece_off(lane), pre[a][i]);
                    __syncwarp();
                    if (c + 16 < nmma) fetch(c + 16);
                    uint32_t frag[3][2][4];
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int j = 0; j < 2; ++j) ldmatrix4_trans(wb + 1024 * a + 512 * j + fo, frag[a][j]);
                    tmem_frag_wait(v0, v1);
                    float dot[2][2];
                    tn_swiglu_backward(frag, v0, v1, gbuf + 4u * c, tpair, dot);
                    __syncwarp();                              // every lane has its fragments of the stash
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int j = 0; j < 2; ++j)
                            stmatrix4_trans(wb + 1024 * a + 512 * j + fo, frag[a][j][0], frag[a][j][1], frag[a][j][2], frag[a][j][3]);
                    __syncwarp();
#pragma unroll
                    for (int a = 0; a < 3; ++a)
                        tn_write_rows<2>(dst[a], args.ep.ldo, wb + 1024 * a, row0 + c, rows - c, fcol, args.Mw, lane);
                    tn_write_dots(args.ep, dot, row0 + c, rows - c, tpair, fcol, args.Mw, lane);
                    __syncwarp();
                }
            } else if constexpr (KIND == TN_B2S) {
                // The same with the stash and the results travelling as boxes of 64 features, whole 128-byte lines, between global and
                // shared memory, in the buffers' place; a warp works on its 32 of them.  Where K is short, 16-byte loads and stores of
                // half lines, one step ahead, are more than half of a tile's time.
                const int fcol = ti.mt * 256 + 128 * (int)rank + 32 * quarter;      // first f column of this warp
                const int sub = 4 * (quarter & 1);                                  // its first 16-byte piece of a line
                const uint32_t fo2 = (uint32_t)((lane & 7) * 128 + (((sub + (lane >> 3)) ^ (lane & 7)) << 4));
                bf16* const dst[3] = {args.ep.out0, args.ep.out1, args.ep.out2};
#pragma unroll 1
                for (int c = 0; c < nmma; c += 16, ++steps) {
                    const int b = steps % BUFS;
                    const uint32_t st = stash + b * 3 * TN_STASH_BYTES;
                    float v0[8], v1[8];
                    tmem_frag2(taddr + c, v0);
                    tmem_frag2(taddr + (16u << 16) + c, v1);
                    bool ok = mbar_wait_warp(stash_bar(stash_pair, b), (uint32_t)(steps / BUFS) & 1u, abort_flag, args.status, STATUS_WAIT_FULL, lane);
                    uint32_t frag[3][2][4];
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int j = 0; j < 2; ++j) ldmatrix4_trans(st + a * TN_STASH_BYTES + 1024 * j + fo2, frag[a][j]);
                    // the step before left its buffer to the store that reads it: once that is done, the step after this one
                    if (copies && c > 0 && c + 16 * (BUFS - 1) < nmma) {
                        tma_store_wait_read<0>();
                        fetch_stash(steps + BUFS - 1, row0 + c + 16 * (BUFS - 1));
                    }
                    tmem_frag_wait(v0, v1);
                    float dot[2][2];
                    tn_swiglu_backward(frag, v0, v1, gbuf + 4u * c, tpair, dot);
                    __syncwarp();                              // every lane has its fragments of the stash
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int j = 0; j < 2; ++j)
                            stmatrix4_trans(st + a * TN_STASH_BYTES + 1024 * j + fo2, frag[a][j][0], frag[a][j][1], frag[a][j][2], frag[a][j][3]);
                    const bool whole = c + 16 <= rows;
                    // (in either case: TMA reads these bytes now, or writes the next tile's stash over them)
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    if (!whole) {                              // the rows after the tile's are another expert's: row by row
                        __syncwarp();
                        const int tok = lane >> 2, col = fcol + (lane & 3) * 8;
#pragma unroll
                        for (int a = 0; a < 3; ++a)
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                const uint4 v = lds128(st + a * TN_STASH_BYTES + (8 * i + tok) * 128 + (((sub + (lane & 3)) ^ tok) << 4));
                                if (c + 8 * i + tok < rows && col < args.Mw)
                                    *reinterpret_cast<uint4*>(dst[a] + (size_t)(row0 + c + 8 * i + tok) * args.ep.ldo + col) = v;
                            }
                    }
                    ok = bar_vote_all(pair_bar, 64, ok);       // both halves of the lines are there (or one of the two gives up)
                    if (copies && ok && whole) {
                        const int f0 = ti.mt * 256 + 128 * (int)rank + 64 * (quarter >> 1);
#pragma unroll
                        for (int a = 0; a < 3; ++a)
                            if (f0 < args.Mw) tma_store_2d(&maps.b1[3 + a], st + a * TN_STASH_BYTES, f0, row0 + c);
                        tma_store_commit();
                    }
                    tn_write_dots(args.ep, dot, row0 + c, rows - c, tpair, fcol, args.Mw, lane);
                    if (!ok) { gone = true; break; }
                }
            } else {
                const int mcol = ti.mt * 256 + 128 * (int)rank + 32 * quarter;      // first output column of this warp
#pragma unroll 1
                for (int c = 0; c < nmma; c += 32) {
                    float v0[16], v1[16];
                    tmem_frag4(taddr + c, v0);
                    tmem_frag4(taddr + (16u << 16) + c, v1);
                    tmem_frag_wait(v0, v1);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if constexpr (KIND == TN_F2) {
                            const float2 g = lds64f(gbuf + 4u * (c + 8 * j + tpair));
                            v0[4 * j] *= g.x; v0[4 * j + 1] *= g.y; v0[4 * j + 2] *= g.x; v0[4 * j + 3] *= g.y;
                            v1[4 * j] *= g.x; v1[4 * j + 1] *= g.y; v1[4 * j + 2] *= g.x; v1[4 * j + 3] *= g.y;
                        }
                        stmatrix4_trans(wb + 512 * j + fo, pack_bf16x2(v0[4 * j], v0[4 * j + 1]), pack_bf16x2(v0[4 * j + 2], v0[4 * j + 3]),
                                        pack_bf16x2(v1[4 * j], v1[4 * j + 1]), pack_bf16x2(v1[4 * j + 2], v1[4 * j + 3]));
                    }
                    __syncwarp();
                    tn_write_rows<4>(args.ep.out0, args.ep.ldo, wb, row0 + c, rows - c, mcol, args.Mw, lane);
                    __syncwarp();
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(tempty_bar(buf) & T2_PEER_MASK);
        });
        if (KIND == TN_B2S && copies) tma_store_wait_all();
    }

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
template <int KIND>
inline bool tn_set_smem() {
    return cudaFuncSetAttribute(tn_gemm_kernel<KIND, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, TN_SMEM_BYTES) == cudaSuccess &&
           cudaFuncSetAttribute(tn_gemm_kernel<KIND, KIND != TN_F1G>, cudaFuncAttributeMaxDynamicSharedMemorySize, TN_SMEM_BYTES) == cudaSuccess;
}
inline mop_status tn_init() {
    return tn_set_smem<TN_F1>() && tn_set_smem<TN_F2>() && tn_set_smem<TN_F1G>() && tn_set_smem<TN_B4>() && tn_set_smem<TN_B2>() && tn_set_smem<TN_B2S>()
               ? MOP_OK : MOP_ERR_CUDA;
}

// Tables behind `tiles`: 128-row tiles, (the mixed schedule's second list,) token tiles.
inline int32_t* tn_table(const TcPlan* p, int32_t* tiles) {
    return tiles + 2 * (tc_tile_table_bytes(p->s.T * p->s.k, p->s.E) / 4);
}
inline mop_status tn_build_tiles(TcPlan* p, const int32_t* offsets, int32_t* tiles, bool rows128, cudaStream_t st) {
    p->prof->begin("tn_build_ttiles", st);
    pdl_launch(tn_build_ttiles_kernel, rows128 ? 2 : 1, 1024, 0, st, offsets, p->s.E, tn_table(p, tiles), tiles);
    p->prof->end(st);
    return cudaGetLastError() == cudaSuccess ? MOP_OK : MOP_ERR_CUDA;
}

// Weights that are read by one token tile only need no place in L2: as evict-first lines they leave the activations there, which
// the next kernels of the layer read.  That is so up to about 256 rows per expert (a second tile reads its weight tile again, from
// DRAM if it went: 384 rows, d = 2048, f = 1408: up-projection 230 us, evicted first 235; its backward 204 and 211), and pays
// where the activations fit beside them (d = 7168, 16384 rows: 929 us and 935).  One layer, d = 2048, f = 1408, 64 experts, default
// policy and evict-first: 6 rows per expert 216 and 206 us, 48 rows 245 and 235, 96 rows 264 and 257, 171 rows 290 and 285.
inline bool tn_stream_weights(const mop_moe_shape& s) {
    const uint64_t M = (uint64_t)s.T * s.k;
    return M <= 240ull * s.E && M * (uint64_t)(s.d + s.f) * 2 <= (96ull << 20);
}

inline TnArgs tn_base_args(const TcPlan* p, int32_t* tiles, int kind, int32_t* status) {
    int32_t* table = tn_table(p, tiles);
    TnArgs g{};
    g.next = table + TT_NEXT + kind;
    g.ttiles = reinterpret_cast<const int4*>(table + TT_TILES);
    g.n_ttiles = table;
    g.status = status;
    return g;
}

// Maps of a [rows, cols] bf16 token matrix with boxes of 16, 32, .. 128 rows, as far as a tile can need them.  The caller's tables
// may give one expert every row (indices that name it more than once for a token included): a tile has up to min(rows, 256) rows,
// half of them (rounded up to 8) per CTA.
inline bool tn_token_maps(const TcPlan* p, CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols) {
    const int most = rows < 256 ? (int)rows : 256;
    const int boxes = tn_box(most) + 1;
    for (int i = 0; i < boxes; ++i)
        if (!tc_map_2d(p, &m[i], base, rows, cols, 16 * (i + 1))) return false;
    return true;
}

template <int KIND>
inline mop_status tn_launch(const TcPlan* p, const char* name, const TnMaps& m, const TnArgs& g, cudaStream_t st) {
    p->prof->begin(name, st);
    const bool once = KIND != TN_F1G && tn_stream_weights(p->s);
    pdl_launch(once ? tn_gemm_kernel<KIND, KIND != TN_F1G> : tn_gemm_kernel<KIND, false>, p->sm_count & ~1, TN_THREADS,
               TN_SMEM_BYTES, st, m, g);
    p->prof->end(st);
    return cudaGetLastError() == cudaSuccess ? MOP_OK : MOP_ERR_CUDA;
}

// Up-projection + SwiGLU on the tokens-on-N kernel (`tiles`: the tables of tn_build_tiles).
inline mop_status tn_up_swiglu(TcPlan* p, const TcFwdArgs& a, int32_t* tiles, int32_t* status, bool gemm_follows, cudaStream_t st) {
    const mop_moe_shape& s = p->s;
    const uint64_t M = tc_rows(p);
    TnMaps m;
    if (!tc_map_3d(p, &m.a0, a.W_gate, s.E, s.d, s.f, TN_BK) || !tc_map_3d(p, &m.a1, a.W_up, s.E, s.d, s.f, TN_BK) ||
        !tn_token_maps(p, m.b, a.Xp, M, s.d))
        return MOP_ERR_CUDA;
    TnArgs g = tn_base_args(p, tiles, TN_F1, status);
    g.tiles_m = ceil_div(s.f, 128); g.kblocks = ceil_div(s.d, TN_BK); g.Mw = s.f;
    g.ep.out0 = a.H; g.ep.out1 = a.G_save; g.ep.out2 = a.U_save; g.ep.ldo = s.f; g.ep.M_total = (int)M;
    g.gemm_follows = gemm_follows;
    return tn_launch<TN_F1>(p, "gemm_up_swiglu", m, g, st);
}

// Up-projection + SwiGLU reading its token rows straight from the unpermuted x (no Xp, no stash).
inline mop_status tn_up_swiglu_gather(TcPlan* p, const bf16* x, const TcFwdArgs& a, int32_t* tiles, int32_t* status,
                                      cudaStream_t st) {
    const mop_moe_shape& s = p->s;
    TnMaps m;
    if (!tc_map_2d(p, &m.b[0], x, s.T, s.d, 1) || !tc_map_3d(p, &m.a0, a.W_gate, s.E, s.d, s.f, TN_BK) ||
        !tc_map_3d(p, &m.a1, a.W_up, s.E, s.d, s.f, TN_BK))
        return MOP_ERR_CUDA;
    TnArgs g = tn_base_args(p, tiles, TN_F1G, status);
    g.tiles_m = ceil_div(s.f, 128); g.kblocks = ceil_div(s.d, TN_BK); g.Mw = s.f;
    g.row_src = a.row_src; g.topk = s.k;
    g.ep.out0 = a.H; g.ep.ldo = s.f; g.ep.M_total = s.T * s.k;
    return tn_launch<TN_F1G>(p, "gemm_up_swiglu_gather", m, g, st);
}

// Down-projection + gate on the tokens-on-N kernel.
inline mop_status tn_down_gate(TcPlan* p, const TcFwdArgs& a, int32_t* tiles, int32_t* status, cudaStream_t st) {
    const mop_moe_shape& s = p->s;
    const uint64_t M = tc_rows(p);
    TnMaps m;
    const bool split = s.d % 64 != 0;
    if (!(split ? tc_map_3d(p, &m.a0, a.W_down, s.E, s.f, s.d, TN_BK) : tc_map_chunked_3d(p, &m.a0, a.W_down, s.E, s.f, s.d, 2, TN_BK)) ||
        !tn_token_maps(p, m.b, a.H, M, s.f))
        return MOP_ERR_CUDA;
    TnArgs g = tn_base_args(p, tiles, TN_F2, status);
    g.tiles_m = ceil_div(s.d, 256); g.kblocks = ceil_div(s.f, TN_BK); g.Mw = s.d; g.a_split = split;
    g.ep.out0 = a.Yp; g.ep.gate = a.gate; g.ep.row_src = a.row_src; g.ep.ldo = s.d; g.ep.M_total = (int)M;
    return tn_launch<TN_F2>(p, "gemm_down_gate", m, g, st);
}

// Data gradient of the up-projection on the tokens-on-N kernel: dXp = dG W_gate^T + dU W_up^T.
inline mop_status tn_dgrad_gate_up(TcPlan* p, const TcBwdArgs& a, int32_t* tiles, int32_t* status, cudaStream_t st) {
    const mop_moe_shape& s = p->s;
    const uint64_t M = tc_rows(p);
    TnMaps m;
    if (!tc_map_3d(p, &m.a0, a.W_gate, s.E, s.d, s.f, 128) || !tc_map_3d(p, &m.a1, a.W_up, s.E, s.d, s.f, 128) ||
        !tn_token_maps(p, m.b, a.dG, M, s.f) || !tn_token_maps(p, m.b1, a.dU, M, s.f))
        return MOP_ERR_CUDA;
    TnArgs g = tn_base_args(p, tiles, TN_B4, status);
    g.tiles_m = ceil_div(s.d, 256); g.kblocks = ceil_div(s.f, TN_BK); g.Mw = s.d;
    g.ep.out0 = a.dXp; g.ep.ldo = s.d; g.ep.M_total = (int)M;
    g.gemm_follows = true;
    return tn_launch<TN_B4>(p, "gemm_dgrad_gate_up", m, g, st);
}

// Data gradient of the down-projection with the SwiGLU backward on the tokens-on-N kernel.
// Writes one dgate partial per 32 columns of f (part[f / 32][row]).
inline mop_status tn_dgrad_down(TcPlan* p, const TcBwdArgs& a, int32_t* tiles, int32_t* status, cudaStream_t st) {
    const mop_moe_shape& s = p->s;
    const uint64_t M = tc_rows(p);
    TnMaps m;
    if (!tc_map_3d(p, &m.a0, a.W_down, s.E, s.f, s.d, 128) || !tn_token_maps(p, m.b, a.dYp, M, s.d)) return MOP_ERR_CUDA;
    TnArgs g = tn_base_args(p, tiles, TN_B2, status);
    g.tiles_m = ceil_div(s.f, 256); g.kblocks = ceil_div(s.d, TN_BK); g.Mw = s.f;
    g.ep.out0 = a.dG; g.ep.out1 = a.dU; g.ep.out2 = a.gH; g.ep.in0 = a.G_save; g.ep.in1 = a.U_save; g.ep.in2 = a.H;
    g.ep.gate = a.gate; g.ep.row_src = a.row_src; g.ep.part = a.part; g.ep.ldo = s.f; g.ep.M_total = (int)M;
    g.gemm_follows = true;
    // Boxes where the epilogue (by the rows of a tile) is long beside the main loop (by d).  us, by warps and by boxes: d 512, f 1024,
    // 64 experts of 28 rows 29.3 and 29.0, 64 rows 39.0 and 37.1, 256 rows 86 and 72; d 1000, f 1416, 28 rows 55.5 and 56.4, 64 rows 67.8
    // and 65.9, 256 rows 152 and 119; d 2048, f 1408, 64 rows 91 and 97, 128 rows 106.9 and 109.8, 160 rows 117.1 and 117.5, 200 rows 133
    // and 129, 256 rows 160 and 150.  Longer K, with two buffers and a stage more: d 4096, f 1024, 200 rows 152 and 158; d 7168,
    // f 2048, 32 experts of 96 rows 189 and 197, 600 rows 476 and 493.
    if (s.d > 2048 || (uint64_t)s.T * s.k * 16 <= (uint64_t)s.d * s.E) return tn_launch<TN_B2>(p, "gemm_dgrad_down_dswiglu", m, g, st);
    const void* const boxes[6] = {a.G_save, a.U_save, a.H, a.dG, a.dU, a.gH};
    for (int i = 0; i < 6; ++i)
        if (!tc_map_2d(p, &m.b1[i], boxes[i], M, s.f, 16)) return MOP_ERR_CUDA;
    return tn_launch<TN_B2S>(p, "gemm_dgrad_down_dswiglu", m, g, st);
}

}  // namespace mop
