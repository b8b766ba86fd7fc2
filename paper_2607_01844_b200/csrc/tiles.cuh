// Token tiles of the tokens-on-N kernels: the table and the block that writes it.
#pragma once
#include "common.cuh"

namespace mop {

// Words of the table: [0] number of tiles, [TT_NEXT + kind] work items that a kernel of this kind has handed out, from [TT_TILES]
// on {expert, first row, rows (1..256), position of the tile within its expert | tiles of the expert << 16} per tile.
constexpr int TT_NEXT = 16, TT_KINDS = 8, TT_TILES = 64;
constexpr int TT_MAX_E = 1024;

// Exclusive sum over the NT threads of a block in thread order; `total` is the sum over all.  warp_sum: NT / 32 words.
template <int NT>
__device__ __forceinline__ int block_exclusive_sum(int v, int32_t* warp_sum, int& total) {
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) warp_sum[warp] = inc;
    __syncthreads();
    const int mine = lane < NT / 32 ? warp_sum[lane] : 0;
    int upto = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, upto, o);
        if (lane >= o) upto += u;
    }
    total = __shfl_sync(0xffffffffu, upto, 31);
    const int before = __shfl_sync(0xffffffffu, upto - mine, warp);
    __syncthreads();                       // warp_sum may be used again
    return before + inc - v;
}

// The table from offsets [E + 1] (shared or global memory), by one block of NT threads; an expert's rows are cut into
// ceil(rows / 256) nearly equal tiles.
template <int NT>
__device__ __forceinline__ void write_token_tiles(const int32_t* offsets, int E, int32_t* __restrict__ table, int32_t* warp_sum) {
    constexpr int PER = TT_MAX_E / NT;
    int n = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int e = threadIdx.x * PER + i;
        if (e < E) n += (offsets[e + 1] - offsets[e] + 255) / 256;
    }
    int total;
    int at = block_exclusive_sum<NT>(n, warp_sum, total);
    int4* tiles = reinterpret_cast<int4*>(table + TT_TILES);
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int e = threadIdx.x * PER + i;
        if (e >= E) break;
        const int off = offsets[e], cnt = offsets[e + 1] - off, nt = (cnt + 255) / 256;
        const int sz = nt ? (((cnt + nt - 1) / nt + 15) & ~15) : 0;
        for (int q = 0; q < nt; ++q) tiles[at + q] = make_int4(e, off + q * sz, min(sz, cnt - q * sz), q | (nt << 16));
        at += nt;
    }
    if (threadIdx.x == 0) table[0] = total;
    if (threadIdx.x < TT_KINDS) table[TT_NEXT + threadIdx.x] = 0;
}

// The table as one more block (the first) of a row mover that runs before the GEMMs anyway, so that it costs no launch of its own.
struct TileJob {
    const int32_t* offsets;
    int E;
    int32_t* table;                        // null: no such block
    __host__ __device__ int blocks() const { return table ? 1 : 0; }
};
__device__ __forceinline__ bool tile_block(const TileJob& job) {
    if (!job.table || blockIdx.x != 0) return false;
    __shared__ int32_t warp_sum[8];
    write_token_tiles<256>(job.offsets, job.E, job.table, warp_sum);
    return true;
}

}  // namespace mop
