// Count / prefix-sum permutation of token-expert assignments into expert-contiguous rows, and the
// row movers (scatter x -> Xp, k-row combine Yp -> Y).  The order inside an expert is the assignment id: only counts, whose
// order does not matter, are ever made with atomics (of integers, in shared memory).
#pragma once
#include "tiles.cuh"

namespace mop {

constexpr int PERM_SEG = 512;    // assignments walked by one warp ("unit")
constexpr int PERM_WARPS = 4;    // warps per block in the histogram / rank kernels

// Histogram per unit: partial[u][e] = number of assignments of unit u that go to expert e.
__global__ void __launch_bounds__(PERM_WARPS * 32) perm_hist_kernel(const int32_t* __restrict__ idx,
                                                                    int32_t* __restrict__ partial, int M, int E) {
    pdl_begin();
    extern __shared__ int32_t perm_smem[];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    int32_t* cnt = perm_smem + (size_t)warp * E;
    const int unit = blockIdx.x * PERM_WARPS + warp;
    const int a0 = unit * PERM_SEG;
    if (a0 >= M) return;
    for (int e = lane; e < E; e += 32) cnt[e] = 0;
    __syncwarp();
    for (int it = 0; it < PERM_SEG / 32; ++it) {
        const int a = a0 + it * 32 + lane;
        int e = (a < M) ? idx[a] : -1;
        if (e < 0 || e >= E) e = -1;
        const uint32_t same = __match_any_sync(0xffffffffu, e);
        if (e >= 0 && lane == __ffs(same) - 1) cnt[e] += __popc(same);
        __syncwarp();
    }
    for (int e = lane; e < E; e += 32) partial[(size_t)unit * E + e] = cnt[e];
}

// Scan on one block: counts, offsets (exclusive scan over experts) and, in place of partial[u][e], the first
// row of unit u inside expert e; thread e owns expert e (strided if E > blockDim).  Used when there is nothing
// to permute (it still writes counts and offsets); otherwise perm_scan_cols_kernel + perm_rank_kernel do this.
__global__ void __launch_bounds__(1024) perm_scan_kernel(int32_t* __restrict__ partial, int32_t* __restrict__ counts,
                                                         int32_t* __restrict__ offsets, int units, int E) {
    pdl_begin();
    extern __shared__ int32_t scan_smem[];  // E + 1
    for (int e = threadIdx.x; e < E; e += blockDim.x) {
        int32_t run = 0;
        for (int u = 0; u < units; ++u) {
            const int32_t c = partial[(size_t)u * E + e];
            partial[(size_t)u * E + e] = run;
            run += c;
        }
        counts[e] = run;
        scan_smem[e] = run;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        // exclusive scan over E by one warp, 32 experts per step
        int32_t carry = 0;
        for (int e0 = 0; e0 < E; e0 += 32) {
            const int e = e0 + threadIdx.x;
            const int32_t c = (e < E) ? scan_smem[e] : 0;
            int32_t inc = c;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int32_t o = __shfl_up_sync(0xffffffffu, inc, off);
                if ((int)threadIdx.x >= off) inc += o;
            }
            if (e < E) scan_smem[e] = carry + inc - c;
            carry += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (threadIdx.x == 0) scan_smem[E] = carry;
    }
    __syncthreads();
    for (int e = threadIdx.x; e <= E; e += blockDim.x) offsets[e] = scan_smem[e];
    for (int e = threadIdx.x; e < E; e += blockDim.x) {
        const int32_t o = scan_smem[e];
        for (int u = 0; u < units; ++u) partial[(size_t)u * E + e] += o;
    }
}

// Column scan, spread over the GPU: a block owns 32 experts (a lane each: coalesced 128-byte rows of
// partial[u][.]) and its eight warps own eight contiguous ranges of units.  In place of partial[u][e]: the
// number of rows of expert e in the units before u; counts[e] = the expert's total.  Fixed order, no atomics.
constexpr int PSCAN_WARPS = 8;
__global__ void __launch_bounds__(PSCAN_WARPS * 32) perm_scan_cols_kernel(int32_t* __restrict__ partial,
                                                                          int32_t* __restrict__ counts, int units,
                                                                          int E) {
    pdl_begin();
    __shared__ int32_t tot[PSCAN_WARPS][32];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int e = blockIdx.x * 32 + lane;
    const int per = (units + PSCAN_WARPS - 1) / PSCAN_WARPS;
    const int u0 = min(units, warp * per), u1 = min(units, u0 + per);
    int32_t run = 0;
    if (e < E)
        for (int u = u0; u < u1; ++u) {
            const int32_t c = partial[(size_t)u * E + e];
            partial[(size_t)u * E + e] = run;
            run += c;
        }
    tot[warp][lane] = run;
    __syncthreads();
    int32_t before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < PSCAN_WARPS; ++w) {
        if (w < warp) before += tot[w][lane];
        total += tot[w][lane];
    }
    if (e < E) {
        if (before)
            for (int u = u0; u < u1; ++u) partial[(size_t)u * E + e] += before;
        if (warp == 0) counts[e] = total;
    }
}

// Rank: second walk over the same segments; perm_row[a] = offsets[e] + base[u][e] + rank inside the unit.
// Every block scans counts[] into the experts' offsets for itself (E <= 1024 words of shared memory);
// block 0 also writes them out.
__global__ void __launch_bounds__(PERM_WARPS * 32) perm_rank_kernel(const int32_t* __restrict__ idx,
                                                                    const int32_t* __restrict__ base,
                                                                    const int32_t* __restrict__ counts,
                                                                    int32_t* __restrict__ offsets,
                                                                    int32_t* __restrict__ perm_row,
                                                                    int32_t* __restrict__ row_src, int M, int E) {
    pdl_begin();
    extern __shared__ int32_t perm_smem[];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    int32_t* off = perm_smem + (size_t)PERM_WARPS * E;   // E + 1 words
    for (int e = threadIdx.x; e < E; e += blockDim.x) off[e] = counts[e];
    __syncthreads();
    if (warp == 0) {
        // exclusive scan over E by one warp, 32 experts per step
        int32_t carry = 0;
        for (int e0 = 0; e0 < E; e0 += 32) {
            const int e = e0 + lane;
            const int32_t c = (e < E) ? off[e] : 0;
            int32_t inc = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t v = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += v;
            }
            if (e < E) off[e] = carry + inc - c;
            carry += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (lane == 0) off[E] = carry;
    }
    __syncthreads();
    if (blockIdx.x == 0)
        for (int e = threadIdx.x; e <= E; e += blockDim.x) offsets[e] = off[e];
    int32_t* run = perm_smem + (size_t)warp * E;
    const int unit = blockIdx.x * PERM_WARPS + warp;
    const int a0 = unit * PERM_SEG;
    if (a0 >= M) return;
    for (int e = lane; e < E; e += 32) run[e] = base[(size_t)unit * E + e] + off[e];
    __syncwarp();
    const uint32_t lt = (1u << lane) - 1u;
    for (int it = 0; it < PERM_SEG / 32; ++it) {
        const int a = a0 + it * 32 + lane;
        int e = (a < M) ? idx[a] : -1;
        if (e < 0 || e >= E) e = -1;
        const uint32_t same = __match_any_sync(0xffffffffu, e);
        int32_t p = -1;
        if (e >= 0) p = run[e] + __popc(same & lt);
        __syncwarp();
        if (e >= 0 && lane == __ffs(same) - 1) run[e] += __popc(same);
        __syncwarp();
        if (a < M) {
            perm_row[a] = p;
            if (p >= 0) row_src[p] = a;
        }
    }
}

// The whole permutation in ONE launch: a cluster of up to eight CTAs of 32 warps, each warp with its run of `per_warp` assignments.
// A warp counts its run (counts need no order: atomics on its own row of shared memory), a thread per expert scans the 32 rows of
// its CTA, the CTAs read each other's totals through distributed shared memory, every CTA scans the experts for itself, and the
// warps walk their runs again in order.  Same tables as the three kernels above.  tile_table: the token tiles of the GEMMs too.
// Bounded by latency, and by the scattered row_src entries (a store of 32 of them takes 32 cycles of an SM, and there are eight SMs)
// where there are many: us a call in a graph, three kernels (up to 4096 assignments one block doing their work) and this
// one: M 32, E 8 4.4 and 2.4; 512, 256 11.0 and 3.6; 4096, 64 11.4 and 4.8; 4611, 20 13.0 and 4.6; 24576, 64 15.7 and 6.9; 16384,
// 1024 20.8 and 10.0; 131072, 256 21.9 and 24.0; 262144, 64 25.4 and 37.5.  Hence the line, PC_MAX_M.
constexpr int PC_WARPS = 32;
constexpr int PC_BATCH = 8;            // loads of a lane in flight
constexpr long long PC_MAX_M = 98304;
constexpr int PC_MAX_CTAS = 8;         // the portable cluster size
struct PermSmem {
    int32_t *cnt, *first, *off, *tot, *wsum;
    __device__ PermSmem(int32_t* base, int E) {
        cnt = base;                                    // [PC_WARPS][E] counts of the warps, then the next rows of each
        first = cnt + (size_t)PC_WARPS * E;            // [E] first row of this CTA's assignments of an expert
        off = first + E;                               // [E + 1]
        tot = off + E + 1;                             // [E] this CTA's totals, read by the others
        wsum = tot + E;                                // [32]
    }
};
inline size_t perm_cluster_smem(int E) { return ((size_t)PC_WARPS * E + 3 * E + 1 + 32) * sizeof(int32_t); }

// From the warps' counts to their first rows (less sm.first, which the caller adds), counts, offsets and sm.off.  Every CTA of the
// cluster calls it with all its threads, and waits for the cluster's barrier once more before it leaves (n_ctas > 1).
__device__ __forceinline__ void perm_cluster_scan(const PermSmem& sm, int32_t* __restrict__ counts, int32_t* __restrict__ offsets,
                                                  int E, int n_ctas, int rank) {
    const int tid = threadIdx.x;
    __syncthreads();
    int total = 0;
    if (tid < E) {                                     // E <= 1024: a thread per expert
#pragma unroll
        for (int w0 = 0; w0 < PC_WARPS; w0 += 16) {
            int c[16];
#pragma unroll
            for (int w = 0; w < 16; ++w) c[w] = sm.cnt[(w0 + w) * E + tid];
#pragma unroll
            for (int w = 0; w < 16; ++w) { sm.cnt[(w0 + w) * E + tid] = total; total += c[w]; }
        }
        sm.tot[tid] = total;
    }
    int before = 0;
    if (n_ctas > 1) {
        cluster_sync_all();
        if (tid < E) {
            const uint32_t addr = (uint32_t)__cvta_generic_to_shared(sm.tot + tid);
            total = 0;
            for (int r = 0; r < n_ctas; ++r) {
                int v;
                asm volatile("{\n.reg .b32 a;\nmapa.shared::cluster.u32 a, %1, %2;\nld.shared::cluster.s32 %0, [a];\n}"
                             : "=r"(v) : "r"(addr), "r"(r) : "memory");
                if (r < rank) before += v;
                total += v;
            }
        }
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    }
    int rows;
    const int base = block_exclusive_sum<PC_WARPS * 32>(total, sm.wsum, rows);
    if (tid < E) {
        sm.off[tid] = base;
        sm.first[tid] = base + before;
        if (rank == 0) { counts[tid] = total; offsets[tid] = base; }
    }
    if (tid == 0) {
        sm.off[E] = rows;
        if (rank == 0) offsets[E] = rows;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(PC_WARPS * 32) perm_cluster_kernel(const int32_t* __restrict__ idx, int32_t* __restrict__ counts,
                                                                     int32_t* __restrict__ offsets, int32_t* __restrict__ perm_row,
                                                                     int32_t* __restrict__ row_src, int M, int E, int per_warp,
                                                                     int32_t* __restrict__ tile_table) {
    extern __shared__ int32_t perm_smem[];
    const PermSmem sm(perm_smem, E);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int n_ctas = gridDim.x, rank = blockIdx.x;   // the grid is one cluster
    int32_t* mine = sm.cnt + (size_t)warp * E;
    for (int e = lane; e < E; e += 32) mine[e] = 0;
    __syncwarp();
    pdl_begin();
    const long long a0 = (long long)(rank * PC_WARPS + warp) * per_warp;
    const int n = (int)max(0ll, min((long long)per_warp, M - a0));       // assignments of this warp
    const int32_t* run_idx = idx + a0;
    auto load = [&](int b, int (&ev)[PC_BATCH]) {
#pragma unroll
        for (int i = 0; i < PC_BATCH; ++i) {
            const int o = b + 32 * i + lane;
            const int e = o < n ? run_idx[o] : -1;
            ev[i] = e >= 0 && e < E ? e : -1;
        }
    };
    for (int b = 0; b < n; b += 32 * PC_BATCH) {
        int ev[PC_BATCH];
        load(b, ev);
#pragma unroll
        for (int i = 0; i < PC_BATCH; ++i)
            if (ev[i] >= 0) atomicAdd(&mine[ev[i]], 1);
    }
    perm_cluster_scan(sm, counts, offsets, E, n_ctas, rank);
    if (n > 0) {
        for (int e = lane; e < E; e += 32) mine[e] += sm.first[e];
        __syncwarp();
        const uint32_t lt = (1u << lane) - 1u;
        for (int b = 0; b < n; b += 32 * PC_BATCH) {
            int ev[PC_BATCH];
            load(b, ev);
#pragma unroll
            for (int i = 0; i < PC_BATCH; ++i) {
                if (b + 32 * i >= n) break;
                const int e = ev[i];
                const uint32_t same = __match_any_sync(0xffffffffu, e);
                int32_t p = -1;
                if (e >= 0) p = mine[e] + __popc(same & lt);
                __syncwarp();
                if (e >= 0 && (same & lt) == 0) mine[e] += __popc(same);
                __syncwarp();
                const int o = b + 32 * i + lane;
                if (o < n) {
                    perm_row[a0 + o] = p;
                    if (p >= 0) row_src[p] = (int32_t)(a0 + o);
                }
            }
        }
    }
    if (tile_table && rank == n_ctas - 1) write_token_tiles<PC_WARPS * 32>(sm.off, E, tile_table, sm.wsum);
    __syncwarp();
    if (n_ctas > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
inline bool perm_cluster_init() {
    return cudaFuncSetAttribute(perm_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)perm_cluster_smem(TT_MAX_E)) ==
           cudaSuccess;
}
inline bool perm_cluster_fits(long long M) { return M <= PC_MAX_M; }
inline void launch_perm_cluster(const int32_t* idx, int32_t* counts, int32_t* offsets, int32_t* perm_row, int32_t* row_src, int M,
                                int E, int32_t* tile_table, cudaStream_t st) {
    int ctas = 1;
    while (ctas < PC_MAX_CTAS && ctas * PC_WARPS * 32 < M) ctas *= 2;
    const int per_warp = ceil_div(ceil_div(M, ctas * PC_WARPS), 32) * 32;
    pdl_launch_clusters(perm_cluster_kernel, ctas, ctas, PC_WARPS * 32, perm_cluster_smem(E), st, idx, counts, offsets, perm_row,
                        row_src, M, E, per_warp, tile_table);
}

// Scatter rows: one warp per token reads x[t,:] once (16-byte vectors, coalesced) and writes it to
// its k destination rows.  Used for x -> Xp and for dY -> dYp.
__global__ void __launch_bounds__(256) scatter_rows_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst,
                                                           const int32_t* __restrict__ perm_row, int T, int k,
                                                           int vec_per_row, TileJob job) {
    pdl_begin();
    if (tile_block(job)) return;
    const int warps_per_block = blockDim.x / 32, block = blockIdx.x - job.blocks(), blocks = gridDim.x - job.blocks();
    const int lane = threadIdx.x % 32;
    for (int t = block * warps_per_block + threadIdx.x / 32; t < T; t += blocks * warps_per_block) {
        int32_t myrow = -1;
        if (lane < k) myrow = perm_row[(size_t)t * k + lane];  // k <= 32 checked on the host
        const uint4* s = src + (size_t)t * vec_per_row;
        for (int c0 = 0; c0 < vec_per_row; c0 += 128) {
            uint4 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int c = c0 + q * 32 + lane;
                if (c < vec_per_row) v[q] = __ldg(s + c);
            }
            for (int j = 0; j < k; ++j) {
                const int32_t p = __shfl_sync(0xffffffffu, myrow, j);
                if (p < 0) continue;
                uint4* o = dst + (size_t)p * vec_per_row;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int c = c0 + q * 32 + lane;
                    if (c < vec_per_row) __stcs(o + c, v[q]);
                }
            }
        }
    }
}

// Scatter rows with the whole source row in registers (VPL 16-byte vectors per lane, rows of up to 512 VPL
// bytes): the row is read once and each of its k copies is written as one contiguous run, which DRAM takes
// better than pieces of 2 KiB interleaved over k rows (random 2 KiB pieces: 4.4 TB/s at T = 16384, d = 7168).
template <int VPL>
__global__ void __launch_bounds__(256) scatter_rows_reg_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst,
                                                               const int32_t* __restrict__ perm_row, int T, int k,
                                                               int vec_per_row, TileJob job) {
    pdl_begin();
    if (tile_block(job)) return;
    const int warps_per_block = blockDim.x / 32, block = blockIdx.x - job.blocks(), blocks = gridDim.x - job.blocks();
    const int lane = threadIdx.x % 32;
    for (int t = block * warps_per_block + threadIdx.x / 32; t < T; t += blocks * warps_per_block) {
        int32_t myrow = -1;
        if (lane < k) myrow = perm_row[(size_t)t * k + lane];  // k <= 32 checked on the host
        const uint4* s = src + (size_t)t * vec_per_row;
        uint4 v[VPL];
#pragma unroll
        for (int q = 0; q < VPL; ++q) {
            const int c = q * 32 + lane;
            if (c < vec_per_row) v[q] = __ldg(s + c);
        }
        for (int j = 0; j < k; ++j) {
            const int32_t p = __shfl_sync(0xffffffffu, myrow, j);
            if (p < 0) continue;
            uint4* o = dst + (size_t)p * vec_per_row;
#pragma unroll
            for (int q = 0; q < VPL; ++q) {
                const int c = q * 32 + lane;
                if (c < vec_per_row) __stcs(o + c, v[q]);
            }
        }
    }
}

// Combine: Y[t,:] = bf16(sum_j Yp[perm_row[t*k+j],:]) with the k-row sum kept in fp32 registers, j ascending.  Rows of -1 are left out.
__device__ __forceinline__ void add_bf16x8(float (&a)[8], const uint4& v) {
    a[0] += bf16_lo(v.x); a[1] += bf16_hi(v.x); a[2] += bf16_lo(v.y); a[3] += bf16_hi(v.y);
    a[4] += bf16_lo(v.z); a[5] += bf16_hi(v.z); a[6] += bf16_lo(v.w); a[7] += bf16_hi(v.w);
}
__device__ __forceinline__ uint4 pack_bf16x8(const float (&a)[8]) {
    return make_uint4(pack_bf16x2(a[0], a[1]), pack_bf16x2(a[2], a[3]), pack_bf16x2(a[4], a[5]), pack_bf16x2(a[6], a[7]));
}
// Much to do: a warp takes 2 KiB of a token's row, one of the k rows at a time.  HBM bound (T = 16384, d = 7168, k = 8: 338 us, 0.96 of
// the copy rate), and there one row of 2 KiB at a time does best (T = 8192, d = 4096, k = 4: 55 us, 64 with two rows of 1 KiB, 78 with
// four, 82 with a warp per token and rows of 4 KiB).
constexpr int COMB_SEG = 4;
__global__ void __launch_bounds__(256) combine_rows_kernel(const uint4* __restrict__ Yp, const int32_t* __restrict__ perm_row,
                                                            uint4* __restrict__ Y, int T, int k, int vec_per_row) {
    pdl_begin();
    const int lane = threadIdx.x % 32;
    const uint32_t wpb = blockDim.x / 32, segs = (vec_per_row + 32 * COMB_SEG - 1) / (32 * COMB_SEG);
    const uint32_t items = (uint32_t)T * segs;         // (32 bits: T < 2^31, and the rest of 16-byte vectors fits the device's memory)
    for (uint32_t i = blockIdx.x * wpb + threadIdx.x / 32; i < items; i += gridDim.x * wpb) {
        const int t = (int)(i / segs), c = (int)(i - t * segs) * 32 * COMB_SEG + lane;
        int32_t myrow = -1;
        if (lane < k) myrow = perm_row[(size_t)t * k + lane];
        float acc[COMB_SEG][8];
#pragma unroll
        for (int q = 0; q < COMB_SEG; ++q)
#pragma unroll
            for (int u = 0; u < 8; ++u) acc[q][u] = 0.0f;
        for (int j = 0; j < k; ++j) {
            const int32_t p = __shfl_sync(0xffffffffu, myrow, j);
            if (p < 0) continue;
            const uint4* src = Yp + (size_t)p * vec_per_row + c;
            uint4 v[COMB_SEG];
#pragma unroll
            for (int q = 0; q < COMB_SEG; ++q)
                if (c + 32 * q < vec_per_row) v[q] = __ldcs(src + 32 * q);
#pragma unroll
            for (int q = 0; q < COMB_SEG; ++q) add_bf16x8(acc[q], v[q]);
        }
#pragma unroll
        for (int q = 0; q < COMB_SEG; ++q)
            if (c + 32 * q < vec_per_row) Y[(size_t)t * vec_per_row + c + 32 * q] = pack_bf16x8(acc[q]);
    }
}
// Little to do, or rows too short for that: a thread per vector of Y, R of its rows in flight.  Nothing is left idle where a row is
// no multiple of what a warp takes, and there is little to set up.
template <int R>
__global__ void __launch_bounds__(256) combine_vectors_kernel(const uint4* __restrict__ Yp, const int32_t* __restrict__ perm_row,
                                                              uint4* __restrict__ Y, uint32_t n, int k, uint32_t vec_per_row) {
    pdl_begin();
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const uint32_t t = i / vec_per_row, c = i - t * vec_per_row;
        const int32_t* rows = perm_row + (size_t)t * k;
        float acc[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) acc[u] = 0.0f;
        for (int j = 0; j < k; j += R) {
            uint4 v[R];
            int32_t p[R];
#pragma unroll
            for (int r = 0; r < R; ++r) p[r] = j + r < k ? rows[j + r] : -1;
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (p[r] >= 0) v[r] = __ldcs(Yp + (size_t)p[r] * vec_per_row + c);
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (p[r] >= 0) add_bf16x8(acc, v[r]);
        }
        Y[i] = pack_bf16x8(acc);
    }
}

// Launchers: the register-row forms for rows of up to 16 KiB, the chunked kernels otherwise.
inline void launch_scatter_rows(const uint4* src, uint4* dst, const int32_t* perm_row, int T, int k, int vec_per_row,
                                int sm_count, cudaStream_t st, const TileJob& job = TileJob{}) {
    const int blocks = min(ceil_div(T, 8), sm_count * 8) + job.blocks();
    if (T <= 0) return;
    if (vec_per_row <= 32 * 8) pdl_launch(scatter_rows_reg_kernel<8>, blocks, 256, 0, st, src, dst, perm_row, T, k, vec_per_row, job);
    else if (vec_per_row <= 32 * 16) pdl_launch(scatter_rows_reg_kernel<16>, blocks, 256, 0, st, src, dst, perm_row, T, k, vec_per_row, job);
    else if (vec_per_row <= 32 * 28) pdl_launch(scatter_rows_reg_kernel<28>, blocks, 256, 0, st, src, dst, perm_row, T, k, vec_per_row, job);
    else if (vec_per_row <= 32 * 32) pdl_launch(scatter_rows_reg_kernel<32>, blocks, 256, 0, st, src, dst, perm_row, T, k, vec_per_row, job);
    else pdl_launch(scatter_rows_kernel, blocks, 256, 0, st, src, dst, perm_row, T, k, vec_per_row, job);
}
inline void launch_combine_rows(const uint4* Yp, const int32_t* perm_row, uint4* Y, int T, int k, int vec_per_row,
                                int sm_count, cudaStream_t st) {
    if (T <= 0) return;
    // us, vectors and pieces of rows: T 1000, d 1024 (128 thousand vectors) k 1 1.8 and 1.8, k 8 2.8 and 4.0; d 2048 (256 thousand) k 1
    // 2.3 and 2.2, k 8 4.4 and 4.6; T 4096, d 2048, k 1 4.9 and 4.5, k 4 9.4 and 8.1.  Short rows: T 16384, d 520 k 1 5.0 and 5.7,
    // k 4 10.9 and 14.1, k 8 24.7 and 30.3; d 768 k 1 6.9 and 6.2, k 4 19.4 and 20.5; d 1000, k 6 39.3 and 36.3.
    const long long n = (long long)T * vec_per_row;
    const bool few = n <= 512ll * sm_count;
    if (n <= 1280ll * sm_count || (vec_per_row < 96 && n < (1ll << 31))) {
        const int threads = few ? 128 : 256;
        const int blocks = (int)min((n + threads - 1) / threads, (long long)sm_count * (2048 / threads));
        auto go = [&](auto kernel) { pdl_launch(kernel, blocks, threads, 0, st, Yp, perm_row, Y, (uint32_t)n, k, (uint32_t)vec_per_row); };
        // rows in flight, for the latency of one: T 64, d 7168, k 8 2.2 us with eight, 2.3 with four, 2.5 with two.  With more vectors
        // than a few a thread's registers cost more than they give (T 512, d 2048, k 8 3.5, 2.9 and 3.0).
        if (k == 1) go(combine_vectors_kernel<1>);
        else if (k == 2) go(combine_vectors_kernel<2>);
        else if (k <= 4 || !few) go(combine_vectors_kernel<4>);
        else go(combine_vectors_kernel<8>);
        return;
    }
    const long long items = (long long)T * ceil_div(vec_per_row, 32 * COMB_SEG);
    pdl_launch(combine_rows_kernel, (int)min((items + 7) / 8, 8ll * sm_count), 256, 0, st, Yp, perm_row, Y, T, k, vec_per_row);
}

// dgate[a] = sum over n-tiles of the partial dot products written by the dgrad-down epilogue
// (row p = perm_row[a]; fixed order, so the result is reproducible).
__global__ void dgate_reduce_kernel(const float* __restrict__ part, const int32_t* __restrict__ perm_row,
                                    float* __restrict__ dgate, int M, int ntiles) {
    pdl_begin();
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= M) return;
    const int32_t p = perm_row[a];
    float s = 0.0f;
    if (p >= 0)
        for (int n = 0; n < ntiles; ++n) s += part[(size_t)n * M + p];
    dgate[a] = s;
}

// ---------------------------------------------------------------------------------------------
// Expert-chunked layer (only a fraction of the expert-contiguous buffers is live at a time).
// Chunk i of C takes the experts [eb(i), eb(i+1)) where eb(i) is the first expert whose first row is
// at or past ceil(i M / C): C chunks of at most ceil(M / C) + (rows of one expert) rows each.
// ---------------------------------------------------------------------------------------------

// Tables of one chunk: off_c[e] = first row of expert e inside the chunk's buffers (experts outside the
// chunk get no rows), row_src_c[r] = assignment of chunk row r, perm_c[a] = chunk row of assignment a or -1.
// bounds[0] = first row of the chunk in the whole layer, bounds[1] = its rows.
__global__ void __launch_bounds__(256) chunk_tables_kernel(const int32_t* __restrict__ offsets,
                                                           const int32_t* __restrict__ row_src,
                                                           const int32_t* __restrict__ perm_row,
                                                           int32_t* __restrict__ off_c, int32_t* __restrict__ row_src_c,
                                                           int32_t* __restrict__ perm_c, int32_t* __restrict__ bounds,
                                                           int E, int M, int chunk, int n_chunks) {
    pdl_begin();
    // The first expert at or past a row is the number of experts before it (offsets never decrease): counted by the block, not
    // searched for by one thread (12 us at 64 experts and 16384 assignments, now 9).
    const long long t0 = ((long long)chunk * M + n_chunks - 1) / n_chunks;
    const long long t1 = ((long long)(chunk + 1) * M + n_chunks - 1) / n_chunks;
    int e0 = 0, e1 = 0;
    for (int b = 0; b < E; b += blockDim.x) {
        const int e = b + threadIdx.x;
        const int32_t o = e < E ? offsets[e] : 0x7fffffff;
        e0 += __syncthreads_count(o < t0);
        e1 += __syncthreads_count(o < t1);
    }
    if (chunk + 1 == n_chunks) e1 = E;
    const int lo = offsets[e0], hi = offsets[e1];
    const int gtid = blockIdx.x * blockDim.x + threadIdx.x, gsz = gridDim.x * blockDim.x;
    if (gtid == 0) { bounds[0] = lo; bounds[1] = hi - lo; }
    for (int e = gtid; e <= E; e += gsz) off_c[e] = min(max(offsets[e], lo), hi) - lo;
    for (int r = gtid; r < hi - lo; r += gsz) row_src_c[r] = row_src[lo + r];
    for (int a = gtid; a < M; a += gsz) {
        const int32_t p = perm_row[a];
        perm_c[a] = (p >= lo && p < hi) ? p - lo : -1;
    }
}

// The row copies below give a warp CHUNK_SEG x 32 vectors of one row, all loaded before the first is used: a warp that walks
// a whole row a vector at a time has one DRAM access in flight per lane.
constexpr int CHUNK_SEG = 4;

// Xp_c[r,:] = x[row_src_c[r] / k, :] for the rows of a chunk (16-byte vectors).
// d = 7168, 4096 rows (117 MB): 25 us, 26 with a warp per row.
__global__ void __launch_bounds__(256) gather_rows_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst,
                                                          const int32_t* __restrict__ row_src_c,
                                                          const int32_t* __restrict__ bounds, int k, int vec_per_row,
                                                          TileJob job) {
    pdl_begin();
    if (tile_block(job)) return;
    const int lane = threadIdx.x % 32, wpb = blockDim.x / 32, block = blockIdx.x - job.blocks(), blocks = gridDim.x - job.blocks();
    const int segs = (vec_per_row + 32 * CHUNK_SEG - 1) / (32 * CHUNK_SEG);
    const long long items = (long long)bounds[1] * segs;
    for (long long i = (long long)block * wpb + threadIdx.x / 32; i < items; i += (long long)blocks * wpb) {
        const int r = (int)(i / segs), c = (int)(i % segs) * 32 * CHUNK_SEG + lane;
        const uint4* s = src + (size_t)(row_src_c[r] / k) * vec_per_row;
        uint4* o = dst + (size_t)r * vec_per_row;
        uint4 v[CHUNK_SEG];
#pragma unroll
        for (int u = 0; u < CHUNK_SEG; ++u)
            if (c + 32 * u < vec_per_row) v[u] = __ldg(s + c + 32 * u);
#pragma unroll
        for (int u = 0; u < CHUNK_SEG; ++u)
            if (c + 32 * u < vec_per_row) __stcs(o + c + 32 * u, v[u]);
    }
}

// Accumulating combine: acc[t,:] (+)= sum_j Yp_c[perm_c[t*k+j], :] over the token's rows inside the chunk
// (fp32, j ascending; chunks are added in chunk order, so the result is reproducible).  first: acc is
// written, not read; last: the sum is rounded once to bf16 into out instead of going back to acc.
// d = 7168, 4096 tokens, 4 chunks of 4096 rows (about 225 MB for one in the middle): 47 us, 93 with a warp per
// row; 2 or 7 vectors a lane instead of 4: 47 and 50.
__global__ void __launch_bounds__(256) combine_acc_kernel(const uint4* __restrict__ Yp_c,
                                                          const int32_t* __restrict__ perm_c, float4* __restrict__ acc,
                                                          uint4* __restrict__ out, int T, int k, int vec_per_row,
                                                          int first, int last) {
    pdl_begin();
    const int wpb = blockDim.x / 32, lane = threadIdx.x % 32;
    const int segs = (vec_per_row + 32 * CHUNK_SEG - 1) / (32 * CHUNK_SEG);
    const long long items = (long long)T * segs;
    for (long long i = (long long)blockIdx.x * wpb + threadIdx.x / 32; i < items; i += (long long)gridDim.x * wpb) {
        const int t = (int)(i / segs), c = (int)(i % segs) * 32 * CHUNK_SEG + lane;
        int32_t myrow = -1;
        if (lane < k) myrow = perm_c[(size_t)t * k + lane];
        uint32_t rows = __ballot_sync(0xffffffffu, myrow >= 0);
        if (!rows && !first && !last) continue;             // nothing of this token in the chunk
        float a[CHUNK_SEG][8];
        float4* ap = acc + ((size_t)t * vec_per_row + c) * 2;
#pragma unroll
        for (int u = 0; u < CHUNK_SEG; ++u) {
            float4 a0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), a1 = a0;
            if (!first && c + 32 * u < vec_per_row) { a0 = __ldcs(ap + 64 * u); a1 = __ldcs(ap + 64 * u + 1); }
            a[u][0] = a0.x; a[u][1] = a0.y; a[u][2] = a0.z; a[u][3] = a0.w;
            a[u][4] = a1.x; a[u][5] = a1.y; a[u][6] = a1.z; a[u][7] = a1.w;
        }
        for (; rows; rows &= rows - 1) {
            const uint4* y = Yp_c + (size_t)__shfl_sync(0xffffffffu, myrow, __ffs(rows) - 1) * vec_per_row + c;
            uint4 v[CHUNK_SEG];
#pragma unroll
            for (int u = 0; u < CHUNK_SEG; ++u) v[u] = c + 32 * u < vec_per_row ? __ldcs(y + 32 * u) : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int u = 0; u < CHUNK_SEG; ++u) {
                a[u][0] += bf16_lo(v[u].x); a[u][1] += bf16_hi(v[u].x); a[u][2] += bf16_lo(v[u].y); a[u][3] += bf16_hi(v[u].y);
                a[u][4] += bf16_lo(v[u].z); a[u][5] += bf16_hi(v[u].z); a[u][6] += bf16_lo(v[u].w); a[u][7] += bf16_hi(v[u].w);
            }
        }
#pragma unroll
        for (int u = 0; u < CHUNK_SEG; ++u) {
            if (c + 32 * u >= vec_per_row) continue;
            if (last) {
                uint4 o;
                o.x = pack_bf16x2(a[u][0], a[u][1]); o.y = pack_bf16x2(a[u][2], a[u][3]);
                o.z = pack_bf16x2(a[u][4], a[u][5]); o.w = pack_bf16x2(a[u][6], a[u][7]);
                out[(size_t)t * vec_per_row + c + 32 * u] = o;
            } else {
                ap[64 * u] = make_float4(a[u][0], a[u][1], a[u][2], a[u][3]);
                ap[64 * u + 1] = make_float4(a[u][4], a[u][5], a[u][6], a[u][7]);
            }
        }
    }
}

// dgate of the assignments that lie inside the chunk (others are left alone).
__global__ void dgate_reduce_chunk_kernel(const float* __restrict__ part, const int32_t* __restrict__ perm_c,
                                          float* __restrict__ dgate, int M, int rows_pitch, int ntiles) {
    pdl_begin();
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= M) return;
    const int32_t p = perm_c[a];
    if (p < 0) return;
    float s = 0.0f;
    for (int n = 0; n < ntiles; ++n) s += part[(size_t)n * rows_pitch + p];
    dgate[a] = s;
}

// Zero the weight gradients of the experts that received no row (the chunked backward writes only experts with rows).
__global__ void __launch_bounds__(256) zero_empty_experts_kernel(const int32_t* __restrict__ offsets,
                                                                float4* __restrict__ dWg, float4* __restrict__ dWu,
                                                                float4* __restrict__ dWd, size_t vec_per_expert) {
    pdl_begin();
    const int e = blockIdx.y;
    if (offsets[e + 1] > offsets[e]) return;
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < vec_per_expert; i += (size_t)gridDim.x * blockDim.x) {
        dWg[e * vec_per_expert + i] = z;
        dWu[e * vec_per_expert + i] = z;
        dWd[e * vec_per_expert + i] = z;
    }
}

}  // namespace mop
