// Selection, permutation, token tiles and row copy of a small layer in one launch.
#pragma once
#include "permute.cuh"
#include "route.cuh"

namespace mop {

// From the logits to the expert-contiguous rows, by one cluster: a warp selects for one token, whose assignments are its run (a token's
// experts are distinct, so that its k lanes count and rank side by side), the permutation goes on as in perm_cluster_kernel, and
// the CTA copies the rows of its tokens.  Same tables and gates as the separate kernels.
// What it saves is two launches; what it costs is that eight SMs copy slower than all.  A whole forward, us, separate and in one:
// T 16, d 2048, E 64, k 6 152 and 149; T 256, d 256, E 8, k 2 22.6 and 21.0; 1 MiB of rows 33.6 and 31.4 (T 64, d 1024, k 8), 26.7
// and 26.2 (T 256, d 512, k 4), 31.6 and 31.7 (T 256, d 1024, k 2); 4 MiB 36.0 and 40.6 (T 256, d 1024, k 8; all f 64 but the first two).
constexpr int RP_MAX_T = PC_MAX_CTAS * PC_WARPS;
constexpr int RP_MAX_E = 256;
constexpr long long RP_MAX_BYTES = 1 << 20;        // of the copied rows

template <int Q>
__global__ void __launch_bounds__(PC_WARPS * 32)
route_permute_kernel(const float* __restrict__ z, const float* __restrict__ bias, int32_t* __restrict__ idx, float* __restrict__ gate,
                     int32_t* __restrict__ counts, int32_t* __restrict__ offsets, int32_t* __restrict__ perm_row,
                     int32_t* __restrict__ row_src, int T, int E, int k, int score_fn, int bias_mode, int per_cta,
                     int32_t* __restrict__ tile_table, const uint4* __restrict__ x, uint4* __restrict__ Xp, int vec_per_row) {
    extern __shared__ int32_t perm_smem[];
    const PermSmem sm(perm_smem, E);
    int32_t* rows = sm.wsum + 32;                      // [per_cta][k] rows of this CTA's assignments
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int n_ctas = gridDim.x, rank = blockIdx.x;   // the grid is one cluster
    int32_t* mine = sm.cnt + (size_t)warp * E;
    for (int e = lane; e < E; e += 32) mine[e] = 0;
    __syncwarp();
    pdl_begin();
    const int t0 = rank * per_cta, cta_tokens = max(0, min(per_cta, T - t0));
    const bool has = warp < cta_tokens;                // this warp's token is t0 + warp
    const size_t a = ((size_t)t0 + warp) * k + lane;
    int e = 0;
    if (has) {
        float g;
        select_token<Q>(z + ((size_t)t0 + warp) * E, bias, E, k, score_fn, bias_mode, lane, e, g);
        if (lane < k) {
            idx[a] = e;
            gate[a] = g;
            mine[e] = 1;
        }
    }
    perm_cluster_scan(sm, counts, offsets, E, n_ctas, rank);
    if (has && lane < k) {
        const int p = mine[e] + sm.first[e];
        perm_row[a] = p;
        row_src[p] = (int32_t)a;
        rows[warp * k + lane] = p;
    }
    if (tile_table && rank == n_ctas - 1) write_token_tiles<PC_WARPS * 32>(sm.off, E, tile_table, sm.wsum);
    __syncthreads();
    constexpr int V = 4;                               // vectors of a lane in flight
    const int segs = (vec_per_row + 32 * V - 1) / (32 * V);
    for (int i = warp; i < cta_tokens * segs; i += PC_WARPS) {
        const int t = i / segs, c = (i - t * segs) * 32 * V + lane;
        const uint4* s = x + (size_t)(t0 + t) * vec_per_row + c;
        uint4 v[V];
#pragma unroll
        for (int q = 0; q < V; ++q)
            if (c + 32 * q < vec_per_row) v[q] = __ldg(s + 32 * q);
        for (int j = 0; j < k; ++j) {
            uint4* o = Xp + (size_t)rows[t * k + j] * vec_per_row + c;
#pragma unroll
            for (int q = 0; q < V; ++q)
                if (c + 32 * q < vec_per_row) o[32 * q] = v[q];
        }
    }
    __syncwarp();
    if (n_ctas > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

inline size_t route_permute_smem(int per_cta, int E, int k) { return perm_cluster_smem(E) + (size_t)per_cta * k * sizeof(int32_t); }
inline bool route_permute_init() {
    const int most = (int)route_permute_smem(PC_WARPS, RP_MAX_E, 32);
    return cudaFuncSetAttribute(route_permute_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, most) == cudaSuccess &&
           cudaFuncSetAttribute(route_permute_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, most) == cudaSuccess &&
           cudaFuncSetAttribute(route_permute_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, most) == cudaSuccess;
}
inline bool route_permute_fits(int T, int d, int E, int k) {
    return T > 0 && T <= RP_MAX_T && E <= RP_MAX_E && (long long)T * k * d * 2 <= RP_MAX_BYTES;
}
inline void launch_route_permute(const float* z, const float* bias, int32_t* idx, float* gate, int32_t* counts, int32_t* offsets,
                                 int32_t* perm_row, int32_t* row_src, int T, int d, int E, int k, int score_fn, int bias_mode,
                                 int32_t* tile_table, const uint4* x, uint4* Xp, cudaStream_t st) {
    const int ctas = T >= PC_MAX_CTAS ? PC_MAX_CTAS : 1, per_cta = ceil_div(T, ctas);
    auto go = [&](auto kernel) {
        pdl_launch_clusters(kernel, ctas, ctas, PC_WARPS * 32, route_permute_smem(per_cta, E, k), st, z, bias, idx, gate, counts, offsets,
                            perm_row, row_src, T, E, k, score_fn, bias_mode, per_cta, tile_table, x, Xp, d / 8);
    };
    if (E <= 64) go(route_permute_kernel<2>);
    else if (E <= 128) go(route_permute_kernel<4>);
    else go(route_permute_kernel<8>);
}

}  // namespace mop
