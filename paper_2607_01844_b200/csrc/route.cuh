// Router kernels: warp-per-token top-k with gate renormalisation, the tensor-core scoring path, the router backward
// (the router of the MoE block, Section 2.1 of the paper).
#pragma once
#include "route_score.cuh"

namespace mop {

// Sigmoid of the routing contract: a fixed sequence of fp32 operations, each rounded once
// (explicit-rounding intrinsics so that no contraction or fast path can change a step).
__device__ __forceinline__ float sigmoid_contract(float zv) {
    float u = -zv;
    u = fminf(fmaxf(u, -80.0f), 80.0f);
    const float n = rintf(__fmul_rn(u, 1.44269504088896341f));
    float r = __fmaf_rn(n, -0.693145751953125f, u);
    r = __fmaf_rn(n, -1.42860682030941723e-6f, r);
    float p = __fdiv_rn(1.0f, 720.0f);
    p = __fmaf_rn(p, r, __fdiv_rn(1.0f, 120.0f));
    p = __fmaf_rn(p, r, __fdiv_rn(1.0f, 24.0f));
    p = __fmaf_rn(p, r, __fdiv_rn(1.0f, 6.0f));
    p = __fmaf_rn(p, r, 0.5f);
    p = __fmaf_rn(p, r, 1.0f);
    p = __fmaf_rn(p, r, 1.0f);
    const float scale = __int_as_float(((int)n + 127) << 23);
    const float e = __fmul_rn(p, scale);
    return __fdiv_rn(1.0f, __fadd_rn(1.0f, e));
}

// ---------------------------------------------------------------------------------------------
// Selection: one warp per token, lane l holds the keys of the experts l, l + 32, .. in registers as integers of the same order, the
// largest of them at hand.  k rounds of two warp reductions (largest key; lowest id among the lanes that have it), after which the
// winner's lane looks through its keys again.  "Key greater, or equal and id lower"; k <= 32, lane j keeps the j-th pick.
// Bounded by latency: with keys in shared memory and ten shuffles a round T = 4096, E = 64, k = 6 took 8.4 us.
// ---------------------------------------------------------------------------------------------
constexpr int SEL_WARPS = 4;
constexpr int SEL_MAX_E = 1024;

// Larger key, larger integer; 0 is below every key (a NaN counts as the least key, -0 as +0).
__device__ __forceinline__ uint32_t order_key(float v) {
    const uint32_t u = __float_as_uint(v == v ? __fadd_rn(v, 0.0f) : -INFINITY);
    return u ^ ((uint32_t)((int32_t)u >> 31) | 0x80000000u);
}

// Q = E / 32 rounded up, or more.  On return lane j < k holds the j-th pick and its gate.
template <int Q>
__device__ __forceinline__ void select_token(const float* __restrict__ z, const float* __restrict__ bias, int E, int k,
                                             int score_fn, int bias_mode, int lane, int& my_e, float& my_gate) {
    // The loads of a lane first, all in flight: with the forms of the key inside one loop each load waited for the branch of the one
    // before it (router at T 64, d 64, k 1: E 1024 15.7 us, now 4.2; E 256 5.7 and 3.4; T 16384, E 256, k 8 with a bias 53 and 40).
    float v[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) v[q] = q * 32 + lane < E ? z[q * 32 + lane] : 0.0f;
    if (bias_mode != 0) {
        float b[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) b[q] = q * 32 + lane < E ? bias[q * 32 + lane] : 0.0f;
        if (bias_mode == 1 && score_fn == 1) {
#pragma unroll
            for (int q = 0; q < Q; ++q) v[q] = sigmoid_contract(v[q]);
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) v[q] = __fadd_rn(v[q], b[q]);
    }
    uint32_t key[Q], best = 0;
    int best_q = 0;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        key[q] = q * 32 + lane < E ? order_key(v[q]) : 0;
        if (key[q] > best) { best = key[q]; best_q = q; }
    }
    my_e = 0;
    for (int j = 0; j < k; ++j) {
        const uint32_t most = __reduce_max_sync(0xffffffffu, best);
        const uint32_t e = __reduce_min_sync(0xffffffffu, best == most ? (uint32_t)(best_q * 32 + lane) : 0xffffffffu);
        if (j == lane) my_e = (int)e;
        if ((e & 31u) == (uint32_t)lane) {
            best = 0;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                if (q == (int)(e >> 5)) key[q] = 0;
                if (key[q] > best) { best = key[q]; best_q = q; }
            }
        }
    }
    const bool act = lane < k;
    float zz = act ? z[my_e] : 0.0f;
    if (act && bias_mode == 2) zz = __fadd_rn(zz, bias[my_e]);
    float s;
    if (score_fn == 0) {
        float m = act ? zz : -INFINITY;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        s = act ? expf(zz - m) : 0.0f;
    } else {
        s = act ? sigmoidf_acc(zz) : 0.0f;
    }
    float sum = s;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    my_gate = s / sum;
}

template <int Q>
__global__ void __launch_bounds__(SEL_WARPS * 32) route_select_kernel(const float* __restrict__ z, const float* __restrict__ bias,
                                                                      int32_t* __restrict__ idx, float* __restrict__ gate, int T,
                                                                      int E, int k, int score_fn, int bias_mode) {
    pdl_begin();
    const int lane = threadIdx.x % 32, t = blockIdx.x * SEL_WARPS + threadIdx.x / 32;
    if (t >= T) return;
    int e;
    float g;
    select_token<Q>(z + (size_t)t * E, bias, E, k, score_fn, bias_mode, lane, e, g);
    if (lane < k) {
        idx[(size_t)t * k + lane] = e;
        gate[(size_t)t * k + lane] = g;
    }
}
inline void launch_route_select(const float* z, const float* bias, int32_t* idx, float* gate, int T, int E, int k, int score_fn,
                                int bias_mode, cudaStream_t st) {
    auto go = [&](auto kernel) {
        pdl_launch(kernel, ceil_div(T, SEL_WARPS), SEL_WARPS * 32, 0, st, z, bias, idx, gate, T, E, k, score_fn, bias_mode);
    };
    if (E <= 64) go(route_select_kernel<2>);
    else if (E <= 128) go(route_select_kernel<4>);
    else if (E <= 256) go(route_select_kernel<8>);
    else if (E <= 512) go(route_select_kernel<16>);
    else go(route_select_kernel<32>);
}

// ---------------------------------------------------------------------------------------------
// Fast scoring path: logits on the tensor cores, the contract's chain only where it can matter.
//
// 1. W_r (fp32) is split into three bf16 pieces, hi + mid + lo = W_r to 2^-24 relative (each
//    residual is exact in fp32), and x (bf16) is multiplied by the pieces on the tensor cores: z~
//    (route_score_pair_kernel; the K loop is summed in segments of 192, all three pieces, so that the
//    truncating accumulation inside the tensor core stays short; the segments are added in fp32 registers).
//    Every product is exact; what separates z~ from the contract's logit z (one fp32 fused
//    multiply-add per i, i ascending) is the rounding of the two summations.  Each rounding is at most
//    u = 2^-24 of a partial sum, and the partial sums of a logit grow like a random walk towards
//    ||x|| ||w|| / sqrt(d) for data without a common direction: d roundings give a standard deviation of
//    u ||x|| ||w|| / sqrt(6) per summation, whatever d.  The selection relies on
//        |z~ - z|  <=  eps_z(t) = 24 u ||x_t||_2 max_e ||W_r[:,e]||_2        (40 standard deviations).
//    This is a model, not a worst case (which is d u ||x|| ||w||): the realised maximum over millions
//    of logits is 3 to 6.2 u ||x|| ||w|| on every shape tried, the tests assert it, and every logit that
//    the kernel re-evaluates is compared with half the bound as it runs (mop_route_stats).
//    In key space a logit error e moves sigmoid(z) + b by at most (s (1 - s) + e / 8) e + 4e-7; approximate
//    keys are formed with the fast sigmoid, whose own error (below 1e-6) is added to that.
// 2. Screening pass, one warp per token: the k largest approximate keys, every key with the interval that
//    holds its exact value.  If the intervals of adjacent picks are disjoint and no other expert's
//    interval reaches the weakest pick, the exact keys have the same order and the token is done
//    (more than nine tenths of the tokens when the router is fresh; none of them with the biases of a
//    heavily skewed one).  The others are listed, and the experts in doubt of each go to that expert's list.
//    Chain pass: the contract's chain (__fmaf_rn, i ascending, W_r read through its transposed copy) for
//    every listed pair, 32 tokens of one expert per warp; the exact logits go over z~.  Resolving pass, one
//    warp per listed token: the evaluated intervals are points now and their keys the contract's; it selects
//    again, evaluates what is still in doubt, and so on until nothing that matters overlaps.  Indices and
//    their order are then those of the exact path.
// 3. Gates are ratios of scores, not an order: a pick keeps its approximate logit unless that could move
//    its gate by more than 5e-6 relative (score far from saturation), in which case its chain is
//    evaluated too; the gates then agree with the exact path's to 1e-6 + 1e-5 g.
// ---------------------------------------------------------------------------------------------

// W_r [d,E] -> three bf16 pieces [3,d,E], the transposed copy W_r^T [E,d] (32 x 32 tiles through shared
// memory) and, per 32-row slab, the partial squared column norms (summed by route_wnorm_kernel).
__global__ void __launch_bounds__(256) route_prep_kernel(const float* __restrict__ W_r, bf16* __restrict__ pieces,
                                                         float* __restrict__ W_rT, float* __restrict__ colsq,
                                                         int d, int E) {
    __shared__ float tile[32][33];
    const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
    const size_t n = (size_t)d * E;
    for (int r = ty; r < 32; r += 8) {
        float w = 0.0f;
        if (r0 + r < d && c0 + tx < E) {
            const size_t i = (size_t)(r0 + r) * E + c0 + tx;
            w = W_r[i];
            const bf16 hi = __float2bfloat16_rn(w);
            const float r1 = w - __bfloat162float(hi);          // exact
            const bf16 mid = __float2bfloat16_rn(r1);
            const float r2 = r1 - __bfloat162float(mid);        // exact
            pieces[i] = hi;
            pieces[n + i] = mid;
            pieces[2 * n + i] = __float2bfloat16_rn(r2);
        }
        tile[r][tx] = w;
    }
    __syncthreads();
    for (int c = ty; c < 32; c += 8)
        if (c0 + c < E && r0 + tx < d) W_rT[(size_t)(c0 + c) * d + r0 + tx] = tile[tx][c];
    if (ty == 0 && c0 + tx < E) {
        float sq = 0.0f;
        for (int r = 0; r < 32; ++r) sq = fmaf(tile[r][tx], tile[r][tx], sq);
        colsq[(size_t)blockIdx.y * E + c0 + tx] = sq;
    }
}

// Squared column norms ||W_r[:,e]||^2 from the slab partials: one warp per expert, fixed order (reproducible).
__global__ void __launch_bounds__(256) route_wnorm_kernel(const float* __restrict__ colsq, float* __restrict__ wsq,
                                                          int slabs, int E) {
    const int lane = threadIdx.x % 32;
    const int e = blockIdx.x * 8 + threadIdx.x / 32;
    if (e >= E) return;
    float sq = 0.0f;
    for (int s = lane; s < slabs; s += 32) sq += colsq[(size_t)s * E + e];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
    if (lane == 0) wsq[e] = sq;
}

// ||x_t||_2 per token: one warp per row, 16-byte loads.
__global__ void __launch_bounds__(256) route_xnorm_kernel(const bf16* __restrict__ x, float* __restrict__ xnorm, int T,
                                                          int d) {
    const int lane = threadIdx.x % 32;
    const int t = blockIdx.x * 8 + threadIdx.x / 32;
    if (t >= T) return;
    const uint4* row = reinterpret_cast<const uint4*>(x + (size_t)t * d);
    float sq = 0.0f;
    for (int v = lane; v < d / 8; v += 32) {
        const uint4 q = __ldg(row + v);
        const uint32_t w4[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float a = bf16_lo(w4[j]), b = bf16_hi(w4[j]);
            sq = fmaf(a, a, sq);
            sq = fmaf(b, b, sq);
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
    if (lane == 0) xnorm[t] = sqrtf(sq);
}

constexpr int SELF_WARPS = 2;     // warps per block of the fast selection (a warp that re-evaluates takes ~20 us)
constexpr float ROUTE_EPS_C = 24.0f;      // order:  |z~ - z| <= C 2^-24 ||x_t|| max_e ||W_r[:,e]||  (see below)
constexpr float ROUTE_EPS_GATE_C = 6.0f;  // gates:  the same with the largest error seen, not a bound (a tolerance, not an order)
constexpr float ROUTE_GATE_REL = 5e-6f;   // a pick whose gate could be off by more than this (relative) gets its chain
constexpr int SELF_XCHUNK = 512;  // elements of the token's row staged per step of the exact chains
constexpr int SELF_CAND = 4;      // chains evaluated side by side (one lane each), their W_r^T rows staged in shared memory
constexpr int SELF_WPITCH = SELF_XCHUNK + 4;   // row pitch of the staged W_r^T chunks: lanes read different banks
constexpr int SELF_SMEM_FLOATS = SELF_XCHUNK + SELF_CAND * SELF_WPITCH;   // per warp, besides the 2 E logit / list words

// Order-preserving map of a finite float to an unsigned integer (-0 counts as +0, as in a float comparison).
__device__ __forceinline__ uint32_t key_ord(float f) {
    uint32_t u = __float_as_uint(f);
    if (u == 0x80000000u) u = 0u;
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// k selection rounds over keys held in registers: lane l owns the experts e = l + 32 q, q < Q, key kv[q].
// A round is two warp reductions (largest key among the lanes' best untaken keys, then the lowest expert id
// among the lanes that hold it) and a rescan of the winner's own keys.  Lane j < k keeps the j-th pick: its
// expert, its key and the logit its gate is computed from; `taken` marks this lane's picked experts.
// Same order as route_select_kernel: larger key first, equal keys by lower id.
template <int Q>
__device__ __forceinline__ void select_rounds_reg(const float (&kv)[Q], uint32_t invalid, const float* zg, int k, int lane,
                                                  int& my_e, float& my_key, float& my_z, uint32_t& taken) {
    taken = 0;
    my_e = -1; my_key = 0.0f; my_z = 0.0f;
    float bk = 0.0f; int bq = -1;
    auto rescan = [&]() {
        bq = -1; bk = 0.0f;
        const uint32_t off = taken | invalid;
#pragma unroll
        for (int q = 0; q < Q; ++q)
            if (!((off >> q) & 1u) && (bq < 0 || kv[q] > bk)) { bq = q; bk = kv[q]; }
    };
    rescan();
    for (int j = 0; j < k; ++j) {
        const uint32_t mine = bq >= 0 ? key_ord(bk) : 0u;            // 0 lies below the image of every finite key
        const uint32_t top = __reduce_max_sync(0xffffffffu, mine);
        const int cand = (bq >= 0 && mine == top) ? lane + 32 * bq : 0x7fffffff;
        const int win = __reduce_min_sync(0xffffffffu, cand);
        const float wkey = __shfl_sync(0xffffffffu, bk, win & 31);
        if ((win & 31) == lane) { taken |= 1u << (win >> 5); rescan(); }
        if (j == lane) { my_e = win; my_key = wkey; my_z = zg[win]; }
    }
}

__device__ __forceinline__ float route_key(float zz, float b, int score_fn, int bias_mode) {
    return (score_fn == 1 && bias_mode == 1) ? __fadd_rn(sigmoid_contract(zz), b) : zz;
}
// Key of an approximate logit: the sigmoid by the fast exponential and division.  Against the contract's sequence it is
// off by less than 1e-6 (exponential: 2 + 1.173 |z| ulp, times the slope s (1 - s): at most 8e-8; division 2 ulp;
// the contract's own polynomial 2e-7), which key_error adds to the interval of such a key.
constexpr float ROUTE_FAST_KEY_ERR = 1e-6f;
__device__ __forceinline__ float route_key_approx(float zz, float b, int score_fn, int bias_mode) {
    return (score_fn == 1 && bias_mode == 1) ? sigmoidf_fast(zz) + b : zz;
}

// Bound on the error of an approximate key whose logit is off by at most ez (a little slack covers its own rounding).
__device__ __forceinline__ float key_error(float zz, float ez, int score_fn, int bias_mode) {
    if (!(score_fn == 1 && bias_mode == 1)) return ez;                   // the key is the logit itself
    const float s = sigmoidf_fast(zz);
    return 1.001f * (s * (1.0f - s) + 0.125f * ez) * ez + 4e-7f + ROUTE_FAST_KEY_ERR;   // |s''| <= 0.1
}

// One token, one warp.  RESOLVE = false: the screening pass; if some order or gate is in doubt it lists the experts
// whose chains are needed and returns false.  RESOLVE = true: starts with those logits exact, and evaluates the chains
// still in doubt until everything is settled.
// Lane l holds the keys of the experts l + 32 q in registers (Q = ceil(E / 32) rounded up to a supported size).
// zg: E floats (logits); clist: E ints, xs, ws: staging of the chains (RESOLVE only).
// pair_cnt [E], pair_list [E][T]: tokens listed per expert; pre [T][32]: bit q of word l: expert l + 32 q was listed.
template <bool RESOLVE, int Q>
__device__ __forceinline__ bool route_token(int t, int lane, float* zg, int32_t* clist, float* xs, float* ws,
                                            float* __restrict__ z, const float* __restrict__ z1,
                                            const float* __restrict__ bias,
                                            const bf16* __restrict__ x, const float* __restrict__ W_rT,
                                            const float* __restrict__ xnorm, float wmax, int32_t* __restrict__ idx,
                                            float* __restrict__ gate, int32_t* __restrict__ stats,
                                            int32_t* __restrict__ pair_cnt, int32_t* __restrict__ pair_list,
                                            uint32_t* __restrict__ pre, int T, int d, int E, int k, int score_fn,
                                            int bias_mode) {
    float* zrow = z + (size_t)t * E;
    float kv[Q];
    uint32_t invalid = 0;                            // slots q of this lane beyond E
    uint32_t exact = RESOLVE && pre ? pre[(size_t)t * 32 + lane] : 0;       // this lane's experts that carry the chain's logit
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int e = lane + 32 * q;
        kv[q] = 0.0f;
        if (e < E) {
            float zz = zrow[e];
            if (z1) {                                // the logit GEMM left two partial sums over K: add, keep the sum
                zz += z1[(size_t)t * E + e];
                zrow[e] = zz;
            }
            const float b = bias_mode ? bias[e] : 0.0f;
            if (bias_mode == 2) zz = __fadd_rn(zz, b);
            kv[q] = RESOLVE && ((exact >> q) & 1u) ? route_key(zz, b, score_fn, bias_mode)
                                                   : route_key_approx(zz, b, score_fn, bias_mode);
            zg[e] = zz;
        } else {
            invalid |= 1u << q;
        }
    }
    __syncwarp();
    // Bound of this token's logit error (see above).
    const float scale = 5.9604645e-8f * xnorm[t] * wmax;
    const float ez = ROUTE_EPS_C * scale, ez_gate = ROUTE_EPS_GATE_C * scale;
    int my_e; float my_key, my_z; uint32_t taken;
    int n_chains = 0, n_bad = 0;
    for (int iter = 0; iter <= k + 1; ++iter) {
        select_rounds_reg<Q>(kv, invalid, zg, k, lane, my_e, my_key, my_z, taken);
        // interval [lo, hi] that holds the exact key of each pick (a point once the chain was evaluated)
        const bool pick = lane < k;
        const uint32_t owner_exact = __shfl_sync(0xffffffffu, exact, pick ? (my_e & 31) : 0);
        const uint32_t pick_exact = pick ? (owner_exact >> (my_e >> 5)) & 1u : 1u;
        const float my_err = (pick && !pick_exact) ? key_error(my_z, ez, score_fn, bias_mode) : 0.0f;
        const float lo = pick ? my_key - my_err : INFINITY, hi = pick ? my_key + my_err : -INFINITY;
        const float next_hi = __shfl_down_sync(0xffffffffu, hi, 1), prev_lo = __shfl_up_sync(0xffffffffu, lo, 1);
        // a pick is in doubt if it may swap with a neighbour (NaN compares unsure: inputs must be finite)
        bool doubt = pick && ((lane + 1 < k && !(lo > next_hi)) || (lane > 0 && !(prev_lo > hi)));
        float lo_min = lo;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) lo_min = fminf(lo_min, __shfl_xor_sync(0xffffffffu, lo_min, off));
        // outsiders that could reach the weakest pick, and the picks they could reach.  Nearly all of them
        // fail already with the largest error any key can have (slope 1/4), which costs no transcendental.
        const float err_any = (score_fn == 1 && bias_mode == 1)
                                  ? 1.001f * (0.25f + 0.125f * ez) * ez + 4e-7f + ROUTE_FAST_KEY_ERR : ez;
        float out_hi = -INFINITY;
        int n_c = 0;
        uint32_t cands = 0;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int e = lane + 32 * q;
            bool cand = false;
            if (!(((taken | invalid) >> q) & 1u) && !(kv[q] + err_any < lo_min)) {
                const bool ex = (exact >> q) & 1u;
                const float h = kv[q] + (ex ? 0.0f : key_error(zg[e], ez, score_fn, bias_mode));
                if (!(h < lo_min)) { out_hi = fmaxf(out_hi, h); cand = !ex; }
            }
            if constexpr (RESOLVE) {
                const uint32_t m = __ballot_sync(0xffffffffu, cand);
                if (m) {
                    if (cand) clist[n_c + __popc(m & ((1u << lane) - 1u))] = e;
                    n_c += __popc(m);
                }
            } else {
                if (cand) cands |= 1u << q;
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) out_hi = fmaxf(out_hi, __shfl_xor_sync(0xffffffffu, out_hi, off));
        if (pick && !(lo > out_hi)) doubt = true;
        // gates: d g / g = (1 - s) dz for a sigmoid score, at most dz for a softmax over the picks
        if (pick && !pick_exact) {
            const float sens = (score_fn == 1) ? 1.0f - sigmoidf_fast(my_z) : 1.0f;
            if (sens * ez_gate > ROUTE_GATE_REL) doubt = true;
        }
        // picks in doubt whose logit is still approximate join the list
        const bool need = doubt && !pick_exact;
        const uint32_t m = __ballot_sync(0xffffffffu, need);
        if constexpr (!RESOLVE) {
            if (!m && !__any_sync(0xffffffffu, cands != 0)) break;
            for (uint32_t r = m; r; r &= r - 1) {
                const int e = __shfl_sync(0xffffffffu, my_e, __ffs(r) - 1);
                if ((e & 31) == lane) cands |= 1u << (e >> 5);
            }
            pre[(size_t)t * 32 + lane] = cands;
            for (uint32_t r = cands; r; r &= r - 1) {
                const int e = lane + 32 * (__ffs(r) - 1);
                pair_list[(size_t)e * T + atomicAdd(pair_cnt + e, 1)] = t;
            }
            return false;
        }
        if (need) clist[n_c + __popc(m & ((1u << lane) - 1u))] = my_e;
        n_c += __popc(m);
        if (n_c == 0) break;                         // every order that matters is settled (exact ties go by id)
        __syncwarp();
        for (int c0 = 0; c0 < n_c; c0 += SELF_CAND) {
            const int nc = min(SELF_CAND, n_c - c0);
            const bool mine = lane < nc;
            const int e = mine ? clist[c0 + lane] : 0;
            float acc = 0.0f;
            // All lanes fetch: the token's chunk (16 bytes per lane) and the same chunk of every candidate's row
            // of W_r^T (lane l: 16-byte pieces l, l + 32, ... of the nc rows laid end to end).  The fetch of chunk
            // i + 1 is in flight while the chains run over chunk i.
            constexpr int WV = SELF_CAND * SELF_XCHUNK / 4 / 32;      // 16-byte pieces of W per lane and chunk
            constexpr int XV = SELF_XCHUNK / 8 / 32;                  // 16-byte pieces of x per lane and chunk
            uint4 xq[XV];
            float4 wq[WV];
            auto fetch = [&](int i0) {
                const int n = min(SELF_XCHUNK, d - i0);              // a multiple of 8
#pragma unroll
                for (int u = 0; u < XV; ++u)
                    if (lane + 32 * u < n / 8)
                        xq[u] = __ldg(reinterpret_cast<const uint4*>(x + (size_t)t * d + i0) + lane + 32 * u);
#pragma unroll
                for (int u = 0; u < WV; ++u) {
                    const int v = lane + 32 * u, c = v / (SELF_XCHUNK / 4), j = v % (SELF_XCHUNK / 4);
                    if (c < nc && 4 * j < n)
                        wq[u] = __ldg(reinterpret_cast<const float4*>(W_rT + (size_t)clist[c0 + c] * d + i0) + j);
                }
            };
            fetch(0);
            for (int i0 = 0; i0 < d; i0 += SELF_XCHUNK) {
                const int n = min(SELF_XCHUNK, d - i0);
                __syncwarp();
                // x stays bf16 in shared memory (16 bytes = 8 elements per load in the chains: every shared-memory
                // instruction of a warp costs a wavefront however few lanes take part, and the chains of all
                // resident warps together are bound by those wavefronts when most tokens are listed)
#pragma unroll
                for (int u = 0; u < XV; ++u) reinterpret_cast<uint4*>(xs)[lane + 32 * u] = xq[u];
#pragma unroll
                for (int u = 0; u < WV; ++u) {
                    const int v = lane + 32 * u, c = v / (SELF_XCHUNK / 4), j = v % (SELF_XCHUNK / 4);
                    if (c < nc) *reinterpret_cast<float4*>(ws + c * SELF_WPITCH + 4 * j) = wq[u];
                }
                __syncwarp();
                if (i0 + SELF_XCHUNK < d) fetch(i0 + SELF_XCHUNK);
                if (mine) {
                    // the contract's chain: one fused multiply-add per i, i ascending
                    const float* wrow = ws + lane * SELF_WPITCH;
#pragma unroll 4
                    for (int i = 0; i < n; i += 8) {
                        const float4 w0 = *reinterpret_cast<const float4*>(wrow + i);
                        const float4 w1 = *reinterpret_cast<const float4*>(wrow + i + 4);
                        const uint4 xv = *reinterpret_cast<const uint4*>(reinterpret_cast<const bf16*>(xs) + i);
                        acc = __fmaf_rn(bf16_lo(xv.x), w0.x, acc);
                        acc = __fmaf_rn(bf16_hi(xv.x), w0.y, acc);
                        acc = __fmaf_rn(bf16_lo(xv.y), w0.z, acc);
                        acc = __fmaf_rn(bf16_hi(xv.y), w0.w, acc);
                        acc = __fmaf_rn(bf16_lo(xv.z), w1.x, acc);
                        acc = __fmaf_rn(bf16_hi(xv.z), w1.y, acc);
                        acc = __fmaf_rn(bf16_lo(xv.w), w1.z, acc);
                        acc = __fmaf_rn(bf16_hi(xv.w), w1.w, acc);
                    }
                }
            }
            float newkey = 0.0f;
            if (mine) {
                if (fabsf(zrow[e] - acc) > 0.5f * ez) ++n_bad;       // the model of the error is checked as we go
                zrow[e] = acc;                       // the exact logit replaces the approximate one
                const float b = bias_mode ? bias[e] : 0.0f;
                const float zz = (bias_mode == 2) ? __fadd_rn(acc, b) : acc;
                newkey = route_key(zz, b, score_fn, bias_mode);      // the contract's key
                zg[e] = zz;
            }
            // the evaluated experts' keys go to their owner lanes, which mark them exact
            for (int j = 0; j < nc; ++j) {
                const int ej = clist[c0 + j];
                const float kj = __shfl_sync(0xffffffffu, newkey, j);
                if ((ej & 31) == lane) {
                    exact |= 1u << (ej >> 5);
#pragma unroll
                    for (int q = 0; q < Q; ++q)
                        if (q == (ej >> 5)) kv[q] = kj;
                }
            }
        }
        n_chains += n_c;
        __syncwarp();
    }
    if (RESOLVE && stats && n_chains > 0) {
        n_bad = __reduce_add_sync(0xffffffffu, n_bad);
        if (lane == 0) { atomicAdd(stats + 1, n_chains); if (n_bad) atomicAdd(stats + 2, n_bad); }
    }
    const bool act = lane < k;
    float s;
    if (score_fn == 0) {
        float m = act ? my_z : -INFINITY;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        s = act ? expf(my_z - m) : 0.0f;
    } else {
        s = act ? sigmoidf_acc(my_z) : 0.0f;
    }
    float sum = s;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    if (act) {
        idx[(size_t)t * k + lane] = my_e;
        gate[(size_t)t * k + lane] = s / sum;
    }
    return true;
}

// Largest column norm of W_r, from the squared norms: every lane returns it.
__device__ __forceinline__ float route_wmax(const float* __restrict__ wsq, int E, int lane) {
    float wmax2 = 0.0f;
    for (int e = lane; e < E; e += 32) wmax2 = fmaxf(wmax2, wsq[e]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) wmax2 = fmaxf(wmax2, __shfl_xor_sync(0xffffffffu, wmax2, off));
    return sqrtf(wmax2);
}

// Screening pass: every token, one warp each, little shared memory (high occupancy).  Tokens whose approximate
// keys settle everything are finished here; the others are listed for the resolving pass.  The list's order
// depends on timing, no result does.
constexpr int SCREEN_WARPS = 4;
template <int Q>
__global__ void __launch_bounds__(SCREEN_WARPS * 32) route_screen_kernel(
    float* __restrict__ z, const float* __restrict__ z1, const float* __restrict__ bias,
    const float* __restrict__ xnorm, const float* __restrict__ wsq, int32_t* __restrict__ idx, float* __restrict__ gate,
    int32_t* __restrict__ todo, int32_t* __restrict__ n_todo, int32_t* __restrict__ pair_cnt,
    int32_t* __restrict__ pair_list, uint32_t* __restrict__ pre, int T, int d, int E, int k, int score_fn, int bias_mode) {
    extern __shared__ float sel_smem[];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int t = blockIdx.x * SCREEN_WARPS + warp;
    if (t >= T) return;
    const float wmax = route_wmax(wsq, E, lane);
    const bool done = route_token<false, Q>(t, lane, sel_smem + (size_t)warp * E, nullptr, nullptr, nullptr, z, z1, bias,
                                            nullptr, nullptr, xnorm, wmax, idx, gate, nullptr, pair_cnt, pair_list, pre, T,
                                            d, E, k, score_fn, bias_mode);
    if (!done && lane == 0) todo[atomicAdd(n_todo, 1)] = t;
}

// Chain pass: the listed (token, expert) pairs, 32 tokens of one expert per warp and one chain per lane, so that every
// element of the expert's row of W_r^T is read once for 32 chains and a step of 8 elements costs 3 shared-memory loads
// for all of them (evaluating a token's 1 to 4 chains in a warp of its own spends the same loads and steps on 4 lanes,
// and fetches 28 KB of W_r^T per chain).  Bounded by the rows of x, which come from L2 once per chain.
// d = 7168, E = 256, 16384 tokens with a skewed router (61 thousand chains, 0.88 GB of rows): 191 us, and 93 for the resolving
// pass, which took 873 by itself.  Stages of 128 elements: 252; three stages instead of five: 221.
//
// From 6 listed tokens per SM on: below that the resolving pass evaluates the chains itself.  d = 7168, E = 256, chain pass +
// resolving pass against the resolving pass alone, us: 512 tokens 59 + 14 and 72, 1023 tokens 60 + 14 and 96, 4092 tokens
// 82 + 31 and 278 (d = 2048, E = 64: 24 + 10 and 28, 24 + 10 and 31, 26 + 17 and 68).
// With few listed tokens it is an empty launch more: the two passes are dependent launches, and the lists are emptied beside the
// logit GEMM, so that the whole router costs no more than without it (T 3000, d 7168, E 512: 153 us without, 156 with plain
// launches, 149 so; T 1024, E 1024: 180, 192 and 182; T 8192, E 192: 144, 143 and 136).
constexpr int CHAIN_MIN_PER_SM = 6;
constexpr int CHAIN_WARPS = 4;
constexpr int CHAIN_STAGES = 5;
constexpr int CHAIN_K = 64;                             // elements per stage
constexpr int CHAIN_XPITCH = CHAIN_K * 2 + 16;          // bytes per row of x: eight lanes' 16-byte loads meet different banks
constexpr int CHAIN_STAGE_BYTES = 32 * CHAIN_XPITCH + CHAIN_K * 4;
constexpr int CHAIN_SMEM_BYTES = CHAIN_WARPS * CHAIN_STAGES * CHAIN_STAGE_BYTES;
constexpr int CHAIN_BLOCKS = 227 * 1024 / (CHAIN_SMEM_BYTES + 6144);     // resident per SM
__global__ void __launch_bounds__(CHAIN_WARPS * 32) route_chain_kernel(
    float* __restrict__ z, const bf16* __restrict__ x, const float* __restrict__ W_rT, const float* __restrict__ xnorm,
    const float* __restrict__ wsq, const int32_t* __restrict__ pair_cnt, const int32_t* __restrict__ pair_list,
    int32_t* __restrict__ stats, int min_listed, int T, int d, int E) {
    pdl_begin();
    extern __shared__ __align__(16) char chain_smem[];
    __shared__ int32_t first[1025];                      // first tile of 32 pairs of each expert
    __shared__ int32_t part[CHAIN_WARPS];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (pair_cnt[E] < min_listed) return;                // the resolving pass takes all of them
    const int per = (E + CHAIN_WARPS * 32 - 1) / (CHAIN_WARPS * 32), e0 = threadIdx.x * per;
    int tiles = 0, pairs = 0;
    for (int e = e0; e < min(e0 + per, E); ++e) {
        const int c = pair_cnt[e];
        tiles += (c + 31) / 32;
        pairs += c;
    }
    if (stats && blockIdx.x == 0 && pairs > 0) atomicAdd(stats + 1, pairs);
    int incl = tiles;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
    }
    if (lane == 31) part[warp] = incl;
    __syncthreads();
    int start = incl - tiles;
    for (int w = 0; w < warp; ++w) start += part[w];
    for (int e = e0; e < min(e0 + per, E); ++e) {
        first[e] = start;
        start += (pair_cnt[e] + 31) / 32;
        if (e == E - 1) first[E] = start;
    }
    __syncthreads();
    const int n_tiles = first[E];
    const float wmax = route_wmax(wsq, E, lane);
    char* stages = chain_smem + (size_t)warp * CHAIN_STAGES * CHAIN_STAGE_BYTES;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(stages);
    const int n_chunks = d / CHAIN_K;                    // d is a multiple of 64 on this path
    constexpr int PIECES = CHAIN_K / 8, RSTEP = 32 / PIECES;         // 16-byte pieces of a row; rows per copy of the warp
    const int piece = lane % PIECES;                     // this lane's piece of the rows lane / PIECES + RSTEP u
    int n_bad = 0;
    for (int tile = blockIdx.x * CHAIN_WARPS + warp; tile < n_tiles; tile += gridDim.x * CHAIN_WARPS) {
        int lo = 0, hi = E;                              // the last expert whose first tile is at or before this one
        while (hi - lo > 1) {
            const int mid = (lo + hi) / 2;
            if (first[mid] <= tile) lo = mid; else hi = mid;
        }
        const int e = lo, n_e = pair_cnt[e], i = (tile - first[e]) * 32 + lane;
        const int rows = n_e - (i - lane);               // of this tile; the lanes past them repeat the last one's logit
        const int t = pair_list[(size_t)e * T + min(i, n_e - 1)];
        const float* wrow = W_rT + (size_t)e * d;
        const bf16* xrow[PIECES];
#pragma unroll
        for (int u = 0; u < PIECES; ++u)
            xrow[u] = x + (size_t)__shfl_sync(0xffffffffu, t, lane / PIECES + RSTEP * u) * d + piece * 8;
        auto fetch = [&](int c) {
            if (c < n_chunks) {
                const int i0 = c * CHAIN_K;
                const uint32_t st = sbase + (c % CHAIN_STAGES) * CHAIN_STAGE_BYTES;
#pragma unroll
                for (int u = 0; u < PIECES; ++u)
                    if (lane / PIECES + RSTEP * u < rows)
                        cp_async16(st + (lane / PIECES + RSTEP * u) * CHAIN_XPITCH + piece * 16, xrow[u] + i0, true);
                if (lane < CHAIN_K / 4) cp_async16(st + 32 * CHAIN_XPITCH + lane * 16, wrow + i0 + lane * 4, true);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
#pragma unroll
        for (int c = 0; c < CHAIN_STAGES - 1; ++c) fetch(c);
        float acc = 0.0f;
        for (int c = 0; c < n_chunks; ++c) {
            asm volatile("cp.async.wait_group %0;" ::"n"(CHAIN_STAGES - 2) : "memory");
            __syncwarp();
            fetch(c + CHAIN_STAGES - 1);                 // into the stage that was read last time round
            const char* st = stages + (c % CHAIN_STAGES) * CHAIN_STAGE_BYTES;
            const uint4* xs = reinterpret_cast<const uint4*>(st + min(lane, rows - 1) * CHAIN_XPITCH);
            const float4* ws = reinterpret_cast<const float4*>(st + 32 * CHAIN_XPITCH);
            // the contract's chain: one fused multiply-add per i, i ascending
            auto step = [&](int j) {
                const uint4 xv = xs[j];
                const float4 w0 = ws[2 * j], w1 = ws[2 * j + 1];
                acc = __fmaf_rn(bf16_lo(xv.x), w0.x, acc);
                acc = __fmaf_rn(bf16_hi(xv.x), w0.y, acc);
                acc = __fmaf_rn(bf16_lo(xv.y), w0.z, acc);
                acc = __fmaf_rn(bf16_hi(xv.y), w0.w, acc);
                acc = __fmaf_rn(bf16_lo(xv.z), w1.x, acc);
                acc = __fmaf_rn(bf16_hi(xv.z), w1.y, acc);
                acc = __fmaf_rn(bf16_lo(xv.w), w1.z, acc);
                acc = __fmaf_rn(bf16_hi(xv.w), w1.w, acc);
            };
#pragma unroll
            for (int j = 0; j < CHAIN_K / 8; ++j) step(j);
        }
        __syncwarp();                                    // the next tile's fetches overwrite the stages
        if (i < n_e) {
            float* zp = z + (size_t)t * E + e;
            // the model of the error is checked as we go
            if (fabsf(*zp - acc) > 0.5f * ROUTE_EPS_C * (5.9604645e-8f * xnorm[t] * wmax)) ++n_bad;
            *zp = acc;
        }
    }
    n_bad = __reduce_add_sync(0xffffffffu, n_bad);
    if (stats && lane == 0 && n_bad) atomicAdd(stats + 2, n_bad);
}
inline bool route_chain_init() {
    return cudaFuncSetAttribute(route_chain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, CHAIN_SMEM_BYTES) == cudaSuccess;
}

// Resolving pass: the listed tokens, one warp each, with the staging memory of the chains.
template <int Q>
__global__ void __launch_bounds__(SELF_WARPS * 32) route_resolve_kernel(
    float* __restrict__ z, const float* __restrict__ bias, const bf16* __restrict__ x, const float* __restrict__ W_rT,
    const float* __restrict__ xnorm, const float* __restrict__ wsq, int32_t* __restrict__ idx,
    float* __restrict__ gate, const int32_t* __restrict__ todo, const int32_t* __restrict__ n_todo,
    int32_t* __restrict__ stats, uint32_t* __restrict__ pre, int min_listed, int d, int E, int k, int score_fn, int bias_mode) {
    pdl_begin();
    extern __shared__ float sel_smem[];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int n = *n_todo;
    if (stats && n > 0 && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(stats, n);   // statistics only: no result depends on them
    if ((int)blockIdx.x * SELF_WARPS >= n) return;
    float* zg = sel_smem + (size_t)warp * (2 * E + SELF_SMEM_FLOATS);
    int32_t* clist = reinterpret_cast<int32_t*>(zg + E);   // experts whose exact logit is needed
    float* xs = zg + 2 * E;                                 // a chunk of the token's row, fp32
    float* ws = xs + SELF_XCHUNK;                           // the same chunk of up to SELF_CAND rows of W_r^T
    const float wmax = route_wmax(wsq, E, lane);
    for (int i = blockIdx.x * SELF_WARPS + warp; i < n; i += gridDim.x * SELF_WARPS) {
        route_token<true, Q>(todo[i], lane, zg, clist, xs, ws, z, nullptr, bias, x, W_rT, xnorm, wmax, idx, gate, stats,
                             nullptr, nullptr, n < min_listed ? nullptr : pre, 0, d, E, k, score_fn, bias_mode);
        __syncwarp();
    }
}

// Buffers of the selection that its passes share.
struct RouteLists {
    int32_t* todo;           // [T] listed tokens
    int32_t* pair_cnt;       // [E] listed tokens per expert, then the number of listed tokens: zeroed before the screening
    int32_t* pair_list;      // [E][T]
    uint32_t* pre;           // [T][32]
    int32_t* stats;
    int min_listed;          // the chain pass runs from this number of listed tokens on
};

// The screening and the resolving pass for the smallest supported Q >= ceil(E / 32).
template <int Q>
inline void route_select_fast_q(float* z, const float* z1, const float* bias, const bf16* x, const float* W_rT, const float* xnorm,
                                const float* wsq, int32_t* idx, float* gate, const RouteLists& l, int T, int d, int E, int k,
                                int score_fn, int bias_mode, int pass, int resolve_blocks, cudaStream_t st) {
    if (pass == 0) {
        route_screen_kernel<Q><<<ceil_div(T, SCREEN_WARPS), SCREEN_WARPS * 32, (size_t)SCREEN_WARPS * E * sizeof(float), st>>>(
            z, z1, bias, xnorm, wsq, idx, gate, l.todo, l.pair_cnt + E, l.pair_cnt, l.pair_list, l.pre, T, d, E, k, score_fn,
            bias_mode);
    } else {
        const size_t smem = (size_t)SELF_WARPS * (2 * E + SELF_SMEM_FLOATS) * sizeof(float);
        pdl_launch(route_resolve_kernel<Q>, resolve_blocks, SELF_WARPS * 32, smem, st, z, bias, x, W_rT, xnorm, wsq, idx, gate, l.todo,
                   l.pair_cnt + E, l.stats, l.pre, l.min_listed, d, E, k, score_fn, bias_mode);
    }
}
// Blocks of the resolving pass that are resident at once: its grid.  Every warp then walks its share of the list;
// a larger grid would run in waves of whole walks.
template <int Q>
inline int route_resolve_resident_q(int E, int sm_count) {
    int nb = 0;
    const size_t smem = (size_t)SELF_WARPS * (2 * E + SELF_SMEM_FLOATS) * sizeof(float);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, route_resolve_kernel<Q>, SELF_WARPS * 32, smem) != cudaSuccess || nb < 1)
        nb = 1;
    return nb * sm_count;
}
inline int route_resolve_resident(int E, int sm_count) {
    const int q = ceil_div(E, 32);
    if (q <= 2) return route_resolve_resident_q<2>(E, sm_count);
    if (q <= 4) return route_resolve_resident_q<4>(E, sm_count);
    if (q <= 8) return route_resolve_resident_q<8>(E, sm_count);
    if (q <= 12) return route_resolve_resident_q<12>(E, sm_count);
    if (q <= 16) return route_resolve_resident_q<16>(E, sm_count);
    return route_resolve_resident_q<32>(E, sm_count);
}
inline void route_select_fast(float* z, const float* z1, const float* bias, const bf16* x, const float* W_rT, const float* xnorm,
                              const float* wsq, int32_t* idx, float* gate, const RouteLists& l, int T, int d, int E, int k,
                              int score_fn, int bias_mode, int pass, int resolve_blocks, cudaStream_t st) {
    const int q = ceil_div(E, 32);
#define MOP_ROUTE_Q(QQ)                                                                                                 \
    route_select_fast_q<QQ>(z, z1, bias, x, W_rT, xnorm, wsq, idx, gate, l, T, d, E, k, score_fn, bias_mode, pass,             \
                            resolve_blocks, st)
    if (q <= 2) MOP_ROUTE_Q(2);
    else if (q <= 4) MOP_ROUTE_Q(4);
    else if (q <= 8) MOP_ROUTE_Q(8);
    else if (q <= 12) MOP_ROUTE_Q(12);
    else if (q <= 16) MOP_ROUTE_Q(16);
    else MOP_ROUTE_Q(32);
#undef MOP_ROUTE_Q
}

// ---------------------------------------------------------------------------------------------
// Router backward (selection held fixed).  With g_j = s_j / sum_l s_l over a token's k selected
// experts (s = softmax over all E, whose common denominator cancels, or s = sigmoid):
//   softmax:  dz_j = g_j (dgate_j - sum_l g_l dgate_l)
//   sigmoid:  dz_j = (dgate_j - sum_l g_l dgate_l) / S * s_j (1 - s_j),   S = sum_l s_l
// dz is zero at every expert that was not selected.  Then dW_r = x^T dz, dX += dz W_r^T and, for a
// bias added before the score, dbias = column sums of dz.
// ---------------------------------------------------------------------------------------------

// W_r^T [E,d] from W_r [d,E], a tile of 32 x 32 per block through shared memory: gives the dX kernel contiguous rows.
__device__ __forceinline__ void transpose_tile(const float* __restrict__ in, float* __restrict__ out, int rows, int cols, int block) {
    __shared__ float tile[32][33];
    const int across = (cols + 31) / 32;
    const int c0 = (block % across) * 32, r0 = (block / across) * 32;
    const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
    for (int r = ty; r < 32; r += 8)
        if (r0 + r < rows && c0 + tx < cols) tile[r][tx] = in[(size_t)(r0 + r) * cols + c0 + tx];
    __syncthreads();
    for (int c = ty; c < 32; c += 8)
        if (c0 + c < cols && r0 + tx < rows) out[(size_t)(c0 + c) * rows + r0 + tx] = tile[tx][c];
}

// One warp per token: lane j < k owns the j-th selected expert.  Writes dz per assignment and, in
// expert-contiguous row order (row = perm_row[assignment]), the copy that the dW_r kernel reads.
// The blocks behind the first dz_blocks transpose W_r, which the next kernel reads as well: a launch less.
__global__ void __launch_bounds__(256) route_bwd_dz_kernel(const float* __restrict__ logits,
                                                           const float* __restrict__ bias,
                                                           const int32_t* __restrict__ idx,
                                                           const float* __restrict__ gate,
                                                           const float* __restrict__ dgate,
                                                           const int32_t* __restrict__ perm_row,
                                                           float* __restrict__ dz_sel, float* __restrict__ dz_row,
                                                           int T, int E, int k, int score_fn, int bias_mode, int dz_blocks,
                                                           const float* __restrict__ W_r, float* __restrict__ W_rT, int d) {
    pdl_begin();
    if ((int)blockIdx.x >= dz_blocks) { transpose_tile(W_r, W_rT, d, E, blockIdx.x - dz_blocks); return; }
    const int lane = threadIdx.x % 32;
    const int t = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    if (t >= T) return;
    const bool act = lane < k;
    const size_t a = (size_t)t * k + lane;
    float g = 0.0f, dg = 0.0f, zz = 0.0f;
    if (act) {
        const int e = idx[a];
        g = gate[a];
        dg = dgate[a];
        zz = logits[(size_t)t * E + e];
        if (bias_mode == 2) zz += bias[e];
    }
    float dot = g * dg;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
    float dz;
    if (score_fn == 0) {
        dz = g * (dg - dot);
    } else {
        const float s = act ? sigmoidf_acc(zz) : 0.0f;
        float S = s;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) S += __shfl_xor_sync(0xffffffffu, S, off);
        dz = (dg - dot) / S * s * (1.0f - s);
    }
    if (act) {
        dz_sel[a] = dz;
        const int32_t p = perm_row[a];
        if (p >= 0) dz_row[p] = dz;
    }
}

// dX[t,:] += dz[t,:] W_r^T = sum_j dz[t,j] * W_r^T[e_j,:]: a block takes 256 columns (of blocks `block`, `block` + segments, ..) and its
// warps a token each, twice four columns a lane (neighbouring lanes read neighbouring 16 bytes), with the k rows of W_r^T four at a
// time; dX is read, updated in fp32 and rounded back to bf16.  d is a multiple of 8.
// Bound by what the rows of W_r^T cost: k fp32 columns for each bf16 one of dX.  With the columns fixed, E KiB of them pass through an
// SM's L1 again and again, instead of all E rows through L2.
__device__ __forceinline__ void route_bwd_dx(const float* __restrict__ W_rT, const int32_t* __restrict__ idx,
                                             const float* __restrict__ dz_sel, bf16* __restrict__ dX, int T, int d, int k, int block,
                                             int blocks) {
    const int lane = threadIdx.x % 32, warps = blockDim.x / 32, segs = (d + 255) / 256;
    const int i = (block % segs) * 256 + lane * 4;
    const bool in[2] = {i < d, i + 128 < d};
    const long long t0 = (long long)(block / segs) * warps + threadIdx.x / 32, step = (long long)(blocks / segs) * warps;
    int e_next;
    float dz_next;
    uint2 v_next[2];
    auto fetch = [&](long long t) {
        e_next = 0; dz_next = 0.0f;
        v_next[0] = v_next[1] = make_uint2(0, 0);
        if (t >= T) return;
        if (lane < k) { e_next = idx[(size_t)t * k + lane]; dz_next = dz_sel[(size_t)t * k + lane]; }
        const bf16* px = dX + (size_t)t * d + i;
        if (in[0]) v_next[0] = *reinterpret_cast<const uint2*>(px);
        if (in[1]) v_next[1] = *reinterpret_cast<const uint2*>(px + 128);
    };
    fetch(t0);
    for (long long t = t0; t < T; t += step) {
        const int e = e_next;
        const float dz = dz_next;
        uint2 v[2] = {v_next[0], v_next[1]};
        fetch(t + step);
        bf16* px = dX + (size_t)t * d + i;
        float a[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < 4; ++q) a[h][q] = 0.0f;
#pragma unroll 4
        for (int j = 0; j < k; ++j) {
            const float* w = W_rT + (size_t)__shfl_sync(0xffffffffu, e, j) * d + i;
            const float s = __shfl_sync(0xffffffffu, dz, j);
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (in[h]) {
                    const float4 u = *reinterpret_cast<const float4*>(w + 128 * h);
                    a[h][0] = fmaf(s, u.x, a[h][0]); a[h][1] = fmaf(s, u.y, a[h][1]);
                    a[h][2] = fmaf(s, u.z, a[h][2]); a[h][3] = fmaf(s, u.w, a[h][3]);
                }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (in[h]) {
                v[h].x = pack_bf16x2(bf16_lo(v[h].x) + a[h][0], bf16_hi(v[h].x) + a[h][1]);
                v[h].y = pack_bf16x2(bf16_lo(v[h].y) + a[h][2], bf16_hi(v[h].y) + a[h][3]);
                *reinterpret_cast<uint2*>(px + 128 * h) = v[h];
            }
    }
}

// dW_r[i,e] = sum over the rows p of expert e of Xp[p,i] * dz_row[p].  Block (256 columns i, e): warp w adds the rows w, w + W,
// ... of the expert (eight columns per lane, four rows in flight), the W partial sums are added in order through shared memory.
// Bound by reading Xp once.  With one thread per eight columns walking all rows two at a time (128 threads per 1024 columns)
// there were too few bytes in flight: 141 us at T = 4096, d = 2048, E = 64, k = 6 and 292 us at T = 4096, d = 1024, E = 32,
// k = 8; now 28 and 21.  Fixed order, no atomics.
// The blocks behind these, if any, add the router's share to dX: neither waits for the other.
__global__ void __launch_bounds__(1024) route_bwd_dwr_dx_kernel(const bf16* __restrict__ Xp, const float* __restrict__ dz_row,
                                                                const int32_t* __restrict__ offsets, float* __restrict__ dW_r,
                                                                float* __restrict__ dbias, int d, int E, const float* __restrict__ W_rT,
                                                                const int32_t* __restrict__ idx, const float* __restrict__ dz_sel,
                                                                bf16* __restrict__ dX, int T, int k) {
    pdl_begin();
    extern __shared__ float dwr_smem[];                              // [W][256]
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32, W = blockDim.x / 32;
    const int across = (d + 255) / 256, dwr_blocks = across * E;
    if ((int)blockIdx.x >= dwr_blocks) {
        route_bwd_dx(W_rT, idx, dz_sel, dX, T, d, k, (int)blockIdx.x - dwr_blocks, (int)gridDim.x - dwr_blocks);
        return;
    }
    const int e = blockIdx.x / across, c0 = (blockIdx.x - e * across) * 256, i = c0 + lane * 8;
    const int p0 = offsets[e], p1 = offsets[e + 1];
    float a[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) a[q] = 0.0f;
    if (i < d) {
        for (int p = p0 + warp; p < p1; p += 4 * W) {
            uint4 v[4];
            float w[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int pr = p + r * W;
                w[r] = pr < p1 ? dz_row[pr] : 0.0f;
                v[r] = pr < p1 ? __ldcs(reinterpret_cast<const uint4*>(Xp + (size_t)pr * d + i)) : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                a[0] = fmaf(bf16_lo(v[r].x), w[r], a[0]); a[1] = fmaf(bf16_hi(v[r].x), w[r], a[1]);
                a[2] = fmaf(bf16_lo(v[r].y), w[r], a[2]); a[3] = fmaf(bf16_hi(v[r].y), w[r], a[3]);
                a[4] = fmaf(bf16_lo(v[r].z), w[r], a[4]); a[5] = fmaf(bf16_hi(v[r].z), w[r], a[5]);
                a[6] = fmaf(bf16_lo(v[r].w), w[r], a[6]); a[7] = fmaf(bf16_hi(v[r].w), w[r], a[7]);
            }
        }
    }
    float* mine = dwr_smem + warp * 256 + lane * 8;
    *reinterpret_cast<float4*>(mine) = make_float4(a[0], a[1], a[2], a[3]);
    *reinterpret_cast<float4*>(mine + 4) = make_float4(a[4], a[5], a[6], a[7]);
    __syncthreads();
    if (threadIdx.x < 256 && c0 + (int)threadIdx.x < d) {
        float s = 0.0f;
        for (int w = 0; w < W; ++w) s += dwr_smem[w * 256 + threadIdx.x];
        dW_r[(size_t)(c0 + threadIdx.x) * E + e] = s;
    }
    if (dbias && c0 == 0 && warp == 0) {
        float sb = 0.0f;
        for (int p = p0 + lane; p < p1; p += 32) sb += dz_row[p];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) sb += __shfl_xor_sync(0xffffffffu, sb, off);
        if (lane == 0) dbias[e] = sb;
    }
}
// Warps per block: enough to keep 16 warps and more on every SM (8 warps leave the other blocks room where there are many).
inline int dwr_warps(long long blocks, int sm_count) { return blocks >= 4ll * sm_count ? 8 : blocks >= 2ll * sm_count ? 16 : 32; }

}  // namespace mop
