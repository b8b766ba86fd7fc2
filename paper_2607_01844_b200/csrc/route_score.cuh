// Exact fp32 scoring of the router (Section 2.1 of the paper).
//
// z[t,e] = sum_i x[t,i] * W_r[i,e] as ONE chain of fused multiply-adds per (t,e), i ascending, each step rounded once to fp32.
// The chain order is part of the routing contract (it makes top-k indices reproducible bit for bit), so there is no split over i
// and no tensor core here; parallelism comes from the T*E independent chains.  Each thread owns RT tokens x RE experts; with
// several experts it advances two chains (experts e, e + 1) per instruction with the packed fma.rn.f32x2 of sm_100 (two
// independent IEEE fused multiply-adds: the rounding of each chain is unchanged).
//
// What bounds it: where there are many chains, the packed multiply-adds (2.8 cycles each with three different operands); where there
// are few, the latency of one (4 cycles) and what a warp issues between two of a chain.  A load from shared memory holds its warp up
// for its whole latency once the next load's results are waited for together with it, and costs 4 cycles of the SM per 512 bytes
// returned.  So the warps that multiply do nothing else: as many warps again bring the operands in by cp.async, stages ahead, the
// two kinds meet at barriers only, registers are filled again one by one as the steps go along, and x stays bf16 until a step
// before its use.
// A warp covers LT RT tokens x (32 / LT) RE experts, a block CW times the tokens.
#pragma once
#include <type_traits>

#include "gemm_tc.cuh"

namespace mop {

__device__ __forceinline__ void unpack_f32x2(unsigned long long v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async8(uint32_t dst, const void* src, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(ok ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(ok ? 4 : 0) : "memory");
}

template <int RT, int RE, int LT, int CW, bool TWO>
struct ScoreShape {
    static constexpr bool PAIRS = RE > 1;                       // chains in pairs of experts; else plain chains, and W transposed
    static constexpr int LE = 32 / LT;
    static constexpr int TT = CW * LT * RT, TE = LE * RE;
    static constexpr int TK = 64;                               // steps per stage
    // TWO: two blocks of 64 x 64 on an SM, so that one's multiplications fill the other's waits (registers: six warps of 168; shared
    // memory: four slots of 25 KiB).  A step of theirs takes long enough to load one stage ahead, by half as many warps.
    static constexpr int LOADERS = TWO ? 16 * CW : 32 * CW, THREADS = 32 * CW + LOADERS;   // warps 0 .. CW - 1 multiply, the others load
    static constexpr int AHEAD = TWO ? 1 : PAIRS ? 2 : 8;       // stages in flight from global memory
    static constexpr int READY = 2;                             // stages handed to the multiplying warps
    static constexpr int SLOTS = AHEAD + 1 + READY;             // (filled AHEAD stages early; READY back may still be read; one just released)
    static constexpr int X_PITCH = TK * 2 + 16;                 // neighbouring tokens 16 bytes apart in the banks
    static constexpr int W_PITCH = PAIRS ? TE * 4 : TK * 4 + 16;   // a step's experts, or (transposed) an expert's steps
    static constexpr int X_BYTES = TT * X_PITCH;
    static constexpr int W_BYTES = (PAIRS ? TK : TE) * W_PITCH;
    static constexpr int BAR_BYTES = 128;
    static constexpr int SMEM = BAR_BYTES + SLOTS * (W_BYTES + X_BYTES);
};

__device__ __forceinline__ void lds_b128(uint32_t addr, uint32_t (&v)[4]) {
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr) : "memory");
}

template <int RT, int RE, int LT, int CW, bool TWO>
__global__ void __launch_bounds__(ScoreShape<RT, RE, LT, CW, TWO>::THREADS, TWO ? 2 : 0)
route_score_kernel(const bf16* __restrict__ x, const float* __restrict__ W_r, float* __restrict__ z, int T, int d, int E,
                   int32_t* __restrict__ status) {
    using Sh = ScoreShape<RT, RE, LT, CW, TWO>;
    constexpr bool PAIRS = Sh::PAIRS;
    constexpr int LE = Sh::LE, TT = Sh::TT, TE = Sh::TE, TK = Sh::TK, AHEAD = Sh::AHEAD, READY = Sh::READY, SLOTS = Sh::SLOTS;
    constexpr int LOADERS = Sh::LOADERS;
    constexpr int VE = RE < 4 ? RE : 4;                             // adjacent experts of a thread; further groups LE * VE apart
    static_assert(RE == 1 || RE == 2 || RE % 4 == 0, "experts of a thread");
    static_assert(Sh::W_BYTES % 16 == 0 && Sh::X_BYTES % 16 == 0 && 16 * READY + 4 <= Sh::BAR_BYTES, "16-byte copies, barriers");
    extern __shared__ __align__(16) uint8_t sc_smem[];
    const uint32_t base = smem_u32(sc_smem);
    const uint32_t w_base = base + Sh::BAR_BYTES, x_base = w_base + SLOTS * Sh::W_BYTES;
    auto full_bar = [&](int s) { return base + 16u * (s % READY); };
    auto empty_bar = [&](int s) { return base + 16u * (s % READY) + 8u; };
    auto round_of = [&](int s) { return (uint32_t)(s / READY) & 1u; };
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sc_smem + 16 * READY);
    const int tid = threadIdx.x, warp = warp_index(), lane = tid % 32;
    if (tid == 0) {
        for (int s = 0; s < READY; ++s) { mbar_init(full_bar(s), LOADERS / 32); mbar_init(empty_bar(s), CW); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    pdl_begin();
    const int t0 = blockIdx.x * TT, e0 = blockIdx.y * TE;
    const int stages = (d + TK - 1) / TK;

    if (warp >= CW) {
        // ===================================================================== loading warps
        // A thread's copies of a stage lie at fixed distances, so that a stage costs about an addition per copy.  Tokens past T,
        // experts past E and steps past d are zeros (copies of no bytes: many lanes that read one address instead take turns).
        const int lt = tid - 32 * CW;
        constexpr int XN = TT * (TK / 8) / LOADERS, XR = LOADERS / (TK / 8);      // 16 bytes = 8 steps of one token
        const int xt = lt / (TK / 8), xc = (lt % (TK / 8)) * 8;
        const bf16* xs = x + (size_t)(t0 + xt) * d + xc;
        const size_t x_step = (size_t)XR * d;
        const uint32_t xd = x_base + xt * Sh::X_PITCH + xc * 2;
        auto load = [&](auto width) {
            constexpr int V = decltype(width)::value;                             // floats per copy of W
            constexpr int COLS = TE / V, WN = TK * COLS / LOADERS, WR = LOADERS / COLS;
            static_assert(LOADERS % COLS == 0, "a thread keeps its columns");
            const int wi = lt / COLS, we = (lt % COLS) * V;
            const float* wsrc = W_r + (size_t)wi * E + e0 + we;
            const bool e_ok = e0 + we < E;                                        // (V divides E)
            const uint32_t wd = w_base + (PAIRS ? wi * Sh::W_PITCH + we * 4 : we * Sh::W_PITCH + wi * 4);
            const size_t w_step = (size_t)WR * E, w_stage = (size_t)TK * E;
            int slot = 0;
            auto issue = [&](int s) {
                if (s < stages) {
                    const uint32_t xb = xd + slot * Sh::X_BYTES, wb = wd + slot * Sh::W_BYTES;
                    const bool whole = (s + 1) * TK <= d;
                    const bool xok = whole || s * TK + xc < d;
#pragma unroll
                    for (int p = 0; p < XN; ++p) {
                        const bool ok = xok && t0 + xt + p * XR < T;
                        cp_async16(xb + p * XR * Sh::X_PITCH, ok ? xs + p * x_step : x, ok);
                    }
                    const float* w = wsrc;
#pragma unroll
                    for (int p = 0; p < WN; ++p) {
                        const uint32_t dst = wb + p * WR * (PAIRS ? Sh::W_PITCH : 4);
                        const bool ok = e_ok && (whole || s * TK + wi + p * WR < d);
                        const float* src = ok ? w : W_r;
                        if constexpr (V == 4) cp_async16(dst, src, ok);
                        else if constexpr (V == 2) cp_async8(dst, src, ok);
                        else cp_async4(dst, src, ok);
                        w += w_step;
                    }
                    xs += TK;
                    wsrc += w_stage;
                    slot = slot + 1 == SLOTS ? 0 : slot + 1;
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
#pragma unroll 1
            for (int s = 0; s < AHEAD; ++s) issue(s);
#pragma unroll 1
            for (int s = 0; s < stages; ++s) {
                issue(s + AHEAD);
                asm volatile("cp.async.wait_group %0;" ::"n"(AHEAD) : "memory");  // this thread's part of stage s is there
                if (!mbar_wait_all(empty_bar(s), round_of(s) ^ 1u, abort_flag, status, STATUS_WAIT_EMPTY)) break;
                __syncwarp();
                if (lane == 0) mbar_arrive(full_bar(s));
            }
        };
        if (PAIRS && E % 4 == 0) load(std::integral_constant<int, PAIRS ? 4 : 1>{});
        else if (PAIRS && E % 2 == 0) load(std::integral_constant<int, PAIRS ? 2 : 1>{});
        else load(std::integral_constant<int, 1>{});
        asm volatile("cp.async.wait_all;" ::: "memory");
        return;
    }

    // ===================================================================== multiplying warps
    // Tokens of a thread: tt, tt + LT, ..
    const int tt = warp * LT * RT + (PAIRS ? lane % LT : lane / LE);
    const int te = PAIRS ? (lane / LT) * VE : lane % LE;
    constexpr int G = PAIRS ? 8 : 16;                               // steps whose operands are in registers
    constexpr int NG = TK / G, NP = PAIRS ? RE / 2 : 1;
    static_assert(NG % 2 == 0, "the register buffers of x alternate");
    unsigned long long acc[RT][NP];
    float acc1[RT];
#pragma unroll
    for (int a = 0; a < RT; ++a) {
        acc1[a] = 0.0f;
#pragma unroll
        for (int b = 0; b < NP; ++b) acc[a][b] = 0ull;
    }
    // Registers of W are filled again, with the step G further on, as soon as a step (plain chains: four steps) is done with them;
    // x comes a group ahead in the other of two buffers.  (All loads of a group at its start: one latency per group, 60 to 90 cycles.)
    uint32_t xv[2][RT][G / 8][4], wt[G / 4][4];
    unsigned long long wp[G][NP];
    const uint32_t x_off = tt * Sh::X_PITCH, w_off = PAIRS ? te * 4 : te * Sh::W_PITCH;
    auto load_x = [&](int buf, uint32_t xa) {
#pragma unroll
        for (int a = 0; a < RT; ++a)
#pragma unroll
            for (int q = 0; q < G / 8; ++q) lds_b128(xa + a * LT * Sh::X_PITCH + q * 16, xv[buf][a][q]);
    };
    auto load_w = [&](int j, uint32_t wa) {
        if constexpr (!PAIRS) {
            if (j % 4 == 3) lds_b128(wa + (j / 4) * 16, wt[j / 4]);
        } else if constexpr (VE == 2) {
            asm volatile("ld.shared.b64 %0, [%1];" : "=l"(wp[j][0]) : "r"(wa + j * Sh::W_PITCH) : "memory");
        } else {
#pragma unroll
            for (int b = 0; b < RE / 4; ++b)
                asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(wp[j][2 * b]), "=l"(wp[j][2 * b + 1])
                             : "r"(wa + j * Sh::W_PITCH + b * LE * VE * 4) : "memory");
        }
    };
    // x of a step as fp32 (pairs: twice)
    unsigned long long xq[2][RT];
    float xf[2][RT];
    auto convert = [&](int buf, int j, int to) {
#pragma unroll
        for (int a = 0; a < RT; ++a) {
            const uint32_t v = xv[buf][a][j >> 3][(j >> 1) & 3];
            uint32_t f, h;      // (a byte permutation: shift, mask and move run at half its rate)
            if (j & 1) asm volatile("prmt.b32 %0, %1, 0, 0x3244;" : "=r"(f) : "r"(v));
            else asm volatile("prmt.b32 %0, %1, 0, 0x1044;" : "=r"(f) : "r"(v));
            if constexpr (PAIRS) {
                if (j & 1) asm volatile("prmt.b32 %0, %1, 0, 0x3244;" : "=r"(h) : "r"(v));
                else asm volatile("prmt.b32 %0, %1, 0, 0x1044;" : "=r"(h) : "r"(v));
                asm volatile("mov.b64 %0, {%1, %2};" : "=l"(xq[to][a]) : "r"(f), "r"(h));
            } else xf[to][a] = __uint_as_float(f);
        }
    };
    // Steps past d (d not a multiple of a stage) multiply zeros: fma(0, 0, acc) = acc, exact.
    bool alive = mbar_wait_all(full_bar(0), round_of(0), abort_flag, status, STATUS_WAIT_FULL);
    uint32_t xs = x_base + x_off, ws = w_base + w_off;              // this stage's slot
    if (alive) {
        load_x(0, xs);
#pragma unroll
        for (int j = 0; j < G; ++j) load_w(j, ws);
        convert(0, 0, 0);
    }
    int slot = 0;
#pragma unroll 1
    for (int s = 0; s < stages && alive; ++s) {
        slot = slot + 1 == SLOTS ? 0 : slot + 1;
        // the last group of the last stage loads its own stage's first one again (into registers that nobody reads)
        const bool more = s + 1 < stages;
        const uint32_t xn = more ? x_base + slot * Sh::X_BYTES + x_off : xs, wn = more ? w_base + slot * Sh::W_BYTES + w_off : ws;
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            const int cur = g & 1;
            if (g + 1 == NG && more) alive = mbar_wait_all(full_bar(s + 1), round_of(s + 1), abort_flag, status, STATUS_WAIT_FULL);
            const uint32_t xa = g + 1 < NG ? xs + (g + 1) * G * 2 : xn;
            const uint32_t wa = g + 1 < NG ? ws + (g + 1) * (PAIRS ? G * Sh::W_PITCH : G * 4) : wn;
            load_x(cur ^ 1, xa);
#pragma unroll
            for (int j = 0; j < G; ++j) {
                if (j + 1 < G) convert(cur, j + 1, (j + 1) & 1);
                else convert(cur ^ 1, 0, 0);
#pragma unroll
                for (int a = 0; a < RT; ++a) {
                    if constexpr (!PAIRS)
                        asm volatile("fma.rn.f32 %0, %1, %2, %0;" : "+f"(acc1[a]) : "f"(xf[j & 1][a]), "f"(__uint_as_float(wt[j >> 2][j & 3])));
                    else
#pragma unroll
                        for (int b = 0; b < NP; ++b)
                            asm volatile("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[a][b]) : "l"(xq[j & 1][a]), "l"(wp[j][b]));
                }
                load_w(j, wa);
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty_bar(s));
        xs = xn; ws = wn;
    }
#pragma unroll
    for (int a = 0; a < RT; ++a) {
        const int t = t0 + tt + LT * a;
        if (t >= T) continue;
        if constexpr (!PAIRS) {
            if (e0 + te < E) z[(size_t)t * E + e0 + te] = acc1[a];
        } else {
#pragma unroll
            for (int b = 0; b < NP; ++b) {
                float v[2];
                unpack_f32x2(acc[a][b], v[0], v[1]);
                const int e = e0 + te + (2 * b / VE) * LE * VE + 2 * b % VE;
                float* dst = z + (size_t)t * E + e;
                if (E % 2 == 0 && e + 1 < E) {
                    *reinterpret_cast<float2*>(dst) = make_float2(v[0], v[1]);
                } else {
                    if (e < E) dst[0] = v[0];
                    if (e + 1 < E) dst[1] = v[1];
                }
            }
        }
    }
}

template <int RT, int RE, int LT, int CW, bool TWO>
inline bool route_score_attr() {
    return cudaFuncSetAttribute(route_score_kernel<RT, RE, LT, CW, TWO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                ScoreShape<RT, RE, LT, CW, TWO>::SMEM) == cudaSuccess;
}
inline bool route_score_init() {
    return route_score_attr<2, 1, 4, 2, false>() && route_score_attr<2, 1, 4, 4, false>() && route_score_attr<2, 4, 4, 4, false>() &&
           route_score_attr<4, 4, 4, 4, false>() && route_score_attr<4, 8, 4, 4, false>() && route_score_attr<4, 8, 4, 4, true>();
}
template <int RT, int RE, int LT, int CW, bool TWO>
inline void launch_route_score(const bf16* x, const float* W_r, float* z, int T, int d, int E, int32_t* status, cudaStream_t st) {
    using Sh = ScoreShape<RT, RE, LT, CW, TWO>;
    dim3 grid(ceil_div(T, Sh::TT), ceil_div(E, Sh::TE));
    pdl_launch(route_score_kernel<RT, RE, LT, CW, TWO>, grid, Sh::THREADS, Sh::SMEM, st, x, W_r, z, T, d, E, status);
}
// Shape choice: the least estimated cycles per step on the fullest SM, first + more * (blocks on it - 1), as measured at
// d = 7168 (one block alone on an SM; each further one).  us, with every thread loading and multiplying by turns and now:
// T 64, d 7168, E 256 (16 x 8) 44 and 33; T 1537, d 1000, E 20 (32 x 8) 10.8 and 8.4; T 512, d 7168, E 256 (32 x 32) 101 and 66;
// T 4096, d 2048, E 64 (64 x 32) 39 and 31, E 61 49 and 33; T 2048, d 7168, E 96 (64 x 32) 130 and 102; d 7168, E 256 (64 x 64)
// T 2368 208 and 191, T 16576 1225 and 1189, E 255 1552 and 1374.  The packed multiply-adds alone, three different operands each, take
// 2.8 cycles a warp and scheduler: 53 TFLOP/s.
// 64 x 64 as two blocks on an SM, or as one with twice the loading warps where E is odd and W_r comes in by 4 bytes: d 7168, one
// block's worth per SM (T 2368) E 256 191 and 193 us, E 255 247 and 203; seven (T 16576) E 256 1189 and 1292, E 252 1190 and 1337,
// E 255 1355 and 1374.
inline void route_score(const bf16* x, const float* W_r, float* z, int T, int d, int E, int sm_count, int32_t* status,
                        cudaStream_t st) {
    const bool two = E % 2 == 0;
    const struct { int tt, te; float first, more; } shape[5] = {
        {16, 8, 8.8f, 4.5f}, {32, 8, 11.f, 7.6f}, {32, 32, 16.9f, 13.2f}, {64, 32, 27.8f, 24.8f}, {64, 64, 47.6f, two ? 43.5f : 48.5f}};
    int pick = 0;
    float best = 0.0f;
    for (int i = 0; i < 5; ++i) {
        const long long blocks = (long long)ceil_div(T, shape[i].tt) * ceil_div(E, shape[i].te);
        const float cost = shape[i].first + shape[i].more * (float)((blocks + sm_count - 1) / sm_count - 1);
        if (i == 0 || cost <= best) { best = cost; pick = i; }
    }
    if (pick == 0) launch_route_score<2, 1, 4, 2, false>(x, W_r, z, T, d, E, status, st);
    else if (pick == 1) launch_route_score<2, 1, 4, 4, false>(x, W_r, z, T, d, E, status, st);
    else if (pick == 2) launch_route_score<2, 4, 4, 4, false>(x, W_r, z, T, d, E, status, st);
    else if (pick == 3) launch_route_score<4, 4, 4, 4, false>(x, W_r, z, T, d, E, status, st);
    else if (two) launch_route_score<4, 8, 4, 4, true>(x, W_r, z, T, d, E, status, st);
    else launch_route_score<4, 8, 4, 4, false>(x, W_r, z, T, d, E, status, st);
}

}  // namespace mop
