// Shared device helpers for the routed-expert kernels (sm_100a only).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace mop {

typedef __nv_bfloat16 bf16;

// Codes written to the context's device status word by bounded waits.
enum : int { STATUS_OK = 0, STATUS_WAIT_FULL = 1, STATUS_WAIT_EMPTY = 2, STATUS_WAIT_TMEM_FULL = 3,
             STATUS_WAIT_TMEM_EMPTY = 4, STATUS_BAD_TILE = 5 };

__device__ __forceinline__ float bf16_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

// two fp32 -> packed bf16x2 (round to nearest even), lo in the low half
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&p);
}

__device__ __forceinline__ float sigmoidf_acc(float v) { return 1.0f / (1.0f + expf(-v)); }
// Sigmoid of the SwiGLU epilogues: fast exponential and division (about 2 ulp), far inside the bf16
// rounding of every value it feeds; all GEMM schedules share it, so they stay bit-identical.  (The
// router's gates keep the accurate form above.)
__device__ __forceinline__ float sigmoidf_fast(float v) { return __fdividef(1.0f, 1.0f + __expf(-v)); }

// Programmatic dependent launch: a kernel started by pdl_launch() may be brought up before its predecessor in the stream has
// drained; pdl_begin() waits until the predecessor has finished and its writes are visible.  Nothing may be read or written
// before it, and every kernel started by pdl_launch() calls it, or one of its two forms below, in every thread.
// A grid of few blocks also lets the next kernel come up while it runs (blocks resident, barriers and tensor memory set up).  A
// grid that fills the SMs does not: the next kernel's blocks would pile up on the SMs that empty first (training step at
// T 1537, d 1000, E 20: 346 us without any of this, 391 with every kernel letting its successor in at its start).
__device__ __forceinline__ void pdl_begin() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (gridDim.x * gridDim.y <= 64) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// The exception: a GEMM followed by a GEMM.  Both take a whole SM per CTA, so the next one's CTAs can only come up where one of this
// grid has left, one each, and find their barriers, tensor memory and descriptors ready when the last one leaves.
// `note`: the next kernel runs beside this one, and this one leaves word that everything before it is complete.
struct PdlNote {
    int32_t* word;           // null: no such kernel follows
    int32_t value;           // another one for every pair of kernels since the word was cleared
};
__device__ __forceinline__ void pdl_begin_gemm(bool gemm_follows, const PdlNote& note) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (note.word) {
        if (blockIdx.x == 0 && threadIdx.x == 0)
            asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(note.word), "r"(note.value) : "memory");
        __syncthreads();     // so that the word is on its way before this block lets the next kernel start
    }
    if (gemm_follows) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// A kernel that runs beside the one before it (A), and reads and writes only what kernels before A have written and read.
//  - A waits first (pdl_begin_gemm with the same note), so all grids before A are complete and visible to A when it writes the word;
//    each of those has waited for the one before it in turn.
//  - Only this kernel's own griddepcontrol.wait would make their writes visible to it, and that one waits for A as well.  So the
//    ordering goes through the word: A's release, the acquire here, the barrier, and, because TMA reads through another proxy than
//    the one those kernels wrote through, a proxy fence in every thread.  The word is not waited for: a block that does not find it
//    takes the grid's wait.
//  - What A reads may only be overwritten, and what A writes only be read, by kernels after this one: it waits for A before it
//    leaves (pdl_end_beside), so that its end is the end of both.
__device__ __forceinline__ void pdl_begin_beside(bool gemm_follows, const PdlNote& note) {
    if (gemm_follows) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    int32_t v = note.value;
    if (threadIdx.x == 0) asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(note.word) : "memory");
    if (!__syncthreads_and(v == note.value)) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("fence.proxy.async.global;" ::: "memory");
}
__device__ __forceinline__ void pdl_end_beside() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class... P, class... A>
inline cudaError_t pdl_launch_clusters(void (*kernel)(P...), int cluster, dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                       A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[2] = {};
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster; attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = cluster > 0 ? 2 : 1;      // 0: as the kernel itself declares
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
template <class... P, class... A>
inline cudaError_t pdl_launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
    return pdl_launch_clusters(kernel, 0, grid, block, smem, st, args...);
}

__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

static inline int ceil_div(int a, int b) { return (a + b - 1) / b; }

// Optional per-kernel timing: a pool of CUDA event pairs recorded around every launch on the
// launching stream, aggregated by kernel name when read.  Off by default (no events, no cost).
struct Profiler {
    static constexpr int MAX_REC = 8192;
    bool on = false;
    cudaEvent_t* ev = nullptr;          // 2 * MAX_REC events once enabled
    const char* names[MAX_REC];
    int n = 0;
    void begin(const char* name, cudaStream_t st) {
        if (on && n < MAX_REC) { names[n] = name; cudaEventRecord(ev[2 * n], st); }
    }
    void end(cudaStream_t st) {
        if (on && n < MAX_REC) { cudaEventRecord(ev[2 * n + 1], st); ++n; }
    }
};

}  // namespace mop
