// Warp-MMA building blocks of the kernels that keep the weights of a stage in registers (fused_m32.cu, stream_m64.cu): one
// operand is the weights (rows = outputs), the tokens are N, so results have tokens innermost and every permutation of
// Section 3.3 is a choice of where stmatrix puts a row of 8 tokens.
#pragma once

#include "tc_common.cuh"

namespace monarch {
namespace tc {

__device__ __forceinline__ void ldm4(uint32_t (&r)[4], uint32_t a)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldm4t(uint32_t (&r)[4], uint32_t a)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void stm4(uint32_t a, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3)
{
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(r0), "r"(r1), "r"(r2), "r"(r3) : "memory");
}
__device__ __forceinline__ void stm4(uint32_t a, const uint32_t (&r)[4]) { stm4(a, r[0], r[1], r[2], r[3]); }
__device__ __forceinline__ void stm4t(uint32_t a, const uint32_t (&r)[4])
{
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}
__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *m, int x, int y, int z, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(dst),
                 "l"(m), "r"(bar), "r"(x), "r"(y), "r"(z) : "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap *m, uint32_t src, int x, int y, int z)
{
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(m), "r"(src), "r"(x), "r"(y), "r"(z) : "memory");
}

struct Lane {                                            // rows of the four matrices of an x4 instruction
    int warp, m, r;
    __device__ __forceinline__ Lane() : warp(threadIdx.x >> 5), m((threadIdx.x & 31) >> 3), r(threadIdx.x & 7) {}
};

// After a wait that ran out: no copy into this CTA's shared memory may outlive the CTA.  Nothing is loaded any more (Ring::load),
// and what is under way lands within a millisecond.
__device__ __forceinline__ void let_copies_land(volatile int *dead)
{
    if (*dead)
        for (int i = 0; i < 4096; ++i) __nanosleep(256);
}

// Launched with programmatic serialization: a kernel may begin while the one before it drains.  Before its wait it may read only
// what no kernel of its own call writes (the weights), and only behind a kernel of that call that signals after its own wait: what
// ran before the call has then finished.  Everything else, and all writes, come after the wait.  The kernels of rect_tc.cu
// signal before they wait, so a launch behind one of them reads nothing early.
__device__ __forceinline__ void depend_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void depend_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... Ts, typename... As>
int launch_serialized(void (*kern)(Ts...), dim3 grid, int threads, int smem, cudaStream_t s, As... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (smem > 48 * 1024) MONARCH_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    MONARCH_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, args...));
    note_launch();
    return MONARCH_OK;
}

}  // namespace tc
}  // namespace monarch
