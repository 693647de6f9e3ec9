// Helpers of the tensor-core kernels that run on CTA pairs (tcgen05
// cta_group::2, a cluster of two CTAs on one 256-row tile) with bf16
// operand planes: barriers of the pair, TMA loads that signal the leader's
// barrier, matrix and instruction descriptors, 256-bit stores.
//
// A pair's leader is the CTA of rank 0. Each CTA loads its own half of both
// operands (its 128 rows of A, its half of B's rows) into the same offsets of
// its own shared memory and its loads complete on the leader's "full" barrier;
// one thread of the leader issues the MMAs for both, each CTA's tensor memory
// receives its own 128 rows of the result, and commits are multicast to the
// barriers of both CTAs.
#pragma once

#include <atomic>

#include <cuda_bf16.h>

#include "tc_common.cuh"

namespace csrt {

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The shared::cluster address of a local shared-memory object in CTA `rank`.
__device__ __forceinline__ uint32_t map_to_rank(const void *p, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
    return r;
}
// Arrives on a barrier of either CTA. (With .release.cluster the arrival waits
// for every load the thread has in flight, over 1000 clocks for a prefetch;
// what it has to order here is shared memory behind fence.proxy.async and
// tensor memory behind tcgen05.wait and fence.)
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// 2-D TMA load into this CTA's shared memory, completing on a barrier given
// by its shared::cluster address (the leader's).
__device__ __forceinline__ void tma_load_2d_pair(void *dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
// Bounded wait for a phase of a barrier, or for another role's giving up. The
// thread sleeps in the barrier unit for up to a microsecond per look instead
// of taking issue slots from the warps that work.
constexpr unsigned kPairWaitLooks = 1u << 18;
__device__ __forceinline__ bool pair_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag) {
    const uint32_t addr = smem_u32(bar);
    for (unsigned i = 0; i < kPairWaitLooks; ++i) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(addr), "r"(parity)
            : "memory");
        if (done) return true;
        if (*abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}
// Arrives on the barrier at this offset in both CTAs once every MMA issued
// before by this thread is done.
__device__ __forceinline__ void mma_commit_pair(uint64_t *bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_u32(bar)),
        "h"((uint16_t)3)
        : "memory");
}
// The operands by the low words of their matrix descriptors (the address in
// units of 16 bytes and the part that is the same for all K-major operands of
// 128-byte rows; smem_desc_sw128): offsets are added there in 32 bits, and the
// high word is a constant.
__device__ __forceinline__ uint32_t smem_desc_lo(const void *p) { return (uint32_t)smem_desc_sw128(p); }
__device__ __forceinline__ void mma_bf16_pair(uint32_t tmem_d, uint32_t adesc_lo, uint32_t bdesc_lo, uint32_t idesc,
                                             uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n .reg .b64 a, b;\n setp.ne.b32 p, %4, 0;\n mov.b64 a, {%1, %5};\n mov.b64 b, {%2, %5};\n"
        " tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, p;\n}\n" ::"r"(tmem_d),
        "r"(adesc_lo), "r"(bdesc_lo), "r"(idesc), "r"(accumulate), "n"(kSmemDescHi)
        : "memory");
}

// Instruction descriptor, kind::f16: bf16 operands, both K-major, float32
// accumulators.
__host__ __device__ constexpr uint32_t idesc_bf16(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// Sixteen columns of this warp's 32 tensor-memory lanes.
__device__ __forceinline__ void tmem_ld_16cols(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Eight floats to a 32-byte aligned address in one store (a whole sector).
__device__ __forceinline__ void st_global_f8(float *p, const float *v) {
    asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}

__device__ __forceinline__ void ld_global_f8(const float *p, float (&v)[8]) {
    asm volatile("ld.relaxed.gpu.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(p)
                 : "memory");
}

// Row-major rows x cols matrix of bf16 with row stride ld elements (a multiple
// of 8): boxes of box_rows x 64 elements, 128-byte swizzle.
inline bool make_map_bf16(CUtensorMap *map, const void *base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// Whether this build's kernel can run on the current device as written: it may
// use `smem` bytes of shared memory, and its launches of `threads` threads hold
// `regs` registers, the sum of what its warps lower and raise their shares to
// (setmaxnreg.inc waits without a bound for registers the launch does not
// hold; how many it holds is the compiler's choice). `state`: 64 zeros, one per
// device, asked once.
template <typename K>
inline bool pair_kernel_ready(K kernel, std::atomic<int> *state, int smem, int threads, int regs) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    int known = state[dev].load();
    if (known == 0) {
        cudaFuncAttributes fa{};
        const bool ok =
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess &&
            cudaFuncGetAttributes(&fa, kernel) == cudaSuccess && fa.numRegs * threads >= regs;
        if (!ok) cudaGetLastError();   // (not an error of the call: it takes the other path)
        known = ok ? 1 : 2;
        state[dev].store(known);
    }
    return known == 1;
}

// Launch of a kernel on CTA pairs (grid a multiple of 2) with programmatic
// dependent launch.
template <typename... P, typename... A>
inline cudaError_t launch_pair(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                               A &&...args) {
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace csrt
