// PTX wrappers shared by the tensor-core contractions (tcgen05, mbarrier, TMA
// for sm_103a) and the host's access to the tensor-map encoder.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "fbs_internal.h"

namespace fbs {

namespace {

constexpr long long kWaitCycles = 2000000000LL;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the phase of the given parity; false on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
    long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > kWaitCycles) return false;
    }
    return true;
}

__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// One lane of a converged warp (the same lane each time).  Code under
// elect.sync is known to run on one thread, so the descriptors of its MMAs go
// to uniform registers once; under an ordinary `lane == 0` branch every
// tcgen05.mma costs the issuing thread at least 45 cycles, under elect.sync
// N / 2 (the tensor pipe's own rate at M = 128, K = 16), measured for N = 32..256.
__device__ __forceinline__ bool elect_one() {
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(ok));
    return ok != 0;
}

__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// 2-D tiled TMA load (x = point, y = bin) into shared memory; completion is
// counted in bytes on the mbarrier.  Points past the tensor's end read zero.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y,
                                            uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
        "[%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// Bounded wait that gives up at once after any other wait of the CTA timed
// out (the abort flag is sticky), so no role can strand another.
// `limit` is the launch's hand-off wait limit in clock cycles (about one
// second by default; a plan option shortens it to exercise this path).
__device__ __forceinline__ bool role_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag,
                                          int *err, int code, long long limit) {
    if (mbar_try_wait(bar, parity)) return true;  // ready: no clock read, no flag read
    long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (*abort_flag) return false;
        if (clock64() - t0 > limit) {
            *abort_flag = 1;
            atomicExch(err, code);
            return false;
        }
    }
    return true;
}

// Compensated (Kahan) FP32 running sum: x = sum, y = compensation; the
// value is x - y.  Explicit round-to-nearest operations keep the compiler
// from contracting or reassociating them.
__device__ __forceinline__ void kahan_add(float2 &a, float v) {
    const float y = __fsub_rn(v, a.y);
    const float t = __fadd_rn(a.x, y);
    a.y = __fsub_rn(__fsub_rn(t, a.x), y);
    a.x = t;
}

}  // namespace

// cuTensorMapEncodeTiled through cudaGetDriverEntryPointByVersion, so the
// library links only the CUDA runtime (not libcuda directly).
inline PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    }();
    return fn;
}

// Tensor map of one slab of shell fields: x = point (npts valid, contiguous),
// y = bin (stride slab_stride floats); boxes of `pts` points x all bins, in the
// 128-byte swizzle (32 points) or row by row; points past npts read as zero.
inline CUtensorMap field_map(const float *islab, long long npts, long long slab_stride, int nbins, int rows, int pts,
                             bool swizzled) {
    auto enc = tensor_map_encoder();
    if (!enc) throw Failure{FBS_ERR_CUDA, "cuTensorMapEncodeTiled is not available"};
    if ((reinterpret_cast<uintptr_t>(islab) & 15) || ((slab_stride * 4) & 15) || nbins < 1 || nbins > 256 ||
        rows < nbins || npts < 1 || npts >= (1LL << 31))
        throw Failure{FBS_ERR_ARG, "shell-field slab does not meet the TMA layout rules"};
    CUtensorMap m;
    cuuint64_t dims[2] = {(cuuint64_t)npts, (cuuint64_t)rows};  // rows: nbins per field of a batch
    cuuint64_t strides[1] = {(cuuint64_t)slab_stride * 4};
    cuuint32_t box[2] = {(cuuint32_t)pts, (cuuint32_t)nbins};
    cuuint32_t es[2] = {1u, 1u};
    CUresult r = enc(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float *>(islab), dims, strides, box, es,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, swizzled ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) throw Failure{FBS_ERR_CUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")"};
    return m;
}

}  // namespace fbs
