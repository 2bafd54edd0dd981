// ews_tma.cuh -- mbarrier and TMA wrappers, tensor-map encoding and the z-chunk
// model shared by the z-marching kernels (ews_stencil.cu, ews_fused.cu).
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "ews_internal.cuh"

namespace ews {
namespace {

constexpr unsigned long long kWaitNs = 2000000000ull;  // 2 s per wait
constexpr int r128(int b) { return (b + 127) / 128 * 128; }

// --- PTX wrappers -------------------------------------------------------------

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}

__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait on the phase `parity` of an mbarrier.
__device__ __noinline__ bool mbar_wait_slow(uint64_t* bar, uint32_t parity) {
    const unsigned long long t0 = now_ns();
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if (now_ns() - t0 > kWaitNs) return false;
        __nanosleep(64);
    }
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
    return mbar_try(bar, parity) || mbar_wait_slow(bar, parity);
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar,
                                            int x, int y, int z) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z)
        : "memory");
}

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, uint64_t* bar,
                                            int x, int y, int z, int w) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z),
        "r"(w)
        : "memory");
}

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

// Tensor map of nt pitched [nz][ny][pitch] arrays lying tstride bytes apart,
// as a 4D tensor [array][nz][ny][pitch], with a box of bw x bh x 1 x bt.
bool encode4(CUtensorMap* map, const DevGrid& g, const void* base, CUtensorMapDataType dt,
             int esize, long long tstride, int nt, int bw, int bh, int bt) {
    auto fn = encoder();
    if (!fn) return false;
    cuuint64_t dims[4] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz, (cuuint64_t)nt};
    cuuint64_t strides[3] = {(cuuint64_t)g.pitch * esize, (cuuint64_t)g.plane * esize,
                             (cuuint64_t)tstride};
    cuuint32_t box[4] = {(cuuint32_t)bw, (cuuint32_t)bh, 1, (cuuint32_t)bt};
    cuuint32_t es[4] = {1, 1, 1, 1};
    CUresult r = fn(map, dt, 4, const_cast<void*>(base), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// Tensor map of one pitched [nz][ny][pitch] array with a box of bw x bh x 1.
bool encode(CUtensorMap* map, const DevGrid& g, const void* base, CUtensorMapDataType dt,
            int esize, int bw, int bh) {
    auto fn = encoder();
    if (!fn) return false;
    cuuint64_t dims[3] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz};
    cuuint64_t strides[2] = {(cuuint64_t)g.pitch * esize, (cuuint64_t)g.plane * esize};
    cuuint32_t box[3] = {(cuuint32_t)bw, (cuuint32_t)bh, 1};
    cuuint32_t es[3] = {1, 1, 1};
    CUresult r = fn(map, dt, 3, const_cast<void*>(base), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// Planes per z-chunk of a pass over ntile tile columns with `slots` CTAs
// resident at once: the chunk count n (chunks of at least min_planes
// planes) that minimises the modelled pass time, the waves of (tile, chunk)
// CTAs times the planes each CTA marches through, ceil(ntile n / slots) x
// (nz / n + halo) with `halo` the planes a chunk loads beyond its own on
// each side; ties go to more chunks.  Measured against the earlier rule of
// about four waves (GB300, Gcell/s): 192^3 sponge 48.4 vs 44.5, 192^3 C-PML
// 35.4 vs 33.8, 128^3 sponge 50.5 vs 39.4, 1024 x 1024 x 512 BF16 (32 x 16
// tiles) 78.9 vs 75.9, 256^3 C-PML unchanged (7 chunks either way).  Chunks
// of at least 4 planes: small grids, whose few columns leave most SMs idle,
// get more CTAs (64 x 64 x 32 sponge: 11.3 Gcell/s with 4-plane chunks, 9.1
// with at least 8 planes; 64^3 19.9 vs 17.5).
int chunk_planes(long long ntile, long long slots, int nz, int min_planes, int halo) {
    long long best_n = 1, best_cost = -1;
    for (long long n = 1; n <= std::max(1, nz / min_planes); ++n) {
        const long long zc = (nz + n - 1) / n;
        const long long nn = (nz + zc - 1) / zc;               // chunks of zc planes
        const long long cost = ((ntile * nn + slots - 1) / slots) * (zc + halo);
        if (best_cost < 0 || cost <= best_cost) {
            best_cost = cost;
            best_n = n;
        }
    }
    return (int)((nz + best_n - 1) / best_n);
}

}  // namespace
}  // namespace ews
