// Bulk-tensor loads and their mbarriers, shared by the 3D sweeps (tma3d.cu, tma3d2.cu).
#pragma once

#include <cuda.h>

namespace mxp {

constexpr long long kTmaPollLimit = 1ll << 22;

template <typename S> struct TmaElt;
template <> struct TmaElt<float2> {        // complex64: two 4-byte elements per value
    static constexpr int E = 2, HL = 2;
};
template <> struct TmaElt<__nv_bfloat162> {  // bf16x2: one 4-byte element per value
    static constexpr int E = 1, HL = 4;
};

__device__ __forceinline__ unsigned smem_u32(const void *p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void tma_load3(void *dst, const CUtensorMap *map, int c0, int c1, int c2,
                                          unsigned long long *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];"
        :
        : "r"(smem_u32(dst)), "l"(reinterpret_cast<unsigned long long>(map)), "r"(c0), "r"(c1), "r"(c2),
          "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void mbar_expect(unsigned long long *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// true once the phase with the given parity has completed; false after the limit
__device__ __forceinline__ bool mbar_wait(unsigned long long *bar, unsigned parity)
{
    for (long long it = 0; it < kTmaPollLimit; ++it) {
        unsigned done;
        asm volatile(
            "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
            : "=r"(done)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// Tensor map of a 3D array of 4-byte elements: extents (ex, ey, ez) elements, rows
// `row` and planes `plane` bytes apart, box bx x by x 1; zeros outside.
bool tma3_encode(CUtensorMap *m, const void *base, int64_t ex, int64_t ey, int64_t ez, int64_t row, int64_t plane, int bx,
                 int by);

// Maps of a problem's four work buffers and of its kappa.  Rows are `pitch` values
// apart (n0 rounded up to a multiple of 4: strides must be multiples of 16 bytes).
struct Tma3Maps {
    CUtensorMap p[4], y[4], k;                 // one step: boxes of tma3d.cu
    CUtensorMap p2[2][4], y2[2][4], k2[2];     // two steps: boxes of tma3d2.cu, regions of 32 and 64 columns
    int pitch = 0;
    bool ok = false;
};

template <typename S> bool tma3_maps2(Tma3Maps *t, const Geom &g, void *const *bufs, const float *kappa);

}  // namespace mxp
