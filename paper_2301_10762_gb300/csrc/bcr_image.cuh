// Device helpers of the block images (bcr_solve.h): scales, the FP16 hi / lo split, bulk copies
// (internal header of bcr_solve.cu and bcr_gemm.cu).
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

#include "common.cuh"

namespace helm {

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive_cta(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ uint32_t bs_abs_bits(float x) { return __float_as_uint(x) & 0x7fffffffu; }

// shift s with max * 2^s in [2^14, 2^15) (FP16 range), from the bits of the maximum modulus; NaN
// and infinite maxima get a finite scale and stay NaN or infinite in the split
__device__ __forceinline__ int bs_scale_shift(uint32_t max_bits) { return min(141 - (int)(max_bits >> 23), 100); }
__device__ __forceinline__ float bs_pow2(int s) { return __uint_as_float((uint32_t)(127 + s) << 23); }

// (hi, lo) FP16 split of two scaled values, packed
__device__ __forceinline__ void bs_split2(float a, float b, uint32_t &hi, uint32_t &lo) {
    const __half2 h = __floats2half2_rn(a, b);
    const float2 f = __half22float2(h);
    const __half2 l = __floats2half2_rn(a - f.x, b - f.y);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    lo = *reinterpret_cast<const uint32_t *>(&l);
}
// hi parts of this lane's and the next lane's value (even lanes), lo parts of the lane before's and
// this one's (odd lanes), packed; all lanes of the warp
__device__ __forceinline__ uint32_t bs_split_pair(float x, int lane) {
    const __half h = __float2half_rn(x), l = __float2half_rn(x - __half2float(h));
    const uint32_t t = (uint32_t)__half_as_ushort(h) | (uint32_t)__half_as_ushort(l) << 16;
    const uint32_t o = __shfl_xor_sync(0xffffffffu, t, 1);
    return (lane & 1) ? ((o >> 16) | (t & 0xffff0000u)) : ((t & 0xffffu) | (o << 16));
}
// the 16-byte pieces (hi and lo, real and imaginary) of eight entries times sc
__device__ __forceinline__ void bs_split8(const float2 (&v)[8], float sc, uint4 &rh, uint4 &rl, uint4 &ih, uint4 &il) {
    uint32_t *a = reinterpret_cast<uint32_t *>(&rh), *b = reinterpret_cast<uint32_t *>(&rl);
    uint32_t *c = reinterpret_cast<uint32_t *>(&ih), *d = reinterpret_cast<uint32_t *>(&il);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        bs_split2(v[2 * e].x * sc, v[2 * e + 1].x * sc, a[e], b[e]);
        bs_split2(v[2 * e].y * sc, v[2 * e + 1].y * sc, c[e], d[e]);
    }
}

}  // namespace helm
