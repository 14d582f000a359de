// Block products of the block-cyclic-reduction factor on images (bcr_solve.h) of the operands:
//     C_t = +-A_t B_t^T        written as an image, or        D_t <- D_t - A_t B_t^T    (FP32)
// for n x n blocks A_t, B_t.  The factor's couplings and their products with the inverses never
// exist in FP32: the epilogue writes the next product's operands.  A CTA computes 128 x 128 tiles;
// a copy thread streams the operands' chunks (64 KB for 32 columns of K, contiguous runs, no
// tensor maps) through three stages, one thread issues the products (24 per chunk: hi hi, hi lo,
// lo hi of Ar Br - Ai Bi and Ar Bi + Ai Br, FP16, N = 128), eight warps write the tile.
// The tensor core adds into FP32 with truncation, so the number of additions into the large sum is
// what limits the product (192 at n = 256 in zgemm_tc.cu).  Here every chunk of 32 columns goes
// into a fresh accumulator, which the epilogue warps add to sums in registers, rounding to
// nearest, while the next chunk runs into the other one: 24 additions of a chunk, n / 32 sums.  It
// costs nothing (128 KB of tensor memory read per 1536 cycles of products) and leaves both
// accumulators to the next tile while a tile is written.
// An image's scale has to be known before the tile: 2^15 over the bound 2 n max|A| max|B|, which is
// 2^5 to 2^10 above the true maximum (FP16 keeps 22 bits down to 2^-15 of the scale); the true
// maximum is recorded on the way and bounds the next level.
// 256^2 with 8 frequencies, all products of the factor at levels >= 1: 4.6 ms as TF32 GEMMs of FP32
// blocks with images made afterwards (2.4 ms more).
#include <algorithm>

#include "abi_internal.h"
#include "bcr_image.cuh"
#include "bcr_solve.h"
#include "kernels.h"
#include "tcgen05.cuh"
#include "trace.h"

namespace helm {

namespace {

constexpr int BG_WARPS = 10, BG_THREADS = 32 * BG_WARPS, BG_EPI0 = 2;   // MMA, copy, eight epilogue warps
constexpr int BG_STAGE = 65536, BG_STAGES = 3;
constexpr size_t BG_SMEM = (size_t)BG_STAGES * BG_STAGE + 1024;

__global__ void __launch_bounds__(BG_THREADS, 1) bcr_gemm_kernel(BgArgs a) {
    extern __shared__ uint8_t bg_smem[];
    __shared__ __align__(8) uint64_t full[BG_STAGES], empty[BG_STAGES], acc_full[2], acc_empty[2], done_bar;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < BG_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&acc_full[s], 1);
            mbar_init(&acc_empty[s], BG_WARPS - BG_EPI0);
        }
        mbar_init(&done_bar, 1);
        fence_mbar_init_cluster();
        s_abort = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const uint32_t smem0 = (smem_u32(bg_smem) + 1023u) & ~1023u;
    const int per = a.nt * a.nt;   // tiles of a task
    auto give_up = [&]() {
        atomicOr(a.status, ST_TIMEOUT);
        s_abort = 1;
    };
    auto wait1 = [&](uint64_t *bar, uint32_t parity) -> bool {
        if (mbar_wait_cta(bar, parity, a.tries, &s_abort)) return true;
        give_up();
        return false;
    };
    if (warp == 1) {
        if (elect_one()) {   // copy thread
            int s = 0, issued = 0;
            uint32_t ph = 1;
            bool go = true;
            const size_t im_off = (size_t)a.nzr * 128;
            for (int t = blockIdx.x; go && t < a.n_tiles; t += gridDim.x) {
                const int *task = a.tasks + BG_TASK * (t / per);
                const int m0 = 128 * (t % per / a.nt), n0 = 128 * (t % a.nt);
                const uint32_t ba = 128u * (uint32_t)min(128, a.nzr - m0), bb = 128u * (uint32_t)min(128, a.nzr - n0);
                const unsigned char *pa = a.im.at(task[1], a.mat_bytes) + (size_t)m0 * 128;
                const unsigned char *pb = a.im.at(task[2], a.mat_bytes) + (size_t)n0 * 128;
                for (int c = 0; c < a.n_chunk; ++c, pa += 2 * im_off, pb += 2 * im_off) {
                    if (!wait1(&empty[s], ph)) { go = false; break; }
                    const uint32_t dst = smem0 + (uint32_t)(s * BG_STAGE);
                    mbar_arrive_expect_tx(&full[s], 2 * (ba + bb));
                    bulk_load(dst, pa, ba, &full[s]);
                    bulk_load(dst + 16384, pa + im_off, ba, &full[s]);
                    bulk_load(dst + 32768, pb, bb, &full[s]);
                    bulk_load(dst + 49152, pb + im_off, bb, &full[s]);
                    ++issued;
                    if (++s == BG_STAGES) { s = 0; ph ^= 1u; }
                }
            }
            // no copy may land after the CTA has left
            for (int c = max(0, issued - BG_STAGES); c < issued; ++c)
                mbar_wait_bounded(&full[c % BG_STAGES], (uint32_t)((c / BG_STAGES) & 1), kDefaultWaitTries);
        }
        __syncwarp();
    } else if (warp == 0) {
        if (elect_one()) {   // MMA thread
            int s = 0, cc = 0;
            uint32_t ph = 0;
            bool go = true;
            const uint64_t dstage0 = desc_sw128(smem0);
            for (int t = blockIdx.x; go && t < a.n_tiles; t += gridDim.x) {
                const int n0 = 128 * (t % a.nt), nb = min(128, (a.nzr - n0 + 15) & ~15);
                const uint32_t id = idesc_f16(nb, false), idn = idesc_f16(nb, true);
                for (int c = 0; c < a.n_chunk; ++c, ++cc) {
                    if (!wait1(&acc_empty[cc & 1], (uint32_t)((cc >> 1) & 1) ^ 1u) || !wait1(&full[s], ph)) { go = false; break; }
                    tc_fence_after();
                    const uint64_t ar = dstage0 + (uint64_t)(s * (BG_STAGE / 16)), ai = ar + 1024, br = ar + 2048, bi = ar + 3072;
                    const uint32_t d = tmem + (uint32_t)((cc & 1) * 256);   // Re, Im of the chunk
#pragma unroll
                    for (int p = 0; p < 6; ++p) {   // cross terms first: hi*lo, lo*hi, then hi*hi, two K steps each
                        const int ka = ((p >> 1) == 1 ? 4 : 0) + 2 * (p & 1), kb = (p < 2 ? 4 : 0) + 2 * (p & 1);
                        const uint32_t acc = p > 0 ? 1u : 0u;
                        tc_mma_f16(d, ar + ka, br + kb, id, acc);
                        tc_mma_f16(d + 128, ar + ka, bi + kb, id, acc);
                        tc_mma_f16(d, ai + ka, bi + kb, idn, 1u);
                        tc_mma_f16(d + 128, ai + ka, br + kb, id, 1u);
                    }
                    tc_commit(&empty[s]);
                    tc_commit(&acc_full[cc & 1]);
                    if (++s == BG_STAGES) { s = 0; ph ^= 1u; }
                }
            }
            tc_commit(&done_bar);
            mbar_wait_bounded(&done_bar, 0, kDefaultWaitTries);
        }
        __syncwarp();
    } else {
        // epilogue warps: tensor-memory lanes 32 q .. + 31 = rows m0 + 32 q + lane, 64 columns each
        const int q = warp & 3, hh = (warp - BG_EPI0) >> 2;
        int cc = 0;
        bool go = true;
        const int n_cols = 32 * a.n_chunk;
        for (int t = blockIdx.x; t < a.n_tiles; t += gridDim.x) {
            const int *task = a.tasks + BG_TASK * (t / per);
            const int m0 = 128 * (t % per / a.nt), n0 = 128 * (t % a.nt) + 64 * hh, m = m0 + 32 * q + lane;
            const int flags = task[0], ia = task[1], ib = task[2], out = task[3];
            const float f = bs_pow2(max(-126, min(126, -(a.im.shift[ia] + a.im.shift[ib])))) * ((flags & BG_NEG) ? -1.f : 1.f);
            float re[64], im[64];
#pragma unroll
            for (int e = 0; e < 64; ++e) re[e] = im[e] = 0.f;
            for (int c = 0; c < a.n_chunk; ++c, ++cc) {
                const bool ok = mbar_wait_cta(&acc_full[cc & 1], (uint32_t)((cc >> 1) & 1), a.tries, &s_abort);
                if (!__all_sync(0xffffffffu, ok)) {
                    if (lane == 0) give_up();
                    go = false;
                    break;
                }
                tc_fence_after();
                const uint32_t d = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)((cc & 1) * 256 + 64 * hh);
#pragma unroll
                for (int g = 0; g < 8; g += 2) {
                    uint32_t r0[8], r1[8], i0[8], i1[8];
                    tc_ld8_issue(d + 8 * g, r0);
                    tc_ld8_issue(d + 8 * g + 8, r1);
                    tc_ld8_issue(d + 128 + 8 * g, i0);
                    tc_ld8_issue(d + 128 + 8 * g + 8, i1);
                    tc_wait_ld8(r0);
                    tc_wait_ld8(r1);
                    tc_wait_ld8(i0);
                    tc_wait_ld8(i1);
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        re[8 * g + e] += __uint_as_float(r0[e]);
                        re[8 * g + 8 + e] += __uint_as_float(r1[e]);
                        im[8 * g + e] += __uint_as_float(i0[e]);
                        im[8 * g + 8 + e] += __uint_as_float(i1[e]);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cta(&acc_empty[cc & 1]);
            }
            if (!go) break;
            // image: the bound's scale
            const int eb = (int)(a.im.mx[ia] >> 23) + (int)(a.im.mx[ib] >> 23) - 254 + 2 + a.log2_2k;
            const int sh = max(-100, min(100, 15 - eb));
            const float sc = bs_pow2(sh);
            uint32_t mxv = 0;
            float2 *dst = a.D + (size_t)out * a.nz * a.nz + (size_t)m * a.nz;   // (BG_FP32)
            unsigned char *img = (flags & BG_FP32) ? nullptr : a.im.at(out, a.mat_bytes);
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                const int nn = n0 + 8 * g;
                if (nn >= n_cols) continue;
                float2 v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const bool in = m < a.nz && nn + e < a.nz;
                    v[e] = in ? make_float2(re[8 * g + e] * f, im[8 * g + e] * f) : make_float2(0.f, 0.f);
                }
                if (!img) {   // n is even: pairs of columns on 16-byte boundaries
                    if (m < a.nz) {
#pragma unroll
                        for (int e = 0; e < 8; e += 2)
                            if (nn + e < a.nz) {
                                float4 *w = reinterpret_cast<float4 *>(dst + nn + e);
                                const float4 o = *w;
                                *w = make_float4(o.x + v[e].x, o.y + v[e].y, o.z + v[e + 1].x, o.w + v[e + 1].y);
                            }
                    }
                    continue;
                }
                {
#pragma unroll
                    for (int e = 0; e < 8; ++e) mxv = max(mxv, max(bs_abs_bits(v[e].x), bs_abs_bits(v[e].y)));
                    if (m < a.nzr) {   // 16-byte pieces of the row: eight columns' hi, and lo 64 bytes on
                        const int c = nn >> 5, j = (nn >> 3) & 3;
                        uint4 rh, rl, ih, il;
                        bs_split8(v, sc, rh, rl, ih, il);
                        unsigned char *row = img + ((size_t)(2 * c) * a.nzr + m) * 128;
                        *reinterpret_cast<uint4 *>(row + ((j ^ (m & 7)) << 4)) = rh;
                        *reinterpret_cast<uint4 *>(row + (((j + 4) ^ (m & 7)) << 4)) = rl;
                        row += (size_t)a.nzr * 128;
                        *reinterpret_cast<uint4 *>(row + ((j ^ (m & 7)) << 4)) = ih;
                        *reinterpret_cast<uint4 *>(row + (((j + 4) ^ (m & 7)) << 4)) = il;
                    }
                }
            }
            if (img) {
                if (t % per == 0 && warp == BG_EPI0 && lane == 0) a.im.shift[out] = sh;
                mxv = __reduce_max_sync(0xffffffffu, mxv);
                if (lane == 0 && mxv) atomicMax(a.im.mx + out, mxv);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

}  // namespace

cudaError_t launch_bcr_gemm(BgArgs a, int n_tasks, cudaStream_t st) {
    if (n_tasks <= 0) return cudaSuccess;
    if (a.nz & 1) return cudaErrorInvalidValue;
    const BsLayout l = bs_layout(a.nz);
    a.n_chunk = l.n_chunk;
    a.nzr = l.nzr;
    a.mat_bytes = l.mat_bytes;
    a.nt = (a.nz + 127) / 128;
    a.n_tiles = n_tasks * a.nt * a.nt;
    a.log2_2k = 1;
    while ((1 << a.log2_2k) < 2 * a.nz) ++a.log2_2k;
    cudaError_t e = ensure_dyn_smem((const void *)bcr_gemm_kernel, BG_SMEM);
    if (e != cudaSuccess) return e;
    const int grid = std::min(device_sms(), a.n_tiles);
    HELM_TRACED_W(K_BCR_GEMM, st, 8.0 * a.nz * a.nz * (double)a.nz * n_tasks,
                  (bcr_gemm_kernel<<<grid, BG_THREADS, BG_SMEM, st>>>(a)));
    return cudaGetLastError();
}

}  // namespace helm
