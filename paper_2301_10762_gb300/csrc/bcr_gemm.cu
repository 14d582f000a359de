// Block products of the block-cyclic-reduction factor on images (bcr_solve.h) of the operands:
//     C_t = +-A_t B_t^T    written as an image, or    D_t <- D_t -+ (A_t B_t^T + A'_t B'_t^T)    (FP32)
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
constexpr int BG_STAGE = 65536, BG_STAGES = 3, BG_QD = 4;
constexpr int BG_OUT = 4096;   // staging of an epilogue warp: 32 rows of an image's chunk
constexpr size_t BG_SMEM = (size_t)BG_STAGES * BG_STAGE + (BG_WARPS - BG_EPI0) * BG_OUT + 1024;

__device__ __forceinline__ void red_add2(float2 *p, float x, float y) {
    asm volatile("red.relaxed.gpu.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(x), "f"(y) : "memory");
}

struct BgTile {   // what the MMA thread and the epilogue need of a tile: read ahead by the copy thread
    int flags, terms, out, shift;   // (image: its scale)
    float f[2];                     // +-2^-(shift A + shift B) of the terms
    int out_t, blk;                 // the transposed image's matrix, or -1; the D block
};

__global__ void __launch_bounds__(BG_THREADS, 1) bcr_gemm_kernel(BgArgs a) {
    extern __shared__ uint8_t bg_smem[];
    __shared__ __align__(8) uint64_t full[BG_STAGES], empty[BG_STAGES], acc_full[2], acc_empty[2], done_bar;
    __shared__ __align__(8) uint64_t tq_full[BG_QD], tq_empty[BG_QD];
    __shared__ BgTile tq[BG_QD];
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
        for (int q = 0; q < BG_QD; ++q) {
            mbar_init(&tq_full[q], 1);
            mbar_init(&tq_empty[q], 1 + BG_WARPS - BG_EPI0);
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
    const int per = a.mt * a.nt, mr = (a.m + 7) & ~7, nr = (a.n + 7) & ~7;   // tiles of a task; rows of its operands
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
            int s = 0, issued = 0, i = 0;
            uint32_t ph = 1;
            bool go = true;
            const size_t im_off = (size_t)a.nzr * 128;
            for (int t = blockIdx.x; go && t < a.n_tiles; t += gridDim.x, ++i) {
                int task[BG_TASK];
#pragma unroll
                for (int e = 0; e < BG_TASK; ++e) task[e] = __ldg(a.tasks + BG_TASK * (t / per) + e);
                BgTile tl;
                tl.flags = task[0];
                tl.terms = (tl.flags & BG_TWO) ? 2 : 1;
                tl.out_t = (tl.flags & BG_TR) ? task[4] : -1;
                tl.blk = (tl.flags & BG_STORE) ? task[5] : task[3];
                tl.out = task[3];
                // image: the bound's scale
                const int eb = (int)(a.im.mx[task[1]] >> 23) + (int)(a.im.mx[task[2]] >> 23) - 254 + 2 + a.log2_2k;
                tl.shift = max(-100, min(100, 15 - eb));
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int x = task[u < tl.terms ? 1 + 3 * u : 1], y = task[u < tl.terms ? 2 + 3 * u : 2];
                    tl.f[u] = bs_pow2(max(-126, min(126, -(a.im.shift[x] + a.im.shift[y])))) * ((tl.flags & BG_NEG) ? -1.f : 1.f);
                }
                if (!wait1(&tq_empty[i % BG_QD], (uint32_t)((i / BG_QD) & 1) ^ 1u)) break;
                tq[i % BG_QD] = tl;
                mbar_arrive_cta(&tq_full[i % BG_QD]);
                const int m0 = 128 * (t % per / a.nt), n0 = 128 * (t % a.nt);
                const uint32_t ba = 128u * (uint32_t)min(128, mr - m0), bb = 128u * (uint32_t)min(128, nr - n0);
                const unsigned char *pa = nullptr, *pb = nullptr;
                for (int c = 0, n = a.n_chunk * tl.terms; c < n; ++c, pa += 2 * im_off, pb += 2 * im_off) {
                    if (c % a.n_chunk == 0) {   // the next term
                        pa = a.im.at(c == 0 ? task[1] : task[4], a.mat_bytes) + (size_t)(a.ca >> 5) * 2 * im_off + (size_t)(a.ra + m0) * 128;
                        pb = a.im.at(c == 0 ? task[2] : task[5], a.mat_bytes) + (size_t)(a.cb >> 5) * 2 * im_off + (size_t)(a.rb + n0) * 128;
                    }
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
            int s = 0, cc = 0, i = 0;
            uint32_t ph = 0;
            bool go = true;
            const uint64_t dstage0 = desc_sw128(smem0);
            for (int t = blockIdx.x; go && t < a.n_tiles; t += gridDim.x, ++i) {
                if (!wait1(&tq_full[i % BG_QD], (uint32_t)((i / BG_QD) & 1))) break;
                const int terms = tq[i % BG_QD].terms;
                mbar_arrive_cta(&tq_empty[i % BG_QD]);
                const int n0 = 128 * (t % a.nt), nb = min(128, (nr - n0 + 15) & ~15);
                const uint32_t id = idesc_f16(nb, false), idn = idesc_f16(nb, true);
                for (int c = 0, n = a.n_chunk * terms; c < n; ++c, ++cc) {
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
        int cc = 0, i = 0;
        bool go = true;
        const int n_cols = (a.n + 31) & ~31, m_cols = (a.m + 31) & ~31;
        unsigned char *stage = bg_smem + (smem0 - smem_u32(bg_smem)) + BG_STAGES * BG_STAGE + (warp - BG_EPI0) * BG_OUT;
        auto stage_wait = [&]() {   // the copy out of the staging buffer has read it
            if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            __syncwarp();
        };
        auto stage_store = [&](unsigned char *dst, int bytes) {
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0)
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n cp.async.bulk.commit_group;" ::"l"(dst),
                             "r"(smem_u32(stage)), "r"(bytes)
                             : "memory");
        };
        for (int t = blockIdx.x; t < a.n_tiles; t += gridDim.x, ++i) {
            const int m0 = 128 * (t % per / a.nt), n0 = 128 * (t % a.nt) + 64 * hh, m = m0 + 32 * q + lane;
            if (!__all_sync(0xffffffffu, mbar_wait_cta(&tq_full[i % BG_QD], (uint32_t)((i / BG_QD) & 1), a.tries, &s_abort))) {
                if (lane == 0) give_up();
                break;
            }
            const BgTile tl = tq[i % BG_QD];
            __syncwarp();
            if (lane == 0) mbar_arrive_cta(&tq_empty[i % BG_QD]);
            const int flags = tl.flags, out = tl.out, sh = tl.shift;
            float re[64], im[64];
#pragma unroll
            for (int e = 0; e < 64; ++e) re[e] = im[e] = 0.f;
            for (int c = 0; c < a.n_chunk * tl.terms; ++c, ++cc) {
                const float f = c < a.n_chunk ? tl.f[0] : tl.f[1];
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
                        re[8 * g + e] = fmaf(f, __uint_as_float(r0[e]), re[8 * g + e]);
                        re[8 * g + 8 + e] = fmaf(f, __uint_as_float(r1[e]), re[8 * g + 8 + e]);
                        im[8 * g + e] = fmaf(f, __uint_as_float(i0[e]), im[8 * g + e]);
                        im[8 * g + 8 + e] = fmaf(f, __uint_as_float(i1[e]), im[8 * g + 8 + e]);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cta(&acc_empty[cc & 1]);
            }
            if (!go) break;
            const int mb = m - lane;   // the warp's rows mb .. mb + 31
            if (flags & (BG_FP32 | BG_STORE)) {
                // the update is symmetric: entry (m, n) is added to D[n][m], 256 contiguous bytes of a
                // column's 32 rows at a time, and without a load
                float2 *dst = a.D + ((size_t)tl.blk * a.nz + a.co + n0) * a.nz + a.ro + m;
                if (m < a.m) {
#pragma unroll
                    for (int e = 0; e < 64; ++e)
                        if (n0 + e < a.n) {
                            if (flags & BG_STORE) dst[(size_t)e * a.nz] = make_float2(re[e], im[e]);
                            else red_add2(dst + (size_t)e * a.nz, re[e], im[e]);
                        }
                }
                if (!(flags & BG_STORE)) continue;
            }
            const float sc = bs_pow2(sh);
            uint32_t mxv = 0;
            unsigned char *img = a.im.at(out, a.mat_bytes), *img_t = tl.out_t >= 0 ? a.im.at(tl.out_t, a.mat_bytes) : nullptr;
            const size_t half = (size_t)a.nzr * 128;
            const int rows = min(32, mr - mb);
#pragma unroll
            for (int cb = 0; cb < 64; cb += 32) {
                const int nn = n0 + cb, c = (a.co + nn) >> 5;
                if (nn >= n_cols) continue;
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    float *v = (p ? im : re) + cb;
#pragma unroll
                    for (int e = 0; e < 32; ++e) {
                        if (m >= a.m || nn + e >= a.n) v[e] = 0.f;
                        mxv = max(mxv, bs_abs_bits(v[e]));
                        v[e] *= sc;
                    }
                    if (rows > 0) {   // rows of the image, in its layout: one contiguous piece of memory
                        stage_wait();
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            uint4 hi, lo;
                            bs_split2(v[8 * j], v[8 * j + 1], hi.x, lo.x);
                            bs_split2(v[8 * j + 2], v[8 * j + 3], hi.y, lo.y);
                            bs_split2(v[8 * j + 4], v[8 * j + 5], hi.z, lo.z);
                            bs_split2(v[8 * j + 6], v[8 * j + 7], hi.w, lo.w);
                            *reinterpret_cast<uint4 *>(stage + lane * 128 + ((j ^ (lane & 7)) << 4)) = hi;
                            *reinterpret_cast<uint4 *>(stage + lane * 128 + (((j + 4) ^ (lane & 7)) << 4)) = lo;
                        }
                        stage_store(img + (size_t)(2 * c + p) * half + (size_t)(a.ro + mb) * 128, rows * 128);
                    }
                    if (img_t && mb < m_cols) {
                        // the transpose: the warp's 32 rows are a chunk of row n; even lanes hold the hi
                        // parts of two columns, odd lanes the lo parts, 128 bytes in all
                        stage_wait();
#pragma unroll
                        for (int e = 0; e < 32; ++e) {
                            const int o = (((lane >> 3) + 4 * (lane & 1)) ^ (e & 7)) * 16 + (lane & 6) * 2;
                            *reinterpret_cast<uint32_t *>(stage + e * 128 + o) = bs_split_pair(v[e], lane);
                        }
                        stage_store(img_t + (size_t)(2 * ((a.ro + mb) >> 5) + p) * half + (size_t)(a.co + nn) * 128, min(32, nr - nn) * 128);
                    }
                }
            }
            if (t % per == 0 && warp == BG_EPI0 && lane == 0) {
                a.im.shift[out] = sh;
                if (img_t) a.im.shift[tl.out_t] = sh;
            }
            mxv = __reduce_max_sync(0xffffffffu, mxv);
            if (lane == 0 && mxv) {
                atomicMax(a.im.mx + out, mxv);
                if (img_t) atomicMax(a.im.mx + tl.out_t, mxv);
            }
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

}  // namespace

cudaError_t launch_bcr_gemm(BgArgs a, int n_tasks, int n_products, cudaStream_t st) {
    if (n_tasks <= 0) return cudaSuccess;
    if (a.nz & 1) return cudaErrorInvalidValue;
    const BsLayout l = bs_layout(a.nz);
    if (a.k == 0) a.m = a.n = a.k = a.nz;
    a.n_chunk = (a.k + 31) / 32;
    a.nzr = l.nzr;
    a.mat_bytes = l.mat_bytes;
    a.mt = (a.m + 127) / 128;
    a.nt = (a.n + 127) / 128;
    a.n_tiles = n_tasks * a.mt * a.nt;
    a.log2_2k = 1;
    while ((1 << a.log2_2k) < 2 * a.k) ++a.log2_2k;
    cudaError_t e = ensure_dyn_smem((const void *)bcr_gemm_kernel, BG_SMEM);
    if (e != cudaSuccess) return e;
    const int grid = std::min(device_sms(), a.n_tiles);
    HELM_TRACED_W(K_BCR_GEMM, st, 8.0 * a.m * a.n * (double)a.k * n_products,
                  (bcr_gemm_kernel<<<grid, BG_THREADS, BG_SMEM, st>>>(a)));
    return cudaGetLastError();
}

}  // namespace helm
