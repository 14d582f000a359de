// The solve of a block-cyclic-reduction factor (bcr.cu) as one persistent tensor-core kernel.
//
// Every step of the substitution is a sum of products of a stored n_z x n_z block with a line of
// the right-hand sides of a system (bcr.cu's header; C = diag(cx) the level-0 coupling):
//     level 0, forward    r_k -= C (Dinv_{k-1} r_{k-1} + Dinv_{k+1} r_{k+1})       k even
//     level l, forward    r_k -= W_a r_a + V_c r_c                                 k = 0 mod 2s
//     last line           x_0 = Dinv_0 r_0
//     level l, backward   x_j = Dinv_j r_j - P_j x_{j-s} - Q_j x_{j+s}             j = s mod 2s
//     level 0, backward   x_j = Dinv_j (r_j - C (x_{j-1} + x_{j+1}))               j odd
// The blocks are read once per solve and nothing else comes close in bytes (3.5 n_x n_z^2 complex
// entries per frequency: 3.8 GB at 256^2 with 8 frequencies, 0.56 ms at the measured copy rate),
// so the kernel is laid out as a stream of the blocks through the tensor cores:
//   * The blocks are stored as the tensor core reads them ("image"): every real entry as the sum
//     of two FP16 numbers of its row-scaled value (hi + lo, 22 to 23 bits below the largest entry
//     of the row, as many as the 3xTF32 split of the GEMM keeps; 8 bytes per complex entry as in
//     FP32), real and imaginary parts apart, 32 columns of a row as one 128-byte swizzled row (32
//     hi, then 32 lo).  A chunk of a tile is two contiguous runs of memory: a copy warp streams
//     them with bulk copies, and no thread touches them.
//   * The vectors are split by operand warps as they come (a power-of-two scale per line slice
//     from the maxima that the writers of the vectors leave), 16 KB against 32 KB of block data
//     per chunk at 64 right-hand sides.
//   * One MMA warp issues hi hi + hi lo + lo hi for Re and Im (the negated product by the
//     instruction's negate bit), FP32 accumulation in tensor memory, one accumulator per product
//     term (the terms' scales differ); four epilogue warps scale, sum, add the old line and
//     write, while the next tile's products run into the other accumulators.
//   * The tiles of all levels are taken in order from a device counter by whichever CTA is free.
//     A tile waits until the previous step of its own system is complete (a counter per step and
//     system); only the operand warps wait, so the block stream runs on across steps.  Every
//     wait is for tiles that were taken earlier, so the kernel needs no co-resident grid, and
//     every wait is bounded.
#include <algorithm>

#include "abi_internal.h"
#include "bcr_solve.h"
#include "kernels.h"
#include "tcgen05.cuh"
#include "trace.h"

#include <cuda_fp16.h>

namespace helm {

namespace {

constexpr int BS_WARPS = 14;                 // MMA, copy, 4 epilogue, 8 operand warps
constexpr int BS_THREADS = 32 * BS_WARPS;
constexpr int BS_EPI0 = 2, BS_OP0 = 6, BS_OPW = 8;
constexpr int BS_QD = 4;                     // tile queue of a CTA
constexpr int BS_A = 32768;                  // A bytes of a stage: 128 rows x 128 bytes, Re and Im
constexpr uint32_t BS_TMEM = 512;

template <int NT> struct BsCfg {
    static constexpr int B = NT * 256;                   // B bytes of a stage: NT rows x 128 bytes, Re and Im
    static constexpr int STAGE = BS_A + B;
    static constexpr int STAGES = NT == 64 ? 4 : 5;
    static constexpr int SLOTS = NT == 64 ? 4 : 8;       // accumulators of 2 NT tensor-memory columns
    static constexpr int PAIRS = NT / 16;                // row pairs of a chunk per operand warp
    static constexpr size_t SMEM = (size_t)STAGES * STAGE + 1024;
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t abs_bits(float x) { return __float_as_uint(x) & 0x7fffffffu; }

// shift s with max * 2^s in [2^14, 2^15) (FP16 range), from the bits of the maximum modulus; NaN
// and infinite maxima get a finite scale and stay NaN or infinite in the split
__device__ __forceinline__ int scale_shift(uint32_t max_bits) { return min(141 - (int)(max_bits >> 23), 100); }
__device__ __forceinline__ float pow2(int s) { return __uint_as_float((uint32_t)(127 + s) << 23); }

// (hi, lo) FP16 split of two scaled values, packed
__device__ __forceinline__ void split_h2(float a, float b, uint32_t &hi, uint32_t &lo) {
    const __half2 h = __floats2half2_rn(a, b);
    const float2 f = __half22float2(h);
    const __half2 l = __floats2half2_rn(a - f.x, b - f.y);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    lo = *reinterpret_cast<const uint32_t *>(&l);
}

struct Tile {
    int phase, sys, task, n0, r0, rows;
};
__device__ __forceinline__ Tile decode(const BsArgs &a, int t, int nt_size) {
    int p = 0;
    while (p + 1 < a.n_phase && t >= a.ph[p + 1].tile0) ++p;
    const BsPhase &ph = a.ph[p];
    int q = t - ph.tile0;
    Tile o;
    o.phase = p;
    o.r0 = (q % ph.mt) * ph.mrows;
    q /= ph.mt;
    o.n0 = (q % a.n_tiles) * nt_size;
    q /= a.n_tiles;
    o.sys = q / ph.tasks;
    o.task = ph.task0 + q % ph.tasks;
    o.rows = min(ph.mrows, a.nzr - o.r0);
    return o;
}

template <int NT, bool EVEN>
__global__ void __launch_bounds__(BS_THREADS, 1) bcr_solve_kernel(const __grid_constant__ BsArgs a) {
    using Cfg = BsCfg<NT>;
    constexpr int ST = Cfg::STAGES, SL = Cfg::SLOTS;
    extern __shared__ uint8_t bs_smem[];
    __shared__ __align__(8) uint64_t full_a[ST], full_b[ST], empty[ST];
    __shared__ __align__(8) uint64_t acc_full[SL], acc_empty[SL];
    __shared__ __align__(8) uint64_t tq_full[BS_QD], tq_empty[BS_QD], done_bar;
    __shared__ int tq[BS_QD];
    __shared__ float s_bscale[SL][NT];   // 2^-s of each right-hand side of an accumulator's product
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    if (a.skip && *a.skip) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(&full_a[s], 1);
            mbar_init(&full_b[s], BS_OPW);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < SL; ++s) {
            mbar_init(&acc_full[s], 1);
            mbar_init(&acc_empty[s], 4);
        }
        for (int q = 0; q < BS_QD; ++q) {
            mbar_init(&tq_full[q], 1);
            mbar_init(&tq_empty[q], 1 + 4 + BS_OPW);
        }
        mbar_init(&done_bar, 1);
        fence_mbar_init_cluster();
        s_abort = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(BS_TMEM)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const uint32_t smem0 = (smem_u32(bs_smem) + 1023u) & ~1023u;
    auto give_up = [&]() {
        atomicOr(a.status, ST_TIMEOUT);
        atomicExch(a.ctl + 1, 1u);
        s_abort = 1;
    };
    // bounded wait of a whole warp; false: give up (every lane takes the same decision)
    auto wait = [&](uint64_t *bar, int parity) -> bool {
        const bool ok = mbar_wait_or_abort(bar, (uint32_t)(parity & 1), a.tries, &s_abort);
        if (__all_sync(0xffffffffu, ok)) return true;
        if (lane == 0) give_up();
        return false;
    };
    // next tile of the queue (i-th): its number, or -1 at the end or after a give-up
    auto next_tile = [&](int i) -> int {
        if (!wait(&tq_full[i % BS_QD], i / BS_QD)) return -1;
        const int t = tq[i % BS_QD];
        __syncwarp();
        if (lane == 0) mbar_arrive(&tq_empty[i % BS_QD]);
        return t;
    };

    if (warp == 1) {
        // ---- copy warp: takes tiles, fills the queue, streams the blocks' chunks
        int cc = 0;
        bool go = true;
        for (int i = 0; go; ++i) {
            int t = 0;
            if (lane == 0) {
                for (;;) {   // the tiles of a converged system are passed over
                    t = (int)atomicAdd(a.ctl, 1u);
                    if (t >= a.n_tile_total) { t = -1; break; }
                    if (!a.frozen || !a.frozen[2 * decode(a, t, NT).sys]) break;
                }
            }
            t = __shfl_sync(0xffffffffu, t, 0);
            if (i >= BS_QD && !wait(&tq_empty[i % BS_QD], i / BS_QD - 1)) break;
            if (lane == 0) {
                tq[i % BS_QD] = t;
                mbar_arrive(&tq_full[i % BS_QD]);
            }
            if (t < 0) break;
            const Tile tl = decode(a, t, NT);
            const int *task = a.tasks + 8 * tl.task;
            const int nterms = task[1] >> 4;
            const uint32_t bytes = (uint32_t)tl.rows * 128u;
            for (int u = 0; go && u < nterms; ++u) {
                const unsigned char *m = a.img + (size_t)bs_matrix(a, task[2 + 2 * u], tl.sys) * a.mat_bytes;
                for (int c = 0; c < a.n_chunk; ++c, ++cc) {
                    const int s = cc % ST;
                    if (cc >= ST && !wait(&empty[s], cc / ST - 1)) { go = false; break; }
                    if (lane == 0) {
                        const uint32_t dst = smem0 + (uint32_t)(s * Cfg::STAGE);
                        const unsigned char *src = m + ((size_t)(2 * c) * a.nzr + tl.r0) * 128;
                        mbar_arrive_expect_tx(&full_a[s], 2 * bytes);
                        bulk_load(dst, src, bytes, &full_a[s]);
                        bulk_load(dst + 16384, src + (size_t)a.nzr * 128, bytes, &full_a[s]);
                    }
                    __syncwarp();
                }
            }
        }
        // no copy may land after the CTA has left
        for (int c = max(0, cc - ST); c < cc; ++c) mbar_wait_bounded(&full_a[c % ST], (uint32_t)((c / ST) & 1), kDefaultWaitTries);
    } else if (warp == 0) {
        // ---- MMA warp
        int cc = 0, tt = 0;
        bool go = true;
        constexpr uint32_t id2 = idesc_f16(2 * NT, false), id1 = idesc_f16(NT, false), id1n = idesc_f16(NT, true);
        for (int i = 0; go; ++i) {
            const int t = next_tile(i);
            if (t < 0) break;
            const Tile tl = decode(a, t, NT);
            const int nterms = a.tasks[8 * tl.task + 1] >> 4;
            for (int u = 0; go && u < nterms; ++u, ++tt) {
                const int sl = tt % SL;
                if (tt >= SL && !wait(&acc_empty[sl], tt / SL - 1)) { go = false; break; }
                const uint32_t dre = tmem + (uint32_t)(sl * 2 * NT), dim = dre + NT;
                for (int c = 0; c < a.n_chunk; ++c, ++cc) {
                    const int s = cc % ST;
                    if (!wait(&full_a[s], cc / ST) || !wait(&full_b[s], cc / ST)) { go = false; break; }
                    tc_fence_after();
                    if (lane == 0) {
                        const uint32_t ar = smem0 + (uint32_t)(s * Cfg::STAGE), ai = ar + 16384, br = ar + BS_A,
                                       bi = br + (uint32_t)(NT * 128);
#pragma unroll
                        for (int p = 0; p < 3; ++p) {   // hi*hi, hi*lo, lo*hi (lo 64 bytes into the row)
                            const uint32_t oa = p == 2 ? 64u : 0u, ob = p == 1 ? 64u : 0u;
#pragma unroll
                            for (int kk = 0; kk < 2; ++kk) {   // K = 16 FP16 (32 bytes) per instruction
                                const uint32_t acc = (c > 0 || p > 0 || kk > 0) ? 1u : 0u;
                                const uint32_t ka = oa + 32 * kk, kb = ob + 32 * kk;
                                // [Re | Im] += Ar [Br | Bi];  Re -= Ai Bi;  Im += Ai Br
                                tc_mma_f16(dre, desc_sw128(ar + ka), desc_sw128(br + kb), id2, acc);
                                tc_mma_f16(dre, desc_sw128(ai + ka), desc_sw128(bi + kb), id1n, 1u);
                                tc_mma_f16(dim, desc_sw128(ai + ka), desc_sw128(br + kb), id1, 1u);
                            }
                        }
                        tc_commit(&empty[s]);
                        if (c == a.n_chunk - 1) tc_commit(&acc_full[sl]);
                    }
                    __syncwarp();
                }
            }
        }
        if (lane == 0) tc_commit(&done_bar);   // every MMA issued
        __syncwarp();
        mbar_wait_bounded(&done_bar, 0, kDefaultWaitTries);
    } else if (warp >= BS_OP0) {
        // ---- operand warps: lane half h of row pair i holds right-hand side row(i, h), complex
        // columns 2 j, 2 j + 1 of the chunk (j = lane & 15); rows 4 apart keep the 4-byte stores of
        // the two halves on distinct banks
        const int ow = warp - BS_OP0, h = lane >> 4, j = lane & 15;
        const size_t N = (size_t)a.N;
        int cc = 0, tt = 0, seen = -1;
        bool go = true;
        for (int i = 0; go; ++i) {
            const int t = next_tile(i);
            if (t < 0) break;
            const Tile tl = decode(a, t, NT);
            const int *task = a.tasks + 8 * tl.task;
            const int type = task[1] & 15, nterms = task[1] >> 4;
            // the previous step of this system
            const int key = tl.phase * a.ns + tl.sys;
            if (tl.phase > 0 && key != seen) {
                const unsigned *cnt = a.ctl + 2 + (key - a.ns);
                const unsigned want = (unsigned)a.ph[tl.phase - 1].done;
                bool ok = false;
                for (uint32_t q = 0; q < a.tries; ++q) {
                    if (ld_acquire(cnt) >= want) { ok = true; break; }
                    if (*(volatile int *)&s_abort || ((q & 63) == 63 && ld_acquire(a.ctl + 1))) break;
                    __nanosleep(40);
                }
                if (!__all_sync(0xffffffffu, ok)) {
                    if (lane == 0) give_up();
                    break;
                }
                seen = key;
            }
            int rowi[Cfg::PAIRS];
            bool val[Cfg::PAIRS];
            size_t off[Cfg::PAIRS];
#pragma unroll
            for (int q = 0; q < Cfg::PAIRS; ++q) {
                const int p = ow * Cfg::PAIRS + q;
                rowi[q] = 8 * (p >> 2) + (p & 3) + 4 * h;
                val[q] = tl.n0 + rowi[q] < a.nrhs;
                off[q] = ((size_t)tl.sys * a.nrhs + (val[q] ? tl.n0 + rowi[q] : 0)) * N;
            }
            for (int u = 0; go && u < nterms; ++u, ++tt) {
                const int bl = task[3 + 2 * u], sl = tt % SL;
                const bool is_x = bs_kind(task[2 + 2 * u]) >= BS_P;
                const float2 *vec = is_x ? a.x : a.r;
                // type 4 (level 0, backward): r_j - C (x_{j-1} + x_{j+1})
                const bool l0b = type == BS_BWD0, two = l0b && bl + 1 < a.nx;
                const float *gm = is_x ? a.gx : a.gr;
                auto load1 = [&](const float2 *p, int k) -> float4 {   // entries k, k + 1 of a line slice
                    if constexpr (EVEN) return __ldcg(reinterpret_cast<const float4 *>(p + k));
                    const float2 v0 = __ldcg(p + k), v1 = k + 1 < a.nz ? __ldcg(p + k + 1) : make_float2(0.f, 0.f);
                    return make_float4(v0.x, v0.y, v1.x, v1.y);
                };
                float4 nb[Cfg::PAIRS], na[Cfg::PAIRS], nc[Cfg::PAIRS];
                auto fetch = [&](int c) {
                    const int k = 32 * c + 2 * j;
#pragma unroll
                    for (int q = 0; q < Cfg::PAIRS; ++q) {
                        const bool in = val[q] && k < a.nz;
                        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
                        nb[q] = in ? load1(vec + off[q] + (size_t)bl * a.nz, k) : z;
                        if (l0b) {
                            na[q] = in ? load1(a.x + off[q] + (size_t)(bl - 1) * a.nz, k) : z;
                            nc[q] = in && two ? load1(a.x + off[q] + (size_t)(bl + 1) * a.nz, k) : z;
                        }
                    }
                };
                fetch(0);
                // the slice's maximum (a bound of it on level 0, backward) and its scale
                float sc[Cfg::PAIRS];
                if (tt >= SL && !wait(&acc_empty[sl], tt / SL - 1)) { go = false; break; }
#pragma unroll
                for (int q = 0; q < Cfg::PAIRS; ++q) {
                    auto line_max = [&](const float *g, int line) -> uint32_t {
                        uint32_t mx = 0;
                        for (int e = j; e < a.ng; e += 16)
                            if (val[q])
                                mx = max(mx, __float_as_uint(__ldcg(g + (((size_t)tl.sys * a.nx + line) * a.ng + e) * a.nrhs +
                                                                      tl.n0 + rowi[q])));
                        return mx;
                    };
                    uint32_t mx = line_max(gm, bl);
                    if (l0b) {
                        uint32_t ma = line_max(a.gx, bl - 1), mc = two ? line_max(a.gx, bl + 1) : 0u;
                        for (int o = 8; o > 0; o >>= 1) {
                            ma = max(ma, __shfl_xor_sync(0xffffffffu, ma, o));
                            mc = max(mc, __shfl_xor_sync(0xffffffffu, mc, o));
                        }
                        for (int o = 8; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                        mx = abs_bits(__uint_as_float(mx) +
                                      fabsf(a.cx_in) * (__uint_as_float(ma) + __uint_as_float(mc)));
                    } else {
                        for (int o = 8; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                    }
                    const int sh = scale_shift(mx);
                    sc[q] = pow2(sh);
                    if (j == 0) s_bscale[sl][rowi[q]] = pow2(-sh);
                }
                for (int c = 0; c < a.n_chunk; ++c, ++cc) {
                    const int s = cc % ST, k = 32 * c + 2 * j;
                    float4 v[Cfg::PAIRS];
#pragma unroll
                    for (int q = 0; q < Cfg::PAIRS; ++q) {
                        v[q] = nb[q];
                        if (l0b) {
                            const float c0 = (k == 0 || k == a.nz - 1) ? a.cx_edge : a.cx_in;
                            const float c1 = k + 1 == a.nz - 1 ? a.cx_edge : a.cx_in;
                            v[q].x -= c0 * (na[q].x + nc[q].x);
                            v[q].y -= c0 * (na[q].y + nc[q].y);
                            v[q].z -= c1 * (na[q].z + nc[q].z);
                            v[q].w -= c1 * (na[q].w + nc[q].w);
                        }
                    }
                    if (c + 1 < a.n_chunk) fetch(c + 1);
                    if (cc >= ST && !wait(&empty[s], cc / ST - 1)) { go = false; break; }
                    const uint32_t br = smem0 + (uint32_t)(s * Cfg::STAGE + BS_A), bi = br + (uint32_t)(NT * 128);
#pragma unroll
                    for (int q = 0; q < Cfg::PAIRS; ++q) {
                        uint32_t hi, lo;
                        const int r = rowi[q];
                        const uint32_t in16 = (uint32_t)(j & 3) * 4;
                        const uint32_t oh = sw128(r, j >> 2) + in16, ol = sw128(r, 4 + (j >> 2)) + in16;
                        split_h2(v[q].x * sc[q], v[q].z * sc[q], hi, lo);
                        asm volatile("st.shared.b32 [%0], %1;" ::"r"(br + oh), "r"(hi) : "memory");
                        asm volatile("st.shared.b32 [%0], %1;" ::"r"(br + ol), "r"(lo) : "memory");
                        split_h2(v[q].y * sc[q], v[q].w * sc[q], hi, lo);
                        asm volatile("st.shared.b32 [%0], %1;" ::"r"(bi + oh), "r"(hi) : "memory");
                        asm volatile("st.shared.b32 [%0], %1;" ::"r"(bi + ol), "r"(lo) : "memory");
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&full_b[s]);
                }
            }
        }
    } else {
        // ---- epilogue warps: tensor-memory lanes 32 q .. + 31 = rows r0 + 32 q + lane of the line
        const int q = warp & 3;
        const size_t N = (size_t)a.N;
        int tt = 0;
        bool go = true;
        for (int i = 0; go; ++i) {
            const int t = next_tile(i);
            if (t < 0) break;
            const Tile tl = decode(a, t, NT);
            const int *task = a.tasks + 8 * tl.task;
            const int line = task[0], type = task[1] & 15, nterms = task[1] >> 4;
            const int row = 32 * q + lane, m = tl.r0 + row;
            const bool on = row < tl.rows && m < a.nz, warp_on = 32 * q < tl.rows;
            const bool to_r = type <= BS_FWD;
            float2 *vec = to_r ? a.r : a.x;
            float *gm = to_r ? a.gr : a.gx;
            float f[3] = {0.f, 0.f, 0.f};   // row scale and sign of each term
            if (on)
                for (int u = 0; u < nterms; ++u) {
                    f[u] = __ldg(a.scl + (size_t)bs_matrix(a, task[2 + 2 * u], tl.sys) * a.nz + m);
                    if (type == BS_FWD0) f[u] *= -((m == 0 || m == a.nz - 1) ? a.cx_edge : a.cx_in);
                    if (type == BS_FWD || (type == BS_BWD && u > 0)) f[u] = -f[u];
                }
            for (int u = 0; u < nterms && go; ++u) go = wait(&acc_full[(tt + u) % SL], (tt + u) / SL);
            if (!go) break;
            tc_fence_after();
            float2 *out = vec + ((size_t)tl.sys * a.nrhs + tl.n0) * N + (size_t)line * a.nz + m;
            float *gout = gm + (((size_t)tl.sys * a.nx + line) * a.ng + (tl.r0 >> 5) + q) * a.nrhs + tl.n0;
            const int ncol = min(NT, a.nrhs - tl.n0);
            if (warp_on) {
                for (int c0 = 0; c0 < ncol; c0 += 16) {
                    float2 o[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        o[e] = on && to_r && c0 + e < ncol ? __ldcg(out + (size_t)(c0 + e) * N) : make_float2(0.f, 0.f);
                    for (int u = 0; u < nterms; ++u) {
                        const int sl = (tt + u) % SL;
                        const uint32_t d = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(sl * 2 * NT + c0);
                        float re[16], im[16];
                        tc_ld16(d, re);
                        tc_ld16(d + NT, im);
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            const float sb = s_bscale[sl][c0 + e];
                            o[e].x += (re[e] * f[u]) * sb;
                            o[e].y += (im[e] * f[u]) * sb;
                        }
                    }
                    uint32_t gmax = 0;
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        if (on && c0 + e < ncol) out[(size_t)(c0 + e) * N] = o[e];
                        const uint32_t b = on ? max(abs_bits(o[e].x), abs_bits(o[e].y)) : 0u;
                        const uint32_t w = __reduce_max_sync(0xffffffffu, b);
                        if (lane == e) gmax = w;
                    }
                    if (lane < 16 && c0 + lane < ncol) gout[c0 + lane] = __uint_as_float(gmax);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                for (int u = 0; u < nterms; ++u) mbar_arrive(&acc_empty[(tt + u) % SL]);
                __threadfence();   // the warp's stores before its count
                atomicAdd(a.ctl + 2 + tl.phase * a.ns + tl.sys, 1u);
            }
            tt += nterms;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(BS_TMEM) : "memory");
}

// maxima of the real and imaginary parts of every 32-row group of every line of v:
// g[((sys * nx + line) * ng + group) * nrhs + column]; a warp per (line group, 32 columns)
__global__ void __launch_bounds__(256) line_max_kernel(int nx, int nz, int ng, int nrhs, int n_cb, long long n_items,
                                                       const float2 *v, float *g, const int *skip, const int *frozen) {
    if (skip && *skip) return;
    const int lane = threadIdx.x & 31;
    const long long it = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (it >= n_items) return;
    const int cb = (int)(it % n_cb);
    const long long lg = it / n_cb;
    const int grp = (int)(lg % ng), line = (int)(lg / ng % nx), sys = (int)(lg / ng / nx);
    if (frozen && frozen[2 * sys]) return;
    const int k = 32 * grp + lane, c0 = 32 * cb, nc = min(32, nrhs - c0);
    const float2 *p = v + ((size_t)sys * nrhs + c0) * nx * nz + (size_t)line * nz + k;
    uint32_t mine = 0;
    for (int b = 0; b < nc; b += 8) {
        float2 t[8];
#pragma unroll
        for (int e = 0; e < 8; ++e)
            t[e] = k < nz && b + e < nc ? __ldg(p + (size_t)(b + e) * nx * nz) : make_float2(0.f, 0.f);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const uint32_t w = __reduce_max_sync(0xffffffffu, max(abs_bits(t[e].x), abs_bits(t[e].y)));
            if (lane == b + e) mine = w;
        }
    }
    if (lane < nc) g[(((size_t)sys * nx + line) * ng + grp) * nrhs + c0 + lane] = __uint_as_float(mine);
}

// Image of 32 rows of a block: dst matrix pairs[2 t + 1] from src block pairs[2 t] (n x n row-major,
// transposed if trans), rows 32 blockIdx.x ..; two passes over the rows (their maxima, then the
// split), the second from L2.  Columns beyond n are zero.
__global__ void __launch_bounds__(256) bcr_image_kernel(int n, int n_chunk, int nzr, const float2 *src, long long stride,
                                                        int trans, const int *pairs, unsigned char *img, size_t mat_bytes,
                                                        float *scl) {
    __shared__ float2 t[32][33];
    __shared__ float s_scale[32];
    const int *pr = pairs + 2 * (size_t)blockIdx.y;
    const float2 *A = src + (long long)pr[0] * stride;
    const int r0 = 32 * blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    auto entry = [&](int r, int k) -> float2 {   // (r, k) of the image's block, 0 beyond it
        if (r >= n || k >= n) return make_float2(0.f, 0.f);
        return __ldg(trans ? A + (long long)k * n + r : A + (long long)r * n + k);
    };
    // (loads run along the source's rows: lanes over k, or over r if transposed)
    uint32_t mx[4] = {0, 0, 0, 0};
    for (int c = 0; c < n_chunk; ++c) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int o = w + 8 * q;
            const float2 v = trans ? entry(r0 + lane, 32 * c + o) : entry(r0 + o, 32 * c + lane);
            mx[q] = max(mx[q], max(abs_bits(v.x), abs_bits(v.y)));
        }
    }
    if (trans) {   // lane = row: over the warps' k
        uint32_t m = max(max(mx[0], mx[1]), max(mx[2], mx[3]));
        uint32_t *sm = reinterpret_cast<uint32_t *>(&t[0][0]);
        sm[w * 32 + lane] = m;
        __syncthreads();
        if (w == 0) {
            for (int e = 1; e < 8; ++e) m = max(m, sm[e * 32 + lane]);
            const int sh = scale_shift(m);
            s_scale[lane] = pow2(sh);
            if (r0 + lane < n) scl[(size_t)pr[1] * n + r0 + lane] = pow2(-sh);
        }
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int sh = scale_shift(__reduce_max_sync(0xffffffffu, mx[q])), o = w + 8 * q;
            if (lane == 0) {
                s_scale[o] = pow2(sh);
                if (r0 + o < n) scl[(size_t)pr[1] * n + r0 + o] = pow2(-sh);
            }
        }
    }
    __syncthreads();
    unsigned char *M = img + (size_t)pr[1] * mat_bytes;
    const int row = threadIdx.x >> 3, j = threadIdx.x & 7, kb = 8 * (j & 3);
    for (int c = 0; c < n_chunk; ++c) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int o = w + 8 * q;
            if (trans) t[lane][o] = entry(r0 + lane, 32 * c + o);
            else t[o][lane] = entry(r0 + o, 32 * c + lane);
        }
        __syncthreads();
        if (r0 + row < nzr) {
            const float sc = s_scale[row];
            uint4 re, im;
            uint32_t *pre = reinterpret_cast<uint32_t *>(&re), *pim = reinterpret_cast<uint32_t *>(&im);
#pragma unroll
            for (int e = 0; e < 4; ++e) {   // 16-byte piece j: hi of columns kb .. kb + 7 (j < 4), else lo
                const float2 v0 = t[row][kb + 2 * e], v1 = t[row][kb + 2 * e + 1];
                uint32_t hi, lo;
                split_h2(v0.x * sc, v1.x * sc, hi, lo);
                pre[e] = j < 4 ? hi : lo;
                split_h2(v0.y * sc, v1.y * sc, hi, lo);
                pim[e] = j < 4 ? hi : lo;
            }
            unsigned char *d = M + ((size_t)(2 * c) * nzr + r0 + row) * 128 + ((j ^ (row & 7)) << 4);
            *reinterpret_cast<uint4 *>(d) = re;
            *reinterpret_cast<uint4 *>(d + (size_t)nzr * 128) = im;
        }
        __syncthreads();
    }
}

template <int NT, bool EVEN> cudaError_t launch_nt(const BsArgs &a, int grid, double flops, cudaStream_t st) {
    const void *fn = (const void *)bcr_solve_kernel<NT, EVEN>;
    cudaError_t e = ensure_dyn_smem(fn, BsCfg<NT>::SMEM);
    if (e != cudaSuccess) return e;
    HELM_TRACED_W(K_BCR_SOLVE, st, flops, (bcr_solve_kernel<NT, EVEN><<<grid, BS_THREADS, BsCfg<NT>::SMEM, st>>>(a)));
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_bcr_image(int n, const float2 *src, long long stride, bool trans, const int *pairs_dev, int count,
                             unsigned char *img, float *scl, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    const BsLayout l = bs_layout(n);
    for (int t = 0; t < count; t += 65535) {
        const int nb = std::min(65535, count - t);
        HELM_TRACED(K_BCR_IMAGE, st, (bcr_image_kernel<<<dim3((n + 31) / 32, nb), 256, 0, st>>>(
                                         n, l.n_chunk, l.nzr, src, stride, trans ? 1 : 0, pairs_dev + 2 * (size_t)t, img,
                                         l.mat_bytes, scl)));
    }
    return cudaGetLastError();
}

cudaError_t launch_bcr_solve(BsArgs a, const BsStep *steps, int n_steps, double flops, cudaStream_t st) {
    if (n_steps > BS_MAX_PHASE) return cudaErrorInvalidValue;
    const BsLayout l = bs_layout(a.nz);
    a.nzr = l.nzr;
    a.n_chunk = l.n_chunk;
    a.mat_bytes = l.mat_bytes;
    a.ng = l.ng;
    a.N = a.nx * a.nz;
    const int nt = a.nrhs <= 16 ? 16 : (a.nrhs <= 32 ? 32 : 64);
    a.n_tiles = (a.nrhs + nt - 1) / nt;
    const int sms = device_sms();
    a.n_phase = n_steps;
    int tile = 0;
    for (int p = 0; p < n_steps; ++p) {
        BsPhase &ph = a.ph[p];
        ph.tile0 = tile;
        ph.task0 = steps[p].task0;
        ph.tasks = steps[p].tasks;
        // steps with few lines take lower tiles, so that more SMs share the blocks' stream
        ph.mrows = 128;
        auto tiles_of = [&](int rows) { return ph.tasks * a.ns * a.n_tiles * ((a.nz + rows - 1) / rows); };
        while (ph.mrows > 32 && tiles_of(ph.mrows) < sms) ph.mrows /= 2;
        ph.mt = (a.nz + ph.mrows - 1) / ph.mrows;
        ph.done = 4 * ph.tasks * a.n_tiles * ph.mt;   // four epilogue warps count each tile
        tile += tiles_of(ph.mrows);
    }
    a.n_tile_total = tile;
    cudaError_t e = cudaMemsetAsync(a.ctl, 0, sizeof(unsigned) * bs_ctl_words(n_steps, a.ns), st);
    if (e != cudaSuccess) return e;
    const int n_cb = (a.nrhs + 31) / 32;
    const long long items = (long long)a.ns * a.nx * a.ng * n_cb;
    HELM_TRACED(K_LINEMAX, st, (line_max_kernel<<<(unsigned)((items + 7) / 8), 256, 0, st>>>(
                                   a.nx, a.nz, a.ng, a.nrhs, n_cb, items, a.r, a.gr, a.skip, a.frozen)));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int grid = std::min(sms, tile);
    const bool even = (a.nz & 1) == 0;
    if (nt == 16) return even ? launch_nt<16, true>(a, grid, flops, st) : launch_nt<16, false>(a, grid, flops, st);
    if (nt == 32) return even ? launch_nt<32, true>(a, grid, flops, st) : launch_nt<32, false>(a, grid, flops, st);
    return even ? launch_nt<64, true>(a, grid, flops, st) : launch_nt<64, false>(a, grid, flops, st);
}

}  // namespace helm
