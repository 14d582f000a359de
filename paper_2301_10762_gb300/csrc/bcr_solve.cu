// The solve of a block-cyclic-reduction factor (bcr.cu) as one persistent tensor-core kernel.
//
// Every step of the substitution is a sum of products of a stored n_z x n_z block with a line of
// the right-hand sides of a system (bcr.cu's header; C = diag(cx) the level-0 coupling):
//     level 0, forward    r_k -= C (Dinv_{k-1} r_{k-1} + Dinv_{k+1} r_{k+1})       k even
//     level l, forward    r_k -= W_a r_a + V_c r_c                                 k = 0 mod 2s
//     last line           x_0 = Dinv_0 r_0
//     level l, backward   x_j = Dinv_j r_j - P_j x_{j-s} - Q_j x_{j+s}             j = s mod 2s
//     level 0, backward   x_j = Dinv_j (r_j - C (x_{j-1} + x_{j+1}))               j odd
// The blocks are read once per solve (the odd lines' inverses twice) and nothing else comes close in
// bytes (3.5 n_x n_z^2 complex entries of 8 bytes per frequency: 3.8 GB at 256^2 with 8 frequencies,
// 0.56 ms at the measured copy rate), so the kernel is laid out as a stream of the blocks through the tensor cores:
//   * The blocks are stored as the tensor core reads them ("image"): every real entry as the sum
//     of two FP16 numbers of its scaled value (a power of two per block; hi + lo carry 22 to 23
//     bits for entries down to 2^-15 of the block's largest, as many as the 3xTF32 split keeps, and
//     2^-39 of the largest below that; 8 bytes per complex entry as in FP32), real and imaginary
//     parts apart, 32 columns of a row as one 128-byte swizzled row (32 hi, then 32 lo).  A chunk of a tile is two contiguous runs of memory: a copy warp streams
//     them with bulk copies, and no thread touches them.
//   * The vectors are split by operand warps as they come (a power-of-two scale per line slice
//     from the maxima that the writers of the vectors leave), 16 KB against 32 KB of block data
//     per chunk at 64 right-hand sides.
//   * One thread issues hi hi + hi lo + lo hi of Ar [Br | Bi] and Ai [Br | Bi], FP32 accumulation in
//     tensor memory; four epilogue warps combine and scale them, add the old line and write,
//     while the next tile's products run into the other accumulator.
//   * The tiles of all levels are taken in order from a device counter by whichever CTA is free.
//     A tile waits until the previous step of its own system is complete (a counter per step and
//     system); only the operand warps wait, so the block stream runs on across steps.  Every
//     wait is for tiles that were taken earlier, so the kernel needs no co-resident grid, and
//     every wait is bounded.
// Measured per solve at 256^2, 8 frequencies (block stream 0.56 ms): 1 right-hand side 0.61 ms, 64
// of them 1.12 ms (vectors and products restart at every tile); one GEMM launch per level (18
// launches, 3xTF32, blocks split by operand warps) took 1.9 and 2.4 ms.  With few systems the chain
// of 2 log2(n_x) + 1 steps is what is left, 6 to 17 us a step: 0.12 ms at 128^2.
#include <algorithm>

#include "abi_internal.h"
#include "bcr_image.cuh"
#include "bcr_solve.h"
#include "kernels.h"
#include "tcgen05.cuh"
#include "trace.h"

namespace helm {

namespace {

constexpr int BS_WARPS = 14;                 // MMA, copy, 4 epilogue, 8 operand warps
constexpr int BS_THREADS = 32 * BS_WARPS;
constexpr int BS_OP0 = 6, BS_OPW = 8;        // (epilogue warps 2 .. 5)
constexpr int BS_QD = 4;                     // tile queue of a CTA
constexpr int BS_A = 32768;                  // A bytes of a stage: 128 rows x 128 bytes, Re and Im
constexpr uint32_t BS_TMEM = 512;

constexpr int BS_SLOTS = 2, BS_SLOT_COLS = 256;   // accumulators: one per tile, [Ar Br | Ar Bi | Ai Br | Ai Bi]

// NT: widest tile of the launch (right-hand sides); a step with few lines takes narrower ones
template <int NT> struct BsCfg {
    static constexpr int B = NT * 256;                   // B bytes of a stage: NT rows x 128 bytes, Re and Im
    static constexpr int STAGE = BS_A + B;
    static constexpr int STAGES = NT == 16 ? 5 : 3;
    static constexpr int PAIRS = NT / 16;                // row pairs of a chunk per operand warp
    // raw vector chunks on their way (NT rows x 256 bytes each): five, or three of three vectors in
    // the last step, which takes tiles of at most 32 right-hand sides
    static constexpr int RAW = NT == 64 ? 5 * B : 9 * B;
    static constexpr size_t SMEM = (size_t)STAGES * STAGE + RAW + 1024;
};
constexpr int BS_AHEAD = 4, BS_AHEAD0 = 2;   // vector chunks in flight ahead of the one being split
constexpr int BS_NT_BWD0 = 32;

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
struct BsQ {   // a queue entry: the tile, its task and the shifts of the task's blocks, read ahead by the copy thread
    int t, task[8], sa[3];
};
struct Tile {
    int phase, sys, task, n0, r0, rows, nt;
};
__device__ __forceinline__ Tile decode(const BsArgs &a, int t) {
    int p = 0;
    while (p + 1 < a.n_phase && t >= a.ph[p + 1].tile0) ++p;
    const BsPhase &ph = a.ph[p];
    int q = t - ph.tile0;
    Tile o;
    o.phase = p;
    o.nt = ph.nt;
    o.r0 = (q % ph.mt) * ph.mrows;
    q /= ph.mt;
    o.n0 = (q % ph.n_tiles) * ph.nt;
    q /= ph.n_tiles;
    o.sys = q / ph.tasks;
    o.task = ph.task0 + q % ph.tasks;
    o.rows = min(ph.mrows, a.nzr - o.r0);
    return o;
}

// 16 bytes global -> shared through L2 (zeros if !in), asynchronous
__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void *src, bool in) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ float4 ld_shared4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr)
                 : "memory");
    return v;
}

template <int NT>
__global__ void __launch_bounds__(BS_THREADS, 1) bcr_solve_kernel(const __grid_constant__ BsArgs a) {
    using Cfg = BsCfg<NT>;
    constexpr int ST = Cfg::STAGES, SL = BS_SLOTS, PR = Cfg::PAIRS;
    extern __shared__ uint8_t bs_smem[];
    __shared__ __align__(8) uint64_t full[ST], empty[ST];   // a stage written (the copy warp's bytes and the operand warps), read by its MMAs
    __shared__ __align__(8) uint64_t acc_full[SL], acc_empty[SL];
    __shared__ __align__(8) uint64_t tq_full[BS_QD], tq_empty[BS_QD], done_bar;
    __shared__ BsQ tq[BS_QD];
    __shared__ float s_bscale[SL][NT];   // 2^-S of each right-hand side of an accumulator
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    if (a.skip && *a.skip) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(&full[s], 1 + BS_OPW);
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
        bool ok = a.tries > 0 && mbar_test_cta(bar, (uint32_t)(parity & 1));
        if (__all_sync(0xffffffffu, ok)) return true;
        ok = mbar_wait_cta(bar, (uint32_t)(parity & 1), a.tries, &s_abort);
        if (__all_sync(0xffffffffu, ok)) return true;
        if (lane == 0) give_up();
        return false;
    };
    // the same for one thread on its own
    auto wait1 = [&](uint64_t *bar, uint32_t parity) -> bool {
        if (mbar_wait_cta(bar, parity, a.tries, &s_abort)) return true;
        give_up();
        return false;
    };
    // next tile of the queue (i-th): its number, or -1 at the end or after a give-up
    auto next_tile = [&](int i, BsQ &e) -> int {
        if (!wait(&tq_full[i % BS_QD], i / BS_QD)) return -1;
        e = tq[i % BS_QD];
        __syncwarp();
        if (lane == 0) mbar_arrive_cta(&tq_empty[i % BS_QD]);
        return e.t;
    };

    // the step before tile tl's of the same system is complete (seen: the last one found complete)
    auto step_wait = [&](const Tile &tl, int &seen) -> bool {
        const int key = tl.phase * a.ns + tl.sys;
        if (tl.phase == 0 || key == seen) return true;
        const unsigned *cnt = a.ctl + 2 + (key - a.ns);
        const unsigned want = (unsigned)a.ph[tl.phase - 1].done;
        bool ok = false;
        for (uint32_t q = 0; q < a.tries; ++q) {
            if (ld_acquire(cnt) >= want) { ok = true; break; }
            if (*(volatile int *)&s_abort || ((q & 63) == 63 && ld_acquire(a.ctl + 1))) break;
            __nanosleep(20);
        }
        if (!__all_sync(0xffffffffu, ok)) {
            if (lane == 0) give_up();
            return false;
        }
        seen = key;
        return true;
    };

    if (warp == 1) {
        // ---- copy warp (one thread): takes tiles, fills the queue, streams the blocks' chunks
        if (elect_one()) {
            int cs = 0, issued = 0;
            uint32_t cph = 1;   // parity of the stage's previous release (the first round passes at once)
            bool go = true;
            // the next tile: its ticket, its task and its blocks' shifts, one access after the other and two
            // chunks of the present tile apart (together they take 2 to 3 us)
            BsQ ne;
            Tile ntl{};
            int4 a0, a1;
            int part = 0, frozen = 0;
            auto advance = [&]() {
                if (part == 0) {
                    ne.t = (int)atomicAdd(a.ctl, 1u);
                } else if (part == 1) {
                    if (ne.t >= a.n_tile_total) ne.t = -1;
                    if (ne.t >= 0) {
                        ntl = decode(a, ne.t);
                        a0 = __ldg(reinterpret_cast<const int4 *>(a.tasks + 8 * ntl.task));
                        a1 = __ldg(reinterpret_cast<const int4 *>(a.tasks + 8 * ntl.task) + 1);
                        frozen = a.frozen ? a.frozen[2 * ntl.sys] : 0;
                    }
                } else if (ne.t >= 0) {
                    ne.task[0] = a0.x; ne.task[1] = a0.y; ne.task[2] = a0.z; ne.task[3] = a0.w;
                    ne.task[4] = a1.x; ne.task[5] = a1.y; ne.task[6] = a1.z; ne.task[7] = a1.w;
#pragma unroll
                    for (int u = 0; u < 3; ++u)
                        ne.sa[u] = u < (ne.task[1] >> 4) ? __ldg(a.shift + bs_matrix(a, ne.task[2 + 2 * u], ntl.sys)) : 0;
                }
                ++part;
            };
            for (int i = 0; go; ++i) {
                for (;;) {   // the tiles of a converged system are passed over
                    while (part < 3) advance();
                    if (ne.t < 0 || !frozen) break;
                    part = 0;
                }
                const BsQ e = ne;
                const Tile tl = ntl;
                const int *task = e.task;
                part = 0;
                if (!wait1(&tq_empty[i % BS_QD], (uint32_t)((i / BS_QD) & 1) ^ 1u)) break;
                tq[i % BS_QD] = e;
                mbar_arrive_cta(&tq_full[i % BS_QD]);
                if (e.t < 0) break;
                const int nterms = task[1] >> 4;
                // taking a ticket early keeps the stream of blocks going (256^2, 8 frequencies, 8 columns: 657 -> 614 us), but
                // binds a tile of the next step to this SM while others may be idle (the chain of a 128^2
                // system 117 -> 129 us): only in steps of four tiles an SM and more
                const BsPhase &ph = a.ph[tl.phase];
                const bool ahead = (long long)ph.tasks * a.ns * ph.n_tiles * ph.mt >= 4ll * gridDim.x;
                const uint32_t bytes = (uint32_t)tl.rows * 128u;
                const size_t im_off = (size_t)a.nzr * 128;
                for (int u = 0; go && u < nterms; ++u) {
                    const int code = u == 0 ? task[2] : (u == 1 ? task[4] : task[6]);
                    const unsigned char *src = a.img + (size_t)bs_matrix(a, code, tl.sys) * a.mat_bytes +
                                               (size_t)tl.r0 * 128;
                    for (int c = 0; c < a.n_chunk; ++c, src += 2 * im_off) {
                        if (!wait1(&empty[cs], cph)) { go = false; break; }
                        const uint32_t dst = smem0 + (uint32_t)(cs * Cfg::STAGE);
                        mbar_arrive_expect_tx(&full[cs], 2 * bytes);
                        bulk_load(dst, src, bytes, &full[cs]);
                        bulk_load(dst + 16384, src + im_off, bytes, &full[cs]);
                        ++issued;
                        if (++cs == ST) { cs = 0; cph ^= 1u; }
                        if (ahead && part < 3 && (issued & 1)) advance();
                    }
                }
            }
            // no copy may land after the CTA has left.  (A stage's barrier completes with the operand
            // warps' arrivals too, which an abort may leave out, also one that comes while this waits:
            // then a fixed time is waited)
            for (int c = max(0, issued - ST); c < issued; ++c)
                if (!mbar_wait_cta(&full[c % ST], (uint32_t)((c / ST) & 1), kDefaultWaitTries, &s_abort)) {
                    abort_drain();
                    break;
                }
        }
        __syncwarp();
    } else if (warp == 0) {
        // ---- MMA warp (one thread; its instruction stream paces the whole CTA: a warp-wide vote per
        // wait and two barriers per chunk cost 0.5 us a chunk)
        if (elect_one()) {
            int s = 0, sl = 0;
            uint32_t ph = 0, slph = 1;
            bool go = true;
            const uint64_t dstage0 = desc_sw128(smem0);
            for (int i = 0; go; ++i) {
                if (!wait1(&tq_full[i % BS_QD], (uint32_t)((i / BS_QD) & 1))) break;
                const int t = tq[i % BS_QD].t, nterms = tq[i % BS_QD].task[1] >> 4;
                mbar_arrive_cta(&tq_empty[i % BS_QD]);
                if (t < 0) break;
                const int nt = decode(a, t).nt;
                const uint32_t id = idesc_f16(2 * nt);
                if (!wait1(&acc_empty[sl], slph)) break;
                const uint32_t d0 = tmem + (uint32_t)(sl * BS_SLOT_COLS), d1 = d0 + (uint32_t)(2 * nt);
                for (int c = 0, n = nterms * a.n_chunk; c < n; ++c) {
                    if (!wait1(&full[s], ph)) { go = false; break; }
                    fence_proxy_async_smem();   // the operand warps' stores, ordered by the barrier
                    tc_fence_after();
                    const uint64_t dar = dstage0 + (uint64_t)(s * (Cfg::STAGE / 16)), dai = dar + 1024, dbr = dar + BS_A / 16;
                    // products hi*hi, hi*lo, lo*hi (lo 64 bytes into the row), each two steps of
                    // K = 16 FP16 (32 bytes; 2 in descriptor units): Ar [Br | Bi] and Ai [Br | Bi]
#pragma unroll
                    for (int p = 0; p < 6; ++p) {
                        const int ka = (p >= 4 ? 4 : 0) + 2 * (p & 1), kb = ((p >> 1) == 1 ? 4 : 0) + 2 * (p & 1);
                        const uint32_t acc = p > 0 ? 1u : (c > 0 ? 1u : 0u);
                        tc_mma_f16(d0, dar + ka, dbr + kb, id, acc);
                        tc_mma_f16(d1, dai + ka, dbr + kb, id, acc);
                    }
                    tc_commit(&empty[s]);
                    if (++s == ST) { s = 0; ph ^= 1u; }
                }
                if (go) tc_commit(&acc_full[sl]);
                if (++sl == SL) { sl = 0; slph ^= 1u; }
            }
            tc_commit(&done_bar);   // every MMA issued
            mbar_wait_bounded(&done_bar, 0, kDefaultWaitTries);
        }
        __syncwarp();
    } else if (warp >= BS_OP0) {
        // ---- operand warps: lane half h of row pair q holds right-hand side row0 + 16 q (row0 with
        // 4 h), complex columns 2 j, 2 j + 1 of the chunk (j = lane & 15); rows 4 apart keep the
        // 4-byte stores of the two halves on distinct banks.  The vectors come from L2 or HBM, 1 to
        // 3 us off: every lane copies its own 16 bytes per row into a raw slot asynchronously,
        // BS_AHEAD chunks ahead of the one it splits (loads into registers ran at one latency per
        // chunk whatever the number of sets: their scoreboards are shared)
        const int ow = warp - BS_OP0, h = lane >> 4, j = lane & 15;
        const size_t N = (size_t)a.N;
        const uint32_t raw0 = smem0 + (uint32_t)(ST * Cfg::STAGE);
        int cc = 0, tt = 0, seen = -1;
        bool go = true;
        for (int i = 0; go; ++i) {
            BsQ entry;
            const int t = next_tile(i, entry);
            if (t < 0) break;
            const Tile tl = decode(a, t);
            const int *task = entry.task;
            const int type = task[1] & 15, nterms = task[1] >> 4, np = tl.nt / 16;
            if (!step_wait(tl, seen)) break;
            const int row0 = 8 * (ow >> 2) + (ow & 3) + 4 * h;   // row of pair q: row0 + 16 q
            const float2 *r0p = a.r + ((size_t)tl.sys * a.nrhs + tl.n0 + row0) * N;
            const float2 *x0p = a.x + ((size_t)tl.sys * a.nrhs + tl.n0 + row0) * N;
            const int nval = a.nrhs - tl.n0 - row0;
            auto val = [&](int q) { return q < np && 16 * q < nval; };
            // largest entry of a line of the warp's rows (from the maxima its writer left); the loads of
            // all terms are issued before the first is used
            auto line_max = [&](const float *g, int bl, int q) -> uint32_t {
                const float *p = g + ((size_t)tl.sys * a.nx + bl) * a.ng * a.nrhs + tl.n0 + row0 + 16 * q;
                uint32_t mx = j < a.ng && val(q) ? __float_as_uint(__ldcg(p + (size_t)j * a.nrhs)) : 0u;
                if (a.ng > 16)
                    for (int e = j + 16; e < a.ng; e += 16)
                        if (val(q)) mx = max(mx, __float_as_uint(__ldcg(p + (size_t)e * a.nrhs)));
                return mx;
            };
            auto over_lanes = [&](uint32_t m) {
                for (int o = 8; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
                return m;
            };
            // terms share the tile's accumulator, so their scales share one exponent S per right-hand
            // side: S = min over the terms of (the block's shift + the line's largest shift), and a
            // line's shift is S less its block's.  A term that is small against the largest loses
            // only what the sum does not hold (FP16 keeps all 22 bits 15 octaves down).  S ends at 126,
            // whose 2^-S is the smallest normal number: small lines times blocks of small entries
            // (far from square cells) keep fewer bits there instead of a wrong scale.
            float sc[PR];
            auto put_scale = [&](int q, int S, int sl) {
                if (j == 0 && q < np) s_bscale[sl][row0 + 16 * q] = bs_pow2(max(-126, -S));
            };
            const int sl = tt % SL;
            // split and store one chunk's pairs into stage s
            auto put = [&](int s, const float4 (&v)[PR]) {
                const uint32_t br = smem0 + (uint32_t)(s * Cfg::STAGE + BS_A), bi = br + (uint32_t)(tl.nt * 128);
#pragma unroll
                for (int q = 0; q < PR; ++q) {
                    if (q < np) {
                        uint32_t hi, lo;
                        const int r = row0 + 16 * q;
                        const uint32_t in16 = (uint32_t)(j & 3) * 4;
                        const uint32_t oh = sw128(r, j >> 2) + in16, ol = sw128(r, 4 + (j >> 2)) + in16;
                        bs_split2(v[q].x * sc[q], v[q].z * sc[q], hi, lo);
                        asm volatile("st.shared.b32 [%0], %1;" ::"r"(br + oh), "r"(hi) : "memory");
                        asm volatile("st.shared.b32 [%0], %1;" ::"r"(br + ol), "r"(lo) : "memory");
                        bs_split2(v[q].y * sc[q], v[q].w * sc[q], hi, lo);
                        asm volatile("st.shared.b32 [%0], %1;" ::"r"(bi + oh), "r"(hi) : "memory");
                        asm volatile("st.shared.b32 [%0], %1;" ::"r"(bi + ol), "r"(lo) : "memory");
                    }
                }
                // (the fence that makes these stores visible to the tensor core stands in the MMA
                // warp: here it would also wait for every load the warp has in flight)
                __syncwarp();
                if (lane == 0) mbar_arrive_cta(&full[s]);
            };
            // this lane's 16 bytes of row pair q in raw slot e
            auto raw = [&](int e, int q) { return raw0 + (uint32_t)((e * tl.nt + row0 + 16 * q) * 256 + 16 * j); };
            // copy chunk c of a line (base: its entry of this warp's first row) into raw slot e
            auto fetch = [&](int e, const float2 *base, int c, bool on) {
                const int k = 32 * c + 2 * j;
#pragma unroll
                for (int q = 0; q < PR; ++q) {
                    if (q < np) {
                        const bool in = on && val(q) && k < a.nz;
                        cp_async16_zfill(raw(e, q), in ? base + (size_t)(16 * q) * N + k : a.r, in);
                    }
                }
            };
            if (type == BS_BWD0) {
                // level 0, backward: v = r_j - C (x_{j-1} + x_{j+1}); its maximum is bounded by the parts'
                const int bl = task[3], sa = entry.sa[0];
                const bool two = bl + 1 < a.nx;
                const size_t lo = (size_t)bl * a.nz;
                auto fetch3 = [&](int c) {
                    if (c < a.n_chunk) {
                        const int e = 3 * (c % (BS_AHEAD0 + 1));
                        fetch(e, r0p + lo, c, true);
                        fetch(e + 1, x0p + lo - a.nz, c, true);
                        fetch(e + 2, x0p + lo + a.nz, c, two);
                    }
                    cp_async_commit();
                };
#pragma unroll
                for (int c = 0; c < BS_AHEAD0; ++c) fetch3(c);
                uint32_t m3[3][PR];
#pragma unroll
                for (int q = 0; q < PR; ++q) {
                    m3[0][q] = line_max(a.gr, bl, q);
                    m3[1][q] = line_max(a.gx, bl - 1, q);
                    m3[2][q] = two ? line_max(a.gx, bl + 1, q) : 0u;
                }
                if (tt >= SL && !wait(&acc_empty[sl], tt / SL - 1)) break;
#pragma unroll
                for (int q = 0; q < PR; ++q) {
                    const float bound = __uint_as_float(over_lanes(m3[0][q])) +
                                        fabsf(a.cx_in) * (__uint_as_float(over_lanes(m3[1][q])) +
                                                          __uint_as_float(over_lanes(m3[2][q])));
                    const int sh = min(bs_scale_shift(bs_abs_bits(bound)), 126 - sa);
                    sc[q] = bs_pow2(sh);
                    put_scale(q, sh + sa, sl);
                }
                for (int c = 0; c < a.n_chunk; ++c, ++cc) {
                    const int s = cc % ST, k = 32 * c + 2 * j, e = 3 * (c % (BS_AHEAD0 + 1));
                    const float c0 = (k == 0 || k == a.edge) ? a.cx_edge : a.cx_in;
                    const float c1 = k + 1 == a.edge ? a.cx_edge : a.cx_in;
                    fetch3(c + BS_AHEAD0);
                    cp_async_wait<BS_AHEAD0>();
                    float4 v[PR];
#pragma unroll
                    for (int q = 0; q < PR; ++q) {
                        if (q < np) {
                            const float4 nb = ld_shared4(raw(e, q)), na = ld_shared4(raw(e + 1, q)), nc = ld_shared4(raw(e + 2, q));
                            v[q] = make_float4(nb.x - c0 * (na.x + nc.x), nb.y - c0 * (na.y + nc.y),
                                               nb.z - c1 * (na.z + nc.z), nb.w - c1 * (na.w + nc.w));
                        }
                    }
                    if (cc >= ST && !wait(&empty[s], cc / ST - 1)) { go = false; break; }
                    put(s, v);
                }
                ++tt;
                continue;
            }
            // the chunks of all terms as one sequence
            int fu = 0, fc = 0, fe = 0;
            const float2 *fv = r0p;
            auto fetch_next = [&]() {
                if (fu < nterms) {
                    if (fc == 0) {
                        const int code = fu == 0 ? task[2] : (fu == 1 ? task[4] : task[6]);
                        const int line = fu == 0 ? task[3] : (fu == 1 ? task[5] : task[7]);
                        fv = (bs_kind(code) >= BS_P ? x0p : r0p) + (size_t)line * a.nz;
                    }
                    fetch(fe, fv, fc, true);
                    if (++fc == a.n_chunk) { fc = 0; ++fu; }
                    if (++fe == BS_AHEAD + 1) fe = 0;
                }
                cp_async_commit();
            };
            for (int d = 0; d < BS_AHEAD; ++d) fetch_next();
            uint32_t mx[3][PR];
            const int *sa = entry.sa;
#pragma unroll
            for (int u = 0; u < 3; ++u) {
                const bool in = u < nterms;
#pragma unroll
                for (int q = 0; q < PR; ++q)
                    mx[u][q] = in && q < np
                                   ? line_max(bs_kind(task[2 + 2 * u]) >= BS_P ? a.gx : a.gr, task[3 + 2 * u], q)
                                   : 0u;
            }
            if (tt >= SL && !wait(&acc_empty[sl], tt / SL - 1)) break;
            int S[PR];
#pragma unroll
            for (int q = 0; q < PR; ++q) {
                S[q] = 126;
#pragma unroll
                for (int u = 0; u < 3; ++u) {
                    const int t2 = sa[u] + bs_scale_shift(over_lanes(mx[u][q]));
                    if (u < nterms) S[q] = min(S[q], t2);
                }
                put_scale(q, S[q], sl);
            }
            ++tt;
            int e = 0;
            for (int u = 0; go && u < nterms; ++u) {
                const int su = u == 0 ? sa[0] : (u == 1 ? sa[1] : sa[2]);
#pragma unroll
                for (int q = 0; q < PR; ++q) {   // P and Q enter with a minus sign
                    const float f = bs_pow2(max(-126, min(126, S[q] - su)));
                    sc[q] = type == BS_BWD && u > 0 ? -f : f;
                }
                for (int c = 0; c < a.n_chunk; ++c, ++cc) {
                    const int s = cc % ST;
                    fetch_next();
                    cp_async_wait<BS_AHEAD>();
                    float4 v[PR];
#pragma unroll
                    for (int q = 0; q < PR; ++q)
                        if (q < np) v[q] = ld_shared4(raw(e, q));
                    if (cc >= ST && !wait(&empty[s], cc / ST - 1)) { go = false; break; }
                    put(s, v);
                    if (++e == BS_AHEAD + 1) e = 0;
                }
            }
        }
        cp_async_wait<0>();
    } else {
        // ---- epilogue warps: tensor-memory lanes 32 q .. + 31 = rows r0 + 32 q + lane of the line
        const int q = warp & 3;
        const size_t N = (size_t)a.N;
        int tt = 0, seen = -1;
        bool go = true;
        for (int i = 0; go; ++i) {
            BsQ entry;
            const int t = next_tile(i, entry);
            if (t < 0) break;
            const Tile tl = decode(a, t);
            const int *task = entry.task;
            const int line = task[0], type = task[1] & 15, nt = tl.nt;
            const int row = 32 * q + lane, m = tl.r0 + row;
            const bool on = row < tl.rows && m < a.nz, warp_on = 32 * q < tl.rows;
            const bool to_r = type <= BS_FWD;
            float2 *vec = to_r ? a.r : a.x;
            float *gm = to_r ? a.gr : a.gx;
            // sign and (level 0, forward) the coupling of the row
            const float f = type == BS_FWD ? -1.f
                                           : (type == BS_FWD0 ? -((m == 0 || m == a.edge) ? a.cx_edge : a.cx_in) : 1.f);
            float2 *out = vec + ((size_t)tl.sys * a.nrhs + tl.n0) * N + (size_t)line * a.nz + m;
            float *gout = gm + (((size_t)tl.sys * a.nx + line) * a.ng + (tl.r0 >> 5) + q) * a.nrhs + tl.n0;
            const int ncol = min(nt, a.nrhs - tl.n0), sl = tt % SL;
            // the old line, ahead of the products that are added to it: four groups of 8 columns in flight
            constexpr int OG = 4;
            float2 old[OG][8];
            auto fetch_old = [&](float2 (&o)[8], int c0) {
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    o[e] = on && to_r && c0 + e < ncol ? __ldcg(out + (size_t)(c0 + e) * N) : make_float2(0.f, 0.f);
            };
            if (to_r && !step_wait(tl, seen)) break;
            if (warp_on) {
#pragma unroll
                for (int g = 0; g < OG; ++g) fetch_old(old[g], 8 * g);
            }
            if (!wait(&acc_full[sl], tt / SL)) break;
            tc_fence_after();
            if (warp_on) {
                const uint32_t d = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(sl * BS_SLOT_COLS);
                for (int cb = 0; cb < ncol; cb += 8 * OG) {
#pragma unroll
                    for (int g = 0; g < OG; ++g) {
                        const int c0 = cb + 8 * g;
                        if (c0 >= ncol) break;
                        // Re = Ar Br - Ai Bi, Im = Ar Bi + Ai Br
                        uint32_t rr[8], ri[8], ir[8], ii[8];
                        tc_ld8_issue(d + c0, rr);
                        tc_ld8_issue(d + nt + c0, ri);
                        tc_ld8_issue(d + 2 * nt + c0, ir);
                        tc_ld8_issue(d + 3 * nt + c0, ii);
                        tc_wait_ld8(rr);
                        tc_wait_ld8(ri);
                        tc_wait_ld8(ir);
                        tc_wait_ld8(ii);
                        float2 o[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const float sb = s_bscale[sl][c0 + e] * f;
                            o[e].x = old[g][e].x + (__uint_as_float(rr[e]) - __uint_as_float(ii[e])) * sb;
                            o[e].y = old[g][e].y + (__uint_as_float(ri[e]) + __uint_as_float(ir[e])) * sb;
                        }
                        fetch_old(old[g], c0 + 8 * OG);
                        uint32_t gmax = 0;
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            if (on && c0 + e < ncol) out[(size_t)(c0 + e) * N] = o[e];
                            const uint32_t b = on ? max(bs_abs_bits(o[e].x), bs_abs_bits(o[e].y)) : 0u;
                            const uint32_t w = __reduce_max_sync(0xffffffffu, b);
                            if (lane == e) gmax = w;
                        }
                        if (lane < 8 && c0 + lane < ncol) gout[c0 + lane] = __uint_as_float(gmax);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive_cta(&acc_empty[sl]);
                __threadfence();   // the warp's stores before its count
                atomicAdd(a.ctl + 2 + tl.phase * a.ns + tl.sys, 1u);
            }
            ++tt;
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
            const uint32_t w = __reduce_max_sync(0xffffffffu, max(bs_abs_bits(t[e].x), bs_abs_bits(t[e].y)));
            if (lane == b + e) mine = w;
        }
    }
    if (lane < nc) g[(((size_t)sys * nx + line) * ng + grp) * nrhs + c0 + lane] = __uint_as_float(mine);
}

// largest modulus of the real and imaginary parts of a part of the blocks, as bits (mx zeroed
// beforehand): a CTA takes 32 rows, up to the end of their 128 x 128 block on the diagonal
__global__ void __launch_bounds__(256) bcr_max_kernel(int n, BsPart pt, const float2 *src, long long stride, const int *pairs,
                                                      uint32_t *mx) {
    const int *pr = pairs + 2 * (size_t)blockIdx.y;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, r0 = pt.r0 + 32 * blockIdx.x;
    const int end = min(pt.c0 + pt.n, (r0 | 127) + 1);
    uint32_t m = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int r = r0 + w + 8 * q;
        if (r >= pt.r0 + pt.m) continue;
        const float4 *A = reinterpret_cast<const float4 *>(src + (long long)pr[0] * stride + (long long)r * n + pt.c0);
        for (int e = lane; e < (end - pt.c0) / 2; e += 32) {
            const float4 v = __ldg(A + e);
            m = max(max(m, max(bs_abs_bits(v.x), bs_abs_bits(v.y))), max(bs_abs_bits(v.z), bs_abs_bits(v.w)));
        }
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0 && m) atomicMax(mx + pr[1], m);
}

// Image of a part of a symmetric block (n x n row-major) as matrix pairs[.][1].  A CTA takes 32 rows, a
// thread a row and eight columns at a time; rows and columns beyond n are zero.
__global__ void __launch_bounds__(128) bcr_image_kernel(int n, BsPart pt, int nzr, const float2 *src, long long stride,
                                                        const int *pairs, BsImages im, size_t mat_bytes) {
    __shared__ float2 t[32][33];
    const int *pr = pairs + 2 * (size_t)blockIdx.y;
    const float2 *A = src + (long long)pr[0] * stride;
    const int r0 = pt.r0 + 32 * blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int sh = bs_scale_shift(im.mx[pr[1]]);
    const float sc = bs_pow2(sh);
    if (blockIdx.x == 0 && threadIdx.x == 0) im.shift[pr[1]] = sh;
    const int row = threadIdx.x >> 2, j = threadIdx.x & 3, r = r0 + row;
    const size_t half = (size_t)nzr * 128;
    unsigned char *d = im.at(pr[1], mat_bytes) + (size_t)(pt.c0 >> 5) * 2 * half + (size_t)r * 128;
    for (int c = 0; c < (pt.n + 31) / 32; ++c) {
        const int k0 = pt.c0 + 32 * c;
        const bool up = (r0 >> 7) < (k0 >> 7);   // above the diagonal: the mirror image's rows
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int o = w + 4 * q, rr = (up ? k0 : r0) + o, k = (up ? r0 : k0) + lane;
            const float2 v = rr < n && k < n ? __ldg(A + (long long)rr * n + k) : make_float2(0.f, 0.f);
            if (up) t[lane][o] = v;
            else t[o][lane] = v;
        }
        __syncthreads();
        if (r < nzr) {
            float2 v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = t[row][8 * j + e];
            uint4 rh, rl, ih, il;
            bs_split8(v, sc, rh, rl, ih, il);
            *reinterpret_cast<uint4 *>(d + ((j ^ (r & 7)) << 4)) = rh;
            *reinterpret_cast<uint4 *>(d + (((j + 4) ^ (r & 7)) << 4)) = rl;
            d += half;
            *reinterpret_cast<uint4 *>(d + ((j ^ (r & 7)) << 4)) = ih;
            *reinterpret_cast<uint4 *>(d + (((j + 4) ^ (r & 7)) << 4)) = il;
            d += half;
        }
        __syncthreads();
    }
}

template <int NT> cudaError_t launch_nt(const BsArgs &a, int grid, double flops, cudaStream_t st) {
    const void *fn = (const void *)bcr_solve_kernel<NT>;
    cudaError_t e = ensure_dyn_smem(fn, BsCfg<NT>::SMEM);
    if (e != cudaSuccess) return e;
    HELM_TRACED_W(K_BCR_SOLVE, st, flops, (bcr_solve_kernel<NT><<<grid, BS_THREADS, BsCfg<NT>::SMEM, st>>>(a)));
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_bcr_image(int n, BsPart part, const float2 *src, long long stride, const int *pairs_dev, int count,
                             const BsImages &im, cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    const BsLayout l = bs_layout(n);
    const unsigned rows = (part.m + 31) / 32;
    for (int t = 0; t < count; t += 65535) {
        const dim3 grid(rows, std::min(65535, count - t));
        const int *pr = pairs_dev + 2 * (size_t)t;
        HELM_TRACED(K_BCR_IMAGE, st, (bcr_max_kernel<<<grid, 256, 0, st>>>(n, part, src, stride, pr, im.mx)));
        HELM_TRACED(K_BCR_IMAGE, st, (bcr_image_kernel<<<grid, 128, 0, st>>>(n, part, l.nzr, src, stride, pr, im, l.mat_bytes)));
    }
    return cudaGetLastError();
}

cudaError_t launch_bcr_solve(BsArgs a, const BsStep *steps, int n_steps, bool prepared, double flops, cudaStream_t st) {
    if (n_steps > BS_MAX_PHASE || (a.nz & 1)) return cudaErrorInvalidValue;
    const BsLayout l = bs_layout(a.nz);
    a.nzr = l.nzr;
    a.n_chunk = l.n_chunk;
    a.mat_bytes = l.mat_bytes;
    a.ng = l.ng;
    a.N = a.nx * a.nz;
    const int nt = a.nrhs <= 16 ? 16 : (a.nrhs <= 32 ? 32 : 64);
    const int sms = device_sms();
    a.n_phase = n_steps;
    int tile = 0;
    for (int p = 0; p < n_steps; ++p) {
        BsPhase &ph = a.ph[p];
        ph.tile0 = tile;
        ph.task0 = steps[p].task0;
        ph.tasks = steps[p].tasks;
        // steps with few lines take narrower and then lower tiles, so that more SMs share their
        // products and the blocks' stream
        ph.mrows = 128;
        ph.nt = steps[p].type == BS_BWD0 ? std::min(nt, BS_NT_BWD0) : nt;
        auto tiles_of = [&]() {
            ph.n_tiles = (a.nrhs + ph.nt - 1) / ph.nt;
            ph.mt = (a.nz + ph.mrows - 1) / ph.mrows;
            return ph.tasks * a.ns * ph.n_tiles * ph.mt;
        };
        while (ph.nt > 16 && tiles_of() < sms) ph.nt /= 2;
        while (ph.mrows > 32 && tiles_of() < sms) ph.mrows /= 2;
        tile += tiles_of();
        ph.done = 4 * ph.tasks * ph.n_tiles * ph.mt;   // four epilogue warps count each tile
    }
    a.n_tile_total = tile;
    if (!prepared) {
        cudaError_t e = cudaMemsetAsync(a.ctl, 0, sizeof(unsigned) * bs_ctl_words(n_steps, a.ns), st);
        if (e != cudaSuccess) return e;
        const int n_cb = (a.nrhs + 31) / 32;
        const long long items = (long long)a.ns * a.nx * a.ng * n_cb;
        HELM_TRACED(K_LINEMAX, st, (line_max_kernel<<<(unsigned)((items + 7) / 8), 256, 0, st>>>(
                                       a.nx, a.nz, a.ng, a.nrhs, n_cb, items, a.r, a.gr, a.skip, a.frozen)));
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    const int grid = std::min(sms, tile);
    if (nt == 16) return launch_nt<16>(a, grid, flops, st);
    return nt == 32 ? launch_nt<32>(a, grid, flops, st) : launch_nt<64>(a, grid, flops, st);
}

}  // namespace helm
