// The persistent solve of a block-cyclic-reduction factor (bcr_solve.cu; internal header).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace helm {

// Blocks of the factor in the solve's operand layout: n_chunk chunks of 32 columns, each the rows
// (padded to 8) of the real and then of the imaginary part, 128 bytes a row (32 hi, 32 lo FP16)
struct BsLayout {
    int n_chunk, nzr, ng;   // ng: 32-row groups of a line (the vectors' maxima)
    size_t mat_bytes;
};
__host__ __device__ inline BsLayout bs_layout(int nz) {
    BsLayout l;
    l.n_chunk = (nz + 31) / 32;
    l.nzr = (nz + 7) & ~7;
    l.ng = (nz + 31) / 32;
    l.mat_bytes = (size_t)l.n_chunk * 2 * l.nzr * 128;
    return l;
}

// Kinds of stored blocks: per system n_x inverses, then n_half of W, V, P and Q each (slot line / 2).
// A block of a task is coded kind << 24 | slot; P and Q multiply x, the others r.
enum { BS_DINV = 0, BS_W = 1, BS_V = 2, BS_P = 3, BS_Q = 4 };
// steps (types of tasks): level 0 forward, level forward, last line, level backward, level 0 backward
enum { BS_FWD0 = 0, BS_FWD = 1, BS_LAST = 2, BS_BWD = 3, BS_BWD0 = 4 };
constexpr int BS_MAX_PHASE = 64;

struct BsStep {   // one dependent step of the solve: its tasks (the same for every system)
    int task0, tasks, type;
};
struct BsPhase {
    int tile0, task0, tasks, nt, n_tiles, mt, mrows, done;   // nt x mrows: the step's tiles
};
struct BsArgs {
    int nx, nz, ns, nrhs, half;
    int edge;               // last node of a line (nz - 1, or nz - 2 where nz counts a line's extra node)
    float2 *r, *x;          // [ns][nrhs][nx * nz]: right-hand sides (overwritten) and the result
    float *gr, *gx;         // maxima of r and x: [ns][nx][ng][nrhs] each
    const unsigned char *img;
    const int *shift;       // [matrix]: the image holds the block's entries times 2^shift
    const int *tasks;       // [8] per task: line, type | terms << 4, then (block, line of the vector) per term
    float cx_in, cx_edge;
    unsigned *ctl;          // tile counter, abort word, tiles finished per step and system
    int *status;
    const int *skip, *frozen;
    uint32_t tries;
    // set by launch_bcr_solve
    int N, n_chunk, nzr, ng, n_phase, n_tile_total;
    size_t mat_bytes;
    BsPhase ph[BS_MAX_PHASE];
};
inline size_t bs_ctl_words(int n_steps, int ns) { return 2 + (size_t)n_steps * ns; }
__host__ __device__ inline int bs_kind(int code) { return code >> 24; }
// matrix number of a coded block of system sys
__host__ __device__ inline long long bs_matrix_index(int nx, int ns, int half, int code, int sys) {
    const int kind = code >> 24, slot = code & 0xffffff;
    return kind == BS_DINV ? (long long)sys * nx + slot
                           : (long long)ns * nx + ((long long)(kind - 1) * ns + sys) * half + slot;
}
__device__ __forceinline__ long long bs_matrix(const BsArgs &a, int code, int sys) {
    return bs_matrix_index(a.nx, a.ns, a.half, code, sys);
}

// A family of images: matrices 0 .. n_kept - 1 stay with the factor, the others are its working blocks
struct BsImages {
    unsigned char *kept = nullptr, *work = nullptr;
    int n_kept = 0;
    int *shift = nullptr;      // [matrix]
    uint32_t *mx = nullptr;    // [matrix]: bits of the largest modulus (or a bound); working array of the factor
    // from n_sub on: parts of a block that is being inverted, eight matrices (scales) to a node of its
    // recursion and `sub` to a block, whose parts fill two images from number sub0 (of the working
    // ones) on: the first four of a node one, the others the other
    int n_sub = 0x7fffffff, sub = 8, sub0 = 0;
    __host__ __device__ unsigned char *at(int i, size_t mat_bytes) const {
        if (i < n_kept) return kept + (size_t)i * mat_bytes;
        const int j = i - n_sub;
        return work + (size_t)(j < 0 ? i - n_kept : sub0 + 2 * (j / sub) + ((j >> 2) & 1)) * mat_bytes;
    }
};
struct BsPart {   // rows r0 .. + m and columns c0 .. + n of a block (r0 and c0 multiples of 128)
    int r0, c0, m, n;
};
// images of the part of n x n row-major symmetric blocks src + pairs[.][0] * stride as that part of the
// matrices pairs[.][1]; 128 x 128 blocks above the diagonal are taken from below it (and need not be
// in memory); im.mx zeroed beforehand
cudaError_t launch_bcr_image(int n, BsPart part, const float2 *src, long long stride, const int *pairs_dev, int count,
                             const BsImages &im, cudaStream_t st);

// Products of images (bcr_gemm.cu): tasks of BG_TASK ints (flags, matrix A, matrix B, output, and two
// more): the image of +-A B^T as matrix `output` and, with BG_TR, of its transpose as the matrix in
// the fifth place; or (BG_FP32) D block `output` += +-A B^T, with BG_TWO += +-(A B^T + A' B'^T), A'
// and B' the fifth and sixth; BG_STORE: an image whose transpose is stored to D block in the sixth place.
// The updates (BG_FP32) are symmetric.
constexpr int BG_TASK = 6;
enum { BG_NEG = 1, BG_FP32 = 2, BG_TWO = 4, BG_TR = 8, BG_STORE = 16 };
struct BgArgs {
    int nz;
    const int *tasks;
    BsImages im;
    float2 *D;               // [block][nz][nz]
    int *status;
    uint32_t tries;
    // the products of a launch: m x n of inner length k, from row ra and column ca of A, row rb and
    // column cb of B, to row ro and column co (k = 0: whole blocks)
    int m, n, k, ra, ca, rb, cb, ro, co;
    // set by launch_bcr_gemm
    int n_chunk, nzr, mt, nt, n_tiles, log2_2k;
    size_t mat_bytes;
};
cudaError_t launch_bcr_gemm(BgArgs a, int n_tasks, int n_products, cudaStream_t st);
cudaError_t launch_bcr_solve(BsArgs a, const BsStep *steps, int n_steps, bool prepared, double flops, cudaStream_t st);
int device_sms();   // streaming multiprocessors of the current device

}  // namespace helm
