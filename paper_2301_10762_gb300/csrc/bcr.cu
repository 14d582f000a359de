// Block cyclic reduction (BCR) of the block-tridiagonal line system, mixed precision.
//
// With lines of constant x (n_z nodes each) the discrete operator A(m, w) of the Appendix
// ("Numerical forward model") is block tridiagonal: diagonal blocks D_i (tridiagonal) and the
// diagonal horizontal couplings C between neighbouring lines; A is complex symmetric, so the
// coupling of line k to a line a is the transpose of that of a to k.  Where the line factor
// (factor.cu) runs the Schur recurrence line after line, BCR eliminates every other line of
// the current system at once, level by level (spacing s = 2^l):
//     eliminated j (j = s mod 2s):    Dinv_j = D_j^{-1}
//     kept k (k = 0 mod 2s), a = k - s, c = k + s:
//         D_k <- D_k - L_k Dinv_a U_a - U_k Dinv_c L_c
//         L_k <- -L_k Dinv_a L_a      (coupling to k - 2s)
//         U_k <- -U_k Dinv_c U_c      (coupling to k + 2s)
// until one line is left (line 0, whose inverse ends the factor).  Every level is a batch of
// independent dense block products and inversions over all lines and frequencies, which
// bcr_gemm.cu and the batched block inversion below run; the depth of the
// dependent chain is log2(n_x) levels instead of n_x lines.  By symmetry L_k = U_a^T and
// U_k = L_c^T, so every product is a GEMM of row-major operands:
//     W_a = L_k Dinv_a (= (Dinv_a U_a)^T),   V_c = U_k Dinv_c (= (Dinv_c L_c)^T),
//     D_k -= L_k W_a^T + U_k V_c^T,   L_k <- -L_k V_a^T,   U_k <- -U_k W_c^T,
// and the back substitution takes P_j = V_j^T = Dinv_j L_j, Q_j = W_j^T = Dinv_j U_j.
// Level 0 has the diagonal couplings C: its products are elementwise scalings.
//
// The solve of A x = b (all right-hand sides of a system as the products' N dimension) takes the
// blocks W, V, P, Q and the inverses in the layout of bcr_solve.cu, which runs it:
//     forward, level 0:  b_k -= C (Dinv_a b_a + Dinv_c b_c)
//     forward, level l:  b_k -= W_a b_a + V_c b_c
//     last line:         x_0 = Dinv_0 b_0
//     backward, level l: x_j = Dinv_j b_j - P_j x_{j-s} - Q_j x_{j+s}
//     backward, level 0: x_j = Dinv_j (b_j - C (x_{j-1} + x_{j+1})).
// The factor is the preconditioner of the FP64-residual refinement of the mixed path, exactly as the
// line factor is.  Blocks that are factored further (D) are complex FP32; couplings, their products
// and the inverses exist only as images (bcr_solve.h: every real entry the sum of two FP16 numbers,
// 22 bits), which the products (bcr_gemm.cu) read and write.  Residuals after 1, 2, 3 sweeps at 128^2:
// 1.5e-5, 6.4e-10, 1.5e-13 (with FP32 blocks, 3xTF32 products and truncating sums throughout: 5.7e-9
// after 2 and 1.4e-12 after 3; the line factor 6e-11 and 1.4e-13).  What decides it is the sums: the
// tensor core truncates, so long ones go through registers (bcr_gemm.cu, zinv_kernel).
//
// Level 0 inverts no block (TriGen below).  Above it, a batch of dense inversions: n <= 128 one CTA per
// block (zinv_kernel); larger n by the 2 x 2 block inverse of a symmetric matrix
//     [[D11, D21^T], [D21, D22]]^{-1}:  X11 = D11^{-1}, T = X11 D21^T, S = D22 - D21 T,
//     X22 = S^{-1}, X12 = -T X22, X21 = X12^T, X11 <- X11 - T X21,
// with the products on the tensor cores and the two half-size inverses recursive (invert_images).
// Time at 256^2 with 8 frequencies, of a 6.9 ms factor: level 0 0.9 ms, inversions 1.8, their parts'
// products and images 1.4, the levels' products 2.3, images of the inverses 0.4.
#include <math.h>
#include <stdlib.h>

#include <algorithm>
#include <functional>
#include <initializer_list>
#include <utility>
#include <vector>

#include "abi_internal.h"
#include "bcr_image.cuh"
#include "bcr_solve.h"
#include "kernels.h"
#include "pivot16.cuh"
#include "tcgen05.cuh"
#include "trace.h"

namespace helm {

namespace {

constexpr int INV_MAX = 128;   // largest block inverted in one CTA's shared memory

// ------------------------------------------------------------------- kernels

// couplings of the grid in FP32: horizontal (between lines, row j) and vertical (within line
// i), each halved on a boundary edge; computed once on the host
struct Coup {
    float cx_in, cx_edge, cz_in, cz_edge;
    __device__ __forceinline__ float cx(int j, int nz) const { return (j == 0 || j == nz - 1) ? cx_edge : cx_in; }
    __device__ __forceinline__ float cz(int i, int nx) const { return (i == 0 || i == nx - 1) ? cz_edge : cz_in; }
};
Coup coup_of(const GridGeom &g) {
    return Coup{(float)coup_x(g, 1), (float)coup_x(g, 0), (float)coup_z(g, 1), (float)coup_z(g, 0)};
}

// Level 0: the eliminated lines' blocks are complex symmetric tridiagonal, T = tridiag(cz, d, cz),
// and their inverses semiseparable:
//     X_ij = u_i v_j for i <= j (X symmetric),   u_i = 1 / R_i,  v_j = g_j R_j,
// with the pivots of the elimination from above (delta_k = d_k - cz^2 / delta_{k-1}) and from
// below (gamma_k = d_k - cz^2 / gamma_{k+1}), R_j = prod_{k < j} (-cz / delta_k) and g_j = X_jj =
// 1 / (delta_j + gamma_j - d_j).  So no block is inverted: the recurrences run in FP64 (O(n_z) per
// line), and every kernel that wants X forms its entries from u and v, held as FP32 hi + lo with an
// exponent (R spans hundreds of orders of magnitude), correct to FP32 rounding.  Cyclic reduction
// amplifies level 0's errors most (the Schur complements of the smooth modes lose four in size
// per level): a block Gauss-Jordan inverse carries 1.2e-7 of its norm.
// 256^2 with 8 frequencies: level 0 with its images 0.9 ms, a quarter of it the recurrences (dense inversions by two 128-column
// halves 1.0 ms, images and update 0.6); 512^2 with 8: 19 ms less.
struct TriGen {          // generators of the odd lines' inverses: [line][nz]
    float4 *u, *v;       // hi.x, hi.y, lo.x, lo.y
    int2 *e;             // exponents of u and v
};
struct TriScan {         // working arrays of the recurrences: [k][line]
    double2 *delta, *gamma, *r;
    int *re;
};

// 1 / z, the modulus bounded from below by 1e-12 of `scale` (a pivot there is as good as singular in
// FP32: T is perturbed by no more than that)
__device__ __forceinline__ double2 crecip_guard(double2 z, double scale) {
    double n2 = z.x * z.x + z.y * z.y;
    if (n2 < 1e-24 * scale * scale) {
        z = make_double2(1e-12 * scale, 0.0);
        n2 = z.x * z.x;
    }
    const double r = fast_recip(n2);
    return make_double2(z.x * r, -z.y * r);
}
// z scaled to a largest part in [1, 2), e its exponent (zero and non-finite values as they are)
__device__ __forceinline__ double2 cnormalize(double2 z, int &e) {
    const int hx = (__double2hiint(z.x) >> 20) & 0x7ff, hy = (__double2hiint(z.y) >> 20) & 0x7ff, h = max(hx, hy);
    if (h == 0 || h == 0x7ff) { e = 0; return z; }
    e = h - 1023;
    const double s = __hiloint2double((2046 - h) << 20, 0);   // 2^-e
    return make_double2(z.x * s, z.y * s);
}

// the recurrences: a thread per line and direction.  A chain of n_z steps of about ten dependent
// FP64 operations; 32 chains share a warp because the FP64 pipe takes two lanes a cycle per SM
// however many are active.
__global__ void __launch_bounds__(32) tri_scan_kernel(GridGeom g, int n_line, const double2 *diag, TriScan w) {
    const int t = blockIdx.x * 32 + threadIdx.x, dir = t & 1, l = t >> 1;
    if (l >= n_line) return;
    const int nx = g.nx, nz = g.nz, no = nx / 2, line = 2 * (l % no) + 1;
    const double2 *d = diag + ((size_t)(l / no) * nx + line) * nz;
    const double cz = coup_z(g, line), c2 = cz * cz;
    double2 inv = make_double2(0.0, 0.0), r = make_double2(1.0, 0.0);
    int re = 0;
    double2 nd = d[dir ? nz - 1 : 0];
    for (int q = 0; q < nz; ++q) {
        const int k = dir ? nz - 1 - q : q;
        const double2 dk = nd;
        if (q + 1 < nz) nd = d[dir ? k - 1 : k + 1];
        const double2 p = make_double2(dk.x - c2 * inv.x, dk.y - c2 * inv.y);
        const size_t o = (size_t)k * n_line + l;
        inv = crecip_guard(p, cz);
        if (dir) {
            w.gamma[o] = p;
        } else {
            w.delta[o] = p;
            w.r[o] = r;
            w.re[o] = re;
            int e;
            r = cnormalize(cmul(r, make_double2(-cz * inv.x, -cz * inv.y)), e);
            re += e;
        }
    }
}

// generators, and the scales of the images of X and of -C X C from the bound max_j |v_j| max_{i <= j}
// |u_i| (attained up to the FP32 rounding): a CTA per line
__global__ void __launch_bounds__(256) tri_gen_kernel(GridGeom g, Coup cp, int n_line, const double2 *diag, TriScan w,
                                                      TriGen o, const int *dst, BsImages im) {
    const int l = blockIdx.x, nx = g.nx, nz = g.nz, no = nx / 2, line = 2 * (l % no) + 1;
    const double2 *d = diag + ((size_t)(l / no) * nx + line) * nz;
    const double cz = coup_z(g, line);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ float s_u[8], s_top[8];
    float carry = -1e30f, top = -1e30f;   // log2 of the largest |u| so far and of the largest |X|
    for (int k0 = 0; k0 < nz; k0 += 256) {
        const int k = k0 + tid;
        float lu = -1e30f, lv = -1e30f;
        if (k < nz) {
            const size_t q = (size_t)k * n_line + l;
            const double2 dl = w.delta[q], gm = w.gamma[q], r = w.r[q], dk = d[k];
            int e1, e2;
            const double2 u = cnormalize(crecip_guard(r, 0.0), e1);
            const double2 gg = crecip_guard(make_double2(dl.x + gm.x - dk.x, dl.y + gm.y - dk.y), cz);
            const double2 v = cnormalize(cmul(gg, r), e2);
            const int eu = e1 - w.re[q], ev = e2 + w.re[q];
            const size_t p = (size_t)l * nz + k;
            const float ux = (float)u.x, uy = (float)u.y, vx = (float)v.x, vy = (float)v.y;
            o.u[p] = make_float4(ux, uy, (float)(u.x - ux), (float)(u.y - uy));
            o.v[p] = make_float4(vx, vy, (float)(v.x - vx), (float)(v.y - vy));
            o.e[p] = make_int2(eu, ev);
            lu = 0.5f * __log2f(ux * ux + uy * uy) + (float)eu;
            lv = 0.5f * __log2f(vx * vx + vy * vy) + (float)ev;
        }
        // running maximum of lu over k: warp scan, then the warps before, then the blocks before
        float m = lu;
#pragma unroll
        for (int s = 1; s < 32; s *= 2) {
            const float t = __shfl_up_sync(0xffffffffu, m, s);
            if (lane >= s) m = fmaxf(m, t);
        }
        if (lane == 31) s_u[warp] = m;
        __syncthreads();
        float all = carry;
        for (int s = 0; s < 8; ++s) {
            if (s < warp) m = fmaxf(m, s_u[s]);
            all = fmaxf(all, s_u[s]);
        }
        m = fmaxf(m, carry);
        carry = all;
        top = fmaxf(top, lv + m);
        __syncthreads();
    }
#pragma unroll
    for (int s = 16; s > 0; s /= 2) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, s));
    if (lane == 0) s_top[warp] = top;
    __syncthreads();
    if (tid == 0) {
        for (int s = 1; s < 8; ++s) top = fmaxf(top, s_top[s]);
        // (a NaN is left out of fmaxf: the entries themselves carry it)
        const float mx = exp2f(fminf(fmaxf(top, -120.f), 120.f)) * 1.0001f;
        const float mm = mx * fmaxf(cp.cx_in * cp.cx_in, cp.cx_edge * cp.cx_edge);
        im.mx[dst[2 * l]] = bs_abs_bits(mx);
        im.shift[dst[2 * l]] = bs_scale_shift(bs_abs_bits(mx));
        im.mx[dst[2 * l + 1]] = bs_abs_bits(mm);
        im.shift[dst[2 * l + 1]] = bs_scale_shift(bs_abs_bits(mm));
    }
}

// u v 2^(eu + ev + sh)
__device__ __forceinline__ float2 tri_entry(const float4 &u, const float4 &v, int e) {
    const float re = fmaf(u.x, v.x, fmaf(-u.y, v.y, fmaf(u.x, v.z, fmaf(-u.y, v.w, fmaf(u.z, v.x, -u.w * v.y)))));
    const float im = fmaf(u.x, v.y, fmaf(u.y, v.x, fmaf(u.x, v.w, fmaf(u.y, v.z, fmaf(u.z, v.y, u.w * v.x)))));
    const float s = e < -126 ? 0.f : bs_pow2(min(e, 128));   // (128: infinity)
    return make_float2(re * s, im * s);
}

// images of X (matrix dst[.][0]) and -C X C (dst[.][1]) of a line: a CTA takes 32 rows, a thread a
// row and eight columns at a time.  Bound by the write of the images.
__global__ void __launch_bounds__(128) tri_image_kernel(int n, int n_chunk, int nzr, TriGen tg, const int *dst, Coup cp,
                                                        BsImages im, size_t mat_bytes) {
    const int l = blockIdx.x, row = threadIdx.x >> 2, j = threadIdx.x & 3, r = 32 * blockIdx.y + row;
    if (r >= nzr) return;
    const bool on = r < n;
    const float4 *U = tg.u + (size_t)l * n, *V = tg.v + (size_t)l * n;
    const int2 *E = tg.e + (size_t)l * n;
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 ur = on ? U[r] : z4, vr = on ? V[r] : z4;
    const int2 er = on ? E[r] : make_int2(0, 0);
    const int mx = dst[2 * l], mm = dst[2 * l + 1], shx = im.shift[mx], shm = im.shift[mm];
    const float cr = on ? -cp.cx(r, n) * bs_pow2(shm - shx) : 0.f;   // (|shm - shx|: the couplings' exponent)
    unsigned char *px = im.at(mx, mat_bytes) + (size_t)r * 128, *pm = im.at(mm, mat_bytes) + (size_t)r * 128;
    const int o0 = (j ^ (r & 7)) << 4, o1 = ((j + 4) ^ (r & 7)) << 4;
    const size_t half = (size_t)nzr * 128;
    for (int c = 0; c < n_chunk; ++c, px += 2 * half, pm += 2 * half) {
        float2 x[8], m[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int k = 32 * c + 8 * j + q;
            x[q] = m[q] = make_float2(0.f, 0.f);
            if (on && k < n) {
                const bool up = r <= k;
                const float4 o = __ldg(up ? V + k : U + k);
                const int2 e = __ldg(E + k);
                x[q] = tri_entry(up ? ur : vr, o, (up ? er.x + e.y : er.y + e.x) + shx);
                const float f = cr * cp.cx(k, n);
                m[q] = make_float2(f * x[q].x, f * x[q].y);
            }
        }
        uint4 rh, rl, ih, il;
        bs_split8(x, 1.f, rh, rl, ih, il);
        *reinterpret_cast<uint4 *>(px + o0) = rh;
        *reinterpret_cast<uint4 *>(px + o1) = rl;
        *reinterpret_cast<uint4 *>(px + half + o0) = ih;
        *reinterpret_cast<uint4 *>(px + half + o1) = il;
        bs_split8(m, 1.f, rh, rl, ih, il);
        *reinterpret_cast<uint4 *>(pm + o0) = rh;
        *reinterpret_cast<uint4 *>(pm + o1) = rl;
        *reinterpret_cast<uint4 *>(pm + half + o0) = ih;
        *reinterpret_cast<uint4 *>(pm + half + o1) = il;
    }
}

// level 0 (couplings C = diag(cx)): kept line k (even) with eliminated neighbours k - 1, k + 1:
//   D_k = T_k - C X_{k-1} C - C X_{k+1} C
// a CTA takes 32 rows by 256 columns, a thread two columns (their generators in registers; the
// rows' are the same for the whole CTA)
__global__ void __launch_bounds__(128) bcr_level0_kernel(GridGeom g, int np, Coup cp, float2 *D, const double2 *diag, TriGen tg) {
    const int nz = g.nz, nx = g.nx, no = nx / 2, nk = (nx + 1) / 2;
    const int s = blockIdx.x / nk, k = 2 * (blockIdx.x % nk), c = 256 * blockIdx.z + 2 * threadIdx.x;
    if (c >= np) return;
    const bool has[2] = {k >= 1, k + 1 < nx};
    float4 uc[2][2], vc[2][2];
    int2 ec[2][2];
    size_t base[2];
    float fc[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) fc[h] = cp.cx(c + h, nz);
#pragma unroll
    for (int n = 0; n < 2; ++n) {
        base[n] = ((size_t)s * no + (has[n] ? k / 2 - 1 + n : 0)) * nz;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int cc = min(c + h, nz - 1);
            uc[n][h] = __ldg(tg.u + base[n] + cc);
            vc[n][h] = __ldg(tg.v + base[n] + cc);
            ec[n][h] = __ldg(tg.e + base[n] + cc);
        }
    }
    const float cz = cp.cz(k, nx);
    const double2 *dg = diag + ((size_t)s * nx + k) * nz;
    float2 *Dk = D + ((size_t)s * nk + k / 2) * np * np;   // (the odd lines' blocks are never formed)
    for (int r = 32 * blockIdx.y; r < min(np, 32 * (int)blockIdx.y + 32); ++r) {
        if (r >= nz) {   // an odd line's extra node: decoupled
            *reinterpret_cast<float4 *>(Dk + (size_t)r * np + c) = make_float4(c == r ? 1.f : 0.f, 0.f, c + 1 == r ? 1.f : 0.f, 0.f);
            continue;
        }
        float2 t[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            if (!has[n]) continue;
            const float4 ur = __ldg(tg.u + base[n] + r), vr = __ldg(tg.v + base[n] + r);
            const int2 er = __ldg(tg.e + base[n] + r);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool up = r <= c + h;
                const float2 x = up ? tri_entry(ur, vc[n][h], er.x + ec[n][h].y) : tri_entry(uc[n][h], vr, ec[n][h].x + er.y);
                t[h].x += x.x;
                t[h].y += x.y;
            }
        }
        const float fr = cp.cx(r, nz);
        float2 o[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int cc = c + h;
            float2 d = make_float2(0.f, 0.f);
            if (r == cc) d = to_c64(dg[r]);
            else if (r - cc == 1 || cc - r == 1) d.x = cz;
            const float f = fr * fc[h];
            o[h] = cc < nz ? make_float2(d.x - f * t[h].x, d.y - f * t[h].y) : make_float2(0.f, 0.f);
        }
        *reinterpret_cast<float4 *>(Dk + (size_t)r * np + c) = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
    }
}

struct InvArgs {
    int n;
    float2 *X;                   // blocks, row-major
    long long stride;
    int ld;
    const int *idx;              // [count]: block
    int *status;
    uint32_t tries = 0;          // polls of a bounded mbarrier wait before it gives up
};

// X <- X^{-1} of one n x n block (n <= 128) per CTA by Gauss-Jordan in steps of 16 columns, partial
// pivoting inside each 16 x 16 pivot block.  The block lives in registers: thread (r, h) of
// 512 holds row r, columns 32 h .. + 31 (beyond n: the identity).  A step with the pivot columns
// K = k0 .. k0 + 15 is
//     W <- W' + A' R'  (W' = W with the rows and columns K zeroed;
//                       A'[r][u] = -W[r][k0 + u] off the pivot rows, delta(r - k0, u) on them;
//                       R' = P W[K, :] off the pivot columns, P on them, P = W[K, K]^{-1}),
// one 3xTF32 product of M = 128, N = 2 n, K = 32 reals (R' expanded to real rows) into a fresh
// accumulator in tensor memory, which the threads add to W: the tensor core truncates every sum,
// and a step that accumulated into W itself lost up to an ulp of W twelve times over, which cost
// the inverses of the upper levels a factor of 30 (3e-5 of their norm).
// The chain of pivot blocks is what bounds it, so it runs ahead of the rest: warps 0 to 7 update the
// next pivot block W[K1, K1] first and warp 0 inverts it while the other warps form R',
// the tensor core multiplies and W is updated.
// H groups of 32 columns: four, or two for n <= 64 (256 threads and 86 KB, so that two CTAs share an SM and
// hide each other's chain: 1000 blocks of 16 take 44 us, of 30 81, of 64 143; with four groups 80, 142 and
// 233; a wave of them 14, 23 and 34 us against 16, 25 and 38).
constexpr int ZT_PS = 17;   // row stride (complex) of the 16 x 16 blocks
constexpr int ZT_TS = 65;   // row stride (complex) of 64 columns on their way in or out
template <int H> struct ZtCfg {
    static constexpr int WARPS = 4 * H, THREADS = 32 * WARPS;
    static constexpr int WS = 32 * H + 1;   // row stride (complex) of the pivot rows
    static constexpr uint32_t A = 0, B = 32768, B_BYTES = 8192 * H, WK = B + 2 * B_BYTES, P = WK + 8 * PIV * WS,
                              BLK = P + 2 * 8 * PIV * PIV;
    static constexpr size_t SMEM = BLK + 4 * 8 * PIV * ZT_PS + 1024;
    static constexpr uint32_t TMEM = 64 * H;
};

// 16 x 16 inverse in place by one warp: lane (r, h) holds row r, columns 8 h .. + 7 of M (shared, row
// stride ZT_PS); P row stride 16.  Gauss-Jordan with partial pivoting without row swaps: at step
// q the row p_q eliminates column q, whose slot then holds column p_q of the inverse.  Bounds: the
// chain of a column (maximum, broadcast, reciprocal, update, about 200 cycles); the augmented form
// [M | I] of warp_invert16 has twice the shuffles and products per lane.  False if a pivot was zero
// or not finite.
__device__ bool warp_invert16_inplace(const float2 *M, float2 *P) {
    const int lane = threadIdx.x & 31, r = lane & 15, h = lane >> 4;
    float2 a[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) a[j] = M[r * ZT_PS + 8 * h + j];
    unsigned used = 0;
    unsigned long long perm = 0;
    int qinv = 0;
    bool ok = true;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        const int src = r + 16 * (q >> 3);
        const float2 f = make_float2(__shfl_sync(0xffffffffu, a[q & 7].x, src), __shfl_sync(0xffffffffu, a[q & 7].y, src));
        const float mag = f.x * f.x + f.y * f.y, rd = __frcp_rn(mag);
        unsigned key = (__float_as_uint(fminf(mag, 3.0e38f)) & ~0xFu) | (unsigned)(15 - r);
        if (!(isfinite(f.x) && isfinite(f.y))) key = 0xFFFFFFF0u | (unsigned)(15 - r);
        if ((used >> r) & 1u) key = 0u;
        const unsigned best = __reduce_max_sync(0xffffffffu, key);
        const int p = 15 - (int)(best & 0xFu);
        if ((best >> 4) == 0u || (best >> 23) >= 255u) ok = false;
        used |= 1u << p;
        perm |= (unsigned long long)p << (4 * q);
        // (every lane's reciprocal, next to the maximum: off the chain)
        const float2 inv = make_float2(__shfl_sync(0xffffffffu, f.x * rd, p), __shfl_sync(0xffffffffu, -f.y * rd, p));
        const bool mine = r == p;
        if (mine) qinv = q;
        const float2 g = mine ? make_float2(-inv.x, -inv.y) : cmul(f, inv);
        const int ps = p + 16 * h;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float2 pj = make_float2(__shfl_sync(0xffffffffu, a[j].x, ps), __shfl_sync(0xffffffffu, a[j].y, ps));
            float2 o = mine ? make_float2(0.f, 0.f) : a[j];
            cfms(o, g, pj);
            a[j] = o;
        }
        if (h == (q >> 3)) a[q & 7] = make_float2(-g.x, -g.y);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) P[qinv * PIV + (int)((perm >> (4 * (8 * h + j))) & 15)] = a[j];
    return ok;
}

template <int H> __global__ void __launch_bounds__(ZtCfg<H>::THREADS, 4 / H) zinv_kernel(InvArgs a) {
    using Cfg = ZtCfg<H>;
    constexpr int ZT_WS = Cfg::WS;
    extern __shared__ __align__(16) unsigned char zt_smem[];
    __shared__ __align__(8) uint64_t mma_bar;
    __shared__ uint32_t s_tmem;
    __shared__ int s_bad;
    const int n = a.n, nb = (n + PIV - 1) / PIV, np = nb * PIV;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q = warp & 3, h = warp >> 2, r = 32 * q + lane, lr = lane & 15, lh = lane >> 4;
    const uint32_t base = (smem_u32(zt_smem) + 1023u) & ~1023u;
    unsigned char *gbase = zt_smem + (base - smem_u32(zt_smem));
    float2 *Wk = reinterpret_cast<float2 *>(gbase + Cfg::WK);      // [16][ZT_WS]: the pivot rows
    float2 *Pb = reinterpret_cast<float2 *>(gbase + Cfg::P);       // [2][16][16]: the pivot block's inverse, of even and odd steps
    float2 *Nd = reinterpret_cast<float2 *>(gbase + Cfg::BLK);     // [16][ZT_PS] each: W[K1, K1],
    float2 *Un = Nd + PIV * ZT_PS, *Rn = Un + PIV * ZT_PS;       // W[K1, K] and R'[:, K1] of the next block,
    float2 *Sn = Rn + PIV * ZT_PS;                               // and the next pivot block
    const uint32_t a_hi = base + Cfg::A, a_lo = a_hi + 16384, b_hi = base + Cfg::B, b_lo = b_hi + Cfg::B_BYTES;
    float2 *X = a.X + a.idx[blockIdx.x] * a.stride;
    if (tid == 0) {
        s_bad = 0;
        mbar_init(&mma_bar, 1);
        fence_mbar_init_cluster();
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(Cfg::TMEM)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // the block through shared memory, 64 columns at a time: whole rows of memory, a thread its own row
    float2 *T = reinterpret_cast<float2 *>(gbase);
    float2 w[32];
#pragma unroll 1
    for (int half = 0; half < H / 2; ++half) {
#pragma unroll
        for (int i = 0; i < 128 / Cfg::WARPS; ++i) {
            const int rr = 128 / Cfg::WARPS * warp + i;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int c = 64 * half + 32 * e + lane;
                T[rr * ZT_TS + 32 * e + lane] =
                    rr < n && c < n ? X[(size_t)rr * a.ld + c] : make_float2(rr == c ? 1.f : 0.f, 0.f);
            }
        }
        __syncthreads();
        if ((h >> 1) == half) {
#pragma unroll
            for (int i = 0; i < 32; ++i) w[i] = T[r * ZT_TS + 32 * (h & 1) + i];
        }
        __syncthreads();
    }
    // 16 columns of w by a warp-uniform half
    auto copy16 = [&](float2 *dst, int half) {
#pragma unroll
        for (int u = 0; u < PIV; ++u) dst[lr * ZT_PS + u] = half ? w[16 + u] : w[u];
    };
    if (warp == 0 && lh == 0) copy16(Sn, 0);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t trow = s_tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(64 * h);   // this thread's lane and columns
    if (warp == 0) {
        if (!warp_invert16_inplace(Sn, Pb) && lane == 0) s_bad = 1;
    }
    const uint32_t idesc = idesc_tf32(2 * np);
    int phase = 0;
    bool aborted = false;
#pragma unroll 1
    for (int kb = 0; kb < nb; ++kb) {
        const int k0 = kb * PIV, bk = k0 >> 5, hf = kb & 1, k1 = k0 + PIV, bk1 = k1 >> 5, hf1 = hf ^ 1;
        const bool krow = q == bk && lh == hf;           // this lane's row is a pivot row
        const bool nrow = q == bk1 && lh == hf1;         // ... of the next step
        // (a) the pivot rows; the column panel as A' and for the next pivot block; rows and columns
        // K zeroed
        if (nrow && h == bk1) copy16(Nd, hf1);
        if (h == bk) {
            if (nrow) copy16(Un, hf);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                float4 v;
                if (krow) {
                    v = make_float4(lr == 2 * j ? 1.f : 0.f, 0.f, lr == 2 * j + 1 ? 1.f : 0.f, 0.f);
                } else {
                    const float2 u0 = hf ? w[16 + 2 * j] : w[2 * j], u1 = hf ? w[17 + 2 * j] : w[2 * j + 1];
                    v = make_float4(-u0.x, -u0.y, -u1.x, -u1.y);
                }
                float4 hi, lo;
                split4(v, 1.f, hi, lo);
                st_shared_v4(a_hi + sw128(r, j), hi);
                st_shared_v4(a_lo + sw128(r, j), lo);
            }
        }
        if (krow) {
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                Wk[lr * ZT_WS + 32 * h + i] = w[i];
                w[i] = make_float2(0.f, 0.f);
            }
        }
        if (h == bk) {
#pragma unroll
            for (int u = 0; u < PIV; ++u) {
                if (hf) w[16 + u] = make_float2(0.f, 0.f);
                else w[u] = make_float2(0.f, 0.f);
            }
        }
        fence_proxy_async_smem();   // the A tiles, before the tensor core reads them
        __syncthreads();   // (P of this step was written before the last barrier)
        const float2 *P = Pb + hf * PIV * PIV;
        // (b) the next pivot block: R'[:, K1], then W[K1, K1] - W[K1, K] R'[:, K1], and its inverse
        if (kb + 1 < nb && warp < 8) {
            const int i = tid >> 4, c = tid & 15;
            float2 s0 = make_float2(0.f, 0.f), s1 = make_float2(0.f, 0.f);
#pragma unroll
            for (int u = 0; u < PIV; u += 2) {
                cfma(s0, P[i * PIV + u], Wk[u * ZT_WS + k1 + c]);
                cfma(s1, P[i * PIV + u + 1], Wk[(u + 1) * ZT_WS + k1 + c]);
            }
            Rn[i * ZT_PS + c] = make_float2(s0.x + s1.x, s0.y + s1.y);
            asm volatile("bar.sync 1, 256;" ::: "memory");
            s0 = Nd[i * ZT_PS + c];
            s1 = make_float2(0.f, 0.f);
#pragma unroll
            for (int u = 0; u < PIV; u += 2) {
                cfms(s0, Un[i * ZT_PS + u], Rn[u * ZT_PS + c]);
                cfms(s1, Un[i * ZT_PS + u + 1], Rn[(u + 1) * ZT_PS + c]);
            }
            Sn[i * ZT_PS + c] = make_float2(s0.x + s1.x, s0.y + s1.y);
            asm volatile("bar.sync 1, 256;" ::: "memory");
            if (warp == 0 && !warp_invert16_inplace(Sn, Pb + hf1 * PIV * PIV) && lane == 0) s_bad = 1;
        }
        if (warp > 0) {
            // (c) R' and the expanded B tiles: 32 columns c and u = 2j, 2j + 1 at a time; B row 2c = (Re,
            // -Im), row 2c + 1 = (Im, Re) of R'[u][c], split into hi and lo
#pragma unroll 1
            for (int it = warp - 1; it < 8 * H; it += Cfg::WARPS - 1) {
                const int c = 32 * (it % H) + lane, j = it / H;
                if (c >= np) continue;
                float2 x0, x1;
                const float2 *p0 = P + 2 * j * PIV;
                if (c >= k0 && c < k1) {
                    x0 = p0[c - k0];
                    x1 = p0[PIV + c - k0];
                } else {
                    x0 = x1 = make_float2(0.f, 0.f);
#pragma unroll
                    for (int v = 0; v < PIV; v += 2) {
                        const float2 w0 = Wk[v * ZT_WS + c], w1 = Wk[(v + 1) * ZT_WS + c];
                        const float4 a0 = *reinterpret_cast<const float4 *>(p0 + v);
                        const float4 a1 = *reinterpret_cast<const float4 *>(p0 + PIV + v);
                        cfma(x0, make_float2(a0.x, a0.y), w0);
                        cfma(x1, make_float2(a1.x, a1.y), w0);
                        cfma(x0, make_float2(a0.z, a0.w), w1);
                        cfma(x1, make_float2(a1.z, a1.w), w1);
                    }
                }
                // (lanes 4 apart start with different rows: eight distinct bank groups)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const bool im = ((lane >> 2) & 1) != e;
                    float4 hi, lo;
                    split4(im ? make_float4(x0.y, x0.x, x1.y, x1.x) : make_float4(x0.x, -x0.y, x1.x, -x1.y), 1.f, hi, lo);
                    st_shared_v4(b_hi + sw128(2 * c + im, j), hi);
                    st_shared_v4(b_lo + sw128(2 * c + im, j), lo);
                }
            }
            fence_proxy_async_smem();   // the operand tiles, before the tensor core reads them
            tc_fence_before();
            asm volatile("bar.sync 2, %0;" ::"n"(Cfg::THREADS - 32) : "memory");
            // (d) A' R' into tensor memory, the cross terms first
            if (warp == Cfg::WARPS - 1 && elect_one()) {
                tc_fence_after();
#pragma unroll
                for (int p = 0; p < 3; ++p) {   // lo*hi, hi*lo, hi*hi
                    const uint32_t aa = p == 0 ? a_lo : a_hi, bb = p == 1 ? b_lo : b_hi;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        tc_mma(s_tmem, desc_sw128(aa + 32 * kk), desc_sw128(bb + 32 * kk), idesc, p + kk > 0 ? 1u : 0u);
                }
                tc_commit(&mma_bar);
            }
            __syncwarp();
        }
        // (e) W += A' R'
        const bool done = mbar_wait_bounded(&mma_bar, (uint32_t)phase, a.tries);
        if (__all_sync(0xffffffffu, done)) {
            tc_fence_after();
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                float v[16];
                tc_ld16(trow + (uint32_t)(16 * g), v);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    w[8 * g + e].x += v[2 * e];
                    w[8 * g + e].y += v[2 * e + 1];
                }
            }
        }
        tc_fence_before();
        if (__syncthreads_or(!done)) {   // uniform: every thread leaves the loop
            if (tid == 0) atomicOr(a.status, ST_TIMEOUT);
            aborted = true;
            break;
        }
        tc_fence_after();
        phase ^= 1;
    }
    if (!aborted) {
#pragma unroll 1
        for (int half = 0; half < H / 2; ++half) {
            if ((h >> 1) == half) {
#pragma unroll
                for (int i = 0; i < 32; ++i) T[r * ZT_TS + 32 * (h & 1) + i] = w[i];
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < 128 / Cfg::WARPS; ++i) {
                const int rr = 128 / Cfg::WARPS * warp + i;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int c = 64 * half + 32 * e + lane;
                    if (rr < n && c < n) X[(size_t)rr * a.ld + c] = T[rr * ZT_TS + 32 * e + lane];
                }
            }
            __syncthreads();
        }
    } else {
        mbar_wait_bounded(&mma_bar, (uint32_t)phase, kDefaultWaitTries);   // an MMA that may still be in flight
    }
    if (tid == 0 && s_bad) atomicOr(a.status, ST_SINGULAR);
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(Cfg::TMEM) : "memory");
}

// *out = largest of n words
__global__ void __launch_bounds__(1024) max_words_kernel(size_t n, const uint32_t *v, int *out) {
    __shared__ uint32_t s[32];
    uint32_t m = 0;
    for (size_t i = threadIdx.x; i < n; i += 1024) m = max(m, v[i]);
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = __reduce_max_sync(0xffffffffu, s[threadIdx.x]);
        if (threadIdx.x == 0) *out = (int)m;
    }
}

// ----------------------------------------------------------------- host side

struct TaskBuf {   // device copy of host-built task lists (freed on the stream when done)
    int *dev = nullptr;
    cudaStream_t st = nullptr;
    ~TaskBuf() { dev_free(dev, st); }
};

helm_status upload_ints(const std::vector<int> &h, TaskBuf &b, cudaStream_t st) {
    b.st = st;
    helm_status s = dev_alloc((void **)&b.dev, h.size() * sizeof(int), "bcr: task list", st);
    if (s != HELM_OK) return s;
    cudaError_t e = cudaMemcpyAsync(b.dev, h.data(), h.size() * sizeof(int), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) { helm_set_error("bcr: task upload", e); return HELM_ECUDA; }
    return HELM_OK;
}

// partial tiles of the split-K products of helm_zgemm_batched and helm_zinv_batched: 64 MB (8 products of
// 256 x 256 split 16 ways)
constexpr size_t kSplitElems = (size_t)8 << 20;

// A recorded sequence of launches: every task list goes into one host array, uploaded with a
// single copy before the launches are enqueued (a copy from pageable host memory waits for the
// stream, so one copy per launch would serialise the host with the GPU at every launch).
struct Plan {
    cudaStream_t st;
    std::vector<int> ints;
    std::vector<std::function<helm_status(const int *)>> ops;
    std::vector<void *> scratch;   // device scratch of the launches, released after the last one
    float2 *split = nullptr;       // split-K partial tiles shared by the plan's GEMM launches (one
    size_t split_cap = 0;          // stream: each launch's reduction reads them before the next writes)
    explicit Plan(cudaStream_t s) : st(s) {}
    helm_status with_split(size_t elems) {
        helm_status s = dev_alloc((void **)&split, elems * sizeof(float2), "bcr: split-K tiles", st);
        if (s != HELM_OK) return s;
        scratch.push_back(split);
        split_cap = elems;
        return HELM_OK;
    }
    ~Plan() {
        for (void *p : scratch) dev_free(p, st);
    }
    int add(const std::vector<int> &v) {
        const int off = (int)ints.size();
        ints.insert(ints.end(), v.begin(), v.end());
        return off;
    }
    helm_status run() {
        TaskBuf tb;
        helm_status s = HELM_OK;
        if (!ints.empty() && (s = upload_ints(ints, tb, st)) != HELM_OK) return s;
        for (auto &op : ops)
            if ((s = op(tb.dev)) != HELM_OK) return s;
        return HELM_OK;
    }
};

ZOperand zop(const float2 *base, long long stride, int ld) {
    ZOperand o;
    o.base = base;
    o.stride = stride;
    o.ld = ld;
    return o;
}

helm_status gemm(const ZGemmArgs &a0, const std::vector<int> &tasks, Plan &pl) {
    if (tasks.empty()) return HELM_OK;
    const int off = pl.add(tasks), n = (int)(tasks.size() / 4);
    ZGemmArgs a = a0;
    for (int t = 0; t < n; ++t) {
        a.A.count = std::max<long long>(a.A.count, tasks[4 * t] + 1);
        a.B.count = std::max<long long>(a.B.count, tasks[4 * t + 1] + 1);
    }
    a.tries = wait_tries();
    a.flops = 8.0 * a.M * a.N * a.K * n;
    a.part = pl.split;
    a.part_cap = pl.split_cap;
    const cudaStream_t st = pl.st;
    pl.ops.push_back([a, off, n, st](const int *dev) mutable -> helm_status {
        a.tasks = dev + off;
        const cudaError_t e = launch_zgemm(a, n, st);
        if (e != cudaSuccess) { helm_set_error("bcr: tensor-core GEMM", e); return HELM_ECUDA; }
        return HELM_OK;
    });
    return HELM_OK;
}

// A family of n x n row-major blocks within a family of larger row-major matrices: the block
// at (row r0, column c0) of matrix idx (the larger matrices have row stride ld).
struct Fam {
    float2 *base;
    long long stride;
    int ld;
    Fam sub(int r0, int c0) const { return Fam{base + (long long)r0 * ld + c0, stride, ld}; }
    ZOperand op() const { return zop(base, stride, ld); }
};

// X[i] <- X[i]^{-1} for every block i of the list, n x n, symmetric above INV_MAX columns
helm_status invert_blocks(int n, Fam X, const std::vector<int> &blocks, int *status, Plan &pl) {
    const int count = (int)blocks.size();
    if (count == 0) return HELM_OK;
    const cudaStream_t st = pl.st;
    helm_status s;
    if (n <= INV_MAX) {
        const int off = pl.add(blocks);
        const bool small = n <= 64;
        const size_t smem = small ? ZtCfg<2>::SMEM : ZtCfg<4>::SMEM;
        cudaError_t e = ensure_dyn_smem(small ? (const void *)zinv_kernel<2> : (const void *)zinv_kernel<4>, smem);
        if (e != cudaSuccess) { helm_set_error("bcr: block inversion", e); return HELM_ECUDA; }
        InvArgs a{n, X.base, X.stride, X.ld, nullptr, status};
        a.tries = wait_tries();
        pl.ops.push_back([a, off, count, st, small, smem](const int *dev) mutable -> helm_status {
            a.idx = dev + off;
            if (small) HELM_TRACED(K_ZINV, st, (zinv_kernel<2><<<count, ZtCfg<2>::THREADS, smem, st>>>(a)));
            else HELM_TRACED(K_ZINV, st, (zinv_kernel<4><<<count, ZtCfg<4>::THREADS, smem, st>>>(a)));
            const cudaError_t e2 = cudaGetLastError();
            if (e2 != cudaSuccess) { helm_set_error("bcr: block inversion", e2); return HELM_ECUDA; }
            return HELM_OK;
        });
        return HELM_OK;
    }
    const int n1 = INV_MAX * ((n / INV_MAX + 1) / 2), n2 = n - n1;
    // X11 = D11^{-1}
    if ((s = invert_blocks(n1, X, blocks, status, pl)) != HELM_OK) return s;
    // scratch T (n1 x n2) and Tt = T^T (n2 x n1) per block: allocated now (stream-ordered, usable
    // by the launches enqueued later), released on the stream after the last launch that reads it
    float2 *T = nullptr, *Tt = nullptr;
    const long long ts = (long long)n1 * n2;
    if ((s = dev_alloc((void **)&T, (size_t)count * ts * sizeof(float2), "bcr: inversion scratch", st)) != HELM_OK)
        return s;
    if ((s = dev_alloc((void **)&Tt, (size_t)count * ts * sizeof(float2), "bcr: inversion scratch", st)) != HELM_OK) {
        dev_free(T, st);
        return s;
    }
    // (released by the plan after its last launch)
    pl.scratch.push_back(T);
    pl.scratch.push_back(Tt);
    const Fam X11 = X.sub(0, 0), X12 = X.sub(0, n1), X21 = X.sub(n1, 0), X22 = X.sub(n1, n1);
    const Fam FT{T, ts, n2}, FTt{Tt, ts, n1};
    std::vector<int> tk;
    auto run = [&](int M, int N, int K, Fam A, Fam B, const Fam *C0, Fam C, float sign) -> helm_status {
        // matrices of X by the block, of T and its transpose by the position in the batch
        auto id = [&](const Fam &f, int t) { return f.base == T || f.base == Tt ? t : blocks[t]; };
        tk.clear();
        for (int t = 0; t < count; ++t) tk.insert(tk.end(), {id(A, t), id(B, t), C0 ? id(*C0, t) : 0, id(C, t)});
        ZGemmArgs g;
        g.M = M; g.N = N; g.K = K;
        g.A = A.op();
        g.B = B.op();
        g.sign = sign;
        if (C0) g.C0 = C0->op();
        g.C = C.base;
        g.c_stride = C.stride;
        g.ldc = C.ld;
        g.status = status;
        return gemm(g, tk, pl);
    };
    // (X21 and X22 hold D21 and D22 until they are written)
    // T = X11 D12 = X11 D21^T;  Tt = D21 X11 (= T^T, X11 symmetric)
    if ((s = run(n1, n2, n1, X11, X21, nullptr, FT, 1.f)) != HELM_OK) return s;
    if ((s = run(n2, n1, n1, X21, X11, nullptr, FTt, 1.f)) != HELM_OK) return s;
    // X22 = S = D22 - D21 T, then its inverse
    if ((s = run(n2, n2, n1, X21, FTt, &X22, X22, -1.f)) != HELM_OK) return s;
    if ((s = invert_blocks(n2, X22, blocks, status, pl)) != HELM_OK) return s;
    // X12 = -T X22;  X21 = -X22 T^T;  X11 <- X11 - T X21
    if ((s = run(n1, n2, n2, FT, X22, nullptr, X12, -1.f)) != HELM_OK) return s;
    if ((s = run(n2, n1, n2, X22, FT, nullptr, X21, -1.f)) != HELM_OK) return s;
    return run(n1, n1, n2, FT, X12, &X11, X11, -1.f);
}

// images (bcr_solve.cu) of a part of the blocks in slots pairs[.][0] of D as matrices pairs[.][1]
helm_status image_blocks(const BgArgs &ba, BsPart part, const std::vector<int> &pairs, Plan &pl) {
    if (pairs.empty()) return HELM_OK;
    const int off = pl.add(pairs), count = (int)(pairs.size() / 2);
    const cudaStream_t st = pl.st;
    pl.ops.push_back([=](const int *dev) -> helm_status {
        const cudaError_t e = launch_bcr_image(ba.nz, part, ba.D, (long long)ba.nz * ba.nz, dev + off, count, ba.im, st);
        if (e != cudaSuccess) { helm_set_error("bcr: images", e); return HELM_ECUDA; }
        return HELM_OK;
    });
    return HELM_OK;
}

// products of images (bcr_gemm.cu), one launch
helm_status image_gemm(const BgArgs &ba, const std::vector<int> &tasks, Plan &pl) {
    if (tasks.empty()) return HELM_OK;
    const int off = pl.add(tasks), n = (int)(tasks.size() / BG_TASK);
    int products = n;
    for (int t = 0; t < n; ++t) products += (tasks[BG_TASK * t] & BG_TWO) != 0;
    const cudaStream_t st = pl.st;
    pl.ops.push_back([=](const int *dev) -> helm_status {
        BgArgs a = ba;
        a.tasks = dev + off;
        const cudaError_t e = launch_bcr_gemm(a, n, products, st);
        if (e != cudaSuccess) { helm_set_error("bcr: block products", e); return HELM_ECUDA; }
        return HELM_OK;
    });
    return HELM_OK;
}

// D[slots[t]] <- its inverse on and below the 128 x 128 blocks of the diagonal, for symmetric blocks:
// the 2 x 2 block inverse with the products on images of the parts (invert_blocks has them as 3xTF32
// GEMMs of FP32 blocks, with T^T and X21 as products of their own).  `node`: numbers the recursion.
int invert_nodes(int n) {   // nodes of the recursion on n columns
    if (n <= INV_MAX) return 0;
    const int n1 = INV_MAX * ((n / INV_MAX + 1) / 2);
    return 1 + invert_nodes(n1) + invert_nodes(n - n1);
}
helm_status invert_images(const BgArgs &ba, const std::vector<int> &slots, int r0, int n, int &node, Plan &pl) {
    const int count = (int)slots.size(), nz = ba.nz;
    if (n <= INV_MAX) {
        return invert_blocks(n, Fam{ba.D, (long long)nz * nz, nz}.sub(r0, r0), slots, ba.status, pl);
    }
    const int id = ba.im.n_sub + 8 * node++, n1 = INV_MAX * ((n / INV_MAX + 1) / 2), n2 = n - n1, r1 = r0 + n1;
    enum { D21, X11, T, X22, TT, X12 };
    std::vector<int> pairs, tasks;
    auto image = [&](int part, int pr, int pc, int m, int k) {
        pairs.clear();
        for (int t = 0; t < count; ++t) pairs.insert(pairs.end(), {slots[t], id + ba.im.sub * t + part});
        return image_blocks(ba, BsPart{pr, pc, m, k}, pairs, pl);
    };
    // parts A (row ra, column ca) and B: m x n products of inner length k to row ro, column co
    auto product = [&](int flags, int A, int ra, int ca, int B, int rb, int cb, int m, int nn, int k, int ro, int co, int out,
                       int out_t) {
        BgArgs a = ba;
        a.m = m; a.n = nn; a.k = k;
        a.ra = ra; a.ca = ca; a.rb = rb; a.cb = cb; a.ro = ro; a.co = co;
        tasks.clear();
        for (int t = 0; t < count; ++t) {
            const int v = id + ba.im.sub * t;
            tasks.insert(tasks.end(), {flags, v + A, v + B, (flags & BG_FP32) ? slots[t] : v + out, v + out_t, slots[t]});
        }
        return image_gemm(a, tasks, pl);
    };
    helm_status s;
    if ((s = invert_images(ba, slots, r0, n1, node, pl)) != HELM_OK ||
        (s = image(D21, r1, r0, n2, n1)) != HELM_OK || (s = image(X11, r0, r0, n1, n1)) != HELM_OK ||
        // T = X11 D21^T with T^T, D22 -= D21 T
        (s = product(BG_TR, X11, r0, r0, D21, r1, r0, n1, n2, n1, r0, r1, T, TT)) != HELM_OK ||
        (s = product(BG_NEG | BG_FP32, D21, r1, r0, TT, r1, r0, n2, n2, n1, r1, r1, 0, 0)) != HELM_OK ||
        (s = invert_images(ba, slots, r1, n2, node, pl)) != HELM_OK || (s = image(X22, r1, r1, n2, n2)) != HELM_OK ||
        // X12 = -T X22 (its transpose X21 to memory), X11 -= T X21
        (s = product(BG_NEG | BG_STORE, T, r0, r1, X22, r1, r1, n1, n2, n2, r0, r1, X12, 0)) != HELM_OK)
        return s;
    return product(BG_NEG | BG_FP32, T, r0, r1, X12, r0, r1, n1, n1, n2, r0, r0, 0, 0);
}

}  // namespace

int bcr_line(const GridGeom &g) { return g.nz + (g.nz & 1); }

int solve_line(const helm_factor_t *f) { return f->use_bcr ? bcr_line(f->op->g) : f->op->g.nz; }

bool bcr_supported(const GridGeom &g) { return (g.nz % 2) == 0 && g.nz >= 16 && g.nx >= 4; }

// ------------------------------------------------------------------ factor

helm_status bcr_factor(helm_factor_t *f) {
    helm_op *op = f->op;
    const GridGeom &g = op->g;
    // (an odd line has one more, decoupled, node here: pairs of entries on 16-byte boundaries)
    const int nx = g.nx, nz = bcr_line(g), ns = op->n_omega;
    const long long nz2 = (long long)nz * nz;
    const int half = nx / 2 + 1, quart = nx / 4 + 1, nk = (nx + 1) / 2;
    const cudaStream_t st = op->st;
    BcrData &b = f->bcr;
    b.half = half;
    helm_status s;
    // Images (bcr_solve.h), one family of matrices.  Kept: every line's inverse, and W, V, P, Q of
    // the lines eliminated at levels >= 1.  Working: the couplings.  At level 0 both couplings
    // through an odd line j are M_j = -C Dinv_j C (slot j / 2); above, U_k (to the next line of the
    // spacing) and L_k = U_{k - sp}^T, ping-pong by level.
    const size_t n_kept = (size_t)ns * (nx + 4 * (size_t)half);
    const int m_stride = half, eighth = nx / 8 + 1;
    const size_t m0 = n_kept, u0 = m0 + (size_t)ns * m_stride;
    const size_t n_sub = u0 + 2 * (size_t)ns * (quart + eighth);   // parts of a level's blocks (BsImages)
    const int sub = 8 * std::max(1, invert_nodes(nz));
    const size_t n_mat = n_sub + (nz > INV_MAX ? (size_t)sub * ns * quart : 0);
    const size_t n_img = n_sub + (nz > INV_MAX ? 2 * (size_t)ns * quart : 0);
    const int u_stride[2] = {quart, eighth};
    auto u_base = [&](int buf, int which) {   // first matrix of U (which = 0) or L (1) of a buffer
        return u0 + (size_t)ns * (buf == 0 ? which * quart : 2 * quart + which * eighth);
    };
    const BsLayout lay = bs_layout(nz);
    if ((s = dev_alloc((void **)&b.img, n_kept * lay.mat_bytes, "bcr: blocks", st)) != HELM_OK ||
        (s = dev_alloc((void **)&b.shift, n_mat * sizeof(int), "bcr: scales", st)) != HELM_OK ||
        (s = dev_alloc((void **)&b.gsmall, kSmallMaxima * sizeof(float), "bcr: maxima", st)) != HELM_OK)
        return s;
    // working arrays: the diagonal blocks of the even lines (FP32, an eliminated line's is inverted in
    // place), the working images, level 0's generators (40 bytes an entry) and recurrences (52), the
    // maxima; one allocation, whose size is the same in every factor of a grid (several of different
    // sizes next to the kept blocks left the pool remapping memory: 2.5 ms a factor at 256^2)
    const size_t n_gen = (size_t)ns * (nx / 2) * g.nz;
    auto up = [](size_t v) { return (v + 1023) & ~(size_t)1023; };
    const size_t d_bytes = up((size_t)ns * nk * nz2 * sizeof(float2)), w_bytes = up((n_img - n_kept) * lay.mat_bytes);
    unsigned char *work = nullptr;
    struct Work {
        unsigned char **p;
        cudaStream_t st;
        ~Work() { dev_free(*p, st); }
    } work_owner{&work, st};
    if ((s = dev_alloc((void **)&work, d_bytes + w_bytes + up(n_gen * 92) + n_mat * sizeof(uint32_t), "bcr: work", st)) != HELM_OK)
        return s;
    float2 *D = reinterpret_cast<float2 *>(work);
    BsImages im;
    im.kept = b.img;
    im.work = work + d_bytes;
    im.mx = reinterpret_cast<uint32_t *>(work + d_bytes + w_bytes + up(n_gen * 92));
    im.n_kept = (int)n_kept;
    im.shift = b.shift;
    im.n_sub = (int)n_sub;
    im.sub = sub;
    im.sub0 = (int)(n_sub - n_kept);
    cudaError_t e;
    if ((e = cudaMemsetAsync(im.mx, 0, n_mat * sizeof(uint32_t), st)) != cudaSuccess) {
        helm_set_error("bcr: maxima", e);
        return HELM_ECUDA;
    }
    BgArgs ba{};
    ba.nz = nz;
    ba.im = im;
    ba.D = D;
    ba.status = op->status;
    ba.tries = wait_tries();
    Plan pl(st);
    auto mat = [&](int kind, int sy, int slot) { return (int)bs_matrix_index(nx, ns, half, kind << 24 | slot, sy); };
    auto dblk = [&](int sy, int k) { return sy * nk + k / 2; };   // D block of an even line
    // inverses of the blocks pairs[.][0] of D as matrices pairs[.][1]
    auto invert = [&](const std::vector<int> &pairs) -> helm_status {
        std::vector<int> slots;
        for (size_t t = 0; t < pairs.size(); t += 2) slots.push_back(pairs[t]);
        if (nz > INV_MAX) {
            uint32_t *mxs = im.mx + n_sub;
            const size_t bytes = (size_t)sub * ns * quart * sizeof(uint32_t);
            pl.ops.push_back([=](const int *) -> helm_status {   // (the level before's maxima)
                const cudaError_t e2 = cudaMemsetAsync(mxs, 0, bytes, st);
                if (e2 != cudaSuccess) { helm_set_error("bcr: maxima", e2); return HELM_ECUDA; }
                return HELM_OK;
            });
        }
        int node = 0;
        const helm_status s1 = invert_images(ba, slots, 0, nz, node, pl);
        return s1 != HELM_OK ? s1 : image_blocks(ba, BsPart{0, 0, nz, nz}, pairs, pl);
    };
    // level 0: generators of the odd lines' inverses, their images and the even lines' blocks
    {
        const int no = nx / 2, n_line = ns * no;
        std::vector<int> dst;
        for (int sy = 0; sy < ns; ++sy)
            for (int j = 1; j < nx; j += 2) dst.insert(dst.end(), {mat(BS_DINV, sy, j), (int)m0 + sy * m_stride + j / 2});
        const int off = pl.add(dst);
        TriGen tg;
        TriScan ts;
        tg.u = reinterpret_cast<float4 *>(work + d_bytes + w_bytes);
        tg.v = tg.u + n_gen;
        ts.delta = (double2 *)(tg.v + n_gen);
        ts.gamma = ts.delta + n_gen;
        ts.r = ts.gamma + n_gen;
        tg.e = (int2 *)(ts.r + n_gen);
        ts.re = (int *)(tg.e + n_gen);
        const Coup cp = coup_of(g);
        const double2 *diag = op->diag;
        float2 *D0 = D;
        pl.ops.push_back([=](const int *dev) -> helm_status {
            HELM_TRACED(K_BCR_L0, st, (tri_scan_kernel<<<(2 * n_line + 32 - 1) / 32, 32, 0, st>>>(g, n_line, diag, ts)));
            HELM_TRACED(K_BCR_L0, st, (tri_gen_kernel<<<n_line, 256, 0, st>>>(g, cp, n_line, diag, ts, tg, dev + off, im)));
            HELM_TRACED(K_BCR_IMAGE, st, (tri_image_kernel<<<dim3(n_line, (lay.nzr + 31) / 32), 128, 0, st>>>(
                                             g.nz, lay.n_chunk, lay.nzr, tg, dev + off, cp, im, lay.mat_bytes)));
            HELM_TRACED(K_BCR_L0, st, (bcr_level0_kernel<<<dim3(ns * ((nx + 1) / 2), (nz + 31) / 32, (nz + 255) / 256), 128, 0, st>>>(
                                          g, nz, cp, D0, diag, tg)));
            const cudaError_t e2 = cudaGetLastError();
            if (e2 != cudaSuccess) { helm_set_error("bcr: level 0", e2); return HELM_ECUDA; }
            return HELM_OK;
        });
    }
    int cur = 1, levels = 1;   // U, L of the spacing in buffer cur (from level 2 on)
    for (int sp = 2; sp < nx; sp *= 2, ++levels) {
        std::vector<int> inv;
        for (int sy = 0; sy < ns; ++sy)
            for (int j = sp; j < nx; j += 2 * sp) inv.insert(inv.end(), {dblk(sy, j), mat(BS_DINV, sy, j)});
        if ((s = invert(inv)) != HELM_OK) return s;
        const int nxt = cur ^ 1;
        // couplings of line k to its neighbours at distance sp
        auto Uc = [&](int sy, int k) { return sp == 2 ? (int)m0 + sy * m_stride + k / 2 : (int)u_base(cur, 0) + sy * u_stride[cur] + k / sp; };
        auto Lc = [&](int sy, int k) { return sp == 2 ? (int)m0 + sy * m_stride + k / 2 - 1 : (int)u_base(cur, 1) + sy * u_stride[cur] + k / sp; };
        auto Un = [&](int sy, int k) { return (int)u_base(nxt, 0) + sy * u_stride[nxt] + k / (2 * sp); };
        auto Ln = [&](int sy, int k) { return (int)u_base(nxt, 1) + sy * u_stride[nxt] + k / (2 * sp); };
        std::vector<int> t1, t2;   // V, W with their transposes P, Q; the new couplings and D -= L W^T + U V^T
        auto add = [](std::vector<int> &t, int flags, int ia, int ib, int out, int ia2 = -1, int ib2 = -1) {
            t.insert(t.end(), {flags, ia, ib, out, ia2, ib2});
        };
        for (int sy = 0; sy < ns; ++sy) {
            for (int j = sp; j < nx; j += 2 * sp) {
                const int di = mat(BS_DINV, sy, j), u = Uc(sy, j - sp);
                add(t1, BG_TR, u, di, mat(BS_V, sy, j / 2), mat(BS_P, sy, j / 2));   // V_j = U_{j-s} Dinv_j, P_j = V_j^T
                if (j + sp < nx) add(t1, BG_TR, Lc(sy, j + sp), di, mat(BS_W, sy, j / 2), mat(BS_Q, sy, j / 2));   // W_j, Q_j
            }
            for (int k = 0; k < nx; k += 2 * sp) {
                const int a = k - sp, c = k + sp;
                const int l = a >= 0 ? Lc(sy, k) : -1, w = a >= 0 ? mat(BS_W, sy, a / 2) : -1;   // D_k -= L_k W_a^T + U_k V_c^T
                const int u = c < nx ? Uc(sy, k) : -1, v = c < nx ? mat(BS_V, sy, c / 2) : -1;
                if (a >= 0) add(t2, BG_FP32 | BG_NEG | (c < nx ? BG_TWO : 0), l, w, dblk(sy, k), u, v);
                else if (c < nx) add(t2, BG_FP32 | BG_NEG, u, v, dblk(sy, k));
                if (k >= 2 * sp) add(t2, BG_NEG, Lc(sy, k), mat(BS_V, sy, a / 2), Ln(sy, k));          // L_k <- -L_k V_a^T
                if (k + 2 * sp < nx) add(t2, BG_NEG, Uc(sy, k), mat(BS_W, sy, c / 2), Un(sy, k));      // U_k <- -U_k W_c^T
            }
        }
        uint32_t *mxn = im.mx + u_base(nxt, 0);
        const size_t mxb = 2 * (size_t)ns * u_stride[nxt] * sizeof(uint32_t);
        if ((s = image_gemm(ba, t1, pl)) != HELM_OK) return s;
        pl.ops.push_back([=](const int *) -> helm_status {   // (the buffer's maxima of two levels ago)
            const cudaError_t e2 = cudaMemsetAsync(mxn, 0, mxb, st);
            if (e2 != cudaSuccess) { helm_set_error("bcr: maxima", e2); return HELM_ECUDA; }
            return HELM_OK;
        });
        if ((s = image_gemm(ba, t2, pl)) != HELM_OK) return s;
        cur = nxt;
    }
    // the last line left: line 0
    {
        std::vector<int> last;
        for (int sy = 0; sy < ns; ++sy) last.insert(last.end(), {dblk(sy, 0), mat(BS_DINV, sy, 0)});
        if ((s = invert(last)) != HELM_OK) return s;
        int *out = op->status + 2;   // the largest entry of the inverses (the matrices 0 .. ns nx - 1)
        const uint32_t *mxd = im.mx;
        pl.ops.push_back([=](const int *) -> helm_status {
            HELM_TRACED(K_BCR_IMAGE, st, (max_words_kernel<<<1, 1024, 0, st>>>((size_t)ns * nx, mxd, out)));
            const cudaError_t e2 = cudaGetLastError();
            if (e2 != cudaSuccess) { helm_set_error("bcr: maxima", e2); return HELM_ECUDA; }
            return HELM_OK;
        });
    }
    if ((s = pl.run()) != HELM_OK) return s;
    // the solve's steps and tasks (the same for every system), built once
    std::vector<int> all;
    b.terms = 0;
    auto step = [&](int first) {
        const int n = (int)all.size() / 8 - first;
        if (n > 0) b.steps.push_back(BsStep{first, n, all[8 * (size_t)first + 1] & 15});
    };
    auto add = [&](int line, int type, std::initializer_list<std::pair<int, int>> terms) {
        const size_t o = all.size();
        all.resize(o + 8, 0);
        all[o] = line;
        all[o + 1] = type | (int)terms.size() << 4;
        int q = 2;
        for (auto &t : terms) { all[o + q++] = t.first; all[o + q++] = t.second; }
        b.terms += (long long)terms.size();
    };
    auto blk_of = [](int kind, int slot) { return kind << 24 | slot; };
    auto pair_step = [&](int sp, int type, int kind_a, int kind_c, int shift) {   // kept lines and their two neighbours
        const int first = (int)all.size() / 8;
        for (int k = 0; k < nx; k += 2 * sp) {
            const int a = k - sp, c = k + sp;
            if (a >= 0 && c < nx) add(k, type, {{blk_of(kind_a, a >> shift), a}, {blk_of(kind_c, c >> shift), c}});
            else if (a >= 0) add(k, type, {{blk_of(kind_a, a >> shift), a}});
            else if (c < nx) add(k, type, {{blk_of(kind_c, c >> shift), c}});
        }
        step(first);
    };
    pair_step(1, BS_FWD0, BS_DINV, BS_DINV, 0);
    for (int l = 1, sp = 2; l < levels; ++l, sp *= 2) pair_step(sp, BS_FWD, BS_W, BS_V, 1);
    add(0, BS_LAST, {{blk_of(BS_DINV, 0), 0}});
    step((int)all.size() / 8 - 1);
    for (int l = levels - 1; l >= 0; --l) {
        const int sp = 1 << l, first = (int)all.size() / 8;
        for (int j = sp; j < nx; j += 2 * sp) {
            if (l == 0) add(j, BS_BWD0, {{blk_of(BS_DINV, j), j}});
            else if (j + sp < nx)
                add(j, BS_BWD, {{blk_of(BS_DINV, j), j}, {blk_of(BS_P, j / 2), j - sp}, {blk_of(BS_Q, j / 2), j + sp}});
            else add(j, BS_BWD, {{blk_of(BS_DINV, j), j}, {blk_of(BS_P, j / 2), j - sp}});
        }
        step(first);
    }
    if ((int)b.steps.size() > BS_MAX_PHASE) { helm_set_msg("bcr: too many levels"); return HELM_EINVAL; }
    if ((s = dev_alloc((void **)&b.tasks, all.size() * sizeof(int), "bcr: solve plan", st)) != HELM_OK ||
        (s = dev_alloc((void **)&b.ctl, bs_ctl_words((int)b.steps.size(), ns) * sizeof(unsigned), "bcr: solve counters",
                       st)) != HELM_OK)
        return s;
    if ((e = cudaMemcpyAsync(b.tasks, all.data(), all.size() * sizeof(int), cudaMemcpyHostToDevice, st)) != cudaSuccess) {
        helm_set_error("bcr: solve plan", e);
        return HELM_ECUDA;
    }
    // the work blocks are released on the stream after the last kernel that reads them
    return HELM_OK;
}

void bcr_free(helm_factor_t *f) {
    const cudaStream_t st = f->op ? f->op->st : nullptr;
    BcrData &b = f->bcr;
    dev_free(b.img, st);
    dev_free(b.shift, st);
    dev_free(b.tasks, st);
    dev_free(b.ctl, st);
    dev_free(b.gsmall, st);
    b = BcrData();
}

// ------------------------------------------------------------------- solve

size_t bcr_maxima_elems(const GridGeom &g, size_t cols) { return 2 * cols * g.nx * (size_t)bs_layout(g.nz).ng; }

// x = A~^{-1} r for every system and right-hand side, complex FP32: r [n_sys][nrhs][N] is the
// working vector (overwritten), x [n_sys][nrhs][N] the result.  skip: launches do nothing
// while it is set (refinement finished).  maxima: bcr_maxima_elems floats of scratch; prepared: the
// first half holds the maxima of r already and the factor's counters are zero.
helm_status bcr_solve(const helm_factor_t *f, int nrhs, float2 *r, float2 *x, float *maxima, bool prepared, const int *skip,
                      const int *frozen) {
    const helm_op *op = f->op;
    const GridGeom &g = op->g;
    const BcrData &b = f->bcr;
    BsArgs a{};
    a.nx = g.nx;
    a.nz = bcr_line(g);
    a.edge = g.nz - 1;
    a.ns = op->n_omega;
    a.nrhs = nrhs;
    a.half = b.half;
    a.r = r;
    a.x = x;
    a.gr = maxima;
    a.gx = maxima + bcr_maxima_elems(g, (size_t)a.ns * nrhs) / 2;
    a.img = b.img;
    a.shift = b.shift;
    a.tasks = b.tasks;
    a.cx_in = (float)coup_x(g, 1);
    a.cx_edge = (float)coup_x(g, 0);
    a.ctl = b.ctl;
    a.status = op->status;
    a.skip = skip;
    a.frozen = frozen;
    a.tries = wait_tries();
    const double flops = 8.0 * g.nz * g.nz * nrhs * (double)b.terms * a.ns;
    const cudaError_t e = launch_bcr_solve(a, b.steps.data(), (int)b.steps.size(), prepared, flops, op->st);
    if (e != cudaSuccess) { helm_set_error("bcr solve", e); return HELM_ECUDA; }
    return HELM_OK;
}

// ------------------------------------------------ building blocks at the ABI (helm_blas.h)

helm_status blas_zgemm(int batch, int M, int N, int K, const float2 *A, long long sa, int lda, const float2 *Bt,
                       long long sb, int ldb, float sign, const float2 *C0, float2 *C, long long sc, int ldc,
                       cudaStream_t st, int *status) {
    ZGemmArgs a;
    a.M = M; a.N = N; a.K = K;
    a.A = zop(A, sa, lda);
    a.B = zop(Bt, sb, ldb);
    a.sign = sign;
    if (C0) a.C0 = zop(C0, sc, ldc);
    a.C = C; a.c_stride = sc; a.ldc = ldc;
    a.status = status;
    std::vector<int> tasks;
    for (int t = 0; t < batch; ++t) tasks.insert(tasks.end(), {t, t, t, t});
    Plan pl(st);
    helm_status s = pl.with_split(kSplitElems);
    if (s == HELM_OK) s = gemm(a, tasks, pl);
    return s == HELM_OK ? pl.run() : s;
}

helm_status blas_zinv(int batch, int n, const float2 *A, long long sa, int lda, float2 *X, long long sx, int ldx,
                      cudaStream_t st, int *status) {
    std::vector<int> blocks(batch);
    for (int t = 0; t < batch; ++t) blocks[t] = t;
    if (A != X) {   // copy into X first: the recursion works in place on the output blocks
        // blocks stacked without gaps on both sides are one 2D copy of batch * n rows
        const bool stacked = sa == (long long)n * lda && sx == (long long)n * ldx;
        cudaError_t e = cudaMemcpy2DAsync(X, (size_t)ldx * sizeof(float2), A, (size_t)lda * sizeof(float2),
                                          (size_t)n * sizeof(float2), (size_t)n * (stacked ? batch : 1),
                                          cudaMemcpyDeviceToDevice, st);
        for (int t = 1; !stacked && t < batch && e == cudaSuccess; ++t)
            e = cudaMemcpy2DAsync(X + (long long)t * sx, (size_t)ldx * sizeof(float2), A + (long long)t * sa,
                                  (size_t)lda * sizeof(float2), (size_t)n * sizeof(float2), (size_t)n,
                                  cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) { helm_set_error("helm_zinv_batched: copy", e); return HELM_ECUDA; }
    }
    const Fam f{X, sx, ldx};
    Plan pl(st);
    helm_status s = pl.with_split(kSplitElems);
    if (s == HELM_OK) s = invert_blocks(n, f, blocks, status, pl);
    return s == HELM_OK ? pl.run() : s;
}

}  // namespace helm

// ------------------------------------------------------------------ C ABI (helm_blas.h)

#include "helm_blas.h"

namespace {
struct DevStatus {   // a device status word for the building-block calls
    int *p = nullptr;
    cudaStream_t st;
    explicit DevStatus(cudaStream_t s) : st(s) {}
    ~DevStatus() { ::dev_free(p, st); }
};
}  // namespace

extern "C" helm_status helm_zgemm_batched(int32_t batch, int32_t M, int32_t N, int32_t K, const helm_c64 *A, int64_t sa,
                                          int32_t lda, const helm_c64 *Bt, int64_t sb, int32_t ldb, float sign,
                                          const helm_c64 *C0, helm_c64 *C, int64_t sc, int32_t ldc, void *stream) {
    if (batch < 0 || batch > 65535 || M < 1 || N < 1 || K < 1 || (K & 1) || !A || !Bt || !C || lda < K || ldb < K ||
        ldc < N || (lda & 1) || (ldb & 1) || (sa & 1) || (sb & 1) || (sign != 1.f && sign != -1.f) ||
        ((uintptr_t)A & 15) || ((uintptr_t)Bt & 15)) {
        helm_set_msg("helm_zgemm_batched: bad sizes, strides, alignment or sign");
        return HELM_EINVAL;
    }
    if (batch == 0) return HELM_OK;
    cudaStream_t st = (cudaStream_t)stream;
    DevStatus ds(st);
    helm_status s = dev_alloc((void **)&ds.p, sizeof(int), "helm_zgemm_batched: status", st);
    if (s != HELM_OK) return s;
    cudaError_t e = cudaMemsetAsync(ds.p, 0, sizeof(int), st);
    if (e != cudaSuccess) { helm_set_error("helm_zgemm_batched", e); return HELM_ECUDA; }
    return helm::blas_zgemm(batch, M, N, K, (const float2 *)A, sa, lda, (const float2 *)Bt, sb, ldb, sign,
                            (const float2 *)C0, (float2 *)C, sc, ldc, st, ds.p);
}

extern "C" helm_status helm_zinv_batched(int32_t batch, int32_t n, const helm_c64 *A, int64_t sa, int32_t lda,
                                         helm_c64 *X, int64_t sx, int32_t ldx, void *stream) {
    if (batch < 0 || batch > 65535 || n < 2 || (n & 1) || !A || !X || lda < n || ldx < n || (lda & 1) || (ldx & 1) ||
        (sa & 1) || (sx & 1) || ((uintptr_t)A & 15) || ((uintptr_t)X & 15)) {
        helm_set_msg("helm_zinv_batched: bad sizes, strides or alignment");
        return HELM_EINVAL;
    }
    if (batch == 0) return HELM_OK;
    cudaStream_t st = (cudaStream_t)stream;
    DevStatus ds(st);
    helm_status s = dev_alloc((void **)&ds.p, sizeof(int), "helm_zinv_batched: status", st);
    if (s != HELM_OK) return s;
    cudaError_t e = cudaMemsetAsync(ds.p, 0, sizeof(int), st);
    if (e != cudaSuccess) { helm_set_error("helm_zinv_batched", e); return HELM_ECUDA; }
    if ((s = helm::blas_zinv(batch, n, (const float2 *)A, sa, lda, (float2 *)X, sx, ldx, st, ds.p)) != HELM_OK) return s;
    int h = 0;
    e = cudaMemcpyAsync(&h, ds.p, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) { helm_set_error("helm_zinv_batched", e); return HELM_ECUDA; }
    if (h & helm::ST_SINGULAR) { helm_set_msg("helm_zinv_batched: zero or non-finite pivot"); return HELM_ESINGULAR; }
    return HELM_OK;
}
