// bicgstab.cu -- mixed-precision BiCGStab(l) (Sec. 6.1; Sleijpen and Fokkema)
// on the full-lattice operator M = 2m + D, and its C-ABI entry point.
//
// Each cycle: l BiCG steps (two matvecs each) followed by a minimal-residual
// step over the l new directions, orthogonalised by modified Gram-Schmidt.
// Vectors r_0..r_l, u_0..u_l and the shadow residual live in the sloppy
// format; x, b and true residuals in FP64; every scalar (rho, alpha, omega,
// the Gram-Schmidt coefficients tau, sigma, gamma) is computed on the device
// by the kernels that use it, so a cycle is one fixed kernel sequence (captured
// once as a CUDA graph).  A reliable update (FP64 true residual)
// ends a cycle when |r| has dropped below delta times its maximum since the
// previous one, or when the iterated residual meets the target.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <type_traits>
#include <vector>

#include "blas.h"
#include "cg.h"
#include "codecs.cuh"
#include "internal.h"
#include "launch.cuh"
#include "reduce.cuh"

namespace hisq {

namespace {

constexpr int kMaxL = 8;
constexpr int kBlock = 256;
constexpr int kMaxBlocks = 304;   // blocks with sites of the vector kernels (two a SM; more rows cost the next kernel's sums)
constexpr int kGroup = 4;         // fields of a kind whose loads a thread issues before it stores any (template
                                  // argument G of the u and r updates: one on large lattices, more threads instead)
constexpr int kMaxRows = 4096;    // stencil block sums that the next kernel's blocks sum themselves

struct BState {
    double rho_re[kMaxL], rho_im[kMaxL];          // rho_j of the cycle's steps
    double al_re[kMaxL], al_im[kMaxL];            // alpha_j
    double rhoc_re, rhoc_im, alc_re, alc_im;      // -omega rho and alpha carried from the previous cycle
    double dot[3];                                // Re, Im <rt, v> and |v|^2 where they are summed once
    double tau_re[kMaxL + 1][kMaxL + 1], tau_im[kMaxL + 1][kMaxL + 1];
    double gp_re[kMaxL + 1], gp_im[kMaxL + 1];    // gamma'
    double rr, rr_max, delta2, stop2, tiny2;
    double rt2;   // |rt|^2 of the shadow residual
    double brk2;  // breakdown when |<rt, v>|^2 <= brk2 |rt|^2 |v|^2
    int active, reason, cycles, l;
};

// A cycle is a chain of kernels each of which sums its predecessor's block
// partials itself (every block, one fixed order) and takes its scalars from
// them, so no completion counter, last-block tail or one-thread launch lies
// between: u update (beta from <rt, r_j>), M u_j with <rt, u_{j+1}> in its
// epilogue, r and x update (alpha), M r_j with <rt, r_{j+1}>, the l
// Gram-Schmidt passes, and the final update.  The last block of each grid has
// no sites and writes the scalars to the state.  16^3x32 sites, 20-bit: 45
// launches of about 10 us a cycle before, 21 now.
struct BArgs {
    int vh;
    size_t hb;               // bytes of one half-lattice sloppy field
    size_t fb;               // bytes of one full sloppy field (2 halves)
    char *R;                 // r_0..r_l, fb apart
    char *U;                 // u_0..u_l
    const char *rt;          // shadow residual
    double *x64;             // FP64 full field (two planar halves, 48*vh bytes each)
    int j;                   // step
    int rows;                // rows of partials to sum; 0: the sums are in the state
    double *part_in, *part_out;
    BState *b;
    const int *active;
    int *err;
    RedBuf red;
};

__device__ __forceinline__ bool skip(const int *active) { return active && *(volatile const int *)active == 0; }

__device__ __forceinline__ void cdiv(double ar, double ai, double br, double bi, double &qr, double &qi)
{
    const double d = 1.0 / (br * br + bi * bi);
    qr = (ar * br + ai * bi) * d;
    qi = (ai * br - ar * bi) * d;
}

__device__ void b_stop(BState *b, int reason)
{
    b->reason = reason;
    b->active = 0;
}

// a value in the compute precision as FP64
__device__ __forceinline__ double widen(float v) { return f2d_bits(v); }
__device__ __forceinline__ double widen(double v) { return v; }

// site s of the full lattice: half s / vh, index s % vh of it
struct Site {
    int h, i;
};
__device__ __forceinline__ Site site_of(int s, int vh) { return s < vh ? Site{0, s} : Site{1, s - vh}; }

// The three sums of the pass or kernel before: the state's, or summed here (thread 0 of tot).
template <typename real>
__device__ __forceinline__ void dot_sums(const BArgs &a, double *tot)
{
    if (a.rows == 0) {
        if (threadIdx.x < 3) tot[threadIdx.x] = a.b->dot[threadIdx.x];
        __syncthreads();
        return;
    }
    RedBuf rb{};
    rb.partials = a.part_in;
    sum_partials<3, real>(rb, (unsigned)a.rows, tot);
}

// NR sums over `rows` rows, a warp a value: FP32 rows in FP32 pairs, FP64 rows in FP64; every thread
// may read tot afterwards.
template <int NR, typename real>
__device__ __forceinline__ void sum_rows(const real *part, int rows, double *tot)
{
    constexpr int U = 10, W = kBlock / 32, K = (NR + W - 1) / W;  // values a warp: v0, v0 + W, ..., loaded together
    const int lane = threadIdx.x & 31, v0 = threadIdx.x >> 5;
    if constexpr (std::is_same<real, double>::value) {
        for (int v = v0; v < NR; v += W) {
            double w[1] = {0.0};
            for (int r = lane; r < rows; r += 32) w[0] += __ldcg(part + (size_t)r * NR + v);
            warp_sum<1, double>(w);
            if (lane == 0) tot[v] = w[0];
        }
    } else {
        FF w[K];
#pragma unroll
        for (int k = 0; k < K; k++) w[k] = {0.0f, 0.0f};
        for (int r0 = lane; r0 < rows; r0 += 32 * U) {
            float t[K][U];
#pragma unroll
            for (int k = 0; k < K; k++)
#pragma unroll
                for (int u = 0; u < U; u++)
                    t[k][u] = v0 + k * W < NR && r0 + 32 * u < rows
                                  ? __ldcg(part + (size_t)(r0 + 32 * u) * NR + v0 + k * W) : 0.0f;
#pragma unroll
            for (int u = 0; u < U; u++)
#pragma unroll
                for (int k = 0; k < K; k++) w[k] = ff_add(w[k], FF{t[k][u], 0.0f});
        }
        warp_sum_ff<K>(w);
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < K; k++)
                if (v0 + k * W < NR) tot[v0 + k * W] = (double)w[k].hi + (double)w[k].lo;
    }
    __syncthreads();
}

// one site's <x, y> = conj(x) y and |y|^2 added to v
template <typename real>
__device__ __forceinline__ void dot_site(const real x[6], const real y[6], real v[3])
{
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const real xr = x[2 * c], xi = x[2 * c + 1], yr = y[2 * c], yi = y[2 * c + 1];
        v[0] += xr * yr + xi * yi;
        v[1] += xr * yi - xi * yr;
        v[2] += yr * yr + yi * yi;
    }
}

// The dot sums of many rows once, into the state: a large lattice's stencil pass, whose rows every block of
// the next kernel would read.  FP32 rows are summed in FP32 pairs.
template <typename T>
__global__ void __launch_bounds__(kBlock) dot_rows_kernel(BArgs a)
{
    using V = std::conditional_t<std::is_same<T, double>::value, double, ff>;
    pdl_wait();
    pdl_launch_dependents();
    if (skip(a.active)) return;
    const T *part = reinterpret_cast<const T *>(a.part_in);
    V v[3] = {V(0), V(0), V(0)};
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < a.rows; r += gridDim.x * blockDim.x)
#pragma unroll
        for (int k = 0; k < 3; k++) v[k] = v[k] + V(__ldcg(part + (size_t)r * 3 + k));
    __shared__ double tot[3];
    if (reduce_grid<3>(v, a.red, tot) && threadIdx.x == 0)
        for (int k = 0; k < 3; k++) a.b->dot[k] = tot[k];
}

// <rt, v> and |v|^2 over the full lattice, into the state: r_0 at a start or restart, and the stencil's
// output where its block sums would not fit their buffer
template <int SF, typename real>
__global__ void __launch_bounds__(kBlock) dot_kernel(BArgs a, const char *v)
{
    pdl_wait();
    if (skip(a.active)) return;
    real s3[3] = {0, 0, 0};
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < 2 * a.vh; s += gridDim.x * blockDim.x) {
        const Site q = site_of(s, a.vh);
        real x[6], y[6];
        Spinor<SF>::load(a.rt + q.h * a.hb, a.vh, q.i, x);
        Spinor<SF>::load(v + q.h * a.hb, a.vh, q.i, y);
        dot_site(x, y, s3);
    }
    pdl_launch_dependents();
    __shared__ double tot[3];
    if (reduce_grid<3>(s3, a.red, tot) && threadIdx.x == 0)
        for (int k = 0; k < 3; k++) a.b->dot[k] = tot[k];
}

// u_i = r_i - beta u_i, i = 0..j, with rho1 = <rt, r_j>, beta = alpha rho1 / rho0.
// Breakdown: rho1 (nearly) orthogonal relative to |rt| |r_j|, or a rho0 too small to divide by.
template <int SF, typename real, int G>
__global__ void __launch_bounds__(kBlock) u_multi_kernel(BArgs a)
{
    pdl_wait();
    if (skip(a.active)) return;
    __shared__ double tot[3];
    __shared__ real be_sh[2];
    __shared__ int ok_sh;
    // the first site's fields are loaded before the sums, and the next site's after a site's stores
    constexpr int C = Spinor<SF>::chunks;
    const int step = (int)(gridDim.x - 1) * kBlock;
    int s = blockIdx.x == gridDim.x - 1 ? 2 * a.vh : (int)(blockIdx.x * kBlock + threadIdx.x);
    uint4 cr[G][C], cu[G][C];
    auto load = [&](int at, int i0) {
        if (at >= 2 * a.vh) return;
        const Site q = site_of(at, a.vh);
        const size_t off = q.h * a.hb;
#pragma unroll
        for (int g = 0; g < G; g++)
            if (i0 + g <= a.j) {
                Spinor<SF>::gather(a.R + off + (i0 + g) * a.fb, a.vh, q.i, cr[g]);
                Spinor<SF>::gather(a.U + off + (i0 + g) * a.fb, a.vh, q.i, cu[g]);
            }
    };
    load(s, 0);
    dot_sums<real>(a, tot);
    if (threadIdx.x == 0) {
        BState *b = a.b;
        const int j = a.j;
        const double pr = j ? b->rho_re[j - 1] : b->rhoc_re, pi = j ? b->rho_im[j - 1] : b->rhoc_im;
        const double lr = j ? b->al_re[j - 1] : b->alc_re, li = j ? b->al_im[j - 1] : b->alc_im;
        const double n2 = tot[0] * tot[0] + tot[1] * tot[1];
        const bool ok = pr * pr + pi * pi > b->tiny2 && !(tot[2] > 0.0 && !(n2 > b->brk2 * b->rt2 * tot[2])) &&
                        isfinite(n2);
        if (blockIdx.x == gridDim.x - 1) {
            if (ok) {
                b->rho_re[j] = tot[0];
                b->rho_im[j] = tot[1];
            } else {
                b_stop(b, REASON_BREAKDOWN);
            }
        }
        double qr = 0.0, qi = 0.0;
        if (ok) cdiv(tot[0], tot[1], pr, pi, qr, qi);
        be_sh[0] = (real)(lr * qr - li * qi);
        be_sh[1] = (real)(lr * qi + li * qr);
        ok_sh = ok;
    }
    __syncthreads();
    if (!ok_sh || blockIdx.x == gridDim.x - 1) return;
    const real br = be_sh[0], bi = be_sh[1];
    for (; s < 2 * a.vh; s += step) {
        const Site q = site_of(s, a.vh);
        char *uf = a.U + q.h * a.hb;
        for (int i0 = 0; i0 <= a.j; i0 += G) {
            if (i0 > 0) load(s, i0);
#pragma unroll
            for (int g = 0; g < G; g++) {
                if (i0 + g > a.j) continue;
                real r[6], u[6];
                Spinor<SF>::decode(cr[g], r);
                Spinor<SF>::decode(cu[g], u);
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const real ur = u[2 * c], ui = u[2 * c + 1];
                    u[2 * c] = r[2 * c] - (br * ur - bi * ui);
                    u[2 * c + 1] = r[2 * c + 1] - (br * ui + bi * ur);
                }
                if (!Spinor<SF>::store(uf + (i0 + g) * a.fb, a.vh, q.i, u)) atomicExch(a.err, 1);
            }
        }
        load(s + step, 0);
    }
    pdl_launch_dependents();
}

// r_i -= alpha u_{i+1}, i = 0..j; x += alpha u_0 (FP64), with gamma = <rt, u_{j+1}>, alpha = rho / gamma;
// breakdown relative to |rt| |u_{j+1}|
template <int SF, typename real, int G>
__global__ void __launch_bounds__(kBlock) r_multi_kernel(BArgs a)
{
    pdl_wait();
    if (skip(a.active)) return;
    __shared__ double tot[3];
    __shared__ real al_sh[2];
    __shared__ int ok_sh;
    // loads as in the u update; u_0 and x with them when several fields are in flight anyway (G > 1)
    constexpr int C = Spinor<SF>::chunks;
    const int step = (int)(gridDim.x - 1) * kBlock;
    int s = blockIdx.x == gridDim.x - 1 ? 2 * a.vh : (int)(blockIdx.x * kBlock + threadIdx.x);
    uint4 cr[G][C], cu[G][C], c0[C], cx[Spinor<S_F64>::chunks];
    auto x_field = [&](int h) { return reinterpret_cast<char *>(a.x64) + h * (size_t)48 * a.vh; };
    auto load_x = [&](const Site &q) {
        Spinor<SF>::gather(a.U + q.h * a.hb, a.vh, q.i, c0);
        Spinor<S_F64>::gather(x_field(q.h), a.vh, q.i, cx);
    };
    auto load = [&](int at, int i0) {
        if (at >= 2 * a.vh) return;
        const Site q = site_of(at, a.vh);
        const size_t off = q.h * a.hb;
        if (G > 1 && i0 == 0) load_x(q);
#pragma unroll
        for (int g = 0; g < G; g++)
            if (i0 + g <= a.j) {
                Spinor<SF>::gather(a.U + a.fb + off + (i0 + g) * a.fb, a.vh, q.i, cu[g]);
                Spinor<SF>::gather(a.R + off + (i0 + g) * a.fb, a.vh, q.i, cr[g]);
            }
    };
    load(s, 0);
    dot_sums<real>(a, tot);
    if (threadIdx.x == 0) {
        BState *b = a.b;
        const double n2 = tot[0] * tot[0] + tot[1] * tot[1];
        const bool ok = !(n2 <= b->tiny2) && n2 > b->brk2 * b->rt2 * tot[2] && isfinite(tot[0]) && isfinite(tot[1]);
        double qr = 0.0, qi = 0.0;
        if (ok) cdiv(b->rho_re[a.j], b->rho_im[a.j], tot[0], tot[1], qr, qi);
        if (blockIdx.x == gridDim.x - 1) {
            if (ok) {
                b->al_re[a.j] = qr;
                b->al_im[a.j] = qi;
            } else {
                b_stop(b, REASON_BREAKDOWN);
            }
        }
        al_sh[0] = (real)qr;
        al_sh[1] = (real)qi;
        ok_sh = ok;
    }
    __syncthreads();
    if (!ok_sh || blockIdx.x == gridDim.x - 1) return;
    const real ar = al_sh[0], ai = al_sh[1];
    for (; s < 2 * a.vh; s += step) {
        const Site q = site_of(s, a.vh);
        char *rf = a.R + q.h * a.hb;
        for (int i0 = 0; i0 <= a.j; i0 += G) {
            if (i0 > 0) load(s, i0);
#pragma unroll
            for (int g = 0; g < G; g++) {
                if (i0 + g > a.j) continue;
                real u[6], r[6];
                Spinor<SF>::decode(cu[g], u);
                Spinor<SF>::decode(cr[g], r);
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const real ur = u[2 * c], ui = u[2 * c + 1];
                    r[2 * c] -= ar * ur - ai * ui;
                    r[2 * c + 1] -= ar * ui + ai * ur;
                }
                if (!Spinor<SF>::store(rf + (i0 + g) * a.fb, a.vh, q.i, r)) atomicExch(a.err, 1);
            }
        }
        // x += alpha u_0: the increment in the compute precision, the sum in FP64
        if (G == 1) load_x(q);
        real u0[6];
        double x[6];
        Spinor<SF>::decode(c0, u0);
        Spinor<S_F64>::decode(cx, x);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            x[2 * c] += widen(ar * u0[2 * c] - ai * u0[2 * c + 1]);
            x[2 * c + 1] += widen(ar * u0[2 * c + 1] + ai * u0[2 * c]);
        }
        Spinor<S_F64>::store(x_field(q.h), a.vh, q.i, x);
        load(s + step, 0);
    }
    pdl_launch_dependents();
}

// The most vectors after r_k that pass k's kernel is compiled for.
__host__ __device__ constexpr int mgs_nj(int rest) { return rest == 0 ? 0 : rest == 1 ? 1 : rest <= 3 ? 3 : 7; }

// The sums that pass k - 1 of l left.
template <typename real>
__device__ __forceinline__ void sum_prev(const BArgs &a, int k, int l, double *tot)
{
    const real *part = reinterpret_cast<const real *>(a.part_in);
    switch (mgs_nj(l - k + 1)) {
    case 1: sum_rows<5, real>(part, a.rows, tot); break;
    case 3: sum_rows<9, real>(part, a.rows, tot); break;
    default: sum_rows<17, real>(part, a.rows, tot); break;
    }
}

// Gram-Schmidt pass k = a.j of r_1..r_l, modified in the right-looking order:
// r_i -= tau_{k-1,i} r_{k-1} for i = k..l (k >= 2), each r_i thus projected
// against r_1, r_2, ... one after another as the left-looking order does, then
// the sums of sigma_k = |r_k|^2, <r_k, r_0> and <r_k, r_i>, i > k: l passes
// over the vectors instead of l (l + 1) / 2 (16^3x32, l = 4: ten of 9.9 us).
// NJ: the most vectors after r_k.
template <int SF, typename real, int NJ>
__global__ void __launch_bounds__(kBlock) mgs_kernel(BArgs a)
{
    constexpr int NR = 3 + 2 * NJ, C = Spinor<SF>::chunks;
    pdl_wait();
    if (skip(a.active)) return;
    BState *b = a.b;
    const int k = a.j, rest = b->l - k;  // vectors after r_k
    const bool scalars = blockIdx.x == gridDim.x - 1;
    __shared__ double tot[3 + 2 * kMaxL];
    __shared__ real tau[2 * (NJ + 1)];
    __shared__ int ok_sh;
    // the first site's fields are loaded before the sums
    const int step = (int)(gridDim.x - 1) * kBlock;
    int s = scalars ? 2 * a.vh : (int)(blockIdx.x * kBlock + threadIdx.x);
    uint4 c0[C], cp[C], cr[NJ + 1][C];
    auto load = [&](int at) {
        if (at >= 2 * a.vh) return;
        const Site q = site_of(at, a.vh);
        const char *f = a.R + q.h * a.hb;
        Spinor<SF>::gather(f, a.vh, q.i, c0);
        if (k >= 2) Spinor<SF>::gather(f + (k - 1) * a.fb, a.vh, q.i, cp);
#pragma unroll
        for (int i = 0; i <= NJ; i++)
            if (i <= rest) Spinor<SF>::gather(f + (k + i) * a.fb, a.vh, q.i, cr[i]);
    };
    load(s);
    if (k >= 2) {
        // the previous pass left 3 + 2 * (its NJ) values a row; tau_{k-1,i} = <r_{k-1}, r_i> / sigma_{k-1}
        sum_prev<real>(a, k, b->l, tot);
        const double sg = tot[0];
        const bool ok = sg > 0.0 && isfinite(sg);
        if (threadIdx.x <= rest) {
            const int i = threadIdx.x;  // r_{k+i}
            const double inv = ok ? 1.0 / sg : 0.0, tr = tot[3 + 2 * i] * inv, ti = tot[4 + 2 * i] * inv;
            tau[2 * i] = (real)tr;
            tau[2 * i + 1] = (real)ti;
            if (scalars) {
                b->tau_re[k - 1][k + i] = tr;
                b->tau_im[k - 1][k + i] = ti;
                if (i == 0) {
                    b->gp_re[k - 1] = tot[1] * inv;
                    b->gp_im[k - 1] = tot[2] * inv;
                    if (!ok) b_stop(b, REASON_BREAKDOWN);
                }
            }
        }
        if (threadIdx.x == 0) ok_sh = ok;
        __syncthreads();
        if (!ok_sh) return;
    }
    if (scalars) return;
    real v[NR];
#pragma unroll
    for (int q = 0; q < NR; q++) v[q] = 0;
    for (; s < 2 * a.vh; s += step) {
        const Site q = site_of(s, a.vh);
        auto field = [&](int i) { return a.R + i * a.fb + q.h * a.hb; };
        real r0[6], rp[6], rk[6];
        Spinor<SF>::decode(c0, r0);
        if (k >= 2) Spinor<SF>::decode(cp, rp);
#pragma unroll
        for (int i = 0; i <= NJ; i++) {
            if (i > rest) continue;
            real r[6];
            Spinor<SF>::decode(cr[i], r);
            if (k >= 2) {
                const real tr = tau[2 * i], ti = tau[2 * i + 1];
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const real pr = rp[2 * c], pi = rp[2 * c + 1];
                    r[2 * c] -= tr * pr - ti * pi;
                    r[2 * c + 1] -= tr * pi + ti * pr;
                }
                if (!Spinor<SF>::store(field(k + i), a.vh, q.i, r)) atomicExch(a.err, 1);
            }
            if (i == 0) {
                real w[3] = {0, 0, 0};
                dot_site(r, r0, w);
                v[1] += w[0];
                v[2] += w[1];
                real n2 = 0;
#pragma unroll
                for (int c = 0; c < 6; c++) {
                    rk[c] = r[c];
                    n2 += r[c] * r[c];
                }
                v[0] += n2;
            } else {
                real w[3] = {0, 0, 0};
                dot_site(rk, r, w);
                v[1 + 2 * i] += w[0];
                v[2 + 2 * i] += w[1];
            }
        }
        load(s + step);
    }
    pdl_launch_dependents();
    store_partial_at<NR, real>(v, reinterpret_cast<real *>(a.part_out), blockIdx.x);
}

// x += gamma_1 r_0 + sum gamma''_j r_j;  r_0 -= gamma'_l r_l + sum gamma'_j r_j;
// u_0 -= gamma_l u_l + sum gamma_j u_j; then <rt, r_0>, |r_0|^2 and the cycle's decisions, with
// gamma_l = gamma'_l, omega = gamma_l; gamma_j = gamma'_j - sum_{i>j} tau_ji gamma_i;
// gamma''_j = gamma_{j+1} + sum_{i=j+1}^{l-1} tau_ji gamma_{i+1}
template <int SF, typename real>
__global__ void __launch_bounds__(kBlock) final_kernel(BArgs a)
{
    pdl_wait();
    if (skip(a.active)) return;
    BState *b = a.b;
    const int l = b->l;
    __shared__ double tot[3];
    __shared__ double g_re[kMaxL + 1], g_im[kMaxL + 1];
    __shared__ real g[kMaxL + 1][2], gp[kMaxL + 1][2], gpp[kMaxL + 1][2];
    __shared__ int ok_sh;
    sum_rows<3, real>(reinterpret_cast<const real *>(a.part_in), a.rows, tot);
    if (threadIdx.x == 0) {
        const double sg = tot[0];
        const bool ok = sg > 0.0 && isfinite(sg);
        ok_sh = ok;
        const double gr = ok ? tot[1] / sg : 0.0, gi = ok ? tot[2] / sg : 0.0;
        g_re[l] = gr;
        g_im[l] = gi;
        for (int j = l - 1; j >= 1; j--) {
            double sr = b->gp_re[j], si = b->gp_im[j];
            for (int i = j + 1; i <= l; i++) {
                sr -= b->tau_re[j][i] * g_re[i] - b->tau_im[j][i] * g_im[i];
                si -= b->tau_re[j][i] * g_im[i] + b->tau_im[j][i] * g_re[i];
            }
            g_re[j] = sr;
            g_im[j] = si;
        }
        for (int j = 1; j <= l; j++) {
            g[j][0] = (real)g_re[j];
            g[j][1] = (real)g_im[j];
            gp[j][0] = (real)(j < l ? b->gp_re[j] : gr);
            gp[j][1] = (real)(j < l ? b->gp_im[j] : gi);
            if (j == l) continue;
            double sr = g_re[j + 1], si = g_im[j + 1];
            for (int i = j + 1; i <= l - 1; i++) {
                sr += b->tau_re[j][i] * g_re[i + 1] - b->tau_im[j][i] * g_im[i + 1];
                si += b->tau_re[j][i] * g_im[i + 1] + b->tau_im[j][i] * g_re[i + 1];
            }
            gpp[j][0] = (real)sr;
            gpp[j][1] = (real)si;
        }
        if (!ok && blockIdx.x == 0) b_stop(b, REASON_BREAKDOWN);
    }
    __syncthreads();
    if (!ok_sh) return;
    real v[3] = {0, 0, 0};
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < 2 * a.vh; s += gridDim.x * blockDim.x) {
        const Site q = site_of(s, a.vh);
        // updates in the compute precision; x's increment is added in FP64
        real dx[6] = {0, 0, 0, 0, 0, 0}, r0[6], u0[6], t[6];
        char *xf = reinterpret_cast<char *>(a.x64) + q.h * (size_t)48 * a.vh;
        char *r0f = a.R + q.h * a.hb, *u0f = a.U + q.h * a.hb;
        uint4 cx[Spinor<S_F64>::chunks];
        constexpr int G = kGroup - 1, C = Spinor<SF>::chunks;  // l - 1 = 3 fields of a kind at the usual l = 4
        uint4 ct[C];
        Spinor<S_F64>::gather(xf, a.vh, q.i, cx);
        Spinor<SF>::gather(a.rt + q.h * a.hb, a.vh, q.i, ct);
        Spinor<SF>::load(r0f, a.vh, q.i, r0);
        Spinor<SF>::load(u0f, a.vh, q.i, u0);
        auto cax = [](real *y, const real *c2, const real *z, real sgn) {
            const real c_r = c2[0] * sgn, c_i = c2[1] * sgn;
#pragma unroll
            for (int c = 0; c < 3; c++) {
                y[2 * c] += c_r * z[2 * c] - c_i * z[2 * c + 1];
                y[2 * c + 1] += c_r * z[2 * c + 1] + c_i * z[2 * c];
            }
        };
        cax(dx, g[1], r0, real(1));
        Spinor<SF>::load(a.R + l * a.fb + q.h * a.hb, a.vh, q.i, t);
        cax(r0, gp[l], t, real(-1));
        Spinor<SF>::load(a.U + l * a.fb + q.h * a.hb, a.vh, q.i, t);
        cax(u0, g[l], t, real(-1));
        for (int j0 = 1; j0 <= l - 1; j0 += G) {
            uint4 cr[G][C], cu[G][C];
#pragma unroll
            for (int w = 0; w < G; w++)
                if (j0 + w <= l - 1) {
                    Spinor<SF>::gather(u0f + (j0 + w) * a.fb, a.vh, q.i, cu[w]);
                    Spinor<SF>::gather(r0f + (j0 + w) * a.fb, a.vh, q.i, cr[w]);
                }
#pragma unroll
            for (int w = 0; w < G; w++) {
                const int j = j0 + w;
                if (j > l - 1) continue;
                Spinor<SF>::decode(cu[w], t);
                cax(u0, g[j], t, real(-1));
                Spinor<SF>::decode(cr[w], t);
                cax(dx, gpp[j], t, real(1));
                cax(r0, gp[j], t, real(-1));
            }
        }
        real rt[6];
        Spinor<SF>::decode(ct, rt);
        double x[6];
        Spinor<S_F64>::decode(cx, x);
#pragma unroll
        for (int k = 0; k < 6; k++) x[k] += widen(dx[k]);
        Spinor<S_F64>::store(xf, a.vh, q.i, x);
        if (!Spinor<SF>::store(r0f, a.vh, q.i, r0)) atomicExch(a.err, 1);
        if (!Spinor<SF>::store(u0f, a.vh, q.i, u0)) atomicExch(a.err, 1);
        dot_site(rt, r0, v);
    }
    pdl_launch_dependents();
    if (reduce_grid<3>(v, a.red, tot) && threadIdx.x == 0) {
        for (int k = 0; k < 3; k++) b->dot[k] = tot[k];
        // the next cycle's rho_0 starts from -omega rho
        const double rr = tot[2], lr = b->rho_re[l - 1], li = b->rho_im[l - 1];
        b->rhoc_re = -(g_re[l] * lr - g_im[l] * li);
        b->rhoc_im = -(g_re[l] * li + g_im[l] * lr);
        b->alc_re = b->al_re[l - 1];
        b->alc_im = b->al_im[l - 1];
        b->rr = rr;
        b->cycles += 1;
        if (!isfinite(rr)) {
            b_stop(b, REASON_BREAKDOWN);
            return;
        }
        if (rr > b->rr_max) b->rr_max = rr;
        if (rr <= b->stop2)
            b_stop(b, REASON_CONVERGED);
        else if (rr < b->delta2 * b->rr_max)
            b_stop(b, REASON_RELIABLE);
    }
}

// after a reliable update: rr = |r_hi|^2 (sums[0]) and iterate again
__global__ void restart_kernel(BState *b, const double *sum)
{
    pdl_wait();
    pdl_launch_dependents();
    b->rr = sum[0];
    b->rr_max = sum[0];
    b->reason = REASON_NONE;
    b->active = isfinite(sum[0]) ? 1 : 0;
    if (!b->active) b->reason = REASON_BREAKDOWN;
}

// Blocks with sites of a vector kernel over the full lattice: kMaxBlocks at most where the next kernel's blocks
// sum its rows or the stencil's; on large lattices (more stencil rows than kMaxRows, summed once) one full wave
// with the scalars' block, since two blocks a SM leave too few loads in flight.  32^3x64, 20-bit, us a launch at
// 304 blocks of four fields at once and here: u update 66.6 and 48.6, r update 107.5 and 77.9, Gram-Schmidt passes
// 66.5, 66.1, 42.3 and 52.0, 53.5, 32.7 (16^3x32 keeps 304: more rows cost the next kernel more than they give)
template <typename K>
int vec_blocks(K kernel, int vh, bool large)
{
    const int need = (2 * vh + kBlock - 1) / kBlock;
    const int most = large ? std::max(wave_blocks(kernel, kBlock) - 1, 1) : kMaxBlocks;
    return need < most ? need : most;
}

// f(integral_constant<spinor format>, a value of the compute type)
template <typename F>
void b_dispatch(const hisq_prec &p, F f)
{
    const bool f64 = p.compute == HISQ_COMPUTE_F64;
    switch (p.spinor) {
    case S_F64: f(std::integral_constant<int, S_F64>{}, double{}); break;
    case S_F32: f(std::integral_constant<int, S_F32>{}, float{}); break;
    case S_HALF: f(std::integral_constant<int, S_HALF>{}, float{}); break;
    case S_INT20: f(std::integral_constant<int, S_INT20>{}, float{}); break;
    case S_INT14: f(std::integral_constant<int, S_INT14>{}, float{}); break;
    case S_INT30:
        if (f64) f(std::integral_constant<int, S_INT30>{}, double{});
        else f(std::integral_constant<int, S_INT30>{}, float{});
        break;
    }
}

struct BRun {
    hisq_ctx *c;
    hisq_gauge *g;
    const hisq_solver_params &p;
    cudaStream_t st;
    Workspace ws;
    int vh, l;
    size_t hb, fb;
    char *R = nullptr, *U = nullptr, *rt = nullptr;
    double *x64 = nullptr, *r64 = nullptr, *ax64 = nullptr;
    double *park = nullptr;  // the even half's |r|^2 while the odd half is reduced
    BState *b = nullptr, *bh = nullptr;
    GaugeView gv_s{}, gv_d{};
    int mv = 0, mv_hi = 0, ru = 0;

    BRun(hisq_ctx *c_, hisq_gauge *g_, const hisq_solver_params &p_, cudaStream_t s_)
        : c(c_), g(g_), p(p_), st(s_), ws(c_, s_), vh(g_->geom.vh), l(p_.l)
    {
    }
    ~BRun()
    {
        cudaStreamSynchronize(st);  // no copy into the state block is in flight
        pinned_put(c, bh);
    }

    BArgs args() const
    {
        BArgs a{};
        a.vh = vh;
        a.hb = hb;
        a.fb = fb;
        a.R = R;
        a.U = U;
        a.rt = rt;
        a.x64 = x64;
        a.b = b;
        a.active = &b->active;
        a.err = cur_err(c);
        a.red = cur_red(c);
        return a;
    }

    bool large() const { return dslash_full_rows(p.sloppy.gauge, vh) > kMaxRows; }
    double sbytes() const { return spinor_site_bytes(p.sloppy.spinor) * 2.0 * vh; }

    // out = 2m in + D in on the full lattice (two half-lattice passes)
    void mfull(const hisq_prec &pr, const GaugeView &gv, const char *in, char *out, size_t half_bytes,
               const int *active, int kind)
    {
        for (int po = 0; po < 2; po++) {
            DslashArgs d{};
            d.g = g->geom;
            d.gv = gv;
            d.err = cur_err(c);
            d.red = cur_red(c);
            d.active = active;
            d.out_parity = po;
            d.in = in + (1 - po) * half_bytes;
            d.out = out + po * half_bytes;
            d.y = in + po * half_bytes;
            d.a = 2.0 * p.mass;
            d.sign = 1;
            d.xpay = 1;
            LaunchScope ls(c, st, kind, stencil_bytes(pr, vh, true));
            launch_dslash(pr.gauge, pr.spinor, pr.compute, pr.long_recon, false, d, st);
        }
    }

    // <rt, v> and |v|^2 into the state
    void dot_to_state(const char *v, const int *act)
    {
        BArgs a = args();
        a.active = act;
        LaunchScope ls(c, st, PROF_BLAS, 2.0 * sbytes());
        b_dispatch(p.sloppy, [&](auto sf, auto rl) {
            auto k = dot_kernel<decltype(sf)::value, decltype(rl)>;
            launch_chained(k, dim3(vec_blocks(k, vh, large())), dim3(kBlock), st, a, v);
        });
    }

    // out = M in with <rt, out> and |out|^2; returns the rows of partials left at red.partials (0: the sums are
    // in the state)
    int mfull_dot(const char *in, char *out)
    {
        const int rows = dslash_full_rows(p.sloppy.gauge, vh);
        const size_t row_bytes = 3 * (p.sloppy.compute == HISQ_COMPUTE_F64 ? 8 : 4);
        const bool fits = rows * row_bytes <= kSplitHalf * sizeof(double);
        DslashArgs d{};
        d.g = g->geom;
        d.gv = gv_s;
        d.err = cur_err(c);
        d.red = cur_red(c);
        if (!fits) d.red.partials = nullptr;
        d.active = &b->active;
        d.in = in;
        d.out = out;
        d.y = in;
        d.a = 2.0 * p.mass;
        d.sign = 1;
        d.xpay = 1;
        d.half_bytes = hb;
        d.dot = rt;
        {
            LaunchScope ls(c, st, PROF_STENCIL, 2.0 * stencil_bytes(p.sloppy, vh, true));
            launch_dslash(p.sloppy.gauge, p.sloppy.spinor, p.sloppy.compute, p.sloppy.long_recon, false, d, st);
        }
        if (!fits) {
            dot_to_state(out, &b->active);
            return 0;
        }
        if (rows <= kMaxRows) return rows;
        BArgs a = args();
        a.rows = rows;
        a.part_in = cur_red(c).partials;
        a.red.partials = cur_red(c).partials + kSplitHalf;
        const dim3 grid(32), block(kBlock);
        LaunchScope ls(c, st, PROF_BLAS, 0.0);
        if (p.sloppy.compute != HISQ_COMPUTE_F64)
            launch_chained(dot_rows_kernel<float>, grid, block, st, a);
        else
            launch_chained(dot_rows_kernel<double>, grid, block, st, a);
        return 0;
    }

    void cycle()
    {
        int nb = 0;  // rows the Gram-Schmidt pass before left
        double *half[2] = {cur_red(c).partials, cur_red(c).partials + kSplitHalf};
        int rows = 0;  // <rt, r_0> is in the state
        for (int j = 0; j < l; j++) {
            BArgs a = args();
            a.j = j;
            a.rows = rows;
            a.part_in = half[0];
            b_dispatch(p.sloppy, [&](auto sf, auto rl) {
                LaunchScope ls(c, st, PROF_BLAS, 3.0 * (j + 1) * sbytes());
                constexpr int SF = decltype(sf)::value;
                using real = decltype(rl);
                auto kern = large() ? u_multi_kernel<SF, real, 1> : u_multi_kernel<SF, real, kGroup>;
                launch_chained(kern, dim3(vec_blocks(kern, vh, large()) + 1), dim3(kBlock), st, a);
            });
            a.rows = mfull_dot(U + j * fb, U + (j + 1) * fb);
            b_dispatch(p.sloppy, [&](auto sf, auto rl) {
                LaunchScope ls(c, st, PROF_BLAS, (3.0 * (j + 1) + 1) * sbytes() + 96.0 * 2 * vh);
                constexpr int SF = decltype(sf)::value;
                using real = decltype(rl);
                auto kern = large() ? r_multi_kernel<SF, real, 1> : r_multi_kernel<SF, real, kGroup>;
                launch_chained(kern, dim3(vec_blocks(kern, vh, large()) + 1), dim3(kBlock), st, a);
            });
            rows = mfull_dot(R + j * fb, R + (j + 1) * fb);
        }
        for (int k = 1; k <= l; k++) {
            BArgs a = args();
            a.j = k;
            a.rows = nb;
            a.part_in = half[(k - 1) & 1];
            a.part_out = half[k & 1];
            b_dispatch(p.sloppy, [&](auto sf, auto rl) {
                constexpr int SF = decltype(sf)::value;
                using real = decltype(rl);
                LaunchScope ls(c, st, PROF_BLAS, ((l - k + 2.0) + (k >= 2 ? l - k + 2.0 : 0.0)) * sbytes());
                auto pass = [&](auto kern) {
                    nb = vec_blocks(kern, vh, large());
                    launch_chained(kern, dim3(nb + 1), dim3(kBlock), st, a);
                };
                switch (mgs_nj(l - k)) {
                case 0: pass(mgs_kernel<SF, real, 0>); break;
                case 1: pass(mgs_kernel<SF, real, 1>); break;
                case 3: pass(mgs_kernel<SF, real, 3>); break;
                default: pass(mgs_kernel<SF, real, 7>); break;
                }
            });
        }
        BArgs a = args();
        a.rows = nb;
        a.part_in = half[l & 1];
        // the final update's own sums go to the other half
        a.red.partials = half[(l + 1) & 1];
        b_dispatch(p.sloppy, [&](auto sf, auto rl) {
            LaunchScope ls(c, st, PROF_BLAS, (2.0 * l + 5.0) * sbytes() + 96.0 * 2 * vh);
            auto kern = final_kernel<decltype(sf)::value, decltype(rl)>;
            launch_chained(kern, dim3(vec_blocks(kern, vh, large())), dim3(kBlock), st, a);
        });
    }

    hisq_status pull()
    {
        cudaMemcpyAsync(bh, b, sizeof(BState), cudaMemcpyDeviceToHost, st);
        const cudaError_t e = cudaStreamSynchronize(st);
        return e == cudaSuccess ? HISQ_OK : cuda_fail(c, e, "BiCGStab state");
    }

    // r_hi = b - M x (FP64), r_0 = r_hi (sloppy); |r_hi|^2 -> red.result[0]
    void true_residual(const double *b64, bool x_zero)
    {
        const size_t h64 = (size_t)48 * vh;
        if (!x_zero) {
            mfull(prec_f64(), gv_d, (const char *)x64, (char *)ax64, h64, nullptr, PROF_STENCIL_HI);
            mv_hi++;
        }
        for (int h = 0; h < 2; h++) {
            BlasArgs a{};
            a.n = vh;
            a.err = cur_err(c);
            a.red = cur_red(c);
            a.b64 = b64 + h * 6 * (size_t)vh;
            a.ax64 = x_zero ? nullptr : ax64 + h * 6 * (size_t)vh;
            a.r64 = r64 + h * 6 * (size_t)vh;
            a.v0 = R + h * hb;
            a.v1 = R + h * hb;
            a.fin = FIN_STORE;
            a.fst = nullptr;
            LaunchScope ls(c, st, PROF_BLAS, (48.0 * 3 + 2.0 * spinor_site_bytes(p.sloppy.spinor)) * vh);
            launch_true_residual(p.sloppy.spinor, p.sloppy.compute, a, st);
            if (h == 0) cudaMemcpyAsync(park, cur_red(c).result, sizeof(double), cudaMemcpyDeviceToDevice, st);
        }
    }

    hisq_status run(const double *b64, bool x_zero, hisq_solve_info *info)
    {
        hisq_status e = gauge_view_for(c, g, p.sloppy, &gv_s);
        if (!e) e = gauge_view_for(c, g, prec_f64(), &gv_d);
        if (e) return e;
        hb = spinor_field_bytes(p.sloppy.spinor, vh);
        fb = 2 * hb;
        const size_t f64b = (size_t)96 * vh;
        e = ws.alloc(fb * (l + 1), (void **)&R);
        if (!e) e = ws.alloc(fb * (l + 1), (void **)&U);
        if (!e) e = ws.alloc(fb, (void **)&rt);
        if (!e) e = ws.alloc(f64b, (void **)&ax64);
        if (!e) e = ws.alloc(64, (void **)&park);
        if (!e) e = ws.alloc(f64b, (void **)&r64);
        if (!e) e = ws.alloc(sizeof(BState), (void **)&b);
        if (e) return e;
        bh = (BState *)pinned_get(c, sizeof(BState));
        if (!bh) return fail(c, HISQ_ENOMEM, "pinned host state");
        tune_stencil(c, g->geom, p.sloppy, gv_s, U, R, st);
        tune_stencil(c, g->geom, prec_f64(), gv_d, (char *)ax64, (char *)r64, st);
        cudaMemsetAsync(U, 0, fb * (l + 1), st);
        cudaMemsetAsync(R, 0, fb * (l + 1), st);
        // |b|^2 over both halves
        double bb = 0.0;
        for (int h = 0; h < 2; h++) {
            BlasArgs a{};
            a.n = vh;
            a.red = cur_red(c);
            a.x64 = const_cast<double *>(b64) + h * 6 * (size_t)vh;
            launch_norm2(a, st);
            double part = 0;
            cudaMemcpyAsync(&part, cur_red(c).result, sizeof part, cudaMemcpyDeviceToHost, st);
            if (cudaStreamSynchronize(st) != cudaSuccess) return cuda_fail(c, cudaGetLastError(), "norm");
            bb += part;
        }
        if (!std::isfinite(bb)) return fail(c, HISQ_EINVAL, "non-finite right-hand side");
        if (bb == 0.0) {
            cudaMemsetAsync(x64, 0, f64b, st);
            cudaStreamSynchronize(st);
            return HISQ_OK;
        }
        // r_0 = b - M x, shadow residual = r_0
        auto residual_norm = [&](bool xz, double &rr) -> hisq_status {
            true_residual(b64, xz);
            double parts[2] = {0, 0};
            cudaMemcpyAsync(&parts[0], park, sizeof(double), cudaMemcpyDeviceToHost, st);
            cudaMemcpyAsync(&parts[1], cur_red(c).result, sizeof(double), cudaMemcpyDeviceToHost, st);
            const cudaError_t ce = cudaStreamSynchronize(st);
            if (ce != cudaSuccess) return cuda_fail(c, ce, "true residual");
            rr = parts[0] + parts[1];
            return HISQ_OK;
        };
        double rr = 0;
        e = residual_norm(x_zero, rr);
        if (e) return e;
        cudaMemcpyAsync(rt, R, fb, cudaMemcpyDeviceToDevice, st);
        BState init{};
        init.rhoc_re = -1.0;  // rho = omega = 1
        init.rr = rr;
        init.rr_max = rr;
        init.delta2 = p.delta * p.delta;
        init.stop2 = p.tol * p.tol * bb;
        init.tiny2 = 1e-300;  // only guards the divisions
        init.rt2 = rr;        // rt = r_0
        init.brk2 = 1e-60;    // |<rt, v>| <= 1e-30 |rt| |v|
        init.active = 1;
        init.l = l;
        *bh = init;
        cudaMemcpyAsync(b, &init, sizeof init, cudaMemcpyHostToDevice, st);
        dot_to_state(R, nullptr);
        hisq_status status = HISQ_OK;
        bool done = rr <= init.stop2;
        const bool graph = p.use_graph && !c->prof.on;
        cudaGraphExec_t exec = nullptr;
        int64_t nodes = 0;
        while (!done) {
            if (mv >= p.maxiter) {
                status = HISQ_ENOTCONV;
                break;
            }
            if (graph) {
                if (!exec) {
                    cudaGraph_t gr = nullptr;
                    set_thread_capturing(true);
                    cudaError_t ce = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
                    if (ce == cudaSuccess) {
                        cycle();
                        ce = cudaStreamEndCapture(st, &gr);
                    }
                    set_thread_capturing(false);
                    if (ce == cudaSuccess) ce = cudaGraphInstantiate(&exec, gr, 0);
                    size_t nn = 0;
                    if (ce == cudaSuccess) ce = graph_kernel_nodes(gr, &nn);
                    if (gr) cudaGraphDestroy(gr);
                    if (ce != cudaSuccess) return cuda_fail(c, ce, "BiCGStab graph capture");
                    nodes = (int64_t)nn;
                }
                cudaGraphLaunch(exec, st);
                c->launches += nodes;
            } else {
                cycle();
            }
            mv += 2 * l;
            e = pull();
            if (e) break;
            if (bh->reason == REASON_BREAKDOWN) {
                status = fail(c, HISQ_EBREAKDOWN, "BiCGStab(%d) breakdown in cycle %d", l, bh->cycles);
                break;
            }
            if (bh->reason == REASON_RELIABLE || bh->reason == REASON_CONVERGED) {
                e = residual_norm(false, rr);
                if (e) break;
                ru++;
                {
                    LaunchScope ls(c, st, PROF_BLAS, 0.0);
                    // total of both halves was assembled on the host; hand it to the device
                    cudaMemcpyAsync(cur_red(c).result, &rr, sizeof rr, cudaMemcpyHostToDevice, st);
                    launch_chained(restart_kernel, dim3(1), dim3(1), st, b, (const double *)cur_red(c).result);
                }
                dot_to_state(R, nullptr);
                e = pull();
                if (e) break;
                done = rr <= init.stop2;
            }
        }
        if (exec) cudaGraphExecDestroy(exec);
        if (e) return e;
        if (status != HISQ_OK) {
            e = residual_norm(false, rr);
            if (e) return e;
        }
        info->iters = bh->cycles;
        info->matvecs = mv;
        info->matvecs_hi = mv_hi;
        info->reliable_updates = ru;
        info->true_residual = std::sqrt(rr / bb);
        if (status == HISQ_ENOTCONV)
            fail(c, HISQ_ENOTCONV, "BiCGStab(%d) reached %d matvecs with true residual %.3e", l, mv,
                 info->true_residual);
        return status;
    }
};

}  // namespace

}  // namespace hisq

using namespace hisq;

extern "C" hisq_status hisq_bicgstabl(hisq_ctx *c, const hisq_gauge *gc, const hisq_solver_params *p,
                                      const double *b, double *x, hisq_solve_info *info)
{
    if (!c || !gc || !b || !x || !info) return fail(c, HISQ_EINVAL, "hisq_bicgstabl: null argument");
    *info = hisq_solve_info{};
    hisq_status e = validate_params(c, p);
    if (e) return e;
    if (p->l < 1 || p->l > 8) return fail(c, HISQ_EINVAL, "l must be in 1..8");
    cudaSetDevice(c->device);
    const auto t0 = std::chrono::steady_clock::now();
    hisq_gauge *g = const_cast<hisq_gauge *>(gc);
    cudaStream_t s = pick_stream(c, p->stream);
    const int64_t vh = g->geom.vh;
    if (!solver_red_fits(vh)) return fail(c, HISQ_EINVAL, "lattice too large for the solvers' reductions");
    Workspace ws(c, s);
    double *b64 = nullptr, *x64 = nullptr;
    e = ws.alloc((size_t)96 * vh, (void **)&b64);
    if (!e) e = ws.alloc((size_t)96 * vh, (void **)&x64);
    if (e) return e;
    // the caller's full-lattice array is [even][odd]: convert per half
    for (int h = 0; h < 2 && !e; h++) e = to_planar(c, ws, b + h * 6 * vh, p->on_device, vh, b64 + h * 6 * vh, s);
    if (!e && p->use_init_guess)
        for (int h = 0; h < 2 && !e; h++) e = to_planar(c, ws, x + h * 6 * vh, p->on_device, vh, x64 + h * 6 * vh, s);
    if (!e && !p->use_init_guess) cudaMemsetAsync(x64, 0, (size_t)96 * vh, s);
    if (e) return e;
    hisq_status st;
    {
        BRun run(c, g, *p, s);
        run.x64 = x64;
        st = run.run(b64, !p->use_init_guess, info);
    }
    if (st != HISQ_OK && st != HISQ_ENOTCONV && st != HISQ_EBREAKDOWN) return st;
    for (int h = 0; h < 2 && !e; h++) e = from_planar(c, ws, x64 + h * 6 * vh, vh, x + h * 6 * vh, p->on_device, s);
    if (e) return e;
    info->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    return st;
}
