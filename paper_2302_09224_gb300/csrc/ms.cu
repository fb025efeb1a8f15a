// ms.cu -- mixed-precision multi-shift CG with refinement (Sec. 3.2) and its
// C-ABI entry point.
//
// Stage 1 (sloppy triplet): one base recurrence on A = M_ee + sigma_0 (the
// smallest shift) with reliable updates on the base system; the other shifts'
// solutions and gradient vectors, which only need the residuals, are brought up
// to date in one kernel per block of iterations (x_i accumulators in the compute
// precision, flushed into FP64 at each reliable update).  Shift i stops updating once its iterated
// residual zeta_i |r| reaches max(tol_i, 10 eps of the sloppy format); the
// stage ends when every shift other than the base has stopped.
// Stage 2 (refinement triplet): CG on the base system continuing from its
// gradient vector (re-projected against the new residual), then CG on each
// other shift from its x_i with a clean restart, skipping shifts whose FP64
// true residual already meets their target.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <numeric>
#include <type_traits>
#include <vector>

#include "blas.h"
#include "blas_update.cuh"
#include "cg.h"
#include "codecs.cuh"
#include "internal.h"
#include "launch.cuh"
#include "reduce.cuh"
#include "finish.cuh"

namespace hisq {

struct MSArgs {
    int n;
    int nshift;
    char *p;              // nshift sloppy fields, p_bytes apart
    size_t p_bytes;
    char *acc;            // nshift accumulator fields (F32 or F64 planar), acc_bytes apart
    size_t acc_bytes;
    double *x64;          // nshift FP64 planar fields, 48*n apart
    int *err;
};

namespace {

constexpr int kBlock = 256;

// An iteration of the stage after the two stencil passes: the residual update
// (every block sums the reducing pass's partials and takes alpha), then the base
// system's gradient vector and accumulator (every block sums the residual
// update's partials and takes beta).  The last block of each grid has no sites:
// its first warp runs the scalar recurrences of all shifts meanwhile.
//
// No kernel tests at its head a word that a block of its own grid writes, where
// a block that starts late would then skip work that counts.  The stage stops in
// the gradient update (m->active), which therefore tests m->go, left by the
// residual update before it: its sites are updated in place (the base's solution
// and gradient vector), so none may be left out of the iteration that stops.  The
// residual update tests m->active, which its own grid clears only on a breakdown,
// where every other block finds the same sums and does nothing.
struct MSIter {
    BlasArgs b;      // n, err, red; v0, v1: r and A p, then r and p of the base; nparts
    char *out;       // the new residual (its own ring slot); then the base's accumulator
    MSState *m;
    MSRing *ring;
    int slot, part;  // the iteration's ring slot, and the part of the block that fills the ring
};

template <typename real>
constexpr int ms_block()
{
    return std::is_same<real, float>::value ? 1024 : 512;
}

template <int SF, typename real>
__global__ void __launch_bounds__(ms_block<real>()) ms_r_update_kernel(const __grid_constant__ MSIter a)
{
    constexpr int BS = ms_block<real>(), U = 2, C = Spinor<SF>::chunks;
    pdl_wait();
    MSState *m = a.m;
    const bool scalars = blockIdx.x == gridDim.x - 1;
    if (*(volatile const int *)&m->active == 0) {  // uniform over the grid but for a breakdown (see above)
        if (scalars && threadIdx.x == 0) m->go = 0;
        return;
    }
    const int step = (int)(gridDim.x - 1) * BS * U;
    int i0 = scalars ? a.b.n : (int)blockIdx.x * BS * U + (int)threadIdx.x;
    uint4 cr[U][C], ca[U][C];
    r_load<SF>(a.b, i0, cr, ca);
    __shared__ double tot[2];
    __shared__ real al_sh;
    __shared__ int ok_sh;
    if (a.b.nparts > 0) sum_partials<2, part_t<real>>(a.b.red, a.b.nparts, tot);
    if (scalars) {
        if (threadIdx.x >= 32) return;
        __syncwarp();
        if (threadIdx.x == 0) {
            m->rr_den = m->rr;
            if (a.slot == 0) {
                a.ring->n = 0;
                a.ring->part = a.part;
            }
        }
        if (a.b.nparts > 0) ms_alpha_warp(m, tot[0]);
        if (threadIdx.x == 0) m->go = m->active;
        return;
    }
    if (threadIdx.x == 0) {
        // without partials the pass ran the finisher itself
        const double al = a.b.nparts > 0 ? m->rr / tot[0] : m->alpha;
        const bool ok = (a.b.nparts == 0 || tot[0] > 0.0) && isfinite(al);
        al_sh = ok ? real(al) : real(0);
        ok_sh = ok;
    }
    __syncthreads();
    if (!ok_sh) return;
    const real alpha = al_sh;
    red_t<real> v[2] = {0, 0};
    for (; i0 < a.b.n; i0 += step) {
        r_group<SF, real>(a.b, i0, cr, ca, alpha, v, a.out);
        r_load<SF>(a.b, i0 + step, cr, ca);
    }
    pdl_launch_dependents();
    store_block_partial<2>(v, split_half(a.b.red));
}

template <int SF, typename real>
__global__ void __launch_bounds__(kBlock) ms_p_update_kernel(const __grid_constant__ MSIter a)
{
    constexpr int C = Spinor<SF>::chunks;
    constexpr int AF = is_ff<real>::value ? S_FF : sizeof(real) == 8 ? S_F64 : S_F32;
    pdl_wait();
    MSState *m = a.m;
    if (m->go == 0) return;  // written by the kernel before, uniform over the grid
    const bool scalars = blockIdx.x == gridDim.x - 1;
    const int n = a.b.n, i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    const bool mine = !scalars && i < n;
    uint4 cr[C], cp[C], cx[Spinor<AF>::chunks];
    if (mine) {
        Spinor<SF>::gather(a.b.v0, n, i, cr);
        Spinor<SF>::gather(a.b.v1, n, i, cp);
        Spinor<AF>::gather(a.out, n, i, cx);
    }
    __shared__ double tot[2];
    __shared__ real al_sh, be_sh;
    __shared__ int ok_sh;
    warp0_sum_partials<2, part_t<real>>(split_half(a.b.red), a.b.nparts, tot);
    if (scalars) {
        if (threadIdx.x >= 32) return;
        __syncwarp();
        ms_beta_warp(m, a.ring, a.slot, tot[0]);
        return;
    }
    if (threadIdx.x == 0) {
        const double be = tot[0] / m->rr_den;
        ok_sh = isfinite(tot[0]) && isfinite(be);
        be_sh = real(be);
        al_sh = real(m->alpha);
    }
    __syncthreads();
    if (!mine || !ok_sh) return;
    const real al = al_sh, be = be_sh;
    real r[6], p[6], x[6];
    Spinor<SF>::decode(cr, r);
    Spinor<SF>::decode(cp, p);
    Spinor<AF>::decode(cx, x);
#pragma unroll
    for (int k = 0; k < 6; k++) {
        x[k] += al * p[k];
        p[k] = r[k] + be * p[k];
    }
    pdl_launch_dependents();
    if (!Spinor<SF>::store(a.b.v1, n, i, p)) atomicExch(a.b.err, 1);
    Spinor<AF>::store(a.out, n, i, x);
}

// The recorded iterations of every shift but the base, whose gradient vectors
// and accumulators need nothing but the residuals r_1, r_2, ... of the block (kept
// in a ring): per iteration j in which the shift was live, acc_i += alpha_ij p_i,
// p_i = zeta_ij r_j + beta_ij p_i.  A shift's fields are read and written once
// per block of iterations instead of every one (12 shifts at 16^3x32, FP64-class:
// 36.8 us an iteration before), and p_i stays in the compute precision between
// the block's iterations.  The last residual goes to r0, where the next part
// starts.
template <int SF, typename real>
__global__ void __launch_bounds__(kBlock) shift_ring_kernel(MSArgs a, const MSRing *ring, int part, char *r0,
                                                              char *r_ring)
{
    pdl_wait();
    pdl_launch_dependents();
    if (ring->part != part) return;  // the block stopped before this part (uniform over the grid)
    constexpr int AF = is_ff<real>::value ? S_FF : sizeof(real) == 8 ? S_F64 : S_F32;
    // iterations whose residuals a thread holds at once: decoded for FP32, as records otherwise
    constexpr bool kDecoded = std::is_same<real, float>::value;
    constexpr int RB = 8, C = Spinor<SF>::chunks;
    __shared__ real cs[3][kMaxBuf][kMaxShift];
    __shared__ unsigned live[kMaxBuf];
    const int n = ring->n;
    for (int k = threadIdx.x; k < n * kMaxShift; k += blockDim.x) {
        const int j = k / kMaxShift, s = k % kMaxShift;
        const bool on = s < a.nshift && ring->live[j][s] != 0;
        const unsigned bits = __ballot_sync(__activemask(), on);
        if (s == 0) live[j] = bits;
        if (on) {
            cs[0][j][s] = (real)ring->a[j][s];
            cs[1][j][s] = (real)ring->z[j][s];
            cs[2][j][s] = (real)ring->b[j][s];
        }
    }
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n || n == 0) return;
    for (int j0 = 0; j0 < n; j0 += RB) {
        const int m = n - j0 < RB ? n - j0 : RB;
        uint4 cr[RB][C];
        real r[kDecoded ? RB : 1][6];
        unsigned any = 0;
#pragma unroll
        for (int j = 0; j < RB; j++)
            if (j < m) {
                Spinor<SF>::gather(r_ring + (size_t)(j0 + j) * a.p_bytes, a.n, i, cr[j]);
                any |= live[j0 + j];
            }
        if (j0 + m == n) {
#pragma unroll
            for (int j = 0; j < RB; j++)
                if (j == m - 1) Spinor<SF>::put(r0, a.n, i, cr[j]);
        }
        if constexpr (kDecoded) {
#pragma unroll
            for (int j = 0; j < RB; j++)
                if (j < m) Spinor<SF>::decode(cr[j], r[j]);
        }
        for (int s = 1; s < a.nshift; s++) {
            if (!((any >> s) & 1u)) continue;
            real p[6], x[6];
            char *ps = a.p + (size_t)s * a.p_bytes;
            char *xs = a.acc + (size_t)s * a.acc_bytes;
            Spinor<SF>::load(ps, a.n, i, p);
            Spinor<AF>::load(xs, a.n, i, x);
#pragma unroll
            for (int j = 0; j < RB; j++) {
                if (j >= m || !((live[j0 + j] >> s) & 1u)) continue;
                const real al = cs[0][j0 + j][s], z = cs[1][j0 + j][s], be = cs[2][j0 + j][s];
                real rv[6];
                if constexpr (!kDecoded) Spinor<SF>::decode(cr[j], rv);
#pragma unroll
                for (int k = 0; k < 6; k++) {
                    x[k] += al * p[k];
                    p[k] = z * (kDecoded ? r[j][k] : rv[k]) + be * p[k];
                }
            }
            if (!Spinor<SF>::store(ps, a.n, i, p)) atomicExch(a.err, 1);
            Spinor<AF>::store(xs, a.n, i, x);
        }
    }
}

// x64_i += acc_i and acc_i = 0 for every shift.
template <int AF>
__global__ void __launch_bounds__(kBlock) acc_flush_kernel(MSArgs a)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    for (int s = 0; s < a.nshift; s++) {
        char *xs = a.acc + (size_t)s * a.acc_bytes;
        char *x64 = reinterpret_cast<char *>(a.x64) + (size_t)s * 48 * a.n;
        double acc[6], x[6];
        Spinor<AF>::load(xs, a.n, i, acc);
        Spinor<S_F64>::load(x64, a.n, i, x);
#pragma unroll
        for (int k = 0; k < 6; k++) {
            x[k] += acc[k];
            acc[k] = 0.0;
        }
        Spinor<S_F64>::store(x64, a.n, i, x);
        Spinor<AF>::store(xs, a.n, i, acc);
    }
}

template <int SI, int SO>
__global__ void __launch_bounds__(kBlock) convert_kernel(int n, const char *in, char *out, int *err)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double v[6];
    Spinor<SI>::load(in, n, i, v);
    if (!Spinor<SO>::store(out, n, i, v)) atomicExch(err, 1);
}

template <int SI>
void convert_to(int so, int n, const char *in, char *out, int *err, cudaStream_t s)
{
    const int nb = (n + kBlock - 1) / kBlock;
    switch (so) {
    case S_F64: convert_kernel<SI, S_F64><<<nb, kBlock, 0, s>>>(n, in, out, err); break;
    case S_F32: convert_kernel<SI, S_F32><<<nb, kBlock, 0, s>>>(n, in, out, err); break;
    case S_HALF: convert_kernel<SI, S_HALF><<<nb, kBlock, 0, s>>>(n, in, out, err); break;
    case S_INT20: convert_kernel<SI, S_INT20><<<nb, kBlock, 0, s>>>(n, in, out, err); break;
    case S_INT14: convert_kernel<SI, S_INT14><<<nb, kBlock, 0, s>>>(n, in, out, err); break;
    case S_INT30: convert_kernel<SI, S_INT30><<<nb, kBlock, 0, s>>>(n, in, out, err); break;
    }
}

int nblk(int n) { return (n + kBlock - 1) / kBlock; }

double format_eps(int sf)
{
    switch (sf) {
    case S_F32: return std::ldexp(1.0, -24);
    case S_HALF: return std::ldexp(1.0, -15);  // Sec. 2
    case S_INT20: return std::ldexp(1.0, -19); // Sec. 4
    case S_INT30: return std::ldexp(1.0, -29); // Sec. 4
    case S_INT14: return std::ldexp(1.0, -13);
    default: return std::ldexp(1.0, -52);
    }
}

}  // namespace

// field conversion between storage formats (any pair), exposed to the drivers
void launch_convert(int si, int so, int n, const char *in, char *out, int *err, cudaStream_t s)
{
    switch (si) {
    case S_F64: convert_to<S_F64>(so, n, in, out, err, s); break;
    case S_F32: convert_to<S_F32>(so, n, in, out, err, s); break;
    case S_HALF: convert_to<S_HALF>(so, n, in, out, err, s); break;
    case S_INT20: convert_to<S_INT20>(so, n, in, out, err, s); break;
    case S_INT14: convert_to<S_INT14>(so, n, in, out, err, s); break;
    case S_INT30: convert_to<S_INT30>(so, n, in, out, err, s); break;
    }
}

namespace {

struct MSRun {
    hisq_ctx *c;
    hisq_gauge *g;
    const hisq_solver_params &p;
    cudaStream_t s;
    Workspace ws;
    int vh, ns;
    size_t sb, accb;
    int acc_fmt;
    std::vector<double> sig, tol;
    char *r_s = nullptr, *w_s = nullptr, *tmp_s = nullptr, *P = nullptr, *ACC = nullptr;
    double *X = nullptr, *r64 = nullptr, *ax64 = nullptr, *tmp64 = nullptr;
    MSState *m = nullptr, *mh = nullptr;
    MSRing *ring = nullptr;
    GaugeView gv_s{}, gv_d{};
    int ru = 0, mv_hi = 0;
    int parts = 1;  // iterations whose residuals are kept before the shifts are brought up to date

    MSRun(hisq_ctx *c_, hisq_gauge *g_, const hisq_solver_params &p_, cudaStream_t s_)
        : c(c_), g(g_), p(p_), s(s_), ws(c_, s_), vh(g_->geom.vh), ns(0)
    {
    }
    ~MSRun()
    {
        cudaStreamSynchronize(s);  // no copy into the state block is in flight
        pinned_put(c, mh);
    }

    double *x64(int i) { return X + (size_t)i * 6 * vh; }
    char *pf(int i) { return P + (size_t)i * sb; }

    MSArgs args() const
    {
        MSArgs a{};
        a.n = vh;
        a.nshift = ns;
        a.p = P;
        a.p_bytes = sb;
        a.acc = ACC;
        a.acc_bytes = accb;
        a.x64 = X;
        a.err = cur_err(c);
        return a;
    }

    hisq_status pull()
    {
        cudaMemcpyAsync(mh, m, sizeof(MSState), cudaMemcpyDeviceToHost, s);
        const cudaError_t e = cudaStreamSynchronize(s);
        return e == cudaSuccess ? HISQ_OK : cuda_fail(c, e, "multi-shift state");
    }

    void flush_acc()
    {
        MSArgs a = args();
        LaunchScope ls(c, s, PROF_BLAS, (double)ns * (96.0 + 2.0 * spinor_site_bytes(acc_fmt)) * vh);
        if (acc_fmt == S_F64)
            acc_flush_kernel<S_F64><<<nblk(vh), kBlock, 0, s>>>(a);
        else if (acc_fmt == S_FF)
            acc_flush_kernel<S_FF><<<nblk(vh), kBlock, 0, s>>>(a);
        else
            acc_flush_kernel<S_F32><<<nblk(vh), kBlock, 0, s>>>(a);
    }

    // FP64 |b - (M_ee + sigma) x|^2 into red.result[0]; also leaves r64/r_s.
    void residual(int shift, int fin, void *fst)
    {
        const double diag = 4.0 * p.mass * p.mass + sig[shift];
        apply_mee(c, g->geom, prec_f64(), gv_d, diag, (const char *)x64(shift), (char *)tmp64, (char *)ax64, FIN_NONE,
                  nullptr, 0, nullptr, PROF_STENCIL_HI, s);
        mv_hi++;
        BlasArgs b{};
        b.n = vh;
        b.err = cur_err(c);
        b.red = cur_red(c);
        b.b64 = b64;
        b.ax64 = ax64;
        b.r64 = r64;
        b.v0 = r_s;
        b.v1 = pf(0);
        b.fin = fin;
        b.fst = fst;
        LaunchScope ls(c, s, PROF_BLAS, (48.0 * 3 + 2.0 * spinor_site_bytes(p.sloppy.spinor)) * vh);
        launch_true_residual(p.sloppy.spinor, p.sloppy.compute, b, s);
    }

    const double *b64 = nullptr;

    // SF and compute type of the sloppy triplet
    template <typename F>
    void dispatch(F f)
    {
        const bool f64 = p.sloppy.compute == HISQ_COMPUTE_F64;
        switch (p.sloppy.spinor) {
        case S_F64: f(std::integral_constant<int, S_F64>{}, double{}); break;
        case S_F32: f(std::integral_constant<int, S_F32>{}, float{}); break;
        case S_HALF: f(std::integral_constant<int, S_HALF>{}, float{}); break;
        case S_INT20: f(std::integral_constant<int, S_INT20>{}, float{}); break;
        case S_INT14: f(std::integral_constant<int, S_INT14>{}, float{}); break;
        case S_INT30:
            if (f64) f(std::integral_constant<int, S_INT30>{}, ff{});  // FP64-class compute in FP32 pairs
            else f(std::integral_constant<int, S_INT30>{}, float{});
            break;
        }
    }

    // the residual a part starts from (0) and those of its iterations, in the FP64 work fields
    char *r_slot(int j) { return j == 0 ? r_s : (char *)r64 + (size_t)(j - 1) * sb; }

    void iterate_block(int nit)
    {
        const double diag0 = 4.0 * p.mass * p.mass + sig[0];
        const int *act = &m->active;
        for (int it = 0; it < nit; it++) {
            const unsigned np = apply_mee(c, g->geom, p.sloppy, gv_s, diag0, pf(0), tmp_s, w_s, FIN_MS_ALPHA, m, 0, act,
                                          PROF_STENCIL, s, true);
            MSIter a{};
            a.b.n = vh;
            a.b.err = cur_err(c);
            a.b.red = cur_red(c);
            a.m = m;
            a.ring = ring;
            a.slot = it % parts;
            a.part = it / parts;
            dispatch([&](auto sf, auto rl) {
                constexpr int SF = decltype(sf)::value;
                using real = decltype(rl);
                constexpr int BS = ms_block<real>();
                static const int wave = wave_blocks(ms_r_update_kernel<SF, real>, BS);
                const int need = (vh + 2 * BS - 1) / (2 * BS);
                const int nb = std::max(1, std::min(need, wave - 1));
                a.b.v0 = r_slot(a.slot);
                a.b.v1 = w_s;
                a.out = r_slot(a.slot + 1);
                a.b.nparts = np;
                {
                    LaunchScope ls(c, s, PROF_BLAS, 3.0 * spinor_site_bytes(SF) * vh);
                    launch_chained(ms_r_update_kernel<SF, real>, dim3(nb + 1), dim3(BS), s, a);
                }
                a.b.v0 = r_slot(a.slot + 1);
                a.b.v1 = pf(0);
                a.out = ACC;
                a.b.nparts = nb;
                LaunchScope ls(c, s, PROF_BLAS, (3.0 * spinor_site_bytes(SF) + 2.0 * spinor_site_bytes(acc_fmt)) * vh);
                launch_chained(ms_p_update_kernel<SF, real>, dim3(nblk(vh) + 1), dim3(kBlock), s, a);
            });
            if (a.slot != parts - 1 && it != nit - 1) continue;
            int live = 0;
            for (int i = 1; i < ns; i++) live += mh->live[i];
            dispatch([&](auto sf, auto rl) {
                constexpr int SF = decltype(sf)::value;
                LaunchScope ls(c, s, PROF_BLAS,
                               ((a.slot + 2.0) * spinor_site_bytes(SF) +
                                live * 2.0 * (spinor_site_bytes(SF) + spinor_site_bytes(acc_fmt))) * vh);
                launch_chained(shift_ring_kernel<SF, decltype(rl)>, dim3(nblk(vh)), dim3(kBlock), s, args(),
                               (const MSRing *)ring, a.part, r_s, (char *)r64);
            });
        }
    }

    hisq_status run(const double *b64_, int nshift, const double *sigma, const double *tolv, hisq_solve_info *info,
                    bool refine = true)
    {
        b64 = b64_;
        ns = nshift;
        sig.assign(sigma, sigma + ns);
        tol.assign(tolv, tolv + ns);
        hisq_status e = gauge_view_for(c, g, p.sloppy, &gv_s);
        if (!e) e = gauge_view_for(c, g, prec_f64(), &gv_d);
        if (e) return e;
        sb = spinor_field_bytes(p.sloppy.spinor, vh);
        acc_fmt = p.sloppy.compute != HISQ_COMPUTE_F64 ? S_F32 : p.sloppy.spinor == S_INT30 ? S_FF : S_F64;
        accb = spinor_field_bytes(acc_fmt, vh);
        const size_t b48 = (size_t)48 * vh;
        const int N = std::max(1, p.nbuf);
        e = ws.alloc(sb, (void **)&r_s);
        if (!e) e = ws.alloc(sizeof(MSRing), (void **)&ring);
        if (!e) e = ws.alloc(sb, (void **)&w_s);
        if (!e) e = ws.alloc(sb, (void **)&tmp_s);
        if (!e) e = ws.alloc(sb * ns, (void **)&P);
        if (!e) e = ws.alloc(accb * ns, (void **)&ACC);
        if (!e) e = ws.alloc(b48 * ns, (void **)&X);
        // true residuals' work fields; between them, a block's residuals (as many as fit)
        if (!e) e = ws.alloc(3 * b48, (void **)&r64);
        ax64 = r64 + (size_t)6 * vh;
        tmp64 = ax64 + (size_t)6 * vh;
        parts = std::min(N, (int)(3 * b48 / sb));
        if (!e) e = ws.alloc(sizeof(MSState), (void **)&m);
        if (e) return e;
        mh = (MSState *)pinned_get(c, sizeof(MSState));
        if (!mh) return fail(c, HISQ_ENOMEM, "pinned host state");
        cudaMemsetAsync(ACC, 0, accb * ns, s);
        cudaMemsetAsync(X, 0, b48 * ns, s);
        tune_stencil(c, g->geom, p.sloppy, gv_s, w_s, tmp_s, s);
        tune_stencil(c, g->geom, prec_f64(), gv_d, (char *)ax64, (char *)tmp64, s);
        // r = p_i = b
        {
            LaunchScope ls(c, s, PROF_CONVERT, (48.0 + spinor_site_bytes(p.sloppy.spinor)) * vh);
            launch_convert(S_F64, p.sloppy.spinor, vh, (const char *)b64, r_s, cur_err(c), s);
        }
        for (int i = 0; i < ns; i++) cudaMemcpyAsync(pf(i), r_s, sb, cudaMemcpyDeviceToDevice, s);
        {
            BlasArgs a{};
            a.n = vh;
            a.red = cur_red(c);
            a.x64 = const_cast<double *>(b64);
            LaunchScope ls(c, s, PROF_BLAS, 48.0 * vh);
            launch_norm2(a, s);
        }
        double bb = 0;
        cudaMemcpyAsync(&bb, cur_red(c).result, sizeof bb, cudaMemcpyDeviceToHost, s);
        if (cudaStreamSynchronize(s) != cudaSuccess) return cuda_fail(c, cudaGetLastError(), "norm");
        if (!std::isfinite(bb)) return fail(c, HISQ_EINVAL, "non-finite right-hand side");
        info->nshift = ns;
        if (bb == 0.0) return HISQ_OK;  // all x_i = 0
        MSState init{};
        init.rr = bb;
        init.rr_max = bb;
        init.bb = bb;
        init.delta2 = p.delta * p.delta;
        init.alpha_prev = 1.0;
        init.beta_prev = 0.0;
        init.nshift = ns;
        init.active = 1;
        const double floor = 10.0 * format_eps(p.sloppy.spinor);
        for (int i = 0; i < ns; i++) {
            init.shift[i] = sig[i] - sig[0];
            const double t = std::max(tol[i], floor);
            init.stop2[i] = t * t * bb;
            init.zeta[i] = init.zeta_prev[i] = 1.0;
            init.live[i] = 1;
        }
        *mh = init;
        cudaMemcpyAsync(m, &init, sizeof init, cudaMemcpyHostToDevice, s);
        const bool graph = p.use_graph && !c->prof.on;
        cudaGraphExec_t exec = nullptr;
        int64_t nodes = 0;
        hisq_status status = HISQ_OK;
        while (true) {
            if (mh->k >= p.maxiter) {
                status = HISQ_ENOTCONV;
                break;
            }
            if (graph) {
                if (!exec) {
                    cudaGraph_t gr = nullptr;
                    set_thread_capturing(true);
                    cudaError_t ce = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
                    if (ce == cudaSuccess) {
                        iterate_block(N);
                        ce = cudaStreamEndCapture(s, &gr);
                    }
                    set_thread_capturing(false);
                    if (ce == cudaSuccess) ce = cudaGraphInstantiate(&exec, gr, 0);
                    size_t nn = 0;
                    if (ce == cudaSuccess) ce = graph_kernel_nodes(gr, &nn);
                    if (gr) cudaGraphDestroy(gr);
                    if (ce != cudaSuccess) return cuda_fail(c, ce, "multi-shift graph capture");
                    nodes = (int64_t)nn;
                }
                cudaGraphLaunch(exec, s);
                c->launches += nodes;
            } else {
                iterate_block(N);
            }
            e = pull();
            if (e) break;
            if (mh->reason == REASON_BREAKDOWN) {
                status = fail(c, HISQ_EBREAKDOWN, "multi-shift CG breakdown at iteration %d", mh->k);
                break;
            }
            if (mh->reason == REASON_CONVERGED) break;
            if (mh->reason == REASON_RELIABLE) {
                flush_acc();
                residual(0, FIN_MS_TRUE, m);
                ru++;
                e = pull();
                if (e) break;
            }
        }
        if (exec) cudaGraphExecDestroy(exec);
        if (e) return e;
        flush_acc();
        info->iters = mh->k;
        info->matvecs += mh->k;
        info->reliable_updates += ru;
        for (int i = 0; i < ns; i++) info->shift_iters[i] = mh->live[i] ? mh->k : mh->frozen_at[i];
        // FP64 true residual of every shift after the multi-shift stage (Table 3's r_sigma), then its refinement:
        // the base system keeps its gradient vector, the others restart
        const double rr_base = mh->rr;
        const bool refining = status != HISQ_EBREAKDOWN && refine;
        hisq_status worst = status;
        for (int i = 0; i < ns; i++) {
            residual(i, FIN_STORE, nullptr);
            double rr = 0;
            cudaMemcpyAsync(&rr, cur_red(c).result, sizeof rr, cudaMemcpyDeviceToHost, s);
            if (cudaStreamSynchronize(s) != cudaSuccess) return cuda_fail(c, cudaGetLastError(), "residual");
            const double rs = std::sqrt(rr / bb);
            info->shift_resid_ms[i] = rs;
            info->shift_resid[i] = rs;
            if (!refining || rs <= tol[i]) continue;
            CGConfig cfg = config_from(&p, sig[i]);
            cfg.sloppy = p.refine;
            cfg.tol = tol[i];
            cfg.ax_init = ax64;  // A x_i, just applied
            if (i == 0) {
                cfg.p_init = pf(0);
                cfg.p_init_fmt = p.sloppy.spinor;
                cfg.rr_prev_init = rr_base;
            }
            hisq_solve_info ri{};
            const hisq_status st = run_cg(c, g, cfg, b64, x64(i), false, &ri, s);
            info->refine_iters[i] = ri.iters;
            info->matvecs += ri.matvecs;
            info->matvecs_hi += ri.matvecs_hi;
            info->reliable_updates += ri.reliable_updates;
            info->shift_resid[i] = ri.true_residual;
            if (st == HISQ_ENOTCONV || st == HISQ_EBREAKDOWN) {
                worst = st;
            } else if (st != HISQ_OK) {
                return st;
            }
        }
        if (!refining) {
            info->matvecs_hi += mv_hi;
            info->true_residual = info->shift_resid[0];
            return status;
        }
        info->matvecs_hi += mv_hi;
        info->true_residual = info->shift_resid[0];
        return worst;
    }
};

}  // namespace

hisq_status run_multishift_stage(hisq_ctx *c, hisq_gauge *g, const hisq_solver_params &p, int ns, const double *sigma,
                                 const double *tol, const double *b64, double *const *x64_out, hisq_solve_info *info,
                                 cudaStream_t s)
{
    MSRun run(c, g, p, s);
    const hisq_status st = run.run(b64, ns, sigma, tol, info, false);
    if (st != HISQ_OK && st != HISQ_ENOTCONV && st != HISQ_EBREAKDOWN) return st;
    for (int i = 0; i < ns; i++)
        cudaMemcpyAsync(x64_out[i], run.x64(i), (size_t)48 * g->geom.vh, cudaMemcpyDeviceToDevice, s);
    const cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(c, e, "multi-shift stage results");
    return st;
}

}  // namespace hisq

using namespace hisq;

extern "C" hisq_status hisq_multishift_cg(hisq_ctx *c, const hisq_gauge *gc, const hisq_solver_params *p, int nshift,
                                          const double *sigma, const double *tol, const double *b, double *const *x,
                                          hisq_solve_info *info)
{
    if (!c || !gc || !sigma || !tol || !b || !x || !info) return fail(c, HISQ_EINVAL, "hisq_multishift_cg: null argument");
    *info = hisq_solve_info{};
    hisq_status e = validate_params(c, p);
    if (e) return e;
    e = check_prec(c, p->refine);
    if (e) return e;
    if (nshift < 1 || nshift > HISQ_MAX_SHIFTS || nshift > kMaxShift)
        return fail(c, HISQ_EINVAL, "nshift must be in 1..%d", HISQ_MAX_SHIFTS);
    for (int i = 0; i < nshift; i++) {
        if (!std::isfinite(sigma[i]) || !(tol[i] > 0.0) || !x[i])
            return fail(c, HISQ_EINVAL, "shift %d: sigma must be finite, tol > 0, x non-null", i);
        if (4.0 * p->mass * p->mass + sigma[i] <= 0.0)
            return fail(c, HISQ_EINVAL, "shift %d: 4m^2 + sigma must be positive", i);
    }
    cudaSetDevice(c->device);
    const auto t0 = std::chrono::steady_clock::now();
    hisq_gauge *g = const_cast<hisq_gauge *>(gc);
    cudaStream_t s = pick_stream(c, p->stream);
    const int64_t vh = g->geom.vh;
    if (!solver_red_fits(vh)) return fail(c, HISQ_EINVAL, "lattice too large for the solvers' reductions");
    // ascending shifts: the smallest is the base system
    std::vector<int> ord(nshift);
    std::iota(ord.begin(), ord.end(), 0);
    std::stable_sort(ord.begin(), ord.end(), [&](int a, int bb) { return sigma[a] < sigma[bb]; });
    std::vector<double> ss(nshift), tt(nshift);
    for (int i = 0; i < nshift; i++) {
        ss[i] = sigma[ord[i]];
        tt[i] = tol[ord[i]];
    }
    Workspace ws(c, s);
    double *b64 = nullptr;
    e = ws.alloc((size_t)48 * vh, (void **)&b64);
    if (!e) e = to_planar(c, ws, b, p->on_device, vh, b64, s);
    if (e) return e;
    hisq_solve_info si{};
    hisq_status st;
    {
        MSRun run(c, g, *p, s);
        st = run.run(b64, nshift, ss.data(), tt.data(), &si);
        if (st != HISQ_OK && st != HISQ_ENOTCONV && st != HISQ_EBREAKDOWN) return st;
        for (int i = 0; i < nshift; i++) {
            e = from_planar(c, ws, run.x64(i), vh, x[ord[i]], p->on_device, s);
            if (e) return e;
        }
    }
    // report per shift in the caller's order
    *info = si;
    for (int i = 0; i < nshift; i++) {
        info->shift_iters[ord[i]] = si.shift_iters[i];
        info->shift_resid_ms[ord[i]] = si.shift_resid_ms[i];
        info->shift_resid[ord[i]] = si.shift_resid[i];
        info->refine_iters[ord[i]] = si.refine_iters[i];
    }
    info->true_residual = si.shift_resid[0];
    info->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    return st;
}
