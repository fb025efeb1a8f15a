// cg_block.cuh -- the CG iteration of a lattice that fits on the chip at once:
// whole blocks of iterations in one cooperative launch.
//
// On a small lattice an iteration of four dependent kernels (two stencil
// passes, the residual and the gradient update) is bound by their latencies:
// 22 us an iteration on 8^4 and 26 us on 16^4 (20-bit), where the links read
// from L2 take under 4 us.  This kernel: 9.8 and 15.3 us.  Every thread group
// owns one site (of each parity) for the whole launch: r, p, A p and the step
// of x stay in registers, only p and the odd-site intermediate go through
// memory (L2), and the kernels' boundaries become four grid-wide exchanges, two
// barriers and two sums:
//   tmp = D_oe p | barrier | A p = diag p - D_eo tmp, <p, A p> | sum barrier |
//   r -= alpha A p, |r|^2, <r, r_old> | sum barrier | p = r + beta p | barrier.
// Every block sums the blocks' partials in one fixed order, takes alpha, beta and
// the decision to stop from them as FP64 would (in FP32 pairs wherever these
// cannot differ, see cg_scalars.cuh: an FP64 division in the way of every block
// costs half a microsecond) and keeps its own copy of the solver's state, so the
// decision needs no further exchange; block 0 writes it back.
//
// S lanes share a site (one or more directions each, their sums combined by
// shuffles): four or two while that takes one block of at most 512 threads an SM,
// else one, with up to 1024 threads (cg_block_shape), so that 8^4 occupies the
// whole chip and 16^3x64 still fits.
//
// The blocks of the launch wait for one another: the launch is cooperative
// (all of them resident or none; with 40 SMs taken by another stream's kernel for
// two seconds a 16^3x32 solve began after that and gave the same bits), every
// wait is bounded, and a wait that gives up sets bit 2 of the error word and ends
// its block.
#pragma once

#include <cuda_runtime.h>

#include "cg.h"
#include "cg_scalars.cuh"
#include "codecs.cuh"
#include "dslash.cuh"
#include "finish.cuh"
#include "internal.h"
#include "reduce.cuh"

namespace hisq {

// Lanes s of the S lanes of site cb: the terms of their directions of D in at
// output parity po, summed over the lanes (every lane returns all of it), in
// units of the fat scale.
template <int GF, int SF, int LREC, int S>
__device__ __forceinline__ void lane_stencil(const DslashArgs &a, const char *in, int po, int lane_s, int xh, int y,
                                             int z, int t, int cb, size_t pstride, float lsc, float ratio, float o[6])
{
    SiteAccPacked acc;
    acc.zero();
    const int x = 2 * xh + ((y + z + t + po) & 1);
    const int lex = 2 * cb + (x & 1);
#pragma unroll
    for (int k = 0; k < 4 / S; k++) {
        const int mu = lane_s * (4 / S) + k;
        const int cmu = mu == 0 ? x : mu == 1 ? y : mu == 2 ? z : t;
        const int phase_sum = mu == 0 ? 0 : mu == 1 ? x : mu == 2 ? x + y : x + y + z;
        // other blocks write `in` between barriers (plain loads); the links are read every pass (kept in L2)
        stencil_direction<GF, SF, float, LREC, 2, true>(a, in, mu, cmu, t, lex, cb, po, pstride, lsc, ratio,
                                                           phase_sum, acc);
    }
#pragma unroll
    for (int k = 0; k < 6; k++) {
        o[k] = acc.get(k);
#pragma unroll
        for (int off = 1; off < S; off *= 2) o[k] += __shfl_xor_sync(0xffffffffu, o[k], off);
    }
}

// Every block arrives, then waits until all have (target arrivals in all since
// the launch began); thread 0 runs `meanwhile` between its arrival and its
// wait.  False when the wait gave up.
template <typename F>
__device__ __forceinline__ bool grid_arrive_wait(const CGBlockArgs &a, unsigned target, int *ok_sh, F meanwhile)
{
    __syncthreads();  // the block's writes precede the release
    if (threadIdx.x == 0) {
        red_release_add(a.bar, 1u);
        meanwhile();
        unsigned polls = 0;
        int ok = 1;
        while (ld_acquire(a.bar) < target + a.wait_extra)
            if (++polls > a.wait_polls) {
                atomicOr(a.err, 2);
                ok = 0;
                break;
            }
        *ok_sh = ok;
    }
    __syncthreads();
    return *ok_sh != 0;
}

// Sum of two values over the grid, in every block (warp 0; lane 0 holds tot).
// Each block writes its FP32 sums, as two 64-bit words of value and tag, into
// the inbox of every block, and warp 0 of each block reads its own inbox until
// every word carries this sum's tag: the words are barrier and data at once.
// Nothing else is ordered by it.  The two sets of inboxes alternate: a block can
// only write into a set again after every block has written, hence read past,
// the sum in between.  Partials are summed in FP32 pairs in a fixed order.
// Measured on 152 blocks, in cycles: an arrival counter and a second round of
// loads 4600 to 5000; one shared row of words that every block polls 7200 (152
// SMs reading the same lines); inboxes 3000 to 3600.
__device__ __forceinline__ bool grid_sum(const CGBlockArgs &a, float v[2], unsigned tag, FF tot[2], float (*sh)[2])
{
    block_sum<2, float>(v, sh);
    if (threadIdx.x >= 32) return true;
    const unsigned nb = gridDim.x, want = tag + a.wait_extra;
    ulonglong2 *set = a.inbox + (size_t)(tag & 1u) * nb * nb;
    const unsigned long long t64 = (unsigned long long)tag << 32;
    const unsigned long long s0 = t64 | __float_as_uint(__shfl_sync(0xffffffffu, v[0], 0));
    const unsigned long long s1 = t64 | __float_as_uint(__shfl_sync(0xffffffffu, v[1], 0));
    for (unsigned b = threadIdx.x; b < nb; b += 32)
        asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(set + (size_t)b * nb + blockIdx.x), "l"(s0),
                     "l"(s1)
                     : "memory");
    const ulonglong2 *slots = set + (size_t)blockIdx.x * nb;
    bool ok = true;
    tot[0] = tot[1] = FF{0.0f, 0.0f};
    constexpr int U = 5;  // words of that many blocks in flight a lane: one round for 152 blocks
    for (unsigned b0 = threadIdx.x; b0 < nb; b0 += 32 * U) {
        unsigned long long w0[U], w1[U];
        unsigned polls = 0;
        for (;;) {
            bool all = true;
#pragma unroll
            for (int u = 0; u < U; u++) {
                const unsigned b = b0 + 32 * u < nb ? b0 + 32 * u : b0;
                asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];"
                             : "=l"(w0[u]), "=l"(w1[u])
                             : "l"(slots + b)
                             : "memory");
            }
#pragma unroll
            for (int u = 0; u < U; u++)
                all = all && (unsigned)(w0[u] >> 32) == want && (unsigned)(w1[u] >> 32) == want;
            if (all) break;
            if (++polls > a.wait_polls) {
                ok = false;
                break;
            }
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (b0 + 32 * u >= nb) continue;
            tot[0] = ff_add(tot[0], FF{__uint_as_float((unsigned)w0[u]), 0.0f});
            tot[1] = ff_add(tot[1], FF{__uint_as_float((unsigned)w1[u]), 0.0f});
        }
    }
    warp_sum_ff<2>(tot);
    ok = __all_sync(0xffffffffu, ok);
    if (!ok && threadIdx.x == 0) atomicOr(a.err, 2);
    return ok;
}

template <int GF, int SF, int LREC, int S, int T>
__global__ void __launch_bounds__(T, 1) cg_block_kernel(const __grid_constant__ CGBlockArgs a)
{
    constexpr int C = Spinor<SF>::chunks;
    __shared__ CGState st;  // this block's copy
    __shared__ float sums_sh[32][2];
    __shared__ FF tot_ap[2], tot_r[2];  // <p, A p>, |A p|^2 and |r|^2, <r, r_old> of the iteration
    __shared__ float step_sh;           // alpha, then beta
    __shared__ float ring_sh[kMaxBuf];  // the steps of the ring's slots
    __shared__ int ok_sh;
    const Geom &g = a.d.g;
    const int vh = g.vh;
    for (int k = threadIdx.x; k < (int)(sizeof(CGState) / 4); k += blockDim.x)
        reinterpret_cast<unsigned *>(&st)[k] = reinterpret_cast<const unsigned *>(a.st)[k];
    if (threadIdx.x < kMaxBuf) ring_sh[threadIdx.x] = 0.0f;  // a breakdown's flush reads every slot
    const unsigned tag0 = __ldcg(a.seq);  // of the launch's first sum
    unsigned tag = tag0;
    const unsigned nb = gridDim.x;
    // Every block counts itself out, whichever way it ends; the last one zeroes the counters for the next launch
    // and moves the first tag past every tag in the slots.  The fence: this block's arrivals precede its leaving.
    auto leave = [&] {
        if (threadIdx.x != 0) return;
        __threadfence();
        if (atomicAdd(a.bar + 8, 1u) != nb - 1) return;
        a.bar[0] = 0u;
        a.bar[8] = 0u;
        *a.seq = tag0 + 2u * (unsigned)a.iters + 2u;
    };
    __syncthreads();
    if (st.active == 0) {  // uniform over the grid, unless a wait of an earlier block has given up already
        leave();
        return;
    }
    if (threadIdx.x == 0 && blockIdx.x != 0) st.hist = nullptr;  // block 0 keeps the history

    const int group = (int)((blockIdx.x * blockDim.x + threadIdx.x) / S), lane_s = threadIdx.x % S;
    const bool lead = group < vh && lane_s == 0;
    const int cb = group < vh ? group : vh - 1;  // idle groups repeat the last site, without storing it
    int q = cb / g.xh;
    const int xh = cb - q * g.xh;
    const int y = q % g.L[1];
    q /= g.L[1];
    const int z = q % g.L[2], t = q / g.L[2];
    const size_t pstride = (size_t)8 * vh * 16;
    constexpr bool kScaled = LinkScaled<GF>::value;
    const float fsc = kScaled ? a.d.gv.fat_scale_f : 1.0f;
    const float lsc = kScaled ? a.d.gv.lng_scale_f : 1.0f;
    const float ratio = lsc / fsc;
    const float diag = (float)a.diag;
    const int pr = st.pr;
    // Thread 0: the recurrence's scalars in FP32 pairs (FP64 divisions, and even conversions, of a launch's every
    // iteration would stand in every block's way), FP64 deciding where a pair cannot.  The sums are pairs, so
    // their doubles are known exactly; those of the launch's start stay in st.  The state receives the doubles at
    // the end of the launch, or each iteration where a history or the error-estimate trigger asks for the FP64
    // finishers.
    const bool fp64 = st.dyn || a.st->hist != nullptr;
    ff rr(st.rr), rr_prev(0.0f), rr_max(st.rr_max);
    const float delta2 = (float)st.delta2, stop2 = (float)st.stop2;
    int steps = 0;          // updates of rr so far: the first makes rr, the second rr_prev a sum's pair
    bool max_sum = false;   // rr_max is a sum's pair
    float al_used = 0.0f, be_used = 0.0f;

    float r[6], p[6], dx[6] = {0, 0, 0, 0, 0, 0};
    {
        uint4 c[C];
        gather_coherent<SF>(a.r, vh, cb, c);
        Spinor<SF>::decode(c, r);
        gather_coherent<SF>(a.ring, vh, cb, c);
        Spinor<SF>::decode(c, p);
    }
    unsigned arrived = 0;  // the target of the next barrier
    bool bad = false, gave_up = false;
    auto f64 = [](FF v) { return (double)v.hi + (double)v.lo; };
    auto rr64 = [&] { return steps > 0 ? (double)rr : st.rr; };
    auto max64 = [&] { return max_sum ? (double)rr_max : st.rr_max; };
    // thread 0, after iteration i: the finishers' decisions
    auto finish = [&](int i) {
        if (fp64) {
            double tot[2] = {f64(tot_ap[0]), f64(tot_ap[1])};
            run_finisher(FIN_CG_ALPHA, tot, &st, i);
            tot[0] = f64(tot_r[0]);
            tot[1] = f64(tot_r[1]);
            run_finisher(FIN_CG_BETA, tot, &st, i);
        } else {
            st.k += 1;
            if (decide_less(rr_max.hi, rr.hi, [&](double &x, double &y) { x = max64(), y = (double)rr; })) {
                rr_max = rr;
                max_sum = true;
            }
            if (!decide_less(stop2, rr.hi, [&](double &x, double &y) { x = st.stop2, y = (double)rr; }))
                stop_iterating(&st, REASON_CONVERGED);
            else if (decide_less(rr.hi, delta2 * rr_max.hi,
                                 [&](double &x, double &y) { x = (double)rr, y = st.delta2 * max64(); }))
                stop_iterating(&st, REASON_RELIABLE);
        }
        ring_sh[i] = i == a.nslots - 1 ? 0.0f : al_used;
        if (i == a.nslots - 1)
            for (int j = 0; j < kMaxBuf; j++) ring_sh[j] = 0.0f;
    };

    for (int it = 0; it < a.iters; it++) {
        const int i = it % a.nslots;
        // odd sites: tmp = D_oe p
        float o[6];
        lane_stencil<GF, SF, LREC, S>(a.d, a.ring + (size_t)i * a.slot_bytes, 1, lane_s, xh, y, z, t, cb, pstride, lsc,
                                      ratio, o);
        uint4 c[C];
#pragma unroll
        for (int k = 0; k < 6; k++) o[k] *= fsc;
        bad = !Spinor<SF>::encode(o, c) || bad;
        if (lead) Spinor<SF>::put(a.tmp, vh, cb, c);
        if (!grid_arrive_wait(a, arrived += nb, &ok_sh, [] {})) {
            gave_up = true;
            break;
        }

        // even sites: A p and its sums
        float ap[6];
        lane_stencil<GF, SF, LREC, S>(a.d, a.tmp, 0, lane_s, xh, y, z, t, cb, pstride, lsc, ratio, ap);
        float v[2] = {0.0f, 0.0f};
#pragma unroll
        for (int k = 0; k < 6; k++) {
            ap[k] = diag * p[k] - fsc * ap[k];
            v[0] += p[k] * ap[k];
            v[1] += ap[k] * ap[k];
        }
        if (!lead) v[0] = v[1] = 0.0f;
        FF tot[2];
        bool got = grid_sum(a, v, tag++, tot, sums_sh);
        if (threadIdx.x == 0) {
            tot_ap[0] = tot[0];
            tot_ap[1] = tot[1];
            step_sh = al_used = step_quotient(rr, ff(0.0f), ff(tot[0].hi, tot[0].lo), [&](double &n, double &d) {
                n = rr64();
                d = f64(tot[0]);
            });
            ok_sh = !got ? 0 : tot[0].hi > 0.0f && isfinite(al_used) ? 1 : 2;
        }
        __syncthreads();
        if (ok_sh != 1) {  // the wait gave up, or a breakdown: every block has the same sums
            gave_up = ok_sh == 0;
            if (ok_sh == 2 && threadIdx.x == 0) stop_iterating(&st, REASON_BREAKDOWN);
            break;
        }

        // r, its sums, and the step of x
        const float alpha = step_sh;
        v[0] = v[1] = 0.0f;
#pragma unroll
        for (int k = 0; k < 6; k++) {
            const float rn = r[k] - alpha * ap[k];
            v[0] += rn * rn;
            v[1] += rn * r[k];
            r[k] = rn;
            dx[k] += alpha * p[k];
        }
        if (!lead) v[0] = v[1] = 0.0f;
        got = grid_sum(a, v, tag++, tot, sums_sh);
        if (threadIdx.x == 0) {
            tot_r[0] = tot[0];
            tot_r[1] = tot[1];
            const ff rn(tot[0].hi, tot[0].lo);
            step_sh = be_used = step_quotient(rn, pr ? ff(tot[1].hi, tot[1].lo) : ff(0.0f), rr, [&](double &n, double &d) {
                n = pr ? f64(tot[0]) - f64(tot[1]) : f64(tot[0]);
                d = rr64();
            });
            rr_prev = rr;
            rr = rn;
            steps++;
            ok_sh = !got ? 0 : isfinite(tot[0].hi) && isfinite(be_used) ? 1 : 2;
        }
        __syncthreads();
        if (ok_sh == 0) {
            gave_up = true;
            break;
        }
        if (i == a.nslots - 1) {  // the ring is full: x is brought up to date
            if (lead) {
                uint4 cx[Spinor<S_F64>::chunks];
                double x[6];
                char *xf = reinterpret_cast<char *>(a.x64);
                gather_coherent<S_F64>(xf, vh, cb, cx);
                Spinor<S_F64>::decode(cx, x);
#pragma unroll
                for (int k = 0; k < 6; k++) x[k] += f2d_bits(dx[k]);
                Spinor<S_F64>::encode(x, cx);
                Spinor<S_F64>::put(xf, vh, cb, cx);
            }
#pragma unroll
            for (int k = 0; k < 6; k++) dx[k] = 0.0f;
            // r as a launch that ended here would leave it: where the launches are cut changes no bit
            bad = !Spinor<SF>::encode(r, c) || bad;
            Spinor<SF>::decode(c, r);
        }
        if (ok_sh == 2) {
            if (threadIdx.x == 0) {
                finish(i);
                stop_iterating(&st, REASON_BREAKDOWN);
            }
            break;
        }

        // p, as the next pass reads it
        const float beta = step_sh;
#pragma unroll
        for (int k = 0; k < 6; k++) p[k] = r[k] + beta * p[k];
        bad = !Spinor<SF>::encode(p, c) || bad;
        if (lead) Spinor<SF>::put(a.ring + (size_t)((i + 1) % a.nslots) * a.slot_bytes, vh, cb, c);
        Spinor<SF>::decode(c, p);
        if (!grid_arrive_wait(a, arrived += nb, &ok_sh, [&] { finish(i); })) {
            gave_up = true;
            break;
        }
        if (st.active == 0) break;  // stopped by this iteration's decisions, the same in every block
    }

    uint4 c[C];
    bad = !Spinor<SF>::encode(r, c) || bad;
    if (lead) Spinor<SF>::put(a.r, vh, cb, c);
    if (bad && lead) atomicOr(a.err, 1);
    if (threadIdx.x == 0) {
        if (!fp64) {
            if (steps > 0) {
                st.rr_prev = steps > 1 ? (double)rr_prev : st.rr;
                st.rr = (double)rr;
            }
            st.rr_max = max64();
            st.pAp = f64(tot_ap[0]);
            st.apap = f64(tot_ap[1]);
            st.alpha = (double)al_used;
        }
        st.beta = (double)be_used;
        for (int j = 0; j < a.nslots; j++) st.alpha_ring[j] = (double)ring_sh[j];
        if (gave_up) {  // the host stops here; the error word tells why
            st.active = 0;
            st.reason = REASON_BREAKDOWN;
        }
    }
    __syncthreads();
    if (blockIdx.x == 0)
        for (int k = threadIdx.x; k < (int)(sizeof(CGState) / 4); k += blockDim.x)
            reinterpret_cast<unsigned *>(a.st)[k] = reinterpret_cast<const unsigned *>(&st)[k];
    leave();
}

template <int GF, int SF, int LREC, int S, int T>
bool launch_cg_block_s(const CGBlockArgs &a, int nb, int threads, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nb);
    cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, cg_block_kernel<GF, SF, LREC, S, T>, a) == cudaSuccess;
}

template <int GF, int SF, int LREC>
bool launch_cg_block_r(const CGBlockShape &sh, const CGBlockArgs &a, cudaStream_t s)
{
    if (sh.lanes == 4) return launch_cg_block_s<GF, SF, LREC, 4, 512>(a, sh.blocks, sh.threads, s);
    if (sh.lanes == 2) return launch_cg_block_s<GF, SF, LREC, 2, 512>(a, sh.blocks, sh.threads, s);
    if (sh.threads <= 512) return launch_cg_block_s<GF, SF, LREC, 1, 512>(a, sh.blocks, sh.threads, s);
    return launch_cg_block_s<GF, SF, LREC, 1, 1024>(a, sh.blocks, sh.threads, s);
}

template <int GF, int SF>
bool launch_cg_block_t(int long_recon, const CGBlockShape &sh, const CGBlockArgs &a, cudaStream_t s)
{
    if (long_recon == 12) return launch_cg_block_r<GF, SF, 12>(sh, a, s);
    if (long_recon == 18) return launch_cg_block_r<GF, SF, 18>(sh, a, s);
    return false;
}

}  // namespace hisq
