// blas_update.cuh -- the residual and gradient-vector updates of a CG iteration
// on groups of U sites a thread (every load of a group issued before any is
// used), shared by the single-system and the batched kernels.
#pragma once

#include <cuda_runtime.h>

#include "blas.h"
#include "codecs.cuh"
#include "reduce.cuh"

namespace hisq {

// A solver scalar (FP64 in the state) in the compute precision.  For FP32
// pairs the conversion runs on GB300's narrow FP64 pipe, so one thread of the
// block converts and the block reads the pair from shared memory.  Every
// thread of the block calls it, at most once per kernel.
template <typename real>
__device__ __forceinline__ real block_scalar(const double *src)
{
    if constexpr (is_ff<real>::value) {
        __shared__ ff sh;
        if (threadIdx.x == 0) sh = ff(*src);
        __syncthreads();
        return sh;
    } else {
        return (real)*src;
    }
}

// The partials' second half: the split chain's residual update leaves its block
// sums there while it reads the stencil pass's from the first.
inline __device__ RedBuf split_half(RedBuf rb)
{
    rb.partials += kSplitHalf;
    return rb;
}

// Loads of r (v0) and Ap (v1) at the U sites i0 + u * blockDim.x.
template <int SF, int U, int C>
__device__ __forceinline__ void r_load(const BlasArgs &a, int i0, uint4 (&cr)[U][C], uint4 (&ca)[U][C])
{
#pragma unroll
    for (int u = 0; u < U; u++) {
        const int i = i0 + u * blockDim.x;
        if (i < a.n) {
            Spinor<SF>::gather(a.v0, a.n, i, cr[u]);
            Spinor<SF>::gather(a.v1, a.n, i, ca[u]);
        }
    }
}

// r - alpha Ap at those sites, stored in out (r itself or another field); |r_new|^2 and Re<r_new, r_old> added to v.
template <int SF, typename real, int U, int C>
__device__ __forceinline__ void r_group(const BlasArgs &a, int i0, const uint4 (&cr)[U][C], const uint4 (&ca)[U][C],
                                        real alpha, red_t<real> v[2], char *out)
{
#pragma unroll
    for (int u = 0; u < U; u++) {
        const int i = i0 + u * blockDim.x;
        if (i >= a.n) continue;
        if constexpr (SF == S_INT30 && is_ff<real>::value) {
            // FP64-class: the update in FP32 pairs; |r|^2 and Re<r_new, r_old> exactly in integers
            // from the stored 30-bit records (products of 30-bit integers, sums below 2^62)
            int32_t qr[6];
            const uint32_t Er = Spinor<S_INT30>::raw(cr[u], qr);
            ff r[6], ap[6], rn[6];
            Spinor<S_INT30>::decode(cr[u], r);
            Spinor<S_INT30>::decode(ca[u], ap);
#pragma unroll
            for (int k = 0; k < 6; k++) rn[k] = r[k] - alpha * ap[k];
            uint32_t qn[6], En;
            if (!Spinor<S_INT30>::store_ff_q(out, a.n, i, rn, qn, En)) atomicExch(a.err, 1);
            long long n2 = 0, d = 0;
#pragma unroll
            for (int k = 0; k < 6; k++) {
                asm("mad.wide.s32 %0, %1, %1, %0;" : "+l"(n2) : "r"((int)qn[k]));
                asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(d) : "r"((int)qn[k]), "r"(qr[k]));
            }
            // a record's value is q 2^(E-127)
            v[0] += ff_ldexp(ff_from_ll(n2), 2 * (int)En - 254);
            v[1] += ff_ldexp(ff_from_ll(d), (int)En + (int)Er - 254);
        } else {
            real r[6], ap[6], rn[6];
            Spinor<SF>::decode(cr[u], r);
            Spinor<SF>::decode(ca[u], ap);
            real n2 = real(0), d = real(0);  // in the compute precision; the block sums the threads
#pragma unroll
            for (int k = 0; k < 6; k++) {
                rn[k] = r[k] - alpha * ap[k];
                n2 += rn[k] * rn[k];
                d += rn[k] * r[k];
            }
            v[0] += (red_t<real>)n2;
            v[1] += (red_t<real>)d;
            if (!Spinor<SF>::store(out, a.n, i, rn)) atomicExch(a.err, 1);
        }
    }
}

template <int SF, int U, int C>
__device__ __forceinline__ void p_load(const BlasArgs &a, int i0, uint4 (&cr)[U][C], uint4 (&cp)[U][C])
{
#pragma unroll
    for (int u = 0; u < U; u++) {
        const int i = i0 + u * blockDim.x;
        if (i < a.n) {
            Spinor<SF>::gather(a.v0, a.n, i, cr[u]);
            Spinor<SF>::gather(a.v1, a.n, i, cp[u]);
        }
    }
}

// p' = r + beta p at those sites, stored into v2.
template <int SF, typename real, int U, int C>
__device__ __forceinline__ void p_group(const BlasArgs &a, int i0, const uint4 (&cr)[U][C], const uint4 (&cp)[U][C],
                                        real beta)
{
#pragma unroll
    for (int u = 0; u < U; u++) {
        const int i = i0 + u * blockDim.x;
        if (i >= a.n) continue;
        real r[6], p[6];
        Spinor<SF>::decode(cr[u], r);
        Spinor<SF>::decode(cp[u], p);
#pragma unroll
        for (int k = 0; k < 6; k++) p[k] = r[k] + beta * p[k];
        if (!Spinor<SF>::store(a.v2, a.n, i, p)) atomicExch(a.err, 1);
    }
}

}  // namespace hisq
