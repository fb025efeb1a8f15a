// convert.cu -- format conversion kernels: spinor pack/unpack between the
// caller's FP64 [site][6] layout and the storage formats, and the gauge
// loader's scale, compression check and quantisation passes.
#include <cuda_runtime.h>

#include <cstdint>

#include "codecs.cuh"
#include "internal.h"
#include "launch.cuh"

namespace hisq {

namespace {

constexpr int kBlock = 256;

// The conversions between the caller's [site][6] arrays and the storage formats
// are bound by their bytes: full-line accesses through shared memory and FP64
// <-> FP32 on the integer pipe (codecs.cuh).  20-bit, 663589 sites: pack 10.6
// us, unpack 19.0 us with strided accesses and the conversion instructions.
template <int SF, typename T>
__device__ __forceinline__ bool pack_warp(int64_t n, const T *in, char *out, T *sh)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t i0 = i & ~(int64_t)31;
    if (i0 >= n) return true;
    T v[6];
    warp_load_sites(in, i0, n, v, sh);
    return i >= n || Spinor<SF>::store(out, (int)n, (int)i, v);
}

// Sites that cannot be encoded: counted on the device, and (host not null) reported to a host-mapped word,
// which stays zero otherwise, so that the caller has nothing to copy back.
__device__ __forceinline__ void report_bad(int *bad, int *host)
{
    atomicAdd(bad, 1);
    if (host != nullptr) *(volatile int *)host = 1;
}

// FP64 input; FP32 input goes through the FP32 store (the one FP32-compute kernels use)
template <int SF, typename T>
__global__ void __launch_bounds__(kBlock) pack_kernel(int64_t n, const T *in, char *out, int *bad, int *host)
{
    __shared__ __align__(16) T sh[kBlock / 32][192];
    if (!pack_warp<SF>(n, in, out, sh[threadIdx.x >> 5])) report_bad(bad, host);
}

// FP32-pair input [n][6][hi, lo] through the pair store (FP64-class kernels)
__global__ void pack_pair_kernel(int64_t n, const float *in, char *out, int *bad, int *host)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    ff v[6];
#pragma unroll
    for (int k = 0; k < 6; k++) v[k] = ff(in[12 * i + 2 * k], in[12 * i + 2 * k + 1]);
    if (!Spinor<S_INT30>::store(out, (int)n, (int)i, v)) report_bad(bad, host);
}

// Field blockIdx.y of several (the halves of the stencil entry point's inputs)
template <int SF>
__global__ void __launch_bounds__(kBlock) pack_fields_kernel(int64_t n, const __grid_constant__ PackFields f)
{
    __shared__ __align__(16) double sh[kBlock / 32][192];
    pdl_wait();
    const int y = (int)blockIdx.y;
    const double *in = y == 0 ? f.in[0] : y == 1 ? f.in[1] : y == 2 ? f.in[2] : f.in[3];
    char *out = y == 0 ? f.out[0] : y == 1 ? f.out[1] : y == 2 ? f.out[2] : f.out[3];
    const bool ok = pack_warp<SF>(n, in, out, sh[threadIdx.x >> 5]);
    pdl_launch_dependents();
    if (!ok) {
        *(volatile int *)f.bad = 1;
        *(volatile int *)f.bad_host = 1;
    }
}

template <int SF, typename real>
__global__ void __launch_bounds__(kBlock) unpack_kernel(int64_t n, const char *in, double *out)
{
    __shared__ __align__(16) double sh[kBlock / 32][192];
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t i0 = i & ~(int64_t)31;
    if (i0 >= n) return;
    double v[6];
    if (i < n) {
        uint4 c[Spinor<SF>::chunks];
        Spinor<SF>::gather(in, (int)n, (int)i, c);
        decode_f64<SF, real>(c, v);
    }
    warp_store_sites(out, i0, n, v, sh[threadIdx.x >> 5]);
}

__device__ __forceinline__ void atomic_max_nonneg(double *addr, double v)
{
    // non-negative doubles order like their bit patterns (NaN sorts above Inf)
    atomicMax(reinterpret_cast<unsigned long long *>(addr), (unsigned long long)__double_as_longlong(v));
}

__device__ __forceinline__ void lex_coords(const Geom &g, int lex, int c[4])
{
    c[0] = lex % g.L[0];
    int r = lex / g.L[0];
    c[1] = r % g.L[1];
    r /= g.L[1];
    c[2] = r % g.L[2];
    c[3] = r / g.L[2];
}

// idx = mu V + lex, without a 64-bit division
__device__ __forceinline__ void link_index(int64_t idx, int V, int &mu, int &lex)
{
    mu = (idx >= V) + (idx >= 2LL * V) + (idx >= 3LL * V);
    lex = (int)(idx - (int64_t)mu * V);
}

// A warp's 32 consecutive links of an FP64 [mu][lex][18] field, from idx0 on
// (fewer at the field's end), to shared memory in full lines; a link's 18 reals
// are kLinkPad apart there (a lane's walk over its own link then meets no bank
// conflict).  f(bits, address) sees every real once, by the lane that loaded it.
constexpr int kLinkPad = 19;
constexpr int kLinkBlock = 128;
template <typename F>
__device__ __forceinline__ void warp_load_links(const double *links, int64_t idx0, int64_t n, double *sh, F f)
{
    const int lane = threadIdx.x & 31;
    const int m = 18 * (int)(n - idx0 < 32 ? n - idx0 : 32);
    // as bit patterns: an absolute value written on doubles becomes an FP64 instruction
    const unsigned long long *src = reinterpret_cast<const unsigned long long *>(links) + 18 * idx0;
    unsigned long long v[18];
#pragma unroll
    for (int k = 0; k < 18; k++) {
        const int j = lane + 32 * k;
        v[k] = j < m ? __ldcs(src + j) : 0ull;
    }
#pragma unroll
    for (int k = 0; k < 18; k++) {
        const int j = lane + 32 * k;
        if (j >= m) continue;
        reinterpret_cast<unsigned long long *>(sh)[j / 18 * kLinkPad + j % 18] = v[k];
        f(v[k], 18 * idx0 + j);
    }
    __syncwarp();
}

// Row 2's deviation from sign * conj(row0 x row1), and the deviation of U U^+
// from 1, of one link in FP64.
__device__ __noinline__ double r12_dev64(const double *u, double sign)
{
    double R[18], m = 0.0;
    for (int j = 0; j < 18; j++) R[j] = u[j];
    rebuild_row2(R, sign);
    for (int j = 12; j < 18; j++) {
        const double d = fabs(R[j] - u[j]);
        m = (d > m || d != d) ? d : m;
    }
    return m;
}

__device__ __noinline__ double u3_dev64(const double *u)
{
    double m = 0.0;
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) {
            double re = 0.0, im = 0.0;  // sum_k U_ik conj(U_jk)
            for (int k = 0; k < 3; k++) {
                const double ar = u[2 * (3 * i + k)], ai = u[2 * (3 * i + k) + 1];
                const double br = u[2 * (3 * j + k)], bi = u[2 * (3 * j + k) + 1];
                re += ar * br + ai * bi;
                im += ai * br - ar * bi;
            }
            const double d = fmax(fabs(re - (i == j ? 1.0 : 0.0)), fabs(im));
            m = (d > m || d != d) ? d : m;
        }
    return m;
}

// A double as an FP32 pair on the integer and FP32 pipes: the top 24 bits, and
// the other 29 rounded to FP32 (below 2^-126 as zero); |d| < 2^127.
__device__ __forceinline__ ff d2ff_bits(double d)
{
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    const uint32_t e = (hi >> 20) & 0x7ffu, sg = hi & 0x80000000u;
    if (e < 897u) return ff(0.0f);
    const float h = __uint_as_float(sg | __funnelshift_l(lo, (hi & 0x7fffffffu) - (896u << 20), 3));
    if (e < 950u) return ff(h);
    const float sc = __uint_as_float(sg | ((e - 948u) << 23));  // 2^(e - 1075)
    return ff(h, __fmul_rn(__uint2float_rn(lo & 0x1fffffffu), sc));
}

// The same two deviations in FP32 pairs (about 46 bits): FP64 arithmetic at
// GB300's rate bounded the checks (70 and 171 us for a field of 524288 links,
// 11 us of bytes).
__device__ __forceinline__ float r12_dev_ff(const ff u[18], float sign)
{
    float m = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const int k = (c + 1) % 3, l = (c + 2) % 3;
        const ff *ak = u + 2 * k, *al = u + 2 * l, *bk = u + 6 + 2 * k, *bl = u + 6 + 2 * l;
        const ff cr = (ak[0] * bl[0] - ak[1] * bl[1]) - (al[0] * bk[0] - al[1] * bk[1]);
        const ff ci = (ak[0] * bl[1] + ak[1] * bl[0]) - (al[0] * bk[1] + al[1] * bk[0]);
        const float dr = fabsf((ff_scale(cr, sign) - u[12 + 2 * c]).hi);
        const float di = fabsf((ff_scale(ci, -sign) - u[13 + 2 * c]).hi);
        m = fmaxf(m, fmaxf(dr, di));
    }
    return m;
}

// near: row 2 is the product of rows 0 and 1 to 1e-8.  Then U U^+ follows from
// the first two rows (each further entry is off by at most a few times theirs
// plus the row's own deviation), and only the first three pairs are formed.
__device__ __forceinline__ float u3_dev_ff(const ff u[18], bool near)
{
    float m = 0.0f;
#pragma unroll
    for (int j = 0; j < 3; j++)
#pragma unroll
        for (int i = 0; i <= j; i++) {  // (j, i) is its conjugate
            if (j == 2 && near && m < 1e-8f) continue;
            ff re(i == j ? -1.0f : 0.0f), im(0.0f);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const ff *a = u + 2 * (3 * i + k), *b = u + 2 * (3 * j + k);
                re += a[0] * b[0] + a[1] * b[1];
                if (i != j) im += a[1] * b[0] - a[0] * b[1];
            }
            m = fmaxf(m, fmaxf(fabsf(re.hi), fabsf(im.hi)));
        }
    return m;
}

// A gauge field at load, in one pass over its links (five passes before, two of
// them bound by FP64 arithmetic): the resident copy (COPY), the bits of the
// largest |element| (out[0]; non-negative doubles order like their bits, NaN
// above infinity), whether some link's row 2 is not sign * conj(row0 x row1)
// to 1e-6 (out[1], k = 1 fat, k = 3 long) and, for the long links, whether some
// link is not unitary to 1e-6 (out[2]).  The deviations are taken in FP32 pairs;
// a link whose deviation comes within 0.1 % of the bound, or whose elements
// exceed 16, is decided in FP64.
constexpr double kCompressTol = 1e-6;
template <bool LONG, bool COPY>
__global__ void __launch_bounds__(kLinkBlock) gauge_scan_kernel(Geom g, const double *links, double *copy,
                                                                unsigned long long *out)
{
    __shared__ double sh[kLinkBlock / 32][32 * kLinkPad];
    __shared__ unsigned long long mx_sh[kLinkBlock / 32];
    const int V = 2 * g.vh, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t n = 4LL * V;
    const int64_t idx = (int64_t)blockIdx.x * kLinkBlock + threadIdx.x, idx0 = idx - lane;
    unsigned long long mx = 0;
    if (idx0 < n) {
        warp_load_links(links, idx0, n, sh[wid], [&](unsigned long long v, int64_t at) {
            const unsigned long long b = v & 0x7fffffffffffffffull;
            mx = b > mx ? b : mx;
            if constexpr (COPY) reinterpret_cast<unsigned long long *>(copy)[at] = v;
        });
    }
    bool bad12 = false, bad3 = false;
    if (idx < n) {
        const double *u = sh[wid] + lane * kLinkPad;
        int mu, lex;
        link_index(idx, V, mu, lex);
        int c[4];
        lex_coords(g, lex, c);
        int ps = 0;
        for (int nu = 0; nu < mu; nu++) ps += c[nu];
        const bool flip = g.antiperiodic_t && mu == 3 && c[3] + (LONG ? 3 : 1) >= g.L[3];
        const float sign = ((ps & 1) != 0) != flip ? -1.0f : 1.0f;
        ff w[18];
        unsigned top = 0;
#pragma unroll
        for (int k = 0; k < 18; k++) {
            const double v = u[k];
            const unsigned h = (unsigned)__double2hiint(v) & 0x7fffffffu;
            top = h > top ? h : top;
            w[k] = d2ff_bits(v);
        }
        const bool big = top >= 0x40300000u;  // 16
        const float lo = (float)(0.999 * kCompressTol), hi = (float)(1.001 * kCompressTol);
        const float d12 = r12_dev_ff(w, sign);
        bad12 = big || !(d12 < lo);
        if (bad12 && (big || d12 <= hi)) {
            const double d = r12_dev64(u, (double)sign);
            bad12 = !(isfinite(d) && d <= kCompressTol);
        }
        if constexpr (LONG) {
            const float d3 = u3_dev_ff(w, d12 < 1e-8f);
            bad3 = big || !(d3 < lo);
            if (bad3 && (big || d3 <= hi)) {
                const double d = u3_dev64(u);
                bad3 = !(isfinite(d) && d <= kCompressTol);
            }
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_down_sync(0xffffffffu, mx, off);
        mx = o > mx ? o : mx;
    }
    if (lane == 0) mx_sh[wid] = mx;
    const int any12 = __syncthreads_or(bad12), any3 = __syncthreads_or(bad3);
    if (threadIdx.x == 0) {
        // (a field that does not compress has bad links everywhere: one store, not one per link)
        volatile unsigned long long *flag = out;
        if (any12 && flag[1] == 0) flag[1] = 1ull;
        if (any3 && flag[2] == 0) flag[2] = 1ull;
        for (int w = 1; w < kLinkBlock / 32; w++) mx = mx_sh[w] > mx ? mx_sh[w] : mx;
        if (mx > *(volatile unsigned long long *)out) atomicMax(out, mx);
    }
}

// FP64 [mu][lex][18] -> stored copy [plane][parity][mu][Vh] in format GF with
// RECON reals per link.  Fixed point: q = rint(x * inv) clamped to +-qmax,
// inv = qmax / global max (Sec. 2 footnote; Sec. 4 for 32 bits).
// rint(fl(x inv)) for |x inv| <= 32767 (1 + 2^-52) without FP64 arithmetic, which
// bounded the 16-bit quantisation (two operations a real, 44 us for 524288
// 18-real links): the product in FP32 pairs is within 2^-30 of x inv, so its
// nearest integer is the one wanted unless it lies that close to a tie, where
// the FP64 rounding decides.
// (The FP64 form is a function of its own, not inlined: written in place it is
// evaluated for every real and then selected.)
__device__ __noinline__ int quantise_f64(double x, double inv)
{
    return __double2loint(__dadd_rn(__dmul_rn(x, inv), 6755399441055744.0));
}

__device__ __forceinline__ int quantise16(double x, double inv, ff inv_ff)
{
    const ff v = d2ff_bits(x) * inv_ff;
    const float t = __fadd_rn(v.hi, 12582912.0f);  // 1.5 2^23: its low bits are v.hi's nearest integer
    const float rest = __fadd_rn(__fsub_rn(v.hi, __fsub_rn(t, 12582912.0f)), v.lo);
    if (fabsf(fabsf(rest) - 0.5f) < 1e-6f) return quantise_f64(x, inv);
    return (int)__float_as_uint(t) - 0x4B400000 + (rest > 0.5f ? 1 : rest < -0.5f ? -1 : 0);
}

// A thread a link in the caller's order, so that both the reads (through shared
// memory) and the writes (16 consecutive links of each parity a warp) are full
// lines.  The fixed-point integers take two FP64 operations a real: the product,
// and the sum with 1.5 2^52, whose low word is the product rounded to the
// nearest even integer (rint, two clamps and a conversion took five; 93 us for
// 524288 18-real links to 16 bits).
template <int GF, int RECON>
__global__ void __launch_bounds__(kLinkBlock) quantise_kernel(Geom g, const double *links, double inv, char *out)
{
    __shared__ double sh[kLinkBlock / 32][32 * kLinkPad];
    const int vh = g.vh;
    const int64_t n = 8LL * vh;
    const int64_t idx = (int64_t)blockIdx.x * kLinkBlock + threadIdx.x;
    const int lane = threadIdx.x & 31;
    if (idx - lane < n) warp_load_links(links, idx - lane, n, sh[threadIdx.x >> 5], [](unsigned long long, int64_t) {});
    if (idx >= n) return;
    int mu, lex;
    link_index(idx, 2 * vh, mu, lex);
    int cc[4];
    lex_coords(g, lex, cc);
    const int t = cc[3];
    const int par = (cc[0] + cc[1] + cc[2] + cc[3]) & 1;
    const int64_t li = (int64_t)(par * 4 + mu) * vh + lex / 2;
    const double *src = sh[threadIdx.x >> 5] + lane * kLinkPad;
    const size_t pstride = (size_t)n * 16;
    constexpr int n16 = link_n16(GF, RECON), tail = link_tail(GF, RECON);
    if constexpr (RECON == 8) {
        // 8 reals of V = sign U (V in SU(3); sign: the long link's staggered phase and boundary
        // sign): arg V00 / pi, arg V20 / pi, V01, V02, V10.  Angles are stored as the format
        // stores a real in [-1, 1] (fixed point: rint(t qmax)), elements as every other element.
        int ps = 0;
        for (int nu = 0; nu < mu; nu++) ps += cc[nu];
        double sg = (ps & 1) ? -1.0 : 1.0;
        if (g.antiperiodic_t && mu == 3 && t + 3 >= g.L[3]) sg = -sg;
        const double inv_pi = 0.31830988618379067154;
        const double pv[8] = {atan2(sg * src[1], sg * src[0]) * inv_pi, atan2(sg * src[13], sg * src[12]) * inv_pi,
                              sg * src[2], sg * src[3], sg * src[4], sg * src[5], sg * src[6], sg * src[7]};
        if constexpr (GF == G_F64) {
            for (int k = 0; k < 4; k++)
                reinterpret_cast<double2 *>(out + k * pstride)[li] = make_double2(pv[2 * k], pv[2 * k + 1]);
        } else if constexpr (GF == G_F32) {
            for (int k = 0; k < 2; k++)
                reinterpret_cast<float4 *>(out + k * pstride)[li] =
                    make_float4((float)pv[4 * k], (float)pv[4 * k + 1], (float)pv[4 * k + 2], (float)pv[4 * k + 3]);
        } else {
            constexpr double qmax = GF == G_FIX16 ? 32767.0 : 2147483647.0;
            int q[8];
            for (int k = 0; k < 8; k++) {
                double v = rint(__dmul_rn(pv[k], k < 2 ? qmax : inv));
                q[k] = (int)fmin(qmax, fmax(-qmax, v));
            }
            if constexpr (GF == G_FIX16) {
                int4 w;
                w.x = (int)((q[0] & 0xffff) | ((uint32_t)q[1] << 16));
                w.y = (int)((q[2] & 0xffff) | ((uint32_t)q[3] << 16));
                w.z = (int)((q[4] & 0xffff) | ((uint32_t)q[5] << 16));
                w.w = (int)((q[6] & 0xffff) | ((uint32_t)q[7] << 16));
                reinterpret_cast<int4 *>(out)[li] = w;
            } else {
                reinterpret_cast<int4 *>(out)[li] = make_int4(q[0], q[1], q[2], q[3]);
                reinterpret_cast<int4 *>(out + pstride)[li] = make_int4(q[4], q[5], q[6], q[7]);
            }
        }
        return;
    }
    if constexpr (GF == G_F64) {
        for (int k = 0; k < RECON / 2; k++)
            reinterpret_cast<double2 *>(out + k * pstride)[li] = make_double2(src[2 * k], src[2 * k + 1]);
    } else if constexpr (GF == G_F32) {
        for (int k = 0; k < n16; k++)
            reinterpret_cast<float4 *>(out + k * pstride)[li] =
                make_float4(d2f_bits(src[4 * k]), d2f_bits(src[4 * k + 1]), d2f_bits(src[4 * k + 2]),
                            d2f_bits(src[4 * k + 3]));
        if constexpr (tail == 8)
            reinterpret_cast<float2 *>(out + n16 * pstride)[li] =
                make_float2(d2f_bits(src[4 * n16]), d2f_bits(src[4 * n16 + 1]));
    } else if constexpr (GF == G_SE15) {
        // per link: 15-bit integers with one exponent, the 30-bit rule in FP64 with scale 2^14 - 1
        // (t = max |x| / (2^14 - 1), 2^(E-127) the power of two just above t); half k = q_k << 1 | bit k
        // of E (k < 8); a link whose exponent does not fit is stored as zero with E = 1
        double mx = 0.0;
        bool ok = true;
        for (int k = 0; k < RECON; k++) {
            ok = ok && isfinite(src[k]);
            mx = fmax(mx, fabs(src[k]));
        }
        const double tq = mx / 16383.0;
        int ex = 0;
        if (tq > 0.0) frexp(tq, &ex);
        int E = tq > 0.0 ? ex + 127 : 1;
        if (E < 1) E = 1;
        if (E > 254) ok = false;
        if (!ok) E = 1;
        uint32_t h[RECON];
        for (int k = 0; k < RECON; k++) {
            const int q = ok ? (int)rint(ldexp(src[k], -(E - 127))) : 0;
            h[k] = (((uint32_t)q & 0x7fffu) << 1) | (k < 8 ? ((uint32_t)E >> k) & 1u : 0u);
        }
        for (int k = 0; k < n16; k++)
            reinterpret_cast<uint4 *>(out + k * pstride)[li] =
                make_uint4(h[8 * k] | (h[8 * k + 1] << 16), h[8 * k + 2] | (h[8 * k + 3] << 16),
                           h[8 * k + 4] | (h[8 * k + 5] << 16), h[8 * k + 6] | (h[8 * k + 7] << 16));
        if constexpr (tail == 4)
            reinterpret_cast<uint32_t *>(out + n16 * pstride)[li] = h[8 * n16] | (h[8 * n16 + 1] << 16);
        else if constexpr (tail == 8)
            reinterpret_cast<uint2 *>(out + n16 * pstride)[li] =
                make_uint2(h[8 * n16] | (h[8 * n16 + 1] << 16), h[8 * n16 + 2] | (h[8 * n16 + 3] << 16));
    } else {
        constexpr double qmax = GF == G_FIX16 ? 32767.0 : 2147483647.0;
        // |x inv| <= qmax (1 + 2^-52), so the rounded product stays within +-qmax
        int q[RECON];
        const ff inv_ff = GF == G_FIX16 ? d2ff_bits(inv) : ff(0.0f);
        // Outside [2^-73, 1e12) the FP64 form: a smaller field's inv overflows, or a real's tail leaves FP32's
        // range; a larger one's inv loses its own tail (below 2^-73), and its elements leave d2ff_bits' (at 2^127).
        if (!(inv >= 0x1p-73 && inv < 1e12)) {
            for (int k = 0; k < RECON; k++) q[k] = (int)fmin(qmax, fmax(-qmax, rint(__dmul_rn(src[k], inv))));
        } else {
#pragma unroll
            for (int k = 0; k < RECON; k++)
                q[k] = GF == G_FIX16 ? quantise16(src[k], inv, inv_ff)
                                     : __double2loint(__dadd_rn(__dmul_rn(src[k], inv), 6755399441055744.0));
        }
        if constexpr (GF == G_FIX16) {
            for (int k = 0; k < n16; k++) {
                int4 w;
                w.x = (int)((q[8 * k] & 0xffff) | ((uint32_t)q[8 * k + 1] << 16));
                w.y = (int)((q[8 * k + 2] & 0xffff) | ((uint32_t)q[8 * k + 3] << 16));
                w.z = (int)((q[8 * k + 4] & 0xffff) | ((uint32_t)q[8 * k + 5] << 16));
                w.w = (int)((q[8 * k + 6] & 0xffff) | ((uint32_t)q[8 * k + 7] << 16));
                reinterpret_cast<int4 *>(out + k * pstride)[li] = w;
            }
            if constexpr (tail == 4) {
                reinterpret_cast<int *>(out + n16 * pstride)[li] =
                    (int)((q[8 * n16] & 0xffff) | ((uint32_t)q[8 * n16 + 1] << 16));
            } else if constexpr (tail == 8) {
                reinterpret_cast<int2 *>(out + n16 * pstride)[li] =
                    make_int2((int)((q[8 * n16] & 0xffff) | ((uint32_t)q[8 * n16 + 1] << 16)),
                              (int)((q[8 * n16 + 2] & 0xffff) | ((uint32_t)q[8 * n16 + 3] << 16)));
            }
        } else {
            for (int k = 0; k < n16; k++)
                reinterpret_cast<int4 *>(out + k * pstride)[li] =
                    make_int4(q[4 * k], q[4 * k + 1], q[4 * k + 2], q[4 * k + 3]);
            if constexpr (tail == 8)
                reinterpret_cast<int2 *>(out + n16 * pstride)[li] = make_int2(q[4 * n16], q[4 * n16 + 1]);
        }
    }
    if constexpr (RECON == 13) {
        // the 13th real: arg det U as a fraction of pi (row 2 = det(U) conj(row0 x row1) for unitary U)
        double u[18];
        for (int k = 0; k < 18; k++) u[k] = src[k];
        auto mre = [&](int i, int j) { return u[2 * (3 * i + j)]; };
        auto mim = [&](int i, int j) { return u[2 * (3 * i + j) + 1]; };
        auto cof = [&](int a, int b, int c, int d, double &r, double &im) {  // m(1,a) m(2,b) - m(1,c) m(2,d)
            r = mre(1, a) * mre(2, b) - mim(1, a) * mim(2, b) - (mre(1, c) * mre(2, d) - mim(1, c) * mim(2, d));
            im = mre(1, a) * mim(2, b) + mim(1, a) * mre(2, b) - (mre(1, c) * mim(2, d) + mim(1, c) * mre(2, d));
        };
        double c0r, c0i, c1r, c1i, c2r, c2i;
        cof(1, 2, 2, 1, c0r, c0i);
        cof(2, 0, 0, 2, c1r, c1i);
        cof(0, 1, 1, 0, c2r, c2i);
        const double dr = mre(0, 0) * c0r - mim(0, 0) * c0i + mre(0, 1) * c1r - mim(0, 1) * c1i + mre(0, 2) * c2r -
                          mim(0, 2) * c2i;
        const double di = mre(0, 0) * c0i + mim(0, 0) * c0r + mre(0, 1) * c1i + mim(0, 1) * c1r + mre(0, 2) * c2i +
                          mim(0, 2) * c2r;
        const double t = atan2(di, dr) * 0.31830988618379067154;  // 1/pi
        char *pp = out + n16 * pstride + (size_t)tail * n;
        if constexpr (GF == G_F64)
            reinterpret_cast<double *>(pp)[li] = t;
        else if constexpr (GF == G_F32)
            reinterpret_cast<float *>(pp)[li] = (float)t;
        else if constexpr (GF == G_FIX16)
            reinterpret_cast<short *>(pp)[li] = (short)rint(t * 32767.0);
        else
            reinterpret_cast<int *>(pp)[li] = (int)rint(t * 2147483647.0);
    }
}

// Error of the long links of a field stored with 8 reals, |U_stored - U| per
// real: the largest (out[0]) and the sum of squares (out[1]).  The stored
// parameters are decoded and V rebuilt in FP64 (the device rebuilds in the
// compute precision), so the result is the storage's own error, amplified
// where the rebuild is ill-conditioned (N = 1 - |V00|^2 or |V20| small).
// el: the element scale (gmax/qmax or 1), an: the angle scale (1/qmax or 1).
template <int GF>
__global__ void r8_check_kernel(Geom g, const double *links, const char *stored, double el, double an, double *out)
{
    const int vh = g.vh;
    const int64_t n = 8LL * vh;
    const size_t pstride = (size_t)n * 16;
    double m = 0.0, q = 0.0;
    for (int64_t li = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; li < n; li += (int64_t)gridDim.x * blockDim.x) {
        const int cb = (int)(li % vh);
        const int pm = (int)(li / vh);
        const int par = pm >> 2, mu = pm & 3;
        int r = cb / g.xh;
        const int xh = cb - r * g.xh;
        const int y = r % g.L[1];
        r /= g.L[1];
        const int z = r % g.L[2];
        const int t = r / g.L[2];
        const int x = 2 * xh + ((y + z + t + par) & 1);
        const int lex = 2 * cb + (x & 1);
        const double *src = links + ((int64_t)mu * 2 * vh + lex) * 18;
        int ps = 0;
        const int cc[4] = {x, y, z, t};
        for (int nu = 0; nu < mu; nu++) ps += cc[nu];
        double sg = (ps & 1) ? -1.0 : 1.0;
        if (g.antiperiodic_t && mu == 3 && t + 3 >= g.L[3]) sg = -sg;
        double p[8];
        if constexpr (GF == G_F64) {
            for (int k = 0; k < 4; k++) {
                const double2 v = reinterpret_cast<const double2 *>(stored + k * pstride)[li];
                p[2 * k] = v.x;
                p[2 * k + 1] = v.y;
            }
        } else if constexpr (GF == G_F32) {
            for (int k = 0; k < 2; k++) {
                const float4 v = reinterpret_cast<const float4 *>(stored + k * pstride)[li];
                p[4 * k] = v.x; p[4 * k + 1] = v.y; p[4 * k + 2] = v.z; p[4 * k + 3] = v.w;
            }
        } else if constexpr (GF == G_FIX16) {
            const int4 w = reinterpret_cast<const int4 *>(stored)[li];
            const int ws[4] = {w.x, w.y, w.z, w.w};
            for (int k = 0; k < 4; k++) {
                p[2 * k] = (double)(short)(ws[k] & 0xffff);
                p[2 * k + 1] = (double)(ws[k] >> 16);
            }
        } else {
            const int4 a = reinterpret_cast<const int4 *>(stored)[li], b = reinterpret_cast<const int4 *>(stored + pstride)[li];
            p[0] = a.x; p[1] = a.y; p[2] = a.z; p[3] = a.w; p[4] = b.x; p[5] = b.y; p[6] = b.z; p[7] = b.w;
        }
        const double t1 = p[0] * an, t2 = p[1] * an;
        const double a2r = p[2] * el, a2i = p[3] * el, a3r = p[4] * el, a3i = p[5] * el, b1r = p[6] * el, b1i = p[7] * el;
        const double N = a2r * a2r + a2i * a2i + a3r * a3r + a3i * a3i;
        const double ra = sqrt(fmax(1.0 - N, 0.0)), rc = sqrt(fmax(N - b1r * b1r - b1i * b1i, 0.0));
        double s1, c1, s2, c2;
        sincospi(t1, &s1, &c1);
        sincospi(t2, &s2, &c2);
        const double a1r = ra * c1, a1i = ra * s1, cr = rc * c2, ci = rc * s2;
        // b2 = -(conj(a1) a2 b1 + conj(a3) conj(c1)) / N, b3 = (conj(a2) conj(c1) - conj(a1) a3 b1) / N
        const double a1a2r = a1r * a2r + a1i * a2i, a1a2i = a1r * a2i - a1i * a2r;    // conj(a1) a2
        const double t3r = a1a2r * b1r - a1a2i * b1i, t3i = a1a2r * b1i + a1a2i * b1r;  // * b1
        const double t4r = a3r * cr - a3i * ci, t4i = -(a3r * ci + a3i * cr);           // conj(a3) conj(c1)
        const double b2r = -(t3r + t4r) / N, b2i = -(t3i + t4i) / N;
        const double t5r = a2r * cr - a2i * ci, t5i = -(a2r * ci + a2i * cr);           // conj(a2) conj(c1)
        const double a1a3r = a1r * a3r + a1i * a3i, a1a3i = a1r * a3i - a1i * a3r;      // conj(a1) a3
        const double t6r = a1a3r * b1r - a1a3i * b1i, t6i = a1a3r * b1i + a1a3i * b1r;  // * b1
        const double b3r = (t5r - t6r) / N, b3i = (t5i - t6i) / N;
        // c2 = conj(a3 b1 - a1 b3), c3 = conj(a1 b2 - a2 b1)
        const double c2r = (a3r * b1r - a3i * b1i) - (a1r * b3r - a1i * b3i);
        const double c2i = -((a3r * b1i + a3i * b1r) - (a1r * b3i + a1i * b3r));
        const double c3r = (a1r * b2r - a1i * b2i) - (a2r * b1r - a2i * b1i);
        const double c3i = -((a1r * b2i + a1i * b2r) - (a2r * b1i + a2i * b1r));
        const double V[18] = {a1r, a1i, a2r, a2i, a3r, a3i, b1r, b1i, b2r, b2i, b3r, b3i, cr, ci, c2r, c2i, c3r, c3i};
        for (int k = 0; k < 18; k++) {
            const double d = fabs(sg * V[k] - src[k]);
            m = (d > m || d != d) ? d : m;
            q += d * d;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const double o = __shfl_down_sync(0xffffffffu, m, off);
        m = (o > m || o != o) ? o : m;
        q += __shfl_down_sync(0xffffffffu, q, off);
    }
    if ((threadIdx.x & 31) == 0) {
        atomic_max_nonneg(out, m);
        atomicAdd(out + 1, q);
    }
}

int nblocks(int64_t n, int b) { return (int)((n + b - 1) / b); }

}  // namespace

void launch_pack_spinor(int sf, int64_t n, const double *in, char *out, int *bad, cudaStream_t s, int *host)
{
    if (n <= 0) return;
    const int nb = nblocks(n, kBlock);
    switch (sf) {
    case S_F64: pack_kernel<S_F64, double><<<nb, kBlock, 0, s>>>(n, in, out, bad, host); break;
    case S_F32: pack_kernel<S_F32, double><<<nb, kBlock, 0, s>>>(n, in, out, bad, host); break;
    case S_HALF: pack_kernel<S_HALF, double><<<nb, kBlock, 0, s>>>(n, in, out, bad, host); break;
    case S_INT20: pack_kernel<S_INT20, double><<<nb, kBlock, 0, s>>>(n, in, out, bad, host); break;
    case S_INT14: pack_kernel<S_INT14, double><<<nb, kBlock, 0, s>>>(n, in, out, bad, host); break;
    case S_INT30: pack_kernel<S_INT30, double><<<nb, kBlock, 0, s>>>(n, in, out, bad, host); break;
    default: break;
    }
}

void launch_pack_fields(int sf, int64_t n, const PackFields &f, cudaStream_t s)
{
    if (n <= 0 || f.nfields <= 0) return;
    const dim3 nb(nblocks(n, kBlock), f.nfields), b(kBlock);
    switch (sf) {
    case S_F64: launch_chained(pack_fields_kernel<S_F64>, nb, b, s, n, f); break;
    case S_F32: launch_chained(pack_fields_kernel<S_F32>, nb, b, s, n, f); break;
    case S_HALF: launch_chained(pack_fields_kernel<S_HALF>, nb, b, s, n, f); break;
    case S_INT20: launch_chained(pack_fields_kernel<S_INT20>, nb, b, s, n, f); break;
    case S_INT14: launch_chained(pack_fields_kernel<S_INT14>, nb, b, s, n, f); break;
    case S_INT30: launch_chained(pack_fields_kernel<S_INT30>, nb, b, s, n, f); break;
    default: break;
    }
}

void launch_pack32_spinor(int sf, int64_t n, const float *in, char *out, int *bad, cudaStream_t s, int *host)
{
    if (n <= 0) return;
    const int nb = nblocks(n, kBlock);
    switch (sf) {
    case S_F32: pack_kernel<S_F32, float><<<nb, kBlock, 0, s>>>(n, in, out, bad, host); break;
    case S_HALF: pack_kernel<S_HALF, float><<<nb, kBlock, 0, s>>>(n, in, out, bad, host); break;
    case S_INT20: pack_kernel<S_INT20, float><<<nb, kBlock, 0, s>>>(n, in, out, bad, host); break;
    case S_INT14: pack_kernel<S_INT14, float><<<nb, kBlock, 0, s>>>(n, in, out, bad, host); break;
    case S_INT30: pack_kernel<S_INT30, float><<<nb, kBlock, 0, s>>>(n, in, out, bad, host); break;
    default: break;
    }
}

void launch_pack_pair_int30(int64_t n, const float *in, char *out, int *bad, cudaStream_t s, int *host)
{
    if (n <= 0) return;
    pack_pair_kernel<<<nblocks(n, kBlock), kBlock, 0, s>>>(n, in, out, bad, host);
}

void launch_unpack_spinor(int sf, int cf, int64_t n, const char *in, double *out, cudaStream_t s)
{
    if (n <= 0) return;
    const int nb = nblocks(n, kBlock);
    const bool f64 = cf == HISQ_COMPUTE_F64;
    switch (sf) {
    case S_F64:
        if (f64) unpack_kernel<S_F64, double><<<nb, kBlock, 0, s>>>(n, in, out);
        else unpack_kernel<S_F64, float><<<nb, kBlock, 0, s>>>(n, in, out);
        break;
    case S_F32: unpack_kernel<S_F32, float><<<nb, kBlock, 0, s>>>(n, in, out); break;
    case S_HALF: unpack_kernel<S_HALF, float><<<nb, kBlock, 0, s>>>(n, in, out); break;
    case S_INT20: unpack_kernel<S_INT20, float><<<nb, kBlock, 0, s>>>(n, in, out); break;
    case S_INT14: unpack_kernel<S_INT14, float><<<nb, kBlock, 0, s>>>(n, in, out); break;
    case S_INT30:
        if (f64) unpack_kernel<S_INT30, double><<<nb, kBlock, 0, s>>>(n, in, out);
        else unpack_kernel<S_INT30, float><<<nb, kBlock, 0, s>>>(n, in, out);
        break;
    default: break;
    }
}

void launch_gauge_scan(const Geom &g, bool lng, const double *links, double *copy, unsigned long long *out,
                       cudaStream_t s)
{
    const int nb = nblocks(8LL * g.vh, kLinkBlock);
    if (lng && copy)
        gauge_scan_kernel<true, true><<<nb, kLinkBlock, 0, s>>>(g, links, copy, out);
    else if (lng)
        gauge_scan_kernel<true, false><<<nb, kLinkBlock, 0, s>>>(g, links, copy, out);
    else if (copy)
        gauge_scan_kernel<false, true><<<nb, kLinkBlock, 0, s>>>(g, links, copy, out);
    else
        gauge_scan_kernel<false, false><<<nb, kLinkBlock, 0, s>>>(g, links, copy, out);
}

void launch_r8_check(const Geom &g, int gf, const double *links, const char *stored, double el, double an,
                     double *out, cudaStream_t s)
{
    const int nb = (int)std::min<int64_t>(nblocks(8LL * g.vh, kBlock), 4096);
    switch (gf) {
    case G_F64: r8_check_kernel<G_F64><<<nb, kBlock, 0, s>>>(g, links, stored, el, an, out); break;
    case G_F32: r8_check_kernel<G_F32><<<nb, kBlock, 0, s>>>(g, links, stored, el, an, out); break;
    case G_FIX16: r8_check_kernel<G_FIX16><<<nb, kBlock, 0, s>>>(g, links, stored, el, an, out); break;
    case G_FIX32: r8_check_kernel<G_FIX32><<<nb, kBlock, 0, s>>>(g, links, stored, el, an, out); break;
    }
}

void launch_quantise_links(const Geom &g, int gf, int recon, const double *links, double inv, char *out,
                           cudaStream_t s)
{
    const int nb = nblocks(8LL * g.vh, kLinkBlock);
#define Q(GF, R) quantise_kernel<GF, R><<<nb, kLinkBlock, 0, s>>>(g, links, inv, out)
    if (recon == 18) {
        switch (gf) {
        case G_F64: Q(G_F64, 18); break;
        case G_F32: Q(G_F32, 18); break;
        case G_FIX16: Q(G_FIX16, 18); break;
        case G_FIX32: Q(G_FIX32, 18); break;
        case G_SE15: Q(G_SE15, 18); break;
        }
    } else if (recon == 8) {
        switch (gf) {
        case G_F64: Q(G_F64, 8); break;
        case G_F32: Q(G_F32, 8); break;
        case G_FIX16: Q(G_FIX16, 8); break;
        case G_FIX32: Q(G_FIX32, 8); break;
        }
    } else if (recon == 13) {
        switch (gf) {
        case G_F64: Q(G_F64, 13); break;
        case G_F32: Q(G_F32, 13); break;
        case G_FIX16: Q(G_FIX16, 13); break;
        case G_FIX32: Q(G_FIX32, 13); break;
        }
    } else {
        switch (gf) {
        case G_F64: Q(G_F64, 12); break;
        case G_F32: Q(G_F32, 12); break;
        case G_FIX16: Q(G_FIX16, 12); break;
        case G_FIX32: Q(G_FIX32, 12); break;
        case G_SE15: Q(G_SE15, 12); break;
        }
    }
#undef Q
}

}  // namespace hisq
