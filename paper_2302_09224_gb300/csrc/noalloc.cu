// noalloc.cu -- hisq_dslash_noalloc: the stencil entry point for callers that
// must not allocate device memory.  Its scratch (the input and xpay fields in
// the storage format) is one file-scope device array sized for at most HISQ_NOALLOC_MAX_SITES sites per parity;
// every GPU that loads the library holds it until the process exits.
#include <cuda_runtime.h>

#include <mutex>

#include "internal.h"

namespace hisq {

namespace {

constexpr int64_t kMaxSites = HISQ_NOALLOC_MAX_SITES;
constexpr size_t kFieldBytes = (size_t)48 * 2 * kMaxSites;  // one full-lattice field, widest format
constexpr size_t kScratchBytes = 2 * kFieldBytes;

static __device__ __align__(256) unsigned char noalloc_scratch[kScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex addr_mu;
char *addr_of[kMaxDevices] = {};

// Device address of the scratch array for the current device, looked up once
// per device (host code only holds a stand-in for the symbol).
hisq_status scratch_address(hisq_ctx *c, char **out)
{
    if (c->device < 0 || c->device >= kMaxDevices) return fail(c, HISQ_EINVAL, "device index out of range");
    std::lock_guard<std::mutex> lk(addr_mu);
    if (!addr_of[c->device]) {
        void *p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, noalloc_scratch);
        if (e != cudaSuccess || !p) return cuda_fail(c, e, "cudaGetSymbolAddress(noalloc scratch)");
        addr_of[c->device] = static_cast<char *>(p);
    }
    *out = addr_of[c->device];
    return HISQ_OK;
}

}  // namespace

}  // namespace hisq

using namespace hisq;

extern "C" hisq_status hisq_dslash_noalloc(hisq_ctx *c, const hisq_gauge *g, hisq_prec prec, int out_parity,
                                           double a, const double *xpay_in, const double *in, double *out,
                                           void *stream)
{
    if (!c || !g || !in || !out) return fail(c, HISQ_EINVAL, "hisq_dslash_noalloc: null argument");
    if (out_parity < 0 || out_parity > 2) return fail(c, HISQ_EINVAL, "out_parity must be 0, 1 or 2");
    const bool xpay = a != 0.0;
    if (xpay && !xpay_in) return fail(c, HISQ_EINVAL, "xpay_in is required when a != 0");
    const int64_t vh = g->geom.vh;
    if (vh > kMaxSites)
        return fail(c, HISQ_EINVAL, "hisq_dslash_noalloc: %lld sites per parity exceed its fixed scratch (%lld)",
                    (long long)vh, (long long)kMaxSites);
    if (c->device < 0 || c->device >= kMaxDevices) return fail(c, HISQ_EINVAL, "device index out of range");
    cudaError_t e = cudaSetDevice(c->device);
    if (e != cudaSuccess) return cuda_fail(c, e, "hisq_dslash_noalloc: cudaSetDevice");
    cudaStream_t s = pick_stream(c, stream);
    // the synchronisation below cannot be captured
    if (stream_capturing(s))
        return fail(c, HISQ_EINVAL, "hisq_dslash_noalloc cannot be called while its stream is being captured");
    GaugeView gv{};
    hisq_status st = gauge_view_existing(c, g, prec, &gv);
    if (st) return st;
    char *sc = nullptr;
    st = scratch_address(c, &sc);
    if (st) return st;
    StencilCall call{g, gv, prec, out_parity, a, xpay ? xpay_in : nullptr, in, out, sc, sc + kFieldBytes, nullptr};
    return run_stencil_call(c, call, nullptr, s, "hisq_dslash_noalloc");
}
