// Dispatch from a runtime precision triplet to the compiled stencil kernels,
// and the launch-shape tuner: the first time a (triplet, lattice) pair is
// prepared outside graph capture every launch shape is timed on the device and
// the fastest is kept for the rest of the process.
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <atomic>
#include <map>
#include <mutex>

#include "dslash.cuh"
#include "internal.h"

namespace hisq {

bool launch_dslash_f64(int, bool, int, const DslashArgs &, cudaStream_t);
bool launch_dslash_f32(int, bool, int, const DslashArgs &, cudaStream_t);
bool launch_dslash_half(int, bool, int, const DslashArgs &, cudaStream_t);
bool launch_dslash_int20(int, bool, int, const DslashArgs &, cudaStream_t);
bool launch_dslash_int14(int, bool, int, const DslashArgs &, cudaStream_t);
bool launch_dslash_int20se(int, bool, int, const DslashArgs &, cudaStream_t);
bool launch_dslash_int30d(int, bool, int, const DslashArgs &, cudaStream_t);
bool launch_dslash_int30f(int, bool, int, const DslashArgs &, cudaStream_t);

bool launch_mee_f32(int, int, const MeeArgs &, cudaStream_t);
bool launch_mee_half(int, int, const MeeArgs &, cudaStream_t);
bool launch_mee_int20(int, int, const MeeArgs &, cudaStream_t);
bool launch_mee_int30f(int, int, const MeeArgs &, cudaStream_t);

std::atomic<int> fused_mode{0};

bool mee_fused_asked() { return fused_mode.load() != 0; }

bool mee_fused_available(int gf, int sf, int cf, const Geom &g)
{
    if (cf != HISQ_COMPUTE_F32 || g.L[3] > kMaxFusedLt || fused_mode.load() == 0) return false;
    return (gf == G_F32 && sf == S_F32) || (gf == G_FIX16 && (sf == S_HALF || sf == S_INT20)) ||
           (gf == G_FIX32 && sf == S_INT30);
}

extern std::atomic<int> fused_lag, fused_bps;
extern std::atomic<unsigned> fused_wait_polls, fused_wait_extra;
extern std::atomic<bool> resident_refused;

bool launch_mee_fused(int gf, int sf, int cf, int long_recon, const MeeArgs &m_in, cudaStream_t s)
{
    if (!mee_fused_available(gf, sf, cf, m_in.d1.g) || m_in.d2.red.sync == nullptr) return false;
    MeeArgs m = m_in;
    m.lag = fused_lag.load();
    m.blocks_per_sm = fused_bps.load();
    m.wait_polls = fused_wait_polls.load();
    m.wait_extra = fused_wait_extra.load();
    const int cfg = 4;
    if (gf == G_F32) return launch_mee_f32(long_recon, cfg, m, s);
    if (sf == S_HALF) return launch_mee_half(long_recon, cfg, m, s);
    if (sf == S_INT20) return launch_mee_int20(long_recon, cfg, m, s);
    return launch_mee_int30f(long_recon, cfg, m, s);
}

namespace {

bool launch_with(int gf, int sf, int cf, int lrec, bool red, int cfg, const DslashArgs &a, cudaStream_t s)
{
    const bool f64 = cf == HISQ_COMPUTE_F64;
    if (gf == G_F64 && sf == S_F64 && f64) return launch_dslash_f64(lrec, red, cfg, a, s);
    if (gf == G_F32 && sf == S_F32 && !f64) return launch_dslash_f32(lrec, red, cfg, a, s);
    if (gf == G_FIX16 && sf == S_HALF && !f64) return launch_dslash_half(lrec, red, cfg, a, s);
    if (gf == G_FIX16 && sf == S_INT20 && !f64) return launch_dslash_int20(lrec, red, cfg, a, s);
    if (gf == G_FIX16 && sf == S_INT14 && !f64) return launch_dslash_int14(lrec, red, cfg, a, s);
    if (gf == G_SE15 && sf == S_INT20 && !f64) return launch_dslash_int20se(lrec, red, cfg, a, s);
    if (gf == G_FIX32 && sf == S_INT30) {
        if (f64) return launch_dslash_int30d(lrec, red, cfg, a, s);
        return launch_dslash_int30f(lrec, red, cfg, a, s);
    }
    return false;
}

using TuneKey = std::array<int, 9>;
std::mutex tune_mu;
std::map<TuneKey, int> tune_cache;

TuneKey key_of(int gf, int sf, int cf, int lrec, bool red, const Geom &g)
{
    return {gf, sf, cf, lrec, red ? 1 : 0, g.L[0], g.L[1], g.L[2], g.L[3]};
}

}  // namespace

std::atomic<int> forced_config{-1};
std::atomic<int> forced_config_red{-1};

namespace {

int forced_for(bool red)
{
    const int fr = forced_config_red.load();
    return red && fr >= 0 ? fr : forced_config.load();
}

}  // namespace

int stencil_config(int gf, int sf, int cf, int lrec, bool red, const Geom &g)
{
    const int f = forced_for(red);
    if (f >= 0 && stencil_config_valid(f, gf)) return f;
    std::lock_guard<std::mutex> lk(tune_mu);
    auto it = tune_cache.find(key_of(gf, sf, cf, lrec, red, g));
    return it == tune_cache.end() ? 0 : it->second;
}

int stencil_config_in_use(int gf, int sf, int cf, int lrec, bool red, const Geom &g)
{
    const int f = forced_for(red);
    if (f >= 0 && stencil_config_valid(f, gf)) return f;
    std::lock_guard<std::mutex> lk(tune_mu);
    auto it = tune_cache.find(key_of(gf, sf, cf, lrec, red, g));
    return it == tune_cache.end() ? -1 : it->second;
}

bool launch_dslash(int gf, int sf, int cf, int long_recon, bool reduce, const DslashArgs &a, cudaStream_t s)
{
    return launch_with(gf, sf, cf, long_recon, reduce, stencil_config(gf, sf, cf, long_recon, reduce, a.g), a, s);
}

namespace {

// Times every launch shape of one kernel variant; the reducing variant (whose
// register budget differs) is timed as the solvers use it, with xpay and both
// sums, and with no finisher.
void tune_variant(int gf, int sf, int cf, int lrec, bool red, const DslashArgs &args, cudaStream_t s)
{
    if (const int f = forced_for(red); f >= 0 && stencil_config_valid(f, gf)) return;  // shape fixed by the caller
    const TuneKey key = key_of(gf, sf, cf, lrec, red, args.g);
    {
        std::lock_guard<std::mutex> lk(tune_mu);
        if (tune_cache.count(key)) return;
    }
    DslashArgs a = args;
    a.fin = FIN_NONE;
    a.active = nullptr;
    if (gf == G_F64 && !red) {
        // the shapes serve the passes with a thread a site: none on lattices where both the pass over one parity
        // and the one over both share a site among lanes
        if (dslash_f64_lanes(args.g.vh) > 1 && dslash_f64_lanes(2LL * args.g.vh) > 1) return;
        a.one_lane = 1;
    }
    if (red) {
        a.xpay = 1;
        a.y = a.out;
        a.a = 1.0;
    }
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return;
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return;
    }
    float ms_of[kNumStencilConfigs];
    auto time_shape = [&](int cfg, int reps) {
        cudaEventRecord(e0, s);
        for (int r = 0; r < reps; r++) launch_with(gf, sf, cf, lrec, red, cfg, a, s);
        cudaEventRecord(e1, s);
        float ms = 0.f;
        return cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess ? ms / reps
                                                                                                           : 1e30f;
    };
    int best = 0, second = -1;
    for (int cfg = 0; cfg < kNumStencilConfigs; cfg++) {
        ms_of[cfg] = 1e30f;
        if (!stencil_config_valid(cfg, gf)) continue;
        launch_with(gf, sf, cf, lrec, red, cfg, a, s);  // warm
        ms_of[cfg] = time_shape(cfg, 3);
        if (ms_of[cfg] < ms_of[best]) {
            second = best;
            best = cfg;
        } else if (cfg != best && (second < 0 || ms_of[cfg] < ms_of[second])) {
            second = cfg;
        }
    }
    // three passes of 10 us are noisy: the two fastest are timed again, in turn (16^3x32 solves differed by
    // up to 13 % between processes by the shape picked).  From 40 us a pass on the first look decides: 16 more
    // passes would cost a first call more than they tell it (FP64 16^3x32: 6.5 ms against 4.1 without).
    if (second >= 0 && ms_of[best] < 0.04f && ms_of[second] < 1.15f * ms_of[best]) {
        float b2 = 1e30f, s2 = 1e30f;
        for (int r = 0; r < 2; r++) {
            b2 = std::min(b2, time_shape(best, 4));
            s2 = std::min(s2, time_shape(second, 4));
        }
        if (s2 < b2) best = second;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    (void)cudaGetLastError();
    // first result wins: a thread that tuned the same pair concurrently keeps
    // the shape already in use, so every launch after the first insertion of a
    // key (and hence every block-sum order) is the same for the whole process
    std::lock_guard<std::mutex> lk(tune_mu);
    tune_cache.emplace(key, best);
}

}  // namespace

void tune_dslash(int gf, int sf, int cf, int lrec, const DslashArgs &args, cudaStream_t s)
{
    tune_variant(gf, sf, cf, lrec, false, args, s);
    if (args.red.partials != nullptr && args.red.counter != nullptr) tune_variant(gf, sf, cf, lrec, true, args, s);
}

}  // namespace hisq

namespace hisq {

bool launch_mrhs_f32(int, bool, int, int, const DslashMArgs &, cudaStream_t);
bool launch_mrhs_half(int, bool, int, int, const DslashMArgs &, cudaStream_t);
bool launch_mrhs_int20(int, bool, int, int, const DslashMArgs &, cudaStream_t);

bool launch_dslash_mrhs(int gf, int sf, int cf, int long_recon, bool reduce, int T, int variant, const DslashMArgs &a,
                        cudaStream_t s)
{
    if (T != 1 && T != 2 && T != 4 && T != 8 && T != 16) return false;
    if (a.nrhs < 1 || a.nrhs > kMaxRHS || a.nrhs % T) return false;
    if (cf != HISQ_COMPUTE_F32) return false;
    if (gf == G_F32 && sf == S_F32) return launch_mrhs_f32(long_recon, reduce, T, variant, a, s);
    if (gf == G_FIX16 && sf == S_HALF) return launch_mrhs_half(long_recon, reduce, T, variant, a, s);
    if (gf == G_FIX16 && sf == S_INT20) return launch_mrhs_int20(long_recon, reduce, T, variant, a, s);
    return false;
}

}  // namespace hisq

namespace hisq {

bool launch_cg_block_f32(int, const CGBlockShape &, const CGBlockArgs &, cudaStream_t);
bool launch_cg_block_half(int, const CGBlockShape &, const CGBlockArgs &, cudaStream_t);
bool launch_cg_block_int20(int, const CGBlockShape &, const CGBlockArgs &, cudaStream_t);

// The most lanes a site (4, 2 or 1) with at most 512 threads on each SM (128
// registers a thread: no spills), else one lane and up to 1024 threads while
// the links of both passes take at most 200 MB (FP32 ones beyond that, 252 MB at
// 16^3x64 to 276 MB at 20^3x36, measured 54 to 66 us against 57 to 61 for the
// separate kernels, no clear gain), spread over every SM.  Per iteration, here
// against the separate kernels, 20-bit: 8^4 9.8 us against 22, 12^4 12.0 / 21.6,
// 16^4 15.2 / 24.4, 16^3x32 20.4 / 32.2, 16^3x64 33.8 / 47.5, 20^3x36 38.9 /
// 47.5; FP32: 16^3x32 17.7 / 32.3.  Two lanes on 864 threads (64 registers)
// lost to one lane on 431: 24.7 against 22.9 us on 16^3x32, in an earlier form.
CGBlockShape cg_block_shape(int gf, int sf, int cf, int long_recon, int vh)
{
    const bool has = cf == HISQ_COMPUTE_F32 && (long_recon == 12 || long_recon == 18) &&
                     ((gf == G_F32 && sf == S_F32) || (gf == G_FIX16 && (sf == S_HALF || sf == S_INT20)));
    static const int sms = [] {
        int dev = 0, n = 0, coop = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
        return coop ? n : 0;
    }();
    for (int lanes = 4; has && lanes >= 1; lanes /= 2) {
        const long long all = (long long)vh * lanes;
        if (all > (long long)sms * (lanes > 1 ? 512 : 1024)) continue;
        if (all > (long long)sms * 512 && 16LL * vh * (link_bytes(gf, 18) + link_bytes(gf, long_recon)) > 200000000LL)
            continue;
        const int per = (int)((all + sms - 1) / sms);
        const int threads = per <= 64 ? 64 : (per + 31) / 32 * 32;
        return {lanes, threads, (int)((all + threads - 1) / threads)};
    }
    return {0, 0, 0};
}

bool launch_cg_block(int gf, int sf, int long_recon, const CGBlockShape &sh, const CGBlockArgs &args, cudaStream_t s)
{
    CGBlockArgs a = args;
    a.wait_polls = std::min(fused_wait_polls.load(), 1u << 20);  // about half a second of L2 round trips
    a.wait_extra = fused_wait_extra.load();
    if (resident_refused.load()) return false;
    if (gf == G_F32) return launch_cg_block_f32(long_recon, sh, a, s);
    if (sf == S_HALF) return launch_cg_block_half(long_recon, sh, a, s);
    return launch_cg_block_int20(long_recon, sh, a, s);
}

}  // namespace hisq

extern "C" int hisq_stencil_config_reduce(int cfg)
{
    if (cfg < -1 || cfg >= hisq::kNumStencilConfigs) return -2;
    return hisq::forced_config_red.exchange(cfg);
}

extern "C" int hisq_stencil_config_in_use(const hisq_gauge *g, hisq_prec p, int reduce)
{
    if (!g) return -1;
    return hisq::stencil_config_in_use(p.gauge, p.spinor, p.compute, p.long_recon, reduce != 0, g->geom);
}

extern "C" int hisq_mee_fused(int mode)
{
    if (mode < 0 || mode > 1) return -2;
    return hisq::fused_mode.exchange(mode);
}

namespace hisq {
std::atomic<int> fused_lag{4}, fused_bps{0};
std::atomic<unsigned> fused_wait_polls{kMeeWaitPolls}, fused_wait_extra{0};
std::atomic<bool> resident_refused{false};
}

extern "C" void hisq_mee_fused_wait_test(unsigned polls, int unreachable)
{
    hisq::fused_wait_polls.store(polls > 0 ? polls : hisq::kMeeWaitPolls);
    hisq::fused_wait_extra.store(unreachable && unreachable != 2 ? 1u : 0u);
    hisq::resident_refused.store(unreachable == 2);
}

extern "C" void hisq_mee_fused_shape(int lag, int blocks_per_sm)
{
    if (lag >= 0) hisq::fused_lag.store(lag);
    if (blocks_per_sm >= 0) hisq::fused_bps.store(blocks_per_sm);
}

namespace hisq {
std::atomic<int> pdl_mode{1};
}

extern "C" int hisq_programmatic_launch(int mode)
{
    if (mode < 0 || mode > 1) return -2;
    return hisq::pdl_mode.exchange(mode);
}

namespace hisq {
std::atomic<int> split_mode{1};
}

extern "C" int hisq_cg_split_scalars(int mode)
{
    if (mode < 0 || mode > 1) return -2;
    return hisq::split_mode.exchange(mode);
}

extern "C" int hisq_stencil_config(int cfg)
{
    if (cfg < -1 || cfg >= hisq::kNumStencilConfigs) return -2;
    return hisq::forced_config.exchange(cfg);
}
