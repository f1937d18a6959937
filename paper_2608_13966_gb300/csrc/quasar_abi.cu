// C ABI of the QUASAR reconstruction library: argument validation, kernel
// selection and launch configuration.  Declarations and contracts are in
// include/quasar.h.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include "params.h"
#include "quasar.h"

namespace quasar {
// integer-code kernels: one entry per (one chunk of 8 candidates, or more;
// clamp-set size)
#define QUASAR_INT_ENTRY(n, s) const void* int_kernel_nch##n##_ss##s(int epl, bool batch, bool adam, bool var);
QUASAR_INT_ENTRY(1, 8) QUASAR_INT_ENTRY(1, 4) QUASAR_INT_ENTRY(1, 3) QUASAR_INT_ENTRY(1, 2)
QUASAR_INT_ENTRY(1, 1)
QUASAR_INT_ENTRY(2, 4) QUASAR_INT_ENTRY(2, 2) QUASAR_INT_ENTRY(2, 1)
#undef QUASAR_INT_ENTRY
const void* nvfp4_kernel(bool batch);
const void* nvfp4_amax_ahead_kernel();
const void* nvfp4_adamw_ahead_kernel();
const void* amax_kernel(bool batch);
const void* amax_init_kernel(bool batch);
const void* amax_to_scale_kernel(bool batch);
const void* lut_kernel();
const void* adamw_amax_kernel();
const void* sym_kernel_ss8(int epl);
const void* sym_kernel_ss4(int epl);
const void* sym_kernel_ss3(int epl);
const void* sym_kernel_ss2(int epl);
const void* sym_kernel_ss1(int epl);
}  // namespace quasar

// Per-device status word (bit 0: a kernel timed out on a wait).
__device__ unsigned int g_quasar_status_word;

namespace {

using namespace quasar;

// Threads of the CTAs of the absmax and AdamW passes alone.
constexpr int kThreads = 256;
constexpr uint64_t kDefaultTimeoutNs = 1000000000ull;  // 1 s per wait

std::atomic<int64_t> g_force_timeout_ns{0};
std::atomic<unsigned int*> g_stats{nullptr};
std::atomic<int> g_hoist{-1};  // -1: the environment's choice (tuning().hoist)

// The error bounds' defaults are the smallest values their derivations allow
// (the summation-depth bound of the candidate errors, the NVFP4 direct-sum
// bound, the fit error that triggers the compensated fit): an environment
// value below one is raised to it, so a setting can make the careful paths
// run more often but never skip one that correctness needs.  Larger values
// are capped where a float overflow would start to matter.
constexpr float kTieKappaMin = 16.0f;
constexpr float kTieScaleMin = 1.0f;
constexpr float kFitUlpsMin = 8.0f;

struct Tuning {
    int stages = 0;            // 0: each kernel's choice
    float tie_kappa = kTieKappaMin;  // NVFP4 tie bound, in ulps
    float tie_scale = kTieScaleMin;  // multiplier of the integer kernel's summation-depth bound
    float fit_ulps = kFitUlpsMin;
    int hoist = 1;             // 0: the integer kernel's code-clamp sets hold one candidate
};

// A float from the environment, clamped to [lo, hi] (non-numbers give lo).
float env_float(const char* s, float lo, float hi)
{
    const double x = std::atof(s);
    return !(x >= lo) ? lo : (x > hi ? hi : (float)x);
}

const Tuning& tuning()
{
    static const Tuning t = [] {
        Tuning x;
        if (const char* s = std::getenv("QUASAR_STAGES")) x.stages = std::min(std::max(std::atoi(s), 0), 8);
        if (const char* s = std::getenv("QUASAR_TIE_KAPPA")) x.tie_kappa = env_float(s, kTieKappaMin, 1e4f);
        if (const char* s = std::getenv("QUASAR_TIE_SCALE")) x.tie_scale = env_float(s, kTieScaleMin, 1e3f);
        if (const char* s = std::getenv("QUASAR_FIT_ULPS")) x.fit_ulps = env_float(s, kFitUlpsMin, 1e4f);
        if (const char* s = std::getenv("QUASAR_HOIST")) x.hoist = std::atoi(s);
        return x;
    }();
    return t;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

bool overlaps(const void* a, size_t na, const void* b, size_t nb)
{
    if (!a || !b || na == 0 || nb == 0) return false;
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return x < y + nb && y < x + na;
}

size_t dtype_size(quasar_dtype d) { return d == QUASAR_BF16 ? 2 : 4; }

bool valid_dtype(quasar_dtype d) { return d == QUASAR_F32 || d == QUASAR_BF16; }

// Checks shared by both reconstruction entry points.  On success fills n.
quasar_status check_common(const float* w, const void* g, quasar_dtype g_dtype, const float* v,
                           float beta2, const float* clip, int n_clip, int64_t rows, int64_t cols,
                           const void* r, quasar_dtype r_dtype, int64_t* n)
{
    if (rows < 0 || cols < 0) return QUASAR_ERR_INVALID_ARG;
    if (rows != 0 && cols > (int64_t(1) << 62) / rows) return QUASAR_ERR_INVALID_ARG;
    *n = rows * cols;
    if (!(beta2 >= 0.0f && beta2 < 1.0f)) return QUASAR_ERR_INVALID_ARG;
    if (!clip || n_clip < 1 || n_clip > kMaxClip) return QUASAR_ERR_INVALID_ARG;
    for (int k = 0; k < n_clip; ++k)
        if (!(clip[k] > 0.0f && clip[k] <= 1.0f)) return QUASAR_ERR_INVALID_ARG;
    if (!valid_dtype(r_dtype) || (g && !valid_dtype(g_dtype))) return QUASAR_ERR_INVALID_ARG;
    if (*n == 0) return QUASAR_OK;
    if (!w || !v || !r) return QUASAR_ERR_INVALID_ARG;
    if (!aligned16(w) || !aligned16(v) || !aligned16(r) || (g && !aligned16(g)))
        return QUASAR_ERR_INVALID_ARG;
    return QUASAR_OK;
}

// Output byte ranges must not overlap w, g or v.
bool outputs_alias_inputs(const float* w, const void* g, quasar_dtype g_dtype, const float* v,
                          int64_t n, const void* const* outs, const size_t* out_bytes, int n_out)
{
    const size_t nb = (size_t)n;
    for (int i = 0; i < n_out; ++i) {
        if (overlaps(outs[i], out_bytes[i], w, nb * 4)) return true;
        if (overlaps(outs[i], out_bytes[i], v, nb * 4)) return true;
        if (g && overlaps(outs[i], out_bytes[i], g, nb * dtype_size(g_dtype))) return true;
    }
    return false;
}

void fill_clip(const float* clip, int n_clip, float* f, float* invf)
{
    for (int k = 0; k < kMaxClip; ++k) {
        const float fk = clip[std::min(k, n_clip - 1)];
        f[k] = fk;
        invf[k] = (float)(1.0 / (double)fk);
    }
}

// Code clamps of the integer kernels.  A set of consecutive candidate slots
// shares one clamp of |w - centre| (asymmetric) or |w| (symmetric codes) when
// the capped value has the largest code for every factor of the set and no
// value below the cap exceeds it.  Asymmetric, J = (qmax - 1) / 2: some tau
// with J f_max (1 + 1e-3) <= tau <= (J + 1) f_min (1 - 1e-3); then
// min(|d|, tau range / qmax) P_k has the code min(floor(|d| P_k), J) for every
// slot k of the set (a capped |d| gives cap P_k ~ tau / f_k in [J, J + 1), and
// below the cap |d| P_k < J + 1).  Symmetric, codes rounded to at most Q: the
// same with Q - 1/2 and Q + 1/2 for J and J + 1, and the cap tau amax / Q.  The
// margin covers the fp32 roundings of the cap, of R and of P.  The largest set
// size of 8, 4, 3, 2, 1 whose sets all qualify is taken (a set of one always
// does), and no larger than max_size; every slot holds its set's tau / qmax (or
// tau / Q).  Also the centre factor of each 8-candidate chunk.
void fill_caps(IntParams* p, int max_size, bool sets_8_3 = false, bool symmetric = false)
{
    const int J = p->qmax >> 1;
    const int Q = (p->qmax - 1) >> 1;
    const double below = symmetric ? Q - 0.5 : J, above = symmetric ? Q + 0.5 : J + 1;
    // the sets of a size: consecutive runs of `size` slots; 3: the runs 3, 3,
    // 2 of every 8 slots (3 and 8: only where the kernel is built for them)
    auto first_of = [](int size, int k) { return size == 3 ? 8 * (k / 8) + 3 * ((k % 8) / 3) : k - k % size; };
    auto len_of = [](int size, int k0) { return size == 3 ? (k0 % 8 == 6 ? 2 : 3) : size; };
    auto cap_of = [&](int k0, int n, double* tau) {
        double fmax = 0.0, fmin = 2.0;
        for (int k = k0; k < k0 + n; ++k) {
            fmax = std::max(fmax, (double)p->f[k]);
            fmin = std::min(fmin, (double)p->f[k]);
        }
        const double lo = below * fmax * (1.0 + 1e-3), hi = above * fmin * (1.0 - 1e-3);
        *tau = 0.5 * (lo + hi);
        return lo < hi;
    };
    int size = 1;
    for (int cand : {8, 4, 3, 2}) {
        if ((cand == 3 || cand == 8) ? (!sets_8_3 || max_size < 4) : cand > max_size) continue;
        bool ok = true;
        double tau;
        for (int k0 = 0; k0 < kMaxClip && ok; k0 += len_of(cand, k0)) ok = cap_of(k0, len_of(cand, k0), &tau);
        if (ok) {
            size = cand;
            break;
        }
    }
    p->set_size = size;
    for (int k = 0; k < kMaxClip; ++k) {
        const int k0 = first_of(size, k);
        double tau = 0.0;
        cap_of(k0, len_of(size, k0), &tau);
        p->cap[k] = (float)(tau / (symmetric ? Q : p->qmax));
    }
    for (int c = 0; c < kMaxClip / 8; ++c) {
        double lo = 1e300, hi = 0.0;
        for (int k = 8 * c; k < 8 * c + 8 && k < std::max(p->n_clip, 8 * c + 1); ++k) {
            lo = std::min(lo, 1.0 / (double)p->f[k]);
            hi = std::max(hi, 1.0 / (double)p->f[k]);
        }
        p->invfc[c] = (float)(0.5 * (lo + hi));
    }
}

struct Launch {
    int stages;
    uint32_t stage_bytes;
    size_t smem;
};

// Per-device facts looked up once: SM count and the status word's address.
constexpr int kMaxDevices = 64;
struct DeviceInfo {
    std::atomic<int> ready{0};
    int nsm = 0;
    unsigned int* status = nullptr;
};
DeviceInfo g_dev[kMaxDevices];
std::mutex g_mu;

// Launch configuration of one kernel at one shared-memory size and block size, per device.
struct KernelConfig {
    const void* fn = nullptr;
    size_t smem = 0;
    int threads = 0;
    int dev = -1;
    int occupancy = 0;
};
constexpr int kMaxConfigs = 256;
KernelConfig g_cfg[kMaxConfigs];
int g_ncfg = 0;
// Kernels whose dynamic shared-memory limit was raised, per device.  The
// limit is always set to the device's opt-in maximum, so it never has to be
// raised again or lowered for another size (a full table only repeats the
// same setting).
struct SmemLimit {
    const void* fn = nullptr;
    int dev = -1;
};
constexpr int kMaxLimits = 256;
SmemLimit g_limit[kMaxLimits];
int g_nlimit = 0;

quasar_status device_info(int* dev_out, const DeviceInfo** info)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return QUASAR_ERR_CUDA;
    if (dev < 0 || dev >= kMaxDevices) return QUASAR_ERR_UNSUPPORTED;
    DeviceInfo& d = g_dev[dev];
    if (!d.ready.load(std::memory_order_acquire)) {
        std::lock_guard<std::mutex> lock(g_mu);
        if (!d.ready.load(std::memory_order_relaxed)) {
            void* ptr = nullptr;
            if (cudaDeviceGetAttribute(&d.nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
                return QUASAR_ERR_CUDA;
            if (cudaGetSymbolAddress(&ptr, g_quasar_status_word) != cudaSuccess)
                return QUASAR_ERR_CUDA;
            d.status = static_cast<unsigned int*>(ptr);
            d.ready.store(1, std::memory_order_release);
        }
    }
    *dev_out = dev;
    *info = &d;
    return QUASAR_OK;
}

quasar_status status_ptr(unsigned int** p)
{
    int dev;
    const DeviceInfo* info;
    const quasar_status st = device_info(&dev, &info);
    if (st != QUASAR_OK) return st;
    *p = info->status;
    return QUASAR_OK;
}

// Resident CTAs per SM for (fn, smem) on device dev.  The kernel's dynamic
// shared-memory limit is set once per device, to the device's opt-in
// maximum, so every configuration cached earlier stays launchable.
quasar_status occupancy(const void* fn, size_t smem, int threads, int dev, int* occ)
{
    std::lock_guard<std::mutex> lock(g_mu);
    for (int i = 0; i < g_ncfg; ++i)
        if (g_cfg[i].fn == fn && g_cfg[i].dev == dev && g_cfg[i].smem == smem && g_cfg[i].threads == threads) {
            *occ = g_cfg[i].occupancy;
            return QUASAR_OK;
        }
    bool raised = false;
    for (int i = 0; i < g_nlimit && !raised; ++i) raised = g_limit[i].fn == fn && g_limit[i].dev == dev;
    if (!raised) {
        int optin = 0;
        if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
            return QUASAR_ERR_CUDA;
        if (smem > (size_t)optin) return QUASAR_ERR_UNSUPPORTED;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin) != cudaSuccess)
            return QUASAR_ERR_CUDA;
        if (g_nlimit < kMaxLimits) g_limit[g_nlimit++] = SmemLimit{fn, dev};
    }
    int o = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, fn, threads, smem) != cudaSuccess)
        return QUASAR_ERR_CUDA;
    if (g_ncfg < kMaxConfigs) g_cfg[g_ncfg++] = KernelConfig{fn, smem, threads, dev, o};
    *occ = o;
    return QUASAR_OK;
}

// Persistent launch: at most (#SMs x resident CTAs) CTAs of `warps` warps, and
// no more than there are units of work: a launch with fewer units than warps
// spreads them over the SMs (the kernels give a CTA's first warp the first of
// its units) instead of filling a few CTAs, whose warps would share a
// scheduler.
// extra_warps: warps a CTA has beside those (a fused pass of its own, which takes
// every resident CTA); extra: that pass's parameters, the kernel's second.
quasar_status launch_persistent(const void* fn, void* params, size_t smem, int64_t n_units,
                                cudaStream_t stream, int warps, void* extra = nullptr,
                                int extra_warps = 0)
{
    int dev = 0, occ = 0;
    const DeviceInfo* info = nullptr;
    quasar_status st = device_info(&dev, &info);
    if (st != QUASAR_OK) return st;
    const int threads = (warps + extra_warps) * 32;
    if ((st = occupancy(fn, smem, threads, dev, &occ)) != QUASAR_OK) return st;
    if (occ < 1) return QUASAR_ERR_UNSUPPORTED;
    const int64_t all = (int64_t)info->nsm * occ;
    const int grid = (int)std::max<int64_t>(1, extra_warps ? all : std::min<int64_t>(all, n_units));
    void* args[] = {params, extra};
    if (cudaLaunchKernel(fn, dim3(grid), dim3(threads), args, smem, stream) != cudaSuccess)
        return QUASAR_ERR_CUDA;
    return QUASAR_OK;
}


// Variant options of a call (quasar_options; NULL means the defaults).
struct Opts {
    int h_mode = kSalEma;
    bool packed = false;
    bool symmetric = false;
};

quasar_status read_options(const quasar_options* o, Opts* out)
{
    *out = Opts{};
    if (!o) return QUASAR_OK;
    if (o->saliency != QUASAR_SALIENCY_EMA && o->saliency != QUASAR_SALIENCY_EMA_SQUARED &&
        o->saliency != QUASAR_SALIENCY_UNIFORM)
        return QUASAR_ERR_INVALID_ARG;
    if (o->codes_layout != QUASAR_CODES_U8 && o->codes_layout != QUASAR_CODES_PACKED)
        return QUASAR_ERR_INVALID_ARG;
    if (o->grid != QUASAR_GRID_ASYMMETRIC && o->grid != QUASAR_GRID_SYMMETRIC)
        return QUASAR_ERR_INVALID_ARG;
    out->symmetric = o->grid == QUASAR_GRID_SYMMETRIC;
    out->h_mode = o->saliency == QUASAR_SALIENCY_EMA_SQUARED ? kSalEmaSquared
                  : o->saliency == QUASAR_SALIENCY_UNIFORM   ? kSalUniform
                                                             : kSalEma;
    out->packed = o->codes_layout == QUASAR_CODES_PACKED;
    return QUASAR_OK;
}


// Validation of one tensor of an integer-code call; fills its descriptor
// (unit0 is set by the caller).
quasar_status int_tensor(const float* w, const void* g, quasar_dtype g_dtype, float* v,
                         float beta2, const float* clip, int n_clip, int64_t rows, int64_t cols,
                         void* r, quasar_dtype r_dtype, uint8_t* codes, float* a, float* b,
                         uint8_t* cand_idx, int group_size, IntTensor* T, int bits = 8,
                         bool packed = false)
{
    int64_t n = 0;
    quasar_status st = check_common(w, g, g_dtype, v, beta2, clip, n_clip, rows, cols, r, r_dtype, &n);
    if (st != QUASAR_OK) return st;
    if (group_size <= 0 || cols % group_size != 0) return QUASAR_ERR_INVALID_ARG;
    const int64_t n_groups = n / group_size;
    if (n > 0) {
        if (!a || !b) return QUASAR_ERR_INVALID_ARG;
        if (codes && !aligned16(codes)) return QUASAR_ERR_INVALID_ARG;
        const void* outs[] = {r, codes, a, b, cand_idx};
        const size_t code_bytes = packed ? (size_t)n / 8 * (size_t)bits : (size_t)n;
        const size_t bytes[] = {(size_t)n * dtype_size(r_dtype), codes ? code_bytes : 0,
                                (size_t)n_groups * 4, (size_t)n_groups * 4,
                                cand_idx ? (size_t)n_groups : 0};
        if (outputs_alias_inputs(w, g, g_dtype, v, n, outs, bytes, 5)) return QUASAR_ERR_INVALID_ARG;
    }
    *T = IntTensor{w, g, v, nullptr, r, codes, a, b, cand_idx, n_groups, 0};
    return QUASAR_OK;
}

// Settings shared by the tensors of an integer-code call (no CUDA calls).
quasar_status int_check(int bits, int group_size)
{
    if (bits < 1 || bits > 8) return QUASAR_ERR_INVALID_ARG;
    if (group_size <= 0) return QUASAR_ERR_INVALID_ARG;
    if (group_size != 32 && group_size != 64 && group_size != 128 && group_size != 256)
        return QUASAR_ERR_UNSUPPORTED;
    return QUASAR_OK;
}

// Hyper-parameters of the fused AdamW step (validated by the caller).
struct AdamHp {
    float lr, beta1, eps, weight_decay;
    int64_t step;
};

// The CTA of an integer kernel: one per SM, with a ring of S slots of one unit
// tile each (w, v, m for the fused AdamW step, then the gradient region, which
// is also the candidate table and so at least kIntTableBytes for each 8
// candidates), S + 1 mbarriers, S sequence words and the next tile's number.
// As many warps as the registers allow, but one fewer than the slots that fit
// (a copy in flight), and up to kRingAhead slots in flight (QUASAR_STAGES
// overrides).  One slot in flight beyond the warps is enough: AdamW + INT4 g128
// with fp32 gradients, 14 slots, 949 us with 13 warps and 974 with 12; group
// 256, 7 slots, 518 with 6 and 556 with 5.  Of slots that are left, 8 in flight
// are a little better than 4 or 6 in small groups (INT2 g64, 16 factors: 1,408,
// 1,424 and 1,413 us).
constexpr int kRingAhead = 8;
constexpr size_t kCtaSmem = 227 * 1024;  // what a CTA may have

Launch plan_ring(int group_size, int g_kind, bool adam, int n_clip, int* warps)
{
    const uint32_t gbytes = g_kind == 2 ? 2u : (g_kind == 1 ? 4u : 0u);
    const uint32_t unit = (uint32_t)(kIntGroups * group_size);
    const uint32_t tile = unit * (adam ? 12u : 8u) + std::max(unit * gbytes, (uint32_t)((n_clip + 7) / 8) * kIntTableBytes);
    Launch L;
    L.stage_bytes = (tile + 127u) & ~127u;
    constexpr size_t kPerSlot = 8 + 4, kPerCta = 8 + 4;
    const int fit = (int)((kCtaSmem - kPerCta) / (L.stage_bytes + kPerSlot));
    *warps = std::min(int_max_warps(group_size / kIntLanes), fit - 1);
    L.stages = std::min(*warps + (tuning().stages > 0 ? tuning().stages : kRingAhead), fit);
    L.smem = (size_t)L.stages * (L.stage_bytes + kPerSlot) + kPerCta;
    return L;
}

// Parameters shared by the tensors of an integer-code call (adam: the
// AdamW-fused variant's step, else nullptr).
quasar_status int_params(quasar_dtype g_dtype, bool has_g, float beta2, int bits, int group_size,
                         const float* clip, int n_clip, quasar_dtype r_dtype, IntParams* p,
                         const AdamHp* adam = nullptr, const Opts& opt = Opts{})
{
    quasar_status st0 = int_check(bits, group_size);
    if (st0 != QUASAR_OK) return st0;
    *p = IntParams{};
    p->g_kind = has_g ? (g_dtype == QUASAR_BF16 ? 2 : 1) : 0;
    p->r_bf16 = r_dtype == QUASAR_BF16;
    p->h_mode = opt.h_mode;
    p->codes_packed = opt.packed;
    p->bits = bits;
    p->qmax = (1 << bits) - 1;
    p->n_clip = n_clip;
    p->beta2 = beta2;
    p->c1 = 1.0f - beta2;
    // each candidate sum is accumulated over at most G/8 terms a packed half
    // (4 lanes a group), plus the halves' sum and the lane tree (2 levels); the
    // terms' own roundings and those that form N, D and E make up the rest
    p->tie_kappa = tuning().tie_scale * (float)(group_size / 8 + 8);
    p->fit_ulps = tuning().fit_ulps;
    p->timeout_ns = kDefaultTimeoutNs;
    p->force_timeout_ns = (uint64_t)std::max<int64_t>(0, g_force_timeout_ns.load());
    p->stats = g_stats.load();
    // a factor below 2^-90 acts as 2^-90, which keeps q_max / (f range) finite
    // (only weights below that part of their group's range could tell)
    float f[kMaxClip];
    for (int k = 0; k < n_clip; ++k) f[k] = std::max(clip[k], std::ldexp(1.0f, -90));
    fill_clip(f, n_clip, p->f, p->invf);
    bool up = true, down = true;
    for (int k = 1; k < n_clip; ++k) {
        up &= p->invf[k] >= p->invf[k - 1];
        down &= p->invf[k] <= p->invf[k - 1];
    }
    p->monotone = up || down;
    quasar_status st;
    if ((st = status_ptr(&p->status)) != QUASAR_OK) return st;
    if (adam) {
        // fp32 constants of the step, formed in double from the fp32
        // hyper-parameters: w' = w - (w*lr*wd + step_size * m' / den),
        // den = sqrt(v') / sqrt(1 - beta2^t) + eps
        const double t = (double)adam->step;
        p->beta1 = adam->beta1;
        p->c1b = 1.0f - adam->beta1;
        p->lr_wd = (float)((double)adam->lr * (double)adam->weight_decay);
        p->step_size = (float)((double)adam->lr / (1.0 - std::pow((double)adam->beta1, t)));
        p->isbc2 = (float)(1.0 / std::sqrt(1.0 - std::pow((double)beta2, t)));
        p->eps = adam->eps;
    }
    return QUASAR_OK;
}

// Number the tensors' units consecutively and launch over all of them.
template <int MAXT>
quasar_status int_launch(IntLaunch<MAXT>& Lp, int group_size, int n_clip, cudaStream_t stream,
                         bool adam = false, bool symmetric = false)
{
    int64_t units = 0;
    for (int i = 0; i < Lp.n_t; ++i) {
        Lp.t[i].unit0 = units;
        units += (Lp.t[i].n_groups + kIntGroups - 1) / kIntGroups;
    }
    Lp.n_units = units;
    if (units == 0) return QUASAR_OK;
    int warps = 0;
    const Launch L = plan_ring(group_size, Lp.p.g_kind, adam, n_clip, &warps);
    Lp.p.stages = L.stages;
    Lp.p.stage_bytes = L.stage_bytes;
    const int epl = group_size / kIntLanes;
    const bool one_chunk = n_clip <= 8;
    const bool batch = MAXT > 1;
    const bool var = Lp.p.h_mode != kSalEma || Lp.p.codes_packed;
    // clamp sets: as large as the factors allow, unless switched off (sets of one)
    const int hoist_on = g_hoist.load() < 0 ? tuning().hoist : g_hoist.load();
    if (symmetric) {
        if (MAXT == 1) return QUASAR_ERR_UNSUPPORTED;
        fill_caps(&Lp.p, hoist_on ? 4 : 1, true, true);
        const int ss = Lp.p.set_size;
        const void* fn = (ss == 8   ? sym_kernel_ss8
                          : ss == 4 ? sym_kernel_ss4
                          : ss == 3 ? sym_kernel_ss3
                          : ss == 2 ? sym_kernel_ss2
                                    : sym_kernel_ss1)(epl);
        if (!fn) return QUASAR_ERR_UNSUPPORTED;
        return launch_persistent(fn, &Lp, L.smem, units, stream, warps);
    }
    // (sets of 8 or 3-3-2 with a single chunk)
    fill_caps(&Lp.p, hoist_on ? 4 : 1, one_chunk);
    using Entry = const void* (*)(int, bool, bool, bool);
    static const Entry table[2][5] = {
        {int_kernel_nch1_ss8, int_kernel_nch1_ss4, int_kernel_nch1_ss3, int_kernel_nch1_ss2, int_kernel_nch1_ss1},
        {nullptr, int_kernel_nch2_ss4, nullptr, int_kernel_nch2_ss2, int_kernel_nch2_ss1}};
    const int ci = one_chunk ? 0 : 1;
    const int ss = Lp.p.set_size;
    const int si = ss == 8 ? 0 : (ss == 4 ? 1 : (ss == 3 ? 2 : (ss == 2 ? 3 : 4)));
    if (!table[ci][si]) return QUASAR_ERR_UNSUPPORTED;
    const void* fn = table[ci][si](epl, batch, adam, var);
    if (!fn) return QUASAR_ERR_UNSUPPORTED;
    return launch_persistent(fn, &Lp, L.smem, units, stream, warps);
}

// Validation of one tensor of an NVFP4 call; fills its descriptor and its
// absmax/scale item (unit0 is set later).
quasar_status nvfp4_tensor(const float* w, const void* g, quasar_dtype g_dtype, float* v,
                           float beta2, const float* clip, int n_clip, int64_t rows, int64_t cols,
                           const float* tensor_amax, void* r, quasar_dtype r_dtype, uint8_t* codes,
                           uint8_t* block_scale, float* tensor_scale, uint8_t* cand_idx,
                           Nvfp4Tensor* T, AmaxItem* A, bool packed = false)
{
    int64_t n = 0;
    quasar_status st = check_common(w, g, g_dtype, v, beta2, clip, n_clip, rows, cols, r, r_dtype, &n);
    if (st != QUASAR_OK) return st;
    if (cols % 16 != 0) return QUASAR_ERR_INVALID_ARG;
    if (!tensor_scale || (reinterpret_cast<uintptr_t>(tensor_scale) & 3u) != 0)
        return QUASAR_ERR_INVALID_ARG;
    if (tensor_amax && (reinterpret_cast<uintptr_t>(tensor_amax) & 3u) != 0)
        return QUASAR_ERR_INVALID_ARG;
    const int64_t n_blocks = n / 16;
    if (n > 0) {
        if (!block_scale) return QUASAR_ERR_INVALID_ARG;
        if (codes && !aligned16(codes)) return QUASAR_ERR_INVALID_ARG;
        const void* outs[] = {r, codes, block_scale, tensor_scale, cand_idx};
        const size_t bytes[] = {(size_t)n * dtype_size(r_dtype),
                                codes ? (packed ? (size_t)n / 2 : (size_t)n) : 0, (size_t)n_blocks, 4,
                                cand_idx ? (size_t)n_blocks : 0};
        if (outputs_alias_inputs(w, g, g_dtype, v, n, outs, bytes, 5)) return QUASAR_ERR_INVALID_ARG;
        if (tensor_amax && overlaps(tensor_amax, 4, tensor_scale, 4)) return QUASAR_ERR_INVALID_ARG;
    }
    *T = Nvfp4Tensor{w, g, v, r, codes, block_scale, cand_idx, tensor_amax ? tensor_amax : tensor_scale,
                     n_blocks, 0};
    *A = AmaxItem{w, n, tensor_scale, tensor_amax};
    return QUASAR_OK;
}

quasar_status nvfp4_params(bool has_g, quasar_dtype g_dtype, float beta2, const float* clip,
                           int n_clip, quasar_dtype r_dtype, Nvfp4Params* p,
                           const Opts& opt = Opts{})
{
    *p = Nvfp4Params{};
    p->g_kind = has_g ? (g_dtype == QUASAR_BF16 ? 2 : 1) : 0;
    p->r_bf16 = r_dtype == QUASAR_BF16;
    p->h_mode = opt.h_mode;
    p->codes_packed = opt.packed;
    p->n_clip = n_clip;
    p->beta2 = beta2;
    p->c1 = 1.0f - beta2;
    p->tie_kappa = tuning().tie_kappa;
    p->timeout_ns = kDefaultTimeoutNs;
    p->force_timeout_ns = (uint64_t)std::max<int64_t>(0, g_force_timeout_ns.load());
    p->stats = g_stats.load();
    fill_clip(clip, n_clip, p->f, p->invf);
    return status_ptr(&p->status);
}

// The absmax slots of a batch set to 0 (those of the tensors whose amax is
// computed, or all of them), in one launch.
template <int MAXT>
quasar_status zero_amax_slots(const AmaxBatch<MAXT>& B, bool all, cudaStream_t s)
{
    static_assert(MAXT == 1 || MAXT == kMaxBatch, "the sizes the kernel is built for");
    int flag = all ? 1 : 0;
    void* args[] = {(void*)&B, (void*)&flag};
    if (cudaLaunchKernel(amax_init_kernel(MAXT > 1), dim3(1), dim3(256), args, 0, s) != cudaSuccess)
        return QUASAR_ERR_CUDA;
    return QUASAR_OK;
}

// Absmax of the tensors whose amax is not supplied, into their scale slots
// (zeroed first by the caller of each slot), beside nothing.
template <int MAXT>
quasar_status launch_amax(const AmaxBatch<MAXT>& B, cudaStream_t s)
{
    static_assert(MAXT == 1 || MAXT == kMaxStage, "the sizes k_amax is built for");
    int dev = 0;
    const DeviceInfo* info = nullptr;
    const quasar_status st = device_info(&dev, &info);
    if (st != QUASAR_OK) return st;
    int64_t nmax = 0;
    for (int i = 0; i < B.n_t; ++i)
        if (!B.t[i].amax_in) nmax = std::max(nmax, B.t[i].n);
    if (nmax == 0) return QUASAR_OK;
    const int64_t want = (nmax / 4 + kThreads - 1) / kThreads;
    const int64_t per_sm = std::max<int64_t>(1, (int64_t)info->nsm * 8 / B.n_t);
    const int gx = (int)std::max<int64_t>(1, std::min<int64_t>(per_sm, want));
    void* args[] = {(void*)&B};
    if (cudaLaunchKernel(amax_kernel(MAXT > 1), dim3(gx, B.n_t), dim3(kThreads), args, 0, s) !=
        cudaSuccess)
        return QUASAR_ERR_CUDA;
    return QUASAR_OK;
}

// Every slot := s_T.
template <int MAXT>
quasar_status launch_to_scale(const AmaxBatch<MAXT>& B, cudaStream_t s)
{
    static_assert(MAXT == 1 || MAXT == kMaxBatch, "the sizes the kernel is built for");
    void* args[] = {(void*)&B};
    if (cudaLaunchKernel(amax_to_scale_kernel(MAXT > 1), dim3(1), dim3(256), args, 0, s) != cudaSuccess)
        return QUASAR_ERR_CUDA;
    return QUASAR_OK;
}

// Number the units of a launch's tensors and plan the tiles of its warps that
// reconstruct from the start; returns the units.
template <int MAXT>
int64_t nvfp4_number_units(Nvfp4Launch<MAXT>& Lp, int warps, size_t* smem)
{
    int64_t units = 0;
    for (int i = 0; i < Lp.n_t; ++i) {
        Lp.t[i].unit0 = units;
        units += (Lp.t[i].n_blocks + kBlocksPerUnit - 1) / kBlocksPerUnit;
    }
    Lp.n_units = units;
    const int gbytes = Lp.p.g_kind == 2 ? 2 : (Lp.p.g_kind == 1 ? 4 : 0);
    // one tile a warp and its barrier (the tile is in registers, and the next copy
    // under way, before the search begins), the failure hook's, the next unit's number
    Lp.p.stage_bytes = (uint32_t)(kBlocksPerUnit * 16 * (8 + gbytes));
    *smem = (size_t)warps * (Lp.p.stage_bytes + 8) + 16;
    return units;
}

// The reconstruction of a launch's tensors, beside nothing.
template <int MAXT>
quasar_status nvfp4_recon(Nvfp4Launch<MAXT>& Lp, cudaStream_t s)
{
    size_t smem = 0;
    const int64_t units = nvfp4_number_units(Lp, kNvfp4Warps, &smem);
    if (units == 0) return QUASAR_OK;
    NoAheadArg none;
    return launch_persistent(nvfp4_kernel(MAXT > 1), &Lp, smem, units, s, kNvfp4Warps, &none);
}

// The AdamW steps of a launch's tensors, beside nothing.
quasar_status launch_adamw(const AdamwBatch<kMaxStage>& B, cudaStream_t s)
{
    int dev = 0;
    const DeviceInfo* info = nullptr;
    const quasar_status st = device_info(&dev, &info);
    if (st != QUASAR_OK) return st;
    int64_t nmax = 0;
    for (int i = 0; i < B.n_t; ++i) nmax = std::max(nmax, B.t[i].n);
    if (nmax == 0) return QUASAR_OK;
    const int64_t want = (nmax / 4 + kThreads - 1) / kThreads;
    const int64_t per = std::max<int64_t>(1, (int64_t)info->nsm * 8 / B.n_t);
    const int gx = (int)std::max<int64_t>(1, std::min<int64_t>(per, want));
    void* args[] = {(void*)&B};
    if (cudaLaunchKernel(adamw_amax_kernel(), dim3(gx, B.n_t), dim3(kThreads), args, 0, s) != cudaSuccess)
        return QUASAR_ERR_CUDA;
    return QUASAR_OK;
}

// A batch is cut into stages of whole tensors whose absmax (or AdamW) pass
// runs beside the reconstruction of the stage before: about kStages of them, so
// that little of either pass runs alone, but none smaller than kStageMin
// weights, about 40 us of reconstruction, below which the launches' own ends
// cost more than the overlap gives.
constexpr int kStages = 8;
constexpr int64_t kStageMin = int64_t(1) << 23;

// The NVFP4 call over n tensors.  fill(i, T, A, W) describes tensor i (validated
// before); hp: the AdamW step, or nullptr for none.
template <class Fill>
quasar_status nvfp4_batch(int n, const Fill& fill, const Nvfp4Params& p, const AdamwHp* hp, cudaStream_t s)
{
    // kept off the stack
    static thread_local Nvfp4Launch<kMaxBatch> alone;
    static thread_local Nvfp4Launch<kMaxStage> staged;
    static thread_local AmaxBatch<kMaxBatch> slots;
    static thread_local AmaxBatch<kMaxStage> amax;
    static thread_local AdamwBatch<kMaxStage> adamw;
    quasar_status st;
    Nvfp4Tensor T;
    AmaxItem A;
    AdamwItem W;
    int64_t total = 0;
    bool ahead = false;  // some tensor needs a pass before its reconstruction
    for (int i = 0; i < n; ++i) {
        fill(i, &T, &A, &W);
        total += A.n;
        ahead |= hp != nullptr || (!A.amax_in && A.n > 0);
    }
    auto all_slots = [&](auto&& launch) {
        for (int i0 = 0; i0 < n; i0 += kMaxBatch) {
            slots.n_t = std::min(kMaxBatch, n - i0);
            for (int i = 0; i < slots.n_t; ++i) fill(i0 + i, &T, &slots.t[i], &W);
            if ((st = launch()) != QUASAR_OK) return st;
        }
        return QUASAR_OK;
    };
    // scale slots of tensors whose amax is computed start at 0
    if (all_slots([&] {
            bool any = hp != nullptr;
            for (int i = 0; i < slots.n_t; ++i) any |= !slots.t[i].amax_in;
            return any ? zero_amax_slots(slots, hp != nullptr, s) : QUASAR_OK;
        }) != QUASAR_OK)
        return st;
    const int64_t target = std::max<int64_t>(kStageMin, total / kStages);
    auto stage_end = [&](int i) {
        int64_t sum = 0;
        const int most = ahead ? kMaxStage : kMaxBatch;
        int j = i;
        while (j < n && j - i < most && (!ahead || sum < target)) {
            fill(j++, &T, &A, &W);
            sum += A.n;
        }
        return j;
    };
    // the pass of the tensors [i0, i1): described, and launched alone
    auto describe_ahead = [&](int i0, int i1) {
        amax.n_t = adamw.n_t = i1 - i0;
        if (hp) adamw.hp = *hp;
        adamw.n_units = 0;
        for (int i = i0; i < i1; ++i) {
            AdamwItem& w = adamw.t[i - i0];
            fill(i, &T, &amax.t[i - i0], &w);
            if (!hp) continue;
            w.unit0 = adamw.n_units;
            adamw.n_units += (w.n + kAheadUnit - 1) / kAheadUnit;
        }
    };
    auto ahead_alone = [&] { return hp ? launch_adamw(adamw, s) : launch_amax(amax, s); };
    int a0 = 0, a1 = stage_end(0);
    if (ahead) {
        describe_ahead(a0, a1);
        if ((st = ahead_alone()) != QUASAR_OK) return st;
    }
    while (a0 < n) {
        const int b1 = a1 < n ? stage_end(a1) : a1;
        size_t smem = 0;
        bool fused = false;
        if (ahead && b1 > a1) {
            describe_ahead(a1, b1);
            staged.p = p;
            staged.n_t = a1 - a0;
            for (int i = a0; i < a1; ++i) fill(i, &staged.t[i - a0], &A, &W);
            const int extra = hp ? kAdamwWarps : kAmaxWarps, warps = (hp ? kNvfp4AdamwWarps : kNvfp4Warps) - extra;
            const int64_t units = nvfp4_number_units(staged, warps, &smem);
            smem = (smem + 127) & ~size_t(127);
            staged.p.ahead_smem = (uint32_t)smem;
            staged.p.ahead_bytes = ahead_region(
                hp ? std::max(staged.p.stage_bytes, kAheadTiles * (kAheadUnit * (hp->g_kind == 2 ? 14u : 16u) + 8u))
                   : staged.p.stage_bytes);
            smem += extra * staged.p.ahead_bytes;
            fused = units > 0;
            st = fused ? launch_persistent(hp ? nvfp4_adamw_ahead_kernel() : nvfp4_amax_ahead_kernel(), &staged,
                                           smem, units, s, warps, hp ? (void*)&adamw : (void*)&amax, extra)
                       : ahead_alone();
            if (st != QUASAR_OK) return st;
        }
        if (!fused) {
            alone.p = p;
            alone.n_t = a1 - a0;
            for (int i = a0; i < a1; ++i) fill(i, &alone.t[i - a0], &A, &W);
            if ((st = nvfp4_recon(alone, s)) != QUASAR_OK) return st;
        }
        a0 = a1;
        a1 = b1;
    }
    return all_slots([&] { return launch_to_scale(slots, s); });
}

}  // namespace

extern "C" {

quasar_status quasar_recon_int(const float* w, const void* g, quasar_dtype g_dtype, float* v,
                               float beta2, int bits, int group_size, const float* clip,
                               int n_clip, int64_t rows, int64_t cols, void* r,
                               quasar_dtype r_dtype, uint8_t* codes, float* a, float* b,
                               uint8_t* cand_idx, quasar_stream_t stream)
{
    IntLaunch<1> Lp;
    quasar_status st = int_tensor(w, g, g_dtype, v, beta2, clip, n_clip, rows, cols, r, r_dtype,
                                  codes, a, b, cand_idx, group_size > 0 ? group_size : 1, &Lp.t[0]);
    if (st != QUASAR_OK) return st;
    if ((st = int_check(bits, group_size)) != QUASAR_OK) return st;
    if (Lp.t[0].n_groups == 0) return QUASAR_OK;  // empty: no-op
    if ((st = int_params(g_dtype, g != nullptr, beta2, bits, group_size, clip, n_clip, r_dtype,
                         &Lp.p)) != QUASAR_OK)
        return st;
    Lp.n_t = 1;
    return int_launch(Lp, group_size, n_clip, reinterpret_cast<cudaStream_t>(stream));
}

quasar_status quasar_recon_int_batch(const quasar_int_tensor* tensors, int n_tensors,
                                     quasar_dtype g_dtype, float beta2, int bits, int group_size,
                                     const float* clip, int n_clip, quasar_dtype r_dtype,
                                     quasar_stream_t stream)
{
    return quasar_recon_int_batch_ex(tensors, n_tensors, g_dtype, beta2, bits, group_size, clip,
                                     n_clip, r_dtype, nullptr, stream);
}

quasar_status quasar_recon_int_batch_ex(const quasar_int_tensor* tensors, int n_tensors,
                                        quasar_dtype g_dtype, float beta2, int bits,
                                        int group_size, const float* clip, int n_clip,
                                        quasar_dtype r_dtype, const quasar_options* options,
                                        quasar_stream_t stream)
{
    Opts opt;
    if (read_options(options, &opt) != QUASAR_OK) return QUASAR_ERR_INVALID_ARG;
    if (n_tensors < 0 || (n_tensors > 0 && !tensors)) return QUASAR_ERR_INVALID_ARG;
    if (opt.symmetric && bits < 2) return QUASAR_ERR_INVALID_ARG;  // Q = 2^(bits-1) - 1 >= 1
    if (n_tensors == 0) return QUASAR_OK;
    // all non-empty tensors carry a gradient, or none does
    int with_g = 0, non_empty = 0;
    for (int i = 0; i < n_tensors; ++i)
        if (tensors[i].rows != 0 && tensors[i].cols != 0) {
            ++non_empty;
            with_g += tensors[i].g != nullptr;
        }
    if (with_g != 0 && with_g != non_empty) return QUASAR_ERR_INVALID_ARG;
    const bool has_g = with_g != 0;
    static thread_local IntLaunch<kMaxBatch> Lp;  // 20 KB: kept off the stack
    quasar_status st = int_check(bits, group_size);
    if (st != QUASAR_OK) return st;
    // validate every tensor before launching anything
    int64_t total = 0;
    for (int i = 0; i < n_tensors; ++i) {
        const quasar_int_tensor& x = tensors[i];
        IntTensor T;
        if ((st = int_tensor(x.w, x.g, g_dtype, x.v, beta2, clip, n_clip, x.rows, x.cols, x.r,
                             r_dtype, x.codes, x.a, x.b, x.cand_idx, group_size, &T, bits,
                             opt.packed)) != QUASAR_OK)
            return st;
        total += T.n_groups;
    }
    if (total == 0) return QUASAR_OK;
    if ((st = int_params(g_dtype, has_g, beta2, bits, group_size, clip, n_clip, r_dtype, &Lp.p,
                         nullptr, opt)) != QUASAR_OK)
        return st;
    const cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    for (int i0 = 0; i0 < n_tensors; i0 += kMaxBatch) {
        Lp.n_t = std::min(kMaxBatch, n_tensors - i0);
        for (int i = 0; i < Lp.n_t; ++i) {
            const quasar_int_tensor& x = tensors[i0 + i];
            int_tensor(x.w, x.g, g_dtype, x.v, beta2, clip, n_clip, x.rows, x.cols, x.r, r_dtype,
                       x.codes, x.a, x.b, x.cand_idx, group_size, &Lp.t[i], bits, opt.packed);
        }
        if ((st = int_launch(Lp, group_size, n_clip, s, false, opt.symmetric)) != QUASAR_OK) return st;
    }
    return QUASAR_OK;
}

quasar_status quasar_adamw_recon_int_batch(const quasar_adamw_tensor* tensors, int n_tensors,
                                           quasar_dtype g_dtype, float lr, float beta1,
                                           float beta2, float eps, float weight_decay,
                                           int64_t step, int bits, int group_size,
                                           const float* clip, int n_clip, quasar_dtype r_dtype,
                                           const quasar_options* options, quasar_stream_t stream)
{
    Opts opt;
    if (read_options(options, &opt) != QUASAR_OK) return QUASAR_ERR_INVALID_ARG;
    if (opt.symmetric) return QUASAR_ERR_UNSUPPORTED;  // no fused AdamW kernel for symmetric codes
    if (n_tensors < 0 || (n_tensors > 0 && !tensors)) return QUASAR_ERR_INVALID_ARG;
    if (!(std::isfinite(lr) && lr >= 0.0f) || !(beta1 >= 0.0f && beta1 < 1.0f) ||
        !(std::isfinite(eps) && eps > 0.0f) ||
        !(std::isfinite(weight_decay) && weight_decay >= 0.0f) || step < 1)
        return QUASAR_ERR_INVALID_ARG;
    if (n_tensors == 0) return QUASAR_OK;
    static thread_local IntLaunch<kMaxBatch> Lp;
    quasar_status st = int_check(bits, group_size);
    if (st != QUASAR_OK) return st;
    // one tensor's descriptor; checks beyond those of the reconstruction:
    // g and m present, and w, g, m, v pairwise disjoint
    auto describe = [&](const quasar_adamw_tensor& x, IntTensor* T) {
        quasar_status s1 = int_tensor(x.w, x.g, g_dtype, x.v, beta2, clip, n_clip, x.rows, x.cols,
                                      x.r, r_dtype, x.codes, x.a, x.b, x.cand_idx, group_size, T,
                                      bits, opt.packed);
        if (s1 != QUASAR_OK) return s1;
        T->m = x.m;
        if (T->n_groups == 0) return QUASAR_OK;
        if (!x.g || !x.m || !aligned16(x.m)) return QUASAR_ERR_INVALID_ARG;
        const size_t n = (size_t)(x.rows * x.cols);
        const void* outs[] = {x.r, x.codes, x.a, x.b, x.cand_idx};
        const size_t bytes[] = {n * dtype_size(r_dtype), x.codes ? (opt.packed ? n / 8 * bits : n) : 0,
                                (size_t)T->n_groups * 4, (size_t)T->n_groups * 4,
                                x.cand_idx ? (size_t)T->n_groups : 0};
        for (int i = 0; i < 5; ++i)
            if (overlaps(outs[i], bytes[i], x.m, n * 4)) return QUASAR_ERR_INVALID_ARG;
        const void* state[] = {x.w, x.g, x.m, x.v};
        const size_t sbytes[] = {n * 4, n * dtype_size(g_dtype), n * 4, n * 4};
        for (int i = 0; i < 4; ++i)
            for (int j = i + 1; j < 4; ++j)
                if (overlaps(state[i], sbytes[i], state[j], sbytes[j])) return QUASAR_ERR_INVALID_ARG;
        return QUASAR_OK;
    };
    int64_t total = 0;
    for (int i = 0; i < n_tensors; ++i) {
        IntTensor T;
        if ((st = describe(tensors[i], &T)) != QUASAR_OK) return st;
        total += T.n_groups;
    }
    if (total == 0) return QUASAR_OK;
    const AdamHp hp{lr, beta1, eps, weight_decay, step};
    if ((st = int_params(g_dtype, true, beta2, bits, group_size, clip, n_clip, r_dtype, &Lp.p,
                         &hp, opt)) != QUASAR_OK)
        return st;
    const cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    for (int i0 = 0; i0 < n_tensors; i0 += kMaxBatch) {
        Lp.n_t = std::min(kMaxBatch, n_tensors - i0);
        for (int i = 0; i < Lp.n_t; ++i) describe(tensors[i0 + i], &Lp.t[i]);
        if ((st = int_launch(Lp, group_size, n_clip, s, true)) != QUASAR_OK) return st;
    }
    return QUASAR_OK;
}

quasar_status quasar_tensor_amax(const float* w, int64_t n, float* amax_out, quasar_stream_t stream)
{
    if (n < 0 || !amax_out) return QUASAR_ERR_INVALID_ARG;
    if (n > 0 && (!w || !aligned16(w))) return QUASAR_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(amax_out) & 3u) != 0) return QUASAR_ERR_INVALID_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(amax_out, 0, sizeof(float), s) != cudaSuccess) return QUASAR_ERR_CUDA;
    if (n == 0) return QUASAR_OK;
    AmaxBatch<1> B;
    B.n_t = 1;
    B.t[0] = AmaxItem{w, n, amax_out, nullptr};
    return launch_amax(B, s);
}

quasar_status quasar_recon_nvfp4(const float* w, const void* g, quasar_dtype g_dtype, float* v,
                                 float beta2, const float* clip, int n_clip, int64_t rows,
                                 int64_t cols, const float* tensor_amax, void* r,
                                 quasar_dtype r_dtype, uint8_t* codes, uint8_t* block_scale,
                                 float* tensor_scale, uint8_t* cand_idx, quasar_stream_t stream)
{
    Nvfp4Launch<1> Lp;
    AmaxBatch<1> B;
    quasar_status st = nvfp4_tensor(w, g, g_dtype, v, beta2, clip, n_clip, rows, cols, tensor_amax, r,
                                    r_dtype, codes, block_scale, tensor_scale, cand_idx, &Lp.t[0],
                                    &B.t[0]);
    if (st != QUASAR_OK) return st;
    Lp.n_t = B.n_t = 1;
    if ((st = nvfp4_params(g != nullptr, g_dtype, beta2, clip, n_clip, r_dtype, &Lp.p)) != QUASAR_OK)
        return st;
    const cudaStream_t cs = reinterpret_cast<cudaStream_t>(stream);
    if (!tensor_amax &&
        ((st = zero_amax_slots(B, false, cs)) != QUASAR_OK || (st = launch_amax(B, cs)) != QUASAR_OK))
        return st;
    if ((st = nvfp4_recon(Lp, cs)) != QUASAR_OK) return st;
    return launch_to_scale(B, cs);
}

quasar_status quasar_recon_nvfp4_batch(const quasar_nvfp4_tensor* tensors, int n_tensors,
                                       quasar_dtype g_dtype, float beta2, const float* clip,
                                       int n_clip, quasar_dtype r_dtype, quasar_stream_t stream)
{
    return quasar_recon_nvfp4_batch_ex(tensors, n_tensors, g_dtype, beta2, clip, n_clip, r_dtype,
                                       nullptr, stream);
}

quasar_status quasar_recon_nvfp4_batch_ex(const quasar_nvfp4_tensor* tensors, int n_tensors,
                                          quasar_dtype g_dtype, float beta2, const float* clip,
                                          int n_clip, quasar_dtype r_dtype,
                                          const quasar_options* options, quasar_stream_t stream)
{
    Opts opt;
    if (read_options(options, &opt) != QUASAR_OK) return QUASAR_ERR_INVALID_ARG;
    if (opt.symmetric) return QUASAR_ERR_INVALID_ARG;  // an integer-code option
    if (n_tensors < 0 || (n_tensors > 0 && !tensors)) return QUASAR_ERR_INVALID_ARG;
    if (n_tensors == 0) return QUASAR_OK;
    int with_g = 0, non_empty = 0;
    for (int i = 0; i < n_tensors; ++i)
        if (tensors[i].rows != 0 && tensors[i].cols != 0) {
            ++non_empty;
            with_g += tensors[i].g != nullptr;
        }
    if (with_g != 0 && with_g != non_empty) return QUASAR_ERR_INVALID_ARG;
    const bool has_g = with_g != 0;
    // one tensor's checks; fills its descriptors
    auto describe = [&](int i, Nvfp4Tensor* T, AmaxItem* A) {
        const quasar_nvfp4_tensor& x = tensors[i];
        return nvfp4_tensor(x.w, x.g, g_dtype, x.v, beta2, clip, n_clip, x.rows, x.cols, x.tensor_amax, x.r,
                            r_dtype, x.codes, x.block_scale, x.tensor_scale, x.cand_idx, T, A, opt.packed);
    };
    quasar_status st;
    for (int i = 0; i < n_tensors; ++i) {  // validate everything first
        Nvfp4Tensor T;
        AmaxItem A;
        if ((st = describe(i, &T, &A)) != QUASAR_OK) return st;
    }
    Nvfp4Params p;
    if ((st = nvfp4_params(has_g, g_dtype, beta2, clip, n_clip, r_dtype, &p, opt)) != QUASAR_OK) return st;
    return nvfp4_batch(n_tensors, [&](int i, Nvfp4Tensor* T, AmaxItem* A, AdamwItem*) { describe(i, T, A); }, p,
                       nullptr, reinterpret_cast<cudaStream_t>(stream));
}

quasar_status quasar_recon_lut_batch(const quasar_lut_tensor* tensors, int n_tensors,
                                     quasar_dtype g_dtype, float beta2, const float* clip,
                                     int n_clip, quasar_dtype r_dtype, const quasar_options* options,
                                     quasar_stream_t stream)
{
    Opts opt;
    if (read_options(options, &opt) != QUASAR_OK) return QUASAR_ERR_INVALID_ARG;
    if (opt.symmetric) return QUASAR_ERR_INVALID_ARG;  // an integer-code option
    if (n_tensors < 0 || (n_tensors > 0 && !tensors)) return QUASAR_ERR_INVALID_ARG;
    if (n_tensors == 0) return QUASAR_OK;
    int with_g = 0, non_empty = 0;
    for (int i = 0; i < n_tensors; ++i)
        if (tensors[i].rows != 0 && tensors[i].cols != 0) {
            ++non_empty;
            with_g += tensors[i].g != nullptr;
        }
    if (with_g != 0 && with_g != non_empty) return QUASAR_ERR_INVALID_ARG;
    const bool has_g = with_g != 0;
    // one tensor's checks; fills its descriptor (unit0 set later)
    auto describe = [&](const quasar_lut_tensor& x, LutTensor* T) {
        int64_t n = 0;
        quasar_status s1 = check_common(x.w, x.g, g_dtype, x.v, beta2, clip, n_clip, x.rows, x.cols,
                                        x.r, r_dtype, &n);
        if (s1 != QUASAR_OK) return s1;
        if (x.rows % kLutRows != 0 || x.cols % kLutCols != 0) return QUASAR_ERR_INVALID_ARG;
        const int64_t n_blocks = n / kLutBlock;
        if (n_blocks > (int64_t)UINT32_MAX) return QUASAR_ERR_INVALID_ARG;  // 32-bit block indices
        if (n > 0) {
            if (!x.book || !aligned16(x.book)) return QUASAR_ERR_INVALID_ARG;
            if (x.codes && !aligned16(x.codes)) return QUASAR_ERR_INVALID_ARG;
            const void* outs[] = {x.r, x.codes, x.book, x.cand_idx};
            const size_t bytes[] = {(size_t)n * dtype_size(r_dtype),
                                    x.codes ? (opt.packed ? (size_t)n / 8 * 3 : (size_t)n) : 0,
                                    (size_t)n_blocks * 8, x.cand_idx ? (size_t)n_blocks : 0};
            if (outputs_alias_inputs(x.w, x.g, g_dtype, x.v, n, outs, bytes, 4))
                return QUASAR_ERR_INVALID_ARG;
        }
        const uint64_t nbc = (uint64_t)std::max<int64_t>(1, x.cols / kLutCols);
        *T = LutTensor{x.w, x.g, x.v, x.r, x.codes, x.book, x.cand_idx, x.cols, n_blocks, 0, (uint32_t)nbc,
                       (uint32_t)std::min<uint64_t>(UINT32_MAX, (uint64_t(1) << 32) / nbc)};
        return QUASAR_OK;
    };
    static thread_local LutLaunch<kMaxBatch> Lp;
    int64_t total = 0;
    quasar_status st;
    for (int i = 0; i < n_tensors; ++i) {
        LutTensor T;
        if ((st = describe(tensors[i], &T)) != QUASAR_OK) return st;
        total += T.n_blocks;
    }
    if (total == 0) return QUASAR_OK;
    LutParams& p = Lp.p;
    p = LutParams{};
    p.g_kind = has_g ? (g_dtype == QUASAR_BF16 ? 2 : 1) : 0;
    p.r_bf16 = r_dtype == QUASAR_BF16;
    p.h_mode = opt.h_mode;
    p.codes_packed = opt.packed;
    p.n_clip = n_clip;
    p.beta2 = beta2;
    p.c1 = 1.0f - beta2;
    p.tie_kappa = tuning().tie_scale;
    p.force_timeout_ns = (uint64_t)std::max<int64_t>(0, g_force_timeout_ns.load());
    p.stats = g_stats.load();
    fill_clip(clip, n_clip, p.f, p.invf);
    p.invf_max = *std::max_element(p.invf, p.invf + n_clip);
    if ((st = status_ptr(&p.status)) != QUASAR_OK) return st;
    const uint32_t gbytes = p.g_kind == 2 ? 2 : (p.g_kind == 1 ? 4 : 0);
    p.stage_bytes = (std::max(kLutBlock * (8 + gbytes), kLutListBytes) + 127u) & ~127u;
    // (and the next unit's number)
    const size_t smem = (size_t)kLutWarps * (p.stage_bytes + kLutScratchBytes) + sizeof(int);
    const cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    for (int i0 = 0; i0 < n_tensors; i0 += kMaxBatch) {
        Lp.n_t = std::min(kMaxBatch, n_tensors - i0);
        int64_t units = 0;
        for (int i = 0; i < Lp.n_t; ++i) {
            describe(tensors[i0 + i], &Lp.t[i]);
            Lp.t[i].unit0 = units;
            units += Lp.t[i].n_blocks;
        }
        Lp.n_units = units;
        if (units == 0) continue;
        if ((st = launch_persistent(lut_kernel(), &Lp, smem, units, s, kLutWarps)) != QUASAR_OK) return st;
    }
    return QUASAR_OK;
}

quasar_status quasar_adamw_recon_nvfp4_batch(const quasar_adamw_nvfp4_tensor* tensors,
                                             int n_tensors, quasar_dtype g_dtype, float lr,
                                             float beta1, float beta2, float eps,
                                             float weight_decay, int64_t step, const float* clip,
                                             int n_clip, quasar_dtype r_dtype,
                                             const quasar_options* options, quasar_stream_t stream)
{
    Opts opt;
    if (read_options(options, &opt) != QUASAR_OK) return QUASAR_ERR_INVALID_ARG;
    if (opt.symmetric) return QUASAR_ERR_INVALID_ARG;  // an integer-code option
    if (n_tensors < 0 || (n_tensors > 0 && !tensors)) return QUASAR_ERR_INVALID_ARG;
    if (!(std::isfinite(lr) && lr >= 0.0f) || !(beta1 >= 0.0f && beta1 < 1.0f) ||
        !(std::isfinite(eps) && eps > 0.0f) ||
        !(std::isfinite(weight_decay) && weight_decay >= 0.0f) || step < 1 || !valid_dtype(g_dtype))
        return QUASAR_ERR_INVALID_ARG;
    if (n_tensors == 0) return QUASAR_OK;
    // one tensor: the reconstruction's checks (without a gradient: v is
    // updated by the AdamW pass), plus g and m present and w, g, m, v
    // pairwise disjoint
    auto describe = [&](const quasar_adamw_nvfp4_tensor& x, Nvfp4Tensor* T, AmaxItem* A,
                        AdamwItem* W) {
        quasar_status s1 = nvfp4_tensor(x.w, nullptr, g_dtype, x.v, beta2, clip, n_clip, x.rows,
                                        x.cols, nullptr, x.r, r_dtype, x.codes, x.block_scale,
                                        x.tensor_scale, x.cand_idx, T, A, opt.packed);
        if (s1 != QUASAR_OK) return s1;
        const int64_t n = x.rows * x.cols;
        *W = AdamwItem{x.w, x.g, x.m, x.v, n, x.tensor_scale, 0};
        if (n == 0) return QUASAR_OK;
        if (!x.g || !x.m || !aligned16(x.g) || !aligned16(x.m)) return QUASAR_ERR_INVALID_ARG;
        const size_t nb = (size_t)n;
        const void* outs[] = {x.r, x.codes, x.block_scale, x.tensor_scale, x.cand_idx};
        const size_t bytes[] = {nb * dtype_size(r_dtype), x.codes ? (opt.packed ? nb / 2 : nb) : 0,
                                nb / 16, 4, x.cand_idx ? nb / 16 : 0};
        for (int i = 0; i < 5; ++i)
            if (overlaps(outs[i], bytes[i], x.m, nb * 4) ||
                overlaps(outs[i], bytes[i], x.g, nb * dtype_size(g_dtype)))
                return QUASAR_ERR_INVALID_ARG;
        const void* state[] = {x.w, x.g, x.m, x.v};
        const size_t sbytes[] = {nb * 4, nb * dtype_size(g_dtype), nb * 4, nb * 4};
        for (int i = 0; i < 4; ++i)
            for (int j = i + 1; j < 4; ++j)
                if (overlaps(state[i], sbytes[i], state[j], sbytes[j])) return QUASAR_ERR_INVALID_ARG;
        return QUASAR_OK;
    };
    quasar_status st;
    for (int i = 0; i < n_tensors; ++i) {
        Nvfp4Tensor T;
        AmaxItem A;
        AdamwItem W;
        if ((st = describe(tensors[i], &T, &A, &W)) != QUASAR_OK) return st;
    }
    Nvfp4Params p;
    if ((st = nvfp4_params(false, g_dtype, beta2, clip, n_clip, r_dtype, &p, opt)) != QUASAR_OK) return st;
    const double t = (double)step;
    AdamwHp hp;
    hp.g_kind = g_dtype == QUASAR_BF16 ? 2 : 1;
    hp.beta1 = beta1;
    hp.c1b = 1.0f - beta1;
    hp.beta2 = beta2;
    hp.c1 = 1.0f - beta2;
    hp.lr_wd = (float)((double)lr * (double)weight_decay);
    hp.step_size = (float)((double)lr / (1.0 - std::pow((double)beta1, t)));
    hp.isbc2 = (float)(1.0 / std::sqrt(1.0 - std::pow((double)beta2, t)));
    hp.eps = eps;
    return nvfp4_batch(
        n_tensors, [&](int i, Nvfp4Tensor* T, AmaxItem* A, AdamwItem* W) { describe(tensors[i], T, A, W); }, p, &hp,
        reinterpret_cast<cudaStream_t>(stream));
}

quasar_status quasar_get_device_status(quasar_stream_t stream)
{
    if (cudaStreamSynchronize(reinterpret_cast<cudaStream_t>(stream)) != cudaSuccess)
        return QUASAR_ERR_CUDA;
    unsigned int word = 0;
    if (cudaMemcpyFromSymbol(&word, g_quasar_status_word, sizeof(word)) != cudaSuccess)
        return QUASAR_ERR_CUDA;
    if (word == 0) return QUASAR_OK;
    const unsigned int zero = 0;
    if (cudaMemcpyToSymbol(g_quasar_status_word, &zero, sizeof(zero)) != cudaSuccess)
        return QUASAR_ERR_CUDA;
    return (word & kStatusTimeout) ? QUASAR_ERR_TIMEOUT : QUASAR_OK;
}

void quasar_debug_force_timeout(int64_t nanoseconds) { g_force_timeout_ns.store(nanoseconds); }

void quasar_debug_set_stats(unsigned int* device_counters) { g_stats.store(device_counters); }

void quasar_debug_set_hoist(int enable) { g_hoist.store(enable ? 1 : 0); }

const char* quasar_status_string(quasar_status status)
{
    switch (status) {
    case QUASAR_OK: return "QUASAR_OK";
    case QUASAR_ERR_INVALID_ARG: return "QUASAR_ERR_INVALID_ARG";
    case QUASAR_ERR_UNSUPPORTED: return "QUASAR_ERR_UNSUPPORTED";
    case QUASAR_ERR_CUDA: return "QUASAR_ERR_CUDA";
    case QUASAR_ERR_TIMEOUT: return "QUASAR_ERR_TIMEOUT";
    default: return "QUASAR_ERR_UNKNOWN";
    }
}

int quasar_version(void) { return 100; }

}  // extern "C"
