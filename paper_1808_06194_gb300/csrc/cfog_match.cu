// The FFT matcher's host side: kernel variants, the queue of the batched
// launch, tuned plans, and the C entry points.  The kernel itself is in
// cfog_match_fft.cuh, one translation unit per geometry.
#include "cfog_internal.cuh"
#include "cfog_match_common.cuh"
#include "cfog_plan.cuh"

#include <cuda.h>

#include <algorithm>
#include <array>
#include <climits>
#include <cstdint>
#include <cstring>
#include <map>
#include <mutex>
#include <vector>

namespace cfog {
namespace {

constexpr int kNumVariants = 4;

// A kernel variant: the geometry that runs it, the bound on the FFT plane
// P_y * P_x, and its plan table in that geometry.
struct VariantInfo {
    MatchKernel (*kernel)();
    MatchKernel (*tall)();   // one CTA of twice the threads per SM (few CPs), same results
    int per_sm;    // CTAs per SM
    int maxe;
    int table;
};
const VariantInfo &variant_info(int v) {
    static const VariantInfo t[kNumVariants] = {
        {match_kernel_wide, match_kernel_wide_tall, 2, 16384, 0},   // planes up to 128 x 128 (one CTA per SM above 109 KB)
        {match_kernel_pair, match_kernel_pair_tall, 2, 9216, 0},    // planes up to 96 x 96
        {match_kernel_trio, nullptr, 3, 7680, 0},    // three CPs per SM
        {match_kernel_pair, match_kernel_pair_tall, 2, 9216, 1},    // pair geometry with plans of its own
    };
    return t[v - 1];
}

// An SM holds 228 KB of shared memory: of a CTA's share, 1 KB is reserved and
// about 4 KB are static.
PlanLimits variant_limits(int v) {
    const VariantInfo &i = variant_info(v);
    return PlanLimits{i.maxe, i.per_sm >= 3 ? 71 * 1024 : 109 * 1024,
                      fft_tmem_cols(i.per_sm) / (kFftThreads / 128), kFftThreads};
}

// Queue order for the persistent kernel: CPs sorted by search-window side
// N + 2r, largest first (a proxy of their FFT cost), so that the expensive CPs
// start early and the cheap ones fill the tail.  One CTA: histogram over the
// window side, exclusive scan, scatter.  Also resets the queue counter.
constexpr int kOrderThreads = 1024;
constexpr int kSideMax = kMaxFft + 64;

__global__ void __launch_bounds__(kOrderThreads)
order_queue_kernel(const int *__restrict__ tmpl, const int *__restrict__ radius, int n,
                   int *__restrict__ counter, int *__restrict__ order) {
    __shared__ int hist[kSideMax + 2];
    for (int i = threadIdx.x; i < kSideMax + 2; i += kOrderThreads) hist[i] = 0;
    if (threadIdx.x == 0) *counter = 0;
    __syncthreads();
    auto key = [&](int i) {
        const int side = tmpl[i] + 2 * radius[i];
        const int s = side < 0 ? 0 : (side > kSideMax ? kSideMax : side);
        return kSideMax - s;   // descending side
    };
    for (int i = threadIdx.x; i < n; i += kOrderThreads) atomicAdd(&hist[key(i)], 1);
    __syncthreads();
    if (threadIdx.x == 0) {
        int acc = 0;
        for (int b = 0; b <= kSideMax; ++b) {
            const int c = hist[b];
            hist[b] = acc;
            acc += c;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kOrderThreads) order[atomicAdd(&hist[key(i)], 1)] = i;
}

// ------------------------------------------------------------------- host --
// Host mirror of the tuned-plan tables and the AUTO variant choices.
struct Tuning {
    std::mutex mu;
    int32_t plan[kNumVariants][kMaxFft + 1][kMaxRadius + 1] = {};
    int count[kNumVariants] = {};
    unsigned gen = 1;   // bumped by every change of the plan tables
    std::map<std::array<int, 4>, int> auto_variant;   // (m, tmpl_max, radius_max, precision)
};
Tuning &tuning() {
    static Tuning t;
    return t;
}

// Write n entries of variant v's plan table on the current device, in every
// kernel that runs the variant.
cfog_status write_plans(int v, size_t offset, const int32_t *src, size_t n) {
    const VariantInfo &info = variant_info(v);
    cfog_status st = info.kernel().write_plans(info.table, offset, src, n);
    if (st == CFOG_OK && info.tall) st = info.tall().write_plans(info.table, offset, src, n);
    return st;
}

// Tuned plan code of (variant, N, r) for m, or -1.
int tuned_code(int v, int N, int r, int m) {
    const int e = tuning().plan[v - 1][N][r];
    return (e != 0 && (e >> 16) == m) ? (e & 0xffff) - 1 : -1;
}

// Two CTAs hold 2 x 256 tensor-memory columns: a launch whose planes would let
// more of them share an SM reserves enough shared memory that they do not.
constexpr int kMinSmem = 77 * 1024;

constexpr int kTallCps = 2;
constexpr int kTallSmem = 222 * 1024;   // of the 227 KB a CTA may use, 5 KB for static memory

// Largest dynamic shared memory over every class (N <= tmpl_max, r <= radius_max)
// of a launch, for CTAs of kFftThreads and of kFftThreadsTall (-1: a class has no plan).
struct SmemNeed {
    int normal, tall;
    void add(const MatchPlan &p, int N, int r) {
        normal = std::max(normal, plan_smem_bytes(p, N, r, kFftThreads, p.G));
        tall = std::max(tall, plan_smem_bytes(p, N, r, kFftThreadsTall, p.G));
    }
};

// Over the cost-model plan and any tuned plan alike (a device whose table was not
// written uses the cost model).  The search over the cost model is made once per
// bounds; a change of the tuned plans costs a look through the table only.
SmemNeed max_plan_smem(int v, int tmpl_max, int radius_max, int m) {
    struct Entry {
        SmemNeed model, all;
        unsigned gen;
    };
    static std::map<std::array<int, 4>, Entry> cache;   // guarded by the tuning's mutex
    Tuning &T = tuning();
    std::lock_guard<std::mutex> lock(T.mu);
    const PlanLimits lim = variant_limits(v);
    auto [it, fresh] = cache.try_emplace({v, tmpl_max, radius_max, m}, Entry{{0, 0}, {0, 0}, 0});
    Entry &e = it->second;
    if (fresh) {
        for (int N = 1; N <= tmpl_max && e.model.normal >= 0; ++N)
            for (int r = 0; r <= radius_max; ++r) {
                MatchPlan p;
                if (!make_plan_host(N, r, m, lim, &p)) {
                    e.model = SmemNeed{-1, -1};
                    break;
                }
                e.model.add(p, N, r);
            }
    }
    if (e.gen != T.gen) {
        e.gen = T.gen;
        e.all = e.model;
        for (int N = 1; N <= tmpl_max && T.count[v - 1] > 0 && e.model.normal >= 0; ++N)
            for (int r = 0; r <= radius_max; ++r) {
                MatchPlan p;
                const int t = T.plan[v - 1][N][r];
                if (t != 0 && (t >> 16) == m && plan_for_code(N, r, m, (t & 0xffff) - 1, lim, &p) >= 0)
                    e.all.add(p, N, r);
            }
    }
    return e.all;
}

// Kernel, shared memory and plan table of a launch of variant v.  One CTA of
// twice the threads per SM, transforming twice the planes at once where they
// fit, runs a launch of at most kTallCps CPs per SM: every CP then has an SM to
// itself and the queue keeps balancing, where two CTAs per SM would start all
// CPs at once and leave the largest ones sharing their SMs (256 CPs of N
// 64/96, r 10..20 take 0.35 instead of 0.43 ms, with 36 channels 1.59 instead
// of 2.18 ms, 304 CPs 0.41 instead of 0.45; 400 CPs take 0.44 with two CTAs).
// The same for any launch whose planes leave an SM one CTA only.
cfog_status prepare(int v, MatchArgs *a, MatchKernel *K) {
    const VariantInfo &info = variant_info(v);
    *K = info.kernel();
    const SmemNeed need = max_plan_smem(v, a->tmpl_max, a->radius_max, a->m);
    int smem = need.normal;
    if (info.tall && smem > 0 && (a->n <= kTallCps * sm_count() || smem > variant_limits(v).smem_cap)) {
        *K = info.tall();
        smem = std::max(need.tall, kTallSmem);
    }
    if (smem <= 0) {
        set_error("cfog_match: no FFT plan for tmpl_max %d radius_max %d", a->tmpl_max, a->radius_max);
        return CFOG_E_INVAL;
    }
    smem = std::max(smem, info.per_sm == 2 ? kMinSmem : 16 * 1024);
    a->lim = variant_limits(v);
    a->smem_bytes = smem;
    {
        // the kernel consults the variant's tuned-plan table if it has entries
        Tuning &T = tuning();
        std::lock_guard<std::mutex> lock(T.mu);
        a->plan_table = T.count[v - 1] > 0 ? info.table : -1;
    }
    return ensure_dynamic_smem(K->fn, smem, "cfog_match");
}

// The variant AUTO runs for a launch class: the autotuner's choice if one is
// recorded, else WIDE (it plans every class with the fewest template blocks).
int auto_variant(int m, int tmpl_max, int radius_max, int precision) {
    Tuning &T = tuning();
    std::lock_guard<std::mutex> lock(T.mu);
    auto it = T.auto_variant.find({m, tmpl_max, radius_max, precision});
    return it != T.auto_variant.end() ? it->second : CFOG_MATCH_VARIANT_WIDE;
}

cfog_status check_common(int32_t n, const void *cps, const void *tmpl, const void *radius,
                         const void *out, int32_t tmpl_max, int32_t radius_max, int32_t m,
                         int32_t precision, int32_t variant) {
    CFOG_REQUIRE(n >= 0, "cfog_match: n = %d < 0", n);
    CFOG_REQUIRE(n == 0 || (cps && tmpl && radius && out), "cfog_match: null CP array");
    CFOG_REQUIRE(m >= 1 && m <= 64, "cfog_match: m = %d outside [1, 64]", m);
    CFOG_REQUIRE(tmpl_max >= 1 && tmpl_max <= kMaxFft, "cfog_match: tmpl_max %d outside [1, %d]",
                 tmpl_max, kMaxFft);
    CFOG_REQUIRE(radius_max >= 0 && radius_max <= 32, "cfog_match: radius_max %d outside [0, 32]",
                 radius_max);
    CFOG_REQUIRE(n <= (1 << 30), "cfog_match: n too large");
    CFOG_REQUIRE(variant >= 0 && variant <= 4, "cfog_match: unknown variant %d", variant);
    CFOG_REQUIRE(precision == CFOG_PREC_FP32_FFT || precision == CFOG_PREC_BF16_DIRECT,
                 "cfog_match: unknown precision %d", precision);
    if (precision == CFOG_PREC_BF16_DIRECT && tmpl_max > 128) {
        set_error("cfog_match: BF16 direct precision supports templates up to 128 (tmpl_max %d)",
                  tmpl_max);
        return CFOG_E_UNSUPPORTED;
    }
    return CFOG_OK;
}

}  // namespace
}  // namespace cfog

using namespace cfog;

extern "C" cfog_status cfog_match(const cfog_features *ref, const cfog_features *sen,
                                  const cfog_point *cps_dev, int32_t n, const int32_t *tmpl_dev,
                                  const int32_t *radius_dev, int32_t tmpl_max, int32_t radius_max,
                                  const cfog_point *prior_dev, int32_t precision,
                                  cfog_match_result *out_dev, float *surface_dev, void *stream) {
    CFOG_TRACE("cfog_match");
    CFOG_REQUIRE(ref && sen, "cfog_match: ref and sen must be non-NULL");
    CFOG_REQUIRE(ref->m == sen->m, "cfog_match: channel counts %d/%d", ref->m, sen->m);
    cfog_status st = check_common(n, cps_dev, tmpl_dev, radius_dev, out_dev, tmpl_max, radius_max,
                                  ref->m, precision, 0);
    if (st != CFOG_OK || n == 0) return st;
    CFOG_REQUIRE(ref->data && sen->data && sen->sqnorm, "cfog_match: null feature pointer");

    MatchArgs a{};
    a.ref = ref->data;
    a.ref_sq = ref->sqnorm;
    a.ref_h = ref->h;
    a.ref_w = ref->w;
    a.ref_rp = ref->row_pitch;
    a.ref_pp = ref->plane_pitch;
    a.sen = sen->data;
    a.sen_sq = sen->sqnorm;
    a.sen_h = sen->h;
    a.sen_w = sen->w;
    a.sen_rp = sen->row_pitch;
    a.sen_pp = sen->plane_pitch;
    a.jobs = nullptr;
    a.job_of_cp = nullptr;
    a.n_jobs = 0;
    a.m = ref->m;
    a.cps = cps_dev;
    a.tmpl = tmpl_dev;
    a.radius = radius_dev;
    a.prior = prior_dev;
    a.n = n;
    a.out = out_dev;
    a.surface = surface_dev;
    a.surf_side = 2 * radius_max + 1;
    a.tmpl_max = tmpl_max;
    a.radius_max = radius_max;
    a.plan_table = -1;
    if (precision == CFOG_PREC_BF16_DIRECT) return launch_bf16_direct(a, nullptr, nullptr, as_stream(stream));
    MatchKernel K;
    st = prepare(CFOG_MATCH_VARIANT_WIDE, &a, &K);
    if (st != CFOG_OK) return st;
    return K.launch(a, nullptr, nullptr, n, a.smem_bytes, as_stream(stream));
}

extern "C" size_t cfog_match_workspace_bytes(int32_t n) {
    if (n < 0) return 0;
    return 256 + (size_t)n * sizeof(int32_t);
}

extern "C" cfog_status cfog_match_batched(const cfog_job *jobs_dev, int32_t n_jobs,
                                          const int32_t *job_of_cp_dev, const cfog_point *cps_dev,
                                          int32_t n, const int32_t *tmpl_dev,
                                          const int32_t *radius_dev, int32_t tmpl_max,
                                          int32_t radius_max, int32_t m,
                                          const cfog_point *prior_dev, int32_t precision,
                                          int32_t variant, cfog_match_result *out_dev,
                                          void *workspace_dev, size_t workspace_bytes,
                                          void *stream) {
    CFOG_TRACE("cfog_match_batched");
    cfog_status st = check_common(n, cps_dev, tmpl_dev, radius_dev, out_dev, tmpl_max, radius_max,
                                  m, precision, variant);
    if (st != CFOG_OK || n == 0) return st;
    CFOG_REQUIRE(jobs_dev && n_jobs >= 1, "cfog_match_batched: empty job table");
    CFOG_REQUIRE(workspace_dev, "cfog_match_batched: workspace is NULL");
    if (workspace_bytes < cfog_match_workspace_bytes(n)) {
        set_error("cfog_match_batched: workspace %zu bytes < %zu needed", workspace_bytes,
                  cfog_match_workspace_bytes(n));
        return CFOG_E_NOMEM;
    }
    CFOG_REQUIRE(((uintptr_t)workspace_dev & 255) == 0,
                 "cfog_match_batched: workspace must be 256-byte aligned");
    MatchArgs a{};
    a.jobs = jobs_dev;
    a.job_of_cp = job_of_cp_dev;
    a.n_jobs = n_jobs;
    a.m = m;
    a.cps = cps_dev;
    a.tmpl = tmpl_dev;
    a.radius = radius_dev;
    a.prior = prior_dev;
    a.n = n;
    a.out = out_dev;
    a.surface = nullptr;
    a.surf_side = 2 * radius_max + 1;
    a.tmpl_max = tmpl_max;
    a.radius_max = radius_max;
    a.plan_table = -1;
    const int v = variant == 0 ? auto_variant(m, tmpl_max, radius_max, precision) : variant;
    int *counter = static_cast<int *>(workspace_dev);
    int *order = reinterpret_cast<int *>(static_cast<char *>(workspace_dev) + 256);
    cudaStream_t s = as_stream(stream);
    if (precision == CFOG_PREC_BF16_DIRECT) {
        order_queue_kernel<<<1, kOrderThreads, 0, s>>>(tmpl_dev, radius_dev, n, counter, order);
        st = check_launch("cfog_match_batched: order launch");
        if (st != CFOG_OK) return st;
        return launch_bf16_direct(a, counter, order, s);
    }
    MatchKernel K;
    st = prepare(v, &a, &K);
    if (st != CFOG_OK) return st;
    int per_sm = 0;
    st = persistent_ctas_per_sm(K.fn, K.threads, a.smem_bytes, &per_sm, "cfog_match_batched: occupancy");
    if (st != CFOG_OK) return st;
    // CTAs hold their tensor-memory columns for life: at most 512 / columns per SM
    per_sm = std::min(per_sm, 512 / K.tmem_cols);
    const int grid = (int)std::min<long long>((long long)n, (long long)sm_count() * per_sm);
    order_queue_kernel<<<1, kOrderThreads, 0, s>>>(tmpl_dev, radius_dev, n, counter, order);
    st = check_launch("cfog_match_batched: order launch");
    if (st != CFOG_OK) return st;
    return K.launch(a, counter, order, grid, a.smem_bytes, s);
}

// Plan of (N, r, m) in variant v: the tuned plan if one is recorded (host
// mirror), else the cost model's.
static bool plan_in_use(int tmpl, int radius, int m, int v, MatchPlan *p) {
    const PlanLimits lim = variant_limits(v);
    int code;
    {
        Tuning &T = tuning();
        std::lock_guard<std::mutex> lock(T.mu);
        code = tuned_code(v, tmpl, radius, m);
    }
    if (code >= 0 && plan_for_code(tmpl, radius, m, code, lim, p) >= 0) return true;
    return make_plan_host(tmpl, radius, m, lim, p);
}

static void plan_row(const MatchPlan &p, int v, int N, int r, int32_t *out8) {
    out8[0] = p.y.nb;
    out8[1] = p.x.nb;
    out8[2] = p.y.P;
    out8[3] = p.x.P;
    out8[4] = p.y.bs;
    out8[5] = p.x.bs;
    out8[6] = (p.y.B > 1 ? 2 : 1) + (p.x.B > 1 ? 2 : 1);
    out8[7] = plan_smem_bytes(p, N, r, variant_limits(v).threads, p.G);
}

#define CFOG_CHECK_CLASS(who, tmpl, radius, m)                                                \
    CFOG_REQUIRE(tmpl >= 1 && tmpl <= kMaxFft && radius >= 0 && radius <= 32 && m >= 1 && m <= 64, \
                 who ": (N=%d, r=%d, m=%d) outside the supported range", tmpl, radius, m)

extern "C" cfog_status cfog_plan_info(int32_t tmpl, int32_t radius, int32_t m, int32_t variant,
                                      int32_t *out8) {
    CFOG_REQUIRE(out8, "cfog_plan_info: out8 is NULL");
    CFOG_CHECK_CLASS("cfog_plan_info", tmpl, radius, m);
    CFOG_REQUIRE(variant >= 0 && variant <= 4, "cfog_plan_info: unknown variant %d", variant);
    const int v = variant == 0 ? CFOG_MATCH_VARIANT_WIDE : variant;
    MatchPlan p;
    CFOG_REQUIRE(plan_in_use(tmpl, radius, m, v, &p), "cfog_plan_info: no plan");
    plan_row(p, v, tmpl, radius, out8);
    return CFOG_OK;
}

extern "C" cfog_status cfog_plan_candidates(int32_t tmpl, int32_t radius, int32_t m,
                                            int32_t variant, int32_t max_out, int32_t *out9,
                                            int32_t *n_out) {
    CFOG_REQUIRE(out9 && n_out, "cfog_plan_candidates: null output");
    CFOG_CHECK_CLASS("cfog_plan_candidates", tmpl, radius, m);
    CFOG_REQUIRE(variant >= 1 && variant <= 4, "cfog_plan_candidates: variant %d not in 1..4",
                 variant);
    CFOG_REQUIRE(max_out >= 0, "cfog_plan_candidates: max_out = %d", max_out);
    std::vector<std::pair<long long, int>> c;
    for (int code = 0; code < kPlanCodes; ++code) {
        MatchPlan p;
        const long long cost = plan_for_code(tmpl, radius, m, code, variant_limits(variant), &p);
        if (cost >= 0) c.emplace_back(cost, code);
    }
    std::sort(c.begin(), c.end());
    // distinct plans only (two codes can name the same plan when a block
    // split degenerates), in order of the model's cost
    int n = 0;
    std::vector<MatchPlan> seen;
    for (const auto &e : c) {
        if (n >= max_out) break;
        MatchPlan p;
        plan_for_code(tmpl, radius, m, e.second, variant_limits(variant), &p);
        bool dup = false;
        for (const MatchPlan &q : seen)
            dup = dup || (q.y.nb == p.y.nb && q.x.nb == p.x.nb && q.y.P == p.y.P && q.x.P == p.x.P);
        if (dup) continue;
        seen.push_back(p);
        out9[9 * n] = e.second;
        plan_row(p, variant, tmpl, radius, out9 + 9 * n + 1);
        ++n;
    }
    *n_out = n;
    return CFOG_OK;
}

extern "C" cfog_status cfog_match_set_plan(int32_t variant, int32_t m, int32_t tmpl,
                                           int32_t radius, int32_t code) {
    CFOG_TRACE("cfog_match_set_plan");
    CFOG_CHECK_CLASS("cfog_match_set_plan", tmpl, radius, m);
    CFOG_REQUIRE(variant >= 1 && variant <= 4, "cfog_match_set_plan: variant %d not in 1..4",
                 variant);
    MatchPlan p;
    CFOG_REQUIRE(code == -1 || plan_for_code(tmpl, radius, m, code, variant_limits(variant), &p) >= 0,
                 "cfog_match_set_plan: code %d names no feasible plan for (N=%d, r=%d, m=%d)", code,
                 tmpl, radius, m);
    const int32_t e = code < 0 ? 0 : (int32_t)((m << 16) | (code + 1));
    Tuning &T = tuning();
    std::lock_guard<std::mutex> lock(T.mu);
    cfog_status st = write_plans(variant, (size_t)tmpl * (kMaxRadius + 1) + radius, &e, 1);
    if (st != CFOG_OK) return st;
    int32_t &h = T.plan[variant - 1][tmpl][radius];
    T.count[variant - 1] += (e != 0) - (h != 0);
    h = e;
    ++T.gen;
    return CFOG_OK;
}

extern "C" cfog_status cfog_match_set_auto_variant(int32_t m, int32_t tmpl_max,
                                                   int32_t radius_max, int32_t precision,
                                                   int32_t variant) {
    CFOG_CHECK_CLASS("cfog_match_set_auto_variant", tmpl_max, radius_max, m);
    CFOG_REQUIRE(variant >= 0 && variant <= 4, "cfog_match_set_auto_variant: variant %d", variant);
    CFOG_REQUIRE(precision == CFOG_PREC_FP32_FFT || precision == CFOG_PREC_BF16_DIRECT,
                 "cfog_match_set_auto_variant: unknown precision %d", precision);
    Tuning &T = tuning();
    std::lock_guard<std::mutex> lock(T.mu);
    const std::array<int, 4> key{m, tmpl_max, radius_max, precision};
    if (variant == 0)
        T.auto_variant.erase(key);
    else
        T.auto_variant[key] = variant;
    return CFOG_OK;
}

extern "C" int32_t cfog_match_auto_variant(int32_t m, int32_t tmpl_max, int32_t radius_max,
                                           int32_t precision) {
    return auto_variant(m, tmpl_max, radius_max, precision);
}

extern "C" cfog_status cfog_match_clear_tuning(void) {
    CFOG_TRACE("cfog_match_clear_tuning");
    Tuning &T = tuning();
    std::lock_guard<std::mutex> lock(T.mu);
    static const int32_t zeros[(kMaxFft + 1) * (kMaxRadius + 1)] = {};
    for (int v = 1; v <= kNumVariants; ++v) {
        cfog_status st = write_plans(v, 0, zeros, sizeof(zeros) / sizeof(zeros[0]));
        if (st != CFOG_OK) return st;
    }
    std::memset(T.plan, 0, sizeof(T.plan));
    for (int &c : T.count) c = 0;
    T.auto_variant.clear();
    ++T.gen;
    return CFOG_OK;
}

// ------------------------------------------------ allocation-free variant --
// Batched matching for callers that cannot allocate device memory.  The
// queue scratch of cfog_match_batched (a counter and the order of up to
// kNoAllocMaxCps CPs) lives in this file-scope array instead of a caller
// workspace.  Every GPU that loads the library holds it until the process
// exits.  In host code the symbol is only a host-side stand-in: the device
// address comes from cudaGetSymbolAddress, looked up with the device current.
// The address belongs to one CUDA context (a device reset, or a second
// context on the same device, loads the module again elsewhere), so the
// cached address is keyed by the driver's context ID, which is never reused
// within a process; a call from another context looks the address up again.
namespace cfog {
namespace {
constexpr int kNoAllocMaxCps = 65536;
constexpr size_t kNoAllocBytes = 256 + (size_t)kNoAllocMaxCps * sizeof(int32_t);
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

struct NoAllocSlot {
    void *ptr;
    unsigned long long ctx_id;   // 0: unknown, never matches
};
std::mutex g_noalloc_mu;
NoAllocSlot g_noalloc[64] = {};

// ID of the current CUDA context (0 if there is none or the driver calls are
// unavailable).  The two driver functions are resolved through the runtime,
// so the library does not link libcuda itself.
unsigned long long current_ctx_id() {
    using GetCurrentFn = CUresult (*)(CUcontext *);
    using GetIdFn = CUresult (*)(CUcontext, unsigned long long *);
    static GetCurrentFn get_current = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess || q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<GetCurrentFn>(f);
    }();
    static GetIdFn get_id = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess || q != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<GetIdFn>(f);
    }();
    CUcontext ctx = nullptr;
    unsigned long long id = 0;
    if (!get_current || !get_id || get_current(&ctx) != CUDA_SUCCESS || !ctx) return 0;
    if (get_id(ctx, &id) != CUDA_SUCCESS) return 0;
    return id;
}

// Device address of g_noalloc_scratch in the current context (looked up on
// the first call made in that context).
cfog_status noalloc_scratch(void **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return check_cuda(e, "cfog_match_batched_noalloc: cudaGetDevice");
    if (dev < 0 || dev >= 64) {
        set_error("cfog_match_batched_noalloc: device %d outside the supported range [0, 64)", dev);
        return CFOG_E_UNSUPPORTED;
    }
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    const unsigned long long id = current_ctx_id();
    if (g_noalloc[dev].ptr && id != 0 && g_noalloc[dev].ctx_id == id) {
        *out = g_noalloc[dev].ptr;
        return CFOG_OK;
    }
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p)
        return check_cuda(e != cudaSuccess ? e : cudaErrorInvalidSymbol,
                          "cfog_match_batched_noalloc: cudaGetSymbolAddress");
    // the lookup makes the device's primary context current if none was
    g_noalloc[dev].ptr = p;
    g_noalloc[dev].ctx_id = id != 0 ? id : current_ctx_id();
    *out = p;
    return CFOG_OK;
}
}  // namespace
}  // namespace cfog

extern "C" int32_t cfog_match_batched_noalloc_max_cps(void) { return kNoAllocMaxCps; }

extern "C" cfog_status cfog_match_batched_noalloc(const cfog_job *jobs_dev, int32_t n_jobs,
                                                  const int32_t *job_of_cp_dev,
                                                  const cfog_point *cps_dev, int32_t n,
                                                  const int32_t *tmpl_dev,
                                                  const int32_t *radius_dev, int32_t tmpl_max,
                                                  int32_t radius_max, int32_t m,
                                                  const cfog_point *prior_dev, int32_t precision,
                                                  int32_t variant, cfog_match_result *out_dev,
                                                  void *stream) {
    CFOG_TRACE("cfog_match_batched_noalloc");
    if (n > kNoAllocMaxCps) {
        set_error("cfog_match_batched_noalloc: n = %d CPs exceeds the built-in scratch for %d CPs;"
                  " split the batch or use cfog_match_batched with a workspace",
                  n, kNoAllocMaxCps);
        return CFOG_E_INVAL;
    }
    void *scratch = nullptr;
    if (n > 0) {
        cfog_status st = noalloc_scratch(&scratch);
        if (st != CFOG_OK) return st;
    }
    return cfog_match_batched(jobs_dev, n_jobs, job_of_cp_dev, cps_dev, n, tmpl_dev, radius_dev,
                              tmpl_max, radius_max, m, prior_dev, precision, variant, out_dev,
                              scratch, kNoAllocBytes, stream);
}
