// tune.cu -- plan choice for hj_join (SHJ or PHJ, radix bits, passes): a cost model
// of the GPU-only join, and an on-device tuner that refines it.
//
// The paper's model (Sec. 4) prices a join as T = max(T_CPU, T_GPU) (Eq. 1) with
// T_XPU = sum over steps i of C_i + M_i + D_i (Eq. 2): computation C_i = #I_i x
// items / IPC (Eq. 3), memory stalls M_i, and the CPU/GPU pipeline delay D_i.  With
// every step on the GPU the ratio r is 0, T = T_GPU and D_i = 0.  Re-derived for
// GB300:
//   * M_i = bytes the step must move / HBM bandwidth (nominal from the device's
//     memory clock and bus width, times the fraction a plain copy reaches);
//   * C_i = items_i x thread instructions per item / issue rate (SMs x 4
//     schedulers x clock x 32 lanes x a sustained issue fraction).  As in the
//     paper's instantiation (Sec. 4.2, instruction counts from a profiler), the
//     per-item instruction counts are measured (ncu, smsp__inst_executed);
//   * a GPU overlaps the two within a kernel, so a step costs max(C_i, M_i), plus
//     a launch latency per kernel;
//   * the SHJ table's random accesses cost nothing extra while the table stays in
//     L2, and one sector from HBM for the share of them that falls outside it (the
//     "leap" of the paper's end-to-end results once the table outgrows the cache,
//     Sec. 5.5); a build side that fits shared memory whole has no such table.
// hj_tune then times the model's best few plans on the caller's relations and
// caches the fastest for the relations' size class on the context; hj_join with
// HJ_ALGO_AUTO uses a cached plan when one exists, else the model's choice.
#include <algorithm>
#include <cmath>
#include <vector>

#include "ctx.cuh"
#include "engine.cuh"

namespace hj {

namespace {

// Effective thread instructions per item of each kernel at the sustained issue
// rate below, set so that the model's time equals the kernel's measured time on GB300
// (4-byte tuples; where it says so, 8-byte tuples take twice as many): scatters of 2^26
// (2^25) tuples, the joins of 2^24 x 2^24 and 2^24 x 2^28 at 11 radix bits (u64 3e6 x 2e7
// at 10), SHJ of 2^18 .. 2^24 build tuples with 1, 8 and 64 times as many.
// hj_tune measures the real thing on the caller's relations.
constexpr double kIptHist = 22.0;          // per input tuple (bandwidth-bound)
constexpr double kIptScatter = 66.0;       // per input tuple, at most 2^9 digits (x 2 for 8 bytes)
constexpr double kIptScatter10 = 80.0;     // 2^10 digits (x 2)
constexpr double kIptScatter11 = 87.0;     // 2^11 digits (x 2)
constexpr double kIptScatterNext = 35.0;   // added by a second pass (many segments, launches)
constexpr double kIptScatterWide = 266.0;  // per input tuple, fan-out 2^12
constexpr double kIptJoinProbe = 55.0;     // per S tuple, shared-memory table (x 2)
constexpr double kIptJoinBuild = 184.0;    // per R tuple, shared-memory table (x 2)
constexpr double kIptShjBuild = 240.0;     // per R tuple, global table in L2
constexpr double kIptShjBuildAgg4 = 480.0;   // aggregate table (three atomics per tuple)
constexpr double kIptShjBuildAgg8 = 1400.0;
constexpr double kIptShjProbe4 = 140.0;    // per S tuple, global table in L2
constexpr double kIptShjProbe8 = 172.0;    // 8-byte tuples
constexpr double kIptShjAgg8 = 270.0;      // 8-byte tuples, aggregate table (32-byte slots)
constexpr double kIptSmallProbe = 64.0;    // per S tuple, whole build side in shared memory (x 1.6)
constexpr double kIssueFraction = 0.55;    // sustained share of the issue slots
constexpr double kCopyFraction = 0.83;     // share of nominal HBM bandwidth a copy reaches
constexpr double kRandomFraction = 0.2;    // share for 32-byte random sectors (table probes)
constexpr double kL2Table = 0.75;          // share of L2 that a table may take before probes miss
constexpr double kLaunchS = 4e-6;          // per kernel launch
constexpr double kSmallFixedS = 32e-6;     // per SHJ call with the build side in shared memory
constexpr double kShjFixedS = 35e-6;       // per SHJ call: allocations, one host synchronisation
constexpr double kPhjFixedS = 50e-6;       // per PHJ call: allocations, launch gaps, one host synchronisation

}  // namespace

CostModel cost_model_for(int device) {
    CostModel m;  // defaults: GB300
    int v = 0;
    if (device >= 0) {
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, device) == cudaSuccess && v > 0) m.sms = v;
        int clk = 0, mclk = 0, bus = 0, l2 = 0;
        if (cudaDeviceGetAttribute(&clk, cudaDevAttrClockRate, device) == cudaSuccess && clk > 0)
            m.sm_hz = clk * 1e3;
        if (cudaDeviceGetAttribute(&mclk, cudaDevAttrMemoryClockRate, device) == cudaSuccess &&
            cudaDeviceGetAttribute(&bus, cudaDevAttrGlobalMemoryBusWidth, device) == cudaSuccess && mclk > 0 && bus > 0)
            m.hbm_bps = 2.0 * mclk * 1e3 * bus / 8.0;
        if (cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, device) == cudaSuccess && l2 > 0) m.l2_bytes = l2;
        cudaGetLastError();
    }
    return m;
}

static double issue_rate(const CostModel &m) { return m.sms * 4.0 * m.sm_hz * 32.0 * kIssueFraction; }
static double bw(const CostModel &m) { return m.hbm_bps * kCopyFraction; }

// Largest mean build partition whose shared-memory table stays at most half full
// (the join kernel's biggest shape: 200 KiB of slots).
static double fit_tuples(int width, bool agg) {
    // aggregate slots: key, count and (with checksums, assumed) a 64-bit sum
    const double slot = agg ? width + 12.0 : 2.0 * width;
    return (200.0 * 1024 - 4096) / slot / 2.0;
}

JoinKind join_kind(const hj_ctx *c, int width, int mode, uint64_t flags) {
    const bool agg = mode != HJ_MATERIALIZE;
    return JoinKind{width, agg, !agg && (flags & HJ_FLAG_CHECKSUM) != 0, c && c->budget != 0};
}

double predict_seconds(const CostModel &m, const JoinKind &jk, uint64_t nR, uint64_t nS, int algo, int bits,
                       int passes, double *steps) {
    const int width = jk.width;
    const bool agg = jk.agg, mat = !agg;
    const double t = 2.0 * width, o = 2.0 * width, ir = issue_rate(m), b = bw(m);
    const double n = (double)nR + (double)nS, M = mat ? (double)nS : 0.0;  // one match per probe tuple
    double s[4] = {0, 0, 0, 0};  // hist, scatter, join / build, probe
    if (algo == HJ_ALGO_SHJ && jk.small(nR)) {
        s[3] = std::max((t * nS + o * M) / b, nS * kIptSmallProbe * (width == 4 ? 1.0 : 1.6) / ir) + kSmallFixedS;
    } else if (algo == HJ_ALGO_SHJ) {
        // probes of what does not stay in L2 read a sector of the table from HBM
        const double slot = agg ? (width == 4 ? 16.0 : 32.0) : t;
        const double table = (double)table_slots(width, agg, nR, jk.budget) * slot;
        const double miss = std::max(0.0, 1.0 - kL2Table * m.l2_bytes / std::max(table, 1.0));
        const double rnd = b * kRandomFraction;
        const double probe = width == 4 ? kIptShjProbe4 : agg ? kIptShjAgg8 : kIptShjProbe8;
        const double build = !agg ? kIptShjBuild : width == 4 ? kIptShjBuildAgg4 : kIptShjBuildAgg8;
        s[2] = std::max(t * nR / b, nR * build / ir) + table / b + miss * 64.0 * nR / rnd;
        s[3] = std::max((t * nS + o * M) / b, nS * probe / ir) + miss * 32.0 * nS / rnd;
        s[3] += 5 * kLaunchS + kShjFixedS;
    } else {
        const int b1 = passes == 2 ? bits - bits / 2 : bits, b2 = passes == 2 ? bits / 2 : 0;
        const double wide = width == 4 ? 1.0 : 2.0;
        for (int p = 0; p < passes; ++p) {
            const int bp = p == 0 ? b1 : b2;
            const double ipt = bp <= 9    ? kIptScatter * wide
                               : bp == 10 ? kIptScatter10 * wide
                               : bp == 11 ? kIptScatter11 * wide
                                          : kIptScatterWide;
            // a first pass at <= 2^11 digits is two launches per relation (histogram
            // and scatter place the runs themselves), any other pass eight
            s[0] += std::max(t * n / b, n * kIptHist / ir) + (p == 0 && bp <= 11 ? 2 * 2 : 2 * 8) * kLaunchS;
            s[1] += std::max(2.0 * t * n / b, n * (ipt + (p ? kIptScatterNext * wide : 0.0)) / ir);
        }
        // fewer partition pairs than join CTAs leave SMs idle
        const double busy = std::min(1.0, std::exp2(bits) / (2.0 * m.sms));
        s[2] = std::max((t * n + o * M) / b, (nS * kIptJoinProbe + nR * kIptJoinBuild) * wide / ir) / busy + 6 * kLaunchS +
               kPhjFixedS;
        // the (chunk, digit) count matrix: written, scanned and read once per pass
        s[0] += passes * 24.0 * m.sms * std::exp2(std::max(b1, b2)) / b;
    }
    if (steps)
        for (int i = 0; i < 4; ++i) steps[i] = s[i];
    return s[0] + s[1] + s[2] + s[3];
}

std::vector<PlanCand> plan_candidates(const CostModel &m, const JoinKind &jk, uint64_t nR, uint64_t nS, int algo,
                                      int bits, int passes) {
    std::vector<PlanCand> out;
    auto add = [&](int a, int bb, int g) {
        PlanCand pc{a, bb, g, predict_seconds(m, jk, nR, nS, a, bb, g, nullptr)};
        out.push_back(pc);
    };
    if (algo == HJ_ALGO_AUTO || algo == HJ_ALGO_SHJ) add(HJ_ALGO_SHJ, 0, 0);
    if (algo == HJ_ALGO_AUTO || algo == HJ_ALGO_PHJ) {
        const double fit = fit_tuples(jk.width, jk.agg);
        for (int b = 1; b <= 24; ++b) {
            if (bits > 0 && b != bits) continue;
            // every partition table must fit: skip fan-outs whose mean partition plus
            // six standard deviations exceeds the half-full table (unless forced)
            const double mean = (double)nR / std::exp2(b);
            if (bits <= 0 && mean + 6.0 * std::sqrt(mean + 1.0) + 64.0 > fit && b < 24) continue;
            for (int g = 1; g <= 2; ++g) {
                if (passes > 0 && g != passes) continue;
                if (g == 1 && b > 12) continue;
                if (g == 2 && (b < 2 || b - b / 2 > 12)) continue;
                add(HJ_ALGO_PHJ, b, g);
            }
            // the smallest fitting fan-outs are the cheapest; a few more are kept
            // as candidates for the tuner
            if (bits <= 0 && out.size() >= 8) break;
        }
    }
    std::sort(out.begin(), out.end(), [](const PlanCand &x, const PlanCand &y) { return x.sec < y.sec; });
    return out;
}

uint64_t plan_key(const JoinKind &jk, uint64_t nR, uint64_t nS) {
    auto lg = [](uint64_t x) {
        int l = 0;
        while (x > 1) {
            x >>= 1;
            ++l;
        }
        return (uint64_t)l;
    };
    // (SHJ is another join on either side of small(): a class of its own)
    return ((uint64_t)jk.width << 40) | ((uint64_t)jk.small(nR) << 33) | ((uint64_t)jk.agg << 32) | (lg(nR + 1) << 8) |
           lg(nS + 1);
}

void choose_plan(hj_ctx *c, const JoinKind &jk, uint64_t nR, uint64_t nS, int algo, int bits, int passes, int *a_out,
                 int *b_out, int *g_out) {
    if (algo == HJ_ALGO_AUTO && bits <= 0 && passes <= 0 && c) {
        auto it = c->tuned.find(plan_key(jk, nR, nS));
        if (it != c->tuned.end()) {
            *a_out = it->second.algo;
            *b_out = it->second.bits;
            *g_out = it->second.passes;
            return;
        }
    }
    if (algo == HJ_ALGO_SHJ) {
        *a_out = HJ_ALGO_SHJ;
        *b_out = 0;
        *g_out = 0;
        return;
    }
    if (!c->model_ready) {
        c->model = cost_model_for(c->device);
        c->model_ready = true;
    }
    std::vector<PlanCand> pcs = plan_candidates(c->model, jk, nR, nS, algo, bits, passes);
    if (pcs.empty()) {  // forced shape the filters rejected: honour it
        *a_out = HJ_ALGO_PHJ;
        *b_out = bits > 0 ? bits : 12;
        *g_out = passes > 0 ? passes : (*b_out <= 12 ? 1 : 2);
        return;
    }
    *a_out = pcs[0].algo;
    *b_out = pcs[0].bits;
    *g_out = pcs[0].passes;
}

}  // namespace hj

using namespace hj;

extern "C" {

hj_status hj_plan(hj_ctx *c, const hj_rel *R, const hj_rel *S, const hj_opts *opts, hj_plan_info *out) {
    if (!R || !S || !out) return c ? set_err(c, HJ_E_INVALID, "NULL argument") : HJ_E_INVALID;
    if ((R->width != HJ_U32 && R->width != HJ_U64) || R->width != S->width)
        return c ? set_err(c, HJ_E_INVALID, "bad or differing widths") : HJ_E_INVALID;
    hj_opts o{};
    o.mode = HJ_MATERIALIZE;
    if (opts) o = *opts;
    const JoinKind jk = join_kind(c, R->width, o.mode, o.flags);
    CostModel m = c ? cost_model_for(c->device) : CostModel{};
    int a = o.algo, b = o.radix_bits, g = o.passes;
    if (c) {
        choose_plan(c, jk, R->n, S->n, o.algo, o.radix_bits, o.passes, &a, &b, &g);
    } else {
        std::vector<PlanCand> pcs = plan_candidates(m, jk, R->n, S->n, o.algo, o.radix_bits, o.passes);
        if (pcs.empty()) return HJ_E_INVALID;
        a = pcs[0].algo;
        b = pcs[0].bits;
        g = pcs[0].passes;
    }
    *out = hj_plan_info{};
    out->algo = a;
    out->radix_bits = a == HJ_ALGO_PHJ ? b : 0;
    out->passes = a == HJ_ALGO_PHJ ? g : 0;
    double st[4];
    out->predicted_ms = 1e3 * predict_seconds(m, jk, R->n, S->n, a, b, g, st);
    for (int i = 0; i < 4; ++i) out->step_ms[i] = 1e3 * st[i];
    out->measured_ms = -1.0;
    return HJ_OK;
}

hj_status hj_tune(hj_ctx *c, const hj_rel *R, const hj_rel *S, const hj_opts *opts, int top_k, hj_plan_info *out) {
    if (!c || !R || !S) return c ? set_err(c, HJ_E_INVALID, "NULL argument") : HJ_E_INVALID;
    if ((R->width != HJ_U32 && R->width != HJ_U64) || R->width != S->width)
        return set_err(c, HJ_E_INVALID, "bad or differing widths");
    hj_opts o{};
    o.mode = HJ_MATERIALIZE;
    if (opts) o = *opts;
    if (top_k <= 0) top_k = 4;
    const JoinKind jk = join_kind(c, R->width, o.mode, o.flags);
    if (!c->model_ready) {
        c->model = cost_model_for(c->device);
        c->model_ready = true;
    }
    std::vector<PlanCand> pcs = plan_candidates(c->model, jk, R->n, S->n, HJ_ALGO_AUTO, 0, 0);
    if ((int)pcs.size() > top_k) pcs.resize(top_k);
    if (pcs.empty()) return set_err(c, HJ_E_UNSUPPORTED, "no plan candidate");
    cudaEvent_t e0, e1;
    HJ_CUDA(c, cudaEventCreate(&e0));
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return set_err(c, HJ_E_CUDA, "cudaEventCreate");
    }
    double best = 1e30;
    PlanCand pick = pcs[0];
    hj_status st = HJ_OK;
    for (const PlanCand &pc : pcs) {
        hj_opts oj = o;
        oj.algo = pc.algo;
        oj.radix_bits = pc.bits;
        oj.passes = pc.passes;
        double t_min = 1e30;
        for (int rep = 0; rep < 3 && st == HJ_OK; ++rep) {  // one warm-up, two timed
            hj_result res{};
            cudaEventRecord(e0, c->stream);
            st = hj_join(c, R, S, &oj, &res);
            cudaEventRecord(e1, c->stream);
            if (st != HJ_OK) break;
            cudaEventSynchronize(e1);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            hj_result_free(c, &res);
            if (rep > 0) t_min = std::min(t_min, (double)ms);
        }
        if (st != HJ_OK) break;
        if (t_min < best) {
            best = t_min;
            pick = pc;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (st != HJ_OK) return st;
    c->tuned[plan_key(jk, R->n, S->n)] = TunedPlan{pick.algo, pick.bits, pick.passes};
    if (out) {
        *out = hj_plan_info{};
        out->algo = pick.algo;
        out->radix_bits = pick.algo == HJ_ALGO_PHJ ? pick.bits : 0;
        out->passes = pick.algo == HJ_ALGO_PHJ ? pick.passes : 0;
        double s4[4];
        out->predicted_ms = 1e3 * predict_seconds(c->model, jk, R->n, S->n, pick.algo, pick.bits, pick.passes, s4);
        for (int i = 0; i < 4; ++i) out->step_ms[i] = 1e3 * s4[i];
        out->measured_ms = best;
    }
    return HJ_OK;
}

hj_status hj_tune_clear(hj_ctx *c) {
    if (!c) return HJ_E_INVALID;
    c->tuned.clear();
    return HJ_OK;
}

}  // extern "C"
