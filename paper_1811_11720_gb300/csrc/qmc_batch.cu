// qmc_batch.cu -- qmc_batch_sums / qmc_batch_autotune: many integrals in one launch.
#include <cuda_runtime.h>

#include <algorithm>
#include <new>
#include <cstdint>
#include <cstring>
#include <vector>

#include "qmc_gb300.h"
#include "qmc_hostutil.h"
#include "qmc_internal.h"
#include "qmc_reduce.cuh"

using namespace qmc;
using namespace qmc::host;

namespace qmc {

// Block (q, component, k): fold item q's tiles for shift k.
__global__ void __launch_bounds__(kRedThreads)
    batch_reduce_kernel(const Integral *items, int m, int cplx, const double *partials,
                        double *sums) {
    const int per_item = m * (cplx ? 2 : 1);
    const int q = blockIdx.x / per_item;
    const int rest = blockIdx.x % per_item;
    const int comp = rest / m, k = rest % m;
    const uint64_t tiles = items[q].tiles;
    const SumPair acc =
        fold_tiles(partials + items[q].partial_off + 2 * (uint64_t)comp * tiles * m, tiles, m, k);
    if (threadIdx.x == 0) {
        double *o = sums + (size_t)items[q].slot * 4 * m + 2 * (size_t)comp * m + 2 * k;
        o[0] = acc.hi;
        o[1] = acc.lo;
    }
}

// One warp per item and component: Qbar and sigma (Eq. (lattice), Eq. (lattice-error)).  (One
// thread per item, its m divisions one after the other, took 33 us for 64 items.)
constexpr int kBatchFinThreads = 128;

__global__ void __launch_bounds__(kBatchFinThreads)
    batch_finalize_kernel(const Integral *__restrict__ items, int count, int m, int cplx,
                          const double *__restrict__ sums, double *__restrict__ results) {
    const int ncomp = cplx ? 2 : 1;
    const int w = (blockIdx.x * kBatchFinThreads + threadIdx.x) >> 5;
    const int q = w / ncomp, comp = w - q * ncomp;
    if (q >= count) return;
    const double dn = (double)items[q].n;
    const size_t slot = items[q].slot;
    const double *__restrict__ sc = sums + slot * 4 * m + 2 * (size_t)comp * m;
    double *res = results + 4 * slot;
    shift_stats(m, [&](int k) { return (sc[2 * k] + sc[2 * k + 1]) / dn; }, res + 2 * comp);
    if (!cplx && (threadIdx.x & 31) < 2) res[2 + (threadIdx.x & 31)] = 0.0;
}

cudaError_t launch_batch(int family, int tkind, int max_d, const Integral *items, const uint64_t *tb,
                         int count, uint64_t first_tile, uint64_t end_tile, int m, int spb, int chain,
                         double *partials, unsigned long long *counters, cudaStream_t s) {
    LatticeLaunch lp{};
    lp.items = items;
    lp.tile_begin = tb;
    lp.count = count;
    lp.m = m;
    lp.spb = spb;
    lp.chain = chain;
    lp.first_tile = first_tile;
    lp.end_tile = end_tile;
    lp.partials = partials;
    lp.counters = counters;
    return launch_sums_any(family, tkind, lp, max_d, s);
}

bool batch_family_supported(int fam) {
    return fam == QMC_GENZ_OSCILLATORY || fam == QMC_GENZ_PRODUCT_PEAK || fam == QMC_GENZ_CORNER_PEAK ||
           fam == QMC_GENZ_GAUSSIAN || fam == QMC_SECTOR || fam == QMC_FEYNMAN;
}

cudaError_t launch_batch_reduce(const Integral *d_items, int count, int m, int cplx,
                                const double *partials, double *sums, cudaStream_t s) {
    const uint64_t blocks = (uint64_t)count * m * (cplx ? 2 : 1);
    batch_reduce_kernel<<<(unsigned)blocks, kRedThreads, 0, s>>>(d_items, m, cplx, partials, sums);
    return cudaGetLastError();
}

cudaError_t launch_batch_finalize(const Integral *d_items, int count, int m, int cplx,
                                  const double *sums, double *results, cudaStream_t s) {
    const int per = kBatchFinThreads / 32, warps = count * (cplx ? 2 : 1);
    batch_finalize_kernel<<<(warps + per - 1) / per, kBatchFinThreads, 0, s>>>(d_items, count, m, cplx, sums, results);
    return cudaGetLastError();
}

int fill_batch_item(Integral &it, const qmc_batch_item &b, int m, int spb, uint32_t Lcfg, int fam) {
    int st = check_integrand_shape(&b.f);
    if (st) return st;
    if ((st = check_rule(&b.rule))) return st;
    if (b.f.family != fam || (int)b.rule.m != m) return QMC_ERR_ARG;
    if (b.f.dim != b.rule.dim) return QMC_ERR_DIM;
    if (b.i_end <= b.i_begin || b.i_end > b.rule.n) return QMC_ERR_RANGE;
    const uint64_t range = b.i_end - b.i_begin;
    uint32_t L = Lcfg;
    if (L == 0) {
        Geometry g = geometry(range, m);
        L = (g.spb == spb) ? g.L : points_per_stream(range, (uint64_t)spb);
    }
    fill_integral(it, &b.f, &b.rule, b.i_begin, b.i_end, spb, L);
    return QMC_OK;
}

}  // namespace qmc

namespace {

struct BatchPlan {
    std::vector<Integral> items;        // grouped by transform kind, in input order within one
    struct Group {
        int kind, begin, end, max_d;
    };
    std::vector<Group> groups;          // one launch each
    std::vector<uint64_t> tile_begin;   // count + 1
    uint64_t total_tiles = 0;
    uint64_t partial_doubles = 0;
    int m = 0, spb = 0, family = 0, cplx = 0;
    size_t off_items = 0, off_tb = 0, off_partials = 0, bytes = 0;
};

// Validates the batch and lays out descriptors, tile prefix sums and partials.
int plan_batch(const qmc_batch_item *in, int count, const qmc_batch_config *cfg, BatchPlan &P) {
    if (!in || count < 1) return QMC_ERR_ARG;
    const int m = (int)in[0].rule.m;
    const int fam = in[0].f.family;
    if (m < 1 || m > kMaxShiftGroup) return QMC_ERR_M;
    if (!batch_family_supported(fam)) return QMC_ERR_INTEGRAND;
    int spb = (cfg && cfg->streams_per_block > 0) ? cfg->streams_per_block : std::max(1, kSumsThreads / m);
    if (spb * m > kSumsThreads) return QMC_ERR_ARG;
    const uint32_t Lcfg = cfg ? cfg->points_per_stream : 0;
    P.m = m;
    P.spb = spb;
    P.family = fam;
    P.cplx = is_complex_family(fam);
    P.items.resize(count);
    P.tile_begin.resize(count + 1);
    P.groups.clear();
    for (int q = 0; q < count; ++q) {
        int st = fill_batch_item(P.items[q], in[q], m, spb, Lcfg, fam);
        if (st) return st;
        P.items[q].slot = q;
    }
    // the kernel is compiled per transform kind: a batch of one kind (the usual one) is one
    // launch in input order, a mixed one a launch per kind.  These overlap: alone, each of 24
    // integrals' six launches (n = 1021, m = 32) leaves the chip half empty and takes its own
    // latency, 286 us with the reduction, 134 overlapped (272 for one launch of all kinds compiled
    // together).
    std::stable_sort(P.items.begin(), P.items.end(),
                     [](const Integral &a, const Integral &b) { return a.t.kind < b.t.kind; });
    uint64_t tiles = 0, poff = 0;
    for (int q = 0; q < count; ++q) {
        Integral &it = P.items[q];
        it.tile_begin = tiles;
        it.partial_off = poff;
        P.tile_begin[q] = tiles;
        tiles += it.tiles;
        poff += it.tiles * (uint64_t)m * 2 * (P.cplx ? 2 : 1);
        if (P.groups.empty() || P.groups.back().kind != it.t.kind) P.groups.push_back({it.t.kind, q, q, 0});
        P.groups.back().end = q + 1;
        P.groups.back().max_d = std::max(P.groups.back().max_d, it.d);
    }
    P.tile_begin[count] = tiles;
    P.total_tiles = tiles;
    P.partial_doubles = poff;
    size_t o = 0;
    P.off_items = o;
    o += align256(sizeof(Integral) * count);
    P.off_tb = o;
    o += align256(sizeof(uint64_t) * (count + 1));
    P.off_partials = o;
    o += align256(sizeof(double) * poff);
    P.bytes = o;
    return QMC_OK;
}

// Kernels only (descriptors already in the workspace): capturable in a CUDA graph.
int launch_planned(const BatchPlan &P, int count, void *workspace, double *sums, double *results,
                   unsigned long long *counters, cudaStream_t s) {
    char *ws = (char *)workspace;
    Integral *d_items = (Integral *)(ws + P.off_items);
    uint64_t *d_tb = (uint64_t *)(ws + P.off_tb);
    double *d_part = (double *)(ws + P.off_partials);
    for (const auto &g : P.groups)
        if (launch_batch(P.family, g.kind, g.max_d, d_items + g.begin, d_tb + g.begin, g.end - g.begin,
                         P.tile_begin[g.begin], P.tile_begin[g.end], P.m, P.spb,
                         P.groups.size() == 1 ? kNoChain : g.begin == 0 ? kChainFirst : kChainLater, d_part,
                         counters, s) != cudaSuccess)
            return QMC_ERR_CUDA;
    if (launch_batch_reduce(d_items, count, P.m, P.cplx, d_part, sums, s) != cudaSuccess) return QMC_ERR_CUDA;
    if (results) {
        if (P.m < 2) return QMC_ERR_M;
        if (launch_batch_finalize(d_items, count, P.m, P.cplx, sums, results, s) != cudaSuccess)
            return QMC_ERR_CUDA;
    }
    return QMC_OK;
}

int run_batch(const BatchPlan &P, int count, void *workspace, double *sums, double *results,
              unsigned long long *counters, cudaStream_t s) {
    char *ws = (char *)workspace;
    if (cudaMemcpyAsync(ws + P.off_items, P.items.data(), sizeof(Integral) * count, cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(ws + P.off_tb, P.tile_begin.data(), sizeof(uint64_t) * (count + 1), cudaMemcpyHostToDevice, s) != cudaSuccess)
        return QMC_ERR_CUDA;
    return launch_planned(P, count, workspace, sums, results, counters, s);
}

}  // namespace

struct qmc_batch_plan {
    BatchPlan P;
    int count;
    void *workspace;
};

extern "C" int qmc_batch_plan_create(const qmc_batch_item *items, int count,
                                     const qmc_batch_config *cfg, void *workspace,
                                     size_t workspace_bytes, void *stream, qmc_batch_plan **out) {
    if (!workspace || !out) return QMC_ERR_ARG;
    qmc_batch_plan *plan = new (std::nothrow) qmc_batch_plan;
    if (!plan) return QMC_ERR_ARG;
    int st = plan_batch(items, count, cfg, plan->P);
    if (!st && workspace_bytes < plan->P.bytes) st = QMC_ERR_WORKSPACE;
    if (!st) st = device_ok();
    if (!st) {
        cudaStream_t s = (cudaStream_t)stream;
        char *ws = (char *)workspace;
        if (cudaMemcpyAsync(ws + plan->P.off_items, plan->P.items.data(), sizeof(Integral) * count,
                            cudaMemcpyHostToDevice, s) != cudaSuccess ||
            cudaMemcpyAsync(ws + plan->P.off_tb, plan->P.tile_begin.data(),
                            sizeof(uint64_t) * (count + 1), cudaMemcpyHostToDevice, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            st = QMC_ERR_CUDA;
    }
    if (st) {
        delete plan;
        return st;
    }
    plan->count = count;
    plan->workspace = workspace;
    *out = plan;
    return QMC_OK;
}

extern "C" int qmc_batch_plan_run(const qmc_batch_plan *plan, double *sums, double *results,
                                  unsigned long long *counters, void *stream) {
    if (!plan || !sums) return QMC_ERR_ARG;
    return launch_planned(plan->P, plan->count, plan->workspace, sums, results, counters,
                          (cudaStream_t)stream);
}

extern "C" void qmc_batch_plan_destroy(qmc_batch_plan *plan) { delete plan; }

extern "C" size_t qmc_batch_workspace_bytes(const qmc_batch_item *items, int count,
                                            const qmc_batch_config *cfg) {
    BatchPlan P;
    if (plan_batch(items, count, cfg, P) != QMC_OK) return 0;
    return P.bytes;
}

extern "C" int qmc_batch_sums(const qmc_batch_item *items, int count, const qmc_batch_config *cfg,
                              void *workspace, size_t workspace_bytes, double *sums,
                              double *results, unsigned long long *counters, void *stream) {
    if (!workspace || !sums) return QMC_ERR_ARG;
    BatchPlan P;
    int st = plan_batch(items, count, cfg, P);
    if (st) return st;
    if (workspace_bytes < P.bytes) return QMC_ERR_WORKSPACE;
    if ((st = device_ok())) return st;
    return run_batch(P, count, workspace, sums, results, counters, (cudaStream_t)stream);
}

extern "C" int qmc_batch_autotune(const qmc_batch_item *items, int count, void *workspace,
                                  size_t workspace_bytes, double *sums, void *stream,
                                  qmc_batch_config *best) {
    if (!workspace || !sums || !best || !items || count < 1) return QMC_ERR_ARG;
    int st = device_ok();
    if (st) return st;
    cudaStream_t s = (cudaStream_t)stream;
    // a sample of the batch: every step-th item, at most 256 items
    const int step = std::max(1, count / 256);
    std::vector<qmc_batch_item> sample;
    for (int q = 0; q < count; q += step) sample.push_back(items[q]);
    // bounded cost per candidate: at most ~2^23 points in all, each item's range cut to its
    // share from its start (the candidates are compared on the same work)
    const uint64_t share = std::max<uint64_t>(1u << 16, (1u << 23) / sample.size());
    for (auto &it : sample)
        if (it.i_end > it.i_begin + share) it.i_end = it.i_begin + share;
    const int m = (int)items[0].rule.m;
    if (m < 1 || m > kMaxShiftGroup) return QMC_ERR_M;
    const int spb_max = std::max(1, kSumsThreads / m);
    const int spbs[] = {spb_max, std::max(1, spb_max / 2), std::max(1, spb_max / 4)};
    const uint32_t Ls[] = {16, 32, 64, 128, 256, 512};
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return QMC_ERR_CUDA;
    float best_ms = -1.0f;
    qmc_batch_config cand;
    for (int si = 0; si < 3; ++si) {
        if (si > 0 && spbs[si] == spbs[si - 1]) continue;
        for (uint32_t L : Ls) {
            cand.streams_per_block = spbs[si];
            cand.points_per_stream = L;
            BatchPlan P;
            if ((st = plan_batch(sample.data(), (int)sample.size(), &cand, P))) break;
            if (P.bytes > workspace_bytes) continue;
            // warm once, then time one run
            if ((st = run_batch(P, (int)sample.size(), workspace, sums, nullptr, nullptr, s))) break;
            cudaEventRecord(e0, s);
            if ((st = run_batch(P, (int)sample.size(), workspace, sums, nullptr, nullptr, s))) break;
            cudaEventRecord(e1, s);
            if (cudaEventSynchronize(e1) != cudaSuccess) { st = QMC_ERR_CUDA; break; }
            float ms = 0.0f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (best_ms < 0.0f || ms < best_ms) {
                best_ms = ms;
                *best = cand;
            }
        }
        if (st) break;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (st) return st;
    return best_ms < 0.0f ? QMC_ERR_WORKSPACE : QMC_OK;
}
