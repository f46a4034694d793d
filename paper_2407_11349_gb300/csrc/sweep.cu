// Host side of the FP32 pair sweep (kernels in sweep_kernel.cuh): kernel
// variants, their work lists, and launch.  This unit instantiates the
// space-time background's kernels; sweep_bgt.cu the time-only background's
// and sweep_ll.cu the log-likelihood-only ones.
#include <algorithm>
#include <string>
#include <vector>

#include "sweep_kernel.cuh"
#include "units.cuh"

namespace hk {

static const Variant kVariants[] = HK_SWEEP_VARIANTS(false, false);
static_assert(sizeof(kVariants) / sizeof(kVariants[0]) == kNumVariants, "variant count");

// The kernel family of a call: the time-only background keeps its own kernels
// (with the log-likelihood-only flag it forms every moment and the gradient is
// dropped at finalisation).
static const Variant& variant_of(int v, bool bgt, bool ll) {
    return bgt ? sweep_variants_bgt()[v] : ll ? sweep_variants_ll()[v] : kVariants[v];
}

int sweep_num_variants() { return kNumVariants; }
int sweep_variant_rows(int v) { return kVariants[v].tr; }

cudaError_t sweep_setup_attributes() {
    for (int k = 0; k < 3 * kNumVariants; ++k) {
        const int fam = k / kNumVariants;
        const Variant& v = variant_of(k % kNumVariants, fam == 1, fam == 2);
        for (SweepFn f : {v.win, v.sym, v.batch}) {
            cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 static_cast<int>(v.smem));
            if (e != cudaSuccess) return e;
        }
    }
    return split_setup_attributes();
}

int sweep_blocks_per_sm(int v) {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kVariants[v].sym, THREADS,
                                                      kVariants[v].smem) != cudaSuccess)
        return 1;
    return nb > 0 ? nb : 1;
}

// The plan (sweep_plan.h) on variant v.
SweepPlan sweep_plan(const int64_t* ns, size_t count, int sms, int v, int chunk, bool band) {
    return sweep_plan(ns, count, sms, PlanKernels{kVariants[v].tr, kVariants[v].minb, split_rows()}, chunk, band);
}

// The tuning caches' part of a key that says which kernels the times are of: a
// number to raise when the sweep's kernels or plans change, and each variant's plan
// (c column split alone, r row tiles).  Sizes of one power of two may differ in it,
// and on a c the variants' times are one kernel's.
std::string sweep_plans_key(const int64_t* ns, size_t count, int sms) {
    std::string key = "kernels=2|plans=";
    for (int v = 0; v < kNumVariants; ++v) key += sweep_plan(ns, count, sms, v, CHUNK, true).split ? 'c' : 'r';
    return key + "|";
}

// Symmetric work list over problems of sizes ns[] for plan pl (variant v on
// the row-tile kernel): items (row tile, column tiles [jb, je), problem) in
// chunks of pl.chunk column tiles.  order 0: all items longest first (ties: later row tiles first);
// order 1: problem by problem, largest problem first, each problem's items
// longest first, so that the source tiles and accumulators of the problems
// in flight stay in L2 while the tail still ends on the smallest items.
std::vector<int4> sweep_items_batch(const std::vector<int64_t>& ns, const SweepPlan& pl, int v,
                                    int order) {
    const int tr = pl.split ? split_rows() : kVariants[v].tr, chunk = pl.chunk;
    auto longest_first = [](const int4& a, const int4& b) {
        return (a.z - a.y) > (b.z - b.y) || ((a.z - a.y) == (b.z - b.y) && a.x > b.x);
    };
    std::vector<size_t> pidx(ns.size());
    for (size_t p = 0; p < ns.size(); ++p) pidx[p] = p;
    if (order == 1)
        std::stable_sort(pidx.begin(), pidx.end(), [&](size_t a, size_t b) { return ns[a] > ns[b]; });
    std::vector<int4> items;
    for (size_t p : pidx) {
        const int64_t n = ns[p];
        const int64_t nI = (n + tr - 1) / tr;
        const size_t first = items.size();
        for (int64_t I = 0; I < nI; ++I) {
            const int nJ = static_cast<int>(pl.band ? I * tr / TC : (std::min<int64_t>((I + 1) * tr, n) + TC - 1) / TC);
            for (int jb = 0; jb < nJ; jb += chunk)
                items.push_back(make_int4(static_cast<int>(I), jb, std::min(jb + chunk, nJ),
                                          static_cast<int>(p)));
        }
        if (order == 1) std::stable_sort(items.begin() + first, items.end(), longest_first);
    }
    if (order == 0) std::stable_sort(items.begin(), items.end(), longest_first);
    return items;
}

// Items of the diagonal band, for the column-split kernel: the columns that the
// row tiles of a plan with `band` leave out.
std::vector<int4> sweep_band(const std::vector<int64_t>& ns, const SweepPlan& pl, int v) {
    std::vector<int4> items;
    if (!pl.band) return items;
    const int tr = kVariants[v].tr, rows = split_rows();
    for (size_t p = 0; p < ns.size(); ++p)
        for (int64_t r = 0; r < ns[p]; r += rows)
            items.push_back(make_int4(static_cast<int>(r / rows), static_cast<int>(r / tr * (tr / TC)),
                                      static_cast<int>((std::min<int64_t>(r + rows, ns[p]) + TC - 1) / TC),
                                      static_cast<int>(p)));
    std::stable_sort(items.begin(), items.end(), [](const int4& a, const int4& b) { return a.z - a.y > b.z - b.y; });
    return items;
}

std::vector<int4> sweep_items(int64_t n, const SweepPlan& pl, int v) {
    return sweep_items_batch({n}, pl, v, 0);
}

static ProbDesc desc_of(const hawkes_ctx* c) {
    return ProbDesc{c->t, c->rec, c->lo, c->hi, c->tb, c->cc, c->acc, c->n, c->npad};
}

// Row-tile sweep of one problem over the work list items[0, nitems) and the
// diagonal band's items behind it (the whole lists, or one shard's part of them).
cudaError_t launch_sweep_list(hawkes_ctx* c, const int4* items, int nitems, int nband, bool bgt, bool ll) {
    const Variant& v = variant_of(c->variant, bgt, ll);
    const int grid_cap = c->sms * c->variant_bpsm;
    const int grid = nitems < grid_cap ? nitems : grid_cap;
    if (grid > 0) {
        const cudaError_t e = launch_chained(v.sym, grid, THREADS, v.smem, c->stream, desc_of(c), nullptr, items,
                                             nitems, c->ctr, 0, c->n, nband > 0 ? 1 : 0, 0);
        if (e != cudaSuccess) return e;
    }
    if (nband == 0) return cudaSuccess;
    return launch_sweep_split(c->stream, c->sms, desc_of(c), nullptr, 0, items + nitems, nband, c->ctr, bgt, ll,
                              nitems > 0);
}

cudaError_t launch_sweep(hawkes_ctx* c, bool sym, int64_t row_begin, int64_t row_end, bool bgt,
                         bool ll) {
    const Variant& v = variant_of(c->variant, bgt, ll);
    const int grid_cap = c->sms * c->variant_bpsm;
    const ProbDesc one = desc_of(c);
    if (sym && c->plan.split) {
        return launch_sweep_split(c->stream, c->sms, one, nullptr, 0, c->items, c->nitems, c->ctr, bgt,
                                  ll, false);
    } else if (sym) {
        return launch_sweep_list(c, c->items, c->nitems, c->nband, bgt, ll);
    } else {
        const int item0 = static_cast<int>(row_begin / v.tr);
        const int nrt = static_cast<int>((row_end + v.tr - 1) / v.tr) - item0;
        const int ncol = static_cast<int>((c->n + TC - 1) / TC);
        const int nch = (ncol + CHUNK - 1) / CHUNK;
        const int nitems = nrt * nch;
        const int grid = nitems < grid_cap ? nitems : grid_cap;
        if (grid <= 0) return cudaSuccess;
        return launch_chained(v.win, grid, THREADS, v.smem, c->stream, one, nullptr, nullptr, nitems, c->ctr,
                              row_begin, row_end, item0, nch);
    }
}

// Persistent launches over the items of many problems; ctr[CT_WORK] and
// ctr[CT_BAND] must be zero when they start.
cudaError_t launch_sweep_batch(cudaStream_t st, const SweepPlan& pl, int sms, int variant, int grid,
                               const ProbDesc* probs, int nprobs, const int4* items, int nitems, int nband,
                               int* ctr, bool bgt, bool ll) {
    if (pl.split)
        return launch_sweep_split(st, sms, ProbDesc{}, probs, nprobs, items, nitems, ctr, bgt, ll, false);
    const Variant& v = variant_of(variant, bgt, ll);
    if (grid > nitems) grid = nitems;
    ProbDesc none{};
    if (grid > 0) {
        const cudaError_t e = launch_chained(v.batch, grid, THREADS, v.smem, st, none, probs, items, nitems, ctr, 0, 0,
                                             nband > 0 ? 1 : 0, nprobs);
        if (e != cudaSuccess) return e;
    }
    if (nband == 0) return cudaSuccess;
    return launch_sweep_split(st, sms, none, probs, nprobs, items + nitems, nband, ctr, bgt, ll, nitems > 0);
}

}  // namespace hk
