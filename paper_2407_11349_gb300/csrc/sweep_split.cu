// Column-split pair sweep: the symmetric sweep of sweep_kernel.cuh with the
// tile's columns, not its rows, divided among the CTA's warps.
//
// The row-tile kernel gives each warp its own 256 rows, so its unit of work is
// 2,048 rows x 256 columns.  At N = 2,000 that is one row tile, hence one SM
// of 152 (0.43 ms), and near the diagonal the warps whose rows lie above a
// column tile idle (14% of the units at N = 20,000).  Here all eight warps
// hold the same 128 rows and each takes 32 of the tile's 256 columns, so the
// unit is 128 x 256 pairs, a sixteenth of the other.  Like the row-tile
// kernel it is bound by the FP32 pipe, with the same arithmetic per pair
// (chunk_pass), plus the row flush below once per item.  Sweep times before
// (row tiles, 16 column tiles per item) and after, space-time background:
// N = 2,000 0.425 -> 0.014 ms, 10,000 0.945 -> 0.062, 17,103 0.943 -> 0.144,
// 30,000 0.87 -> 0.40.  sweep_plan.h says which kernel runs.  Larger sums (and some of the
// smaller, as 17,103) take the row-tile kernel below the diagonal and this one for
// the band of each row tile's own columns.
// What changes:
//   - a column belongs to one warp: its sums go from the warp's registers to
//     the FP64 accumulators, without the shared-memory pass;
//   - a row's sums are spread over the eight warps: at the end of an item they
//     meet in shared memory (FP32, a fixed tree of eight) and each row is
//     flushed once per item.
#include <algorithm>
#include <vector>

#include "sweep_kernel.cuh"
#include "units.cuh"

namespace hk {

// 2 row pairs per lane (128 rows) and 2 CTAs per SM: measured against 4 pairs
// and one CTA it was 0.0143 to 0.0208 ms at N = 2,000, 0.0622 to 0.0786 at
// 10,000, 0.402 to 0.410 at 30,000 and 1.056 to 1.040 at 50,000 (where the two
// kernels together take 0.956).
constexpr int SPLIT_RP = 2, SPLIT_BPSM = 2;
constexpr int STAGE = 2;  // column tiles per shared-memory buffer (one CTA barrier each)

template <int RP>
struct SGeo {
    static constexpr int R = 2 * RP;
    static constexpr int ROWS = 32 * R;  // rows of an item, shared by all warps
    static_assert(TB % ROWS == 0, "an item's rows share one time block");
    static constexpr size_t SMEM_TILES = 2 * STAGE * TC * sizeof(Rec);
    static constexpr size_t SMEM_RED = 6 * WARPS * ROWS * sizeof(float);
    static constexpr size_t SMEM_LO = ROWS * sizeof(int);
    static constexpr size_t SMEM_RACC = 3 * RP * THREADS * sizeof(float4);  // BGT kernels only
    static constexpr size_t smem(bool bgt) {
        return SMEM_TILES + SMEM_RED + SMEM_LO + (bgt ? SMEM_RACC : 0);
    }
};
static_assert(TC == 32 * WARPS, "one 32-column chunk of a tile per warp");

// Persistent sweep over items (row group of ROWS rows, first column tile, end
// column tile, problem); modes as in k_sweep.
template <int RP, int MINB, int MODE, bool BGT, bool LL>
__global__ void __launch_bounds__(THREADS, MINB)
    k_sweep_cs(ProbDesc one, const ProbDesc* __restrict__ probs, const int4* __restrict__ items,
               int nitems, int* __restrict__ ctr, int nprobs, int band) {
    using G = SGeo<RP>;
    constexpr int R = G::R, ROWS = G::ROWS;
    extern __shared__ __align__(128) unsigned char smem[];
    Rec* tiles = reinterpret_cast<Rec*>(smem);
    float* red = reinterpret_cast<float*>(smem + G::SMEM_TILES);
    int* slo = reinterpret_cast<int*>(smem + G::SMEM_TILES + G::SMEM_RED);
    float4* racc = reinterpret_cast<float4*>(smem + G::SMEM_TILES + G::SMEM_RED + G::SMEM_LO) +
                   threadIdx.x;
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ int s_item, s_abort, s_bad;
    __shared__ __align__(16) ProbDesc s_pd;  // the current item's problem (MODE_BATCH)
    volatile ProbDesc* vpd = &s_pd;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // As the band of a row-tile sweep, this kernel starts while that one runs: its
    // inputs were complete when that one passed its chain_wait, which it publishes
    // before the chain_next that lets this one start; this one's end waits for its.
    if (!band) chain_wait();
    if (tid == 0) {
        s_abort = 0;
        if (band && !acquire_ready(ctr)) {
            set_error(ctr, HAWKES_ERR_TIMEOUT);
            s_abort = 1;
        }
    }
    __syncthreads();
    if (MODE != MODE_BATCH && one.cc[CC_VALID] == 0.0) {
        if (band) chain_wait();
        return;
    }
    if (tid == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        fence_barrier_init();
    }
    __syncthreads();
    uint32_t parbits = 0u;   // bit b: parity of the next phase of buffer b
    uint32_t pendbits = 0u;  // thread 0, bit b: a copy into buffer b is in flight
    int* mylo = slo + lane * R;

    for (;;) {
        if (tid == 0) {
            const int k = atomicAdd(ctr + (band ? CT_BAND : CT_WORK), 1);
            s_item = k;
            if (kDebug) s_bad = 0;
            if (kDebug && MODE == MODE_BATCH && k < nitems &&
                !(items[k].w >= 0 && items[k].w < nprobs)) {
                s_bad = 1;  // problem index out of range: do not read its descriptor
            } else if (MODE == MODE_BATCH && k < nitems) {
                const ProbDesc d = probs[items[k].w];
                vpd->t = d.t; vpd->rec = d.rec; vpd->lo = d.lo; vpd->hi = d.hi; vpd->tb = d.tb;
                vpd->cc = d.cc; vpd->acc = d.acc; vpd->n = d.n; vpd->npad = d.npad;
            }
        }
        __syncthreads();
        const int item = s_item;
        if (item >= nitems || s_abort) {
            chain_next();
            break;
        }
#define HK_PD(field) (MODE == MODE_BATCH ? vpd->field : one.field)
        const int4 it = items[item];
        const int64_t r0 = static_cast<int64_t>(it.x) * ROWS;
        const int jb = it.y, nJ = it.z - it.y;
        if (kDebug) {  // the item must lie inside its problem's causal triangle
            bool ok = !s_bad;
            const int64_t nn = ok ? HK_PD(n) : 0, np = ok ? HK_PD(npad) : 0;
            const int64_t jmax = (min(r0 + ROWS, nn) + TC - 1) / TC;
            ok = ok && it.x >= 0 && r0 < nn && r0 + ROWS <= np && jb >= 0 && jb < it.z &&
                 it.z <= jmax && static_cast<int64_t>(it.z) * TC <= np;
            if (!ok) {
                if (tid == 0) set_error(ctr, HAWKES_ERR_BOUNDS);
                __syncthreads();
                continue;
            }
        }
        const double* cc = HK_PD(cc);
        if (MODE == MODE_BATCH && cc[CC_VALID] == 0.0) {  // problem with invalid parameters
            __syncthreads();
            continue;
        }
        const float omt = static_cast<float>(cc[CC_OMT]);
        const float2 nomt = f2(-omt, -omt);
        const double kt = cc[CC_KT];
        const int64_t n = HK_PD(n);
        const double skipdt = cc[CC_SKIPDT];
        if (skipdt > 0.0) {  // whole item below the FP32 underflow bound
            const double* tt = HK_PD(t);
            const int64_t lastc = min(static_cast<int64_t>(it.z) * TC, n) - 1;
            if ((tt[r0] - tt[lastc]) * kt > skipdt) {
                __syncthreads();
                continue;
            }
        }
        // Buffer q holds the item's tiles [q STAGE, (q + 1) STAGE), then every
        // second group of STAGE after it (tiles are contiguous: one copy each).
        auto load_stage = [&](int q, int J) {  // thread 0
            const uint32_t bytes = min(STAGE, nJ - J) * static_cast<uint32_t>(TC * sizeof(Rec));
            mbar_arrive_expect_tx(&bars[q], bytes);
            tma_load_1d(tiles + q * STAGE * TC, HK_PD(rec) + static_cast<int64_t>(jb + J) * TC, bytes,
                        &bars[q]);
            pendbits |= 1u << q;
        };
        if (tid == 0)
            for (int q = 0; q < 2 && q * STAGE < nJ; ++q) load_stage(q, q * STAGE);

        Rows<RP> rr;
        float t0[R];
#pragma unroll
        for (int p = 0; p < RP; ++p) {
            const Rec* rec = HK_PD(rec);
            const int32_t* plo = HK_PD(lo);
            const int64_t i0 = r0 + lane + 64 * p, i1 = i0 + 32;
            const float4 a0 = *rec_q(rec, i0, 0), b0 = *rec_q(rec, i0, 1), c0 = *rec_q(rec, i0, 2);
            const float4 a1 = *rec_q(rec, i1, 0), b1 = *rec_q(rec, i1, 1), c1 = *rec_q(rec, i1, 2);
            t0[2 * p] = -a0.x;
            t0[2 * p + 1] = -a1.x;
            rr.xh[p] = f2(-a0.z, -a1.z);
            rr.xl[p] = f2(-b0.x, -b1.x);
            rr.yh[p] = f2(-b0.z, -b1.z);
            rr.yl[p] = f2(-c0.x, -c1.x);
            rr.sB[p] = rr.sBr[p] = rr.sBt[p] = rr.sE[p] = rr.sEt[p] = rr.sEq[p] = f2(0.f, 0.f);
            if (BGT)
                for (int q = 0; q < 3; ++q) racc[(3 * p + q) * THREADS] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (warp == 0) {
                mylo[2 * p] = plo[i0];
                mylo[2 * p + 1] = plo[i1];
            }
        }
        const int lo_first = HK_PD(lo)[r0];
        const double trow = HK_PD(tb)[r0 / TB];
        __syncthreads();  // slo

        const double* tbp = HK_PD(tb);
        float dT = static_cast<float>((trow - tbp[jb]) * kt);  // row times against the tile's base
        for (int J = 0; J < nJ; J += STAGE) {
            const int buf = (J / STAGE) & 1;
            if (!mbar_wait(&bars[buf], (parbits >> buf) & 1u)) {
                set_error(ctr, HAWKES_ERR_TIMEOUT);
                s_abort = 1;
            }
            parbits ^= 1u << buf;
            pendbits &= ~(1u << buf);
#pragma unroll 1
            for (int u = 0; u < STAGE && J + u < nJ; ++u) {
                const int jt = jb + J + u;
                const int j0 = jt * TC, c0 = j0 + 32 * warp;  // this warp's columns [c0, c0 + 32)
                // columns at or past the last row (or the last event) hold no pair
                bool run = c0 < min(r0 + ROWS, n);
                if (run && skipdt > 0.0) {
                    const double* tt = HK_PD(t);
                    if ((tt[r0] - tt[min(static_cast<int64_t>(c0) + 32, n) - 1]) * kt > skipdt) run = false;
                }
                const float dTj = dT;
                if (J + u + 1 < nJ) dT = static_cast<float>((trow - tbp[jt + 1]) * kt);
                if (!run) continue;
#pragma unroll
                for (int p = 0; p < RP; ++p) rr.tp[p] = f2(t0[2 * p] + dTj, t0[2 * p + 1] + dTj);
                const float4* tile = reinterpret_cast<const float4*>(tiles + (buf * STAGE + u) * TC);
                float2 cB, cBr, cBt;
                // (the unmasked pass fully unrolled: 1-2% over an unroll of 8, which
                // refills the pipeline four times a chunk)
                if (c0 + 32 > lo_first)
                    chunk_pass<RP, 8, M_LOWER, true, true, BGT, LL>(tile, warp, j0, lane, rr, nomt, mylo, mylo, cB, cBr, cBt);
                else
                    chunk_pass<RP, 32, M_NONE, true, true, BGT, LL>(tile, warp, j0, lane, rr, nomt, mylo, mylo, cB, cBr, cBt);
                if (BGT) fold_rows<RP>(rr, racc);
                const float v0 = cB.x + cB.y, v1 = cBr.x + cBr.y, v2 = cBt.x + cBt.y;
                if (v0 != 0.f || v1 != 0.f || v2 != 0.f) {
                    double* acc = HK_PD(acc) + c0 + lane;
                    const int64_t npad = HK_PD(npad);
                    atomicAdd(acc, static_cast<double>(v0));
                    if (!LL) {
                        if (!BGT) atomicAdd(acc + npad, static_cast<double>(v1) * cc[CC_SR]);
                        atomicAdd(acc + 2 * npad, static_cast<double>(v2) * cc[CC_ST]);
                    }
                }
            }
            __syncthreads();
            if (tid == 0 && J + 2 * STAGE < nJ && !s_abort) load_stage(buf, J + 2 * STAGE);
            if (s_abort) break;
        }

        // The eight warps' row sums meet in shared memory, moment by moment
        // (red[q][warp][row]), and go to the FP64 accumulators.
#pragma unroll
        for (int p = 0; p < RP; ++p) {
            float2 v[6] = {rr.sB[p], rr.sBr[p], rr.sBt[p], rr.sE[p], rr.sEt[p], rr.sEq[p]};
            if (BGT) {
                const float4 a = racc[(3 * p + 0) * THREADS];
                const float4 b = racc[(3 * p + 1) * THREADS];
                const float4 e = racc[(3 * p + 2) * THREADS];
                v[0] = f2(a.x, a.y); v[1] = f2(a.z, a.w); v[2] = f2(b.x, b.y);
                v[3] = f2(b.z, b.w); v[4] = f2(e.x, e.y); v[5] = f2(e.z, e.w);
            }
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                if ((LL && q != 0 && q != 3) || (BGT && q == 1)) continue;
                float* dst = red + (q * WARPS + warp) * ROWS + lane + 64 * p;
                dst[0] = v[q].x;
                dst[32] = v[q].y;
            }
        }
        __syncthreads();
        if (!s_abort) {
            for (int k = tid; k < 6 * ROWS; k += THREADS) {
                const int q = k / ROWS, row = k % ROWS;
                if ((LL && q != 0 && q != 3) || (BGT && q == 1) || r0 + row >= n) continue;
                const float* src = red + q * WARPS * ROWS + row;
                const float a = (src[0] + src[ROWS]) + (src[2 * ROWS] + src[3 * ROWS]);
                const float b = (src[4 * ROWS] + src[5 * ROWS]) + (src[6 * ROWS] + src[7 * ROWS]);
                const float v = a + b;
                if (v == 0.f) continue;
                const double f = q == 1 ? cc[CC_SR] : q == 2 ? cc[CC_ST] : q == 4 ? cc[CC_SET]
                                 : q == 5 ? -cc[CC_SEQ] : 1.0;
                atomicAdd(HK_PD(acc) + q * HK_PD(npad) + r0 + row, static_cast<double>(v) * f);
            }
        }
        __syncthreads();  // thread 0 replaces s_item and s_pd next
        if (s_abort) break;
#undef HK_PD
    }
    // A wait that gave up may leave bulk copies in flight: let them land
    // (bounded) before the CTA's shared memory is released.
    if (tid == 0)
        for (int q = 0; q < 2; ++q)
            if ((pendbits >> q) & 1u) (void)mbar_wait(&bars[q], (parbits >> q) & 1u);
    if (band) chain_wait();
}

using SplitFn = void (*)(ProbDesc, const ProbDesc*, const int4*, int, int*, int, int);

struct SplitKernel {
    SplitFn sym, batch;
    size_t smem;
};

#define HK_SPLIT(BGT, LL)                                                                     \
    {k_sweep_cs<SPLIT_RP, SPLIT_BPSM, MODE_SYM, BGT, LL>,                                     \
     k_sweep_cs<SPLIT_RP, SPLIT_BPSM, MODE_BATCH, BGT, LL>, SGeo<SPLIT_RP>::smem(BGT)}
// space-time background, time-only background, log-likelihood only
static const SplitKernel kSplit[3] = {HK_SPLIT(false, false), HK_SPLIT(true, false),
                                      HK_SPLIT(false, true)};

cudaError_t split_setup_attributes() {
    for (const SplitKernel& k : kSplit)
        for (SplitFn f : {k.sym, k.batch}) {
            const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       static_cast<int>(k.smem));
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

int split_rows() { return SGeo<SPLIT_RP>::ROWS; }

// One problem (probs null) or the items of many; band: launched behind a row-tile
// sweep of the same problems that lets it start early.
cudaError_t launch_sweep_split(cudaStream_t st, int sms, const ProbDesc& one, const ProbDesc* probs,
                               int nprobs, const int4* items, int nitems, int* ctr, bool bgt, bool ll, bool band) {
    const SplitKernel& k = kSplit[bgt ? 1 : ll ? 2 : 0];
    const int grid = std::min(nitems, sms * SPLIT_BPSM);
    if (grid <= 0) return cudaSuccess;
    return launch_chained(probs ? k.batch : k.sym, grid, THREADS, k.smem, st, one, probs, items, nitems, ctr,
                          nprobs, band ? 1 : 0);
}

}  // namespace hk
