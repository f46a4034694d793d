// Surrogate network of the log-likelihood and its gradient: a 7 -> 256 -> 256
// -> 7 multilayer perceptron (tanh hidden units), trained on the GPU with
// these kernels and evaluated inside HMC leapfrog trajectories.  The paper has
// no surrogate: this is the learned part layered on its method.
//
// Inputs are the six standardised log-parameters and a seventh input that is
// either a constant 1 or a standardised per-sample feature; outputs are the
// standardised log-likelihood and its six log-parameter partials.
// Weights are kept in FP32 (Adam state and master copy); the 256 x 256 layer
// runs on the 5th-generation tensor cores (tcgen05.mma, accumulator in tensor
// memory) from BF16 copies of W2 and W2^T with BF16 activations and FP32
// accumulation; the 7-wide layers run in FP32.  A training step is two
// launches (k_mlp, k_update), a prediction one.
//   forward:  h1 = tanh(x W1^T + b1), h2 = tanh(h1 W2^T + b2), y = h2 W3^T + b3
//   loss:     mean over the batch and the 7 outputs of (y - t)^2
#include <cuda_bf16.h>

#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "common.cuh"

namespace {

using bf16 = __nv_bfloat16;
constexpr int DIN = 7, DH = 256, DOUT = 7;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + DH * DIN, OFF_W2 = OFF_B1 + DH, OFF_B2 = OFF_W2 + DH * DH,
              OFF_W3 = OFF_B2 + DH, OFF_B3 = OFF_W3 + DOUT * DH, NPARAMS = OFF_B3 + DOUT;
static_assert(NPARAMS == HAWKES_MLP_NPARAMS, "parameter count");
constexpr int BMAX = 4096;  // largest batch (a multiple of 64)

// Philox4x32-10 (Salmon et al. 2011) for minibatch draws and initialisation.
__device__ __forceinline__ uint4 philox4x32(uint4 c, uint2 k) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) {
            k.x += 0x9E3779B9u;
            k.y += 0xBB67AE85u;
        }
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    }
    return c;
}

// ---------------------------------------------------------------------------
// A training step is two kernels: k_mlp takes the minibatch from its draw to the
// error signals, k_update forms the gradients and applies them.  Predictions
// are k_mlp's first half.
//
// k_mlp: a cluster of four CTAs takes 128 rows; each CTA owns 64 of the 256
// hidden units in both layers.  A thread owns one row and 32 of its CTA's
// units, and keeps h1 and h2 of those in registers; what the other CTAs need
// goes straight into their shared memory: the BF16 operands (h1, dz2) by bulk
// copies that complete on the receiver's barrier, h2 to the CTA that forms its
// row's outputs and the output errors back by stores and a cluster barrier.
// The products run on the 5th-generation tensor cores (tcgen05, M = 128, N = 64
// per CTA) from those operands and the CTA's slices of W2 and W2^T, which one
// bulk copy each brings in:
//     z2 = h1 W2^T       A = h1,  B = W2 slice     (K-major)
//     dz1 = dz2 W2       A = dz2, B = W2^T slice   (K-major)
// k_update: dW2 = dz2^T h1 over all rows, in 128 x 32 tiles, from the same
// operands read along the other axis (MN-major); the 7-wide gradients and
// biases by one block per hidden unit; each followed by its Adam update.
//
// Every sum keeps one fixed order, whatever the number of clusters: outputs
// along the hidden units, dW2 along the rows, the small gradients over 256
// strided chains and a binary tree.  The BF16 roundings make training
// sensitive to the last bit, so that order is part of what the network learns.
//
// What bounds it: latency.  At batch 512 16 CTAs work through four exchanges and
// two products.  (As eleven kernels, three products of 4 CTAs staged through
// registers at 34 to 44 us each among them, a step took 170 us.)
//
// Operand layout: 8 x 16-byte core matrices without swizzle.  In k_mlp the core
// matrix (row group i, unit group j) is at byte (32 i + j) * 128: as a K-major
// operand (rows x units) the step between core matrices along K is 128 and
// between row groups 4096.  In device memory: see store_units.
// A wait that gives up latches HAWKES_ERR_TIMEOUT in *err (pinned host memory)
// and the kernel runs on to its end, so no barrier is left waiting.
// ---------------------------------------------------------------------------
constexpr int CL = 4, MT = 128, NS = DH / CL, MLP_THREADS = 256;
static_assert(BMAX % MT == 0, "whole clusters");
constexpr uint32_t SLICE_BYTES = NS * DH * 2;
constexpr int UT_M = 128, UT_N = 32;  // dW2 tile of k_update: input units x output units

// Byte of element (n, k) in the sliced BF16 copies of W2 (n = output unit) and
// W2^T (n = input unit): slice n / 64, then core matrices as above.
__host__ __device__ __forceinline__ uint32_t slice_off(int n, int k) {
    const int r = n % NS;
    return (n / NS) * SLICE_BYTES + ((r >> 3) * (DH / 8) + (k >> 3)) * 128 + (r & 7) * 16 + (k & 7) * 2;
}

struct MlpSmem {
    unsigned char h1[MT * DH * 2];  // BF16 operands of all 256 units
    unsigned char dz[MT * DH * 2];  // (before dz2: h2 of this CTA's 32 output rows, FP32)
    unsigned char w[SLICE_BYTES];   // W2 slice
    unsigned char wt[SLICE_BYTES];  // W2^T slice
    float x[MT][8], t[MT][8], dy[MT][8];
    float w3o[8][DH + 4];           // W3 by output
    float w1[NS][8];                // W1 of the unit, then b1
    float w3[NS][8];                // W3 of the unit, then b2
    float b3[8];
    uint64_t bar[6];                // W2, z2, dz1, small layers, peers' h1, peers' dz2
    uint32_t tmem;
};
static_assert(sizeof(MlpSmem) <= 227 * 1024, "fits a CTA");
constexpr int YROWS = MT / CL, YPITCH = DH + 4;  // output rows per CTA, floats between them
static_assert(YROWS == 32 && YROWS * YPITCH * 4 <= MT * DH * 2, "a warp's rows; fits the dz buffer");

enum { MLP_PREDICT = 0, MLP_TRAIN = 1, MLP_GIVEN = 2 };

struct MlpArgs {
    const float* P;
    const float *W1p, *W3p;        // per hidden unit: W1 row and b1; W3 column and b2 (8 floats)
    const bf16 *W2s, *W2Ts;        // sliced copies
    int B;                         // rows
    // MLP_TRAIN: rows drawn with replacement from the standardised data set
    const float *Xs, *Ts;          // (MLP_GIVEN: the rows themselves)
    int64_t n;
    uint64_t seed, step, nrec;     // nrec = floor((2^64 - 1) / n)
    // MLP_PREDICT
    const double *q, *f, *stats;
    double* pred;
    // for k_update: BF16 operands, FP32 signals by unit [DH][rows], inputs and
    // output errors [rows][8]
    unsigned char *h1op, *dzop;
    float *h2t, *dz2t, *dz1t, *xin, *dyo;
    float* Y;                      // MLP_GIVEN: outputs (or null)
    double* loss;                  // summed loss (or null)
    volatile int* err;
};

// Instruction descriptor: FP32 accumulator (bits 4-5 = 1), BF16 A and B (bits
// 7-9, 10-12 = 1), A and B major (bits 15, 16: 0 K, 1 MN), N >> 3 at bit 17,
// M >> 4 at bit 24.
constexpr uint32_t TC_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((NS >> 3) << 17) | ((MT >> 4) << 24);
constexpr uint32_t TC_GROUP = 128, TC_ROWS = (DH / 8) * 128;  // core-matrix steps: unit group, row group

// Shared-memory matrix descriptor: start, leading and stride byte offsets (all
// >> 4), descriptor version 1, no swizzle.  K-major: leading = step along K,
// stride = step along M or N.  MN-major: leading = step along K (8 rows),
// stride = step along M or N (8 units).
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return static_cast<uint64_t>((saddr >> 4) & 0x3FFFu) |
           (static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16) |
           (static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     hk::smem_u32(bar))
                 : "memory");
}
// 32 accumulator columns of the thread's row.
__device__ __forceinline__ void tc_load32(uint32_t addr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int q = 0; q < 32; ++q) v[q] = __uint_as_float(r[q]);
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer(uint32_t saddr, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
    return r;
}

// The thread's 32 values as BF16 into the CTA's operand buffer.
__device__ __forceinline__ void store_bf16(const float (&v)[32], unsigned char* base, int row, int group0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t u[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const __nv_bfloat162 b = __floats2bfloat162_rn(v[8 * q + 2 * k], v[8 * q + 2 * k + 1]);
            u[k] = *reinterpret_cast<const uint32_t*>(&b);
        }
        *reinterpret_cast<uint4*>(base + (row >> 3) * TC_ROWS + (group0 + q) * TC_GROUP + (row & 7) * 16) =
            make_uint4(u[0], u[1], u[2], u[3]);
    }
}

// Copy this CTA's units of an operand buffer to the three peers, a row group (1
// KB) per thread and peer, completing on the peers' barrier `bar` (which
// expects PEER_BYTES).  The CTA's stores to it are made visible first.
constexpr uint32_t GROUP_BYTES = (NS / 8) * TC_GROUP, PEER_BYTES = (CL - 1) * (MT / 8) * GROUP_BYTES;
__device__ __forceinline__ void share_units(uint32_t base, uint64_t* bar, int rank, int tid) {
    asm volatile("fence.proxy.async;" ::: "memory");
    __syncthreads();
    if (tid < (CL - 1) * (MT / 8)) {
        const int to = (rank + 1 + tid / (MT / 8)) & (CL - 1);
        const uint32_t at = base + (tid % (MT / 8)) * TC_ROWS + rank * GROUP_BYTES;
        asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         peer(at, to)),
                     "r"(at), "r"(GROUP_BYTES), "r"(peer(hk::smem_u32(bar), to))
                     : "memory");
    }
    __syncwarp();
}

__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
    const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

// Store this CTA's units of an operand buffer to device memory, PIECE bytes of
// a row group per copy: for every block of BLOCK units the 16 row groups are
// contiguous, so k_update brings a block of 128 rows in with one copy.
template <int BLOCK>
__device__ __forceinline__ void store_units(uint32_t base, unsigned char* dst, int cl, int unit0, int tid) {
    constexpr uint32_t BLOCK_BYTES = BLOCK / 8 * TC_GROUP;  // of a row group
    constexpr uint32_t PIECE = BLOCK < NS ? BLOCK_BYTES : GROUP_BYTES;
    constexpr int PIECES = GROUP_BYTES / PIECE;
    if (tid >= 64 && tid < 64 + PIECES * (MT / 8)) {
        const int rg = (tid - 64) % (MT / 8), unit = unit0 + (tid - 64) / (MT / 8) * BLOCK;
        const int64_t at = ((static_cast<int64_t>(cl) * (DH / BLOCK) + unit / BLOCK) * (MT / 8) + rg) * BLOCK_BYTES +
                           unit % BLOCK / 8 * TC_GROUP;
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst + at),
                     "r"(base + rg * TC_ROWS + unit / 8 * TC_GROUP), "r"(PIECE)
                     : "memory");
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    }
    __syncwarp();
}

template <int MODE>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(MLP_THREADS, 1) k_mlp(const __grid_constant__ MlpArgs a) {
    extern __shared__ __align__(1024) unsigned char mlp_smem[];
    MlpSmem& sm = *reinterpret_cast<MlpSmem*>(mlp_smem);
    constexpr bool BWD = MODE != MLP_PREDICT;
    constexpr uint32_t TMEM_COLS = BWD ? 2 * NS : NS;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = blockIdx.x & (CL - 1), cl = blockIdx.x / CL;
    const int row = (warp & 3) * 32 + lane, half = warp >> 2;  // a warp reads TMEM lanes 32 (warp & 3) ..
    const int row0 = cl * MT, unit0 = rank * NS, u0 = half * 32;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(hk::smem_u32(&sm.tmem)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int b = 0; b < 6; ++b) hk::mbar_init(&sm.bar[b], 1);
        hk::fence_barrier_init();
        hk::mbar_arrive_expect_tx(&sm.bar[4], PEER_BYTES);
        if (BWD) hk::mbar_arrive_expect_tx(&sm.bar[5], PEER_BYTES);
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // A training minibatch comes from the data set, which no launch before this
    // one writes; other inputs may come from the caller's last kernel.
    if (MODE != MLP_TRAIN) asm volatile("griddepcontrol.wait;" ::: "memory");
    {  // inputs (threads 0-127) and targets (128-255) of row tid & 127
        const int r = tid & (MT - 1), b = row0 + r;
        float* dst = tid < MT ? sm.x[r] : sm.t[r];
        float v[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (MODE == MLP_PREDICT) {
            if (tid < MT && b < a.B) {
                for (int k = 0; k < 6; ++k)
                    v[k] = static_cast<float>((a.q[b * 6 + k] - a.stats[k]) * a.stats[28 + k]);
                v[6] = a.f ? static_cast<float>((a.f[b] - a.stats[26]) * a.stats[34]) : 1.f;
            }
        } else if (b < a.B) {
            int64_t src = b;
            if (MODE == MLP_TRAIN) {  // Philox counter: row slot, completed steps
                const uint4 d = philox4x32(make_uint4(static_cast<uint32_t>(b), static_cast<uint32_t>(a.step),
                                                      static_cast<uint32_t>(a.step >> 32), 0x4d4c50u),
                                           make_uint2(static_cast<uint32_t>(a.seed), static_cast<uint32_t>(a.seed >> 32)));
                // u mod n from the reciprocal (the quotient is at most 2 short)
                const uint64_t u = (static_cast<uint64_t>(d.x) << 32) | d.y, nn = static_cast<uint64_t>(a.n);
                uint64_t r = u - __umul64hi(u, a.nrec) * nn;
                if (r >= nn) r -= nn;
                if (r >= nn) r -= nn;
                src = static_cast<int64_t>(r);
            }
            const float* p = tid < MT ? a.Xs + src * DIN : a.Ts + src * DOUT;
            for (int k = 0; k < 7; ++k) v[k] = p[k];
        }
        for (int k = 0; k < 7; ++k) dst[k] = v[k];
    }
    // What stands above needs no weights, so it overlaps the end of the launch
    // that updates them (programmatic launch; this waits for it to complete).
    if (MODE == MLP_TRAIN) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (tid == 0) {
        asm volatile("fence.proxy.async;" ::: "memory");
        constexpr uint32_t PACK = NS * 8 * sizeof(float), ROW = DH * sizeof(float);
        hk::mbar_arrive_expect_tx(&sm.bar[3], 2 * PACK + DOUT * ROW + sizeof(sm.b3));
        hk::tma_load_1d(sm.w1, a.W1p + unit0 * 8, PACK, &sm.bar[3]);
        hk::tma_load_1d(sm.w3, a.W3p + unit0 * 8, PACK, &sm.bar[3]);
        for (int o = 0; o < DOUT; ++o) hk::tma_load_1d(sm.w3o[o], a.P + OFF_W3 + o * DH, ROW, &sm.bar[3]);
        hk::tma_load_1d(sm.b3, a.P + OFF_B3, sizeof(sm.b3), &sm.bar[3]);  // (P is allocated in whole vectors)
        hk::mbar_arrive_expect_tx(&sm.bar[0], (BWD ? 2 : 1) * SLICE_BYTES);
        hk::tma_load_1d(sm.w, a.W2s + rank * (SLICE_BYTES / 2), SLICE_BYTES, &sm.bar[0]);
        if (BWD) hk::tma_load_1d(sm.wt, a.W2Ts + rank * (SLICE_BYTES / 2), SLICE_BYTES, &sm.bar[0]);
    }
    const int64_t rows = static_cast<int64_t>(gridDim.x / CL) * MT;  // with padding
    __syncwarp();
    tc_fence_before();
    cluster_sync();  // every CTA runs, and its own set-up is visible
    tc_fence_after();
    const uint32_t tmem = sm.tmem;
    const uint32_t tm = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + static_cast<uint32_t>(u0);

    if (!hk::mbar_wait(&sm.bar[3], 0)) *a.err = HAWKES_ERR_TIMEOUT;
    __syncwarp();
    // layer 1: h1 = tanh(x W1^T + b1)
    float h1[32];
    {
        float x[7];
        for (int k = 0; k < 7; ++k) x[k] = sm.x[row][k];
#pragma unroll
        for (int u = 0; u < 32; ++u) {
            float w[8];
            load8(sm.w1[u0 + u], w);
            float z = w[7];
#pragma unroll
            for (int k = 0; k < DIN; ++k) z = fmaf(w[k], x[k], z);
            h1[u] = tanhf(z);
        }
    }
    const uint32_t sh1 = hk::smem_u32(sm.h1), sdz = hk::smem_u32(sm.dz);
    const int group0 = (unit0 + u0) / 8;
    store_bf16(h1, sm.h1, row, group0);
    share_units(sh1, &sm.bar[4], rank, tid);
    if (BWD) store_units<UT_M>(sh1, a.h1op, cl, unit0, tid);

    // layer 2: h2 = tanh(h1 W2^T + b2)
    if (tid == 0) {
        if (!hk::mbar_wait(&sm.bar[0], 0) || !hk::mbar_wait(&sm.bar[4], 0)) *a.err = HAWKES_ERR_TIMEOUT;
        tc_fence_after();
        const uint32_t sw = hk::smem_u32(sm.w);
        for (int k = 0; k < DH / 16; ++k)
            tc_mma(tmem, smem_desc(sh1 + 2 * k * TC_GROUP, TC_GROUP, TC_ROWS),
                   smem_desc(sw + 2 * k * TC_GROUP, TC_GROUP, TC_ROWS), TC_IDESC, k > 0);
        tc_commit(&sm.bar[1]);
    }
    __syncwarp();
    if (!hk::mbar_wait(&sm.bar[1], 0)) *a.err = HAWKES_ERR_TIMEOUT;
    __syncwarp();
    tc_fence_after();
    float h2[32];
    tc_load32(tm, h2);
#pragma unroll
    for (int u = 0; u < 32; ++u) h2[u] = tanhf(h2[u] + sm.w3[u0 + u][7]);

    // outputs: y = h2 W3^T + b3, one chain along the hidden units per row and
    // output.  The 32 rows of a warp go to CTA warp & 3, whose warps 0 and 1
    // form outputs 0-3 and 4-6 of a row per lane.
    {
        const uint32_t at = peer(sdz + (lane * YPITCH + unit0 + u0) * 4, warp & 3);
#pragma unroll
        for (int q = 0; q < 8; ++q)
            asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at + 16 * q), "f"(h2[4 * q]),
                         "f"(h2[4 * q + 1]), "f"(h2[4 * q + 2]), "f"(h2[4 * q + 3])
                         : "memory");
    }
    __syncwarp();
    cluster_sync();
    if (warp < 2) {
        const int r = rank * YROWS + lane;  // row of the cluster
        const bool real = row0 + r < a.B;
        const float4* h = reinterpret_cast<const float4*>(sm.dz) + lane * (YPITCH / 4);
        float y[4], dv[4];
#pragma unroll
        for (int o = 0; o < 4; ++o) y[o] = sm.b3[4 * warp + o];
#pragma unroll 4
        for (int j = 0; j < DH / 4; ++j) {
            const float4 v = h[j];
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                const float4 w = *reinterpret_cast<const float4*>(&sm.w3o[4 * warp + o][4 * j]);
                y[o] = fmaf(w.x, v.x, y[o]);
                y[o] = fmaf(w.y, v.y, y[o]);
                y[o] = fmaf(w.z, v.z, y[o]);
                y[o] = fmaf(w.w, v.w, y[o]);
            }
        }
        double sq = 0.0;
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            const int oo = 4 * warp + o;
            dv[o] = 0.f;
            if (oo >= DOUT) continue;
            if (MODE == MLP_PREDICT) {
                if (real)
                    a.pred[static_cast<int64_t>(row0 + r) * DOUT + oo] =
                        a.stats[12 + oo] + a.stats[19 + oo] * static_cast<double>(y[o]);
            } else {
                const float d = real ? y[o] - sm.t[r][oo] : 0.f;
                dv[o] = 2.f * d / static_cast<float>(DOUT * a.B);
                if (a.loss) sq += static_cast<double>(d) * d;
                if (MODE == MLP_GIVEN && a.Y && real) a.Y[(row0 + r) * DOUT + oo] = y[o];
            }
        }
        if (BWD) {
            const uint32_t at = hk::smem_u32(&sm.dy[r][4 * warp]);
#pragma unroll
            for (int c = 0; c < CL; ++c)
                asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(peer(at, c)), "f"(dv[0]), "f"(dv[1]),
                             "f"(dv[2]), "f"(dv[3])
                             : "memory");
            if (a.loss) {
                for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
                if (lane == 0) atomicAdd(a.loss, sq / (DOUT * a.B));
            }
        }
    }
    __syncwarp();
    if (BWD) {
        cluster_sync();
        // dz2 = (dy W3) (1 - h2^2)
        float dz[32];
        {
            float dy[8];
            load8(sm.dy[row], dy);
#pragma unroll
            for (int u = 0; u < 32; ++u) {
                float w[8];
                load8(sm.w3[u0 + u], w);
                float g = 0.f;
#pragma unroll
                for (int o = 0; o < DOUT; ++o) g = fmaf(dy[o], w[o], g);
                dz[u] = g * (1.f - h2[u] * h2[u]);
            }
        }
        store_bf16(dz, sm.dz, row, group0);
        share_units(sdz, &sm.bar[5], rank, tid);
        store_units<UT_N>(sdz, a.dzop, cl, unit0, tid);
        if (tid == 0) {
            if (!hk::mbar_wait(&sm.bar[5], 0)) *a.err = HAWKES_ERR_TIMEOUT;
            tc_fence_after();
            const uint32_t swt = hk::smem_u32(sm.wt);
            for (int k = 0; k < DH / 16; ++k)
                tc_mma(tmem + NS, smem_desc(sdz + 2 * k * TC_GROUP, TC_GROUP, TC_ROWS),
                       smem_desc(swt + 2 * k * TC_GROUP, TC_GROUP, TC_ROWS), TC_IDESC, k > 0);
            tc_commit(&sm.bar[2]);
        }
        __syncwarp();
        // (stores to device memory stay behind the barriers, which would wait for them)
        {
            const int64_t r = row0 + (tid >> 1);
            if (rank == 0)
                reinterpret_cast<float4*>(a.dyo + r * 8)[tid & 1] = reinterpret_cast<const float4*>(sm.dy[tid >> 1])[tid & 1];
            if (rank == 1)
                reinterpret_cast<float4*>(a.xin + r * 8)[tid & 1] = reinterpret_cast<const float4*>(sm.x[tid >> 1])[tid & 1];
        }
#pragma unroll
        for (int u = 0; u < 32; ++u) {
            const int64_t at = (unit0 + u0 + u) * rows + row0 + row;
            a.h2t[at] = h2[u];
            a.dz2t[at] = dz[u];
        }
        if (!hk::mbar_wait(&sm.bar[2], 0)) *a.err = HAWKES_ERR_TIMEOUT;
        __syncwarp();
        tc_fence_after();
        tc_load32(tm + NS, dz);
#pragma unroll
        for (int u = 0; u < 32; ++u)
            a.dz1t[(unit0 + u0 + u) * rows + row0 + row] = dz[u] * (1.f - h1[u] * h1[u]);
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    if (tid == 0) {  // (again, bounded, if a wait above gave up)
        (void)hk::mbar_wait(&sm.bar[4], 0);
        if (BWD) (void)hk::mbar_wait(&sm.bar[5], 0);
    }
    __syncwarp();
    // A CTA's copies to its peers read its shared memory; past this barrier they
    // have landed (each peer has waited for them).
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
}

// ---------------------------------------------------------------------------
// Gradients of one minibatch and, with UPDATE, the Adam step (bias-corrected;
// step: completed steps) and the refreshed BF16 copies of W2; without it the
// gradient goes to G.
//   blocks [0, 16): 128 input units x 32 output units of W2: dW2 = dz2^T h1 over
//     the rows, 128 rows per two-stage buffer, on the tensor cores; operands
//     MN-major (units contiguous): the step along the units is 128 bytes, along
//     K (8 rows) a row group of the stage's tile;
//   blocks 16 + j, j < 256: unit j's row of W1, b1, b2 and column of W3;
//   the last block: b3.
// ---------------------------------------------------------------------------
constexpr int UT_BLOCKS = (DH / UT_M) * (DH / UT_N), UPDATE_BLOCKS = UT_BLOCKS + DH + 1;
constexpr uint32_t UT_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((UT_N >> 3) << 17) |
                              ((UT_M >> 4) << 24);
constexpr uint32_t UT_RA = (UT_M / 8) * 128, UT_RB = (UT_N / 8) * 128;  // row group of the stage's A and B
struct UpdateSmem {
    unsigned char a[2][MT / 8 * UT_RA], b[2][MT / 8 * UT_RB];
    uint64_t full[2], done[2], all;  // stage loaded, stage read, every product done
    uint32_t tmem;
};

struct UpdateArgs {
    const unsigned char *h1op, *dzop;
    const float *h2t, *dz2t, *dz1t, *xin, *dyo;
    int B, clusters;
    float *P, *M, *V, *G;
    uint64_t step;
    float lr;
    float *W1p, *W3p;
    bf16 *W2s, *W2Ts;
    volatile int* err;
};

template <bool UPDATE>
__device__ __forceinline__ float apply(const UpdateArgs& a, int i, float g, float p0, float m0, float v0,
                                       float c1, float c2) {
    if (!UPDATE) {
        a.G[i] = g;
        return 0.f;
    }
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float m = b1 * m0 + (1.f - b1) * g;
    const float v = b2 * v0 + (1.f - b2) * g * g;
    a.M[i] = m;
    a.V[i] = v;
    const float mh = m / c1, vh = v / c2;
    const float p = p0 - a.lr * mh / (sqrtf(vh) + eps);
    a.P[i] = p;
    return p;
}

template <bool UPDATE>
__global__ void __launch_bounds__(MLP_THREADS) k_update(const __grid_constant__ UpdateArgs a) {
    extern __shared__ __align__(1024) unsigned char mlp_smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const float tt = static_cast<float>(a.step + 1);  // this update's 1-based step number
    const float c1 = 1.f - powf(0.9f, tt), c2 = 1.f - powf(0.999f, tt);
    if (blockIdx.x < UT_BLOCKS) {
        UpdateSmem& sm = *reinterpret_cast<UpdateSmem*>(mlp_smem);
        const int i0 = (blockIdx.x / (DH / UT_N)) * UT_M, j0 = (blockIdx.x % (DH / UT_N)) * UT_N;
        if (warp == 0) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(hk::smem_u32(&sm.tmem)),
                         "r"(UT_N)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        if (tid == 0) {
            for (int b = 0; b < 2; ++b) {
                hk::mbar_init(&sm.full[b], 1);
                hk::mbar_init(&sm.done[b], 1);
            }
            hk::mbar_init(&sm.all, 1);
            hk::fence_barrier_init();
        }
        __syncwarp();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        const uint32_t tmem = sm.tmem;
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (warp == 0) {
            asm volatile("fence.proxy.async;" ::: "memory");
            bool ok = true;
            // stage c & 1 <- rows [128 c, 128 c + 128)
            auto load = [&](int c) {
                const int s = c & 1;
                if (lane == 0) {
                    hk::mbar_arrive_expect_tx(&sm.full[s], sizeof(sm.a[0]) + sizeof(sm.b[0]));
                    hk::tma_load_1d(sm.a[s], a.h1op + (static_cast<int64_t>(c) * (DH / UT_M) + i0 / UT_M) * sizeof(sm.a[0]),
                                    sizeof(sm.a[0]), &sm.full[s]);
                    hk::tma_load_1d(sm.b[s], a.dzop + (static_cast<int64_t>(c) * (DH / UT_N) + j0 / UT_N) * sizeof(sm.b[0]),
                                    sizeof(sm.b[0]), &sm.full[s]);
                }
                __syncwarp();
            };
            for (int c = 0; c < 2 && c < a.clusters; ++c) load(c);
            for (int c = 0; c < a.clusters; ++c) {
                const int s = c & 1;
                if (lane == 0) {
                    ok = hk::mbar_wait(&sm.full[s], (c >> 1) & 1) && ok;
                    tc_fence_after();
                    const uint32_t sa = hk::smem_u32(sm.a[s]), sb = hk::smem_u32(sm.b[s]);
                    for (int k = 0; k < MT / 16; ++k)
                        tc_mma(tmem, smem_desc(sa + 2 * k * UT_RA, UT_RA, 128), smem_desc(sb + 2 * k * UT_RB, UT_RB, 128),
                               UT_IDESC, c > 0 || k > 0);
                    tc_commit(&sm.done[s]);
                }
                __syncwarp();
                if (c + 2 < a.clusters) {
                    ok = hk::mbar_wait(&sm.done[s], (c >> 1) & 1) && ok;
                    __syncwarp();
                    load(c + 2);
                }
            }
            if (lane == 0) tc_commit(&sm.all);
            if (!ok) *a.err = HAWKES_ERR_TIMEOUT;
        }
        __syncwarp();
        const int i = i0 + (warp & 3) * 32 + lane, u0 = (warp >> 2) * (UT_N / 2);
        float p[16], m[16], v[16];  // loaded together, ahead of the stores
        if (UPDATE)
#pragma unroll
            for (int u = 0; u < 16; ++u) {
                const int at = OFF_W2 + (j0 + u0 + u) * DH + i;
                p[u] = a.P[at];
                m[u] = a.M[at];
                v[u] = a.V[at];
            }
        if (!hk::mbar_wait(&sm.all, 0)) *a.err = HAWKES_ERR_TIMEOUT;
        __syncwarp();
        tc_fence_after();
        uint32_t r[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
              "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
            : "r"(tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16) + static_cast<uint32_t>(u0)));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            const int j = j0 + u0 + u;
            const float w = apply<UPDATE>(a, OFF_W2 + j * DH + i, __uint_as_float(r[u]), p[u], m[u], v[u], c1, c2);
            if (UPDATE) {
                const bf16 b = __float2bfloat16_rn(w);
                a.W2s[slice_off(j, i) / 2] = b;
                a.W2Ts[slice_off(i, j) / 2] = b;
            }
        }
        tc_fence_before();
        __syncthreads();
        if (warp == 0)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(UT_N) : "memory");
        return;
    }
    // Sums over the batch: thread t takes rows t, t + 256, ...; then a binary
    // tree over the threads.
    float(*red)[256] = reinterpret_cast<float(*)[256]>(mlp_smem);
    const int j = blockIdx.x - UT_BLOCKS;
    const int64_t rows = static_cast<int64_t>(a.clusters) * MT;
    float g[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) g[q] = 0.f;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (j < DH) {
        for (int b = tid; b < a.B; b += 256) {
            const float h2 = a.h2t[j * rows + b], d2 = a.dz2t[j * rows + b], d1 = a.dz1t[j * rows + b];
            float dy[8], x[8];
            load8(a.dyo + static_cast<int64_t>(b) * 8, dy);
            load8(a.xin + static_cast<int64_t>(b) * 8, x);
#pragma unroll
            for (int o = 0; o < 7; ++o) {
                g[o] = fmaf(dy[o], h2, g[o]);
                g[8 + o] = fmaf(d1, x[o], g[8 + o]);
            }
            g[7] += d2;
            g[15] += d1;
        }
    } else {
        for (int b = tid; b < a.B; b += 256) {
            float dy[8];
            load8(a.dyo + static_cast<int64_t>(b) * 8, dy);
#pragma unroll
            for (int o = 0; o < 7; ++o) g[o] += dy[o];
        }
    }
#pragma unroll
    for (int q = 0; q < 16; ++q) red[q][tid] = g[q];
    __syncthreads();
    for (int w = 128; w >= 32; w >>= 1) {
        for (int k = tid; k < 16 * w; k += 256) red[k / w][k % w] += red[k / w][k % w + w];
        __syncthreads();
    }
#pragma unroll
    for (int q = warp; q < 16; q += 8) {
        float v = red[q][lane];
        for (int w = 16; w > 0; w >>= 1) v += __shfl_down_sync(0xffffffffu, v, w);
        if (lane == 0) red[q][0] = v;
    }
    __syncthreads();
    if (tid < (j < DH ? 16 : DOUT)) {
        const int at = j == DH ? OFF_B3 + tid : tid < 7 ? OFF_W3 + tid * DH + j : tid == 7 ? OFF_B2 + j
                       : tid < 15 ? OFF_W1 + j * DIN + tid - 8 : OFF_B1 + j;
        const float w = UPDATE ? apply<true>(a, at, red[tid][0], a.P[at], a.M[at], a.V[at], c1, c2)
                               : apply<false>(a, at, red[tid][0], 0.f, 0.f, 0.f, c1, c2);
        if (UPDATE && j < DH) (tid < 8 ? a.W3p : a.W1p)[j * 8 + (tid & 7)] = w;
    }
}

// The copies of the weights that k_mlp reads, from the parameters.
__global__ void k_refresh(const float* __restrict__ P, float* __restrict__ W1p, float* __restrict__ W3p,
                          bf16* __restrict__ W2s, bf16* __restrict__ W2Ts) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= DH * DH) return;
    const int r = i / DH, c = i % DH;
    const bf16 v = __float2bfloat16_rn(P[OFF_W2 + i]);
    W2s[slice_off(r, c) / 2] = v;
    W2Ts[slice_off(c, r) / 2] = v;
    if (i < DH * 8) {
        const int u = i >> 3, k = i & 7;
        W1p[i] = k < DIN ? P[OFF_W1 + u * DIN + k] : P[OFF_B1 + u];
        W3p[i] = k < DOUT ? P[OFF_W3 + k * DH + u] : P[OFF_B2 + u];
    }
}

// Column means and standard deviations (FP64) of X[n x 6], Y[n x 7] and the
// optional feature F[n], then the standardised FP32 copies (the 7th input is
// the standardised feature, or the constant 1 without one).
__global__ void k_stats(const double* __restrict__ X, const double* __restrict__ Y,
                        const double* __restrict__ F, int64_t n,
                        double* stats /* mean_in[6] sd_in[6] mean_out[7] sd_out[7] mean_f sd_f, then 1/sd_in[6] 1/sd_f */) {
    const int col = blockIdx.x;  // 0..5 inputs, 6..12 outputs, 13 the feature
    if (col == 13 && !F) {
        if (threadIdx.x == 0) {
            stats[26] = 0.0;
            stats[27] = 1.0;
            stats[34] = 1.0;
        }
        return;
    }
    const double* src = col < 6 ? X : col < 13 ? Y : F;
    const int w = col < 6 ? 6 : col < 13 ? 7 : 1, c = col < 6 ? col : col < 13 ? col - 6 : 0;
    double s = 0.0, s2 = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        const double v = src[i * w + c];
        s += v;
        s2 += v * v;
    }
    __shared__ double r1[256], r2[256];
    r1[threadIdx.x] = s;
    r2[threadIdx.x] = s2;
    __syncthreads();
    for (int k = blockDim.x / 2; k > 0; k >>= 1) {
        if (threadIdx.x < k) {
            r1[threadIdx.x] += r1[threadIdx.x + k];
            r2[threadIdx.x] += r2[threadIdx.x + k];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double mean = r1[0] / n;
        double var = r2[0] / n - mean * mean;
        double sd = var > 0.0 ? sqrt(var) : 0.0;
        if (!(sd > 1e-12 * (fabs(mean) + 1e-300))) sd = 1.0;  // constant column
        if (col < 6) {
            stats[col] = mean;
            stats[6 + col] = sd;
            stats[28 + col] = 1.0 / sd;
        } else if (col < 13) {
            stats[12 + c] = mean;
            stats[19 + c] = sd;
        } else {
            stats[26] = mean;
            stats[27] = sd;
            stats[34] = 1.0 / sd;
        }
    }
}

__global__ void k_standardise(const double* __restrict__ X, const double* __restrict__ Y,
                              const double* __restrict__ F, int64_t n,
                              const double* __restrict__ st, float* __restrict__ Xs,
                              float* __restrict__ Ts) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        for (int k = 0; k < 6; ++k) Xs[i * DIN + k] = static_cast<float>((X[i * 6 + k] - st[k]) / st[6 + k]);
        Xs[i * DIN + 6] = F ? static_cast<float>((F[i] - st[26]) / st[27]) : 1.f;
        if (Y)
            for (int k = 0; k < 7; ++k)
                Ts[i * DOUT + k] = static_cast<float>((Y[i * 7 + k] - st[12 + k]) / st[19 + k]);
    }
}

__global__ void k_init_params(float* P, uint64_t seed) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NPARAMS) return;
    float lim = 0.f;  // biases start at zero
    if (i < OFF_B1) lim = sqrtf(6.f / (DH + DIN));
    else if (i >= OFF_W2 && i < OFF_B2) lim = sqrtf(6.f / (DH + DH));
    else if (i >= OFF_W3 && i < OFF_B3) lim = sqrtf(6.f / (DOUT + DH));
    const uint4 r = philox4x32(make_uint4(static_cast<uint32_t>(i), 0u, 0u, 0x494e4954u),
                               make_uint2(static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32)));
    const float u = (r.x >> 8) * (1.f / 16777216.f);
    P[i] = lim * (2.f * u - 1.f);
}

}  // namespace

struct hawkes_mlp {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    float *P = nullptr, *G = nullptr, *M = nullptr, *V = nullptr;
    float *W1p = nullptr, *W3p = nullptr;  // packed copies of the 7-wide layers (MlpArgs)
    bf16 *W2s = nullptr, *W2Ts = nullptr;  // sliced BF16 copies of W2 and W2^T
    uint64_t step = 0;                     // completed Adam steps
    double* loss = nullptr;
    double* stats = nullptr;  // 28 values, then reciprocals (k_stats)
    bool have_stats = false;
    bool have_feature = false;  // the 7th input is a feature (else the constant 1)
    int64_t n = 0;
    float *Xs = nullptr, *Ts = nullptr;  // standardised data set
    float *X = nullptr, *T = nullptr, *Y = nullptr;  // one batch given by the caller
    unsigned char *h1op = nullptr, *dzop = nullptr;  // k_mlp to k_update (see MlpArgs)
    float *h2t = nullptr, *dz2t = nullptr, *dz1t = nullptr, *xin = nullptr, *dyo = nullptr;
    double* hbuf = nullptr;  // pinned host copy of the loss
    int* err = nullptr;      // pinned host: latched device error (a wait that gave up)
};

namespace {

int st_of(cudaError_t e) {
    if (e == cudaSuccess) return HAWKES_OK;
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? HAWKES_ERR_OOM : HAWKES_ERR_CUDA;
}
#define HM_TRY(expr)                      \
    do {                                  \
        int _rc = (expr);                 \
        if (_rc != HAWKES_OK) return _rc; \
    } while (0)
#define HM_CUDA(expr) HM_TRY(st_of(expr))

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) cudaSetDevice(dev);
    }
    ~DeviceGuard() {
        int cur = -1;
        if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
    }
};

template <typename T>
int alloc(T** p, size_t count) {
    return st_of(cudaMalloc(reinterpret_cast<void**>(p), (count ? count : 1) * sizeof(T)));
}

// Wait for the queued work; the latched device error, cleared.
int take_err(hawkes_mlp* m) {
    HM_CUDA(cudaStreamSynchronize(m->stream));
    const int e = *static_cast<volatile int*>(m->err);
    *static_cast<volatile int*>(m->err) = 0;
    return e;
}

MlpArgs args_of(const hawkes_mlp* m, int B) {
    MlpArgs a{};
    a.P = m->P;
    a.W1p = m->W1p;
    a.W3p = m->W3p;
    a.W2s = m->W2s;
    a.W2Ts = m->W2Ts;
    a.B = B;
    a.h1op = m->h1op;
    a.dzop = m->dzop;
    a.h2t = m->h2t;
    a.dz2t = m->dz2t;
    a.dz1t = m->dz1t;
    a.xin = m->xin;
    a.dyo = m->dyo;
    a.err = m->err;
    return a;
}

template <int MODE>
int launch_mlp(hawkes_mlp* m, const MlpArgs& a) {
    return st_of(hk::launch_chained(k_mlp<MODE>, CL * ((a.B + MT - 1) / MT), MLP_THREADS, sizeof(MlpSmem), m->stream, a));
}

template <bool UPDATE>
int launch_update(hawkes_mlp* m, int B, float lr) {
    UpdateArgs a{};
    a.h1op = m->h1op; a.dzop = m->dzop;
    a.h2t = m->h2t; a.dz2t = m->dz2t; a.dz1t = m->dz1t; a.xin = m->xin; a.dyo = m->dyo;
    a.B = B;
    a.clusters = (B + MT - 1) / MT;
    a.P = m->P; a.M = m->M; a.V = m->V; a.G = m->G;
    a.step = m->step;
    a.lr = lr;
    a.W1p = m->W1p; a.W3p = m->W3p;
    a.W2s = m->W2s; a.W2Ts = m->W2Ts;
    a.err = m->err;
    return st_of(hk::launch_chained(k_update<UPDATE>, UPDATE_BLOCKS, MLP_THREADS, sizeof(UpdateSmem), m->stream, a));
}

}  // namespace

extern "C" {

int hawkes_mlp_create(hawkes_mlp** out, int device, void* cuda_stream, uint64_t seed) {
    HK_NVTX("hawkes_mlp_create");
    if (!out) return HAWKES_ERR_ARG;
    *out = nullptr;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) {
        cudaGetLastError();
        return device < 0 ? HAWKES_ERR_ARG : HAWKES_ERR_CUDA;
    }
    DeviceGuard g(device);
    hawkes_mlp* m = new (std::nothrow) hawkes_mlp();
    if (!m) return HAWKES_ERR_OOM;
    m->device = device;
    int rc = HAWKES_OK;
    do {
        if (cuda_stream) {
            m->stream = static_cast<cudaStream_t>(cuda_stream);
        } else {
            if ((rc = st_of(cudaStreamCreateWithFlags(&m->stream, cudaStreamNonBlocking)))) break;
            m->own_stream = true;
        }
        if ((rc = alloc(&m->P, NPARAMS + 1)) || (rc = alloc(&m->W1p, DH * 8)) || (rc = alloc(&m->W3p, DH * 8)) ||
            (rc = alloc(&m->G, NPARAMS)) || (rc = alloc(&m->M, NPARAMS)) ||
            (rc = alloc(&m->V, NPARAMS)) || (rc = alloc(&m->W2s, DH * DH)) || (rc = alloc(&m->W2Ts, DH * DH)) ||
            (rc = alloc(&m->loss, 1)) || (rc = alloc(&m->stats, 40)) || (rc = alloc(&m->X, BMAX * DIN)) ||
            (rc = alloc(&m->T, BMAX * DOUT)) || (rc = alloc(&m->Y, BMAX * DOUT)) ||
            (rc = alloc(&m->h1op, BMAX * DH * 2)) || (rc = alloc(&m->dzop, BMAX * DH * 2)) ||
            (rc = alloc(&m->h2t, BMAX * DH)) || (rc = alloc(&m->dz2t, BMAX * DH)) ||
            (rc = alloc(&m->dz1t, BMAX * DH)) || (rc = alloc(&m->xin, BMAX * 8)) || (rc = alloc(&m->dyo, BMAX * 8)))
            break;
        if ((rc = st_of(cudaMallocHost(reinterpret_cast<void**>(&m->hbuf), sizeof(double))))) break;
        if ((rc = st_of(cudaMallocHost(reinterpret_cast<void**>(&m->err), sizeof(int))))) break;
        *m->err = 0;
        for (const void* f : {reinterpret_cast<const void*>(k_mlp<MLP_PREDICT>),
                              reinterpret_cast<const void*>(k_mlp<MLP_TRAIN>),
                              reinterpret_cast<const void*>(k_mlp<MLP_GIVEN>)})
            if ((rc = st_of(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 static_cast<int>(sizeof(MlpSmem))))))
                break;
        for (const void* f : {reinterpret_cast<const void*>(k_update<true>), reinterpret_cast<const void*>(k_update<false>)})
            if (rc == HAWKES_OK)
                rc = st_of(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                static_cast<int>(sizeof(UpdateSmem))));
        if (rc) break;
        k_init_params<<<(NPARAMS + 255) / 256, 256, 0, m->stream>>>(m->P, seed);
        k_refresh<<<DH * DH / 256, 256, 0, m->stream>>>(m->P, m->W1p, m->W3p, m->W2s, m->W2Ts);
        if ((rc = st_of(cudaMemsetAsync(m->M, 0, NPARAMS * sizeof(float), m->stream))) ||
            (rc = st_of(cudaMemsetAsync(m->V, 0, NPARAMS * sizeof(float), m->stream))) ||
            (rc = st_of(cudaMemsetAsync(m->loss, 0, sizeof(double), m->stream))) ||
            (rc = st_of(cudaStreamSynchronize(m->stream))))
            break;
    } while (0);
    if (rc != HAWKES_OK) {
        hawkes_mlp_destroy(m);
        return rc;
    }
    *out = m;
    return HAWKES_OK;
}

void hawkes_mlp_destroy(hawkes_mlp* m) {
    HK_NVTX("hawkes_mlp_destroy");
    if (!m) return;
    DeviceGuard g(m->device);
    if (m->stream) cudaStreamSynchronize(m->stream);
    for (void* p : {(void*)m->P, (void*)m->G, (void*)m->M, (void*)m->V, (void*)m->W1p, (void*)m->W3p,
                    (void*)m->W2s, (void*)m->W2Ts,
                    (void*)m->loss, (void*)m->stats, (void*)m->Xs, (void*)m->Ts, (void*)m->X, (void*)m->T,
                    (void*)m->Y, (void*)m->h1op, (void*)m->dzop, (void*)m->h2t, (void*)m->dz2t, (void*)m->dz1t,
                    (void*)m->xin, (void*)m->dyo})
        if (p) cudaFree(p);
    if (m->err) cudaFreeHost(m->err);
    if (m->hbuf) cudaFreeHost(m->hbuf);
    if (m->own_stream && m->stream) cudaStreamDestroy(m->stream);
    cudaGetLastError();
    delete m;
}

int hawkes_mlp_get_params(hawkes_mlp* m, float* params) {
    HK_NVTX("hawkes_mlp_get_params");
    if (!m || !params) return HAWKES_ERR_ARG;
    DeviceGuard g(m->device);
    HM_CUDA(cudaMemcpyAsync(params, m->P, NPARAMS * sizeof(float), cudaMemcpyDeviceToHost, m->stream));
    return st_of(cudaStreamSynchronize(m->stream));
}

int hawkes_mlp_set_params(hawkes_mlp* m, const float* params) {
    HK_NVTX("hawkes_mlp_set_params");
    if (!m || !params) return HAWKES_ERR_ARG;
    DeviceGuard g(m->device);
    HM_CUDA(cudaMemcpyAsync(m->P, params, NPARAMS * sizeof(float), cudaMemcpyHostToDevice, m->stream));
    k_refresh<<<DH * DH / 256, 256, 0, m->stream>>>(m->P, m->W1p, m->W3p, m->W2s, m->W2Ts);
    HM_CUDA(cudaMemsetAsync(m->M, 0, NPARAMS * sizeof(float), m->stream));
    HM_CUDA(cudaMemsetAsync(m->V, 0, NPARAMS * sizeof(float), m->stream));
    m->step = 0;
    return st_of(cudaStreamSynchronize(m->stream));
}

int hawkes_mlp_set_data(hawkes_mlp* m, int64_t n, const double* X, const double* F,
                        const double* Y) {
    HK_NVTX("hawkes_mlp_set_data");
    if (!m || n < 2 || !X || !Y) return HAWKES_ERR_ARG;
    DeviceGuard g(m->device);
    HM_CUDA(cudaStreamSynchronize(m->stream));
    if (m->Xs) cudaFree(m->Xs);
    if (m->Ts) cudaFree(m->Ts);
    m->Xs = m->Ts = nullptr;
    m->have_stats = false;
    double *dX = nullptr, *dY = nullptr, *dF = nullptr;
    int rc = HAWKES_OK;
    if ((rc = alloc(&m->Xs, n * DIN)) || (rc = alloc(&m->Ts, n * DOUT)) || (rc = alloc(&dX, n * 6)) ||
        (rc = alloc(&dY, n * 7)) || (F && (rc = alloc(&dF, n)))) {
        if (dX) cudaFree(dX);
        if (dY) cudaFree(dY);
        if (dF) cudaFree(dF);
        return rc;
    }
    cudaStream_t st = m->stream;
    if ((rc = st_of(cudaMemcpyAsync(dX, X, n * 6 * sizeof(double), cudaMemcpyHostToDevice, st))) == HAWKES_OK &&
        (rc = st_of(cudaMemcpyAsync(dY, Y, n * 7 * sizeof(double), cudaMemcpyHostToDevice, st))) == HAWKES_OK &&
        (!F || (rc = st_of(cudaMemcpyAsync(dF, F, n * sizeof(double), cudaMemcpyHostToDevice, st))) == HAWKES_OK)) {
        k_stats<<<14, 256, 0, st>>>(dX, dY, dF, n, m->stats);
        k_standardise<<<256, 256, 0, st>>>(dX, dY, dF, n, m->stats, m->Xs, m->Ts);
        rc = st_of(cudaStreamSynchronize(st));
    }
    cudaFree(dX);
    cudaFree(dY);
    if (dF) cudaFree(dF);
    if (rc != HAWKES_OK) return rc;
    m->n = n;
    m->have_stats = true;
    m->have_feature = F != nullptr;
    return HAWKES_OK;
}

int hawkes_mlp_train(hawkes_mlp* m, int64_t steps, int batch, double lr, uint64_t seed,
                     double* last_loss) {
    HK_NVTX("hawkes_mlp_train");
    if (!m || steps < 0 || batch < 64 || batch > BMAX || batch % 64 != 0 || !(lr > 0)) return HAWKES_ERR_ARG;
    if (!m->have_stats || !m->Xs) return HAWKES_ERR_STATE;
    DeviceGuard g(m->device);
    MlpArgs a = args_of(m, batch);
    a.Xs = m->Xs;
    a.Ts = m->Ts;
    a.n = m->n;
    a.seed = seed;
    a.nrec = ~0ull / static_cast<uint64_t>(m->n);
    if (steps > 0) HM_CUDA(cudaMemsetAsync(m->loss, 0, sizeof(double), m->stream));  // (no step: the last loss stays)
    for (int64_t s = 0; s < steps; ++s) {
        a.step = m->step;
        a.loss = s == steps - 1 ? m->loss : nullptr;  // the last minibatch's
        HM_TRY(launch_mlp<MLP_TRAIN>(m, a));
        HM_TRY(launch_update<true>(m, batch, static_cast<float>(lr)));
        m->step += 1;
    }
    HM_CUDA(cudaGetLastError());
    if (last_loss) HM_CUDA(cudaMemcpyAsync(m->hbuf, m->loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream));
    const int rc = take_err(m);
    if (last_loss) *last_loss = m->hbuf[0];
    return rc;
}

int hawkes_mlp_loss_grad(hawkes_mlp* m, int batch, const float* Xs, const float* Ts, double* loss,
                         float* grad, float* Y) {
    HK_NVTX("hawkes_mlp_loss_grad");
    if (!m || batch < 64 || batch > BMAX || batch % 64 != 0 || !Xs || !Ts) return HAWKES_ERR_ARG;
    DeviceGuard g(m->device);
    cudaStream_t st = m->stream;
    HM_CUDA(cudaMemcpyAsync(m->X, Xs, batch * DIN * sizeof(float), cudaMemcpyHostToDevice, st));
    HM_CUDA(cudaMemcpyAsync(m->T, Ts, batch * DOUT * sizeof(float), cudaMemcpyHostToDevice, st));
    HM_CUDA(cudaMemsetAsync(m->loss, 0, sizeof(double), st));
    MlpArgs a = args_of(m, batch);
    a.Xs = m->X;
    a.Ts = m->T;
    a.Y = m->Y;
    a.loss = m->loss;
    HM_TRY(launch_mlp<MLP_GIVEN>(m, a));
    HM_TRY(launch_update<false>(m, batch, 0.f));
    if (grad) HM_CUDA(cudaMemcpyAsync(grad, m->G, NPARAMS * sizeof(float), cudaMemcpyDeviceToHost, st));
    if (Y) HM_CUDA(cudaMemcpyAsync(Y, m->Y, batch * DOUT * sizeof(float), cudaMemcpyDeviceToHost, st));
    HM_CUDA(cudaMemcpyAsync(m->hbuf, m->loss, sizeof(double), cudaMemcpyDeviceToHost, st));
    const int rc = take_err(m);
    if (loss) *loss = m->hbuf[0];
    return rc;
}

int hawkes_mlp_predict(hawkes_mlp* m, int64_t count, const double* d_logp, const double* d_feature,
                       double* d_out) {
    HK_NVTX("hawkes_mlp_predict");
    if (!m || count < 1 || count > BMAX || !d_logp || !d_out || !hk::aligned8(d_logp) ||
        !hk::aligned8(d_out) || !hk::aligned8(d_feature))
        return HAWKES_ERR_ARG;
    if (!m->have_stats || (d_feature != nullptr) != m->have_feature) return HAWKES_ERR_STATE;
    DeviceGuard g(m->device);
    MlpArgs a = args_of(m, static_cast<int>(count));
    a.q = d_logp;
    a.f = d_feature;
    a.stats = m->stats;
    a.pred = d_out;
    return launch_mlp<MLP_PREDICT>(m, a);
}

int hawkes_mlp_stats(hawkes_mlp* m, double* stats28) {
    HK_NVTX("hawkes_mlp_stats");
    if (!m || !stats28) return HAWKES_ERR_ARG;
    if (!m->have_stats) return HAWKES_ERR_STATE;
    DeviceGuard g(m->device);
    HM_CUDA(cudaMemcpyAsync(stats28, m->stats, 28 * sizeof(double), cudaMemcpyDeviceToHost, m->stream));
    return st_of(cudaStreamSynchronize(m->stream));
}

int hawkes_mlp_wait(hawkes_mlp* m) {
    HK_NVTX("hawkes_mlp_wait");
    if (!m) return HAWKES_ERR_ARG;
    DeviceGuard g(m->device);
    return take_err(m);
}

}  // extern "C"
