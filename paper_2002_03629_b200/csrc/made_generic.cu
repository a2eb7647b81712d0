// CUDA-core path of the masked-MLP sampler: one persistent cooperative kernel
// that runs the whole solver (Algorithms 1-3 of arXiv 2002.03629, or the strict
// feedforward order of Eq. 1) on the device.  It serves fp32 models, shapes the
// tensor-core path does not cover, and the fine-grained sweeps of Jacobi-GS.
//
// Every CTA executes the same driver loop; decisions are taken from values all
// CTAs read identically after a grid barrier, so control flow never diverges
// between CTAs.  Each output value is accumulated in a fixed order over k that
// does not depend on what else is skipped, so h_t is the same function in every
// iteration (the convergence proofs need that).
#include <limits.h>

#include <algorithm>

#include "js_common.cuh"
#include "made_driver.cuh"
#include "js_model.h"
#include "tc_common.cuh"

namespace {

constexpr int KC = 64;         // inputs per step of a product
constexpr int NTHREADS = 128;
constexpr int SUM_ROW = 40;    // row stride of partial sums: rows r .. r + 3 by columns c .. c + 7 lie in different banks
constexpr int ROWF = KC + 4;   // row stride in shared memory: the 16-byte pieces of eight rows lie in different banks
// The products go by tiles of 16 rows x 32 columns.  What bounds a layer is its longest tile (one chain over all inputs, with
// every wait of a step in it), so small tiles win although they read shared memory more often: 256 samples through
// 784 - 1024 - 1024 - 1568, five passes: 298 us, with 16 x 64 tiles 343, with 32 x 64 552; 16 samples: 228, 309, 488.
constexpr int MR = 2, NR = 2, BMt = 8 * MR, BNt = 16 * NR;
// Instances: fp32 products (operands by TMA: a fifth warp loads), bf16 products (operands converted on their way through
// registers), and for either type Jacobi-GS's, whose micro-steps are a warp per inner product and want many warps per SM
// but few CTAs at the thousands of grid barriers between them: 256 threads, tiles of 16 x 64 (with 128 threads a call of
// T = 784, H = 1024 x 2 in blocks of 98 took 7.56 ms for one sample, 6.41 so; T = 16, H = 64, batch 8 150 us, 133 so).
// SPLIT: fp32 products with the inputs of a tile dealt to the warps, see split_tile.
template <typename T, bool JGS, bool SPLIT = false> struct Conf {
    static constexpr bool TMA = sizeof(T) == 4 && !JGS;
    static constexpr int NTH = JGS ? 2 * NTHREADS : NTHREADS, BN = BNt * (NTH / NTHREADS);
    static constexpr int STAGES = JGS ? 2 : 4, STAGE_F = (BMt + BN) * (TMA ? 2 * KC : ROWF), CTAS = JGS ? 3 : 2;
    static constexpr int SUMS = SPLIT ? 4 * BMt * SUM_ROW : 0;            // the warps' partial sums
    static constexpr int SMEM_BYTES = (STAGES * STAGE_F + SUMS) * (int)sizeof(float) + (TMA ? 1024 : 0);
    static constexpr int THREADS = TMA ? NTH + 32 : NTH;
};
constexpr int JTHREADS = Conf<float, true>::NTH;
// TMA instance: stages of TK inputs in boxes of 32 (128-byte rows)
constexpr int TK = 2 * KC, BOX_K = 32, TMA_STAGES = 4, TMA_STAGE_BYTES = (BMt + BNt) * TK * 4;

// The stages; for the micro-steps of Jacobi-GS the list of units to evaluate.  Named where it is used, not reached through a
// pointer: the compiler must see that the accesses go to shared memory (as generic loads they took twice the wavefronts
// and global-memory latency, 57 cycles per input of a 16 x 64 tile).
extern __shared__ __align__(16) float g_sm[];

struct Smem {
    int list_n;
    int wcnt[JTHREADS / 32];
    uint64_t full[TMA_STAGES], empty[TMA_STAGES];
};

// The ring of the TMA instance; it is drained at the end of every layer.
struct Ring {
    int st = 0;
    uint32_t ph = 0;
    bool dead = false;
    __device__ void advance()
    {
        if (++st == TMA_STAGES) { st = 0; ph ^= 1u; }
    }
};
__device__ __forceinline__ uint32_t ring_base() { return (smem_u32(g_sm) + 1023u) & ~1023u; }
__device__ __forceinline__ float4 lds_f4(uint32_t a)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}

// The product with operands by TMA.  A stage holds TK inputs of the tile's rows: for every 32 of them the activation rows,
// behind all those the weight rows likewise, 128 bytes a row, 16-byte pieces permuted by the row number (128-byte swizzle,
// which keeps the reads of eight rows in different banks).  cp.async, 16 bytes a lane, cost the shared-memory pipe as much
// as the operand reads (14 wavefronts for 512 bytes).
__device__ __forceinline__ void tma_tile_load(Smem &s, Ring &rg, const MadeDev &m, int l, int meta, int m0, int n0, JsCtl *ctl)
{
    const CUtensorMap *ma = (const CUtensorMap *)m.tma_a + l, *mw = (const CUtensorMap *)m.tma_w + l;
    const int kend = m.t_kend[l][meta];
    // Inputs from kend on are masked.  Their weights are zeros, but a continuous state may be infinite there (its noise is, or
    // an iterate on its way), and zero times that is no zero: where a tile ends inside the four inputs that are multiplied at
    // a time, its last box comes through a map that ends at kend too, and the copy fills the rest with zeros.  (Cutting them
    // in the product cost 2 to 5 % of it.)
    const CUtensorMap *mc = (kend & 3) ? (const CUtensorMap *)m.tma_cut + m.cut_off[l] + meta : ma;
    for (int k0 = 0; k0 < kend; k0 += TK) {
        if (!__all_sync(0xffffffffu, mbar_wait(&s.empty[rg.st], rg.ph ^ 1u, ctl))) { rg.dead = true; return; }
        if (elect_one()) {
            const uint32_t base = ring_base() + (uint32_t)(rg.st * TMA_STAGE_BYTES);
            const int boxes = min(TK / BOX_K, (kend - k0 + BOX_K - 1) / BOX_K);
            mbar_expect_tx(&s.full[rg.st], (uint32_t)(boxes * (BMt + BNt) * BOX_K * 4));
            for (int h = 0; h < boxes; ++h) {
                tma_load_2d(base + (uint32_t)(h * BMt * 128), k0 + (h + 1) * BOX_K >= kend ? mc : ma, &s.full[rg.st], k0 + h * BOX_K, m0);
                tma_load_2d(base + (uint32_t)(TK / BOX_K * BMt * 128 + h * BNt * 128), mw, &s.full[rg.st], k0 + h * BOX_K, n0);
            }
        }
        __syncwarp();
        rg.advance();
    }
}

__device__ __forceinline__ void tma_tile(Smem &s, Ring &rg, int kend, int lr, int wc, JsCtl *ctl, float (&acc)[MR][NR])
{
#pragma unroll
    for (int i = 0; i < MR; ++i)
#pragma unroll
        for (int j = 0; j < NR; ++j) acc[i][j] = 0.0f;
    const uint32_t xa = (uint32_t)(lr & 7) << 4, xb = (uint32_t)(wc & 7) << 4;       // row + 4: the piece's bit 2 flips
    for (int k0 = 0; k0 < kend; k0 += TK) {
        // (A thread whose wait gives up goes on with what is there and waits no more: the warp has to stay together here and in
        // the caller, and the grid barrier behind the layer sees the abort flag.)
        if (!rg.dead && !mbar_wait(&s.full[rg.st], rg.ph, ctl)) rg.dead = true;
        uint32_t ra = ring_base() + (uint32_t)(rg.st * TMA_STAGE_BYTES), rb = ra + (uint32_t)(TK / BOX_K * BMt * 128 + wc * 128);
        ra += (uint32_t)(lr * 128);
        auto read = [&](int q, float4 (&a)[MR], float4 (&b)[NR]) {      // inputs 4 q .. 4 q + 3 from ra, rb on
            const uint32_t h = (uint32_t)(q >> 3), p = (uint32_t)(q & 7) << 4;
#pragma unroll
            for (int i = 0; i < MR; ++i) a[i] = lds_f4(ra + h * (BMt * 128) + (uint32_t)(i * 1024) + (p ^ xa));
#pragma unroll
            for (int j = 0; j < NR; ++j) b[j] = lds_f4(rb + h * (BNt * 128) + (uint32_t)(j * 512) + (p ^ xb ^ (uint32_t)((j & 1) << 6)));
        };
        auto mul = [&](const float4 (&a)[MR], const float4 (&b)[NR]) {
#pragma unroll
            for (int i = 0; i < MR; ++i)
#pragma unroll
                for (int j = 0; j < NR; ++j) acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]);
#pragma unroll
            for (int i = 0; i < MR; ++i)
#pragma unroll
                for (int j = 0; j < NR; ++j) acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
#pragma unroll
            for (int i = 0; i < MR; ++i)
#pragma unroll
                for (int j = 0; j < NR; ++j) acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]);
#pragma unroll
            for (int i = 0; i < MR; ++i)
#pragma unroll
                for (int j = 0; j < NR; ++j) acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
        };
        const int nq = min(TK / 4, (kend - k0 + 3) / 4);                 // (weights beyond kend are masked: zeros)
        constexpr int QU = 16, AHEAD = 3;                                // reads three quadruples ahead of their use
#pragma unroll 1
        for (int q0 = 0; q0 < nq; q0 += QU) {
            if (nq - q0 >= QU) {
                float4 a[AHEAD + 1][MR], b[AHEAD + 1][NR];
#pragma unroll
                for (int q = 0; q < AHEAD; ++q) read(q, a[q], b[q]);
#pragma unroll
                for (int q = 0; q < QU; ++q) {
                    if (q + AHEAD < QU) read(q + AHEAD, a[(q + AHEAD) % (AHEAD + 1)], b[(q + AHEAD) % (AHEAD + 1)]);
                    mul(a[q % (AHEAD + 1)], b[q % (AHEAD + 1)]);
                }
            } else {
#pragma unroll 1
                for (int q = 0; q < nq - q0; ++q) {
                    float4 a[MR], b[NR];
                    read(q, a, b);
                    mul(a, b);
                }
            }
            ra += QU / 8 * BMt * 128;
            rb += QU / 8 * BNt * 128;
        }
        __syncwarp();
        if ((threadIdx.x & 31) == 0) mbar_arrive(&s.empty[rg.st]);
        rg.advance();
    }
}

// The same with the inputs dealt to the warps, for models that only this kernel serves (made_small.cu sums like tma_tile, and the
// solvers of one model must return the same floats): warp w takes inputs 32 w .. 32 w + 31 of every 128, all rows and columns of the
// tile, 4 x 4 outputs a thread, and the four sums of an output are added in order.  With 2 x 2 outputs a thread the operand
// reads (4 of 16 bytes for 16 multiply-adds, 8 for 64 here) kept the shared-memory pipe busier than the multiply-adds the
// others.  T = 784, H = 1024 x 2, 256, 64, 16 samples and one: 279, 220, 209, 167 us, 264, 201, 190, 152 so; with tiles of 32 rows
// 338 for 256, with stages of 64 inputs 213 for 64.
__device__ __forceinline__ void split_tile(Smem &s, Ring &rg, int kend, int lr, int wc, JsCtl *ctl, float (&acc)[MR][NR])
{
    constexpr int PR = BMt / 4, PC = BNt / 8;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r = lane & 3, c = lane >> 2;      // rows r + 4 i, columns c + 8 j
    float p[PR][PC];
#pragma unroll
    for (int i = 0; i < PR; ++i)
#pragma unroll
        for (int j = 0; j < PC; ++j) p[i][j] = 0.0f;
    for (int k0 = 0; k0 < kend; k0 += TK) {
        if (!rg.dead && !mbar_wait(&s.full[rg.st], rg.ph, ctl)) rg.dead = true;       // (see tma_tile)
        const uint32_t st = ring_base() + (uint32_t)(rg.st * TMA_STAGE_BYTES);
        const uint32_t ra = st + (uint32_t)(warp * BMt * 128 + r * 128), rb = st + (uint32_t)(TK / BOX_K * BMt * 128 + warp * BNt * 128 + c * 128);
        const int nq = min(BOX_K / 4, (kend - k0 - BOX_K * warp + 3) / 4);
        auto quad = [&](int q) {                         // four inputs
            float4 a[PR], b[PC];
#pragma unroll
            for (int i = 0; i < PR; ++i) a[i] = lds_f4(ra + (uint32_t)(i * 512) + (uint32_t)((q ^ (r | (i & 1) << 2)) << 4));
#pragma unroll
            for (int j = 0; j < PC; ++j) b[j] = lds_f4(rb + (uint32_t)(j * 1024) + (uint32_t)((q ^ c) << 4));
#pragma unroll
            for (int i = 0; i < PR; ++i)
#pragma unroll
                for (int j = 0; j < PC; ++j) p[i][j] = fmaf(a[i].x, b[j].x, p[i][j]);
#pragma unroll
            for (int i = 0; i < PR; ++i)
#pragma unroll
                for (int j = 0; j < PC; ++j) p[i][j] = fmaf(a[i].y, b[j].y, p[i][j]);
#pragma unroll
            for (int i = 0; i < PR; ++i)
#pragma unroll
                for (int j = 0; j < PC; ++j) p[i][j] = fmaf(a[i].z, b[j].z, p[i][j]);
#pragma unroll
            for (int i = 0; i < PR; ++i)
#pragma unroll
                for (int j = 0; j < PC; ++j) p[i][j] = fmaf(a[i].w, b[j].w, p[i][j]);
        };
        if (nq == BOX_K / 4) {
#pragma unroll
            for (int q = 0; q < BOX_K / 4; ++q) quad(q);
        } else {
#pragma unroll 1
            for (int q = 0; q < nq; ++q) quad(q);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&s.empty[rg.st]);
        rg.advance();
    }
    const uint32_t sums = ring_base() + (uint32_t)(TMA_STAGES * TMA_STAGE_BYTES);
#pragma unroll
    for (int i = 0; i < PR; ++i)
#pragma unroll
        for (int j = 0; j < PC; ++j)
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(sums + 4u * (uint32_t)((warp * BMt + r + 4 * i) * SUM_ROW + c + 8 * j)), "f"(p[i][j]) : "memory");
    asm volatile("bar.sync 1, 128;" ::: "memory");
#pragma unroll
    for (int i = 0; i < MR; ++i)
#pragma unroll
        for (int j = 0; j < NR; ++j) {
            float v[4];
#pragma unroll
            for (int w = 0; w < 4; ++w)
                asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v[w]) : "r"(sums + 4u * (uint32_t)((w * BMt + lr + 8 * i) * SUM_ROW + wc + 4 * j)) : "memory");
            acc[i][j] = ((v[0] + v[1]) + v[2]) + v[3];
        }
    asm volatile("bar.sync 1, 128;" ::: "memory");          // the next tile's sums go to the same place
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// One tile of  out = A[rows][K] * W[N][K]^T  over k in [0, kend): 8 MR rows x BN columns, NT threads of MR x NR outputs
// (row lr + 8 i, column 4 NR warp + lc + 4 j).  Operand rows are copied as they lie in memory, 16 bytes at a time, three
// steps of 64 inputs in flight; a thread reads four inputs of a row at once, the next four while it multiplies.  lr takes bits
// 0, 3, 4 of the lane and lc bits 1, 2: a 16-byte shared-memory load whose address does not depend on bit 0, or not on bit 1,
// takes two cycles for a warp instead of four.  Every output is one chain of fused multiply-adds over k in ascending order.
template <typename T, int STAGES, int STAGE_F, int NT, int BN>
__device__ __forceinline__ void gemm_tile(const T *A, int lda, const T *__restrict__ W, int ldw, int N, int kend,
                                          int m0, int n0, int lr, int wc, float (&acc)[MR][NR])
{
    constexpr int EPP = 16 / sizeof(T);      // values per 16-byte piece
    constexpr int PPR = KC / EPP, RPE = NT / PPR;          // pieces per row, rows per round of the threads
    constexpr int E = (BMt + BN + RPE - 1) / RPE;      // rounds: the activations' rows, behind them the weights'
    constexpr bool EVEN = (BMt + BN) % RPE == 0;
    const int steps = (kend + KC - 1) / KC;
    float *tile = g_sm;
#pragma unroll
    for (int i = 0; i < MR; ++i)
#pragma unroll
        for (int j = 0; j < NR; ++j) acc[i][j] = 0.0f;
    const int prow = threadIdx.x / PPR, pk = (threadIdx.x % PPR) * EPP;       // this thread's piece: row (+ RPE e), inputs
    const uint32_t dst0 = smem_addr(tile) + 4u * (uint32_t)(prow * ROWF + pk);
    // (weight rows beyond the last column: the last one again, their outputs are not stored)
    auto src_of = [&](int e) {
        const int row = prow + RPE * e;
        const bool act = BMt % RPE == 0 ? e < BMt / RPE : row < BMt;
        return act ? A + (size_t)(m0 + row) * lda + pk : W + (size_t)min(n0 + row - BMt, N - 1) * ldw + pk;
    };
    uint4 reg[sizeof(T) == 2 ? E : 1];
    auto fetch = [&](int c, int st) {               // fp32: asynchronous copies; bf16: into registers, converted by put()
        const int vals = max(0, min(EPP, kend - (c * KC + pk))), off = vals > 0 ? c * KC : -pk;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (!EVEN && prow + RPE * e >= BMt + BN) break;
            const T *src = src_of(e) + off;
            if constexpr (sizeof(T) == 4)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst0 + 4u * (uint32_t)(st * STAGE_F + RPE * e * ROWF)),
                             "l"(src), "r"(vals * 4) : "memory");
            else
                reg[e] = vals > 0 ? __ldcg(reinterpret_cast<const uint4 *>(src)) : make_uint4(0, 0, 0, 0);
        }
    };
    auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
    auto put = [&](int c, int st) {
        const int vals = kend - (c * KC + pk);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (!EVEN && prow + RPE * e >= BMt + BN) break;
            const uint32_t w[4] = {reg[sizeof(T) == 2 ? e : 0].x, reg[sizeof(T) == 2 ? e : 0].y, reg[sizeof(T) == 2 ? e : 0].z, reg[sizeof(T) == 2 ? e : 0].w};
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = i < vals ? __uint_as_float((i & 1) ? (w[i / 2] & 0xffff0000u) : (w[i / 2] << 16)) : 0.0f;
            float4 *dst = reinterpret_cast<float4 *>(tile + st * STAGE_F + (prow + RPE * e) * ROWF + pk);
            dst[0] = make_float4(v[0], v[1], v[2], v[3]);
            dst[1] = make_float4(v[4], v[5], v[6], v[7]);
        }
    };
    __syncthreads();                                // the stages are free
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int c = 0; c < STAGES - 1; ++c) {
            if (c < steps) fetch(c, c);
            commit();
        }
    } else if (steps > 0) {
        fetch(0, 0);
    }
    int st = 0;
    for (int c = 0; c < steps; ++c) {
        if constexpr (sizeof(T) == 4) asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
        else put(c, st);
        __syncthreads();
        if constexpr (sizeof(T) == 4) {
            if (c + STAGES - 1 < steps) fetch(c + STAGES - 1, st == 0 ? STAGES - 1 : st - 1);
            commit();
        } else if (c + 1 < steps) {
            fetch(c + 1, 0);
        }
        const float *ta = tile + st * STAGE_F + lr * ROWF, *tb = tile + st * STAGE_F + (BMt + wc) * ROWF;
        float4 a[2][MR], b[2][NR];
        auto read = [&](int k, int u) {
#pragma unroll
            for (int i = 0; i < MR; ++i) a[u][i] = *reinterpret_cast<const float4 *>(ta + 8 * i * ROWF + k);
#pragma unroll
            for (int j = 0; j < NR; ++j) b[u][j] = *reinterpret_cast<const float4 *>(tb + 4 * j * ROWF + k);
        };
        read(0, 0);
#pragma unroll
        for (int k = 0; k < KC; k += 4) {
            const int u = (k >> 2) & 1;
            if (k + 4 < KC) read(k + 4, u ^ 1);
#pragma unroll
            for (int i = 0; i < MR; ++i)
#pragma unroll
                for (int j = 0; j < NR; ++j) acc[i][j] = fmaf(a[u][i].x, b[u][j].x, acc[i][j]);
#pragma unroll
            for (int i = 0; i < MR; ++i)
#pragma unroll
                for (int j = 0; j < NR; ++j) acc[i][j] = fmaf(a[u][i].y, b[u][j].y, acc[i][j]);
#pragma unroll
            for (int i = 0; i < MR; ++i)
#pragma unroll
                for (int j = 0; j < NR; ++j) acc[i][j] = fmaf(a[u][i].z, b[u][j].z, acc[i][j]);
#pragma unroll
            for (int i = 0; i < MR; ++i)
#pragma unroll
                for (int j = 0; j < NR; ++j) acc[i][j] = fmaf(a[u][i].w, b[u][j].w, acc[i][j]);
        }
        if (++st == STAGES) st = 0;
    }
}

__device__ __forceinline__ size_t a0_at(const MadeDev &m, size_t i);

// What becomes of an output tile: logits to memory, or, with one or two outputs per position, sampled on the spot.
struct OutArgs {
    float *zout;               // logits [batch][T*C], or NULL: sample
    bool flag;
    int fslot;
};

// Change flags of many positions: the per-sample word by a plain store, the batch-level words once per warp (an atomic per
// changed position on two words for the whole batch took longer than the forward pass).
struct Changes {
    int first = INT_MAX;
    __device__ __forceinline__ void note(const RunArgs &r, int fslot, int b, int d)
    {
        r.smp_changed[fslot * r.batch + b] = 1;
        first = min(first, d);
    }
    __device__ __forceinline__ void flush(const RunArgs &r, int fslot)
    {
        const int f = __reduce_min_sync(0xffffffffu, first);
        if (f != INT_MAX && (threadIdx.x & 31) == 0) {
            atomicMin(&r.ctl->agg_minfirst[fslot], f);
            atomicOr(&r.ctl->agg_any[fslot], 1);
        }
        first = INT_MAX;
    }
};

// Layer l over the window: hidden layers store act(pre) into `out`; the output layer (l == L) see OutArgs.  Tiles with the
// longest inner products first, dealt to the CTAs back and forth.
template <typename T, bool JGS, bool SPLIT>
__device__ void gemm_phase(Smem &s, Ring &rg, const MadeDev &m, const RunArgs &r, int l, const T *Asrc, T *out, const OutArgs &oa, const Win &w,
                           unsigned long long &issued, unsigned long long &skipped)
{
    constexpr int BN = Conf<T, JGS>::BN;
    static_assert(JS_GT % BN == 0, "a tile lies in one tile of the metadata");
    const int N = m.n[l + 1], K = m.n[l], batch = r.batch;
    const int mt = (batch + BMt - 1) / BMt, nt = (N + BN - 1) / BN, G = (int)gridDim.x;
    const bool is_out = (l == m.L);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lr = (lane & 1) | ((lane >> 3) << 1), wc = 4 * NR * warp + ((lane >> 1) & 3);
    const bool loader = Conf<T, JGS>::TMA && warp == NTHREADS / 32;
    Changes chg;
    for (int round = 0; round * G < mt * nt; ++round) {
        const int tile = round * G + ((round & 1) ? G - 1 - (int)blockIdx.x : (int)blockIdx.x);
        if (tile >= mt * nt) continue;
        const int tn = nt - 1 - tile / mt, tm = tile % mt, m0 = tm * BMt, n0 = tn * BN, meta = n0 / JS_GT;
        const int dmin = m.t_dmin[l][meta], dmax = m.t_dmax[l][meta];
        bool live;
        if (is_out) live = (dmax - 1 >= w.olo) && (dmin - 1 < w.ohi);
        else live = (dmax > w.hdeg_lo) && (dmin <= w.hdeg_hi);
        if (!live) { if (threadIdx.x == 0) skipped++; continue; }
        if constexpr (Conf<T, JGS>::TMA) {
            if (loader) {
                if (rg.dead) break;
                tma_tile_load(s, rg, m, l, meta, m0, n0, r.ctl);
                continue;
            }
        }
        if (threadIdx.x == 0) issued++;
        // what the epilogue needs from memory is asked for before the product: biases, and where positions are sampled in the
        // tile their noise and present values (one after the other behind the product they cost 2 us an output)
        float acc[MR][NR], bv[NR], nz[MR][NR], xo[MR][NR];
        const bool sample = is_out && !oa.zout;
        auto position = [&](int j) { return r.real ? (n0 + wc + 4 * j) >> 1 : n0 + wc + 4 * j; };
        auto mine = [&](int i, int j) {
            const int row = m0 + lr + 8 * i, col = n0 + wc + 4 * j, d = position(j);
            return row < batch && col < N && d >= w.plo && d < w.phi && !(r.real && (col & 1));
        };
#pragma unroll
        for (int j = 0; j < NR; ++j) bv[j] = n0 + wc + 4 * j < N ? __ldg(&m.bias[l][n0 + wc + 4 * j]) : 0.0f;
        bool frozen[MR];
        if (sample)
#pragma unroll
            for (int i = 0; i < MR; ++i) {
                const int row = m0 + lr + 8 * i;
                // a sample whose stopping test has fired keeps the iterate it stopped at (with eps > 0 a further update
                // would still move it)
                frozen[i] = r.real && oa.flag && row < batch && r.smp_state[row] != 0;
#pragma unroll
                for (int j = 0; j < NR; ++j) {
                    const bool in = mine(i, j);
                    const size_t at = (size_t)(in ? row : 0) * m.T + (in ? position(j) : 0);
                    nz[i][j] = in ? __ldg(r.noise + at) : 0.0f;
                    xo[i][j] = !in ? 0.0f : r.real ? r.xr[at] : (float)r.x[at];
                }
            }
        if constexpr (SPLIT) {
            split_tile(s, rg, m.t_kend[l][meta], lr, wc, r.ctl, acc);
        } else if constexpr (Conf<T, JGS>::TMA) {
            tma_tile(s, rg, m.t_kend[l][meta], lr, wc, r.ctl, acc);
        } else {
            gemm_tile<T, Conf<T, JGS>::STAGES, Conf<T, JGS>::STAGE_F, Conf<T, JGS>::NTH, BN>(Asrc, K, (const T *)m.W[l], K, N, m.t_kend[l][meta], m0, n0, lr, wc, acc);
        }
#pragma unroll
        for (int i = 0; i < MR; ++i) {
            const int row = m0 + lr + 8 * i;
#pragma unroll
            for (int j = 0; j < NR; ++j) {
                const int col = n0 + wc + 4 * j;
                const float pre = acc[i][j] + bv[j];
                if (!sample) {
                    if (row < batch && col < N) {
                        if (is_out) oa.zout[(size_t)row * N + col] = pre;
                        else out[(size_t)row * N + col] = from_f32<T>(js_act_fn(m.act, pre));
                    }
                    continue;
                }
                // Continuous states with logistic conditionals (Section 5.3.1, Appendix C.3 of arXiv 2002.03629): logit 2t is the
                // location m_t, logit 2t+1 (the neighbouring column: lane bit 1) the log-scale l_t, and the position's
                // reserved noise e_t = logit(u_t) gives x_t = m_t + exp(l_t) e_t (inverse CDF of the logistic law).  A position
                // counts as changed when it moved by more than eps, so "no position changed" is the stopping rule
                // max_t |x^k_t - x^{k-1}_t| <= eps  of Section 2.2.1 in the maximum norm.
                const float scale = r.real ? __shfl_xor_sync(0xffffffffu, pre, 2) : 0.0f;
                if (!mine(i, j) || frozen[i]) continue;
                const int d = position(j);
                const size_t at = (size_t)row * m.T + d;
                if (r.real) {
                    const float xn = fmaf(expf(scale), nz[i][j], pre);
                    r.xr[at] = xn;
                    ((T *)m.a[0])[a0_at(m, at)] = from_f32<T>(xn);
                    if (oa.flag && !(fabsf(xn - xo[i][j]) <= r.eps)) chg.note(r, oa.fslot, row, d);     // a NaN difference is a change
                } else {
                    const int xn = js_sample_binary(r.nk, pre, nz[i][j]);
                    if ((float)xn != xo[i][j]) {
                        r.x[at] = (uint8_t)xn;
                        ((T *)m.a[0])[a0_at(m, at)] = from_f32<T>(m.lut[xn]);
                        if (oa.flag) chg.note(r, oa.fslot, row, d);
                    }
                }
            }
        }
    }
    if (oa.flag && !loader) chg.flush(r, oa.fslot);
}

// place in a[0] (rows of n[0] >= T values) of element i = sample * T + position
__device__ __forceinline__ size_t a0_at(const MadeDev &m, size_t i)
{
    return m.n[0] == m.T ? i : i / m.T * m.n[0] + i % m.T;
}

// x = init (or zeros), a[0] = lut[x]; also clears the per-sample bookkeeping.
template <typename T>
__device__ void init_phase(const MadeDev &m, const RunArgs &r, const uint8_t *src)
{
    const size_t n = (size_t)r.batch * m.T;
    T *a0 = (T *)m.a[0];
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const uint8_t v = src ? src[i] : (uint8_t)0;
        if (r.x) r.x[i] = v;
        a0[a0_at(m, i)] = from_f32<T>(m.lut[v]);
    }
    if (blockIdx.x == 0) {
        clear_flags(r);
        for (int i = threadIdx.x; i < 2 * r.batch; i += blockDim.x) r.smp_state[i] = 0;
    }
}

// Sample C-way positions [plo, phi) of every sample from the logits scratch, compare with the current iterate, store the
// new symbol and its encoding: a warp per position.
template <typename T>
__device__ void sample_phase(const MadeDev &m, const RunArgs &r, const float *z, int plo, int phi, bool flag,
                             int fslot)
{
    const int T_ = m.T, C = m.C, np = phi - plo;
    T *a0 = (T *)m.a[0];
    const int lane = threadIdx.x & 31;
    const size_t warps = ((size_t)gridDim.x * blockDim.x) >> 5;
    const size_t n = (size_t)r.batch * np;
    Changes chg;
    for (size_t i = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += warps) {
        const int b = (int)(i / np), d = plo + (int)(i % np);
        const size_t at = (size_t)b * T_ + d;
        const int bi = js_warp_sample_cat(r.nk, z + at * C, r.noise + (r.nk == JS_NOISE_GUMBEL ? at * C : at), C, lane);
        if (lane == 0 && bi != r.x[at]) {
            r.x[at] = (uint8_t)bi;
            a0[a0_at(m, at)] = from_f32<T>(m.lut[bi]);
            if (flag) chg.note(r, fslot, b, d);
        }
    }
    if (flag) chg.flush(r, fslot);
}

// Continuous states: x = start values (or zeros), a[0] = x (rounded like any activation in a bf16 model).
template <typename T>
__device__ void init_phase_real(const MadeDev &m, const RunArgs &r, const float *src)
{
    const size_t n = (size_t)r.batch * m.T;
    T *a0 = (T *)m.a[0];
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float v = src ? src[i] : 0.0f;
        if (r.xr) r.xr[i] = v;
        a0[a0_at(m, i)] = from_f32<T>(v);
    }
    if (blockIdx.x == 0) {
        clear_flags(r);
        for (int i = threadIdx.x; i < 2 * r.batch; i += blockDim.x) r.smp_state[i] = 0;
    }
}

// ---- Jacobi-GS micro-steps (Algorithm 2): warp-per-dot-product evaluation of
// the units that become computable at step j of every block's sequential sweep.
// A unit of block i reads, from the layer below, units of earlier blocks at the
// previous outer iterate (`old`) and units of its own block at the current one.
template <typename T>
__device__ float mixed_dot(const MadeDev &m, int l, int unit, int blk, int B, const T *old_row, const T *new_row,
                           int kend)
{
    const int lane = threadIdx.x & 31;
    const T *w = (const T *)m.W[l] + (size_t)unit * m.n[l];
    const int *dg = m.deg[l];
    float acc = 0.0f;
    for (int k = lane; k < kend; k += 32) {
        const bool use_old = ((dg[k] - 1) / B) < blk;
        acc = fmaf(to_f32<T>(w[k]), to_f32<T>(use_old ? old_row[k] : new_row[k]), acc);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    return acc;
}

template <typename T>
__device__ void jgs_hidden_phase(Smem &s, const MadeDev &m, const RunArgs &r, int l, int j, int B, int blk_lo)
{
    // units of layer l+1 whose degree g satisfies g % B == j, in blocks >= blk_lo.
    // The list is built in index order so that every CTA holds the same list.
    int *list = reinterpret_cast<int *>(g_sm);
    const int N = m.n[l + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t warps = ((size_t)gridDim.x * blockDim.x) >> 5;
    for (int ubase = 0; ubase < N; ubase += 4096) {
        const int uend = min(N, ubase + 4096);
        if (threadIdx.x == 0) s.list_n = 0;
        __syncthreads();
        for (int base = ubase; base < uend; base += JTHREADS) {
            const int i = base + threadIdx.x;
            bool pred = false;
            if (i < uend) {
                const int g = m.deg[l + 1][i];
                pred = (g % B == j) && ((g - 1) / B >= blk_lo);
            }
            const unsigned bal = __ballot_sync(0xffffffffu, pred);
            if (lane == 0) s.wcnt[warp] = __popc(bal);
            __syncthreads();
            int off = s.list_n;
            for (int w2 = 0; w2 < warp; ++w2) off += s.wcnt[w2];
            if (pred) list[off + __popc(bal & ((1u << lane) - 1u))] = i;
            __syncthreads();
            if (threadIdx.x == 0) {
                int tot = 0;
                for (int w2 = 0; w2 < JTHREADS / 32; ++w2) tot += s.wcnt[w2];
                s.list_n += tot;
            }
            __syncthreads();
        }
        const int cnt = s.list_n;
        const size_t items = (size_t)cnt * r.batch;
        for (size_t it = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items; it += warps) {
            const int unit = list[it / r.batch], b = (int)(it % r.batch);
            const int g = m.deg[l + 1][unit];
            const float pre = mixed_dot<T>(m, l, unit, (g - 1) / B, B, (const T *)m.a_old[l] + (size_t)b * m.n[l],
                                           (const T *)m.a[l] + (size_t)b * m.n[l], m.t_kend[l][unit / JS_GT]) +
                              m.bias[l][unit];
            if (lane == 0) ((T *)m.a[l + 1])[(size_t)b * N + unit] = from_f32<T>(js_act_fn(m.act, pre));
        }
        __syncthreads();
    }
}

template <typename T>
__device__ void jgs_output_phase(const MadeDev &m, const RunArgs &r, int j, int B, int blk_lo)
{
    const int L = m.L, C = m.C, nblk = (m.T + B - 1) / B;
    const size_t warps = ((size_t)gridDim.x * blockDim.x) >> 5;
    const size_t items = (size_t)(nblk - blk_lo) * C * r.batch;
    const int lane = threadIdx.x & 31;
    for (size_t it = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items; it += warps) {
        const int b = (int)(it % r.batch);
        const int c = (int)((it / r.batch) % C);
        const int blk = blk_lo + (int)(it / ((size_t)r.batch * C));
        const int t = blk * B + j;
        if (t >= m.T) continue;
        const int unit = t * C + c;
        const float z = mixed_dot<T>(m, L, unit, blk, B, (const T *)m.a_old[L] + (size_t)b * m.n[L],
                                     (const T *)m.a[L] + (size_t)b * m.n[L], m.t_kend[L][unit / JS_GT]) +
                        m.bias[L][unit];
        if (C == 1) {
            if (lane == 0) {
                const size_t at = (size_t)b * m.T + t;
                const int xn = js_sample_binary(r.nk, z, r.noise[at]);
                r.x[at] = (uint8_t)xn;
                ((T *)m.a[0])[a0_at(m, at)] = from_f32<T>(m.lut[xn]);
            }
        } else if (lane == 0) {
            m.logits[(size_t)b * m.n[L + 1] + unit] = z;
        }
    }
}

// categorical commit of position blk*B + j for every block (no change flags here)
template <typename T>
__device__ void jgs_commit_phase(const MadeDev &m, const RunArgs &r, int j, int B, int blk_lo)
{
    const int C = m.C, nblk = (m.T + B - 1) / B;
    const size_t warps = ((size_t)gridDim.x * blockDim.x) >> 5;
    const size_t items = (size_t)(nblk - blk_lo) * r.batch;
    const int lane = threadIdx.x & 31;
    for (size_t it = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items; it += warps) {
        const int b = (int)(it % r.batch);
        const int t = (blk_lo + (int)(it / r.batch)) * B + j;
        if (t >= m.T) continue;
        const size_t at = (size_t)b * m.T + t;
        const int bi = js_warp_sample_cat(r.nk, m.logits + at * C, r.noise + (r.nk == JS_NOISE_GUMBEL ? at * C : at), C, lane);
        if (lane == 0) {
            r.x[at] = (uint8_t)bi;
            ((T *)m.a[0])[a0_at(m, at)] = from_f32<T>(m.lut[bi]);
        }
    }
}

// x_old = x and a_old[0] = a[0] (start of an outer iteration); or compare x with
// x_old and raise change flags (end of an outer iteration).
template <typename T>
__device__ void jgs_copy_or_compare(const MadeDev &m, const RunArgs &r, bool compare, int fslot)
{
    Changes chg;
    const size_t n = (size_t)r.batch * m.T;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        if (compare) {
            if (r.x[i] != r.x_old[i]) chg.note(r, fslot, (int)(i / m.T), (int)(i % m.T));
        } else {
            r.x_old[i] = r.x[i];
            ((T *)m.a_old[0])[a0_at(m, i)] = ((const T *)m.a[0])[a0_at(m, i)];
        }
    }
    if (compare) chg.flush(r, fslot);
}

// ------------------------------------------------------------------ engine
template <typename T, bool JGS, bool SPLIT>
struct GenericEngine {
    static constexpr bool has_jgs = JGS;
    Smem &s;
    const MadeDev &m;
    const RunArgs &r;
    unsigned epoch = 0;
    unsigned long long issued = 0, skipped = 0;
    Ring rg;

    __device__ GenericEngine(Smem &s_, const MadeDev &m_, const RunArgs &r_) : s(s_), m(m_), r(r_)
    {
    }
    __device__ bool barrier()
    {
        // activations stored by threads are read by TMA after the barrier: the proxy fence is on the reading side
        const bool ok = grid_barrier(r.ctl, epoch, r.spin_limit);
        if constexpr (Conf<T, JGS>::TMA) fence_proxy_async();
        return ok;
    }
    __device__ void init(const uint8_t *src)
    {
        if (r.real)
            init_phase_real<T>(m, r, r.kmode == KM_FORWARD ? r.xin_r : r.kmode == KM_SEQ ? (const float *)nullptr : r.init_r);
        else
            init_phase<T>(m, r, src);
    }
    __device__ void look_ahead(int) {}
    __device__ int compact(int) { return 0; }      // the CUDA-core path keeps the batch as it is
    // One forward pass over the window; then either the logits go to zout (teacher forcing) or positions [w.plo, w.phi) are
    // sampled and committed: in the output tiles themselves where a position has one logit or a location and a log-scale,
    // from the logits scratch where it has more.
    __device__ bool step(const Win &w, bool flag, int fslot, float *zout)
    {
        const bool fused = !zout && (m.C == 1 || r.real);
        for (int l = 0; l <= m.L; ++l) {
            const OutArgs oa = {zout ? zout : fused ? (float *)nullptr : m.logits, fused && flag && l == m.L, fslot};
            gemm_phase<T, JGS, SPLIT>(s, rg, m, r, l, (const T *)m.a[l], l < m.L ? (T *)m.a[l + 1] : (T *)nullptr, oa, w, issued, skipped);
            if (!barrier()) return false;
        }
        if (zout || fused) return true;
        sample_phase<T>(m, r, m.logits, w.plo, w.phi, flag, fslot);
        return barrier();
    }
    // one outer iteration of Algorithm 2
    __device__ bool jgs_outer(int fslot, int fin_h, int blk_lo, int &iterations)
    {
        const int B = r.block, T_ = m.T;
        jgs_copy_or_compare<T>(m, r, false, fslot);
        if (!barrier()) return false;
        // hidden activations of the previous outer iterate
        const Win w = make_win(fin_h, T_, T_, T_);
        for (int l = 0; l < m.L; ++l) {
            gemm_phase<T, JGS, SPLIT>(s, rg, m, r, l, (const T *)m.a_old[l], (T *)m.a_old[l + 1], OutArgs{nullptr, false, 0}, w, issued, skipped);
            if (!barrier()) return false;
        }
        const int jmax = min(B, T_);
        for (int j = 0; j < jmax; ++j) {
            if (j >= 1)
                for (int l = 0; l < m.L; ++l) {
                    jgs_hidden_phase<T>(s, m, r, l, j, B, blk_lo);
                    if (!barrier()) return false;
                }
            jgs_output_phase<T>(m, r, j, B, blk_lo);
            if (!barrier()) return false;
            if (m.C > 1) {
                jgs_commit_phase<T>(m, r, j, B, blk_lo);
                if (!barrier()) return false;
            }
            iterations++;
        }
        jgs_copy_or_compare<T>(m, r, true, fslot);
        return barrier();
    }
};

template <typename T, bool JGS, bool SPLIT>
__global__ void __launch_bounds__(Conf<T, JGS, SPLIT>::THREADS, Conf<T, JGS, SPLIT>::CTAS) made_generic_kernel(const __grid_constant__ MadeDev m, const __grid_constant__ RunArgs r)
{
    __shared__ Smem s;
    if constexpr (Conf<T, JGS>::TMA) {
        if (threadIdx.x == 0) {
            for (int i = 0; i < TMA_STAGES; ++i) { mbar_init(&s.full[i], 1); mbar_init(&s.empty[i], NTHREADS / 32); }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            fence_proxy_async();
        }
        __syncthreads();
    }
    GenericEngine<T, JGS, SPLIT> e(s, m, r);
    DriverResult res = made_driver(e, m.T, r);
    if constexpr (Conf<T, JGS>::TMA) {
        // after an aborted wait copies may still be on their way into this CTA's shared memory
        if (__syncthreads_or(e.rg.dead || !res.alive)) {
            for (int i = 0; i < 2000; ++i) __nanosleep(1000);
            res.alive = false;
        }
        __syncthreads();
    }
    driver_finish(r, res, e.issued, e.skipped);
}

}  // namespace

struct GenericInstance { const void *kernel; int smem, threads; };
template <typename T, bool JGS, bool SPLIT>
static GenericInstance generic_instance()
{
    using CF = Conf<T, JGS, SPLIT>;
    return {(const void *)made_generic_kernel<T, JGS, SPLIT>, CF::SMEM_BYTES, CF::THREADS};
}
static GenericInstance generic_of(int prec, bool jgs, bool split)
{
    if (prec == JS_BF16) return jgs ? generic_instance<__nv_bfloat16, true, false>() : generic_instance<__nv_bfloat16, false, false>();
    return jgs ? generic_instance<float, true, false>() : split ? generic_instance<float, false, true>() : generic_instance<float, false, false>();
}

// Tensor maps of an fp32 model's activations and masked weights: boxes of 32 inputs x 16 rows (activations) or 32 rows, 128-byte
// swizzle; and of the activations once more for every 64-wide tile of outputs, with the inputs that it reads.
int js_generic_prepare(js_model *mo)
{
    MadeDev &v = mo->made;
    v.tma_a = v.tma_w = v.tma_cut = nullptr;
    if (v.prec != JS_F32) return JS_OK;
    std::vector<CUtensorMap> maps(2 * (v.L + 1));
    for (int l = 0; l <= v.L; ++l) {
        if (!js_encode_map_2d(&maps[l], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, v.a[l], mo->rows, v.n[l], BOX_K, BMt) ||
            !js_encode_map_2d(&maps[v.L + 1 + l], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, v.W[l], v.n[l + 1], v.n[l], BOX_K, BNt))
            return JS_ERR_CUDA;
        v.cut_off[l] = (int)maps.size() - 2 * (v.L + 1);
        for (int kend : mo->host_kend[l]) {
            maps.emplace_back();
            if (!js_encode_map_2d(&maps.back(), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, v.a[l], mo->rows, std::max(kend, 1), BOX_K, BMt, v.n[l])) return JS_ERR_CUDA;
        }
    }
    void *p = nullptr;
    if (cudaMalloc(&p, maps.size() * sizeof(CUtensorMap)) != cudaSuccess) return JS_ERR_CUDA;
    mo->allocs.push_back(p);
    if (cudaMemcpy(p, maps.data(), maps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice) != cudaSuccess) return JS_ERR_CUDA;
    v.tma_a = p;
    v.tma_w = (const CUtensorMap *)p + v.L + 1;
    v.tma_cut = (const CUtensorMap *)p + 2 * (v.L + 1);
    return JS_OK;
}

// most CTAs that are resident at a time (a cooperative launch); jgs: of the instance that serves Jacobi-GS
int js_made_generic_max_grid(int prec, bool jgs, bool split)
{
    static_assert(Conf<float, true>::SMEM_BYTES >= 4096 * 4, "the unit list of the micro-steps shares the stages' memory");
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return -1;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
    const GenericInstance g = generic_of(prec, jgs, split);
    cudaError_t e = cudaFuncSetAttribute(g.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, g.smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, g.kernel, g.threads, g.smem);
    if (e != cudaSuccess || per_sm < 1) return -1;
    return sms * per_sm;
}

int js_launch_made_generic(const MadeDev &m, const RunArgs &r, bool split, int grid, cudaStream_t stream)
{
    void *args[2] = {(void *)&m, (void *)&r};
    const GenericInstance g = generic_of(m.prec, r.kmode == KM_JACOBI_GS, split);
    cudaError_t e = cudaLaunchCooperativeKernel(g.kernel, dim3(grid), dim3(g.threads), args, g.smem, stream);
    return e == cudaSuccess ? 0 : (int)e;
}
