// Cached sequential sweeps of a masked MLP with binary positions, on the sm_100a tensor cores.
//
// A sweep computes positions a .. b-1 of a block strictly in order (Eq. 1 of arXiv 2002.03629),
// each from the positions before it: positions < a are given (their hidden activations come from
// a forward pass on the previous iterate), positions inside the block are the fresh ones.  That is
// the inner loop of Jacobi-GS (Algorithm 2: all blocks in parallel, a sweep inside each) and, with
// one block covering every position, the feedforward pass itself with every hidden unit evaluated
// once (the cached sampler of Section 4.2).
//
// Work decomposition.  A job is (128, 64 or 32 samples, one block); jobs never talk to each other, so the
// kernel needs no grid-wide synchronisation at all.  Inside a job the positions are taken in
// groups of G.  With sorted degrees, everything a group needs from before the group - inputs and
// hidden units of degree <= t0, the group's first position - is a PREFIX of every layer's units,
// so its contribution to the group's G output logits and to the handful of hidden units of degree
// t0+1 .. t0+G is a GEMM  [128 samples x prefix] x [prefix x (<= 32 units)]  per layer: TMA feeds
// the prefix of the activations (from the previous iterate's activations up to the block's start,
// from the job's own buffer F after it) and 16-row weight boxes, tcgen05.mma accumulates in tensor
// memory.  What the units of the group contribute to one another is a triangular system of at most
// 32 x 32 weights per layer, solved position by position: logit, sample against the fixed noise
// (Appendix A.3), then the hidden units that the new symbol makes computable.  A warp takes four or eight sample
// rows, lane = unit of the group, every layer's running sums in registers; a value that becomes known
// goes to all lanes by shuffle and is added to 32 running sums by one multiply-add per row.  (With thread = row and the
// running sums in shared memory a position moved 24 KB through it: 0.6 us for two hidden layers.)  The group's
// activations then go to F, where the next group's GEMMs find them.  What those GEMMs read of earlier groups (all full K
// blocks below the group's first unit) does not wait for that: it is loaded and multiplied while the positions are solved.
//
// What bounds it: the chain of the positions.  256 samples of a 784-1024-1024-784 model, one block (8 jobs of 32 rows): 431 us
// (1117 with thread = row), per group 5.7 us of positions, 2.6 us from the operands of its late K blocks to the sums, 1.6 us to
// store its activations.  512 samples of a 4096-wide model in 32 blocks (128 jobs of 128 rows): 1245 us for three outer
// iterations (1613); a sweep is 220 us, of which the base GEMMs of the longest prefixes take 95 and the positions 75.
//
// Every value is a fixed function of the iterate: the split into prefix and group depends on the
// block size and the position alone.  Waits are bounded as in the other tensor-core kernels.
#include <cuda.h>

#include <algorithm>
#include <vector>

#include "js_common.cuh"
#include "js_model.h"
#include "made_driver.cuh"
#include "tc_common.cuh"

namespace {

constexpr int BM = TC_BM, BK = TC_BK;
constexpr int NEW = 16;                      // epilogue warps: four per tensor-memory quadrant
constexpr int NEP = 32 * NEW;
constexpr int NTH = 64 + NEP;
constexpr int NUP = 32;                      // most units of one layer inside a group
constexpr int GMAX = 32;                     // most positions per group
constexpr int WS = NUP + 1;                  // row stride of the table of weights inside a group: read by targets, written by sources
constexpr int A_BYTES = BM * BK * 2;
constexpr int NB = 128;                      // units per chunk of a base GEMM
constexpr int GPB = 8;                       // groups per base: a base GEMM serves the next GPB groups
constexpr int W_BYTES = NB * BK * 2;
constexpr int STAGE_BYTES = A_BYTES + W_BYTES;          // 32 KB, a multiple of 1 KB
constexpr int BASE_COL = 256;                // tensor-memory columns of the two base accumulators (NB each)
constexpr int MAX_STAGES = 10;
constexpr int SMEM_DYN_MAX = 227 * 1024 - 4 * 1024;

struct SwShared {
    uint64_t full[MAX_STAGES], empty[MAX_STAGES], tfull, tempty, vread, gdone, bfull[2], bempty[2];
    int kbs[JS_MAXL + 1], ub0[JS_MAXL + 1];  // current base: its K blocks per layer (0: none), its first unit
    uint32_t tmem_base;
    int stop;
    int gave_up[2];                          // an epilogue warp's wait ran out: for a base, for a group
    float lut_s[2];
    // geometry of the current group, per GEMM l (activations a[l] -> a[l+1])
    int kin0[JS_MAXL + 1], nin[JS_MAXL + 1], u0[JS_MAXL + 1], nu[JS_MAXL + 1], kb_n[JS_MAXL + 1];
    int cs[JS_MAXL + 1][GMAX + 2];           // cs[l][i] = units of a[l] with degree <= t0 + i   (l >= 1)
    uint4 pk[GMAX][2];                       // units of layer slot l (a word each) that position i completes: the first one, + 32 x how
                                             // many, + 65536 x the byte offset of the first one's weights
    int most[GMAX];                          // most units of one layer that position i completes
    float bias_s[JS_MAXL + 1][NUP];
};

struct Geo { int kin0, kb_n, nin, u0, nu, npad; };
struct Base { int kbs, ub0, nb; };           // K blocks [0, kbs), units [ub0, ub0 + nb)

// shared-memory accesses by 32-bit shared address: the position loop runs on one warp per scheduler, and
// a generic load (which is what a pointer kept in a structure compiles to) waits much longer than ld.shared
__device__ __forceinline__ void sts_f4(uint32_t a, float4 v)
{
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ float lds_f(uint32_t a)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void lds_u4(uint32_t a, uint32_t *v)
{
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(a));
}
__device__ __forceinline__ void sts_f(uint32_t a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }

struct SweepEngine {
    const MadeDev &m;
    const SweepDev &sw;
    const RunArgs &r;
    SwShared &sh;
    uint8_t *ring;
    float *V;            // [L+1][128 rows][NUP]: running sums, then activations, of the group's units; a row's
                         // eight 16-byte chunks are permuted by the row number (conflict-free 16-byte accesses)
    float *Wg;           // [L+1][NUP][WS]: weights between the group's units, [source][target]
    int warp, lane;
    int stage = 0;
    uint32_t spar = 0;
    uint32_t tf_par = 0, te_par = 0, gd_par = 0, vr_par = 0;
    int bbuf = 0;                  // base accumulator in turn; bit b of bb_par: parity of its next use
    uint32_t bb_par = 0;
    bool dead = false;
    uint32_t tmem_base = 0;
    unsigned long long mma_flops = 0;

    __device__ SweepEngine(const MadeDev &m_, const SweepDev &sw_, const RunArgs &r_, SwShared &sh_, uint8_t *ring_)
        : m(m_), sw(sw_), r(r_), sh(sh_), ring(ring_)
    {
        warp = threadIdx.x >> 5;
        lane = threadIdx.x & 31;
        // The running sums V live in the operand ring's memory: the ring is idle from the moment a group's
        // prefix sums are complete until the next group's loads start, which is exactly when V is in use
        // (the threads fence their accesses against the asynchronous proxy before they let the loads go).
        V = reinterpret_cast<float *>(ring);
        uint8_t *p = ring + (size_t)sw.ring_bytes;
        Wg = reinterpret_cast<float *>(p);
    }

    // optional device timeline (JS_OPT_TRACE, js_get_trace) of the first CTA: one row of stamps per group;
    // slots: 0 operands may be loaded, 1 last MMA issued, 2 group tables ready, 3 prefix sums complete,
    // 4 prefix sums read, 5 positions done, 6 activations stored, 7 group geometry ready, 8 the group's
    // weights staged
    int group_no = 0;
    __device__ void trace(int slot) const
    {
        if (r.trace == nullptr || blockIdx.x != 0 || group_no >= JS_TRACE_PHASES) return;
        r.trace[(size_t)group_no * JS_TRACE_SLOTS + slot] = global_ns();
    }

    // units of a[l] with degree <= d (a[0]: the positions themselves, degree = position + 1)
    __device__ int cnt(int l, int d) const { return l == 0 ? d : __ldg(&sw.cnt[l][d]); }

    // group [t0, t1) of a block ending at b: hidden degrees (t0, hi] are evaluated inside it
    __device__ Geo geo(int l, int t0, int t1, int hi) const
    {
        Geo g;
        g.kin0 = cnt(l, t0);
        g.kb_n = (g.kin0 + BK - 1) / BK;
        g.nin = cnt(l, hi) - g.kin0;
        if (l < m.L) {
            g.u0 = cnt(l + 1, t0);
            g.nu = cnt(l + 1, hi) - g.u0;
        } else {
            g.u0 = t0;
            g.nu = t1 - t0;
        }
        g.npad = (g.nu + 15) & ~15;
        return g;
    }

    // Base of the GPB groups that start at position s0 (block ends at b): per layer, the sums over all FULL
    // K blocks below the first group's prefix boundary, for every unit those groups will evaluate.  The
    // groups' own GEMMs then run only over the K blocks from there on.
    __device__ Base base_of(int l, int s0, int b) const
    {
        const int sE = min(s0 + GPB * sw.G, b), hiS = min(sE, b - 1);
        Base g;
        g.kbs = cnt(l, s0) / BK;
        if (l < m.L) {
            g.ub0 = cnt(l + 1, s0);
            g.nb = cnt(l + 1, hiS) - g.ub0;
        } else {
            g.ub0 = s0;
            g.nb = sE - s0;
        }
        if (g.nb <= 0) g.kbs = 0;
        return g;
    }
    __device__ int base_start(int a, int t0) const { return a + ((t0 - a) / (GPB * sw.G)) * (GPB * sw.G); }

    __device__ uint8_t *stage_a(int s) const { return ring + (size_t)s * STAGE_BYTES; }
    __device__ uint8_t *stage_b(int s) const { return ring + (size_t)s * STAGE_BYTES + A_BYTES; }
    __device__ void advance_stage()
    {
        spar ^= 1u << stage;
        if (++stage == sw.n_stages) stage = 0;
    }

    // K blocks [kb, kb_end) of layer l through the ring (whole warp, one elected lane issues): activations from the previous
    // iterate below the block's start, else from the job's own buffer F, and a box of weight rows from row0 on
    __device__ void load_blocks(int l, int kb, int kb_end, int kb_old, int rt, int slot, const CUtensorMap *mw, int row0, uint32_t bytes)
    {
        while (kb < kb_end) {
            const int run = mbar_wait_run(sh.empty, stage, sw.n_stages, ~spar, kb_end - kb, r.ctl);
            if (run == 0) { dead = true; return; }
            for (int i = 0; i < run; ++i, ++kb) {
                if (elect_one()) {
                    mbar_expect_tx(&sh.full[stage], bytes);
                    if (kb < kb_old) tma_load_2d(smem_u32(stage_a(stage)), sw.tmAold + sw.rj_idx * (m.L + 1) + l, &sh.full[stage], kb * BK, rt * sw.rj);
                    else tma_load_3d(smem_u32(stage_a(stage)), sw.tmF + sw.rj_idx * (m.L + 1) + l, &sh.full[stage], (kb - kb_old) * BK, 0, slot);
                    tma_load_2d(smem_u32(stage_b(stage)), mw, &sh.full[stage], kb * BK, row0);
                }
                advance_stage();
            }
        }
    }
    // the MMAs of n K blocks into the accumulator d (which they start or, with `more`, continue)
    __device__ void mma_blocks(int n, uint32_t d, uint32_t idesc, bool more)
    {
        for (int kb = 0; kb < n;) {
            const int run = mbar_wait_run(sh.full, stage, sw.n_stages, spar, n - kb, r.ctl);
            if (run == 0) { dead = true; return; }
            tc_fence_after();
            for (int i = 0; i < run; ++i, ++kb) {
                const uint64_t adesc = smem_desc_sw128(smem_u32(stage_a(stage)));
                const uint64_t bdesc = smem_desc_sw128(smem_u32(stage_b(stage)));
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)
                        umma_bf16(d, adesc + (uint64_t)(2 * k), bdesc + (uint64_t)(2 * k), idesc, (more || kb > 0 || k > 0) ? 1u : 0u);
                    umma_commit(&sh.empty[stage]);
                }
                advance_stage();
            }
        }
    }

    // What the loading and the MMA warp need to know of a group, lane l for layer l (a dependent chain of loads from the
    // unit counts; one after the other for every layer they took 1 us per group): its K blocks kb0 .. kb_n, of which those
    // below kb_e hold no unit of the previous group.
    struct Steps { int kb0, kb_e, kb_n, u0, nu; };
    __device__ Steps steps_of(int a, int t0, int b) const
    {
        Steps g = {0, 0, 0, 0, 0};
        if (lane > m.L) return g;
        const int t1 = min(t0 + sw.G, b), s0 = base_start(a, t0);
        const Geo e = geo(lane, t0, t1, min(t1, b - 1));
        g.u0 = e.u0;
        g.nu = e.nu;
        if (e.nu == 0) return g;
        g.kb0 = base_of(lane, s0, b).kbs;
        g.kb_n = e.kb_n;
        g.kb_e = t0 == s0 ? g.kb0 : max(g.kb0, cnt(lane, t0 - sw.G) / BK);
        return g;
    }
    __device__ Steps of_layer(const Steps &g, int l) const
    {
        return {__shfl_sync(0xffffffffu, g.kb0, l), __shfl_sync(0xffffffffu, g.kb_e, l), __shfl_sync(0xffffffffu, g.kb_n, l),
                __shfl_sync(0xffffffffu, g.u0, l), __shfl_sync(0xffffffffu, g.nu, l)};
    }

    // ------------------------------------------------------------------ roles
    // the K blocks of a group, those that hold units of the previous group (late) or the others
    __device__ void load_group(const Steps &all, bool late, int kb_old_l, int rt, int slot)
    {
        for (int l = 0; l <= m.L && !dead; ++l) {
            const Steps g = of_layer(all, l);
            if (g.nu == 0) continue;
            const int npad = (g.nu + 15) & ~15, kb = late ? g.kb_e : g.kb0, kb_end = late ? g.kb_n : g.kb_e;
            mma_flops += 2ull * BM * BK * (unsigned long long)npad * (unsigned long long)(kb_end - kb);
            // one box of 16 or of 32 weight rows (a load per 16 rows cost a fifth of the K loop)
            load_blocks(l, kb, kb_end, __shfl_sync(0xffffffffu, kb_old_l, l), rt, slot, sw.tmW16 + (npad == 32 ? m.L + 1 : 0) + l, g.u0,
                        (uint32_t)(sw.rj + npad) * BK * 2);
        }
    }

    __device__ void producer(int rt, int slot, int a, int b)
    {
        const int kb_old_l = lane <= m.L ? cnt(lane, a) / BK : 0;
        for (int t0 = a; t0 < b && !dead; t0 += sw.G) {
            const Steps g = steps_of(a, t0, b);
            if (t0 > a) {
                // the previous group's running sums are in registers: the ring is free again
                if (!__all_sync(0xffffffffu, mbar_wait_idle(&sh.vread, vr_par, r.ctl))) { dead = true; break; }
                vr_par ^= 1u;
                load_group(g, false, kb_old_l, rt, slot);
                if (dead) break;
            }
            // the previous group's activations (or the job's start values) are in F
            if (!__all_sync(0xffffffffu, mbar_wait_idle(&sh.gdone, gd_par, r.ctl))) { dead = true; break; }
            gd_par ^= 1u;
            fence_proxy_async();
            if (lane == 0) trace(0);
            const int s0 = base_start(a, t0);
            if (t0 == s0) {
                // the base GEMMs of the next GPB groups: NB units at a time over the full K blocks of the prefix
                for (int l = 0; l <= m.L && !dead; ++l) {
                    const Base bs = base_of(l, s0, b);
                    const int kb_old = __shfl_sync(0xffffffffu, kb_old_l, l);
                    for (int c = 0; c * NB < bs.nb && bs.kbs > 0 && !dead; ++c) {
                        mma_flops += 2ull * BM * BK * NB * (unsigned long long)bs.kbs;
                        load_blocks(l, 0, bs.kbs, kb_old, rt, slot, sw.tmW16 + 2 * (m.L + 1) + l, bs.ub0 + c * NB, sw.rj * BK * 2 + NB * BK * 2);
                    }
                }
            }
            load_group(g, true, kb_old_l, rt, slot);
            group_no++;
        }
    }

    __device__ void mma_group(const Steps &all, bool late)
    {
        for (int l = 0; l <= m.L && !dead; ++l) {
            const Steps g = of_layer(all, l);
            if (g.nu == 0) continue;
            mma_blocks(late ? g.kb_n - g.kb_e : g.kb_e - g.kb0, tmem_base + (uint32_t)(l * NUP), instr_desc_bf16((g.nu + 15) & ~15), late && g.kb_e > g.kb0);
        }
    }

    __device__ void mma_issuer(int a, int b)
    {
        for (int t0 = a; t0 < b && !dead; t0 += sw.G) {
            const Steps g = steps_of(a, t0, b);
            // the epilogue has read the previous group's accumulators
            if (!__all_sync(0xffffffffu, mbar_wait_idle(&sh.tempty, te_par ^ 1u, r.ctl))) { dead = true; break; }
            te_par ^= 1u;
            tc_fence_after();
            const int s0 = base_start(a, t0);
            mma_group(g, false);
            if (dead) break;
            if (t0 == s0) {
                const uint32_t idescb = instr_desc_bf16(NB);
                for (int l = 0; l <= m.L && !dead; ++l) {
                    const Base bs = base_of(l, s0, b);
                    for (int c = 0; c * NB < bs.nb && bs.kbs > 0 && !dead; ++c) {
                        // the epilogue has copied this accumulator's previous chunk away
                        if (!__all_sync(0xffffffffu, mbar_wait(&sh.bempty[bbuf], ((bb_par >> bbuf) & 1u) ^ 1u, r.ctl))) { dead = true; break; }
                        tc_fence_after();
                        const uint32_t d_base = tmem_base + (uint32_t)(BASE_COL + bbuf * NB);
                        mma_blocks(bs.kbs, d_base, idescb, false);
                        if (dead) break;
                        if (elect_one()) umma_commit(&sh.bfull[bbuf]);
                        bb_par ^= 1u << bbuf;
                        bbuf ^= 1;
                    }
                }
                if (dead) break;
            }
            mma_group(g, true);
            if (dead) break;
            const bool any = __any_sync(0xffffffffu, g.kb_n > g.kb0);
            if (elect_one()) {
                if (any) umma_commit(&sh.tfull);
                else mbar_arrive(&sh.tfull);      // a group with empty prefixes (the very first positions)
                trace(1);
            }
            group_no++;
        }
    }

    __device__ void ep_sync() { asm volatile("bar.sync 1, %0;" ::"n"(NEP) : "memory"); }

    // unit j of the group in layer slot l, sample row `row`: its shared-memory address
    __device__ uint32_t vat(int l, int j, int row) const
    {
        return smem_u32(V) + 4u * (uint32_t)(((l * BM + row) * NUP) + ((((j >> 2) ^ (row & 7)) << 2) | (j & 3)));
    }

    // start of a job: the job's buffer F holds, per layer, the units from the K block that contains
    // the block's first old unit onwards: copies of the old activations up to degree a, zeros after
    __device__ void job_init(int rt, int slot, int a, int b)
    {
        const int row = (warp & 3) * 32 + lane, part = (warp - 2) >> 2;
        if (row < sw.rj)
            for (int l = 0; l <= m.L; ++l) {
                const int k_old = cnt(l, a), kb0 = (k_old / BK) * BK;
                const int ncopy = k_old - kb0;
                const int cols = min(sw.WF[l], ((cnt(l, min(b, m.T)) - kb0 + BK - 1) / BK) * BK);
                __nv_bfloat16 *f = sw.F[l] + ((size_t)slot * BM + row) * sw.WF[l];
                const __nv_bfloat16 *old = (const __nv_bfloat16 *)m.a[l] + (size_t)(rt * sw.rj + row) * m.n[l] + kb0;
                for (int c = 8 * part; c < cols; c += 8 * (NEW / 4)) {
                    uint4 v = make_uint4(0u, 0u, 0u, 0u);
                    if (c + 8 <= ncopy) {
                        v = __ldcg(reinterpret_cast<const uint4 *>(old + c));
                    } else if (c < ncopy) {
                        __nv_bfloat16 tmp[8];
                        for (int i = 0; i < 8; ++i) tmp[i] = c + i < ncopy ? old[c + i] : __float2bfloat16_rn(0.0f);
                        v = *reinterpret_cast<const uint4 *>(tmp);
                    }
                    *reinterpret_cast<uint4 *>(f + c) = v;
                }
            }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.gdone);
    }

    // the encodings of the rows' symbols at position i of the group, in every lane
    template <int RPW>
    __device__ __forceinline__ void sample(const float (&logit)[RPW], const float (&nz)[RPW], int i, float lut0, float lut1, float (&val)[RPW]) const
    {
        if (r.nk == JS_NOISE_LOGISTIC) {
#pragma unroll
            for (int rr = 0; rr < RPW; ++rr) val[rr] = __shfl_sync(0xffffffffu, logit[rr] + nz[rr], i);      // as js_sample_binary
#pragma unroll
            for (int rr = 0; rr < RPW; ++rr) val[rr] = val[rr] > 0.0f ? lut1 : lut0;
        } else {
            uint32_t mk = symbols(logit, nz);
            mk = __shfl_sync(0xffffffffu, mk, i);
#pragma unroll
            for (int rr = 0; rr < RPW; ++rr) val[rr] = (mk >> rr & 1u) ? lut1 : lut0;
        }
    }
    // the symbols of this lane's position, a bit per row
    template <int RPW>
    __device__ __forceinline__ uint32_t symbols(const float (&logit)[RPW], const float (&nz)[RPW]) const
    {
        uint32_t mk = 0;
#pragma unroll
        for (int rr = 0; rr < RPW; ++rr) mk |= (uint32_t)js_sample_binary(r.nk, logit[rr], nz[rr]) << rr;
        return mk;
    }
    // Two activations that are known, as every reader sees them: rounded to bf16.
    template <int ACT>
    static __device__ __forceinline__ uint32_t act2(float s0, float s1)
    {
        if (ACT == JS_ACT_RELU) {
            uint32_t v;
            asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(v) : "f"(s1), "f"(s0));
            return v;
        }
        return pack_bf16x2(tc_act_fn(ACT, s0), tc_act_fn(ACT, s1));
    }
    // The value of unit j (lane j of the running sums S, which keep it: the weights from what comes later are zero) for the
    // warp's rows, in every lane.  Two rows travel in one shuffle.
    template <int ACT, int RPW>
    static __device__ __forceinline__ void complete_unit(const float (&S)[RPW], int j, float (&val)[RPW])
    {
        uint32_t p[RPW / 2];
#pragma unroll
        for (int c = 0; c < RPW / 2; ++c) p[c] = act2<ACT>(S[2 * c], S[2 * c + 1]);
#pragma unroll
        for (int c = 0; c < RPW / 2; ++c) {
            p[c] = __shfl_sync(0xffffffffu, p[c], j);
            val[2 * c] = __uint_as_float(p[c] << 16);
            val[2 * c + 1] = __uint_as_float(p[c] & 0xffff0000u);
        }
    }
    // Units u % 32 and, with TWO, (u + 1) % 32 of S, of which as many as bits 5 and 6 of u say are complete, added to the
    // running sums of the next layer.
    template <int ACT, bool TWO, int RPW>
    static __device__ __forceinline__ void complete_units(const float (&S)[RPW], uint32_t u, float (&next)[RPW], float w0, float w1)
    {
        const bool one = (u & 96u) != 0u, two = (u & 64u) != 0u;
        uint32_t p[RPW / 2], p1[RPW / 2];
#pragma unroll
        for (int c = 0; c < RPW / 2; ++c) p[c] = act2<ACT>(S[2 * c], S[2 * c + 1]);
#pragma unroll
        for (int c = 0; c < RPW / 2; ++c) {
            if (TWO) p1[c] = __shfl_sync(0xffffffffu, p[c], (int)u + 1);
            p[c] = __shfl_sync(0xffffffffu, p[c], (int)u);
        }
#pragma unroll
        for (int c = 0; c < RPW / 2; ++c) {
            const float n0 = one ? fmaf(w0, __uint_as_float(p[c] << 16), next[2 * c]) : next[2 * c];
            const float n1 = one ? fmaf(w0, __uint_as_float(p[c] & 0xffff0000u), next[2 * c + 1]) : next[2 * c + 1];
            next[2 * c] = TWO && two ? fmaf(w1, __uint_as_float(p1[c] << 16), n0) : n0;
            next[2 * c + 1] = TWO && two ? fmaf(w1, __uint_as_float(p1[c] & 0xffff0000u), n1) : n1;
        }
    }
    // shared-memory address of the weight from source k of a[l] to target j
    __device__ __forceinline__ uint32_t wat(int l, int k, int j) const { return smem_u32(Wg) + 4u * (uint32_t)((l * NUP + k) * WS + j); }
    template <int RPW>
    static __device__ __forceinline__ void add(float (&S)[RPW], float w, const float (&val)[RPW])
    {
#pragma unroll
        for (int rr = 0; rr < RPW; ++rr) S[rr] = fmaf(w, val[rr], S[rr]);
    }

    // The positions of a group in order: S = the running sums of the warp's rows.  Afterwards every lane's S are those of its
    // units and of its position: what comes later has weight zero there.
    template <int L, int RPW, int ACT>
    __device__ __forceinline__ void solve(float (&S)[L + 1][RPW], const float (&nz)[RPW], int ng, bool last) const
    {
        const int most = __reduce_max_sync(0xffffffffu, lane < ng ? sh.most[lane] : 0);
        if (most <= 1) {
            solve_few<L, RPW, ACT, false>(S, nz, ng, last);
        } else if (most == 2) {
            solve_few<L, RPW, ACT, true>(S, nz, ng, last);
        } else {
            const float lut0 = sh.lut_s[0], lut1 = sh.lut_s[1];
            for (int i = 0; i < ng; ++i) {
                if (last && i == ng - 1) break;
                float val[RPW];
                sample(S[L], nz, i, lut0, lut1, val);
                add(S[0], lds_f(wat(0, i, lane)), val);
#pragma unroll
                for (int l = 0; l < L; ++l) {
                    const int j0 = sh.cs[l + 1][i] - sh.u0[l], j1 = sh.cs[l + 1][i + 1] - sh.u0[l];
                    for (int j = j0; j < j1; ++j) {
                        complete_unit<ACT>(S[l], j, val);
                        add(S[l + 1], lds_f(wat(l + 1, j, lane)), val);
                    }
                }
            }
        }
    }
    // The same where a position completes at most one (TWO: two) units of a layer: no branch.  With one warp per scheduler a
    // position costs the chain of its shuffles (some 200 cycles for two layers), with four of them the instructions: 11 or 16
    // a row and 35 besides.
    template <int L, int RPW, int ACT, bool TWO>
    __device__ __forceinline__ void solve_few(float (&S)[L + 1][RPW], const float (&nz)[RPW], int ng, bool last) const
    {
        const float lut0 = sh.lut_s[0], lut1 = sh.lut_s[1];
        const uint32_t wl = wat(0, 0, lane), pks = smem_u32(sh.pk);
        uint32_t pk[8];
        lds_u4(pks, pk);
        if (L > 4) lds_u4(pks + 16u, pk + 4);
        for (int i = 0; i < ng; ++i) {
            if (last && i == ng - 1) break;
            float w[L + 1][2];                           // asked for before the symbol is known
            w[0][0] = lds_f(wl + (uint32_t)(i * WS * 4));
            uint32_t u[L];
#pragma unroll
            for (int l = 0; l < L; ++l) {
                u[l] = pk[l];
                w[l + 1][0] = lds_f(wl + (u[l] >> 16));
                w[l + 1][1] = TWO ? lds_f(wl + (u[l] >> 16) + WS * 4) : 0.0f;
            }
            const uint32_t at = pks + 32u * (uint32_t)min(i + 1, GMAX - 1);
            lds_u4(at, pk);
            if (L > 4) lds_u4(at + 16u, pk + 4);
            float val[RPW];
            sample(S[L], nz, i, lut0, lut1, val);
            add(S[0], w[0][0], val);
#pragma unroll
            for (int l = 0; l < L; ++l) complete_units<ACT, TWO>(S[l], u[l], S[l + 1], w[l + 1][0], w[l + 1][1]);
        }
    }

    template <int L, int RPW>
    __device__ void epilogue(int rt, int slot, int a, int b, uint32_t &changed)
    {
        const int q = warp & 3, part = (warp - 2) >> 2, row = q * 32 + lane, tid = threadIdx.x - 64;
        const int r0 = RPW * (warp - 2);                 // this warp's rows in the position loop
        const bool active = r0 < sw.rj;
        const float lut0 = sh.lut_s[0], lut1 = sh.lut_s[1];
        int kb_old[L + 1];
#pragma unroll
        for (int l = 0; l <= L; ++l) kb_old[l] = cnt(l, a) / BK;
        job_init(rt, slot, a, b);
        for (int t0 = a; t0 < b && !dead; t0 += sw.G) {
            const int t1 = min(t0 + sw.G, b), hi = min(t1, b - 1), ng = t1 - t0;
            // ---- geometry, small tables, the weights between the group's units, noise (while the GEMMs run)
            ep_sync();                                   // everybody is done with the previous group's tables
            const int s0 = base_start(a, t0);
            if (tid <= L) {
                const Geo g = geo(tid, t0, t1, hi);
                sh.kin0[tid] = g.kin0; sh.nin[tid] = g.nin; sh.u0[tid] = g.u0; sh.nu[tid] = g.nu; sh.kb_n[tid] = g.kb_n;
                const Base bs = base_of(tid, s0, b);
                sh.kbs[tid] = bs.kbs; sh.ub0[tid] = bs.ub0;
            }
            for (int i = tid; i < (L + 1) * (GMAX + 2); i += NEP) {
                const int l = i / (GMAX + 2), k = i % (GMAX + 2);
                if (l >= 1) sh.cs[l][k] = cnt(l, min(t0 + k, m.T));
            }
            // noise and the symbols the positions hold now, lane = position (asked for now, used behind the GEMMs)
            float nz[RPW];
            uint32_t xold = 0;                           // bit rr: row rr's symbol; bit 8 + rr: it holds no symbol yet
#pragma unroll
            for (int rr = 0; rr < RPW; ++rr) {
                const int s2 = rt * sw.rj + r0 + rr;
                const bool in = active && s2 < r.batch && lane < ng;
                nz[rr] = in ? __ldg(r.noise + (size_t)s2 * m.T + t0 + lane) : 0.0f;
                const uint32_t xo = in ? r.x[(size_t)s2 * m.T + t0 + lane] : 0u;
                xold |= (xo & 1u) << rr | (uint32_t)(xo > 1u) << (8 + rr);
            }
            ep_sync();
            if (tid == 0) trace(7);
            {
                // warp = two targets per layer, lane = source: every load of the thread first (coalesced over the sources),
                // the stores to the source-major table after them
                const int j = 2 * (warp - 2);
                __nv_bfloat16 wv[L + 1][2];
#pragma unroll
                for (int l = 0; l <= L; ++l) {
                    const __nv_bfloat16 *Wl = (const __nv_bfloat16 *)m.W[l] + (size_t)(sh.u0[l] + j) * m.n[l] + sh.kin0[l] + lane;
#pragma unroll
                    for (int jj = 0; jj < 2; ++jj)
                        wv[l][jj] = (j + jj < sh.nu[l] && lane < sh.nin[l]) ? Wl[(size_t)jj * m.n[l]] : __float2bfloat16_rn(0.0f);
                }
                float bv = 0.0f;
                if (tid < (L + 1) * NUP && (tid & 31) < sh.nu[tid >> 5]) bv = __ldg(m.bias[tid >> 5] + sh.u0[tid >> 5] + (tid & 31));
#pragma unroll
                for (int l = 0; l <= L; ++l) {
                    sts_f(wat(l, lane, j), __bfloat162float(wv[l][0]));
                    sts_f(wat(l, lane, j + 1), __bfloat162float(wv[l][1]));
                }
                if (tid < (L + 1) * NUP) sh.bias_s[tid >> 5][tid & 31] = bv;
                if (tid < ng) {
                    uint32_t pk[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                    int most = 0;
#pragma unroll
                    for (int l = 0; l < L; ++l) {
                        const int n = sh.cs[l + 1][tid + 1] - sh.cs[l + 1][tid], j = (sh.cs[l + 1][tid] - sh.u0[l]) & 31;
                        most = max(most, n);
                        pk[l] = (uint32_t)(j | min(n, 2) << 5 | ((l + 1) * NUP + j) * WS * 4 << 16);
                    }
                    sh.pk[tid][0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    sh.pk[tid][1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                    sh.most[tid] = most;
                }
            }
            ep_sync();
            if (tid == 0) trace(2);
            // ---- a new base: its sums go from tensor memory to this job's part of S, chunk by chunk, as the
            // MMAs deliver them; a warp takes 32 columns of its quadrant's rows
            if (t0 == s0) {
                for (int l = 0; l <= L && !dead; ++l) {
                    const Base bs = base_of(l, s0, b);
                    float *Sl = sw.S + (((size_t)slot * (L + 1) + l) * sw.nbs) * BM + row;
                    for (int c = 0; c * NB < bs.nb && bs.kbs > 0; ++c) {
                        if (!__all_sync(0xffffffffu, mbar_wait(&sh.bfull[bbuf], (bb_par >> bbuf) & 1u, r.ctl))) { dead = true; break; }
                        tc_fence_after();
                        static_assert(NB == 32 * (NEW / 4), "32 columns of a chunk per warp");
                        if (q * 32 < sw.rj) {
                            float v[32];
                            tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(BASE_COL + bbuf * NB + 32 * part), v);
#pragma unroll
                            for (int i = 0; i < 32; ++i) __stcg(Sl + (size_t)(c * NB + 32 * part + i) * BM, v[i]);
                        }
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&sh.bempty[bbuf]);
                        bb_par ^= 1u << bbuf;
                        bbuf ^= 1;
                    }
                }
                if (dead) sh.gave_up[0] = 1;
                __threadfence_block();
                ep_sync();                               // a row's sums are read by another warp of its quadrant
                if (*(volatile int *)&sh.gave_up[0]) { dead = true; break; }     // all leave at the same place
            }
            // ---- the next group's tables (weights between its units, noise, symbols) are touched once per
            // sweep and would come from DRAM, two dependent round trips of 2.5 us each: ask for them now
            if (t1 < b) {
                const int t2 = min(t1 + sw.G, b), hi2 = min(t2, b - 1);
                for (int i = tid; i < (L + 1) * NUP; i += NEP) {
                    const int l = i / NUP, j = i % NUP;
                    const Geo g = geo(l, t1, t2, hi2);
                    if (j < g.nu && g.nin > 0) {
                        const __nv_bfloat16 *pw = (const __nv_bfloat16 *)m.W[l] + (size_t)(g.u0 + j) * m.n[l] + g.kin0;
                        prefetch_l2(pw);
                        prefetch_l2(pw + g.nin - 1);
                    }
                }
                const int row2 = tid & 127, smp = rt * sw.rj + row2, what = tid >> 7;
                if (row2 < sw.rj && smp < r.batch) {
                    const float *np = r.noise + (size_t)smp * m.T + t1;
                    if (what == 0) prefetch_l2(np);
                    else if (what == 1) prefetch_l2(np + (t2 - t1) - 1);
                    else if (what == 2) prefetch_l2(r.x + (size_t)smp * m.T + t1);
                }
            }
            // ---- prefix sums out of tensor memory
            if (!__all_sync(0xffffffffu, mbar_wait(&sh.tfull, tf_par, r.ctl))) sh.gave_up[1] = 1;
            tf_par ^= 1u;
            tc_fence_after();
            if (tid == 0) trace(3);
            if (q * 32 < sw.rj)
                for (int l = part; l <= L; l += NEW / 4) {
                    float v[32];
                    if (sh.nu[l] > 0 && sh.kb_n[l] > sh.kbs[l]) {
                        tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(l * NUP), v);
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; ++i) v[i] = 0.0f;
                    }
                    if (sh.kbs[l] > 0 && sh.nu[l] > 0) {
                        // base + the group's own K blocks (in that order, always)
                        const float *Sl = sw.S + (((size_t)slot * (L + 1) + l) * sw.nbs + (sh.u0[l] - sh.ub0[l])) * BM + row;
                        const int nuv = sh.nu[l];
                        float sv[32];
#pragma unroll
                        for (int i = 0; i < 32; ++i) sv[i] = i < nuv ? __ldcg(Sl + (size_t)i * BM) : 0.0f;
#pragma unroll
                        for (int i = 0; i < 32; ++i) v[i] = sv[i] + v[i];
                    }
                    // running pre-activation of every unit of the group: prefix sum + bias; the group's own
                    // contributions are added below, each as soon as its source exists
                    const uint32_t v4 = smem_u32(V) + 4u * (uint32_t)((l * BM + row) * NUP);
#pragma unroll
                    for (int c = 0; c < NUP / 4; ++c)
                        sts_f4(v4 + 16u * (uint32_t)(c ^ (row & 7)),
                               make_float4(v[4 * c] + sh.bias_s[l][4 * c], v[4 * c + 1] + sh.bias_s[l][4 * c + 1],
                                           v[4 * c + 2] + sh.bias_s[l][4 * c + 2], v[4 * c + 3] + sh.bias_s[l][4 * c + 3]));
                }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.tempty);
            ep_sync();
            if (*(volatile int *)&sh.gave_up[1]) { dead = true; break; }
            if (tid == 0) trace(4);
            // ---- the group's positions in order.  A value that becomes known (a sampled symbol, then the hidden units it
            // completes, layer by layer) is added at once to the running sums of everything in the group that reads it; each
            // target receives its sources in index order.
            float S[L + 1][RPW];
#pragma unroll
            for (int l = 0; l <= L; ++l)
#pragma unroll
                for (int rr = 0; rr < RPW; ++rr) S[l][rr] = active ? lds_f(vat(l, lane, r0 + rr)) : 0.0f;
            fence_proxy_async_smem();         // the next group's loads overwrite the running sums' memory
            __syncwarp();
            if (t1 < b && lane == 0) mbar_arrive(&sh.vread);
            const bool last = t0 + ng > hi;              // the block's last position completes nothing that the block reads
            if (!active) {
            } else if (m.act == JS_ACT_RELU) solve<L, RPW, JS_ACT_RELU>(S, nz, ng, last);
            else solve<L, RPW, JS_ACT_GELU_TANH>(S, nz, ng, last);
            const uint32_t bits = active ? symbols(S[L], nz) : 0u;
            if (tid == 0) trace(5);
            // ---- the group's activations into F, for the GEMMs of the groups that follow; symbols that changed
            if (t1 < b) {
                if (active && lane < ng) {
                    __nv_bfloat16 *dst = sw.F[0] + ((size_t)slot * BM + r0) * sw.WF[0] + (t0 - kb_old[0] * BK) + lane;
#pragma unroll
                    for (int rr = 0; rr < RPW; ++rr) dst[(size_t)rr * sw.WF[0]] = __float2bfloat16_rn((bits >> rr & 1u) ? lut1 : lut0);
                }
#pragma unroll
                for (int l = 1; l <= L; ++l)
                    if (active && lane < sh.nin[l]) {
                        __nv_bfloat16 *dst = sw.F[l] + ((size_t)slot * BM + r0) * sw.WF[l] + (sh.kin0[l] - kb_old[l] * BK) + lane;
#pragma unroll
                        for (int c = 0; c < RPW / 2; ++c) {
                            const uint32_t v = m.act == JS_ACT_RELU ? act2<JS_ACT_RELU>(S[l - 1][2 * c], S[l - 1][2 * c + 1])
                                                                    : act2<JS_ACT_GELU_TANH>(S[l - 1][2 * c], S[l - 1][2 * c + 1]);
                            dst[(size_t)(2 * c) * sw.WF[l]] = __ushort_as_bfloat16((unsigned short)v);
                            dst[(size_t)(2 * c + 1) * sw.WF[l]] = __ushort_as_bfloat16((unsigned short)(v >> 16));
                        }
                    }
                fence_proxy_async();          // F for the next group's loads
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.gdone);
            }
            if (active && lane < ng)
#pragma unroll
                for (int rr = 0; rr < RPW; ++rr) {
                    const int s2 = rt * sw.rj + r0 + rr;
                    if (s2 < r.batch && (((bits ^ xold) | xold >> 8) >> rr & 1u)) {
                        r.x[(size_t)s2 * m.T + t0 + lane] = (uint8_t)(bits >> rr & 1u);
                        changed |= 1u << rr;
                    }
                }
            if (tid == 0) trace(6);
            group_no++;
        }
    }
};

// LT = the model's number of hidden layers, RPW = sample rows per epilogue warp
template <int LT, int RPW>
__global__ void __launch_bounds__(NTH, 1)
made_sweep_kernel(const __grid_constant__ MadeDev m, const __grid_constant__ SweepDev sw, const __grid_constant__ RunArgs r)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ SwShared sh;
    uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) { mbar_init(&sh.full[s], 1); mbar_init(&sh.empty[s], 1); }
        mbar_init(&sh.tfull, 1);
        mbar_init(&sh.tempty, NEW);
        mbar_init(&sh.vread, NEW);
        mbar_init(&sh.gdone, NEW);
        for (int i = 0; i < 2; ++i) { mbar_init(&sh.bfull[i], 1); mbar_init(&sh.bempty[i], NEW); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
        sh.gave_up[0] = sh.gave_up[1] = 0;
        sh.lut_s[0] = m.lut[0];
        sh.lut_s[1] = m.lut[1];
    }
    if (warp == 1) tmem_alloc(&sh.tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    SweepEngine e(m, sw, r, sh, ring);
    e.tmem_base = sh.tmem_base;
    // jobs: (row tile, block), the blocks with the longest prefixes first
    const int B = r.block, nblk = (m.T + B - 1) / B, MT = (r.batch + sw.rj - 1) / sw.rj;
    const int njobs = MT * (nblk - r.blk_lo);
    for (int job = blockIdx.x; job < njobs; job += gridDim.x) {
        const int blk = nblk - 1 - job / MT, rt = job % MT;
        const int a = blk * B, b = min(a + B, m.T);
        // The accumulators and the ring are idle between jobs; the roles meet here so that a job's
        // start values are never written while the previous job is still being read, and so that
        // all of them see the same answer to "has a wait given up".
        __syncthreads();
        if (threadIdx.x == 0) sh.stop = ld_volatile_i32(&r.ctl->abort);
        __syncthreads();
        if (sh.stop) break;
        if (warp == 0) {
            e.producer(rt, blockIdx.x, a, b);
        } else if (warp == 1) {
            e.mma_issuer(a, b);
        } else {
            uint32_t changed = 0;
            e.template epilogue<LT, RPW>(rt, blockIdx.x, a, b, changed);
            changed = __reduce_or_sync(0xffffffffu, changed);
            if (e.lane < RPW && (changed >> e.lane & 1u)) r.smp_changed[rt * sw.rj + RPW * (warp - 2) + e.lane] = 1;
        }
        __syncwarp();
    }
    DriverResult res = {JS_OK, 0, m.T, !e.dead};
    tc_fence_before();
    __syncthreads();
    if (!res.alive || ld_volatile_i32(&r.ctl->abort) != 0) {
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);      // let copies still in flight land
        res.alive = false;
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(e.tmem_base, 512);
    }
    driver_finish(r, res, 0, 0, e.mma_flops, 0);
}

// Per-sample bookkeeping of Jacobi-GS after outer iteration k (one CTA): a sample whose iterate did
// not change stops counting; the flags are cleared for the next iteration and the host learns
// whether anything changed.
__global__ void jgs_book_kernel(int batch, int k, int at_cap, int *changed, int *done, int32_t *out_iters, int *any_out)
{
    __shared__ int any;
    if (threadIdx.x == 0) any = 0;
    __syncthreads();
    for (int b = threadIdx.x; b < batch; b += blockDim.x) {
        const int c = changed[b];
        if (c) any = 1;
        if (!done[b] && (c == 0 || at_cap)) {
            done[b] = 1;
            if (out_iters) out_iters[b] = k;
        }
        changed[b] = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        // the host polls this word and returns when it is there: everything the block has written comes before it
        __threadfence_system();
        *reinterpret_cast<volatile int *>(any_out) = any;
    }
}

}  // namespace

// --------------------------------------------------------------- host side
typedef void (*SweepKernelFn)(const MadeDev, const SweepDev, const RunArgs);
template <int L>
static SweepKernelFn sweep_kernel_of(int rj_idx)
{
    // eight warps of four rows for 32 rows: a position costs a warp 40 instructions besides those of its rows
    return rj_idx == 2 ? made_sweep_kernel<L, 8> : made_sweep_kernel<L, 4>;
}
static SweepKernelFn sweep_kernel_of(int L, int rj_idx)
{
    switch (L) {
    case 1: return sweep_kernel_of<1>(rj_idx);
    case 2: return sweep_kernel_of<2>(rj_idx);
    case 3: return sweep_kernel_of<3>(rj_idx);
    case 4: return sweep_kernel_of<4>(rj_idx);
    case 5: return sweep_kernel_of<5>(rj_idx);
    case 6: return sweep_kernel_of<6>(rj_idx);
    default: return sweep_kernel_of<7>(rj_idx);
    }
}

// Builds what the sweeps need beside the tensor-core view of the model: prefix counts per degree,
// the group size, the jobs' buffers F and the tensor maps.  Returns 1 if the model qualifies
// (binary positions, sorted degrees, bf16), 0 if not, negative on CUDA errors.  Called on first use.
int js_sweep_prepare(js_model *mo)
{
    if (mo->sweep_state != 0) return mo->sweep_state > 0 ? 1 : 0;
    mo->sweep_state = -1;
    const MadeDev &v = mo->made;
    SweepDev &s = mo->sweep;
    if (!mo->tc_ok || v.C != 1 || v.prec != JS_BF16 || !js_tensor_maps()) return 0;
    if ((v.L + 1) * NUP > BASE_COL) return 0;              // the groups' accumulators end where the base's begin
    const int L = v.L, T = v.T;
    // prefix counts; the group size is the largest one that keeps every layer's units of a group within NUP
    std::vector<std::vector<int>> cnt(L + 1);
    for (int l = 1; l <= L; ++l) {
        cnt[l].assign(T + 1, 0);
        const std::vector<int> &dg = mo->host_deg[l];
        for (size_t i = 1; i < dg.size(); ++i)
            if (dg[i] < dg[i - 1]) return 0;                       // needs sorted degrees
        size_t p = 0;
        for (int d = 0; d <= T; ++d) {
            while (p < dg.size() && dg[p] <= d) ++p;
            cnt[l][d] = (int)p;
        }
    }
    int G = GMAX;
    for (; G >= 1; --G) {
        bool ok = true;
        for (int l = 1; l <= L && ok; ++l)
            for (int d = 0; d < T && ok; ++d)
                if (cnt[l][std::min(d + G, T)] - cnt[l][d] > NUP) ok = false;
        if (ok) break;
    }
    if (G < 1) return 0;
    s.G = G;
    const int v_bytes = (L + 1) * NUP * BM * 4;            // shares the ring's memory
    const int fixed = ((L + 1) * NUP + 1) * WS * 4;      // one row more: a pair of rows is read at the last one too
    s.n_stages = std::min(MAX_STAGES, (SMEM_DYN_MAX - 1024 - fixed) / STAGE_BYTES);
    if (s.n_stages < 2) return 0;
    s.ring_bytes = std::max(s.n_stages * STAGE_BYTES, (v_bytes + 1023) / 1024 * 1024);
    if (1024 + s.ring_bytes + fixed > SMEM_DYN_MAX) return 0;
    s.smem_bytes = 1024 + s.ring_bytes + fixed;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms < 1) return 0;
    s.slots = sms;
    auto fail = [&]() { cudaGetLastError(); return JS_ERR_CUDA; };
    // activations: boxes of 32, 64 and 128 sample rows; weights: of 16, of 32 and of NB rows
    std::vector<CUtensorMap> mapsA(3 * (L + 1)), mapsF(3 * (L + 1)), mapsW(3 * (L + 1));
    for (int l = 0; l <= L; ++l) {
        if (l >= 1) {
            void *p = nullptr;
            if (cudaMalloc(&p, (T + 1) * sizeof(int)) != cudaSuccess) return fail();
            mo->allocs.push_back(p);
            if (cudaMemcpy(p, cnt[l].data(), (T + 1) * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess) return fail();
            s.cnt[l] = (const int *)p;
        } else {
            s.cnt[l] = nullptr;
        }
        s.WF[l] = (v.n[l] + BK - 1) / BK * BK + BK;
        void *f = nullptr;
        const size_t bytes = (size_t)s.slots * BM * s.WF[l] * 2;
        if (cudaMalloc(&f, bytes) != cudaSuccess) return fail();
        mo->allocs.push_back(f);
        if (cudaMemset(f, 0, bytes) != cudaSuccess) return fail();
        s.F[l] = (__nv_bfloat16 *)f;
        {
            const cuuint64_t dims[3] = {(cuuint64_t)s.WF[l], (cuuint64_t)BM, (cuuint64_t)s.slots};
            const cuuint64_t strides[2] = {(cuuint64_t)s.WF[l] * 2, (cuuint64_t)s.WF[l] * 2 * BM};
            const cuuint64_t dimsA[2] = {(cuuint64_t)v.n[l], (cuuint64_t)mo->rows}, stridesA[1] = {(cuuint64_t)v.n[l] * 2};
            for (int i = 0; i < 3; ++i) {
                const cuuint32_t box[3] = {(cuuint32_t)BK, 32u << i, 1};
                if (!js_encode_map(&mapsF[i * (L + 1) + l], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, f, 3, dims, strides, box)) return 0;
                if (!js_encode_map(&mapsA[i * (L + 1) + l], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, v.a[l], 2, dimsA, stridesA, box)) return 0;
            }
        }
        for (int big = 0; big < 3; ++big) {
            const cuuint64_t dims[2] = {(cuuint64_t)v.n[l], (cuuint64_t)v.n[l + 1]};
            const cuuint64_t strides[1] = {(cuuint64_t)v.n[l] * 2};
            const cuuint32_t box[2] = {(cuuint32_t)BK, big == 2 ? (cuuint32_t)NB : 16u << big};
            if (!js_encode_map(&mapsW[big * (L + 1) + l], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, v.W[l], 2, dims, strides, box)) return 0;
        }
    }
    void *pf = nullptr, *pw = nullptr, *pa = nullptr;
    if (cudaMalloc(&pf, 3 * (L + 1) * sizeof(CUtensorMap)) != cudaSuccess) return fail();
    mo->allocs.push_back(pf);
    if (cudaMalloc(&pa, 3 * (L + 1) * sizeof(CUtensorMap)) != cudaSuccess) return fail();
    mo->allocs.push_back(pa);
    if (cudaMemcpy(pa, mapsA.data(), 3 * (L + 1) * sizeof(CUtensorMap), cudaMemcpyHostToDevice) != cudaSuccess) return fail();
    if (cudaMalloc(&pw, 3 * (L + 1) * sizeof(CUtensorMap)) != cudaSuccess) return fail();
    mo->allocs.push_back(pw);
    if (cudaMemcpy(pf, mapsF.data(), 3 * (L + 1) * sizeof(CUtensorMap), cudaMemcpyHostToDevice) != cudaSuccess) return fail();
    if (cudaMemcpy(pw, mapsW.data(), 3 * (L + 1) * sizeof(CUtensorMap), cudaMemcpyHostToDevice) != cudaSuccess) return fail();
    s.tmF = (const CUtensorMap *)pf;
    s.tmW16 = (const CUtensorMap *)pw;
    s.tmAold = (const CUtensorMap *)pa;
    {
        // base sums: per slot and layer, room for the units of GPB groups (rounded up to whole chunks)
        int nbs = NB;
        for (int l = 1; l <= L; ++l)
            for (int d = 0; d < T; ++d) nbs = std::max(nbs, cnt[l][std::min(d + GPB * G, T)] - cnt[l][d]);
        nbs = std::max(nbs, GPB * G);
        s.nbs = (nbs + NB - 1) / NB * NB;
        void *p = nullptr;
        const size_t bytes = (size_t)s.slots * (L + 1) * s.nbs * BM * sizeof(float);
        if (cudaMalloc(&p, bytes) != cudaSuccess) return fail();
        mo->allocs.push_back(p);
        s.S = (float *)p;
    }
    {
        void *p = nullptr;
        if (cudaMalloc(&p, 2 * (size_t)mo->rows * sizeof(int)) != cudaSuccess) return fail();
        mo->allocs.push_back(p);
        if (cudaMemset(p, 0, 2 * (size_t)mo->rows * sizeof(int)) != cudaSuccess) return fail();
        mo->sw_flags = (int *)p;
        if (cudaHostAlloc((void **)&mo->h_any, sizeof(int), cudaHostAllocMapped) != cudaSuccess) return fail();
        if (cudaHostGetDevicePointer((void **)&mo->d_any, mo->h_any, 0) != cudaSuccess) return fail();
    }
    for (int i = 1; i < 3; ++i)
        if (cudaFuncSetAttribute(sweep_kernel_of(L, i), cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_DYN_MAX) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
    mo->sweep_state = 1;
    return 1;
}

// One launch: sweeps of every block >= r.blk_lo (block size r.block) for every row tile.
int js_launch_made_sweep(const js_model *mo, const RunArgs &r, cudaStream_t stream)
{
    SweepDev s = mo->sweep;
    const int nblk = (mo->made.T + r.block - 1) / r.block - r.blk_lo;
    // Sample rows per job: as few (32, 64) as leave every job an SM of its own.  A position costs a job the chain of its
    // layers, and beyond 32 rows the issue slots of several warps per scheduler.
    s.rj_idx = 0;
    while (s.rj_idx < 2 && (r.batch + (32 << s.rj_idx) - 1) / (32 << s.rj_idx) * nblk > s.slots) s.rj_idx++;
    s.rj = 32 << s.rj_idx;
    const int njobs = (r.batch + s.rj - 1) / s.rj * nblk;
    if (njobs < 1) return (int)cudaErrorInvalidValue;
    const int grid = std::min(njobs, s.slots);
    sweep_kernel_of(mo->made.L, s.rj_idx)<<<grid, NTH, s.smem_bytes, stream>>>(mo->made, s, r);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? 0 : (int)e;
}

int js_launch_jgs_book(const js_model *mo, int batch, int k, int at_cap, int32_t *out_iters, cudaStream_t stream)
{
    jgs_book_kernel<<<1, 256, 0, stream>>>(batch, k, at_cap, mo->sw_flags, mo->sw_flags + mo->rows, out_iters, mo->d_any);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? 0 : (int)e;
}
