// Binary bf16 masked MLPs of ordinary size on the sm_100a tensor cores: every thread-block cluster solves its own samples.
//
// Samples never look at one another.  made_tc.cu still runs all of them in step: a layer is a phase of the whole grid, ended
// by a grid barrier, its activations written to and read back from L2; at 10 us a phase (fill 1.4, K loop 4, epilogue 2,
// barrier 1.6) such a call is bound by the chain of its phases, not by its work.  Here a cluster of CS <= 8 CTAs takes R <= 64
// samples through the whole solve, and nothing waits for other clusters:
//   - a layer is cut into tiles of 64 units, dealt to the CTAs so that their K ranges even out (masks are triangular: a tile
//     needs 1 .. all K blocks).  A tile is D[64 units x R samples] = W[64 x K] * A[R x K]^T: the weights are the M side of
//     tcgen05.mma, so that few samples do not waste its rows.  Two threads issue, one the even K blocks into one accumulator,
//     one the odd ones into another (the looks at a K block's barriers and its four MMAs take a thread 200 cycles, the tensor
//     core 96); the epilogue adds the two;
//   - every CTA holds the activations that its tiles read, for its R samples, in shared memory, K block by K block in the layout
//     the MMA reads.  A finished tile IS one K block of the layer above: it is written in place and sent to the other CTAs by
//     one bulk copy each (cp.async.bulk to distributed shared memory, completing on the receiver's mbarrier for that block).
//     An MMA waits for the K blocks it reads, not for a layer: there is no barrier inside a pass;
//   - weights stream from L2 through a ring, two K blocks a load, independent of all that: the next tile's, and in Jacobi mode the
//     next pass's, weights are on their way while a layer waits for its inputs;
//   - noise, symbols and biases of the CTA's own output positions stay in shared memory.
// A pass ends with one exchange of change masks (64 bits, one per sample) between the CTAs.
// What bounds it: the chain of a pass (per layer: last K block arrives -> MMAs -> epilogue -> copy), and for wide models
// the weight stream (each cluster reads all live weights per pass).  784 positions, 1024 units x 2, 24 samples a cluster: 12 us a
// pass, of which three layers at 3.2 and 1.5 from the last mask to the next pass's first MMA; 16.5 before the loads took two
// blocks, one thread of a warp looked for weights, activations and room at once (a look is 150 cycles), and every role
// saw the masks itself.
//
// Solvers: Jacobi (Algorithm 1) and GS-Jacobi (Algorithm 3), the control logic of made_driver.cuh on the cluster's samples.
// Warps: 0 weight loads, 1 and 7 MMA (1 owns tensor memory), 2-5 epilogue, 6 arms and drains the activation barriers.
// All waits are bounded, as in the other tensor-core kernels.
#include <cuda.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "js_common.cuh"
#include "js_model.h"
#include "made_driver.cuh"
#include "tc_common.cuh"

namespace {

constexpr int BK = TC_BK;
constexpr int TM = 64;                       // units per tile
constexpr int NTH = 256;
constexpr int STAGE = TM * BK * 2;           // 8 KB of weights
constexpr int MAX_STAGES = 16;               // of 8 KB; they are used in pairs, an even K block and the odd one behind it
constexpr int NSLOT = 2, ACC = 64;           // accumulator slots; columns of one accumulator (two per slot: even, odd K blocks)
constexpr int MAXOWN = CL_TILES / 8;         // own tiles per layer (the cluster size grows with the tile count)
constexpr int SMEM_MAX = 227 * 1024 - 4 * 1024;      // beside ClShared

struct ClShared {
    uint64_t full[MAX_STAGES / 2], empty[MAX_STAGES / 2], tfull[NSLOT], tempty[NSLOT];
    uint64_t xbar[2][CL_TILES];              // K block of the encoded iterate complete in this CTA, by pass parity
    uint64_t hbar[CL_MAXL][CL_TILES];        // K block of a[l + 1] complete in this CTA
    uint64_t pbar[2];                        // by pass parity: every CTA of the cluster has finished the pass, their masks are here
    uint64_t go;                             // the next pass may start (or the roles may leave)
    uint64_t ack;                            // the loading and MMA warps are done with the pass's ranges
    uint32_t tmem_base;
    int stop, dead;
    int2 rng[2][CL_MAXL + 1];                // per pass parity and layer: the tiles that are computed
    int nown[CL_MAXL + 1];                   // this CTA's tiles per layer, ascending, and the K blocks they read
    int2 own[CL_MAXL + 1][MAXOWN];
    uint32_t chg[2][2];                      // per pass parity: change mask of this CTA's positions
    int first[2];
    uint4 flags[2][8];                       // per pass parity and CTA: change mask, smallest changed position
    int count[64];
    int issued, consumed[2];                 // weight loads; K blocks multiplied, even and odd ones
    int consumed_loads;
    uint64_t apar[2][CL_MAXL + 2];           // of either MMA thread: parity of the next completion of every K block's barrier
    unsigned tiles;
    unsigned sums[2];                        // of the whole cluster (in its first CTA): tiles, K blocks
    unsigned char place[CL_MAXL][MAXOWN];    // this CTA's hidden tiles: K block of a[l + 1] that it keeps them in
};
static_assert(sizeof(ClShared) <= 4 * 1024, "SMEM_MAX leaves this much");

__device__ __forceinline__ void copy_to_peer(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "r"(src), "r"(bytes), "r"(bar) : "memory");
}
// 16 bytes into another CTA's shared memory, counted on the barrier there as they arrive
__device__ __forceinline__ void send16(uint32_t dst, uint4 v, uint32_t bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar) : "memory");
}
// two 8 x 8 blocks in that order of the threads, transposed: lane i (and i + 8) gives the address of the first (second) block's column i
__device__ __forceinline__ void stmatrix2_trans(uint32_t addr, uint32_t a, uint32_t b)
{
    asm volatile("stmatrix.sync.aligned.m8n8.x2.trans.shared.b16 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr) : "memory");
}

struct ClEngine {
    const MadeDev &m;
    const ClusterDev &cd;
    const RunArgs &r;
    ClShared &sh;
    uint8_t *ring, *acts;
    uint8_t *stag;                // [pass parity][own output tile][R x 128 bytes]: encodings on their way to the CTAs
    float *nz;                    // [own output tile][R][64]
    uint64_t *xs;                 // [own output tile][64]: bit s = symbol of sample s
    float *bias;                  // [own tile of layer 0, 1, ..][64]
    const int R;
    int rank, CS, L, NP, warp, lane;          // NP: pairs in the weight ring
    uint32_t blk_bytes;           // one K block of activations: R x 128 bytes
    int b_off[CL_MAXL + 1];       // first own tile of layer l in `bias`

    __device__ ClEngine(const MadeDev &m_, const ClusterDev &cd_, const RunArgs &r_, ClShared &sh_, uint8_t *base, int R_)
        : m(m_), cd(cd_), r(r_), sh(sh_), ring(base), R(R_)
    {
        CS = cd.CS;
        rank = CS > 1 ? (int)cluster_rank() : 0;
        L = m.L;
        NP = cd.n_stages >> 1;
        warp = threadIdx.x >> 5;
        lane = threadIdx.x & 31;
        blk_bytes = (uint32_t)R * 128u;
        acts = ring + (size_t)(2 * NP) * STAGE;
        stag = acts + (size_t)cd.blocks * blk_bytes;
        nz = reinterpret_cast<float *>(stag + (size_t)(2 * cd.own_out) * blk_bytes);
        xs = reinterpret_cast<uint64_t *>(nz + (size_t)cd.own_out * R * TM);
        bias = reinterpret_cast<float *>(xs + (size_t)cd.own_out * TM);
        int at = 0;
#pragma unroll
        for (int l = 0; l <= CL_MAXL; ++l) {
            b_off[l] = at;
            if (l <= L) at += (cd.nt[l] + CS - 1) >> cd.cs_log2;
        }
    }
    // A CTA keeps the K blocks of a[l] that its own tiles of layer l read, cd.need of them, and behind those what it sends
    // of its tiles beyond (js_cluster_prepare: 39 blocks instead of 45 where 784 positions meet 1024 units x 2, which leaves
    // the weights a fourth load in flight; 112 samples with three, four and five: 71.5, 66.7 and 66.0 us).
    __device__ uint8_t *block(int l, int kb) const { return acts + (size_t)(cd.off[l][rank] + kb) * blk_bytes; }
    __device__ uint32_t block_in(int peer, int l, int kb) const { return peer_addr(smem_u32(acts) + (uint32_t)(cd.off[l][peer] + kb) * blk_bytes, peer); }
    __device__ uint64_t *block_bar(int l, int kb, unsigned pass) const { return l == 0 ? &sh.xbar[pass & 1][kb] : &sh.hbar[l - 1][kb]; }

    // Tiles are dealt largest K range first, back and forth over the CTAs, in opposite directions in neighbouring layers.
    __device__ int owner(int l, int tile) const
    {
        const int q = cd.nt[l] - 1 - tile, round = q >> cd.cs_log2, pos = q & (CS - 1);
        return ((round ^ l) & 1) ? CS - 1 - pos : pos;
    }
    // tiles of layer l that the window touches: degrees are monotone, so they are a range (one warp)
    __device__ int2 live_range(int l, const Win &w) const
    {
        int lo = INT_MAX, hi = 0;
        for (int t = lane; t < cd.nt[l]; t += 32) {
            const int dmin = cd.tiles.dmin[l][t], dmax = cd.tiles.dmax[l][t];
            const bool on = l == L ? dmax > w.olo && dmin <= w.ohi : dmax > w.hdeg_lo && dmin <= w.hdeg_hi;
            if (on) { lo = min(lo, t); hi = max(hi, t + 1); }
        }
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        return make_int2(min(lo, hi), hi);
    }
    static __device__ bool in(const int2 &range, int tile) { return tile >= range.x && tile < range.y; }
    // K blocks of a[l] that change before layer l reads them in this pass: x blocks sampled in the pass before, hidden tiles
    // of this pass
    __device__ int2 fresh(int l, unsigned pass) const
    {
        return l > 0 ? sh.rng[pass & 1][l - 1] : pass > 0 ? sh.rng[(pass + 1) & 1][L] : make_int2(0, 0);
    }

    // ---- bounded waits: they give up after spin_limit polls or 2 s, or when any CTA has given up
    __device__ bool give_up() const
    {
        *(volatile int *)&sh.dead = 1;
        atomicExch(&r.ctl->abort, 1);
        return false;
    }
    __device__ bool hopeless(unsigned i, uint64_t &t0) const
    {
        if (i >= r.spin_limit) return true;
        if ((i & 31u) != 31u) return false;
        if (*(volatile int *)&sh.dead || ld_volatile_i32(&r.ctl->abort) != 0) return true;
        if (t0 == 0) t0 = global_ns();
        return global_ns() - t0 > MBAR_WAIT_NS;
    }
    template <bool CLUSTER>
    static __device__ __forceinline__ bool try_wait(uint64_t *bar, uint32_t parity)
    {
        if constexpr (!CLUSTER) return mbar_try_wait(bar, parity);
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
        return ok != 0;
    }
    template <bool CLUSTER>
    __device__ __noinline__ bool wait_slow(uint64_t *bar, uint32_t parity) const
    {
        uint64_t t0 = 0;
        for (unsigned i = 0; !hopeless(i, t0); ++i)
            if (try_wait<CLUSTER>(bar, parity)) return true;
        return give_up();
    }
    template <bool CLUSTER = false>
    __device__ __forceinline__ bool wait(uint64_t *bar, uint32_t parity) const
    {
        if (try_wait<CLUSTER>(bar, parity)) return true;
        return wait_slow<CLUSTER>(bar, parity);
    }
    // May pass `pass` start?  In Jacobi mode every role sees for itself, in the masks of the pass before, whether there is another one
    // (told by the epilogue warps, behind their bookkeeping, it came 0.9 us later); else they are told, and learn the window.
    __device__ bool next_pass(unsigned pass, bool jacobi) const
    {
        if (pass == 0 || !jacobi) return wait(&sh.go, pass & 1) && !*(volatile int *)&sh.stop;
        if (!wait<true>(&sh.pbar[(pass - 1) & 1], (pass - 1) >> 1 & 1)) return false;
        uint32_t any = 0;
        for (int i = 0; i < CS; ++i) {
            const volatile uint4 &f = sh.flags[(pass - 1) & 1][i];
            any |= f.x | f.y;
        }
        const int cap = r.max_iters > 0 && r.max_iters < m.T ? r.max_iters : m.T;
        return any != 0 && (int)pass < cap && !*(volatile int *)&sh.dead;
    }
    // A stage of the weight ring is a pair of K blocks, an even one and the odd one behind it, brought by one load and freed by
    // both consumers.  (A load costs the loading thread 0.2 us, barrier and all, whatever its size: block by block, and with a
    // ring of its own for either consumer, the weights of a pass of 45 blocks took 11 us of the pass's 16.)  Each consumer waits
    // for every stage, also where the last pair of a tile lacks its block: so it cannot take a stage for full, or free one, in a
    // use of it other than its own (a parity does not tell a phase from the one after the next).

    // ---------------------------------------------------------------- roles
    // (one thread)
    __device__ bool room(uint64_t *bar, uint32_t parity, bool stoppable) const
    {
        uint64_t t0 = 0;
        for (unsigned i = 0;; ++i) {
            if (mbar_test_wait(bar, parity)) return true;
            if (stoppable && *(volatile int *)&sh.stop) return false;
            if (hopeless(i, t0)) return give_up();
        }
    }
    __device__ void producer(bool jacobi)
    {
        int n = 0, st = 0;
        uint32_t ph = 1;
        bool on = true;
        const uint32_t ring0 = smem_u32(ring);
        for (unsigned pass = 0; on; ++pass) {
            if (!jacobi && !next_pass(pass, false)) break;
            for (int l = 0; l <= L && on; ++l) {
                // in Jacobi mode every tile is computed in every pass: the stream needs no go-ahead
                const int2 rg = jacobi ? make_int2(0, cd.nt[l]) : sh.rng[pass & 1][l];
                const CUtensorMap *map = cd.tmW + 2 * l;
                const int npad = cd.npad[l], own = sh.nown[l];
                for (int j = 0; j < own && on; ++j) {
                    const int2 o = sh.own[l][j];
                    if (!in(rg, o.x)) continue;
                    for (int kb = 0; kb < o.y; kb += 2) {
                        if (!room(&sh.empty[st], ph, jacobi)) { on = false; break; }
                        const uint32_t to = ring0 + (uint32_t)st * (2 * STAGE);
                        if (kb + 1 < o.y) {
                            mbar_expect_tx(&sh.full[st], 2 * STAGE);
                            tma_load_3d(to, map + 1, &sh.full[st], 0, o.x * TM, kb);
                        } else {
                            mbar_expect_tx(&sh.full[st], STAGE);
                            tma_load_2d(to, map, &sh.full[st], 0, kb * npad + o.x * TM);
                        }
                        ++n;
                        if (++st == NP) { st = 0; ph ^= 1u; }
                    }
                }
            }
            if (!jacobi) mbar_arrive(&sh.ack);
        }
        sh.issued = n;
    }

    // bits lo .. hi - 1
    static __device__ uint64_t bits(const int2 &r)
    {
        return r.y <= r.x ? 0ull : (~0ull >> (64 - (r.y - r.x))) << r.x;
    }
    __device__ __noinline__ bool wait_both(uint64_t *a, uint32_t pa, uint64_t *b, uint32_t pb) const
    {
        return (mbar_test_wait(a, pa) || wait_slow<false>(a, pa)) && (mbar_test_wait(b, pb) || wait_slow<false>(b, pb));
    }
    // One thread; half 0 issues the even K blocks of every tile, half 1 the odd ones.  It looks for the next block's weights and
    // activations (150 cycles) before it issues this one's MMAs (96).
    __device__ void mma_issuer(int half, bool jacobi)
    {
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(R >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
        const uint64_t ring_desc = smem_desc_sw128(smem_u32(ring) + (uint32_t)(half * STAGE));
        const uint32_t blk = blk_bytes >> 4;
        int n = 0, loads = 0, slot = 0, st = 0;  // st, ph: the ring's next stage and the parity of its use
        uint32_t ph = 0, spar = 0;               // spar: parity of the accumulator slots' next use
        bool on = true;
        unsigned tiles = 0;
        for (unsigned pass = 0; on; ++pass) {
            if (!next_pass(pass, jacobi)) break;
#pragma unroll 1
            for (int l = 0; l <= L && on; ++l) {
                const int2 fr = fresh(l, pass), rg = sh.rng[pass & 1][l];
                uint64_t *const apar = &sh.apar[half][l == 0 && (pass & 1) ? CL_MAXL + 1 : l];       // parities of the K blocks' barriers; x: two sets
                const uint64_t ap = *apar, isfresh = bits(fr);
                const uint64_t act_desc = smem_desc_sw128(smem_u32(block(l, 0))) + (uint64_t)(half * blk);
                uint64_t *const bars = block_bar(l, half, pass);
#pragma unroll 1
                for (int j = 0; j < sh.nown[l]; ++j) {
                    const int2 o = sh.own[l][j];
                    if (!in(rg, o.x)) continue;
                    ++tiles;
                    const int mine = (o.y + 1 - half) >> 1, pairs = (o.y + 1) >> 1;
                    const uint32_t d = sh.tmem_base + (uint32_t)((2 * slot + half) * ACC);
                    uint64_t bd = act_desc, am = ap >> half, fm = isfresh >> half, *ab = bars;
                    auto look = [&](int i) {         // block i of this half
                        const bool w = mbar_test_wait(&sh.full[st], ph), a = mbar_test_wait(ab, (uint32_t)am & 1u);
                        return w & (a | (i >= mine) | !(fm & 1ull));
                    };
                    bool ready = look(0);
                    if (!wait(&sh.tempty[slot], (spar >> slot & 1u) ^ 1u)) { on = false; break; }
#pragma unroll 1
                    for (int i = 0; i < pairs; ++i) {
                        if (!ready) {
                            const bool need = i < mine && (fm & 1ull);
                            if (!wait_both(&sh.full[st], ph, need ? ab : &sh.full[st], need ? (uint32_t)am & 1u : ph)) { on = false; break; }
                        }
                        tc_fence_after();
                        const int cur = st;
                        const uint64_t ad = ring_desc + (uint64_t)(cur * (2 * STAGE >> 4)), b = bd;
                        if (++st == NP) { st = 0; ph ^= 1u; }
                        bd += 2 * blk;
                        am >>= 2;
                        fm >>= 2;
                        ab += 2;
                        ready = i + 1 < pairs && look(i + 1);
                        if (i < mine)
#pragma unroll
                            for (int k = 0; k < BK / 16; ++k)
                                umma_bf16(d, ad + (uint64_t)(2 * k), b + (uint64_t)(2 * k), idesc, (i > 0 || k > 0) ? 1u : 0u);
                        umma_commit(&sh.empty[cur]);
                    }
                    if (!on) break;
                    umma_commit(&sh.tfull[slot]);      // (with no K block of its own too: all its earlier MMAs are done)
                    n += mine;
                    loads += pairs;
                    spar ^= 1u << slot;
                    slot ^= 1;
                }
                *apar = ap ^ isfresh;
            }
            if (!jacobi) mbar_arrive(&sh.ack);
        }
        sh.consumed[half] = n;
        if (half == 0) { sh.tiles = tiles; sh.consumed_loads = loads; }
    }

    // Barrier keeper (one warp, lane = K block).  Every block another CTA sends completes its barrier once per pass in
    // which it is live: armed here with the bytes to come, and waited for before the pass may end, so that no copy is in
    // flight when its source or its barrier is used again.  (Bytes that arrive before the arming are counted all the same:
    // the phase cannot complete without it, and the phase before was waited for in the pass before.)
    __device__ void keeper(bool early, bool jacobi)
    {
        uint64_t apar[CL_MAXL + 2];
#pragma unroll
        for (int l = 0; l < CL_MAXL + 2; ++l) apar[l] = 0;
        bool on = true;
        auto arm = [&](int l, unsigned pass) {
            const int2 fr = fresh(l, pass);
            for (int kb = lane; kb < cd.nkb[l]; kb += 32)
                if (in(fr, kb) && kb < cd.need[l][rank] && (l == 0 || owner(l - 1, kb) != rank)) mbar_expect_tx(block_bar(l, kb, pass), blk_bytes);
        };
        auto drain = [&](int l, unsigned pass) {
            const int2 fr = fresh(l, pass);
            const int set = l == 0 ? (pass & 1 ? CL_MAXL + 1 : 0) : l;
            uint64_t ap = 0;
#pragma unroll
            for (int q = 0; q < CL_MAXL + 2; ++q) ap = q == set ? apar[q] : ap;
            for (int kb = lane; kb < cd.nkb[l]; kb += 32)
                if (in(fr, kb) && kb < cd.need[l][rank]) {
                    if (!wait(block_bar(l, kb, pass), (uint32_t)(ap >> kb) & 1u)) on = false;
                    ap ^= 1ull << kb;
                }
#pragma unroll
            for (int q = 0; q < CL_MAXL + 2; ++q) apar[q] = q == set ? ap : apar[q];
        };
        for (unsigned pass = 0;; ++pass) {
            if (!__all_sync(0xffffffffu, next_pass(pass, jacobi))) {
                if (*(volatile int *)&sh.dead) break;
                if (early) { arm(0, pass); drain(0, pass); }         // encodings sent ahead for a pass that is not run
                return;
            }
            if (lane == 0) mbar_expect_tx(&sh.pbar[pass & 1], (uint32_t)(16 * CS));
            for (int l = 0; l <= L; ++l) arm(l, pass);
            for (int l = 0; l <= L; ++l) drain(l, pass);
            on = __all_sync(0xffffffffu, on);
            if (!on) break;
            asm volatile("bar.arrive 2, 160;" ::: "memory");
        }
        asm volatile("bar.arrive 2, 160;" ::: "memory");      // an epilogue that waits for this warp must not be left alone
    }

    __device__ void ep_sync() const { asm volatile("bar.sync 1, 128;" ::: "memory"); }
    // the same, and did every thread say yes: a wait that gave up must take all of them out at the same place
    __device__ bool ep_all(bool ok) const
    {
        int all;
        asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbar.red.and.pred q, 1, 128, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
                     : "=r"(all) : "r"((int)ok) : "memory");
        return all != 0;
    }
    // Tile `tile` of layer l - 1 lies complete in this CTA's K block `place` of a[l]: to the others that read it.  Each epilogue warp serves
    // two CTAs (the copies of one warp leave one after the other, 60 cycles apart).
    __device__ void send(int l, int tile, int place)
    {
        const int peer = (warp & 3) * 2 + lane;
        if (lane < 2 && peer < CS && tile < cd.need[l][peer]) {
            if (peer == rank) mbar_arrive(&sh.hbar[l - 1][tile]);
            else copy_to_peer(block_in(peer, l, tile), smem_u32(block(l, place)), blk_bytes, peer_addr(smem_u32(&sh.hbar[l - 1][tile]), peer));
        }
    }
    // Encodings of output tile `tile` from their staging buffer to every CTA, this one included, for pass `next`.  (They
    // cannot be written in place: the copies of the pass before may still read them when a tile with a short K range is
    // sampled again.  A staging buffer is used again two passes later, and every CTA has seen its copies arrive before it
    // ended the pass in between.)
    __device__ void send_x(int tile, const uint8_t *src, unsigned next)
    {
        const int peer = (warp & 3) * 2 + lane;
        if (lane < 2 && peer < CS && tile < cd.need[0][peer])
            copy_to_peer(block_in(peer, 0, tile), smem_u32(src), blk_bytes,
                         peer_addr(smem_u32(&sh.xbar[next & 1][tile]), peer));
    }
    // byte offset of unit u (0..63) of sample s inside a K block
    __device__ static uint32_t at_block(int s, int u) { return (uint32_t)(s * 128 + ((((u >> 3) ^ (s & 7)) << 4) | ((u & 7) << 1))); }

    // The column loops of the epilogue, eight samples at a time, the next eight on their way out of tensor memory.  They are
    // kept rolled and free of branches: unrolled over a whole tile they missed the instruction cache (2.1 us a tile of 24
    // samples instead of 0.5).  tb: the even K blocks' accumulator, the odd ones' lies ACC columns on.
    __device__ __forceinline__ void load_sums(uint32_t tb, uint32_t (&a)[8], uint32_t (&b)[8], bool two)
    {
        tmem_ld8(tb, a);
        if (two) tmem_ld8(tb + ACC, b);
    }
    // bt: bias of the tile's units.  A value goes from the thread that has it to its sample's row by a transposing store, eight samples
    // of eight units at a time: lane = unit, with half the lanes idle and a 2-byte store per value, took 0.4 us longer.
    template <int ACT>
    __device__ __forceinline__ void hidden_columns(uint32_t dst, uint32_t tb, bool two, const float *bt, int q)
    {
        const float b0 = bt[q * 16 + (lane >> 2)], b1 = bt[q * 16 + (lane >> 2) + 8];
        uint32_t na[4], nb[4] = {0, 0, 0, 0};
        tmem_ld_16x8(tb, na);
        if (two) tmem_ld_16x8(tb + ACC, nb);
        uint32_t at = dst + (uint32_t)((lane & 7) * 128 + (((2 * q + (lane >> 3 & 1)) ^ (lane & 7)) << 4));
#pragma unroll 1
        for (int s0 = 0; s0 < R; s0 += 8, at += 1024) {
            float v[4];
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(na[i]) + __uint_as_float(nb[i]);
            if (s0 + 8 < R) {
                tmem_ld_16x8(tb + (uint32_t)(s0 + 8), na);
                if (two) tmem_ld_16x8(tb + ACC + (uint32_t)(s0 + 8), nb);
            }
            stmatrix2_trans(at, pack_bf16x2(tc_act_fn(ACT, v[0] + b0), tc_act_fn(ACT, v[1] + b0)), pack_bf16x2(tc_act_fn(ACT, v[2] + b1), tc_act_fn(ACT, v[3] + b1)));
        }
    }
    template <int NK>
    __device__ __forceinline__ uint64_t sample_columns(const float *nzt, uint32_t tb, bool two, float bv)
    {
        uint64_t x = 0;
        uint32_t na[8], nb[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        load_sums(tb, na, nb, two);
#pragma unroll 1
        for (int s0 = 0; s0 < R; s0 += 8) {
            float e[8], v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) e[i] = nzt[(s0 + i) * TM];
            uint32_t bits = 0;
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(na[i]) + __uint_as_float(nb[i]);
            load_sums(tb + (uint32_t)min(s0 + 8, R - 8), na, nb, two);
#pragma unroll
            for (int i = 0; i < 8; ++i) bits |= (uint32_t)js_sample_binary(NK, v[i] + bv, e[i]) << i;
            x |= (uint64_t)bits << s0;
        }
        tmem_wait_ld();
        return x;
    }

    __device__ int epilogue(bool jacobi, bool early, int nrow, int &status, int &passes)
    {
        const int q = warp & 3, tid = threadIdx.x - 64;
        const int u = q * 16 + (lane & 15);       // this thread's unit of a tile: the lower half of a warp's lanes
        const bool act_lane = lane < 16;
        const int T = m.T, B = jacobi ? T : r.block;
        const __nv_bfloat16 e0 = __float2bfloat16_rn(m.lut[0]), e1 = __float2bfloat16_rn(m.lut[1]), z0 = __float2bfloat16_rn(0.0f);
        const uint64_t rows = nrow >= 64 ? ~0ull : (1ull << nrow) - 1ull;
        uint64_t done = 0;
        int slot = 0;
        uint32_t spar = 0;
        int fin_x = 0, fin_h = 0, a = 0, lo = 0, k = 0;
        unsigned pass = 0;
        for (;; ++pass) {
            const int par = pass & 1;
            const int bend = min(a + B, T), len = bend - a;
            k += 1;
            // In Jacobi mode every tile is computed in every pass (skipping final ones would save work, which is not what
            // bounds a pass, and the weight stream could not run ahead); blocks take the window of made_driver.cuh.
            const Win w = jacobi ? make_win(0, T, 0, T)
                                 : r.frontier_skip ? make_win(fin_h, bend - 1, lo, bend) : make_win(0, T, a, bend);
#pragma unroll 1
            for (int l = 0; l <= L; ++l)
                for (int j = 0; j < sh.nown[l]; ++j) {
                    const int tile = sh.own[l][j].x;
                    if (!in(sh.rng[par][l], tile)) continue;
                    const bool two = sh.own[l][j].y > 1;
                    const float *bt = bias + (size_t)(b_off[l] + j) * TM;
                    const bool ok = __all_sync(0xffffffffu, wait(&sh.tfull[slot], spar >> slot & 1u));
                    tc_fence_after();
                    const uint32_t tb = sh.tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(2 * slot * ACC);
                    if (l < L) {
                        const uint32_t dst = smem_u32(block(l + 1, sh.place[l][j]));
                        if (m.act == JS_ACT_RELU) hidden_columns<JS_ACT_RELU>(dst, tb, two, bt, q);
                        else hidden_columns<JS_ACT_GELU_TANH>(dst, tb, two, bt, q);
                    } else {
                        const int p = tile * TM + u;
                        const float bv = bt[u];
                        const bool mine = act_lane && p >= w.plo && p < w.phi;
                        uint8_t *dst = stag + (size_t)(par * cd.own_out + j) * blk_bytes;
                        const float *nzt = nz + (size_t)j * R * TM + u;
                        const uint64_t xold = xs[j * TM + u];
                        const uint64_t xnew = r.nk == JS_NOISE_LOGISTIC ? sample_columns<JS_NOISE_LOGISTIC>(nzt, tb, two, bv)
                                                                        : sample_columns<JS_NOISE_UNIFORM_ICDF>(nzt, tb, two, bv);
                        const uint64_t diff = mine ? (xnew ^ xold) & rows : 0ull, x = xold ^ diff;
                        if (act_lane) {
                            if (diff) xs[j * TM + u] = x;
                            const __nv_bfloat16 c0 = p < T ? e0 : z0, c1 = p < T ? e1 : z0;
#pragma unroll 1
                            for (int s0 = 0; s0 < R; s0 += 8, dst += 1024) {
                                const uint32_t bits = (uint32_t)(x >> s0);
#pragma unroll
                                for (int i = 0; i < 8; ++i)
                                    *reinterpret_cast<__nv_bfloat16 *>(dst + at_block(i, u)) = (bits >> i & 1) ? c1 : c0;
                            }
                        }
                        const uint32_t clo = __reduce_or_sync(0xffffffffu, (uint32_t)diff);
                        const uint32_t chi = __reduce_or_sync(0xffffffffu, (uint32_t)(diff >> 32));
                        const int f = __reduce_min_sync(0xffffffffu, diff ? p : INT_MAX);
                        if (lane == 0 && (clo | chi)) {
                            atomicOr(&sh.chg[par][0], clo);
                            atomicOr(&sh.chg[par][1], chi);
                            atomicMin(&sh.first[par], f);
                        }
                    }
                    tc_fence_before();
                    fence_proxy_async_smem();
                    if (!ep_all(ok)) return -1;
                    if (tid == 0) mbar_arrive(&sh.tempty[slot]);
                    if (l < L) send(l + 1, tile, sh.place[l][j]);
                    spar ^= 1u << slot;
                    slot = (slot + 1) % NSLOT;
                }
            // Encodings may leave as soon as every CTA of the cluster has done its first layer (which reads them): known here
            // where this CTA's last output tile read hidden units of every CTA (`early`, see js_cluster_prepare), else when
            // the pass has ended everywhere.
            auto send_all_x = [&] {
                for (int j = 0; j < sh.nown[L]; ++j) {
                    const int tile = sh.own[L][j].x;
                    if (in(sh.rng[par][L], tile)) send_x(tile, stag + (size_t)(par * cd.own_out + j) * blk_bytes, pass + 1);
                }
            };
            if (early) send_all_x();
            // ---- end of the pass: masks to everybody, once this CTA's MMAs are done and all its copies have landed
            asm volatile("bar.sync 2, 160;" ::: "memory");
            // (data and signal in one: a store and a releasing arrival behind it took two trips between CTAs, 1.5 us)
            if (tid < CS)
                send16(peer_addr(smem_u32(&sh.flags[par][rank]), tid), make_uint4(sh.chg[par][0], sh.chg[par][1], (uint32_t)sh.first[par], 0u),
                       peer_addr(smem_u32(&sh.pbar[par]), tid));
            bool fine = wait<true>(&sh.pbar[par], pass >> 1 & 1);
            if (!jacobi && tid == 0) fine = wait(&sh.ack, pass & 1) && fine;
            if (!ep_all(fine && *(volatile int *)&sh.dead == 0)) return -1;
            uint32_t clo = 0, chi = 0;
            int mf = INT_MAX;
            if (lane < CS) {
                const uint4 f = sh.flags[par][lane];
                clo = f.x; chi = f.y; mf = (int)f.z;
            }
            clo = __reduce_or_sync(0xffffffffu, clo);
            chi = __reduce_or_sync(0xffffffffu, chi);
            mf = __reduce_min_sync(0xffffffffu, mf);
            const uint64_t chg = (uint64_t)chi << 32 | clo;
            const bool any = chg != 0;
            const int cap = (r.max_iters > 0 && r.max_iters < len) ? r.max_iters : len;
            const uint64_t stops = (k == cap ? rows : rows & ~chg) & ~done;
            for (int s = tid; s < 64; s += 128)
                if (stops >> s & 1) sh.count[s] = jacobi ? k : sh.count[s] + k;
            done |= stops;
            fin_h = max(fin_h, min(fin_x, jacobi ? T : bend - 1));
            lo = any ? max(lo + 1, min(mf + 1, bend)) : bend;
            fin_x = max(fin_x, lo);
            bool over = false;
            if (!(any && k < cap)) {
                if (any && cap < len) status = JS_NOT_CONVERGED;
                if (!jacobi) {
                    fin_x = bend;
                    done = 0;
                    a = bend;
                    lo = a;
                    k = 0;
                }
                over = jacobi || a >= T;
            }
            if (!over && !early) send_all_x();
            if (tid < 32) {
                if (!over && !jacobi) {
                    const int nb = min(a + B, T);
                    const Win nw = r.frontier_skip ? make_win(fin_h, nb - 1, lo, nb) : make_win(0, T, a, nb);
                    for (int l = 0; l <= L; ++l) {
                        const int2 rg = live_range(l, nw);
                        if (lane == 0) sh.rng[par ^ 1][l] = rg;
                    }
                }
                if (lane == 0) {
                    if (over) *(volatile int *)&sh.stop = 1;
                    sh.chg[par ^ 1][0] = sh.chg[par ^ 1][1] = 0;
                    sh.first[par ^ 1] = INT_MAX;
                    __threadfence_block();
                    if (!jacobi) mbar_arrive(&sh.go);
                }
            }
            if (over) break;
            ep_sync();
        }
        passes = (int)pass + 1;
        return fin_x;
    }
};

__global__ void __launch_bounds__(NTH, 1)
made_cluster_kernel(const __grid_constant__ MadeDev m, const __grid_constant__ ClusterDev cd, const __grid_constant__ RunArgs r, const int R)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ ClShared sh;
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    ClEngine e(m, cd, r, sh, base, R);
    const int tid = threadIdx.x, warp = e.warp, lane = e.lane, CS = e.CS, L = m.L, T = m.T;
    const int cluster = (int)(blockIdx.x >> cd.cs_log2), row0 = cluster * R, nrow = min(R, r.batch - row0);
    const bool jacobi = r.kmode == KM_JACOBI, early = jacobi && cd.early_ok != 0;

    // this CTA's tiles, per layer a warp; the first pass's ranges; barriers
    if (warp <= L) {
        const int l = warp;
        int n = 0, beyond = 0;
        const int need = l < L ? cd.need[l + 1][e.rank] : 0;
        for (int t0 = 0; t0 < cd.nt[l]; t0 += 32) {
            const int t = t0 + lane;
            const bool mine = t < cd.nt[l] && e.owner(l, t) == e.rank;
            const unsigned bal = __ballot_sync(0xffffffffu, mine);
            const unsigned far = __ballot_sync(0xffffffffu, mine && t >= need), before = (1u << lane) - 1u;
            if (mine) {
                const int j = n + __popc(bal & before);
                sh.own[l][j] = make_int2(t, cd.tiles.kbe[l][t]);
                if (l < L) sh.place[l][j] = (unsigned char)(t < need ? t : need + beyond + __popc(far & before));
            }
            n += __popc(bal);
            beyond += __popc(far);
        }
        const int bend = min(jacobi ? T : r.block, T);
        // (the whole of every layer in Jacobi mode)
        const int2 rg = jacobi ? make_int2(0, cd.nt[l]) : e.live_range(l, r.frontier_skip ? make_win(0, bend - 1, 0, bend) : make_win(0, T, 0, bend));
        if (lane == 0) { sh.nown[l] = n; sh.rng[0][l] = sh.rng[1][l] = rg; }
    }
    if (warp == 4 && lane == 0) {
        for (int s = 0; s < MAX_STAGES / 2; ++s) { mbar_init(&sh.full[s], 1); mbar_init(&sh.empty[s], 2); }
        for (int s = 0; s < NSLOT; ++s) { mbar_init(&sh.tfull[s], 2); mbar_init(&sh.tempty[s], 1); }
        mbar_init(&sh.pbar[0], 1);
        mbar_init(&sh.pbar[1], 1);
        mbar_init(&sh.go, 1);
        mbar_init(&sh.ack, 3);
        sh.stop = sh.dead = 0;
        for (int i = 0; i < 2 * (CL_MAXL + 2); ++i) (&sh.apar[0][0])[i] = 0;
        sh.issued = sh.consumed_loads = sh.consumed[0] = sh.consumed[1] = 0;
        sh.tiles = sh.sums[0] = sh.sums[1] = 0;
        for (int i = 0; i < 2; ++i) { sh.chg[i][0] = sh.chg[i][1] = 0; sh.first[i] = INT_MAX; }
    }
    for (int i = tid; i < 2 * CL_TILES; i += NTH) mbar_init(&(&sh.xbar[0][0])[i], 1);
    for (int i = tid; i < CL_MAXL * CL_TILES; i += NTH) mbar_init(&(&sh.hbar[0][0])[i], 1);
    for (int i = tid; i < 64; i += NTH) sh.count[i] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (warp == 5) tmem_alloc(&sh.tmem_base, NSLOT * 2 * ACC);
    __syncthreads();
    // noise of the own positions: asynchronous copies, waited for below
    for (int j = 0; j < sh.nown[L]; ++j) {
        const int tile = sh.own[L][j].x;
        for (int i = tid; i < R * TM; i += NTH) {
            const int s = i / TM, p = tile * TM + i % TM;
            const bool in = s < nrow && p < T;
            const float *src = r.noise + (in ? (size_t)(row0 + s) * T + p : 0);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(e.nz + (size_t)j * R * TM + i)), "l"(src), "r"(in ? 4 : 0)
                         : "memory");
        }
        for (int i = tid; i < TM; i += NTH) {
            uint64_t x = 0;
            const int p = tile * TM + i;
            if (r.init && p < T) {
#pragma unroll 8
                for (int s = 0; s < nrow; ++s) x |= (uint64_t)(r.init[(size_t)(row0 + s) * T + p] != 0) << s;
            }
            e.xs[j * TM + i] = x;
        }
    }
    // biases of the own tiles, likewise
    for (int l = 0; l <= L; ++l)
        for (int i = tid; i < sh.nown[l] * TM; i += NTH) {
            const int u = sh.own[l][i / TM].x * TM + i % TM;
            const bool in = u < m.n[l + 1];
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(e.bias + e.b_off[l] * TM + i)), "l"(m.bias[l] + (in ? u : 0)), "r"(in ? 4 : 0)
                         : "memory");
        }
    // In a window a tile may read K blocks that are not computed yet: zeros.
    if (!jacobi)
        for (int i = tid; i < cd.blocks * (int)(e.blk_bytes / 16); i += NTH) reinterpret_cast<uint4 *>(e.acts)[i] = make_uint4(0, 0, 0, 0);
    {
        // The iterate's encodings, eight positions (16 bytes) at a time.  From zeros the K blocks that lie inside the image are one value
        // throughout, whatever the order of their chunks (samples that are not there included: nothing is taken from their columns);
        // zeros behind the last position.
        const __nv_bfloat16 e0 = __float2bfloat16_rn(m.lut[0]), e1 = __float2bfloat16_rn(m.lut[1]), z0 = __float2bfloat16_rn(0.0f);
        const int need = cd.need[0][e.rank], whole = r.init ? 0 : min(need, T / TM);
        if (!jacobi) __syncthreads();
        const __nv_bfloat162 e2 = __halves2bfloat162(e0, e0);
        const uint32_t w = *reinterpret_cast<const uint32_t *>(&e2);
        for (int i = tid; i < whole * (int)(e.blk_bytes / 16); i += NTH) reinterpret_cast<uint4 *>(e.block(0, 0))[i] = make_uint4(w, w, w, w);
        const int c0 = whole * (TM / 8), chunks = need * (TM / 8);
        for (int s = warp; s < R; s += NTH / 32)
            for (int c = c0 + lane; c < chunks; c += 32) {
                const int p0 = c * 8;
                alignas(16) __nv_bfloat16 v[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const bool in = s < nrow && p0 + k < T, one = in && r.init && r.init[(size_t)(row0 + s) * T + p0 + k] != 0;
                    v[k] = in ? (one ? e1 : e0) : z0;
                }
                *reinterpret_cast<uint4 *>(e.block(0, p0 / TM) + ClEngine::at_block(s, p0 % TM)) = *reinterpret_cast<const uint4 *>(v);
            }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (CS > 1) cluster_sync();          // every CTA's barriers are initialised
    if (tid == 0) mbar_arrive(&sh.go);       // the first pass

    int status = JS_OK, passes = 0, fin = 0;
    if (warp == 0) {
        if (elect_one()) e.producer(jacobi);
    } else if (warp == 1 || warp == 7) {
        if (elect_one()) e.mma_issuer(warp == 7, jacobi);
    } else if (warp == 6) {
        e.keeper(early, jacobi);
    } else {
        fin = e.epilogue(jacobi, early, nrow, status, passes);
        if (fin < 0 && tid == 64) {          // a wait gave up: the other roles must not wait for a next pass
            *(volatile int *)&sh.stop = 1;
            __threadfence_block();
            mbar_arrive(&sh.go);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    const bool alive = sh.dead == 0 && ld_volatile_i32(&r.ctl->abort) == 0;
    if (tid == 0 && alive)                   // weights that ran ahead: let them land
        for (int n = sh.consumed_loads, q = cd.n_stages >> 1; n < sh.issued; ++n) e.wait(&sh.full[n % q], (uint32_t)(n / q) & 1u);
    // results: symbols of the own positions, counts
    if (warp >= 2 && warp < 6 && alive) {
        const int u = (warp & 3) * 16 + (lane & 15);
        for (int j = 0; j < sh.nown[L]; ++j) {
            const int p = sh.own[L][j].x * TM + u;
            if (p >= T) continue;
            const uint64_t x = e.xs[j * TM + u];
            for (int s = lane >> 4; s < nrow; s += 2) r.x[(size_t)(row0 + s) * T + p] = (uint8_t)(x >> s & 1);
        }
        if (e.rank == 0 && r.out_iters)
            for (int s = tid - 64; s < nrow; s += 128) r.out_iters[row0 + s] = sh.count[s];
    }
    if (tid == 0) {
        peer_add(peer_addr(smem_u32(&sh.sums[0]), 0), sh.tiles);
        peer_add(peer_addr(smem_u32(&sh.sums[1]), 0), (unsigned)(sh.consumed[0] + sh.consumed[1]));
    }
    if (!alive)
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);      // copies still in flight land before shared memory goes away
    __syncthreads();
    if (warp == 5) {
        tc_fence_after();
        tmem_dealloc(sh.tmem_base, NSLOT * 2 * ACC);
    }
    if (CS > 1) cluster_sync();
    if (warp == 2 && e.rank == 0) {
        int most = 0;
        for (int s = lane; s < nrow; s += 32) most = max(most, sh.count[s]);
        most = __reduce_max_sync(0xffffffffu, most);
        if (lane == 0)
            cluster_report(r.words, cluster, alive && ld_volatile_i32(&r.ctl->abort) == 0, status, passes, fin, sh.sums[0], most, sh.sums[1]);
    }
}

}  // namespace

// --------------------------------------------------------------- host side
static size_t cluster_smem(const ClusterDev &c, const MadeDev &v, int R, int n_stages)
{
    int own = 0;
    for (int l = 0; l <= v.L; ++l) own += (c.nt[l] + c.CS - 1) / c.CS;
    return 1024 + (size_t)n_stages * STAGE + (size_t)(c.blocks + 2 * c.own_out) * R * 128 + (size_t)c.own_out * (R * TM * 4 + TM * 8) + (size_t)own * TM * 4;
}

// which CTA of a cluster has a tile (ClEngine::owner)
static int cluster_owner(const ClusterDev &c, int l, int tile)
{
    const int q = c.nt[l] - 1 - tile, round = q >> c.cs_log2, pos = q & (c.CS - 1);
    return ((round ^ l) & 1) ? c.CS - 1 - pos : pos;
}

// Builds the view of a model for this kernel: 1 if it qualifies, 0 if not, negative on CUDA errors.  Needs the tile-major
// weights of js_tc_prepare.
int js_cluster_prepare(js_model *mo)
{
    const MadeDev &v = mo->made;
    ClusterDev &c = mo->cluster;
    mo->cluster_ok = 0;
    if (!mo->tc_ok || v.C != 1 || v.L > CL_MAXL) return 0;
    int most = 0;
    for (int l = 0; l <= v.L; ++l) {
        c.nt[l] = (v.n[l + 1] + TM - 1) / TM;
        c.nkb[l] = (v.n[l] + BK - 1) / BK;
        most = std::max(most, std::max(c.nt[l], c.nkb[l]));
    }
    if (most > CL_TILES) return 0;
    // two tiles per CTA and layer are a balanced pair (a short and a long K range)
    c.CS = most <= 2 ? 1 : most <= 4 ? 2 : most <= 8 ? 4 : 8;
    c.cs_log2 = c.CS == 1 ? 0 : c.CS == 2 ? 1 : c.CS == 4 ? 2 : 3;
    c.own_out = (c.nt[v.L] + c.CS - 1) / c.CS;
    std::vector<CUtensorMap> maps(2 * (v.L + 1));
    c.kblocks = 0;
    for (int l = 0; l <= v.L; ++l) {
        const std::vector<int> &din = mo->host_deg[l], &dout = mo->host_deg[l + 1];
        const int N = v.n[l + 1], K = v.n[l];
        for (int t = 0; t < c.nt[l]; ++t) {
            int lo = INT32_MAX, hi = 0;
            for (int u = t * TM; u < std::min(N, (t + 1) * TM); ++u) { lo = std::min(lo, dout[u]); hi = std::max(hi, dout[u]); }
            int ke = K;
            while (ke > 0 && !(l == v.L ? din[ke - 1] < hi : din[ke - 1] <= hi)) --ke;
            c.tiles.kbe[l][t] = (unsigned char)std::max(1, (ke + BK - 1) / BK);
            c.kblocks += c.tiles.kbe[l][t];
            c.tiles.dmin[l][t] = (short)lo;
            c.tiles.dmax[l][t] = (short)hi;
        }
        c.npad[l] = mo->tc.lay[l].npad;
        if (!js_encode_map_2d(&maps[2 * l], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, mo->tc_weights[l], c.nkb[l] * c.npad[l], BK, BK, TM)) return 0;
        const cuuint64_t dims[3] = {BK, (cuuint64_t)c.npad[l], (cuuint64_t)c.nkb[l]}, strides[2] = {BK * 2, (cuuint64_t)c.npad[l] * BK * 2};
        const cuuint32_t box[3] = {BK, TM, 2};
        if (!js_encode_map(&maps[2 * l + 1], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, mo->tc_weights[l], 3, dims, strides, box)) return 0;
    }
    c.kblocks = (c.kblocks + c.CS - 1) / c.CS;
    // K blocks of activations per CTA: those that its tiles read, then its own tiles beyond them
    c.blocks = 0;
    for (int i = 0; i < c.CS; ++i) {
        int at = 0;
        for (int l = 0; l <= v.L; ++l) {
            int need = 0, own = 0;
            for (int t = 0; t < c.nt[l]; ++t)
                if (cluster_owner(c, l, t) == i) need = std::max(need, (int)c.tiles.kbe[l][t]);
            for (int t = need; l > 0 && t < c.nt[l - 1]; ++t) own += cluster_owner(c, l - 1, t) == i;
            c.off[l][i] = (unsigned char)at;
            c.need[l][i] = (unsigned char)need;
            at += need + own;
        }
        c.blocks = std::max(c.blocks, at);
    }
    // Encodings may be sent before the pass has ended everywhere if each CTA's last output tile reads hidden units of every
    // CTA, in a layer above the first: a CTA issues its MMAs in order, so all of them have then done the first layer.
    c.early_ok = v.L >= 2 && c.nt[v.L] >= c.CS ? 1 : 0;
    for (int i = 0; i < c.CS && c.early_ok; ++i) {
        unsigned seen = 0;
        for (int kb = 0; kb < c.tiles.kbe[v.L][c.nt[v.L] - 1 - i]; ++kb) {
            seen |= 1u << cluster_owner(c, v.L - 1, kb);
        }
        if (seen != (1u << c.CS) - 1u) c.early_ok = 0;
    }
    void *p = nullptr;
    if (cudaMalloc(&p, maps.size() * sizeof(CUtensorMap)) != cudaSuccess) return JS_ERR_CUDA;
    mo->allocs.push_back(p);
    if (cudaMemcpy(p, maps.data(), maps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice) != cudaSuccess) return JS_ERR_CUDA;
    c.tmW = (const CUtensorMap *)p;
    if (cudaFuncSetAttribute(made_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)c.CS);
    cfg.blockDim = dim3(NTH);
    cfg.dynamicSmemBytes = SMEM_MAX;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)c.CS;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&c.max_clusters, made_cluster_kernel, &cfg) != cudaSuccess || c.max_clusters < 1) {
        cudaGetLastError();
        return 0;
    }
    mo->cluster_ok = 1;
    return 1;
}

// samples per cluster for a batch (a multiple of 8; 0: does not fit), and the ring stages left beside them
static int cluster_rows(const js_model *mo, int batch, int *n_stages)
{
    const ClusterDev &c = mo->cluster;
    const int want = std::min(64, ((batch + c.max_clusters - 1) / c.max_clusters + 7) / 8 * 8);
    for (int R = want; R >= 8; R -= 8)
        for (int st = MAX_STAGES; st >= 4; st -= 2)            // (they are used in pairs)
            if (cluster_smem(c, mo->made, R, st) <= SMEM_MAX) {
                *n_stages = st;
                return R;
            }
    return 0;
}

// Jacobi and GS-Jacobi calls whose samples go through in one round of clusters, or in two where a CTA's share of the weights is small and
// its ring long; the grid-wide kernel shares every weight tile among 128 samples and is the better one for more.
bool js_cluster_serves(const js_model *mo, const RunArgs &r)
{
    if (!mo->cluster_ok || (r.kmode != KM_JACOBI && r.kmode != KM_GS_JACOBI) || mo->opt_trace) return false;
    int st = 0;
    const int R = cluster_rows(mo, r.batch, &st);
    if (R == 0) return false;
    // A CTA streams its share of the weights every pass, whatever the batch.  One round, 16 and 100 samples, us here and grid-wide: T = 1600,
    // H = 2048 x 3 (241 K blocks) 151 and 177, 163 and 197; T = 1936 (264) 175 and 191, 190 and 218; T = 2500, H = 2500 x 3 (410), 8 samples 404 and 229.
    // Two rounds: 784, 1024 x 2, 512 samples (47 K blocks, 8 stages) 126 and 167; 1024, 1536 x 2, 480 (91, 10) 180 and 202; 1444, 1444 x 2,
    // 300 (104, 8) 198 and 272; but 1024, 2048 x 2, 250 (136, 6) 231 and 202; 1600, 1024, 512 (55, 6) 233 and 221; 1936, 1500 x 2, 250 (138, 4)
    // 340 and 196.
    // One round, but so many samples a cluster that the ring holds two loads (four stages): a pass waits for weights, and the grid-wide
    // kernel, which pays by the layer, is the better one from 45 K blocks a layer on, if it moves whole rows (widths of 16 positions).  Jacobi, 128
    // or 200 samples, here and there: 1296, 2048 x 2 (53 a layer) 264 and 232; 1024, 2240 x 2 (53) 215 and 193; 1936, 1500 x 2 (46) 261 and 237;
    // but 1296, 1024, 1600, 1750 (35) 165 and 185; 1936, 576, 2000 (36) 193 and 214; rows of any length: 1156, 2048 x 2 (50) 247 and 283; 1444,
    // 2240, 1650 (52) 254 and 277.  GS-Jacobi in four blocks gains with all of them (1296, 2048 x 2: 256 and 452).  Three loads: 1024, 2048 x 2 (45),
    // 128 and 200 samples 121 and 160, 171 and 200; 1936, 2304 (75) 254 and 262.
    const int clusters = (r.batch + R - 1) / R, rounds = (clusters + mo->cluster.max_clusters - 1) / mo->cluster.max_clusters;
    if (clusters > JS_MAX_CLUSTERS) return false;
    // (Buffers on any float boundary stay here: the grid-wide kernel does not take them, and the CUDA-core kernel is no match.)
    const bool aligned = (((uintptr_t)r.noise | (uintptr_t)r.x) & 15u) == 0;
    const bool starved = st < 6 && r.kmode == KM_JACOBI && mo->tc.bin_bulk && aligned;
    return rounds == 1 ? mo->cluster.kblocks <= (starved ? std::min(270, 45 * (mo->made.L + 1)) : 270) : rounds == 2 && mo->cluster.kblocks <= 104 && st >= 8;
}

int js_launch_made_cluster(const js_model *mo, const RunArgs &r, cudaStream_t stream, ClusterWork *work)
{
    ClusterDev c = mo->cluster;
    const int R = cluster_rows(mo, r.batch, &c.n_stages);
    *work = ClusterWork{(r.batch + R - 1) / R, 0, 2LL * TM * BK * R, STAGE};
    for (int l = 0; l <= mo->made.L; ++l) work->tiles += c.nt[l];
    memset(mo->h_words, 0, 2 * sizeof(unsigned long long) * (size_t)work->clusters);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(work->clusters * c.CS));
    cfg.blockDim = dim3(NTH);
    cfg.dynamicSmemBytes = cluster_smem(c, mo->made, R, c.n_stages);
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)c.CS;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return (int)cudaLaunchKernelEx(&cfg, made_cluster_kernel, mo->made, c, r, R);
}
