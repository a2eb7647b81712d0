// Masked-convolution sampler (PixelCNN-style stack) on the sm_100a tensor cores.
//
// Every masked 3x3 convolution is an implicit GEMM: M = 128 consecutive pixels of one
// image (whole rows), N = output channels, K = live taps x input channels.  Only the
// five taps the causal mask keeps are visited (row above: left, centre, right; same
// row: left, centre); the centre tap's colour-group mask is already folded into the
// packed weights.  The A operand of tap (ky, kx) is the activation tensor shifted by
// (ky-1, kx-1): a 4-D TMA box {64 channels, width, rows, 1 image} whose start
// coordinate may lie outside the image, where TMA fills zeros - that is the zero
// padding.  The 1x1 head is a plain GEMM with one 256-class sub-pixel per N tile, and
// its epilogue is the sampling step (Gumbel-max against the fixed noise, compare,
// re-encode), as in the masked-MLP kernel.  Solver loops: made_driver.cuh.
//
// What bounds it: 16 images of 32 x 32 through eight layers of 128 channels (one tile per SM) take 6.7 us per layer (8.6 with a grid
// barrier behind each): 1.7 us from a tile's stamps to its first pixels, 2.8 us of K loop (272 KB per tile at the 108 GB/s that an
// SM takes in), 2.2 us of epilogue, half of which is the fence in front of the stamp.  A head tile takes 2.3 to 3.5 us (7 with
// the noise read by the threads).  A call of 13 passes: 891 us, 1290 before.
#include <cuda.h>

#include <cstring>
#include <vector>

#include "js_common.cuh"
#include "js_model.h"
#include "made_driver.cuh"
#include "tc_common.cuh"

namespace {

constexpr int BM = TC_BM, BK = TC_BK;
// warp 0 loads pixels, warp 1 MMA, warps 2-9 epilogue: two per tensor-memory lane quadrant, warp 10 loads weights, 11 the head's noise
constexpr int NTH = 384;
constexpr int ACC_COLS = 256;
constexpr int A_BYTES = BM * BK * 2;
// Two rings, each with a loading warp of its own: weights, which wait for nothing but room and so are there before the layer
// in front has finished, and pixels.  A load takes about 1 us, the MMAs of a K block 0.14: with one ring of 4 stages for both,
// filled when the pixels were there, the ten K blocks of a tile took 2.9 us.
constexpr int W_RING = 80 * 1024;                     // 64 weight rows: 8 KB, 10 stages; 128: 5 stages; the head's 256: 2 stages
constexpr int A_RING = 120 * 1024;                    // pixels of 64 channels: 128 of them, or with the image row above them
constexpr int MAX_STAGES = 10;
constexpr int STAGING_BYTES = 16 * 1024;              // 2 KB per epilogue warp
constexpr int HEAD_STAGES = 2;                        // a tile of the head is one or two K blocks: pixel stages that leave room for the noise
constexpr int NOISE_BUFS = 3;                         // per half of the classes: boxes of 128 pixels x 32 classes
constexpr int NOISE_BOX = 128 * 32 * 4;
constexpr int NOISE_AT = W_RING + HEAD_STAGES * A_BYTES;      // over the rest of the layers' pixel ring and the staging rows
constexpr int SMEM_BYTES = W_RING + A_RING + STAGING_BYTES + 1024;
static_assert(NOISE_AT + 2 * NOISE_BUFS * NOISE_BOX <= SMEM_BYTES - 1024 && NOISE_AT % 1024 == 0, "room for the noise");
constexpr int MAX_IMAGES = 256;

enum { EPI_HIDDEN = 0, EPI_LOGITS = 1, EPI_CAT = 3 };
// which activations a layer reads and writes.  SRC_NEW: the working set.  SRC_OLD: the set of the previous
// outer iterate (Jacobi-GS).  SRC_MIXED: the row above from the previous outer iterate, the own row from
// the working set - the view a one-row block has in Algorithm 2.
enum { SRC_NEW = 0, SRC_OLD = 1, SRC_MIXED = 2 };

struct ConvShared {
    uint64_t wfull[MAX_STAGES], wempty[MAX_STAGES], afull[MAX_STAGES], aempty[MAX_STAGES], tfull[2], tempty[2], nfull[2][NOISE_BUFS], nempty[2][NOISE_BUFS];
    uint32_t tmem_base;
    alignas(16) float bias_s[8][128];     // of the channels or classes of an epilogue warp
    float xbest[2][4][32];    // head: the upper class half's best score and class, by tile parity and quadrant
    int xbi[2][4][32];
    float lut_s[256];         // input encoding table
    int img[2][MAX_IMAGES];   // images still iterating, by engine's icur: this pass's and, while it is being looked at, the next one's
    int n_img[2];
};

struct ConvEngine {
    static constexpr bool has_jgs = true;
    const ConvDev &m;
    const RunArgs &r;
    const CUtensorMap &tm_noise;
    ConvShared &sh;
    uint8_t *ring, *staging;
    unsigned epoch = 0;
    unsigned long long issued = 0, skipped = 0, mma_flops = 0, weight_bytes = 0;
    int warp, lane;
    // the rings: stage in turn, bit s = parity of the next use of stage s, present cut
    int wst = 0, ast = 0;
    uint32_t wpar = 0, apar = 0;
    int w_stages = 1, w_bytes = 0, a_stages = 1, a_bytes = 0;
    int acc = 0;
    uint32_t aphase = 0;
    bool dead = false;
    uint32_t tmem_base = 0;

    // Order of the layers of a pass.  A tile of a conv layer needs its own pixels and those of the tile above from the layer
    // before it, so the layers of a pass are not separated by grid barriers: every tile carries a stamp, the number of the
    // last layer that wrote it, and the loading warp waits for the two stamps (a layer of one tile per SM: 8.6 us with a
    // barrier behind it, of which 3 us were the barrier and the way back to the first load).
    int layer_no = 0;              // layers done by this launch, the current one included (the same in every CTA)
    int conv_lo = 0, conv_hi = 0;  // row tiles that the conv layers of this pass recompute
    // head: next noise buffer (loaded or read by this warp), bit b = parity of buffer b's next use
    int nz_buf = 0;
    uint32_t nz_par = 0;

    __device__ ConvEngine(const ConvDev &m_, const RunArgs &r_, const CUtensorMap &tm_noise_, ConvShared &sh_, uint8_t *ring_)
        : m(m_), r(r_), tm_noise(tm_noise_), sh(sh_), ring(ring_), staging(ring_ + W_RING + A_RING)
    {
        warp = threadIdx.x >> 5;
        lane = threadIdx.x & 31;
    }

    // optional device timeline (JS_OPT_TRACE, js_get_trace): first and last (or chosen) CTA, one row of stamps per
    // layer: 0 epilogue warps start, 1 first operands have landed, 2 last MMA issued, 3 last accumulator
    // complete, 4 epilogues done, 5 grid barrier passed (all layers but a pass's last: the CTA is through with the layer)
    int phase_no = 0;
    int icur = 0;                  // which list of images is this pass's
    int raised_img = -1, raised_phase = -1;      // last (image, phase) this warp reported a change for
    __device__ void trace(int slot) const
    {
        if (r.trace == nullptr || phase_no >= JS_TRACE_PHASES) return;
        const int who = js_trace_who(r);
        if (who < 0) return;
        r.trace[((size_t)who * JS_TRACE_PHASES + phase_no) * JS_TRACE_SLOTS + slot] = global_ns();
    }

    __device__ bool barrier()
    {
        // One proxy fence, on the side of the TMA loads that read what threads stored before the barrier.  (One in front too made
        // every thread wait for its stores a second time.)
        const bool ok = grid_barrier(r.ctl, epoch, r.spin_limit);
        fence_proxy_async();
        if (threadIdx.x == 0) trace(5);
        return ok;
    }

    __device__ void init(const uint8_t *src)
    {
        const size_t n = (size_t)r.batch * m.T;
        __nv_bfloat16 *a0 = (__nv_bfloat16 *)m.act[0];
        for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
            const uint8_t v = src ? src[i] : (uint8_t)0;
            if (r.x) r.x[i] = v;
            const size_t pix = i / m.in_ch;                 // global pixel index (image-major)
            a0[pix * 64 + (i % m.in_ch)] = __float2bfloat16_rn(m.lut[v]);
        }
        if (blockIdx.x == 0) {
            clear_flags(r);
            for (int i = threadIdx.x; i < 2 * r.batch; i += blockDim.x) r.smp_state[i] = 0;
            for (int i = threadIdx.x; i < r.batch * m.nyt * 8; i += blockDim.x) m.stamp[i] = 0;
        }
        for (int i = threadIdx.x; i < r.batch; i += blockDim.x) sh.img[icur][i] = i;
        if (threadIdx.x == 0) sh.n_img[icur] = r.batch;
        __syncthreads();
    }

    // Images whose iterate did not change are at their fixed point: they drop out of the
    // tile lists.  Every CTA derives the same list from the per-sample flags; rows do not
    // move, so nothing has to be rebuilt.  The list is made by one warp while another one asks what changed at all (the two
    // round trips to L2 and a block barrier one after the other cost 1 us per pass): the flags of all images in flight at
    // once, then a ballot per 32 images.
    __device__ void look_ahead(int fslot)
    {
        if (warp != 1) return;
        const int n = sh.n_img[icur];
        int img[MAX_IMAGES / 32];
        bool keep[MAX_IMAGES / 32];
#pragma unroll
        for (int i = 0; i < MAX_IMAGES / 32; ++i) {
            const bool in = 32 * i + lane < n;
            img[i] = in ? sh.img[icur][32 * i + lane] : 0;
            keep[i] = in && ld_volatile_i32(&r.smp_changed[fslot * r.batch + img[i]]) != 0;
        }
        int k = 0;
#pragma unroll
        for (int i = 0; i < MAX_IMAGES / 32; ++i) {
            const unsigned bal = __ballot_sync(0xffffffffu, keep[i]);
            if (keep[i]) sh.img[icur ^ 1][k + __popc(bal & ((1u << lane) - 1u))] = img[i];
            k += __popc(bal);
        }
        if (lane == 0) sh.n_img[icur ^ 1] = k;
    }
    // takes the list that look_ahead has made; always returns 0 (no remapping)
    __device__ int compact(int)
    {
        icur ^= 1;
        if (blockIdx.x == 0 && threadIdx.x == 0) { r.ctl->compactions += 1; r.ctl->live = sh.n_img[icur]; }
        return 0;
    }

    // The rings are cut anew for the head and behind it (the parity of a stage's barriers is kept per stage).  At the start of a
    // pass the grid barrier has drained them; a loading warp that goes over to the head waits until its ring is.
    __device__ void cut_rings(bool head)
    {
        const int bytes = (head ? 256 : m.ch) * BK * 2;
        if (bytes != w_bytes) {
            w_bytes = bytes;
            w_stages = min(MAX_STAGES, W_RING / bytes);
            wst = 0;
        }
        const int as = head ? HEAD_STAGES : min(MAX_STAGES, A_RING / m.stage_a);
        if (as != a_stages) {
            a_stages = as;
            a_bytes = head ? A_BYTES : m.stage_a;
            ast = 0;
        }
    }
    __device__ bool drained(uint64_t *empty, int n, uint32_t par)
    {
        for (int s = 0; s < n; ++s)
            if (!__all_sync(0xffffffffu, mbar_wait(&empty[s], ((par >> s) & 1u) ^ 1u, r.ctl))) return false;
        return true;
    }
    __device__ uint8_t *stage_w(int s) const { return ring + (size_t)s * w_bytes; }
    __device__ uint8_t *stage_a(int s) const { return ring + W_RING + (size_t)s * a_bytes; }
    __device__ void advance_w()
    {
        wpar ^= 1u << wst;
        if (++wst == w_stages) wst = 0;
    }
    __device__ void advance_a()
    {
        apar ^= 1u << ast;
        if (++ast == a_stages) ast = 0;
    }

    // Whole warp: waits until tiles ya and yb of image n carry stamp `want` or a later one (an index outside the tiles
    // that this pass recomputes: nothing to wait for).  Eight stamps per tile, one per warp that writes it.
    __device__ bool wait_stamps(int n, int ya, int yb, int want)
    {
        const int y = lane < 8 ? ya : yb;
        const bool look = lane < 16 && y >= conv_lo && y < conv_hi;
        const int *st = m.stamp + 8 * (size_t)(n * m.nyt + (look ? y : 0)) + (lane & 7);
        uint64_t t0 = 0;
        for (unsigned i = 1;; ++i) {
            if (__all_sync(0xffffffffu, !look || (int)ld_acquire_u32(reinterpret_cast<const unsigned *>(st)) >= want)) break;
            if ((i & 31u) == 0u) {
                if (t0 == 0) t0 = global_ns();
                if (__any_sync(0xffffffffu, ld_volatile_i32(&r.ctl->abort) != 0 || global_ns() - t0 > MBAR_WAIT_NS)) {
                    if (lane == 0) atomicExch(&r.ctl->abort, 1);
                    return false;
                }
            }
        }
        __syncwarp();             // the polls were acquires
        fence_proxy_async();
        return true;
    }
    __device__ void advance_acc()
    {
        acc ^= 1;
        if (acc == 0) aphase ^= 1u;
    }

    // row tiles (of every image) that the window touches.  A hidden unit of colour group g at
    // pixel p reads positions < 3p + g ("degree"); position t = 3p + c.
    __device__ void live_rows(bool head, const Win &w, int &yt_lo, int &yt_hi) const
    {
        const int lo_key = head ? w.olo : w.hdeg_lo + 1;      // live iff largest degree/position >= lo_key
        const int hi_key = head ? w.ohi - 1 : w.hdeg_hi;      // live iff smallest degree/position <= hi_key
        yt_lo = m.nyt;
        yt_hi = 0;
        for (int yt = 0; yt < m.nyt; ++yt) {
            const int p0 = yt * m.R * m.width;
            const int p1 = min(m.height, (yt + 1) * m.R) * m.width - 1;
            const int dmin = p0 * m.in_ch, dmax = p1 * m.in_ch + m.in_ch - 1;
            if (dmax >= lo_key && dmin <= hi_key) { yt_lo = min(yt_lo, yt); yt_hi = max(yt_hi, yt + 1); }
        }
        if (yt_hi < yt_lo) yt_lo = yt_hi = 0;
    }

    // tile id -> (image, row tile, sub-pixel); `per` = 1 for conv layers, in_ch for the head
    __device__ void locate(int id, int nyl, int yt_lo, int per, int &n, int &yt, int &c) const
    {
        c = id % per;
        const int t2 = id / per;
        yt = yt_lo + t2 % nyl;
        n = sh.img[icur][t2 / nyl];
    }

    __device__ int kblocks(int l) const
    {
        return l < m.n_conv ? 5 * (m.cin_pad[l] / BK) : m.ch / BK;
    }

    __device__ void load_weights(int l, int ntiles)
    {
        const bool head = (l == m.n_conv);
        const int per = head ? m.in_ch : 1, kcs = head ? m.ch / BK : m.cin_pad[l] / BK, kcs_log2 = kcs == 2 ? 1 : 0;
        const int nkb = kblocks(l);
        const CUtensorMap *mw = m.tmW + l;
        if (head && w_bytes != 0 && !drained(sh.wempty, w_stages, wpar)) { dead = true; return; }
        cut_rings(head);
        for (int id = blockIdx.x; id < ntiles; id += gridDim.x) {
            const int c = id % per;
            for (int kb = 0; kb < nkb;) {
                const int run = mbar_wait_run(sh.wempty, wst, w_stages, ~wpar, nkb - kb, r.ctl);
                if (run == 0) { dead = true; return; }
                for (int i = 0; i < run; ++i, ++kb) {
                    if (elect_one()) {
                        mbar_expect_tx(&sh.wfull[wst], (uint32_t)w_bytes);
                        tma_load_2d(smem_u32(stage_w(wst)), mw, &sh.wfull[wst], (kb & (kcs - 1)) * BK, head ? c * 256 : (kb >> kcs_log2) * m.ch);
                    }
                    advance_w();
                }
            }
        }
    }

    // Pixel loads of a tile: a box per K block, or, where the ring holds them all (m.share), a box per horizontal shift and 64
    // channels that has the image row above the tile too, and serves the taps of both rows.  (Not for a one-row block, which
    // takes the two rows from different sets.)
    __device__ bool shares(bool head, int src) const { return !head && m.share && src != SRC_MIXED; }
    __device__ void load_pixels(int l, int yt_lo, int nyl, int ntiles, int src)
    {
        const bool head = (l == m.n_conv), share = shares(head, src);
        const int per = head ? m.in_ch : 1, kcs = head ? m.ch / BK : m.cin_pad[l] / BK, kcs_log2 = kcs == 2 ? 1 : 0;       // 64 or 128 channels
        const int n_loads = share ? 3 * kcs : kblocks(l);
        const CUtensorMap *ma_new = m.tmAct + l, *ma_old = m.tmActOld + l, *ma_two = (src == SRC_OLD ? m.tmActOld2 : m.tmAct2) + l;
        if (head && w_bytes != 0 && !drained(sh.aempty, a_stages, apar)) { dead = true; return; }
        cut_rings(head);
        for (int id = blockIdx.x; id < ntiles; id += gridDim.x) {
            int n, yt, c;
            locate(id, nyl, yt_lo, per, n, yt, c);
            const int y0 = yt * m.R;
            // The head writes the image, which the tile below reads in the first layer: it waits for that tile too.
            if (l > 0 && !wait_stamps(n, yt, head ? yt + 1 : yt - 1, layer_no - 1)) { dead = true; return; }
            for (int k = 0; k < n_loads;) {
                const int run = mbar_wait_run(sh.aempty, ast, a_stages, ~apar, n_loads - k, r.ctl);
                if (run == 0) { dead = true; return; }
                for (int i = 0; i < run; ++i, ++k) {
                    const int tap = k >> kcs_log2, kc = k & (kcs - 1);
                    // taps in the order of the packed weights: the three of the row above, then left and centre
                    const int dy = head || tap >= 3 ? 0 : -1, dx = head ? 0 : tap >= 3 ? tap - 4 : tap - 1;
                    const bool two = share && tap < 2;
                    const CUtensorMap *ma = two ? ma_two : (src == SRC_OLD || (src == SRC_MIXED && dy < 0)) ? ma_old : ma_new;
                    if (elect_one()) {
                        mbar_expect_tx(&sh.afull[ast], two ? A_BYTES + m.width * BK * 2 : A_BYTES);
                        tma_load_4d(smem_u32(stage_a(ast)), ma, &sh.afull[ast], kc * BK, dx, y0 + dy, n);
                    }
                    advance_a();
                }
            }
        }
    }

    // One thread of the warp issues everything (the ring and accumulator state of this role lives in it).  It asks for the next
    // K block's barriers before it issues the MMAs of this one: a look at a barrier takes 150 cycles, the MMAs of a K block 256,
    // and with look and issue one after the other a K block took 600.
    __device__ void mma_issuer(int l, int src, int ntiles)
    {
        cut_rings(l == m.n_conv);
        __syncwarp();
        if (elect_one()) mma_tiles(l, src, ntiles);
        __syncwarp();
        if (lane == 0) trace(2);
    }
    __device__ void mma_tiles(int l, int src, int ntiles)
    {
        const bool head = (l == m.n_conv), share = shares(head, src);
        const uint32_t idesc = instr_desc_bf16(head ? 256 : m.ch);
        const int nkb = kblocks(l), kcs = head ? m.ch / BK : m.cin_pad[l] / BK;
        const int n_loads = share ? 3 * kcs : nkb;
        const uint32_t row = (uint32_t)m.width * BK * 2;             // one image row of a stage
        bool first = true;
        for (int id = blockIdx.x; id < ntiles && !dead; id += gridDim.x) {
            if (!mbar_wait(&sh.tempty[acc], aphase ^ 1u, r.ctl)) { dead = true; break; }
            const uint32_t d_tmem = tmem_base + (uint32_t)(acc * ACC_COLS);
            const int a0 = ast;
            bool w_ok = false, a_ok = false;
            for (int kb = 0; kb < nkb; ++kb) {
                const bool again = kb >= n_loads;
                if (!w_ok && !mbar_wait(&sh.wfull[wst], (wpar >> wst) & 1u, r.ctl)) { dead = true; break; }
                if (!again && !a_ok && !mbar_wait(&sh.afull[ast], (apar >> ast) & 1u, r.ctl)) { dead = true; break; }
                tc_fence_after();
                if (first) trace(1);
                first = false;
                // taps 3 and 4 (left, centre) of a shared load are one image row further down in the stages of taps 0 and 1
                int a_now = again ? a0 + kb - n_loads : ast;
                if (a_now >= a_stages) a_now -= a_stages;
                const int w_now = wst;
                const uint64_t adesc = smem_desc_sw128(smem_u32(stage_a(a_now)) + (again ? row : 0u));
                const uint64_t bdesc = smem_desc_sw128(smem_u32(stage_w(w_now)));
                advance_w();
                if (!again) advance_a();
                if (kb + 1 < nkb) {
                    w_ok = mbar_test_wait(&sh.wfull[wst], (wpar >> wst) & 1u);
                    a_ok = kb + 1 >= n_loads || mbar_test_wait(&sh.afull[ast], (apar >> ast) & 1u);
                }
#pragma unroll
                for (int k = 0; k < BK / 16; ++k)
                    umma_bf16(d_tmem, adesc + (uint64_t)(2 * k), bdesc + (uint64_t)(2 * k), idesc, (kb > 0 || k > 0) ? 1u : 0u);
                if (!share || kb >= 2 * kcs) umma_commit(&sh.aempty[a_now]);
                umma_commit(&sh.wempty[w_now]);
            }
            if (dead) break;
            umma_commit(&sh.tfull[acc]);
            advance_acc();
        }
    }

    __device__ void release_acc()
    {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.tempty[acc]);
    }

    // conv layer: ReLU(acc + bias) -> bf16, through the staging buffer so that the NHWC stores are coalesced.  A warp takes half
    // the channels (64 or 32) of its quadrant's 32 pixels, 32 at a time: rows of 64 bytes, 16-byte chunks permuted by the row.
    __device__ void epi_hidden_tile(int n, int y0, uint32_t tbase, int half, __nv_bfloat16 *out)
    {
        const uint32_t stg = smem_u32(staging) + 2048u * (uint32_t)(warp - 2), bs = smem_u32(sh.bias_s[warp - 2]);
        const int bn = m.ch, mine = bn / 2, q = warp & 3;
        const int rows_valid = (min(m.height, y0 + m.R) - y0) * m.width;            // pixels of the tile inside the image
        // readback: four lanes per pixel, eight pixels at once
        const int ch = lane & 3, r0 = lane >> 2;
        __nv_bfloat16 *dst = out + ((size_t)n * m.height * m.width + (size_t)y0 * m.width + q * 32 + r0) * bn + half * mine + ch * 8;
#pragma unroll 1
        for (int c0 = 0; c0 < mine; c0 += 32) {
            float v[32];
            tmem_ld32(tbase + (uint32_t)(half * mine + c0), v);
            if (c0 + 32 == mine) release_acc();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint32_t pk[4];
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int j = 8 * i + 4 * k;
                    float4 b;
                    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w) : "r"(bs + 4u * (uint32_t)(c0 + j)));
                    pk[2 * k] = pack_bf16x2(fmaxf(v[j] + b.x, 0.0f), fmaxf(v[j + 1] + b.y, 0.0f));
                    pk[2 * k + 1] = pack_bf16x2(fmaxf(v[j + 2] + b.z, 0.0f), fmaxf(v[j + 3] + b.w, 0.0f));
                }
                asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(stg + 64u * (uint32_t)lane + 16u * (uint32_t)(i ^ ((lane >> 1) & 3))),
                             "r"(pk[0]), "r"(pk[1]), "r"(pk[2]), "r"(pk[3]) : "memory");
            }
            __syncwarp();
#pragma unroll
            for (int it = 0; it < 4; ++it) {
                const int rl = 8 * it + r0;
                uint32_t x, y, z, w;
                asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(x), "=r"(y), "=r"(z), "=r"(w)
                             : "r"(stg + 64u * (uint32_t)rl + 16u * (uint32_t)(ch ^ ((rl >> 1) & 3))));
                if (q * 32 + rl < rows_valid) *reinterpret_cast<uint4 *>(dst + (size_t)(8 * it) * bn + c0) = make_uint4(x, y, z, w);
            }
            __syncwarp();
        }
        // (The reader's proxy fence, behind its look at the stamp, orders these stores before its TMA loads.)
        if (lane == 0) {
            __threadfence();
            *reinterpret_cast<volatile int *>(m.stamp + 8 * (size_t)(n * m.nyt + y0 / m.R) + warp - 2) = layer_no;
        }
    }

    static __device__ __forceinline__ float4 lds_f4(uint32_t a)
    {
        float4 v;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
        return v;
    }

    // ---- head: the noise of a tile goes through shared memory, from a warp of its own, in boxes of 128 pixels x 32 classes.
    // (Read by the threads, a lane per pixel, every 16-byte load of a warp touched 32 lines: 7 us per tile, a quarter of a whole
    // pass.  Asked for by the epilogue warps themselves, a box cost them 0.23 us each, of 0.9 per 32 classes.)
    __device__ uint8_t *noise_buf(int half, int b) const { return ring + NOISE_AT + (size_t)(half * NOISE_BUFS + b) * NOISE_BOX; }
    // Head, epilogue warps and the one that loads the noise: every warp is through with its staging rows and has seen this CTA's
    // last accumulator, so the layers' pixel ring is drained too.
    __device__ void noise_may_come()
    {
        asm volatile("bar.sync 5, 288;" ::: "memory");
        fence_proxy_async();
    }
    __device__ void load_noise(int yt_lo, int nyl, int ntiles)
    {
        for (int id = blockIdx.x; id < ntiles; id += gridDim.x) {
            int n, yt, c;
            locate(id, nyl, yt_lo, m.in_ch, n, yt, c);
            const int pix = (n * m.height + yt * m.R) * m.width;
            for (int k = 0; k < 4; ++k) {
                for (int half = 0; half < 2; ++half) {
                    if (!__all_sync(0xffffffffu, mbar_wait(&sh.nempty[half][nz_buf], ((nz_par >> nz_buf) & 1u) ^ 1u, r.ctl))) { dead = true; return; }
                    if (elect_one()) {
                        uint64_t *bar = &sh.nfull[half][nz_buf];
                        mbar_expect_tx(bar, NOISE_BOX);
                        tma_load_3d(smem_u32(noise_buf(half, nz_buf)), &tm_noise, bar, half * 128 + k * 32, c, pix);
                    }
                    __syncwarp();
                }
                nz_par ^= 1u << nz_buf;
                if (++nz_buf == NOISE_BUFS) nz_buf = 0;
            }
        }
    }

    // Inverse CDF of the softmax from one uniform number u: the first class c with u * S < sum_{i<=c} e_i,
    // e_i = exp(z_i - max z).  Three readings of the thread's 256 logits out of tensor memory: the maximum,
    // the running sums (kept at the chunk ends), the class inside the chunk found.  Kept out of line: it
    // must not cost the Gumbel path registers.
    __device__ __noinline__ int head_icdf(uint32_t tbase, const float *bias, float u)
    {
        float mx = -INFINITY;
        for (int c0 = 0; c0 < 256; c0 += 32) {
            float v[32];
            __syncwarp();
            tmem_ld32(tbase + (uint32_t)c0, v);
#pragma unroll
            for (int i = 0; i < 32; ++i) mx = fmaxf(mx, v[i] + __ldg(bias + c0 + i));
        }
        float run = 0.0f, cum[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            float v[32];
            __syncwarp();
            tmem_ld32(tbase + (uint32_t)(k * 32), v);
#pragma unroll
            for (int i = 0; i < 32; ++i) run += __expf((v[i] + __ldg(bias + k * 32 + i)) - mx);
            cum[k] = run;
        }
        const float target = u * run;
        int ck = 8;
        float base = 0.0f;
#pragma unroll
        for (int k = 7; k >= 0; --k)
            if (target < cum[k]) { ck = k; base = k > 0 ? cum[k - 1] : 0.0f; }
        int bi = (run == run) ? 255 : 0;          // u at the very top of the range; no finite score: class 0
        for (int k = 0; k < 8; ++k) {
            float v[32];
            __syncwarp();
            tmem_ld32(tbase + (uint32_t)(k * 32), v);         // warp-wide load: every lane takes part
            if (k != ck) continue;
            float s2 = base;
            int hit = -1;
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                s2 += __expf((v[i] + __ldg(bias + k * 32 + i)) - mx);
                hit = (hit < 0 && target < s2) ? i : hit;
            }
            bi = k * 32 + (hit < 0 ? 31 : hit);
        }
        return bi;
    }

    __device__ void epilogue(int l, int kind, const Win &w, bool flag, int fslot, float *zout, int yt_lo, int nyl,
                             int ntiles, int src)
    {
        const bool head = (l == m.n_conv);
        const int per = head ? m.in_ch : 1;
        const int q = warp & 3;
        // Two warps share a quadrant (a warp reaches only the tensor-memory lanes of its own quadrant).  The
        // second one takes the upper half of the channels or of the 256 classes (the argmax is bound by instruction
        // issue, one warp per scheduler was not enough); behind uniform noise it only hands the accumulator back.
        const int half = (warp - 2) >> 2;
        if (warp == 4 && lane == 0) trace(0);
        int tile_par = 0;
        const bool split_head = head && kind == EPI_CAT && r.nk == JS_NOISE_GUMBEL;
        bool any_changed = false;
        int first = INT_MAX;
        if (split_head) noise_may_come();
        int id = blockIdx.x;
        for (; id < ntiles && !dead; id += gridDim.x) {
            int n, yt, c;
            locate(id, nyl, yt_lo, per, n, yt, c);
            const int y0 = yt * m.R;
            if (half == 1 && head && !split_head && kind != EPI_LOGITS) {
                if (!__all_sync(0xffffffffu, mbar_wait(&sh.tfull[acc], aphase, r.ctl))) { dead = true; break; }
                tc_fence_after();
                release_acc();
                advance_acc();
                continue;
            }
            if (!head || split_head) {
                const float *bias = head ? m.bias[l] + (size_t)c * 256 + half * 128 : m.bias[l] + half * (m.ch / 2);
                float *bs = sh.bias_s[warp - 2];
                __syncwarp();
                if (4 * lane < (head ? 128 : m.ch / 2))
                    *reinterpret_cast<float4 *>(bs + 4 * lane) = __ldg(reinterpret_cast<const float4 *>(bias) + lane);
                __syncwarp();
            }
            if (!__all_sync(0xffffffffu, mbar_wait(&sh.tfull[acc], aphase, r.ctl))) { dead = true; break; }
            tc_fence_after();
            if (warp == 4 && lane == 0) trace(3);
            const uint32_t tbase = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * ACC_COLS);
            if (!head) {
                epi_hidden_tile(n, y0, tbase, half, (__nv_bfloat16 *)(src == SRC_OLD ? m.act_old[l + 1] : m.act[l + 1]));
            } else {
                // thread = one pixel of the tile; 256 logits of sub-pixel c
                const int prow = q * 32 + lane;
                const int rows_valid = (min(m.height, y0 + m.R) - y0) * m.width;
                const bool valid = prow < rows_valid;
                const int pix = y0 * m.width + prow;
                const int t = pix * m.in_ch + c;
                const size_t at = (size_t)n * m.T + t;
                const float *bias = m.bias[m.n_conv] + (size_t)c * 256;
                float best = -INFINITY;
                int bi = 0;
                // the current symbol, asked for now: its latency passes while the classes are reduced
                const bool commit = kind == EPI_CAT && valid && t >= w.plo && t < w.phi;
                int xold = 0;
                if (commit) xold = (int)__ldcg(r.x + at);
                if (kind == EPI_CAT && r.nk == JS_NOISE_UNIFORM_CAT) {
                    bi = head_icdf(tbase, bias, commit ? __ldg(r.noise + at) : 0.5f);
                } else
                for (int c0 = half * 128; c0 < half * 128 + 128; c0 += 32) {
                    float v[32];
                    __syncwarp();
                    tmem_ld32(tbase + (uint32_t)c0, v);
                    if (kind == EPI_LOGITS) {
                        if (!valid) continue;
#pragma unroll
                        for (int i = 0; i < 32; ++i) zout[at * 256 + c0 + i] = v[i] + bias[c0 + i];
                    } else {
                        if (!__all_sync(0xffffffffu, mbar_wait(&sh.nfull[half][nz_buf], (nz_par >> nz_buf) & 1u, r.ctl))) { dead = true; break; }
                        // lane = pixel: rows of 128 bytes, their 16-byte chunks permuted by the row number (the box's swizzle)
                        const uint32_t gg = smem_u32(noise_buf(half, nz_buf)) + 128u * (uint32_t)prow;
                        const uint32_t bb = smem_u32(sh.bias_s[warp - 2]) + 4u * (uint32_t)(c0 - half * 128);
                        float sc[32];
#pragma unroll
                        for (int i = 0; i < 32; i += 4) {
                            const float4 b4 = lds_f4(bb + 4u * (uint32_t)i), g4 = lds_f4(gg + 16u * (uint32_t)((i >> 2) ^ (lane & 7)));
                            sc[i] = (v[i] + b4.x) + g4.x;
                            sc[i + 1] = (v[i + 1] + b4.y) + g4.y;
                            sc[i + 2] = (v[i + 2] + b4.z) + g4.z;
                            sc[i + 3] = (v[i + 3] + b4.w) + g4.w;
                        }
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&sh.nempty[half][nz_buf]);
                        nz_par ^= 1u << nz_buf;
                        if (++nz_buf == NOISE_BUFS) nz_buf = 0;
                        argmax_chunk32(sc, c0, best, bi);
                    }
                }
                release_acc();        // the accumulator has been read: the next tile's MMAs may have it
                if (split_head) {
                    // the two halves meet: the upper half's result wins only if strictly larger (lowest index on ties)
                    if (half == 1) {
                        sh.xbest[tile_par][q][lane] = best;
                        sh.xbi[tile_par][q][lane] = bi;
                    }
                    asm volatile("bar.sync %0, 64;" ::"r"(1 + q) : "memory");
                    if (half == 0) {
                        const float b1 = sh.xbest[tile_par][q][lane];
                        if (b1 > best) { best = b1; bi = sh.xbi[tile_par][q][lane]; }
                    }
                    tile_par ^= 1;
                }
                if (half == 1) { advance_acc(); continue; }
                bool ch = false;
                if (commit && xold != bi) {
                    r.x[at] = (uint8_t)bi;
                    ((__nv_bfloat16 *)m.act[0])[((size_t)n * m.height * m.width + pix) * 64 + c] =
                        __float2bfloat16_rn(sh.lut_s[bi]);
                    ch = true;
                }
                if (flag) {
                    // every pixel of the tile belongs to image n: one lane reports for the warp, with a
                    // plain store (a load to look first would be an L2 round trip per tile), and only
                    // once per image and phase
                    if (__any_sync(0xffffffffu, ch) && (raised_img != n || raised_phase != phase_no)) {
                        if (lane == 0) r.smp_changed[fslot * r.batch + n] = 1;
                        raised_img = n;
                        raised_phase = phase_no;
                    }
                    if (ch) {
                        any_changed = true;
                        first = min(first, t);
                    }
                }
            }
            advance_acc();
        }
        // a warp that gave up lets its partner through the meetings it will not come to
        if (split_head && dead)
            for (; id < ntiles; id += gridDim.x) asm volatile("bar.arrive %0, 64;" ::"r"(1 + q) : "memory");
        if (warp == 4 && lane == 0) trace(4);
        if (warp == 4 && lane == 0) trace(5);            // (a pass's last layer: overwritten behind the grid barrier)
        if (flag) {
            const bool wany = __any_sync(0xffffffffu, any_changed);
            if (wany) {
                const int wmin = __reduce_min_sync(0xffffffffu, first);
                if (lane == 0) {
                    atomicMin(&r.ctl->agg_minfirst[fslot], wmin);
                    atomicOr(&r.ctl->agg_any[fslot], 1);
                }
            }
        }
    }

    __device__ void layer_phase(int l, int kind, const Win &w, bool flag, int fslot, float *zout, int src = SRC_NEW)
    {
        const bool head = (l == m.n_conv);
        int yt_lo, yt_hi;
        live_rows(head, w, yt_lo, yt_hi);
        const int nyl = yt_hi - yt_lo;
        const int ntiles = sh.n_img[icur] * nyl * (head ? m.in_ch : 1);
        if (threadIdx.x == 0) {
            for (int id = blockIdx.x; id < ntiles; id += gridDim.x) {
                issued++;
                mma_flops += 2ull * BM * BK * (unsigned long long)(head ? 256 : m.ch) * (unsigned long long)kblocks(l);
            }
            // a layer's packed weights serve every tile: the pass streams them once
            if (blockIdx.x == 0 && ntiles > 0)
                weight_bytes += 2ull * BK * (unsigned long long)kblocks(l) * (unsigned long long)(head ? 256 * m.in_ch : m.ch);
            if (blockIdx.x == 0) skipped += (unsigned long long)(r.batch * m.nyt - sh.n_img[icur] * nyl) * (head ? m.in_ch : 1);
        }
        if (ntiles == 0) return;
        phase_no++;
        layer_no++;
        if (!head) conv_lo = yt_lo, conv_hi = yt_hi;
        if (warp == 0) {
            load_pixels(l, yt_lo, nyl, ntiles, src);
        } else if (warp == 1) {
            mma_issuer(l, src, ntiles);
        } else if (warp == 10) {
            load_weights(l, ntiles);
        } else if (warp == 11) {
            if (head && kind == EPI_CAT && r.nk == JS_NOISE_GUMBEL) {
                noise_may_come();
                load_noise(yt_lo, nyl, ntiles);
            }
        } else {
            epilogue(l, kind, w, flag, fslot, zout, yt_lo, nyl, ntiles, src);
        }
    }

    // One pass.  Inside it the tiles wait for one another by their stamps; the grid barrier at its end lets the next pass
    // overwrite what this one read, and makes the flags complete.
    __device__ bool step(const Win &w, bool flag, int fslot, float *zout, int src = SRC_NEW)
    {
        conv_lo = conv_hi = 0;
        const int l_end = src == SRC_OLD ? m.n_conv - 1 : m.n_conv;      // the old set needs no head
        for (int l = 0; l <= l_end; ++l) {
            const bool last = (l == m.n_conv);
            layer_phase(l, last ? (zout ? EPI_LOGITS : EPI_CAT) : EPI_HIDDEN, w, last && flag, fslot, zout, src);
        }
        return barrier();
    }

    // One outer iteration of Algorithm 2 with one-image-row blocks.  A block's sequential sweep yields the
    // unique solution of the block's own triangular system given the rows above at the previous outer
    // iterate; Jacobi iterations on that sub-system reach the very same solution in at most |B| steps
    // (Proposition 1 applied to the block), and they can run for all rows of all images at once as
    // forward passes in which every layer reads the row above from the activations of x^{k-1} and its
    // own row from the working activations.  So: the hidden layers once on x^{k-1} (the "old" set),
    // then mixed passes until no symbol changes, then the comparison with x^{k-1} for the outer flags,
    // which are left in the flag slot `fslot`.
    __device__ bool jgs_outer(int fslot, int, int, int &iterations)
    {
        const size_t n = (size_t)r.batch * m.T;
        const size_t npix64 = (size_t)r.batch * m.height * m.width * 64 / 8;       // uint4 units of the padded image
        for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
            r.x_old[i] = r.x[i];
        {
            const uint4 *src = reinterpret_cast<const uint4 *>(m.act[0]);
            uint4 *dst = reinterpret_cast<uint4 *>(m.act_old[0]);
            for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < npix64; i += (size_t)gridDim.x * blockDim.x)
                dst[i] = src[i];
        }
        if (!barrier()) return false;
        // every CTA has read the previous outer iteration's flags by now: all slots start clean
        if (blockIdx.x == 0) clear_flags(r);
        const Win w = make_win(0, m.T, 0, m.T);
        if (!step(w, false, 0, nullptr, SRC_OLD)) return false;
        iterations++;
        const int cap = m.width * m.in_ch;
        int q = fslot;
        for (int k = 1; k <= cap; ++k) {
            q = next_slot(q);
            if (!step(w, true, q, nullptr, SRC_MIXED)) return false;
            iterations++;
            const int any = ld_volatile_i32(&r.ctl->agg_any[q]);
            clear_old_slot(r, q);
            if (!barrier()) return false;
            if (!any) break;
        }
        // all flag slots start clean, then the outer comparison fills slot `fslot`
        if (blockIdx.x == 0) clear_flags(r);
        if (!barrier()) return false;
        for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
            if (r.x[i] != r.x_old[i]) note_change(r, fslot, (int)(i / m.T), (int)(i % m.T));
        return barrier();
    }
};

__global__ void __launch_bounds__(NTH, 1)
conv_tc_kernel(const __grid_constant__ ConvDev m, const __grid_constant__ RunArgs r, const __grid_constant__ CUtensorMap tm_noise)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ ConvShared sh;
    uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) { mbar_init(&sh.wfull[s], 1); mbar_init(&sh.wempty[s], 1); }
        for (int s = 0; s < MAX_STAGES; ++s) { mbar_init(&sh.afull[s], 1); mbar_init(&sh.aempty[s], 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(&sh.tfull[a], 1); mbar_init(&sh.tempty[a], 8); }
        for (int h = 0; h < 2; ++h)
            for (int i = 0; i < NOISE_BUFS; ++i) { mbar_init(&sh.nfull[h][i], 1); mbar_init(&sh.nempty[h][i], 4); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    for (int i = threadIdx.x; i < 256; i += blockDim.x) sh.lut_s[i] = m.lut[i];
    if (warp == 1) tmem_alloc(&sh.tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    ConvEngine e(m, r, tm_noise, sh, ring);
    e.tmem_base = sh.tmem_base;
    DriverResult res = made_driver(e, m.T, r);
    if (e.dead) res.alive = false;

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
    driver_finish(r, res, e.issued, e.skipped, e.mma_flops, e.weight_bytes);
}

}  // namespace

// --------------------------------------------------------------- host side
static bool encode_nd(CUtensorMap *out, const void *base, int rank, const cuuint64_t *dims, const cuuint64_t *strides,
                      const cuuint32_t *box, CUtensorMapDataType type = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16)
{
    return js_encode_map(out, type, base, rank, dims, strides, box);
}

template <typename T>
static bool upload(js_model *mo, const T *host, size_t count, T **dev)
{
    void *p = nullptr;
    if (cudaMalloc(&p, std::max<size_t>(count * sizeof(T), 16)) != cudaSuccess) return false;
    mo->allocs.push_back(p);
    if (host) {
        if (cudaMemcpy(p, host, count * sizeof(T), cudaMemcpyHostToDevice) != cudaSuccess) return false;
    } else if (cudaMemset(p, 0, count * sizeof(T)) != cudaSuccess) {
        return false;
    }
    *dev = (T *)p;
    return true;
}

// Builds the device model of a masked-conv stack.  JS_OK, JS_ERR_UNSUPPORTED for shapes the
// kernel does not cover, JS_ERR_CUDA on runtime failures.
int js_conv_build(js_model *mo, const js_conv_desc *d)
{
    ConvDev &v = mo->conv;
    if (d->prec != JS_BF16 || d->C != 256 || d->n_lut != 256) return JS_ERR_UNSUPPORTED;
    if (d->in_ch < 1 || d->in_ch > 8 || (d->ch != 64 && d->ch != 128)) return JS_ERR_UNSUPPORTED;
    if (d->width < 8 || d->width > 128 || (128 % d->width) != 0 || d->height < 1) return JS_ERR_UNSUPPORTED;
    if (d->n_conv < 1 || d->n_conv > JS_MAXL || d->max_batch > MAX_IMAGES) return JS_ERR_UNSUPPORTED;
    if (!js_tensor_maps()) return JS_ERR_UNSUPPORTED;
    v.height = d->height; v.width = d->width; v.in_ch = d->in_ch; v.ch = d->ch; v.n_conv = d->n_conv; v.C = d->C;
    v.T = d->height * d->width * d->in_ch;
    v.R = 128 / d->width;
    v.nyt = (d->height + v.R - 1) / v.R;
    const int ch = d->ch, nb = mo->max_batch;
    const size_t npix = (size_t)nb * d->height * d->width;
    auto group = [&](int k) { return (int)(((long long)d->in_ch * k) / ch); };

    // a pixel stage with the row above the tile, if three shifts of all channels fit into the ring
    const int two = (v.R + 1) * d->width * BK * 2;
    v.share = 3 * (ch / BK) * two <= A_RING;
    v.stage_a = v.share ? two : A_BYTES;
    std::vector<CUtensorMap> mapsA(d->n_conv + 1), mapsAold(d->n_conv + 1), mapsA2(d->n_conv + 1), mapsAold2(d->n_conv + 1), mapsW(d->n_conv + 1);
    for (int l = 0; l <= d->n_conv; ++l) {
        const int c_l = l == 0 ? 64 : ch;                 // channels of act[l] (the image is padded to 64)
        if (l < d->n_conv) v.cin_pad[l] = c_l;
        // two sets: the working activations, and those of the previous outer iterate (Jacobi-GS)
        for (int set = 0; set < 2; ++set) {
            __nv_bfloat16 *a = nullptr;
            if (!upload<__nv_bfloat16>(mo, nullptr, npix * c_l, &a)) return JS_ERR_CUDA;
            (set == 0 ? v.act[l] : v.act_old[l]) = a;
            const cuuint64_t dims[4] = {(cuuint64_t)c_l, (cuuint64_t)d->width, (cuuint64_t)d->height, (cuuint64_t)nb};
            const cuuint64_t strides[3] = {(cuuint64_t)c_l * 2, (cuuint64_t)d->width * c_l * 2,
                                           (cuuint64_t)d->height * d->width * c_l * 2};
            const cuuint32_t box[4] = {(cuuint32_t)BK, (cuuint32_t)d->width, (cuuint32_t)v.R, 1};
            const cuuint32_t box2[4] = {(cuuint32_t)BK, (cuuint32_t)d->width, (cuuint32_t)v.R + 1, 1};
            if (!encode_nd(set == 0 ? &mapsA[l] : &mapsAold[l], a, 4, dims, strides, box)) return JS_ERR_UNSUPPORTED;
            if (!encode_nd(set == 0 ? &mapsA2[l] : &mapsAold2[l], a, 4, dims, strides, box2)) return JS_ERR_UNSUPPORTED;
        }
    }
    static const int tky[5] = {0, 0, 0, 1, 1}, tkx[5] = {0, 1, 2, 0, 1};
    for (int l = 0; l < d->n_conv; ++l) {
        const int cin = l == 0 ? d->in_ch : ch, cpad = v.cin_pad[l];
        std::vector<__nv_bfloat16> wp((size_t)5 * ch * cpad, __float2bfloat16_rn(0.0f));
        for (int tap = 0; tap < 5; ++tap)
            for (int co = 0; co < ch; ++co)
                for (int ci = 0; ci < cin; ++ci) {
                    bool keep = true;
                    if (tap == 4) {                       // centre tap: colour-group mask, type A then type B
                        const int gi = l == 0 ? ci : group(ci), go = group(co);
                        keep = l == 0 ? (gi < go) : (gi <= go);
                    }
                    const float w = keep ? d->W[l][(((size_t)co * 3 + tky[tap]) * 3 + tkx[tap]) * cin + ci] : 0.0f;
                    wp[((size_t)tap * ch + co) * cpad + ci] = __float2bfloat16_rn(w);
                }
        __nv_bfloat16 *wd = nullptr;
        if (!upload<__nv_bfloat16>(mo, wp.data(), wp.size(), &wd)) return JS_ERR_CUDA;
        const cuuint64_t dims[2] = {(cuuint64_t)cpad, (cuuint64_t)5 * ch};
        const cuuint64_t strides[1] = {(cuuint64_t)cpad * 2};
        const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)ch};
        if (!encode_nd(&mapsW[l], wd, 2, dims, strides, box)) return JS_ERR_UNSUPPORTED;
        float *bd = nullptr;
        if (!upload<float>(mo, d->b[l], ch, &bd)) return JS_ERR_CUDA;
        v.bias[l] = bd;
    }
    {
        const int nout = d->in_ch * d->C;
        std::vector<__nv_bfloat16> wh((size_t)nout * ch);
        for (int o = 0; o < nout; ++o)
            for (int ci = 0; ci < ch; ++ci)
                wh[(size_t)o * ch + ci] =
                    __float2bfloat16_rn(group(ci) <= o / d->C ? d->W[d->n_conv][(size_t)o * ch + ci] : 0.0f);
        __nv_bfloat16 *wd = nullptr;
        if (!upload<__nv_bfloat16>(mo, wh.data(), wh.size(), &wd)) return JS_ERR_CUDA;
        const cuuint64_t dims[2] = {(cuuint64_t)ch, (cuuint64_t)nout};
        const cuuint64_t strides[1] = {(cuuint64_t)ch * 2};
        const cuuint32_t box[2] = {(cuuint32_t)BK, 256};
        if (!encode_nd(&mapsW[d->n_conv], wd, 2, dims, strides, box)) return JS_ERR_UNSUPPORTED;
        float *bd = nullptr;
        if (!upload<float>(mo, d->b[d->n_conv], nout, &bd)) return JS_ERR_CUDA;
        v.bias[d->n_conv] = bd;
    }
    {
        std::vector<float> lut(d->lut, d->lut + d->n_lut);
        for (auto &f : lut) f = __bfloat162float(__float2bfloat16_rn(f));
        float *ld = nullptr;
        if (!upload<float>(mo, lut.data(), lut.size(), &ld)) return JS_ERR_CUDA;
        v.lut = ld;
    }
    if (!upload<int>(mo, nullptr, (size_t)nb * v.nyt * 8, &v.stamp)) return JS_ERR_CUDA;
    CUtensorMap *pa = nullptr, *pw = nullptr, *pao = nullptr, *pa2 = nullptr, *pao2 = nullptr;
    if (!upload<CUtensorMap>(mo, mapsA2.data(), mapsA2.size(), &pa2)) return JS_ERR_CUDA;
    if (!upload<CUtensorMap>(mo, mapsAold2.data(), mapsAold2.size(), &pao2)) return JS_ERR_CUDA;
    v.tmAct2 = pa2;
    v.tmActOld2 = pao2;
    if (!upload<CUtensorMap>(mo, mapsAold.data(), mapsAold.size(), &pao)) return JS_ERR_CUDA;
    v.tmActOld = pao;
    if (!upload<CUtensorMap>(mo, mapsA.data(), mapsA.size(), &pa)) return JS_ERR_CUDA;
    if (!upload<CUtensorMap>(mo, mapsW.data(), mapsW.size(), &pw)) return JS_ERR_CUDA;
    v.tmAct = pa;
    v.tmW = pw;
    if (cudaFuncSetAttribute(conv_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES) != cudaSuccess) {
        cudaGetLastError();
        return JS_ERR_UNSUPPORTED;
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    mo->conv_max_grid = sms;
    mo->conv_T = v.T;
    mo->conv_C = v.C;
    return JS_OK;
}

int js_launch_conv_tc(const js_model *mo, const RunArgs &r, cudaStream_t stream)
{
    const ConvDev &v = mo->conv;
    const int tiles = r.batch * v.nyt * v.in_ch;
    const int grid = std::max(1, std::min(mo->conv_max_grid, tiles));
    CUtensorMap noise;
    std::memset(&noise, 0, sizeof noise);
    if (r.nk == JS_NOISE_GUMBEL && r.noise) {
        // {class, sub-pixel, pixel}, a box per 128 pixels and 32 classes of one sub-pixel
        const cuuint64_t dims[3] = {256, (cuuint64_t)v.in_ch, (cuuint64_t)r.batch * v.height * v.width};
        const cuuint64_t strides[2] = {1024, (cuuint64_t)v.in_ch * 1024};
        const cuuint32_t box[3] = {32, 1, 128};
        if (!encode_nd(&noise, r.noise, 3, dims, strides, box, CU_TENSOR_MAP_DATA_TYPE_FLOAT32)) return (int)cudaErrorInvalidValue;
    }
    void *args[3] = {(void *)&v, (void *)&r, (void *)&noise};
    cudaError_t e = cudaLaunchCooperativeKernel((const void *)conv_tc_kernel, dim3(grid), dim3(NTH), args, SMEM_BYTES,
                                                stream);
    return e == cudaSuccess ? 0 : (int)e;
}
