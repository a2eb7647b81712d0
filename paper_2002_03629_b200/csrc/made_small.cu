// Small fp32 masked MLPs (binary positions, or continuous states with two outputs per position), Jacobi mode.
//
// Samples never look at one another, so a solve needs no grid-wide step at all: a thread-block cluster of
// CS <= 8 CTAs takes a few samples through every iteration until they stop changing.  The masked weights stay in
// shared memory for the whole call (CTA c of a cluster owns the units c, c + CS, c + 2 CS ... of every layer), and
// so do the samples' activations (every CTA of the cluster holds all of them): a layer is a matrix product out of
// shared memory, its results are written into all CTAs of the cluster, and one hardware cluster barrier (0.2 us,
// against 1.5 us plus a memory round trip for the grid barrier of made_generic.cu) ends it.
//
// What bounds it: latency - the dependent chain  layer -> barrier -> layer  and the launch itself; the arithmetic
// of these models is a few microseconds of one SM at most.
// Every output is one chain of fused multiply-adds over k in ascending order, exactly as in made_generic.cu, so
// both kernels return the same bits.
//
// Measured (B200, the call as a Python program sees it, 3 or 4 iterations): T = 16, H = 64, batch 8: 58 us with
// made_generic.cu, 19 us here, of which launch and report are 7.
#include <algorithm>
#include <cstring>
#include <vector>

#include "js_common.cuh"
#include "js_model.h"
#include "made_driver.cuh"
#include "tc_common.cuh"

namespace {

constexpr int NTH = 256;
constexpr int RMAX = 64;                 // samples per cluster
constexpr int SMEM_MAX = 220 * 1024;
constexpr int KS = 16;                   // inputs per step of a product; rows of weights and activations are padded to it
__host__ __device__ inline int pad_k(int k) { return (k + KS - 1) / KS * KS; }

struct SmallShared {
    uint64_t wbar;
    int chg[2][RMAX];                    // per parity: did the sample change in this CTA's positions
    int first[2];                        // per parity: smallest changed position of this CTA
    int done[RMAX], count[RMAX];
    unsigned tiles, skipped;
};

__device__ __forceinline__ void st_peer_f(uint32_t addr, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ int ld_peer_i(uint32_t addr)
{
    int v;
    asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}

// shared memory after the packed weights: activations a[l][k][RS], noise and symbols of the CTA's own positions
struct Layout {
    int a[JS_MAXL + 1];                  // float offsets
    int nz, xs, total;
};
__host__ __device__ inline Layout small_layout(const MadeDev &m, const SmallDev &s, int RS)
{
    Layout o;
    int at = s.pack_floats;
    for (int l = 0; l <= m.L; ++l) { o.a[l] = at; at += pad_k(m.n[l]) * RS; }
    const int own = (m.T + s.CS - 1) / s.CS;
    o.nz = at; at += own * RS;
    o.xs = at; at += own * RS;
    o.total = at;
    return o;
}

// KS rows of RG activations.  RG == 1 has a row stride of 1 (see rows_group): four rows per load.
template <int RG>
__device__ __forceinline__ void load_rows(const float *a, int RS, float (&av)[KS][RG])
{
    if constexpr (RG == 1) {
#pragma unroll
        for (int q = 0; q < KS; q += 4) {
            const float4 v = *reinterpret_cast<const float4 *>(a + q);
            av[q][0] = v.x; av[q + 1][0] = v.y; av[q + 2][0] = v.z; av[q + 3][0] = v.w;
        }
    } else {
#pragma unroll
        for (int q = 0; q < KS; ++q) {
            if constexpr (RG == 4) {
                const float4 v = *reinterpret_cast<const float4 *>(a + q * RS);
                av[q][0] = v.x; av[q][1] = v.y; av[q][2] = v.z; av[q][3] = v.w;
            } else {
                const float2 v = *reinterpret_cast<const float2 *>(a + q * RS);
                av[q][0] = v.x; av[q][1] = v.y;
            }
        }
    }
}

// RG: samples per thread in the products (a row of RG activations is one vector load, broadcast over the warp)
// REAL: continuous states; CL: the cluster has more than one CTA
template <int RG, bool REAL, bool CL>
__global__ void __launch_bounds__(NTH)
made_small_kernel(const __grid_constant__ MadeDev m, const __grid_constant__ SmallDev s, const __grid_constant__ RunArgs r,
                  const int R)
{
    extern __shared__ __align__(16) float sm[];
    __shared__ SmallShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int CS = CL ? s.CS : 1, csh = CL ? s.cs_log2 : 0, c = CL ? (int)cluster_rank() : 0;
    const int RS = (R + RG - 1) / RG * RG;               // row stride of the activations
    const int row0 = (int)(blockIdx.x >> csh) * R, nrow = min(R, r.batch - row0);
    const Layout lo_ = small_layout(m, s, RS);
    const int T = m.T, L = m.L;
    const float lut0 = REAL ? 0.0f : __ldg(m.lut), lut1 = REAL ? 0.0f : __ldg(m.lut + 1);

    if (tid == 0) {
        mbar_init(&sh.wbar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_proxy_async();
    }
    __syncthreads();
    // this CTA's weights, biases and degrees: one contiguous piece, brought in while the iterate is set up
    if (tid == 0) {
        const uint32_t bytes = (uint32_t)s.pack_floats * 4u;
        mbar_expect_tx(&sh.wbar, bytes);
        const uint8_t *src = reinterpret_cast<const uint8_t *>(s.pack) + (size_t)c * bytes;
        for (uint32_t at = 0; at < bytes; at += 32768u)
            bulk_load(smem_u32(sm) + at, src + at, min(32768u, bytes - at), &sh.wbar);
    }
    float *a0 = sm + lo_.a[0], *nz = sm + lo_.nz, *xs = sm + lo_.xs;
    const int own = (T - c + CS - 1) >> csh;             // own positions: c + CS * j
    for (int rr = warp; rr < RS; rr += NTH / 32)
        for (int t = lane; t < T; t += 32) {
            float v = 0.0f, e = 0.0f;
            if (rr < nrow) {
                const size_t at = (size_t)(row0 + rr) * T + t;
                e = __ldg(r.noise + at);
                if constexpr (REAL) v = r.init_r ? r.init_r[at] : 0.0f;
                else v = r.init ? (float)r.init[at] : 0.0f;
            }
            if ((t & (CS - 1)) == c) {
                const int j = t >> csh;
                xs[j * RS + rr] = v;
                nz[j * RS + rr] = e;
            }
            a0[t * RS + rr] = REAL ? v : v != 0.0f ? lut1 : lut0;
        }
    for (int l = 0; l <= L; ++l)                         // padding rows are multiplied by zero weights: keep them finite
        for (int i = (l == 0 ? T : m.n[l]) * RS + tid; i < pad_k(m.n[l]) * RS; i += NTH) sm[lo_.a[l] + i] = 0.0f;
    for (int i = tid; i < 2 * RMAX; i += NTH) {
        sh.chg[i / RMAX][i % RMAX] = 0;
        if (i < RMAX) { sh.done[i] = 0; sh.count[i] = 0; }
    }
    if (tid < 2) sh.first[tid] = INT_MAX;
    if (tid == 0) sh.tiles = sh.skipped = 0u;
    // A CTA whose weights do not come says so where every CTA of the cluster looks for the first iteration's changes: all of
    // them leave at the same place then.  (A spin limit of zero: the first look decides, as at the grid barriers.)
    bool here = mbar_test_wait(&sh.wbar, 0);
    if (!here && r.spin_limit != 0) here = mbar_wait(&sh.wbar, 0, r.ctl);
    const bool gave_up = !__syncthreads_and(here);
    if (gave_up && tid == 0) {
        atomicExch(&r.ctl->abort, 1);
        sh.first[1] = -1;
    }
    if constexpr (CL) cluster_sync();          // every CTA of the cluster has started: its shared memory may be written
    else __syncthreads();

    const int cap = (r.max_iters > 0 && r.max_iters < T) ? r.max_iters : T;
    int fin_x = 0, fin_h = 0, lo = 0, k = 0, status = JS_OK;
    unsigned tiles = 0, skipped = 0;
    int mf;
    for (;;) {
        ++k;
        const int par = k & 1;
        const int hlo = r.frontier_skip ? fin_h : 0, plo = r.frontier_skip ? lo : 0;
        for (int l = 0; l <= L; ++l) {
            const bool out = l == L;
            const int K = m.n[l], nc = s.nc[l], ncs = s.ncs[l];
            const float *W = sm + s.w_off[l], *bias = sm + s.b_off[l];
            const uint32_t *deg = reinterpret_cast<const uint32_t *>(sm + s.d_off[l]);      // degree, inputs << 16
            const float *A = sm + lo_.a[l];
            // a warp's work: 32 own outputs of one group of RG samples
            const int nblk = (nc + 31) / 32, nrg = RS / RG;
            for (int rg = 0, blk = warp;; blk += NTH / 32) {
                while (blk >= nblk) { blk -= nblk; ++rg; }
                if (rg >= nrg) break;
                const int ib = blk * 32, i = ib + lane;
                const bool mine = i < nc;
                const int ii = min(i, nc - 1), dg = (int)(deg[ii] & 0xffffu);
                // live: hidden units of degree > hlo, output positions (degree - 1) >= plo
                const bool live = mine && (out ? dg > plo : dg > hlo);
                if (!__any_sync(0xffffffffu, live)) { skipped++; continue; }
                tiles++;
                // inputs beyond the largest degree of the warp's units are masked: exact zeros
                const int kend = min(K, s.kend[l][min(ib / 32, SMALL_KENDS - 1)]);
                // Inputs up to the unit's own last live one.  The warp's units lie CS apart, so the warp reads far beyond it for
                // some; a continuous state may be infinite there (its noise is, or an iterate on its way), and a zero weight
                // does not make that a zero.
                const int kl = REAL ? (int)(deg[ii] >> 16) : 0;
                const int kall = REAL ? (int)__reduce_min_sync(0xffffffffu, (unsigned)kl) : 0;
                float acc[RG];
#pragma unroll
                for (int q = 0; q < RG; ++q) acc[q] = 0.0f;
                // KS steps at a time: their loads in flight together, then the multiply-adds in order
                const float *w = W + ii, *a = A + rg * RG;
                int k0 = 0;
                if (RG > 1 || !REAL)
                    for (; k0 < (REAL ? min(kend, kall / KS * KS) : kend); k0 += KS) {
                        float wv[KS], av[KS][RG];
#pragma unroll
                        for (int q = 0; q < KS; ++q) wv[q] = w[(k0 + q) * ncs];
                        load_rows<RG>(a + k0 * RS, RS, av);
#pragma unroll
                        for (int kk = 0; kk < KS; ++kk)
#pragma unroll
                            for (int q = 0; q < RG; ++q) acc[q] = fmaf(av[kk][q], wv[kk], acc[q]);
                    }
                if constexpr (REAL)
                    for (; k0 < kend; k0 += KS) {
                        float wv[KS], av[KS][RG];
#pragma unroll
                        for (int q = 0; q < KS; ++q) wv[q] = w[(k0 + q) * ncs];
                        load_rows<RG>(a + k0 * RS, RS, av);
#pragma unroll
                        for (int kk = 0; kk < KS; ++kk)
#pragma unroll
                            for (int q = 0; q < RG; ++q)
                                if (k0 + kk < kl) acc[q] = fmaf(av[kk][q], wv[kk], acc[q]);
                    }
                const float bv = bias[ii];
#pragma unroll
                for (int q = 0; q < RG; ++q) {
                    const int rr = rg * RG + q;
                    const float pre = acc[q] + bv;
                    if (!out) {
                        if (live) {
                            const float v = js_act_fn(m.act, pre);
                            const uint32_t at = smem_u32(sm + lo_.a[l + 1] + (size_t)(c + CS * i) * RS + rr);
                            if constexpr (!CL) sm[lo_.a[l + 1] + (size_t)i * RS + rr] = v;
                            else
                                for (int p = 0; p < CS; ++p) st_peer_f(peer_addr(at, p), v);
                        }
                        continue;
                    }
                    int j = i;
                    float xn, xo;
                    if constexpr (REAL) {
                        // a pair of lanes holds location and log-scale of a position
                        const float ls = __shfl_down_sync(0xffffffffu, pre, 1);
                        j = i >> 1;
                        if (!live || (i & 1) || rr >= nrow || sh.done[rr]) continue;
                        xo = xs[j * RS + rr];
                        xn = fmaf(expf(ls), nz[j * RS + rr], pre);
                        xs[j * RS + rr] = xn;
                        if (!(fabsf(xn - xo) <= r.eps)) {        // a NaN difference is a change
                            sh.chg[par][rr] = 1;
                            atomicMin(&sh.first[par], c + CS * j);
                        }
                    } else {
                        if (!live || rr >= nrow) continue;
                        xo = xs[j * RS + rr];
                        xn = (float)js_sample_binary(r.nk, pre, nz[j * RS + rr]);
                        if (xn == xo) continue;
                        xs[j * RS + rr] = xn;
                        sh.chg[par][rr] = 1;
                        atomicMin(&sh.first[par], c + CS * j);
                    }
                    const float enc = REAL ? xn : xn != 0.0f ? lut1 : lut0;
                    const uint32_t at = smem_u32(a0 + (size_t)(c + CS * j) * RS + rr);
                    if constexpr (!CL) a0[(size_t)j * RS + rr] = enc;
                    else
                        for (int p = 0; p < CS; ++p) st_peer_f(peer_addr(at, p), enc);
                }
            }
            if constexpr (CL) cluster_sync();
            else __syncthreads();
        }
        // Every warp reads the flags of all CTAs of the cluster (they are kept until two iterations later, so no
        // further barrier is needed); the first keeps the samples' counts, the second clears the other parity's flags,
        // last read before the barriers of this iteration.
        int any = 0;
        mf = INT_MAX;
        for (int rr = lane; rr < nrow; rr += 32) {
            int ch = 0;
            if constexpr (CL)
                for (int p = 0; p < CS; ++p) ch |= ld_peer_i(peer_addr(smem_u32(&sh.chg[par][rr]), p));
            else ch = sh.chg[par][rr];
            any |= ch;
            if (warp == 0 && !sh.done[rr] && (ch == 0 || k == cap)) { sh.done[rr] = 1; sh.count[rr] = k; }
        }
        if (lane < CS) mf = CL ? ld_peer_i(peer_addr(smem_u32(&sh.first[par]), lane)) : sh.first[par];
        mf = __reduce_min_sync(0xffffffffu, mf);
        any = __any_sync(0xffffffffu, any != 0 && mf >= 0);
        if (warp == 1) {
            for (int rr = lane; rr < R; rr += 32) sh.chg[par ^ 1][rr] = 0;
            if (lane == 0) sh.first[par ^ 1] = INT_MAX;
        }
        fin_h = max(fin_h, fin_x);
        lo = any ? max(lo + 1, min(mf + 1, T)) : T;
        fin_x = max(fin_x, lo);
        if (any && k < cap) continue;
        if (any && cap < T) status = JS_NOT_CONVERGED;
        break;
    }
    const bool alive = mf >= 0;
    // results: symbols or states of the own positions; counts by the first CTA of the cluster
    for (int i = tid; alive && i < own * nrow; i += NTH) {
        const int rr = i / own, j = i - rr * own;
        const size_t at = (size_t)(row0 + rr) * T + c + CS * j;
        if constexpr (REAL) r.xr[at] = xs[j * RS + rr];
        else r.x[at] = (uint8_t)xs[j * RS + rr];
    }
    if (c == 0 && r.out_iters && alive)
        for (int rr = tid; rr < nrow; rr += NTH) r.out_iters[row0 + rr] = sh.count[rr];
    if (lane == 0) {
        if constexpr (!CL) {
            atomicAdd(&sh.tiles, tiles);
            atomicAdd(&sh.skipped, skipped);
        } else {
            peer_add(peer_addr(smem_u32(&sh.tiles), 0), tiles);
            peer_add(peer_addr(smem_u32(&sh.skipped), 0), skipped);
        }
    }
    if (gave_up)
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);      // weights still on their way land before shared memory goes away
    if constexpr (CL) cluster_sync();          // no CTA leaves while others may still read its flags
    else __syncthreads();
    if (tid == 0 && c == 0) cluster_report(r.words, (int)(blockIdx.x >> csh), alive, status, k, fin_x, sh.tiles, k, sh.skipped);
}

// packed weights of CTA c: per layer [K][ncs] (column i = unit of the i-th own output), then biases, then degrees
__global__ void pack_small_weights(const MadeDev m, const SmallDev s, float *pack)
{
    const int c = blockIdx.y;
    float *dst = pack + (size_t)c * s.pack_floats;
    const int C = m.C;
    for (int l = 0; l <= m.L; ++l) {
        const int per = l == m.L ? C : 1;        // outputs of a position stay together
        const int K = m.n[l], nc = s.nc[l], ncs = s.ncs[l];
        const int mine = l == m.L ? ((m.T - c + s.CS - 1) / s.CS) * C : (m.n[l + 1] - c + s.CS - 1) / s.CS;
        auto unit = [&](int i) { return (c + s.CS * (i / per)) * per + i % per; };
        const float *W = (const float *)m.W[l];
        for (int at = blockIdx.x * blockDim.x + threadIdx.x; at < pad_k(K) * ncs; at += gridDim.x * blockDim.x) {
            const int i = at % ncs, k = at / ncs;
            dst[s.w_off[l] + at] = i < mine && k < K ? W[(size_t)unit(i) * K + k] : 0.0f;
        }
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nc; i += gridDim.x * blockDim.x) {
            dst[s.b_off[l] + i] = i < mine ? m.bias[l][unit(i)] : 0.0f;
            // degree and last live input (continuous states), 16 bits each: weights for more inputs do not fit a CTA.  An output
            // beyond the CTA's own ones is never live and limits nobody.
            uint32_t v = 0xffffu << 16;
            if (i < mine) {
                const int dg = m.deg[l + 1][unit(i)];
                int ke = K;
                if (C == 2)
                    while (ke > 0 && !(l == m.L ? m.deg[l][ke - 1] < dg : m.deg[l][ke - 1] <= dg)) --ke;
                v = (uint32_t)dg | (uint32_t)ke << 16;
            }
            reinterpret_cast<uint32_t *>(dst + s.d_off[l])[i] = v;
        }
    }
}

typedef void (*SmallKernelFn)(const MadeDev, const SmallDev, const RunArgs, const int);
template <bool REAL, bool CL>
SmallKernelFn small_kernel_rg(int rg)
{
    return rg == 1 ? made_small_kernel<1, REAL, CL> : rg == 2 ? made_small_kernel<2, REAL, CL> : made_small_kernel<4, REAL, CL>;
}
SmallKernelFn small_kernel_of(int rg, bool real, bool cl)
{
    return real ? (cl ? small_kernel_rg<true, true>(rg) : small_kernel_rg<true, false>(rg))
                : (cl ? small_kernel_rg<false, true>(rg) : small_kernel_rg<false, false>(rg));
}
int rows_group(int R) { return R == 1 ? 1 : R == 2 ? 2 : 4; }

// samples per cluster of a call: as few as spread the batch over the GPU, bounded by what shared memory holds
int rows_of(const js_model *mo, int batch)
{
    const SmallDev &s = mo->small;
    const int clusters = std::max(1, s.sms * 7 / (8 * s.CS));       // clusters that fit at a time (GPCs are not multiples of CS)
    int R = std::min(RMAX, (batch + clusters - 1) / clusters);
    auto fits = [&](int q) {
        const int g = rows_group(q), rs = (q + g - 1) / g * g;
        return small_layout(mo->made, s, rs).total * 4 <= SMEM_MAX;
    };
    while (R > 1 && !fits(R)) --R;
    return fits(R) && (batch + R - 1) / R <= JS_MAX_CLUSTERS ? R : 0;
}

}  // namespace

// Decides whether the model is served by this kernel and packs its weights.  The cluster size grows with the widest
// layer, so that a CTA has one or two warps' worth of units per layer and a layer is a short chain; the weights of a
// CTA have to fit its shared memory beside at least one sample's activations.  Larger models stay with the
// grid-wide kernel, which streams the weights.
int js_small_prepare(js_model *mo)
{
    const MadeDev &v = mo->made;
    SmallDev &s = mo->small;
    mo->small_ok = 0;
    if (v.prec != JS_F32 || !(v.C == 1 || v.C == 2)) return 0;
    int widest = v.T * v.C;
    for (int l = 0; l <= v.L; ++l) widest = std::max(widest, v.n[l + 1]);
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&s.sms, cudaDevAttrMultiProcessorCount, dev);
    for (int CS = widest <= 96 ? 1 : widest <= 192 ? 2 : widest <= 384 ? 4 : 8; CS <= 8; CS *= 2) {
        s.CS = CS;
        s.cs_log2 = CS == 1 ? 0 : CS == 2 ? 1 : CS == 4 ? 2 : 3;
        int at = 0;
        for (int l = 0; l <= v.L; ++l) {
            s.nc[l] = l == v.L ? ((v.T + CS - 1) / CS) * v.C : (v.n[l + 1] + CS - 1) / CS;
            s.ncs[l] = s.nc[l];
            s.w_off[l] = at; at += pad_k(v.n[l]) * s.ncs[l];
            at = (at + 3) / 4 * 4;
            s.b_off[l] = at; at += s.nc[l];
            s.d_off[l] = at; at += s.nc[l];
        }
        s.pack_floats = (at + 3) / 4 * 4;
        static_assert(190 * 1024 / 4 < 0x10000, "degrees and inputs in 16 bits");
        if (small_layout(v, s, 1).total * 4 > SMEM_MAX || s.pack_floats * 4 > 190 * 1024) continue;
        // last live input of every block of 32 own outputs, over all CTAs of the cluster
        for (int l = 0; l <= v.L; ++l) {
            const std::vector<int> &din = mo->host_deg[l], &dout = mo->host_deg[l + 1];
            const int per = l == v.L ? v.C : 1;
            for (int b = 0; b < SMALL_KENDS; ++b) s.kend[l][b] = 0;
            for (int u = 0; u < v.n[l + 1]; ++u) {
                const int b = std::min(SMALL_KENDS - 1, ((u / per / CS) * per + u % per) / 32);
                int ke = v.n[l];
                while (ke > s.kend[l][b] && !(l == v.L ? din[ke - 1] < dout[u] : din[ke - 1] <= dout[u])) --ke;
                s.kend[l][b] = std::max(s.kend[l][b], ke);
            }
        }
        void *p = nullptr;
        if (cudaMalloc(&p, (size_t)CS * s.pack_floats * 4) != cudaSuccess) return JS_ERR_CUDA;
        mo->allocs.push_back(p);
        pack_small_weights<<<dim3(32, CS), 256>>>(v, s, (float *)p);
        if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) return JS_ERR_CUDA;
        s.pack = (const float *)p;
        for (int rg : {1, 2, 4})
            if (cudaFuncSetAttribute(small_kernel_of(rg, v.C == 2, CS > 1), cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX) != cudaSuccess) {
                cudaGetLastError();
                return 0;
            }
        mo->small_ok = 1;
        return 1;
    }
    return 0;
}

bool js_small_serves(const js_model *mo, const RunArgs &r)
{
    return mo->small_ok && r.kmode == KM_JACOBI && (r.real != 0) == (mo->made.C == 2) && rows_of(mo, r.batch) > 0;
}

int js_launch_made_small(const js_model *mo, const RunArgs &r, cudaStream_t stream, ClusterWork *work)
{
    const SmallDev &s = mo->small;
    const int R = rows_of(mo, r.batch), rg = rows_group(R), RS = (R + rg - 1) / rg * rg;
    *work = ClusterWork{(r.batch + R - 1) / R, 0, 0, 0};
    memset(mo->h_words, 0, 2 * sizeof(unsigned long long) * (size_t)work->clusters);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(work->clusters * s.CS));
    cfg.blockDim = dim3(NTH);
    cfg.dynamicSmemBytes = (size_t)small_layout(mo->made, s, RS).total * 4;
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)s.CS;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = s.CS > 1 ? 1 : 0;
    return (int)cudaLaunchKernelEx(&cfg, small_kernel_of(rg, r.real != 0, s.CS > 1), mo->made, s, r, R);
}
