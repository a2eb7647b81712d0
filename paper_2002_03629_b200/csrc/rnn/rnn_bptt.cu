// Back-propagation through time of a one-layer recurrent network as a triangular system (arXiv 2002.03629,
// Section 5.1; appendix "Backpropagation"): forward pass, exact back-substitution, truncated Jacobi
// iterations (Algorithm 1) and the parameter gradients.  fp32 fused multiply-adds in a fixed order.
//
// Forward pass and back-substitution are chains of T matrix-vector products: what counts is the latency of one
// step, so a step is spread over four threads per component (see the kernels).  A Jacobi iteration has parallel slack,
// all T states at once, a [T x H] x [H x H] product per iteration: a register-tiled product out of shared memory in
// which the iterate (premultiplied by the activation derivative and shifted by one step) and the weights stay; a small
// batch shares each sequence among the CTAs of a cluster, which hand over one row per iteration.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <cstdio>

#include "../../../include/rnn_bptt.h"

namespace {

constexpr int MT = RNN_MAX_T, MH = RNN_MAX_H, MIO = RNN_MAX_IO;

char g_err[256] = "";

int launch_status()
{
    const cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) return RNN_OK;
    snprintf(g_err, sizeof g_err, "%s", cudaGetErrorString(e));
    return RNN_ERR_CUDA;
}

// Four neighbouring floats of global memory.  VEC: every pointer of the call lies on 16 bytes (rows do then too, H being a
// multiple of 4) and they move as one piece; otherwise (views into a larger buffer, say) one by one.
template <bool VEC>
__device__ __forceinline__ float4 ldg4(const float *p)
{
    if constexpr (VEC) return __ldg(reinterpret_cast<const float4 *>(p));
    return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
}
template <bool VEC>
__device__ __forceinline__ void stg4(float *p, float4 v)
{
    if constexpr (VEC) { *reinterpret_cast<float4 *>(p) = v; return; }
    p[0] = v.x; p[1] = v.y; p[2] = v.z; p[3] = v.w;
}

// ------------------------------------------------------------------ one step of a chain
// A matrix-vector product with a 128 x 128 matrix in the registers of 128 threads.  Thread (warp w, lane) holds a 4 x 32
// tile: the four outputs 4 g .. 4 g + 3, g = 8 w + lane % 8, by the inputs k = 16 m + 4 q + e (m < 8, e < 4), q = lane / 8;
// the inputs come from shared memory, eight 16-byte loads per thread.  (Lanes of a warp read four different pieces, eight
// neighbouring lanes the same one: such a load takes two cycles of the shared-memory pipe.  With the four pieces in turn
// over the lanes it takes four, and more threads with smaller tiles pay for more loads: both were slower.)  Three shuffles
// add the quarters and leave output 4 g + q to each thread, so what follows - an activation and its derivative - is
// computed once per output.
constexpr int CT = 128;          // threads

struct MatvecTile {
    float w[4][MH / 4];
};
__device__ __forceinline__ void tile_dot(const MatvecTile &t, const float *v, int q, float (&out)[4])
{
    const float4 *p = reinterpret_cast<const float4 *>(v) + q;
    float c0[4], c1[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) { c0[u] = 0.0f; c1[u] = 0.0f; }
#pragma unroll
    for (int m = 0; m < MH / 16; ++m) {
        const float4 x = p[4 * m];
        // eight chains in turn: a multiply-add never waits for the one before it
#pragma unroll
        for (int u = 0; u < 4; ++u) c0[u] = fmaf(t.w[u][4 * m], x.x, c0[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) c1[u] = fmaf(t.w[u][4 * m + 1], x.y, c1[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) c0[u] = fmaf(t.w[u][4 * m + 2], x.z, c0[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) c1[u] = fmaf(t.w[u][4 * m + 3], x.w, c1[u]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) out[u] = c0[u] + c1[u];
}
// sums over the four lanes q = 0..3 of a group; lane q keeps the sum of v[q]
__device__ __forceinline__ float scatter_sum(const float (&v)[4], int lane)
{
    const bool b1 = lane & 16, b0 = lane & 8;
    const float r0 = __shfl_xor_sync(0xffffffffu, b1 ? v[0] : v[2], 16);
    const float r1 = __shfl_xor_sync(0xffffffffu, b1 ? v[1] : v[3], 16);
    const float k0 = (b1 ? v[2] : v[0]) + r0, k1 = (b1 ? v[3] : v[1]) + r1;
    return (b0 ? k1 : k0) + __shfl_xor_sync(0xffffffffu, b0 ? k0 : k1, 8);
}

template <int N>
struct Count {
    static constexpr int value = N;
};

// ------------------------------------------------------------------ forward
// Two groups of 128 threads.  The first carries the chain and nothing else: product, softplus, new state (0.33 us per
// step).  The second follows it with what does not feed back.  Its four warps take the steps in turn, lane = four units,
// and each spreads the work on its step over four iterations, which keeps every iteration shorter than the chain's:
//   0  state to global memory, the derivative's exponential     1  outputs y_t, residuals, direct gradient l_t, loss
//   2  l_t and derivative to global memory                       3  input part W_x x + b of the next step of the chain
// One block barrier per iteration keeps the groups together.  With all of it between two steps of the chain a step took
// 0.57 us; with every warp of the second group doing a quarter of each kind of work in every iteration, 0.8 us.
// T = 100, H = 128, one input and output (B200): batch 1 86 -> 40 us, batch 592 209 -> 118 us; 16 inputs and outputs, T = 128:
// 200 -> 132 and 613 -> 326 us.
// NS sequences per CTA: the weights in registers serve NS independent chains, whose latencies overlap.  MANY: sums of several
// outputs go through the shuffles side by side; for one output and few inputs the plain loop is the shorter step (T = 100,
// batch 1: 40 us against 46; two outputs 52 against 48).
template <int NS, bool VEC, bool MANY>
__global__ void __launch_bounds__(2 * CT, 1)
rnn_forward_kernel(const float *__restrict__ Wh, const float *__restrict__ Wx, const float *__restrict__ b,
                   const float *__restrict__ Wo, const float *__restrict__ bo, const float *__restrict__ x,
                   const float *__restrict__ r, int B, int T, int H, int d_in, int d_out, float *__restrict__ h,
                   float *__restrict__ d, float *__restrict__ l, float *__restrict__ loss)
{
    __shared__ __align__(16) float hs[2][NS][MH];       // the states of two steps, zero beyond H
    __shared__ __align__(16) float as[2][NS][MH];       // their pre-activations
    __shared__ __align__(16) float xin[2][NS][MH];                  // input parts of two steps
    __shared__ float red[NS][CT / 32], bos[MIO];
    extern __shared__ __align__(16) float dyn[];        // Wo [d_out][MH], Wx [d_in][MH], x [NS][T d_in], r [NS][T d_out]
    float *wos = dyn, *wxs = wos + d_out * MH, *xs = wxs + d_in * MH, *rs = xs + NS * T * d_in;
    const int tid = threadIdx.x, lane = tid & 31, warp = (tid >> 5) & 3, seq0 = blockIdx.x * NS;
    const int ns = min(NS, B - seq0);
    for (int p = tid; p < d_out * MH; p += 2 * CT) {
        const int c = p / MH, i = p % MH;
        wos[p] = i < H ? Wo[(size_t)c * H + i] : 0.0f;
    }
    if (tid < d_out) bos[tid] = bo[tid];
    for (int p = tid; p < d_in * MH; p += 2 * CT) {
        const int c = p / MH, i = p % MH;
        wxs[p] = i < H ? Wx[(size_t)i * d_in + c] : 0.0f;
    }
    for (int p = tid; p < ns * T * d_in; p += 2 * CT) xs[p] = x[(size_t)seq0 * T * d_in + p];
    for (int p = tid; p < ns * T * d_out; p += 2 * CT) rs[p] = r[(size_t)seq0 * T * d_out + p];
    for (int p = tid; p < NS * MH; p += 2 * CT) (&hs[0][0][0])[p] = 0.0f;
    if (tid < CT) {
        const int g = 8 * warp + (lane & 7), q = lane >> 3, j = 4 * g + q;      // j: this thread's hidden unit
        const bool on = j < H;
        MatvecTile w;
#pragma unroll
        for (int m = 0; m < MH / 16; ++m) {
            const int k = 16 * m + 4 * q;               // H is a multiple of 4
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 v = (4 * g < H && k < H) ? ldg4<VEC>(Wh + (size_t)(4 * g + u) * H + k) : make_float4(0, 0, 0, 0);
                w.w[u][4 * m] = v.x; w.w[u][4 * m + 1] = v.y; w.w[u][4 * m + 2] = v.z; w.w[u][4 * m + 3] = v.w;
            }
        }
        __syncthreads();                                // the tables are there
        __syncthreads();                                // and the first step's input part
        for (int it = 0; it < T + 3; ++it) {
            if (it < T) {
                const int cur = it & 1;
#pragma unroll
                for (int n = 0; n < NS; ++n) {
                    float v[4];
                    tile_dot(w, hs[cur][n], q, v);
                    const float a = xin[cur][n][j] + scatter_sum(v, lane);
                    hs[cur ^ 1][n][j] = on ? fmaxf(a, 0.0f) + log1pf(expf(-fabsf(a))) : 0.0f;
                    as[cur][n][j] = a;
                }
            }
            __syncthreads();
        }
    } else {
        const int j4 = 4 * lane;                         // this lane's units (H is a multiple of 4)
        const bool on = j4 < H;
        const float4 b4 = on ? ldg4<VEC>(b + j4) : make_float4(0, 0, 0, 0);
        float part[NS];
        float4 hv[NS], lv[NS], nv[NS], ev[NS];           // of this warp's step: state, direct gradient, sigmoid as a fraction
#pragma unroll
        for (int n = 0; n < NS; ++n) { part[n] = 0.0f; hv[n] = lv[n] = nv[n] = ev[n] = make_float4(0, 0, 0, 0); }
        auto fma4 = [](float x, float4 w, float4 a) {
            return make_float4(fmaf(w.x, x, a.x), fmaf(w.y, x, a.y), fmaf(w.z, x, a.z), fmaf(w.w, x, a.w));
        };
        auto input_part = [&](int t) {
            float4 a[NS];
#pragma unroll
            for (int n = 0; n < NS; ++n) a[n] = b4;
#pragma unroll MANY ? 4 : 1
            for (int c = 0; c < d_in; ++c) {
                const float4 wv = *reinterpret_cast<const float4 *>(wxs + c * MH + j4);
#pragma unroll
                for (int n = 0; n < NS; ++n) a[n] = fma4(xs[(n * T + t) * d_in + c], wv, a[n]);
            }
#pragma unroll
            for (int n = 0; n < NS; ++n) *reinterpret_cast<float4 *>(&xin[t & 1][n][j4]) = a[n];
        };
        // Outputs c .. c + G - 1 of step t for all sequences: their sums over the units go through the shuffles side by side
        // (a shuffle's latency is 25 cycles and a sum takes five, one after the other).
        auto outputs = [&](auto g_, int t, int c) {
            constexpr int G = decltype(g_)::value;
            float4 wv[G];
            float y[NS][G];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                wv[g] = *reinterpret_cast<const float4 *>(wos + (c + g) * MH + j4);
#pragma unroll
                for (int n = 0; n < NS; ++n)
                    y[n][g] = fmaf(wv[g].w, hv[n].w, fmaf(wv[g].z, hv[n].z, fmaf(wv[g].y, hv[n].y, wv[g].x * hv[n].x)));
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1)
#pragma unroll
                for (int n = 0; n < NS; ++n)
#pragma unroll
                    for (int g = 0; g < G; ++g) y[n][g] += __shfl_xor_sync(0xffffffffu, y[n][g], off);
#pragma unroll
            for (int g = 0; g < G; ++g)
#pragma unroll
                for (int n = 0; n < NS; ++n) {
                    const float res = y[n][g] + bos[c + g] - rs[(n * T + t) * d_out + c + g];
                    lv[n] = fma4(res, wv[g], lv[n]);
                    part[n] = fmaf(0.5f * res, res, part[n]);
                }
        };
        // derivative of softplus from the pre-activation: the exponential's argument is never positive
        auto fraction = [](float a, float &num, float &den) {
            const float e = expf(-fabsf(a));
            num = a >= 0.0f ? 1.0f : e;
            den = 1.0f + e;
        };
        __syncthreads();
        if (warp == 0) input_part(0);
        __syncthreads();
        for (int it = 0; it < T + 3; ++it) {
            const int phase = (it - warp) & 3, t = it - 1 - phase;       // this warp's step
            if (phase == 3) {
                if (it + 1 < T) input_part(it + 1);
            } else if (t >= 0 && t < T) {
                const size_t o = ((size_t)seq0 * T + t) * H + j4, next = (size_t)T * H;
                if (phase == 0) {
#pragma unroll
                    for (int n = 0; n < NS; ++n) {
                        hv[n] = *reinterpret_cast<const float4 *>(&hs[it & 1][n][j4]);
                        const float4 a = *reinterpret_cast<const float4 *>(&as[t & 1][n][j4]);
                        fraction(a.x, nv[n].x, ev[n].x);
                        fraction(a.y, nv[n].y, ev[n].y);
                        fraction(a.z, nv[n].z, ev[n].z);
                        fraction(a.w, nv[n].w, ev[n].w);
                        if (on && n < ns) stg4<VEC>(h + o + n * next, hv[n]);
                    }
                } else if (phase == 1) {
                    constexpr int GM = NS <= 2 ? 4 : 2;          // sums side by side: six to eight, four for one sequence
#pragma unroll
                    for (int n = 0; n < NS; ++n) lv[n] = make_float4(0, 0, 0, 0);
                    int c = 0;
                    if constexpr (MANY) {
#pragma unroll 1
                        for (; c + GM <= d_out; c += GM) outputs(Count<GM>(), t, c);
                        if (GM == 4 && c + 2 <= d_out) { outputs(Count<2>(), t, c); c += 2; }
                        if (c < d_out) outputs(Count<1>(), t, c);
                    } else {
#pragma unroll 1
                        for (; c < d_out; ++c) outputs(Count<1>(), t, c);
                    }
                } else if (on) {
#pragma unroll
                    for (int n = 0; n < NS; ++n)
                        if (n < ns) {
                            stg4<VEC>(l + o + n * next, lv[n]);
                            stg4<VEC>(d + o + n * next, make_float4(nv[n].x / ev[n].x, nv[n].y / ev[n].y, nv[n].z / ev[n].z, nv[n].w / ev[n].w));
                        }
                }
            }
            __syncthreads();
        }
#pragma unroll
        for (int n = 0; n < NS; ++n)
            if (lane == 0) red[n][warp] = part[n];
    }
    __syncthreads();
    if (tid < ns) {
        float s = 0.0f;
        for (int i = 0; i < CT / 32; ++i) s += red[tid][i];
        loss[seq0 + tid] = s;
    }
}

// ------------------------------------------------------------------ exact back-substitution
// The same product with the transposed weights.  A step is shorter than a trip to L2, so the steps' l and d come in
// chunks of SC through two shared-memory buffers, the next chunk's copies in flight while one is worked off.
// T = 100, H = 128 (B200): batch 1 39 -> 25 us, batch 592 110 -> 64 us.
constexpr int SC = 16;

template <bool VEC>
__device__ __forceinline__ void copy4_async(float *dst, const float *src, bool in)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(dst);
    if constexpr (VEC) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(a), "l"(src), "r"(in ? 16 : 0) : "memory");
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(a + 4u * e), "l"(src + e), "r"(in ? 4 : 0) : "memory");
    }
}

template <int NS, bool VEC>
__global__ void __launch_bounds__(CT, NS == 1 ? 3 : 2)
rnn_bptt_sequential_kernel(const float *__restrict__ Wh, const float *__restrict__ l, const float *__restrict__ d,
                           int B, int T, int H, float *__restrict__ s)
{
    extern __shared__ __align__(16) float ring[];       // [NS][2][l, d][SC][MH]; row g of a chunk: step t0 - g
    __shared__ __align__(16) float u[NS][2][MH];        // d_{t+1} * s_{t+1}
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, seq0 = blockIdx.x * NS;
    const int g = 8 * warp + (lane & 7), q = lane >> 3, i = 4 * g + q;
    const bool on = i < H;
    MatvecTile w;
#pragma unroll
    for (int m = 0; m < MH / 4; ++m) {
        const int k = 16 * (m >> 2) + 4 * q + (m & 3);
        const float4 v = (4 * g < H && k < H) ? ldg4<VEC>(Wh + (size_t)k * H + 4 * g) : make_float4(0, 0, 0, 0);
        w.w[0][m] = v.x; w.w[1][m] = v.y; w.w[2][m] = v.z; w.w[3][m] = v.w;
    }
    auto chunk = [&](int n, int buf, int which) { return ring + (((n * 2 + buf) * 2 + which) * SC) * MH; };
    auto fetch = [&](int t0, int buf) {
        for (int p = tid; p < SC * MH / 4; p += CT) {
            const int r = p / (MH / 4), c = (p % (MH / 4)) * 4, t = t0 - r;
#pragma unroll
            for (int n = 0; n < NS; ++n) {
                const bool in = t >= 0 && c < H && seq0 + n < B;
                const size_t at = in ? ((size_t)(seq0 + n) * T + t) * H + c : 0;
                copy4_async<VEC>(chunk(n, buf, 0) + r * MH + c, l + at, in);
                copy4_async<VEC>(chunk(n, buf, 1) + r * MH + c, d + at, in);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int n = 0; n < NS; ++n) { u[n][0][tid] = 0.0f; u[n][1][tid] = 0.0f; }
    fetch(T - 1, 0);
    for (int t0 = T - 1, buf = 0; t0 >= 0; t0 -= SC, buf ^= 1) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                                // the chunk is here, and its predecessor has been read
        if (t0 >= SC) fetch(t0 - SC, buf ^ 1);
        const int ng = min(SC, t0 + 1);
        for (int e = 0; e < ng; ++e) {
            const int t = t0 - e;
#pragma unroll
            for (int n = 0; n < NS; ++n) {
                float v[4];
                tile_dot(w, u[n][(t + 1) & 1], q, v);
                const float acc = chunk(n, buf, 0)[e * MH + i] + scatter_sum(v, lane);
                u[n][t & 1][i] = on ? chunk(n, buf, 1)[e * MH + i] * acc : 0.0f;
                if (on && seq0 + n < B) s[((size_t)(seq0 + n) * T + t) * H + i] = acc;
            }
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------------ Jacobi iterations
// A sequence is solved by a cluster of csz CTAs (1 where the batch fills the GPU); CTA c owns the steps
// [c rpc, (c + 1) rpc).  V[k][r] = d_{t+1}[k] * s_{t+1}[k] of the current iterate for t = c rpc + r (zero where t + 1 >= T
// or k >= H), so that  s_new[t][i] = l[t][i] + sum_k V[k][r] * W_h[k][i];  the value of a CTA's first step belongs to the
// CTA before it.  A thread owns a tile of 4 steps x 8 components.  Neighbouring lanes take the same columns and
// neighbouring tile rows: a 16-byte shared-memory load then takes two cycles for a warp instead of the four it takes when
// neighbouring lanes read sixteen pieces of a weight row, and the product is bound by its multiply-adds (8 cycles per
// warp and k against 6).  Steps are laid out without padding to 128, for which 100 steps paid 28 %.  Row k of V starts at
// vrow(k): the four floats of slack after every fourth row spread the transposed stores over the banks.
// Three forms:
//   JAC_PAIR   two sequences per CTA, each with its own threads and its own (named) barrier, for batches beyond one per
//              SM: one sequence's stores and waits pass while the other multiplies, and 26 warps balance better over
//              four schedulers than 13.  One buffer for V, refilled between two barriers.
//   JAC_ONE    one sequence per CTA, two buffers.
//   JAC_SPLIT  one sequence per cluster: a CTA has so few steps that the k range is cut into four parts for as many
//              thread groups; part p adds the four sums of every tile's row p (in order) and finishes it.
// After k iterations the last k states are final (Proposition 1), and a repeated evaluation would give the same bits:
// they are stored when they become final and not computed again; their warps drop out.
// Bound: issue of fp32 multiply-adds (a plain FFMA loop reaches 61 TFLOP/s on this GPU).  T = 100, H = 128, 20 iterations:
// batch 1 285 -> 73 us (cluster of 8), batch 592 1148 -> 895 us (40 TFLOP/s of what is still computed).
enum { JAC_PAIR = 0, JAC_ONE = 1, JAC_SPLIT = 2 };

__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ int vrow(int k, int VS) { return k * VS + (k & ~3); }

template <int FORM, int NT, bool VEC>
__global__ void __launch_bounds__(NT, 1)
rnn_bptt_jacobi_kernel(const float *__restrict__ Wh, const float *__restrict__ l, const float *__restrict__ d,
                       int B, int T, int H, int n_iters, const float *__restrict__ s0, float *__restrict__ s, int csz, int rpc)
{
    constexpr int TR = 4, KS = FORM == JAC_SPLIT ? TR : 1, NSQ = FORM == JAC_PAIR ? 2 : 1;
    constexpr bool DB = FORM != JAC_PAIR;
    extern __shared__ __align__(16) float sm[];
    const int tid = threadIdx.x, nth = blockDim.x;
    const int seq0 = blockIdx.x / csz * NSQ, c = FORM == JAC_SPLIT ? blockIdx.x % csz : 0;
    const int NG = (H + 7) / 8, VS = (rpc + 3) / 4 * 4, VB = H * (VS + 1);      // VB: one buffer of a sequence's iterate
    float *W = sm;                                       // [H][MH]: component 4 ig + e at 4 ig + e, 4 (ig + NG) + e at 64 + 4 ig + e
    float *V = sm + (size_t)H * MH;                      // [NSQ][1 or 2][VB]
    float *part = V + (size_t)(NSQ * (DB ? 2 : 1)) * VB; // JAC_SPLIT: [4 parts][4 rows][8][threads of a part]
    const int t0 = c * rpc, nr = max(0, min(rpc, T - t0));
    for (int p = tid; p < NSQ * (DB ? 2 : 1) * VB; p += nth) V[p] = 0.0f;
    for (int p = tid; p < H * 2 * NG; p += nth) {
        const int k = p / (2 * NG), g = p - k * 2 * NG;
        *reinterpret_cast<float4 *>(W + (size_t)k * MH + (g < NG ? 4 * g : 64 + 4 * (g - NG))) =
            4 * g < H ? ldg4<VEC>(Wh + (size_t)k * H + 4 * g) : make_float4(0, 0, 0, 0);
    }
    if (n_iters <= 0) {
        for (int n = 0; n < NSQ && seq0 + n < B; ++n)
            for (int p = tid; p < nr * H; p += nth) {
                const size_t at = (size_t)(seq0 + n) * T * H + (size_t)t0 * H + p;
                s[at] = s0 != nullptr ? s0[at] : 0.0f;
            }
        return;                                          // every CTA of the cluster leaves here
    }
    // thread = (sequence n or part ks, tile row tg, column group ig); a sequence's threads are whole warps
    const int tgs = ((rpc + TR - 1) / TR + 1) / 2 * 2, per_seq = tgs * NG;
    const int grp = FORM == JAC_ONE ? nth : nth / (NSQ * KS), gi = FORM == JAC_ONE ? 0 : tid / grp, ti = tid - gi * grp;
    const int n = FORM == JAC_PAIR ? gi : 0, ks = FORM == JAC_SPLIT ? gi : 0;
    const int ig = (ti >> 1) % NG, tg = (ti >> 1) / NG * 2 + (ti & 1), r0 = tg * TR;
    const bool here = ti < per_seq && seq0 + n < B;
    const float *lp = l + (size_t)(seq0 + n) * T * H, *dp = d + (size_t)(seq0 + n) * T * H;
    float *sp = s + (size_t)(seq0 + n) * T * H;
    float *Vn = V + n * VB;
    __syncthreads();
    if (s0 != nullptr)
        for (int m = 0; m < NSQ && seq0 + m < B; ++m)
            for (int p = tid; p < nr * H; p += nth) {
                const int r = p / H, k = p - r * H, t = t0 + r + 1;
                const size_t at = (size_t)(seq0 + m) * T * H + (size_t)t * H + k;
                if (t < T) V[m * VB + vrow(k, VS) + r] = d[at] * s0[at];
            }
    // the CTA before this one: where the value of our first step goes
    uint32_t prev = 0;
    if (FORM == JAC_SPLIT && c > 0) {
        const uint32_t mine = (uint32_t)__cvta_generic_to_shared(Vn);
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(prev) : "r"(mine), "r"(c - 1));
    }
    auto load4 = [&](const float *src, int r, int hf) {          // l or d of step t0 + r, components 4 (ig + hf NG) ..
        const int i = 4 * (ig + hf * NG);
        return r < nr && i < H ? ldg4<VEC>(src + (size_t)(t0 + r) * H + i) : make_float4(0, 0, 0, 0);
    };
    float4 lk[2], dk[2];                                 // JAC_SPLIT: l and d of this part's row
    if (FORM == JAC_SPLIT && here)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) { lk[hf] = load4(lp, r0 + ks, hf); dk[hf] = load4(dp, r0 + ks, hf); }
    if (FORM == JAC_SPLIT) cluster_barrier();
    else __syncthreads();
    const int iters = min(n_iters, T), kc = (H / 4 + KS - 1) / KS * 4;     // k per part (H is a multiple of 4)
    const int k0 = ks * kc, k1 = min(H, k0 + kc);
    for (int it = 0; it < iters; ++it) {
        const int cur = DB ? (it & 1) * VB : 0, nxt = DB ? VB - cur : 0;
        const int live = min(nr, T - it - t0);           // steps beyond are final
        const bool work = here && r0 < live;             // (pairs of tile rows drop out of the warps together)
        const bool last = it + 1 == iters;
        // a finished row: to global memory when it is final, to the next iterate unless this was the last iteration
        auto finish = [&](int r, const float (&v)[8], const float4 (&dv)[2]) {
            const int t = t0 + r;
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const int i = 4 * (ig + hf * NG);
                if (i >= H) continue;
                if (last || t == T - 1 - it)
                    stg4<VEC>(sp + (size_t)t * H + i, make_float4(v[4 * hf], v[4 * hf + 1], v[4 * hf + 2], v[4 * hf + 3]));
                if (last) continue;
                const float dd[4] = {dv[hf].x, dv[hf].y, dv[hf].z, dv[hf].w};
                const int row = nxt + vrow(i, VS);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float val = dd[e] * v[4 * hf + e];
                    if (r >= 1) Vn[row + e * VS + r - 1] = val;
                    else if (FORM == JAC_SPLIT && c > 0)
                        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(prev + 4u * (uint32_t)(row + e * VS + rpc - 1)), "f"(val) : "memory");
                }
            }
        };
        float acc[TR][8];
        if (work) {
#pragma unroll
            for (int rr = 0; rr < TR; ++rr)
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const float4 a = FORM == JAC_SPLIT ? make_float4(0, 0, 0, 0) : load4(lp, r0 + rr, hf);
                    acc[rr][4 * hf] = a.x; acc[rr][4 * hf + 1] = a.y; acc[rr][4 * hf + 2] = a.z; acc[rr][4 * hf + 3] = a.w;
                }
            const float *vp = Vn + cur + r0 + vrow(k0, VS), *wp = W + 4 * ig + (size_t)k0 * MH;
            for (int k = k0; k < k1; k += 4, vp += 4 * VS + 4, wp += 4 * MH)
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const float4 a = *reinterpret_cast<const float4 *>(vp + kk * VS);
                    const float4 w0 = *reinterpret_cast<const float4 *>(wp + kk * MH);
                    const float4 w1 = *reinterpret_cast<const float4 *>(wp + kk * MH + 64);
                    const float av[TR] = {a.x, a.y, a.z, a.w};
                    const float wv[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
                    for (int rr = 0; rr < TR; ++rr)
#pragma unroll
                        for (int e = 0; e < 8; ++e) acc[rr][e] = fmaf(av[rr], wv[e], acc[rr][e]);
                }
            if (FORM == JAC_SPLIT)
#pragma unroll
                for (int e = 0; e < 32; ++e) part[(ks * 32 + e) * grp + ti] = acc[e >> 3][e & 7];
        }
        if (FORM == JAC_SPLIT) {
            __syncthreads();                             // the parts' sums are there
            if (work && r0 + ks < live) {
                float v[8] = {lk[0].x, lk[0].y, lk[0].z, lk[0].w, lk[1].x, lk[1].y, lk[1].z, lk[1].w};
#pragma unroll
                for (int p = 0; p < KS; ++p)
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[e] += part[(p * 32 + ks * 8 + e) * grp + ti];
                finish(r0 + ks, v, dk);
            }
            cluster_barrier();
        } else {
            if (FORM == JAC_PAIR) asm volatile("bar.sync %0, %1;" ::"r"(1 + n), "r"(grp) : "memory");     // V has been read
            if (work)
#pragma unroll
                for (int rr = 0; rr < TR; ++rr)
                    if (r0 + rr < live) {
                        const float4 dv[2] = {load4(dp, r0 + rr, 0), load4(dp, r0 + rr, 1)};
                        finish(r0 + rr, acc[rr], dv);
                    }
            if (FORM == JAC_PAIR) asm volatile("bar.sync %0, %1;" ::"r"(1 + n), "r"(grp) : "memory");
            else __syncthreads();
        }
    }
}

// ------------------------------------------------------------------ parameter gradients
// dWh = sum_t g_t h_{t-1}^T with g_t = d_t * s_t: a [128 x T] x [T x 64] product per CTA (two CTAs per sequence), 128
// threads with 8 x 8 outputs each (rows 4 ty.. and 64 + 4 ty.., columns 4 tx.. and 32 + 4 tx..).  The steps come in
// chunks of GC through two small shared-memory buffers, the next chunk's loads in registers while one is multiplied, so
// that several CTAs share an SM and one's loads and stores hide behind another's arithmetic; before, a CTA held all
// steps (128 KB) and its three stages ran one after another.  db and dWx ride along: the same sums with 1 and x_t on
// the right.  T = 100, H = 128 (B200): batch 1 31 -> 17 us, batch 592 191 -> 79 us (60 MB in, 39 MB out).
constexpr int GC = 16, GN = 64, GTH = 128;

template <bool VEC>
__global__ void __launch_bounds__(GTH)
rnn_param_grads_kernel(const float *__restrict__ s, const float *__restrict__ d, const float *__restrict__ h,
                       const float *__restrict__ x, int T, int H, int d_in, float *__restrict__ dWh,
                       float *__restrict__ dWx, float *__restrict__ db)
{
    __shared__ __align__(16) float g[2][GC][MH];         // d_t * s_t
    __shared__ __align__(16) float hh[2][GC][GN];        // h_{t-1}, this CTA's columns
    __shared__ float xs[MT * MIO];
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3, seq = blockIdx.x, n0 = blockIdx.y * GN;
    const size_t base = (size_t)seq * T * H;
    const bool extra = blockIdx.y == 0;                  // this CTA also sums db and dWx: thread = component
    if (extra)
        for (int p = tid; p < T * d_in; p += GTH) xs[p] = x[(size_t)seq * T * d_in + p];
    // a chunk: 16 x 128 values of g (four float4 per thread) and 16 x 64 of h (two)
    float4 rg[4], rh[2];
    auto fetch = [&](int tc) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int t = tc + ty / 4 + 4 * e, i = (tid & 31) * 4;
            const bool in = t < T && i < H;
            const size_t at = base + (size_t)t * H + i;
            const float4 a = in ? ldg4<VEC>(d + at) : make_float4(0, 0, 0, 0);
            const float4 b = in ? ldg4<VEC>(s + at) : make_float4(0, 0, 0, 0);
            rg[e] = make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w);
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int t = tc + tid / 16 + 8 * e, i = n0 + (tid & 15) * 4;
            rh[e] = (t >= 1 && t < T && i < H) ? ldg4<VEC>(h + base + (size_t)(t - 1) * H + i) : make_float4(0, 0, 0, 0);
        }
    };
    float acc[8][8], sb = 0.0f, sx[MIO];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[a][c] = 0.0f;
#pragma unroll
    for (int c = 0; c < MIO; ++c) sx[c] = 0.0f;
    fetch(0);
    for (int tc = 0, buf = 0; tc < T; tc += GC, buf ^= 1) {
#pragma unroll
        for (int e = 0; e < 4; ++e) *reinterpret_cast<float4 *>(&g[buf][ty / 4 + 4 * e][(tid & 31) * 4]) = rg[e];
#pragma unroll
        for (int e = 0; e < 2; ++e) *reinterpret_cast<float4 *>(&hh[buf][tid / 16 + 8 * e][(tid & 15) * 4]) = rh[e];
        __syncthreads();                                 // (a buffer is refilled after the barrier that follows its reading)
        if (tc + GC < T) fetch(tc + GC);
        const int ke = min(GC, T - tc);
#pragma unroll 4
        for (int k = 0; k < ke; ++k) {
            const float4 g0 = *reinterpret_cast<const float4 *>(&g[buf][k][4 * ty]);
            const float4 g1 = *reinterpret_cast<const float4 *>(&g[buf][k][64 + 4 * ty]);
            const float4 h0 = *reinterpret_cast<const float4 *>(&hh[buf][k][4 * tx]);
            const float4 h1 = *reinterpret_cast<const float4 *>(&hh[buf][k][32 + 4 * tx]);
            const float gv[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
            const float hv[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int c = 0; c < 8; ++c) acc[a][c] = fmaf(gv[a], hv[c], acc[a][c]);
        }
        if (extra) {
            for (int k = 0; k < ke; ++k) {
                const float gv = g[buf][k][tid];
                sb += gv;
#pragma unroll
                for (int c = 0; c < MIO; ++c)
                    if (c < d_in) sx[c] = fmaf(gv, xs[(tc + k) * d_in + c], sx[c]);
            }
        }
    }
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        const int j = (a < 4 ? 0 : 60) + 4 * ty + a;
        if (j >= H) continue;
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
            const int i = n0 + 32 * hf + 4 * tx;
            if (i < H)
                stg4<VEC>(dWh + ((size_t)seq * H + j) * H + i,
                          make_float4(acc[a][4 * hf], acc[a][4 * hf + 1], acc[a][4 * hf + 2], acc[a][4 * hf + 3]));
        }
    }
    if (extra && tid < H) {
        db[(size_t)seq * H + tid] = sb;
#pragma unroll
        for (int c = 0; c < MIO; ++c)
            if (c < d_in) dWx[((size_t)seq * H + tid) * d_in + c] = sx[c];
    }
}

bool sizes_ok(int B, int T, int H) { return B >= 1 && T >= 1 && T <= MT && H >= 1 && H <= MH && H % 4 == 0; }

constexpr size_t JACOBI_SMEM_MAX = (size_t)(2 * MH * (MT + 1) + MH * MH) * sizeof(float);

int sm_count()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return 148;
    return sms;
}

template <bool VEC>
auto forward_kernel_of(int ns, bool many)
{
    return ns == 1 ? (many ? rnn_forward_kernel<1, VEC, true> : rnn_forward_kernel<1, VEC, false>)
         : ns == 2 ? rnn_forward_kernel<2, VEC, true> : ns == 3 ? rnn_forward_kernel<3, VEC, true> : rnn_forward_kernel<4, VEC, true>;
}

// one sequence per CTA until three of them per SM are not enough (the most its registers allow)
int seqs_per_cta(int B) { return B <= 3 * sm_count() ? 1 : 2; }

// A kernel's dynamic shared memory limit, raised once per device (the attribute call costs as much as a launch).
template <typename K>
bool allow_smem(K kernel, size_t bytes, int which)
{
    static std::atomic<unsigned long long> done[10];      // bit = device; one word per instance
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && dev < 64 && (done[which].load(std::memory_order_relaxed) >> dev & 1ull)) return true;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess) {
        launch_status();
        return false;
    }
    if (dev < 64) done[which].fetch_or(1ull << dev);
    return true;
}

// do all these pointers lie on 16 bytes?
template <typename... P>
bool vectors(const P *...p)
{
    return ((... | reinterpret_cast<uintptr_t>(p)) & 15u) == 0;
}

}  // namespace

extern "C" {

int rnn_forward(const float *Wh, const float *Wx, const float *b, const float *Wo, const float *bo, const float *x,
                const float *r, int B, int T, int H, int d_in, int d_out, float *h, float *d, float *l, float *loss,
                void *stream)
{
    if (!Wh || !Wx || !b || !Wo || !bo || !x || !r || !h || !d || !l || !loss) return RNN_ERR_INVALID;
    if (!sizes_ok(B, T, H) || d_in < 1 || d_in > MIO || d_out < 1 || d_out > MIO) return RNN_ERR_INVALID;
    const int sms = sm_count(), ns = std::min(4, (B + sms - 1) / sms);          // sequences per CTA: one CTA per SM, up to four
    const bool many = d_out > 1 || d_in > 4;
    const bool vec = vectors(Wh, b, h, d, l);
    auto kernel = vec ? forward_kernel_of<true>(ns, many) : forward_kernel_of<false>(ns, many);
    const size_t smem = (size_t)((d_in + d_out) * (MH + ns * T)) * sizeof(float);
    if (!allow_smem(kernel, (size_t)(2 * MIO * (MH + 4 * MT)) * sizeof(float), (ns == 1 && !many ? 0 : ns) + (vec ? 0 : 5))) return RNN_ERR_CUDA;
    kernel<<<(B + ns - 1) / ns, 2 * CT, smem, (cudaStream_t)stream>>>(Wh, Wx, b, Wo, bo, x, r, B, T, H, d_in, d_out, h, d, l, loss);
    return launch_status();
}

int rnn_bptt_sequential(const float *Wh, const float *l, const float *d, int B, int T, int H, float *s, void *stream)
{
    if (!Wh || !l || !d || !s || !sizes_ok(B, T, H)) return RNN_ERR_INVALID;
    const int ns = seqs_per_cta(B);
    const bool vec = vectors(Wh, l, d);
    auto kernel = vec ? (ns == 1 ? rnn_bptt_sequential_kernel<1, true> : rnn_bptt_sequential_kernel<2, true>)
                      : (ns == 1 ? rnn_bptt_sequential_kernel<1, false> : rnn_bptt_sequential_kernel<2, false>);
    const size_t smem = (size_t)ns * 4 * SC * MH * sizeof(float);
    if (!allow_smem(kernel, smem, ns - 1 + (vec ? 0 : 2))) return RNN_ERR_CUDA;
    kernel<<<(B + ns - 1) / ns, CT, smem, (cudaStream_t)stream>>>(Wh, l, d, B, T, H, s);
    return launch_status();
}

int rnn_bptt_jacobi(const float *Wh, const float *l, const float *d, int B, int T, int H, int n_iters, const float *s0,
                    float *s, void *stream)
{
    if (!Wh || !l || !d || !s || !sizes_ok(B, T, H) || n_iters < 0) return RNN_ERR_INVALID;
    // CTAs per sequence: 15 clusters of 8 or 33 of 4 fit the GPU at a time, and two rounds of 4 still beat whole sequences
    // on single CTAs; shares of fewer than eight steps would be mostly barriers
    const int sms = sm_count();
    int csz = B <= 15 && T >= 64 ? 8 : B <= 66 && T >= 32 ? 4 : 1;
    const int rpc = (T + csz - 1) / csz, NG = (H + 7) / 8, VS = (rpc + 3) / 4 * 4;
    const int grp = (((rpc + 3) / 4 + 1) / 2 * 2 * NG + 31) / 32 * 32;       // threads of a sequence's share
    // Pairs where an even number of rounds of one sequence per SM would be needed: a round of pairs takes 1.9 times as long
    // (T = 100, H = 128, 20 iterations: 450 and 236 us), so that for 300 sequences two of them, 904 us, lose to three rounds
    // of one, 705 us, and for 592 two, 900 us, win over four, 945 us.
    const int rounds = (B + sms - 1) / sms;
    const int form = csz > 1 || (grp <= 128 && rounds == 1) ? JAC_SPLIT : rounds % 2 == 0 && grp <= 416 ? JAC_PAIR : JAC_ONE;
    const bool vec = vectors(Wh, l, d, s);
    auto kernel = form == JAC_PAIR ? (vec ? rnn_bptt_jacobi_kernel<JAC_PAIR, 832, true> : rnn_bptt_jacobi_kernel<JAC_PAIR, 832, false>)
                : form == JAC_SPLIT ? (vec ? rnn_bptt_jacobi_kernel<JAC_SPLIT, 512, true> : rnn_bptt_jacobi_kernel<JAC_SPLIT, 512, false>)
                                    : (vec ? rnn_bptt_jacobi_kernel<JAC_ONE, 512, true> : rnn_bptt_jacobi_kernel<JAC_ONE, 512, false>);
    if (!allow_smem(kernel, JACOBI_SMEM_MAX, form + (vec ? 0 : 3))) return RNN_ERR_CUDA;
    const int nsq = form == JAC_PAIR ? 2 : 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((B + nsq - 1) / nsq * csz));
    cfg.blockDim = dim3((unsigned)(form == JAC_PAIR ? 2 * grp : form == JAC_SPLIT ? 4 * grp : grp));
    cfg.dynamicSmemBytes = (size_t)(H * MH + 2 * H * (VS + 1) + (form == JAC_SPLIT ? 128 * grp : 0)) * sizeof(float);
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)csz;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = csz > 1 ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, Wh, l, d, B, T, H, n_iters, s0, s, csz, rpc);
    return launch_status();
}

int rnn_param_grads(const float *s, const float *d, const float *h, const float *x, int B, int T, int H, int d_in,
                    float *dWh, float *dWx, float *db, void *stream)
{
    if (!s || !d || !h || !x || !dWh || !dWx || !db || !sizes_ok(B, T, H) || d_in < 1 || d_in > MIO) return RNN_ERR_INVALID;
    auto kernel = vectors(s, d, h, dWh) ? rnn_param_grads_kernel<true> : rnn_param_grads_kernel<false>;
    kernel<<<dim3(B, (H + GN - 1) / GN), GTH, 0, (cudaStream_t)stream>>>(s, d, h, x, T, H, d_in, dWh, dWx, db);
    return launch_status();
}

const char *rnn_last_error(void) { return g_err; }

}  // extern "C"
