// Back-propagation through time of a one-layer recurrent network as a triangular system (arXiv 2002.03629,
// Section 5.1; appendix "Backpropagation"): forward pass, exact back-substitution, truncated Jacobi
// iterations (Algorithm 1) and the parameter gradients.  Everything is summed in a fixed order: by fp32 fused multiply-adds in the forward pass,
// the back-substitution and the gradients of up to 24 steps, by tensor-core products of bf16 pieces that carry fp32's 24 bits in the others.
//
// Forward pass and back-substitution are chains of T matrix-vector products: what counts is the latency of one
// step, so a step is spread over four threads per component (see the kernels).  A Jacobi iteration is a product for all T
// states at once, [T x H] x [H x H]: it runs on the tensor cores, in pieces of bf16 that add up to fp32.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <cstdio>

#include "../../../include/rnn_bptt.h"
#include "../tc_common.cuh"

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

// two fp32 values in a register pair; a multiply-add on both
__device__ __forceinline__ unsigned long long pair(float lo, float hi)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
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
// The same by packed multiply-adds, the same values: half the instructions leave the schedulers to the forward pass's second group of
// warps (batch 1: 38 -> 35 us, 592: 116 -> 111, T = 64, H = 64, batch 30: 27 -> 23).  Back-substitution, which has the schedulers to
// itself, is slower with them (24 -> 26, 61 -> 65 us).
__device__ __forceinline__ void tile_dot2(const MatvecTile &t, const float *v, int q, float (&out)[4])
{
    const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(v) + q;
    // eight chains, two to a packed multiply-add (inputs of even and of odd number)
    unsigned long long c[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) c[u] = 0ull;
#pragma unroll
    for (int m = 0; m < MH / 16; ++m) {
        const ulonglong2 x = p[4 * m];
#pragma unroll
        for (int u = 0; u < 4; ++u) c[u] = fma2(pair(t.w[u][4 * m], t.w[u][4 * m + 1]), x.x, c[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) c[u] = fma2(pair(t.w[u][4 * m + 2], t.w[u][4 * m + 3]), x.y, c[u]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) out[u] = __uint_as_float((uint32_t)c[u]) + __uint_as_float((uint32_t)(c[u] >> 32));
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
// T = 100, H = 128, one input and output (B200): batch 1 86 -> 35 us, batch 592 209 -> 111 us; 16 inputs and outputs, T = 128 (before
// packed multiply-adds): 200 -> 132 and 613 -> 326 us.
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
                    tile_dot2(w, hs[cur][n], q, v);
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
// On the tensor cores.  An iteration is a product with the recurrent weights for all steps at once,
//     s_new[t][i] = l[t][i] + sum_k U[t + 1][k] * W_h[k][i],   U[t][k] = d[t][k] * s[t][k],
// computed transposed: D[i][c] = sum_k A[i][k] * B[k][c] with A = W_h^T, 128 x 128, constant, in tensor memory, and the iterate U in
// shared memory.  Column c of a CTA's unit is step t = c % T of its sequence c / T (a unit is one sequence, or as many whole
// ones as 128 columns hold): as the steps of a batch lie one after another in memory, so do the columns, and U, taken as
// zero at t = 0, keeps a sequence from reaching into the one before it.
// fp32 values are cut into three bf16 pieces (8 + 8 + 8 bits; what is left is below 2^-26 of the value) and the six products
// of pieces down to 2^-18 are summed.  Both sides are cut 2^24 times as large and the sums brought back by 2^-48, both exact: the last
// bit of any fp32 value then lies above the smallest bf16 number, where as they are the pieces of values below 6e-33 lose bits.  The tensor core rounds its running sums towards zero, so the five small products
// come first, while the sum is small, and the large one, high by high, is shared by two accumulators: four steps of full size each.
//   warps 0-7   epilogue: thread = (component i, JC columns of each slot); l and d of these stay in registers, s = l + D, U goes back to
//               shared memory as three pieces, eight columns (16 bytes) a store.  JC = 32; up to 64 components the rows of A lie
//               in tensor memory twice, so that all eight warps find work: 16 columns each
//   warps 8, 9  MMA, a slot each (their warpgroup hands its registers to the others)
// The columns go in two slots of up to 64, each with accumulators of its own: one slot's MMAs run while the other's epilogue
// does.  A slot's last column takes its sum from the first column of the slot behind it, which is therefore the first in every round.
// l and d of the next unit come into shared memory (bulk copies, where the pointers lie on 16 bytes) while this one is worked on.
// Values that three pieces cannot carry (infinities, NaN, states beyond 1e24, factors beyond 2e31) show as non-finite
// states: such a unit is computed again with plain multiply-adds before anything of it is stored.
// Bound: at 65 to 128 components the MMAs, 96 of 17 to 32 cycles an iteration (1.6 us of the 1.7 measured for 100 steps of 128
// components; multiply-adds on the CUDA cores, 40 TFLOP/s, took 10); below that the way from a slot's last product to its next
// first one (0.3 us of waits, 0.3 to 0.6 of epilogue).  T = 100, H = 128, 20 iterations: batch 1 71 -> 43 us, batch 592 894 -> 168 us;
// T = 50, H = 64, 10 iterations, batch 300: 61 -> 28 us.  Against 64 bits the states are off by 1.0e-7 (2-norm), 1.1e-7 to 3.4e-7 before.
constexpr int JE = 256, JTH = JE + 128;      // epilogue threads, all threads
constexpr int J_SLOT = 64;                   // columns of a slot
constexpr int J_PIECE = MH * J_SLOT * 2;     // bytes of one piece of a slot's operand: [128 k][64 columns], 128-byte swizzle
constexpr size_t J_OPS = 6 * J_PIECE;        // then l and d of a unit, [columns][H] each
constexpr uint32_t J_DCOL = 3 * (MH / 2);    // tensor memory: three pieces of A, then per slot the two accumulators

// The waits of a call: how long one may take, and where the caller wants to read that one gave up (or NULL).
struct Waits {
    unsigned long long ns;
    int *status;
};
// What the waits of a CTA share.  (The patience lies in shared memory: as a kernel argument in every wait it cost the loops registers, 170 us
// instead of 168 for 592 sequences of 100 steps and 20 iterations.)
struct CtaWaits {
    unsigned long long ns;
    int dead;                                // a wait gave up
};
struct JacShared {
    uint64_t ready[2], full[2];              // the slot's operand is there; its products are
    uint32_t tmem;
    uint64_t staged;                         // the unit's l and d are in shared memory
    CtaWaits waits;
};

// D[tmem] (+)= A[tmem] * B[smem], 128 x N x 16
__device__ __forceinline__ void umma_ts_bf16(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, bool accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
                 ::"r"(d), "r"(a), "l"(b), "r"(idesc), "r"((uint32_t)accumulate) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
                   "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ uint32_t tmem_ld1(uint32_t taddr)
{
    uint32_t r;
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr) : "memory");
    return r;
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint32_t (&r)[4])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}
__device__ __forceinline__ void sts4(uint32_t at, const uint32_t (&r)[4])
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}
constexpr float PIECES_UP = 0x1p24f, SUMS_DOWN = 0x1p-48f;      // before the cut, after the products
// two values in three bf16 pieces each, packed (the first in the low half)
__device__ __forceinline__ void cut3(float a, float b, uint32_t &h, uint32_t &m, uint32_t &l)
{
    h = pack_bf16x2(a, b);
    a -= __uint_as_float(h << 16);
    b -= __uint_as_float(h & 0xffff0000u);
    m = pack_bf16x2(a, b);
    a -= __uint_as_float(m << 16);
    b -= __uint_as_float(m & 0xffff0000u);
    l = pack_bf16x2(a, b);
}
// bounded: true once the barrier's phase has completed, false when the time is over (0: at once) or another wait of the CTA has given up
__device__ __forceinline__ bool jac_wait(CtaWaits &w, uint64_t *bar, uint32_t parity)
{
    if (mbar_test_wait(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    const unsigned long long ns = *(volatile unsigned long long *)&w.ns;
    for (unsigned i = 1; ns != 0; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 63u) == 0u && (*(volatile int *)&w.dead || global_ns() - t0 > ns)) break;
    }
    *(volatile int *)&w.dead = 1;
    return false;
}
// The end of a CTA in which a wait gave up (all threads, behind a barrier): the caller is told, and shared and tensor memory are kept until
// the copies and MMAs that are on their way, microseconds' worth, have ended.
__device__ __noinline__ void gave_up(const Waits &w)
{
    if (threadIdx.x == 0 && w.status != nullptr) *(volatile int *)w.status = RNN_ERR_TIMEOUT;
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
}
// barrier of the epilogue warps: did every thread say yes?
__device__ __forceinline__ bool jac_all(bool ok)
{
    int all;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbar.red.and.pred q, 1, 256, p;\n\tselp.b32 %0, 1, 0, q;\n\t}" : "=r"(all) : "r"((int)ok) : "memory");
    return all != 0;
}

// One sequence by plain multiply-adds, thread = component, U in shared memory.  Steps in ascending order: step t reads U[t + 1], not yet
// overwritten, and then replaces U[t], which nobody reads any more.  Sixteen weights in flight: 592 sequences of 100 steps and 20 iterations,
// an infinity in each, 20 ms (50 with four).  Eight steps a thread for every weight take 8 ms, but the registers that the compiler gives
// them cost the units that never come here 3 to 6 % (300 sequences of 50 steps, H = 64).
__device__ __forceinline__ void jac_plain(const float *Wh, const float *l, const float *d, int T, int H, int iters, const float *s0, float *s,
                                          float *U, int tid)
{
    for (int p = tid; p < T * MH; p += JE) {
        const int t = p / MH, k = p % MH;
        U[p] = k < H && s0 != nullptr ? d[t * H + k] * s0[t * H + k] : 0.0f;
    }
#pragma unroll 1
    for (int it = 0; it < iters; ++it)
#pragma unroll 1
        for (int t = 0; t < T; ++t) {
            jac_all(true);
            if (tid >= H) continue;
            const int at = t * H + tid;
            float acc = l[at];
            if (t + 1 < T)
#pragma unroll 16
                for (int k = 0; k < H; ++k) acc = fmaf(U[(t + 1) * MH + k], __ldg(Wh + k * H + tid), acc);
            if (it + 1 == iters) s[at] = acc;
            else U[t * MH + tid] = d[at] * acc;
        }
    jac_all(true);
}

// MANY: units of several sequences
template <int JC, bool MANY>
__global__ void __launch_bounds__(JTH, 1)
rnn_bptt_jacobi_kernel(const float *__restrict__ Wh, const float *l, const float *d, int B, int T, int H, int iters, const float *s0, float *s,
                       int per_unit, const Waits waits)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ JacShared sh;
    uint8_t *ops = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);   // [slot][piece]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int ROWS = MH * JC / 32, G = J_SLOT / JC;              // rows of A before they repeat, groups of columns
    const int row = (warp & 3) * 32 + lane;                                  // epilogue: tensor memory lane,
    const int i = row % ROWS, g = (warp >> 2) * (G / 2) + row / ROWS;        // component, group of columns
    const uint32_t quad = (uint32_t)((warp & 3) * 32) << 16;
    const int width = per_unit * T;                                          // columns of a unit
    const bool two = width > J_SLOT;
    const int units = (B - 1) / per_unit + 1, nk = (H + 15) / 16;
    // the columns of unit u (B T need not fit 31 bits)
    auto unit_columns = [&](int u) { return min(per_unit, B - u * per_unit) * T; };
    // the columns of a slot that its MMAs compute
    auto slot_columns = [&](int k) { return max(0, min(J_SLOT, width - k * J_SLOT) + 15) / 16 * 16; };
    float *const ls = reinterpret_cast<float *>(ops + J_OPS), *const ds = ls + width * H;
    const bool stages = ((reinterpret_cast<uintptr_t>(l) | reinterpret_cast<uintptr_t>(d)) & 15u) == 0;
    auto stage = [&](int u) {
        if (u >= units || !stages) return;
        const uint32_t bytes = (uint32_t)(unit_columns(u) * H) * 4u;
        const size_t from = (size_t)u * per_unit * T * H;
        mbar_expect_tx(&sh.staged, 2 * bytes);
        bulk_load(smem_u32(ls), l + from, bytes, &sh.staged);
        bulk_load(smem_u32(ds), d + from, bytes, &sh.staged);
    };
    if (tid == 0) {
        for (int k = 0; k < 2; ++k) { mbar_init(&sh.ready[k], JE / 32); mbar_init(&sh.full[k], 1); }
        mbar_init(&sh.staged, 1);
        sh.waits = CtaWaits{waits.ns, 0};
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        stage(blockIdx.x);
    }
    if (warp == 8) tmem_alloc(&sh.tmem, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = sh.tmem;
    const int nmma = iters - (s0 == nullptr ? 1 : 0);                        // from zero the first iteration gives l
    bool fine = true;                                                        // this thread's weights are finite
    if (warp < 8) {
        float chk = 0.0f;
#pragma unroll 2
        for (int c4 = 0; c4 < 8; ++c4) {                                     // 32 words of every piece, 64 k
            const int k0 = (warp >> 2) * 64 + c4 * 8;
            if (k0 >= nk * 16) break;
            uint32_t ph[4], pm[4], pl[4];
            float w[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                w[e] = k0 + e < H && i < H ? __ldg(Wh + (k0 + e) * H + i) : 0.0f;
                chk = fmaf(w[e], 0.0f, chk);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) cut3(w[2 * e] * PIECES_UP, w[2 * e + 1] * PIECES_UP, ph[e], pm[e], pl[e]);
            const uint32_t at = tm + quad + (uint32_t)(k0 / 2);
            tmem_st4(at, ph);
            tmem_st4(at + MH / 2, pm);
            tmem_st4(at + MH, pl);
        }
        fine = chk == 0.0f;
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();

    if (warp >= 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");                 // 384 threads x 168 registers = 256 x 232 + 128 x 40
        if (warp < 10) {
            const int slot = warp - 8, cols = slot_columns(slot);
            if (cols > 0) {
                // B lies with neighbouring columns together ("MN-major": bit 16)
                const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(MH >> 4) << 24) | ((uint32_t)(cols >> 3) << 17);
                const uint32_t d0 = tm + J_DCOL + (uint32_t)(slot * 128), d1 = d0 + J_SLOT;
                // swizzled, 64 columns a row of 128 bytes, groups of eight k rows 1024 bytes apart
                const uint64_t bd = smem_desc_sw128(smem_u32(ops + (size_t)slot * 3 * J_PIECE)) | ((uint64_t)(1024 >> 4) << 16);
                constexpr uint64_t PC = J_PIECE >> 4, K16 = 2048 >> 4;
                uint32_t par = 0;
                bool on = true;
                for (int u = blockIdx.x; u < units && on; u += gridDim.x)
                    for (int it = 0; it < nmma && on; ++it, par ^= 1u) {
                        on = __all_sync(0xffffffffu, jac_wait(sh.waits, &sh.ready[slot], par));
                        if (!on) break;
                        tc_fence_after();
                        if (elect_one()) {
                            // (rolled: straight-line code of 96 MMAs cost 10 us of instruction fetches in the first iterations)
                            uint32_t a = tm;
                            uint64_t b = bd;
#pragma unroll 2
                            for (int k = 0; k < nk; ++k, a += 8, b += K16) {
                                umma_ts_bf16(d1, a + MH, b, idesc, k > 0);
                                umma_ts_bf16(d1, a, b + 2 * PC, idesc, true);
                                umma_ts_bf16(d1, a + MH / 2, b + PC, idesc, true);
                                umma_ts_bf16(d1, a + MH / 2, b, idesc, true);
                                umma_ts_bf16(d1, a, b + PC, idesc, true);
                            }
                            a = tm;
                            b = bd;
#pragma unroll 2
                            for (int k = 0; k < nk; ++k, a += 8, b += K16) umma_ts_bf16(k < nk / 2 ? d1 : d0, a, b, idesc, k != nk / 2);
                            umma_commit(&sh.full[slot]);
                        }
                        __syncwarp();
                    }
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 232;");
        uint32_t par = 0, staged_par = 0;
        for (int u = blockIdx.x; u < units; u += gridDim.x) {
            const int cols = unit_columns(u);
            const size_t base = (size_t)u * per_unit * T * H + i;
            bool ok = *(volatile int *)&sh.waits.dead == 0;                        // (a wait that gave up ends the CTA's work)
            if (ok && stages) ok = jac_wait(sh.waits, &sh.staged, staged_par);
            staged_par ^= 1u;
            const float *lp = stages ? ls + i : l + base, *dp = stages ? ds + i : d + base;
            float lv[2][JC], dv[2][JC], l0 = 0.0f;
            uint32_t first[2];
            // This thread's columns of slot k are 64 k + JC g + 1 + j, its operand columns one less; column 0 feeds nothing.
            // (Row offsets are run along anew for every array: kept for all columns they would take 64 registers.)
            auto rows = [&](int k, auto f) {
                int step = H;
                asm volatile("" : "+r"(step));
                const int c0 = k * J_SLOT + g * JC + 1, left = i < H ? cols - c0 : 0;
                int at = c0 * step;
#pragma unroll
                for (int j0 = 0; j0 < JC; j0 += 8) {
                    if (j0 + 8 <= left) {
#pragma unroll
                        for (int j = j0; j < j0 + 8; ++j, at += step) f(j, at, true);
                    } else {
#pragma unroll
                        for (int j = j0; j < j0 + 8; ++j, at += step) f(j, at, j < left);
                    }
                }
            };
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                rows(k, [&](int j, int at, bool in) { lv[k][j] = in ? lp[at] : 0.0f; });
                rows(k, [&](int j, int at, bool in) { dv[k][j] = in ? dp[at] * PIECES_UP : 0.0f; });
                // first steps of the unit's other sequences: no U, not even of an infinite state
                first[k] = 0;
                if (MANY)
                    for (int c = T; c < cols; c += T) {
                        const int j = c - (k * J_SLOT + g * JC + 1);
                        if (j >= 0 && j < JC) first[k] |= 1u << j;
                    }
            }
            if (g == 0 && i < H) l0 = lp[0];
            ok = jac_all(ok);                                                // everything has been read
            if (tid == 0 && ok) stage(u + (int)gridDim.x);
            const bool idle = (i & ~31) >= H;                                // no component of this warp's (and no k that the MMAs read)
            // eight columns of the operand of slot k from their states: pieces of U = d s (d as large as they want it)
            auto put8 = [&](int k, int j0, const float (&v)[8]) {
                uint32_t ph[4], pm[4], pl[4];
                float w[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) w[e] = dv[k][j0 + e] * v[e];
                if (MANY)
#pragma unroll
                    for (int e = 0; e < 8; ++e) w[e] = first[k] >> (j0 + e) & 1u ? 0.0f : w[e];
#pragma unroll
                for (int e = 0; e < 4; ++e) cut3(w[2 * e], w[2 * e + 1], ph[e], pm[e], pl[e]);
                const uint32_t at = smem_u32(ops + (size_t)k * 3 * J_PIECE) + (uint32_t)(i * 128 + (((JC / 8 * g + (j0 >> 3)) ^ (i & 7)) << 4));
                sts4(at, ph);
                sts4(at + J_PIECE, pm);
                sts4(at + 2 * J_PIECE, pl);
            };
            // this warp's part of the operand of slot k is written and its sums are read
            auto hand_over = [&](int k) {
                fence_proxy_async_smem();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.ready[k]);
            };
            float edge = 0.0f;                                               // the last group's: column 64's sum
            // A slot's sums to states: into the operand, or, in the last iteration, in place of l.  The last of a thread's columns is
            // the first of the other thread's, or of the slot behind.
            auto finish = [&](int k, bool last) {
                const uint32_t at = tm + quad + J_DCOL + (uint32_t)(k * 128 + g * JC);
                const int mine = slot_columns(k) - g * JC;                   // a multiple of 16
                if (idle) return;
                if (k == 1 && g == G - 1) {
                    const uint32_t first = tm + quad + J_DCOL + 128u, e0 = tmem_ld1(first), e1 = tmem_ld1(first + J_SLOT);
                    tmem_wait_ld();
                    edge = __uint_as_float(e0) + __uint_as_float(e1);
                }
                if (mine <= 0) return;
                // sixteen columns in hand, the next ones on their way
                uint32_t a[JC / 16][16], b[JC / 16][16], an = 0, bn = 0;
                tmem_ld16(at, a[0]);
                tmem_ld16(at + J_SLOT, b[0]);
                if (JC == 32) tmem_wait_ld();
                if (JC == 32 && mine > 16) {
                    tmem_ld16(at + 16, a[JC / 16 - 1]);
                    tmem_ld16(at + J_SLOT + 16, b[JC / 16 - 1]);
                }
                if (g < G - 1 && mine > JC) { an = tmem_ld1(at + JC); bn = tmem_ld1(at + J_SLOT + JC); }
                if (JC == 16) tmem_wait_ld();
                auto sum = [&](int c) { return __uint_as_float(a[c >> 4][c & 15]) + __uint_as_float(b[c >> 4][c & 15]); };
                auto beyond = [&] { return g < G - 1 ? __uint_as_float(an) + __uint_as_float(bn) : k == 0 ? edge : 0.0f; };
                auto take = [&](int j0, float (&w)[8]) {
                    if (last) {
#pragma unroll
                        for (int e = 0; e < 8; ++e) lv[k][j0 + e] = fmaf(w[e], SUMS_DOWN, lv[k][j0 + e]);
                    } else {
#pragma unroll
                        for (int e = 0; e < 8; ++e) w[e] = fmaf(w[e], SUMS_DOWN, lv[k][j0 + e]);
                        put8(k, j0, w);
                    }
                };
                float w[8];
                if (g == 0 && k == 0 && last) l0 = fmaf(sum(0), SUMS_DOWN, l0);
#pragma unroll
                for (int e = 0; e < 8; ++e) w[e] = sum(1 + e);
                take(0, w);
#pragma unroll
                for (int e = 0; e < 7; ++e) w[e] = sum(9 + e);
                if constexpr (JC == 16) {
                    w[7] = beyond();
                    take(8, w);
                } else {
                    tmem_wait_ld();
                    w[7] = mine > 16 ? sum(16) : 0.0f;                       // (a seventeenth column that is nobody's)
                    take(8, w);
                    if (mine > 16) {
#pragma unroll
                        for (int e = 0; e < 8; ++e) w[e] = sum(17 + e);
                        take(16, w);
#pragma unroll
                        for (int e = 0; e < 7; ++e) w[e] = sum(25 + e);
                        w[7] = beyond();
                        take(24, w);
                    }
                }
            };
            // the start: U of s0, or of the first iteration from zero, which gives l
            if (nmma > 0) {
#pragma unroll
                for (int k = 1; k >= 0; --k) {
                    if (k == 1 && !two) continue;
                    float v[JC];
                    if (s0 != nullptr) rows(k, [&](int j, int at, bool in) { v[j] = in ? (s0 + base)[at] : 0.0f; });
#pragma unroll
                    for (int j0 = 0; j0 < JC; j0 += 8) {
                        if (idle || j0 >= slot_columns(k) - g * JC) break;
                        float w[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) w[j] = s0 != nullptr ? v[j0 + j] : lv[k][j0 + j];
                        put8(k, j0, w);
                    }
                    hand_over(k);
                }
            }
            for (int it = 0; it < nmma && ok; ++it, par ^= 1u) {
                const bool last = it + 1 == nmma;
#pragma unroll
                for (int k = 1; k >= 0; --k) {
                    if (k == 1 && !two) continue;
                    ok = __all_sync(0xffffffffu, jac_wait(sh.waits, &sh.full[k], par));
                    if (!ok) break;
                    tc_fence_after();
                    finish(k, last);
                    if (!last) hand_over(k);
                }
            }
            // Non-finite anywhere?  (Whatever became non-finite on the way either shows here or has left at a first step.)
            float chk = fine ? l0 * 0.0f : NAN;
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int j = 0; j < JC; ++j) chk = fmaf(lv[k][j], 0.0f, chk);
            const bool plain = !jac_all(chk == 0.0f);
            ok = jac_all(ok);
            if (!ok) {
                // the operands did not come or the MMAs did not end: nothing is known about the states
                for (int c = g; c < cols; c += G)
                    if (i < H) s[base + (size_t)c * H] = NAN;
            } else if (plain) {
                for (int q = 0; q < per_unit && u * per_unit + q < B; ++q) {
                    const size_t o = (size_t)(u * per_unit + q) * T * H;
                    jac_plain(Wh, l + o, d + o, T, H, iters, s0 != nullptr ? s0 + o : nullptr, s + o, reinterpret_cast<float *>(ops), tid);
                }
            } else if (i < H) {
#pragma unroll
                for (int k = 0; k < 2; ++k) rows(k, [&](int j, int at, bool in) { if (in) (s + base)[at] = lv[k][j]; });
                if (g == 0) s[base] = l0;
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (sh.waits.dead != 0) gave_up(waits);
    if (warp == 8) {
        tc_fence_after();
        tmem_dealloc(tm, 512);
    }
}

// n_iters == 0: the start iterate
__global__ void rnn_copy_kernel(const float *s0, float *s, size_t n)
{
    for (size_t p = (size_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (size_t)gridDim.x * blockDim.x) s[p] = s0 != nullptr ? s0[p] : 0.0f;
}

// ------------------------------------------------------------------ parameter gradients
// dWh = sum_t g_t h_{t-1}^T with g_t = d_t * s_t: a [128 x T] x [T x 128] product per sequence, on the tensor cores like the Jacobi
// iterations: three bf16 pieces of either side (2^24 times as large), six products, the five small ones in an accumulator of their own.  Both operands lie
// in shared memory as they come, components together, steps in rows (PK of them at a time, so that two CTAs share an SM and one's
// loads and stores pass while the other multiplies).  A CTA computes `cols` columns of one sequence: all of them, or a half or a
// quarter where there are few sequences.  db and dWx, the same sums with 1 and x_t on the right, are taken up while the operands are cut:
// a warp sums the steps that it cuts, the warps' sums are added in order.
// Sums that are not finite (an operand beyond 2e31, a product beyond 1e24) are made again by plain multiply-adds, as in jac_plain.
// T = 100, H = 128 (B200): batch 592 45 us (91 MB in, 39 MB out: 20 us), batch 1 11; multiply-adds on the CUDA cores took 75 and 16.  Against 64 bits
// dWh is off by 1.1e-7 in the 2-norm, 1.8e-7 before.  Bound: a CTA's chain of loads, cutting, MMAs and stores, twice per SM.
constexpr int PK = 64, PGT = 256;            // steps at a time, threads
constexpr int P_PIECE = PK * MH * 2;         // bytes of a piece: [two groups of 64 components][PK steps][128 bytes, swizzled]
constexpr size_t P_SMEM = 6 * P_PIECE + 1024;

// NX: room for that many inputs
template <bool VEC, int NX>
__global__ void __launch_bounds__(PGT, 2)
rnn_param_grads_kernel(const float *__restrict__ s, const float *__restrict__ d, const float *__restrict__ h,
                       const float *__restrict__ x, int T, int H, int d_in, int cols, float *__restrict__ dWh,
                       float *__restrict__ dWx, float *__restrict__ db, const Waits waits)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t done;
    __shared__ uint32_t tmem;
    __shared__ CtaWaits own;
    uint8_t *ops = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);    // pieces of g, then of h
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, seq = blockIdx.x, n0 = blockIdx.y * cols;
    const size_t base = (size_t)seq * T * H;
    const bool extra = blockIdx.y == 0;
    if (tid == 0) {
        mbar_init(&done, 1);
        own = CtaWaits{waits.ns, 0};
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(&tmem, 256);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = tmem;
    const int i4 = lane * 4;
    float sx[1 + NX][4];                                 // db, then dWx
#pragma unroll
    for (int c = 0; c <= NX; ++c)
#pragma unroll
        for (int e = 0; e < 4; ++e) sx[c][e] = 0.0f;
    bool ok = true;
    // four neighbouring components of step row r of an operand, in pieces
    auto put = [&](uint8_t *op, int r, const float (&v)[4]) {
        uint32_t ph[2], pm[2], pl[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) cut3(v[2 * e] * PIECES_UP, v[2 * e + 1] * PIECES_UP, ph[e], pm[e], pl[e]);
        const uint32_t at = smem_u32(op) + (uint32_t)((i4 >> 6) * (PK * 128) + r * 128 + ((((i4 & 63) >> 3) ^ (r & 7)) << 4) + (i4 & 7) * 2);
        asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(at), "r"(ph[0]), "r"(ph[1]) : "memory");
        asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(at + P_PIECE), "r"(pm[0]), "r"(pm[1]) : "memory");
        asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(at + 2 * P_PIECE), "r"(pl[0]), "r"(pl[1]) : "memory");
    };
    uint32_t par = 0;
    for (int t0 = 0; t0 < T; t0 += PK, par ^= 1u) {
        if (t0 > 0) {                                    // the steps before have been multiplied
            ok = jac_wait(own, &done, par ^ 1u);
            if (!__syncthreads_and(ok)) { ok = false; break; }
        }
        const int rows = (min(PK, T - t0) + 15) / 16 * 16;
#pragma unroll (NX <= 4 ? 4 : 2)
        for (int r = warp; r < rows; r += PGT / 32) {
            const int t = t0 + r;
            const bool in = t < T && i4 < H, hin = in && t >= 1;
            const size_t at = base + (size_t)t * H + i4;
            const float4 a = in ? ldg4<VEC>(d + at) : make_float4(0, 0, 0, 0), b = in ? ldg4<VEC>(s + at) : make_float4(0, 0, 0, 0);
            const float4 hv = hin ? ldg4<VEC>(h + at - H) : make_float4(0, 0, 0, 0);
            const float gv[4] = {a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w};
            put(ops, r, gv);
            const float hh[4] = {hv.x, hv.y, hv.z, hv.w};
            put(ops + 3 * P_PIECE, r, hh);
            if (extra && t < T) {
#pragma unroll
                for (int e = 0; e < 4; ++e) sx[0][e] += gv[e];
#pragma unroll
                for (int c = 0; c < NX; ++c)
                    if (c < d_in) {
                        const float xv = __ldg(x + ((size_t)seq * T + t) * d_in + c);
#pragma unroll
                        for (int e = 0; e < 4; ++e) sx[c + 1][e] = fmaf(gv[e], xv, sx[c + 1][e]);
                    }
            }
        }
        fence_proxy_async_smem();
        tc_fence_before();
        __syncthreads();
        if (warp == 0 && elect_one()) {
            tc_fence_after();
            // both operands lie with neighbouring components together ("MN-major": bits 15 and 16)
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (3u << 15) | ((uint32_t)(MH >> 4) << 24) | ((uint32_t)(cols >> 3) << 17);
            // groups of 64 components PK x 128 bytes apart, of eight steps 1024
            const uint64_t lead = (uint64_t)((PK * 128 >> 4) - 1) << 16;      // (the descriptor comes with 1)
            const uint64_t ad0 = smem_desc_sw128(smem_u32(ops)) + lead;
            const uint64_t bd0 = smem_desc_sw128(smem_u32(ops + 3 * P_PIECE + (n0 >> 6) * (PK * 128)) + (uint32_t)((n0 & 63) * 2)) + lead;
            constexpr uint64_t PC = P_PIECE >> 4, K16 = 2048 >> 4;
            const uint32_t dm = tm, dc = tm + MH;
            uint64_t a = ad0, b = bd0;
#pragma unroll 1
            for (int k = 0; k < rows; k += 16, a += K16, b += K16) {
                const bool on = t0 > 0 || k > 0;
                umma_bf16(dc, a + 2 * PC, b, idesc, on);
                umma_bf16(dc, a, b + 2 * PC, idesc, 1u);
                umma_bf16(dc, a + PC, b + PC, idesc, 1u);
                umma_bf16(dc, a + PC, b, idesc, 1u);
                umma_bf16(dc, a, b + PC, idesc, 1u);
                umma_bf16(dm, a, b, idesc, on);
            }
            umma_commit(&done);
        }
        __syncwarp();
    }
    if (ok) ok = jac_wait(own, &done, par ^ 1u);
    ok = __syncthreads_and(ok) != 0;
    tc_fence_after();
    float *out = dWh + (size_t)seq * H * H;
    float chk = 0.0f;                                    // non-zero (NaN): a sum that is not finite
    if (ok) {
        // a warp takes sixteen rows of its quadrant and half of the columns at a time: eight rows of 32 bytes a store
        const int q = warp & 3, half = cols / 2, c0 = (warp >> 2) * half;
#pragma unroll 1
        for (int rr = 0; rr < 32; rr += 16)
#pragma unroll 1
            for (int c = c0; c < c0 + half; c += 8) {
                const uint32_t at = tm + ((uint32_t)(q * 32 + rr) << 16) + (uint32_t)c;
                uint32_t a[4], b[4];
                tmem_ld_16x8(at, a);
                tmem_ld_16x8(at + MH, b);
                tmem_wait_ld();
                float v[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = (__uint_as_float(a[e]) + __uint_as_float(b[e])) * SUMS_DOWN;
                const int j = n0 + c + 2 * (lane & 3);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int i = q * 32 + rr + (lane >> 2) + 8 * e;
                    if (i < H && j < H) {                // (H is even)
                        float *to = out + (size_t)i * H + j;
                        if constexpr (VEC) *reinterpret_cast<float2 *>(to) = make_float2(v[2 * e], v[2 * e + 1]);
                        else { to[0] = v[2 * e]; to[1] = v[2 * e + 1]; }
                        chk = fmaf(v[2 * e], 0.0f, fmaf(v[2 * e + 1], 0.0f, chk));
                    }
                }
            }
    }
    // Not finite: an operand that the pieces cannot carry, or a product or a sum beyond 1e24, whose pieces may leave fp32 with either sign.  (Whatever
    // does not carry shows here: each operand meets every one of the other side, be it a zero.)
    if (!__syncthreads_and(ok && chk == 0.0f))
        for (int p = tid; p < H * cols; p += PGT) {
            const int i = p / cols, j = n0 + p % cols;
            if (j >= H) continue;
            const float *gd = d + base + i, *gs = s + base + i, *hj = h + base + j;
            float acc = ok ? 0.0f : NAN;
#pragma unroll 4
            for (int t = H; t < T * H; t += H) acc = fmaf(gd[t] * gs[t], hj[t - H], acc);
            out[(size_t)i * H + j] = acc;
        }
    if (extra) {
        // the warps' sums through the operands' memory
        float *sums = reinterpret_cast<float *>(ops);        // [warp][1 + d_in][MH]
        const int n = 1 + d_in;
        if (ok)                                              // (else the MMAs may still read there)
#pragma unroll
            for (int c = 0; c <= NX; ++c)
                if (c < n) *reinterpret_cast<float4 *>(sums + (warp * n + c) * MH + i4) = make_float4(sx[c][0], sx[c][1], sx[c][2], sx[c][3]);
        __syncthreads();
        for (int p = tid; p < n * MH; p += PGT) {
            const int c = p / MH, i = p % MH;
            if (i >= H) continue;
            float t = ok ? 0.0f : NAN;
            for (int w = 0; ok && w < PGT / 32; ++w) t += sums[(w * n + c) * MH + i];
            if (c == 0) db[(size_t)seq * H + i] = t;
            else dWx[((size_t)seq * H + i) * d_in + c - 1] = t;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (own.dead != 0) gave_up(waits);
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tm, 256);
    }
}

// Few steps: multiply-adds on the CUDA cores, a [128 x T] x [T x 64] product per CTA (two CTAs per sequence), 128 threads with 8 x 8 outputs
// each (rows 4 ty.. and 64 + 4 ty.., columns 4 tx.. and 32 + 4 tx..), the steps in chunks of GC through two small shared-memory buffers, the
// next chunk's loads in registers while one is multiplied.  db and dWx ride along: the same sums with 1 and x_t on the right.
constexpr int GC = 16, GN = 64, GTH = 128;

template <bool VEC>
__global__ void __launch_bounds__(GTH)
rnn_param_grads_short_kernel(const float *__restrict__ s, const float *__restrict__ d, const float *__restrict__ h,
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

int rnn_bptt_jacobi_bounded(const float *Wh, const float *l, const float *d, int B, int T, int H, int n_iters, const float *s0,
                            float *s, unsigned long long wait_ns, int *status, void *stream)
{
    if (!Wh || !l || !d || !s || !sizes_ok(B, T, H) || n_iters < 0) return RNN_ERR_INVALID;
    const int sms = sm_count();
    if (n_iters == 0) {
        const size_t n = (size_t)B * T * H;
        rnn_copy_kernel<<<(unsigned)std::min<size_t>((n + 255) / 256, (size_t)sms * 8), 256, 0, (cudaStream_t)stream>>>(s0, s, n);
        return launch_status();
    }
    // several sequences in a unit of 128 columns only where there are more of them than SMs
    const int per_unit = std::max(1, std::min(2 * J_SLOT / T, (B - 1) / sms + 1));
    auto kernel = per_unit > 1 ? (H > 64 ? rnn_bptt_jacobi_kernel<32, true> : rnn_bptt_jacobi_kernel<16, true>)
                               : (H > 64 ? rnn_bptt_jacobi_kernel<32, false> : rnn_bptt_jacobi_kernel<16, false>);
    if (!allow_smem(kernel, 1024 + J_OPS + (size_t)2 * MT * MH * sizeof(float), (H > 64) + 2 * (per_unit > 1))) return RNN_ERR_CUDA;
    const size_t smem = 1024 + J_OPS + (size_t)2 * per_unit * T * H * sizeof(float);
    kernel<<<std::min(sms, (B - 1) / per_unit + 1), JTH, smem, (cudaStream_t)stream>>>(
        Wh, l, d, B, T, H, std::min(n_iters, T), s0, s, per_unit, Waits{wait_ns, status});
    return launch_status();
}

int rnn_bptt_jacobi(const float *Wh, const float *l, const float *d, int B, int T, int H, int n_iters, const float *s0,
                    float *s, void *stream)
{
    return rnn_bptt_jacobi_bounded(Wh, l, d, B, T, H, n_iters, s0, s, MBAR_WAIT_NS, nullptr, stream);
}

int rnn_param_grads_bounded(const float *s, const float *d, const float *h, const float *x, int B, int T, int H, int d_in,
                            float *dWh, float *dWx, float *db, unsigned long long wait_ns, int *status, void *stream)
{
    if (!s || !d || !h || !x || !dWh || !dWx || !db || !sizes_ok(B, T, H) || d_in < 1 || d_in > MIO) return RNN_ERR_INVALID;
    const bool vec = vectors(s, d, h, dWh);
    // Tensor memory and operands cost a CTA about a microsecond: 12 steps, H = 32, batch 1 and 300: 4.2 and 8.2 us that way, 3.5 and 5.4 this;
    // 13 steps, H = 92, batch 2: 4.4 and 3.9; 30 steps, H = 60, batch 592: 12.5 and 16.8; 31 steps, batch 59: 5.9 and 6.4.
    if (T <= 24) {
        auto few = vec ? rnn_param_grads_short_kernel<true> : rnn_param_grads_short_kernel<false>;
        few<<<dim3(B, (H + GN - 1) / GN), GTH, 0, (cudaStream_t)stream>>>(s, d, h, x, T, H, d_in, dWh, dWx, db);
        return launch_status();
    }
    auto kernel = d_in <= 4 ? (vec ? rnn_param_grads_kernel<true, 4> : rnn_param_grads_kernel<false, 4>)
                            : (vec ? rnn_param_grads_kernel<true, MIO> : rnn_param_grads_kernel<false, MIO>);
    // columns per CTA: all where there are sequences for all SMs, else a half, a quarter
    const int sms = sm_count(), all = (H + 31) / 32 * 32;
    const int cols = B >= sms ? all : B >= sms / 2 ? std::min(all, MH / 2) : std::min(all, MH / 4);
    if (!allow_smem(kernel, P_SMEM, vec + 2 * (d_in <= 4))) return RNN_ERR_CUDA;
    kernel<<<dim3(B, (H + cols - 1) / cols), PGT, P_SMEM, (cudaStream_t)stream>>>(s, d, h, x, T, H, d_in, cols, dWh, dWx, db, Waits{wait_ns, status});
    return launch_status();
}

int rnn_param_grads(const float *s, const float *d, const float *h, const float *x, int B, int T, int H, int d_in,
                    float *dWh, float *dWx, float *db, void *stream)
{
    return rnn_param_grads_bounded(s, d, h, x, B, T, H, d_in, dWh, dWx, db, MBAR_WAIT_NS, nullptr, stream);
}

const char *rnn_last_error(void) { return g_err; }

}  // extern "C"
