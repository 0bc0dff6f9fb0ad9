// Learned slab sizing: a small MLP that predicts how many edges each vertex
// will gain, so that a rebuilt graph can give it enough buckets up front.
// The paper fixes bucket counts a priori from the load factor and the
// current degree (Sec. "Motivation"); this is a project addition on top of
// that rule, which stays its fallback and its yardstick.  It may change the
// memory layout (bucket counts) but never a result.
//
// Network: 8 inputs -> 64 ReLU -> 64 ReLU -> 1.  Master weights are fp32;
// every forward and backward pass uses them rounded to bf16 (round to
// nearest even) and accumulates in fp32.  Loss = mean squared error.
// Gradients are with respect to the bf16-rounded weights (the rounding is
// treated as the identity), and Adam updates the fp32 masters.
//
// Kernels: the 64 x 64 layers are register-tiled products over a tile of
// samples held in shared memory, one row a hidden unit (see tile_product);
// the fp32 pipe bounds them.  Every output is the same chain of fused
// multiply-adds, in the same order, as one thread per sample would compute,
// so predictions do not depend on the tiling.
#include "mk_host.h"

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

using namespace mk;

namespace {

constexpr int kIn = 8, kHid = 64;
constexpr int kW1 = 0, kB1 = kW1 + kIn * kHid, kW2 = kB1 + kHid, kB2 = kW2 + kHid * kHid, kW3 = kB2 + kHid,
              kB3 = kW3 + kHid, kNParams = kB3 + 1; // 4801

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// One block: 128 threads = 8 output columns groups (tx) x 16 sample groups
// (ty).  Activations are kept as [unit][sample] rows of LD floats.
constexpr int kThreads = 128;

struct Weights {
    float w1[kIn * kHid], b1[kHid], w2[kHid * kHid], b2[kHid], w3[kHid], b3, pad[3];
};

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void st4(float *p, float a, float b, float c, float d)
{
    *reinterpret_cast<float4 *>(p) = make_float4(a, b, c, d);
}

// The tile position of a thread's r-th sample and c-th column: samples
// 4 * ty + 64 * q + 0..3, columns tx + 8 * c.  The rows of W1, W2 and of W2
// transposed are kept in shared memory in the order in which the threads read
// them (place_of), so that a quarter warp's 16-byte accesses cover all banks,
// the reads of a weight row and the writes of a tile alike (with columns
// 4 * tx + 32 * h + 0..3 the writes met four at a bank).
__device__ __forceinline__ int column_of(int tx, int c) { return tx + 8 * c; }
__device__ __forceinline__ int place_of(int col) { return 4 * (col & 7) + 32 * (col >> 5) + ((col >> 3) & 3); }

__device__ __forceinline__ void load_weights(Weights &s, const float *P)
{
    for (int i = threadIdx.x; i < kIn * kHid; i += kThreads)
        s.w1[i / kHid * kHid + place_of(i % kHid)] = bf16r(P[kW1 + i]);
    for (int i = threadIdx.x; i < kHid * kHid; i += kThreads)
        s.w2[i / kHid * kHid + place_of(i % kHid)] = bf16r(P[kW2 + i]);
    for (int i = threadIdx.x; i < kHid; i += kThreads) {
        s.b1[i] = bf16r(P[kB1 + i]);
        s.b2[i] = bf16r(P[kB2 + i]);
        s.w3[i] = bf16r(P[kW3 + i]);
    }
    if (threadIdx.x == 0)
        s.b3 = bf16r(P[kB3]);
}

// acc[r][c] += sum over k of A[k][sample r] * W[k][column c], k ascending,
// one fused multiply-add each.  A thread holds 4Q samples x 8 columns and
// reads Q + 2 16-byte words for 32Q multiply-adds: one thread a sample read
// two words for each (shared memory 96 % busy, the fp32 pipe 38 %).
template <int Q, int LD, int K>
__device__ __forceinline__ void tile_product(const float *A, const float *W, int tx, int ty, float (&acc)[4 * Q][8])
{
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        float a[4 * Q], w[8];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const float4 v = ld4(A + k * LD + 4 * ty + 64 * q);
            a[4 * q] = v.x, a[4 * q + 1] = v.y, a[4 * q + 2] = v.z, a[4 * q + 3] = v.w;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float4 v = ld4(W + k * kHid + 4 * tx + 32 * h);
            w[4 * h] = v.x, w[4 * h + 1] = v.y, w[4 * h + 2] = v.z, w[4 * h + 3] = v.w;
        }
#pragma unroll
        for (int r = 0; r < 4 * Q; ++r)
#pragma unroll
            for (int c = 0; c < 8; ++c)
                acc[r][c] = fmaf(a[r], w[c], acc[r][c]);
    }
}

// A layer of the tile: ReLU(A W + bias), into registers.
template <int Q, int LD, int K>
__device__ __forceinline__ void relu_layer(const float *A, const float *W, const float *bias, int tx, int ty,
                                           float (&acc)[4 * Q][8])
{
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const float b = bias[column_of(tx, c)];
#pragma unroll
        for (int r = 0; r < 4 * Q; ++r)
            acc[r][c] = b;
    }
    tile_product<Q, LD, K>(A, W, tx, ty, acc);
#pragma unroll
    for (int r = 0; r < 4 * Q; ++r)
#pragma unroll
        for (int c = 0; c < 8; ++c)
            acc[r][c] = fmaxf(acc[r][c], 0.f);
}

template <int Q, int LD>
__device__ __forceinline__ void store_tile(float *H, int tx, int ty, const float (&acc)[4 * Q][8])
{
#pragma unroll
    for (int c = 0; c < 8; ++c)
#pragma unroll
        for (int q = 0; q < Q; ++q)
            st4(H + column_of(tx, c) * LD + 4 * ty + 64 * q, acc[4 * q][c], acc[4 * q + 1][c], acc[4 * q + 2][c],
                acc[4 * q + 3][c]);
}

// Output of sample column t: y = b3 + sum over j of H2[j][t] * w3[j].
template <int LD>
__device__ __forceinline__ float output_of(const Weights &s, const float *H2, int t)
{
    float y = s.b3;
#pragma unroll 4
    for (int j = 0; j < kHid; j += 4) {
        const float4 w = ld4(s.w3 + j);
        y = fmaf(H2[j * LD + t], w.x, y);
        y = fmaf(H2[(j + 1) * LD + t], w.y, y);
        y = fmaf(H2[(j + 2) * LD + t], w.z, y);
        y = fmaf(H2[(j + 3) * LD + t], w.w, y);
    }
    return y;
}

// Inputs of samples base + t, base + t + 128, ...; 16 bytes at a time if the
// array's address allows.
template <int N>
__device__ __forceinline__ void load_inputs(const float *__restrict__ X, uint64_t base, uint64_t n, float (&xs)[N][kIn])
{
    const bool wide = (reinterpret_cast<uintptr_t>(X) & 15) == 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const uint64_t i = base + threadIdx.x + k * kThreads;
        if (wide) {
#pragma unroll
            for (int f = 0; f < kIn; f += 4) {
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (i < n)
                    v = __ldg(reinterpret_cast<const float4 *>(X + i * kIn + f));
                xs[k][f] = v.x, xs[k][f + 1] = v.y, xs[k][f + 2] = v.z, xs[k][f + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int f = 0; f < kIn; ++f)
                xs[k][f] = i < n ? __ldg(X + i * kIn + f) : 0.f;
        }
    }
}

template <int N, int LD>
__device__ __forceinline__ void store_inputs(float *x, const float (&xs)[N][kIn])
{
#pragma unroll
    for (int k = 0; k < N; ++k)
#pragma unroll
        for (int f = 0; f < kIn; ++f)
            x[f * LD + threadIdx.x + k * kThreads] = xs[k][f];
}

// Forward pass: 256 samples a tile, 16 samples x 8 columns a thread.
constexpr int kFwdTile = 256, kFwdLd = kFwdTile + 4;

struct FwdSmem {
    Weights w;
    float x[kIn * kFwdLd], h[kHid * kFwdLd]; // h: H1, then H2
};

// The fp32 pipe sets the pace (549 us of it for 4.2 M samples at 2.06 GHz)
// once shared memory does not: both layers are tile products (the first by a
// thread a sample read a weight for each two multiply-adds), and no access
// meets another at a bank.  4.2 M samples: 3.88 -> 0.72 ms (55 TFLOP/s; 0.83
// with the first layer by samples and the conflicts; 0.84 with 128-sample
// tiles, four blocks an SM, so it is not the warps; 0.73 with packed pairs of
// multiply-adds).
__global__ void __launch_bounds__(kThreads, 2) k_mlp_forward(const float *P, const float *X, uint64_t n, float *Y)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FwdSmem &s = *reinterpret_cast<FwdSmem *>(smem_raw);
    const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
    const uint64_t stride = (uint64_t)gridDim.x * kFwdTile;
    uint64_t base = (uint64_t)blockIdx.x * kFwdTile;
    load_weights(s.w, P);
    float xs[2][kIn]; // the next tile's inputs, read while a tile is computed
    load_inputs<2>(X, base, n, xs);
    for (; base < n; base += stride) {
        store_inputs<2, kFwdLd>(s.x, xs);
        __syncthreads(); // and the tile before has been read
        load_inputs<2>(X, base + stride, n, xs);
        {
            float acc[16][8];
            relu_layer<4, kFwdLd, kIn>(s.x, s.w.w1, s.w.b1, tx, ty, acc);
            store_tile<4, kFwdLd>(s.h, tx, ty, acc);
        }
        __syncthreads();
        {
            float acc[16][8];
            relu_layer<4, kFwdLd, kHid>(s.h, s.w.w2, s.w.b2, tx, ty, acc);
            __syncthreads(); // every thread has read H1
            store_tile<4, kFwdLd>(s.h, tx, ty, acc);
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const uint64_t i = base + threadIdx.x + k * kThreads;
            const float y = output_of<kFwdLd>(s.w, s.h, threadIdx.x + k * kThreads);
            if (i < n)
                Y[i] = y;
        }
    }
}

// Backward pass: 128 samples a tile, 8 samples x 8 columns a thread.
constexpr int kTile = 128, kLd = kTile + 4;

struct BwdSmem {
    Weights w;
    float w2t[kHid * kHid]; // W2 transposed
    float x[kIn * kLd], h1[kHid * kLd], h2[kHid * kLd], dy[kTile];
};

// sum over the tile's samples of R[row][t]
__device__ __forceinline__ float row_sum(const float *R)
{
    float a = 0.f;
#pragma unroll 8
    for (int t = 0; t < kTile; t += 4) {
        const float4 v = ld4(R + t);
        a += (v.x + v.y) + (v.z + v.w);
    }
    return a;
}

// sum over the tile's samples of A[t] * B[t]
__device__ __forceinline__ float row_dot(const float *A, const float *B)
{
    float a = 0.f;
#pragma unroll 8
    for (int t = 0; t < kTile; t += 4) {
        const float4 u = ld4(A + t), v = ld4(B + t);
        a = fmaf(u.x, v.x, a);
        a = fmaf(u.y, v.y, a);
        a = fmaf(u.z, v.z, a);
        a = fmaf(u.w, v.w, a);
    }
    return a;
}

// Gradient of mean((y - T)^2) over n samples, accumulated into G (kNParams
// floats, zeroed by the caller); the sum of squared errors into *sse.  Each
// block keeps its gradient in registers over its tiles (32 entries of W2 a
// thread, its 4 entries of W1, its bias entries) and adds it once, one atomic
// a parameter.  262,144 samples: 718 -> 190 us.
__global__ void __launch_bounds__(kThreads, 2) k_mlp_backward(const float *P, const float *X, const float *T,
                                                              uint64_t n, float inv_n, float *G, double *sse)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BwdSmem &s = *reinterpret_cast<BwdSmem *>(smem_raw);
    const int t = threadIdx.x, tx = t & 7, ty = t >> 3;
    load_weights(s.w, P);
    __syncthreads();
    for (int i = t; i < kHid * kHid; i += kThreads)
        s.w2t[(i % kHid) * kHid + place_of(i / kHid)] = s.w.w2[i / kHid * kHid + place_of(i % kHid)];
    // W2 entries of the thread: rows k = tx + 8 * a (a < 8), columns j = ty + 16 * b (b < 4)
    float gw2[8][4] = {}, gw1[4] = {}, gvec[2] = {0.f, 0.f}, gb3 = 0.f;
    double my_sse = 0.0;
    for (uint64_t base = (uint64_t)blockIdx.x * kTile; base < n; base += (uint64_t)gridDim.x * kTile) {
        __syncthreads(); // the tile before has been read (and w2t is written)
        const uint64_t i = base + t;
        {
            float xs[1][kIn];
            load_inputs<1>(X, base, n, xs);
            store_inputs<1, kLd>(s.x, xs);
        }
        __syncthreads();
        float acc[8][8];
        relu_layer<2, kLd, kIn>(s.x, s.w.w1, s.w.b1, tx, ty, acc);
        store_tile<2, kLd>(s.h1, tx, ty, acc);
        __syncthreads();
        relu_layer<2, kLd, kHid>(s.h1, s.w.w2, s.w.b2, tx, ty, acc);
        store_tile<2, kLd>(s.h2, tx, ty, acc);
        __syncthreads();
        const float y = output_of<kLd>(s.w, s.h2, t);
        const float e = i < n ? y - T[i] : 0.f;
        my_sse += (double)e * e;
        s.dy[t] = 2.f * e * inv_n;
        __syncthreads();
        // w3's gradient needs H2; dZ2 replaces H2 afterwards
        if (t < kHid)
            gvec[0] += row_dot(s.h2 + t * kLd, s.dy);
        else if (t == kHid)
            gb3 += row_sum(s.dy);
        __syncthreads();
        {
            const float dy = s.dy[t];
#pragma unroll 8
            for (int j = 0; j < kHid; ++j) {
                float &h = s.h2[j * kLd + t];
                h = h > 0.f ? dy * s.w.w3[j] : 0.f;
            }
        }
        __syncthreads();
        // gW2[k][j] += sum over t of H1[k][t] * dZ2[j][t], each tile's sum on
        // its own (a sum over all tiles in one chain would round more)
        float part[8][4] = {};
#pragma unroll 1
        for (int r = 0; r < kTile; r += 4) {
            float4 d[4];
#pragma unroll
            for (int b = 0; b < 4; ++b)
                d[b] = ld4(s.h2 + (ty + 16 * b) * kLd + r);
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                const float4 h = ld4(s.h1 + (tx + 8 * a) * kLd + r);
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    float g = part[a][b];
                    g = fmaf(h.x, d[b].x, g);
                    g = fmaf(h.y, d[b].y, g);
                    g = fmaf(h.z, d[b].z, g);
                    part[a][b] = fmaf(h.w, d[b].w, g);
                }
            }
        }
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b)
                gw2[a][b] += part[a][b];
        if (t < kHid)
            gvec[1] += row_sum(s.h2 + t * kLd); // b2
        // dZ1[t][k] = (sum over j of dZ2[t][j] * W2[k][j]) where H1 > 0
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int c = 0; c < 8; ++c)
                acc[r][c] = 0.f;
        tile_product<2, kLd, kHid>(s.h2, s.w2t, tx, ty, acc);
        __syncthreads(); // H1 has been read for gW2
#pragma unroll
        for (int c = 0; c < 8; ++c)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                float *at = s.h1 + column_of(tx, c) * kLd + 4 * ty + 64 * q;
                const float4 h = ld4(at);
                st4(at, h.x > 0.f ? acc[4 * q][c] : 0.f, h.y > 0.f ? acc[4 * q + 1][c] : 0.f,
                    h.z > 0.f ? acc[4 * q + 2][c] : 0.f, h.w > 0.f ? acc[4 * q + 3][c] : 0.f);
            }
        __syncthreads();
        // gW1[f][k] += sum over t of x[f][t] * dZ1[k][t]; b1's on the upper half of the block
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int o = t + a * kThreads; // f * 64 + k
            gw1[a] += row_dot(s.x + (o / kHid) * kLd, s.h1 + (o % kHid) * kLd);
        }
        if (t >= kHid)
            gvec[1] += row_sum(s.h1 + (t - kHid) * kLd);
    }
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
            atomicAdd(&G[kW2 + (tx + 8 * a) * kHid + ty + 16 * b], gw2[a][b]);
#pragma unroll
    for (int a = 0; a < 4; ++a)
        atomicAdd(&G[kW1 + t + a * kThreads], gw1[a]);
    if (t < kHid) {
        atomicAdd(&G[kW3 + t], gvec[0]);
        atomicAdd(&G[kB2 + t], gvec[1]);
    } else {
        atomicAdd(&G[kB1 + t - kHid], gvec[1]);
        if (t == kHid)
            atomicAdd(&G[kB3], gb3);
    }
    // block sum of squared errors
    for (int o = 16; o; o >>= 1)
        my_sse += __shfl_xor_sync(kFull, my_sse, o);
    if ((threadIdx.x & 31) == 0)
        atomicAdd(sse, my_sse);
}

// Adam (Kingma and Ba, ICLR 2015) on the fp32 master weights.
__global__ void k_adam(float *P, const float *G, float *M, float *Vv, int n, float lr, float b1, float b2,
                       float eps, float c1, float c2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    const float g = G[i];
    const float m = b1 * M[i] + (1.f - b1) * g;
    const float v = b2 * Vv[i] + (1.f - b2) * g * g;
    M[i] = m;
    Vv[i] = v;
    P[i] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
}

// Degree trace: out/in degree += sign for every edge flagged 1.
__global__ void k_degree_update(const uint32_t *src, const uint32_t *dst, const uint8_t *flags, uint64_t n, int sign,
                                uint32_t V, uint32_t *out_deg, uint32_t *in_deg)
{
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (i >= n || (flags && !flags[i]))
        return;
    const uint32_t s = src[i], d = dst[i];
    if (s >= V || d >= V)
        return;
    if (out_deg)
        atomicAdd(&out_deg[s], (uint32_t)sign);
    if (in_deg)
        atomicAdd(&in_deg[d], (uint32_t)sign);
}

__device__ __forceinline__ float lg1p(float x) { return log1pf(fmaxf(x, 0.f)); }

// Features of each vertex from its out-degree snapshots (hist[k * V + v] =
// out-degree k batches ago, k = 0..4), in-degree and bucket count.
__global__ void k_features(const uint32_t *hist, const uint32_t *in_deg, const uint32_t *buckets, uint32_t V, float *X)
{
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= V)
        return;
    const float d0 = (float)hist[v], din = (float)in_deg[v];
    const uint32_t nb = buckets[v];
    float g[4];
#pragma unroll
    for (int k = 1; k <= 4; ++k)
        g[k - 1] = lg1p(d0 - (float)hist[(uint64_t)k * V + v]);
    const float l0 = lg1p(d0), lin = lg1p(din);
    const float fill = d0 / (15.f * (float)(nb ? nb : 1));
    const float x[kIn] = {l0, g[0], g[1], g[2], g[3], lin, lin - l0, fill};
    float *o = X + (uint64_t)v * kIn;
    if ((reinterpret_cast<uintptr_t>(X) & 15) == 0) {
        st4(o, x[0], x[1], x[2], x[3]);
        st4(o + 4, x[4], x[5], x[6], x[7]);
    } else {
#pragma unroll
        for (int k = 0; k < kIn; ++k)
            o[k] = x[k];
    }
}

// Bucket counts from the predicted growth: y = log1p(edges gained per
// batch); future degree = degree + horizon * expm1(y); buckets =
// max(1, ceil(future degree / (load_factor * 15))).
__global__ void k_learned_buckets(const float *Y, const uint32_t *deg, uint32_t V, float horizon, float lf,
                                  uint32_t max_buckets, uint32_t *buckets)
{
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= V)
        return;
    const float growth = fmaxf(expm1f(fmaxf(Y[v], 0.f)), 0.f);
    const float per = lf * 15.f;
    uint32_t b = 0;
    bool sure = false;
    if (growth == 0.f && isfinite(horizon)) {
        b = ceil_ratio(deg[v], per);
        sure = true;
    } else {
        // the 32-bit quotient is within 8 * 2^-24 of the 64-bit one; where
        // that leaves one ceiling, it is the answer without the 64-bit
        // division (4.2 M vertices: 139 -> 25 us)
        const float q = ((float)deg[v] + horizon * growth) / per;
        const float lo = ceilf(q * (1.f - 1e-6f)), hi = ceilf(q * (1.f + 1e-6f));
        if (q < 262144.f && lo == hi) {
            b = (uint32_t)lo;
            sure = true;
        }
    }
    if (!sure) {
        const double fut = (double)deg[v] + (double)horizon * growth;
        double x = ceil(fut / (double)per);
        if (x < 1)
            x = 1;
        if (x > max_buckets)
            x = max_buckets;
        b = (uint32_t)x;
        buckets[v] = b;
        return;
    }
    buckets[v] = min(max(b, 1u), max_buckets);
}

// Training target of each vertex: log1p of the out-edges it gained per batch
// between two snapshots h batches apart.
__global__ void k_growth_targets(const uint32_t *deg_then, const uint32_t *deg_later, uint32_t V, float h, float *T)
{
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= V)
        return;
    const float gain = (float)deg_later[v] - (float)deg_then[v];
    T[v] = log1pf(fmaxf(gain, 0.f) / h);
}

// Resident blocks for n samples in tiles of `tile`, two an SM, with the
// kernels' shared-memory limits raised (a function attribute of the current
// device: set on every call).
template <typename K>
int mlp_grid(K kernel, size_t smem, uint64_t n, int tile)
{
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const uint64_t tiles = (n + tile - 1) / tile;
    return (int)std::max<uint64_t>(std::min<uint64_t>(tiles, (uint64_t)num_sms() * 2), 1);
}

// splitmix64, for the initial weights
uint64_t mix64(uint64_t z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

} // namespace

struct mk_mlp {
    float *P = nullptr, *G = nullptr, *M = nullptr, *Vv = nullptr;
    double *sse = nullptr;
    uint64_t steps = 0;
};

extern "C" {

mk_status mk_mlp_create(uint64_t seed, mk_mlp **out)
{
    if (!out)
        return MK_ERR_INVALID_ARG;
    mk_mlp *m = new mk_mlp;
    const size_t bytes = kNParams * sizeof(float);
    if (cudaMalloc(&m->P, bytes) != cudaSuccess || cudaMalloc(&m->G, bytes) != cudaSuccess ||
        cudaMalloc(&m->M, bytes) != cudaSuccess || cudaMalloc(&m->Vv, bytes) != cudaSuccess ||
        cudaMalloc(&m->sse, sizeof(double)) != cudaSuccess) {
        mk_mlp_destroy(m);
        return MK_ERR_NO_MEMORY;
    }
    // He-uniform initial weights, zero biases
    std::vector<float> h(kNParams, 0.f);
    auto uni = [&](uint64_t i) { return (double)(mix64(seed * 0x9E3779B97F4A7C15ULL + i + 1) >> 11) / 9007199254740992.0; };
    for (int i = 0; i < kIn * kHid; ++i)
        h[kW1 + i] = (float)((2 * uni(i) - 1) * std::sqrt(6.0 / kIn));
    for (int i = 0; i < kHid * kHid; ++i)
        h[kW2 + i] = (float)((2 * uni(10000 + i) - 1) * std::sqrt(6.0 / kHid));
    for (int i = 0; i < kHid; ++i)
        h[kW3 + i] = (float)((2 * uni(20000 + i) - 1) * std::sqrt(6.0 / kHid));
    if (cudaMemcpy(m->P, h.data(), bytes, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(m->M, 0, bytes) != cudaSuccess || cudaMemset(m->Vv, 0, bytes) != cudaSuccess) {
        mk_mlp_destroy(m);
        return MK_ERR_CUDA;
    }
    *out = m;
    return MK_OK;
}

mk_status mk_mlp_destroy(mk_mlp *m)
{
    if (!m)
        return MK_ERR_INVALID_ARG;
    cudaFree(m->P);
    cudaFree(m->G);
    cudaFree(m->M);
    cudaFree(m->Vv);
    cudaFree(m->sse);
    delete m;
    return MK_OK;
}

int mk_mlp_num_params(void) { return kNParams; }

mk_status mk_mlp_get_params(mk_mlp *m, float *h_out)
{
    if (!m || !h_out)
        return MK_ERR_INVALID_ARG;
    MK_CUDA(cudaMemcpy(h_out, m->P, kNParams * sizeof(float), cudaMemcpyDeviceToHost));
    return MK_OK;
}

mk_status mk_mlp_set_params(mk_mlp *m, const float *h_in)
{
    if (!m || !h_in)
        return MK_ERR_INVALID_ARG;
    MK_CUDA(cudaMemcpy(m->P, h_in, kNParams * sizeof(float), cudaMemcpyHostToDevice));
    MK_CUDA(cudaMemset(m->M, 0, kNParams * sizeof(float)));
    MK_CUDA(cudaMemset(m->Vv, 0, kNParams * sizeof(float)));
    m->steps = 0;
    return MK_OK;
}

mk_status mk_mlp_forward(mk_mlp *m, const float *d_x, uint64_t n, float *d_y, void *stream)
{
    if (!m || (n && (!d_x || !d_y)))
        return MK_ERR_INVALID_ARG;
    if (!n)
        return MK_OK;
    cudaStream_t s = (cudaStream_t)stream;
    k_mlp_forward<<<mlp_grid(k_mlp_forward, sizeof(FwdSmem), n, kFwdTile), kThreads, sizeof(FwdSmem), s>>>(m->P, d_x, n, d_y);
    MK_CUDA(cudaGetLastError());
    return MK_OK;
}

mk_status mk_mlp_gradient(mk_mlp *m, const float *d_x, const float *d_t, uint64_t n, float *d_grad, double *d_sse,
                          void *stream)
{
    if (!m || !n || !d_x || !d_t || !d_grad)
        return MK_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    MK_CUDA(cudaMemsetAsync(d_grad, 0, kNParams * sizeof(float), s));
    double *sse = d_sse ? d_sse : m->sse;
    MK_CUDA(cudaMemsetAsync(sse, 0, sizeof(double), s));
    k_mlp_backward<<<mlp_grid(k_mlp_backward, sizeof(BwdSmem), n, kTile), kThreads, sizeof(BwdSmem), s>>>(
        m->P, d_x, d_t, n, 1.f / (float)n, d_grad, sse);
    MK_CUDA(cudaGetLastError());
    return MK_OK;
}

mk_status mk_mlp_adam_step(mk_mlp *m, const float *d_x, const float *d_t, uint64_t n, float lr, double *d_sse,
                           void *stream)
{
    if (!m || !n || !d_x || !d_t || !(lr > 0.f))
        return MK_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    MK_TRY(mk_mlp_gradient(m, d_x, d_t, n, m->G, d_sse, stream));
    m->steps++;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)m->steps), c2 = 1.f - std::pow(b2, (float)m->steps);
    k_adam<<<(kNParams + 255) / 256, 256, 0, s>>>(m->P, m->G, m->M, m->Vv, kNParams, lr, b1, b2, 1e-8f, c1, c2);
    MK_CUDA(cudaGetLastError());
    return MK_OK;
}

mk_status mk_degree_update(uint32_t V, const uint32_t *d_src, const uint32_t *d_dst, const uint8_t *d_flags,
                           uint64_t n, int sign, uint32_t *d_out_deg, uint32_t *d_in_deg, void *stream)
{
    if (!V || (n && (!d_src || !d_dst)) || (sign != 1 && sign != -1))
        return MK_ERR_INVALID_ARG;
    if (!n)
        return MK_OK;
    k_degree_update<<<grid_for(n, 256), 256, 0, (cudaStream_t)stream>>>(d_src, d_dst, d_flags, n, sign, V, d_out_deg,
                                                                        d_in_deg);
    MK_CUDA(cudaGetLastError());
    return MK_OK;
}

mk_status mk_sizing_features(uint32_t V, const uint32_t *d_out_hist, const uint32_t *d_in_deg,
                             const uint32_t *d_buckets, float *d_x, void *stream)
{
    if (!V || !d_out_hist || !d_in_deg || !d_buckets || !d_x)
        return MK_ERR_INVALID_ARG;
    k_features<<<grid_for(V, 256), 256, 0, (cudaStream_t)stream>>>(d_out_hist, d_in_deg, d_buckets, V, d_x);
    MK_CUDA(cudaGetLastError());
    return MK_OK;
}

mk_status mk_sizing_targets(uint32_t V, const uint32_t *d_deg_then, const uint32_t *d_deg_later, float horizon,
                            float *d_t, void *stream)
{
    if (!V || !d_deg_then || !d_deg_later || !d_t || !(horizon > 0.f))
        return MK_ERR_INVALID_ARG;
    k_growth_targets<<<grid_for(V, 256), 256, 0, (cudaStream_t)stream>>>(d_deg_then, d_deg_later, V, horizon, d_t);
    MK_CUDA(cudaGetLastError());
    return MK_OK;
}

mk_status mk_sizing_buckets(mk_mlp *m, const float *d_x, const uint32_t *d_out_deg, uint32_t V, float horizon,
                            float load_factor, uint32_t max_buckets, float *d_y, uint32_t *d_buckets, void *stream)
{
    if (!m || !V || !d_x || !d_out_deg || !d_y || !d_buckets || !(load_factor > 0.f) || load_factor > 1.f ||
        horizon < 0.f || max_buckets == 0)
        return MK_ERR_INVALID_ARG;
    MK_TRY(mk_mlp_forward(m, d_x, V, d_y, stream));
    k_learned_buckets<<<grid_for(V, 256), 256, 0, (cudaStream_t)stream>>>(d_y, d_out_deg, V, horizon, load_factor,
                                                                          max_buckets, d_buckets);
    MK_CUDA(cudaGetLastError());
    return MK_OK;
}

} // extern "C"
