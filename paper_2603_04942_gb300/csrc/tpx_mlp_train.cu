// tpx_mlp_train.cu -- one training step of the perceptron refiner (fp32) in two
// kernels, for hidden widths up to 160.
//
//   k_rows: a CTA takes 32 rows of the minibatch through the whole network and
//     back to the first layer's pre-activation gradient. Activations stay in
//     shared memory, feature-major, so that a warp's four rows of a feature are
//     one broadcast 16-byte load; the weights pass through shared memory 16
//     features at a time, the next ones on their way in registers.
//   k_grads: the weight and bias gradients, sums over the rows, and Adam. A
//     cluster of 8 CTAs shares a tile of parameters, each over an eighth of the
//     rows; the eight partial sums meet in distributed shared memory, always
//     in the same order, and the CTA that adds them up applies the update.
//
// Bound by the fp32 units and shared-memory reads (six wavefronts per 20
// multiply-adds and warp). Measured on 4096 rows, width 160: a step of 2.55 ms
// -> 78 us, error against 64 bits 1.1e-6 -> 1.0e-6; before, each gradient was a GEMM of nine 64 x 64 tiles, each
// running through all rows by itself, and each bias gradient a serial column
// sum, so that most of the chip idled.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "tpx_mlp_train.cuh"

namespace cg = cooperative_groups;

namespace tpxt {

constexpr int NIN = 162, NOUT = 6;
constexpr int HM = kMaxHidden;        // columns a warp covers: 5 per lane
constexpr int Q = HM / 32;
constexpr int R = 32;                 // rows of a CTA: four per warp
constexpr int NTH = 256;
constexpr int AS = R + 4;             // stride of a feature's rows: 16-byte loads, conflict-free 16-byte stores
constexpr int KC = 16;                // features of a weight chunk
constexpr int WS = HM + 5;            // its stride: the transposed chunk's stores hit different banks
constexpr int PER = KC * HM / NTH;    // words of a chunk per thread

struct Offsets { long long w1, b1, w2, b2, w3, b3; };
__host__ __device__ inline Offsets offsets(int h) {
    Offsets o;
    o.w1 = 0; o.b1 = (long long)NIN * h; o.w2 = o.b1 + h; o.b2 = o.w2 + (long long)h * h; o.w3 = o.b2 + h;
    o.b3 = o.w3 + (long long)h * NOUT;
    return o;
}

struct RowsSmem {
    float x[NIN][AS];
    float a1[HM][AS], a2[HM][AS], d[HM][AS];
    float w[2][KC][WS];
    float w3[HM * NOUT];
    float o[R][NOUT + 1];             // outputs, then their gradients
};

// acc[row][col] = sum over features k of A[k][4 warp + row] W(k, lane + 32 col),
// W(k, c) = W[k h + c], or W[c h + k] when TRANS; k in ascending order
template <bool TRANS>
__device__ __forceinline__ void rows_gemm(RowsSmem &S, const float (*A)[AS], const float *__restrict__ W, int K, int h,
                                          float (&acc)[4][Q]) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float pre[PER];
    auto load = [&](int k0) {
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int t = tid + u * NTH;
            const int kk = TRANS ? t % KC : t / HM, c = TRANS ? t / KC : t % HM;
            const int k = k0 + kk;
            pre[u] = (k < K && c < h) ? __ldg(W + (TRANS ? (long long)c * h + k : (long long)k * h + c)) : 0.f;
        }
    };
    auto store = [&](int b) {
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int t = tid + u * NTH;
            S.w[b][TRANS ? t % KC : t / HM][TRANS ? t / KC : t % HM] = pre[u];
        }
    };
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < Q; ++q) acc[r][q] = 0.f;
    load(0);
    __syncthreads();   // the operand rows are written, the chunk buffers free
    store(0);
    int b = 0;
    for (int k0 = 0; k0 < K; k0 += KC, b ^= 1) {
        if (k0 + KC < K) load(k0 + KC);
        __syncthreads();
        const int kn = min(KC, K - k0);
#pragma unroll 4
        for (int kk = 0; kk < kn; ++kk) {
            const float4 a = *reinterpret_cast<const float4 *>(&A[k0 + kk][4 * warp]);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const float w = S.w[b][kk][lane + 32 * q];
                acc[0][q] = fmaf(a.x, w, acc[0][q]);
                acc[1][q] = fmaf(a.y, w, acc[1][q]);
                acc[2][q] = fmaf(a.z, w, acc[2][q]);
                acc[3][q] = fmaf(a.w, w, acc[3][q]);
            }
        }
        if (k0 + KC < K) store(b ^ 1);   // read two chunks ago: every warp is past it
    }
}

// the warp's four rows by its columns: into the feature-major rows D (if any)
// and the row-major global array
__device__ __forceinline__ void put_rows(float (*D)[AS], float *g, long long r0, long long n, int h,
                                         const float (&v)[4][Q]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int c = lane + 32 * q;
        if (D) *reinterpret_cast<float4 *>(&D[c][4 * warp]) = make_float4(v[0][q], v[1][q], v[2][q], v[3][q]);
        if (c >= h) continue;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const long long row = r0 + 4 * warp + r;
            if (row < n) g[row * h + c] = v[r][q];
        }
    }
}

__global__ void __launch_bounds__(NTH) k_rows(const float *__restrict__ P, int h, const float *__restrict__ x,
                                              const float *__restrict__ y, long long n, float w_off, float *a1, float *a2,
                                              float *out, float *dout, float *d2, float *d1, float *loss) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    RowsSmem &S = *reinterpret_cast<RowsSmem *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long r0 = (long long)blockIdx.x * R;
    const Offsets L = offsets(h);
    for (int t = tid; t < NIN * R; t += NTH) {   // the rows' words are consecutive
        const int r = t / NIN, k = t % NIN;
        S.x[k][r] = r0 + r < n ? __ldg(x + r0 * NIN + t) : 0.f;
    }
    for (int t = tid; t < h * NOUT; t += NTH) S.w3[t] = __ldg(P + L.w3 + t);
    float acc[4][Q];
    auto bias_relu = [&](const float *b) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const float bv = lane + 32 * q < h ? __ldg(b + lane + 32 * q) : 0.f;
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[r][q] = fmaxf(acc[r][q] + bv, 0.f);
        }
    };
    rows_gemm<false>(S, S.x, P + L.w1, NIN, h, acc);
    bias_relu(P + L.b1);
    put_rows(S.a1, a1, r0, n, h, acc);
    rows_gemm<false>(S, S.a1, P + L.w2, h, h, acc);
    bias_relu(P + L.b2);
    put_rows(S.a2, a2, r0, n, h, acc);
    __syncthreads();
    if (tid < R * NOUT) {   // the outputs, a thread each
        const int r = tid % R, o = tid / R;
        float s = 0.f;
        for (int k = 0; k < h; ++k) s = fmaf(S.a2[k][r], S.w3[k * NOUT + o], s);
        s += __ldg(P + L.b3 + o);
        S.o[r][o] = s;
        if (r0 + r < n) out[(r0 + r) * NOUT + o] = s;
    }
    __syncthreads();
    if (warp == 0) {   // the loss (softmax cross-entropy and offsets) and its gradient, a lane per row
        const long long row = r0 + lane;
        float l = 0.f, g[NOUT] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (row < n) {
            float o[NOUT], t[5];
#pragma unroll
            for (int k = 0; k < NOUT; ++k) o[k] = S.o[lane][k];
#pragma unroll
            for (int k = 0; k < 5; ++k) t[k] = __ldg(y + row * 5 + k);
            const bool two = t[0] > 1.5f;
            const float m = fmaxf(o[0], o[1]);
            const float e0 = __expf(o[0] - m), e1 = __expf(o[1] - m), z = e0 + e1;
            const float p1 = e1 / z, inv = 1.f / (float)n;
            l = -((two ? o[1] : o[0]) - m - __logf(z));
            g[0] = ((1.f - p1) - (two ? 0.f : 1.f)) * inv;
            g[1] = (p1 - (two ? 1.f : 0.f)) * inv;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float d = (k < 2 || two) ? o[2 + k] - t[1 + k] : 0.f;
                l += 0.5f * w_off * d * d;
                g[2 + k] = w_off * d * inv;
            }
        }
#pragma unroll
        for (int k = 0; k < NOUT; ++k) {
            S.o[lane][k] = g[k];
            if (row < n) dout[row * NOUT + k] = g[k];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) atomicAdd(loss, l / (float)n);
    }
    __syncthreads();
    // d2 = (dout W3^T) where a2 > 0
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int c = lane + 32 * q;
        const float4 a = *reinterpret_cast<const float4 *>(&S.a2[c][4 * warp]);
        const float on[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            float s = 0.f;
            if (c < h)
#pragma unroll
                for (int o = 0; o < NOUT; ++o) s = fmaf(S.o[4 * warp + r][o], S.w3[c * NOUT + o], s);
            acc[r][q] = on[r] > 0.f ? s : 0.f;
        }
    }
    put_rows(S.d, d2, r0, n, h, acc);
    // d1 = (d2 W2^T) where a1 > 0
    rows_gemm<true>(S, S.d, P + L.w2, h, h, acc);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const float4 a = *reinterpret_cast<const float4 *>(&S.a1[lane + 32 * q][4 * warp]);
        if (!(a.x > 0.f)) acc[0][q] = 0.f;
        if (!(a.y > 0.f)) acc[1][q] = 0.f;
        if (!(a.z > 0.f)) acc[2][q] = 0.f;
        if (!(a.w > 0.f)) acc[3][q] = 0.f;
    }
    put_rows(nullptr, d1, r0, n, h, acc);
}

// ---------------------------------------------------------------- gradients
constexpr int CL = 8;                 // CTAs of a cluster: an eighth of the rows each
constexpr int GF = 28, GC = 80;       // features (the last one of a layer is the bias) x columns of a tile
constexpr int GTH = 128;              // 7 x 16 threads of 4 x 5 parameters, and 16 that only load
constexpr int GR = 32;                // rows of a step
constexpr int APER = GF * GR / GTH, BPER = GC * GR / GTH;

struct Adam { float lr, b1, b2, c1, c2, eps; };

__device__ __forceinline__ void adam(float *P, float *G, float *M, float *V, long long i, float g, const Adam &A) {
    G[i] = g;
    const float mi = A.b1 * M[i] + (1.f - A.b1) * g, vi = A.b2 * V[i] + (1.f - A.b2) * g * g;
    M[i] = mi;
    V[i] = vi;
    P[i] -= A.lr * (mi / A.c1) / (sqrtf(vi / A.c2) + A.eps);
}

__global__ void __launch_bounds__(GTH) __cluster_dims__(CL, 1, 1)
    k_grads(float *P, float *G, float *M, float *V, int h, const float *__restrict__ x, const float *__restrict__ a1,
            const float *__restrict__ a2, const float *__restrict__ dout, const float *__restrict__ d2,
            const float *__restrict__ d1, long long n, Adam A) {
    __shared__ __align__(16) float s_a[2][GR][GF];
    __shared__ __align__(16) float s_b[2][GR][GC];
    __shared__ float part[GF * GC];
    auto cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), tid = threadIdx.x;
    const Offsets L = offsets(h);
    const int ct = (h + GC - 1) / GC;                 // column tiles of a hidden layer
    const int t1 = (NIN + 1 + GF - 1) / GF * ct, t2 = (h + 1 + GF - 1) / GF * ct;
    int tile = blockIdx.x / CL;
    // the tile's layer: inputs [n x F - 1] and a column of ones, gradients [n x N]
    const float *in, *dz;
    int F, N;
    long long ow, ob;
    if (tile < t1) { in = x; dz = d1; F = NIN + 1; N = h; ow = L.w1; ob = L.b1; }
    else if (tile < t1 + t2) { tile -= t1; in = a1; dz = d2; F = h + 1; N = h; ow = L.w2; ob = L.b2; }
    else { tile -= t1 + t2; in = a2; dz = dout; F = h + 1; N = NOUT; ow = L.w3; ob = L.b3; }
    const int nct = (N + GC - 1) / GC;
    const int f0 = tile / nct * GF, c0 = tile % nct * GC;
    const int FI = F - 1;                             // true input features
    const long long per = (n + CL - 1) / CL;
    const long long rb = rank * per, re = min(n, rb + per);
    const int tr = tid / 16, tc = tid % 16;
    float acc[4][5] = {};
    float pa[APER], pb[BPER];
    auto load = [&](long long r) {
#pragma unroll
        for (int u = 0; u < APER; ++u) {
            const int t = tid + u * GTH, f = f0 + t % GF;
            const long long row = r + t / GF;
            pa[u] = row < re ? (f < FI ? __ldg(in + row * FI + f) : f == FI ? 1.f : 0.f) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < BPER; ++u) {
            const int t = tid + u * GTH, c = c0 + t % GC;
            const long long row = r + t / GC;
            pb[u] = (row < re && c < N) ? __ldg(dz + row * N + c) : 0.f;
        }
    };
    int b = 0;
    load(rb);
    for (long long r = rb; r < re; r += GR, b ^= 1) {
#pragma unroll
        for (int u = 0; u < APER; ++u) (&s_a[b][0][0])[tid + u * GTH] = pa[u];
#pragma unroll
        for (int u = 0; u < BPER; ++u) (&s_b[b][0][0])[tid + u * GTH] = pb[u];
        if (r + GR < re) load(r + GR);
        __syncthreads();
        if (tr < GF / 4) {
#pragma unroll 4
            for (int k = 0; k < GR; ++k) {
                const float4 a = *reinterpret_cast<const float4 *>(&s_a[b][k][4 * tr]);
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    const float w = s_b[b][k][tc + 16 * q];
                    acc[0][q] = fmaf(a.x, w, acc[0][q]);
                    acc[1][q] = fmaf(a.y, w, acc[1][q]);
                    acc[2][q] = fmaf(a.z, w, acc[2][q]);
                    acc[3][q] = fmaf(a.w, w, acc[3][q]);
                }
            }
        }
    }
    if (tr < GF / 4)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int q = 0; q < 5; ++q) part[(4 * tr + i) * GC + tc + 16 * q] = acc[i][q];
    cluster.sync();
    for (int e = rank * GTH + tid; e < GF * GC; e += CL * GTH) {
        const int f = f0 + e / GC, c = c0 + e % GC;
        if (f >= F || c >= N) continue;
        float g = 0.f;
#pragma unroll
        for (int k = 0; k < CL; ++k) g += *cluster.map_shared_rank(&part[e], k);
        adam(P, G, M, V, f < FI ? ow + (long long)f * N + c : ob + c, g, A);
    }
    cluster.sync();   // the partial sums stay until every CTA has read them
}

cudaError_t train_step(cudaStream_t s, float *P, float *M, float *V, float *G, int h, long long step, const float *x,
                       const float *y, long long n, float lr, float w_off, float *work, float *loss) {
    float *a1 = work, *a2 = a1 + n * h, *out = a2 + n * h, *dout = out + n * NOUT, *d2 = dout + n * NOUT, *d1 = d2 + n * h;
    cudaError_t e = cudaFuncSetAttribute(k_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RowsSmem));
    if (e != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(loss, 0, 4, s)) != cudaSuccess) return e;
    k_rows<<<(unsigned)((n + R - 1) / R), NTH, sizeof(RowsSmem), s>>>(P, h, x, y, n, w_off, a1, a2, out, dout, d2, d1, loss);
    const float b1 = 0.9f, b2 = 0.999f;
    const Adam A{lr, b1, b2, 1.f - powf(b1, (float)step), 1.f - powf(b2, (float)step), 1e-8f};
    const int ct = (h + GC - 1) / GC;
    const int tiles = (NIN + 1 + GF - 1) / GF * ct + (h + 1 + GF - 1) / GF * ct + (h + 1 + GF - 1) / GF;
    k_grads<<<(unsigned)(tiles * CL), GTH, 0, s>>>(P, G, M, V, h, x, a1, a2, dout, d2, d1, n, A);
    return cudaGetLastError();
}

}  // namespace tpxt
