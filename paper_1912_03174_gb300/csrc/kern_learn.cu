// The learned form: the per-atom shift network (forward, backward, Adam) and the
// closed-form leapfrog window with a frozen Hamiltonian.
//
// Network: y = w3 . tanh(W2^T tanh(W1^T x + b1) + b2) + b3 per sample, weights used in
// bfloat16 (rounded from FP32 masters when staged into shared memory), FP32
// accumulation.  Training minimises the mean squared error with Adam; the backward pass
// keeps a block of 128 samples' activations in shared memory and forms the weight
// gradients as block-level sums (X^T dz1, h1^T dz2) added to the global gradient.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <cmath>
#include <cstdint>

#include "tdb_internal.h"

namespace tdb {
namespace learn {
namespace {
namespace cg = cooperative_groups;

constexpr int kBlockSamples = 128;

__device__ __forceinline__ float bf(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// Packed parameter offsets (W1 F x H, b1 H, W2 H x H, b2 H, w3 H, b3).
struct Layout {
    int F, H, oW1, ob1, oW2, ob2, ow3, ob3, n;
};
__host__ __device__ inline Layout layout(int F, int H) {
    Layout L;
    L.F = F;
    L.H = H;
    L.oW1 = 0;
    L.ob1 = F * H;
    L.oW2 = L.ob1 + H;
    L.ob2 = L.oW2 + H * H;
    L.ow3 = L.ob2 + H;
    L.ob3 = L.ow3 + H;
    L.n = L.ob3 + 1;
    return L;
}

// Stage the parameters into shared memory, weight matrices rounded to bfloat16.
__device__ void stage(const Layout& L, const float* __restrict__ p, float* s) {
    for (int i = threadIdx.x; i < L.n; i += blockDim.x) {
        const bool weight = i < L.ob1 || (i >= L.oW2 && i < L.ob2) || (i >= L.ow3 && i < L.ob3);
        s[i] = weight ? bf(p[i]) : p[i];
    }
}

__global__ void k_net_forward(int F, int H, const float* __restrict__ params,
                              const float* __restrict__ X, long n, float* __restrict__ Y) {
    extern __shared__ float sp[];
    const Layout L = layout(F, H);
    stage(L, params, sp);
    __syncthreads();
    const long s = static_cast<long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (s >= n) return;
    float h1[64];
    const float* x = X + s * F;
    for (int j = 0; j < H; ++j) {
        float z = sp[L.ob1 + j];
        for (int f = 0; f < F; ++f) z = fmaf(x[f], sp[L.oW1 + f * H + j], z);
        h1[j] = tanhf(z);
    }
    float y = sp[L.ob3];
    for (int j = 0; j < H; ++j) {
        float z = sp[L.ob2 + j];
        for (int i = 0; i < H; ++i) z = fmaf(h1[i], sp[L.oW2 + i * H + j], z);
        y = fmaf(tanhf(z), sp[L.ow3 + j], y);
    }
    Y[s] = y;
}

// Gradient of the mean squared error over n samples (scale = 1 / n), added to grad;
// the sum of squared residuals is added to *sse.  One block takes 128 samples and works
// layer by layer, all threads on each layer's 128 x H outputs (one sample's row is read
// as a broadcast, the weights along consecutive columns); W2 is staged with rows padded
// to H + 1 so that its transposed use in the backward pass is conflict-free too.  The
// weight and bias gradients are the block's column sums, one global atomic per element.
// Rows past n carry x = 0 and dy = 0, so they add nothing.
__global__ void __launch_bounds__(256)
    k_net_grad(int F, int H, const float* __restrict__ params, const float* __restrict__ X,
               const float* __restrict__ Y, long n, float scale, float* __restrict__ grad,
               double* __restrict__ sse) {
    extern __shared__ float sm[];
    const Layout L = layout(F, H);
    const int FS = F + 1, HS = H + 1, t = threadIdx.x, nt = blockDim.x;
    constexpr int S = kBlockSamples;
    float* sW1 = sm;                        // F x H
    float* sb1 = sW1 + F * H;               // H
    float* sW2 = sb1 + H;                   // H x (H + 1)
    float* sb2 = sW2 + H * HS;              // H
    float* sw3 = sb2 + H;                   // H
    float* sx = sw3 + H + 1;                // [S][F + 1]   (b3 sits at sw3[H])
    float* sh1 = sx + S * FS;               // [S][H + 1]
    float* sh2 = sh1 + S * HS;              // [S][H + 1]
    float* sd1 = sh2 + S * HS;              // [S][H + 1]
    float* sd2 = sd1 + S * HS;              // [S][H + 1]
    float* sdy = sd2 + S * HS;              // [S]
    float* sr2 = sdy + S;                   // [S] squared residuals
    for (int i = t; i < F * H; i += nt) sW1[i] = bf(params[L.oW1 + i]);
    for (int i = t; i < H * H; i += nt) sW2[(i / H) * HS + i % H] = bf(params[L.oW2 + i]);
    for (int i = t; i < H; i += nt) {
        sb1[i] = params[L.ob1 + i];
        sb2[i] = params[L.ob2 + i];
        sw3[i] = bf(params[L.ow3 + i]);
    }
    if (t == 0) sw3[H] = params[L.ob3];
    const long s0 = static_cast<long>(blockIdx.x) * S;
    for (int e = t; e < S * F; e += nt) {
        const int q = e / F, f = e % F;
        sx[q * FS + f] = s0 + q < n ? X[(s0 + q) * F + f] : 0.f;
    }
    __syncthreads();
    // h1 = tanh(x W1 + b1)
    for (int e = t; e < S * H; e += nt) {
        const int q = e / H, j = e % H;
        float z = sb1[j];
        for (int f = 0; f < F; ++f) z = fmaf(sx[q * FS + f], sW1[f * H + j], z);
        sh1[q * HS + j] = tanhf(z);
    }
    __syncthreads();
    // h2 = tanh(h1 W2 + b2)
    for (int e = t; e < S * H; e += nt) {
        const int q = e / H, j = e % H;
        float z = sb2[j];
        for (int i = 0; i < H; ++i) z = fmaf(sh1[q * HS + i], sW2[i * HS + j], z);
        sh2[q * HS + j] = tanhf(z);
    }
    __syncthreads();
    // y = h2 w3 + b3, dy = 2 (y - Y) / n
    for (int q = t; q < S; q += nt) {
        float y = sw3[H];
        for (int j = 0; j < H; ++j) y = fmaf(sh2[q * HS + j], sw3[j], y);
        const bool ok = s0 + q < n;
        const float r = ok ? y - Y[s0 + q] : 0.f;
        sdy[q] = 2.f * r * scale;
        sr2[q] = r * r;
    }
    __syncthreads();
    // dz2 = dy w3 (1 - h2^2)
    for (int e = t; e < S * H; e += nt) {
        const int q = e / H, j = e % H;
        const float h2 = sh2[q * HS + j];
        sd2[q * HS + j] = sdy[q] * sw3[j] * (1.f - h2 * h2);
    }
    __syncthreads();
    // dz1 = (dz2 W2^T) (1 - h1^2)
    for (int e = t; e < S * H; e += nt) {
        const int q = e / H, i = e % H;
        float g = 0.f;
        for (int j = 0; j < H; ++j) g = fmaf(sd2[q * HS + j], sW2[i * HS + j], g);
        const float h1 = sh1[q * HS + i];
        sd1[q * HS + i] = g * (1.f - h1 * h1);
    }
    __syncthreads();
    // column sums over the block's samples
    const int nW1 = F * H, nW2 = H * H;
    for (int e = t; e < nW1 + nW2 + 3 * H + 1; e += nt) {
        float g = 0.f;
        int dst;
        if (e < nW1) {
            const int f = e / H, j = e % H;
            for (int q = 0; q < S; ++q) g = fmaf(sx[q * FS + f], sd1[q * HS + j], g);
            dst = L.oW1 + e;
        } else if (e < nW1 + nW2) {
            const int e2 = e - nW1, i = e2 / H, j = e2 % H;
            for (int q = 0; q < S; ++q) g = fmaf(sh1[q * HS + i], sd2[q * HS + j], g);
            dst = L.oW2 + e2;
        } else {
            const int e3 = e - nW1 - nW2, j = e3 % H;
            if (e3 < H) {                       // b1
                for (int q = 0; q < S; ++q) g += sd1[q * HS + j];
                dst = L.ob1 + j;
            } else if (e3 < 2 * H) {            // b2
                for (int q = 0; q < S; ++q) g += sd2[q * HS + j];
                dst = L.ob2 + j;
            } else if (e3 < 3 * H) {            // w3
                for (int q = 0; q < S; ++q) g = fmaf(sh2[q * HS + j], sdy[q], g);
                dst = L.ow3 + j;
            } else {                            // b3
                for (int q = 0; q < S; ++q) g += sdy[q];
                dst = L.ob3;
            }
        }
        atomicAdd(&grad[dst], g);
    }
    if (t < 32) {
        float r2 = 0.f;
        for (int q = t; q < S; q += 32) r2 += sr2[q];
        for (int o = 16; o > 0; o >>= 1) r2 += __shfl_xor_sync(0xffffffffu, r2, o);
        if (t == 0) atomicAdd(sse, static_cast<double>(r2));
    }
}

// One epoch of Adam in one thread-block cluster: every CTA keeps the whole network in shared
// memory (weights rounded to bfloat16) and owns 1/NC of the parameters' FP32 masters and Adam
// moments.  Per mini-batch the CTAs take equal shares of the samples (chunks of 32), write their
// gradient sums into their own shared memory, and after a cluster barrier each owner adds the NC
// sums of its parameters in rank order through distributed shared memory, updates them and
// stores the new values into all NC networks.  The arithmetic per sample is that of k_net_grad.
// A mini-batch is a few MFLOP, so what bounds it is latency: two launches, an atomic sum and
// layers with one output per thread cost 121 us a batch of 512 at 16 x 64 (4 blocks of 128
// samples), this 17.8; here a thread takes 2 samples x 4 hidden units, and nothing leaves the
// cluster between batches.  Hidden units are padded to 64 with zero weights, which add nothing.
constexpr int kES = 32, kEH = 64, kEF = 32, kEStride = kEH + 4, kEThreads = 256;
constexpr int kEMaxOwn = 4;            // parameters per thread and CTA: 6337 / 8 / 256
struct EpochSmem {
    float W1[kEF][kEH], W2[kEH][kEH], W2T[kEH][kEH];
    float b1[kEH], b2[kEH], w3[kEH], b3;
    alignas(16) float x[kES][kEF + 4], h1[kES][kEStride], h2[kES][kEStride], d1[kES][kEStride],
        d2[kES][kEStride];
    float y[kES], dy[kES];
    double sse[kEThreads / 32];
    float g[kEF * kEH + 2 * kEH + kEH * kEH + kEH + 1];
};

// network value of packed parameter i (used by the owner to fill every CTA's copy)
__device__ void put_param(const Layout& L, EpochSmem& s, int i, float v) {
    const int H = L.H;
    if (i < L.ob1) {
        s.W1[i / H][i % H] = bf(v);
    } else if (i < L.oW2) {
        s.b1[i - L.ob1] = v;
    } else if (i < L.ob2) {
        const int k = i - L.oW2;
        s.W2[k / H][k % H] = bf(v);
        s.W2T[k % H][k / H] = bf(v);
    } else if (i < L.ow3) {
        s.b2[i - L.ob2] = v;
    } else if (i < L.ob3) {
        s.w3[i - L.ow3] = bf(v);
    } else {
        s.b3 = v;
    }
}

// acc[q][j] += sum_k A[2 ty + q][k] W[k][4 tx + j], k < K (a multiple of 4)
__device__ __forceinline__ void layer(const float* A, int lda, const float* W, int K, int tx, int ty,
                                      float (&acc)[2][4]) {
#pragma unroll 4
    for (int k = 0; k < K; k += 4) {
        const float4 a0 = *reinterpret_cast<const float4*>(A + 2 * ty * lda + k);
        const float4 a1 = *reinterpret_cast<const float4*>(A + (2 * ty + 1) * lda + k);
        const float av[2][4] = {{a0.x, a0.y, a0.z, a0.w}, {a1.x, a1.y, a1.z, a1.w}};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float4 w = *reinterpret_cast<const float4*>(W + (k + u) * kEH + 4 * tx);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                acc[q][0] = fmaf(av[q][u], w.x, acc[q][0]);
                acc[q][1] = fmaf(av[q][u], w.y, acc[q][1]);
                acc[q][2] = fmaf(av[q][u], w.z, acc[q][2]);
                acc[q][3] = fmaf(av[q][u], w.w, acc[q][3]);
            }
        }
    }
}
__device__ __forceinline__ void put2(float (*o)[kEStride], int tx, int ty, const float (&v)[2][4]) {
#pragma unroll
    for (int q = 0; q < 2; ++q)
        *reinterpret_cast<float4*>(&o[2 * ty + q][4 * tx]) =
            make_float4(v[q][0], v[q][1], v[q][2], v[q][3]);
}

__global__ void __launch_bounds__(kEThreads)
    k_net_epoch(int F, int H, float* __restrict__ params, float* __restrict__ am,
                float* __restrict__ av, const float* __restrict__ X, const float* __restrict__ Y,
                long n, long batch, float lr, float beta1, float beta2, float eps, long t0,
                double* __restrict__ sse) {
    extern __shared__ __align__(16) uint8_t epoch_raw[];
    EpochSmem& s = *reinterpret_cast<EpochSmem*>(epoch_raw);
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = static_cast<int>(cluster.block_rank()), NC = static_cast<int>(cluster.num_blocks());
    const Layout L = layout(F, H);
    const int t = threadIdx.x, tx = t % 16, ty = t / 16;
    // everything starts at zero (padded rows and columns stay there)
    for (int i = t; i < static_cast<int>(sizeof(EpochSmem) / 4); i += kEThreads)
        reinterpret_cast<uint32_t*>(epoch_raw)[i] = 0;
    __syncthreads();
    for (int i = t; i < L.n; i += kEThreads) put_param(L, s, i, params[i]);
    // this CTA's parameters
    const int own = (L.n + NC - 1) / NC, o0 = rank * own;
    float pp[kEMaxOwn], pm[kEMaxOwn], pv[kEMaxOwn];
#pragma unroll
    for (int u = 0; u < kEMaxOwn; ++u) {
        const int k = t + u * kEThreads, i = o0 + k;
        const bool mine = k < own && i < L.n;
        pp[u] = mine ? params[i] : 0.f;
        pm[u] = mine ? am[i] : 0.f;
        pv[u] = mine ? av[i] : 0.f;
    }
    double sq = 0.0;
    long step = t0;
    // this thread's values of a chunk, loaded one chunk ahead (rows past the share: x = 0)
    constexpr int kPre = kES * kEF / kEThreads;
    float xn[kPre], yn = 0.f;
    auto fetch = [&](long b0, long c0) {
        const long nb = batch < n - b0 ? batch : n - b0;
        const long per = (nb + NC - 1) / NC, lo = rank * per, hi = lo + per < nb ? lo + per : nb;
#pragma unroll
        for (int u = 0; u < kPre; ++u) {
            const int e = t + u * kEThreads, q = e / F;
            const long r = lo + c0 + q;
            xn[u] = q < kES && r < hi ? __ldg(X + (b0 + r) * F + (e - q * F)) : 0.f;
        }
        yn = t < kES && lo + c0 + t < hi ? __ldg(Y + b0 + lo + c0 + t) : 0.f;
    };
    fetch(0, 0);
    for (long b0 = 0; b0 < n; b0 += batch) {
        const long nb = batch < n - b0 ? batch : n - b0;
        const long per = (nb + NC - 1) / NC, lo = rank * per, hi = lo + per < nb ? lo + per : nb;
        const float scale = 1.0f / static_cast<float>(nb);
        for (long c0 = 0; c0 < per; c0 += kES) {
            // samples lo + c0 .. of the batch (rows past the share carry x = 0 and dy = 0)
            __syncthreads();
#pragma unroll
            for (int u = 0; u < kPre; ++u) {
                const int e = t + u * kEThreads, q = e / F;
                if (q < kES) s.x[q][e - q * F] = xn[u];
            }
            if (t < kES) s.y[t] = yn;
            __syncthreads();
            if (c0 + kES < per)
                fetch(b0, c0 + kES);
            else if (b0 + batch < n)
                fetch(b0 + batch, 0);
            float v[2][4], dv[2][4];
            auto bias = [&](const float* b) {
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int j = 0; j < 4; ++j) v[q][j] = b[4 * tx + j];
            };
            // h1 = tanh(x W1 + b1); rows of W1 past F are zero
            bias(s.b1);
            layer(&s.x[0][0], kEF + 4, &s.W1[0][0], (F + 3) & ~3, tx, ty, v);
            float h1[2][4];
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int j = 0; j < 4; ++j) h1[q][j] = tanhf(v[q][j]);
            put2(s.h1, tx, ty, h1);
            __syncthreads();
            // h2 = tanh(h1 W2 + b2)
            bias(s.b2);
            layer(&s.h1[0][0], kEStride, &s.W2[0][0], kEH, tx, ty, v);
            float h2[2][4];
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int j = 0; j < 4; ++j) h2[q][j] = tanhf(v[q][j]);
            put2(s.h2, tx, ty, h2);
            // y = h2 w3 + b3, dy = 2 (y - Y) / nb: the 16 threads of a sample pair
            float z[2] = {0.f, 0.f};
#pragma unroll
            for (int q = 0; q < 2; ++q) {
#pragma unroll
                for (int j = 0; j < 4; ++j) z[q] = fmaf(h2[q][j], s.w3[4 * tx + j], z[q]);
                for (int o = 8; o > 0; o >>= 1) z[q] += __shfl_xor_sync(0xffffffffu, z[q], o);
                const long r = lo + c0 + 2 * ty + q;
                const float res = r < hi ? z[q] + s.b3 - s.y[2 * ty + q] : 0.f;
                z[q] = 2.f * res * scale;
                if (tx == 0) {
                    s.dy[2 * ty + q] = z[q];
                    sq += static_cast<double>(res * res);
                }
            }
            // dz2 = dy w3 (1 - h2^2)
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    dv[q][j] = z[q] * s.w3[4 * tx + j] * (1.f - h2[q][j] * h2[q][j]);
            put2(s.d2, tx, ty, dv);
            __syncthreads();
            // dz1 = (dz2 W2^T) (1 - h1^2)
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int j = 0; j < 4; ++j) v[q][j] = 0.f;
            layer(&s.d2[0][0], kEStride, &s.W2T[0][0], kEH, tx, ty, v);
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int j = 0; j < 4; ++j) v[q][j] *= 1.f - h1[q][j] * h1[q][j];
            put2(s.d1, tx, ty, v);
            // gradient sums of W2 (rows 4 ty .., columns 4 tx ..): h1^T dz2
            {
                float g2[4][4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) g2[i][j] = 0.f;
#pragma unroll 4
                for (int q = 0; q < kES; ++q) {
                    const float4 a = *reinterpret_cast<const float4*>(&s.h1[q][4 * ty]);
                    const float4 d = *reinterpret_cast<const float4*>(&s.d2[q][4 * tx]);
                    const float ai[4] = {a.x, a.y, a.z, a.w}, dj[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) g2[i][j] = fmaf(ai[i], dj[j], g2[i][j]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (4 * ty + i < H && 4 * tx + j < H) {
                            float& o = s.g[L.oW2 + (4 * ty + i) * H + 4 * tx + j];
                            o = c0 ? o + g2[i][j] : g2[i][j];
                        }
            }
            __syncthreads();
            // W1: x^T dz1 (rows ty, ty + 16); then the biases, w3 and b3
#pragma unroll
            for (int r = 0; r < kEF / 16; ++r) {
                const int f = ty + 16 * r;
                if (f >= F) break;
                float g1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
                for (int q = 0; q < kES; ++q) {
                    const float4 d = *reinterpret_cast<const float4*>(&s.d1[q][4 * tx]);
                    const float xf = s.x[q][f];
                    g1[0] = fmaf(xf, d.x, g1[0]);
                    g1[1] = fmaf(xf, d.y, g1[1]);
                    g1[2] = fmaf(xf, d.z, g1[2]);
                    g1[3] = fmaf(xf, d.w, g1[3]);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (4 * tx + j < H) {
                        float& o = s.g[L.oW1 + f * H + 4 * tx + j];
                        o = c0 ? o + g1[j] : g1[j];
                    }
            }
            {
                const int kind = t / kEH, j = t % kEH;
                float g = 0.f;
                if (kind == 0)
#pragma unroll 8
                    for (int q = 0; q < kES; ++q) g += s.d1[q][j];
                else if (kind == 1)
#pragma unroll 8
                    for (int q = 0; q < kES; ++q) g += s.d2[q][j];
                else if (kind == 2)
#pragma unroll 8
                    for (int q = 0; q < kES; ++q) g = fmaf(s.h2[q][j], s.dy[q], g);
                else if (j == 0)
                    for (int q = 0; q < kES; ++q) g += s.dy[q];
                if ((kind < 3 && j < H) || (kind == 3 && j == 0)) {
                    float& o = s.g[kind == 0 ? L.ob1 + j : kind == 1 ? L.ob2 + j
                                                       : kind == 2   ? L.ow3 + j
                                                                     : L.ob3];
                    o = c0 ? o + g : g;
                }
            }
        }
        cluster.sync();
        // owners: sum over the CTAs in rank order, Adam, new values into every network
        ++step;
        const float c1 = 1.0f - powf(beta1, static_cast<float>(step));
        const float c2 = 1.0f - powf(beta2, static_cast<float>(step));
#pragma unroll
        for (int u = 0; u < kEMaxOwn; ++u) {
            const int k = t + u * kEThreads, i = o0 + k;
            if (k < own && i < L.n) {
                float g = 0.f;
#pragma unroll 8
                for (int c = 0; c < NC; ++c) g += *cluster.map_shared_rank(&s.g[i], c);
                pm[u] = beta1 * pm[u] + (1.f - beta1) * g;
                pv[u] = beta2 * pv[u] + (1.f - beta2) * g * g;
                pp[u] -= lr * (pm[u] / c1) / (sqrtf(pv[u] / c2) + eps);
                for (int c = 0; c < NC; ++c) put_param(L, *cluster.map_shared_rank(&s, c), i, pp[u]);
            }
        }
        cluster.sync();
    }
#pragma unroll
    for (int u = 0; u < kEMaxOwn; ++u) {
        const int k = t + u * kEThreads, i = o0 + k;
        if (k < own && i < L.n) {
            params[i] = pp[u];
            am[i] = pm[u];
            av[i] = pv[u];
        }
    }
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (t % 32 == 0) s.sse[t / 32] = sq;
    __syncthreads();
    if (t == 0) {
        double x = 0.0;
        for (int w = 0; w < kEThreads / 32; ++w) x += s.sse[w];
        atomicAdd(sse, x);
    }
}

__global__ void k_adam(int n, float* __restrict__ p, const float* __restrict__ g,
                       float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2,
                       float c1, float c2, float eps) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    m[i] = b1 * m[i] + (1.f - b1) * g[i];
    v[i] = b2 * v[i] + (1.f - b2) * g[i] * g[i];
    p[i] -= lr * (m[i] / c1) / (sqrtf(v[i] / c2) + eps);
}

// Closed-form leapfrog window in the eigenbasis: for element (a, b), theta = (e_a - e_b) dt,
// the leapfrog modes are l+ = exp(-i phi), l- = -exp(i phi) with phi = asin(theta);
// (x0, x1) = (x_{n-1}, x_n) -> (x_{n-1+k}, x_{n+k}).
__global__ void k_window(int N, const double* __restrict__ eps, double dt, int k,
                         double* __restrict__ x0re, double* __restrict__ x0im,
                         double* __restrict__ x1re, double* __restrict__ x1im) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    const int a = blockIdx.y * blockDim.y + threadIdx.y;
    if (a >= N || b >= N) return;
    const size_t i = static_cast<size_t>(a) * N + b;
    const double th = (eps[a] - eps[b]) * dt;
    const double c = sqrt(1.0 - th * th);
    const double phi = asin(th);
    // A = (x1 - l- x0) / (2c), l- = (-c, -th);  B = x0 - A
    const double lmr = -c, lmi = -th;
    const double ar = (x1re[i] - (lmr * x0re[i] - lmi * x0im[i])) / (2.0 * c);
    const double ai = (x1im[i] - (lmr * x0im[i] + lmi * x0re[i])) / (2.0 * c);
    const double br = x0re[i] - ar, bi = x0im[i] - ai;
    double out[2][2];
    for (int q = 0; q < 2; ++q) {
        const int m = k + q;
        double sn, cs;
        sincos(m * phi, &sn, &cs);
        const double sg = (m & 1) ? -1.0 : 1.0;
        // l+^m = (cs, -sn), l-^m = sg (cs, sn)
        out[q][0] = (ar * cs + ai * sn) + sg * (br * cs - bi * sn);
        out[q][1] = (ai * cs - ar * sn) + sg * (bi * cs + br * sn);
    }
    x0re[i] = out[0][0];
    x0im[i] = out[0][1];
    x1re[i] = out[1][0];
    x1im[i] = out[1][1];
}

__global__ void k_add_step(DevScalars* sc, int k) {
    if (threadIdx.x == 0 && blockIdx.x == 0) sc->step += k;
}

}  // namespace

int n_params(int F, int H) { return layout(F, H).n; }

size_t grad_smem(int F, int H) {
    return sizeof(float) * (F * H + H + H * (H + 1) + 3 * H + 1 + kBlockSamples * (F + 1) +
                            4 * kBlockSamples * (H + 1) + 2 * kBlockSamples);
}

// The attributes are set for the largest network (32 features, 64 hidden), so that
// networks of different sizes can live side by side.
cudaError_t prepare(int, int) {
    cudaError_t e = cudaFuncSetAttribute(k_net_grad, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(grad_smem(32, 64)));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_net_epoch, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(sizeof(EpochSmem)));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_net_epoch, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_net_forward, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(sizeof(float) * layout(32, 64).n));
    return e;
}

void launch_forward(int F, int H, const float* params, const float* X, long n, float* Y,
                    cudaStream_t st) {
    const int blocks = static_cast<int>((n + 127) / 128);
    k_net_forward<<<blocks, 128, sizeof(float) * layout(F, H).n, st>>>(F, H, params, X, n, Y);
}

void launch_grad(int F, int H, const float* params, const float* X, const float* Y, long n,
                 float scale, float* grad, double* sse, cudaStream_t st) {
    const int blocks = static_cast<int>((n + kBlockSamples - 1) / kBlockSamples);
    k_net_grad<<<blocks, 256, grad_smem(F, H), st>>>(F, H, params, X, Y, n, scale, grad, sse);
}

void launch_adam(int n, float* p, const float* g, float* m, float* v, float lr, float b1,
                 float b2, float c1, float c2, float eps, cudaStream_t st) {
    k_adam<<<(n + 255) / 256, 256, 0, st>>>(n, p, g, m, v, lr, b1, b2, c1, c2, eps);
}

namespace {
// launch of the epoch kernel as one cluster of nc CTAs
struct EpochLaunch {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    EpochLaunch(int nc, cudaStream_t st) {
        cfg.gridDim = dim3(nc);
        cfg.blockDim = dim3(kEThreads);
        cfg.dynamicSmemBytes = sizeof(EpochSmem);
        cfg.stream = st;
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = nc;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
    }
};
}  // namespace

// CTAs of the epoch kernel's cluster: 16 where the device can place such a cluster, else 8.
int epoch_cluster() {
    int fits = 0;
    EpochLaunch l(16, nullptr);
    if (cudaOccupancyMaxActiveClusters(&fits, k_net_epoch, &l.cfg) != cudaSuccess) cudaGetLastError();
    return fits > 0 ? 16 : 8;
}

cudaError_t launch_epoch(int nc, int F, int H, float* params, float* m, float* v, const float* X,
                         const float* Y, long n, long batch, float lr, float b1, float b2, float eps,
                         long t0, double* sse, cudaStream_t st) {
    EpochLaunch l(nc, st);
    return cudaLaunchKernelEx(&l.cfg, k_net_epoch, F, H, params, m, v, X, Y, n, batch, lr, b1, b2,
                              eps, t0, sse);
}

void launch_window(int N, const double* eps, double dt, int k, double* x0re, double* x0im,
                   double* x1re, double* x1im, cudaStream_t st) {
    dim3 b(32, 8);
    dim3 g((N + 31) / 32, (N + 7) / 8);
    k_window<<<g, b, 0, st>>>(N, eps, dt, k, x0re, x0im, x1re, x1im);
}

void launch_add_step(DevScalars* sc, int k, cudaStream_t st) { k_add_step<<<1, 32, 0, st>>>(sc, k); }

}  // namespace learn
}  // namespace tdb
