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
#include <cstddef>
#include <cstdint>

#include "tdb_internal.h"
#include "tdb_learn.h"

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

// One parameter's Adam step with the bias corrections c1, c2 (k_adam and k_net_epoch; the
// roundings are written out, so that both are the same).
__device__ __forceinline__ void adam(float& p, float& m, float& v, float g, float lr, float b1, float b2,
                                     float c1, float c2, float eps) {
    m = fmaf(b1, m, __fmul_rn(1.f - b1, g));
    v = fmaf(b2, v, __fmul_rn(__fmul_rn(1.f - b2, g), g));
    p -= lr * (m / c1) / (sqrtf(v / c2) + eps);
}

// Mini-batches of Adam in one thread-block cluster: every CTA keeps the whole network in shared
// memory (weights rounded to bfloat16).  The CTAs work in groups of four; a group takes a block
// of 128 samples of the mini-batch, each of its CTAs (members) the activations of 32 of them.
// They hand those on through distributed shared memory, all first-layer activations to every
// member and the rest to the member whose 16 columns they belong to, and after a cluster barrier
// each member forms its columns' gradient sums over the block's 128 samples.  After another
// barrier each owner adds the groups' sums of its parameters in group order, updates them (FP32
// masters and moments in registers) and stores the new values into every network.
//
// The sums round as those of k_net_grad do: a chain over the 128 samples of a block for each
// parameter, blocks added one after another, and per sample the same chains.  Where a mini-batch has
// one block or two (a sum of two does not depend on its order) the results are bit for bit those
// of k_net_grad and k_adam; with more, k_net_grad's atomic order varies from run to run and this
// is one of its orders up to one block a group.  (Sums in other chains are as accurate, but a master
// near a tie of the bfloat16 rounding then rounds the other way now and then, and an epoch's
// parameters moved by up to 2e-5 against 1e-5 between two runs of k_net_grad.)
//
// A mini-batch is a few MFLOP, so what bounds it is latency: two launches, an atomic sum and
// layers with one output per thread cost 121 us a batch of 512 at 16 x 64 (4 blocks of 128
// samples), this 14.2; with sums over 32 samples in every CTA and block barriers between the layers it was
// 17.9.  A thread takes 2 samples x 4 hidden units; a warp's four samples need no other
// warp, so the layers follow one another without a block barrier.  Hidden units are padded to
// 64 with zero weights and zero activations.  Bias corrections 1 - beta^t come from the host.
constexpr int kES = 32, kEMembers = 4, kEH = 64, kEF = 32, kEC = kEH / kEMembers, kEStride = kEH + 4,
              kEThreads = 256;
constexpr int kESlice = (kEF + kEH + 3) * kEC + 1;   // gradient sums of a member: W1, W2, b1, b2, w3, b3
static_assert(kES * kEMembers == kBlockSamples, "sizes");
struct EpochSmem {
    float W1[kEF][kEH], W2[kEH][kEH], W2T[kEH][kEH];
    float b1[kEH], b2[kEH], w3[kEH], b3;
    alignas(16) float h2[kES][kEStride], d2[kES][kEStride];   // own samples
    // the block's samples: inputs (of this batch and the next), activations, columns of this member
    alignas(16) float x[2][kBlockSamples][kEF + 4], h1[kBlockSamples][kEStride];
    float h2c[kBlockSamples][kEC + 4], d1c[kBlockSamples][kEC + 4], d2c[kBlockSamples][kEC + 4];
    float dy[kBlockSamples], r2[kBlockSamples];
    float g[kESlice];
};

// Entry e of member's gradient slice: its packed parameter (-1: none).
__device__ __forceinline__ int slice_param(const Layout& L, int member, int e) {
    if (e == (L.F + L.H + 3) * kEC) return member == 0 ? L.ob3 : -1;
    const int row = e / kEC, col = kEC * member + e % kEC;
    if (col >= L.H) return -1;
    if (row < L.F) return L.oW1 + row * L.H + col;
    if (row < L.F + L.H) return L.oW2 + (row - L.F) * L.H + col;
    return (row == L.F + L.H ? L.ob1 : row == L.F + L.H + 1 ? L.ob2 : L.ow3) + col;
}
// Where packed parameter i lies in a network, in floats from its start: `at` (and `at2`, W2
// transposed, or -1); true for a weight, which is kept rounded to bfloat16.
__device__ __forceinline__ bool param_place(const Layout& L, int i, int& at, int& at2) {
    auto f = [](size_t bytes) { return static_cast<int>(bytes / sizeof(float)); };
    at2 = -1;
    if (i < L.ob1) {
        at = f(offsetof(EpochSmem, W1)) + i / L.H * kEH + i % L.H;
    } else if (i < L.oW2) {
        at = f(offsetof(EpochSmem, b1)) + i - L.ob1;
        return false;
    } else if (i < L.ob2) {
        const int r = (i - L.oW2) / L.H, c = (i - L.oW2) % L.H;
        at = f(offsetof(EpochSmem, W2)) + r * kEH + c;
        at2 = f(offsetof(EpochSmem, W2T)) + c * kEH + r;
    } else if (i < L.ow3) {
        at = f(offsetof(EpochSmem, b2)) + i - L.ob2;
        return false;
    } else if (i < L.ob3) {
        at = f(offsetof(EpochSmem, w3)) + i - L.ow3;
    } else {
        at = f(offsetof(EpochSmem, b3));
        return false;
    }
    return true;
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
__device__ __forceinline__ void put4(float* o, const float (&v)[4]) {
    *reinterpret_cast<float4*>(o) = make_float4(v[0], v[1], v[2], v[3]);
}
// Column sums over the block of a tile of 2 rows x 4 columns: g[r][j] = sum_q A[q][r] D[q][j], q in order
__device__ __forceinline__ void column_sums(const float* A, int lda, const float* D, float (&g)[2][4]) {
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) g[r][j] = 0.f;
#pragma unroll 8
    for (int q = 0; q < kBlockSamples; ++q) {
        const float2 a = *reinterpret_cast<const float2*>(A + q * lda);
        const float4 d = *reinterpret_cast<const float4*>(D + q * (kEC + 4));
        const float ar[2] = {a.x, a.y}, dj[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int j = 0; j < 4; ++j) g[r][j] = fmaf(ar[r], dj[j], g[r][j]);
    }
}

// NG: groups of the cluster
template <int NG>
__global__ void __launch_bounds__(kEThreads)
    k_net_epoch(int F, int H, float* __restrict__ params, float* __restrict__ am,
                float* __restrict__ av, const float* __restrict__ X, const float* __restrict__ Y,
                long n, long batch, float lr, float beta1, float beta2, float eps,
                const __grid_constant__ Corrections corr, double* __restrict__ sse) {
    extern __shared__ __align__(16) uint8_t epoch_raw[];
    EpochSmem& s = *reinterpret_cast<EpochSmem*>(epoch_raw);
    float* const net = reinterpret_cast<float*>(epoch_raw);
    cg::cluster_group cluster = cg::this_cluster();
    constexpr int NC = NG * kEMembers, kOwn = (kESlice + NG * kEThreads - 1) / (NG * kEThreads);
    const int rank = static_cast<int>(cluster.block_rank());
    const int group = rank / kEMembers, member = rank % kEMembers;
    const Layout L = layout(F, H);
    const int t = threadIdx.x, lane = t % 32, warp = t / 32, tx = t % 16, ty = t / 16;
    // everything starts at zero (padded rows and columns stay there)
    for (int i = t; i < static_cast<int>(sizeof(EpochSmem) / 4); i += kEThreads)
        reinterpret_cast<uint32_t*>(epoch_raw)[i] = 0;
    __syncthreads();
    for (int i = t; i < L.n; i += kEThreads) {
        int at, at2;
        const float v = params[i], w = param_place(L, i, at, at2) ? bf(v) : v;
        net[at] = w;
        if (at2 >= 0) net[at2] = w;
    }
    // this CTA's parameters: its share of the member's slice
    const int slice = (F + H + 3) * kEC + 1, own = (slice + NG - 1) / NG;
    float pp[kOwn], pm[kOwn], pv[kOwn];
    int pe[kOwn], pi[kOwn], at[kOwn], at2[kOwn];
    bool weight[kOwn];
#pragma unroll
    for (int u = 0; u < kOwn; ++u) {
        const int k = t + u * kEThreads;
        pe[u] = group * own + k;
        pi[u] = k < own && pe[u] < slice ? slice_param(L, member, pe[u]) : -1;
        pp[u] = pm[u] = pv[u] = 0.f;
        at[u] = at2[u] = -1;
        weight[u] = false;
        if (pi[u] >= 0) {
            pp[u] = params[pi[u]];
            pm[u] = am[pi[u]];
            pv[u] = av[pi[u]];
            weight[u] = param_place(L, pi[u], at[u], at2[u]);
        }
    }
    // block `round NG + group` of the mini-batch at b0: its inputs into x[buf] (rows past the batch:
    // zero), asynchronously, and this lane's target
    const bool vec = F % 4 == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    const int row = kES * member + 4 * warp + (lane & 3);   // of the block: this lane's sample
    float yn = 0.f;
    auto fetch = [&](long b0, long round, int buf) {
        const long nb = batch < n - b0 ? batch : n - b0, r0 = (round * NG + group) * kBlockSamples;
        const int q = t >> 1;
        const bool in = r0 + q < nb;
        const float* src = X + (in ? b0 + r0 + q : b0) * F;
        float* dst = s.x[buf][q];
        if (vec)
            for (int c = 4 * (t & 1); c < F; c += 8)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                                 static_cast<uint32_t>(__cvta_generic_to_shared(dst + c))),
                             "l"(src + c), "r"(in ? 16 : 0) : "memory");
        else
            for (int c = t & 1; c < F; c += 2)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                                 static_cast<uint32_t>(__cvta_generic_to_shared(dst + c))),
                             "l"(src + c), "r"(in ? 4 : 0) : "memory");
        yn = r0 + row < nb ? __ldg(Y + b0 + r0 + row) : 0.f;
    };
    double sq = 0.0;
    int buf = 0;
    fetch(0, 0, 0);
    cluster.sync();   // no CTA writes into another one's memory before that is cleared
    for (long b0 = 0, step = 0; b0 < n; b0 += batch, ++step) {
        const long nb = batch < n - b0 ? batch : n - b0;
        const long blocks = (nb + kBlockSamples - 1) / kBlockSamples, rounds = (blocks + NG - 1) / NG;
        const float scale = 1.0f / static_cast<float>(nb);
        for (long round = 0; round < rounds; ++round, buf ^= 1) {
            const bool real = (round * NG + group) * kBlockSamples + row < nb;   // this lane's sample
            const float y_ref = yn;
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
            if (round + 1 < rounds)
                fetch(b0, round + 1, buf ^ 1);
            else if (b0 + batch < n)
                fetch(b0 + batch, 0, buf ^ 1);
            const int r = kES * member + 2 * ty;   // of the block: this thread's first sample
            float v[2][4], h1[2][4], h2[2][4];
            auto bias = [&](const float* b) {
#pragma unroll
                for (int q = 0; q < 2; ++q)
#pragma unroll
                    for (int j = 0; j < 4; ++j) v[q][j] = b[4 * tx + j];
            };
            // h1 = tanh(x W1 + b1) to every member; rows of W1 past F are zero.  (Padded units are
            // set to zero: an infinite input times their zero weights is not.)
            bias(s.b1);
            layer(s.x[buf][kES * member], kEF + 4, &s.W1[0][0], (F + 3) & ~3, tx, ty, v);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
#pragma unroll
                for (int j = 0; j < 4; ++j) h1[q][j] = 4 * tx + j < H ? tanhf(v[q][j]) : 0.f;
#pragma unroll
                for (int m = 0; m < kEMembers; ++m) {
                    float* o = &s.h1[r + q][4 * tx];   // (this CTA reads its own rows in a moment)
                    put4(m == member ? o : cluster.map_shared_rank(o, group * kEMembers + m), h1[q]);
                }
            }
            __syncwarp();
            // h2 = tanh(h1 W2 + b2)
            bias(s.b2);
            layer(s.h1[kES * member], kEStride, &s.W2[0][0], kEH, tx, ty, v);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
#pragma unroll
                for (int j = 0; j < 4; ++j) h2[q][j] = tanhf(v[q][j]);
                put4(&s.h2[2 * ty + q][4 * tx], h2[q]);
            }
            __syncwarp();
            // y = h2 w3 + b3, dy = 2 (y - Y) / nb, every lane for one of the warp's four samples
            float y = s.b3;
#pragma unroll 4
            for (int j = 0; j < kEH; j += 4) {
                const float4 h = *reinterpret_cast<const float4*>(&s.h2[4 * warp + (lane & 3)][j]);
                const float4 w = *reinterpret_cast<const float4*>(&s.w3[j]);
                y = fmaf(h.x, w.x, y);
                y = fmaf(h.y, w.y, y);
                y = fmaf(h.z, w.z, y);
                y = fmaf(h.w, w.w, y);
            }
            const float res = real ? y - y_ref : 0.f;
            const float dy = 2.f * res * scale;
            // lane l stores the sample l & 3 to member l >> 2
            if (lane < 4 * kEMembers) {
                EpochSmem* to = cluster.map_shared_rank(&s, group * kEMembers + (lane >> 2));
                to->dy[row] = dy;
                to->r2[row] = res * res;
            }
            // dz2 = dy w3 (1 - h2^2); this thread's four columns belong to member tx / 4
            EpochSmem* to = cluster.map_shared_rank(&s, group * kEMembers + tx / 4);
            const int col = 4 * (tx % 4);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float z = __shfl_sync(0xffffffffu, dy, 2 * (ty & 1) + q);
#pragma unroll
                for (int j = 0; j < 4; ++j) v[q][j] = z * s.w3[4 * tx + j] * (1.f - h2[q][j] * h2[q][j]);
                put4(&s.d2[2 * ty + q][4 * tx], v[q]);
                put4(&to->d2c[r + q][col], v[q]);
                put4(&to->h2c[r + q][col], h2[q]);
            }
            __syncwarp();
            // dz1 = (dz2 W2^T) (1 - h1^2)
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int j = 0; j < 4; ++j) v[q][j] = 0.f;
            layer(&s.d2[0][0], kEStride, &s.W2T[0][0], kEH, tx, ty, v);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
#pragma unroll
                for (int j = 0; j < 4; ++j) v[q][j] *= 1.f - h1[q][j] * h1[q][j];
                put4(&to->d1c[r + q][col], v[q]);
            }
            cluster.sync();
            // gradient sums of the block: W2 by warps 0 - 3, W1 by 4 and 5, the rest by 6 and 7
            auto add = [&](int e, float g) { s.g[e] = round ? s.g[e] + g : g; };
            if (warp < 6) {
                const bool first = warp >= 4;
                const int k = first ? t - 128 : t, i = 2 * (k / 4), c = 4 * (k % 4);
                if (i < (first ? F : H)) {
                    float g[2][4];
                    if (first)
                        column_sums(&s.x[buf][0][i], kEF + 4, &s.d1c[0][c], g);
                    else
                        column_sums(&s.h1[0][i], kEStride, &s.d2c[0][c], g);
#pragma unroll
                    for (int q = 0; q < 2; ++q)
                        if (i + q < (first ? F : H))
#pragma unroll
                            for (int j = 0; j < 4; ++j) add(((first ? 0 : F) + i + q) * kEC + c + j, g[q][j]);
                }
            } else {
                const int k = t - 192, kind = k / kEC, c = k % kEC;
                float g = 0.f;
                if (kind == 0)
#pragma unroll 8
                    for (int q = 0; q < kBlockSamples; ++q) g += s.d1c[q][c];
                else if (kind == 1)
#pragma unroll 8
                    for (int q = 0; q < kBlockSamples; ++q) g += s.d2c[q][c];
                else if (kind == 2)
#pragma unroll 8
                    for (int q = 0; q < kBlockSamples; ++q) g = fmaf(s.h2c[q][c], s.dy[q], g);
                else if (c == 0)
#pragma unroll 8
                    for (int q = 0; q < kBlockSamples; ++q) g += s.dy[q];
                if (kind < 3 || c == 0) add((F + H + kind) * kEC + c, g);
                if (warp == 6 && member == 0) {
                    float r2 = 0.f;
#pragma unroll
                    for (int q = 0; q < kBlockSamples; q += 32) r2 += s.r2[q + lane];
                    for (int o = 16; o > 0; o >>= 1) r2 += __shfl_xor_sync(0xffffffffu, r2, o);
                    sq += static_cast<double>(r2);
                }
            }
            cluster.sync();   // the block's sums are complete, and its activations read
        }
        // owners: sum over the groups in order, Adam, new values into every network
        const float2 c = corr.c[step];
#pragma unroll
        for (int u = 0; u < kOwn; ++u)
            if (pi[u] >= 0) {
                float g = 0.f;
#pragma unroll
                for (int k = 0; k < NG; ++k)
                    g += *cluster.map_shared_rank(&s.g[pe[u]], k * kEMembers + member);
                adam(pp[u], pm[u], pv[u], g, lr, beta1, beta2, c.x, c.y, eps);
                const float w = weight[u] ? bf(pp[u]) : pp[u];
#pragma unroll 4
                for (int k = 0; k < NC; ++k) {
                    float* o = cluster.map_shared_rank(net, k);
                    o[at[u]] = w;
                    if (at2[u] >= 0) o[at2[u]] = w;
                }
            }
        cluster.sync();
    }
#pragma unroll
    for (int u = 0; u < kOwn; ++u)
        if (pi[u] >= 0) {
            params[pi[u]] = pp[u];
            am[pi[u]] = pm[u];
            av[pi[u]] = pv[u];
        }
    if (warp == 6 && member == 0 && lane == 0) atomicAdd(sse, sq);
}

__global__ void k_adam(int n, float* __restrict__ p, const float* __restrict__ g,
                       float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2,
                       float c1, float c2, float eps) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    adam(p[i], m[i], v[i], g[i], lr, b1, b2, c1, c2, eps);
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
        e = cudaFuncSetAttribute(k_net_epoch<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(sizeof(EpochSmem)));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_net_epoch<4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(sizeof(EpochSmem)));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_net_epoch<4>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
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
    if (cudaOccupancyMaxActiveClusters(&fits, k_net_epoch<4>, &l.cfg) != cudaSuccess) cudaGetLastError();
    return fits > 0 ? 16 : 8;
}

cudaError_t launch_epoch(int nc, int F, int H, float* params, float* m, float* v, const float* X,
                         const float* Y, long n, long batch, float lr, float b1, float b2, float eps,
                         const Corrections& corr, double* sse, cudaStream_t st) {
    EpochLaunch l(nc, st);
    auto kernel = nc == 16 ? k_net_epoch<4> : k_net_epoch<2>;
    return cudaLaunchKernelEx(&l.cfg, kernel, F, H, params, m, v, X, Y, n, batch, lr, b1, b2, eps, corr,
                              sse);
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
