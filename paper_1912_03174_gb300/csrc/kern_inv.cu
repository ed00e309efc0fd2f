// S^-1 of a small overlap matrix (moving nuclei: every step, Sec. 2.3) without a library call or
// a host synchronisation: Gauss-Jordan in FP32 by one block with the matrix in registers, then
// two Newton-Schulz steps X <- X + X E, E = 1 - S X, which square the FP32 inverse's residual
// (1e-6 of the synthetic overlaps) twice; E needs an FP64 product, X E only corrects and is an
// FP32 one.  A result whose residual before the last step was still large (an ill-conditioned S)
// is replaced by an FP64 Gauss-Jordan in the same launch sequence.  The result depends on S
// alone, so a state loaded from a checkpoint continues bit for bit.
//
// Bound by latency: N / 4 dependent blocks of pivots of one shared-memory round trip each (no
// pivoting: S is positive definite), then four products of a few microseconds.  cuSOLVER's potrf
// + potri took 912 us at N = 132.
#include <cmath>

#include "pdl.cuh"
#include "tdb_internal.h"

namespace tdb {

namespace {

// Inverse of a 4 x 4 symmetric positive definite block in place; false if a pivot is not positive.
__device__ __forceinline__ bool invert4(float (&p)[4][4]) {
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        ok &= p[k][k] > 0.f;
        const float inv = __fdividef(1.f, p[k][k]);   // refined in FP64 afterwards
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (j != k) p[k][j] *= inv;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i != k) {
                const float f = p[i][k];
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (j != k) p[i][j] = fmaf(-f, p[k][j], p[i][j]);
                p[i][k] = -f * inv;
            }
        p[k][k] = inv;
    }
    return ok;
}

// In-place Gauss-Jordan inversion by blocks of four pivots, thread (tx, ty) of 16 x 16 holding
// the elements (ty + 16 a, tx + 16 b), a, b < T (rows and columns past N: identity).  A pivot that
// is not positive makes the result NaN.  One barrier a block: the four pivot rows and columns go
// through double-buffered shared memory, and every thread inverts the pivot block for itself.  Bound
// by the issue of the 4 T^2 updates plus that round trip and the block's inversion.  At N = 132 the
// inverse by single pivots took 70 us, by blocks of four 58 (the whole S^-1: 95).
template <int T>
__global__ void __launch_bounds__(256)
    k_inv_f32(int N, const double* S, double* X, float* Xf,
              unsigned* norm) {
    __shared__ __align__(16) float row_s[2][16 * T][4], col_s[2][16 * T][4];   // [index][pivot]
    const int tx = threadIdx.x, ty = threadIdx.y;
    float r[T][T];
    pdl_launch_dependents();
    pdl_wait();
    if (tx == 0 && ty == 0) *norm = 0u;
#pragma unroll
    for (int a = 0; a < T; ++a)
#pragma unroll
        for (int b = 0; b < T; ++b) {
            const int i = ty + 16 * a, j = tx + 16 * b;
            r[a][b] = i < N && j < N ? static_cast<float>(S[(size_t)i * N + j]) : (i == j ? 1.f : 0.f);
        }
    bool good = true;
    int s = 0;
#pragma unroll
    for (int kb = 0; kb < T; ++kb)
#pragma unroll 1   // the body stays in the instruction cache
        for (int kq = 0; kq < 4 && kb * 16 + 4 * kq < N; ++kq, s ^= 1) {
            const bool my_row = ty / 4 == kq, my_col = tx / 4 == kq;   // this block's pivots
            if (my_row)
#pragma unroll
                for (int b = 0; b < T; ++b) row_s[s][tx + 16 * b][ty & 3] = r[kb][b];
            if (my_col)
#pragma unroll
                for (int a = 0; a < T; ++a) col_s[s][ty + 16 * a][tx & 3] = r[a][kb];
            __syncthreads();
            float p[4][4];   // the pivot block: p[i][j] = element (pivot i, pivot j)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 c = *reinterpret_cast<const float4*>(row_s[s][kb * 16 + 4 * kq + j]);
                p[0][j] = c.x, p[1][j] = c.y, p[2][j] = c.z, p[3][j] = c.w;
            }
            good &= invert4(p);
            // V = P^-1 (pivot rows); the pivot columns themselves become P^-1
            float v[T][4];
#pragma unroll
            for (int b = 0; b < T; ++b) {
                const float4 c = *reinterpret_cast<const float4*>(row_s[s][tx + 16 * b]);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    v[b][q] = fmaf(p[q][0], c.x, fmaf(p[q][1], c.y, fmaf(p[q][2], c.z, p[q][3] * c.w)));
            }
            float pc[4];   // column tx & 3 of P^-1
#pragma unroll
            for (int q = 0; q < 4; ++q)
                pc[q] = (tx & 3) == 0 ? p[q][0] : (tx & 3) == 1 ? p[q][1] : (tx & 3) == 2 ? p[q][2] : p[q][3];
            if (my_col)
#pragma unroll
                for (int q = 0; q < 4; ++q) v[kb][q] = pc[q];
#pragma unroll
            for (int a = 0; a < T; ++a) {
                const float4 c = *reinterpret_cast<const float4*>(col_s[s][ty + 16 * a]);
                if (my_col) r[a][kb] = 0.f;   // rows below: -(column) P^-1
#pragma unroll
                for (int b = 0; b < T; ++b)
                    r[a][b] = fmaf(-c.x, v[b][0], fmaf(-c.y, v[b][1], fmaf(-c.z, v[b][2], fmaf(-c.w, v[b][3], r[a][b]))));
            }
            // the pivot rows: P^-1 (row), and P^-1 in the pivot block
            if (my_row)
#pragma unroll
                for (int b = 0; b < T; ++b)
                    r[kb][b] = (ty & 3) == 0 ? v[b][0] : (ty & 3) == 1 ? v[b][1] : (ty & 3) == 2 ? v[b][2] : v[b][3];
        }
#pragma unroll
    for (int a = 0; a < T; ++a)
#pragma unroll
        for (int b = 0; b < T; ++b) {
            const int i = ty + 16 * a, j = tx + 16 * b;
            if (i < N && j < N) {
                const float x = good ? r[a][b] : __int_as_float(0x7fffffff);
                X[(size_t)i * N + j] = static_cast<double>(x);
                Xf[(size_t)i * N + j] = x;
            }
        }
}

// The products of a Newton-Schulz step, 8 x 8 tiles of one output per thread; the next 64-deep
// block is loaded while this one is multiplied.
constexpr int kT = 8, kKB = 64;

template <typename T>
struct TileProduct {
    T As[kT][kKB + 2], Bs[kKB][kT + 1];
    // sum over K of A (row m0 + ty) B (column n0 + tx), K in order
    __device__ __forceinline__ T run(int N, int m0, int n0, const T* A, const T* B) {
        const int tid = threadIdx.x, tx = tid % kT, ty = tid / kT;
        T ra[kT], rb[kT], acc = 0;
        auto load = [&](int k0) {
#pragma unroll
            for (int i = 0; i < kT; ++i) {
                const int k = k0 + ty + kT * i;
                ra[i] = m0 + i < N && k0 + tid < N ? A[(size_t)(m0 + i) * N + k0 + tid] : T(0);
                rb[i] = k < N && n0 + tx < N ? B[(size_t)k * N + n0 + tx] : T(0);
            }
        };
        load(0);
        for (int k0 = 0; k0 < N; k0 += kKB) {
            if (k0) __syncthreads();
#pragma unroll
            for (int i = 0; i < kT; ++i) {
                As[i][tid] = ra[i];
                Bs[ty + kT * i][tx] = rb[i];
            }
            __syncthreads();
            if (k0 + kKB < N) load(k0 + kKB);
            const int len = N - k0 < kKB ? N - k0 : kKB;
#pragma unroll 8
            for (int k = 0; k < len; ++k) acc = fma(As[ty][k], Bs[k][tx], acc);
        }
        return acc;
    }
};

// E = 1 - S X (FP64 product, FP32 result); the largest |E| into *norm (float bits; NaN as
// infinity) where set
__global__ void __launch_bounds__(kT* kT)
    k_ns_resid(int N, const double* S, const double* X, float* E,
               unsigned* norm) {
    __shared__ TileProduct<double> tile;
    const int m0 = blockIdx.y * kT, n0 = blockIdx.x * kT;
    const int i = m0 + threadIdx.x / kT, j = n0 + threadIdx.x % kT;
    pdl_wait();
    const float e = static_cast<float>((i == j ? 1.0 : 0.0) - tile.run(N, m0, n0, S, X));
    pdl_launch_dependents();
    const bool in = i < N && j < N;
    if (in) E[(size_t)i * N + j] = e;
    if (norm) {
        const float f = in ? fabsf(e) : 0.f;
        const unsigned m = __reduce_max_sync(0xffffffffu, f >= 0.f ? __float_as_uint(f) : 0x7f800000u);
        if ((threadIdx.x & 31) == 0) atomicMax(norm, m);
    }
}

// X' = X + Xf E (FP32 product) with its FP32 copy; with `last` only tiles on and above the
// diagonal, mirrored: X' exactly symmetric, no copy
__global__ void __launch_bounds__(kT* kT)
    k_ns_step(int N, const double* X, const float* Xf, const float* E,
              int last, double* Xn, float* Xnf) {
    __shared__ TileProduct<float> tile;
    const int m0 = blockIdx.y * kT, n0 = blockIdx.x * kT;
    const int i = m0 + threadIdx.x / kT, j = n0 + threadIdx.x % kT;
    pdl_wait();
    if (last && m0 > n0) return;
    const float acc = tile.run(N, m0, n0, Xf, E);
    pdl_launch_dependents();
    if (i >= N || j >= N || (last && i > j)) return;
    const double x = X[(size_t)i * N + j] + static_cast<double>(acc);
    Xn[(size_t)i * N + j] = x;
    if (last)
        Xn[(size_t)j * N + i] = x;
    else
        Xnf[(size_t)i * N + j] = static_cast<float>(x);
}

// X = S^-1 by Gauss-Jordan in FP64, one block, if N *norm exceeds 1e-7 (the residual after the
// last Newton-Schulz step is its square); otherwise nothing.  NaN where S is not positive
// definite.
__global__ void __launch_bounds__(1024)
    k_inv_repair(int N, const double* S, double* X,
                 const unsigned* norm) {
    extern __shared__ double rc[];   // pivot row and column
    pdl_launch_dependents();
    pdl_wait();
    if (static_cast<float>(N) * __uint_as_float(__ldcg(norm)) <= 1e-7f) return;
    double *row = rc, *col = rc + N;
    const int t = threadIdx.x, NN = N * N;
    for (int e = t; e < NN; e += 1024) X[e] = S[e];
    bool bad = false;
    for (int k = 0; k < N; ++k) {
        __syncthreads();
        const double piv = X[(size_t)k * N + k];
        bad |= !(piv > 0.0);
        for (int j = t; j < N; j += 1024) {
            row[j] = X[(size_t)k * N + j] / piv;
            col[j] = X[(size_t)j * N + k];
        }
        __syncthreads();
        for (int e = t; e < NN; e += 1024) {
            const int i = e / N, j = e - i * N;
            double v;
            if (i == k)
                v = j == k ? 1.0 / piv : row[j];
            else
                v = j == k ? -col[i] / piv : fma(-col[i], row[j], X[e]);
            X[e] = v;
        }
    }
    __syncthreads();
    // exactly symmetric, from the upper triangle
    for (int e = t; e < NN; e += 1024) {
        const int i = e / N, j = e - i * N;
        if (bad)
            X[e] = __longlong_as_double(0x7ff8000000000000ll);
        else if (i > j)
            X[e] = X[(size_t)j * N + i];
    }
}

}  // namespace

void launch_small_inverse(int N, const double* S, double* Sinv, double* t0, double* t1, double* t2,
                          unsigned* norm, cudaStream_t st) {
    // t0: X0, X1 (FP64); t1: E; t2: X0, X1 (FP32)
    const size_t NN = (size_t)N * N;
    double *x0 = t0, *x1 = Sinv;
    float *x0f = reinterpret_cast<float*>(t2), *x1f = x0f + NN, *e = reinterpret_cast<float*>(t1);
    const dim3 b(16, 16);
    switch ((N + 15) / 16) {
        case 1: launch_pdl(k_inv_f32<1>, dim3(1), b, 0, st, N, S, x0, x0f, norm); break;
        case 2: launch_pdl(k_inv_f32<2>, dim3(1), b, 0, st, N, S, x0, x0f, norm); break;
        case 3: launch_pdl(k_inv_f32<3>, dim3(1), b, 0, st, N, S, x0, x0f, norm); break;
        case 4: launch_pdl(k_inv_f32<4>, dim3(1), b, 0, st, N, S, x0, x0f, norm); break;
        case 5: launch_pdl(k_inv_f32<5>, dim3(1), b, 0, st, N, S, x0, x0f, norm); break;
        case 6: launch_pdl(k_inv_f32<6>, dim3(1), b, 0, st, N, S, x0, x0f, norm); break;
        case 7: launch_pdl(k_inv_f32<7>, dim3(1), b, 0, st, N, S, x0, x0f, norm); break;
        case 8: launch_pdl(k_inv_f32<8>, dim3(1), b, 0, st, N, S, x0, x0f, norm); break;
        case 9: launch_pdl(k_inv_f32<9>, dim3(1), b, 0, st, N, S, x0, x0f, norm); break;
        case 10: launch_pdl(k_inv_f32<10>, dim3(1), b, 0, st, N, S, x0, x0f, norm); break;
        case 11: launch_pdl(k_inv_f32<11>, dim3(1), b, 0, st, N, S, x0, x0f, norm); break;
        default: launch_pdl(k_inv_f32<12>, dim3(1), b, 0, st, N, S, x0, x0f, norm); break;
    }
    const dim3 g((N + kT - 1) / kT, (N + kT - 1) / kT), tb(kT * kT);
    launch_pdl(k_ns_resid, g, tb, 0, st, N, S, (const double*)x0, e, (unsigned*)nullptr);
    launch_pdl(k_ns_step, g, tb, 0, st, N, (const double*)x0, (const float*)x0f, (const float*)e, 0, x1, x1f);
    launch_pdl(k_ns_resid, g, tb, 0, st, N, S, (const double*)x1, e, norm);
    // in place: a thread reads X at (i, j), i <= j, and writes (i, j) and its mirror
    launch_pdl(k_ns_step, g, tb, 0, st, N, (const double*)x1, (const float*)x1f, (const float*)e, 1, Sinv,
               (float*)nullptr);
    launch_pdl(k_inv_repair, dim3(1), dim3(1024), 2 * sizeof(double) * N, st, N, S, Sinv,
               (const unsigned*)norm);
}

}  // namespace tdb
