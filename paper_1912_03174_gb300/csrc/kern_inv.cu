// S^-1 of a small overlap matrix (moving nuclei: every step, Sec. 2.3) without a library call or
// a host synchronisation: Gauss-Jordan in FP32 by one block with the matrix in registers, then
// two Newton-Schulz steps X <- X + X (1 - S X) in FP64, which square the FP32 inverse's residual
// (1e-6 of the synthetic overlaps) twice.  A result whose residual before the last step was still
// large (an ill-conditioned S) is replaced by an FP64 Gauss-Jordan in the same launch sequence.
// The result depends on S alone, so a state loaded from a checkpoint continues bit for bit.
//
// Bound by latency: N dependent pivots of one shared-memory round trip each (no pivoting: S is
// positive definite), then four products of a few microseconds.  cuSOLVER's potrf + potri took
// 912 us at N = 132.
#include <cmath>

#include "pdl.cuh"
#include "tdb_internal.h"

namespace tdb {

namespace {

// In-place Gauss-Jordan inversion, thread (tx, ty) of 16 x 16 holding the elements
// (ty + 16 a, tx + 16 b), a, b < T (rows and columns past N: identity).  A pivot that is not
// positive makes the result NaN.  One barrier a pivot: the pivot row and column go through
// double-buffered shared memory.  Bound by the issue of the T^2 updates plus that round trip; 256
// threads with large register tiles rather than 1024 with small ones, which spent their time on
// the shared-memory reads, the fix-ups and the barrier.
template <int T>
__global__ void __launch_bounds__(256)
    k_inv_f32(int N, const double* __restrict__ S, double* __restrict__ X, unsigned* __restrict__ norm) {
    __shared__ float row_s[2][16 * T], col_s[2][16 * T];
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
    bool bad = false;
    int s = 0;
#pragma unroll
    for (int kb = 0; kb < T; ++kb)
#pragma unroll 1   // the body stays in the instruction cache
        for (int kk = 0; kk < 16 && kb * 16 + kk < N; ++kk, s ^= 1) {
            if (ty == kk)
#pragma unroll
                for (int b = 0; b < T; ++b) row_s[s][tx + 16 * b] = r[kb][b];
            if (tx == kk)
#pragma unroll
                for (int a = 0; a < T; ++a) col_s[s][ty + 16 * a] = r[a][kb];
            __syncthreads();
            const float piv = col_s[s][kb * 16 + kk];
            bad |= !(piv > 0.f);
            const float inv = __fdividef(1.f, piv);   // refined in FP64 afterwards
            float rj[T];
#pragma unroll
            for (int b = 0; b < T; ++b) rj[b] = row_s[s][tx + 16 * b] * inv;
#pragma unroll
            for (int a = 0; a < T; ++a) {
                const float ci = col_s[s][ty + 16 * a];
#pragma unroll
                for (int b = 0; b < T; ++b) r[a][b] = fmaf(-ci, rj[b], r[a][b]);
                if (tx == kk) r[a][kb] = -ci * inv;
            }
            if (ty == kk) {
#pragma unroll
                for (int b = 0; b < T; ++b) r[kb][b] = rj[b];
                if (tx == kk) r[kb][kb] = inv;
            }
        }
#pragma unroll
    for (int a = 0; a < T; ++a)
#pragma unroll
        for (int b = 0; b < T; ++b) {
            const int i = ty + 16 * a, j = tx + 16 * b;
            if (i < N && j < N)
                X[(size_t)i * N + j] = bad ? __longlong_as_double(0x7ff8000000000000ll)
                                           : static_cast<double>(r[a][b]);
        }
}

// The products of a Newton-Schulz step, 8 x 8 tiles of one output per thread (FP64, K in order):
//   kResid: C = 1 - A B, the largest |C| into *norm (float bits; NaN as infinity)
//   kStep:  C = A + A B
//   kLast:  the same for tiles on and above the diagonal, mirrored: C exactly symmetric
enum NsMode { kResid, kStep, kLast };
constexpr int kT = 8, kKB = 64;

template <int MODE>
__global__ void __launch_bounds__(kT* kT)
    k_ns_product(int N, const double* __restrict__ A, const double* __restrict__ B,
                 double* __restrict__ C, unsigned* __restrict__ norm) {
    __shared__ double As[kT][kKB + 2], Bs[kKB][kT + 1];
    const int tid = threadIdx.x, tx = tid % kT, ty = tid / kT;
    const int m0 = blockIdx.y * kT, n0 = blockIdx.x * kT;
    pdl_launch_dependents();
    pdl_wait();
    if (MODE == kLast && m0 > n0) return;
    double acc = 0.0;
    for (int k0 = 0; k0 < N; k0 += kKB) {
#pragma unroll
        for (int i = 0; i < kT; ++i)
            As[i][tid] = m0 + i < N && k0 + tid < N ? A[(size_t)(m0 + i) * N + k0 + tid] : 0.0;
#pragma unroll
        for (int i = 0; i < kKB / kT; ++i) {
            const int k = ty + kT * i;
            Bs[k][tx] = k0 + k < N && n0 + tx < N ? B[(size_t)(k0 + k) * N + n0 + tx] : 0.0;
        }
        __syncthreads();
        const int len = N - k0 < kKB ? N - k0 : kKB;
#pragma unroll 8
        for (int k = 0; k < len; ++k) acc = fma(As[ty][k], Bs[k][tx], acc);
        __syncthreads();
    }
    const int i = m0 + ty, j = n0 + tx;
    const bool in = i < N && j < N;
    if (MODE == kResid) {
        const double e = (i == j ? 1.0 : 0.0) - acc;
        if (in) C[(size_t)i * N + j] = e;
        if (norm) {
            const float f = in ? fabsf(static_cast<float>(e)) : 0.f;
            const unsigned m = __reduce_max_sync(0xffffffffu, f >= 0.f ? __float_as_uint(f) : 0x7f800000u);
            if ((tid & 31) == 0) atomicMax(norm, m);
        }
    } else if (MODE == kStep) {
        if (in) C[(size_t)i * N + j] = A[(size_t)i * N + j] + acc;
    } else if (in && i <= j) {
        const double x = A[(size_t)i * N + j] + acc;
        C[(size_t)i * N + j] = x;
        C[(size_t)j * N + i] = x;
    }
}

// X = S^-1 by Gauss-Jordan in FP64, one block, if N *norm exceeds 1e-7 (the residual after the
// last Newton-Schulz step is its square); otherwise nothing.  NaN where S is not positive
// definite.
__global__ void __launch_bounds__(1024)
    k_inv_repair(int N, const double* __restrict__ S, double* __restrict__ X,
                 const unsigned* __restrict__ norm) {
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
    const dim3 b(16, 16);
    switch ((N + 15) / 16) {
        case 1: launch_pdl(k_inv_f32<1>, dim3(1), b, 0, st, N, S, t0, norm); break;
        case 2: launch_pdl(k_inv_f32<2>, dim3(1), b, 0, st, N, S, t0, norm); break;
        case 3: launch_pdl(k_inv_f32<3>, dim3(1), b, 0, st, N, S, t0, norm); break;
        case 4: launch_pdl(k_inv_f32<4>, dim3(1), b, 0, st, N, S, t0, norm); break;
        case 5: launch_pdl(k_inv_f32<5>, dim3(1), b, 0, st, N, S, t0, norm); break;
        case 6: launch_pdl(k_inv_f32<6>, dim3(1), b, 0, st, N, S, t0, norm); break;
        case 7: launch_pdl(k_inv_f32<7>, dim3(1), b, 0, st, N, S, t0, norm); break;
        case 8: launch_pdl(k_inv_f32<8>, dim3(1), b, 0, st, N, S, t0, norm); break;
        case 9: launch_pdl(k_inv_f32<9>, dim3(1), b, 0, st, N, S, t0, norm); break;
        case 10: launch_pdl(k_inv_f32<10>, dim3(1), b, 0, st, N, S, t0, norm); break;
        case 11: launch_pdl(k_inv_f32<11>, dim3(1), b, 0, st, N, S, t0, norm); break;
        default: launch_pdl(k_inv_f32<12>, dim3(1), b, 0, st, N, S, t0, norm); break;
    }
    const dim3 g((N + kT - 1) / kT, (N + kT - 1) / kT), tb(kT * kT);
    unsigned* none = nullptr;
    launch_pdl(k_ns_product<kResid>, g, tb, 0, st, N, S, static_cast<const double*>(t0), t1, none);
    launch_pdl(k_ns_product<kStep>, g, tb, 0, st, N, static_cast<const double*>(t0),
               static_cast<const double*>(t1), t2, none);
    launch_pdl(k_ns_product<kResid>, g, tb, 0, st, N, S, static_cast<const double*>(t2), t1, norm);
    launch_pdl(k_ns_product<kLast>, g, tb, 0, st, N, static_cast<const double*>(t2),
               static_cast<const double*>(t1), Sinv, none);
    launch_pdl(k_inv_repair, dim3(1), dim3(1024), 2 * sizeof(double) * N, st, N, S, Sinv,
               static_cast<const unsigned*>(norm));
}

}  // namespace tdb
