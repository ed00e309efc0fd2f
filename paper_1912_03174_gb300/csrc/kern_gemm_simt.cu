// SIMT matrix products (row-major C = A B).  FP64 (DFMA) for the FP64 form of
// the propagator and for the setup; FP32 (FFMA) for the TDB_FP32 form.  The
// B operand can be formed while it is loaded (the SCC Hamiltonian of eq:hscc,
// H_kj = H0_kj + 1/2 S_kj (v_k + v_j)), so H is never stored.
#include "pdl.cuh"
#include "tdb_internal.h"

namespace tdb {

namespace {

// B operands: raw(k, j) are the loads of an element (anything outside the matrix), value(raw, v_j)
// the element formed from them, col(j) what a column needs once.  (Ham loads without a branch:
// under one, the compiler forms the element at the load and waits for it there.)
struct Dense {
    const double* p;
    int ld;
    struct Raw {
        double x;
    };
    __device__ __forceinline__ Raw raw(int r, int c, bool in) const {
        return {in ? p[(size_t)r * ld + c] : 0.0};
    }
    __device__ __forceinline__ double col(int, bool) const { return 0.0; }
    __device__ __forceinline__ double value(const Raw& x, double) const { return x.x; }
};

// H_kj = H0_kj + 1/2 S_kj (v_k + v_j)
struct Ham {
    const double *H0, *S, *v;
    int N;
    struct Raw {
        double h, s, vk;
    };
    __device__ __forceinline__ Raw raw(int k, int j, bool in) const {
        const size_t i = in ? (size_t)k * N + j : 0;
        return {H0[i], S[i], v[in ? k : 0]};
    }
    __device__ __forceinline__ double col(int j, bool in) const { return in ? v[j] : 0.0; }
    __device__ __forceinline__ double value(const Raw& x, double vj) const {
        return x.h + 0.5 * x.s * (x.vk + vj);
    }
};

// FP64: an 8 x 8 tile of C per block of 64 threads, one output each; blockIdx.z picks one of
// two products that share A.  DFMA issues at two lanes a clock per SM on this part, so the
// product is bound by that pipe whatever the tile, and the tile only has to spread the work:
// 64 x 64 tiles left all but N^2 / 4096 of the 152 SMs idle below N = 800.  Each output sums
// its K terms in order.  A frozen FP64 step at N = 40: 173 us with 64 x 64 tiles and three
// product launches, 18.7 us with these and two (whole steps in one launch: 11.2, k_small_steps).
constexpr int kT8 = 8, kK8 = 64;

template <class LB>
__global__ void __launch_bounds__(kT8* kT8)
    k_gemm_f64(int M, int Ncol, int K, const double* A, int lda, LB lb0, LB lb1, double* C0, double* C1,
               int ldc) {
    __shared__ double As[kT8][kK8 + 2];
    __shared__ double Bs[kK8][kT8 + 1];
    const int tid = threadIdx.x, tx = tid % kT8, ty = tid / kT8;
    const int m0 = blockIdx.y * kT8, n0 = blockIdx.x * kT8;
    const LB lb = blockIdx.z ? lb1 : lb0;
    pdl_wait();
    double acc = 0.0, ra[kT8];
    typename LB::Raw rb[kT8];
    const double vj = lb.col(n0 + tx, n0 + tx < Ncol);
    auto load = [&](int k0) {
#pragma unroll
        for (int i = 0; i < kT8; ++i) {
            const int gm = m0 + i, ga = k0 + tid, gk = k0 + ty + kT8 * i, gn = n0 + tx;
            ra[i] = (gm < M && ga < K) ? A[(size_t)gm * lda + ga] : 0.0;
            rb[i] = lb.raw(gk, gn, gk < K && gn < Ncol);
        }
    };
    load(0);
    for (int k0 = 0; k0 < K; k0 += kK8) {
        if (k0) __syncthreads();
#pragma unroll
        for (int i = 0; i < kT8; ++i) {
            As[i][tid] = ra[i];
            const bool in = k0 + ty + kT8 * i < K && n0 + tx < Ncol;
            Bs[ty + kT8 * i][tx] = in ? lb.value(rb[i], vj) : 0.0;
        }
        __syncthreads();
        if (k0 + kK8 < K) load(k0 + kK8);   // while this block is multiplied
        const int len = K - k0 < kK8 ? K - k0 : kK8;
#pragma unroll 8
        for (int kk = 0; kk < len; ++kk) acc = fma(As[ty][kk], Bs[kk][tx], acc);
    }
    pdl_launch_dependents();   // at the end: see pdl.cuh
    const int gm = m0 + ty, gn = n0 + tx;
    if (gm < M && gn < Ncol) (blockIdx.z ? C1 : C0)[(size_t)gm * ldc + gn] = acc;
}

// FP32, large systems: a 64 x 64 tile of C per block of 128 threads, 8 x 4 consecutive outputs
// each, for one of up to three products of the same shape (blockIdx.z).  Bound by FFMA issue: a
// warp's step of K reads 2 + 2 shared-memory wavefronts for its 32 FFMA, and the next 32-deep
// block is loaded into registers while this one is multiplied (32 rather than 16: a block's
// multiplications then outlast a load).  Nothing may use a loaded value before the
// multiplications: delta H is formed where B goes to shared memory (formed in the load, it made
// delta M at N = 1024 take 113 us, now 75; X 178, now 173).  Each output sums its K terms in order.
constexpr int kF32Tile = 64, kF32K = 32, kF32Threads = 128, kF32Loads = 4;

struct F32Parts {
    F32Part p[3];
};

// B operand: dense, or delta H_kj = 1/2 S_kj (dv_k + dv_j) with S = b and dv set
template <bool DHAM>
__global__ void __launch_bounds__(kF32Threads, 3)
    k_gemm_f32(int M, int Ncol, int K, const __grid_constant__ F32Parts parts,
               const float* dv, const float* add, float* C2) {
    // A transposed; row r of k lies at r ^ 4 (k / 4 mod 8): the transposing stores hit all 32 banks
    __shared__ __align__(16) float As[2][kF32K][kF32Tile];
    __shared__ __align__(16) float Bs[2][kF32K][kF32Tile];
    const F32Part& P = parts.p[blockIdx.z];
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
    const int m0 = blockIdx.y * kF32Tile, n0 = blockIdx.x * kF32Tile;
    // loads of a block: A rows ar + 16 h (4 consecutive k each), B rows bk + 8 h (4 consecutive
    // columns each)
    const int ar = tid / 8, ak = 4 * (tid % 8), bk = tid / 16, bn = 4 * (tid % 16);
    const bool va = (P.lda % 4 == 0) && (reinterpret_cast<uintptr_t>(P.A) & 15) == 0;
    const bool vb = (P.ldb % 4 == 0) && (reinterpret_cast<uintptr_t>(P.B) & 15) == 0;
    float ra[kF32Loads][4], rb[kF32Loads][4], dk[kF32Loads];
    float dvn[4] = {0.f, 0.f, 0.f, 0.f};
    pdl_wait();
    if (DHAM)
#pragma unroll
        for (int j = 0; j < 4; ++j) dvn[j] = n0 + bn + j < Ncol ? dv[n0 + bn + j] : 0.f;
    auto load = [&](int k0) {
#pragma unroll
        for (int h = 0; h < kF32Loads; ++h) {
            const int gm = m0 + ar + 16 * h, ga = k0 + ak;
            const float* pa = P.A + (size_t)gm * P.lda + ga;
            if (va && gm < M && ga + 4 <= K) {
                const float4 v = *reinterpret_cast<const float4*>(pa);
                ra[h][0] = v.x, ra[h][1] = v.y, ra[h][2] = v.z, ra[h][3] = v.w;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) ra[h][j] = gm < M && ga + j < K ? pa[j] : 0.f;
            }
            const int gk = k0 + bk + 8 * h, gn = n0 + bn;
            const float* pb = P.B + (size_t)gk * P.ldb + gn;
            if (vb && gk < K && gn + 4 <= Ncol) {
                const float4 v = *reinterpret_cast<const float4*>(pb);
                rb[h][0] = v.x, rb[h][1] = v.y, rb[h][2] = v.z, rb[h][3] = v.w;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j) rb[h][j] = gk < K && gn + j < Ncol ? pb[j] : 0.f;
            }
            if (DHAM) dk[h] = gk < K ? dv[gk] : 0.f;
        }
    };
    auto store = [&](int s) {
#pragma unroll
        for (int h = 0; h < kF32Loads; ++h) {
#pragma unroll
            for (int j = 0; j < 4; ++j) As[s][ak + j][(ar + 16 * h) ^ ak] = ra[h][j];
            if (DHAM)
#pragma unroll
                for (int j = 0; j < 4; ++j) rb[h][j] = 0.5f * rb[h][j] * (dk[h] + dvn[j]);
            *reinterpret_cast<float4*>(&Bs[s][bk + 8 * h][bn]) =
                make_float4(rb[h][0], rb[h][1], rb[h][2], rb[h][3]);
        }
    };
    float acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    load(0);
    store(0);
    __syncthreads();
    int s = 0;
    for (int k0 = 0; k0 < K; k0 += kF32K, s ^= 1) {
        const bool more = k0 + kF32K < K;
        if (more) load(k0 + kF32K);
#pragma unroll
        for (int kk = 0; kk < kF32K; ++kk) {
            const float4 a0 = *reinterpret_cast<const float4*>(&As[s][kk][(8 * ty) ^ (kk & ~3)]);
            const float4 a1 = *reinterpret_cast<const float4*>(&As[s][kk][(8 * ty + 4) ^ (kk & ~3)]);
            const float4 b0 = *reinterpret_cast<const float4*>(&Bs[s][kk][4 * tx]);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float b[4] = {b0.x, b0.y, b0.z, b0.w};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        if (more) {
            store(s ^ 1);
            __syncthreads();
        }
    }
    pdl_launch_dependents();
    const int gn = n0 + 4 * tx;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int gm = m0 + 8 * ty + i;
        if (gm >= M) break;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (gn + j < Ncol) {
                P.C[(size_t)gm * P.ldc + gn + j] = acc[i][j];
                // M = M_gs + delta M beside delta M
                if (DHAM && C2) C2[(size_t)gm * P.ldc + gn + j] = add[(size_t)gm * Ncol + gn + j] + acc[i][j];
            }
    }
}

// FP32, up to one 64 x 64 tile per SM and product: smaller tiles, TM x TN of C per block, RM x RN
// outputs per thread (rows CY apart, columns in groups of four consecutive ones), for one of up to
// three products of the same shape (blockIdx.z).  With so little work per SM what bounds it is
// the latency of each K block: operands go to shared memory by asynchronous copies two blocks
// ahead, A as it lies in memory (a thread reads four K of its rows at a time), so that a block
// costs one barrier and few instructions beside its FFMA.  Each output sums its K terms in order.
// Microseconds, delta M / the three X products, 64 x 64 tiles of k_gemm_f32 and this: N = 40 7.6 / 5.8
// and 3.8 / 2.7, N = 260 16.8 / 17.3 and 11.1 / 8.2, N = 532 28.7 / 45.8 and 25.6 / 30.6.
template <int TM, int TN, int RM, int RN, int KB, int ST>
struct F32Tile {
    static constexpr int M = TM, N = TN, R = RM, C = RN, K = KB, S = ST, CX = TN / RN, CY = TM / RM,
                         T = CX * CY;
    static constexpr int KA = KB / 4, NB = TN / 4, LA = TM * KA / T, LB = KB * NB / T;
    static_assert(T % KA == 0 && T % NB == 0 && RN % 4 == 0 && LA * T == TM * KA && LB * T == KB * NB, "");
};

// 16 bytes (or 4) to shared memory, of which the first `bytes` are read and the rest are zero
__device__ __forceinline__ void copy16(float* dst, const float* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy4(float* dst, const float* src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src), "r"(bytes) : "memory");
}
// Four elements p[0 .. 3] of which the first n (any integer) exist; base is any valid address.
__device__ __forceinline__ void copy_row4(float* dst, const float* p, const float* base, int n, bool vec) {
    n = max(0, min(n, 4));
    if (vec) {
        copy16(dst, n ? p : base, 4 * n);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) copy4(dst + j, j < n ? p + j : base, j < n ? 4 : 0);
    }
}

template <bool DHAM, class X>
__global__ void __launch_bounds__(X::T)
    k_gemm_f32_small(int M, int Ncol, int K, const __grid_constant__ F32Parts parts,
               const float* dv, const float* add, float* C2) {
    __shared__ __align__(16) float As[X::S][X::M][X::K + 4];
    __shared__ __align__(16) float Bs[X::S][X::K][X::N];
    __shared__ float dks[DHAM ? X::S : 1][X::LB][X::T];
    const F32Part& P = parts.p[blockIdx.z];
    const int tid = threadIdx.x, tx = tid % X::CX, ty = tid / X::CX;
    const int m0 = blockIdx.y * X::M, n0 = blockIdx.x * X::N;
    const int ar = tid / X::KA, ak = 4 * (tid % X::KA), bk = tid / X::NB, bn = 4 * (tid % X::NB);
    const bool va = (P.lda % 4 == 0) && (reinterpret_cast<uintptr_t>(P.A) & 15) == 0;
    const bool vb = (P.ldb % 4 == 0) && (reinterpret_cast<uintptr_t>(P.B) & 15) == 0;
    const bool vc = (P.ldc % 4 == 0) && (reinterpret_cast<uintptr_t>(P.C) & 15) == 0;
    float dvn[4] = {0.f, 0.f, 0.f, 0.f};
    pdl_wait();
    if (DHAM)
#pragma unroll
        for (int j = 0; j < 4; ++j) dvn[j] = n0 + bn + j < Ncol ? dv[n0 + bn + j] : 0.f;
    auto load = [&](int k0, int s) {
        if (k0 < K) {
#pragma unroll
            for (int h = 0; h < X::LA; ++h) {
                const int r = ar + X::T / X::KA * h, gm = m0 + r;
                copy_row4(&As[s][r][ak], P.A + (size_t)gm * P.lda + k0 + ak, P.A,
                          gm < M ? K - k0 - ak : 0, va);
            }
#pragma unroll
            for (int h = 0; h < X::LB; ++h) {
                const int r = bk + X::T / X::NB * h, gk = k0 + r;
                copy_row4(&Bs[s][r][bn], P.B + (size_t)gk * P.ldb + n0 + bn, P.B,
                          gk < K ? Ncol - n0 - bn : 0, vb);
                if (DHAM) copy4(&dks[s][h][tid], gk < K ? dv + gk : dv, gk < K ? 4 : 0);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[X::R][X::C];
#pragma unroll
    for (int i = 0; i < X::R; ++i)
#pragma unroll
        for (int j = 0; j < X::C; ++j) acc[i][j] = 0.f;
#pragma unroll
    for (int s = 0; s < X::S - 1; ++s) load(s * X::K, s);
    int s = 0;
    for (int k0 = 0; k0 < K; k0 += X::K, s = s + 1 == X::S ? 0 : s + 1) {
        asm volatile("cp.async.wait_group %0;" ::"n"(X::S - 2) : "memory");
        if (DHAM)   // each thread turns the elements of S that it has copied into delta H
#pragma unroll
            for (int h = 0; h < X::LB; ++h) {
                float4* b = reinterpret_cast<float4*>(&Bs[s][bk + X::T / X::NB * h][bn]);
                const float dk = dks[s][h][tid];
                float4 v = *b;
                v.x = 0.5f * v.x * (dk + dvn[0]);
                v.y = 0.5f * v.y * (dk + dvn[1]);
                v.z = 0.5f * v.z * (dk + dvn[2]);
                v.w = 0.5f * v.w * (dk + dvn[3]);
                *b = v;
            }
        __syncthreads();
        load(k0 + (X::S - 1) * X::K, s == 0 ? X::S - 1 : s - 1);
#pragma unroll
        for (int k4 = 0; k4 < X::K; k4 += 4) {
            float4 a4[X::R];
#pragma unroll
            for (int i = 0; i < X::R; ++i) a4[i] = *reinterpret_cast<const float4*>(&As[s][ty + X::CY * i][k4]);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                float b[X::C];
#pragma unroll
                for (int q = 0; q < X::C; q += 4) {
                    const float4 v = *reinterpret_cast<const float4*>(&Bs[s][k4 + kk][4 * tx + X::CX * q]);
                    b[q] = v.x, b[q + 1] = v.y, b[q + 2] = v.z, b[q + 3] = v.w;
                }
#pragma unroll
                for (int i = 0; i < X::R; ++i) {
                    const float a = kk == 0 ? a4[i].x : kk == 1 ? a4[i].y : kk == 2 ? a4[i].z : a4[i].w;
#pragma unroll
                    for (int j = 0; j < X::C; ++j) acc[i][j] = fmaf(a, b[j], acc[i][j]);
                }
            }
        }
    }
    pdl_launch_dependents();
#pragma unroll
    for (int i = 0; i < X::R; ++i) {
        const int gm = m0 + ty + X::CY * i;
        if (gm >= M) break;
#pragma unroll
        for (int q = 0; q < X::C; q += 4) {
            const int gn = n0 + 4 * tx + X::CX * q;
            float* c = P.C + (size_t)gm * P.ldc + gn;
            if (vc && gn + 4 <= Ncol) {
                *reinterpret_cast<float4*>(c) = make_float4(acc[i][q], acc[i][q + 1], acc[i][q + 2], acc[i][q + 3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (gn + j < Ncol) c[j] = acc[i][q + j];
            }
            // M = M_gs + delta M beside delta M
            if (DHAM && C2)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (gn + j < Ncol)
                        C2[(size_t)gm * P.ldc + gn + j] = add[(size_t)gm * Ncol + gn + j] + acc[i][q + j];
        }
    }
}

// 64 x 32 tiles, or 32 x 32 where they leave fewer outputs on the fullest SM (N = 532: 36 and 31 us
// for X; where both leave as many the larger tile reads less, N = 700: 57 and 71).
using F32Wide = F32Tile<64, 32, 4, 4, 32, 3>;
using F32Narrow = F32Tile<32, 32, 4, 4, 32, 3>;

template <bool DHAM>
void run_f32(int M, int Ncol, int K, const F32Parts& p, int nparts, const float* dv, const float* add,
             float* C2, cudaStream_t st) {
    auto tiles = [&](int tm, int tn) { return ((M + tm - 1) / tm) * ((Ncol + tn - 1) / tn); };
    bool aligned = true;
    for (int z = 0; z < nparts; ++z)
        aligned = aligned && p.p[z].lda % 4 == 0 && p.p[z].ldb % 4 == 0 &&
                  ((reinterpret_cast<uintptr_t>(p.p[z].A) | reinterpret_cast<uintptr_t>(p.p[z].B)) & 15) == 0;
    // rows without 16-byte alignment are copied element by element, four times the copies of a block:
    // a step with these tiles / 64 x 64 ones, us: N = 70 23.5 / 30.7, 161 30.9 / 40.0, 193 32.8 / 43.3, 321
    // 47.1 / 57.3, 385 62.6 / 71.7, 513 95.0 / 90.8, 641 144 / 126.  (The line at 9 tiles, N = 192, is on
    // the safe side of that crossover.)
    auto go = [&](auto kernel, int tm, int tn, int threads) {
        launch_pdl(kernel, dim3((Ncol + tn - 1) / tn, (M + tm - 1) / tm, nparts), dim3(threads), 0, st, M,
                   Ncol, K, p, dv, add, C2);
    };
    if (tiles(64, 64) > (aligned ? kSmCount : 9)) {
        go(k_gemm_f32<DHAM>, kF32Tile, kF32Tile, kF32Threads);
    } else {
        auto fullest = [&](int tm, int tn) { return (tiles(tm, tn) * nparts + kSmCount - 1) / kSmCount * tm * tn; };
        const bool narrow = tiles(64, 32) * nparts > kSmCount && fullest(32, 32) < fullest(64, 32);
        if (narrow)
            go(k_gemm_f32_small<DHAM, F32Narrow>, F32Narrow::M, F32Narrow::N, F32Narrow::T);
        else
            go(k_gemm_f32_small<DHAM, F32Wide>, F32Wide::M, F32Wide::N, F32Wide::T);
    }
}

template <class LB>
void run_f64(int M, int Ncol, int K, const double* A, int lda, LB lb0, LB lb1, double* C0, double* C1,
             int ldc, cudaStream_t st) {
    const dim3 g((Ncol + kT8 - 1) / kT8, (M + kT8 - 1) / kT8, C1 ? 2 : 1);
    launch_pdl(k_gemm_f64<LB>, g, dim3(kT8 * kT8), 0, st, M, Ncol, K, A, lda, lb0, lb1, C0, C1, ldc);
}

}  // namespace

void gemm_f64(int M, int Ncol, int K, const double* A, int lda, const double* B, int ldb,
              double* C, int ldc, cudaStream_t st) {
    const Dense b{B, ldb};
    run_f64(M, Ncol, K, A, lda, b, b, C, static_cast<double*>(nullptr), ldc, st);
}

void gemm_f64_pair(int N, const double* A, const double* B0, const double* B1, double* C0,
                   double* C1, cudaStream_t st) {
    run_f64(N, N, N, A, N, Dense{B0, N}, Dense{B1, N}, C0, C1, N, st);
}

void gemm_f64_ham(int N, const double* A, const double* H0, const double* S, const double* v_orb,
                  double* C, cudaStream_t st) {
    const Ham h{H0, S, v_orb, N};
    run_f64(N, N, N, A, N, h, h, C, static_cast<double*>(nullptr), N, st);
}

void gemm_f32(int M, int Ncol, int K, const F32Part* parts, int nparts, cudaStream_t st) {
    F32Parts p{};
    for (int z = 0; z < nparts; ++z) p.p[z] = parts[z];
    run_f32<false>(M, Ncol, K, p, nparts, nullptr, nullptr, nullptr, st);
}

void gemm_f32_dham(int N, const float* A, const float* S, const float* dv, float* dM, float* Msum,
                   int ldc, const float* Mgs, cudaStream_t st) {
    F32Parts p{};
    p.p[0] = {A, N, S, N, dM, ldc};
    run_f32<true>(N, N, N, p, 1, dv, Mgs, Msum, st);
}

}  // namespace tdb
