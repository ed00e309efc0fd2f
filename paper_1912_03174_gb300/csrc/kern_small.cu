// Many steps of a small frozen-nuclei system in the FP64 form, one launch of one thread-block
// cluster (eq:leapfrog, eq:eomrho, eq:hscc, eq:qmulik; Sec. 2.2 dipole).
//
// At N = 40 a step is 0.2 MFLOP in five dependent kernels of three to four microseconds each.
// Here the CTAs of a cluster share out the rows of every matrix (R = ceil(N / CTAs) each), keep
// both density levels and H whole in their own shared memory, and exchange what the others need
// (rows of H, X transposed, rows of the new density with its Mulliken row sums) by stores into
// distributed shared memory, with three cluster barriers a step.  Bound by the latency of those
// exchanges and of the sums between them: the 3 R N^2 DFMA of a step and CTA take 3.5 of 11.2 us at
// N = 40 (two lanes a clock per SM).  Every sum is taken in the order of the separate
// kernels (k_charges, k_potential, k_gemm_f64, k_update), so both paths give the same bits.
// Measured, SCC off, N = 40: 11.2 us a step, 18.7 in separate kernels replayed as a graph.
#include <cooperative_groups.h>

#include <cmath>

#include "field.cuh"
#include "tdb_internal.h"

namespace tdb {

namespace {
namespace cg = cooperative_groups;

constexpr int kThreads = 256, kMaxN = kSmallStepN, kMaxRows = 4;
static_assert(kMaxRows * kMaxN <= kThreads && kMaxN <= 16 * kMaxRows && kMaxN % kTile == 0, "sizes");
constexpr int kTiles = kMaxN / kTile;

struct Smem {
    double rho[2][2][kMaxN][kMaxN];                  // [level][re, im], all rows
    double H[kMaxN][kMaxN];
    double xt[2][kMaxRows][kMaxN];                   // X[:, own rows] (re, im), pushed by the others
    double sinv[kMaxRows][kMaxN], s[kMaxRows][kMaxN], h0[kMaxRows][kMaxN];   // own rows
    double m[kMaxRows][kMaxN];
    double pv[kMaxRows][kTiles][kTile + 1];
    double partial[kMaxN][kTiles];                   // Mulliken row sums, all rows
    double dq[kMaxN], v[kMaxN], R[3 * kMaxN];
    double gamma[kMaxN][kMaxN];
    double red[4][kThreads / 32];
    double E[2][3];                                  // field of even and odd steps
};

__device__ __forceinline__ double wsum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__global__ void __launch_bounds__(kThreads)
    k_small_steps(SmallStepArgs a) {
    extern __shared__ __align__(16) unsigned char raw[];
    Smem& s = *reinterpret_cast<Smem*>(raw);
    cg::cluster_group cl = cg::this_cluster();
    const int nc = static_cast<int>(cl.num_blocks()), rank = static_cast<int>(cl.block_rank());
    const int N = a.N, nat = a.nat, nper = a.nper, nct = (N + kTile - 1) / kTile;
    const int rows = (N + nc - 1) / nc, r0 = rank * rows;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    DevScalars* sc = a.sc;
    // whole matrices and own rows (rows past N stay unused)
    for (int e = t; e < N * N; e += kThreads) {
        const int i = e / N, j = e - i * N;
        for (int l = 0; l < 2; ++l) {
            s.rho[l][0][i][j] = a.rho_re[l][e];
            s.rho[l][1][i][j] = a.rho_im[l][e];
        }
        if (i >= r0 && i < r0 + rows) {
            s.sinv[i - r0][j] = a.Sinv[e];
            s.s[i - r0][j] = a.S[e];
            s.h0[i - r0][j] = a.H0[e];
        }
    }
    for (int e = t; e < N * nct; e += kThreads) s.partial[e / nct][e % nct] = a.partial[e];
    for (int e = t; e < 3 * nat; e += kThreads) s.R[e] = a.R[e];
    for (int e = t; e < nat * nat; e += kThreads) s.gamma[e / nat][e % nat] = a.gamma[e];
    const long long n0 = sc->step;
    if (t == kThreads - 32)
        field_at(sc->field, sc->t_base + (double)(n0 - sc->n_base) * sc->dt, s.E[0]);
    // this thread's element (own row lr, column j)
    const int lr = t / N, j = t - lr * N, r = r0 + lr;
    const bool mine = lr < rows && r < N;
    cl.sync();
    int cur = a.cur;
    for (long k = 0; k < a.steps; ++k, cur ^= 1) {
        const int prv = cur ^ 1;
        const double* E = s.E[k & 1];
        // charges of rho_n: eight lanes per atom (nper nct <= 8 row sums; the other lanes of a
        // whole-warp sum would add zeros), all atoms at once
        for (int A0 = 0; A0 < nat; A0 += kThreads / 8) {
            const int A = A0 + (t >> 3), l = t & 7;
            double q = 0.0;
            if (A < nat && l < nper * nct) q += s.partial[A * nper + l / nct][l % nct];
            for (int o = 4; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
            if (A < nat && l == 0) s.dq[A] = q - a.q0[A];
        }
        __syncthreads();
        // potentials: sixteen lanes per atom up to sixteen atoms (the same argument), else a warp,
        // over the partners
        const int width = nat <= 16 ? 16 : 32;
        for (int A0 = 0; A0 < nat; A0 += kThreads / width) {
            const int A = A0 + t / width, l = t % width;
            double x = 0.0;
            if (a.scc && A < nat)
                for (int B = l; B < nat; B += 32) x += s.gamma[A][B] * s.dq[B];
            for (int o = width / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if (A < nat && l == 0)
                s.v[A] = x + s.R[3 * A] * E[0] + s.R[3 * A + 1] * E[1] + s.R[3 * A + 2] * E[2];
        }
        __syncthreads();
        // own rows of H = H0 + 1/2 S (v_r + v_j) into every CTA
        if (mine) {
            const double h = s.h0[lr][j] + 0.5 * s.s[lr][j] * (s.v[r / nper] + s.v[j / nper]);
            for (int c = 0; c < nc; ++c) *cl.map_shared_rank(&s.H[r][j], c) = h;
        }
        cl.sync();
        if (rank == nc - 1) {
            // dipole of rho_n into the ring (the totals of k_potential), on the last CTA, which has
            // the fewest rows or none
            double m0 = 0, m1 = 0, m2 = 0, ee = 0;
            for (int A = t; A < nat; A += kThreads) {
                const double d = s.dq[A];
                m0 -= d * s.R[3 * A];
                m1 -= d * s.R[3 * A + 1];
                m2 -= d * s.R[3 * A + 2];
                ee += d * (s.R[3 * A] * E[0] + s.R[3 * A + 1] * E[1] + s.R[3 * A + 2] * E[2]);
            }
            if (warp < 2) {   // nat <= 64
                m0 = wsum(m0);
                m1 = wsum(m1);
                m2 = wsum(m2);
                ee = wsum(ee);
            }
            if (lane == 0) {
                s.red[0][warp] = m0;
                s.red[1][warp] = m1;
                s.red[2][warp] = m2;
                s.red[3][warp] = ee;
            }
            __syncthreads();
            if (t < 4) {
                double x = 0;
                for (int w = 0; w < kThreads / 32; ++w) x += s.red[t][w];
                if (t < 3) {
                    sc->mu[t] = x;
                    sc->E[t] = E[t];
                    const long long slot = (n0 + k) % sc->hist_cap;
                    const long long s2 = slot < 0 ? slot + sc->hist_cap : slot;
                    a.hist[3 * s2 + t] = x;
                } else {
                    sc->e_ext = x;
                }
            }
        }
        // own rows of M = S^-1 H
        double acc = 0.0;
        if (mine) {
#pragma unroll 8
            for (int q = 0; q < N; ++q) acc = fma(s.sinv[lr][q], s.H[q][j], acc);
            s.m[lr][j] = acc;
        }
        // the next step's field, beside the products
        if (t == kThreads - 32 && k + 1 < a.steps)
            field_at(sc->field, sc->t_base + (double)(n0 + k + 1 - sc->n_base) * sc->dt, s.E[(k + 1) & 1]);
        __syncthreads();
        // own rows of X = M rho_n; X_rj goes to the owner of row j
        double xr = 0.0, xi = 0.0;
        if (mine) {
#pragma unroll 8
            for (int q = 0; q < N; ++q) {
                const double m = s.m[lr][q];
                xr = fma(m, s.rho[cur][0][q][j], xr);
                xi = fma(m, s.rho[cur][1][q][j], xi);
            }
            const int c = j / rows, jl = j - c * rows;
            *cl.map_shared_rank(&s.xt[0][jl][r], c) = xr;
            *cl.map_shared_rank(&s.xt[1][jl][r], c) = xi;
        }
        cl.sync();
        // leapfrog update of the own rows (base level prv), Mulliken row sums
        if (mine) {
            const double dre = xi + s.xt[1][lr][j], dim = s.xt[0][lr][j] - xr;
            const double nre = s.rho[prv][0][r][j] + a.factor * dre;
            const double nim = s.rho[prv][1][r][j] + a.factor * dim;
            for (int c = 0; c < nc; ++c) {
                *cl.map_shared_rank(&s.rho[prv][0][r][j], c) = nre;
                *cl.map_shared_rank(&s.rho[prv][1][r][j], c) = nim;
            }
            s.pv[lr][j / kTile][j % kTile] = nre * s.s[lr][j];
        }
        __syncthreads();
        if (t < rows * nct) {
            const int l = t / nct, ct = t - l * nct, row = r0 + l;
            if (row < N) {
                double sum = 0.0;
                const int len = N - ct * kTile < kTile ? N - ct * kTile : kTile;
                for (int q = 0; q < len; ++q) sum += s.pv[l][ct][q];
                for (int c = 0; c < nc; ++c) *cl.map_shared_rank(&s.partial[row][ct], c) = sum;
            }
        }
        cl.sync();
    }
    // own rows of both levels and of the row sums; the step counter
    if (mine)
        for (int l = 0; l < 2; ++l) {
            a.rho_re[l][(size_t)r * N + j] = s.rho[l][0][r][j];
            a.rho_im[l][(size_t)r * N + j] = s.rho[l][1][r][j];
        }
    if (t < rows * nct && r0 + t / nct < N)
        a.partial[(size_t)(r0 + t / nct) * nct + t % nct] = s.partial[r0 + t / nct][t % nct];
    if (rank == 0 && t == 0) sc->step = n0 + a.steps;
}

struct Launch {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    explicit Launch(cudaStream_t st) {
        cfg.gridDim = dim3(16);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = sizeof(Smem);
        cfg.stream = st;
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 16;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
    }
};

}  // namespace

bool small_steps_prepare() {
    int fits = 0;
    Launch l(nullptr);
    const bool ok = cudaFuncSetAttribute(k_small_steps, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         sizeof(Smem)) == cudaSuccess &&
                    cudaFuncSetAttribute(k_small_steps, cudaFuncAttributeNonPortableClusterSizeAllowed,
                                         1) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&fits, k_small_steps, &l.cfg) == cudaSuccess;
    if (!ok) cudaGetLastError();
    return ok && fits > 0;
}

cudaError_t launch_small_steps(const SmallStepArgs& a, cudaStream_t st) {
    Launch l(st);
    return cudaLaunchKernelEx(&l.cfg, k_small_steps, a);
}

}  // namespace tdb
