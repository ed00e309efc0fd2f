// O(N^2) kernels of the propagation step and of the setup: model build
// (S, H0, gamma), Mulliken charges, SCC potential, leapfrog update, kick
// helpers and observable reductions.  All arithmetic is FP64.
#include <algorithm>
#include <cmath>

#include <cuda_fp16.h>

#include "field.cuh"
#include "pdl.cuh"
#include "tc_split.cuh"
#include "tdb_internal.h"

namespace tdb {

namespace {

__device__ __forceinline__ uint16_t to16(float x, int bf16) {
    if (bf16) return __bfloat16_as_ushort(__float2bfloat16_rn(x));
    return __half_as_ushort(__float2half_rn(x));
}
__device__ __forceinline__ float from16(uint16_t x, int bf16) {
    if (bf16) return __bfloat162float(__ushort_as_bfloat16(x));
    return __half2float(__ushort_as_half(x));
}

// head (integer, |h| <= 127) + two FP16 tails of a scaled FP32 value (exact split)
__device__ __forceinline__ void split_head3(float x, uint16_t (&q)[3]) {
    const float h = fminf(fmaxf(rintf(x), -127.f), 127.f);
    const float r = x - h;
    const __half rh = __float2half_rn(r);
    q[0] = __half_as_ushort(__float2half_rn(h));
    q[1] = __half_as_ushort(rh);
    q[2] = __half_as_ushort(__float2half_rn(r - __half2float(rh)));
}

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Short-range part zeta(R) of gamma for exponents ta, tb (tau = 16 U / 5):
// Coulomb integral of two normalised exp(-tau r) densities is 1/R - zeta(R).
__device__ double gamma_short(double ta, double tb, double R) {
    const double tmax = ta > tb ? ta : tb;
    if (fabs(ta - tb) < 3e-4 * tmax) {
        const double t = 0.5 * (ta + tb);
        return exp(-t * R) * (1.0 / R + 11.0 * t / 16.0 + 3.0 * t * t * R / 16.0 +
                              t * t * t * R * R / 48.0);
    }
    double z = 0.0;
    for (int s = 0; s < 2; ++s) {
        const double a = s ? tb : ta, b = s ? ta : tb;
        const double a2 = a * a, b2 = b * b, d = a2 - b2;
        const double b4 = b2 * b2;
        z += exp(-a * R) * (b4 * a / (2.0 * d * d) - (b4 * b2 - 3.0 * a2 * b4) / (d * d * d * R));
    }
    return z;
}

// One thread per atom pair A <= B (blockIdx.y = A) writes the nper x nper blocks (A, B) and
// (B, A) of S and H0 and gamma_AB = gamma_BA (eq:coul).  Off-site: Slater-Koster s/p table with
// direction cosines c of R_B - R_A:
//   ss = K0, s-a = c_a K1, a-s = -c_a K1, a-b = c_a c_b (K2 - K3) + delta_ab K3,
// with hopping K = eta t0 exp(-r/lam_H) and overlap K = -eta s0 exp(-r/lam_S); the block (B, A)
// is the transpose, element for element.  FP64 issue bounds it (two lanes a clock per SM): every
// pair is evaluated once.
constexpr int kPairThreads = 64;

__global__ void __launch_bounds__(kPairThreads)
    k_build_pair(int nat, int nper, const double* R, const double* onsite,
                 const double* U, ModelParams mp, double* S,
                 double* H0, double* G) {
    const int A = blockIdx.y, B = blockIdx.x * kPairThreads + threadIdx.x;
    pdl_wait();
    if (B < A || B >= nat) return;
    const int N = nat * nper;
    double hb[4][4], sb[4][4];
    if (A == B) {
        for (int i = 0; i < 4; ++i)
            for (int j = 0; j < 4; ++j) {
                sb[i][j] = (i == j) ? 1.0 : 0.0;
                hb[i][j] = (i == j && i < nper) ? onsite[A * nper + i] : 0.0;
            }
        G[(size_t)A * nat + A] = U[A];
    } else {
        const double dx = R[3 * B] - R[3 * A], dy = R[3 * B + 1] - R[3 * A + 1],
                     dz = R[3 * B + 2] - R[3 * A + 2];
        const double r = sqrt(dx * dx + dy * dy + dz * dz);
        const double c[3] = {dx / r, dy / r, dz / r};
        const double eh = exp(-r / mp.lam_H), es = exp(-r / mp.lam_S);
        double kh[4], ks[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            kh[k] = mp.eta[k] * mp.t0 * eh;
            ks[k] = -mp.eta[k] * mp.s0 * es;
        }
        hb[0][0] = kh[0];
        sb[0][0] = ks[0];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            hb[0][1 + a] = c[a] * kh[1];
            sb[0][1 + a] = c[a] * ks[1];
            hb[1 + a][0] = -hb[0][1 + a];
            sb[1 + a][0] = -sb[0][1 + a];
#pragma unroll
            for (int b = 0; b <= a; ++b) {
                const double cc = c[a] * c[b];
                hb[1 + a][1 + b] = cc * (kh[2] - kh[3]) + (a == b ? kh[3] : 0.0);
                sb[1 + a][1 + b] = cc * (ks[2] - ks[3]) + (a == b ? ks[3] : 0.0);
                hb[1 + b][1 + a] = hb[1 + a][1 + b];
                sb[1 + b][1 + a] = sb[1 + a][1 + b];
            }
        }
        // the two exponents' terms are summed in the order of the row's atom, as ever
        const double ta = 3.2 * U[A], tb = 3.2 * U[B];
        const double g = 1.0 / r - gamma_short(ta, tb, r);
        G[(size_t)A * nat + B] = g;
        G[(size_t)B * nat + A] = ta == tb ? g : 1.0 / r - gamma_short(tb, ta, r);
    }
    if (nper == 4) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const size_t ab = (size_t)(4 * A + i) * N + 4 * B, ba = (size_t)(4 * B + i) * N + 4 * A;
            double2 *s0 = reinterpret_cast<double2*>(S + ab), *h0 = reinterpret_cast<double2*>(H0 + ab);
            s0[0] = make_double2(sb[i][0], sb[i][1]);
            s0[1] = make_double2(sb[i][2], sb[i][3]);
            h0[0] = make_double2(hb[i][0], hb[i][1]);
            h0[1] = make_double2(hb[i][2], hb[i][3]);
            if (A != B) {
                double2 *s1 = reinterpret_cast<double2*>(S + ba), *h1 = reinterpret_cast<double2*>(H0 + ba);
                s1[0] = make_double2(sb[0][i], sb[1][i]);
                s1[1] = make_double2(sb[2][i], sb[3][i]);
                h1[0] = make_double2(hb[0][i], hb[1][i]);
                h1[1] = make_double2(hb[2][i], hb[3][i]);
            }
        }
    } else {
        S[(size_t)A * N + B] = S[(size_t)B * N + A] = sb[0][0];
        H0[(size_t)A * N + B] = H0[(size_t)B * N + A] = hb[0][0];
    }
}

// Row-major upper triangle -> lower triangle (after a column-major lower potri).
__global__ void k_sym_upper_to_lower(int N, double* A) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y * blockDim.y + threadIdx.y;
    if (r < N && c < N && r > c) A[(size_t)r * N + c] = A[(size_t)c * N + r];
}

__global__ void k_transpose(int N, const double* __restrict__ in, double* __restrict__ out) {
    __shared__ double t[kTile][kTile + 1];
    const int bx = blockIdx.x * kTile, by = blockIdx.y * kTile;
    for (int y = threadIdx.y; y < kTile; y += blockDim.y) {
        const int r = by + y, c = bx + threadIdx.x;
        if (r < N && c < N) t[y][threadIdx.x] = in[(size_t)r * N + c];
    }
    __syncthreads();
    for (int y = threadIdx.y; y < kTile; y += blockDim.y) {
        const int r = bx + y, c = by + threadIdx.x;
        if (r < N && c < N) out[(size_t)r * N + c] = t[threadIdx.x][y];
    }
}

// Sum of a row of 32 products, in column order.  The order is kept everywhere: a state loaded
// from a checkpoint continues bitwise, and the reduced forms round differently (1e-9 .. 1e-7 of
// the dipole) for ground-state charges that differ in their last bits.
__device__ __forceinline__ double tile_row_sum_f64(const double* row) {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < kTile; ++k) s += row[k];
    return s;
}

// partial[row][ct] = sum over the 32 columns of tile ct of Re rho[row][col] * S[row][col]
// (eq:qmulik: q_A = sum_{nu in A} Re (rho S)_{nu nu}; S is symmetric).  Summed as the update
// kernel sums them, so a state loaded from a checkpoint continues bitwise.
__global__ void __launch_bounds__(256)
    k_mulliken_partials(int N, int nct, const double* rre, const double* S,
                        double* partial) {
    __shared__ double pv_s[kTile][kTile + 1];
    const int ct = blockIdx.x;
    const int col = ct * kTile + threadIdx.x;
    pdl_launch_dependents();
    pdl_wait();
#pragma unroll
    for (int k = 0; k < kTile / 8; ++k) {
        const int y = threadIdx.y + 8 * k, row = blockIdx.y * kTile + y;
        double v = 0.0;
        if (row < N && col < N) v = rre[(size_t)row * N + col] * S[(size_t)row * N + col];
        pv_s[y][threadIdx.x] = v;
    }
    __syncthreads();
    if (threadIdx.y == 0) {
        const int row = blockIdx.y * kTile + threadIdx.x;
        const double sum = tile_row_sum_f64(pv_s[threadIdx.x]);
        if (row < N) partial[(size_t)row * nct + ct] = sum;
    }
}

// q_A = sum of the Mulliken row partials of A's orbitals (contiguous in the
// [row][ct] layout): one warp per atom.
__global__ void k_charges(int nat, int nper, int nct, const double* partial,
                          const double* q0, double* q,
                          double* dq, double* reset0, double* reset1,
                          tc::DynScales* dyn, int cur,
                          const double* qbase) {
    const int lane = threadIdx.x & 31;
    const int A = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    // the potentials kernel may start once the previous step's update is complete: it then
    // evaluates the field at this step's time while the charges are summed
    pdl_wait();
    pdl_launch_dependents();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (reset0) *reset0 = 0.0;
        if (reset1) *reset1 = 0.0;
        if (dyn) {
            // FP16X6 bookkeeping of a step: the maximum of the deviation written by the
            // previous update now describes buffer cur; start this step's maxima
            dyn->max_drho[cur] = dyn->max_drho[2];
            dyn->max_drho[2] = 0.0;
            for (int k = 0; k < tc::kMaxParts; ++k) dyn->max_x[k] = 0.0;
        }
    }
    if (A >= nat) return;
    const double* p = partial + (size_t)A * nper * nct;
    double s = 0.0;
#pragma unroll 4
    for (int i = lane; i < nper * nct; i += 32) s += p[i];
    s = warp_sum(s);
    if (lane == 0) {
        if (qbase) s += qbase[A];   // partials of the deviation rho - rho_ref
        q[A] = s;
        dq[A] = s - q0[A];
    }
}

// Warp per atom A: gdq_A = sum_B gamma_AB dq_B;  v_A = [scc] gdq_A + R_A . E(t_n)
// (eq:hscc, eq:hsccvext with V_ext,A = R_A . E).  With `record`, one more block (the last) puts
// E(t_n), the dipole mu = -sum_A dq_A R_A (also into the history ring) and sum_A dq_A V_ext,A
// into sc.  `early` (launched behind k_charges, whose blocks release it after the step counter's
// writer has finished): the field is evaluated before the wait for the charges.
__global__ void __launch_bounds__(256)
    k_potential(int nat, int nper, int scc, const double* gamma,
                const double* dq, const double* R,
                DevScalars* sc, double* v_orb,
                double* v_atom, double* gdq,
                double* hist, const double* v_ref,
                float* dv_f, double* max_dv, int record, int early) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarp = blockDim.x >> 5;
    const int nab = gridDim.x - (record ? 1 : 0);
    __shared__ double E_sh[3];
    if (!early) pdl_wait();
    const long long n = sc->step;
    // the field at t_n, evaluated once per block
    if (threadIdx.x == 0) {
        const double t = sc->t_base + (double)(n - sc->n_base) * sc->dt;
        field_at(sc->field, t, E_sh);
    }
    if (early) pdl_wait();
    pdl_launch_dependents();
    __syncthreads();
    const double E[3] = {E_sh[0], E_sh[1], E_sh[2]};
    if ((int)blockIdx.x < nab) {
        for (int A = blockIdx.x * nwarp + warp; A < nat; A += nab * nwarp) {
            double s = 0.0;
            if (scc) {
                const double* g = gamma + (size_t)A * nat;
#pragma unroll 8
                for (int B = lane; B < nat; B += 32) s += g[B] * dq[B];
            }
            s = warp_sum(s);
            const double vA = s + R[3 * A] * E[0] + R[3 * A + 1] * E[1] + R[3 * A + 2] * E[2];
            if (lane < nper) {
                const int o = A * nper + lane;
                v_orb[o] = vA;
                if (dv_f) dv_f[o] = (float)(vA - v_ref[o]);
            }
            if (lane == 0) {
                v_atom[A] = vA;
                gdq[A] = s;
                if (max_dv)
                    atomicMax(reinterpret_cast<unsigned long long*>(max_dv),
                              (unsigned long long)__double_as_longlong(fabs(vA - v_ref[A * nper])));
            }
        }
        return;
    }
    __shared__ double red[4][32];
    double m0 = 0, m1 = 0, m2 = 0, ee = 0;
    for (int A = threadIdx.x; A < nat; A += blockDim.x) {
        const double d = dq[A];
        m0 -= d * R[3 * A];
        m1 -= d * R[3 * A + 1];
        m2 -= d * R[3 * A + 2];
        ee += d * (R[3 * A] * E[0] + R[3 * A + 1] * E[1] + R[3 * A + 2] * E[2]);
    }
    m0 = warp_sum(m0);
    m1 = warp_sum(m1);
    m2 = warp_sum(m2);
    ee = warp_sum(ee);
    if (lane == 0) {
        red[0][warp] = m0;
        red[1][warp] = m1;
        red[2][warp] = m2;
        red[3][warp] = ee;
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        double a = 0;
        for (int w = 0; w < nwarp; ++w) a += red[threadIdx.x][w];
        if (threadIdx.x < 3) {
            sc->mu[threadIdx.x] = a;
            sc->E[threadIdx.x] = E[threadIdx.x];
            const long long slot = n % sc->hist_cap;
            const long long s2 = slot < 0 ? slot + sc->hist_cap : slot;
            hist[3 * s2 + threadIdx.x] = a;
        } else {
            sc->e_ext = a;
        }
    }
}

__global__ void k_build_hamiltonian(int N, const double* __restrict__ H0,
                                    const double* __restrict__ S, const double* __restrict__ v,
                                    double* __restrict__ H) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y * blockDim.y + threadIdx.y;
    if (r >= N || c >= N) return;
    const size_t i = (size_t)r * N + c;
    H[i] = H0[i] + 0.5 * S[i] * (v[r] + v[c]);
}

// Leapfrog / Euler update of the FP64 form (eq:leapfrog with eq:eomrho):
//   out = base + factor * rhodot,  rhodot = -i (X - X^dagger) - (Z + Z^dagger),
//   X = S^-1 H rho, Z = S^-1 D rho (moving nuclei only).
// Re rhodot_ij = Im X_ij + Im X_ji;  Im rhodot_ij = -(Re X_ij - Re X_ji).
// A block (32 x 8 threads) owns the tile pair (bi, bj), bi <= bj: rhodot is formed once and used
// for both halves, so rho stays exactly Hermitian.  Z joins X when the tiles are loaded,
//   rhodot_re,ij = b_ij + b_ji, rhodot_im,ij = a_ji - a_ij, a = Re X + Im Z, b = Im X - Re Z.
// The Mulliken row partials of the new rho are fused in.  Bound by HBM and, about equally, by FP64
// issue (two lanes a clock per SM).
__global__ void __launch_bounds__(256)
    k_update(int N, int nct, const double* Xre, const double* Xim,
             const double* bre, const double* bim,
             double* ore, double* oim, double factor,
             const double* S, double* partial,
             DevScalars* sc, const double* zre,
             const double* zim) {
    // block b = bj (bj + 1) / 2 + bi
    const int blk = blockIdx.x;
    int bj = (int)((sqrtf(8.0f * (float)blk + 1.0f) - 1.0f) * 0.5f);
    while (bj * (bj + 1) / 2 > blk) --bj;
    while ((bj + 1) * (bj + 2) / 2 <= blk) ++bj;
    const int bi = blk - bj * (bj + 1) / 2;
    constexpr int RPT = kTile / 8;   // rows per thread
    __shared__ double t_re[kTile][kTile + 1], t_im[kTile][kTile + 1];   // (j, i) tile of X, then rhodot
    __shared__ double pv_s[2][kTile][kTile + 1];   // products of both halves
    const int tx = threadIdx.x, ty = threadIdx.y;
    pdl_launch_dependents();
    pdl_wait();
    double a_ij[RPT], b_ij[RPT];
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
        const int y = ty + 8 * k;
        int r = bi * kTile + y, c = bj * kTile + tx;
        double a = 0, b = 0;
        if (r < N && c < N) {
            const size_t i = (size_t)r * N + c;
            a = Xre[i];
            b = Xim[i];
            if (zre) {
                a += zim[i];
                b -= zre[i];
            }
        }
        a_ij[k] = a;
        b_ij[k] = b;
        r = bj * kTile + y;
        c = bi * kTile + tx;
        a = 0;
        b = 0;
        if (r < N && c < N) {
            const size_t i = (size_t)r * N + c;
            a = Xre[i];
            b = Xim[i];
            if (zre) {
                a += zim[i];
                b -= zre[i];
            }
        }
        t_re[y][tx] = a;
        t_im[y][tx] = b;
    }
    __syncthreads();
    // rhodot of the (i, j) tile into registers; then, through shared memory, to the other half
    double dre[RPT], dim[RPT];
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
        const int y = ty + 8 * k;
        dre[k] = b_ij[k] + t_im[tx][y];
        dim[k] = t_re[tx][y] - a_ij[k];
    }
    if (bi != bj) {
        __syncthreads();
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            t_re[ty + 8 * k][tx] = dre[k];
            t_im[ty + 8 * k][tx] = dim[k];
        }
        __syncthreads();
    }
    for (int half = 0; half < (bi == bj ? 1 : 2); ++half) {
        const int ti = half ? bj : bi, tj = half ? bi : bj;
        double b_re[RPT], b_im[RPT], s_v[RPT];
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            const int r = ti * kTile + ty + 8 * k, c = tj * kTile + tx;
            b_re[k] = b_im[k] = s_v[k] = 0.0;
            if (r < N && c < N) {
                const size_t i = (size_t)r * N + c;
                b_re[k] = bre[i];
                b_im[k] = bim[i];
                s_v[k] = S[i];
            }
        }
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            const int y = ty + 8 * k;
            const int r = ti * kTile + y, c = tj * kTile + tx;
            double pv = 0.0;
            if (r < N && c < N) {
                const double d0 = half ? t_re[tx][y] : dre[k];
                const double d1 = half ? -t_im[tx][y] : dim[k];
                const size_t i = (size_t)r * N + c;
                const double nre = b_re[k] + factor * d0;
                const double nim = b_im[k] + factor * d1;
                ore[i] = nre;
                oim[i] = nim;
                pv = nre * s_v[k];
            }
            pv_s[half][y][tx] = pv;
        }
    }
    __syncthreads();
    // one warp per half
    if (ty < (bi == bj ? 1 : 2)) {
        const int r = (ty ? bj : bi) * kTile + tx;
        const double sum = tile_row_sum_f64(pv_s[ty][tx]);
        if (r < N) partial[(size_t)r * nct + (ty ? bi : bj)] = sum;
    }
    if (blk == 0 && threadIdx.x == 0 && threadIdx.y == 0) sc->step += 1;
}

// C = diag(p) P diag(conj p), p_mu = exp(-i E0 dir . R_A(mu)): the phase factors of
// eq:rhokick with V = -E0 diag(dir . R).
__global__ void k_kick_phase(int N, int nper, const double* __restrict__ R, double E0, double d0,
                             double d1, double d2, const double* __restrict__ Pre,
                             const double* __restrict__ Pim, double* __restrict__ Cre,
                             double* __restrict__ Cim) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y * blockDim.y + threadIdx.y;
    if (r >= N || c >= N) return;
    const int A = r / nper, B = c / nper;
    const double xa = d0 * R[3 * A] + d1 * R[3 * A + 1] + d2 * R[3 * A + 2];
    const double xb = d0 * R[3 * B] + d1 * R[3 * B + 1] + d2 * R[3 * B + 2];
    // p_r conj(p_c) = exp(-i E0 (x_a - x_b))
    double sn, cs;
    sincos(-E0 * (xa - xb), &sn, &cs);
    const size_t i = (size_t)r * N + c;
    const double pr = Pre[i], pi = Pim[i];
    Cre[i] = cs * pr - sn * pi;
    Cim[i] = cs * pi + sn * pr;
}

// out = 1/2 (T + T^dagger)
__global__ void k_hermitian_half(int N, const double* __restrict__ Tre,
                                 const double* __restrict__ Tim, double* __restrict__ ore,
                                 double* __restrict__ oim) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y * blockDim.y + threadIdx.y;
    if (r >= N || c >= N) return;
    const size_t i = (size_t)r * N + c, j = (size_t)c * N + r;
    ore[i] = 0.5 * (Tre[i] + Tre[j]);
    oim[i] = 0.5 * (Tim[i] - Tim[j]);
}

// Per block (persistent over tile pairs bi <= bj): sum Re rho * H0, sum Re rho * S, sum Im rho *
// S, max |rho_ij - conj rho_ji|; the transposed tiles go through shared memory.
__global__ void __launch_bounds__(256)
    k_obs_reduce(int N, int npair, const double* __restrict__ rre, const double* __restrict__ rim,
                 const double* __restrict__ H0, const double* __restrict__ S, double* __restrict__ out) {
    __shared__ double t_re[kTile][kTile + 1], t_im[kTile][kTile + 1];
    const int tx = threadIdx.x, ty = threadIdx.y;
    double a = 0, b = 0, c = 0, m = 0;
    for (int blk = blockIdx.x; blk < npair; blk += gridDim.x) {
        int bj = (int)((sqrtf(8.0f * (float)blk + 1.0f) - 1.0f) * 0.5f);
        while (bj * (bj + 1) / 2 > blk) --bj;
        while ((bj + 1) * (bj + 2) / 2 <= blk) ++bj;
        const int bi = blk - bj * (bj + 1) / 2;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kTile / 8; ++k) {
            const int y = ty + 8 * k, r = bj * kTile + y, col = bi * kTile + tx;
            double re = 0, im = 0;
            if (r < N && col < N) {
                const size_t i = (size_t)r * N + col;
                re = rre[i];
                im = rim[i];
                if (bi != bj) {
                    a = fma(re, H0[i], a);
                    b = fma(re, S[i], b);
                    c = fma(im, S[i], c);
                }
            }
            t_re[y][tx] = re;
            t_im[y][tx] = im;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kTile / 8; ++k) {
            const int y = ty + 8 * k, r = bi * kTile + y, col = bj * kTile + tx;
            if (r < N && col < N) {
                const size_t i = (size_t)r * N + col;
                const double re = rre[i], im = rim[i];
                a = fma(re, H0[i], a);
                b = fma(re, S[i], b);
                c = fma(im, S[i], c);
                const double e1 = fabs(re - t_re[tx][y]), e2 = fabs(im + t_im[tx][y]);
                m = fmax(m, fmax(e1, e2));
            }
        }
    }
    __shared__ double red[4][8];
    a = warp_sum(a);
    b = warp_sum(b);
    c = warp_sum(c);
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (tx == 0) {
        red[0][ty] = a;
        red[1][ty] = b;
        red[2][ty] = c;
        red[3][ty] = m;
    }
    __syncthreads();
    if (ty == 0 && tx < 4) {
        double s = red[tx][0];
        for (int k = 1; k < 8; ++k) s = tx == 3 ? fmax(s, red[3][k]) : s + red[tx][k];
        out[4 * blockIdx.x + tx] = s;
    }
}

// One warp per quantity: the block sums (and the maximum, quantity 3).
__global__ void k_obs_finish(int nb, const double* __restrict__ in, double* __restrict__ out) {
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    double s = 0;
    for (int k = lane; k < nb; k += 32) s = q == 3 ? fmax(s, in[4 * k + q]) : s + in[4 * k + q];
    for (int o = 16; o > 0; o >>= 1) {
        const double t = __shfl_xor_sync(0xffffffffu, s, o);
        s = q == 3 ? fmax(s, t) : s + t;
    }
    if (lane == 0) out[q] = s;
}

// out[m][k] = in[m][k] * f[k]
__global__ void k_scale_cols(int N, const double* __restrict__ in, const double* __restrict__ f,
                             double* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y * blockDim.y + threadIdx.y;
    if (r >= N || c >= N) return;
    out[(size_t)r * N + c] = in[(size_t)r * N + c] * f[c];
}

inline dim3 grid2(int nx, int ny, dim3 b) {
    return dim3((nx + b.x - 1) / b.x, (ny + b.y - 1) / b.y);
}

}  // namespace

void launch_build_pair(const Ctx& c, const double* R, double* S, double* H0, double* gamma,
                       cudaStream_t st) {
    const dim3 g((c.nat + kPairThreads - 1) / kPairThreads, c.nat);
    launch_pdl(k_build_pair, g, dim3(kPairThreads), 0, st, c.nat, c.nper, R, c.d_onsite, c.d_U, c.mp, S,
               H0, gamma);
}

void launch_symmetrize_upper_to_lower(int N, double* A, cudaStream_t st) {
    dim3 b(32, 8);
    k_sym_upper_to_lower<<<grid2(N, N, b), b, 0, st>>>(N, A);
}

void launch_transpose(int N, const double* in, double* out, cudaStream_t st) {
    dim3 b(kTile, 8);
    dim3 g((N + kTile - 1) / kTile, (N + kTile - 1) / kTile);
    k_transpose<<<g, b, 0, st>>>(N, in, out);
}

void launch_mulliken_partials(int N, const double* rho_re, const double* S, double* partial,
                              cudaStream_t st) {
    const int nct = (N + kTile - 1) / kTile;
    launch_pdl(k_mulliken_partials, dim3(nct, nct), dim3(kTile, 8), 0, st, N, nct, rho_re, S, partial);
}

void launch_charges(const Ctx& c, const double* partial, double* q, double* dq, cudaStream_t st,
                    double* reset0, double* reset1, tc::DynScales* dyn, int cur,
                    const double* qbase) {
    launch_pdl(k_charges, dim3((c.nat + 7) / 8), dim3(256), 0, st, c.nat, c.nper, c.nct, partial,
               (const double*)c.d_q0, q, dq, reset0, reset1, dyn, cur, qbase);
}

void launch_potential(const Ctx& c, const double* gamma, const double* dq, const double* R,
                      DevScalars* sc, double* v_orb, double* v_atom, double* gdq, double* hist,
                      const double* v_ref, float* dv_orb, cudaStream_t st, double* max_dv,
                      int record, int after_charges) {
    const int warps = 8;
    const int blocks = (c.nat + warps - 1) / warps + (record ? 1 : 0);
    launch_pdl(k_potential, dim3(blocks), dim3(warps * 32), 0, st, c.nat, c.nper, c.prm.scc, gamma, dq, R,
               sc, v_orb, v_atom, gdq, hist, v_ref, dv_orb, max_dv, record, after_charges);
}

void launch_build_hamiltonian(int N, const double* H0, const double* S, const double* v_orb,
                              double* H, cudaStream_t st) {
    dim3 b(32, 8);
    k_build_hamiltonian<<<grid2(N, N, b), b, 0, st>>>(N, H0, S, v_orb, H);
}

void launch_update(const Ctx& c, const double* Xre, const double* Xim, const double* base_re,
                   const double* base_im, double* out_re, double* out_im, double factor,
                   const double* S, double* partial, DevScalars* sc, cudaStream_t st,
                   const double* zre, const double* zim) {
    launch_pdl(k_update, dim3(c.nct * (c.nct + 1) / 2), dim3(kTile, 8), 0, st, c.N, c.nct, Xre, Xim,
               base_re, base_im, out_re, out_im, factor, S, partial, sc, zre, zim);
}

void launch_kick_phase(int N, int n_per, const double* R, double strength, const double* dir,
                       const double* Pre, const double* Pim, double* Cre, double* Cim,
                       cudaStream_t st) {
    dim3 b(32, 8);
    k_kick_phase<<<grid2(N, N, b), b, 0, st>>>(N, n_per, R, strength, dir[0], dir[1], dir[2], Pre,
                                               Pim, Cre, Cim);
}

void launch_hermitian_half(int N, const double* Tre, const double* Tim, double* out_re,
                           double* out_im, cudaStream_t st) {
    dim3 b(32, 8);
    k_hermitian_half<<<grid2(N, N, b), b, 0, st>>>(N, Tre, Tim, out_re, out_im);
}

void launch_obs_reduce(int N, const double* rho_re, const double* rho_im, const double* H0,
                       const double* S, double* block_out, int n_blocks, cudaStream_t st) {
    const int nt = (N + kTile - 1) / kTile;
    k_obs_reduce<<<n_blocks, dim3(kTile, 8), 0, st>>>(N, nt * (nt + 1) / 2, rho_re, rho_im, H0, S,
                                                      block_out);
}

void launch_obs_finish(int n_blocks, const double* block_out, double* out4, cudaStream_t st) {
    k_obs_finish<<<1, 128, 0, st>>>(n_blocks, block_out, out4);
}

void launch_scale_rows_f(int N, const double* in, const double* f, double* out, cudaStream_t st) {
    dim3 b(32, 8);
    k_scale_cols<<<grid2(N, N, b), b, 0, st>>>(N, in, f, out);
}

}  // namespace tdb

namespace tdb {

namespace {

__global__ void k_f64_to_f32(size_t n, const double* __restrict__ in, float* __restrict__ out) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        out[i] = (float)in[i];
}

// Start of the Newton-Schulz inverse at the next geometry: X <- 2 X - P (the line through the
// last two inverses; P = null: X stays), P <- X, and a zeroed residual norm.
__global__ void k_ns_start(size_t n, double* X, double* P, int line,
                           unsigned* norm) {
    pdl_launch_dependents();
    pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0) *norm = 0u;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
        const double x = X[i];
        if (line) X[i] = 2.0 * x - P[i];
        P[i] = x;
    }
}

// X <- X + 1/2 (Q + Q^T) for a symmetric X: one block per tile pair, so X stays exactly
// symmetric.  With a gate: nothing if *gate (float bits) is below `below`.
__global__ void __launch_bounds__(256)
    k_ns_update(int N, double* X, const double* Q,
                const unsigned* gate, float below) {
    __shared__ double a[kTile][kTile + 1], b[kTile][kTile + 1];
    const int bi = blockIdx.y, bj = blockIdx.x;
    pdl_launch_dependents();
    pdl_wait();
    if (bi > bj || (gate && __uint_as_float(__ldcg(gate)) < below)) return;
    const int tx = threadIdx.x;
    for (int y = threadIdx.y; y < kTile; y += 8) {
        const int r = bi * kTile + y, c = bj * kTile + tx, r2 = bj * kTile + y, c2 = bi * kTile + tx;
        a[y][tx] = r < N && c < N ? Q[(size_t)r * N + c] : 0.0;
        b[y][tx] = r2 < N && c2 < N ? Q[(size_t)r2 * N + c2] : 0.0;
    }
    __syncthreads();
    for (int y = threadIdx.y; y < kTile; y += 8) {
        const int r = bi * kTile + y, c = bj * kTile + tx, r2 = bj * kTile + y, c2 = bi * kTile + tx;
        if (r < N && c < N) X[(size_t)r * N + c] += 0.5 * (a[y][tx] + b[tx][y]);
        if (bi != bj && r2 < N && c2 < N) X[(size_t)r2 * N + c2] += 0.5 * (b[y][tx] + a[tx][y]);
    }
}

__global__ void k_f32_to_f64(size_t n, const float* __restrict__ in, double* __restrict__ out) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        out[i] = (double)in[i];
}

// Block sums of the pair repulsion rep_A exp(-r/rep_b): blocks take atoms A in turn, their
// threads the partners B > A.
__global__ void __launch_bounds__(128)
    k_repulsion(int nat, const double* __restrict__ R, double rep_A, double rep_b,
                double* __restrict__ part) {
    double er = 0;
    for (int A = blockIdx.x; A < nat; A += gridDim.x)
        for (int B = A + 1 + threadIdx.x; B < nat; B += 128) {
            const double dx = R[3 * B] - R[3 * A], dy = R[3 * B + 1] - R[3 * A + 1],
                         dz = R[3 * B + 2] - R[3 * A + 2];
            er += rep_A * exp(-sqrt(dx * dx + dy * dy + dz * dz) / rep_b);
        }
    er = warp_sum(er);
    __shared__ double red[4];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = er;
    __syncthreads();
    if (threadIdx.x == 0) part[blockIdx.x] = (red[0] + red[1]) + (red[2] + red[3]);
}

// out[0] = 1/2 sum_A dq_A (gamma dq)_A (eq:coul), out[1] = sum_{A<B} rep_A exp(-r/rep_b) from its
// nrep block sums, out[2] = nuclear kinetic energy (moving nuclei only)
__global__ void k_small_energies(int nat, const double* __restrict__ dq,
                                 const double* __restrict__ gdq, const double* __restrict__ V,
                                 const double* __restrict__ mass, int nrep,
                                 const double* __restrict__ rep, int kinetic,
                                 double* __restrict__ out) {
    double ec = 0, er = 0, ek = 0;
    for (int k = threadIdx.x; k < nrep; k += blockDim.x) er += rep[k];
    for (int A = threadIdx.x; A < nat; A += blockDim.x) {
        ec += 0.5 * dq[A] * gdq[A];
        if (kinetic)
            ek += 0.5 * mass[A] * 1822.888486 *
                  (V[3 * A] * V[3 * A] + V[3 * A + 1] * V[3 * A + 1] + V[3 * A + 2] * V[3 * A + 2]);
    }
    __shared__ double red[3][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    ec = warp_sum(ec);
    er = warp_sum(er);
    ek = warp_sum(ek);
    if (lane == 0) {
        red[0][w] = ec;
        red[1][w] = er;
        red[2][w] = ek;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double a = 0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) a += red[threadIdx.x][k];
        out[threadIdx.x] = a;
    }
}

// out = max |x| (out must start at 0): non-negative doubles order like their bit patterns
__global__ void k_absmax(size_t n, const double* __restrict__ x, const double* __restrict__ sub,
                         double* __restrict__ out) {
    double m = 0.0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        m = fmax(m, fabs(sub ? x[i] - sub[i] : x[i]));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0)
        atomicMax(reinterpret_cast<unsigned long long*>(out), (unsigned long long)__double_as_longlong(m));
}

}  // namespace

void launch_absmax(size_t n, const double* x, double* out, cudaStream_t st, const double* sub) {
    k_absmax<<<608, 256, 0, st>>>(n, x, sub, out);
}

void launch_ns_start(int N, double* X, double* P, int line, unsigned* norm, cudaStream_t st) {
    launch_pdl(k_ns_start, dim3(1216), dim3(256), 0, st, (size_t)N * N, X, P, line, norm);
}

void launch_ns_update(int N, double* X, const double* Q, const unsigned* gate, float below,
                      cudaStream_t st) {
    const int nt = (N + kTile - 1) / kTile;
    launch_pdl(k_ns_update, dim3(nt, nt), dim3(kTile, 8), 0, st, N, X, Q, gate, below);
}

void launch_f32_to_f64(size_t n, const float* in, double* out, cudaStream_t st) {
    k_f32_to_f64<<<1216, 256, 0, st>>>(n, in, out);
}

void launch_f64_to_f32(size_t n, const double* in, float* out, cudaStream_t st) {
    k_f64_to_f32<<<1216, 256, 0, st>>>(n, in, out);
}

void launch_small_energies(const Ctx& c, double* out, double* scratch, int nscratch, cudaStream_t st) {
    const int nrep = c.mp.rep_A != 0.0 ? std::min(c.nat, nscratch) : 0;
    if (nrep) k_repulsion<<<nrep, 128, 0, st>>>(c.nat, c.d_R, c.mp.rep_A, c.mp.rep_b, scratch);
    k_small_energies<<<1, 256, 0, st>>>(c.nat, c.dq, c.gdq, c.d_Vn, c.d_mass, nrep, scratch,
                                        c.prm.move_nuclei, out);
}

}  // namespace tdb

// ---------------------------------------------------------------------------
// Reduced-precision forms: the density master is rho - rho_ref held as an FP32
// pair (hi + lo, ~48 bits) per element, so the per-step update runs without FP64
// arithmetic (FP64 issues at 1/64 of the FP32 rate on this part).  The FP64
// matrices rho_re / rho_im are a view, materialised for observables, kicks and
// checkpoints.
// ---------------------------------------------------------------------------

namespace tdb {

namespace {

// s + e = a + b exactly (Knuth's two-sum)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// (hi, lo) += inc, renormalised
__device__ __forceinline__ void df_add(float& hi, float& lo, float inc) {
    float s, e;
    two_sum(hi, inc, s, e);
    e += lo;
    hi = s + e;
    lo = e - (hi - s);
}

// FP32-pair ("double-float", ~48 bits) sums and products.  FP64 issues at a small fraction
// of the FP32 rate on this part, so the per-step reductions use these.  The sum is
// commutative bit for bit (the rounded sum and its exact error do not depend on the
// order), so butterfly reductions give the same value on every lane.
__device__ __forceinline__ float2 df2_add(float2 a, float2 b) {
    float s, e;
    two_sum(a.x, b.x, s, e);
    e += a.y + b.y;
    const float h = s + e;
    return make_float2(h, e - (h - s));
}
// a * b with the exact product of the high parts (FMA) and the cross terms
__device__ __forceinline__ float2 df2_mul(float2 a, float2 b) {
    const float p = a.x * b.x;
    const float e = fmaf(a.x, b.x, -p) + (a.x * b.y + a.y * b.x);
    return make_float2(p, e);
}
__device__ __forceinline__ float2 df2_shfl_xor(float2 v, int o) {
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}
__device__ __forceinline__ float2 df2_warp_sum(float2 v) {
    for (int o = 16; o > 0; o >>= 1) v = df2_add(v, df2_shfl_xor(v, o));
    return v;
}
__device__ __forceinline__ float2 ldcg2(const float2* p) { return __ldcg(p); }

// Mulliken product of one element of the deviation master with FP32 S: (re_hi + re_lo) S
// as (hi, lo) with the high product exact
__device__ __forceinline__ float2 mulliken_elem(float rh, float rl, float s) {
    const float p = rh * s;
    return make_float2(p, fmaf(rh, s, -p) + rl * s);
}
// Sum of the 32 element values of a tile row (column order fixed: four interleaved
// partial sums, then combined), shared by the update and the master partials.
__device__ __forceinline__ float2 tile_row_sum(const float2* row) {
    float2 a[4] = {row[0], row[1], row[2], row[3]};
#pragma unroll
    for (int k = 4; k < kTile; k += 4)
#pragma unroll
        for (int j = 0; j < 4; ++j) a[j] = df2_add(a[j], row[k + j]);
    return df2_add(df2_add(a[0], a[1]), df2_add(a[2], a[3]));
}

// Power-of-two scale mapping a bound m into (63.5, 127] (FP32 form of tc::pscale; an
// FP32 quotient that rounds up to a power of two gives a scale one step too large, which
// only moves a little more of a value into its FP16 tails: the heads stay within +-127).
__device__ __forceinline__ float pscale_f(float m) {
    if (!(m > 0.f)) return 1099511627776.0f;   // 2^40
    int e;
    frexpf(127.0f / m, &e);
    e -= 1;
    e = min(40, max(-40, e));
    return ldexpf(1.0f, e);
}

// E(t) of eq:pumpf with the phase formed and reduced modulo 2 pi in FP64 and the sine and
// envelope in FP32 (relative error ~1e-7, far below the reduced forms' product error).
__device__ void field_at_f(const FieldDev& f, double t, float E[3]) {
    if (!f.on) {
        E[0] = E[1] = E[2] = 0.f;
        return;
    }
    const double kTwoPi = 6.283185307179586476925;
    float env = 1.f;
    if (f.envelope == 1) {
        const double x = t - f.t_center;
        const double y = x * x * (4.0 * 0.69314718055994530942 / (f.fwhm * f.fwhm));
        const float yf = (float)y;
        env = expf(-yf) * (1.f - (float)(y - (double)yf));
    } else if (f.envelope == 2) {
        if (t >= 0.0 && t <= f.fwhm) {
            const float sv = sinf((float)(3.14159265358979323846 * t / f.fwhm));
            env = sv * sv;
        } else {
            env = 0.f;
        }
    }
    double ph = f.omega * t + f.phase;
    ph -= kTwoPi * rint(ph * (1.0 / kTwoPi));
    const float a = (float)f.E0 * sinf((float)ph) * env;
    E[0] = a * (float)f.dir[0];
    E[1] = a * (float)f.dir[1];
    E[2] = a * (float)f.dir[2];
}

// Counter increment with acquire-release semantics at GPU scope: after a block barrier it
// publishes what the block wrote (release is cumulative over the barrier) and, for the block
// that completes a count, makes what the others published visible (acquire; the barrier
// that follows extends it to the block).  One such atomic per block replaces per-thread
// fences, which serialise across the GPU.
__device__ __forceinline__ int atom_add_acq_rel(int* p, int v) {
    int old;
    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v)
                 : "memory");
    return old;
}

// Evaluation of a level from its Mulliken row partials, in two kernels of one block per
// kLvAtoms atoms (64 threads, two warps, per atom).
//
// Charges (block blk): dq_A = sum of the partials of atom A's rows (thread t of the atom sums
// partials t, t + 64, ... in order; each warp reduces by a butterfly, and the atom's two
// warps are added), into dq[A]; the block's sums of dq_A R_A and dq_A into bsum[blk]
// (dipole and trace parts).
__device__ void level_dq_block(const LevelArgs& a, int blk) {
    __shared__ float2 half_sum[8];
    __shared__ float2 red[kLvAtoms][4];
    __shared__ float2 r_sh[3 * kLvAtoms];
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const float2 z = make_float2(0.f, 0.f);
    const int A0 = blk * kLvAtoms;
    const int A = A0 + (warp >> 1), t = (warp & 1) * 32 + lane;
    const int len = a.nper * a.nct;
    if (tid < 3 * kLvAtoms) r_sh[tid] = A0 * 3 + tid < 3 * a.nat ? __ldg(a.R2 + 3 * A0 + tid) : z;
    // the potentials kernel may be scheduled now (it loads its constants, then waits)
    pdl_launch_dependents();
    pdl_wait();
    float2 s = z;
    if (A < a.nat) {
        const float2* p = a.partial + (size_t)A * len;
        for (int k0 = t; k0 < len; k0 += 512) {
            float2 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = k0 + 64 * u < len ? ldcg2(p + k0 + 64 * u) : z;
#pragma unroll
            for (int u = 0; u < 8; ++u) s = df2_add(s, v[u]);
        }
    }
    s = df2_warp_sum(s);
    if (lane == 0) half_sum[warp] = s;
    __syncthreads();
    if (tid < kLvAtoms) {
        const int Aa = A0 + tid;
        float2 m[4] = {z, z, z, z};
        if (Aa < a.nat) {
            const float2 d = df2_add(half_sum[2 * tid], half_sum[2 * tid + 1]);
            a.dq[Aa] = d;
#pragma unroll
            for (int k = 0; k < 3; ++k) m[k] = df2_mul(d, r_sh[3 * tid + k]);
            m[3] = d;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) red[tid][k] = m[k];
    }
    __syncthreads();
    if (tid < 4) {
        float2 x = red[0][tid];
#pragma unroll
        for (int i = 1; i < kLvAtoms; ++i) x = df2_add(x, red[i][tid]);
        a.bsum[4 * blk + tid] = x;
    }
}

// Potentials and the level's scalars.  Blocks 0 .. level_blocks(nat) - 1 (kLvAtoms atoms
// each): dv_A = sum_B gamma_AB dq_B (eq:hscc; thread t of atom A takes B = t, t + 64, ...
// in order, each warp reduces by a butterfly, the atom's two warps are added) + R_A . E(t)
// + the SCC residual of rho_ref, written per orbital (dv_f), and the maximum |dv| over the
// blocks.  Block level_blocks(nat) (the totals block): Tr(rho S) and the renormalisation
// factor of level `slot` from the charge blocks' sums, the dipole mu = mu_ref - sum_A dq_A
// R_A into sc->mu and the history slot of step n_lvl, the field record.  The block that
// arrives last sets the FP16X6 scales of the next products and, with step_end, the step
// counter (to n_lvl) and the FP16X6 maxima (the new level is in `slot`); it resets the
// counters.  trace_only (one block): only Tr(rho S) and f - 1.
__device__ void level_final_block(const LevelArgs& a, int slot, long long n_lvl, bool trace_only,
                                  bool step_end, int blk, int nblk) {
    __shared__ float2 half_sum[8];
    __shared__ float2 tot[4];
    __shared__ float E_sh[3];
    __shared__ float rc_sh[kLvAtoms][4];
    __shared__ float mx_sh;
    __shared__ int last;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    DevScalars* sc = a.sc;
    const float2 z = make_float2(0.f, 0.f);
    const int nab = level_blocks(a.nat);
    // constants first (gamma of this thread's first products, positions, residuals); the
    // charges and scalars of the previous kernels after pdl_wait
    const int A0 = blk * kLvAtoms;
    const int A = A0 + (warp >> 1), t = (warp & 1) * 32 + lane;
    const bool atoms = !trace_only && blk < nab;
    float2 gv[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int b = t + 64 * u;
        gv[u] = (atoms && a.scc && A < a.nat && b < a.nat) ? __ldg(a.gam2 + (size_t)A * a.nat + b) : z;
    }
    if (atoms && tid < kLvAtoms) {
        const int Aa = A0 + tid;
        const bool ok = Aa < a.nat;
        rc_sh[tid][0] = ok ? __ldg(&a.R2[3 * Aa].x) : 0.f;
        rc_sh[tid][1] = ok ? __ldg(&a.R2[3 * Aa + 1].x) : 0.f;
        rc_sh[tid][2] = ok ? __ldg(&a.R2[3 * Aa + 2].x) : 0.f;
        rc_sh[tid][3] = ok ? __ldg(a.c_res + Aa) : 0.f;
    }
    pdl_wait();
    if (tid == 0) {
        float E[3] = {0.f, 0.f, 0.f};
        if (!trace_only && sc->field.on) {
            const double t = sc->t_base + (double)(n_lvl - sc->n_base) * sc->dt;
            field_at_f(sc->field, t, E);
        }
        E_sh[0] = E[0];
        E_sh[1] = E[1];
        E_sh[2] = E[2];
        mx_sh = 0.f;
    }
    if (trace_only || blk == nab) {
        // the totals block: sums of the charge blocks' dipole and trace parts (warps 0-3)
        if (warp < 4) {
            float2 s = z;
            for (int r = lane; r < nab; r += 32) s = df2_add(s, ldcg2(a.bsum + 4 * r + warp));
            s = df2_warp_sum(s);
            if (lane == 0) tot[warp] = s;
        }
        __syncthreads();
        if (tid == 0) {
            // Tr(rho S) = N_e - c0 + sum_A dq_A;  f - 1 = (N_e - Tr) / Tr ~ (c0 - sum dq) / N_e
            const float2 d = tot[3];
            const float eps = (((float)sc->c0_trace - d.x) - d.y) * a.inv_ne;
            sc->eps_lvl[slot] = eps;
            sc->trace_lvl[slot] = (sc->n_e - sc->c0_trace) + ((double)d.x + (double)d.y);
        }
        if (trace_only) return;
        if (warp == 1) {
            // dipole (lanes 0-2, one component each) into sc and the history slot of step n_lvl
            const int k = lane < 3 ? lane : 0;
            const double mu = sc->mu_ref[k] - ((double)tot[k].x + (double)tot[k].y);
            const double ek = mu * (double)E_sh[k];
            const double e_ext = -(ek + __shfl_down_sync(0xffffffffu, ek, 1) +
                                   __shfl_down_sync(0xffffffffu, ek, 2));
            if (lane < 3) {
                long long h = n_lvl % sc->hist_cap;
                if (h < 0) h += sc->hist_cap;
                sc->mu[k] = mu;
                sc->E[k] = (double)E_sh[k];
                a.hist[3 * h + k] = mu;
            }
            if (lane == 0) sc->e_ext = e_ext;
        }
    } else {
        float2 acc = z;
        if (a.scc && A < a.nat) {
            const float2* g = a.gam2 + (size_t)A * a.nat;
            for (int b0 = t; b0 < a.nat; b0 += 512) {
                float2 qv[8];
                if (b0 != t)
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int b = b0 + 64 * u;
                        gv[u] = b < a.nat ? __ldg(g + b) : z;
                    }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int b = b0 + 64 * u;
                    qv[u] = b < a.nat ? ldcg2(a.dq + b) : z;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) acc = df2_add(acc, df2_mul(gv[u], qv[u]));
            }
        }
        acc = df2_warp_sum(acc);
        if (lane == 0) half_sum[warp] = acc;
        __syncthreads();
        if (warp == 0) {
            float mx = 0.f;
            const int Aa = A0 + lane;
            if (lane < kLvAtoms && Aa < a.nat) {
                const float2 s = df2_add(half_sum[2 * lane], half_sum[2 * lane + 1]);
                const float ext = fmaf(rc_sh[lane][0], E_sh[0],
                                       fmaf(rc_sh[lane][1], E_sh[1], rc_sh[lane][2] * E_sh[2]));
                const float dv = s.x + (s.y + (ext + rc_sh[lane][3]));
                for (int k = 0; k < a.nper; ++k) a.dv_f[Aa * a.nper + k] = dv;
                mx = fabsf(dv);
            }
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            if (lane == 0) mx_sh = mx;
        }
    }
    // arrival of every block (atom blocks carry their maximum |dv|)
    __syncthreads();
    int* max_bits = a.count + 1;     // max |dv| of this evaluation (float bits, >= 0)
    if (tid == 0) {
        if (blk < nab) atomicMax(max_bits, __float_as_int(mx_sh));
        last = atom_add_acq_rel(a.count, 1) == nblk - 1;
    }
    __syncthreads();
    if (!last || tid != 0) return;
    const float m = __int_as_float(__ldcg(max_bits));
    tc::DynScales* dy = a.dyn;
    if (dy) {
        dy->max_dv = (double)m;
        if (a.has_scales) {
            dy->s_dh = pscale_f(m);
            dy->s_dm = pscale_f(m * (float)dy->sinv_norm);
        }
        for (int k = 0; k < tc::kMaxParts; ++k) dy->max_x[k] = 0.0;
        if (step_end) {
            // the maximum the update's blocks accumulated (atomics, read through L2)
            dy->max_drho[slot] = __ldcg(&dy->max_drho[2]);
            dy->max_drho[2] = 0.0;
        }
    }
    if (step_end) sc->step = n_lvl;
    // the counters, after this thread's read of the maximum
    a.count[0] = 0;
    a.count[1] = 0;
}

// Update of the FP32-pair master (eq:leapfrog, eq:eomrho, frozen nuclei): the same
// tile-pair scheme and operands as k_update, with the increment factor * rhodot formed
// as fh * d + fl * d (factor = fh + fl) so the step length carries no FP32 rounding.
// Every kRenormEvery steps the base level is first renormalised to Tr(rho S) = N_e:
// rho_base <- f rho_base with f = 1 + eps from its trace (Sec. 2.3: the exact leapfrog
// conserves the electron number; the reduced products do not, by ~1e-14 of N_e per step),
// i.e. the deviation gains eps (rho_ref + deviation).  Mulliken row partials of the new
// deviation in FP32-pair arithmetic, from which two small kernels evaluate the new level
// (level_dq_block, level_final_block).
// Steps between renormalisations of a leapfrog level (the reduced forms drift by ~1e-14 of
// N_e per step, so Tr(rho S) stays within ~1e-12 of N_e in between).
constexpr int kRenormEvery = 8;

__device__ __forceinline__ void update_df_block(const UpdateDfArgs& A, int b) {
    const int N = A.N, nct = A.nct;
    const MasterPtrs& base = A.base;
    const MasterPtrs& out = A.out;
    const float fh = A.fh, fl = A.fl;
    const double factor = A.factor;
    const float* __restrict__ Sf = A.Sf;
    const float* __restrict__ rgs = A.rgs;
    DevScalars* __restrict__ sc = A.sc;
    const UpdateOperands& ops = A.ops;
    const LevelArgs& lv = A.lv;
    // one block per tile pair bi <= bj: block b = bj (bj + 1) / 2 + bi
    int bj = (int)((sqrtf(8.0f * (float)b + 1.0f) - 1.0f) * 0.5f);
    while (bj * (bj + 1) / 2 > b) --bj;
    while ((bj + 1) * (bj + 2) / 2 <= b) ++bj;
    const int bi = b - bj * (bj + 1) / 2;
    // a thread takes four consecutive columns x .. x + 3 of row y of a tile: 16-byte accesses where
    // the rows are aligned (N a multiple of 4), a quarter of the memory instructions
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    const int y = tid >> 3, x = 4 * (tid & 7);
    const bool vec = (N & 3) == 0;
    auto load4 = [&](const float* p, int r, int c, float (&v)[4]) {
        v[0] = v[1] = v[2] = v[3] = 0.f;
        if (r >= N || c >= N) return;
        const float* q = p + (size_t)r * N + c;
        if (vec) {
            const float4 f = *reinterpret_cast<const float4*>(q);
            v[0] = f.x, v[1] = f.y, v[2] = f.z, v[3] = f.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (c + j < N) v[j] = q[j];
        }
    };
    auto store4 = [&](float* p, int r, int c, const float (&v)[4]) {
        float* q = p + (size_t)r * N + c;
        if (vec) {
            *reinterpret_cast<float4*>(q) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (c + j < N) q[j] = v[j];
        }
    };
    // base level and S of a half: constants of this step (their writer finished two kernels ago)
    float rh[4], rl[4], ih[4], il[4], sv[4];
    auto load_base = [&](int half) {
        const int r = (half ? bj : bi) * kTile + y, c = (half ? bi : bj) * kTile + x;
        load4(base.re_hi, r, c, rh);
        load4(base.re_lo, r, c, rl);
        load4(base.im_hi, r, c, ih);
        load4(base.im_lo, r, c, il);
        load4(Sf, r, c, sv);
    };
    // before the wait for X: the first half's operands into registers, the second's lines (rows of
    // 32 floats = one 128-byte line) into L2
    load_base(0);
    if (bi != bj) {
        const int arr = tid >> 5, row = tid & 31;
        if (arr < 5) {
            const float* p = arr == 0 ? base.re_hi : arr == 1 ? base.re_lo : arr == 2 ? base.im_hi
                             : arr == 3 ? base.im_lo : Sf;
            const int r = bj * kTile + row, c = bi * kTile;
            if (r < N && c < N) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + (size_t)r * N + c));
        }
    }
    // X, the scalars and the outputs belong to the previous kernels from here on
    pdl_wait();
    __shared__ float xr_ij[kTile][kTile + 1], xi_ij[kTile][kTile + 1];
    __shared__ float xr_ji[kTile][kTile + 1], xi_ji[kTile][kTile + 1];
    __shared__ float2 pv_s[2][kTile][kTile + 1];   // Mulliken products of both halves
    // X = sum of its partial products, in a fixed order: Re X = ((t0 + t1) + t2) + t3, Im X = t0 + t1;
    // the first round's loads of both tiles in flight together, a second round for two K slices
    {
        float t[2][3][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = (h ? bj : bi) * kTile + y, c = (h ? bi : bj) * kTile + x;
            load4(ops.xre[0], r, c, t[h][0]);
            if (ops.nre > 1) load4(ops.xre[1], r, c, t[h][1]);
            load4(ops.xim[0], r, c, t[h][2]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (ops.nre > 1) t[h][0][j] += t[h][1][j];
        if (ops.nre > 2) {
            float u[2][3][4];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = (h ? bj : bi) * kTile + y, c = (h ? bi : bj) * kTile + x;
                load4(ops.xre[2], r, c, u[h][0]);
                load4(ops.xre[3], r, c, u[h][1]);
                load4(ops.xim[1], r, c, u[h][2]);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    t[h][0][j] = (t[h][0][j] + u[h][0][j]) + u[h][1][j];
                    t[h][2][j] += u[h][2][j];
                }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                (h ? xr_ji : xr_ij)[y][x + j] = t[h][0][j];
                (h ? xi_ji : xi_ij)[y][x + j] = t[h][2][j];
            }
    }
    __shared__ float s_bound;
    __shared__ float eps_sh;
    if (tid == 0) {
        // both leapfrog chains are renormalised once every kRenormEvery steps
        const long long n = sc->step;
        eps_sh = (n % kRenormEvery) < 2 ? sc->eps_lvl[ops.base_slot] : 0.f;
        if (ops.dyn) {
            // |X| <= the sum of the maxima of its partial products
            const tc::DynScales* d = ops.dyn;
            float mre = 0.f, mim = 0.f;
            for (int q = 0; q < ops.nre; ++q) mre += (float)d->max_x[q];
            for (int q = 0; q < ops.nim; ++q) mim += (float)d->max_x[ops.nre + q];
            s_bound = pscale_f((float)d->max_drho[ops.base_slot] * (1.f + fabsf(eps_sh)) +
                               8.f * fabsf(eps_sh) +
                               fabsf((float)factor) * 2.0f * fmaxf(mre, mim));
        }
    }
    __syncthreads();
    const float op_scale = ops.dyn ? s_bound : ops.scale;
    const float eps = eps_sh;
    float dmax = 0.f;
    for (int half = 0; half < (bi == bj ? 1 : 2); ++half) {
        const int ti = half ? bj : bi, tj = half ? bi : bj;
        const int r = ti * kTile + y, c0 = tj * kTile + x;
        if (half) load_base(1);
        float gv[4] = {0.f, 0.f, 0.f, 0.f};
        if (eps != 0.f) load4(rgs, r, c0, gv);
        const bool in = r < N && c0 < N;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float x_ij_re = (half ? xr_ji : xr_ij)[y][x + j], x_ij_im = (half ? xi_ji : xi_ij)[y][x + j];
            const float x_ji_re = (half ? xr_ij : xr_ji)[x + j][y], x_ji_im = (half ? xi_ij : xi_ji)[x + j][y];
            // rhodot = -i (X - X^dagger); the (j,i) element repeats these operations on
            // the swapped operands, so the master stays exactly Hermitian
            const float dre = x_ij_im + x_ji_im;
            const float dim = -(x_ij_re - x_ji_re);
            const float ire = fmaf(fh, dre, fl * dre);
            const float iim = fmaf(fh, dim, fl * dim);
            if (eps != 0.f) {
                // renormalised base: f (rho_ref + dev) - rho_ref = dev + eps (rho_ref + dev)
                df_add(rh[j], rl[j], eps * (gv[j] + rh[j]));
                df_add(ih[j], il[j], eps * ih[j]);
            }
            df_add(rh[j], rl[j], ire);
            df_add(ih[j], il[j], iim);
            const bool here = in && c0 + j < N;
            pv_s[half][y][x + j] = here ? mulliken_elem(rh[j], rl[j], sv[j]) : make_float2(0.f, 0.f);
            if (ops.dyn && here) dmax = fmaxf(dmax, fmaxf(fabsf(rh[j]), fabsf(ih[j])));
        }
        if (!in) continue;
        store4(out.re_hi, r, c0, rh);
        store4(out.re_lo, r, c0, rl);
        store4(out.im_hi, r, c0, ih);
        store4(out.im_lo, r, c0, il);
        if (ops.re[0]) {
            // operands of the tensor-core products are K-major: Re rho is symmetric, the transpose
            // of Im rho is -Im rho; four pieces per 8-byte store (rows are padded to 64 columns;
            // a ragged row writes zeros past N)
            const size_t jr = (size_t)r * ops.ld_re + c0, ji = (size_t)r * ops.ld_im + c0;
            uint32_t a[3], b[3];
            auto put = [&](uint16_t* const* dst, size_t o, const float (&v)[4], float f) {
                if (ops.re[2]) {
                    tc::split_pair<tc::kHead3>(v[0] * f, v[1] * f, 0, a);
                    tc::split_pair<tc::kHead3>(v[2] * f, v[3] * f, 0, b);
                } else {
                    tc::split_pair<tc::kHiLo>(v[0] * f, v[1] * f, ops.bf16, a);
                    tc::split_pair<tc::kHiLo>(v[2] * f, v[3] * f, ops.bf16, b);
                }
#pragma unroll
                for (int t = 0; t < 3; ++t)
                    if (t < 2 || ops.re[2]) *reinterpret_cast<uint2*>(dst[t] + o) = make_uint2(a[t], b[t]);
            };
            put(ops.re, jr, rh, op_scale);
            put(ops.im, ji, ih, -op_scale);
        }
    }
    __syncthreads();
    // row sums, one warp per half
    const int tx = tid & 31, ty = tid >> 5;
    if (ty < (bi == bj ? 1 : 2)) {
        const int r = (ty ? bj : bi) * kTile + tx;
        const float2 sum = tile_row_sum(pv_s[ty][tx]);
        if (r < N) const_cast<float2*>(lv.partial)[(size_t)r * nct + (ty ? bi : bj)] = sum;
    }
    if (ops.dyn) {
        // one atomic per block (the warps' maxima through shared memory)
        __shared__ float wmax[8];
        for (int o = 16; o > 0; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
        if (tx == 0) wmax[ty] = dmax;
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < 8; ++w) dmax = fmaxf(dmax, wmax[w]);
            atomicMax(reinterpret_cast<unsigned long long*>(&ops.dyn->max_drho[2]),
                      (unsigned long long)__double_as_longlong((double)dmax));
            if (bi == 0 && bj == 0) ops.dyn->s_rho = op_scale;
        }
    }
}

__global__ void __launch_bounds__(256, 4) k_update_df(UpdateDfArgs a) { update_df_block(a, blockIdx.x); }

__global__ void __launch_bounds__(256, 4)
    k_update_df_grouped(const UpdateDfArgs* __restrict__ args, const int2* __restrict__ work) {
    const int2 w = work[blockIdx.x];
    update_df_block(args[w.x], w.y);
}

// The charges of a level (after an update, or of the current level outside a step).
__global__ void __launch_bounds__(256) k_level_dq(LevelArgs lv) { level_dq_block(lv, blockIdx.x); }

__global__ void __launch_bounds__(256)
    k_level_dq_grouped(const LevelFinalArgs* __restrict__ args, const int2* __restrict__ work) {
    const int2 w = work[blockIdx.x];
    level_dq_block(args[w.x].lv, w.y);
}

// The potentials and scalars of a level after k_level_dq: after an update (step_end, the new
// level n + 1 in slot) or of the current level.
__global__ void __launch_bounds__(256) k_level_final(LevelArgs lv, int slot, int trace_only, int step_end) {
    const long long n_lvl = lv.sc->step + (step_end ? 1 : 0);
    level_final_block(lv, slot, n_lvl, trace_only != 0, step_end != 0, blockIdx.x, gridDim.x);
}

__global__ void __launch_bounds__(256)
    k_level_final_grouped(const LevelFinalArgs* __restrict__ args, const int2* __restrict__ work) {
    const int2 w = work[blockIdx.x];
    const LevelFinalArgs& f = args[w.x];
    const long long n_lvl = f.lv.sc->step + 1;
    level_final_block(f.lv, f.slot, n_lvl, false, true, w.y, level_blocks(f.lv.nat) + 1);
}

// FP64 populations from the (hi, lo) row partials of the deviation: one warp per atom
__global__ void k_charges_df(int nat, int nper, int nct, const float2* __restrict__ partial,
                             const double* __restrict__ qbase, const double* __restrict__ q0,
                             double* __restrict__ q, double* __restrict__ dq) {
    const int lane = threadIdx.x & 31;
    const int A = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (A >= nat) return;
    const float2* p = partial + (size_t)A * nper * nct;
    double s = 0.0;
    for (int i = lane; i < nper * nct; i += 32) s += (double)p[i].x + (double)p[i].y;
    s = warp_sum(s);
    if (lane == 0) {
        s += qbase[A];
        q[A] = s;
        dq[A] = s - q0[A];
    }
}

// master (hi, lo) of rho - rho_ref from the FP64 view
__global__ void k_view_to_master(size_t n, const double* __restrict__ rre,
                                 const double* __restrict__ rim, const double* __restrict__ ref,
                                 MasterPtrs m) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
        const double d = rre[i] - ref[i];
        const float h = (float)d;
        m.re_hi[i] = h;
        m.re_lo[i] = (float)(d - (double)h);
        const double e = rim[i];
        const float g = (float)e;
        m.im_hi[i] = g;
        m.im_lo[i] = (float)(e - (double)g);
    }
}

// FP64 view rho = rho_ref + hi + lo from the master
__global__ void k_master_to_view(size_t n, MasterPtrs m, const double* __restrict__ ref,
                                 double* __restrict__ rre, double* __restrict__ rim) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
        rre[i] = ref[i] + ((double)m.re_hi[i] + (double)m.re_lo[i]);
        rim[i] = (double)m.im_hi[i] + (double)m.im_lo[i];
    }
}

// Mulliken row partials of the deviation held by the master, with the arithmetic of
// k_update_df (exact high products, FP32-pair sums in the same column order)
__global__ void k_master_partials(int N, int nct, MasterPtrs m, const float* __restrict__ Sf,
                                  float2* __restrict__ partial) {
    __shared__ float2 pv_s[kTile][kTile + 1];
    const int ct = blockIdx.x;
    const int col = ct * kTile + threadIdx.x;
    for (int y = threadIdx.y; y < kTile; y += blockDim.y) {
        const int row = blockIdx.y * kTile + y;
        float2 v = make_float2(0.f, 0.f);
        if (row < N && col < N) {
            const size_t i = (size_t)row * N + col;
            v = mulliken_elem(m.re_hi[i], m.re_lo[i], Sf[i]);
        }
        pv_s[y][threadIdx.x] = v;
    }
    __syncthreads();
    if (threadIdx.y == 0) {
        const int row = blockIdx.y * kTile + threadIdx.x;
        const float2 sum = tile_row_sum(pv_s[threadIdx.x]);
        if (row < N) partial[(size_t)row * nct + ct] = sum;
    }
}

// max(|re_hi|, |im_hi|) into out (out must start at 0)
__global__ void k_master_absmax(size_t n, MasterPtrs m, double* __restrict__ out) {
    float mx = 0.f;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        mx = fmaxf(mx, fmaxf(fabsf(m.re_hi[i]), fabsf(m.im_hi[i])));
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0)
        atomicMax(reinterpret_cast<unsigned long long*>(out),
                  (unsigned long long)__double_as_longlong((double)mx));
}

// operand pieces of the master deviation (the update's arithmetic); the scale is
// pscale(*mx_exact) (FP16X6, exact maximum), else *dev_scale (FP16X6, restored), else
// the constant ops.scale
__global__ void k_master_pieces(int N, MasterPtrs m, UpdateOperands ops, const double* mx_exact,
                                const float* dev_scale) {
    __shared__ float s_sh;
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        s_sh = mx_exact ? tc::pscale(*mx_exact) : dev_scale ? *dev_scale : ops.scale;
        if (mx_exact && ops.dyn && blockIdx.x == 0 && blockIdx.y == 0) ops.dyn->s_rho = s_sh;
    }
    __syncthreads();
    const float sc = s_sh;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y * blockDim.y + threadIdx.y;
    if (r >= N || c >= N) return;
    const size_t i = (size_t)r * N + c;
    const float rh = m.re_hi[i], ih = m.im_hi[i];
    const size_t jr = (size_t)r * ops.ld_re + c;
    const size_t ji = (size_t)r * ops.ld_im + c;
    if (ops.re[2]) {
        uint16_t q[3];
        split_head3(rh * sc, q);
        ops.re[0][jr] = q[0];
        ops.re[1][jr] = q[1];
        ops.re[2][jr] = q[2];
        split_head3(-ih * sc, q);
        ops.im[0][ji] = q[0];
        ops.im[1][ji] = q[1];
        ops.im[2][ji] = q[2];
    } else {
        const float xa = rh * sc;
        const uint16_t h1 = to16(xa, ops.bf16);
        ops.re[0][jr] = h1;
        ops.re[1][jr] = to16(xa - from16(h1, ops.bf16), ops.bf16);
        const float yb = -ih * sc;
        const uint16_t h2 = to16(yb, ops.bf16);
        ops.im[0][ji] = h2;
        ops.im[1][ji] = to16(yb - from16(h2, ops.bf16), ops.bf16);
    }
}

}  // namespace

UpdateDfArgs update_df_args(const Ctx& c, const MasterPtrs& base, const MasterPtrs& out,
                            double factor, DevScalars* sc, const UpdateOperands& ops,
                            const LevelArgs& lv) {
    UpdateDfArgs a{};
    a.N = c.N;
    a.nct = c.nct;
    a.out_slot = out.re_hi == c.ms[0].re_hi ? 0 : 1;
    a.base = base;
    a.out = out;
    a.fh = (float)factor;
    a.fl = (float)(factor - (double)a.fh);
    a.factor = factor;
    a.Sf = c.S_f;
    a.rgs = c.rref_f;
    a.sc = sc;
    a.ops = ops;
    a.lv = lv;
    return a;
}

void launch_update_df(const Ctx& c, const MasterPtrs& base, const MasterPtrs& out, double factor,
                      DevScalars* sc, const UpdateOperands& ops, const LevelArgs& lv,
                      cudaStream_t st) {
    launch_pdl(k_update_df, dim3(c.nct * (c.nct + 1) / 2), dim3(kTile, 8), 0, st,
               update_df_args(c, base, out, factor, sc, ops, lv));
}

void launch_update_df_grouped(const UpdateDfArgs* args, const int2* work, int nwork,
                              cudaStream_t st) {
    launch_pdl(k_update_df_grouped, dim3(nwork), dim3(kTile, 8), 0, st, args, work);
}

void launch_level(const Ctx& c, const LevelArgs& lv, int slot, int trace_only, cudaStream_t st) {
    k_level_dq<<<level_blocks(c.nat), dim3(kTile, 8), 0, st>>>(lv);
    k_level_final<<<trace_only ? 1 : level_blocks(c.nat) + 1, dim3(kTile, 8), 0, st>>>(
        lv, slot, trace_only, 0);
}

void launch_level_dq(const Ctx& c, const LevelArgs& lv, cudaStream_t st) {
    launch_pdl(k_level_dq, dim3(level_blocks(c.nat)), dim3(kTile, 8), 0, st, lv);
}

void launch_level_dq_grouped(const LevelFinalArgs* args, const int2* work, int nwork,
                             cudaStream_t st) {
    launch_pdl(k_level_dq_grouped, dim3(nwork), dim3(kTile, 8), 0, st, args, work);
}

void launch_level_final(const Ctx& c, const LevelArgs& lv, int slot, cudaStream_t st) {
    launch_pdl(k_level_final, dim3(level_blocks(c.nat) + 1), dim3(kTile, 8), 0, st, lv, slot, 0, 1);
}

void launch_level_final_grouped(const LevelFinalArgs* args, const int2* work, int nwork,
                                cudaStream_t st) {
    launch_pdl(k_level_final_grouped, dim3(nwork), dim3(kTile, 8), 0, st, args, work);
}

void launch_charges_df(const Ctx& c, const float2* partial, double* q, double* dq, cudaStream_t st) {
    k_charges_df<<<(c.nat + 7) / 8, 256, 0, st>>>(c.nat, c.nper, c.nct, partial, c.qbase, c.d_q0, q,
                                                  dq);
}

void launch_view_to_master(const Ctx& c, const double* rre, const double* rim, const MasterPtrs& m,
                           cudaStream_t st) {
    k_view_to_master<<<1216, 256, 0, st>>>((size_t)c.N * c.N, rre, rim, c.rho_ref, m);
}

void launch_master_to_view(const Ctx& c, const MasterPtrs& m, double* rre, double* rim,
                           cudaStream_t st) {
    k_master_to_view<<<1216, 256, 0, st>>>((size_t)c.N * c.N, m, c.rho_ref, rre, rim);
}

void launch_master_partials(const Ctx& c, const MasterPtrs& m, float2* partial, cudaStream_t st) {
    dim3 b(kTile, 8);
    k_master_partials<<<dim3(c.nct, c.nct), b, 0, st>>>(c.N, c.nct, m, c.S_f, partial);
}

void launch_master_absmax(const Ctx& c, const MasterPtrs& m, double* out, cudaStream_t st) {
    k_master_absmax<<<608, 256, 0, st>>>((size_t)c.N * c.N, m, out);
}

void launch_master_pieces(const Ctx& c, const MasterPtrs& m, const UpdateOperands& ops,
                          const double* mx_exact, const float* dev_scale, cudaStream_t st) {
    dim3 b(32, 8);
    k_master_pieces<<<grid2(c.N, c.N, b), b, 0, st>>>(c.N, m, ops, mx_exact, dev_scale);
}

}  // namespace tdb
