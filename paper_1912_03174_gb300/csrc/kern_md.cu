// Moving nuclei (Ehrenfest dynamics): forces (eq:forces), the non-adiabatic
// coupling matrix D (eq:nac, eq:onsite), the work rate P and velocity Verlet
// (Sec. 2.3).  FP64 throughout.  Gradients of the two-centre blocks are
// recomputed from the geometry where they are used and never stored.
#include <cmath>

#include "pdl.cuh"
#include "tdb_internal.h"

namespace tdb {

namespace {

__device__ __forceinline__ double warp_sum_d(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// d gamma_AB / dR for exponents ta, tb (tau = 16 U / 5): derivative of
// 1/R - zeta(R), with the equal-exponent form below a 3e-4 relative gap.
__device__ double gamma_dR(double ta, double tb, double R) {
    const double tmax = ta > tb ? ta : tb;
    double dz;
    if (fabs(ta - tb) < 3e-4 * tmax) {
        const double t = 0.5 * (ta + tb);
        const double e = exp(-t * R);
        const double poly = 1.0 / R + 11.0 * t / 16.0 + 3.0 * t * t * R / 16.0 + t * t * t * R * R / 48.0;
        const double dpoly = -1.0 / (R * R) + 3.0 * t * t / 16.0 + t * t * t * R / 24.0;
        dz = e * (dpoly - t * poly);
    } else {
        dz = 0.0;
        for (int s = 0; s < 2; ++s) {
            const double a = s ? tb : ta, b = s ? ta : tb;
            const double a2 = a * a, b2 = b * b, d = a2 - b2;
            const double c1 = b2 * b2 * a / (2.0 * d * d);
            const double c2 = (b2 * b2 * b2 - 3.0 * a2 * b2 * b2) / (d * d * d);
            dz += exp(-a * R) * (-a * (c1 - c2 / R) + c2 / (R * R));
        }
    }
    return -1.0 / (R * R) - dz;
}

// Gradient with respect to d = R_B - R_A of the weighted block sum sum_ij w_ij T_ij(d) of a
// two-centre s/p block (T_00 = K0, T_0a = c_a K1, T_a0 = -c_a K1, T_ab = c_a c_b (K2 - K3)
// + delta_ab K3, c = d / r), contracted before differentiating: with p_a = w_0a - w_a0 and
// M_ab = w_ab the sum is w_00 K0 + (p.c) K1 + (c.Mc) (K2 - K3) + tr(M) K3, and with
// dc_a/dd_q = (delta_aq - c_a c_q) / r and dr/dd = c its gradient is
//   c [w_00 K0' + (p.c) K1' + (c.Mc)(K2' - K3') + tr(M) K3' - ((p.c) K1 + 2 (c.Mc)(K2 - K3)) / r]
//   + [p K1 + (M + M^T) c (K2 - K3)] / r.
// nper = 1 (s only): w_00 K0' c.
__device__ __forceinline__ void block_sum_grad(int nper, const double (&w)[16], const double c[3],
                                               double inv_r, const double K[4],
                                               const double dK[4], double g[3]) {
    if (nper == 1) {
        for (int q = 0; q < 3; ++q) g[q] = w[0] * dK[0] * c[q];
        return;
    }
    const double p[3] = {w[1] - w[4], w[2] - w[8], w[3] - w[12]};
    double Mc[3], MTc[3];
    for (int a = 0; a < 3; ++a) {
        Mc[a] = w[4 * (a + 1) + 1] * c[0] + w[4 * (a + 1) + 2] * c[1] + w[4 * (a + 1) + 3] * c[2];
        MTc[a] = w[4 + a + 1] * c[0] + w[8 + a + 1] * c[1] + w[12 + a + 1] * c[2];
    }
    const double pc = p[0] * c[0] + p[1] * c[1] + p[2] * c[2];
    const double cMc = c[0] * Mc[0] + c[1] * Mc[1] + c[2] * Mc[2];
    const double tr = w[5] + w[10] + w[15];
    const double d23 = K[2] - K[3];
    const double par = w[0] * dK[0] + pc * dK[1] + cMc * (dK[2] - dK[3]) + tr * dK[3] -
                       (pc * K[1] + 2.0 * cMc * d23) * inv_r;
    for (int q = 0; q < 3; ++q)
        g[q] = par * c[q] + (p[q] * K[1] + (Mc[q] + MTc[q]) * d23) * inv_r;
}

// Pair terms of the forces (eq:forces, energy-weighted form of the S-derivative terms, velocity
// terms dropped), one thread per pair A < B (blockIdx.y = A): the force on A,
//   sum over the (A, B) block of 2 Re rho_ij dH_ij/dR_B + (Re rho_ij (v_A + v_B) - 2 Re W_ij)
//   dS_ij/dR_B, plus -dq_A dq_B dgamma/dR_A + rep_A/rep_b e^{-r/rep_b} u;
// W = 1/2 (X + X^dagger), X = S^-1 H rho, is formed from the blocks (A, B) and (B, A) of Re X.
// The force on B is its negative: pf[A][B] = f, pf[B][A] = -f, so that an atom's row sums to its
// force.  Bound by FP64 issue (two lanes a clock per SM): the block sums are differentiated in
// contracted form (block_sum_grad) and each pair is evaluated once.
constexpr int kPairThreads = 64;

__global__ void __launch_bounds__(kPairThreads)
    k_pair_forces(int nat, int nper, int scc, const double* R,
                  const double* rre, const double* xre,
                  const double* v_atom, const double* dq,
                  const double* U, ModelParams mp, double* pf) {
    const int A = blockIdx.y, B = blockIdx.x * kPairThreads + threadIdx.x;
    pdl_wait();
    if (B < A || B >= nat) return;
    const size_t ab = 3 * ((size_t)A * nat + B), ba = 3 * ((size_t)B * nat + A);
    if (A == B) {
        for (int q = 0; q < 3; ++q) pf[ab + q] = 0.0;
        return;
    }
    const int N = nat * nper;
    const double d[3] = {R[3 * B] - R[3 * A], R[3 * B + 1] - R[3 * A + 1], R[3 * B + 2] - R[3 * A + 2]};
    const double vv = v_atom[A] + v_atom[B];
    double wh[16], ws[16];
    if (nper == 4) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const double2* pr = reinterpret_cast<const double2*>(rre + (size_t)(4 * A + i) * N + 4 * B);
            const double2* px = reinterpret_cast<const double2*>(xre + (size_t)(4 * A + i) * N + 4 * B);
            const double2 p0 = pr[0], p1 = pr[1], x0 = px[0], x1 = px[1];
            wh[4 * i] = p0.x, wh[4 * i + 1] = p0.y, wh[4 * i + 2] = p1.x, wh[4 * i + 3] = p1.y;
            ws[4 * i] = x0.x, ws[4 * i + 1] = x0.y, ws[4 * i + 2] = x1.x, ws[4 * i + 3] = x1.y;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const double2* px = reinterpret_cast<const double2*>(xre + (size_t)(4 * B + j) * N + 4 * A);
            const double2 x0 = px[0], x1 = px[1];
            const double x[4] = {x0.x, x0.y, x1.x, x1.y};
#pragma unroll
            for (int i = 0; i < 4; ++i) ws[4 * i + j] = fma(wh[4 * i + j], vv, -(ws[4 * i + j] + x[i]));
        }
    } else {
        for (int k = 0; k < 16; ++k) wh[k] = ws[k] = 0.0;
        wh[0] = rre[(size_t)A * N + B];
        ws[0] = wh[0] * vv - (xre[(size_t)A * N + B] + xre[(size_t)B * N + A]);
    }
    const double r = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    const double inv_r = 1.0 / r;
    const double c[3] = {d[0] * inv_r, d[1] * inv_r, d[2] * inv_r};
    // the hopping block carries 2 Re rho
    const double eh = 2.0 * mp.t0 * exp(-r / mp.lam_H), es = -mp.s0 * exp(-r / mp.lam_S);
    const double ih = -1.0 / mp.lam_H, is = -1.0 / mp.lam_S;
    double K[4], dK[4], g[3], f[3];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        K[k] = mp.eta[k] * eh;
        dK[k] = K[k] * ih;
    }
    block_sum_grad(nper, wh, c, inv_r, K, dK, f);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        K[k] = mp.eta[k] * es;
        dK[k] = K[k] * is;
    }
    block_sum_grad(nper, ws, c, inv_r, K, dK, g);
    double s = 0.0;
    if (scc) s = dq[A] * dq[B] * gamma_dR(3.2 * U[A], 3.2 * U[B], r);
    if (mp.rep_A != 0.0) s -= mp.rep_A / mp.rep_b * exp(-r / mp.rep_b);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const double t = f[q] + g[q] + s * c[q];   // u = (R_A - R_B) / r = -c
        pf[ab + q] = t;
        pf[ba + q] = -t;
    }
}

// F_A = sum_B pf[A][B] - dq_A E(t), one warp per atom; then V_n = V_{n-1/2} + F_n dt / 2m (V_0
// itself at the first step).
__global__ void __launch_bounds__(128)
    k_force_sum(int nat, const double* pf, const double* dq,
                const DevScalars* sc, const double* Vh,
                const double* mass, double dt, int first, double* F,
                double* Vn) {
    const int lane = threadIdx.x & 31, A = blockIdx.x * 4 + (threadIdx.x >> 5);
    pdl_launch_dependents();
    pdl_wait();
    if (A >= nat) return;
    double f[3] = {0.0, 0.0, 0.0};
    const double* p = pf + 3 * (size_t)A * nat;
    for (int B = lane; B < nat; B += 32)
        for (int q = 0; q < 3; ++q) f[q] += p[3 * B + q];
    for (int q = 0; q < 3; ++q) f[q] = warp_sum_d(f[q]);
    if (lane < 3) {
        const int i = 3 * A + lane;
        const double x = (lane == 0 ? f[0] : lane == 1 ? f[1] : f[2]) - dq[A] * sc->E[lane];
        F[i] = x;
        Vn[i] = first ? Vh[i] : Vh[i] + x * dt / (2.0 * (mass[A] * 1822.888486));
    }
}

// The non-adiabatic coupling D_mu_nu = Rdot_B . grad_B S_mu_nu (mu in A, nu in B != A, on-site
// blocks 0; eq:nac, eq:onsite), or with `transposed` its transpose, and the pair sums of the work
// rate P = Re Tr[S^-1 H rho (D - D^T)].  One thread per pair A < B (blockIdx.y = A): both blocks
// of a pair are directional derivatives of one s/p block T(d), d = R_B - R_A,
//   D_AB,ij = V_B . grad T_ij,  D_BA,ji = -V_A . grad T_ij,
// with d(c_a) = (V_a - c_a (c.V)) / r and d(K) = K' (c.V) along V.
__device__ __forceinline__ void block_along(int nper, const double c[3], double inv_r, const double K[4],
                                            const double dK[4], const double V[3], double (&o)[16]) {
    const double cv = c[0] * V[0] + c[1] * V[1] + c[2] * V[2];
    o[0] = dK[0] * cv;
    if (nper == 1) return;
    double dc[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) dc[a] = (V[a] - c[a] * cv) * inv_r;
    const double k1 = dK[1] * cv, d23 = K[2] - K[3], k23 = (dK[2] - dK[3]) * cv, k3 = dK[3] * cv;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double sa = dc[a] * K[1] + c[a] * k1;
        o[1 + a] = sa;
        o[4 * (1 + a)] = -sa;
#pragma unroll
        for (int b = 0; b <= a; ++b) {
            const double pp = (dc[a] * c[b] + c[a] * dc[b]) * d23 + c[a] * c[b] * k23 + (a == b ? k3 : 0.0);
            o[4 * (1 + a) + 1 + b] = pp;
            o[4 * (1 + b) + 1 + a] = pp;
        }
    }
}

__global__ void __launch_bounds__(kPairThreads)
    k_nac_power(int nat, int nper, const double* R, const double* V,
                ModelParams mp, const double* xre, int transposed, double* D,
                double* part) {
    const int A = blockIdx.y, B = blockIdx.x * kPairThreads + threadIdx.x;
    const int N = nat * nper;
    double p = 0.0;
    pdl_wait();
    if (B >= A && B < nat) {
        double ab[16], ba[16];   // blocks (A, B) and, transposed, (B, A) of D
        if (A == B) {
#pragma unroll
            for (int k = 0; k < 16; ++k) ab[k] = ba[k] = 0.0;
        } else {
            const double d[3] = {R[3 * B] - R[3 * A], R[3 * B + 1] - R[3 * A + 1],
                                 R[3 * B + 2] - R[3 * A + 2]};
            const double r = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
            const double inv_r = 1.0 / r;
            const double c[3] = {d[0] * inv_r, d[1] * inv_r, d[2] * inv_r};
            const double es = -mp.s0 * exp(-r / mp.lam_S), is = -1.0 / mp.lam_S;
            double K[4], dK[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                K[k] = mp.eta[k] * es;
                dK[k] = K[k] * is;
            }
            const double vb[3] = {V[3 * B], V[3 * B + 1], V[3 * B + 2]};
            const double va[3] = {-V[3 * A], -V[3 * A + 1], -V[3 * A + 2]};
            block_along(nper, c, inv_r, K, dK, vb, ab);
            block_along(nper, c, inv_r, K, dK, va, ba);
            // P: X_AB,ij (D_BA,ji - D_AB,ij) + X_BA,ji (D_AB,ij - D_BA,ji)
            if (nper == 4) {
                double x[16];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const double2* px = reinterpret_cast<const double2*>(xre + (size_t)(4 * A + i) * N + 4 * B);
                    const double2 x0 = px[0], x1 = px[1];
                    x[4 * i] = x0.x, x[4 * i + 1] = x0.y, x[4 * i + 2] = x1.x, x[4 * i + 3] = x1.y;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const double2* px = reinterpret_cast<const double2*>(xre + (size_t)(4 * B + j) * N + 4 * A);
                    const double2 x0 = px[0], x1 = px[1];
                    const double y[4] = {x0.x, x0.y, x1.x, x1.y};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        p = fma(x[4 * i + j] - y[i], ba[4 * i + j] - ab[4 * i + j], p);
                }
            } else {
                p = (xre[(size_t)A * N + B] - xre[(size_t)B * N + A]) * (ba[0] - ab[0]);
            }
        }
        // (A, B) holds ab and (B, A) the transpose of ba; in D^T the two change places
        if (nper == 4) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                double2* o = reinterpret_cast<double2*>(D + (size_t)(4 * A + i) * N + 4 * B);
                const double* s = transposed ? ba : ab;
                o[0] = make_double2(s[4 * i], s[4 * i + 1]);
                o[1] = make_double2(s[4 * i + 2], s[4 * i + 3]);
            }
            if (A != B)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    double2* o = reinterpret_cast<double2*>(D + (size_t)(4 * B + j) * N + 4 * A);
                    const double* s = transposed ? ab : ba;
                    o[0] = make_double2(s[j], s[4 + j]);
                    o[1] = make_double2(s[8 + j], s[12 + j]);
                }
        } else {
            D[(size_t)A * N + B] = transposed ? ba[0] : ab[0];
            if (A != B) D[(size_t)B * N + A] = transposed ? ab[0] : ba[0];
        }
    }
    p = warp_sum_d(p);
    __shared__ double red[kPairThreads / 32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = p;
    __syncthreads();
    if (threadIdx.x == 0) part[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = red[0] + red[1];
}

// Sum the block partials into P_n; work_n = work_{n-1} + dt/2 (P_n + P_{n-1}) (none at
// the first step).  commit = 0: only report (observables of the current state).
__global__ void __launch_bounds__(1024)
    k_power_finish(int nb, const double* part, MdScalars* md, double dt,
                   int first, int commit) {
    double p = 0.0;
    pdl_launch_dependents();
    pdl_wait();
    for (int k = threadIdx.x; k < nb; k += 1024) p += part[k];
    p = warp_sum_d(p);
    __shared__ double red[32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = p;
    __syncthreads();
    if (threadIdx.x >= 32) return;
    p = warp_sum_d(red[threadIdx.x]);
    if (threadIdx.x != 0) return;
    const double w = first ? md->work : md->work + 0.5 * dt * (p + md->P_prev);
    md->P_now = p;
    md->work_now = w;
    if (commit) {
        md->work = w;
        md->P_prev = p;
    }
}

// V_{n+1/2} = V_n + F_n dt / 2m;  R_{n+1} = R_n + dt V_{n+1/2}.
__global__ void k_vv(int nat, const double* __restrict__ Vn, const double* __restrict__ F,
                     const double* __restrict__ mass, double dt, double* __restrict__ Vh,
                     double* __restrict__ R) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 3 * nat) return;
    const double m = mass[i / 3] * 1822.888486;
    const double vh = Vn[i] + F[i] * dt / (2.0 * m);
    Vh[i] = vh;
    R[i] += dt * vh;
}

}  // namespace

size_t pair_blocks(int nat) { return (size_t)nat * ((nat + kPairThreads - 1) / kPairThreads); }

void launch_forces(const Ctx& c, const double* rre, const double* xre, double* F, int first,
                   cudaStream_t st) {
    const dim3 g((c.nat + kPairThreads - 1) / kPairThreads, c.nat);
    launch_pdl(k_pair_forces, g, dim3(kPairThreads), 0, st, c.nat, c.nper, c.prm.scc, c.d_R, rre, xre,
               c.v_atom, c.dq, c.d_U, c.mp, c.md_pf);
    launch_pdl(k_force_sum, dim3((c.nat + 3) / 4), dim3(128), 0, st, c.nat, c.md_pf, c.dq, c.sc, c.d_V,
               c.d_mass, c.prm.dt, first, F, c.d_Vn);
}

void launch_nac_power(const Ctx& c, const double* V, const double* xre, int transposed, double* D,
                      int first, int commit, cudaStream_t st) {
    const dim3 g((c.nat + kPairThreads - 1) / kPairThreads, c.nat);
    launch_pdl(k_nac_power, g, dim3(kPairThreads), 0, st, c.nat, c.nper, c.d_R, V, c.mp, xre, transposed,
               D, c.pw_part);
    launch_pdl(k_power_finish, dim3(1), dim3(1024), 0, st, (int)pair_blocks(c.nat), c.pw_part, c.md,
               c.prm.dt, first, commit);
}

void launch_vv(const Ctx& c, const double* F, cudaStream_t st) {
    k_vv<<<(3 * c.nat + 255) / 256, 256, 0, st>>>(c.nat, c.d_Vn, F, c.d_mass, c.prm.dt, c.d_V,
                                                   c.d_R);
}

}  // namespace tdb
