// Damped one-sided Fourier transforms of sampled dipole signals: the transforms behind the
// absorption cross section (eq:alpha, eq:sigma, Sec. 2.2) and the transient absorption of
// pump-probe runs (eq:alphaeff, eq:sigmaeff, Sec. 3.2):
//
//   F_s(w) = dt sum_{n < K} x_s[n] exp(-n dt / t_damp) exp(+i w n dt).
//
// FP64 results by two paths, picked by the number of sample-frequency-signal products (see
// kTensorWork):
//  - direct: a thread per frequency, up to nine signals at once (they share its twiddles),
//    the samples split over blocks whose partial sums a second kernel adds in order;
//  - blocked: samples in blocks of 512, F_s(w) = sum_b e^{z_w b 512 dt} P_s,b(w) with
//    P_s,b(w) = sum_{j < 512} x_s[512 b + j] e^{z_w j dt}: one 512-deep matrix product over all
//    (s, b) and w, run as integer slices on the tensor cores (scheme kSeven, FP64-accurate),
//    then one multiply-add per (s, b, w).
// FP64 issues at two lanes a clock per SM on this part, which is what bounds the direct path;
// the blocked path needs it for the twiddles of one block and the outer sums only.
#include <algorithm>
#include <cmath>
#include <vector>

#include "tdb_internal.h"
#include "tdb_oz.h"

namespace tdb {
void set_last_error(const char* msg);
}

namespace {

using namespace tdb;

constexpr int kFreqs = 128;   // frequencies (threads) per block
constexpr int kSamp = 256;    // samples staged per pass
constexpr int kExact = 32;    // samples between exact twiddles
constexpr int kMaxSigs = 9;   // signals per thread of the direct path
constexpr int kBlk = 512;     // samples per block of the blocked path
// From this many products on the blocked path is the faster one.  Whole call, microseconds,
// direct / blocked: 3e6 358 / 366, 1.0e7 349 / 354, 1.5e7 413 / 359, 2.7e7 484 / 383,
// 3.6e8 (9 signals x 20000 samples x 2000 frequencies) 2010 / 521; about 280 of each is the
// call's allocation and copies.  (One thread per frequency over all samples, eight signal
// slots: 14500 for the last.)
constexpr double kTensorWork = 1.2e7;
constexpr size_t kChunkBytes = size_t(256) << 20;   // bound on the blocked path's products

// exp((i w - inv_td) n dt): the phase w n dt to about twice the working precision, so that its
// rounding does not grow with n
__device__ void twiddle(double w, double dt, double inv_td, double n, double& re, double& im) {
    const double t = n * dt, te = fma(n, dt, -t);
    const double p = w * t, pe = fma(w, t, -p) + w * te;
    double sn, cs;
    sincos(p, &sn, &cs);
    const double d = exp(-t * inv_td);
    re = d * fma(-sn, pe, cs);
    im = d * fma(cs, pe, sn);
}

// Partial sums of the samples [n0, n1) of blockIdx.z for the signals of blockIdx.y, or without
// `part` the results themselves (one block takes all samples).  The
// twiddle is exact every 32 samples and advanced by the one-step factor in between, which keeps
// its error at a few tens of ulps.
template <int SIGS>
__global__ void __launch_bounds__(kFreqs)
    k_damped_transform(int nsig, long long K, long long span, const double* __restrict__ x, double dt,
                       double inv_td, int nw, const double* __restrict__ omega,
                       double2* __restrict__ part, double* __restrict__ re,
                       double* __restrict__ im) {
    __shared__ double xs[SIGS][kSamp];
    const int k = blockIdx.x * kFreqs + threadIdx.x;
    const int s0 = blockIdx.y * SIGS;
    const long long b0 = blockIdx.z * span, b1 = b0 + span < K ? b0 + span : K;
    const double w = k < nw ? omega[k] : 0.0;
    double c1, s1;
    twiddle(w, dt, inv_td, 1.0, c1, s1);
    double ar[SIGS], ai[SIGS];
#pragma unroll
    for (int s = 0; s < SIGS; ++s) ar[s] = ai[s] = 0.0;
    for (long long n0 = b0; n0 < b1; n0 += kSamp) {
        __syncthreads();
        for (int i = threadIdx.x; i < SIGS * kSamp; i += kFreqs) {
            const int s = i / kSamp;
            const long long n = n0 + i % kSamp;
            xs[s][i % kSamp] = (s0 + s < nsig && n < b1) ? x[(size_t)(s0 + s) * K + n] : 0.0;
        }
        __syncthreads();
        const int len = (int)(b1 - n0 < kSamp ? b1 - n0 : kSamp);
        for (int b = 0; b < len; b += kExact) {
            double tr, ti;
            twiddle(w, dt, inv_td, (double)(n0 + b), tr, ti);
            const int e = len - b < kExact ? len - b : kExact;
#pragma unroll 2
            for (int j = 0; j < e; ++j) {
#pragma unroll
                for (int s = 0; s < SIGS; ++s) {
                    const double v = xs[s][b + j];
                    ar[s] = fma(v, tr, ar[s]);
                    ai[s] = fma(v, ti, ai[s]);
                }
                const double nr = tr * c1 - ti * s1;
                ti = fma(tr, s1, ti * c1);
                tr = nr;
            }
        }
    }
    if (k >= nw) return;
#pragma unroll
    for (int s = 0; s < SIGS; ++s)
        if (s0 + s < nsig) {
            const size_t i = ((size_t)blockIdx.z * nsig + s0 + s) * nw + k;
            if (part) {
                part[i] = make_double2(ar[s], ai[s]);
            } else {
                re[i] = dt * ar[s];
                im[i] = dt * ai[s];
            }
        }
}

// dt times the sum of nz partial sums, in order
__global__ void k_sum_parts(int nz, size_t n, const double2* __restrict__ part, double dt,
                            double* __restrict__ re, double* __restrict__ im) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double a = 0.0, b = 0.0;
    for (int z = 0; z < nz; ++z) {
        const double2 v = part[(size_t)z * n + i];
        a += v.x;
        b += v.y;
    }
    re[i] = dt * a;
    im[i] = dt * b;
}

// Twiddles of one block, transposed: rows 2 k (re) and 2 k + 1 (im) of frequency k, kBlk
// columns; a thread fills 32 columns, the first exact.
__global__ void k_block_twiddles(int nw, const double* __restrict__ omega, double dt, double inv_td,
                                 double* __restrict__ T) {
    const int seg = threadIdx.x % (kBlk / kExact);
    const int k = (blockIdx.x * blockDim.x + threadIdx.x) / (kBlk / kExact);
    if (k >= nw) return;
    const double w = omega[k];
    double c1, s1, tr, ti;
    twiddle(w, dt, inv_td, 1.0, c1, s1);
    twiddle(w, dt, inv_td, (double)(seg * kExact), tr, ti);
    double* o = T + (size_t)2 * k * kBlk + seg * kExact;
    for (int j = 0; j < kExact; ++j) {
        o[j] = tr;
        o[kBlk + j] = ti;
        const double nr = tr * c1 - ti * s1;
        ti = fma(tr, s1, ti * c1);
        tr = nr;
    }
}

// Outer twiddles E[b][k] = exp(z_k b kBlk dt)
__global__ void k_outer_twiddles(int nb, int nw, const double* __restrict__ omega, double dt,
                                 double inv_td, double2* __restrict__ E) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x, b = blockIdx.y;
    if (k >= nw) return;
    double2 e;
    twiddle(omega[k], dt, inv_td, (double)b * kBlk, e.x, e.y);
    E[(size_t)b * nw + k] = e;
}

// F_s(w_k) = dt sum_b E[b][k] P[s nb + b][2 k .. 2 k + 1]; *nonfinite set where a sum is not finite
__global__ void k_outer_sum(int nb, int nw, const double2* __restrict__ E, const double2* __restrict__ P,
                            double dt, int ldo, double* __restrict__ re, double* __restrict__ im,
                            int* __restrict__ nonfinite) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x, s = blockIdx.y;
    if (k >= nw) return;
    double a = 0.0, c = 0.0;
#pragma unroll 4
    for (int b = 0; b < nb; ++b) {
        const double2 e = E[(size_t)b * nw + k], p = P[((size_t)s * nb + b) * nw + k];
        a = fma(e.x, p.x, fma(-e.y, p.y, a));
        c = fma(e.x, p.y, fma(e.y, p.x, c));
    }
    re[(size_t)s * ldo + k] = dt * a;
    im[(size_t)s * ldo + k] = dt * c;
    if (!isfinite(a) || !isfinite(c)) *nonfinite = 1;
}

tdb_status fail(tdb_status st, const char* msg) {
    tdb::set_last_error(msg);
    return st;
}

template <int SIGS>
void run_direct(dim3 grid, int nsig, long long K, long long span, const double* x, double dt,
                double inv_td, int nw, const double* omega, double2* part, double* re, double* im,
                cudaStream_t st) {
    k_damped_transform<SIGS><<<grid, kFreqs, 0, st>>>(nsig, K, span, x, dt, inv_td, nw, omega, part, re,
                                                      im);
}

size_t up(size_t b) { return (b + 255) & ~(size_t)255; }

// The transform by the blocked or the direct path (checked arguments).  The blocked path sets
// nonfinite where a result is not finite: its slices make a block with an infinite sample NaN.
tdb_status transform(bool blocked, int nsig, long K, const double* x, double dt, double inv_td, int nw,
                     const double* omega, double* re, double* im, bool& nonfinite) {
    const long long nb = ((long long)K + kBlk - 1) / kBlk;
    const long long rows = nb * nsig;
    int cw = nw;   // frequencies per chunk
    if (blocked) {
        const long long fit = (long long)(kChunkBytes / 16) / rows;
        cw = (int)std::min<long long>(std::min<long long>(nw, fit), 8192);
    }
    // direct path: signals per block in equal groups, the samples over enough blocks to fill
    // the chip (at least 256 each)
    const int groups = (nsig + kMaxSigs - 1) / kMaxSigs, sigs = (nsig + groups - 1) / groups;
    const int gx = (nw + kFreqs - 1) / kFreqs;
    long long nz = std::max<long long>(1, std::min<long long>((K + kSamp - 1) / kSamp,
                                                              4 * kSmCount / std::max(1, gx * groups)));
    const long long span = ((K + nz - 1) / nz + kExact - 1) / kExact * kExact;
    nz = (K + span - 1) / span;

    const size_t no = (size_t)nsig * (size_t)nw;
    const size_t xrow = blocked ? (size_t)nb * kBlk : (size_t)K;
    const size_t bx = up(sizeof(double) * nsig * xrow), bw = up(sizeof(double) * nw),
                 bo = up(sizeof(double) * no);
    size_t bt = 0, be = 0, bp = 0, bsa = 0, bsb = 0;
    if (blocked) {
        bt = up(sizeof(double) * 2 * cw * kBlk);
        be = up(sizeof(double2) * nb * cw);
        bp = up(sizeof(double2) * rows * cw);
        bsa = up(oz::sliced_bytes((int)rows, kBlk, oz::kSeven));
        bsb = up(oz::sliced_bytes(2 * cw, kBlk, oz::kSeven));
    } else if (nz > 1) {
        bp = up(sizeof(double2) * nz * no);   // 4 kSmCount x 128 x 9 partial sums at most
    }
    tdb_status rc = TDB_OK;
    cudaStream_t st = nullptr;
    char* base = nullptr;
    auto ok = [&](cudaError_t e) {
        if (e != cudaSuccess && rc == TDB_OK) rc = e == cudaErrorMemoryAllocation ? TDB_ERR_NOMEM : TDB_ERR_CUDA;
        return e == cudaSuccess;
    };
    ok(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
    if (!ok(cudaMalloc(&base, bx + bw + 2 * bo + bt + be + bp + bsa + bsb + 256))) cudaGetLastError();
    if (rc == TDB_OK) {
        double* dx = reinterpret_cast<double*>(base);
        double* dw = reinterpret_cast<double*>(base + bx);
        double* dre = reinterpret_cast<double*>(base + bx + bw);
        double* dim_ = reinterpret_cast<double*>(base + bx + bw + bo);
        char* q = base + bx + bw + 2 * bo;
        int* err = reinterpret_cast<int*>(q + bt + be + bp + bsa + bsb);
        int h_err[2] = {0, 0};
        if (blocked && xrow != (size_t)K) ok(cudaMemsetAsync(dx, 0, bx, st));
        ok(cudaMemcpy2DAsync(dx, sizeof(double) * xrow, x, sizeof(double) * K, sizeof(double) * K, nsig,
                             cudaMemcpyHostToDevice, st));
        ok(cudaMemcpyAsync(dw, omega, sizeof(double) * nw, cudaMemcpyHostToDevice, st));
        if (blocked) {
            double* T = reinterpret_cast<double*>(q);
            double2* E = reinterpret_cast<double2*>(q + bt);
            double* P = reinterpret_cast<double*>(q + bt + be);
            oz::Sliced a, b;
            ok(cudaMemsetAsync(err, 0, 2 * sizeof(int), st));
            ok(oz::prepare());
            if (!oz::sliced_init(a, q + bt + be + bp, (int)rows, kBlk, 128, oz::kSeven)) rc = TDB_ERR_CUDA;
            oz::slice_rows(dx, kBlk, 1.0, a, st);
            for (int w0 = 0; w0 < nw && rc == TDB_OK; w0 += cw) {
                const int w = std::min(cw, nw - w0);
                if (!oz::sliced_init(b, q + bt + be + bp + bsa, 2 * w, kBlk, 64, oz::kSeven)) {
                    rc = TDB_ERR_CUDA;
                    break;
                }
                const int per = kBlk / kExact, nth = 128;
                k_block_twiddles<<<(w * per + nth - 1) / nth, nth, 0, st>>>(w, dw + w0, dt, inv_td, T);
                k_outer_twiddles<<<dim3((w + 127) / 128, (unsigned)nb), 128, 0, st>>>(
                    (int)nb, w, dw + w0, dt, inv_td, E);
                oz::slice_rows(T, kBlk, 1.0, b, st);
                oz::Part part;
                part.b = &b;
                part.C = P;
                part.ldc = 2 * w;
                ok(oz::gemm(a, &part, 1, err, st));
                k_outer_sum<<<dim3((w + 63) / 64, nsig), 64, 0, st>>>(
                    (int)nb, w, E, reinterpret_cast<const double2*>(P), dt, nw, dre + w0, dim_ + w0,
                    err + 1);
            }
            ok(cudaMemcpyAsync(h_err, err, 2 * sizeof(int), cudaMemcpyDeviceToHost, st));
        } else {
            double2* part = nz > 1 ? reinterpret_cast<double2*>(q) : nullptr;
            const dim3 grid(gx, groups, (unsigned)nz);
            auto go = [&](auto fn) {
                fn(grid, nsig, (long long)K, span, dx, dt, inv_td, nw, dw, part, dre, dim_, st);
            };
            switch (sigs) {
                case 1: go(run_direct<1>); break;
                case 2: go(run_direct<2>); break;
                case 3: go(run_direct<3>); break;
                case 4: go(run_direct<4>); break;
                case 5: go(run_direct<5>); break;
                case 6: go(run_direct<6>); break;
                case 7: go(run_direct<7>); break;
                case 8: go(run_direct<8>); break;
                default: go(run_direct<9>); break;
            }
            if (part)
                k_sum_parts<<<(unsigned)((no + 127) / 128), 128, 0, st>>>((int)nz, no, part, dt, dre, dim_);
        }
        ok(cudaGetLastError());
        ok(cudaMemcpyAsync(re, dre, sizeof(double) * no, cudaMemcpyDeviceToHost, st));
        ok(cudaMemcpyAsync(im, dim_, sizeof(double) * no, cudaMemcpyDeviceToHost, st));
        ok(cudaStreamSynchronize(st));
        nonfinite = h_err[1] != 0;
        if (rc == TDB_OK && h_err[0] != 0) {
            cudaFree(base);
            cudaStreamDestroy(st);
            return fail(TDB_ERR_TIMEOUT, "tdb_damped_transform: a bounded device wait timed out");
        }
    }
    cudaFree(base);
    if (st) cudaStreamDestroy(st);
    if (rc != TDB_OK) tdb::set_last_error("tdb_damped_transform: a CUDA call failed");
    return rc;
}

}  // namespace

extern "C" tdb_status tdb_damped_transform(int nsig, long K, const double* x, double dt,
                                           double t_damp, int nw, const double* omega, double* re,
                                           double* im) {
    if (nsig < 1 || K < 1 || nw < 1 || !x || !omega || !re || !im || !std::isfinite(dt) ||
        !(dt > 0) || std::isnan(t_damp) || t_damp < 0 || nsig > 65535 * 8)
        return fail(TDB_ERR_ARG, "tdb_damped_transform: invalid sizes, pointers, dt or t_damp");
    for (int k = 0; k < nw; ++k)
        if (!std::isfinite(omega[k]))
            return fail(TDB_ERR_ARG, "tdb_damped_transform: non-finite frequency");
    const double inv_td = (t_damp == 0.0 || std::isinf(t_damp)) ? 0.0 : 1.0 / t_damp;
    // blocked path: rows (signal, block) of 512 samples, the frequencies in chunks whose
    // products stay within kChunkBytes.  The slices are exact relative to a row's largest
    // value, so the damping must not spread a block's twiddles over many binades (e^-8 at most).
    // Where its buffers do not fit, the direct path's do with less; where a result is not finite, the
    // direct path takes infinite samples as FP64 arithmetic does.
    const long long nb = ((long long)K + kBlk - 1) / kBlk;
    const bool blocked = (double)nsig * (double)K * nw >= kTensorWork && nb <= 65535 &&
                         kBlk * dt * inv_td <= 8.0 &&
                         nsig <= 65535 && nb * nsig * 2048 <= (long long)kChunkBytes;
    bool nonfinite = false;
    tdb_status rc = transform(blocked, nsig, K, x, dt, inv_td, nw, omega, re, im, nonfinite);
    if (blocked && (rc == TDB_ERR_NOMEM || (rc == TDB_OK && nonfinite)))
        rc = transform(false, nsig, K, x, dt, inv_td, nw, omega, re, im, nonfinite);
    return rc;
}
