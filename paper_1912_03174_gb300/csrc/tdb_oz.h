// Host interface of the integer-slice GEMM (kern_oz.cu): FP64 products on the FP16
// tensor cores with exact accumulation.
//
// Each row of A is scaled by a power of two 2^-e so that its entries lie in (-1, 1),
// rounded to b S - 1 bits and cut into S signed b-bit integer digits (|a_s| <= 2^(b-1)):
//     A_ik = 2^(e_i - (b-1)) sum_s a_s,ik 2^(-b s) + r_ik,   |r_ik| <= 2^(e_i - b S).
// Columns of B are treated alike (stored as rows of B^T).  Every digit product a_s b_t is
// an integer of magnitude <= 2^(2b-2), so the K-sums of all pairs of equal weight
// w = s + t over a chunk of K stay below 2^24 and are exact in the tensor core's FP32
// accumulator; the sum over weights and chunks is exact in 64-bit integers, rounded once.
// Pairs with s + t < W are kept.  Two schemes:
//
//   kSix    6 digits of 7 bits, W = 6 (21 pairs), chunks of 512: error about 7 2^-42 of
//           K max_k|A_ik| max_k|B_kj| -- the TDB_FP64_SLICED form.
//   kSeven  7 digits of 8 bits, W = 8 (34 pairs), chunks of 128: 55-bit operands, the
//           first dropped weight is 2^-64.  On the products of the propagation (S^-1 H,
//           M Re rho, M Im rho; N = 132 .. 520) its error is 0.29 to 0.61 of the DFMA
//           product's in the 2-norm and 0.03 to 0.14 in the largest element: it replaces
//           the DFMA product of the TDB_FP64 form where N is large enough (see use_slices).
//
// The bounds are relative to the largest entry of a row of A times that of a column of B: an element
// of C far below those (rows of S^-1 and rho decay with distance) has their absolute error, not,
// as from DFMA, a relative one of its own.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace tdb {
namespace oz {

enum Scheme { kSix = 0, kSeven = 1, kLow = 2 };   // kLow: leading slices of kSix operands
constexpr int kMaxSlices = 7;
constexpr int kMaxK = 4096;     // keeps the 64-bit sums below 2^63
__host__ __device__ constexpr int n_slices(int scheme) { return scheme == kSeven ? 7 : scheme == kLow ? 3 : 6; }

// Slices of the rows of a rows x K matrix: s[q] is rows x ld 16-bit (FP16 integers),
// ld a multiple of 64; e[i] the power-of-two exponent of row i (kNonFinite: the row holds
// an Inf or NaN and its products are NaN).  The tensor maps cover rows x K (zero fill
// beyond K) with boxes of 32 (K) x box_rows.
struct Sliced {
    uint16_t* s[kMaxSlices] = {};
    int* e = nullptr;
    int rows = 0, K = 0, ld = 0, scheme = kSix;
    CUtensorMap map[kMaxSlices];
};
constexpr int kNonFinite = 1 << 24;

// Bytes of device memory a Sliced of rows x K needs (slices + exponents).
size_t sliced_bytes(int rows, int K, int scheme = kSix);
// Lays a Sliced out in base (256-byte aligned) and encodes its tensor maps; box_rows
// is 128 for an A operand and 64 for a B operand.  False if a map cannot be encoded.
bool sliced_init(Sliced& s, void* base, int rows, int K, int box_rows, int scheme = kSix);

// A matrix to slice by rows: sign * A (rows x K, row-major FP64 with row stride lda), or,
// with S set, the SCC Hamiltonian A + 1/2 S (v_r + v_c) formed element by element
// (eq:hscc; S with the stride of A).  For a B operand that is symmetric (sign 1) or
// antisymmetric (sign -1) this is also the slicing of B^T.
struct SliceJob {
    const double* A = nullptr;
    int lda = 0;
    double sign = 1.0;
    Sliced* out = nullptr;
    const double* S = nullptr;
    const double* v = nullptr;
    unsigned* resid = nullptr;   // slice 1 - A instead; atomicMax of its largest absolute row sum
                                 // (FP32, as float bits)
};
// A launch that does nothing if *norm (float bits, device) is below `below`.
struct Gate {
    const unsigned* norm = nullptr;
    float below = 0.f;
};
// njobs <= 3 matrices of the same rows, K and scheme in one launch.
void slice_rows(const SliceJob* jobs, int njobs, cudaStream_t st, Gate gate = {});
void slice_rows(const double* A, int lda, double sign, Sliced& out, cudaStream_t st);
// Slices of B^T (scheme kSix) for a general B (K x cols, row-major FP64, row stride ldb);
// colmax is a device scratch of cols doubles.
void slice_cols(const double* B, int ldb, Sliced& out, double* colmax, cudaStream_t st);

// One product sharing the A operand: C (M x N, row-major FP64, row stride ldc) = A B.
struct Part {
    const Sliced* b = nullptr;
    double* C = nullptr;
    int ldc = 0;
};
// Once per process and device before the first launch (outside stream capture).
cudaError_t prepare();
// C_z = A B_z for z < nparts (<= 2); M = a.rows, N = b.rows, K = a.K = b.K (<= kMaxK), all
// of one scheme.  err: device flag, set to 1-3 if a bounded wait expired.
// low: only the three leading slices of each operand and the six pairs s + t < 3 (kSix;
// relative error about 2^-20 of K max|A_i.| max|B_.j|).
cudaError_t gemm(const Sliced& a, const Part* parts, int nparts, int* err, cudaStream_t st,
                 Gate gate = {}, bool low = false);

}  // namespace oz
}  // namespace tdb
