// Integer-slice GEMM on the tcgen05 tensor cores (see tdb_oz.h for the arithmetic).
//
// Data path per 128 x 64 output tile: TMA loads the slices of A and of B^T for a 32-deep K
// block into a shared-memory ring; one thread issues the slice products (pairs s + t < W) of
// each 16-deep step as MMAs of N <= 256 into W TMEM accumulators, one per weight w = s + t;
// after every chunk of K sixteen drain warps move the (exact, integer-valued) accumulators
// into 64-bit integer sums in registers and hand the TMEM back in two halves, so that the
// next chunk's products start while the second half is still read; the last drain rounds the
// sums to FP64, applies the row and column scales and writes C.  All waits are bounded; a
// time-out records an error code and the kernel frees its TMEM and returns.
//
// What bounds it: the ring feed (72 KB for each 32-deep block of 21 pairs) and the
// shared-memory reads of the MMAs.  FP64 arithmetic and 64-bit conversions issue at two lanes
// a clock per SM on this part, so nothing in the kernels of this file uses them: the drain
// converts to 32-bit integers and accumulates with 32 x 32 + 64-bit multiply-adds, the
// rounding to FP64 and the slicing work on the bits.
#include <cuda.h>
#include <cuda_fp16.h>

#include <cstdint>

#include "pdl.cuh"
#include "tc_ptx.cuh"
#include "tdb_oz.h"
#include "tdb_tc.h"

namespace tdb {
namespace oz {

namespace {
using namespace tc::ptx;

constexpr int BM = 128, BN = 64, BK = 32;
constexpr int kDrainWarps = 16;               // four per TMEM lane quarter, 16 columns each
constexpr int kThreads = 128 + 32 * kDrainWarps;   // warps 0-3: TMA, MMA, TMEM; then the drain
constexpr int A_TILE = BM * BK * 2;           // 8 KiB per A slice
constexpr int B_TILE = BN * BK * 2;           // 4 KiB per B slice
constexpr uint32_t TMEM_COLS = 512;
constexpr int kHalfW = 4;                     // weights 0-3 and 4- are handed back separately

template <int SCH>
struct Cfg;
template <>
struct Cfg<kSix> {
    static constexpr int NS = 6, NW = 6, BITS = 7, CHUNK = 512, STAGES = 3;
};
template <>
struct Cfg<kSeven> {
    static constexpr int NS = 7, NW = 8, BITS = 8, CHUNK = 128, STAGES = 2;
};
template <>
struct Cfg<kLow> {
    static constexpr int NS = 3, NW = 3, BITS = 7, CHUNK = 512, STAGES = 4;
};
template <int SCH>
constexpr int stage_bytes() {
    return Cfg<SCH>::NS * (A_TILE + B_TILE);
}
template <int SCH>
constexpr int smem_bytes() {
    return Cfg<SCH>::STAGES * stage_bytes<SCH>() + 1024 + 256;
}
// largest number of digit pairs of one weight
template <int SCH>
constexpr int max_pairs() {
    return Cfg<SCH>::NW <= Cfg<SCH>::NS ? Cfg<SCH>::NW : Cfg<SCH>::NS;
}
static_assert(smem_bytes<kSix>() <= 227 * 1024 && smem_bytes<kSeven>() <= 227 * 1024 &&
                  smem_bytes<kLow>() <= 227 * 1024,
              "shared memory");
static_assert(Cfg<kSix>::NW * BN <= 512 && Cfg<kSeven>::NW * BN <= 512, "accumulators must fit in TMEM");
static_assert(max_pairs<kSix>() * Cfg<kSix>::CHUNK * 64 * 64 < (1 << 24) &&
                  max_pairs<kSeven>() * Cfg<kSeven>::CHUNK * 128 * 128 < (1 << 24),
              "chunk sums must stay exact in FP32");

struct Maps {
    CUtensorMap a[kMaxSlices];
    CUtensorMap b[2][kMaxSlices];
};

struct Params {
    int M, N, K;
    const int* ea;
    const int* eb[2];
    double* C[2];
    int ldc[2];
    int* err;
    uint32_t idesc[5];   // [nb]: instruction descriptor of an N = 64 nb product
    Gate gate;
};

// (hi 2^SHIFT + lo) 2^x as the nearest double (ties to even), in integer arithmetic.
template <int SHIFT>
__device__ __forceinline__ double scaled_sum(long long hi, long long lo, int x) {
    unsigned long long l = static_cast<unsigned long long>(hi) << SHIFT;
    long long h = hi >> (64 - SHIFT);
    const unsigned long long l2 = l + static_cast<unsigned long long>(lo);
    h += (lo >> 63) + (l2 < l ? 1 : 0);
    l = l2;
    const unsigned long long sign = static_cast<unsigned long long>(h) & 0x8000000000000000ull;
    if (sign) {
        l = 0ull - l;
        h = -h - (l != 0 ? 1 : 0);
    }
    const unsigned long long hm = static_cast<unsigned long long>(h);
    if ((hm | l) == 0) return 0.0;
    // top 64 bits m of the 128-bit magnitude, the leading one at bit 63; below: the rest
    const int lz = hm ? __clzll(hm) : 64 + __clzll(l);
    unsigned long long m, below;
    if (lz >= 64) {
        m = l << (lz - 64);
        below = 0;
    } else {
        m = lz ? (hm << lz) | (l >> (64 - lz)) : hm;
        below = l << lz;
    }
    const unsigned r = static_cast<unsigned>(m) & 0x7ffu;
    m >>= 11;
    if (r > 0x400u || (r == 0x400u && (below != 0 || (m & 1)))) ++m;
    // value = m 2^(127 - lz - 52 + x) with m in [2^52, 2^53]
    const int be = 1023 + 127 - lz + x;
    if (be >= 1 && be < 2046)
        return __longlong_as_double(static_cast<long long>(
            sign | ((static_cast<unsigned long long>(be - 1) << 52) + m)));
    const double v = ldexp(static_cast<double>(m), be - 1023 - 52);
    return sign ? -v : v;
}

// The same for hi 2^SHIFT + lo below 2^63 in magnitude (kSix: 2^24 chunk sums, weights to 2^35, 8
// chunks): a third of the instructions, which the epilogue is bound by.
template <int SHIFT>
__device__ __forceinline__ double scaled_sum64(long long hi, long long lo, int x) {
    const long long t = static_cast<long long>(static_cast<unsigned long long>(hi) << SHIFT) + lo;
    if (t == 0) return 0.0;
    const unsigned long long sign = static_cast<unsigned long long>(t) & 0x8000000000000000ull;
    unsigned long long m = static_cast<unsigned long long>(t < 0 ? -t : t);
    const int lz = __clzll(m);
    m <<= lz;
    const unsigned r = static_cast<unsigned>(m) & 0x7ffu;
    m >>= 11;
    if (r > 0x400u || (r == 0x400u && (m & 1))) ++m;
    // value = m 2^(63 - lz - 52 + x) with m in [2^52, 2^53]
    const int be = 1023 + 63 - lz + x;
    if (be >= 1 && be < 2046)
        return __longlong_as_double(static_cast<long long>(
            sign | ((static_cast<unsigned long long>(be - 1) << 52) + m)));
    const double v = ldexp(static_cast<double>(m), be - 1023 - 52);
    return sign ? -v : v;
}

// One CTA per 128 x 64 output tile; every CTA issues its own TMA loads of the A and B
// slices it multiplies.  One product at N = 1024 (128 tiles), kSix: 41 us (79 us when the drain
// used 64-bit conversions and the rounding FP64 arithmetic), kSeven: 68 us; at N = 2048 291 and
// 509 us.
template <int SCH>
__global__ void __launch_bounds__(kThreads, 1)
    k_oz_gemm(const __grid_constant__ Maps maps, Params p) {
    using C = Cfg<SCH>;
    constexpr int NS = C::NS, NW = C::NW, STAGES = C::STAGES;
    constexpr int SB = stage_bytes<SCH>(), kChunkKB = C::CHUNK / BK;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* gbase = smem_raw + (base - raw);
    uint64_t* bars = reinterpret_cast<uint64_t*>(gbase + STAGES * SB);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 3);
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + STAGES);
    const uint32_t cfull = smem_u32(bars + 2 * STAGES), cempty = smem_u32(bars + 2 * STAGES + 1);

    if (p.gate.norm) {
        pdl_wait();
        if (__uint_as_float(__ldcg(p.gate.norm)) < p.gate.below) return;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int z = blockIdx.z;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int nkb = (p.K + BK - 1) / BK;
    const int nchunk = (nkb + kChunkKB - 1) / kChunkKB;

    if (warp == 3 && lane < 2 * NS) prefetch_map(lane < NS ? &maps.a[lane] : &maps.b[z][lane - NS]);
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        mbar_init(cfull, 1);
        mbar_init(cempty, kDrainWarps);       // one arrival per drain warp and half
        mbar_init(cempty + 8, kDrainWarps);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        fence_before();
    }
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    // the slices and exponents belong to the previous kernels from here on
    pdl_wait();

    if (warp == 0) {
        if (lane == 0) {
            // TMA producer: the slices of A, then of B^T, of one K block per stage
            for (int kb = 0; kb < nkb; ++kb) {
                const int s = kb % STAGES, round = kb / STAGES;
                if (kb >= STAGES && !mbar_wait(empty0 + 8 * s, (round - 1) & 1, p.err, 1)) break;
                const uint32_t st = base + s * SB, fb = full0 + 8 * s;
                mbar_expect_tx(fb, SB);
#pragma unroll
                for (int q = 0; q < NS; ++q) {
                    tma_load_2d(st + q * A_TILE, &maps.a[q], kb * BK, m0, fb);
                    tma_load_2d(st + NS * A_TILE + q * B_TILE, &maps.b[z][q], kb * BK, n0, fb);
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            for (int kb = 0; kb < nkb; ++kb) {
                const int s = kb % STAGES, round = kb / STAGES;
                const int c = kb / kChunkKB;
                const bool first = (kb % kChunkKB) == 0;
                if (!mbar_wait(full0 + 8 * s, round & 1, p.err, 2)) break;
                // a new chunk overwrites the accumulators once the previous one is drained:
                // weights below kHalfW now, the others after this block's first MMA
                if (first && c > 0 && !mbar_wait(cempty, (c - 1) & 1, p.err, 2)) break;
                fence_after();
                const uint32_t st = base + s * SB;
                bool drained = true;
#pragma unroll
                for (int k = 0; k < BK / 16; ++k) {
                    uint64_t a[NS], b[NS];
#pragma unroll
                    for (int q = 0; q < NS; ++q) {
                        a[q] = sdesc(st + q * A_TILE + k * 32);
                        b[q] = sdesc(st + NS * A_TILE + q * B_TILE + k * 32);
                    }
                    // pair (sa, tb) into the accumulator of weight sa + tb.  The B slices lie
                    // one after another in shared memory and the accumulators by weight in
                    // TMEM, so one MMA of N = 64 nb takes the pairs (sa, tb .. tb + nb - 1)
                    // into the accumulators sa + tb .. sa + tb + nb - 1.  In a chunk's first
                    // step the sa = 0 products start the accumulators 0 .. NS - 1 afresh and
                    // the last pair of sa = 1 the accumulator NS, where one is kept.
                    const bool fresh = first && k == 0;
#pragma unroll
                    for (int sa = 0; sa < NS; ++sa)
#pragma unroll
                        for (int tb = 0; tb < NS && sa + tb < NW; tb += 4) {
                            int nb = 4;
                            if (nb > NS - tb) nb = NS - tb;
                            if (nb > NW - sa - tb) nb = NW - sa - tb;
                            const uint32_t d = tmem + static_cast<uint32_t>((sa + tb) * BN);
                            if (fresh && sa == 0) {
                                if (tb >= kHalfW && c > 0) drained = mbar_wait(cempty + 8, (c - 1) & 1, p.err, 2);
                                if (tb >= kHalfW) fence_after();
                                mma_f16(d, a[sa], b[tb], p.idesc[nb], 0u);
                            } else if (sa == 1 && NW > NS && sa + tb + nb - 1 == NS && fresh) {
                                if (nb > 1) mma_f16(d, a[sa], b[tb], p.idesc[nb - 1], 1u);
                                mma_f16(tmem + static_cast<uint32_t>(NS * BN), a[sa], b[tb + nb - 1],
                                        p.idesc[1], 0u);
                            } else {
                                mma_f16(d, a[sa], b[tb], p.idesc[nb], 1u);
                            }
                        }
                }
                if (!drained) break;
                // free the stage for a refill (none follows the last STAGES blocks, so no
                // arrival is left in flight when the CTA exits)
                if (kb + STAGES < nkb) mma_commit(empty0 + 8 * s);
                if ((kb % kChunkKB) == kChunkKB - 1 || kb == nkb - 1) mma_commit(cfull);
            }
        }
    } else if (warp >= 4) {
        // drain warps: TMEM lane quarter (warp % 4) and 16 columns each
        const int quarter = warp & 3, cg = (warp - 4) >> 2;
        const int row = m0 + quarter * 32 + lane, col0 = n0 + cg * 16;
        const uint32_t lane_off = static_cast<uint32_t>(quarter * 32) << 16;
        // sum over the chunks of the weights below NW/2 (hi) and above (lo), each in units of
        // its smallest weight: value = hi 2^(BITS NL) + lo
        constexpr int NH = NW / 2, NL = NW - NH, BITS = C::BITS;
        long long hi[16], lo[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) hi[j] = lo[j] = 0;
        bool ok = true;
        for (int c = 0; c < nchunk && ok; ++c) {
            ok = __all_sync(0xffffffffu, mbar_wait(cfull, c & 1, p.err, 3) ? 1 : 0) != 0;
            if (!ok) break;
            fence_after();
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                uint32_t r[16];
                tmem_ld(tmem + static_cast<uint32_t>(w * BN + cg * 16) + lane_off, r);
                tmem_wait_ld();
                // integers below 2^24: exact in 32-bit integers
                const int wgt = 1 << (BITS * ((w < NH ? NH : NW) - 1 - w));
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const long long v =
                        static_cast<long long>(__float2int_rn(__uint_as_float(r[j]))) * wgt;
                    if (w < NH)
                        hi[j] += v;
                    else
                        lo[j] += v;
                }
                constexpr int kFirst = (kHalfW < NW ? kHalfW : NW) - 1;
                if (w == kFirst || w == NW - 1) {
                    fence_before();
                    __syncwarp();
                    if (lane == 0 && w == kFirst) mbar_arrive(cempty);
                    if (lane == 0 && w == NW - 1) mbar_arrive(cempty + 8);
                }
            }
        }
        // the tiles are summed: the next kernel's blocks may be scheduled
        pdl_launch_dependents();
        if (ok && row < p.M) {
            const int ea = p.ea[row];
            const int ex = ea - 2 * (BITS - 1) - BITS * (NW - 1);
            const int* eb = p.eb[z] + col0;
            double* out = p.C[z] + static_cast<size_t>(row) * p.ldc[z] + col0;
            const bool vec = col0 + 16 <= p.N && (reinterpret_cast<uintptr_t>(out) & 31) == 0;
#pragma unroll
            for (int j0 = 0; j0 < 16; j0 += 4) {
                double v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int e = col0 + j0 + j < p.N ? eb[j0 + j] : 0;
                    v[j] = SCH == kSeven ? scaled_sum<BITS * NL>(hi[j0 + j], lo[j0 + j], ex + e)
                                         : scaled_sum64<BITS * NL>(hi[j0 + j], lo[j0 + j], ex + e);
                    if (ea >= kNonFinite || e >= kNonFinite)
                        v[j] = __longlong_as_double(0x7ff8000000000000ll);
                }
                if (vec) {
                    // whole 32-byte sectors: one row of the tile per lane
                    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(out + j0),
                                 "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3])
                                 : "memory");
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (col0 + j0 + j < p.N) out[j0 + j] = v[j];
                }
            }
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 2) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(TMEM_COLS)
                     : "memory");
    }
}

// ---- slicing ----
// Everything on the bits of the FP64 values: the row maximum needs only the high words, the
// scaled value v = round(x 2^(T - e)), T = BITS NS - 1 (ties to even), is a shift of the
// mantissa, and adding 2^(BITS-1) to every digit below the top one turns the balanced digits
// (|d| <= 2^(BITS-1)) into plain bit fields.

struct SlicePtrs {
    uint16_t* s[kMaxSlices];
    int* e;
    int ld;
};

// exponent e of a row whose largest high word (sign cleared) is mh: |x| < 2^e
__device__ __forceinline__ int row_exponent(uint32_t mh) {
    if (mh >= 0x7ff00000u) return kNonFinite;
    const int be = static_cast<int>(mh >> 20);
    return (be > 1 ? be : 1) - 1022;
}

// The digit fields of x in a row of exponent e: u holds d_q + 2^(BITS-1) in its bit fields
// (the top digit without the offset).
template <int NS, int BITS>
__device__ __forceinline__ long long digit_fields(double x, int e) {
    const long long b = __double_as_longlong(x);
    const int be = static_cast<int>((b >> 52) & 0x7ff);
    unsigned long long m = static_cast<unsigned long long>(b) & 0xfffffffffffffull;
    if (be) m |= 0x10000000000000ull;
    const int sh = (be ? be : 1) - 1075 + (BITS * NS - 1) - e;   // v = m 2^sh
    if (sh >= 0) {
        m <<= sh;                 // sh <= BITS NS - 54: 2 at most
    } else {
        const int r = sh < -60 ? 60 : -sh;
        const unsigned long long q = m >> r, rest = m << (64 - r);
        m = q + ((rest > 0x8000000000000000ull || (rest == 0x8000000000000000ull && (q & 1))) ? 1 : 0);
    }
    long long v = static_cast<long long>(m);
    if (b < 0) v = -v;
    long long off = 0;
#pragma unroll
    for (int q = 0; q < NS - 1; ++q) off |= 1ll << (BITS * q + BITS - 1);
    return v + off;
}
// Digit q of two values as packed halves: the integer field added to the bits of the half
// 1536 (unit spacing), minus 1536.
template <int NS, int BITS>
__device__ __forceinline__ uint32_t digit_pair(long long u0, long long u1, int q) {
    const int sh = BITS * (NS - 1 - q);
    int f0 = static_cast<int>(u0 >> sh), f1 = static_cast<int>(u1 >> sh);
    if (q > 0) {
        f0 = (f0 & ((1 << BITS) - 1)) - (1 << (BITS - 1));
        f1 = (f1 & ((1 << BITS) - 1)) - (1 << (BITS - 1));
    }
    const uint32_t bits = static_cast<uint32_t>((f0 + 0x6600) & 0xffff) |
                          (static_cast<uint32_t>(f1 + 0x6600) << 16);
    __half2 h;
    memcpy(&h, &bits, 4);
    h = __hsub2(h, __half2half2(__ushort_as_half(0x6600)));
    uint32_t o;
    memcpy(&o, &h, 4);
    return o;
}

__device__ __forceinline__ double flip(double x, unsigned long long sgn) {
    return __longlong_as_double(__double_as_longlong(x) ^ static_cast<long long>(sgn));
}

struct RowJob {
    const double *A, *S, *v;
    unsigned* resid;
    int lda;
    unsigned long long sgn;
    SlicePtrs out;
};
struct RowJobs {
    RowJob j[3];
    Gate gate;
};

// One block per row (blockIdx.x) and matrix (blockIdx.y); every thread keeps its 4 PASS
// consecutive values in registers between the row maximum and the digits, so the matrix is
// read once.  8 bytes in, 2 NS out per value.
template <int SCH, int PASS>
__global__ void __launch_bounds__(256)
    k_slice_rows(const __grid_constant__ RowJobs jobs, int K) {
    constexpr int NS = Cfg<SCH>::NS, BITS = Cfg<SCH>::BITS;
    const RowJob& job = jobs.j[blockIdx.y];
    const int row = blockIdx.x, step = 4 * blockDim.x;
    const double* a = job.A + static_cast<size_t>(row) * job.lda;
    const double* s = job.S ? job.S + static_cast<size_t>(row) * job.lda : nullptr;
    __shared__ uint32_t red[8];
    __shared__ float red_f[8];
    double x[PASS][4];
    uint32_t mh = 0;
    float abs_sum = 0.f;
    pdl_launch_dependents();
    pdl_wait();
    if (jobs.gate.norm && __uint_as_float(__ldcg(jobs.gate.norm)) < jobs.gate.below) return;
    const double vr = job.S ? job.v[row] : 0.0;
    const bool vec = ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(s)) & 15) == 0;
#pragma unroll
    for (int i = 0; i < PASS; ++i) {
        const int k = 4 * threadIdx.x + i * step;
        if (vec && k + 4 <= K) {
            const double2 u0 = *reinterpret_cast<const double2*>(a + k);
            const double2 u1 = *reinterpret_cast<const double2*>(a + k + 2);
            x[i][0] = u0.x;
            x[i][1] = u0.y;
            x[i][2] = u1.x;
            x[i][3] = u1.y;
            if (s) {
                const double2 t0 = *reinterpret_cast<const double2*>(s + k);
                const double2 t1 = *reinterpret_cast<const double2*>(s + k + 2);
                const double t[4] = {t0.x, t0.y, t1.x, t1.y};
#pragma unroll
                for (int j = 0; j < 4; ++j) x[i][j] += 0.5 * t[j] * (vr + job.v[k + j]);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                x[i][j] = k + j < K ? a[k + j] : 0.0;
                if (s && k + j < K) x[i][j] += 0.5 * s[k + j] * (vr + job.v[k + j]);
            }
        }
        if (job.resid) {
            // row of 1 - A: only the diagonal needs arithmetic
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                x[i][j] = k + j == row ? 1.0 - x[i][j] : flip(x[i][j], 0x8000000000000000ull);
                abs_sum += fabsf(static_cast<float>(x[i][j]));
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            mh = max(mh, static_cast<uint32_t>(__double2hiint(x[i][j])) & 0x7fffffffu);
    }
    mh = __reduce_max_sync(0xffffffffu, mh);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mh;
    if (job.resid) {
        for (int o = 16; o > 0; o >>= 1) abs_sum += __shfl_xor_sync(0xffffffffu, abs_sum, o);
        if ((threadIdx.x & 31) == 0) red_f[threadIdx.x >> 5] = abs_sum;
    }
    __syncthreads();
    if (job.resid && threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) t += red_f[w];
        // a NaN counts as the largest norm
        atomicMax(job.resid, t >= 0.f ? __float_as_uint(t) : 0x7f800000u);
    }
    for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) mh = max(mh, red[w]);
    const int e = row_exponent(mh);
    if (threadIdx.x == 0) job.out.e[row] = e;
#pragma unroll
    for (int i = 0; i < PASS; ++i) {
        const int k = 4 * threadIdx.x + i * step;
        if (k >= K) break;
        long long u[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            u[j] = digit_fields<NS, BITS>(e == kNonFinite ? 0.0 : flip(x[i][j], job.sgn),
                                          e == kNonFinite ? 0 : e);
        const size_t o = static_cast<size_t>(row) * job.out.ld + k;   // ld: a multiple of 64
#pragma unroll
        for (int q = 0; q < NS; ++q)
            *reinterpret_cast<uint2*>(job.out.s[q] + o) =
                make_uint2(digit_pair<NS, BITS>(u[0], u[1], q), digit_pair<NS, BITS>(u[2], u[3], q));
    }
}

// Largest high words of |B| per column (colmax starts at zero): 32 columns x 8 row groups per
// block.
__global__ void k_colmax(const double* __restrict__ B, int ldb, int K, int cols,
                         uint32_t* __restrict__ colmax) {
    const int c = blockIdx.x * 32 + threadIdx.x;
    uint32_t m = 0;
    if (c < cols)
        for (int r = blockIdx.y * 8 + threadIdx.y; r < K; r += gridDim.y * 8)
            m = max(m, static_cast<uint32_t>(__double2hiint(B[static_cast<size_t>(r) * ldb + c])) &
                           0x7fffffffu);
    __shared__ uint32_t red[8][33];
    red[threadIdx.y][threadIdx.x] = m;
    __syncthreads();
    if (threadIdx.y == 0 && c < cols) {
        for (int y = 1; y < 8; ++y) m = max(m, red[y][threadIdx.x]);
        atomicMax(colmax + c, m);
    }
}

// Slices of B^T through a 64 x 32 shared-memory transpose (coalesced on both sides).
__global__ void k_slice_cols(const double* __restrict__ B, int ldb, int K, int cols,
                             const uint32_t* __restrict__ colmax, SlicePtrs out) {
    constexpr int NS = Cfg<kSix>::NS, BITS = Cfg<kSix>::BITS;
    __shared__ double t[64][33];
    const int k0 = blockIdx.y * 64, c0 = blockIdx.x * 32;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int r = k0 + threadIdx.y + 8 * i, c = c0 + threadIdx.x;
        t[threadIdx.y + 8 * i][threadIdx.x] =
            (r < K && c < cols) ? B[static_cast<size_t>(r) * ldb + c] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int n = c0 + threadIdx.y + 8 * i, k = k0 + 2 * threadIdx.x;
        if (n >= cols || k >= K) continue;
        const int e = row_exponent(colmax[n]);
        if (k == 0) out.e[n] = e;
        const bool fin = e != kNonFinite;
        const double x0 = fin ? t[2 * threadIdx.x][threadIdx.y + 8 * i] : 0.0;
        const double x1 = fin ? t[2 * threadIdx.x + 1][threadIdx.y + 8 * i] : 0.0;
        const long long u0 = digit_fields<NS, BITS>(x0, fin ? e : 0);
        const long long u1 = digit_fields<NS, BITS>(x1, fin ? e : 0);
        const size_t o = static_cast<size_t>(n) * out.ld + k;
#pragma unroll
        for (int q = 0; q < NS; ++q)
            *reinterpret_cast<uint32_t*>(out.s[q] + o) = digit_pair<NS, BITS>(u0, u1, q);
    }
}

SlicePtrs ptrs(const Sliced& s) {
    SlicePtrs p{};
    for (int q = 0; q < n_slices(s.scheme); ++q) p.s[q] = s.s[q];
    p.e = s.e;
    p.ld = s.ld;
    return p;
}

size_t up256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

template <int SCH>
void run_slice_rows(const RowJobs& j, int njobs, int rows, int K, cudaStream_t st) {
    // four values per thread and pass, 256 threads at most
    int nt = ((K + 3) / 4 + 31) / 32 * 32;
    if (nt > 256) nt = 256;
    const dim3 g(rows, njobs), b(nt);
    const int pass = (K + 4 * nt - 1) / (4 * nt);
    if (pass <= 1)
        launch_pdl(k_slice_rows<SCH, 1>, g, b, 0, st, j, K);
    else if (pass <= 2)
        launch_pdl(k_slice_rows<SCH, 2>, g, b, 0, st, j, K);
    else
        launch_pdl(k_slice_rows<SCH, 4>, g, b, 0, st, j, K);
}

template <int SCH>
cudaError_t run_gemm(const Maps& m, const Params& p, dim3 grid, cudaStream_t st) {
    return launch_pdl(k_oz_gemm<SCH>, grid, dim3(kThreads), smem_bytes<SCH>(), st, m, p);
}

}  // namespace

size_t sliced_bytes(int rows, int K, int scheme) {
    const size_t ld = static_cast<size_t>((K + 63) / 64 * 64);
    return n_slices(scheme) * up256(2 * ld * rows) + up256(sizeof(int) * rows);
}

bool sliced_init(Sliced& s, void* base, int rows, int K, int box_rows, int scheme) {
    s.rows = rows;
    s.K = K;
    s.scheme = scheme;
    s.ld = (K + 63) / 64 * 64;
    char* p = static_cast<char*>(base);
    const int ns = n_slices(scheme);
    for (int q = 0; q < ns; ++q) {
        s.s[q] = reinterpret_cast<uint16_t*>(p);
        p += up256(2 * static_cast<size_t>(s.ld) * rows);
    }
    s.e = reinterpret_cast<int*>(p);
    for (int q = 0; q < ns; ++q)
        if (!tc::make_map(&s.map[q], s.s[q], rows, K, s.ld, 0, box_rows)) return false;
    return true;
}

void slice_rows(const SliceJob* jobs, int njobs, cudaStream_t st, Gate gate) {
    RowJobs j{};
    j.gate = gate;
    for (int i = 0; i < njobs; ++i)
        j.j[i] = {jobs[i].A, jobs[i].S, jobs[i].v, jobs[i].resid, jobs[i].lda,
                  jobs[i].sign < 0 ? 0x8000000000000000ull : 0ull, ptrs(*jobs[i].out)};
    const Sliced& o = *jobs[0].out;
    if (o.scheme == kSeven)
        run_slice_rows<kSeven>(j, njobs, o.rows, o.K, st);
    else
        run_slice_rows<kSix>(j, njobs, o.rows, o.K, st);
}

void slice_rows(const double* A, int lda, double sign, Sliced& out, cudaStream_t st) {
    SliceJob j;
    j.A = A;
    j.lda = lda;
    j.sign = sign;
    j.out = &out;
    slice_rows(&j, 1, st);
}

void slice_cols(const double* B, int ldb, Sliced& out, double* colmax, cudaStream_t st) {
    const int cols = out.rows, K = out.K;
    uint32_t* cm = reinterpret_cast<uint32_t*>(colmax);
    cudaMemsetAsync(cm, 0, sizeof(uint32_t) * cols, st);
    k_colmax<<<dim3((cols + 31) / 32, 16), dim3(32, 8), 0, st>>>(B, ldb, K, cols, cm);
    const dim3 g((cols + 31) / 32, (K + 63) / 64), b(32, 8);
    k_slice_cols<<<g, b, 0, st>>>(B, ldb, K, cols, cm, ptrs(out));
}

cudaError_t prepare() {
    cudaError_t e = cudaFuncSetAttribute(k_oz_gemm<kSix>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         smem_bytes<kSix>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_oz_gemm<kSeven>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 smem_bytes<kSeven>());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_oz_gemm<kLow>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 smem_bytes<kLow>());
    return e;
}

cudaError_t gemm(const Sliced& a, const Part* parts, int nparts, int* err, cudaStream_t st,
                 Gate gate, bool low) {
    if (nparts < 1 || nparts > 2 || a.K < 1 || a.K > kMaxK || (low && a.scheme != kSix))
        return cudaErrorInvalidValue;
    const int scheme = low ? static_cast<int>(kLow) : a.scheme;
    const int N = parts[0].b->rows, ns = n_slices(scheme);
    Maps m{};
    Params p{};
    for (int q = 0; q < ns; ++q) m.a[q] = a.map[q];
    for (int z = 0; z < nparts; ++z) {
        const Sliced& b = *parts[z].b;
        if (b.K != a.K || b.rows != N || b.scheme != a.scheme) return cudaErrorInvalidValue;
        for (int q = 0; q < ns; ++q) m.b[z][q] = b.map[q];
        p.eb[z] = b.e;
        p.C[z] = parts[z].C;
        p.ldc[z] = parts[z].ldc;
    }
    p.M = a.rows;
    p.N = N;
    p.K = a.K;
    p.ea = a.e;
    p.err = err;
    p.gate = gate;
    for (int nb = 1; nb <= 4; ++nb) p.idesc[nb] = tc::idesc_f16(0, nb * BN);
    const dim3 grid((N + BN - 1) / BN, (a.rows + BM - 1) / BM, nparts);
    if (scheme == kLow) return run_gemm<kLow>(m, p, grid, st);
    return scheme == kSeven ? run_gemm<kSeven>(m, p, grid, st) : run_gemm<kSix>(m, p, grid, st);
}

}  // namespace oz
}  // namespace tdb
