// tallskinny.cu -- FP64 products of tall, narrow matrices on the tensor cores.
//
//   ts_tn: C = A^T B      (A n x p, B n x q, C p x q)
//   ts_nn: Out = beta Out + alpha A C
//
// with p, q <= 64, for the eigensolvers' orthogonalisation and projections.
// GB300's FP64 units do two fused multiply-adds per clock and SM (1.2 TFLOP/s
// on the GPU), so these products, written in FP64 arithmetic, took 80-90% of an
// eigensolver restart while their memory traffic would take a tenth of that.
// Here the products run on the FP16 tensor cores without rounding: the method
// is the splitting of Ozaki, Ogita, Oishi and Rump (Numerical Algorithms 59,
// 2012), on tensor cores as in Mukunoki et al. (ISC 2020), with fixed-point
// digits:
//   * Every column of a tile of kTsRows rows (ts_tn), every row of A and every
//     column of C (ts_nn) is scaled by a power of two so that its largest
//     magnitude lies in [2^61, 2^62), and each element becomes a 64-bit
//     integer: eight signed base-256 digits, most significant first.
//   * Digit products are at most 2^14, so the sum of all products of digits i
//     and j with i + j = d <= 7 over up to 64 terms of the inner dimension is
//     an integer of at most 8 * 64 * 2^14 = 2^23, exact in an FP32
//     accumulator: 36 FP16 mma with 8 accumulators ("diagonals" d = 0..7).
//   * The diagonals are combined in integers, rounded once to FP64 and added in
//     FP64 (one FP64 addition per element and tile instead of kTsRows fused
//     multiply-adds).
// What is left out (i + j >= 8, and bits below 2^-62 of the largest element) is
// at most 2^-58.8 of the product of the two scales per term.  By itself that is a
// bound on the norm: where the large elements of the two operands do not meet, an
// FP64 sum is far more accurate (one element of 1 among 1e-8 in each column, in
// different rows: 1e-12 of sum |a||b| against 2e-17).  So every element's sum of
// |a||b| is found from below as well (magnitudes cut to bf16, one mma beside the
// 36), and an element whose sum is below 2^-5 of the scales' product takes the
// products in FP64 arithmetic instead.  Above that line what is left out is less
// than kTsRows * 2^-53 * sum |a||b| (0.6 of it), the bound of an FP64 sum of as
// many products: the error bound of each element is that of FP64 arithmetic,
// whatever the data.  FP64 arithmetic also takes the elements whose columns (rows)
// hold subnormal numbers or whose scales are near the ends of the exponent range.
// Share of the elements that do, block Krylov-Schur on a symmetrised R-MAT graph,
// first cycles / converged: A^T B below 0.01% / 0.6%, the subtraction of V C none,
// Ritz vectors none / 0.2%.  W R^-1 would have up to 13%, and a kernel for triangular
// factors is as fast in FP64 arithmetic (eigs.cu).
// A tile (row) with an infinity or a NaN gives NaN.
// Largest error against quadruple precision, FP64 kernels -> digits: A^T B,
// 20,000 x 48 by 16, orthonormal columns 7.7e-18 -> 4.9e-18, with rows of very
// different size 4.9e-16 -> 2.0e-16, power-law rows 3.3e-16 -> 6.9e-17; A C, 2-norm
// of the error, 4.6e-17 -> 9.3e-18, 8.7e-16 -> 1.6e-16, 5.1e-16 -> 8.6e-17.
// Digits are made with integer instructions only, since conversions to and from
// FP64 run at the rate of the FP64 units.  Measured, two cycles of the block
// Krylov-Schur solver (one restart) on 148,444 vertices, basis 64, block 16, the
// sums of their launches: A^T B 8.5 -> 1.7 ms (1.3 without the magnitudes' pass),
// A C 3.8 -> 1.9 ms (0.5 of it W R^-1 in FP64 arithmetic; 1.6 with digits throughout
// and no guard), reductions of partials 0.73 -> 0.37 ms; the FP64 units alone would
// need about 7 ms.  Neither memory (DRAM 7-14%, L2 6%) nor the tensor pipe (9-24%)
// bounds these kernels: with 12 warps an SM (168 registers) they issue on 35-51% of
// the cycles.  A warp of ts_tn waits on fixed latencies, loads and the tensor pipe in
// about equal parts; one of ts_nn on fixed latencies and on shared memory and FP64
// results, the FP64 pipe being 31-46% busy with the additions into Out.
#include <algorithm>

#include <cuda_fp16.h>

#include "tallskinny.h"

namespace spmm {

namespace {

constexpr int kTsRows = 64;          // rows per tile of ts_tn: diagonal sums stay within 2^23
constexpr int kTsWarps = 12;         // warps per block, one block per SM (at most 168 registers a thread)
constexpr int kDigits = 8;

// A magnitude is kept as its high word without the sign, the last bit set where
// the low word is not zero: 0 for a zero only.  The largest of a set gives its
// biased exponent: kNoExp where all are zero, kSpecial where an infinity or a NaN
// is among them.
constexpr int kSpecial = 1 << 20;
constexpr int kNoExp = -100000;
__device__ __forceinline__ uint32_t magnitude(uint32_t lo, uint32_t hi) { return (hi & 0x7fffffffu) | min(lo, 1u); }
__device__ __forceinline__ uint32_t magnitude(double x) {
    return magnitude((uint32_t)__double2loint(x), (uint32_t)__double2hiint(x));
}
__device__ __forceinline__ uint32_t magnitude_at(const double* p) {
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
    return magnitude(v.x, v.y);
}
__device__ __forceinline__ int exponent_of(uint32_t h) {
    return h == 0 ? kNoExp : (h >> 20) >= 0x7ffu ? kSpecial : (int)(h >> 20);
}

// A magnitude over its set's scale 2^(emax - 1022), cut to a bf16 (so not above
// it), as a bf16 pair; below 2^-125 zero.
__device__ __forceinline__ uint32_t bf16_below(uint32_t h, int emax) {
    const int de = emax - (int)(h >> 20);
    return (uint32_t)de < 125u ? (uint32_t)(126 - de) << 7 | ((h >> 13) & 0x7fu) : 0u;
}
__device__ __forceinline__ uint32_t bf16_pair(uint32_t h0, uint32_t h1, int e0, int e1) {
    return bf16_below(h0, e0) | bf16_below(h1, e1) << 16;
}

// Whether an element with scales 2^(ea - 1022), 2^(eb - 1022) and at least `low`
// of their product as its sum of |a||b| takes FP64 arithmetic: below the line, with
// subnormal elements that count (sub), or with a result that could leave the normal
// numbers.  Products with a zero set are exact, those with an infinity or a NaN are
// NaN.
constexpr float kLowLine = 0x1p-5f;
__device__ __forceinline__ bool needs_fp64(float low, int ea, int eb, bool sub) {
    if (max(ea, eb) >= kSpecial) return false;
    if (sub) return true;
    if (min(ea, eb) < -50000) return false;
    return !(low >= kLowLine) || ea + eb < 1090 || ea + eb > 3061;
}

// x as eight digits + 128, most significant in the top byte: the 62-bit fixed
// point of x / 2^(emax - 1022), truncated towards zero, plus 0x80 in every byte.
// emax: biased exponent that no element of the scaled set exceeds.  Subnormal
// elements count as zero.
__device__ __forceinline__ uint2 digits_of(double x, int emax) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int e = (int)((hi >> 20) & 0x7ffu);
    const int d = e == 0 ? 63 : min(max(emax - e, 0), 63);
    const uint64_t m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 9;   // < 2^62
    const uint64_t v = m >> d;
    const uint32_t s = (uint32_t)((int32_t)hi >> 31);                               // 0 or ~0
    const uint64_t sv = (v ^ ((uint64_t)s << 32 | s)) - (uint64_t)(int64_t)(int32_t)s;
    const uint64_t y = sv + 0x8080808080808080ull;
    return make_uint2((uint32_t)y, (uint32_t)(y >> 32));
}

// digit i (0 = most significant) of two elements as a pair of FP16 integers:
// byte b under the exponent of 1024 is 1024 + b, less 1152
template <int I>
__device__ __forceinline__ uint32_t digit_pair(uint2 a, uint2 b) {
    constexpr int byte = (kDigits - 1 - I) & 3;
    const uint32_t wa = I < 4 ? a.y : a.x, wb = I < 4 ? b.y : b.x;
    const uint32_t p = __byte_perm(wa, wb, byte | (byte << 4) | ((byte + 4) << 8) | ((byte + 4) << 12));
    uint32_t h = (p & 0x00ff00ffu) | 0x64006400u;
    const __half2 r = __hsub2(*reinterpret_cast<__half2*>(&h), __half2(__float2half(1152.f), __float2half(1152.f)));
    return *reinterpret_cast<const uint32_t*>(&r);
}

__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// all digits of one operand fragment: four (A) or two (B) registers per digit
template <int I>
__device__ __forceinline__ void a_digits(uint32_t (&f)[kDigits][4], const uint2 (&y)[8]) {
    if constexpr (I < kDigits) {
#pragma unroll
        for (int r = 0; r < 4; ++r) f[I][r] = digit_pair<I>(y[2 * r], y[2 * r + 1]);
        a_digits<I + 1>(f, y);
    }
}
template <int I>
__device__ __forceinline__ void b_digits(uint32_t (&f)[kDigits][2], const uint2 (&y)[4]) {
    if constexpr (I < kDigits) {
        f[I][0] = digit_pair<I>(y[0], y[1]);
        f[I][1] = digit_pair<I>(y[2], y[3]);
        b_digits<I + 1>(f, y);
    }
}

// The 36 digit products of one 16 x 8 x 16 step.  Consecutive mma go to
// different diagonals.
__device__ __forceinline__ void mma_digits(float (&acc)[kDigits][4], const uint32_t (&a)[kDigits][4],
                                           const uint32_t (&b)[kDigits][2]) {
#pragma unroll
    for (int i = 0; i < kDigits; ++i)
#pragma unroll
        for (int j = 0; j + i < kDigits; ++j) mma_f16(acc[i + j], a[i], b[j][0], b[j][1]);
}

// sum_d S_d 2^(56 - 8d) * 2^(ea + eb - 2112), rounded once to FP64: the value
// of one element from its eight diagonals and the two biased exponents (a normal
// number or zero unless needs_fp64).
__device__ __forceinline__ double from_diagonals(const float (&acc)[kDigits][4], int c, int ea, int eb) {
    int64_t h = 0, l = 0;
#pragma unroll
    for (int d = 0; d < 4; ++d) h = (h << 8) + (int64_t)__float2int_rn(acc[d][c]);
#pragma unroll
    for (int d = 4; d < 8; ++d) l = (l << 8) + (int64_t)__float2int_rn(acc[d][c]);
    int64_t hs = h + (l >> 32);                  // T = hs * 2^32 + w
    uint32_t w = (uint32_t)l;
    const bool neg = hs < 0;
    if (neg) {
        w = 0u - w;
        hs = ~hs + (w == 0 ? 1 : 0);
    }
    int e2 = ea + eb - 2112;
    uint64_t t = (uint64_t)hs;
    if (t == 0) {                                // only the low word is left
        t = w;
        w = 0;
        e2 -= 32;
    }
    double r = 0.0;
    if (t != 0) {
        const int lz = __clzll((long long)t);    // 17..63: |h| < 2^47
        uint64_t m = t << lz;
        m |= lz >= 32 ? (uint64_t)w << (lz - 32) : (uint64_t)(w >> (32 - lz));
        int be = 1023 + 95 - lz + e2;            // biased exponent of m * 2^(32 - lz + e2)
        const uint64_t q = m + 1024u;            // round to nearest at bit 11
        if (q < m) ++be;                         // carried out: the mantissa is 1.0
        const uint64_t bits = (uint64_t)be << 52 | (q < m ? 0ull : (q >> 11) & 0xfffffffffffffull);
        r = __longlong_as_double((long long)(bits | (neg ? 0x8000000000000000ull : 0ull)));
    }
    // a set with an infinity or a NaN
    return max(ea, eb) >= kSpecial ? __longlong_as_double(0x7ff8000000000000ll) : r;
}

// Warp w of the launch owns unit w % units (16 columns of A by 16 of B) and the
// row tiles w / units, + kgroups, ...; no shared memory and no barriers: a
// tile's column scales and the sums of its magnitudes are found in a first pass,
// which also brings the tile into L1 for the second.  In a fragment, lane 4g + t
// holds rows 2t, 2t+1, 2t+8, 2t+9 of a 16-row step and columns g, g+8.
// SAME: A is B; units are the tile pairs of the upper triangle.
template <bool SAME>
__global__ void __launch_bounds__(kTsWarps * 32, 1)
ts_tn_kernel(const double* __restrict__ A, int64_t lda, int p, const double* __restrict__ B, int64_t ldb, int q,
             int64_t n, int nt, int units, int kgroups, double* __restrict__ partial) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int w = blockIdx.x * kTsWarps + (threadIdx.x >> 5);
    const int unit = w % units, kg = w / units;
    if (kg >= kgroups) return;
    int mi, ni;
    if constexpr (SAME) {
        mi = 0;
        int u = unit;
        while (u >= nt - mi) u -= nt - mi, ++mi;
        ni = mi + u;
    } else {
        mi = unit / nt;
        ni = unit % nt;
    }
    const bool diag = SAME && mi == ni;
    // columns past the last repeat it: their results are not stored
    const double* A0 = A + min(mi * 16 + g, p - 1);
    const double* A1 = A + min(mi * 16 + 8 + g, p - 1);
    const double* B0 = B + min(ni * 16 + g, q - 1);
    const double* B1 = B + min(ni * 16 + 8 + g, q - 1);
    double sum[2][4];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int c = 0; c < 4; ++c) sum[j][c] = 0.0;
    const int64_t tiles = (n + kTsRows - 1) / kTsRows;
    for (int64_t tile = kg; tile < tiles; tile += kgroups) {
        const int64_t r0 = tile * kTsRows;
        // row r of step ks; rows past the last repeat it (and count as zero in the products)
        auto row_of = [&](int ks, int r) { return min(r0 + ks * 16 + 2 * t + (r & 1) + (r >> 1) * 8, n - 1); };
        uint32_t h[kTsRows / 16][4][4], hm[4] = {0, 0, 0, 0};     // A0, A1, B0, B1
#pragma unroll
        for (int ks = 0; ks < kTsRows / 16; ++ks)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int64_t ra = row_of(ks, r) * lda, rb = row_of(ks, r) * ldb;
                h[ks][0][r] = magnitude_at(A0 + ra);
                h[ks][1][r] = magnitude_at(A1 + ra);
                h[ks][2][r] = diag ? 0u : magnitude_at(B0 + rb);
                h[ks][3][r] = diag ? 0u : magnitude_at(B1 + rb);
            }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
#pragma unroll
            for (int ks = 0; ks < kTsRows / 16; ++ks)
#pragma unroll
                for (int r = 0; r < 4; ++r) hm[i] = max(hm[i], h[ks][i][r]);
#pragma unroll
            for (int off = 1; off < 4; off <<= 1) hm[i] = max(hm[i], __shfl_xor_sync(0xffffffffu, hm[i], off));
        }
        if (diag) hm[2] = hm[0], hm[3] = hm[1];
        const int ea0 = exponent_of(hm[0]), ea1 = exponent_of(hm[1]), eb0 = exponent_of(hm[2]), eb1 = exponent_of(hm[3]);
        // bit 4j + c: element c of columns 8j.. takes FP64 arithmetic
        uint32_t fp64 = 0;
        {
            float low[2][4];
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int c = 0; c < 4; ++c) low[j][c] = 0.f;
#pragma unroll
            for (int ks = 0; ks < kTsRows / 16; ++ks) {
                uint32_t ua[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    uint32_t h0 = h[ks][i & 1][i & 2], h1 = h[ks][i & 1][(i & 2) + 1];
                    if (r0 + ks * 16 + 2 * t + (i & 2) * 4 >= n) h0 = 0;
                    if (r0 + ks * 16 + 2 * t + (i & 2) * 4 + 1 >= n) h1 = 0;
                    ua[i] = bf16_pair(h0, h1, (i & 1) ? ea1 : ea0, (i & 1) ? ea1 : ea0);
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const uint32_t(&hb)[4] = h[ks][2 + j];
                    const int eb = j ? eb1 : eb0;
                    const uint32_t b0 = diag ? ua[j] : bf16_pair(hb[0], hb[1], eb, eb);
                    const uint32_t b1 = diag ? ua[2 + j] : bf16_pair(hb[2], hb[3], eb, eb);
                    mma_bf16(low[j], ua, b0, b1);
                }
            }
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int eb = __shfl_sync(0xffffffffu, j ? eb1 : eb0, 4 * (2 * t + (c & 1)));
                    const int ea = c < 2 ? ea0 : ea1;
                    const bool inside = mi * 16 + g + (c < 2 ? 0 : 8) < p && ni * 16 + 8 * j + 2 * t + (c & 1) < q;
                    // near the smallest normal numbers a subnormal element is not below the last digit
                    const bool tiny = min(ea, eb) < 128 && min(ea, eb) >= 0;
                    if (inside && needs_fp64(low[j][c], ea, eb, tiny)) fp64 |= 1u << (4 * j + c);
                }
        }
        float acc[2][kDigits][4];
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int d = 0; d < kDigits; ++d)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[j][d][c] = 0.f;
#pragma unroll 1
        for (int ks = 0; ks < kTsRows / 16; ++ks) {
            double xa[8], xb[8];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int64_t ra = row_of(ks, r) * lda, rb = row_of(ks, r) * ldb;
                xa[r] = A0[ra];
                xa[4 + r] = A1[ra];
                if (!diag) {
                    xb[r] = B0[rb];
                    xb[4 + r] = B1[rb];
                }
            }
            if (r0 + kTsRows > n) {
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    if (r0 + ks * 16 + 2 * t + (r & 1) + (r >> 1) * 8 >= n) xa[r] = xa[4 + r] = 0.0;
            }
            uint32_t fa[kDigits][4];
            {
                // registers of the A fragment: (g, rows 2t..), (g+8, rows 2t..), (g, rows 2t+8..), (g+8, ...)
                uint2 y[8];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    y[r] = digits_of(xa[r], ea0);
                    y[2 + r] = digits_of(xa[4 + r], ea1);
                    y[4 + r] = digits_of(xa[2 + r], ea0);
                    y[6 + r] = digits_of(xa[6 + r], ea1);
                }
                a_digits<0>(fa, y);
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                uint32_t fb[kDigits][2];
                if (diag) {
#pragma unroll
                    for (int d = 0; d < kDigits; ++d) fb[d][0] = fa[d][j], fb[d][1] = fa[d][2 + j];
                } else {
                    uint2 y[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) y[r] = digits_of(xb[4 * j + r], j ? eb1 : eb0);
                    b_digits<0>(fb, y);
                }
                mma_digits(acc[j], fa, fb);
            }
        }
        // element (row g or g+8 of the unit, column 8j + 2t + {0, 1}): its column's
        // exponent sits in lane 4 (2t + {0, 1})
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int eb = __shfl_sync(0xffffffffu, j ? eb1 : eb0, 4 * (2 * t + (c & 1)));
                if (!(fp64 >> (4 * j + c) & 1)) sum[j][c] += from_diagonals(acc[j], c, c < 2 ? ea0 : ea1, eb);
            }
        if (__any_sync(0xffffffffu, fp64 != 0)) {
            const int rows = (int)min((int64_t)kTsRows, n - r0);
#pragma unroll 1
            for (int e = 0; e < 8; ++e) {
                double f = 0.0;
                if (fp64 >> e & 1) {
                    const double* a = ((e & 2) ? A1 : A0) + r0 * lda;
                    const double* b = B + ni * 16 + 8 * (e >> 2) + 2 * t + (e & 1) + r0 * ldb;
#pragma unroll 4
                    for (int r = 0; r < rows; ++r) f = fma(a[r * lda], b[r * ldb], f);
                }
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (u == e && (fp64 >> u & 1)) sum[u >> 2][u & 3] += f;
            }
        }
    }
    double* out = partial + (int64_t)kg * p * q;
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int r = mi * 16 + g + (c < 2 ? 0 : 8), s = ni * 16 + 8 * j + 2 * t + (c & 1);
            if (r < p && s < q) {
                out[r * q + s] = sum[j][c];
                if (SAME && !diag) out[s * q + r] = sum[j][c];
            }
        }
}

// out[e] = sum over the row groups' partials in a fixed order: 8 elements by 32
// strands per block, the strands added by a fixed tree.
__global__ void __launch_bounds__(256) ts_reduce_kernel(const double* __restrict__ partial, int nparts, int pq,
                                                        double* __restrict__ out) {
    __shared__ double sh[32][8];
    const int el = threadIdx.x & 7, strand = threadIdx.x >> 3;
    const int e = blockIdx.x * 8 + el;
    double s0 = 0.0, s1 = 0.0;
    if (e < pq) {
        int c = strand;
        for (; c + 32 < nparts; c += 64) {
            s0 += partial[(int64_t)c * pq + e];
            s1 += partial[(int64_t)(c + 32) * pq + e];
        }
        if (c < nparts) s0 += partial[(int64_t)c * pq + e];
    }
    sh[strand][el] = s0 + s1;
    __syncthreads();
    for (int off = 16; off > 0; off >>= 1) {
        if (strand < off) sh[strand][el] += sh[strand + off][el];
        __syncthreads();
    }
    if (strand == 0 && e < pq) out[e] = sh[0][el];
}

// Out = beta Out + alpha A C.  Row k of C is scaled to a largest magnitude in
// [1, 2) and its scale goes to column k of A, so that a row of A is scaled by its
// largest product, whatever the sizes of A's columns that C compensates (R^-1
// in CholQR); then every column of C is scaled by its largest element.  The
// digits of C sit in shared memory in fragment order (made once per block); a
// warp takes 16 rows of A at a time and for each 16 columns of Out multiplies
// the digits of up to 64 columns of A into one set of accumulators.
// The largest element of each column of C is left out of the digits and its
// product added by one FP64 multiply-add: C is often near a diagonal matrix (the
// Ritz vectors once they converge, V^T W of a restarted cycle), so that an element of
// Out is about one element of A, often far below its row's largest, and the digits
// then hold only the small rest.  An element takes FP64 arithmetic only if neither
// its sum of magnitudes nor that largest product is above the line; with Out added
// unscaled, an element of Out that is larger than what could be left out times 2^53
// hides it too.
__global__ void __launch_bounds__(kTsWarps * 32, 1)
ts_nn_kernel(const double* __restrict__ A, int64_t lda, int p, const double* __restrict__ C, int q, double* Out,
             int64_t ldo, int64_t n, double alpha, double beta, int vec2) {
    extern __shared__ __align__(16) unsigned char ts_smem[];
    const int steps = (p + 15) >> 4, ntiles = (q + 7) >> 3;
    uint2* cd = reinterpret_cast<uint2*>(ts_smem);                                   // [ntile][step][digit][lane]
    uint2* cb = cd + (int64_t)ntiles * steps * kDigits * 32;                         // [ntile][step][lane]: magnitudes
    int* ce = reinterpret_cast<int*>(cb + (int64_t)ntiles * steps * 32);             // exponent of column j of C
    int* cr = ce + 64;                                                               // exponent of row k of C - 1023
    int* cp = cr + 64;                                                               // row of column j's largest element
    double* cs = reinterpret_cast<double*>(cp + 64);                                 // C
    for (int i = threadIdx.x; i < p * q; i += blockDim.x) cs[i] = C[i];
    __syncthreads();
    for (int j = threadIdx.x; j < 64; j += blockDim.x) {
        uint32_t h = 0;
        int row = 0;
        if (j < q)
            for (int k = 0; k < p; ++k) {
                const uint32_t x = magnitude(cs[k * q + j]);
                if (x > h) h = x, row = k;
            }
        cp[j] = row;
    }
    __syncthreads();
    bool sub = false;                                // a subnormal element of C
    for (int k = threadIdx.x; k < 64; k += blockDim.x) {
        uint32_t h = 0;
        if (k < p)
            for (int j = 0; j < q; ++j) {
                const uint32_t x = magnitude(cs[k * q + j]);
                if (cp[j] != k) h = max(h, x);
                sub |= x != 0 && (x >> 20) == 0;
            }
        cr[k] = (h >> 20) == 0 ? kNoExp : (int)(h >> 20) - 1023;
    }
    const bool c_sub = __syncthreads_or(sub) != 0;
    for (int j = threadIdx.x; j < ntiles * 8; j += blockDim.x) {
        int e = 0;
        bool special = false, zero = true;
        if (j < q)
            for (int k = 0; k < p; ++k) {
                const uint32_t h = magnitude(cs[k * q + j]);
                const int x = (int)(h >> 20);
                special |= x == 0x7ff;
                if (cp[j] == k) continue;
                zero &= h == 0;
                if (x > 0) e = max(e, x - cr[k]);
            }
        ce[j] = special ? kSpecial : zero ? kNoExp : e;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    for (int f = warp; f < ntiles * steps; f += kTsWarps) {
        const int nt = f / steps, ks = f % steps, col = nt * 8 + g;
        uint2 y[4];
        uint32_t m[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int k = ks * 16 + 2 * t + (r & 1) + (r >> 1) * 8;
            const double c = k < p && col < q && k != cp[col] ? cs[k * q + col] : 0.0;
            y[r] = digits_of(c, ce[col] + cr[k]);
            m[r] = bf16_below(magnitude(c), ce[col] + cr[k]);
        }
        cb[f * 32 + lane] = make_uint2(m[0] | m[1] << 16, m[2] | m[3] << 16);
        uint32_t fb[kDigits][2];
        b_digits<0>(fb, y);
#pragma unroll
        for (int d = 0; d < kDigits; ++d) cd[((int64_t)f * kDigits + d) * 32 + lane] = make_uint2(fb[d][0], fb[d][1]);
    }
    __syncthreads();
    const int64_t rtiles = (n + 15) >> 4;
    // |Out| >= p 2^-4 of the scales' product: the last rounding is no less than what is left out
    const bool hides = beta == 1.0 && (alpha == 1.0 || alpha == -1.0);
    const int hidden = 1025 - (32 - __clz(p - 1));
    for (int64_t rt = (int64_t)blockIdx.x * kTsWarps + warp; rt < rtiles; rt += (int64_t)gridDim.x * kTsWarps) {
        const int64_t row0 = rt * 16 + g, row1 = row0 + 8;
        // rows past the last repeat it, columns past the last too (C's digits are zero there)
        const double *p0 = A + min(row0, n - 1) * lda, *p1 = A + min(row1, n - 1) * lda;
        // fragment columns 2t, 2t+1 and 2t+8, 2t+9 of rows g and g+8 of one 16-column step
        auto load8 = [&](int ks, double (&x)[8]) {
            const int k = ks * 16 + 2 * t;
            if (vec2) {
                const int ka = min(k, p - 2), kb = min(k + 8, p - 2);
                const double2 a = *reinterpret_cast<const double2*>(p0 + ka), b = *reinterpret_cast<const double2*>(p1 + ka);
                const double2 c = *reinterpret_cast<const double2*>(p0 + kb), d = *reinterpret_cast<const double2*>(p1 + kb);
                x[0] = a.x, x[1] = a.y, x[2] = b.x, x[3] = b.y, x[4] = c.x, x[5] = c.y, x[6] = d.x, x[7] = d.y;
            } else {
#pragma unroll
                for (int r = 0; r < 8; ++r) x[r] = ((r & 2) ? p1 : p0)[min(k + (r & 1) + (r >> 2) * 8, p - 1)];
            }
        };
        int e0 = kNoExp, e1 = kNoExp, sub0 = 0, sub1 = 0;
        uint32_t h[4][8];
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
            if (ks < steps) {
                double x[8];
                load8(ks, x);
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const int k = ks * 16 + 2 * t + (r & 1) + (r >> 2) * 8;
                    h[ks][r] = k < p ? magnitude(x[r]) : 0u;
                    const int x20 = (int)(h[ks][r] >> 20);
                    const int e = x20 == 0x7ff ? kSpecial : x20 == 0 ? kNoExp : x20 + cr[k];
                    const int sb = x20 == 0 && h[ks][r] != 0;
                    if (r & 2) e1 = max(e1, e), sub1 |= sb;
                    else e0 = max(e0, e), sub0 |= sb;
                }
            }
        }
#pragma unroll
        for (int off = 1; off < 4; off <<= 1) {
            e0 = max(e0, __shfl_xor_sync(0xffffffffu, e0, off));
            e1 = max(e1, __shfl_xor_sync(0xffffffffu, e1, off));
            sub0 |= __shfl_xor_sync(0xffffffffu, sub0, off);
            sub1 |= __shfl_xor_sync(0xffffffffu, sub1, off);
        }
        // bit 4 (tile of 8 columns) + c: that element takes FP64 arithmetic
        uint32_t fp64 = 0;
        {
            uint32_t ua[4][4];
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                if (ks < steps) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int* c = cr + ks * 16 + 2 * t + (i >> 1) * 8;
                        const int e = (i & 1) ? e1 : e0;
                        ua[ks][i] = bf16_pair(h[ks][2 * i], h[ks][2 * i + 1], e - c[0], e - c[1]);
                    }
                }
            for (int nt = 0; nt < ntiles; ++nt) {
                float low[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    if (ks < steps) {
                        const uint2 v = cb[(nt * steps + ks) * 32 + lane];
                        mma_bf16(low, ua[ks], v.x, v.y);
                    }
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int col = nt * 8 + 2 * t + (c & 1), e = c < 2 ? e0 : e1;
                    if (col < q && (c < 2 ? row0 : row1) < n &&
                        needs_fp64(low[c], e, ce[col], c_sub || (c < 2 ? sub0 : sub1)))
                        fp64 |= 1u << (4 * nt + c);
                }
            }
        }
        for (int np = 0; np < ntiles; np += 2) {
            float acc[2][kDigits][4];
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int d = 0; d < kDigits; ++d)
#pragma unroll
                    for (int c = 0; c < 4; ++c) acc[j][d][c] = 0.f;
#pragma unroll 1
            for (int ks = 0; ks < steps; ++ks) {
                double x[8];
                load8(ks, x);
                uint2 y[8];
#pragma unroll
                for (int r = 0; r < 8; ++r)
                    y[r] = digits_of(x[r], ((r & 2) ? e1 : e0) - cr[ks * 16 + 2 * t + (r & 1) + (r >> 2) * 8]);
                uint32_t fa[kDigits][4];
                a_digits<0>(fa, y);
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    if (np + j < ntiles) {
                        uint32_t fb[kDigits][2];
                        const uint2* src = cd + ((int64_t)((np + j) * steps + ks) * kDigits) * 32 + lane;
#pragma unroll
                        for (int d = 0; d < kDigits; ++d) {
                            const uint2 v = src[d * 32];
                            fb[d][0] = v.x;
                            fb[d][1] = v.y;
                        }
                        mma_digits(acc[j], fa, fb);
                    }
            }
#pragma unroll
            for (int j = 0; j < 2; ++j)
                if (np + j < ntiles) {
                    const int col = (np + j) * 8 + 2 * t;
                    double v[4], o[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int64_t row = min(c < 2 ? row0 : row1, n - 1);
                        o[c] = beta != 0.0 ? Out[row * ldo + min(col + (c & 1), q - 1)] : 0.0;
                    }
                    uint32_t f64 = fp64 >> (4 * (np + j)) & 15u;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int e = c < 2 ? e0 : e1, ec = ce[col + (c & 1)], top = cp[col + (c & 1)];
                        const double a = (c < 2 ? p0 : p1)[top], d = cs[top * q + min(col + (c & 1), q - 1)];
                        v[c] = fma(a, d, from_diagonals(acc[j], c, e, ec));
                        // hidden behind the largest product (or a zero factor, exponent field 0: not), or behind Out
                        const int xa = (int)(magnitude(a) >> 20), xd = (int)(magnitude(d) >> 20);
                        if (!c_sub && !(c < 2 ? sub0 : sub1) && e + ec >= 1090 && e + ec <= 3061 &&
                            ((xa > 0 && xd > 0 && xa + xd >= e + ec - 3) ||
                             (hides && (int)(magnitude(o[c]) >> 20) >= e + ec - hidden)))
                            f64 &= ~(1u << c);
                    }
                    // the warp's elements in need, one a lane: the FP64 units take as long for one as for 32
                    uint32_t need[4];
                    int first[5] = {0, 0, 0, 0, 0};
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        need[c] = __ballot_sync(0xffffffffu, f64 >> c & 1);
                        first[c + 1] = first[c] + __popc(need[c]);
                    }
#pragma unroll 1
                    for (int base = 0; base < first[4]; base += 32) {
                        const int i = base + lane;
                        double f = 0.0;
                        if (i < first[4]) {
                            int c = 0;
                            uint32_t mask = need[0], nth = i + 1;
#pragma unroll
                            for (int u = 1; u < 4; ++u)
                                if (i >= first[u]) c = u, mask = need[u], nth = i - first[u] + 1;
                            const int src = __fns(mask, 0, nth);         // the lane whose element it is
                            const double* a = A + (rt * 16 + (src >> 2) + (c < 2 ? 0 : 8)) * lda;
                            const double* cc = cs + (np + j) * 8 + 2 * (src & 3) + (c & 1);
#pragma unroll 4
                            for (int k = 0; k < p; ++k) f = fma(a[k], cc[k * q], f);
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int at = first[u] + __popc(need[u] & ((1u << lane) - 1u)) - base;
                            const double mine = __shfl_sync(0xffffffffu, f, at & 31);
                            if ((f64 >> u & 1) && at >= 0 && at < 32) v[u] = mine;
                        }
                    }
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        if (alpha != 1.0) v[c] = alpha == -1.0 ? -v[c] : alpha * v[c];
                        if (beta != 0.0) v[c] = (beta == 1.0 ? o[c] : beta * o[c]) + v[c];
                    }
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int64_t row = c < 2 ? row0 : row1;
                        if (row < n && col + (c & 1) < q) Out[row * ldo + col + (c & 1)] = v[c];
                    }
                }
        }
    }
}

// partial[block][j] = sum of (AU - theta U)^2 over the block's rows: thread t
// keeps column t % q (256 / q rows at a time), its rows' strands are added in
// order.
constexpr int kResidualBlocks = 4;
__global__ void __launch_bounds__(256) ts_residual_kernel(const double* __restrict__ AU, const double* __restrict__ U,
                                                          const double* __restrict__ theta, int q, int64_t n,
                                                          double* __restrict__ partial) {
    __shared__ double sh[256];
    const int strands = 256 / q, j = threadIdx.x % q, strand = threadIdx.x / q;
    double s = 0.0;
    if (strand < strands) {
        const double th = theta[j];
#pragma unroll 4
        for (int64_t i = (int64_t)blockIdx.x * strands + strand; i < n; i += (int64_t)gridDim.x * strands) {
            const double r = fma(-th, U[i * q + j], AU[i * q + j]);
            s = fma(r, r, s);
        }
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.x < q) {
        double a = 0.0;
        for (int k = 0; k < strands; ++k) a += sh[k * q + threadIdx.x];
        partial[(int64_t)blockIdx.x * q + threadIdx.x] = a;
    }
}

int sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 1;
    return std::max(1, sms);
}

size_t nn_smem(int p, int q) {
    const int steps = (p + 15) / 16, ntiles = (q + 7) / 8;
    return (size_t)ntiles * steps * (kDigits + 1) * 32 * sizeof(uint2) + 3 * 64 * sizeof(int) + (size_t)p * q * sizeof(double);
}

// row groups of one ts_tn launch: one warp per unit and group, a wave of blocks
int tn_groups(int64_t n, int units) {
    const int64_t tiles = (n + kTsRows - 1) / kTsRows;
    return (int)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)sm_count() * kTsWarps / units));
}

}  // namespace

size_t ts_partial_doubles(int64_t n, int m) {
    // groups x p x q: groups x units fills the launch's warps and a unit has at most 256 elements (512 with
    // its mirror image when A is B); ts_residuals writes one row of q per block
    const size_t tiles = (size_t)((n + kTsRows - 1) / kTsRows), mm = (size_t)m * m;
    const size_t wave = std::max(mm, (size_t)sm_count() * kTsWarps * 512);
    return std::max((size_t)sm_count() * kResidualBlocks * m, std::min(std::max<size_t>(tiles, 1) * mm, wave));
}

cudaError_t ts_tn(const double* A, int64_t lda, int p, const double* B, int64_t ldb, int q, int64_t n,
                  double* partial, double* out, cudaStream_t s) {
    const int mt = (p + 15) / 16, nt = (q + 15) / 16;
    const bool same = A == B && lda == ldb && p == q;
    const int units = same ? mt * (mt + 1) / 2 : mt * nt;
    const int kg = tn_groups(n, units);
    const unsigned grid = (unsigned)((kg * units + kTsWarps - 1) / kTsWarps);
    if (same) ts_tn_kernel<true><<<grid, kTsWarps * 32, 0, s>>>(A, lda, p, B, ldb, q, n, nt, units, kg, partial);
    else ts_tn_kernel<false><<<grid, kTsWarps * 32, 0, s>>>(A, lda, p, B, ldb, q, n, nt, units, kg, partial);
    ts_reduce_kernel<<<(p * q + 7) / 8, 256, 0, s>>>(partial, kg, p * q, out);
    return cudaGetLastError();
}

cudaError_t ts_nn(const double* A, int64_t lda, int p, const double* C, int q, double* Out, int64_t ldo, int64_t n,
                  double alpha, double beta, cudaStream_t s) {
    const size_t smem = nn_smem(p, q);
    // the attribute is the current device's: set where this launch needs it
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(ts_nn_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const int64_t rtiles = (n + 15) / 16;
    const unsigned grid =
        (unsigned)std::max<int64_t>(1, std::min<int64_t>((rtiles + kTsWarps - 1) / kTsWarps, sm_count()));
    const int vec2 = p % 2 == 0 && lda % 2 == 0 && ((uintptr_t)A & 15) == 0;
    ts_nn_kernel<<<grid, kTsWarps * 32, smem, s>>>(A, lda, p, C, q, Out, ldo, n, alpha, beta, vec2);
    return cudaGetLastError();
}

cudaError_t ts_residuals(const double* AU, const double* U, const double* theta, int q, int64_t n, double* partial,
                         double* out, cudaStream_t s) {
    const int blocks = sm_count() * kResidualBlocks;
    ts_residual_kernel<<<blocks, 256, 0, s>>>(AU, U, theta, q, n, partial);
    ts_reduce_kernel<<<(q + 7) / 8, 256, 0, s>>>(partial, blocks, q, out);
    return cudaGetLastError();
}

}  // namespace spmm
