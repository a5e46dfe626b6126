// gfip_ozaki.cu -- FP64 GEMM emulated on the tcgen05 tensor cores with exact BF16 digit
// products (the Ozaki splitting scheme: Ozaki, Ogita, Oishi, Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix multiplication
// and its applications", Numer. Algorithms 59 (2012); here with BF16 digits and FP32
// accumulation).
//
// Splitting (a pack-time transform, like the slicing that the GEMMFIP paper's future work,
// Sec. 5, folds into packing): every row i of op(A) gets an exponent e_i with
// max_p |a_ip| < 2^e_i, and every element becomes exactly
//     a_ip = 2^(e_i + 1) * (sum_{s=1..S} d_s * 2^(-6 s) + r),   |d_s| <= 32,
// with integer digits d_s (exact in BF16) and |r| <= 2^(-6 S - 1) (the scaled element is below
// 1/2, so even the first digit is at most 32).  Columns of op(B) are split the same way with
// exponents f_j.  A product of two digits is an integer of at most 2^10, so a sum of up to
// 16384 of them is an integer of at most 2^24 and the tensor cores' FP32 accumulation of it
// is exact.  The result is
//     C_ij = alpha * 2^(e_i + f_j + 2) * sum_{s+t <= S+1} 2^(-6(s+t)) * sum_p d_s d_t
//            + beta * C_ij,
// dropping the digit pairs with s + t > S + 1 (triangular truncation).  The tile core
// (gfip_tc.cuh) sums the digit products; while the whole sum fits 63 bits it is formed
// exactly as an integer and rounded to FP64 once, else the exact sums of four classes s + t
// and one k chunk are added in FP64.
#include <cstdint>

#include "gfip_tc.cuh"

namespace gfip {
namespace oz {

using tc::KB;
using tc::PLANE_BYTES;
using tc::TM;

// e with max_p |x_rp| < 2^e for each row r, by atomicMax into exp[] (preset below every
// exponent).  Block (rb, ks) of an operand covers rows rb*128 .. +127 and the ks-th of its
// equal k-ranges.  Row r of the operand has element (r, p) at X[r + p*ld] when contig_rows,
// else X[p + r*ld].  One launch covers both operands.  Bound by HBM: each element is read once.
struct ExpArgs {
    const double *X;
    int64_t ld;
    int rows, contig_rows, row_blocks, ks;
    int *exp;
};

// |x| as an integer with the same order as the magnitudes of finite doubles.
__device__ __forceinline__ unsigned long long mag_bits(double x)
{
    return static_cast<unsigned long long>(__double_as_longlong(x)) & 0x7FFFFFFFFFFFFFFFull;
}

constexpr int NO_EXP = -0x7F7F7F80;   // four bytes 0x80: the preset

// e with |x| < 2^e for the double whose magnitude bits are b (NO_EXP for zero).
__device__ __forceinline__ int exp_of(unsigned long long b)
{
    if (b == 0) return NO_EXP;
    const int ex = static_cast<int>(b >> 52);
    if (ex == 0) return -1074 + 64 - __clzll(static_cast<long long>(b));  // subnormal
    return ex - 1022;   // |x| = 1.f * 2^(ex-1023) < 2^(ex-1022)
}

__global__ void __launch_bounds__(256) exponent_kernel(ExpArgs a, ExpArgs b, int kdim)
{
    __shared__ unsigned long long red[256];
    const int tid = threadIdx.x;
    const int a_blocks = a.row_blocks * a.ks;
    int blk = blockIdx.x;
    if (blk >= a_blocks) {
        blk -= a_blocks;
        a = b;
    }
    const int rb = blk % a.row_blocks, ks = blk / a.row_blocks;
    const int kr = (kdim + a.ks - 1) / a.ks;
    const int p0 = ks * kr, p1 = min(kdim, p0 + kr);
    const int r0 = rb * TM;
    if (a.contig_rows) {
        // two threads per row, consecutive rows in consecutive threads
        const int r = r0 + (tid % TM);
        unsigned long long mx = 0;
        if (r < a.rows) {
#pragma unroll 8
            for (int p = p0 + tid / TM; p < p1; p += 2) {
                const unsigned long long v = mag_bits(a.X[r + (int64_t)p * a.ld]);
                mx = v > mx ? v : mx;
            }
        }
        red[tid] = mx;
        __syncthreads();
        if (tid < TM) {
            const unsigned long long u = red[tid], v = red[tid + TM];
            atomicMax(a.exp + r0 + tid, exp_of(u > v ? u : v));
        }
    } else {
        // one warp per row, lanes along the contiguous k
        const int lane = tid & 31, w = tid >> 5;
        for (int rr = w; rr < TM; rr += 8) {
            const int r = r0 + rr;
            unsigned long long mx = 0;
            if (r < a.rows) {
#pragma unroll 4
                for (int p = p0 + lane; p < p1; p += 32) {
                    const unsigned long long v = mag_bits(a.X[p + (int64_t)r * a.ld]);
                    mx = v > mx ? v : mx;
                }
            }
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
                mx = v > mx ? v : mx;
            }
            if (lane == 0) atomicMax(a.exp + r, exp_of(mx));
        }
    }
}

// x * 2^-(e+1) as a signed fixed-point number with 63 fractional bits, truncated toward zero
// (|x| < 2^e, so the result is below 2^62 in magnitude).  Integer operations on the IEEE bit
// pattern only.  For an integer x the truncation drops nothing.
__device__ __forceinline__ long long to_fixed(double x, int e)
{
    const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(x));
    const int ex = static_cast<int>((bits >> 52) & 0x7FF);
    long long mant = static_cast<long long>(bits & 0xFFFFFFFFFFFFFull);
    int ee = ex;
    if (ex == 0) ee = 1; else mant |= 1ll << 52;   // x = +-mant * 2^(ee - 1075)
    const int sh = ee - 1075 + 62 - e;              // x * 2^(62 - e) = mant * 2^sh
    long long v;
    if (sh >= 0) v = mant << sh;
    else v = (sh > -64) ? (mant >> -sh) : 0;
    return (bits >> 63) ? -v : v;
}

// Digit planes of one 128 x 32 block of an operand.  The block is read coalesced into shared
// memory; each thread then takes 8 consecutive k of one row and writes one 16-byte chunk per
// digit, consecutive threads consecutive chunks of the plane tile.
//
// With X the 63-bit fixed-point copy of an element and w_s = 2^(63-6s), digit s is X's
// remainder below w_(s-1) (its low bits, sign-extended) rounded to a multiple of w_s: the 6-bit
// field of X at w_s taken as a signed number, plus the bit below it.  So no digit waits for
// another, and as 128 + i is the BF16 number with fraction i (i < 128), a pair of digits is
// two field extractions and one exact BF16 subtraction of 160.  (The remainders formed one
// after the other in 64-bit arithmetic took 190 us an operand at 4096 x 4096, seven digits; this
// takes 71, 0.34 GB of it HBM traffic.)
struct SplitArgs {
    const double *X;
    int64_t ld;
    int rows, contig_rows, row_blocks;
    const int *exp;
    uint8_t *planes;
};

constexpr int SPITCH = TM + 1;

__global__ void __launch_bounds__(256) split_kernel(SplitArgs a, SplitArgs b, int kdim,
                                                    int kblocks, int S)
{
    __shared__ double tile[KB * SPITCH];   // element (r, c) at c * SPITCH + r
    const int tid = threadIdx.x;
    int64_t blk = blockIdx.x;
    if (blk >= (int64_t)a.row_blocks * kblocks) {
        blk -= (int64_t)a.row_blocks * kblocks;
        a = b;
    }
    const int rb = static_cast<int>(blk % a.row_blocks), kb = static_cast<int>(blk / a.row_blocks);
    constexpr int PER = TM * KB / 256;   // 16 elements per thread
    double v[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int r = a.contig_rows ? tid % TM : tid / KB + 8 * q;
        const int c = a.contig_rows ? tid / TM + 2 * q : tid % KB;
        const int gr = rb * TM + r, gc = kb * KB + c;
        const int64_t at = a.contig_rows ? gr + (int64_t)gc * a.ld : gc + (int64_t)gr * a.ld;
        v[q] = (gr < a.rows && gc < kdim) ? a.X[at] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int r = a.contig_rows ? tid % TM : tid / KB + 8 * q;
        const int c = a.contig_rows ? tid / TM + 2 * q : tid % KB;
        tile[c * SPITCH + r] = v[q];
    }
    __syncthreads();
    uint8_t *dst = a.planes + ((int64_t)rb * kblocks + kb) * S * PLANE_BYTES;
#pragma unroll 1
    for (int o = tid; o < TM * 4; o += 256) {
        const int r = o >> 2, chunk = (o & 3) ^ ((r >> 1) & 3);
        const int ex = a.exp[rb * TM + r];
        const int e = ex == NO_EXP ? 0 : ex;
        long long y[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) y[i] = to_fixed(tile[(chunk * 8 + i) * SPITCH + r], e);
        for (int s = 1; s <= S; ++s) {
            const int sh = 62 - 6 * s;   // the bit below the digit's field
            uint32_t w[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                // field + 32 (its sign bit flipped) and the bit below it, then their sum
                const uint32_t lo = (static_cast<uint32_t>(y[2 * h] >> sh) & 0x7Fu) ^ 0x40u;
                const uint32_t hi = (static_cast<uint32_t>(y[2 * h + 1] >> sh) & 0x7Fu) ^ 0x40u;
                const uint32_t sum = ((lo | (hi << 16)) + 0x00010001u) >> 1;
                const uint32_t bits = (sum & 0x007F007Fu) | 0x43004300u;   // 160 + digit
                __nv_bfloat162 d;
                *reinterpret_cast<uint32_t *>(&d) = bits;
                d = __hsub2(d, __float2bfloat162_rn(160.f));
                w[h] = *reinterpret_cast<const uint32_t *>(&d);
            }
            *reinterpret_cast<uint4 *>(dst + (s - 1) * PLANE_BYTES + o * 16) =
                make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

}  // namespace oz

cudaError_t launch_ozaki(const OzakiParams &p, int sms, cudaStream_t s)
{
    // every row's exponent starts below all exponents (bytes 0x80)
    const int64_t rows_pad = (int64_t)(p.mt + p.nt) * tc::TM;
    cudaError_t e = cudaMemsetAsync(p.exp, 0x80, rows_pad * sizeof(int), s);
    if (e != cudaSuccess) return e;
    int *ea = p.exp, *eb = p.exp + (int64_t)p.mt * tc::TM;
    const oz::ExpArgs xa{p.A, p.lda, p.m, p.a_contig_rows, p.mt, p.ks_a, ea};
    const oz::ExpArgs xb{p.B, p.ldb, p.n, p.b_contig_rows, p.nt, p.ks_b, eb};
    oz::exponent_kernel<<<p.mt * p.ks_a + p.nt * p.ks_b, 256, 0, s>>>(xa, xb, p.k);
    const oz::SplitArgs sa{p.A, p.lda, p.m, p.a_contig_rows, p.mt, ea, p.pa};
    const oz::SplitArgs sb{p.B, p.ldb, p.n, p.b_contig_rows, p.nt, eb, p.pb};
    oz::split_kernel<<<(p.mt + p.nt) * p.kt, 256, 0, s>>>(sa, sb, p.k, p.kt, p.slices);
    TcParams t{};
    t.pa = p.pa;
    t.pb = p.pb;
    t.C = p.C;
    t.ldc = p.ldc;
    t.m = p.m;
    t.n = p.n;
    t.alpha = p.alpha;
    t.beta = p.beta;
    t.planes = p.slices;
    t.mt = p.mt;
    t.nt = p.nt;
    t.kt = p.kt;
    t.tiles = p.mt * p.nt;
    t.splits = 1;
    t.units = t.tiles;
    t.ea = ea;
    t.eb = eb;
    t.status = p.status;
    t.wait_ns = p.wait_ns;
    t.inject_timeout = p.inject_timeout;
    // |sum| <= k / 4 in units of 2^0, its last digit weighs 2^(-6 (S + 1)): exact in 63 bits
    // while 6 (S + 1) - 2 + log2(k) <= 62
    int bits = 6 * (p.slices + 1) - 2;
    for (int64_t q = 1; q < p.k; q *= 2) ++bits;
    return bits <= 62 ? tc::launch<tc::KIND_DIGITS_INT>(t, sms, s)
                      : tc::launch<tc::KIND_DIGITS_F64>(t, sms, s);
}

}  // namespace gfip
