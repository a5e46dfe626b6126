// gfip_f32_tc.cu -- large FP32 GEMMs on the tensor cores: operands split into three BF16 planes.
//
// x = x1 + x2 + x3 with x1 = BF16(x), x2 = BF16(x - x1), x3 = x - x1 - x2, exactly: each rounding to
// nearest leaves a remainder of at most 2^-8 of what it rounded, and 24 significant bits fit
// three planes of 8.  The tile core (gfip_tc.cuh) forms a1 b1 + (a1 b2 + a2 b1 + a1 b3 + a2 b2 +
// a3 b1 + a2 b3 + a3 b2); the one product left out, a3 b3, is at most 2^-32 of |a b|, a 256th of
// half an ulp, so a sum that one product dominates comes out rounded as a multiply-add rounds it.
// (Without a2 b3 + a3 b2, up to 2^-24 of |a b|, 4 % of such sums were an ulp off and the worst
// error was 1.7 times a multiply-add's; the two products cost 4096^3 20 %.)  a1 b1 and the
// smaller products are accumulated apart, for 32 to 128 k at a time (launch_tc in gfip_api.cu),
// and the chunks are added in FP32 with rounding to nearest, which keeps the sum at least as
// exact as the FFMA core's chains of FP32 multiply-adds, also where all terms have one sign.
// Packing is where the split happens: one pass reads the strided operands (masking triangular
// ones) and writes the plane tiles the MMA reads.
//
// Every element is zero or of magnitude in [2^-100, 2^47), k at most 2^17: the planes are exact
// and normal BF16 numbers, and no sum overflows.  Products may lie below FP32's normal range,
// where the tensor cores' sums lose up to an ulp, 2^-149, a step; so the operands are scaled by
// powers of two, 256 together, and the sum is scaled back, rounded once, at its end: what is lost
// weighs 2^-157 a step, where a chain of multiply-adds rounds to 2^-149 each time.  (Unscaled,
// 700 x 690 x 660 of operands near 2^-65 was off by 95 x 2^-149, the FFMA core by 37.)  An element
// outside (NaN and infinities among them) sets the gate word; the tile core then does nothing and
// the FFMA launch that follows computes the product, as it would without this path.
#include <cstdint>

#include "gfip_kernels.cuh"
#include "gfip_tc.cuh"

namespace gfip {
namespace f32tc {

using tc::KB;
using tc::PLANE_BYTES;
using tc::TM;

constexpr int PITCH = TM + 1;

// Planes of one 128 x 32 block of an operand (one launch covers both).  The block is read
// coalesced into shared memory; each thread then takes 8 consecutive k of one row and writes
// one 16-byte chunk per plane, consecutive threads consecutive chunks.  Bound by HBM: 4 bytes
// read and 6 written per element (both operands of 4096^3: 335 MB in 63 us).
__global__ void __launch_bounds__(256) split_kernel(F32SplitArgs a, F32SplitArgs b, int kdim,
                                                    int kblocks, unsigned int *counter,
                                                    int counters, unsigned int *gate)
{
    __shared__ float tile[KB * PITCH];   // element (r, c) at c * PITCH + r
    const int tid = threadIdx.x;
    // arrival counters of split tiles start at zero
    for (int64_t c = (int64_t)blockIdx.x * 256 + tid; c < counters; c += (int64_t)gridDim.x * 256)
        counter[c] = 0u;
    int64_t blk = blockIdx.x;
    if (blk >= (int64_t)a.row_blocks * kblocks) {
        blk -= (int64_t)a.row_blocks * kblocks;
        a = b;
    }
    const int rb = static_cast<int>(blk % a.row_blocks), kb = static_cast<int>(blk / a.row_blocks);
    const int cls = tmask_class(a.mask, rb * TM, TM, kb * KB, KB);
    if (cls == 2) return;   // wholly outside the triangle: no tile reads it
    constexpr int PER = TM * KB / 256;
    float v[PER];
    bool bad = false;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int r = a.contig_rows ? tid % TM : tid / KB + 8 * q;
        const int c = a.contig_rows ? tid / TM + 2 * q : tid % KB;
        const int gr = rb * TM + r, gc = kb * KB + c;
        const int64_t at = a.contig_rows ? gr + (int64_t)gc * a.ld : gc + (int64_t)gr * a.ld;
        const bool in = gr < a.rows && gc < kdim && (cls == 0 || tmask_keep(a.mask, gr, gc));
        v[q] = in ? a.X[at] : 0.f;
    }
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int r = a.contig_rows ? tid % TM : tid / KB + 8 * q;
        const int c = a.contig_rows ? tid / TM + 2 * q : tid % KB;
        bad = bad || tc::outside_split(v[q]);
        tile[c * PITCH + r] = v[q];
    }
    if (__syncthreads_or(bad)) {
        if (tid == 0) atomicOr(gate, 1u);
        return;   // the planes will not be used
    }
    uint8_t *dst = a.planes + ((int64_t)rb * kblocks + kb) * 3 * PLANE_BYTES;
#pragma unroll
    for (int o = tid; o < TM * 4; o += 256) {
        const int r = o >> 2, chunk = (o & 3) ^ ((r >> 1) & 3);
        const float *src = tile + chunk * 8 * PITCH + r;
        uint32_t p[3][4];
#pragma unroll
        for (int h = 0; h < 4; ++h)
            tc::split_pair(a.scale * src[2 * h * PITCH], a.scale * src[(2 * h + 1) * PITCH],
                           p[0][h], p[1][h], p[2][h]);
#pragma unroll
        for (int s = 0; s < 3; ++s)
            *reinterpret_cast<uint4 *>(dst + s * PLANE_BYTES + o * 16) =
                make_uint4(p[s][0], p[s][1], p[s][2], p[s][3]);
    }
}

}  // namespace f32tc

cudaError_t launch_f32_split(const F32SplitArgs &a, int k, int kt, unsigned int *gate,
                             cudaStream_t s)
{
    F32SplitArgs none{};
    f32tc::split_kernel<<<static_cast<unsigned int>((int64_t)a.row_blocks * kt), 256, 0, s>>>(
        a, none, k, kt, nullptr, 0, gate);
    return cudaGetLastError();
}

cudaError_t launch_f32_tc(const TcParams &p, const F32SplitArgs &a, const F32SplitArgs &b, int k,
                          unsigned int *gate, int sms, cudaStream_t s)
{
    const int64_t blocks = (int64_t)(a.row_blocks + b.row_blocks) * p.kt;
    f32tc::split_kernel<<<static_cast<unsigned int>(blocks), 256, 0, s>>>(
        a, b, k, p.kt, p.counter, p.splits > 1 ? p.tiles * tc::EPI_WARPS : 0, gate);
    return tc::launch<tc::KIND_F32>(p, sms, s);
}

}  // namespace gfip
