// gfip_f32_skinny.cu -- large FP32 products with at most 128 rows or columns, on the tensor cores.
//
// For large operands whose rows (of op(A), or columns of op(B)) run along memory.  Each of their
// elements meets one tile line of C only, so a packed copy of it would
// be read once (the option table of Sec. 3.3 packs no such operand): here it is read where it
// lies and split into its BF16 planes (see gfip_f32_tc.cu) on the way to the MMA.  The small
// operand is split beforehand.  At 64 x 8192 x 8192 the split pass over the large operand and the
// reads of its planes were 1.1 GB of traffic for 268 MB of operand, 207 us.
//
// One CTA per SM, persistent over units (128 rows of the large operand x a range of k):
//   warp 0     copies the small operand's planes (three bulk copies a k block);
//   warp 1     issues the MMAs: the large operand's 128 rows are the MMA's M, the small
//              operand's rows (16 to 128) its N; accumulators as in gfip_tc.cuh;
//   warps 2-17 read the large operand three k blocks ahead into registers, split and store it to
//              the stage as the MMA reads it; drain the accumulators a chunk behind; store the
//              unit's partial sums.  (Eight such warps, with twice the elements each, were 20 %
//              slower; two groups of eight taking turns at the blocks, 35 %.)
// Partial sums of all k ranges are added, in order, by a launch of its own, which also applies
// alpha and beta: C is untouched when an element outside the range of the split turned up and
// the FFMA launch behind has to compute the product.  Every CTA then stops at its next look.
//
// Measured: 64 x 8192 x 8192 207 us from planes -> 120 to 129 here.
// Bound: the latencies of the split (about 1550 clocks a block, for 600 of its instructions, 770
// of MMAs and shared-memory traffic, and 600 of HBM at full rate).
#include <cstdint>

#include "gfip_tc.cuh"

namespace gfip {
namespace skinny {

using tc::KB;
using tc::PLANE_BYTES;
using tc::TM;

constexpr int PLANES = 3;
constexpr int STAGES = 4;
constexpr int DEPTH = 3;           // k blocks of the large operand in registers
constexpr int SPLIT_WARPS = 16;
constexpr int THREADS = 64 + SPLIT_WARPS * 32;
constexpr int PER = 8;             // its elements per thread and block
static_assert(SPLIT_WARPS * 32 * PER == TM * KB, "a block");
static_assert(2 * PLANES * STAGES <= tc::SLOTS && STAGES <= tc::MAX_BSTAGES, "stages fit");

struct Unit {
    int tile, kb0, kb1;
};

__device__ __forceinline__ Unit unit_of(const SkinnyParams &p, int u)
{
    const int split = u / p.tiles;
    return Unit{u - split * p.tiles, static_cast<int>((int64_t)p.kt * split / p.splits),
                static_cast<int>((int64_t)p.kt * (split + 1) / p.splits)};
}

// Stage layout: planes of the large operand, then of the small one.
__device__ __forceinline__ uint8_t *big_plane(tc::Smem &sm, int stage, int s)
{
    return sm.plane[stage * 2 * PLANES + s];
}

__device__ void producer(const SkinnyParams &p, tc::Smem &sm)
{
    const bool leader = tc::elect_one();
    const uint32_t bytes = p.n16 * KB * 2;   // the rows of a plane that are used
    int stage = 0;
    uint32_t lap = 0;
    bool ok = true;
    bool skip = p.inject_timeout && blockIdx.x == 0;   // test hook: the first block never arrives
    for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
        const Unit x = unit_of(p, u);
        const uint8_t *src = p.planes + (int64_t)x.kb0 * PLANES * PLANE_BYTES;
        for (int kb = x.kb0; kb < x.kb1; ++kb, src += PLANES * PLANE_BYTES) {
            // another CTA met an element outside the range: stop (no wait has run out)
            if ((kb & 7) == 7 && leader && *(volatile const unsigned int *)p.gate != 0u)
                tc::set_aborted(sm);
            ok = tc::mbar_wait(&sm.aempty[stage], (lap & 1u) ^ 1u, sm, p.status, p.wait_ns);
            if (!ok) break;
            if (leader && !skip) {
                tc::mbar_expect_tx(&sm.bfull[stage], PLANES * bytes);
                for (int s = 0; s < PLANES; ++s)
                    tc::bulk_copy(big_plane(sm, stage, PLANES + s), src + s * PLANE_BYTES, bytes,
                                  &sm.bfull[stage]);
            }
            skip = false;
            if (++stage == STAGES) {
                stage = 0;
                ++lap;
            }
        }
    }
    // no copy may outlive the CTA
    for (int i = 0; i < STAGES; ++i)
        if (i < stage || lap > 0)
            tc::mbar_wait_drain(&sm.bfull[i], (i < stage ? lap : lap - 1) & 1u, p.wait_ns);
}

__device__ __forceinline__ void mma(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc,
                                    uint32_t accumulate)
{
#pragma unroll
    for (int kk = 0; kk < KB / 16; ++kk)
        asm volatile(
            "{\n .reg .pred p;\n .reg .b64 a, b;\n mov.b64 a, {%1, %5};\n mov.b64 b, {%2, %5};\n"
            " setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n}" ::"r"(d),
            "r"(a + 2 * kk), "r"(b + 2 * kk), "r"(idesc), "r"(kk ? 1u : accumulate),
            "n"(tc::DESC_HIGH)
            : "memory");
}

__device__ void issuer(const SkinnyParams &p, tc::Smem &sm, uint32_t tmem)
{
    const bool leader = tc::elect_one();
    const uint32_t idesc = (tc::IDESC<128> & ~(0x3Fu << 17)) | ((uint32_t)(p.n16 >> 3) << 17);
    int stage = 0;
    uint32_t phase = 0, chunks = 0;
    bool ok = true;
    const uint32_t base = tc::desc_low(tc::saddr(sm.plane[0]));
    for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
        const Unit x = unit_of(p, u);
        for (int k0 = x.kb0; k0 < x.kb1 && ok; k0 += p.chunk, ++chunks) {
            const int k1 = min(x.kb1, k0 + p.chunk);
            const uint32_t buf = chunks & 1u;
            ok = tc::mbar_wait(&sm.tempty[buf], ((chunks >> 1) & 1u) ^ 1u, sm, p.status,
                               p.wait_ns);
            if (!ok) break;
            tc::tc_fence_after();
            const uint32_t d = tmem + buf * 256;
            uint32_t accumulate = 0;
            for (int kb = k0; kb < k1; ++kb) {
                // both operands' planes: the copies', and the splitting warps'
                ok = tc::mbar_wait(&sm.bfull[stage], phase, sm, p.status, p.wait_ns) &&
                     tc::mbar_wait(&sm.afull[stage], phase, sm, p.status, p.wait_ns);
                if (!ok) break;
                tc::tc_fence_after();
                if (leader) {
                    const uint32_t a1 = base + stage * 2 * PLANES * tc::PLANE_DESC;
                    const uint32_t a2 = a1 + tc::PLANE_DESC, a3 = a2 + tc::PLANE_DESC;
                    const uint32_t b1 = a3 + tc::PLANE_DESC, b2 = b1 + tc::PLANE_DESC;
                    mma(d, a1, b1, idesc, accumulate);
                    mma(d + 128, a1, b2, idesc, accumulate);
                    mma(d + 128, a1, b2 + tc::PLANE_DESC, idesc, 1u);
                    mma(d + 128, a2, b1, idesc, 1u);
                    mma(d + 128, a2, b2, idesc, 1u);
                    mma(d + 128, a2, b2 + tc::PLANE_DESC, idesc, 1u);
                    mma(d + 128, a3, b1, idesc, 1u);
                    mma(d + 128, a3, b2, idesc, 1u);
                    tc::mma_commit(&sm.aempty[stage]);
                }
                accumulate = 1;
                if (++stage == STAGES) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
            if (ok && leader) tc::mma_commit(&sm.tfull[buf]);
        }
    }
    if (leader) tc::mma_commit(&sm.drain);
    tc::mbar_wait_drain(&sm.drain, 0, p.wait_ns);
}

// Thread t takes 8 k of row t % 128 of a block: lanes along the contiguous rows.
struct Block {
    int row, k;
    __device__ __forceinline__ explicit Block(int t) : row(t & (TM - 1)), k((t >> 7) * PER) {}

    // left: how many of the k exist (the pointer runs: eight offsets kept would spill)
    __device__ __forceinline__ void load(const float *src, int64_t ld, int64_t left,
                                         float (&v)[PER]) const
    {
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            v[i] = i < left ? __ldg(src) : 0.f;
            src += ld;
            asm volatile("" : "+l"(src));
        }
    }

    // Splits the elements and stores them to the stage's planes.
    __device__ __forceinline__ void store(uint8_t *plane, const float (&v)[PER], uint32_t &high,
                                          uint32_t &low) const
    {
        uint32_t q[PLANES][PER / 2];
#pragma unroll
        for (int h = 0; h < PER / 2; ++h) {
            const float e0 = v[2 * h], e1 = v[2 * h + 1];
            const uint32_t m0 = __float_as_uint(e0) & 0x7FFFFFFFu;
            const uint32_t m1 = __float_as_uint(e1) & 0x7FFFFFFFu;
            high = max(high, max(m0, m1));
            low = min(low, min(m0 - 1u, m1 - 1u));   // a zero wraps around
            tc::split_pair(e0, e1, q[0][h], q[1][h], q[2][h]);
        }
#pragma unroll
        for (int s = 0; s < PLANES; ++s)
            *reinterpret_cast<uint4 *>(plane + s * PLANE_BYTES + tc::plane_off(row, k)) =
                make_uint4(q[s][0], q[s][1], q[s][2], q[s][3]);
    }
};

// An element met so far lies outside the range of the split.
__device__ __forceinline__ bool outside(uint32_t high, uint32_t low)
{
    return high >= tc::HIGH_BITS || low < tc::LOW_BITS - 1u;
}

// A wait that gives up has raised the abort flag, and every later one returns at once; the unit
// is run to its end all the same (its result is invalid, its accesses are the same), so that the
// lanes of a warp stay together for the warp-wide instructions, and the warp leaves after it.  (A
// vote of the lanes behind every drain's wait took 6 % of the kernel.)
__device__ void splitter(const SkinnyParams &p, tc::Smem &sm, uint32_t tmem)
{
    const int t = threadIdx.x - 64, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int quarter = warp & 3, part = (warp - 2) >> 2;   // tensor-memory lanes and columns
    const int cols = p.n16 / 4;              // accumulator columns of this part
    const Block mine(t);
    const int lag = p.chunk > 2 ? 2 : 1;
    int stage = 0;
    uint32_t lap = 0;
    uint32_t drained = 0;                    // chunks drained, over all units
    uint32_t high = 0, low = ~0u;            // largest magnitude, smallest nonzero one less 1 (bits)
    bool ok = true;
    for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
        const Unit x = unit_of(p, u);
        const int len = x.kb1 - x.kb0;
        float acc[32];
#pragma unroll
        for (int c = 0; c < 32; ++c) acc[c] = 0.f;
        int chunks = 0;   // of this unit drained
        auto drain_to = [&](int want) {
            for (; chunks < want; ++chunks, ++drained) {
                const uint32_t buf = drained & 1u;
                ok &= tc::mbar_wait(&sm.tfull[buf], (drained >> 1) & 1u, sm, p.status, p.wait_ns);
                tc::tc_fence_after();
                const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + buf * 256 +
                                       (uint32_t)(part * cols);
#pragma unroll
                for (int h = 0; h < 8; ++h) {
                    if (h * 4 >= cols) break;
                    uint32_t v[2][4];
                    tc::tmem_ld(taddr + h * 4, v[0]);
                    tc::tmem_ld(taddr + 128 + h * 4, v[1]);
                    tc::tmem_wait_ld(v);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        acc[h * 4 + i] += __uint_as_float(v[0][i]) + __uint_as_float(v[1][i]);
                }
                tc::tc_fence_before();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&sm.tempty[buf]);
            }
        };
        const int64_t row = (int64_t)x.tile * TM + mine.row;
        // the k that exist of the next block loaded (none in a row past the edge)
        int64_t left = row < p.rows ? p.k - (int64_t)x.kb0 * KB - mine.k : 0;
        const float *src = p.X + row + ((int64_t)x.kb0 * KB + mine.k) * p.ld;
        const int64_t step = KB * p.ld;
        float v[DEPTH][PER];
#pragma unroll
        for (int d = 0; d < DEPTH; ++d) {
            if (d < len) mine.load(src, p.ld, left, v[d]);
            src += step;
            left -= KB;
        }
        // blocks before the next look at what has been split so far: 3, 6, 12, 24, 48, 72 ...
        int check = DEPTH;
        bool stopped = false;
        for (int b0 = 0; b0 < len; b0 += DEPTH) {
            if (b0 == check) {
                check += min(check, 8 * DEPTH);
                const bool stop = outside(high, low) || tc::aborted(sm);
                stopped = __any_sync(0xffffffffu, stop) != 0;
                if (stopped) {   // the product is the launch's behind: no more of it here
                    tc::set_aborted(sm);
                    break;
                }
            }
#pragma unroll
            for (int d = 0; d < DEPTH; ++d) {
                const int b = b0 + d;   // block within the unit
                if (b >= len) break;
                // a chunk is drained a block or two into the next, when its MMAs are through
                if ((b & (p.chunk - 1)) == (lag & (p.chunk - 1))) drain_to((b - lag) / p.chunk);
                ok &= tc::mbar_wait(&sm.aempty[stage], (lap & 1u) ^ 1u, sm, p.status, p.wait_ns);
                mine.store(big_plane(sm, stage, 0), v[d], high, low);
                // the MMA reads these through the async proxy
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&sm.afull[stage]);
                if (++stage == STAGES) {
                    stage = 0;
                    ++lap;
                }
                if (b + DEPTH < len) mine.load(src, p.ld, left, v[d]);
                src += step;
                left -= KB;
            }
        }
        if (!stopped) drain_to((len + p.chunk - 1) / p.chunk);
        ok = __all_sync(0xffffffffu, ok && !stopped) != 0;
        if (!ok) break;
        // partial sums of the unit: [small row][128 rows of the large operand]
        float *out = p.partial + ((int64_t)u * p.n16 + part * cols) * TM + quarter * 32 + lane;
#pragma unroll
        for (int c = 0; c < 32; ++c)
            if (c < cols) __stcg(out + c * TM, acc[c]);
    }
    if (__any_sync(0xffffffffu, outside(high, low)) && lane == 0) atomicOr(p.gate, 1u);
}

__global__ void __launch_bounds__(THREADS, 1) skinny_kernel(const SkinnyParams p)
{
    extern __shared__ uint8_t smem_raw[];
    tc::Smem &sm = *reinterpret_cast<tc::Smem *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid == 0) {
        for (int i = 0; i < STAGES; ++i) {
            tc::mbar_init(&sm.afull[i], SPLIT_WARPS);
            tc::mbar_init(&sm.bfull[i], 1);
            tc::mbar_init(&sm.aempty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&sm.tfull[i], 1);
            tc::mbar_init(&sm.tempty[i], SPLIT_WARPS);
        }
        tc::mbar_init(&sm.drain, 1);
        sm.abort = 0;
        sm.timeout_bit = 0x8u;   // mirrors GFIP_STATUS_WAIT_TIMEOUT
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         tc::saddr(&sm.tmem_base)),
                     "r"(tc::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc::tc_fence_before();
    // an element of the small operand lies outside the range, or another CTA has met one
    const bool skip =
        __syncthreads_or(tid == 0 && *(volatile const unsigned int *)p.gate != 0u) != 0;
    tc::tc_fence_after();
    const uint32_t tmem = sm.tmem_base;
    if (!skip) {
        if (warp == 0)
            producer(p, sm);
        else if (warp == 1)
            issuer(p, sm, tmem);
        else
            splitter(p, sm, tmem);
    }
    tc::tc_fence_before();
    __syncwarp();
    __syncthreads();
    tc::tc_fence_after();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(tc::TMEM_COLS)
                     : "memory");
}

// C := alpha * (the k ranges' partial sums, in order) + beta * C.  A CTA takes 32 rows of the
// large operand and all of the small one's: reads along the large operand, writes along C's rows.
__global__ void __launch_bounds__(256) add_kernel(const SkinnyParams p, float *C, int64_t ldc,
                                                  int small_rows, int big_is_row, float alpha,
                                                  float beta)
{
    __shared__ float tile[128][33];   // [small row][row of the large operand]
    if (*p.gate != 0u) return;        // the launch behind computes the product
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int b0 = blockIdx.x * 32;
    const int64_t unit = (int64_t)p.n16 * TM;
    for (int s = w; s < small_rows; s += 8) {
        const float *src =
            p.partial + (int64_t)(b0 / TM) * unit + (int64_t)s * TM + b0 % TM + lane;
        float v = 0.f;
        for (int q = 0; q < p.splits; ++q) {
            const float e = __ldcg(src + (int64_t)q * p.tiles * unit);
            v = q == 0 ? e : v + e;
        }
        tile[s][lane] = v;
    }
    __syncthreads();
    const bool read_c = beta != 0.f;
    for (int e = tid; e < 32 * small_rows; e += 256) {
        const int b = big_is_row ? e & 31 : e / small_rows;
        const int s = big_is_row ? e >> 5 : e - b * small_rows;
        if (b0 + b >= p.rows) continue;
        float *c = C + (big_is_row ? (b0 + b) + (int64_t)s * ldc : s + (int64_t)(b0 + b) * ldc);
        const float v = alpha * (tile[s][b] * tc::F32_UNSCALE);
        *c = read_c ? fmaf(beta, *c, v) : v;
    }
}

}  // namespace skinny

cudaError_t launch_f32_skinny(const SkinnyParams &p, const F32SplitArgs &small, float *C,
                              int64_t ldc, int big_is_row, float alpha, float beta, int sms,
                              cudaStream_t s)
{
    using namespace skinny;
    static bool configured = false;
    if (!configured) {
        const cudaError_t e =
            cudaFuncSetAttribute(skinny_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(tc::smem_bytes()));
        if (e != cudaSuccess) return e;
        configured = true;
    }
    const cudaError_t e = launch_f32_split(small, p.k, p.kt, p.gate, s);
    if (e != cudaSuccess) return e;
    const int grid = p.units < sms ? p.units : sms;
    skinny_kernel<<<grid, THREADS, tc::smem_bytes(), s>>>(p);
    add_kernel<<<(p.rows + 31) / 32, 256, 0, s>>>(p, C, ldc, small.rows, big_is_row, alpha, beta);
    return cudaGetLastError();
}

}  // namespace gfip
