// gfip_tc.cuh -- tcgen05 tile core for products of split operands.
//
// Both operands arrive as S BF16 planes each (plane s of element x is its s-th part, the
// largest first); the kernel forms the sum over the plane pairs (s, t) with s + t <= S + 1:
//
//  * KIND_DIGITS (FP64 emulated, gfip_ozaki.cu): planes are 6-bit integer digits.  Pairs with
//    the same s + t (a "class") have the same weight, so they share one FP32 accumulator:
//    sums of up to 16384 digit products stay exact.
//  * KIND_F32 (FP32 GEMM, gfip_f32_tc.cu): three planes hold an FP32 value's 24 bits exactly.
//    a1 b1 has an accumulator of its own, seven smaller products share a second one.
//
// Why this shape.  A CTA computes a 128 x 128 tile of C.  The tensor pipe takes 128 clocks for
// one pair of a 32-wide k block, and one 8 KB plane of each operand serves up to S pairs; so
// the kernel walks k once per group of four classes and multiplies every pair of the group
// from one set of planes: at S = 7 a k block's 14 planes (112 KB) feed 18 pairs, 50 bytes a
// clock from L2.  (One pass over k per pair, with two pairs sharing an A plane, took 94 bytes a
// clock and left the tensor pipe 38 % busy at 4096^3.)  Four classes x 128 columns fill the
// 512 columns of tensor memory.  Neighbouring classes sit in neighbouring columns and
// neighbouring B planes in neighbouring shared memory, so pairs (s, t), (s, t + 1) are one
// MMA of N = 256: it reads 12 KB of operands per 128 clocks where two of N = 128 read 16 KB.
//
// Measured on one GB300: 4096^3 with 7 digits 4710 -> 2416 us (tensor pipe 75 % busy), 8192^3 38 ->
// 63 TFLOP/s FP64-equivalent; FP32 4096^3 2513 us on the FFMA core -> 644 (213 TFLOP/s; 704 where
// the power cap binds, 1024 clocks of MMAs a k block).
//
// Roles (one CTA per SM, 10 warps, persistent over the units of work):
//   warp 0      producer.  Digits: per k block one bulk copy of the B planes the group needs (two
//               to four blocks in flight) and one per A plane into a ring of single-plane
//               slots, each refilled as soon as the MMAs reading it are done.  FP32: both
//               operands' three planes of a block as one 48 KB stage of four;
//   warp 1      allocates tensor memory and issues tcgen05.mma;
//   warps 2-9   drain the accumulators at the end of each k chunk into registers (exact
//               integers, or FP32 sums rounded to nearest) and write C, overlapping the next
//               unit's MMAs.
// The producer and issuer warps run converged, with one elected lane issuing copies and MMAs, and
// wait for one barrier per A plane (digits) or block (FP32): the instructions between two MMAs
// are a serial chain in one warp (a first form with a barrier per plane of either operand, run
// by one lane, spent 800 clocks a step on them and ran the MMAs at a third of their rate; three
// barriers a block took FP32, with six products, 1107 clocks a block, one 904, for 768 of MMAs).
// Every mbarrier wait is bounded by a global-timer budget; on a timeout the kernel raises a
// status bit, the roles skip their remaining work, the producer waits for its copies in
// flight, and tensor memory is released before exit.
#pragma once

#include <cstdint>
#include <type_traits>

#include <cuda_bf16.h>

#include "gfip_internal.h"

namespace gfip {
namespace tc {

constexpr int TM = 128;                  // tile rows (M of the MMA), rows of a plane tile
constexpr int TN = 128;                  // tile columns, rows of a B plane tile
constexpr int KB = 32;                   // k per plane tile: 32 BF16 = one 64-byte row
constexpr int PLANE_BYTES = TM * KB * 2; // 8 KB
constexpr int SLOTS = 28;                // plane slots in shared memory (224 KB)
constexpr int MAX_ASLOTS = 16;
constexpr int MAX_BSTAGES = 4;
constexpr int THREADS = 320;
constexpr int EPI_WARPS = 8;
constexpr uint32_t TMEM_COLS = 512;
constexpr int DIGIT_BITS = 6;
constexpr int EXACT_TERMS = 16384;       // digit products whose sum FP32 holds exactly
constexpr long long WAIT_POLLS = 1ll << 32;          // backstop, should the timer stall

enum Kind : int { KIND_DIGITS_INT = 0, KIND_DIGITS_F64 = 1, KIND_F32 = 2 };

struct Smem {
    uint8_t plane[SLOTS][PLANE_BYTES];  // 1024-byte aligned; A ring first, then B stages
    uint64_t afull[MAX_ASLOTS];
    uint64_t aempty[MAX_ASLOTS];
    uint64_t bfull[MAX_BSTAGES];
    uint64_t bempty[MAX_BSTAGES];
    uint64_t tfull[2];                  // accumulators of a chunk complete
    uint64_t tempty[2];                 // ... and read by the epilogue warps
    uint64_t drain;
    uint32_t tmem_base;
    int abort;
    unsigned timeout_bit;               // status bit of a wait that gave up
};

__device__ __forceinline__ bool aborted(const Smem &sm)
{
    return *(volatile const int *)&sm.abort != 0;
}

__device__ __forceinline__ void set_aborted(Smem &sm)
{
    *(volatile int *)&sm.abort = 1;
}

__device__ __forceinline__ uint32_t saddr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(bar)), "r"(count)
                 : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(bar)) : "memory");
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool mbar_try(uint32_t a, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    return done != 0;
}

// Waits for the phase with the given parity to complete; gives up after budget_ns of the
// global timer, or when another role has aborted.  Returns false if it gave up; a timeout
// sets the CTA's abort flag and the status bit.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, Smem &sm,
                                          unsigned *status, unsigned long long budget_ns)
{
    const uint32_t a = saddr(bar);
    if (mbar_try(a, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (long long it = 0; it < WAIT_POLLS; ++it) {
        if (mbar_try(a, parity)) return true;
        if (aborted(sm)) return false;
        if ((it & 63) == 63 && global_ns() - t0 > budget_ns) break;
    }
    set_aborted(sm);
    atomicOr(status, sm.timeout_bit);
    return false;
}

// The same wait by a whole converged warp, whose lanes go on or give up together: each lane sees
// the timer and the abort flag at its own moment, and a lane that left alone would be missed by
// the warp-wide instructions behind the wait.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t *bar, uint32_t parity, Smem &sm,
                                               unsigned *status, unsigned long long budget_ns)
{
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, sm, status, budget_ns)) != 0;
}

// The same wait, used while draining after an abort: ignores the abort flag and raises
// nothing; returns when the budget runs out.
__device__ __forceinline__ void mbar_wait_drain(uint64_t *bar, uint32_t parity,
                                                unsigned long long budget_ns)
{
    const uint32_t a = saddr(bar);
    const unsigned long long t0 = global_ns();
    for (long long it = 0; it < WAIT_POLLS; ++it) {
        if (mbar_try(a, parity)) return;
        if ((it & 63) == 63 && global_ns() - t0 > budget_ns) return;
    }
}

// Global -> shared bulk copy (TMA engine), completing on an mbarrier.
__device__ __forceinline__ void bulk_copy(void *dst, const void *src, uint32_t bytes,
                                          uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(saddr(dst)), "l"(src), "r"(bytes), "r"(saddr(bar))
        : "memory");
}

// Shared-memory matrix descriptor of a K-major tile in the 64-byte swizzle layout: 8-row
// groups of 64-byte rows, 512 bytes apart (stride byte offset); descriptor version 1.  The low
// word holds the start address / 16 and the leading byte offset (unused here, 1); addresses
// within shared memory add to it without carries.
constexpr uint32_t DESC_HIGH = (512u >> 4) | (1u << 14) | (4u << 29);

__device__ __forceinline__ uint32_t desc_low(uint32_t addr)
{
    return (addr >> 4) | (1u << 16);
}

constexpr uint32_t PLANE_DESC = PLANE_BYTES >> 4;   // one plane further

// Instruction descriptor: kind::f16 with BF16 A and B, FP32 D, both K-major, M = 128.
template <int N>
constexpr uint32_t IDESC = (1u << 4)                      // D: F32
                           | (1u << 7)                    // A: BF16
                           | (1u << 10)                   // B: BF16
                           | ((uint32_t)(N >> 3) << 17)   // N
                           | ((uint32_t)(TM >> 4) << 24); // M

template <int N>
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint32_t adesc, uint32_t bdesc,
                                         uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n .reg .b64 a, b;\n mov.b64 a, {%1, %5};\n mov.b64 b, {%2, %5};\n"
        " setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n}" ::"r"(tmem_d),
        "r"(adesc), "r"(bdesc), "r"(IDESC<N>), "r"(accumulate), "n"(DESC_HIGH)
        : "memory");
}

// One plane pair (N = 128), or two with neighbouring B planes (N = 256), over a 32-wide block;
// accumulate: 0 for the first product of an accumulation.
template <int N>
__device__ __forceinline__ void mma_block(uint32_t tmem_d, uint32_t a, uint32_t b,
                                          uint32_t accumulate)
{
    mma_bf16<N>(tmem_d, a, b, accumulate);
    mma_bf16<N>(tmem_d, a + 2, b + 2, 1u);   // 16 k = 32 bytes further
}

// The same one lane of a converged warp, every time.
__device__ __forceinline__ bool elect_one()
{
    uint32_t r;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(r));
    return r != 0;
}

__device__ __forceinline__ void mma_commit(uint64_t *bar)
{
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            saddr(bar))
        : "memory");
}

__device__ __forceinline__ void tc_fence_before()
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_after()
{
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// 4 consecutive FP32 columns of this thread's tensor-memory lane, as their bits.
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr)
                 : "memory");
}

// ... and 8.
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7])
        : "r"(taddr)
        : "memory");
}

// Waits for this thread's tensor-memory loads; the loaded values pass through it, so no use
// of them can move above the wait.
template <int R, int W> __device__ __forceinline__ void tmem_wait_ld(uint32_t (&v)[R][W])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int a = 0; a < R; ++a)
#pragma unroll
        for (int i = 0; i < W; ++i) asm volatile("" : "+r"(v[a][i]));
}

// Byte offset of element (r, c) (r < 128 rows, c < 32 k) in a plane tile: 8-row groups of 512
// bytes; a row is 64 bytes whose four 16-byte chunks are XOR-permuted by (r / 2) % 4 (the
// 64-byte swizzle the MMA descriptor names).
__host__ __device__ __forceinline__ uint32_t plane_off(int r, int c)
{
    return (uint32_t)(r * 64 + ((((c >> 3) ^ ((r >> 1) & 3))) << 4) + (c & 7) * 2);
}

// The classes of one group: s + t in c0 .. c1; A planes s = 1 .. c1 - 1, for each the B planes
// t = tlo(s) .. c1 - s.  chunk: k blocks per accumulation.
struct Group {
    int c0, c1, chunk;

    __device__ __forceinline__ int tlo(int s) const { return max(1, c0 - s); }
};

__device__ __forceinline__ int group_count(int planes)
{
    return (planes + 3) / 4;
}

__device__ __forceinline__ Group group_of(int g, int planes)
{
    const int c0 = 2 + 4 * g, c1 = min(c0 + 3, planes + 1);
    return Group{c0, c1, EXACT_TERMS / (c1 - 1) / KB};   // a class has at most c1 - 1 pairs
}

// One unit of work: a tile of C over a range of k blocks.
struct Unit {
    int i, j, kb0, kb1, tile, split;
};

__device__ __forceinline__ Unit unit_of(const TcParams &p, int u)
{
    Unit x;
    const int mask = p.tmask_a ? p.tmask_a : p.tmask_b;
    if (mask) {
        // A triangular operand leaves tiles of 1 to all of the k blocks (TRMM): the longest come
        // first, and every other round of the grid runs backwards, so that a CTA with a
        // long tile gets a short one next (2048 x 2048: 68 blocks on the busiest SM, 96 in
        // band order).
        const int grid = static_cast<int>(gridDim.x);
        const int round = u / grid, at = u - round * grid;
        if (round & 1) u = round * grid + min(grid, p.units - round * grid) - 1 - at;
    }
    x.split = u / p.tiles;
    x.tile = u - x.split * p.tiles;
    if (mask) {
        const int across = p.tmask_a ? p.nt : p.mt, along = p.tmask_a ? p.mt : p.nt;
        const int rank = x.tile / across, other = x.tile - rank * across;
        const int line = (mask & TMASK_KEEP_GE) ? along - 1 - rank : rank;
        x.i = p.tmask_a ? line : other;
        x.j = p.tmask_a ? other : line;
    } else if (p.tri != TRI_NONE) {
        // row r of the lower triangle holds tiles r (r + 1) / 2 .. + r
        int r = static_cast<int>((sqrtf(8.f * static_cast<float>(x.tile) + 1.f) - 1.f) * 0.5f);
        while (r * (r + 1) / 2 > x.tile) --r;
        while ((r + 1) * (r + 2) / 2 <= x.tile) ++r;
        const int c = x.tile - r * (r + 1) / 2;
        x.i = p.tri == TRI_LOWER ? r : c;
        x.j = p.tri == TRI_LOWER ? c : r;
    } else {
        // CTAs that run at the same time cover a band of tile rows, so they share planes of A
        // (within the band) and of B (across it) in L2
        constexpr int BAND = 8;
        const int band = x.tile / (BAND * p.nt);
        const int in_band = x.tile - band * BAND * p.nt;
        const int rows = min(BAND, p.mt - band * BAND);
        x.i = band * BAND + in_band % rows;
        x.j = in_band / rows;
    }
    int lo = 0, hi = p.kt;
    if (mask) {   // the k blocks that the tile's rows of the triangular operand keep
        const int x0 = (p.tmask_a ? x.i : x.j) * TM;
        const int strict = (mask & TMASK_STRICT) ? 1 : 0;
        if (mask & TMASK_KEEP_GE)
            hi = min(hi, (x0 + TM - 1 - strict) / KB + 1);
        else
            lo = min(hi - 1, (x0 + strict) / KB);
    }
    const int len = hi - lo;
    x.kb0 = lo + static_cast<int>((int64_t)len * x.split / p.splits);
    x.kb1 = lo + static_cast<int>((int64_t)len * (x.split + 1) / p.splits);
    return x;
}

// FP32: a stage holds a k block's three planes of A, then of B, on one barrier pair (`afull`,
// `aempty`): its 14 MMAs are issued after a single wait.
constexpr int F32_PLANES = 3;
constexpr int F32_STAGES = 4;
constexpr uint32_t F32_BYTES = F32_PLANES * PLANE_BYTES;
static_assert(F32_STAGES * 2 * F32_PLANES <= SLOTS && F32_STAGES <= MAX_ASLOTS, "stages fit");

// The range in which an FP32 element's split into three BF16 planes is exact and safe
// (gfip_f32_tc.cu): zero, or a magnitude in [2^-100, 2^47).  The operands' planes are those of
// the elements times powers of two that multiply to 1 / F32_UNSCALE.
constexpr uint32_t LOW_BITS = (127u - 100u) << 23;   // 2^-100
constexpr uint32_t HIGH_BITS = (127u + 47u) << 23;   // 2^47
constexpr float F32_UNSCALE = 1.f / 256.f;

__device__ __forceinline__ bool outside_split(float x)
{
    const uint32_t m = __float_as_uint(x) & 0x7FFFFFFFu;
    return m != 0u && m - LOW_BITS >= HIGH_BITS - LOW_BITS;
}

// Two floats' planes as BF16 pairs (first element in the low half).
__device__ __forceinline__ void split_pair(float x0, float x1, uint32_t &p1, uint32_t &p2,
                                           uint32_t &p3)
{
    auto pack = [](float lo, float hi) -> uint32_t {
        const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
        return *reinterpret_cast<const uint32_t *>(&v);
    };
    p1 = pack(x0, x1);
    const float r0 = x0 - __uint_as_float(p1 << 16);
    const float r1 = x1 - __uint_as_float(p1 & 0xFFFF0000u);
    p2 = pack(r0, r1);
    p3 = pack(r0 - __uint_as_float(p2 << 16), r1 - __uint_as_float(p2 & 0xFFFF0000u));
}

// Digits: `na` A slots used round robin, then `nb` B stages of `planes` slots.
struct Ring {
    int na, nb;
};

__device__ __forceinline__ Ring ring_of(int planes)
{
    // half of the slots for B, at least two k blocks
    const int nb = min(MAX_BSTAGES, max(2, SLOTS / 2 / planes));
    return Ring{min(MAX_ASLOTS, SLOTS - nb * planes), nb};
}

// ---- producer -----------------------------------------------------------------------------------

__device__ __forceinline__ void digit_producer(const TcParams &p, Smem &sm)
{
    const Ring rg = ring_of(p.planes);
    const bool leader = elect_one();
    int a_slot = 0, b_stage = 0;
    uint32_t a_lap = 0, b_lap = 0;   // laps of the rings; their parity is the next fill's phase
    const bool withhold = p.inject_timeout && blockIdx.x == 0;
    bool skip = withhold;   // test hook: the first A plane is never copied
    bool ok = true;
    const int64_t block = (int64_t)p.planes * PLANE_BYTES;
    const int groups = group_count(p.planes);
    for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
        const Unit x = unit_of(p, u);
        for (int g = 0; g < groups && ok; ++g) {
            const Group q = group_of(g, p.planes);
            const uint8_t *a = p.pa + ((int64_t)x.i * p.kt + x.kb0) * block;
            const uint8_t *b = p.pb + ((int64_t)x.j * p.kt + x.kb0) * block;
            const uint32_t b_bytes = (q.c1 - 1) * PLANE_BYTES;
            for (int kb = x.kb0; kb < x.kb1 && ok; ++kb, a += block, b += block) {
                ok = mbar_wait(&sm.bempty[b_stage], (b_lap & 1u) ^ 1u, sm, p.status, p.wait_ns);
                if (!ok) break;
                if (leader) {
                    mbar_expect_tx(&sm.bfull[b_stage], b_bytes);
                    bulk_copy(sm.plane[rg.na + b_stage * p.planes], b, b_bytes,
                              &sm.bfull[b_stage]);
                }
                if (++b_stage == rg.nb) {
                    b_stage = 0;
                    ++b_lap;
                }
                for (int s = 0; s < q.c1 - 1; ++s) {
                    ok = mbar_wait(&sm.aempty[a_slot], (a_lap & 1u) ^ 1u, sm, p.status,
                                   p.wait_ns);
                    if (!ok) break;
                    if (leader && !skip) {
                        mbar_expect_tx(&sm.afull[a_slot], PLANE_BYTES);
                        bulk_copy(sm.plane[a_slot], a + s * PLANE_BYTES, PLANE_BYTES,
                                  &sm.afull[a_slot]);
                    }
                    skip = false;
                    if (++a_slot == rg.na) {
                        a_slot = 0;
                        ++a_lap;
                    }
                }
            }
        }
    }
    // No bulk copy may still be writing shared memory when the CTA exits: wait for the last
    // fill of every slot (in this lap below the cursor, in the lap before from it on).
    for (int i = 0; i < rg.na; ++i)
        if ((i < a_slot || a_lap > 0) && !(withhold && i == 0 && a_lap == 0))
            mbar_wait_drain(&sm.afull[i], (i < a_slot ? a_lap : a_lap - 1) & 1u, p.wait_ns);
    for (int i = 0; i < rg.nb; ++i)
        if (i < b_stage || b_lap > 0)
            mbar_wait_drain(&sm.bfull[i], (i < b_stage ? b_lap : b_lap - 1) & 1u, p.wait_ns);
}

__device__ __forceinline__ void f32_producer(const TcParams &p, Smem &sm)
{
    const bool leader = elect_one();
    int stage = 0;
    uint32_t lap = 0;
    bool ok = true;
    bool skip = p.inject_timeout && blockIdx.x == 0;   // test hook: the first block never arrives
    for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
        const Unit x = unit_of(p, u);
        const uint8_t *a = p.pa + ((int64_t)x.i * p.kt + x.kb0) * F32_BYTES;
        const uint8_t *b = p.pb + ((int64_t)x.j * p.kt + x.kb0) * F32_BYTES;
        for (int kb = x.kb0; kb < x.kb1; ++kb, a += F32_BYTES, b += F32_BYTES) {
            ok = mbar_wait(&sm.aempty[stage], (lap & 1u) ^ 1u, sm, p.status, p.wait_ns);
            if (!ok) break;
            if (leader && !skip) {
                uint8_t *dst = sm.plane[stage * 2 * F32_PLANES];
                mbar_expect_tx(&sm.afull[stage], 2 * F32_BYTES);
                bulk_copy(dst, a, F32_BYTES, &sm.afull[stage]);
                bulk_copy(dst + F32_BYTES, b, F32_BYTES, &sm.afull[stage]);
            }
            skip = false;
            if (++stage == F32_STAGES) {
                stage = 0;
                ++lap;
            }
        }
    }
    for (int i = 0; i < F32_STAGES; ++i)   // no copy may outlive the CTA
        if (i < stage || lap > 0)
            mbar_wait_drain(&sm.afull[i], (i < stage ? lap : lap - 1) & 1u, p.wait_ns);
}

// ---- MMA issuer ---------------------------------------------------------------------------------

__device__ __forceinline__ void digit_issuer(const TcParams &p, Smem &sm, uint32_t tmem)
{
    const Ring rg = ring_of(p.planes);
    const bool leader = elect_one();
    int a_slot = 0, b_stage = 0;
    uint32_t a_phase = 0, b_phase = 0;
    uint32_t chunks = 0;
    bool ok = true;
    const uint32_t a_base = desc_low(saddr(sm.plane[0]));
    const uint32_t b_base = a_base + rg.na * PLANE_DESC;
    const int groups = group_count(p.planes);
    for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
        const Unit x = unit_of(p, u);
        for (int g = 0; g < groups && ok; ++g) {
            const Group q = group_of(g, p.planes);
            for (int k0 = x.kb0; k0 < x.kb1 && ok; k0 += q.chunk, ++chunks) {
                const int k1 = min(x.kb1, k0 + q.chunk);
                ok = mbar_wait(&sm.tempty[0], (chunks & 1u) ^ 1u, sm, p.status, p.wait_ns);
                if (!ok) break;
                tc_fence_after();
                uint32_t accumulate = 0;   // the first A plane's products start the sums
                for (int kb = k0; kb < k1; ++kb) {
                    ok = mbar_wait(&sm.bfull[b_stage], b_phase, sm, p.status, p.wait_ns);
                    if (!ok) break;
                    const uint32_t b1 = b_base + b_stage * p.planes * PLANE_DESC;
                    for (int s = 1; s < q.c1; ++s) {
                        ok = mbar_wait(&sm.afull[a_slot], a_phase, sm, p.status, p.wait_ns);
                        if (!ok) break;
                        tc_fence_after();
                        if (leader) {
                            const int lo = q.tlo(s);
                            const uint32_t a = a_base + a_slot * PLANE_DESC;
                            uint32_t b = b1 + (lo - 1) * PLANE_DESC;
                            uint32_t d = tmem + (s + lo - q.c0) * TN;
                            int left = q.c1 - s - lo + 1;
                            for (; left >= 2; left -= 2) {
                                mma_block<256>(d, a, b, accumulate);
                                b += 2 * PLANE_DESC;
                                d += 2 * TN;
                            }
                            if (left) mma_block<128>(d, a, b, accumulate);
                            mma_commit(&sm.aempty[a_slot]);
                        }
                        accumulate = 1;
                        if (++a_slot == rg.na) {
                            a_slot = 0;
                            a_phase ^= 1u;
                        }
                    }
                    if (!ok) break;
                    if (leader) mma_commit(&sm.bempty[b_stage]);
                    if (++b_stage == rg.nb) {
                        b_stage = 0;
                        b_phase ^= 1u;
                    }
                }
                if (ok && leader) mma_commit(&sm.tfull[0]);
            }
        }
    }
    // all MMAs this warp issued have completed once this commit arrives
    if (leader) mma_commit(&sm.drain);
    mbar_wait_drain(&sm.drain, 0, p.wait_ns);
}

__device__ __forceinline__ void f32_issuer(const TcParams &p, Smem &sm, uint32_t tmem)
{
    const bool leader = elect_one();
    int stage = 0;
    uint32_t phase = 0, chunks = 0;
    bool ok = true;
    const uint32_t base = desc_low(saddr(sm.plane[0]));
    for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
        const Unit x = unit_of(p, u);
        for (int k0 = x.kb0; k0 < x.kb1 && ok; k0 += p.chunk, ++chunks) {
            const int k1 = min(x.kb1, k0 + p.chunk);
            const uint32_t buf = chunks & 1u;
            ok = mbar_wait(&sm.tempty[buf], ((chunks >> 1) & 1u) ^ 1u, sm, p.status, p.wait_ns);
            if (!ok) break;
            tc_fence_after();
            // columns 0-127: a1 b1; 128-255: the seven smaller products
            const uint32_t d = tmem + buf * 256;
            uint32_t accumulate = 0;   // the block's first MMA starts both sums
            for (int kb = k0; kb < k1; ++kb) {
                ok = mbar_wait(&sm.afull[stage], phase, sm, p.status, p.wait_ns);
                if (!ok) break;
                tc_fence_after();
                if (leader) {
                    const uint32_t a1 = base + stage * 2 * F32_PLANES * PLANE_DESC;
                    const uint32_t a2 = a1 + PLANE_DESC, a3 = a2 + PLANE_DESC;
                    const uint32_t b1 = a3 + PLANE_DESC, b2 = b1 + PLANE_DESC;
                    mma_block<256>(d, a1, b1, accumulate);
                    mma_block<128>(d + TN, a1, b2 + PLANE_DESC, 1u);
                    mma_block<128>(d + TN, a2, b1, 1u);
                    mma_block<128>(d + TN, a2, b2, 1u);
                    mma_block<128>(d + TN, a2, b2 + PLANE_DESC, 1u);
                    mma_block<128>(d + TN, a3, b1, 1u);
                    mma_block<128>(d + TN, a3, b2, 1u);
                    mma_commit(&sm.aempty[stage]);
                }
                accumulate = 1;
                if (++stage == F32_STAGES) {
                    stage = 0;
                    phase ^= 1u;
                }
            }
            if (ok && leader) mma_commit(&sm.tfull[buf]);
        }
    }
    // all MMAs this warp issued have completed once this commit arrives
    if (leader) mma_commit(&sm.drain);
    mbar_wait_drain(&sm.drain, 0, p.wait_ns);
}

// ---- epilogue -----------------------------------------------------------------------------------

// x * 2^e where the result or x is zero, subnormal or not finite.
[[maybe_unused]] static __device__ __noinline__ double scale2_general(double x, int e)
{
    return ldexp(x, e);
}

// x * 2^e; the fast path adds to the exponent field.
__device__ __forceinline__ double scale2(double x, int e)
{
    const int hi = __double2hiint(x);
    const int ex = ((hi >> 20) & 0x7FF) + e;
    if (((hi >> 20) & 0x7FF) != 0 && ex > 0 && ex < 2047)
        return __hiloint2double(hi + e * (1 << 20), __double2loint(x));
    return scale2_general(x, e);
}

template <int KIND> struct AccOf {
    using type = float;
};
template <> struct AccOf<KIND_DIGITS_INT> {
    using type = long long;
};
template <> struct AccOf<KIND_DIGITS_F64> {
    using type = double;
};

// The value of one element's classes c0 .. c0 + N - 1 in units of the last one's weight, exact.
template <int N, int W>
__device__ __forceinline__ long long digits_value(const uint32_t (&v)[N][W], int i)
{
    long long r = __float2int_rn(__uint_as_float(v[N - 1][i]));
#pragma unroll
    for (int c = 0; c < N - 1; ++c)
        r += (long long)__float2int_rn(__uint_as_float(v[c][i])) *
             (1 << (DIGIT_BITS * (N - 1 - c)));
    return r;
}

// Adds the chunk's accumulators (N classes of 128 columns at taddr) to this thread's 64 sums.
template <int KIND, int N>
__device__ __forceinline__ void drain_digits(uint32_t taddr, int shift, double scale,
                                             typename AccOf<KIND>::type (&acc)[64])
{
    constexpr int W = 4;   // columns at a time: 128 registers hold the sums
#pragma unroll
    for (int g = 0; g < 64 / W; ++g) {
        uint32_t v[N][W];
#pragma unroll
        for (int c = 0; c < N; ++c) tmem_ld(taddr + c * TN + g * W, v[c]);
        tmem_wait_ld(v);
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const long long d = digits_value(v, i);
            if constexpr (KIND == KIND_DIGITS_INT)
                acc[g * W + i] += (long long)((unsigned long long)d << shift);
            else
                acc[g * W + i] = fma((double)d, scale, acc[g * W + i]);
        }
    }
}

template <int KIND> __device__ void epilogue(const TcParams &p, Smem &sm, uint32_t tmem)
{
    constexpr int NBUF = KIND == KIND_F32 ? 2 : 1;
    using Acc = typename AccOf<KIND>::type;
    using T = typename std::conditional<KIND == KIND_F32, float, double>::type;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // tensor-memory lane quarter from warp % 4, column half from (warp - 2) / 4
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    const int groups = KIND == KIND_F32 ? 1 : group_count(p.planes);
    uint32_t chunks = 0;
    for (int u = blockIdx.x; u < p.units; u += gridDim.x) {
        const Unit x = unit_of(p, u);
        const int row = x.i * TM + quarter * 32 + lane;
        const int col0 = x.j * TN + half * 64;
        T *C = static_cast<T *>(p.C);
        const T alpha = (T)p.alpha, beta = (T)p.beta;
        const bool read_c = beta != T(0);
        // bring C to L2 while the products are formed: lane l fetches columns l and l + 32 of
        // the warp's 32 rows (128 bytes of FP32, 256 of FP64)
        if (read_c) {
            const int row0 = row - lane;
            for (int c = lane; c < 64; c += 32)
                if (col0 + c < p.n)
                    for (int r = row0; r < min(row0 + 32, p.m); r += 128 / (int)sizeof(T))
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(
                            C + r + (int64_t)(col0 + c) * p.ldc));
        }
        Acc acc[64];
#pragma unroll
        for (int c = 0; c < 64; ++c) acc[c] = Acc(0);
        for (int g = 0; g < groups; ++g) {
            const Group q =
                KIND == KIND_F32 ? Group{2, 4, p.chunk} : group_of(g, p.planes);
            for (int k0 = x.kb0; k0 < x.kb1; k0 += q.chunk, ++chunks) {
                const int buf = chunks % NBUF;
                if (!mbar_wait_warp(&sm.tfull[buf], (chunks / NBUF) & 1u, sm, p.status,
                                    p.wait_ns))
                    return;
                tc_fence_after();
                const uint32_t taddr =
                    tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * 256 + half * 64);
                if constexpr (KIND == KIND_F32) {
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        uint32_t v[4][8];
                        tmem_ld(taddr + h * 16, v[0]);
                        tmem_ld(taddr + h * 16 + 8, v[1]);
                        tmem_ld(taddr + h * 16 + TN, v[2]);
                        tmem_ld(taddr + h * 16 + TN + 8, v[3]);
                        tmem_wait_ld(v);
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            acc[h * 16 + i] +=
                                __uint_as_float(v[0][i]) + __uint_as_float(v[2][i]);
                            acc[h * 16 + 8 + i] +=
                                __uint_as_float(v[1][i]) + __uint_as_float(v[3][i]);
                        }
                    }
                } else {
                    const int shift = DIGIT_BITS * (p.planes + 1 - q.c1);
                    const double scale = scale2(1.0, -DIGIT_BITS * q.c1);
                    switch (q.c1 - q.c0) {
                    case 0: drain_digits<KIND, 1>(taddr, shift, scale, acc); break;
                    case 1: drain_digits<KIND, 2>(taddr, shift, scale, acc); break;
                    case 2: drain_digits<KIND, 3>(taddr, shift, scale, acc); break;
                    default: drain_digits<KIND, 4>(taddr, shift, scale, acc); break;
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.tempty[buf]);
            }
        }
        if constexpr (KIND == KIND_F32) {
            if (p.splits > 1) {
                // every split stores its partial tile; of each warp's 32 x 64 part the last to
                // arrive adds the splits in k order (no warp waits for another)
                const int64_t tile_elems = (int64_t)TM * TN;
                const int at = (half * 64) * TM + quarter * 32 + lane;
                float *mine = p.partial + ((int64_t)x.tile * p.splits + x.split) * tile_elems + at;
#pragma unroll
                for (int c = 0; c < 64; ++c) __stcg(mine + c * TM, acc[c]);
                __threadfence();
                __syncwarp();
                unsigned int old = 0;
                if (lane == 0) old = atomicAdd(p.counter + x.tile * EPI_WARPS + warp - 2, 1u);
                old = __shfl_sync(0xffffffffu, old, 0);
                if (old != (unsigned int)(p.splits - 1)) continue;
                __threadfence();
                const float *src = p.partial + (int64_t)x.tile * p.splits * tile_elems + at;
#pragma unroll
                for (int c = 0; c < 64; ++c) acc[c] = __ldcg(src + c * TM);
                for (int s = 1; s < p.splits; ++s) {
                    src += tile_elems;
#pragma unroll
                    for (int c = 0; c < 64; ++c) acc[c] += __ldcg(src + c * TM);
                }
            }
        }
        if (row >= p.m) continue;
        int er = 0;
        if constexpr (KIND != KIND_F32) {
            er = p.ea[row] + 2;   // 2^(e_i + 1) 2^(f_j + 1)
            if (KIND == KIND_DIGITS_INT) er -= DIGIT_BITS * (p.planes + 1);
        }
        // The columns this row stores: up to n, and of a triangle the row's part.  (Code that
        // decides per column runs at the rate of instruction fetches: 64 columns of it took
        // 25000 clocks a tile at 2048^3.)
        const int first = p.tri == TRI_UPPER ? row : 0;
        const int end = p.tri == TRI_LOWER ? min(p.n, row + 1) : p.n;
        const uint32_t count = end > first ? static_cast<uint32_t>(end - first) : 0u;
        // C is read W columns at a time, before any of them is written
        constexpr int W = KIND == KIND_F32 ? 32 : 8;
        T *cp = C + row + (int64_t)col0 * p.ldc;
        const T *cr = cp;
#pragma unroll
        for (int g = 0; g < 64 / W; ++g) {
            T cv[W];
            if (read_c) {
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    cv[i] = T(0);
                    if (static_cast<uint32_t>(col0 + g * W + i - first) < count) cv[i] = *cr;
                    cr += p.ldc;
                }
            }
#pragma unroll
            for (int i = 0; i < W; ++i) {
                const int col = col0 + g * W + i;
                const bool in = static_cast<uint32_t>(col - first) < count;
                T v;
                if constexpr (KIND == KIND_F32) {
                    v = alpha * (acc[g * W + i] * F32_UNSCALE);
                    if (read_c) v = fmaf(beta, cv[i], v);
                } else {
                    v = alpha * scale2((double)acc[g * W + i], er + (in ? p.eb[col] : 0));
                    if (read_c) v = fma(beta, cv[i], v);
                }
                if (in) *cp = v;
                cp += p.ldc;
            }
        }
    }
}

template <int KIND> __global__ void __launch_bounds__(THREADS, 1) tc_kernel(const TcParams p)
{
    extern __shared__ uint8_t smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int tid = threadIdx.x, warp = tid >> 5;
    // operands outside the range the planes hold: the launch after this one does the work
    if (p.gate != nullptr && *p.gate != 0u) return;

    if (tid == 0) {
        for (int i = 0; i < MAX_ASLOTS; ++i) {
            mbar_init(&sm.afull[i], 1);
            mbar_init(&sm.aempty[i], 1);
        }
        for (int i = 0; i < MAX_BSTAGES; ++i) {
            mbar_init(&sm.bfull[i], 1);
            mbar_init(&sm.bempty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sm.tfull[i], 1);
            mbar_init(&sm.tempty[i], EPI_WARPS);
        }
        mbar_init(&sm.drain, 1);
        sm.abort = 0;
        // mirrors GFIP_STATUS_WAIT_TIMEOUT and GFIP_STATUS_MMA_TIMEOUT
        sm.timeout_bit = KIND == KIND_F32 ? 0x8u : 0x2u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         saddr(&sm.tmem_base)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm.tmem_base;

    if (warp == 0) {
        if constexpr (KIND == KIND_F32) f32_producer(p, sm);
        else digit_producer(p, sm);
    } else if (warp == 1) {
        if constexpr (KIND == KIND_F32) f32_issuer(p, sm, tmem);
        else digit_issuer(p, sm, tmem);
    } else {
        epilogue<KIND>(p, sm, tmem);
    }
    tc_fence_before();
    __syncwarp();
    __syncthreads();
    tc_fence_after();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(TMEM_COLS)
                     : "memory");
}

inline size_t smem_bytes()
{
    return sizeof(Smem) + 1024;
}

template <int KIND> cudaError_t launch(const TcParams &p, int sms, cudaStream_t s)
{
    static bool configured = false;
    if (!configured) {
        const cudaError_t e =
            cudaFuncSetAttribute(tc_kernel<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(smem_bytes()));
        if (e != cudaSuccess) return e;
        configured = true;
    }
    tc_kernel<KIND><<<p.units < sms ? p.units : sms, THREADS, smem_bytes(), s>>>(p);
    return cudaGetLastError();
}

}  // namespace tc
}  // namespace gfip
