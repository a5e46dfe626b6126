// gfip_trsm_f32.cu -- the panel solves of the blocked triangular solve in FP32.
//
// One CTA solves a panel of at most TRSM_PANEL unknowns for 16 right-hand sides that stay in
// shared memory, by blocks of 32 unknowns:
//
//   * the block's own triangle is solved by one warp, a right-hand side per lane: every
//     unknown's quotient and its multiply-adds on the rest of the block are the lane's own, so
//     the chain holds no shuffle (the panel kernel that held an element per lane broadcast
//     every quotient through one: 270 clocks an unknown);
//   * then its 32 unknowns leave the rows below, 8 rows per half warp at a time, the unknowns in
//     registers and the triangle's entries read as rows of 4 (paired FMAs on 2 rows).
//
// The chain is hidden behind the update: the next block's rows are updated first (warps 0
// and 1), and while warp 0 solves them the other warps go on with the rows further down.  Every
// element still loses its multiples one after the other in increasing column order.
//
// The triangle is packed first, by a launch of its own, into the images the CTAs hold in shared
// memory (zero above the diagonal and beyond the panel), so that every CTA fetches a block's
// columns with one bulk copy, two blocks ahead.  (Staging them by 4-byte copies in each CTA
// took 5400 clocks a block, more than the solve: an odd leading dimension allows no wider ones.)
//
// Bound: the chain, about 2000 clocks a block (500 to update the next block's rows, 1350 to
// solve them), with the updates further down just behind it.  512 unknowns, 512 right-hand
// sides: 67 -> 36 us with the packing launch; 2048 x 2048 with its updates 386 -> 266 us (with
// the caller's copy of B; 286 since the updates form more products in shorter accumulations).
#include <cstdint>

#include "gfip_internal.h"

namespace gfip {
namespace trsm32 {

constexpr int BLK = 32;                      // unknowns per block
constexpr int BLOCKS = TRSM_PANEL / BLK;
constexpr int NV = 16;                       // right-hand sides per CTA
constexpr int WARPS = 8;
constexpr int XP = NV + 1;                   // pitch of the right-hand sides, one row per unknown
constexpr unsigned STATUS_WAIT_TIMEOUT = 0x8u;           // mirrors GFIP_STATUS_WAIT_TIMEOUT

// The packed panel of nb blocks, floats: diagonal entries [32 nb], their reciprocals [32 nb],
// the diagonal blocks [nb][column][row], then each block's columns below it [column][row].
__host__ __device__ constexpr int head_floats(int nb)
{
    return nb * (2 * BLK + BLK * BLK);
}
__host__ __device__ constexpr int below(int nb, int bk)   // rows below block bk
{
    return (nb - 1 - bk) * BLK;
}
__host__ __device__ constexpr int columns_at(int nb, int bk)
{
    // head, then 32 columns of below(nb, 0), below(nb, 1), ... rows
    return head_floats(nb) + BLK * BLK * (bk * (nb - 1) - bk * (bk - 1) / 2);
}

struct Smem {
    float head[head_floats(BLOCKS)];
    float col[2][BLK * (TRSM_PANEL - BLK)];
    float x[TRSM_PANEL * XP];        // right-hand sides, then unknowns: [unknown][side]
    unsigned long long full[3];      // col[0], col[1], head have arrived
};

// The panel's system in solve order, as in gfip_trsm.cu: t(q, d) sits at A0[q sq + d sd].
struct Panel {
    const float *A0;
    int64_t sq, sd;
    int along_q;        // |sq| == 1: a column of the local system is contiguous
    int lower_t, unit;
    int pw;
    __device__ __forceinline__ int row(int q) const { return lower_t ? q : pw - 1 - q; }
};

// Panels of up to this many blocks are staged by every CTA itself: their triangle is a few
// loads a thread, less than the packing launch (64 unknowns and sides with the caller's copy of
// B: 12.1 us a call; 16.4 from 100 unknowns on, with it), and both column buffers hold all
// there is.
constexpr int SELF_BLOCKS = 3;

// Packs the panel: CTA (bi, bj), bi >= bj, writes the 32 x 32 block of rows 32 bi, columns 32 bj.
__global__ void __launch_bounds__(256) pack_kernel(const Panel p, int nb, float *image)
{
    __shared__ float tile[BLK][BLK + 1];   // [column][row]
    int bi = 0, left = blockIdx.x;
    while (left > bi) left -= ++bi;
    const int bj = left, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int c = 0; c < BLK / WARPS; ++c) {
        const int a = w + WARPS * c;   // lanes along the contiguous direction of A
        const int i = p.along_q ? lane : a, j = p.along_q ? a : lane;
        const int q = bi * BLK + i, d = bj * BLK + j;
        tile[j][i] = q > d && q < p.pw ? p.A0[(int64_t)q * p.sq + (int64_t)d * p.sd] : 0.f;
    }
    __syncthreads();
    float *dst = bi == bj ? image + 2 * BLK * nb + bi * BLK * BLK
                          : image + columns_at(nb, bj) + (bi - bj - 1) * BLK;
    const int pitch = bi == bj ? BLK : below(nb, bj);
#pragma unroll
    for (int c = 0; c < BLK / WARPS; ++c) {
        const int j = w + WARPS * c;
        dst[j * pitch + lane] = tile[j][lane];
    }
    if (bi == bj && w == 0) {
        const int q = bi * BLK + lane;
        const float t = !p.unit && q < p.pw ? p.A0[(int64_t)q * (p.sq + p.sd)] : 1.f;
        image[q] = t;
        image[nb * BLK + q] = 1.f / t;
    }
}

__device__ __forceinline__ uint32_t saddr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// One thread: a bulk copy of n floats into shared memory, completing on *bar.
__device__ __forceinline__ void fetch(float *dst, const float *src, int n, unsigned long long *bar)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(bar)),
                 "r"(4 * n)
                 : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(saddr(dst)), "l"(src), "r"(4 * n), "r"(saddr(bar))
        : "memory");
}

// Waits for a phase of *bar; false if it gave up after budget_ns.
__device__ __forceinline__ bool arrived(unsigned long long *bar, uint32_t parity,
                                        unsigned long long budget_ns)
{
    unsigned long long t0 = 0;
    for (long long it = 0; it < (1ll << 32); ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(saddr(bar)), "r"(parity)
            : "memory");
        if (done) return true;
        if ((it & 63) == 63) {
            unsigned long long t;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            if (t0 == 0) t0 = t;
            if (t - t0 > budget_ns) break;
        }
    }
    return false;
}

// Block bk's right-hand side of this lane solved with every special value: b / t is
// (b r corrected by one exact residual step), a zero, infinite or NaN t or a non-finite b
// makes that non-finite and takes the division itself.
__device__ __noinline__ void solve_block_exact(Smem &sm, int nb, int bk, float *x)
{
    const float *t = sm.head + bk * BLK, *r = t + nb * BLK;
    const float *tri = sm.head + 2 * BLK * nb + bk * BLK * BLK;
    for (int j = 0; j < BLK; ++j) {
        const float b = x[j * XP], q0 = b * r[j];
        float q = fmaf(fmaf(-t[j], q0, b), r[j], q0);
        if (!isfinite(q)) q = b / t[j];
        x[j * XP] = q;
        for (int i = j + 1; i < BLK; ++i)
            x[i * XP] = fmaf(-tri[j * BLK + i], q, x[i * XP]);
    }
}

// One warp solves block bk: lane l takes right-hand side l % 16 (the upper half repeats).  The
// quotients' special values are left to a second run of the block when one is not finite
// (with finite values both give the same bits); nothing is stored before the end, so that the
// triangle's reads run ahead of the chain.
__device__ __forceinline__ void solve_block(Smem &sm, int nb, int bk)
{
    const int v = threadIdx.x & (NV - 1);
    float *x = sm.x + bk * BLK * XP + v;
    const float *t = sm.head + bk * BLK, *r = t + nb * BLK;
    const float *tri = sm.head + 2 * BLK * nb + bk * BLK * BLK;
    float b[BLK], q[BLK];
#pragma unroll
    for (int i = 0; i < BLK; ++i) b[i] = x[i * XP];
    float finite = 0.f;   // stays zero while every quotient is finite
#pragma unroll
    for (int j = 0; j < BLK; ++j) {
        const float q0 = b[j] * r[j];
        q[j] = fmaf(fmaf(-t[j], q0, b[j]), r[j], q0);   // unit diagonal: t = r = 1, exact
        finite = fmaf(q[j], 0.f, finite);
        const float2 nx = make_float2(-q[j], -q[j]);
        // rows on and above the diagonal hold zeros here and are done with
#pragma unroll
        for (int i = (j + 1) & ~3; i < BLK; i += 4) {
            const float4 a = *reinterpret_cast<const float4 *>(tri + j * BLK + i);
            const float2 lo = __ffma2_rn(make_float2(a.x, a.y), nx, make_float2(b[i], b[i + 1]));
            const float2 hi =
                __ffma2_rn(make_float2(a.z, a.w), nx, make_float2(b[i + 2], b[i + 3]));
            b[i] = lo.x;
            b[i + 1] = lo.y;
            b[i + 2] = hi.x;
            b[i + 3] = hi.y;
        }
    }
    if (__any_sync(0xffffffffu, !(finite == 0.f))) {
        if ((threadIdx.x & 31) < NV) solve_block_exact(sm, nb, bk, x);
        return;
    }
#pragma unroll
    for (int j = 0; j < BLK; ++j) x[j * XP] = q[j];
}

// Rows 16 unit .. 16 unit + 15 below the block lose its unknowns (negated in nx): 8 rows a half
// warp, a right-hand side per lane.
__device__ __forceinline__ void update_rows(Smem &sm, int nb, int bk, int unit,
                                            const float2 (&nx)[BLK])
{
    const int lane = threadIdx.x & 31, v = lane & (NV - 1);
    const int i0 = unit * 16 + (lane >> 4) * 8, pitch = below(nb, bk);
    const float *col = sm.col[bk & 1] + i0;
    float *x = sm.x + ((bk + 1) * BLK + i0) * XP + v;
    float2 acc[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = make_float2(x[2 * i * XP], x[(2 * i + 1) * XP]);
#pragma unroll
    for (int j = 0; j < BLK; ++j) {
        const float4 a = *reinterpret_cast<const float4 *>(col + j * pitch);
        const float4 b = *reinterpret_cast<const float4 *>(col + j * pitch + 4);
        acc[0] = __ffma2_rn(make_float2(a.x, a.y), nx[j], acc[0]);
        acc[1] = __ffma2_rn(make_float2(a.z, a.w), nx[j], acc[1]);
        acc[2] = __ffma2_rn(make_float2(b.x, b.y), nx[j], acc[2]);
        acc[3] = __ffma2_rn(make_float2(b.z, b.w), nx[j], acc[3]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        x[2 * i * XP] = acc[i].x;
        x[(2 * i + 1) * XP] = acc[i].y;
    }
}

// Copies between B and the right-hand sides in shared memory, lanes along B's contiguous
// direction; element q of side v at B[v vstride + row(q) estride].
template <bool STORE>
__device__ __forceinline__ void move_sides(const Panel &p, float *B, int64_t vstride,
                                           int64_t estride, int nvec, int padded, Smem &sm)
{
    const int v0 = blockIdx.x * NV, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    auto move = [&](int q, int v) {
        const bool in = q < p.pw && v0 + v < nvec;
        float *g = B + (int64_t)(v0 + v) * vstride + (int64_t)p.row(q) * estride;
        if (STORE) {
            if (in) *g = sm.x[q * XP + v];
        } else {
            sm.x[q * XP + v] = in ? *g : 0.f;
        }
    };
    if (vstride == 1) {
#pragma unroll 8
        for (int q = 2 * w + (lane >> 4); q < padded; q += 2 * WARPS) move(q, lane & (NV - 1));
    } else {
#pragma unroll 4
        for (int q = lane; q < padded; q += 32) {
            move(q, 2 * w);
            move(q, 2 * w + 1);
        }
    }
}
static_assert(NV == 2 * WARPS, "two sides a warp");

// The whole triangle of a panel of at most SELF_BLOCKS blocks, straight into the images.
__device__ __forceinline__ void stage_self(const Panel &p, int nb, Smem &sm)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int bi = 0; bi < nb; ++bi)
        for (int bj = 0; bj <= bi; ++bj) {
            float *dst = bi == bj ? sm.head + 2 * BLK * nb + bi * BLK * BLK
                                  : sm.col[bj] + (bi - bj - 1) * BLK;
            const int pitch = bi == bj ? BLK : below(nb, bj);
#pragma unroll
            for (int c = 0; c < BLK / WARPS; ++c) {
                const int a = w + WARPS * c;   // lanes along the contiguous direction of A
                const int i = p.along_q ? lane : a, j = p.along_q ? a : lane;
                const int q = bi * BLK + i, d = bj * BLK + j;
                dst[j * pitch + i] =
                    q > d && q < p.pw ? p.A0[(int64_t)q * p.sq + (int64_t)d * p.sd] : 0.f;
            }
        }
    const int q = threadIdx.x;
    if (q < nb * BLK) {
        const float t = !p.unit && q < p.pw ? p.A0[(int64_t)q * (p.sq + p.sd)] : 1.f;
        sm.head[q] = t;
        sm.head[nb * BLK + q] = 1.f / t;
    }
}
static_assert(SELF_BLOCKS <= 3 && SELF_BLOCKS * BLK <= WARPS * 32, "two column buffers, one pass");

__global__ void __launch_bounds__(WARPS * 32, 1)
    panel_kernel(float *B, int64_t vstride, int64_t estride, int nvec, const Panel p,
                 const float *image, unsigned int *status, unsigned long long wait_ns,
                 int inject_timeout)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5;
    const int nb = (p.pw + BLK - 1) / BLK;
    const bool self = image == nullptr;
    const bool plain = !self && status == nullptr;   // staged by the threads: nothing to wait for
    auto fetch_columns = [&](int bk) {   // block bk's columns below it, if there are any
        if (bk + 1 < nb)
            fetch(sm.col[bk & 1], image + columns_at(nb, bk), BLK * below(nb, bk),
                  &sm.full[bk & 1]);
    };
    auto copy = [&](float *dst, const float *src, int n) {
        for (int i = 4 * tid; i < n; i += 4 * WARPS * 32)
            *reinterpret_cast<float4 *>(dst + i) = *reinterpret_cast<const float4 *>(src + i);
    };
    auto copy_columns = [&](int bk) {
        if (bk + 1 < nb) copy(sm.col[bk & 1], image + columns_at(nb, bk), BLK * below(nb, bk));
    };
    if (tid == 0) {
        for (int i = 0; i < 3; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&sm.full[i]))
                         : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (!self && !plain) {
            if (!(inject_timeout && blockIdx.x == 0))   // test hook: its first copy never starts
                fetch(sm.head, image, head_floats(nb), &sm.full[2]);
            fetch_columns(0);
            fetch_columns(1);
        }
    }
    if (self) stage_self(p, nb, sm);
    if (plain) {
        copy(sm.head, image, head_floats(nb));
        copy_columns(0);
        copy_columns(1);
    }
    move_sides<false>(p, B, vstride, estride, nvec, nb * BLK, sm);
    __syncthreads();
    const bool staged = self || plain;
    // all threads go on or give up together
    bool ok = __syncthreads_and(staged || arrived(&sm.full[2], 0, wait_ns));
    if (warp == 0 && ok) solve_block(sm, nb, 0);
    __syncthreads();
    int bk = 0;
    for (; bk + 1 < nb && ok; ++bk) {
        float2 nx[BLK];
        const float *x = sm.x + bk * BLK * XP + (tid & (NV - 1));
#pragma unroll
        for (int j = 0; j < BLK; ++j) {
            const float v = -x[j * XP];
            nx[j] = make_float2(v, v);
        }
        ok = staged || arrived(&sm.full[bk & 1], (bk >> 1) & 1, wait_ns);
        const int units = (nb - 1 - bk) * (BLK / 16);
        if (warp < 2) {
            update_rows(sm, nb, bk, warp, nx);   // the next block's rows
            asm volatile("bar.sync 1, 64;" ::: "memory");
        }
        if (warp == 0) {
            solve_block(sm, nb, bk + 1);
        } else {
            for (int u = 1 + warp; u < units; u += WARPS - 1) update_rows(sm, nb, bk, u, nx);
        }
        ok = __syncthreads_and(ok);
        // into the buffer just read
        if (plain)
            copy_columns(bk + 2);
        else if (tid == 0 && ok && !self)
            fetch_columns(bk + 2);
    }
    if (!ok) {
        // a copy never arrived: leave B as it is, and no copy behind (fetched, not awaited yet)
        if (tid == 0) {
            atomicOr(status, STATUS_WAIT_TIMEOUT);
            for (int b = bk; b < bk + 2 && b + 1 < nb; ++b)
                arrived(&sm.full[b & 1], (b >> 1) & 1, wait_ns);
        }
        return;
    }
    move_sides<true>(p, B, vstride, estride, nvec, nb * BLK, sm);
}

}  // namespace trsm32

bool trsm_packs(int pw)
{
    return pw > trsm32::SELF_BLOCKS * trsm32::BLK;
}

size_t trsm_image_bytes(int pw)
{
    const int nb = (pw + trsm32::BLK - 1) / trsm32::BLK;
    return sizeof(float) * (size_t)trsm32::columns_at(nb, nb - 1);
}

cudaError_t launch_trsm_panel_f32(float *B, int64_t vstride, int64_t estride, int nvec,
                                  const float *A, int64_t lda, int a_trans, int k0, int pw,
                                  int lower_t, int transpose_t, int unit, float *image,
                                  unsigned int *status, unsigned long long wait_ns,
                                  int inject_timeout, cudaStream_t s)
{
    using namespace trsm32;
    if (nvec <= 0 || pw <= 0) return cudaSuccess;
    if (pw > TRSM_PANEL) return cudaErrorInvalidValue;
    static bool configured = false;
    if (!configured) {
        const cudaError_t e =
            cudaFuncSetAttribute(panel_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(sizeof(Smem)));
        if (e != cudaSuccess) return e;
        configured = true;
    }
    // t(q, d): row index i and column index j of op(A) are k0 + r0 + sgn q and k0 + r0 + sgn d
    // (swapped for side 'R'); op(A)[i, j] is element i + j lda ('N') or j + i lda ('T')
    Panel p;
    const int64_t ci = a_trans ? lda : 1, cj = a_trans ? 1 : lda;
    const int64_t cq = transpose_t ? cj : ci, cd = transpose_t ? ci : cj;
    const int sgn = lower_t ? 1 : -1;
    p.A0 = A + (int64_t)(k0 + (lower_t ? 0 : pw - 1)) * (cq + cd);
    p.sq = sgn * cq;
    p.sd = sgn * cd;
    p.along_q = cq == 1;
    p.lower_t = lower_t;
    p.unit = unit;
    p.pw = pw;
    const int nb = (pw + BLK - 1) / BLK;
    if (!trsm_packs(pw))
        image = nullptr;
    else
        pack_kernel<<<nb * (nb + 1) / 2, 256, 0, s>>>(p, nb, image);
    panel_kernel<<<(nvec + NV - 1) / NV, WARPS * 32, sizeof(Smem), s>>>(
        B, vstride, estride, nvec, p, image, status, wait_ns, inject_timeout);
    return cudaGetLastError();
}

}  // namespace gfip
