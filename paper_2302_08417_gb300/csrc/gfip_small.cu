// gfip_small.cu -- GEMM kernels for small products: one launch, no packing, no workspace words,
// no CTA waits for or counts another.
//
// Below a few hundred rows the persistent cores lose their time around the arithmetic: one or
// two k blocks per CTA, partial tiles through global memory, arrival counters, and tiles padded
// to 32 x 32 (FP64) or 128 x 128 (FP32).  Nothing is reused often enough here to be worth
// packing (Sec. 3.3: every operand is read where it lies), so the kernels below cut C into
// small tiles, one CTA each, split k over the CTA's warps and add the warps' sums in warp
// order through shared memory.
//
// Where C has too few tiles to cover the SMs, a cluster of 2, 4 or 8 CTAs shares a tile's k;
// the first CTA receives the others' sums through distributed shared memory and adds them in
// rank order.
#include <algorithm>
#include <cstdint>

#include "gfip_internal.h"

namespace gfip {
namespace small {

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.aligned;\n barrier.cluster.wait.aligned;" ::: "memory");
}

// Address of the same shared-memory variable in the cluster's first CTA.
__device__ __forceinline__ uint32_t in_first(const void *p)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;"
                 : "=r"(r)
                 : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))));
    return r;
}

__device__ __forceinline__ void store_first(void *p, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(in_first(p)), "d"(v) : "memory");
}

__device__ __forceinline__ void store_first(void *p, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(in_first(p)), "f"(v) : "memory");
}

// Part of C (SYRK) and of k (TRMM) that the MASKED kernels leave out.

// Rows x0 .. x0 + T - 1 of C against columns y0 .. y0 + T - 1: a tile of the requested triangle?
template <int T> __device__ __forceinline__ bool tile_in(int tri, int i0, int j0)
{
    return tri == TRI_LOWER ? i0 + T - 1 >= j0 : tri == TRI_UPPER ? i0 <= j0 + T - 1 : true;
}

__device__ __forceinline__ bool elem_in(int tri, int i, int j)
{
    return tri == TRI_LOWER ? i >= j : tri == TRI_UPPER ? i <= j : true;
}

// Whether a triangular operand keeps element (x, k); a dense one (mask 0) keeps all.
__device__ __forceinline__ bool keeps(int mask, int64_t x, int64_t k)
{
    const int s = (mask & TMASK_STRICT) ? 1 : 0;
    return !(mask & TMASK_ON) || ((mask & TMASK_KEEP_GE) ? x - k >= s : k - x >= s);
}

// The k that rows x0 .. x0 + T - 1 of a triangular operand keep anything of.
template <int T> __device__ __forceinline__ void k_range(int mask, int x0, int64_t &lo, int64_t &hi)
{
    if (!(mask & TMASK_ON)) return;
    const int64_t s = (mask & TMASK_STRICT) ? 1 : 0;
    if (mask & TMASK_KEEP_GE)
        hi = min(hi, x0 + T - s);
    else
        lo = max(lo, x0 + s);
}

// ---- FP64 ----------------------------------------------------------------------------------
//
// 8 x 8 tiles; a lane owns two elements.  The FP64 units take one warp instruction per 64
// clocks, so operands come straight from L1 (three loads per two DFMAs) and the tile is as
// small as that allows: its padding is at most 7 rows or columns.  Either the CTA's four warps
// (one per FP64 unit of the SM) share a tile, each taking every fourth group of U rows of k
// (KW = 4: 256^3 gives 1024 tiles, 6.7 a SM), or each warp has a tile of its own (KW = 1: no sums
// to add, which cost as much DFMA time as 3 rows of k).  Bound: the DFMA pipe, and launch
// plus load latency below 100^3.
// 16^3 9.8 -> 2.1 us, 128^3 19.3 -> 6.4, 256^3 59.9 -> 31.6, 512^3 243 -> 222, 2048^3
// 13923 -> 13755 (1.249 of 1.259 TFLOP/s) against the persistent core; 64 x 64 x 8192 283 -> 101.

constexpr int DT = 8, DWARPS = 4, U = 4;

template <bool ACONTIG, bool BCONTIG, int CS, int KW, bool MASKED>
__global__ void __launch_bounds__(DWARPS * 32) dgemm_kernel(const SmallParams<double> p)
{
    static_assert(KW == 1 || KW == DWARPS, "a tile per warp or per CTA");
    static_assert(CS == 1 || KW == DWARPS, "clusters share a CTA's tile");
    __shared__ double part[DWARPS - 1][2][32];
    __shared__ double ranks[CS > 1 ? CS - 1 : 1][2][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int w = KW > 1 ? warp : 0;   // this warp's part of the tile's k
    const int rank = CS > 1 ? static_cast<int>(cluster_rank()) : 0;
    const int tile = KW > 1 ? blockIdx.x / CS : blockIdx.x * DWARPS + warp;
    if (KW == 1 && tile >= p.tiles) return;
    const int i0 = (tile % p.mt) * DT, j0 = (tile / p.mt) * DT;
    int64_t klo = 0, khi = p.k;
    if (MASKED) {
        if (!tile_in<DT>(p.tri, i0, j0)) return;   // the whole cluster
        k_range<DT>(p.tmask_a, i0, klo, khi);
        k_range<DT>(p.tmask_b, j0, klo, khi);
    }
    const int r = lane & 7, c = lane >> 3;          // elements (r, c) and (r, c + 4)
    // rows and columns beyond the edge repeat the last one; their sums are not stored
    const int row = i0 + r, col0 = j0 + c, col1 = col0 + 4;
    const int ar = min(row, p.m - 1), b0 = min(col0, p.n - 1), b1 = min(col1, p.n - 1);
    const int64_t as = ACONTIG ? p.lda : 1, bs = BCONTIG ? p.ldb : 1;
    const double *A = p.A + (ACONTIG ? ar : (int64_t)ar * p.lda);
    const double *B0 = p.B + (BCONTIG ? b0 : (int64_t)b0 * p.ldb);
    const double *B1 = p.B + (BCONTIG ? b1 : (int64_t)b1 * p.ldb);
    constexpr int STEP = CS * KW * U;   // k from one of this warp's groups to its next
    double s0 = 0.0, s1 = 0.0;
    int64_t k = klo + (rank * KW + w) * U;
    auto load_a = [&](int u) {
        return !MASKED || keeps(p.tmask_a, ar, k + u) ? __ldg(A + u * as) : 0.0;
    };
    auto load_b0 = [&](int u) {
        return !MASKED || keeps(p.tmask_b, b0, k + u) ? __ldg(B0 + u * bs) : 0.0;
    };
    auto load_b1 = [&](int u) {
        return !MASKED || keeps(p.tmask_b, b1, k + u) ? __ldg(B1 + u * bs) : 0.0;
    };
    A += k * as;
    B0 += k * bs;
    B1 += k * bs;
    double a[U], x[U], y[U];
    if (k + U <= khi) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            a[u] = load_a(u);
            x[u] = load_b0(u);
            y[u] = load_b1(u);
        }
        // the next group's loads are under way while this one's multiply-adds run
        while (k + STEP + U <= khi) {
            k += STEP;
            A += STEP * as;
            B0 += STEP * bs;
            B1 += STEP * bs;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                s0 = fma(a[u], x[u], s0);
                s1 = fma(a[u], y[u], s1);
                a[u] = load_a(u);
                x[u] = load_b0(u);
                y[u] = load_b1(u);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            s0 = fma(a[u], x[u], s0);
            s1 = fma(a[u], y[u], s1);
        }
        k += STEP;
        A += STEP * as;
        B0 += STEP * bs;
        B1 += STEP * bs;
    }
#pragma unroll 1
    for (int u = 0; u < U && k + u < khi; ++u) {   // the ragged last group
        const double t = load_a(u);
        s0 = fma(t, load_b0(u), s0);
        s1 = fma(t, load_b1(u), s1);
    }
    if (w > 0) {
        part[w - 1][0][lane] = s0;
        part[w - 1][1][lane] = s1;
    }
    const bool read_c = p.beta != 0.0;
    double *C0 = p.C + row + (int64_t)col0 * p.ldc, *C1 = p.C + row + (int64_t)col1 * p.ldc;
    const bool in0 = row < p.m && col0 < p.n && (!MASKED || elem_in(p.tri, row, col0));
    const bool in1 = row < p.m && col1 < p.n && (!MASKED || elem_in(p.tri, row, col1));
    double c0 = 0.0, c1 = 0.0;
    if (w == 0 && rank == 0 && read_c) {
        if (in0) c0 = *C0;
        if (in1) c1 = *C1;
    }
    if constexpr (KW > 1) {
        __syncthreads();
        if (w == 0) {
#pragma unroll
            for (int q = 0; q < DWARPS - 1; ++q) {
                s0 += part[q][0][lane];
                s1 += part[q][1][lane];
            }
        }
    }
    if constexpr (CS > 1) {
        cluster_sync();   // the first CTA runs: its shared memory can be written
        if (w == 0 && rank > 0) {
            store_first(&ranks[rank - 1][0][lane], s0);
            store_first(&ranks[rank - 1][1][lane], s1);
        }
        cluster_sync();
        if (rank > 0) return;
    }
    if (w > 0) return;
    if constexpr (CS > 1) {
#pragma unroll
        for (int q = 0; q < CS - 1; ++q) {
            s0 += ranks[q][0][lane];
            s1 += ranks[q][1][lane];
        }
    }
    if (p.alpha != 1.0) {
        s0 *= p.alpha;
        s1 *= p.alpha;
    }
    if (in0) *C0 = read_c ? fma(p.beta, c0, s0) : s0;
    if (in1) *C1 = read_c ? fma(p.beta, c1, s1) : s1;
}

// ---- FP32 ----------------------------------------------------------------------------------
//
// A 32 x 32 tile per CTA of eight warps.  All threads copy a slab of 64 k of both operands
// through registers into shared memory (one k per 128-byte row, its 16-byte chunks
// XOR-permuted by k % 8, so copies from either operand order and the fragment reads are free
// of bank conflicts); each warp multiplies 8 of the slab's rows, 8 x 4 elements a lane.
// Bound: load latency, then the load/store pipe (a slab is 512 clocks of FFMA, 768 of fragment
// reads and about 400 of copies).
// 16^3 11.1 -> 2.5 us, 128^3 22.9 -> 3.8, 256^3 54.8 -> 4.7, 512^3 59.8 -> 14.5, 64 x 64 x 8192
// 193 -> 17.9 against the FFMA core.

constexpr int ST = 32, SWARPS = 8, SK = 64;
constexpr int SPER = ST * SK / (SWARPS * 32);   // elements of each operand's slab a thread copies

__device__ __forceinline__ int slab_at(int x, int k)
{
    return k * ST + (((x >> 2) ^ (k & 7)) << 2) + (x & 3);
}

// This thread's q-th element of a slab: lanes along the contiguous direction of memory.
template <bool CONTIG> __device__ __forceinline__ void slab_xk(int q, int &x, int &k)
{
    const int t = threadIdx.x;
    if (CONTIG) {
        x = t & 31;
        k = (t >> 5) + SWARPS * q;
    } else {   // 8 k of 4 rows a warp
        k = (t & 7) + 8 * (q & 7);
        x = (t >> 3) + 32 * (q >> 3);
    }
}

template <bool CONTIG, bool MASKED>
__device__ __forceinline__ void slab_load(const float *X, int64_t ld, int x0, int xn, int64_t k0,
                                          int64_t kn, int mask, float (&v)[SPER])
{
#pragma unroll
    for (int q = 0; q < SPER; ++q) {
        int x, k;
        slab_xk<CONTIG>(q, x, k);
        const int64_t gx = x0 + x, gk = k0 + k;
        const bool in = gx < xn && gk < kn && (!MASKED || keeps(mask, gx, gk));
        v[q] = in ? __ldg(X + (CONTIG ? gx + gk * ld : gk + gx * ld)) : 0.f;
    }
}

template <bool CONTIG> __device__ __forceinline__ void slab_store(float *s, const float (&v)[SPER])
{
#pragma unroll
    for (int q = 0; q < SPER; ++q) {
        int x, k;
        slab_xk<CONTIG>(q, x, k);
        s[slab_at(x, k)] = v[q];
    }
}

template <bool ACONTIG, bool BCONTIG, int CS, bool MASKED>
__global__ void __launch_bounds__(SWARPS * 32, 2) sgemm_kernel(const SmallParams<float> p)
{
    // slabs of A and B; then the warps' sums
    __shared__ __align__(16) float sm[SWARPS * ST * ST];
    static_assert(2 * SK * ST <= SWARPS * ST * ST, "the slabs fit the sums' buffer");
    float *sa = sm, *sb = sm + SK * ST;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int rank = CS > 1 ? static_cast<int>(cluster_rank()) : 0;
    const int tile = blockIdx.x / CS;
    const int i0 = (tile % p.mt) * ST, j0 = (tile / p.mt) * ST;
    int64_t klo = 0, khi = p.k;
    if (MASKED) {
        if (!tile_in<ST>(p.tri, i0, j0)) return;   // the whole cluster
        k_range<ST>(p.tmask_a, i0, klo, khi);
        k_range<ST>(p.tmask_b, j0, klo, khi);
    }
    const int tx = lane & 3, ty = lane >> 2;   // rows 4 tx + {0..3}, + 16; columns 4 ty + {0..3}
    float acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    float va[SPER], vb[SPER];
    const int64_t first = klo + rank * SK;
    slab_load<ACONTIG, MASKED>(p.A, p.lda, i0, p.m, first, khi, p.tmask_a, va);
    slab_load<BCONTIG, MASKED>(p.B, p.ldb, j0, p.n, first, khi, p.tmask_b, vb);
    for (int64_t k0 = first; k0 < khi; k0 += CS * SK) {
        slab_store<ACONTIG>(sa, va);
        slab_store<BCONTIG>(sb, vb);
        __syncthreads();
        if (k0 + CS * SK < khi) {
            slab_load<ACONTIG, MASKED>(p.A, p.lda, i0, p.m, k0 + CS * SK, khi, p.tmask_a, va);
            slab_load<BCONTIG, MASKED>(p.B, p.ldb, j0, p.n, k0 + CS * SK, khi, p.tmask_b, vb);
        }
        // the warp's 8 rows (zeros beyond k): row u of the group sits at chunk position ^ u
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int k = w * 8 + u;
            const float4 a0 = *reinterpret_cast<const float4 *>(sa + k * ST + ((tx ^ u) << 2));
            const float4 a1 =
                *reinterpret_cast<const float4 *>(sa + k * ST + (((tx + 4) ^ u) << 2));
            const float4 b = *reinterpret_cast<const float4 *>(sb + k * ST + ((ty ^ u) << 2));
            const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
        __syncthreads();
    }
    // sums of warp w at [w][column][row]
    float *mine = sm + w * ST * ST;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        *reinterpret_cast<float4 *>(mine + (ty * 4 + j) * ST + tx * 4) =
            make_float4(acc[0][j], acc[1][j], acc[2][j], acc[3][j]);
        *reinterpret_cast<float4 *>(mine + (ty * 4 + j) * ST + 16 + tx * 4) =
            make_float4(acc[4][j], acc[5][j], acc[6][j], acc[7][j]);
    }
    const bool read_c = p.beta != 0.f;
    const int row = i0 + lane;
    float cv[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int col = j0 + w + SWARPS * q;
        const bool in = row < p.m && col < p.n && (!MASKED || elem_in(p.tri, row, col));
        cv[q] = (read_c && in) ? p.C[row + (int64_t)col * p.ldc] : 0.f;
    }
    __syncthreads();
    float sum[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int at = (w + SWARPS * q) * ST + lane;
        sum[q] = sm[at];
#pragma unroll
        for (int g = 1; g < SWARPS; ++g) sum[q] += sm[g * ST * ST + at];
    }
    if constexpr (CS > 1) {
        cluster_sync();   // the first CTA has added its warps' sums: its buffer is free
        if (rank > 0) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                store_first(&sm[(rank - 1) * ST * ST + (w + SWARPS * q) * ST + lane], sum[q]);
        }
        cluster_sync();
        if (rank > 0) return;
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int g = 0; g < CS - 1; ++g)
                sum[q] += sm[g * ST * ST + (w + SWARPS * q) * ST + lane];
    }
    if (row >= p.m) return;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int col = j0 + w + SWARPS * q;
        if (col >= p.n || (MASKED && !elem_in(p.tri, row, col))) continue;
        const float s = sum[q] * p.alpha;
        p.C[row + (int64_t)col * p.ldc] = read_c ? fmaf(p.beta, cv[q], s) : s;
    }
}

// Clocks on the busiest SM with cs CTAs per tile: a CTA takes `per_k` clocks per k and about `fixed`
// around its k loop, a cluster 1500 more.  `wait`: clocks per k that its loads take beyond that.
inline int64_t clocks_of(int cs, int64_t tiles, int64_t k, int64_t per_k, int64_t fixed,
                         int64_t wait, int sms)
{
    const int64_t rounds = (tiles * cs + sms - 1) / sms;
    // the other CTAs of the SM hide the wait
    return (k + cs - 1) / cs * std::max(rounds * per_k, per_k + wait) + rounds * fixed +
           (cs > 1 ? 1500 : 0);
}

// CTAs per tile: the fewest clocks.
inline int cluster_size(int64_t tiles, int64_t k, int64_t group, int64_t per_k, int64_t fixed,
                        int64_t wait, int sms)
{
    int best = 1;
    int64_t least = 0;
    for (int cs = 1; cs <= 8; cs *= 2) {
        if (cs > 1 && cs * group > k) break;
        const int64_t cost = clocks_of(cs, tiles, k, per_k, fixed, wait, sms);
        if (cs == 1 || cost < least) {
            best = cs;
            least = cost;
        }
    }
    return best;
}

// FP64: a CTA's 8 x 8 tile takes 32 DFMA clocks per k.
constexpr int64_t DCLOCKS = 32, DFIXED = 1000;

// Its warps load one group ahead.  Alone on its SM a CTA waits 10 clocks per k more for L2
// (8 x 8 x 200000: 313 ns a step), and up to 36 for HBM, where operands come from that do not stay
// in L2 (from about 50 to 60 MB on), or 60 when one lies along k and the other across (8 x 8 x
// 4000000: 560 and 730 ns a step).
inline int64_t dgemm_wait(int64_t mb, bool mixed)
{
    return mixed ? std::min<int64_t>(60, 14 + std::max<int64_t>(0, mb - 50) * 7 / 4)
                 : std::min<int64_t>(36, 10 + std::max<int64_t>(0, mb - 64) * 2 / 3);
}

// CTAs per tile, FP64: by the DFMA clocks, and by the wait as well where it is HBM's.  (By the DFMA
// clocks alone, 64 x 64 x 200000 ran on 128 CTAs in 3.1 to 4.0 ms.)
inline int dgemm_cluster(int64_t run, int64_t m, int64_t n, int64_t k, int tri, bool mixed,
                         int sms)
{
    const int64_t mb = ((tri == TRI_NONE ? m + n : m) * k) >> 17;
    return cluster_size(run, k, DWARPS * U, DCLOCKS, DFIXED, mb > 50 ? dgemm_wait(mb, mixed) : 0,
                        sms);
}

// Tiles that are not left out: about half of a triangle's square.
inline int64_t computed(int64_t tiles, int tri)
{
    return tri == TRI_NONE ? tiles : (tiles + 1) / 2;
}

template <typename T, typename Kernel>
cudaError_t launch(Kernel kernel, const SmallParams<T> &p, unsigned int blocks, int threads, int cs,
                   cudaStream_t s)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks * cs);
    cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = cs;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = cs > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, p);
}

template <bool AC, bool BC, bool MASKED>
cudaError_t launch_mask(const SmallParams<double> &p, unsigned int blocks, int cs, cudaStream_t s)
{
    constexpr int T = DWARPS * 32;
    if constexpr (!MASKED)
        if (cs == 0) return launch(dgemm_kernel<AC, BC, 1, 1, false>, p, blocks, T, 1, s);
    switch (cs) {
    case 1: return launch(dgemm_kernel<AC, BC, 1, DWARPS, MASKED>, p, blocks, T, cs, s);
    case 2: return launch(dgemm_kernel<AC, BC, 2, DWARPS, MASKED>, p, blocks, T, cs, s);
    case 4: return launch(dgemm_kernel<AC, BC, 4, DWARPS, MASKED>, p, blocks, T, cs, s);
    default: return launch(dgemm_kernel<AC, BC, 8, DWARPS, MASKED>, p, blocks, T, cs, s);
    }
}

template <bool AC, bool BC, bool MASKED>
cudaError_t launch_mask(const SmallParams<float> &p, unsigned int blocks, int cs, cudaStream_t s)
{
    constexpr int T = SWARPS * 32;
    switch (cs) {
    case 1: return launch(sgemm_kernel<AC, BC, 1, MASKED>, p, blocks, T, cs, s);
    case 2: return launch(sgemm_kernel<AC, BC, 2, MASKED>, p, blocks, T, cs, s);
    case 4: return launch(sgemm_kernel<AC, BC, 4, MASKED>, p, blocks, T, cs, s);
    default: return launch(sgemm_kernel<AC, BC, 8, MASKED>, p, blocks, T, cs, s);
    }
}

template <bool AC, bool BC, typename T>
cudaError_t launch_order(const SmallParams<T> &p, unsigned int blocks, int cs, cudaStream_t s)
{
    return p.tri != TRI_NONE || p.tmask_a || p.tmask_b ? launch_mask<AC, BC, true>(p, blocks, cs, s)
                                                       : launch_mask<AC, BC, false>(p, blocks, cs, s);
}

template <typename T>
cudaError_t launch_any(const SmallParams<T> &p, unsigned int blocks, int cs, cudaStream_t s)
{
    if (p.a_contig_m)
        return p.b_contig_n ? launch_order<true, true>(p, blocks, cs, s)
                            : launch_order<true, false>(p, blocks, cs, s);
    return p.b_contig_n ? launch_order<false, true>(p, blocks, cs, s)
                        : launch_order<false, false>(p, blocks, cs, s);
}

}  // namespace small

int64_t small_dgemm_clocks(int64_t m, int64_t n, int64_t k, int tri, int a_contig_m,
                           int b_contig_n, int sms)
{
    using namespace small;
    const int64_t run = computed((m + DT - 1) / DT * ((n + DT - 1) / DT), tri);
    const bool mixed = a_contig_m != b_contig_n;
    const int cs = dgemm_cluster(run, m, n, k, tri, mixed, sms);
    const int64_t mb = ((tri == TRI_NONE ? m + n : m) * k) >> 17;
    const int64_t wait = dgemm_wait(mb, mixed), rounds = (run * cs + sms - 1) / sms;
    const int64_t clocks = clocks_of(cs, run, k, DCLOCKS, DFIXED, wait, sms);
    // large clusters over HBM do not spread evenly (128 x 64 x 500000: 7900 us, 6750 by the rounds)
    if (tri == TRI_NONE) return cs >= 4 && rounds > 2 && mb > 128 ? clocks + clocks / 6 : clocks;
    // the masked kernel's loads wait longer, most where both operands lie across k (SYRK 16 x
    // 300000 993 us along, 1512 across), and its CTAs hide little of it (64 x 64 x 300000 2343)
    return (k + cs - 1) / cs * (rounds * DCLOCKS + wait + (a_contig_m ? 40 : 15)) +
           rounds * DFIXED;
}

template <> cudaError_t launch_small<double>(SmallParams<double> p, int sms, cudaStream_t s,
                                               int *grid)
{
    using namespace small;
    p.mt = (p.m + DT - 1) / DT;
    const int64_t tiles = (int64_t)p.mt * ((p.n + DT - 1) / DT);
    p.tiles = static_cast<int>(tiles);
    const int64_t run = computed(tiles, p.tri);
    const bool mixed = p.a_contig_m != p.b_contig_n, across = p.a_contig_m && p.b_contig_n;
    int cs = dgemm_cluster(run, p.m, p.n, p.k, p.tri, mixed, sms);
    // A tile per warp, where there are enough, all are whole and no DFMA clocks are lost on the
    // busiest unit: 64 a row of k and element; 10 instructions end a shared tile (on one unit,
    // while the others go on), 4 an own one.  Within 1 % the own tile is taken, whose sums are
    // one chain in k order like the persistent core's; but not for a long k across which both
    // operands lie, where a warp's loads of a step touch 32 lines for its tile alone (N/T, us:
    // 500 x 1000 x 10000 9327 own, 8132 shared, 8586 the core; 1000^3 1688 and 1625; but
    // 4000 x 4000 x 100 2671 and 2833).
    const int64_t shared = (run + sms - 1) / sms * (p.k * 32 + 160);
    const int64_t own = (run + 4 * sms - 1) / (4 * sms) * (p.k * 128 + 256);
    const bool masked = p.tri != TRI_NONE || p.tmask_a || p.tmask_b;
    if (cs == 1 && !masked && !(across && p.k >= 512) && run >= 16 * sms && own * 100 <= shared * 101)
        cs = 0;
    const int64_t blocks = cs == 0 ? (tiles + DWARPS - 1) / DWARPS : tiles;
    *grid = static_cast<int>(blocks * std::max(cs, 1));
    return launch_any(p, static_cast<unsigned int>(blocks), cs, s);
}

template <> cudaError_t launch_small<float>(SmallParams<float> p, int sms, cudaStream_t s, int *grid)
{
    using namespace small;
    p.mt = (p.m + ST - 1) / ST;
    const int64_t tiles = (int64_t)p.mt * ((p.n + ST - 1) / ST);
    const int cs = cluster_size(computed(tiles, p.tri), p.k, SK, 22, 1500, 0, sms);
    *grid = static_cast<int>(tiles * cs);
    return launch_any(p, static_cast<unsigned int>(tiles), cs, s);
}

}  // namespace gfip
