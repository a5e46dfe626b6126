// gfip_internal.h -- host/device shared definitions of the fused-in-packing GEMM library.
// Not part of the public ABI (that is include/gemmfip.h).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace gfip {

// Where an operand's tiles come from in one launch of the GEMM kernel.
// Part of C a launch computes: all of it (GEMM), or one triangle of a square C (SYRK).
enum Triangle : int { TRI_NONE = 0, TRI_LOWER = 1, TRI_UPPER = 2 };

// Triangular operand (TRMM): element (x, k) of op(X) (x = row of op(A) or column of op(B),
// k = the summed index) is kept when x - k >= s (KEEP_GE) or k - x >= s, s = 1 for a strictly
// triangular operand (a unit diagonal is added separately), else s = 0; the rest is zero.
enum TriMask : int { TMASK_ON = 1, TMASK_KEEP_GE = 2, TMASK_STRICT = 4 };

enum OperandMode : int {
    MODE_RAW = 0,     // always read the raw strided operand (direct variant, SUP analog)
    MODE_PACKED = 1,  // always read the packed copy, written beforehand by the pack kernel
    MODE_FIP = 2,     // fused: the first tile line packs each (panel, k-block) while
                      // computing with it, later tiles read the packed copy once it is
                      // published (Sec. 3.1 Alg. 1, Sec. 3.2)
};

// Tile shape of one element type.  The CTA computes a BM x BN tile of C, stepping through
// k in blocks of BK; each thread owns an (NCM*CH) x (NCN*CH) register micro-tile (CH =
// elements per 16 bytes).
template <typename T> struct TileCfg;

// FP64: the DFMA pipe (2 lanes per clock per SM) is the bound at every size, so small tiles
// cost no throughput and give fine-grained work units that keep all SMs busy.
#ifndef GFIP_F64_BM
#define GFIP_F64_BM 32
#endif
#ifndef GFIP_F64_BN
#define GFIP_F64_BN 32
#endif
#ifndef GFIP_F64_MIN_BLOCKS
#define GFIP_F64_MIN_BLOCKS 6
#endif
#ifndef GFIP_F64_UNROLL
#define GFIP_F64_UNROLL 2
#endif
// A CTA runs at least 4 warps, one per SM sub-partition (each has its own FP64 unit), with
// 4 x 2 micro-tiles for tiles of up to 1024 elements and 4 x 4 above.
template <> struct TileCfg<double> {
    static constexpr int BM = GFIP_F64_BM, BN = GFIP_F64_BN, BK = 16;
    static constexpr int NCM = 2;
    static constexpr int NCN = (BM * BN / 128 >= 16) ? 2 : 1;       // 4 x 4 or 4 x 2 per thread
    static constexpr int THREADS = BM * BN / (4 * 2 * NCN) < 128 ? 128 : BM * BN / (4 * 2 * NCN);
    static constexpr int STAGES = 3;
    static constexpr int MIN_BLOCKS = GFIP_F64_MIN_BLOCKS;
    static constexpr int UNROLL = GFIP_F64_UNROLL;  // k rows per unrolled compute step
};
#ifndef GFIP_F32_MIN_BLOCKS
#define GFIP_F32_MIN_BLOCKS 2
#endif
#ifndef GFIP_F32_STAGES
#define GFIP_F32_STAGES 3
#endif
#ifndef GFIP_F32_BK
#define GFIP_F32_BK 32
#endif
#ifndef GFIP_F32_NCM
#define GFIP_F32_NCM 2
#endif

// FP32: 128 x 128 tiles, 8 x 8 per thread on 256 threads (NCM = NCN = 2 chunks of 4).
// Shared memory delivers 128 bytes per clock per SM and the FFMA pipe 128 lanes, so an 8 x 8
// micro-tile, reading (8 + 8) x 4 bytes per 64 FMAs, sits at the shared-memory limit; 16 x 8
// (NCM = 4, 128 threads) reads 0.75 B/FMA and measured 4 % faster at 8192 but 5-10 % slower
// at 1024-2048, where only 8 warps per SM are left to hide latency.
#ifndef GFIP_F32_UNROLL
#define GFIP_F32_UNROLL 16
#endif
template <> struct TileCfg<float> {
    static constexpr int BM = 128, BN = 128, BK = GFIP_F32_BK, NCM = GFIP_F32_NCM, NCN = 2;
    static constexpr int THREADS = BM * BN / (NCM * 4 * NCN * 4);
    static constexpr int UNROLL = GFIP_F32_UNROLL;
    static constexpr int STAGES = GFIP_F32_STAGES, MIN_BLOCKS = GFIP_F32_MIN_BLOCKS;
};

// Everything one launch of the GEMM kernel needs.  Plain data, passed by value.
template <typename T> struct GemmParams {
    const T *A;
    const T *B;
    T *C;
    int64_t lda, ldb, ldc;
    int m, n, k;
    T alpha, beta;
    int a_contig_m;   // 1: op(A)[i,p] = A[i + p*lda] (transa 'N'); 0: A[p + i*lda]
    int b_contig_n;   // 1: op(B)[p,j] = B[j + p*ldb] (transb 'T'); 0: B[p + j*ldb]
    int mt, nt, kt;   // tile counts along m, n and k
    int tiles;        // mt * nt
    int band;         // tile rows per band of the consumer tile order (>= 1)
    int tri;          // TRI_NONE: all of C; TRI_LOWER / TRI_UPPER: that triangle (SYRK)
    int a_produces;   // the first tile column packs the A panels
    int b_produces;   // the first tile row packs the B panels
    int shared_pack;  // all CTAs pack the packed operands' tiles first (no line producers)
    int64_t pack_units;  // shared packing: (panel, k-block) tiles to pack in all
    int tmask_a;      // triangular mask of op(A) (TRMM), 0 = dense; see TriMask
    int tmask_b;      // triangular mask of op(B)
    int grid;         // persistent CTAs
    int dp_tiles;     // tiles [0, dp_tiles) are data-parallel, taken in order from tile_next
    int64_t sk_iters; // (tiles - dp_tiles) * kt iterations split evenly over the CTAs
    int mode_a, mode_b;
    unsigned long long *state_a;     // [mt * kt] epoch-tagged ready words of packed A tiles,
                                     // then [mt] words "whole panel published"
    unsigned long long *state_b;     // [nt * kt + nt] same for B
    unsigned long long *tile_count;  // [tiles] epoch-tagged arrival counters of split tiles
    T *pack_a;                       // [mt * kt] tiles of BM * BK elements
    T *pack_b;                       // [nt * kt] tiles of BN * BK elements
    T *partial;                      // [grid * 2] slots of BM * BN elements
    unsigned int *status;            // device status bits (GFIP_STATUS_*)
    unsigned int *launch_count;      // launches so far (the epoch of a launch is this + 1)
    unsigned int *done_count;        // CTAs of the current launch that have finished
    unsigned long long *pack_count;  // shared packing: epoch-tagged count of packed tiles
    unsigned long long *tile_next;   // epoch-tagged count of data-parallel tiles taken
    unsigned int *gate;              // nullable (FP32): the launch does nothing while the word is
                                     // zero, and clears it when it has run
    unsigned long long wait_ns;      // FP32: budget of every mbarrier wait (nanoseconds)
    int inject_timeout;              // FP32 test hook: CTA 0 withholds its first operand's arrival
};

// Parameters of the pack kernel of the pack-then-compute variant.
template <typename T> struct PackParams {
    const T *A;
    const T *B;
    int64_t lda, ldb;
    int m, n, k;
    int a_contig_m, b_contig_n;
    int mt, nt, kt;
    T *pack_a;
    T *pack_b;
};

// One launch of the tensor-core tile core (gfip_tc.cuh): both operands split into `planes`
// BF16 planes, plane tiles of 128 rows x 32 k (8 KB, swizzled as the MMA reads them), laid out
// [128-row block][k block][plane].
struct TcParams {
    const uint8_t *pa;   // planes of op(A), rows of C
    const uint8_t *pb;   // planes of op(B), columns of C
    void *C;             // double (digits) or float
    int64_t ldc;
    int m, n;
    double alpha, beta;
    int planes;
    int mt, nt, kt;      // 128-row blocks of m and n, 32-wide k blocks
    int tiles;           // tiles of C computed
    int tri;             // TRI_*: the triangle of C computed (SYRK)
    int tmask_a, tmask_b;  // triangular operand (TRMM): which k a tile needs, see TriMask
    int splits;          // k-ranges per tile (FP32), added by the last to finish
    int chunk;           // FP32: k blocks per accumulation on the tensor cores
    int units;           // tiles * splits
    const int *ea, *eb;  // digits: row exponents of op(A), column exponents of op(B)
    float *partial;      // [tiles][splits] partial tiles of 128 x 128 (splits > 1)
    unsigned int *counter;  // [tiles][8] arrivals, zero at launch (splits > 1)
    const unsigned int *gate;  // nullable; the launch does nothing when the word is set
    unsigned int *status;
    unsigned long long wait_ns;  // budget of every mbarrier wait (nanoseconds)
    int inject_timeout;  // test hook: CTA 0 withholds its first operand copy
};

// Large FP32 GEMMs on the tensor cores (gfip_f32_tc.cu): one operand of the split pass.
struct F32SplitArgs {
    const float *X;
    int64_t ld;
    int rows;         // rows of op(A) or columns of op(B)
    int contig_rows;  // 1: element (r, p) at X[r + p*ld], 0: X[p + r*ld]
    int row_blocks;   // 0: nothing to split (SYRK: B's planes are A's)
    int mask;         // triangular operand (TRMM), 0 = dense; see TriMask
    uint8_t *planes;
    float scale;      // power of two: the planes are those of the scaled elements
};
// Splits both operands and launches the tile core; an element outside the range of the split
// sets *gate (which also makes the tile core do nothing).
cudaError_t launch_f32_tc(const TcParams &p, const F32SplitArgs &a, const F32SplitArgs &b, int k,
                          unsigned int *gate, int sms, cudaStream_t s);

// Splits one operand only.
cudaError_t launch_f32_split(const F32SplitArgs &a, int k, int kt, unsigned int *gate,
                             cudaStream_t s);

// Large FP32 products with at most 128 rows or columns (gfip_f32_skinny.cu): the large operand is
// read where it lies, the small one from its planes.
struct SkinnyParams {
    const float *X;          // the large operand, element (row, p) at X[row + p*ld]
    int64_t ld;
    int rows, k;
    const uint8_t *planes;   // the small operand's planes, one 128-row block
    int n16;                 // its rows, rounded up to a multiple of 16
    int kt, tiles;           // 32-wide k blocks; 128-row blocks of the large operand
    int splits, units;       // k ranges; tiles * splits
    int chunk;               // k blocks per accumulation on the tensor cores (a power of two)
    float *partial;          // [splits][tiles][n16][128]
    unsigned int *gate;      // set when an element is outside the range of the split
    unsigned int *status;
    unsigned long long wait_ns;
    int inject_timeout;      // test hook: CTA 0 withholds its first copies
};
// Splits the small operand, runs the product and adds the k ranges into C (big_is_row: the large
// operand's rows are C's rows), which is untouched when *gate is set.
cudaError_t launch_f32_skinny(const SkinnyParams &p, const F32SplitArgs &small, float *C,
                              int64_t ldc, int big_is_row, float alpha, float beta, int sms,
                              cudaStream_t s);

// FP64 GEMM emulated with BF16 digit products on the tensor cores (gfip_ozaki.cu).
struct OzakiParams {
    const double *A;
    const double *B;
    double *C;
    int64_t lda, ldb, ldc;
    int m, n, k;
    double alpha, beta;
    int a_contig_rows;   // 1: row i of op(A) runs along memory (transa 'N')
    int b_contig_rows;   // 1: column j of op(B) = row j of its K-major form runs along memory ('T')
    int slices;          // digits per element (S)
    int mt, nt, kt;      // 128-row blocks of m and n, 32-wide k blocks
    int ks_a, ks_b;      // k-ranges the exponent reductions are split into
    int *exp;            // [(mt + nt) * 128] row exponents of op(A), column exponents of op(B)
    uint8_t *pa;         // digit planes of op(A)
    uint8_t *pb;         // digit planes of op(B)
    unsigned int *status;
    unsigned long long wait_ns;  // budget of every mbarrier wait (nanoseconds)
    int inject_timeout;  // test hook: CTA 0 withholds its first operand copy
};
cudaError_t launch_ozaki(const OzakiParams &p, int sms, cudaStream_t s);

// Triangular solve: one launch solves a panel of at most TRSM_PANEL unknowns (op(A)'s diagonal
// block at (k0, k0), transposed for side 'R') for every right-hand side; vector v's element i is
// B[v*vstride + i*estride].  FP64 in gfip_trsm.cu; FP32 in gfip_trsm_f32.cu, which packs the
// panel's triangle into `image` (trsm_image_bytes(), 16-byte aligned) first when trsm_packs().
// status: null when there is no cleared status word; the panel is then staged without waits.
constexpr int TRSM_PANEL = 512;
cudaError_t launch_trsm_panel_f64(double *B, int64_t vstride, int64_t estride, int nvec,
                                  const double *A, int64_t lda, int a_trans, int k0, int pw,
                                  int lower_t, int transpose_t, int unit, cudaStream_t s);
cudaError_t launch_trsm_panel_f32(float *B, int64_t vstride, int64_t estride, int nvec,
                                  const float *A, int64_t lda, int a_trans, int k0, int pw,
                                  int lower_t, int transpose_t, int unit, float *image,
                                  unsigned int *status, unsigned long long wait_ns,
                                  int inject_timeout, cudaStream_t s);
size_t trsm_image_bytes(int pw);
bool trsm_packs(int pw);

// Grouped GEMM (gfip_grouped.cu): many independent problems in one persistent launch, each
// problem with its own warp-tile shape and k-split factor.
template <typename T> struct GroupDesc;
template <typename T> struct GroupParams;
template <typename T> cudaError_t launch_grouped(const GroupParams<T> &gp, cudaStream_t s);
// Bytes of one grouped launch's descriptor arrays for `count` problems (element size es).
size_t grouped_desc_bytes(int count, int es);

// Small products (gfip_small.cu): one launch, no packing, no workspace.  *grid: its CTAs.
template <typename T> struct SmallParams {
    const T *A;
    const T *B;
    T *C;
    int64_t lda, ldb, ldc;
    int m, n, k;
    T alpha, beta;
    int a_contig_m, b_contig_n;   // as in GemmParams
    int tri, tmask_a, tmask_b;    // as in GemmParams
    int mt, tiles;                // tiles along m, and of C (set by the launcher)
};
template <typename T> cudaError_t launch_small(SmallParams<T> p, int sms, cudaStream_t s, int *grid);
// Estimated clocks of the FP64 kernel.
int64_t small_dgemm_clocks(int64_t m, int64_t n, int64_t k, int tri, int a_contig_m,
                           int b_contig_n, int sms);

// Launchers (defined per element type in gfip_f64.cu / gfip_f32.cu).
template <typename T> cudaError_t launch_gemm(const GemmParams<T> &p, cudaStream_t s);
template <typename T> cudaError_t launch_pack(const PackParams<T> &p, cudaStream_t s);
template <typename T>
cudaError_t launch_scale(T *C, int64_t ldc, int m, int n, T beta, int tri, cudaStream_t s);
// CTAs of the GEMM kernel that fit on one SM at once.
template <typename T> int gemm_blocks_per_sm();
// The warp-specialised FP32 tile core (gfip_f32_ws.cu): dense FP32 GEMMs over the whole of C
// (no triangle, no triangular operand) with line producers or no packing.
cudaError_t launch_ws_gemm(const GemmParams<float> &p, cudaStream_t s);
// Its pack kernel (pack-then-compute): packed tiles in the swizzled layout it reads.
cudaError_t launch_ws_pack(const PackParams<float> &p, cudaStream_t s);
int ws_blocks_per_sm();

}  // namespace gfip
