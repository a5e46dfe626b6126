// gfip_testing.h -- test-only entry points of libgemmfip.so.  Not part of the public ABI
// (include/gemmfip.h): nothing in the library's normal use calls them, and the only callers are
// tests.
#pragma once

#include <stdint.h>

#include "../../include/gemmfip.h"

#ifdef __cplusplus
extern "C" {
#endif

/* Test hook for the failure path of gfip_dgemm_ozaki (no counterpart in the paper; the
 * paper's CPU kernels have no waits).  Sets, for this handle's later gfip_dgemm_ozaki calls,
 * the budget of every pipeline wait in nanoseconds (0 restores the default, 2 s), and with
 * enable != 0 makes the first CTA withhold its first operand copy, so that its wait runs out:
 * the call then raises GFIP_STATUS_MMA_TIMEOUT, leaves that CTA's 128 x 128 tile of C
 * unwritten (every other tile is computed), waits for its own copies in flight, releases its
 * tensor memory and returns; the context stays usable.  Nothing else is affected.
 * Returns GFIP_ERR_HANDLE for an invalid handle. */
int gfip_debug_ozaki_timeout(gfip_handle_t handle, int enable, uint64_t wait_ns);

/* The same for the FP32 kernels with pipeline waits: the first CTA's first operand copy never
 * arrives (tensor-core tile core, kernel for at most 128 rows or columns, warp-specialised FFMA
 * core, TRSM panels of more than 96 unknowns), so its wait runs out: the call raises
 * GFIP_STATUS_WAIT_TIMEOUT and its result is invalid (a TRSM panel's right-hand sides of that
 * CTA stay as they are). */
int gfip_debug_f32_timeout(gfip_handle_t handle, int enable, uint64_t wait_ns);

/* Sends this handle's later products (GEMM, SYRK, TRMM, TRSM updates) to one path wherever that
 * path can compute them, whatever their size: the fused-in-packing core alone, the small
 * kernels, the tensor cores from planes, or the tensor cores' kernel for at most 128 rows or
 * columns (FP32; the core, or the planes, where it cannot be used). */
#define GFIP_ROUTE_AUTO 0
#define GFIP_ROUTE_CORE 1
#define GFIP_ROUTE_SMALL 2
#define GFIP_ROUTE_TENSOR 3
#define GFIP_ROUTE_SKINNY 4
int gfip_debug_route(gfip_handle_t handle, int route);

#ifdef __cplusplus
}
#endif
