// Helpers shared by the kernels and the host builders: block barrier, reflection, per-block row offsets,
// programmatic dependent launch.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "apr_internal.h"

namespace aprk {
namespace dev {

constexpr int NT = 256;                // threads of the multi-channel weight gradient and of the other tile kernels' gathering warps
constexpr int NWARP = NT / 32;
static_assert(TZ % 2 == 0 && TX % 2 == 0, "tiles must be even-aligned (coarse cells)");

// Block barrier. The warp is reconverged first: threads of one warp may reach this point at
// different times after data-dependent loops, and the block barrier must be executed by converged
// warps.
__device__ __forceinline__ void block_sync() {
    __syncwarp();
    __syncthreads();
}

__host__ __device__ __forceinline__ int imax(int a, int b) { return a > b ? a : b; }
__host__ __device__ __forceinline__ int imin(int a, int b) { return a < b ? a : b; }

__host__ __device__ __forceinline__ int reflect_idx(int i, int d) {
    // half-sample symmetric reflection into [0, d), repeated for grids smaller than the stencil
    const int p = 2 * d;
    int m = i % p;
    if (m < 0) m += p;
    return m >= d ? p - 1 - m : m;
}

// The rows' y-block offsets: blk_start and row_range serve the exported tile plans (apr_tile.cuh), no kernel.
// First element of y-block j of a row (particles or tree); j >= nb gives the row end.
__host__ __device__ __forceinline__ uint32_t blk_start(const uint32_t *rp, const uint16_t *off, int row0, int off0,
                                                       int nb, int rr, int j) {
    if (j >= nb) return rp[row0 + rr + 1];
    return rp[row0 + rr] + off[off0 + rr * nb + j];
}

// Index range [lo, hi) of a row containing every element with y in [ya, yb) (ya < yb), plus at
// most BY/2 extra elements on each side (callers filter by y). Uses the per-block offsets only:
// at most BY - ra elements of block ja lie at or after ya, at most rb elements of block jb before yb.
__host__ __device__ __forceinline__ void row_range(const uint32_t *rp, const uint16_t *off, int row0, int off0, int nb,
                                                   int rr, int ya, int yb, int &lo, int &hi) {
    const int rs = int(rp[row0 + rr]), re = int(rp[row0 + rr + 1]);
    const int ja = ya / BY, ra = ya - ja * BY;
    const int jb = yb / BY, rb = yb - jb * BY;
    int a = ra <= BY / 2 ? int(blk_start(rp, off, row0, off0, nb, rr, ja))
                         : int(blk_start(rp, off, row0, off0, nb, rr, ja + 1)) - (BY - ra);
    int b = rb <= BY / 2 ? int(blk_start(rp, off, row0, off0, nb, rr, jb)) + rb
                         : int(blk_start(rp, off, row0, off0, nb, rr, jb + 1));
    a = imax(a, rs);
    b = imin(b, re);
    lo = a;
    hi = imax(a, b);
}

// Programmatic dependent launch (launch_pdl): pdl_trigger lets the next kernel on the stream start
// (its blocks run their prologue while this kernel finishes); pdl_wait blocks until the kernel before
// this one on the stream has completed and its writes are visible. In a kernel launched without the
// attribute both are no-ops.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// What an earlier launch may write while this kernel already runs (all but the handle's own arrays) is read after
// pdl_wait, and not through the read-only path, which assumes that it stays as it is for the kernel's lifetime.
__device__ __forceinline__ float load_after_wait(const float *p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

}  // namespace dev
}  // namespace aprk
