// Device helpers of the convolution units (apr_unitplan.cpp), shared by the single-channel and the
// multi-channel kernels: a parent's children, octets at the grid's edges, the images of the data adjoint.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "apr_device.cuh"
#include "apr_internal.h"

namespace aprk {
namespace dev {

// Slots of a plane: the unit's, then three that stay zero (ZERO_SLOT: the neighbours of an image outside
// the grid).
constexpr int PLANE = UNIT_SLOTS + 4;
constexpr unsigned ZERO_SLOT = UNIT_SLOTS;

// The children of a parent from its child map: child c = 2k + e (k = (a, b) the child row, e the child's y
// parity) is a particle (kind 1) or a tree node (kind 2) at index ix[c], or absent (kind 0).
struct Octet {
    int ix[8];
    int kind[8];
    __device__ __forceinline__ Octet(const int4 &pw, const int4 &tw) {
        const int pv[4] = {pw.x, pw.y, pw.z, pw.w}, tv[4] = {tw.x, tw.y, tw.z, tw.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned pm = unsigned(pv[k]) >> 30, tm = unsigned(tv[k]) >> 30;
            const int pi = int(unsigned(pv[k]) & TNP_INDEX), ti = int(unsigned(tv[k]) & TNP_INDEX);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const bool isp = (pm >> e) & 1u, ist = (tm >> e) & 1u;
                kind[2 * k + e] = isp ? 1 : (ist ? 2 : 0);
                ix[2 * k + e] = isp ? pi + (e ? int(pm & 1u) : 0) : ti + (e ? int(tm & 1u) : 0);
            }
        }
    }
};

// An octet at or outside the grid's edge: with reflection a missing child takes its sibling's value and
// a mirrored octet is reversed along the mirrored axes; with the zero boundary the missing children and
// every slot outside the grid are zero.
template <typename T>
__device__ __forceinline__ void edge_octet(T (&v)[8], unsigned info, bool reflect, T zero) {
    const unsigned mir = (info >> UE_MIRROR) & 7u, miss = (info >> UE_MISS) & 7u;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const int m = 1 << ax;
        if (miss & m) {
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (c & m) v[c] = reflect ? v[c ^ m] : zero;
        }
    }
    if (mir && !reflect) {
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = zero;
    }
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const int m = 1 << ax;
        if (mir & m) {
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (c & m) {
                    const T t = v[c];
                    v[c] = v[c ^ m];
                    v[c ^ m] = t;
                }
        }
    }
}

__device__ __forceinline__ unsigned pure_slot(const uint4 &q) {
    return (q.x >> 28) | ((q.y >> 28) << 4) | ((q.z >> 28) << 8);
}

// Nine row slots in the words of a record.
__device__ __forceinline__ void unpack_bases(unsigned w1, const uint2 &r1, const uint2 &r2, unsigned (&b)[9]) {
    b[0] = w1 >> 16;
    b[1] = r1.x & 0xffffu;
    b[2] = r1.x >> 16;
    b[3] = r1.y & 0xffffu;
    b[4] = r1.y >> 16;
    b[5] = r2.x & 0xffffu;
    b[6] = r2.x >> 16;
    b[7] = r2.y & 0xffffu;
    b[8] = r2.y >> 16;
}
__device__ __forceinline__ int4 child_particles(const UnitView &U, unsigned node) {
    return __ldg(reinterpret_cast<const int4 *>(U.nplan + node));
}
// f(particle, c) for the particles among the children.
template <typename F>
__device__ __forceinline__ void for_child_particles(const int4 &pw, F f) {
    const int pv[4] = {pw.x, pw.y, pw.z, pw.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned pm = unsigned(pv[k]) >> 30;
        const int pi = int(unsigned(pv[k]) & TNP_INDEX);
        if (pm & 1u) f(pi, 2 * k);
        if (pm & 2u) f(pi + int(pm & 1u), 2 * k + 1);
    }
}

// Images. With reflection, out-of-grid cells c' within R of the grid add to H of the cell they reflect
// onto. Those cells are the children of parents outside the grid, so their sums are those of a record
// there: the same sums over a neighbourhood shifted along the axis (one layer of it inside the grid, the
// others zero), with the children mirrored. Per axis, from the 3-bit edge code, the shifts that occur:
// bit 0 none, bit 1 by -1 (first parent), bit 2 by +1 (the grid ends with this parent's second child, or
// the grid is a single cell), bit 3 by +2 (an odd grid ends with the next parent's first child; only
// radius 2 reaches back). A missing second child (an odd grid's last parent) is itself the image of its
// sibling.
template <int R>
__device__ __forceinline__ unsigned axis_shifts(unsigned code) {
    const unsigned left = code >> 1;
    return 1u | ((code & 1u) ? 2u : 0u) | (left == 2u || code == 3u ? 4u : 0u) | (R == 2 && left == 3u ? 8u : 0u);
}
// All shift triples of an edge word: bit 16 iz + 4 ix + iy.
template <int R>
__device__ __forceinline__ unsigned long long edge_shifts(unsigned edge) {
    const unsigned z = axis_shifts<R>(edge & 7u), x = axis_shifts<R>((edge >> 3) & 7u), y = axis_shifts<R>((edge >> 6) & 7u);
    unsigned xy = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) xy |= ((x >> i) & 1u) ? y << (4 * i) : 0u;
    unsigned long long m = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) m |= ((z >> i) & 1u) ? (unsigned long long)xy << (16 * i) : 0ull;
    return m;
}
// Layer of the record's neighbourhood that layer d of the image with shift index i reads (-1: zero).
__device__ __forceinline__ int image_layer(int i, int d) {
    if (i == 0) return d;
    return d == (i == 1 ? 2 : 0) ? (i == 3 ? 2 : 1) : -1;
}
__device__ __forceinline__ unsigned missing_children(unsigned edge) {   // axis mask z 4, x 2, y 1
    return ((edge >> 1) & 3u) == 1u ? (((edge >> 4) & 3u) == 1u ? 6u : 4u) | (((edge >> 7) & 3u) == 1u ? 1u : 0u)
                                    : (((edge >> 4) & 3u) == 1u ? 2u : 0u) | (((edge >> 7) & 3u) == 1u ? 1u : 0u);
}

}  // namespace dev
}  // namespace aprk
