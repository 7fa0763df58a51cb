// dlo_frames.cuh -- a rod's initial adapted reference frames (App. A.1) as a parallel scan, in
// FP64, one block per rod and one thread per edge; shared by the frame initialisation
// (dlo_init.cu) and its adjoint (dlo_adjoint.cu).
//
// Space-parallel transport carries a director from edge to edge along the rod.  In its edge's
// normal plane a director is a unit complex number: with a_j the projection of a fixed axis
// (a function of the tangent t_j alone) and b_j = t_j x a_j, transporting a_{j-1} to edge j
// gives cos(w_j) a_j + sin(w_j) b_j, so the transported director is Z_j = z_j z_{j-1} ... z_1
// with z_j = exp(i w_j).  Every z_j needs only the two tangents at its vertex, and their
// products are a prefix scan: log2(edges) dependent steps instead of one chain of transports
// and normalisations over the rod (a chain of FP64 square roots and quotients of about 3 us per
// edge, which cost more than the rollout itself in short rollouts of few rods).
#pragma once
#include "dlo_internal.h"
#include "dlo_physics.cuh"

namespace dlo {

typedef V3<double> D3;

__device__ __forceinline__ D3 ld(float4 a) { return D3{(double)a.x, (double)a.y, (double)a.z}; }
__device__ __forceinline__ D3 unit_d(D3 a) { return rsqrt(dot(a, a)) * a; }
// the projection of a fixed axis (z, or x when t lies within about 25 degrees of z), unit length
__device__ __forceinline__ D3 axis_of(D3 t) { return fabs(t.z) < 0.9 ? D3{0.0, 0.0, 1.0} : D3{1.0, 0.0, 0.0}; }
__device__ __forceinline__ D3 first_director(D3 t) {
    const D3 ax = axis_of(t);
    return unit_d(ax - dot(ax, t) * t);
}

// A rotation in an edge's normal plane; `first` starts a new chain there (an element of a
// segmented scan).
struct Turn {
    double c, s;
    int first;
};
// turn a followed by turn b
__device__ __forceinline__ Turn then(const Turn& a, const Turn& b) {
    if (b.first) return b;
    return Turn{a.c * b.c - a.s * b.s, a.c * b.s + a.s * b.c, a.first};
}

constexpr int kFrameMaxEdges = 256;   // edges per rod (one thread each)
constexpr int kFrameMaxWarps = kFrameMaxEdges / 32;

// Inclusive scan over the block's threads (thread order); wsum: kFrameMaxWarps entries of shared
// memory.  Every thread of the block calls it.
__device__ __forceinline__ Turn scan_turns(Turn z, Turn* wsum) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        Turn p;
        p.c = __shfl_up_sync(0xffffffffu, z.c, o);
        p.s = __shfl_up_sync(0xffffffffu, z.s, o);
        p.first = __shfl_up_sync(0xffffffffu, z.first, o);
        if (lane >= o) z = then(p, z);
    }
    if (lane == 31) wsum[w] = z;
    __syncthreads();
    if (w > 0) {
        Turn p = wsum[0];
        for (int k = 1; k < w; ++k) p = then(p, wsum[k]);
        z = then(p, z);
    }
    return z;
}

// The transport of a unit director a (normal to ta) from tangent ta to tb, as a turn from
// (a2, tb x a2) on the edge of tb.  Of unit length: where two edges nearly reverse, at pi - delta, the
// transport itself is off by 2e-16 / delta^2 (1 + cos cancels), which every later product would carry
// into its director's length.  Elsewhere the length is 1 to a few 1e-16 and needs no square root
// (dividing always: 1024 rods of 16-256 vertices 1416 -> 1434 us).
__device__ __forceinline__ Turn transport_turn(D3 ta, D3 a, D3 tb, D3 a2) {
    const D3 u = transport_d(ta, tb, a);
    Turn z{dot(u, a2), dot(u, cross(tb, a2)), 0};
    const double l2 = z.c * z.c + z.s * z.s;
    if (fabs(l2 - 1.0) > 1e-13) {
        const double i = rsqrt(l2);
        z.c *= i;
        z.s *= i;
    }
    return z;
}

// The parallel-transported director of this thread's edge (tangent t; start: a chain begins at
// this edge), before any holonomy correction.  T, A: shared tangents and in-plane axes of the
// rod's edges (filled here).  Threads at and past ne edges take part with a neutral element.
__device__ __forceinline__ D3 transported_director(D3 t, bool start, int ne, D3* T, D3* A, Turn* wsum) {
    const int j = threadIdx.x;
    D3 a{1.0, 0.0, 0.0};
    if (j < ne) {
        a = first_director(t);
        T[j] = t;
        A[j] = a;
    }
    __syncthreads();
    Turn z{1.0, 0.0, start || j == 0 ? 1 : 0};
    if (j < ne && !z.first) z = transport_turn(T[j - 1], A[j - 1], t, a);
    z = scan_turns(z, wsum);
    return z.c * a + z.s * cross(t, a);
}

}  // namespace dlo
