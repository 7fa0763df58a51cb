// dlo_init.cu -- initial adapted reference frames of every rod, in FP64 (App. A.1).
//
// Edge 0 takes the projection of a fixed axis (z, or x when the first edge lies within about
// 25 degrees of z); later edges get their frame by space-parallel transport.  For closed
// loops the holonomy psi_H (mismatch after transporting the last frame across the closing
// hinge, measured about t^0) is spread as phi^j = -psi_H j / N_e and each (d1, d2) rotated by
// phi^j ("Loop Topology").  The reference twist of each hinge is the signed angle from the
// transported d1 of the previous edge to d1 of the next: 0 along an open rod, whose frames are
// transported ones, and -psi_H / N_e at every hinge of a loop; in rest mode it becomes the rest
// twist, so the rest state stores no twist energy.  A record of several strands (ROD_STRANDS)
// starts each strand like edge 0; a break edge between two strands gets tangent z and d1 = x,
// and the hinges at its two ends a reference (and rest) twist of 0.
//
// One block per rod and one thread per edge, the transport as a scan (dlo_frames.cuh).  Bound by
// the FP64 pipe for large batches (about 200 FP64 operations per edge, 2 lanes per SM and clock)
// and by its latency for small ones.  One thread per rod walking its edges took 421 us for 16
// rods of 64 vertices and 1071 us for 4096 of 128.
#include "dlo_frames.cuh"
#include "dlo_kernels.h"

namespace dlo {

// Vertex j and the edge that starts there: the rest twist (rest mode), or the state.
__device__ __forceinline__ void store_init(const InitParams& P, const RodInfo& R, int j, D3 t, D3 d1, float twist) {
    const int nv = R.nv, v0 = R.v0, e0 = R.e0;
    const bool closed = R.flags & ROD_CLOSED;
    if (P.rest_mode) {
        if (j < nv) P.rest[v0 + j].z = twist;
        return;
    }
    if (j < R.ne) {
        const float th = P.thin ? P.thin[e0 + j] : 0.f;
        P.S.ED[e0 + j] = make_float4((float)d1.x, (float)d1.y, (float)d1.z, th);
        P.S.ET[e0 + j] = make_float4((float)t.x, (float)t.y, (float)t.z, P.ES[e0 + j].x);
    }
    if (j < nv) {
        const float4 x = P.xin[v0 + j], rs = P.rest[v0 + j];
        float4 v = P.vin ? P.vin[v0 + j] : make_float4(0.f, 0.f, 0.f, 0.f);
        const bool end = !closed && j == nv - 1;
        if (end) v.w = 0.f;   // no edge starts at the last vertex of an open rod
        P.S.HG[v0 + j] = end || (!closed && j == 0) ? make_float4(0.f, 0.f, 0.f, 0.f)
                                                    : make_float4(rs.x, rs.y, rs.z, twist);
        P.S.X[v0 + j] = make_float4(x.x, x.y, x.z, P.mass[v0 + j].y);
        P.S.Vl[v0 + j] = v;
    }
}

__global__ void __launch_bounds__(kFrameMaxEdges) init_kernel(InitParams P) {
    __shared__ D3 T[kFrameMaxEdges], A[kFrameMaxEdges];
    __shared__ Turn wsum[kFrameMaxWarps];
    __shared__ double psi_sh;
    __shared__ D3 last_sh;
    const int rod = blockIdx.x, j = threadIdx.x;
    const RodInfo R = P.rods[rod];
    const int nv = R.nv, ne = R.ne, v0 = R.v0, e0 = R.e0;
    const bool closed = R.flags & ROD_CLOSED, strands = R.flags & ROD_STRANDS;
    if (P.n_small && nv <= 32) return;   // init_small's
    if (P.rest_mode && !closed) {   // an open rod's rest twists are zero
        if (j < nv) P.rest[v0 + j].z = 0.f;
        return;
    }
    auto brk = [&](int k) { return strands && !(P.ES[e0 + k].x > 0.f); };
    D3 t{0.0, 0.0, 1.0};
    bool bj = true, start = true;
    if (j < ne) {
        bj = brk(j);
        start = bj || (j > 0 && brk(j - 1));
        if (!bj) t = unit_d(ld(P.xin[v0 + (j + 1 == nv ? 0 : j + 1)]) - ld(P.xin[v0 + j]));
    }
    D3 d1 = transported_director(t, start, ne, T, A, wsum);
    if (bj) d1 = D3{1.0, 0.0, 0.0};
    float twist = 0.f;
    if (closed) {
        if (j == ne - 1) last_sh = d1;
        __syncthreads();
        if (j == 0) {   // holonomy: the last frame carried across the closing hinge, against the first
            const Turn z = transport_turn(T[ne - 1], last_sh, T[0], A[0]);
            psi_sh = atan2(z.s, z.c);
        }
        __syncthreads();
        const double psi = psi_sh, phi = -psi * (double)j / (double)ne;
        d1 = cos(phi) * d1 + sin(phi) * cross(t, d1);
        twist = (float)(-psi / (double)ne);
    }
    store_init(P, R, j, t, d1, twist);
    if (P.rest_mode) return;
    for (int k = j; k < 24; k += blockDim.x) P.S.GP[24LL * rod + k] = P.GP0[24LL * rod + k];
}

// The same for rods of up to W <= 32 vertices, 32 / W of them per warp: an FP64 instruction holds the
// pipe for a whole warp however few of its lanes have an edge, so a large batch of short rods with a
// warp each spends it on idle lanes.  Neighbours meet by shuffles; same operations in the same order
// as above.
template <int W>
__global__ void __launch_bounds__(128) init_small(InitParams P) {
    const unsigned all = 0xffffffffu;
    const long long g = ((long long)blockIdx.x * 128 + threadIdx.x) / W;
    const int j = threadIdx.x % W;
    const bool live = g < P.n_small;   // the last warp's spare groups repeat the last rod and store nothing
    const int rod = P.small[live ? g : P.n_small - 1];
    const RodInfo R = P.rods[rod];
    const int nv = R.nv, ne = R.ne, v0 = R.v0, e0 = R.e0;
    const bool closed = R.flags & ROD_CLOSED, strands = R.flags & ROD_STRANDS;
    auto brk = [&](int k) { return strands && !(P.ES[e0 + k].x > 0.f); };
    auto from = [&](D3 a, int lane) {
        return D3{__shfl_sync(all, a.x, lane, W), __shfl_sync(all, a.y, lane, W), __shfl_sync(all, a.z, lane, W)};
    };
    D3 t{0.0, 0.0, 1.0}, d1 = t;
    float twist = 0.f;
    if (__any_sync(all, closed || !P.rest_mode)) {   // an open rod's rest twists are zero
        D3 a{1.0, 0.0, 0.0};
        bool bj = true, start = true;
        if (j < ne) {
            bj = brk(j);
            start = bj || (j > 0 && brk(j - 1));
            if (!bj) t = unit_d(ld(P.xin[v0 + (j + 1 == nv ? 0 : j + 1)]) - ld(P.xin[v0 + j]));
            a = first_director(t);
        }
        const D3 tp = from(t, j > 0 ? j - 1 : 0), ap = from(a, j > 0 ? j - 1 : 0);
        Turn z{1.0, 0.0, start || j == 0 ? 1 : 0};
        if (j < ne && !z.first) z = transport_turn(tp, ap, t, a);
#pragma unroll
        for (int o = 1; o < W; o <<= 1) {
            Turn p;
            p.c = __shfl_up_sync(all, z.c, o, W);
            p.s = __shfl_up_sync(all, z.s, o, W);
            p.first = __shfl_up_sync(all, z.first, o, W);
            if (j >= o) z = then(p, z);
        }
        d1 = z.c * a + z.s * cross(t, a);
        if (bj) d1 = D3{1.0, 0.0, 0.0};
        if (__any_sync(all, closed)) {
            const D3 tl = from(t, ne - 1), dl = from(d1, ne - 1);
            double psi = 0.0;
            if (closed && j == 0) {
                const Turn y = transport_turn(tl, dl, t, a);
                psi = atan2(y.s, y.c);
            }
            psi = __shfl_sync(all, psi, 0, W);
            if (closed) {
                const double phi = -psi * (double)j / (double)ne;
                d1 = cos(phi) * d1 + sin(phi) * cross(t, d1);
                twist = (float)(-psi / (double)ne);
            }
        }
    }
    if (!live) return;
    store_init(P, R, j, t, d1, twist);
    if (P.rest_mode) return;
    for (int k = j; k < 24; k += W) P.S.GP[24LL * rod + k] = P.GP0[24LL * rod + k];
}

template <int W>
static void launch_small(const InitParams& P, cudaStream_t st) {
    init_small<W><<<(unsigned)(((long long)P.n_small * W + 127) / 128), 128, 0, st>>>(P);
}

cudaError_t launch_init(const InitParams& P, int nv_max, cudaStream_t st) {
    if (P.B <= 0) return cudaSuccess;
    if (P.n_small > 0) {
        if (P.nv_small <= 4) launch_small<4>(P, st);
        else if (P.nv_small <= 8) launch_small<8>(P, st);
        else if (P.nv_small <= 16) launch_small<16>(P, st);
        else launch_small<32>(P, st);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess || P.n_small == P.B) return e;
    }
    init_kernel<<<P.B, nv_max, 0, st>>>(P);
    return cudaGetLastError();
}

}  // namespace dlo
