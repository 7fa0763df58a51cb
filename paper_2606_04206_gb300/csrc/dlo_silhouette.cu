// dlo_silhouette.cu -- the system-identification loss: the projection error between the
// simulated rope's silhouette and a camera's binary mask (Sec. 5, "System Identification"),
// made differentiable.  Each edge is drawn as a capsule of the rod's projected radius, its
// soft occupancy of a pixel is sigma((rho_e - dist) / tau), and a pixel's occupancy is
// 1 - prod_e (1 - sigma_e), composited in log space.  The loss is the mean over cameras and
// pixels of (occupancy - mask)^2.
//
// Per camera, two launches over all rods.  Pass 1, a CTA per rod and 32 x 8 pixel tile: the rod's
// edges whose reach box meets the tile are listed once (in order), then each thread composites
// its pixel over the list and stores dL/d(occupancy) * prod_e (1 - sigma_e), the factor every
// edge's gradient at that pixel shares.  Pass 2, a warp per edge: the lanes walk the pixels of the
// edge's reach box and their sums give its endpoints' gradient.  A last launch (one per group of four
// cameras) adds up each rod's tiles and, per vertex, its edges over the cameras.  Nothing is accumulated with atomics:
// the result is deterministic.  Bound by instruction issue: the exponentials and logarithms of
// the pixels near a rope (at 256 x 256 a rope is near 1 pixel in 25).  One CTA per rod testing
// every pixel against every edge took 2.87 ms for 64 rods of 64 vertices and 2 cameras of
// 256 x 256.
#include <algorithm>
#include <cmath>

#include "dlo_runtime.h"
#include "dlo_vec.cuh"

namespace dlo {
namespace {

constexpr int kTileW = 32, kTileH = 8;   // pixels per CTA of pass 1, one per thread
constexpr int kSilT = kTileW * kTileH;
constexpr int kSilMaxV = 256;            // vertices per rod
constexpr int kEdgesPerCta = 8;          // warps of pass 2
constexpr int kCamsPerGroup = 4;         // cameras whose vertices and edge gradients are held at once
// an edge is skipped at pixels farther than rho_e + kReach tau from it: sigma < 1.4e-11 there
constexpr float kReach = 25.f;
constexpr float kNear = 1e-3f;  // edges with an endpoint this close to the camera plane or behind it are not drawn

struct Cam {
    float fx, fy, cx, cy;
    float R[9];   // world to camera, row major
    float t[3];
};

__device__ __forceinline__ float softplus(float z) { return z > 0.f ? z + log1pf(expf(-z)) : log1pf(expf(z)); }
__device__ __forceinline__ float logistic(float z) {
    if (z >= 0.f) return 1.f / (1.f + expf(-z));
    const float e = expf(z);
    return e / (1.f + e);
}

// (u, v, rho, Z): pixel coordinates, projected radius (fx r / Z), depth
__device__ __forceinline__ float4 project(const Cam& c, V3<float> x, float r) {
    const float X = c.R[0] * x.x + c.R[1] * x.y + c.R[2] * x.z + c.t[0];
    const float Y = c.R[3] * x.x + c.R[4] * x.y + c.R[5] * x.z + c.t[1];
    const float Z = c.R[6] * x.x + c.R[7] * x.y + c.R[8] * x.z + c.t[2];
    const float iz = 1.f / Z;
    return make_float4(c.fx * X * iz + c.cx, c.fy * Y * iz + c.cy, c.fx * r * iz, Z);
}

// signed distance of pixel centre (pu, pv) to the capsule of edge (a, b): distance to the
// segment minus the edge radius; t is the closest point's parameter, (nu, nv) the unit
// direction from the closest point to the pixel (zero when they coincide).  The roundings are
// fixed: at a pixel on the segment's line the direction is decided by them, and both passes
// should see the same one.
__device__ __forceinline__ float dot2(float a, float b, float c, float d) { return __fmaf_rn(a, b, __fmul_rn(c, d)); }
__device__ __forceinline__ float capsule_sd(float pu, float pv, float4 a, float4 b, float rho, float& t, float& nu,
                                            float& nv) {
    const float du = b.x - a.x, dv = b.y - a.y;
    const float l2 = dot2(du, du, dv, dv);
    t = l2 > 0.f ? fminf(fmaxf(dot2(pu - a.x, du, pv - a.y, dv) / l2, 0.f), 1.f) : 0.f;
    const float eu = pu - __fmaf_rn(t, du, a.x), ev = pv - __fmaf_rn(t, dv, a.y);
    const float d = sqrtf(dot2(eu, eu, ev, ev));
    nu = d > 0.f ? eu / d : 0.f;
    nv = d > 0.f ? ev / d : 0.f;
    return d - rho;
}

struct SilParams {
    const RodInfo* rods;
    int B, C, H, W, tiles_x, tiles, edge_ctas;
    int c0, nc;                 // the group's first camera and their number
    float tau;
    const float4* X;
    const float* cams;
    const unsigned char* masks;
    const float* g;
    float *q, *render, *wbuf;   // wbuf: the current camera's pixel factors [B][H][W]
    float4* gx;
    float4 *pv, *ge;            // projected vertices [nc][V]; edge gradients [nc][V][2] (an edge at its first vertex)
    float4* acc;                // [V] the vertices' gradient over the groups before
    double* part;               // [B][tiles] sums of squared differences
    long long V;
};

__device__ __forceinline__ void load_cam(const SilParams& P, int c, Cam& cm) {
    if (threadIdx.x < 16) reinterpret_cast<float*>(&cm)[threadIdx.x] = P.cams[16 * c + threadIdx.x];
    __syncthreads();
}

// Reach box (umin, umax, vmin, vmax) of an edge; empty if it is not drawn.
__device__ __forceinline__ float4 reach_box(float4 a, float4 b, float tau) {
    if (!(a.w > kNear && b.w > kNear)) return make_float4(1.f, -1.f, 1.f, -1.f);
    const float m = 0.5f * (a.z + b.z) + kReach * tau;
    return make_float4(fminf(a.x, b.x) - m, fmaxf(a.x, b.x) + m, fminf(a.y, b.y) - m, fmaxf(a.y, b.y) + m);
}

// every vertex in the group's cameras; one CTA per rod and camera (c: the camera within the group)
__global__ void __launch_bounds__(kSilMaxV) sil_project(SilParams P) {
    __shared__ Cam cm;
    const int c = blockIdx.y, i = threadIdx.x;
    const RodInfo R = P.rods[blockIdx.x];
    load_cam(P, P.c0 + c, cm);
    if (i < R.nv) P.pv[c * P.V + R.v0 + i] = project(cm, f3(P.X[R.v0 + i]), R.radius);
}

__global__ void __launch_bounds__(kSilT) sil_pixels(SilParams P, int c) {
    __shared__ float4 ea[kSilMaxV], eb[kSilMaxV], box[kSilMaxV];   // the listed edges' ends and boxes
    __shared__ int cnt[kSilT / 32];
    __shared__ double red[kSilT / 32];
    const int rod = blockIdx.x / P.tiles, tile = blockIdx.x % P.tiles;
    const RodInfo R = P.rods[rod];
    const int n = R.nv, ne = R.ne, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int x0 = tile % P.tiles_x * kTileW, y0 = tile / P.tiles_x * kTileH;
    // list the edges that reach the tile, in order (the products below keep their order)
    {
        const int e = threadIdx.x;
        bool hit = false;
        float4 a, b, bx;
        if (e < ne) {
            const float4* pv = P.pv + c * P.V + R.v0;
            a = pv[e];
            b = pv[e + 1 == n ? 0 : e + 1];
            bx = reach_box(a, b, P.tau);
            hit = !(bx.x > bx.y || (float)x0 + ((float)kTileW - 0.5f) < bx.x || (float)x0 + 0.5f > bx.y ||
                    (float)y0 + ((float)kTileH - 0.5f) < bx.z || (float)y0 + 0.5f > bx.w);
        }
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        if (lane == 0) cnt[w] = __popc(m);
        __syncthreads();
        int at = __popc(m & ((1u << lane) - 1u));
        for (int k = 0; k < w; ++k) at += cnt[k];
        if (hit) {
            ea[at] = a;
            eb[at] = b;
            box[at] = bx;
        }
    }
    __syncthreads();
    int total = 0;
#pragma unroll
    for (int k = 0; k < kSilT / 32; ++k) total += cnt[k];
    const int i = x0 + lane, j = y0 + w;
    double sq = 0.0;
    if (i < P.W && j < P.H) {
        const float px = (float)i + 0.5f, py = (float)j + 0.5f, inv_tau = 1.f / P.tau;
        float S = 0.f;   // log prod_e (1 - sigma_e)
        for (int e = 0; e < total; ++e) {
            const float4 bx = box[e];
            if (px < bx.x || px > bx.y || py < bx.z || py > bx.w) continue;
            const float4 a = ea[e], b = eb[e];
            float t, nu, nv;
            const float sd = capsule_sd(px, py, a, b, 0.5f * (a.z + b.z), t, nu, nv);
            S -= softplus(-sd * inv_tau);
        }
        const size_t HW = (size_t)P.H * P.W, p = (size_t)j * P.W + i, im = ((size_t)rod * P.C + P.c0 + c) * HW + p;
        const float o = -expm1f(S);
        const float d = o - (P.masks[im] ? 1.f : 0.f);
        sq = (double)d * d;
        const float coef = 2.f * (P.g ? P.g[rod] : 1.f) / ((float)P.C * (float)(P.H * P.W));
        if (P.gx) P.wbuf[(size_t)rod * HW + p] = coef * d * expf(S);
        if (P.render) P.render[im] = o;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (lane == 0) red[w] = sq;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = P.c0 + c ? P.part[blockIdx.x] : 0.0;   // the cameras follow one another on the stream
        for (int k = 0; k < kSilT / 32; ++k) t += red[k];
        P.part[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(32 * kEdgesPerCta) sil_edges(SilParams P, int c) {
    __shared__ Cam cm;
    const int rod = blockIdx.x / P.edge_ctas, lane = threadIdx.x & 31;
    const int e = blockIdx.x % P.edge_ctas * kEdgesPerCta + (threadIdx.x >> 5);
    const RodInfo R = P.rods[rod];
    load_cam(P, P.c0 + c, cm);
    if (e >= R.ne) return;
    const float4* pv = P.pv + c * P.V + R.v0;
    const float4 a = pv[e], b = pv[e + 1 == R.nv ? 0 : e + 1], bx = reach_box(a, b, P.tau);
    const float rho = 0.5f * (a.z + b.z), inv_tau = 1.f / P.tau;
    const float* wr = P.wbuf + (size_t)rod * P.H * P.W;
    float gau = 0.f, gav = 0.f, gbu = 0.f, gbv = 0.f, gr = 0.f;   // d L / d(u_a, v_a, u_b, v_b, rho_e)
    if (bx.x <= bx.y) {
        const int i0 = max(0, (int)floorf(bx.x - 0.5f)), i1 = min(P.W - 1, (int)ceilf(bx.y - 0.5f));
        const int j0 = max(0, (int)floorf(bx.z - 0.5f)), j1 = min(P.H - 1, (int)ceilf(bx.w - 0.5f));
        const int bw = i1 - i0 + 1, bh = j1 - j0 + 1;
        if (bw > 0 && bh > 0) {
            const unsigned area = (unsigned)bw * (unsigned)bh;
            for (unsigned k = lane; k < area; k += 32) {
                const int j = j0 + (int)(k / (unsigned)bw), i = i0 + (int)(k % (unsigned)bw);
                const float px = (float)i + 0.5f, py = (float)j + 0.5f;
                if (px < bx.x || px > bx.y || py < bx.z || py > bx.w) continue;
                float t, nu, nv;
                const float sd = capsule_sd(px, py, a, b, rho, t, nu, nv);
                // dL/d(sd) = w(p) sigma(z) dz/d(sd), z = -sd / tau
                const float gs = -wr[(size_t)j * P.W + i] * logistic(-sd * inv_tau) * inv_tau;
                gau -= gs * (1.f - t) * nu;
                gav -= gs * (1.f - t) * nv;
                gbu -= gs * t * nu;
                gbv -= gs * t * nv;
                gr -= gs;
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        gau += __shfl_xor_sync(0xffffffffu, gau, o);
        gav += __shfl_xor_sync(0xffffffffu, gav, o);
        gbu += __shfl_xor_sync(0xffffffffu, gbu, o);
        gbv += __shfl_xor_sync(0xffffffffu, gbv, o);
        gr += __shfl_xor_sync(0xffffffffu, gr, o);
    }
    // (u, v, rho) = (fx X / Z + cx, fy Y / Z + cy, fx r / Z); then world = R^T camera
    auto to_world = [&](float4 p, float g_u, float g_v, float g_r) {
        const float iz = 1.f / p.w;
        const float Xc = (p.x - cm.cx) * p.w / cm.fx, Yc = (p.y - cm.cy) * p.w / cm.fy;
        const float gX = g_u * cm.fx * iz, gY = g_v * cm.fy * iz;
        const float gZ = -(g_u * cm.fx * Xc + g_v * cm.fy * Yc + g_r * cm.fx * R.radius) * iz * iz;
        return make_float4(cm.R[0] * gX + cm.R[3] * gY + cm.R[6] * gZ, cm.R[1] * gX + cm.R[4] * gY + cm.R[7] * gZ,
                           cm.R[2] * gX + cm.R[5] * gY + cm.R[8] * gZ, 0.f);
    };
    if (lane < 2)
        P.ge[2 * (c * P.V + R.v0 + e) + lane] =
            lane == 0 ? to_world(a, gau, gav, 0.5f * gr) : to_world(b, gbu, gbv, 0.5f * gr);
}

// each rod's loss, and its vertices' gradient over the cameras (kept in acc until the last group, so
// that the gradient may go where the positions are)
__global__ void __launch_bounds__(kSilMaxV) sil_gather(SilParams P) {
    __shared__ double red[kSilMaxV];
    const int rod = blockIdx.x, i = threadIdx.x;
    const RodInfo R = P.rods[rod];
    const bool closed = R.flags & ROD_CLOSED;
    const int n = R.nv, ne = R.ne;
    if (P.gx && i < n) {
        float4 acc = P.c0 ? P.acc[R.v0 + i] : make_float4(0.f, 0.f, 0.f, 0.f);
        for (int c = 0; c < P.nc; ++c) {
            const float4* ge = P.ge + 2 * (c * P.V + R.v0);
            if (closed || i < ne) {   // the edge that starts here
                const float4 o = ge[2 * i];
                acc = make_float4(acc.x + o.x, acc.y + o.y, acc.z + o.z, 0.f);
            }
            if (closed || i > 0) {    // and the one that ends here
                const float4 o = ge[2 * (i == 0 ? ne - 1 : i - 1) + 1];
                acc = make_float4(acc.x + o.x, acc.y + o.y, acc.z + o.z, 0.f);
            }
        }
        (P.c0 + P.nc < P.C ? P.acc : P.gx)[R.v0 + i] = acc;
    }
    if (!P.q || P.c0 + P.nc < P.C) return;
    double t = 0.0;
    for (int k = i; k < P.tiles; k += kSilMaxV) t += P.part[(size_t)rod * P.tiles + k];
    red[i] = t;
    __syncthreads();
    for (int s = kSilMaxV / 2; s > 0; s >>= 1) {
        if (i < s) red[i] += red[i + s];
        __syncthreads();
    }
    if (i == 0) P.q[rod] = (float)(red[0] / ((double)P.C * P.H * P.W));
}

}  // namespace
}  // namespace dlo

using namespace dlo;

extern "C" dlo_status dlo_loss_silhouette(dlo_ctx* c, const float* x, const float* cams, int n_cams, int height,
                                          int width, const unsigned char* masks, float tau, const float* g, float* q,
                                          float* dL_dx, float* render) {
    if (!c) return DLO_ERR_INVALID_ARG;
    if (!x || ((uintptr_t)x & 15u) || (dL_dx && ((uintptr_t)dL_dx & 15u)) || !cams || !masks)
        return set_err(c, DLO_ERR_INVALID_ARG, "x, cams and masks are required; x and dL_dx must be 16-byte aligned");
    if (n_cams < 1 || height < 1 || width < 1 || (long long)height * width > (1LL << 24))
        return set_err(c, DLO_ERR_INVALID_ARG, "need 1 or more cameras and 1..2^24 pixels per image");
    if (!(tau > 0.f)) return set_err(c, DLO_ERR_INVALID_ARG, "tau must be positive");
    for (const auto& R : c->rods_h) {
        if (R.nv > kSilMaxV) return set_err(c, DLO_ERR_INVALID_ARG, "rod too long for the silhouette kernel");
        if (R.flags & ROD_STRANDS)   // its edges are drawn as capsules; nothing joins two strands
            return set_err(c, DLO_ERR_INVALID_ARG, "the silhouette loss needs rods without strands");
    }
    SilParams P{};
    P.rods = c->d_rods;
    P.B = c->B;
    P.C = n_cams;
    P.H = height;
    P.W = width;
    P.tiles_x = (width + kTileW - 1) / kTileW;
    P.tiles = P.tiles_x * ((height + kTileH - 1) / kTileH);
    P.edge_ctas = (c->buckets.back().nv_max + kEdgesPerCta - 1) / kEdgesPerCta;
    P.tau = tau;
    P.X = reinterpret_cast<const float4*>(x);
    P.cams = cams;
    P.masks = masks;
    P.g = g;
    P.q = q;
    P.render = render;
    P.gx = reinterpret_cast<float4*>(dL_dx);
    P.V = c->V;
    // Workspace: projected vertices and edge gradients of one group of cameras, the vertices'
    // gradient, tile sums, one camera's pixel factors.  Its size follows from the rods and the
    // number of pixels alone (no image has more tiles than an eighth of its pixels): a graph that
    // holds a call keeps its workspace when a later call asks for the gradient as well, for
    // other cameras or for another shape of as many pixels.
    const size_t nproj = (size_t)kCamsPerGroup * c->V, ntile = (size_t)c->B * P.tiles, pixels = (size_t)height * width;
    const size_t pv_bytes = 16 * nproj, ge_bytes = 32 * nproj, acc_bytes = 16 * (size_t)c->V;
    const size_t part_bytes = (8 * (size_t)c->B * ((pixels + 7) / 8) + 15) & ~(size_t)15;
    const size_t need = pv_bytes + ge_bytes + acc_bytes + part_bytes + sizeof(float) * (size_t)c->B * pixels;
    if (ntile >= ((size_t)1 << 31) || (size_t)c->B * P.edge_ctas >= ((size_t)1 << 31))
        return set_err(c, DLO_ERR_OOM, "too many rods and pixels for one silhouette call");
    if (need > c->sil_bytes) {
        dev_free(c, c->sil_mem);
        c->sil_mem = dev_alloc(c, need);
        c->sil_bytes = c->sil_mem ? need : 0;
        if (!c->sil_mem) return set_err(c, DLO_ERR_OOM, "silhouette scratch allocation failed");
    }
    char* m = reinterpret_cast<char*>(c->sil_mem);
    P.pv = reinterpret_cast<float4*>(m);
    P.ge = reinterpret_cast<float4*>(m + pv_bytes);
    P.acc = reinterpret_cast<float4*>(m + pv_bytes + ge_bytes);
    P.part = reinterpret_cast<double*>(m + pv_bytes + ge_bytes + acc_bytes);
    P.wbuf = reinterpret_cast<float*>(m + pv_bytes + ge_bytes + acc_bytes + part_bytes);
    cudaError_t e = cudaSuccess;
    for (P.c0 = 0; P.c0 < n_cams && e == cudaSuccess; P.c0 += kCamsPerGroup) {
        P.nc = std::min(n_cams - P.c0, kCamsPerGroup);
        sil_project<<<dim3(c->B, P.nc), kSilMaxV, 0, c->stream>>>(P);
        c->launches++;
        e = cudaGetLastError();
        for (int k = 0; k < P.nc && e == cudaSuccess; ++k) {
            sil_pixels<<<(unsigned)ntile, kSilT, 0, c->stream>>>(P, k);
            c->launches++;
            if (P.gx) {
                sil_edges<<<c->B * P.edge_ctas, 32 * kEdgesPerCta, 0, c->stream>>>(P, k);
                c->launches++;
            }
            e = cudaGetLastError();
        }
        if (e == cudaSuccess && (P.gx || P.c0 + P.nc == n_cams)) {
            sil_gather<<<c->B, kSilMaxV, 0, c->stream>>>(P);
            c->launches++;
            e = cudaGetLastError();
        }
    }
    return cuda_err(c, e, "silhouette launch");
}
