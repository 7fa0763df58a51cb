// dlo_loss.cu -- task losses of App. B ("Reward design") on the device, per rod, with their
// gradient with respect to the vertex positions (the dL/dx_T that dlo_backward takes).
// One CTA per rod; sums are reduced in double in a fixed order, and every gradient is
// gathered without atomics, so results are deterministic.
#include <cmath>

#include "dlo_runtime.h"
#include "dlo_vec.cuh"
#include "dlo_physics.cuh"

namespace dlo {
namespace {

constexpr int kLT = 128;          // threads per rod
constexpr int kMaxPoints = 1024;  // Chamfer point set size per rod
constexpr int kMaxV = 256;        // vertices per rod

__device__ double block_sum(double v, double* sh) {
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int s = kLT / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
        __syncthreads();
    }
    const double r = sh[0];
    __syncthreads();
    return r;
}

__device__ __forceinline__ float gscale(const float* g, int rod) { return g ? g[rod] : 1.f; }

// (1/N) sum_i |x_i - t_i|^2
__global__ void loss_target(const RodInfo* rods, const float4* X, const float4* Tg, const float* g, float* q,
                            float4* gx) {
    __shared__ double sh[kLT];
    const int rod = blockIdx.x;
    const RodInfo R = rods[rod];
    const float c = 2.f * gscale(g, rod) / (float)R.nv;
    double s = 0.0;
    for (int i = threadIdx.x; i < R.nv; i += kLT) {
        const V3<float> d = f3(X[R.v0 + i]) - f3(Tg[R.v0 + i]);
        s += (double)dot(d, d);
        if (gx) gx[R.v0 + i] = f4(c * d, 0.f);
    }
    s = block_sum(s, sh);
    if (q && threadIdx.x == 0) q[rod] = (float)(s / R.nv);
}

// (1/N) sum_i min_j |x_i - y_j|^2 + (1/M) sum_j min_i |x_i - y_j|^2
__global__ void loss_chamfer(const RodInfo* rods, const float4* X, const float4* Y, int m, const float* g,
                             float* q, float4* gx) {
    __shared__ double sh[kLT];
    __shared__ float4 xs[kMaxV];
    __shared__ float4 ys[kMaxPoints];
    __shared__ short nn[kMaxPoints];   // nearest vertex of each point
    const int rod = blockIdx.x;
    const RodInfo R = rods[rod];
    const int n = R.nv;
    for (int i = threadIdx.x; i < n; i += kLT) xs[i] = X[R.v0 + i];
    for (int j = threadIdx.x; j < m; j += kLT) ys[j] = Y[(size_t)rod * m + j];
    __syncthreads();
    const float gs = gscale(g, rod);
    double s = 0.0;
    // points to their nearest vertex
    for (int j = threadIdx.x; j < m; j += kLT) {
        const V3<float> y = f3(ys[j]);
        float best = INFINITY;
        int bi = 0;
        for (int i = 0; i < n; ++i) {
            const V3<float> d = f3(xs[i]) - y;
            const float d2 = dot(d, d);
            if (d2 < best) {
                best = d2;
                bi = i;
            }
        }
        nn[j] = (short)bi;
        s += (double)best / m;
    }
    __syncthreads();
    // vertices to their nearest point, and the gradient of both terms at each vertex
    for (int i = threadIdx.x; i < n; i += kLT) {
        const V3<float> x = f3(xs[i]);
        float best = INFINITY;
        int bj = 0;
        V3<float> acc = zf3();
        for (int j = 0; j < m; ++j) {
            const V3<float> d = x - f3(ys[j]);
            const float d2 = dot(d, d);
            if (d2 < best) {
                best = d2;
                bj = j;
            }
            if (nn[j] == i) acc += (2.f / m) * d;
        }
        s += (double)best / n;
        if (gx) gx[R.v0 + i] = f4(gs * ((2.f / n) * (x - f3(ys[bj])) + acc), 0.f);
    }
    s = block_sum(s, sh);
    if (q && threadIdx.x == 0) q[rod] = (float)s;
}

// (1/2pi) sum over segments of the signed angle they subtend at the post (xy-plane); the sum
// telescopes, so only the two ends of an open rod carry gradient: d(phi_j) = (-a_y, a_x) / |a|^2
__global__ void loss_winding(const RodInfo* rods, const float4* X, const float4* posts, const float* g, float* q,
                             float4* gx) {
    __shared__ double sh[kLT];
    const int rod = blockIdx.x;
    const RodInfo R = rods[rod];
    const bool closed = R.flags & ROD_CLOSED;
    const int n = R.nv, ne = closed ? n : n - 1;
    const float px = posts[rod].x, py = posts[rod].y;
    double s = 0.0;
    for (int j = threadIdx.x; j < ne; j += kLT) {
        const int j1 = (j + 1 == n) ? 0 : j + 1;
        const float ax = X[R.v0 + j].x - px, ay = X[R.v0 + j].y - py;
        const float bx = X[R.v0 + j1].x - px, by = X[R.v0 + j1].y - py;
        s += (double)atan2f(ax * by - ay * bx, ax * bx + ay * by);
    }
    s = block_sum(s, sh);
    if (q && threadIdx.x == 0) q[rod] = (float)(s / (2.0 * M_PI));
    if (!gx) return;
    const float c = gscale(g, rod) / (2.f * (float)M_PI);
    for (int i = threadIdx.x; i < n; i += kLT) {
        const float coef = closed ? 0.f : (i == n - 1 ? 1.f : (i == 0 ? -1.f : 0.f));
        const float ax = X[R.v0 + i].x - px, ay = X[R.v0 + i].y - py;
        const float r2 = ax * ax + ay * ay;
        gx[R.v0 + i] = coef != 0.f && r2 > 0.f ? make_float4(c * coef * -ay / r2, c * coef * ax / r2, 0.f, 0.f)
                                              : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// ---- the Gauss double integral of two straight segments (exact closed form).
// The directions r_2 - r_1 of the pair sweep the parallelogram r13, r14, r24, r23; the integral
// is minus its signed solid angle seen from the origin, taken as two triangles with the
// atan2 form of Van Oosterom and Strackee (IEEE TBME 1983), which stays well conditioned in
// float where the arcsine form of the same angle loses its derivative.
// Both triangles, (r13, r14, r24) and (r13, r24, r23), have the same triple product, r13 . (e1 x e2)
// with e1 and e2 the segments: formed from the segments it keeps the digits that the products of
// the nearly equal r's of a distant pair cancel.  Their denominators are
// |u||v||w| + (u.v)|w| + (u.w)|v| + (v.w)|u|.
// Two vertices much closer to each other than the segments are long turn this round: the product of
// the segments is then off by 1e-7 |e1||e2||r13|, the denominators of the triangles that hold the
// short r shrink with it, and at zero the angle is atan2(rounding, 0).  With an r below a quarter of
// the rod's longest edge each triangle takes the product of its own three vectors, which vanishes with
// its shortest, and the lengths are square roots (zero at zero, where s rsqrt(s) is not a number).

// The gradient of a denominator, times c, added to those of its three vectors (lengths l, inverse
// lengths il, dot products d).
__device__ __forceinline__ void denominator_grad(V3<float> u, V3<float> v, V3<float> w, float lu, float lv, float lw,
                                                 float iu, float iv, float iw, float duv, float duw, float dvw, float c,
                                                 V3<float>& gu, V3<float>& gv, V3<float>& gw) {
    const float au = c * (lv * lw + dvw) * iu, av = c * (lu * lw + duw) * iv, aw = c * (lu * lv + duv) * iw;
    const float auv = c * lw, auw = c * lv, avw = c * lu;
    gu += au * u + auv * v + auw * w;
    gv += av * v + auv * u + avw * w;
    gw += aw * w + auw * u + avw * v;
}

// Omega of the segments p1p2 and p3p4; with GRAD also its gradient with respect to the four ends
// (one reverse pass).  near2: the squared distance below which two vertices count as close.
template <bool GRAD>
__device__ __forceinline__ float gauss_pair(V3<float> p1, V3<float> p2, V3<float> p3, V3<float> p4, float near2,
                                            V3<float>* g) {
    const V3<float> r13 = p3 - p1, r14 = p4 - p1, r23 = p3 - p2, r24 = p4 - p2, e1 = p2 - p1, e2 = p4 - p3;
    float l13, l14, l23, l24, i13, i14, i23, i24;
    len_inv(r13, l13, i13);
    len_inv(r14, l14, i14);
    len_inv(r23, l23, i23);
    len_inv(r24, l24, i24);
    const V3<float> e12 = cross(e1, e2);
    float n1 = dot(r13, e12), n2 = n1;
    const float s13 = dot(r13, r13), s14 = dot(r14, r14), s23 = dot(r23, r23), s24 = dot(r24, r24);
    if (fminf(fminf(s13, s14), fminf(s23, s24)) <= near2) {
        n1 = dot(r13, cross(r14, r24));
        n2 = dot(r13, cross(r24, r23));
        auto root = [](float s, float& l, float& i) {
            l = sqrtf(s);
            i = l > 0.f ? 1.f / l : 0.f;
        };
        root(s13, l13, i13);
        root(s14, l14, i14);
        root(s23, l23, i23);
        root(s24, l24, i24);
    }
    const float da = dot(r13, r14), db = dot(r13, r24), dc = dot(r14, r24), dd = dot(r13, r23), de = dot(r24, r23);
    const float m1 = l13 * l14 * l24 + da * l24 + db * l14 + dc * l13;
    const float m2 = l13 * l24 * l23 + db * l23 + dd * l24 + de * l13;
    if (GRAD) {
        const float q1 = -2.f / (n1 * n1 + m1 * m1), q2 = -2.f / (n2 * n2 + m2 * m2);
        V3<float> g13 = zf3(), g14 = zf3(), g23 = zf3(), g24 = zf3();
        denominator_grad(r13, r14, r24, l13, l14, l24, i13, i14, i24, da, db, dc, -(q1 * n1), g13, g14, g24);
        denominator_grad(r13, r24, r23, l13, l24, l23, i13, i24, i23, db, dd, de, -(q2 * n2), g13, g24, g23);
        const float c = q1 * m1 + q2 * m2;   // of the triple product
        g13 += c * e12;
        const V3<float> h1 = c * cross(e2, r13), h2 = c * cross(r13, e1);
        g[0] = -(g13 + g14) - h1;
        g[1] = h1 - (g23 + g24);
        g[2] = g13 + g23 - h2;
        g[3] = g14 + g24 + h2;
    }
    return -2.f * (atan2f(n1, m1) + atan2f(n2, m2));
}

// Sum of floats as an unevaluated pair (Knuth's exact two-term sum): FP64 accuracy on the FP32
// pipe, which an FP64 addition per pair of edges would leave waiting.
struct PairSum {
    float h = 0.f, l = 0.f;
    __device__ __forceinline__ void add(float v) {
        const float t = __fadd_rn(h, v), b = __fsub_rn(t, h);
        l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(t, b)), __fsub_rn(v, b)));
        h = t;
    }
    __device__ __forceinline__ double value() const { return (double)h + (double)l; }
};

// Sum over ordered pairs of non-adjacent edges of Omega / (4 pi), Omega being symmetric twice the
// sum over unordered ones: edge a meets edge a + k (mod the edge count), k = 1, 2, ... up to half
// of them, all threads at the same k.  GRAD: the thread of a keeps its ends' gradient, and adds
// its partner's to that edge's slots (at one k every thread has another partner; a barrier
// separates the steps).  Bound by instruction issue: about 350 instructions a pair.
template <bool GRAD>
__global__ void __launch_bounds__(kLT) loss_crossing(const RodInfo* rods, const float4* X, const float* g, float* q,
                                                     float4* gx) {
    constexpr int EPT = GRAD ? 1 : kMaxV / kLT;   // edges per thread (GRAD: rods of up to kLT vertices)
    __shared__ double sh[kLT];
    __shared__ float4 xs[kMaxV];
    __shared__ float4 ge0[GRAD ? kLT : 1], ge1[GRAD ? kLT : 1];   // d/d(first, second endpoint) of each edge's sum
    __shared__ unsigned longest[kLT / 32];   // the longest edge squared (non-negative floats order like their bits)
    const int rod = blockIdx.x;
    const RodInfo R = rods[rod];
    if (GRAD && R.nv > kLT) return;   // loss_crossing_long's
    const bool closed = R.flags & ROD_CLOSED;
    const int n = R.nv, ne = closed ? n : n - 1;
    unsigned far2 = 0u;
    for (int i = threadIdx.x; i < n; i += kLT) {
        const float4 x0 = X[R.v0 + i];
        xs[i] = x0;
        if (GRAD) ge0[i] = ge1[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i >= ne) continue;
        const V3<float> e = f3(X[R.v0 + (i + 1 == n ? 0 : i + 1)]) - f3(x0);
        far2 = max(far2, __float_as_uint(dot(e, e)));
    }
    far2 = __reduce_max_sync(0xffffffffu, far2);
    if (threadIdx.x % 32 == 0) longest[threadIdx.x / 32] = far2;
    __syncthreads();
    static_assert(kLT == 128, "four warps");
    const float near2 = 0.0625f * __uint_as_float(max(max(longest[0], longest[1]), max(longest[2], longest[3])));
    PairSum sum;
    V3<float> g0[EPT], g1[EPT];
#pragma unroll
    for (int m = 0; m < EPT; ++m) g0[m] = g1[m] = zf3();
    for (int k = 1; k <= ne / 2; ++k) {
#pragma unroll
        for (int m = 0; m < EPT; ++m) {
            const int a = threadIdx.x + m * kLT;
            // the opposite edge of an even ring of indices, from its lower half alone; neighbours
            // (k = 1, but not the two ends of an open rod) do not cross
            if (a >= ne || (2 * k == ne && a >= k)) continue;
            const int b = a + k >= ne ? a + k - ne : a + k;
            if (abs(a - b) <= 1 || (closed && k == 1)) continue;
            V3<float> gp[4];
            sum.add(gauss_pair<GRAD>(f3(xs[a]), f3(xs[a + 1 == n ? 0 : a + 1]), f3(xs[b]), f3(xs[b + 1 == n ? 0 : b + 1]),
                                         near2, gp));
            if (GRAD) {
                g0[m] += gp[0];
                g1[m] += gp[1];
                ge0[b] = f4(f3(ge0[b]) + gp[2], 0.f);
                ge1[b] = f4(f3(ge1[b]) + gp[3], 0.f);
            }
        }
        if (GRAD) __syncthreads();
    }
    if (GRAD) {
#pragma unroll
        for (int m = 0; m < EPT; ++m) {
            const int a = threadIdx.x + m * kLT;
            if (a >= ne) continue;
            ge0[a] = f4(f3(ge0[a]) + g0[m], 0.f);
            ge1[a] = f4(f3(ge1[a]) + g1[m], 0.f);
        }
    }
    __syncthreads();
    const double s = block_sum(2.0 * sum.value(), sh);
    if (q && threadIdx.x == 0) q[rod] = (float)(s / (4.0 * M_PI));
    if (!GRAD) return;
    // each unordered pair appears twice in the sum: d/dx = 2 sum_b dOmega_ab / (4 pi)
    const float c = gscale(g, rod) / (2.f * (float)M_PI);
    for (int i = threadIdx.x; i < n; i += kLT) {
        V3<float> d = zf3();
        if (closed || i < ne) d += f3(ge0[i]);                         // i starts edge i
        if (closed || i > 0) d += f3(ge1[i == 0 ? ne - 1 : i - 1]);     // and ends edge i-1
        gx[R.v0 + i] = f4(c * d, 0.f);
    }
}

__device__ dualf gauss_pair_d(V3<dualf> p1, V3<dualf> p2, V3<dualf> p3, V3<dualf> p4) {
    const V3<dualf> r13 = p3 - p1, r14 = p4 - p1, r23 = p3 - p2, r24 = p4 - p2;
    const dualf l13 = norm(r13), l14 = norm(r14), l23 = norm(r23), l24 = norm(r24);
    const dualf d13_24 = dot(r13, r24);
    const dualf n1 = dot(r13, cross(r14, r24));
    const dualf m1 = l13 * l14 * l24 + dot(r13, r14) * l24 + d13_24 * l14 + dot(r14, r24) * l13;
    const dualf n2 = dot(r13, cross(r24, r23));
    const dualf m2 = l13 * l24 * l23 + d13_24 * l23 + dot(r13, r23) * l24 + dot(r24, r23) * l13;
    return -2.f * (datan2(n1, m1) + datan2(n2, m2));
}

// The same sum and gradient for rods of more than 128 vertices, on dual numbers: the thread of
// edge a evaluates Omega(a, b) for every b with the six coordinates of a's endpoints seeded in
// turn.  Four times the work of the closed form, which holds one edge's gradient per thread.  (The
// gradient is a sum of thousands of cancelling pairs: the two evaluations agree to 1.1e-5 of it at
// 128 vertices and to 2.5e-5 at 250, each 1e-5 to 2e-5 from FP64.)  A rod's kernel follows from its own
// size, so that its result does not depend on the batch it is in.
__global__ void loss_crossing_long(const RodInfo* rods, const float4* X, const float* g, float* q, float4* gx) {
    __shared__ double sh[kLT];
    __shared__ float4 xs[kMaxV];
    __shared__ float4 ge0[kMaxV], ge1[kMaxV];   // d/d(first, second endpoint) of each edge's sum
    const int rod = blockIdx.x;
    const RodInfo R = rods[rod];
    if (R.nv <= kLT) return;   // loss_crossing's
    const bool closed = R.flags & ROD_CLOSED;
    const int n = R.nv, ne = closed ? n : n - 1;
    for (int i = threadIdx.x; i < n; i += kLT) xs[i] = X[R.v0 + i];
    __syncthreads();
    double s = 0.0;
    for (int a = threadIdx.x; a < ne; a += kLT) {
        const int a1 = (a + 1 == n) ? 0 : a + 1;
        const V3<float> pa = f3(xs[a]), pb = f3(xs[a1]);
        float gq[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int b = 0; b < ne; ++b) {
            int sep = abs(a - b);
            if (closed) sep = min(sep, ne - sep);
            if (sep <= 1) continue;
            const int b1 = (b + 1 == n) ? 0 : b + 1;
            const V3<dualf> p3 = lift(f3(xs[b])), p4 = lift(f3(xs[b1]));
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                V3<float> e1 = zf3(), e2 = zf3();
                if (k < 3) (k == 0 ? e1.x : k == 1 ? e1.y : e1.z) = 1.f;
                else (k == 3 ? e2.x : k == 4 ? e2.y : e2.z) = 1.f;
                const dualf om = gauss_pair_d(lift(pa, e1), lift(pb, e2), p3, p4);
                if (k == 0) s += (double)om.v;
                gq[k] += om.d;
            }
        }
        ge0[a] = make_float4(gq[0], gq[1], gq[2], 0.f);
        ge1[a] = make_float4(gq[3], gq[4], gq[5], 0.f);
    }
    __syncthreads();
    s = block_sum(s, sh);
    if (q && threadIdx.x == 0) q[rod] = (float)(s / (4.0 * M_PI));
    // each unordered pair appears twice in the sum: d/dx = 2 sum_b dOmega_ab / (4 pi)
    const float c = gscale(g, rod) / (2.f * (float)M_PI);
    for (int i = threadIdx.x; i < n; i += kLT) {
        V3<float> d = zf3();
        if (closed || i < ne) d += f3(ge0[i]);                         // i starts edge i
        if (closed || i > 0) d += f3(ge1[i == 0 ? ne - 1 : i - 1]);     // and ends edge i-1
        gx[R.v0 + i] = f4(c * d, 0.f);
    }
}

// min_i |x_i - o|; the subgradient at the nearest vertex (lowest index on a tie)
__global__ void loss_mindist(const RodInfo* rods, const float4* X, const float4* obj, const float* g, float* q,
                             float4* gx) {
    __shared__ float bd[kLT];
    __shared__ int bi[kLT];
    const int rod = blockIdx.x;
    const RodInfo R = rods[rod];
    const V3<float> o = f3(obj[rod]);
    float best = INFINITY;
    int arg = 0;
    for (int i = threadIdx.x; i < R.nv; i += kLT) {
        const V3<float> d = f3(X[R.v0 + i]) - o;
        const float d2 = dot(d, d);
        if (d2 < best) {   // strict: a thread's own vertices come in increasing order
            best = d2;
            arg = i;
        }
    }
    bd[threadIdx.x] = best;
    bi[threadIdx.x] = arg;
    __syncthreads();
    for (int s = kLT / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) {
            const float d2 = bd[threadIdx.x + s];
            const int i2 = bi[threadIdx.x + s];
            if (d2 < bd[threadIdx.x] || (d2 == bd[threadIdx.x] && i2 < bi[threadIdx.x])) {
                bd[threadIdx.x] = d2;
                bi[threadIdx.x] = i2;
            }
        }
        __syncthreads();
    }
    const float dmin = sqrtf(bd[0]);
    const int imin = bi[0];
    if (q && threadIdx.x == 0) q[rod] = dmin;
    if (!gx) return;
    const float c = dmin > 0.f ? gscale(g, rod) / dmin : 0.f;
    for (int i = threadIdx.x; i < R.nv; i += kLT)
        gx[R.v0 + i] = i == imin ? f4(c * (f3(X[R.v0 + i]) - o), 0.f) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// sum over unordered pairs of edges more than k apart of max(0, delta - d)^2, d the distance of
// the segments' closest points.  The closest-point parameters are each optimal for the other
// (or fixed), so the gradient holds them fixed: dd/dx_a0 = (1 - s) n, dd/dx_a1 = s n.
__global__ void loss_repulsion(const RodInfo* rods, const float4* X, const float4* prm, const float* g, float* q,
                               float4* gx) {
    __shared__ double sh[kLT];
    __shared__ float4 xs[kMaxV];
    __shared__ float4 ge0[kMaxV], ge1[kMaxV];
    __shared__ float4 mid[kMaxV];   // each edge's midpoint and half length
    __shared__ unsigned reach[kLT / 32];   // squared distance of the farthest vertex from the first (as its bits)
    const int rod = blockIdx.x;
    const RodInfo R = rods[rod];
    const bool closed = R.flags & ROD_CLOSED;
    const int n = R.nv, ne = closed ? n : n - 1;
    const float delta = prm[rod].x;
    const int k = max(1, (int)prm[rod].y);
    unsigned far2 = 0u;
    for (int i = threadIdx.x; i < n; i += kLT) {
        const float4 x0 = X[R.v0 + i];
        xs[i] = x0;
        if (i >= ne) continue;
        const V3<float> p0 = f3(x0), p1 = f3(X[R.v0 + (i + 1 == n ? 0 : i + 1)]), e = p1 - p0, r = p1 - f3(X[R.v0]);
        mid[i] = f4(0.5f * (p0 + p1), 0.5f * sqrtf(dot(e, e)));
        far2 = max(far2, __float_as_uint(dot(r, r)));
    }
    far2 = __reduce_max_sync(0xffffffffu, far2);
    if (threadIdx.x % 32 == 0) reach[threadIdx.x / 32] = far2;
    __syncthreads();
    far2 = max(max(reach[0], reach[1]), max(reach[2], reach[3]));
    // A penalty that reaches over nearly the whole rod acts on nearly every pair: no test then, and
    // all threads at the same edge (one broadcast).  4096 rods x 256 with delta 1.4 times the reach:
    // 1752 us with the test, 1527 without; with half the reach 663 and 1232.
    const bool all = delta * delta >= 0.81f * __uint_as_float(far2);
    double s = 0.0;
    for (int a = threadIdx.x; a < ne; a += kLT) {
        const int a1 = (a + 1 == n) ? 0 : a + 1;
        const V3<float> pa = f3(xs[a]), pb = f3(xs[a1]);
        V3<float> g0 = zf3(), g1 = zf3();
        auto pair = [&](int b) {
            int sep = abs(a - b);
            if (closed) sep = min(sep, ne - sep);
            if (sep <= k) return;
            const int b1 = (b + 1 == n) ? 0 : b + 1;
            // every pair is solved with its lower edge first, as both of its threads must see
            // the same closest points (the near-parallel rule is not symmetric)
            const bool first = a < b;
            const V3<float> qa = f3(xs[b]), qb = f3(xs[b1]);
            const V3<float> p1 = first ? pa : qa, q1 = first ? pb : qb, p2 = first ? qa : pa, q2 = first ? qb : pb;
            float ps, pu;
            closest_params(p1, q1, p2, q2, ps, pu);
            const V3<float> dv = (p1 + ps * (q1 - p1)) - (p2 + pu * (q2 - p2));
            const float d = sqrtf(dot(dv, dv));
            if (d >= delta) return;
            if (first) s += (double)((delta - d) * (delta - d));
            if (d > 0.f) {
                const V3<float> gd = (-2.f * (delta - d) / d) * dv;   // d(pen)/d(first closest point)
                const float t = first ? ps : pu, sg = first ? 1.f : -1.f;
                g0 += (sg * (1.f - t)) * gd;
                g1 += (sg * t) * gd;
            }
        };
        if (all) {
            for (int b = 0; b < ne; ++b) pair(b);
        } else {
            // the other edges by their distance ahead: neighbouring threads then have near pairs, the
            // ones that cost, at the same step
            const float4 ma = mid[a];
            for (int o = 1; o < ne; ++o) {
                const int b = a + o >= ne ? a + o - ne : a + o;
                // segments in spheres farther apart than delta cannot be closer than delta (the
                // spheres enlarged by more than the roundings): most pairs end here
                const float4 mb = mid[b];
                const V3<float> dm = f3(ma) - f3(mb);
                const float far = 1.0001f * (delta + ma.w + mb.w);
                if (!(dot(dm, dm) > far * far && far >= 0.f)) pair(b);
            }
        }
        ge0[a] = f4(g0, 0.f);
        ge1[a] = f4(g1, 0.f);
    }
    __syncthreads();
    s = block_sum(s, sh);
    if (q && threadIdx.x == 0) q[rod] = (float)s;
    if (!gx) return;
    const float c = gscale(g, rod);
    for (int i = threadIdx.x; i < n; i += kLT) {
        V3<float> d = zf3();
        if (closed || i < ne) d += f3(ge0[i]);
        if (closed || i > 0) d += f3(ge1[i == 0 ? ne - 1 : i - 1]);
        gx[R.v0 + i] = f4(c * d, 0.f);
    }
}

}  // namespace
}  // namespace dlo

using namespace dlo;

extern "C" dlo_status dlo_loss(dlo_ctx* c, int kind, const float* x, const float* aux, int m, const float* g,
                               float* q, float* dL_dx) {
    if (!c) return DLO_ERR_INVALID_ARG;
    const float4* X = reinterpret_cast<const float4*>(x);
    float4* GX = reinterpret_cast<float4*>(dL_dx);
    if (!x || ((uintptr_t)x & 15u) || (dL_dx && ((uintptr_t)dL_dx & 15u)) || (aux && ((uintptr_t)aux & 15u)))
        return set_err(c, DLO_ERR_INVALID_ARG, "x, aux and dL_dx must be non-null device float4 arrays (16-byte aligned)");
    for (const auto& R : c->rods_h) {
        if (R.nv > kMaxV) return set_err(c, DLO_ERR_INVALID_ARG, "rod too long for the loss kernels");
        // the losses over a rod's edges take single DLOs: nothing joins the strands of a record
        if ((R.flags & ROD_STRANDS) &&
            (kind == DLO_LOSS_WINDING || kind == DLO_LOSS_CROSSING || kind == DLO_LOSS_REPULSION))
            return set_err(c, DLO_ERR_INVALID_ARG, "edge-based losses need rods without strands");
    }
    switch (kind) {
        case DLO_LOSS_TARGET:
            if (!aux) return set_err(c, DLO_ERR_INVALID_ARG, "the target loss needs target positions");
            loss_target<<<c->B, kLT, 0, c->stream>>>(c->d_rods, X, reinterpret_cast<const float4*>(aux), g, q, GX);
            break;
        case DLO_LOSS_CHAMFER:
            if (!aux || m < 1 || m > kMaxPoints)
                return set_err(c, DLO_ERR_INVALID_ARG, "the Chamfer loss needs 1..1024 points per rod");
            loss_chamfer<<<c->B, kLT, 0, c->stream>>>(c->d_rods, X, reinterpret_cast<const float4*>(aux), m, g, q, GX);
            break;
        case DLO_LOSS_WINDING:
            if (!aux) return set_err(c, DLO_ERR_INVALID_ARG, "the winding number needs a post per rod");
            loss_winding<<<c->B, kLT, 0, c->stream>>>(c->d_rods, X, reinterpret_cast<const float4*>(aux), g, q, GX);
            break;
        case DLO_LOSS_CROSSING:
            if (!GX) {
                loss_crossing<false><<<c->B, kLT, 0, c->stream>>>(c->d_rods, X, g, q, GX);
                break;
            }
            if (c->buckets.front().nv_max <= kLT)
                loss_crossing<true><<<c->B, kLT, 0, c->stream>>>(c->d_rods, X, g, q, GX);
            if (c->buckets.back().nv_max > kLT) {
                if (c->buckets.front().nv_max <= kLT) c->launches++;   // beside the one counted below
                loss_crossing_long<<<c->B, kLT, 0, c->stream>>>(c->d_rods, X, g, q, GX);
            }
            break;
        case DLO_LOSS_MINDIST:
            if (!aux) return set_err(c, DLO_ERR_INVALID_ARG, "the minimum distance needs an object centre per rod");
            loss_mindist<<<c->B, kLT, 0, c->stream>>>(c->d_rods, X, reinterpret_cast<const float4*>(aux), g, q, GX);
            break;
        case DLO_LOSS_REPULSION:
            if (!aux) return set_err(c, DLO_ERR_INVALID_ARG, "the repulsion penalty needs (delta, k) per rod");
            loss_repulsion<<<c->B, kLT, 0, c->stream>>>(c->d_rods, X, reinterpret_cast<const float4*>(aux), g, q,
                                                        GX);
            break;
        default:
            return set_err(c, DLO_ERR_INVALID_ARG, "unknown loss kind");
    }
    c->launches++;
    return cuda_err(c, cudaGetLastError(), "loss launch");
}
