// dlo_step.cuh -- one rod's frame and substep on one thread group, state in shared memory.
//
// Shared by the forward kernel and the backward kernel's recomputations.  Thread i of the group
// owns vertex i, the edge that starts there and the hinge there.  Per substep (DLO-Lab Sec. 3.1 /
// 3.2 / App. A.1):
//   edge phase    the edge's reference frame by time-parallel transport and its material frame
//   hinge phase   curvature and twist, bending plasticity on the rest curvature, and the
//                 hinge's energy gradient back to its two edges' frames
//   edge phase    the edge's frame reversed once on the sum of its two hinges' seeds; its strain
//   vertex phase  gradient gather + stretching, gravity, damping, symplectic-Euler velocity,
//                 soft SDF contact (planes, boxes, capsule grippers), displacement predict,
//                 kinematic vertices, new reference-frame base; new positions when nothing
//                 projects them
//   PBD phase     N_C x (red-black inextensibility / strain limit, Jacobi self-collision), then
//                 v = d/h, positions x + d, self-contact Coulomb friction
// What a thread's own edge hands from phase to phase stays in its registers; only what a
// neighbour reads goes through shared memory (per edge: its frame, the seeds of the hinge at its
// end, its gradient and strain).
// Per frame: self-contact candidates (every edge pair behind a bounding-sphere filter),
// gripper pose update.
#pragma once
#include <type_traits>
#include "dlo_internal.h"
#include "dlo_kernels.h"
#include "dlo_physics.cuh"

namespace dlo {

// The per-rod constants as the persistent kernels hold them: a copy in registers, or (C) a
// reference to the record in global memory, read where used.
template <bool C>
using RodRef = typename std::conditional<C, const RodInfo&, const RodInfo>::type;

// A rod is stepped by a group of TPR threads (whole warps, at least one thread per vertex);
// phases are separated by the group's barrier (the warp's own for TPR = 32, else a named barrier
// of TPR threads).
template <int TPR>
struct Grp {
    int tid;      // thread index within the rod's group
    int bar;      // named barrier id (1..15) of the group
    float* red;   // 64 floats of the rod's shared header, for group reductions
    __device__ __forceinline__ void sync() const {
        if (TPR == 32)
            __syncwarp();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(TPR) : "memory");
    }
    // the same, returning whether p holds for any thread
    __device__ __forceinline__ bool sync_any(bool p) const {
        if (TPR == 32) {
            const bool r = __any_sync(0xffffffffu, p);
            __syncwarp();
            return r;
        }
        unsigned r;
        asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.or.pred q, %2, %3, p;\n\t"
                     "selp.u32 %0, 1, 0, q;\n\t}" : "=r"(r) : "r"((unsigned)p), "r"(bar), "r"(TPR) : "memory");
        return r != 0;
    }
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum over the group (deterministic order: warps' partial sums added in warp order).
template <int TPR>
__device__ __forceinline__ double grp_sum(double v, const Grp<TPR>& g) {
    v = warp_sum(v);
    if (TPR == 32) return v;
    double* r = reinterpret_cast<double*>(g.red);
    if ((g.tid & 31) == 0) r[g.tid >> 5] = v;
    g.sync();
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < TPR / 32; ++k) s += r[k];
    g.sync();
    return s;
}

template <int TPR>
__device__ __forceinline__ bool grp_any(bool p, const Grp<TPR>& g) {
    const bool w = __any_sync(0xffffffffu, p);
    if (TPR == 32) return w;
    int* r = reinterpret_cast<int*>(g.red) + 32;
    if ((g.tid & 31) == 0) r[g.tid >> 5] = w ? 1 : 0;
    g.sync();
    bool s = false;
#pragma unroll
    for (int k = 0; k < TPR / 32; ++k) s |= r[k] != 0;
    g.sync();
    return s;
}

// Bitwise OR over the group.
template <int TPR>
__device__ __forceinline__ unsigned grp_or(unsigned v, const Grp<TPR>& g) {
    const unsigned w = __reduce_or_sync(0xffffffffu, v);
    if (TPR == 32) return w;
    unsigned* r = reinterpret_cast<unsigned*>(g.red) + 56;
    if ((g.tid & 31) == 0) r[g.tid >> 5] = w;
    g.sync();
    unsigned s = 0u;
#pragma unroll
    for (int k = 0; k < TPR / 32; ++k) s |= r[k];
    g.sync();
    return s;
}

// Largest value over the group (non-negative floats: their bit patterns order like the values).
template <int TPR>
__device__ __forceinline__ float grp_max_nonneg(float v, const Grp<TPR>& g) {
    const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(v));
    if (TPR == 32) return __uint_as_float(w);
    unsigned* r = reinterpret_cast<unsigned*>(g.red) + 24;
    if ((g.tid & 31) == 0) r[g.tid >> 5] = w;
    g.sync();
    unsigned m = 0u;
#pragma unroll
    for (int k = 0; k < TPR / 32; ++k) m = max(m, r[k]);
    g.sync();
    return __uint_as_float(m);
}

// Status bit of a failed bounds check.  Debug builds (-DDLO_DEBUG_BOUNDS) check every index
// the kernels take from data (candidate pairs, kinematic kinds, recorded pair counts, work-
// queue items) before using it: a failed check sets the bit in the rod's flag word (slot 40
// of its reduction scratch, folded into the rod's status when its work ends) and the access
// is skipped.  Release builds compile the checks away.
constexpr unsigned kStatusBounds = 8u;

__device__ __forceinline__ bool in_bounds(bool ok, float* red) {
#ifdef DLO_DEBUG_BOUNDS
    if (!ok) atomicOr(reinterpret_cast<unsigned*>(red) + 40, kStatusBounds);
    return ok;
#else
    (void)ok;
    (void)red;
    return true;
#endif
}

// Start of a rod's work: clear its flag word (debug builds).
template <int TPR>
__device__ __forceinline__ void bounds_begin(const Grp<TPR>& g) {
#ifdef DLO_DEBUG_BOUNDS
    if (g.tid == 0) reinterpret_cast<unsigned*>(g.red)[40] = 0u;
#else
    (void)g;
#endif
}

// End of a rod's work, after a group barrier: fold its flag word into status[rod].
template <int TPR>
__device__ __forceinline__ void bounds_end(const Grp<TPR>& g, unsigned* status, int rod) {
#ifdef DLO_DEBUG_BOUNDS
    if (g.tid == 0 && status) {
        const unsigned f = reinterpret_cast<unsigned*>(g.red)[40];
        if (f) atomicOr(&status[rod], f);
    }
#else
    (void)g;
    (void)status;
    (void)rod;
#endif
}

// Value held by thread 0 of the group.
template <int TPR>
__device__ __forceinline__ int grp_bcast0(int v, const Grp<TPR>& g) {
    if (TPR == 32) return __shfl_sync(0xffffffffu, v, 0);
    int* r = reinterpret_cast<int*>(g.red) + 48;
    if (g.tid == 0) *r = v;
    g.sync();
    const int out = *r;
    g.sync();
    return out;
}

// Exclusive prefix sum over the group.
template <int TPR>
__device__ __forceinline__ int grp_excl_scan(int v, const Grp<TPR>& g) {
    const int l = g.tid & 31, w = g.tid >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (l >= o) incl += y;
    }
    if (TPR == 32) return incl - v;
    int* r = reinterpret_cast<int*>(g.red) + 16;
    if (l == 31) r[w] = incl;
    g.sync();
    int off = 0;
    for (int k = 0; k < w; ++k) off += r[k];
    g.sync();
    return off + incl - v;
}

// One substep's records for the adjoint, in global memory (float4 units from base; NV the size
// class): start state (X0, V, HG, ED, ET), then what the substep itself stores.  With ON
// false nothing is recorded.
template <int NV, bool ON>
struct Rec {
    float4* base;
    int n_iter;
    // [NV]: velocity after the force update, before rigid contact
    __device__ __forceinline__ float4* v1() const { return base + 5 * NV; }
    // [NV]: displacement after the PBD iterations, before friction
    __device__ __forceinline__ float4* dfin() const { return base + 6 * NV; }
    // [n_iter][NV]: per edge, the unit direction and target / length of its inextensibility or
    // strain-limit projection, (0, 0, 0, 1) where it did nothing
    __device__ __forceinline__ float4* pbd(int it) const { return base + (size_t)(7 + it) * NV; }
    // [n_iter][NV]: displacements before each self-contact sweep (frames with candidates)
    __device__ __forceinline__ float4* csnap(int it) const { return base + (size_t)(7 + n_iter + it) * NV; }
    // [pair capacity]: first-iteration projection data of each pair
    __device__ __forceinline__ float4* fr0() const { return base + (size_t)(7 + 2 * n_iter) * NV; }
    __device__ __forceinline__ float4* fr1() const { return base + (size_t)(7 + 2 * n_iter + kPairsPerVertex) * NV; }
};

constexpr float kFixPos = 1073741824.f;     // 2^30: fixed-point scale of position corrections
constexpr float kFixVel = 16777216.f;       // 2^24: fixed-point scale of velocity corrections

__device__ __forceinline__ int to_fix(float v, float scale) {
    float q = v * scale;
    q = fminf(fmaxf(q, -2147483520.f), 2147483520.f);
    return __float2int_rn(q);
}

// Impulse m (v_after - v_before) that one contact response gave the vertex, added to its slot.
__device__ __forceinline__ void add_impulse(float4* slot, float m, V3<float> vb, V3<float> va) {
    float4 a = *slot;
    *slot = make_float4(a.x + m * (va.x - vb.x), a.y + m * (va.y - vb.y), a.z + m * (va.z - vb.z), 0.f);
}

// Squared distance from a gripper's centre beyond which no vertex can touch it: the capsule's
// half length plus the contact's reach, a little enlarged.  Nearly every vertex is rejected by
// this one test (the capsule's own takes a projection on its axis and a quotient).
__device__ __forceinline__ float grip_bound(const SceneDev& sc, const RodInfo& R, const float* o) {
    const V3<float> ax = f3(o[8], o[11], o[14]);
    const float b = sc.grip_hl * sqrtf(dot(ax, ax)) + 1.001f * (sc.grip_r + R.radius + kContactReach * R.eps);
    return 1.0001f * b * b;
}
__device__ __forceinline__ bool grip_far(V3<float> x, V3<float> p, const float* o) {
    const V3<float> d = x - p;
    return dot(d, d) > o[30];
}

// Rigid contact of one vertex against the scene and the rod's grippers (Sec. 3.2).
// sp: the substep's gripper block (Smem::sp).  imp (optional): the vertex's four impulse
// slots (planes, boxes, gripper 0, gripper 1), to which each active response adds the
// impulse it gave the vertex of mass m; the rigid body receives the opposite.
__device__ __forceinline__ V3<float> rigid_contact(const SceneDev& sc, const RodInfo& R, V3<float> x,
                                                    V3<float> v, const float* sp, float4* imp = nullptr,
                                                    float m = 0.f) {
    bool on;
    for (int k = 0; k < sc.n_planes; ++k) {
        V3<float> n = f3(sc.planes[k]);
        float sdf = dot(x, n) - sc.planes[k].w;
        const V3<float> vb = v;
        v = contact_respond(v, sdf, n, zf3(), R.radius, R.eps, sc.mu_rigid, sc.restitution, on);
        if (imp && on) add_impulse(imp, m, vb, v);
    }
    for (int k = 0; k < sc.n_boxes; ++k) {
        V3<float> n;
        float sdf = sdf_box(x, f3(sc.box_c[k]), f3(sc.box_h[k]), n);
        const V3<float> vb = v;
        v = contact_respond(v, sdf, n, zf3(), R.radius, R.eps, sc.mu_rigid, sc.restitution, on);
        if (imp && on) add_impulse(imp + 1, m, vb, v);
    }
    for (int g = 0; g < R.ngrip; ++g) {
        const float* o = sp + 32 * g;
        V3<float> p = f3(o[0], o[1], o[2]);
        if (grip_far(x, p, o)) continue;
        V3<float> ax = f3(o[8], o[11], o[14]);   // column 2 of R0: the capsule axis
        V3<float> a = p - sc.grip_hl * ax, b = p + sc.grip_hl * ax, n;
        if (capsule_far(x, a, b, sc.grip_r + R.radius + kContactReach * R.eps)) continue;
        float sdf = sdf_capsule(x, a, b, sc.grip_r, n);
        if (sdf > R.radius + kContactReach * R.eps) continue;
        V3<float> vp = f3(o[24], o[25], o[26]);
        V3<float> w = f3(o[27], o[28], o[29]);
        V3<float> vrig = vp + cross(w, x - p);
        const V3<float> vb = v;
        v = contact_respond(v, sdf, n, vrig, R.radius, R.eps, sc.mu_rigid, sc.restitution, on);
        if (imp && on) add_impulse(imp + 2 + g, m, vb, v);
    }
    return v;
}

template <int NV, bool CONTACT>
struct Smem {
    float4 *X, *X0, *V, *ED, *ET, *HG, *HB0, *HB1, *HB2;
    float4 *fr0, *fr1;
    int4* acc;
    uint32_t* pairs;
    float* red;
    // gripper block (read by every thread of the rod with broadcasts):
    //   fp  [24] pose at the start of the frame being stepped, per gripper p (3), R (9) row major
    //   sp  [kPoseBatch][64] per substep and gripper (32): p0 (3), p1 (3), R0 (9), R1 (9), vp (3), w (3),
    //       grip_bound (1)
    //   act [12] the frame's actions
    float *fp, *sp, *act;
    __device__ Smem(float4* base) {
        red = reinterpret_cast<float*>(base + warp_smem_bytes(NV, CONTACT) / 16);
        fp = red + 64;
        sp = fp + 24;
        act = sp + 64 * kPoseBatch;
        X = base;
        X0 = base + NV;
        V = base + 2 * NV;
        ED = base + 3 * NV;
        ET = base + 4 * NV;
        HG = base + 5 * NV;
        HB0 = base + 6 * NV;
        HB1 = base + 7 * NV;
        HB2 = base + 8 * NV;
        fr0 = base + 9 * NV;
        fr1 = fr0 + kPairsPerVertex * NV;
        acc = reinterpret_cast<int4*>(fr1 + kPairsPerVertex * NV);
        pairs = reinterpret_cast<uint32_t*>(acc + NV);
    }
};

// ------------------------------------------------------------------ broad phase
// Whether an edge strictly between edges a < b is a break edge (rest length 0): a and b then
// lie on different strands, and the exclusion window does not apply to them.
__device__ __forceinline__ bool break_between(const float4* ET, int a, int b) {
    for (int k = a + 1; k < b; ++k)
        if (!(ET[k].w > 0.f)) return true;
    return false;
}

constexpr int kBpBlock = 8;   // edges per block of the broad phase's first level

// Candidates of one rod: the edge pairs outside the exclusion window whose segments are
// closer than R.contact_d.  A rod has at most 256 edges, so every pair is considered, in two
// levels of exact bounding-sphere tests before the closest-point distance:
//   - each block of kBpBlock consecutive edges lies in the sphere around the centre of its
//     vertices' bounding box, with the distance to its farthest vertex as radius;
//   - each edge's segment lies in the sphere around its midpoint with its half length.
// A segment distance below contact_d implies both sphere distances are below contact_d plus
// the radii.  Level 1 tests every pair of blocks (one pair per thread) and lists the near
// ones; level 2 takes an edge of a listed pair's first block per thread against the eight of its
// second and runs the edge-sphere test and the exclusion window on the eight side by side; level
// 3 the exact distance, on the pairs that passed.  (One edge pair per thread, one after the other, and
// a block's sphere by one thread took 9400 cycles for a loose rope of 128 vertices, a sixth
// of its frame, most of them the latency of dependent loads; this takes 3800.)  Found pairs are
// appended with a shared-memory atomic (rare), so their order
// varies; every use of the list (the Jacobi projection and friction, summed in fixed point,
// the records of the backward's recompute, the pair-list query) is independent of it.
template <int NV, bool CONTACT, int TPR>
__device__ int broad_phase(const RodInfo& R, Smem<NV, CONTACT>& s, const Grp<TPR>& g, bool closed, bool& overflow) {
    float4* mid = s.HB0;                          // midpoint, half length of each edge (-1: a break edge)
    int* cnt = reinterpret_cast<int*>(s.HB1);     // [0] pairs found, [1] near block pairs, [2] listed edge pairs
    constexpr int kList = 4 * kPairsPerVertex * NV;
    uint32_t* list = reinterpret_cast<uint32_t*>(s.fr0);   // free between substeps
    uint32_t* nearb = reinterpret_cast<uint32_t*>(s.HB1) + 4;   // near block pairs kA | kB << 16, kA <= kB
    float4* blk = s.HB2;                          // centre, radius of each block of edges
    static_assert((NV / kBpBlock + 1) * (NV / kBpBlock + 2) / 2 + 4 <= 4 * NV, "block pairs fit in HB1");
    const int ne = R.ne, nv = R.nv;
    const bool strands = R.flags & ROD_STRANDS;
    const int nblk = (ne + kBpBlock - 1) / kBpBlock;
    {   // thread j's edge; its block's box and sphere over the block's kBpBlock neighbouring lanes
        static_assert(TPR >= NV && kBpBlock == 8, "one thread per edge, blocks of eight lanes");
        const int j = g.tid;
        const float inf = __int_as_float(0x7f800000);
        V3<float> p0 = f3(inf, inf, inf), p1 = p0, lo = p0, hi = f3(-inf, -inf, -inf);
        if (j < ne) {
            p0 = f3(s.X0[j]);
            p1 = f3(s.X0[j + 1 == nv ? 0 : j + 1]);
            const V3<float> e = p1 - p0;
            mid[j] = (strands && !(s.ET[j].w > 0.f)) ? make_float4(0.f, 0.f, 0.f, -1.f)
                                                     : f4(0.5f * (p0 + p1), 0.5f * sqrtf(dot(e, e)));
            lo = f3(fminf(p0.x, p1.x), fminf(p0.y, p1.y), fminf(p0.z, p1.z));
            hi = f3(fmaxf(p0.x, p1.x), fmaxf(p0.y, p1.y), fmaxf(p0.z, p1.z));
        }
#pragma unroll
        for (int o = 1; o < kBpBlock; o *= 2) {
            auto other = [&](float v) { return __shfl_xor_sync(0xffffffffu, v, o); };
            lo = f3(fminf(lo.x, other(lo.x)), fminf(lo.y, other(lo.y)), fminf(lo.z, other(lo.z)));
            hi = f3(fmaxf(hi.x, other(hi.x)), fmaxf(hi.y, other(hi.y)), fmaxf(hi.z, other(hi.z)));
        }
        const V3<float> c = 0.5f * (lo + hi), d0 = p0 - c, d1 = p1 - c;
        float r2 = j < ne ? fmaxf(dot(d0, d0), dot(d1, d1)) : 0.f;
#pragma unroll
        for (int o = 1; o < kBpBlock; o *= 2) r2 = fmaxf(r2, __shfl_xor_sync(0xffffffffu, r2, o));
        if (j % kBpBlock == 0 && j < ne) blk[j / kBpBlock] = f4(c, sqrtf(r2));
    }
    if (g.tid == 0) {
        cnt[0] = 0;
        cnt[1] = 0;
        cnt[2] = 0;
    }
    g.sync();
    const float cd = R.contact_d;
    // level 1: pairs of blocks
    constexpr int NB = NV <= 32 ? 4 : NV <= 64 ? 8 : NV <= 128 ? 16 : 32;   // blocks, as a power of two
    for (int q = g.tid; q < nblk * NB; q += TPR) {
        const int ka = q / NB, kb = q % NB;
        if (kb < ka || kb >= nblk) continue;
        const float4 A = blk[ka], B = blk[kb];
        const float dx = A.x - B.x, dy = A.y - B.y, dz = A.z - B.z;
        const float rr = (cd + A.w + B.w) * 1.0001f;
        if (dx * dx + dy * dy + dz * dz < rr * rr) nearb[atomicAdd(&cnt[1], 1)] = (uint32_t)ka | ((uint32_t)kb << 16);
    }
    g.sync();
    // level 2: an edge of the first block of a near pair against the second block's eight, whose
    // spheres are tested side by side.  Those that pass are listed and measured one per thread
    // (level 3), beyond the list's room at once.
    const int nn = cnt[1], cap = R.pair_cap, excl = R.excl;   // not read again after each store
    bool ovf = false;
    auto measure = [&](uint32_t pr) {
        const int a = (int)(pr & 0xffffu), b = (int)(pr >> 16);
        int sep = b - a;
        if (closed) sep = min(sep, ne - sep);
        if (!(sep > excl || (strands && break_between(s.ET, a, b)))) return;
        const int a1 = (a + 1 == nv) ? 0 : a + 1, b1 = (b + 1 == nv) ? 0 : b + 1;
        const V3<float> pa0 = f3(s.X0[a]), pa1 = f3(s.X0[a1]), pb0 = f3(s.X0[b]), pb1 = f3(s.X0[b1]);
        float su, uu;
        closest_params(pa0, pa1, pb0, pb1, su, uu);
        const V3<float> dd = (pa0 + su * (pa1 - pa0)) - (pb0 + uu * (pb1 - pb0));
        if (!(sqrtf(dot(dd, dd)) < cd)) return;
        const int idx = atomicAdd(&cnt[0], 1);
        if (idx < cap)
            s.pairs[idx] = pr;
        else
            ovf = true;
    };
    for (int t = g.tid; t < nn * kBpBlock; t += TPR) {
        const uint32_t bp = nearb[t / kBpBlock];
        const int a = (int)(bp & 0xffffu) * kBpBlock + t % kBpBlock, b0 = (int)(bp >> 16) * kBpBlock;
        const float4 ma = mid[min(a, ne - 1)];
        unsigned hits = 0;
#pragma unroll
        for (int m = 0; m < kBpBlock; ++m) {
            const int b = b0 + m;
            const float4 mb = mid[min(b, ne - 1)];
            const float dx = ma.x - mb.x, dy = ma.y - mb.y, dz = ma.z - mb.z, rr = (cd + ma.w + mb.w) * 1.00001f;
            int sep = b - a;
            if (closed) sep = min(sep, ne - sep);
            const bool near = b > a && b < ne && ma.w >= 0.f && mb.w >= 0.f && (sep > excl || strands) &&
                              dx * dx + dy * dy + dz * dz < rr * rr;
            hits |= near ? 1u << m : 0u;
        }
        if (hits) {
            int at = atomicAdd(&cnt[2], __popc(hits));
            for (; hits; hits &= hits - 1, ++at) {
                const uint32_t pr = (uint32_t)a | (uint32_t)(b0 + __ffs(hits) - 1) << 16;
                if (at < kList)
                    list[at] = pr;
                else
                    measure(pr);
            }
        }
    }
    g.sync();
    // level 3
    for (int t = g.tid; t < min(cnt[2], kList); t += TPR) measure(list[t]);
    g.sync();
    overflow = grp_any<TPR>(ovf, g);
    const int np = cnt[0];
    g.sync();
    return min(np, cap);
}

__device__ __forceinline__ unsigned cell_hash(int ix, int iy, int iz, int mask) {
    return ((unsigned)ix * 73856093u ^ (unsigned)iy * 19349663u ^ (unsigned)iz * 83492791u) & (unsigned)mask;
}

// The same candidates found through a per-rod spatial hash of the edge midpoints (the option
// ROD_HASH).  Cells are the candidate distance plus the frame's longest edge, so that the 27
// cells around an edge's cell hold every edge whose segment can come within the candidate
// distance of it (two midpoints are at most that far apart then).  Midpoints are counting-
// sorted into a table of buckets in shared memory (HB0 and HB1, free at this point); each
// edge then tests the edges of its 27 neighbouring cells.
template <int NV, bool CONTACT, int TPR>
__device__ int broad_phase_hash(const RodInfo& R, Smem<NV, CONTACT>& s, const Grp<TPR>& g, bool closed,
                                bool& overflow) {
    constexpr int TBL = NV <= 32 ? 64 : (NV <= 64 ? 128 : (NV <= 128 ? 256 : 512));
    static_assert(2 * NV + TBL + 1 <= 8 * NV, "the hash table fits in HB0 and HB1");
    int* keys = reinterpret_cast<int*>(s.HB0);
    int* cnt = keys + NV;            // TBL bucket counters, then the pair counter
    int* sorted = cnt + TBL + 1;
    const int ne = R.ne, nv = R.nv;
    const bool strands = R.flags & ROD_STRANDS;
    auto real = [&](int j) { return !strands || s.ET[j].w > 0.f; };   // break edges are no segments
    float lmax = 0.f;
    for (int j = g.tid; j < ne; j += TPR) {
        if (!real(j)) continue;
        const int j1 = (j + 1 == nv) ? 0 : j + 1;
        const V3<float> e = f3(s.X0[j1]) - f3(s.X0[j]);
        lmax = fmaxf(lmax, sqrtf(dot(e, e)));
    }
    for (int k = g.tid; k <= TBL; k += TPR) cnt[k] = 0;
    lmax = grp_max_nonneg<TPR>(lmax, g);
    const float inv_cell = 1.f / (R.contact_d + lmax);
    const V3<float> org = f3(s.X0[0]);
    for (int j = g.tid; j < ne; j += TPR) {
        if (!real(j)) continue;
        const int j1 = (j + 1 == nv) ? 0 : j + 1;
        const V3<float> m = 0.5f * (f3(s.X0[j]) + f3(s.X0[j1])) - org;
        const int ix = min(max(__float2int_rd(m.x * inv_cell), -510), 510) + 512;
        const int iy = min(max(__float2int_rd(m.y * inv_cell), -510), 510) + 512;
        const int iz = min(max(__float2int_rd(m.z * inv_cell), -510), 510) + 512;
        keys[j] = (ix << 20) | (iy << 10) | iz;
        atomicAdd(&cnt[cell_hash(ix, iy, iz, TBL - 1)], 1);
    }
    g.sync();
    {   // exclusive scan of the bucket counts, PER consecutive buckets per thread
        constexpr int PER = (TBL + TPR - 1) / TPR;
        int loc[PER];
        int sum = 0;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            loc[k] = g.tid * PER + k < TBL ? cnt[g.tid * PER + k] : 0;
            sum += loc[k];
        }
        int run = grp_excl_scan<TPR>(sum, g);
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if (g.tid * PER + k < TBL) {
                cnt[g.tid * PER + k] = run;
                run += loc[k];
            }
    }
    g.sync();
    for (int j = g.tid; j < ne; j += TPR) {
        if (!real(j)) continue;
        const int key = keys[j];
        const int pos = atomicAdd(&cnt[cell_hash(key >> 20, (key >> 10) & 1023, key & 1023, TBL - 1)], 1);
        sorted[pos] = j;
    }
    g.sync();
    // after the scatter cnt[h] is the end of bucket h (and the start of bucket h + 1)
    const int cap = R.pair_cap;
    const float cd = R.contact_d;
    bool ovf = false;
    for (int a = g.tid; a < ne; a += TPR) {
        if (!real(a)) continue;
        const int key = keys[a];
        const int ix = key >> 20, iy = (key >> 10) & 1023, iz = key & 1023;
        const int a1 = (a + 1 == nv) ? 0 : a + 1;
        const V3<float> pa0 = f3(s.X0[a]), pa1 = f3(s.X0[a1]);
        for (int dz = -1; dz <= 1; ++dz)
            for (int dy = -1; dy <= 1; ++dy)
                for (int dx = -1; dx <= 1; ++dx) {
                    const int cx = ix + dx, cy = iy + dy, cz = iz + dz;
                    const int nk = (cx << 20) | (cy << 10) | cz;
                    const unsigned hh = cell_hash(cx, cy, cz, TBL - 1);
                    const int beg = hh ? cnt[hh - 1] : 0, end = cnt[hh];
                    for (int q = beg; q < end; ++q) {
                        const int b = sorted[q];
                        if (b <= a || keys[b] != nk) continue;
                        int sep = b - a;
                        if (closed) sep = min(sep, ne - sep);
                        if (sep <= R.excl && !(strands && break_between(s.ET, a, b))) continue;
                        const int b1 = (b + 1 == nv) ? 0 : b + 1;
                        const V3<float> pb0 = f3(s.X0[b]), pb1 = f3(s.X0[b1]);
                        float su, uu;
                        closest_params(pa0, pa1, pb0, pb1, su, uu);
                        const V3<float> dd = (pa0 + su * (pa1 - pa0)) - (pb0 + uu * (pb1 - pb0));
                        if (!(sqrtf(dot(dd, dd)) < cd)) continue;
                        const int idx = atomicAdd(&cnt[TBL], 1);
                        if (idx < cap)
                            s.pairs[idx] = (uint32_t)a | ((uint32_t)b << 16);
                        else
                            ovf = true;
                    }
                }
    }
    g.sync();
    overflow = grp_any<TPR>(ovf, g);
    const int np = cnt[TBL];
    g.sync();
    return min(np, cap);
}

// ------------------------------------------------------------------ PBD pieces
// Length projections (inextensibility, strain limit): edges of even index, then of odd index
// (an odd loop's last edge after both), N_C times.  Thread t of the first pbd_threads takes the
// edges 2t and 2t + 1: vertex 2t + 1 belongs to no other edge and stays in its registers, as do the
// edges' start vectors, targets and weights; only the even vertices go through shared memory,
// one load and one store per colour, between barriers of the projecting warps alone.  (Every
// thread meeting at a barrier per colour and reading both ends' positions, displacements and
// the rest length took about 480 cycles per colour.)
__host__ __device__ constexpr int pbd_threads(int NV) { return NV <= 64 ? 32 : (NV / 2 + 31) / 32 * 32; }

// Barrier of a rod's projecting threads (bar: the rod's own barrier, 1..4 where this one is named).
template <int NV>
__device__ __forceinline__ void pbd_sync(int bar) {
    if (pbd_threads(NV) == 32)
        __syncwarp();
    else
        asm volatile("bar.sync %0, %1;" ::"r"(bar + 7), "r"(pbd_threads(NV)) : "memory");
}

struct ProjEdge {
    bool on;          // an edge with a length and at least one free end
    V3<float> r;      // start vector
    float hi, lo;     // bounds of the length (equal for an inextensible edge)
    float wa, wb, ws;
};

// One projection (App. A.1) of the edge between displacements A and B: C = |x_{j+1} - x_j| -
// target, lambda = C / (w_j + w_{j+1}).  Returns its record (Rec::pbd).
__device__ __forceinline__ float4 project_edge(const ProjEdge& p, bool inext, V3<float>& A, V3<float>& B) {
    const V3<float> e = p.r + (B - A);
    float ell, ie;
    len_inv(e, ell, ie);
    const float target = ell > p.hi ? p.hi : p.lo;
    if (!(p.on && (inext || ell > p.hi || ell < p.lo))) return make_float4(0.f, 0.f, 0.f, 1.f);
    const float lam = (ell - target) / p.ws;
    const V3<float> t = ie * e;
    A += (lam * p.wa) * t;
    B -= (lam * p.wb) * t;
    return f4(t, target * ie);
}

// One Jacobi sweep over the candidate pairs.  With ask, returns whether any pair was closer than
// the two radii (the positions are as they were otherwise).  The group has synchronised on return.
template <int NV, bool CONTACT, int TPR>
__device__ __forceinline__ bool contact_sweep(const RodInfo& R, Smem<NV, CONTACT>& s, const Grp<TPR>& g, int np,
                                              bool first, bool ask) {
    const int nv = R.nv;   // s.acc is zero on entry and is left zero
    const float rsum = 2.f * R.radius;
    bool acts = false;
    for (int p = g.tid; p < np; p += TPR) {
        uint32_t pr = s.pairs[p];
        int a0 = pr & 0xffff, c0 = pr >> 16;
        if (!in_bounds(a0 < nv && c0 < nv && p < R.pair_cap, s.red)) continue;
        int a1 = (a0 + 1 == nv) ? 0 : a0 + 1, c1 = (c0 + 1 == nv) ? 0 : c0 + 1;
        // current positions in coordinates local to the start position of vertex a0
        const V3<float> o = f3(s.X0[a0]);
        float4 A0 = s.X[a0], A1 = s.X[a1], C0 = s.X[c0], C1 = s.X[c1];
        V3<float> pa0 = f3(A0), pa1 = (f3(s.X0[a1]) - o) + f3(A1);
        V3<float> pc0 = (f3(s.X0[c0]) - o) + f3(C0), pc1 = (f3(s.X0[c1]) - o) + f3(C1);
        V3<float> dx[4], n;
        float su, uu, d, W;
        bool on = pair_correction(pa0, pa1, pc0, pc1, A0.w, A1.w, C0.w, C1.w, rsum, dx, su, uu, n, d, W);
        if (first) {
            s.fr0[p] = f4(on ? n : zf3(), on ? d : 0.f);
            s.fr1[p] = make_float4(su, uu, W, on ? 1.f : 0.f);
        }
        if (on) {
            acts = true;
            const int idx[4] = {a0, a1, c0, c1};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                atomicAdd(&s.acc[idx[k]].x, to_fix(dx[k].x, kFixPos));
                atomicAdd(&s.acc[idx[k]].y, to_fix(dx[k].y, kFixPos));
                atomicAdd(&s.acc[idx[k]].z, to_fix(dx[k].z, kFixPos));
            }
        }
    }
    if (ask) {
        if (!g.sync_any(acts)) return false;
    } else {
        g.sync();
    }
    for (int i = g.tid; i < nv; i += TPR) {
        int4 q = s.acc[i];
        if (q.x | q.y | q.z) {
            float4 x = s.X[i];
            const float inv = 1.f / kFixPos;
            s.X[i] = make_float4(x.x + q.x * inv, x.y + q.y * inv, x.z + q.z * inv, x.w);
            s.acc[i] = make_int4(0, 0, 0, 0);
        }
    }
    g.sync();
    return true;
}

template <int NV, bool CONTACT, int TPR>
__device__ __forceinline__ void self_friction(const RodInfo& R, Smem<NV, CONTACT>& s, const Grp<TPR>& g, int np,
                                              float h, float mu) {
    const int nv = R.nv;   // s.acc is zero on entry and is left zero
    for (int p = g.tid; p < np; p += TPR) {
        float4 F1 = s.fr1[p];
        if (!(F1.w > 0.f)) continue;
        float4 F0 = s.fr0[p];
        uint32_t pr = s.pairs[p];
        int a0 = pr & 0xffff, c0 = pr >> 16;
        if (!in_bounds(a0 < nv && c0 < nv && p < R.pair_cap, s.red)) continue;
        int a1 = (a0 + 1 == nv) ? 0 : a0 + 1, c1 = (c0 + 1 == nv) ? 0 : c0 + 1;
        float su = F1.x, uu = F1.y, W = F1.z;
        V3<float> n = f3(F0);
        V3<float> vrel = (1.f - su) * f3(s.V[a0]) + su * f3(s.V[a1]) - (1.f - uu) * f3(s.V[c0]) - uu * f3(s.V[c1]);
        V3<float> vt = vrel - dot(vrel, n) * n;
        float vt2 = dot(vt, vt);
        if (!(vt2 > 1e-24f)) continue;
        float coef = fminf(mu * F0.w / (h * sqrtf(vt2)), 1.f);
        V3<float> dv = (-(coef / W)) * vt;
        const int idx[4] = {a0, a1, c0, c1};
        const float wt[4] = {s.X[a0].w * (1.f - su), s.X[a1].w * su, -s.X[c0].w * (1.f - uu), -s.X[c1].w * uu};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            atomicAdd(&s.acc[idx[k]].x, to_fix(wt[k] * dv.x, kFixVel));
            atomicAdd(&s.acc[idx[k]].y, to_fix(wt[k] * dv.y, kFixVel));
            atomicAdd(&s.acc[idx[k]].z, to_fix(wt[k] * dv.z, kFixVel));
        }
    }
    g.sync();
    for (int i = g.tid; i < nv; i += TPR) {
        int4 q = s.acc[i];
        if (q.x | q.y | q.z) {
            float4 v = s.V[i];
            const float inv = 1.f / kFixVel;
            s.V[i] = make_float4(v.x + q.x * inv, v.y + q.y * inv, v.z + q.z * inv, v.w);
            s.acc[i] = make_int4(0, 0, 0, 0);
        }
    }
    g.sync();
}

// The N_C projection iterations of a substep on the displacements s.X: the length projections of
// both colours and, with SWEEPS, a self-contact sweep.  A rod without length projections stops at
// the first sweep that moves nothing (of the sweeps of 400 knotted ropes after the first three
// quarters move nothing: 1.44 -> 1.13 ms for 20 frames).  The group has synchronised since s.X was
// written; on return it has synchronised after the last iteration.
template <int NV, bool CONTACT, int TPR, bool REC, bool SWEEPS>
__device__ __forceinline__ void run_projections(const RodInfo& R, Smem<NV, CONTACT>& s, const Grp<TPR>& g, int n_iter, int np,
                                        const Rec<NV, REC> rec) {
    const int nv = R.nv, ne = R.ne, i = g.tid;
    const bool closed = R.flags & ROD_CLOSED, lenc = R.flags & (ROD_INEXT | ROD_SLIMIT), inext = R.flags & ROD_INEXT;
    const bool ring = closed && (ne & 1);
    const bool proj = lenc && i < pbd_threads(NV);
    const int j = 2 * i, j2 = j + 2 >= nv ? 0 : j + 2;   // the edges j (to j + 1) and j + 1 (to j2)
    const bool last = ring && j == ne - 1;               // edge j is an odd loop's last: ends at vertex 0
    ProjEdge p0{}, p1{};
    V3<float> mid = zf3();                               // displacement of vertex j + 1
    if (proj) {
        auto edge = [&](int k, int k1) {
            ProjEdge p;
            const float len = s.ET[k].w;
            const float4 xa = s.X0[k], xb = s.X0[k1];
            p.r = f3(xb) - f3(xa);
            p.hi = inext ? len : (1.f + R.slim) * len;
            p.lo = inext ? len : (1.f - R.slim) * len;
            p.wa = xa.w;
            p.wb = xb.w;
            p.ws = xa.w + xb.w;
            p.on = p.ws > 0.f && len > 0.f;   // length 0: the edge between two strands
            return p;
        };
        if (j < ne) p0 = edge(j, last || j + 1 == nv ? 0 : j + 1);
        if (j + 1 < ne) p1 = edge(j + 1, j2);
        if (j + 1 < nv) mid = f3(s.X[j + 1]);
    }
    for (int it = 0; it < n_iter; ++it) {
        if (proj) {
            auto put = [&](int k, float4 q) {
                if (REC) rec.pbd(it)[k] = q;
            };
            if (j < ne && !last) {
                const float4 a4 = s.X[j];
                V3<float> A = f3(a4);
                put(j, project_edge(p0, inext, A, mid));
                s.X[j] = f4(A, a4.w);
            }
            pbd_sync<NV>(g.bar);
            if (j + 1 < ne) {
                const float4 b4 = s.X[j2];
                V3<float> B = f3(b4);
                put(j + 1, project_edge(p1, inext, mid, B));
                s.X[j2] = f4(B, b4.w);
            }
            if (SWEEPS || it + 1 == n_iter)
                if (j + 1 < nv) s.X[j + 1] = f4(mid, p0.wb);
            if (ring) {
                pbd_sync<NV>(g.bar);
                if (last) {
                    const float4 a4 = s.X[j], b4 = s.X[0];
                    V3<float> A = f3(a4), B = f3(b4);
                    put(j, project_edge(p0, inext, A, B));
                    s.X[j] = f4(A, a4.w);
                    s.X[0] = f4(B, b4.w);
                }
            }
            if (!SWEEPS) pbd_sync<NV>(g.bar);
        }
        if (SWEEPS) {
            if (lenc) g.sync();
            // each thread stores its own vertices; the sweep reads s.X and writes only the
            // accumulators before its own barrier
            if (REC && i < nv) rec.csnap(it)[i] = s.X[i];
            if (contact_sweep<NV, CONTACT, TPR>(R, s, g, np, it == 0, !lenc)) {
                if (proj && j + 1 < nv) mid = f3(s.X[j + 1]);
            } else {   // nothing moves any more: the sweeps left would find the same
                if (REC && i < nv)
                    for (int k = it + 1; k < n_iter; ++k) rec.csnap(k)[i] = s.X[i];
                break;
            }
        }
    }
    if (!SWEEPS) g.sync();
}

// With contact sweeps, and the friction, as out-of-line calls.  They run only on frames with
// candidates; kept out of the substep's inlined code they add no registers, and no code, to
// the path every substep takes.  The rod's shared-memory view is rebuilt from its base
// inside (a view passed by reference would be read from memory at every use).
template <int NV, bool CONTACT, int TPR, bool REC>
__device__ __noinline__ void run_projections_call(const RodInfo* Rp, float4* base, int gtid, int gbar, int n_iter, int np,
                                          float4* rec) {
    Smem<NV, CONTACT> s(base);
    const Grp<TPR> g{gtid, gbar, s.red};
    const RodInfo R = *Rp;
    run_projections<NV, CONTACT, TPR, REC, true>(R, s, g, n_iter, np, Rec<NV, REC>{rec, n_iter});
}

template <int NV, bool CONTACT, int TPR>
__device__ __noinline__ void self_friction_call(const RodInfo* R, float4* base, int gtid, int gbar, int np,
                                                float h, float mu) {
    Smem<NV, CONTACT> s(base);
    const Grp<TPR> g{gtid, gbar, s.red};
    self_friction<NV, CONTACT, TPR>(*R, s, g, np, h, mu);
}

// An edge's frame for the hinge phase from its stored (t, |e|), (d1r, cos theta) and
// sin theta: d2r = t x d1r and the material frame, as edge_forward forms them.
__device__ __forceinline__ void load_frame(EdgeF<float>& E, float4 ta, float4 rc, float sn) {
    E.t = f3(ta);
    E.d1r = f3(rc);
    E.c = rc.w;
    E.s = sn;
    material_directors(E);
}

// ------------------------------------------------------------------ one substep
// What a thread keeps of its own vertex and edge for the whole rod.
struct Own {
    int kind;      // 0 free, 1 pinned, 2 / 3 held by gripper 0 / 1
    float invI;    // 1 / axial inertia of the edge that starts here
};

__device__ __forceinline__ Own own_of(const float4* __restrict__ KIN, const float2* __restrict__ ES, const RodInfo& R,
                                      int i) {
    return Own{i < R.nv ? (int)KIN[R.v0 + i].w : 1, i < R.ne ? ES[R.e0 + i].y : 0.f};
}

// Target of a held vertex at the substep's end: the gripper's end pose applied to its grasp offset.
__device__ __forceinline__ V3<float> grasp_target(const float* sp, int kind, float4 kin) {
    const float* o = sp + 32 * (kind - 2);
    const V3<float> off = f3(kin);
    const V3<float> p1 = f3(o[3], o[4], o[5]);
    return p1 + f3(o[15] * off.x + o[16] * off.y + o[17] * off.z, o[18] * off.x + o[19] * off.y + o[20] * off.z,
                   o[21] * off.x + o[22] * off.y + o[23] * off.z);
}

// The group has synchronised since X0, V, ED, ET, HG and sp were written; on return it has
// synchronised after writing them.  sp: the substep's gripper block.  The substep is bound by
// the latency of its phases' dependent arithmetic and of the barriers between them (about a
// third of the issue slots at four 128-vertex rods per SM), so it keeps instructions and
// barriers few: one thread per element, four phases for a rod without projections, and no
// atomics (a hinge's seeds for its previous edge travel through one slot; float atomics on
// shared memory are compare-and-swap loops).  4096 elastic ropes x 128 vertices: 30.2 -> 19.1 us
// per substep of the batch against atomics and elements spread over at most 128 threads; one
// 256-vertex class of the ragged batch 4.2 -> 1.5 ms.
template <int NV, bool CONTACT, int TPR, bool REC>
__device__ __forceinline__ void substep_body(const SceneDev& sc, const float4* __restrict__ KIN, const RodInfo& R,
                                             const Own& own, Smem<NV, CONTACT>& s, const Grp<TPR>& g, float h, int np,
                                             const float* sp, const Rec<NV, REC> rec, float4* imp = nullptr,
                                             float* mv = nullptr) {
    static_assert(TPR >= NV, "one thread per vertex");
    const int nv = R.nv, ne = R.ne;
    const bool closed = R.flags & ROD_CLOSED;
    const bool strands = R.flags & ROD_STRANDS;
    const int i = g.tid;
    const int ip = (i + 1 == nv) ? 0 : i + 1;       // end vertex of the own edge
    const int im = (i == 0) ? nv - 1 : i - 1;       // the edge that ends at the own vertex (if any)
    const bool vtx = i < nv, has_e = i < ne, has_em = vtx && (closed || i > 0);
    // exchanged between neighbours; the displacement array SR = X is rewritten by the vertex
    // phase before it is read
    float4* const FA = s.HB0;   // per edge (t, sin theta)
    float4* const FB = s.HB1;   // per edge (d1r, cos theta)
    float4* const SG = s.HB2;   // per edge (dU/dt, dU/dtheta) of the hinge at its end; then (dU/de, K A strain)
    float4* const SR = s.X;     // per edge dU/dd1r of the hinge at its end
    // --- the own edge's frame.  A break edge (rest length 0) has no frame and no hinge.
    EdgeF<float> E;
    V3<float> tb, d1b;
    float theta = 0.f, eb = 0.f;
    bool real = false;
    if (has_e) {
        const float4 ed = s.ED[i], et = s.ET[i];
        tb = f3(et);
        d1b = f3(ed);
        theta = ed.w;
        eb = et.w;
        real = !(strands && !(eb > 0.f));
        if (real) {
            edge_forward(E, f3(s.X0[i]), f3(s.X0[ip]), tb, d1b, theta);
            FA[i] = f4(E.t, E.s);
            FB[i] = f4(E.d1r, E.c);
        }
    }
    g.sync();
    // --- the own hinge, from its edges' frames: seeds for the own edge (kept) and for the
    // previous one (sent; zero where there is no active hinge)
    V3<float> gtb = zf3(), gd1rb = zf3();
    float ghtb = 0.f;
    if (has_em) {
        V3<float> gta = zf3(), gd1ra = zf3();
        float ghta = 0.f;
        const float eba = s.ET[im].w;
        if (has_e && !(strands && !(eba > 0.f && eb > 0.f))) {
            float4 hg = s.HG[i];
            HingeF<float> H;
            const float4 fa = FA[im], fb = FB[im];
            load_frame(H.a, fa, fb, fa.w);
            H.b = E;
            hinge_core_forward(H, s.ED[im].w, theta, hg.w);
            const float lbar = 0.5f * (eba + eb);
            if (R.flags & ROD_PLASTIC) plastic_update(H.k0, H.k1, hg.x, hg.y, R.sy * lbar, R.rc);
            const float il = 1.f / lbar;
            const float gk0 = R.Bm * il * (H.k0 - hg.x), gk1 = R.Bm * il * (H.k1 - hg.y);
            const float gm = R.beta * il * (H.m - hg.z);
            hinge_core_reverse(H, gk0, gk1, gm, 0.f, gta, gd1ra, gtb, gd1rb, ghta, ghtb);
            s.HG[i] = make_float4(hg.x, hg.y, hg.z, H.mref);
        }
        SG[im] = f4(gta, ghta);
        SR[im] = f4(gd1ra, 0.f);
    }
    g.sync();
    // --- the reverse through the own edge's frame: the gradient on the edge vector.  The
    // stretching strain has an IEEE-rounded square root and quotient (the strains of nearly
    // inextensible ropes are ~1e-4, so a few ulps of the length matter to them).
    V3<float> ge = zf3();
    float gth = 0.f, str = 0.f;
    if (has_e) {
        if (real) {
            const float4 sg = SG[i], sr = SR[i];
            gth = sg.w + ghtb;
            ge = edge_reverse<float, false>(E, tb, d1b, f3(sg) + gtb, f3(sr) + gd1rb, 0.f, nullptr, nullptr);
            if (R.kA > 0.f) str = R.kA * edge_strain(f3(s.X0[ip]) - f3(s.X0[i]), eb);
        }
        SG[i] = f4(ge, str);
    }
    g.sync();
    // --- the own vertex
    const bool lenc = R.flags & (ROD_INEXT | ROD_SLIMIT);
    const bool project = lenc || (CONTACT && np > 0);
    const float ih = 1.f / h;
    // new position (the absolute target for a held vertex) and velocity from the displacement d
    const bool held = own.kind >= 2 && in_bounds(own.kind - 2 < R.ngrip, s.red);
    auto finish = [&](float4 x0, V3<float> d, float om, V3<float> target) {
        float4 x = make_float4(x0.x + d.x, x0.y + d.y, x0.z + d.z, x0.w);
        if (held) x = f4(target, x0.w);
        if (mv) {
            const float dx = x.x - x0.x, dy = x.y - x0.y, dz = x.z - x0.z;
            *mv += sqrtf(dx * dx + dy * dy + dz * dz);
        }
        s.X0[i] = x;
        s.V[i] = make_float4(d.x * ih, d.y * ih, d.z * ih, om);
    };
    if (vtx) {
        const float4 xi4 = s.X0[i];
        const V3<float> xi = f3(xi4);
        V3<float> gr = zf3();
        float4 pe = make_float4(0.f, 0.f, 0.f, 0.f);
        if (has_e) gr -= ge;
        if (has_em) {
            pe = SG[im];
            gr += f3(pe);
        }
        if (R.kA > 0.f) {
            if (real) gr -= str * E.t;
            if (has_em && !(strands && !(s.ET[im].w > 0.f))) gr += pe.w * f3(FA[im]);
        }
        const float4 vi = s.V[i];
        // displacement d of this substep (positions are only formed at its end, so the rebuilt
        // velocity d/h carries no cancellation error from |x| >> |h v|)
        V3<float> d = zf3(), target = zf3();
        if (own.kind == 0) {
            V3<float> grav = f3(0.f, 0.f, -sc.gravity);
            V3<float> acc = (-xi4.w) * gr + grav - R.cd * f3(vi);
            V3<float> v1 = f3(vi) + h * acc;
            if (REC) rec.v1()[i] = f4(v1, 0.f);
            const V3<float> v2 = rigid_contact(sc, R, xi, v1, sp, imp ? imp + 4 * i : nullptr, 1.f / xi4.w);
            d = h * v2;
        } else if (held) {   // a held vertex sits at its target
            target = grasp_target(sp, own.kind, KIN[R.v0 + i]);
            d = target - xi;
        }
        float om1 = vi.w;
        if (has_e) {
            om1 = vi.w + h * (-gth * own.invI - R.cd * vi.w);
            const float th1 = theta + h * om1;
            if (real) {
                s.ED[i] = f4(E.d1r, th1);   // the edge's new reference director
                s.ET[i] = f4(E.t, eb);
            } else {
                s.ED[i] = f4(d1b, th1);
            }
        }
        if (project) {
            s.X[i] = f4(d, xi4.w);
            s.V[i].w = om1;
        } else {
            if (REC) rec.dfin()[i] = f4(d, xi4.w);
            finish(xi4, d, om1, target);
        }
    }
    g.sync();
    if (!project) return;
    // --- PBD
    if (CONTACT && np > 0)
        run_projections_call<NV, CONTACT, TPR, REC>(&R, s.X, g.tid, g.bar, sc.n_iter, np, rec.base);
    else
        run_projections<NV, CONTACT, TPR, REC, false>(R, s, g, sc.n_iter, 0, rec);
    // --- velocity from the displacement, new positions, friction
    if (vtx) {
        const float4 d = s.X[i];
        if (REC) rec.dfin()[i] = d;
        finish(s.X0[i], f3(d), s.V[i].w, held ? grasp_target(sp, own.kind, KIN[R.v0 + i]) : zf3());
    }
    if (CONTACT && REC)
        for (int p = g.tid; p < np; p += TPR) {
            rec.fr0()[p] = s.fr0[p];
            rec.fr1()[p] = s.fr1[p];
        }
    g.sync();
    if (CONTACT && np > 0) self_friction_call<NV, CONTACT, TPR>(&R, s.X, g.tid, g.bar, np, h, sc.mu_self);
}

// Substep pose block of gripper q (32 floats at out + 32 q) from the frame-start pose F
// (per gripper p (3), R (9) row major) and the frame's actions: positions and rotations at
// the substep's start (c0) and end (c1) of the frame, p + c dp and exp(c dphi) R (the start
// rotation of the first substep is the frame's own), and the rigid velocities dp/dt, dphi/dt.
__device__ __forceinline__ void substep_pose(const SceneDev& sc, const RodInfo& R, const float* F, const float* act,
                                             int q, float c0, float c1, bool first, float inv_dt, float* out) {
    const float* f = F + 12 * q;
    const float* a = act + 6 * q;
    M3 RF;
#pragma unroll
    for (int k = 0; k < 9; ++k) RF.m[k] = f[3 + k];
    const M3 R0 = first ? RF : matmul(expmap(f3(c0 * a[3], c0 * a[4], c0 * a[5])), RF);
    const M3 R1 = matmul(expmap(f3(c1 * a[3], c1 * a[4], c1 * a[5])), RF);
    float* o = out + 32 * q;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        o[c] = f[c] + c0 * a[c];
        o[3 + c] = f[c] + c1 * a[c];
        o[24 + c] = a[c] * inv_dt;
        o[27 + c] = a[3 + c] * inv_dt;
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        o[6 + k] = R0.m[k];
        o[15 + k] = R1.m[k];
    }
    o[30] = grip_bound(sc, R, o);
}

// Frame end for gripper q: p += dp, R = exp(dphi) R.
__device__ __forceinline__ void frame_advance(float* F, const float* act, int q) {
    float* f = F + 12 * q;
    const float* a = act + 6 * q;
    M3 RF;
#pragma unroll
    for (int k = 0; k < 9; ++k) RF.m[k] = f[3 + k];
    const M3 Rn = matmul(expmap(f3(a[3], a[4], a[5])), RF);
#pragma unroll
    for (int c = 0; c < 3; ++c) f[c] += a[c];
#pragma unroll
    for (int k = 0; k < 9; ++k) f[3 + k] = Rn.m[k];
}

// ------------------------------------------------------------------ record layout
// Records of a run of frames (a chunk, or the whole rollout), per rod (float4 units; NV the size
// class, n the substeps reserved per frame, N the projection iterations):
//   per frame, kFrameHead + NV:  its start pose (24 floats) and candidate count (int at float 24),
//                                then its candidate pairs (4 NV uint32)
//   per substep, sub_rec(NV, N): start state (X0, V, HG, ED, ET; 5 NV), v1 (NV), dfin (NV),
//                                projection records (N NV), contact snapshots (N NV), first-
//                                iteration pair data fr0, fr1 (4 NV each)
// Only what a frame uses is written and read (projection records for length-constrained rods,
// snapshots and pair data for frames with candidates).
constexpr int kFrameHead = 8;
__host__ __device__ constexpr size_t sub_rec(int NV, int n_iter) {
    return (size_t)(7 + 2 * n_iter + 2 * kPairsPerVertex) * NV;
}
__host__ __device__ constexpr size_t frame_rec(int NV, int n_iter, int nsub) {
    return (size_t)(kFrameHead + NV) + (size_t)nsub * sub_rec(NV, n_iter);
}
// frame-start state of one frame of a segment: X0, V, HG, ED, ET and the pose (24 floats)
__host__ __device__ constexpr size_t seg_state(int NV) { return (size_t)5 * NV + 6; }
// cotangent state carried from one chunk's reverse to the next: LX, LV, LE, LT, LK (two floats,
// and in the upper half of the first 12 the frame-start pose cotangents, a double each), then
// the material sums (5 doubles)
__host__ __device__ constexpr size_t cot_state(int NV) { return (size_t)5 * NV + 6; }

// State snapshot layout in the per-rod scratch: X[NV], V[NV], HG[NV], ED[NV], ET[NV].
template <int NV, bool C, int TPR>
__device__ __forceinline__ void save_state(float4* dst, const RodInfo& R, const Grp<TPR>& g, const Smem<NV, C>& s) {
    for (int i = g.tid; i < R.nv; i += TPR) {
        dst[i] = s.X0[i];
        dst[NV + i] = s.V[i];
        dst[2 * NV + i] = s.HG[i];
    }
    for (int j = g.tid; j < R.ne; j += TPR) {
        dst[3 * NV + j] = s.ED[j];
        dst[4 * NV + j] = s.ET[j];
    }
}

// The records of substep sb of the frame whose record is fb: stores its start state (each thread
// its own vertex and edge) and returns where the substep stores the rest.
template <int NV, bool CONTACT, int TPR>
__device__ __forceinline__ Rec<NV, true> record_substep(float4* fb, int sb, int n_iter, const RodInfo& R,
                                                        const Grp<TPR>& g, const Smem<NV, CONTACT>& s) {
    float4* e3 = fb + kFrameHead + NV + (size_t)sb * sub_rec(NV, n_iter);
    save_state<NV, CONTACT, TPR>(e3, R, g, s);
    return Rec<NV, true>{e3, n_iter};
}
// The frame's candidates, into its record.
template <int NV, bool CONTACT, int TPR>
__device__ __forceinline__ void record_pairs(float4* fb, int np, const Grp<TPR>& g, const Smem<NV, CONTACT>& s) {
    uint32_t* pl = reinterpret_cast<uint32_t*>(fb + kFrameHead);
    for (int p = g.tid; p < np; p += TPR) pl[p] = s.pairs[p];
    if (g.tid == 0) reinterpret_cast<int*>(fb)[24] = np;
}

// One frame of one rod: candidates (if self-contact), nsub substeps, pose update.  The frame's
// start pose is s.fp and its actions s.act, both set (and synchronised) by the caller; s.fp
// holds the end pose on return.  pre(sb) runs before substep sb (after a group barrier), e.g.
// to store the substep state, and returns where the substep's records go.  imp: the rod's
// impulse slots (4 per vertex) when the contact impulses are being accumulated.  mv: adds, per
// thread, the sum over the frame's substeps of its vertex's displacement, a bound on how far it
// moved during the frame.
template <int NV, bool CONTACT, int TPR, class PreSub>
__device__ __forceinline__ int run_frame(const SceneDev& sc, const float4* __restrict__ KIN, const RodInfo& R,
                                         const Own& own, Smem<NV, CONTACT>& s, const Grp<TPR>& g, int nsub, float h,
                                         bool& ovf, PreSub pre, float4* imp = nullptr, float* mv = nullptr) {
    int np = 0;
    if (CONTACT && (R.flags & ROD_SELF))
        np = (R.flags & ROD_HASH) ? broad_phase_hash<NV, CONTACT, TPR>(R, s, g, (R.flags & ROD_CLOSED) != 0, ovf)
                                  : broad_phase<NV, CONTACT, TPR>(R, s, g, (R.flags & ROD_CLOSED) != 0, ovf);
    const float inv_dt = 1.f / sc.dt;
    for (int sb = 0; sb < nsub; ++sb) {
        // the gripper blocks of the next kPoseBatch substeps, one per thread, side by side (two
        // rotation exponentials each: done by one thread every substep they were about a tenth
        // of a lone rod's substep); read after the hinge phase's barrier
        if (sb % kPoseBatch == 0) {
            const int k = sb + (g.tid >> 1), q = g.tid & 1;
            if (g.tid < 2 * kPoseBatch && k < nsub && q < R.ngrip)
                substep_pose(sc, R, s.fp, s.act, q, (float)k / (float)nsub, (float)(k + 1) / (float)nsub, k == 0,
                             inv_dt, s.sp + 64 * (g.tid >> 1));
        }
        substep_body(sc, KIN, R, own, s, g, h, np, s.sp + 64 * (sb % kPoseBatch), pre(sb), imp, mv);
    }
    if (g.tid < R.ngrip) frame_advance(s.fp, s.act, g.tid);
    g.sync();
    return np;
}

}  // namespace dlo
