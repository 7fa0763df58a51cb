// dlo_bwd_kernel.cuh -- hand-written adjoint of the rod stepper with gradient checkpointing.
//
// DLO-Lab (Sec. 3.3) differentiates whole trajectories by caching one state per segment and,
// for each segment in reverse, re-running the forward simulation before back-propagating.
// Here the checkpoints live in HBM (written by the forward kernel every K frames) and the
// rollout is reversed in chunks of frames, last first, by two persistent kernels per chunk:
//   rec_kernel   forward-like (a rod per CTA, see best_shape; not run when the forward stored the
//                records): re-runs the chunk's frames from their start state and stores every
//                substep's records in HBM: its start state, the
//                velocity before rigid contact, the displacement before friction, one record
//                per edge and projection iteration (direction and target / length), the
//                displacements before each contact sweep and the first iteration's pair data;
//                for checkpoints more than a chunk apart it first stores the start state of
//                each of the segment's frames
//   rev_kernel   one group per rod: for each frame and substep, last first, loads the records
//                and applies the vector-Jacobian product of every phase in reverse order; the
//                cotangents of the rod's state are carried to the next chunk in HBM
// Second-order terms of the elastic forces are exact: the hinge gradient (a hand reverse pass)
// is re-run on dual numbers, giving d/de [dU/dz](x + e lambda) for every input z, which is
// the transpose-Jacobian product of the force (U's Hessian is symmetric).  Branches (contact
// on/off, yield, strain-limit activity, pair sets) follow the recomputed forward.
#pragma once
#include "dlo_fwd_kernel.cuh"

namespace dlo {

// ------------------------------------------------------------------ small helpers
__device__ __forceinline__ void atomic_add3(float4* a, V3<float> v) {
    atomicAdd(&a->x, v.x);
    atomicAdd(&a->y, v.y);
    atomicAdd(&a->z, v.z);
}

// J_l(phi)^T lam for the left Jacobian of the rotation exponential:
// exp([phi + d]x) ~ exp([J_l(phi) d]x) exp([phi]x),  J_l = I + A [phi]x + B [phi]x^2.
__device__ __forceinline__ V3<float> jl_t(V3<float> phi, V3<float> lam) {
    float t2 = dot(phi, phi), A, B;
    if (t2 < 1e-8f) {
        A = 0.5f - t2 / 24.f;
        B = 1.f / 6.f - t2 / 120.f;
    } else {
        float t = sqrtf(t2), sh = sinf(0.5f * t);
        A = 2.f * sh * sh / t2;
        B = (t - sinf(t)) / (t2 * t);
    }
    V3<float> c = cross(phi, lam);
    return lam - A * c + B * cross(phi, c);
}

// The linear maps that carry gripper q's substep pose cotangents to the frame's actions and
// start pose (see the pose block of reverse_substep), per gripper: M0 = exp(c0 dphi),
// M1 = exp(c1 dphi), c0 J_l(c0 dphi)^T and c1 J_l(c1 dphi)^T (row major, 9 floats each).  Thread
// t < 4 ngrip builds matrix t % 4 of gripper t / 4, so the eight run side by side.  With
// phi = c dphi: J_l(phi)^T = I - A [phi]x + B [phi]x^2, the coefficients of jl_t above.
__device__ __forceinline__ void pose_rev_mat(const float* act, int t, float c0, float c1, float* pm) {
    const int q = t >> 2, m = t & 3;
    const float c = (m & 1) ? c1 : c0;
    const V3<float> phi = c * f3(act[6 * q + 3], act[6 * q + 4], act[6 * q + 5]);
    float* o = pm + 36 * q + 9 * m;
    if (m < 2) {
        const M3 M = expmap(phi);
#pragma unroll
        for (int k = 0; k < 9; ++k) o[k] = M.m[k];
        return;
    }
    const float t2 = dot(phi, phi);
    float A, B;
    if (t2 < 1e-8f) {
        A = 0.5f - t2 / 24.f;
        B = 1.f / 6.f - t2 / 120.f;
    } else {
        const float th = sqrtf(t2), sh = sinf(0.5f * th);
        A = 2.f * sh * sh / t2;
        B = (th - sinf(th)) / (t2 * th);
    }
    const float p[3] = {phi.x, phi.y, phi.z};
    const float d = 1.f - B * t2;
    // [phi]x = [[0, -z, y], [z, 0, -x], [-y, x, 0]]
    const float K[9] = {0.f, -phi.z, phi.y, phi.z, 0.f, -phi.x, -phi.y, phi.x, 0.f};
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int k = 0; k < 3; ++k) o[3 * r + k] = c * ((r == k ? d : 0.f) - A * K[3 * r + k] + B * p[r] * p[k]);
}

// One rigid primitive acting on a vertex velocity (the k-th of planes, boxes, grippers).
template <class T>
__device__ __forceinline__ V3<T> prim_respond(int k, const SceneDev& sc, const RodInfo& R, V3<T> x, V3<T> v,
                                              V3<T> gp, V3<T> gax, V3<T> vp, V3<T> w, bool& act) {
    V3<T> n;
    T sdf;
    V3<T> vrig = zero3<T>();
    if (k < sc.n_planes) {
        n = mk3(cst<T>(sc.planes[k].x), cst<T>(sc.planes[k].y), cst<T>(sc.planes[k].z));
        sdf = dot(x, n) - sc.planes[k].w;
    } else if (k < sc.n_planes + sc.n_boxes) {
        const int b = k - sc.n_planes;
        sdf = sdf_box(x, f3(sc.box_c[b]), f3(sc.box_h[b]), n);
    } else {
        V3<T> a = gp - sc.grip_hl * gax, bb = gp + sc.grip_hl * gax;
        if (capsule_far(vals(x), vals(a), vals(bb), sc.grip_r + R.radius + kContactReach * R.eps)) {
            act = false;
            return v;
        }
        sdf = sdf_capsule(x, a, bb, sc.grip_r, n);
        vrig = vp + cross(w, x - gp);
    }
    return contact_respond(v, sdf, n, vrig, R.radius, R.eps, sc.mu_rigid, sc.restitution, act);
}

// What the reverse reads of the substep before is copied to shared memory while the present
// one is reversed: each thread's own state rows, and of the projection records (each
// projecting thread its own two edges') the last proj_rows(NV) iterations, the rest as they are
// used up.  Read from memory when needed, the state cost its latency once per substep and the
// records, fetched one iteration ahead, once per iteration: of 4096 cables x 128 vertices the
// reverse takes 8.9 instead of 11.1 ms (16 frames).  Fewer rows where more would leave
// room for fewer CTAs on the SM.
__host__ __device__ constexpr int proj_rows(int NV) { return NV == 64 || NV == 128 ? 10 : 5; }
__device__ __forceinline__ void copy16(float4* dst, const float4* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copies_wait() {   // for all but the last N groups of this thread
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Shared memory of one rod of the reverse kernel: what a neighbour (or another vertex of a
// contact pair) reads, and the frame's gripper data.
template <int NV, bool CONTACT>
struct RevSmem {
    float4 *LD;                 // displacement cotangents, then the force cotangents, then dL/d(edge vectors)
    float4 *F0, *F1, *F2, *F3;  // per edge: its dual frame, replaced by the seeds of the hinge at its end
    float2* GM;                 // [5][NV]: the threads' material sums, each an unevaluated sum of two floats
    float* PA;                  // [24][NV]: the threads' pose terms of the frame: positions (2 x 3),
                                // rotations (2 x 3), actions (2 x 6)
    float4* ST;                 // [6][NV]: X0, V, HG, ED, ET, v1 of the substep reversed next
    float4* PR;                 // [proj_rows][NV]: projection records, iterations in the order of the reverse
    float4* WB;                 // [NV / 2]: weights of the projecting threads' edges
    uint32_t* pairs;
    float *red, *f0, *act;      // reduction scratch, the frame's start pose (24) and actions (12)
    float *sp, *PM;             // per substep of a batch: gripper blocks (64) and pose maps (72)
    double* PC;                 // the carried pose cotangents (12)
    float* GA;                  // the frame's action cotangents carried from the next frame's pose (12)
    static constexpr size_t kHeader = 64 + 24 + 16 + 64 * kPoseBatch + 72 * kPoseBatch + 2 * 12 + 16;
    static constexpr size_t kBytes = 16 * (size_t)((11 + proj_rows(NV)) * NV + NV / 2) + 8 * (size_t)(5 * NV) + 4 * (size_t)(24 * NV) +
                                     (CONTACT ? 4 * (size_t)(kPairsPerVertex * NV) : 0) + 4 * kHeader;
    __device__ explicit RevSmem(float4* b) {
        LD = b;
        F0 = b + NV;
        F1 = b + 2 * NV;
        F2 = b + 3 * NV;
        F3 = b + 4 * NV;
        ST = b + 5 * NV;
        PR = b + 11 * NV;
        WB = PR + proj_rows(NV) * NV;
        GM = reinterpret_cast<float2*>(WB + NV / 2);
        PA = reinterpret_cast<float*>(GM + 5 * NV);
        PC = reinterpret_cast<double*>(PA + 24 * NV);
        red = reinterpret_cast<float*>(PC + 12);
        f0 = red + 64;
        act = f0 + 24;
        sp = act + 16;
        PM = sp + 64 * kPoseBatch;
        GA = PM + 72 * kPoseBatch;
        pairs = reinterpret_cast<uint32_t*>(GA + 16);
    }
};

// row-major 3x3 at o times v
__device__ __forceinline__ V3<float> mul_rm(const float* o, V3<float> v) {
    return f3(o[0] * v.x + o[1] * v.y + o[2] * v.z, o[3] * v.x + o[4] * v.y + o[5] * v.z,
              o[6] * v.x + o[7] * v.y + o[8] * v.z);
}
__device__ __forceinline__ V3<float> mul_rm_t(const float* o, V3<float> v) {
    return f3(o[0] * v.x + o[3] * v.y + o[6] * v.z, o[1] * v.x + o[4] * v.y + o[7] * v.z,
              o[2] * v.x + o[5] * v.y + o[8] * v.z);
}

// Pose cotangents of one substep and gripper (positions and rotations at the substep's start
// and end, rigid velocities) -> the frame-start pose and the frame's actions.  acc: the thread's
// pose terms (RevSmem::PA), stride apart.  Only the threads of held vertices and of vertices
// touching a gripper have any.
__device__ __forceinline__ void add_pose(float* acc, int stride, int m, V3<float> v) {
    acc[m * stride] += v.x;
    acc[(m + 1) * stride] += v.y;
    acc[(m + 2) * stride] += v.z;
}
__device__ __forceinline__ void fold_pose(float* acc, int stride, int q, const float* pm, float c0, float c1, float idt,
                                          V3<float> ps0, V3<float> ph0, V3<float> ps1, V3<float> ph1, V3<float> vp,
                                          V3<float> w) {
    pm += 36 * q;
    add_pose(acc, stride, 3 * q, ps0 + ps1);
    add_pose(acc, stride, 6 + 3 * q, mul_rm_t(pm, ph0) + mul_rm_t(pm + 9, ph1));
    add_pose(acc, stride, 12 + 6 * q, c0 * ps0 + c1 * ps1 + idt * vp);
    add_pose(acc, stride, 15 + 6 * q, mul_rm(pm + 18, ph0) + mul_rm(pm + 27, ph1) + idt * w);
}

struct RevGrip {
    V3<float> lx, lam;
};

// d2r and the material directors of a frame from its tangent, first director and (cos, sin),
// formed where the hinge needs them: as opaque values, or the compiler would carry an edge's own
// 18 numbers across the barrier instead of forming them again (twice the spills).
__device__ __forceinline__ void opaque(dualf& a) { asm volatile("" : "+f"(a.v), "+f"(a.d)); }
__device__ __forceinline__ void material_frame(EdgeF<dualf>& E) {
    opaque(E.t.x);
    opaque(E.t.y);
    opaque(E.t.z);
    opaque(E.d1r.x);
    opaque(E.d1r.y);
    opaque(E.d1r.z);
    opaque(E.c);
    opaque(E.s);
    material_directors(E);
}

// Reverse of an active gripper contact: the cotangents of the vertex position (to add) and of
// the velocity before the contact; the pose cotangents go to acc.  Out of line: few vertices
// touch a gripper, and inlined its registers would be every vertex's.
static __device__ __noinline__ RevGrip gripper_reverse(const BwdParams& P, const RodInfo* Rp, const float* sp,
                                                       const float* pm, float* acc, int stride, int q, float c0, float c1, V3<float> x, V3<float> v,
                                                V3<float> lam) {
    const SceneDev& sc = P.scene;
    const RodInfo& R = *Rp;
    const float* o = sp + 32 * q;
    const V3<float> gp = f3(o[0], o[1], o[2]), gax = f3(o[8], o[11], o[14]), vp = f3(o[24], o[25], o[26]),
                    w = f3(o[27], o[28], o[29]);
    RevGrip r;
    V3<float> lp, lphi, lvp, lw, ntmp;
    if (sdf_capsule(x, gp - sc.grip_hl * gax, gp + sc.grip_hl * gax, sc.grip_r, ntmp) > -sc.grip_r) {
        capsule_contact_rev(x, v, gp, gax, sc.grip_hl, sc.grip_r, vp, w, R.radius, R.eps, sc.mu_rigid, sc.restitution,
                            lam, r.lx, r.lam, lp, lphi, lvp, lw);
    } else {   // the degenerate on-axis contact, by dual numbers, one input direction at a time
        const int k = sc.n_planes + sc.n_boxes + q;
        float lin[18];
#pragma unroll 1
        for (int d = 0; d < 18; ++d) {
            V3<float> e = zf3();
            (d % 3 == 0 ? e.x : d % 3 == 1 ? e.y : e.z) = 1.f;
            const int g = d / 3;
            bool on;
            const V3<dualf> out = prim_respond<dualf>(
                k, sc, R, lift(x, g == 0 ? e : zf3()), lift(v, g == 1 ? e : zf3()), lift(gp, g == 2 ? e : zf3()),
                lift(gax, g == 3 ? cross(e, gax) : zf3()), lift(vp, g == 4 ? e : zf3()), lift(w, g == 5 ? e : zf3()), on);
            lin[d] = dot(ders(out), lam);
        }
        r.lx = f3(lin[0], lin[1], lin[2]);
        r.lam = f3(lin[3], lin[4], lin[5]);
        lp = f3(lin[6], lin[7], lin[8]);
        lphi = f3(lin[9], lin[10], lin[11]);
        lvp = f3(lin[12], lin[13], lin[14]);
        lw = f3(lin[15], lin[16], lin[17]);
    }
    fold_pose(acc, stride, q, pm, c0, c1, 1.f / sc.dt, lp, lphi, zf3(), zf3(), lvp, lw);
    return r;
}

// The k-th rigid primitive (planes, boxes, grippers) acting on a vertex velocity.
__device__ __forceinline__ V3<float> respond_at(int k, const SceneDev& sc, const RodInfo& R, const float* sp, V3<float> x,
                                                V3<float> v, bool& on) {
    const int q = k - sc.n_planes - sc.n_boxes;
    V3<float> gp = zf3(), gax = zf3(), vp = zf3(), w = zf3();
    if (q >= 0) {
        const float* o = sp + 32 * q;
        gp = f3(o[0], o[1], o[2]);
        if (grip_far(x, gp, o)) {
            on = false;
            return v;
        }
        gax = f3(o[8], o[11], o[14]);
        vp = f3(o[24], o[25], o[26]);
        w = f3(o[27], o[28], o[29]);
    }
    return prim_respond<float>(k, sc, R, x, v, gp, gax, vp, w, on);
}

// Reverse of the rigid contact of one vertex: from the cotangent lam of the velocity after it,
// that of the velocity v1 before it; adds the position's to lx.
__device__ __forceinline__ V3<float> rigid_reverse(const BwdParams& P, const RodInfo& R, const RodInfo* Rp, const float* sp,
                                                   const float* pm, float* acc, int stride, float c0, float c1,
                                                   V3<float> x, V3<float> v1, V3<float> lam, V3<float>& lx, bool& touched) {
    const SceneDev& sc = P.scene;
    const int nprim = sc.n_planes + sc.n_boxes + R.ngrip;
    unsigned mask = 0;
    V3<float> v = v1, vb = v1;   // vb: the velocity before the last active primitive
#pragma unroll 1
    for (int k = 0; k < nprim; ++k) {
        bool on;
        const V3<float> nxt = respond_at(k, sc, R, sp, x, v, on);
        if (on) {
            mask |= 1u << k;
            vb = v;
        }
        v = nxt;
    }
    while (mask) {
        const int k = 31 - __clz(mask), q = k - sc.n_planes - sc.n_boxes;
        mask ^= 1u << k;
        if (q >= 0) {
            const RevGrip r = gripper_reverse(P, Rp, sp, pm, acc, stride, q, c0, c1, x, vb, lam);
            lx += r.lx;
            lam = r.lam;
            touched = true;
        } else if (k < sc.n_planes) {   // sdf = n.x - o, constant n
            const V3<float> n = f3(sc.planes[k]);
            V3<float> lv, ln, lvr;
            float lsdf;
            contact_respond_rev(vb, dot(x, n) - sc.planes[k].w, n, zf3(), R.radius, R.eps, sc.mu_rigid, sc.restitution,
                                lam, lv, lsdf, ln, lvr);
            lx += lsdf * n;
            lam = lv;
        } else {
            const int bi = k - sc.n_planes;
            V3<float> lv;
            lx += box_contact_rev(x, vb, f3(sc.box_c[bi]), f3(sc.box_h[bi]), R.radius, R.eps, sc.mu_rigid,
                                  sc.restitution, lam, lv);
            lam = lv;
        }
        if (mask) {   // several at once (rare): the velocity before the one below, again from v1
            const int top = 31 - __clz(mask);
            vb = v1;
            for (int j = 0; j < top; ++j) {
                bool on;
                if ((mask >> j) & 1u) vb = respond_at(j, sc, R, sp, x, vb, on);
            }
        }
    }
    return lam;
}

// Adds v to the unevaluated sum s.x + s.y (Knuth's exact two-term sum): what FP64 addition gave
// these strongly cancelling sums, on the FP32 pipe (an FP64 addition and its conversion take 16
// cycles of the SM each).
__device__ __forceinline__ void add_comp(float2* s, float v) {
    float2 a = *s;
    const float t = __fadd_rn(a.x, v), b = __fsub_rn(t, a.x);
    const float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(t, b)), __fsub_rn(v, b));
    *s = make_float2(t, __fadd_rn(a.y, e));
}

template <bool V>
struct Flag {
    static constexpr bool value = V;
};

// A rod's cotangents as a thread holds them for its own vertex, edge and hinge.
struct Cot {
    V3<float> x, v, d1, t;     // position, velocity, base director, base tangent
    float om, th, k0, k1;      // twist rate, twist angle, rest curvature
};

// The two edges of a projecting thread and their running sums of cotangents.
struct PbdRev {
    bool e0, e1, ring;         // edge 2t, edge 2t + 1 are projected; edge 2t is an odd loop's last (its own colour)
    int i0, i2;                // vertices 2t and the end of edge 2t + 1
    float a0, b0, a1, b1;      // w_a / (w_a + w_b), w_b / (w_a + w_b) of both (RevSmem::WB)
    V3<float> s0, s1;          // sums over the iterations
};

// One projection reversed, from its record q (unit direction t, ratio r = target / length): it
// moved its ends by -+ w lambda t, lambda = (l - target) / (w_a + w_b).  A record that did
// nothing, (0, 0, 0, 1), gives zero.
__device__ __forceinline__ V3<float> project_rev(float4 q, float a, float b, V3<float> la, V3<float> lb) {
    const V3<float> t = f3(q);
    const V3<float> mu = a * la - b * lb;
    return mu - q.w * (mu - dot(mu, t) * t);
}

// Copies of the substep reversed next (RevSmem::ST, PR); base: its records.
template <int NV, bool CONTACT>
__device__ __forceinline__ void fetch_state(const RevSmem<NV, CONTACT>& s, const RodInfo& R, const float4* base, int i) {
    if (i < R.nv) {
        copy16(s.ST + i, base + i);
        copy16(s.ST + NV + i, base + NV + i);
        copy16(s.ST + 2 * NV + i, base + 2 * NV + i);
        copy16(s.ST + 5 * NV + i, base + 5 * NV + i);
    }
    if (i < R.ne) {
        copy16(s.ST + 3 * NV + i, base + 3 * NV + i);
        copy16(s.ST + 4 * NV + i, base + 4 * NV + i);
    }
    copies_commit();
}
// iteration it's records of the edges 2 i and 2 i + 1 into row `row`
template <int NV, bool CONTACT>
__device__ __forceinline__ void fetch_projection(const RevSmem<NV, CONTACT>& s, const RodInfo& R, const float4* base, int it,
                                                 int row, int i) {
    const float4* src = base + (size_t)(7 + it) * NV + 2 * i;
    float4* dst = s.PR + row * NV + 2 * i;
    if (2 * i < R.ne) copy16(dst, src);
    if (2 * i + 1 < R.ne) copy16(dst + 1, src + 1);
}
template <int NV, bool CONTACT>
__device__ __forceinline__ void fetch_projections(const RevSmem<NV, CONTACT>& s, const RodInfo& R, const float4* base,
                                                  int n_iter, int i) {
#pragma unroll 1
    for (int k = 0; k < min(n_iter, proj_rows(NV)); ++k) fetch_projection<NV>(s, R, base, n_iter - 1 - k, k, i);
    copies_commit();
}

// ------------------------------------------------------------------ reverse of one substep
// rec: the substep's records, of which the state and the first projection rows are in s;
// before: the records of the substep reversed next (null: none).  c holds the cotangents of S_{n+1} on entry and of S_n on exit.
// sp, pm: the substep's gripper block and pose maps.  touched: set when the thread adds to its
// pose terms.
// Bound by latency: dependent arithmetic of few warps (registers), barriers and record loads.
// Each thread keeps its vertex's, edge's and hinge's data in registers from phase to phase.
template <int NV, bool CONTACT>
__device__ __forceinline__ void reverse_substep(const BwdParams& P, const RodInfo& R, const RodInfo* Rp, const Own& own,
                                                float4 kin, float eb, float eba, RevSmem<NV, CONTACT>& s,
                                                const Grp<NV>& g, const Rec<NV, true> rec, const float4* before,
                                                float h, float c0, float c1,
                                                int np, const float* sp, const float* pm, Cot& c,
                                                bool& touched) {
    const SceneDev& sc = P.scene;
    const int nv = R.nv, ne = R.ne, i = g.tid;
    const bool closed = R.flags & ROD_CLOSED;
    const float ih = 1.f / h;
    const bool lenc = R.flags & (ROD_INEXT | ROD_SLIMIT);
    const bool project = lenc || (CONTACT && np > 0);
    const bool vtx = i < nv, has_e = i < ne, has_em = vtx && (closed || i > 0);
    const bool strands = R.flags & ROD_STRANDS;
    const bool real = has_e && !(strands && !(eb > 0.f));
    const int ip = (i + 1 == nv) ? 0 : i + 1, im = (i == 0) ? nv - 1 : i - 1;
    const float4* S = rec.base;
    float4 x4 = make_float4(0.f, 0.f, 0.f, 0.f), v4 = x4, xb = x4, hg = x4, ed = x4, et = x4, v1 = x4;
    float tha = 0.f;
    copies_wait<0>();   // the own copies are there
    g.sync();   // so are the other threads'; LD of the substep after this one has been read and the
                // frame's shared data is written
    if (vtx) {
        x4 = s.ST[i];
        v4 = s.ST[NV + i];
        v1 = s.ST[5 * NV + i];
    }
    if (has_e) {
        xb = s.ST[ip];
        ed = s.ST[3 * NV + i];
        et = s.ST[4 * NV + i];
    }
    if (has_em) {
        hg = s.ST[2 * NV + i];
        tha = s.ST[3 * NV + im].w;
    }
    // ---- positions at the substep end, and the velocity rebuilt from the displacement
    const bool held = own.kind >= 2;
    V3<float> ld = held ? zf3() : c.x, dx = zf3(), lp0 = zf3();
    if (CONTACT && np > 0) {   // self-contact friction
        const float4* T0 = rec.csnap(0);   // displacements at the first contact sweep
        const float4 *DF = rec.dfin(), *FR1 = rec.fr1();
        if (vtx) {
            s.F1[i] = f4(c.v, 0.f);
            s.F2[i] = s.F3[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        g.sync();
        for (int p = g.tid; p < np; p += NV) {
            if (!(FR1[p].w > 0.f)) continue;
            const uint32_t pr = s.pairs[p];
            const int a0 = pr & 0xffff, q0 = pr >> 16;
            if (!in_bounds(a0 < nv && q0 < nv, s.red)) continue;
            const int idx[4] = {a0, (a0 + 1 == nv) ? 0 : a0 + 1, q0, (q0 + 1 == nv) ? 0 : q0 + 1};
            const V3<float> o = f3(S[a0]);
            V3<float> Pf[4], Vf[4], lo[4];
            float w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float4 xk = S[idx[k]];
                Pf[k] = (k == 0) ? f3(T0[idx[0]]) : (f3(xk) - o) + f3(T0[idx[k]]);
                Vf[k] = ih * f3(DF[idx[k]]);
                w[k] = xk.w;
                lo[k] = f3(s.F1[idx[k]]);
            }
            V3<float> pb[4], vb[4];
            if (fric_pair_vjp(Pf, Vf, w, 2.f * R.radius, sc.mu_self, h, lo, pb, vb))
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    atomic_add3(&s.F2[idx[k]], pb[k]);
                    atomic_add3(&s.F3[idx[k]], vb[k]);
                }
        }
        g.sync();
        if (vtx) {
            lp0 = f3(s.F2[i]);
            c.v += f3(s.F3[i]);
        }
    }
    ld += ih * c.v;
    // ---- projections in reverse
    if (project) {
        constexpr int PT = pbd_threads(NV);
        const int ncol = lenc ? ((closed && (ne & 1)) ? 3 : 2) : 0;
        const bool proj = lenc && i < PT;
        PbdRev b{};
        int row = 0;   // of PR: the iteration's
        if (proj) {
            const int j = 2 * i;
            b.e0 = j < ne;
            b.e1 = j + 1 < ne;
            b.ring = ncol == 3 && j == ne - 1;
            b.i0 = min(j, nv - 1);
            b.i2 = j + 2 >= nv ? 0 : j + 2;
            const float4 w = b.e0 ? s.WB[i] : make_float4(0.f, 0.f, 0.f, 0.f);
            b.a0 = w.x;
            b.b0 = w.y;
            b.a1 = w.z;
            b.b1 = w.w;
            b.s0 = b.s1 = zf3();
        }
        if (vtx) s.LD[i] = f4(ld, 0.f);
        g.sync();
        for (int it = sc.n_iter - 1; it >= 0; --it) {
            if (CONTACT && np > 0) {
                const float4* Dc = rec.csnap(it);   // displacements before the contact sweep
                if (vtx) s.F3[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                g.sync();
                for (int p = g.tid; p < np; p += NV) {
                    const uint32_t pr = s.pairs[p];
                    const int a0 = pr & 0xffff, c0_ = pr >> 16;
                    if (!in_bounds(a0 < nv && c0_ < nv, s.red)) continue;
                    const int idx[4] = {a0, (a0 + 1 == nv) ? 0 : a0 + 1, c0_, (c0_ + 1 == nv) ? 0 : c0_ + 1};
                    const V3<float> o = f3(S[a0]);
                    V3<float> Pf[4], lo[4];
                    float w[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float4 xk = S[idx[k]];
                        Pf[k] = (k == 0) ? f3(Dc[idx[0]]) : (f3(xk) - o) + f3(Dc[idx[k]]);
                        w[k] = xk.w;
                        lo[k] = f3(s.LD[idx[k]]);
                    }
                    V3<float> pb[4];
                    if (pair_correction_vjp(Pf, w, 2.f * R.radius, lo, pb))
#pragma unroll
                        for (int k = 0; k < 4; ++k) atomic_add3(&s.F3[idx[k]], pb[k]);
                }
                g.sync();
                if (vtx) {
                    V3<float> t = f3(s.F3[i]);
                    if (it == 0) t += lp0;
                    s.LD[i] = f4(f3(s.LD[i]) + t, 0.f);
                    dx += t;
                }
                g.sync();
            }
            if (proj) {
                if (sc.n_iter - 1 - it >= proj_rows(NV)) copies_wait<proj_rows(NV) - 1>();
                const float4 none = make_float4(0.f, 0.f, 0.f, 1.f), r0 = b.e0 ? s.PR[row * NV + 2 * i] : none,
                             r1 = b.e1 ? s.PR[row * NV + 2 * i + 1] : none;
                if (ncol == 3) {
                    if (b.ring) {
                        const V3<float> la = f3(s.LD[b.i0]), lb = f3(s.LD[0]);
                        const V3<float> le = project_rev(r0, b.a0, b.b0, la, lb);
                        s.LD[b.i0] = f4(la - le, 0.f);
                        s.LD[0] = f4(lb + le, 0.f);
                        b.s0 += le;
                    }
                    pbd_sync<NV>(g.bar);
                }
                // vertex 2t + 1 belongs to this thread's two edges alone
                V3<float> lm = b.e0 && !b.ring ? f3(s.LD[2 * i + 1]) : zf3();
                if (b.e1) {
                    const V3<float> lb = f3(s.LD[b.i2]);
                    const V3<float> le = project_rev(r1, b.a1, b.b1, lm, lb);
                    lm = lm - le;
                    s.LD[b.i2] = f4(lb + le, 0.f);
                    b.s1 += le;
                }
                pbd_sync<NV>(g.bar);
                if (b.e0 && !b.ring) {
                    const V3<float> la = f3(s.LD[b.i0]);
                    const V3<float> le = project_rev(r0, b.a0, b.b0, la, lm);
                    s.LD[b.i0] = f4(la - le, 0.f);
                    s.LD[2 * i + 1] = f4(lm + le, 0.f);
                    b.s0 += le;
                }
                if (sc.n_iter > proj_rows(NV)) {   // the row just used up takes the iteration proj_rows further on
                    if (it >= proj_rows(NV)) fetch_projection<NV>(s, R, S, it - proj_rows(NV), row, i);
                    copies_commit();
                }
                row = row + 1 == proj_rows(NV) ? 0 : row + 1;
                pbd_sync<NV>(g.bar);
            }
            if (CONTACT && np > 0) g.sync();
        }
        if (proj) {   // F0: each edge's summed cotangent
            if (b.e0) s.F0[2 * i] = f4(b.s0, 0.f);
            if (b.e1) s.F0[2 * i + 1] = f4(b.s1, 0.f);
            if (before) fetch_projections<NV>(s, R, before, sc.n_iter, i);
        }
        g.sync();
        if (vtx) {
            ld = f3(s.LD[i]);
            if (lenc) {
                if (has_e) dx -= f3(s.F0[i]);
                if (has_em) dx += f3(s.F0[im]);
            }
        }
    }
    // ---- vertex phase (rigid contact, symplectic Euler, gravity, damping, twist rate)
    float4 lg = make_float4(0.f, 0.f, 0.f, 0.f);
    float m_cd = 0.f;
    if (vtx) {
        V3<float> lx = held ? dx : c.x + dx, lv = zf3();
        if (own.kind == 0) {
            V3<float> lam = h * ld;
            lam = rigid_reverse(P, R, Rp, sp, pm, s.PA + i, NV, c0, c1, f3(x4), f3(v1), lam, lx, touched);
            // v1 = v + h (-w g + gravity - c_d v)
            lv = (1.f - h * R.cd) * lam;
            const V3<float> l = (-h * x4.w) * lam;
            lg = f4(l, 0.f);
            m_cd = -h * dot(f3(v4), lam);
        } else if (held && in_bounds(own.kind - 2 < R.ngrip, s.red)) {
            // x = target and d = target - x0, the target moving with the gripper's end pose
            const int q = own.kind - 2;
            const V3<float> y1 = mul_rm(sp + 32 * q + 15, f3(kin)), l = c.x + ld;
            fold_pose(s.PA + i, NV, q, pm, c0, c1, 1.f / sc.dt, zf3(), zf3(), l, cross(y1, l), zf3(), zf3());
            touched = true;
            lx -= ld;
        }
        c.x = lx;
        c.v = lv;
        if (has_e) {
            const float lw1 = c.om + h * c.th;     // d theta_{n+1} / d omega_1 = h
            c.om = (1.f - h * R.cd) * lw1;
            lg.w = -h * own.invI * lw1;
            m_cd -= h * v4.w * lw1;
        } else {
            c.om = 0.f;
        }
        s.LD[i] = lg;
    }
    g.sync();
    if (before) fetch_state<NV>(s, R, before, i);   // everyone has read this substep's
    // ---- the own edge's frame as dual numbers in the direction of the force cotangents, the
    // reverse of its stretching
    EdgeF<dualf> E;
    V3<float> tot = zf3();
    float m_K = 0.f;
    if (real) {
        const float4 lgb = s.LD[ip];
        edge_forward(E, lift(f3(x4), f3(lg)), lift(f3(xb), f3(lgb)), lift(f3(et)), lift(f3(ed)), mkd(ed.w, lg.w));
        s.F0[i] = make_float4(E.t.x.v, E.t.y.v, E.t.z.v, E.c.v);
        s.F1[i] = make_float4(E.t.x.d, E.t.y.d, E.t.z.d, E.c.d);
        s.F2[i] = make_float4(E.d1r.x.v, E.d1r.y.v, E.d1r.z.v, E.s.v);
        s.F3[i] = make_float4(E.d1r.x.d, E.d1r.y.d, E.d1r.z.d, E.s.d);
        if (R.kA > 0.f) {
            const V3<float> les = f3(lgb) - f3(lg), t = vals(E.t);
            const float tl = dot(t, les);
            const float st = edge_strain(f3(xb) - f3(x4), eb);
            tot = R.kA * ((tl / eb) * t + st / E.ell.v * (les - tl * t));
            m_K = st * tl;
        }
    }
    const float lga_w = has_em ? s.LD[im].w : 0.f;   // the previous edge's twist-angle direction
    g.sync();
    // ---- the own hinge: force second order, plasticity and its first-order reverse.  Seeds for
    // the own edge are kept, those for the previous edge replace its frame (read here alone).
    V3<dualf> gt = zero3<dualf>(), gr = zero3<dualf>();
    float gth = 0.f, m_E = 0.f, m_G = 0.f, m_sy = 0.f;
    if (has_em) {
        V3<dualf> gta = zero3<dualf>(), gra = zero3<dualf>();
        float gtha = 0.f;
        auto hinge = [&](auto with_twist) {
            constexpr bool twist = decltype(with_twist)::value;
            const float lbar = 0.5f * (eba + eb), il = 1.f / lbar;
            HingeF<dualf> H;
            {
                const float4 a = s.F0[im], d = s.F1[im], e = s.F2[im], f = s.F3[im];
                H.a.t = mk3(mkd(a.x, d.x), mkd(a.y, d.y), mkd(a.z, d.z));
                H.a.d1r = mk3(mkd(e.x, f.x), mkd(e.y, f.y), mkd(e.z, f.z));
                H.a.c = mkd(a.w, d.w);
                H.a.s = mkd(e.w, f.w);
            }
            H.b = E;
            material_frame(H.a);
            material_frame(H.b);
            hinge_bend_forward(H);
            if (twist) hinge_twist_forward(H, mkd(tha, lga_w), mkd(ed.w, lg.w), mkd(hg.w));
            const float hk0 = H.k0.v, hk1 = H.k1.v;   // the hinge's material curvature (for plasticity)
            float kb0 = hg.x, kb1 = hg.y;
            const bool yielded = (R.flags & ROD_PLASTIC) && plastic_update(hk0, hk1, kb0, kb1, R.sy * lbar, R.rc);
            const dualf e0d = H.k0 - kb0, e1d = H.k1 - kb1, emd = twist ? H.m - hg.z : mkd(0.f);
            dualf gk0 = (R.Bm * il) * e0d, gk1 = (R.Bm * il) * e1d;
            const dualf gmt = (R.beta * il) * emd;
            m_E = il * (e0d.v * e0d.d + e1d.v * e1d.d);
            m_G = il * emd.v * emd.d;
            // rest curvature: cotangent of the one used (-d gk / d .) plus the carried one
            float lk0 = c.k0 - gk0.d, lk1 = c.k1 - gk1.d;
            if (yielded) {
                const float el0 = hk0 - hg.x, el1 = hk1 - hg.y;
                const float n = sqrtf(el0 * el0 + el1 * el1), thr = R.sy * lbar;
                const float gg = R.rc * (n - thr) / n;
                const float kk = R.rc * thr / (n * n * n) * (el0 * lk0 + el1 * lk1);
                const float le0 = gg * lk0 + kk * el0, le1 = gg * lk1 + kk * el1;     // cotangent of kappa_el
                m_sy = -R.rc * lbar * (el0 * lk0 + el1 * lk1) / n;
                // The first-order reverse of kappa from seeds (le0, le1) is needed too.  The hinge
                // reverse is linear in its seeds, so adding them to the derivative part of the
                // dual seeds makes the reverse below return J^T le on top of the Hessian term.
                gk0.d += le0;
                gk1.d += le1;
                lk0 -= le0;
                lk1 -= le1;
            }
            dualf ga_, gb_;
            hinge_core_reverse(H, gk0, gk1, gmt, mkd(0.f), gta, gra, gt, gr, ga_, gb_, twist);
            gtha = ga_.d;
            gth = gb_.d;
            c.k0 = lk0;
            c.k1 = lk1;
        };
        // Without torsional stiffness, and with no sensitivity to it asked for, the twist has no
        // cotangent: 4096 ropes x 128, 16 frames, 5.1 instead of 6.0 ms.  Two whole versions, since a
        // branch around the twist's two parts cost the cables 7 %.
        if (has_e && !(strands && !(eba > 0.f && eb > 0.f))) {
            if (R.beta != 0.f || P.gmat)
                hinge(Flag<true>{});
            else
                hinge(Flag<false>{});
        }
        s.F0[im] = make_float4(gta.x.v, gta.y.v, gta.z.v, gra.x.v);
        s.F1[im] = make_float4(gta.x.d, gta.y.d, gta.z.d, gra.x.d);
        s.F2[im] = make_float4(gra.y.v, gra.z.v, gra.y.d, gra.z.d);
        s.F3[im].x = gtha;
    }
    g.sync();
    // ---- the reverse through the own edge's frame on the sum of its hinges' seeds; the
    // cotangents of the frame it hands on (new base tangent and director) join the derivative
    // parts (the reverse is linear in its seeds, as above)
    if (has_e) {
        if (real) {
            const float4 a = s.F0[i], d = s.F1[i], e = s.F2[i];
            gt += mk3(mkd(a.x, d.x + c.t.x), mkd(a.y, d.y + c.t.y), mkd(a.z, d.z + c.t.z));
            gr += mk3(mkd(a.w, d.w + c.d1.x), mkd(e.x, e.z + c.d1.y), mkd(e.y, e.w + c.d1.z));
            c.th += gth + s.F3[i].x;
            V3<dualf> gtb, gdb;
            tot += ders(edge_reverse<dualf, true>(E, lift(f3(et)), lift(f3(ed)), gt, gr, mkd(0.f), &gtb, &gdb));
            c.t = ders(gtb);
            c.d1 = ders(gdb);
        }
        s.LD[i] = f4(tot, 0.f);
    }
    if (P.gmat && vtx) {
        add_comp(s.GM + i, m_K);
        add_comp(s.GM + NV + i, m_E);
        add_comp(s.GM + 2 * NV + i, m_G);
        add_comp(s.GM + 3 * NV + i, m_sy);
        add_comp(s.GM + 4 * NV + i, m_cd);
    }
    g.sync();
    if (vtx) {
        if (has_e) c.x -= tot;                  // edge i starts here
        if (has_em) c.x += f3(s.LD[im]);        // edge i-1 ends here
    }
}

// CTAs per SM the reverse kernel is compiled for.  Up to 128 vertices 384 threads per SM (168
// registers): with 512 (128 registers) 120 registers spill and 4096 ropes x 128 take 12.1 instead
// of 11.6 ms.  Above, two CTAs: with one (255 registers, no spills) 1024 bands x 200 in contact
// take 5.8 instead of 4.8 ms.
__host__ __device__ constexpr int rev_min_ctas(int NV) { return NV <= 128 ? 384 / NV : 2; }
static_assert(rev_min_ctas(256) * (RevSmem<256, true>::kBytes + 1024) <= 228 * 1024 &&
                  rev_min_ctas(128) * (RevSmem<128, true>::kBytes + 1024) <= 228 * 1024,
              "as many rods as registers allow fit the SM's shared memory (1 KB of it reserved per CTA)");

// ------------------------------------------------------------------ the recompute kernel
// Persistent, forward-like (a group of threads per rod, state in shared memory).  RECORD false:
// from the checkpoint of the segment that holds frame fa, store the start state of each of the
// segment's frames (L2).  RECORD true: from the start state of frame fa (a checkpoint, or the
// segment's stored state), run frames fa .. fb-1 storing every substep's records (R3).
template <int NV, bool CONTACT, bool RECORD>
__global__ void __launch_bounds__(kFwdMaxThreads) rec_kernel(BwdParams P) {
    constexpr int TPR = threads_per_rod(NV);
    extern __shared__ float4 dyn_smem[];
    const int slot = threadIdx.x / TPR;
    Smem<NV, CONTACT> s(dyn_smem + slot * (rod_smem_bytes(NV, CONTACT) / 16));
    const Grp<TPR> g{(int)(threadIdx.x % TPR), 1 + slot, s.red};
    const SceneDev& sc = P.scene;
    const int n_iter = sc.n_iter;
    const size_t FR = frame_rec(NV, n_iter, P.nsub_max);
    if (CONTACT)   // the contact accumulators start at zero; every sweep leaves them at zero
        for (int i = g.tid; i < NV; i += TPR) s.acc[i] = make_int4(0, 0, 0, 0);
    for (;;) {
        const int k = grp_bcast0<TPR>(g.tid == 0 ? atomicAdd(P.counter, 1) : 0, g);
        if (k >= P.n_items) break;
        const int rod = P.order[P.item0 + k];
        bounds_begin<TPR>(g);
        if (!in_bounds(rod >= 0 && rod < P.B && P.rods[rod].nv <= NV, s.red)) {
            g.sync();
            bounds_end<TPR>(g, P.status, (rod >= 0 && rod < P.B) ? rod : 0);
            continue;
        }
        // with self-contact read from memory where used: a register copy spills the
        // contact variant of the kernel (its broad phase and sweeps) past the launch bound
        RodRef<CONTACT> R = P.rods[rod];
        const int nsub = P.force_nsub > 0 ? P.force_nsub : R.nsub;
        const float h = sc.dt / (float)nsub;
        const int seg = P.fa / P.ck_every, f0 = seg * P.ck_every;
        float4* L2 = P.L2 + (size_t)k * P.l2_rod;
        if (!RECORD || P.fa == f0) {   // the segment's checkpoint
            const long long oV = seg * P.ck_strideV, oE = seg * P.ck_strideE;
            for (int i = g.tid; i < R.nv; i += TPR) {
                const float4 x = P.ck.X[oV + R.v0 + i];
                s.X0[i] = x;
                s.V[i] = P.ck.Vl[oV + R.v0 + i];
                s.HG[i] = P.ck.HG[oV + R.v0 + i];
            }
            for (int j = g.tid; j < R.ne; j += TPR) {
                s.ED[j] = P.ck.ED[oE + R.e0 + j];
                s.ET[j] = P.ck.ET[oE + R.e0 + j];
            }
            if (g.tid < 24) s.fp[g.tid] = P.ck.GP[seg * P.ck_strideB + 24LL * rod + g.tid];
        } else {                            // the stored start state of frame fa
            const float4* e = L2 + (size_t)(P.fa - f0) * seg_state(NV);
            for (int i = g.tid; i < R.nv; i += TPR) {
                const float4 x = e[i];
                s.X0[i] = x;
                s.V[i] = e[NV + i];
                s.HG[i] = e[2 * NV + i];
            }
            for (int j = g.tid; j < R.ne; j += TPR) {
                s.ED[j] = e[3 * NV + j];
                s.ET[j] = e[4 * NV + j];
            }
            if (g.tid < 24) s.fp[g.tid] = reinterpret_cast<const float*>(e + 5 * NV)[g.tid];
        }
        const Own own = own_of(P.KIN, P.ES, R, g.tid);
        g.sync();
        bool ovf = false;
        if constexpr (!RECORD) {
            const int f1 = min(f0 + P.ck_every, P.frames);
            for (int f = f0; f < f1; ++f) {
                float4* e = L2 + (size_t)(f - f0) * seg_state(NV);
                save_state<NV, CONTACT, TPR>(e, R, g, s);
                if (g.tid < 24) reinterpret_cast<float*>(e + 5 * NV)[g.tid] = s.fp[g.tid];
                if (f + 1 == f1) break;   // the segment's last frame only needs its start state
                if (g.tid < 12) s.act[g.tid] = P.actions[((size_t)f * P.B + rod) * 12 + g.tid];
                g.sync();
                run_frame<NV, CONTACT, TPR>(sc, P.KIN, R, own, s, g, nsub, h, ovf,
                                            [](int) { return Rec<NV, false>{nullptr, 0}; });
            }
        } else {
            float4* R3 = P.R3 + (size_t)k * P.r3_rod;
            for (int f = P.fa; f < P.fb; ++f) {
                float4* fb = R3 + (size_t)(f - P.fa) * FR;
                if (g.tid < 24) reinterpret_cast<float*>(fb)[g.tid] = s.fp[g.tid];
                if (g.tid < 12) s.act[g.tid] = P.actions[((size_t)f * P.B + rod) * 12 + g.tid];
                g.sync();
                const int np = run_frame<NV, CONTACT, TPR>(sc, P.KIN, R, own, s, g, nsub, h, ovf, [&](int sb) {
                    return record_substep<NV, CONTACT, TPR>(fb, sb, n_iter, R, g, s);
                });
                if (CONTACT) record_pairs<NV, CONTACT, TPR>(fb, np, g, s);
            }
        }
        g.sync();
        bounds_end<TPR>(g, P.status, rod);
    }
}

// ------------------------------------------------------------------ the reverse kernel
// Persistent, one CTA of one thread per vertex for each rod: for frames fb-1 .. fa, last first,
// and each frame's substeps, last first, applies the reverse of every phase (reverse_substep)
// from the substep's records.  The cotangents of the rod's state at frame fb come from
// dL/d(final state) on the first chunk (fb = F), else from the previous chunk's launch (CS);
// those at fa go to CS, or to the outputs on the last chunk (fa = 0).
template <int NV, bool CONTACT>
__global__ void __launch_bounds__(NV, rev_min_ctas(NV)) rev_kernel(BwdParams P) {
    constexpr int TPR = NV;
    extern __shared__ float4 dyn_smem[];
    RevSmem<NV, CONTACT> s(dyn_smem);
    const Grp<TPR> g{(int)threadIdx.x, 1, s.red};
    const int i = g.tid;
    const SceneDev& sc = P.scene;
    const int n_iter = sc.n_iter;
    const size_t SR = sub_rec(NV, n_iter), FR = frame_rec(NV, n_iter, P.nsub_max);
    for (;;) {
        const int k = grp_bcast0<TPR>(i == 0 ? atomicAdd(P.counter, 1) : 0, g);
        if (k >= P.n_items) break;
        const int rod = P.order[P.item0 + k];
        bounds_begin<TPR>(g);
        if (!in_bounds(rod >= 0 && rod < P.B && P.rods[rod].nv <= NV, s.red)) {
            g.sync();
            bounds_end<TPR>(g, P.status, (rod >= 0 && rod < P.B) ? rod : 0);
            continue;
        }
        const RodInfo* Rp = P.rods + rod;
        const RodInfo R = *Rp;
        const int nsub = P.force_nsub > 0 ? P.force_nsub : R.nsub;
        const float h = sc.dt / (float)nsub;
        const bool vtx = i < R.nv, has_e = i < R.ne, closed = R.flags & ROD_CLOSED;
        const Own own = own_of(P.KIN, P.ES, R, i);
        const float4 kin = own.kind >= 2 ? P.KIN[R.v0 + i] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float eb = has_e ? P.ES[R.e0 + i].x : 0.f;   // rest lengths of the own and the previous edge
        const float eba = vtx && (closed || i > 0) ? P.ES[R.e0 + (i == 0 ? R.ne - 1 : i - 1)].x : 0.f;
        float4* CS = P.CS + (size_t)k * P.cs_rod;
        Cot c{zf3(), zf3(), zf3(), zf3(), 0.f, 0.f, 0.f, 0.f};
        if (P.first_chunk) {
            if (vtx) {
                const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
                const float4 dx = P.dLdx ? P.dLdx[R.v0 + i] : z, dv = P.dLdv ? P.dLdv[R.v0 + i] : z;
                c.x = f3(dx);
                c.v = f3(dv);
                c.om = !closed && i == R.nv - 1 ? 0.f : dv.w;
            }
            if (has_e && P.dLdth) c.th = P.dLdth[R.e0 + i];
        } else {
            if (vtx) {
                const float4 lv = CS[NV + i], lk = CS[4 * NV + i];
                c.x = f3(CS[i]);
                c.v = f3(lv);
                c.om = lv.w;
                c.k0 = lk.x;
                c.k1 = lk.y;
            }
            if (has_e) {
                const float4 le = CS[2 * NV + i];
                c.d1 = f3(le);
                c.th = le.w;
                c.t = f3(CS[3 * NV + i]);
            }
        }
        // carried sums: the pose cotangents of frame fb's start, positions (2 x 3) then rotations
        if (i < 12) s.PC[i] = P.first_chunk ? 0.0 : reinterpret_cast<const double*>(CS + 4 * NV)[2 * i + 1];
        for (int m = 0; m < 5; ++m) s.GM[m * NV + i] = make_float2(0.f, 0.f);
        bool touched = true;
        {   // the copies of the last substep, and the projecting threads' weights (the inverse masses
            // are the same in every record)
            const float4* last = P.R3 + (size_t)k * P.r3_rod + (size_t)(P.fb - 1 - P.fa) * FR + kFrameHead + NV +
                                 (size_t)(nsub - 1) * SR;
            g.sync();   // the rod before has been reversed
            fetch_state<NV>(s, R, last, i);
            if ((R.flags & (ROD_INEXT | ROD_SLIMIT)) && i < pbd_threads(NV)) {
                fetch_projections<NV>(s, R, last, n_iter, i);
                const int j = 2 * i;
                const float w0 = j < R.ne ? last[j].w : 0.f, w1 = j < R.ne ? last[j + 1 == R.nv ? 0 : j + 1].w : 0.f,
                            w2 = j + 1 < R.ne ? last[j + 2 >= R.nv ? 0 : j + 2].w : 0.f;
                if (j < NV)
                    s.WB[i] = make_float4(w0 + w1 > 0.f ? w0 / (w0 + w1) : 0.f, w0 + w1 > 0.f ? w1 / (w0 + w1) : 0.f,
                                          w1 + w2 > 0.f ? w1 / (w1 + w2) : 0.f, w1 + w2 > 0.f ? w2 / (w1 + w2) : 0.f);
            }
        }
        for (int f = P.fb - 1; f >= P.fa; --f) {
            const float4* fb = P.R3 + (size_t)k * P.r3_rod + (size_t)(f - P.fa) * FR;
            g.sync();   // the previous frame's reverse has finished reading the frame's shared data
            if (i < 12) s.act[i] = P.actions[((size_t)f * P.B + rod) * 12 + i];
            if (i < 24) s.f0[i] = reinterpret_cast<const float*>(fb)[i];
            int np = 0;
            if (CONTACT) {
                np = reinterpret_cast<const int*>(fb)[24];
                if (!in_bounds(np >= 0 && np <= R.pair_cap, s.red)) np = 0;
                const uint32_t* pl = reinterpret_cast<const uint32_t*>(fb + kFrameHead);
                for (int p = i; p < np; p += TPR) s.pairs[p] = pl[p];
            }
            if (touched) {
#pragma unroll 1
                for (int m = 0; m < 24; ++m) s.PA[m * NV + i] = 0.f;
                touched = false;
            }
            g.sync();
            // the pose cotangent of frame f+1's start through the frame's motion: into its actions
            // and its own start pose
            if (i < R.ngrip) {
                const V3<float> dphi = f3(s.act[6 * i + 3], s.act[6 * i + 4], s.act[6 * i + 5]);
                double* lr = s.PC + 6 + 3 * i;
                const V3<float> l = f3((float)lr[0], (float)lr[1], (float)lr[2]);
                const V3<float> jr = jl_t(dphi, l), nr = mulT(expmap(dphi), l);
#pragma unroll
                for (int m = 0; m < 3; ++m) s.GA[6 * i + m] = (float)s.PC[3 * i + m];
                s.GA[6 * i + 3] = jr.x;
                s.GA[6 * i + 4] = jr.y;
                s.GA[6 * i + 5] = jr.z;
                lr[0] = nr.x;
                lr[1] = nr.y;
                lr[2] = nr.z;
            }
#pragma unroll 1
            for (int sb = nsub - 1; sb >= 0; --sb) {
                const int slot = sb % kPoseBatch;
                if (slot == kPoseBatch - 1 || sb == nsub - 1) {
                    // gripper blocks and pose maps of this and the earlier substeps of the batch,
                    // one per thread, side by side (read after the substep's first barrier)
                    if (sb != nsub - 1) g.sync();
                    for (int m = i; m < 10 * (slot + 1); m += TPR) {
                        const int u = m / 10, w = m % 10, sk = sb - slot + u;
                        const float k0 = (float)sk / (float)nsub, k1 = (float)(sk + 1) / (float)nsub;
                        if (w < 2) {
                            if (w < R.ngrip)
                                substep_pose(sc, R, s.f0, s.act, w, k0, k1, sk == 0, 1.f / sc.dt, s.sp + 64 * u);
                        } else if (w - 2 < 4 * R.ngrip) {
                            pose_rev_mat(s.act, w - 2, k0, k1, s.PM + 72 * u);
                        }
                    }
                }
                const Rec<NV, true> rec{const_cast<float4*>(fb) + kFrameHead + NV + (size_t)sb * SR, n_iter};
                const float4* before = sb > 0     ? rec.base - SR
                                       : f > P.fa ? fb - FR + kFrameHead + NV + (size_t)(nsub - 1) * SR
                                                  : nullptr;
                reverse_substep<NV, CONTACT>(P, R, Rp, own, kin, eb, eba, s, g, rec, before, h, (float)sb / (float)nsub,
                                             (float)(sb + 1) / (float)nsub, np, s.sp + 64 * slot, s.PM + 72 * slot, c,
                                             touched);
            }
            // the frame's pose terms: one thread per term adds those of the threads that have any, in
            // order (a tree of FP64 shuffles over every term took a third of the rollout's reverse)
            unsigned* hit = reinterpret_cast<unsigned*>(s.red);
            const unsigned warp_hit = __ballot_sync(0xffffffffu, touched);
            if ((i & 31) == 0) hit[i >> 5] = warp_hit;
            g.sync();
            if (i < 24) {
                double v = 0.0;
                for (int w = 0; w < TPR / 32; ++w)
                    for (unsigned m = hit[w]; m; m &= m - 1) v += (double)s.PA[i * NV + 32 * w + __ffs(m) - 1];
                if (i < 12) {
                    if (i % 6 < 3 * R.ngrip) s.PC[i] += v;
                } else if (P.gact) {
                    const int m = i - 12;
                    P.gact[((size_t)f * P.B + rod) * 12 + m] = m < 6 * R.ngrip ? (float)((double)s.GA[m] + v) : 0.f;
                }
            }
        }
        g.sync();   // the last frame's pose terms have been added
        double gm[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
        if (P.gmat)
#pragma unroll 1
            for (int m = 0; m < 5; ++m) {
                const float2 a = s.GM[m * NV + i];
                gm[m] = grp_sum<TPR>((double)a.x + (double)a.y, g);
                if (!P.first_chunk) gm[m] += reinterpret_cast<const double*>(CS + 5 * NV)[m];
            }
        g.sync();
        const float4 lx = f4(c.x, 0.f), lv = f4(c.v, c.om);
        if (P.last_chunk) {   // outputs: the cotangents of the initial state and the material
            if (vtx) {
                if (P.gx0) P.gx0[R.v0 + i] = lx;
                if (P.gv0) P.gv0[R.v0 + i] = lv;
            }
            if (has_e) {
                if (P.gth0) P.gth0[R.e0 + i] = c.th;
                P.gtb0[R.e0 + i] = f4(c.t, 0.f);
                P.gd1b0[R.e0 + i] = f4(c.d1, 0.f);
            }
            if (i == 0 && P.gmat) {
                const double r = R.radius, A = 3.14159265358979323846 * r * r, r2 = r * r;
                P.gmat[5 * rod + 0] = R.kA > 0.f ? (float)(gm[0] * A) : 0.f;   // K_stretch
                P.gmat[5 * rod + 1] = (float)(gm[1] * A * r2 / 4.0);            // E_bend
                P.gmat[5 * rod + 2] = (float)(gm[2] * A * r2 / 2.0);            // G_twist
                P.gmat[5 * rod + 3] = (float)gm[3];                             // yield curvature
                P.gmat[5 * rod + 4] = (float)gm[4];                             // damping
            }
        } else {   // carry to the next chunk: cotangents, material and pose sums
            if (vtx) {
                CS[i] = lx;
                CS[NV + i] = lv;
                reinterpret_cast<float2*>(CS + 4 * NV)[2 * i] = make_float2(c.k0, c.k1);
            }
            if (has_e) {
                CS[2 * NV + i] = f4(c.d1, c.th);
                CS[3 * NV + i] = f4(c.t, 0.f);
            }
            if (i == 0 && P.gmat) {
                double* d = reinterpret_cast<double*>(CS + 5 * NV);
#pragma unroll
                for (int m = 0; m < 5; ++m) d[m] = gm[m];
            }
            if (i < 12) reinterpret_cast<double*>(CS + 4 * NV)[2 * i + 1] = s.PC[i];
        }
        g.sync();
        bounds_end<TPR>(g, P.status, rod);
    }
}

// ------------------------------------------------------------------ launch helpers
template <int NV, bool C>
static int rev_occ_t(int rpc) {   // one rod per CTA
    if (rpc != 1) return 0;
    const size_t smem = RevSmem<NV, C>::kBytes;
    auto k = rev_kernel<NV, C>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, NV, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}
template <int NV, bool C>
static cudaError_t launch_rev_t(const BwdParams& P, int grid, int, cudaStream_t st) {
    const size_t smem = RevSmem<NV, C>::kBytes;
    auto k = rev_kernel<NV, C>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<grid, NV, smem, st>>>(P);
    return cudaGetLastError();
}
template <int NV, bool C>
static int rec_occ_t(int rpc) {
    if (rpc < 1 || rpc * threads_per_rod(NV) > kFwdMaxThreads) return 0;
    size_t smem = rod_smem_bytes(NV, C) * rpc;
    auto k = rec_kernel<NV, C, true>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, threads_per_rod(NV) * rpc, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}
template <int NV, bool C>
static cudaError_t launch_rec_t(const BwdParams& P, int grid, int rpc, cudaStream_t st) {
    size_t smem = rod_smem_bytes(NV, C) * rpc;
    auto k = P.mode ? rec_kernel<NV, C, true> : rec_kernel<NV, C, false>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<grid, threads_per_rod(NV) * rpc, smem, st>>>(P);
    return cudaGetLastError();
}

}  // namespace dlo
