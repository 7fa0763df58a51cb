// dlo_adjoint.cu -- host side of the hand-written adjoint with gradient checkpointing, and the
// FP64 adjoint of the initial reference frames.
//
// DLO-Lab (Sec. 3.3) differentiates whole trajectories by caching one state per segment and,
// for each segment in reverse, re-running the forward simulation before back-propagating.
// Here the checkpoints live in HBM (written by the forward kernel every K frames).  The
// rollout is reversed in chunks of C frames, last first; per chunk, rec_kernel re-runs the
// chunk's frames from their start state storing every substep's records, then rev_kernel
// reverses them (dlo_bwd_kernel.cuh).  C is a multiple of K when C >= K, so that every chunk
// starts at a checkpoint; otherwise the frame-start states of each segment are stored first.
// When one chunk holds the whole rollout and an earlier call left a workspace with room for it, the
// forward stores the records there and rec_kernel does not run.
#include <algorithm>
#include <cstring>
#include <vector>

#include "dlo_runtime.h"
#include "dlo_kernels.h"
#include "dlo_frames.cuh"

namespace dlo {

// ------------------------------------------------------------------ initial frames adjoint
__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// reverse of u = adapt(w, t), the unit projection of w normal to t: returns lambda_w, adds lambda_t
__device__ __forceinline__ D3 adapt_rev(D3 w, D3 t, D3 lu, D3& lt) {
    D3 dd = w - dot(w, t) * t;
    double n = sqrt(dot(dd, dd));
    D3 u = dd / n;
    D3 ldd = (lu - dot(lu, u) * u) / n;
    lt += -dot(w, t) * ldd - dot(ldd, t) * w;
    return ldd - dot(ldd, t) * t;
}
// reverse of u = transport(a, b, d): adds lambda_a, lambda_b, returns lambda_d
__device__ __forceinline__ D3 transport_rev(D3 A, D3 Bv, D3 d, D3 lu, D3& la, D3& lb) {
    double c = dot(A, Bv);
    D3 k = cross(A, Bv);
    double kd = dot(k, d), luk = dot(lu, k), q = 1.0 / (1.0 + c);
    double lc = dot(lu, d) - kd * luk * q * q;
    D3 lk = cross(d, lu) + (kd * q) * lu + (luk * q) * d;
    la += lc * Bv + cross(Bv, lk);
    lb += lc * A + cross(lk, A);
    return c * lu + cross(lu, k) + (luk * q) * k;
}

// Reverse of the frame construction of dlo_set_state (space-parallel transport, holonomy
// spread for loops): cotangents of the initial base (t, d1) -> positions.  FP64, one block per
// rod and one thread per edge.  A transported director is determined by its edge's tangent and
// its turn about it, and a turn adds to every later director's, so the cotangent that reaches
// the transport into edge j is W_j (t_j x d_j) with W_j the sum over the edges k >= j of their
// cotangents' parts along t_k x d_k: a suffix sum instead of a chain, after which every edge's
// reverse is local.  Bound by the FP64 pipe for large batches and by its latency for small
// ones; one thread per rod walking its edges (with the frames in device memory) took 1395 us
// for one rod of 128 vertices and 1795 us for 4096.
__global__ void __launch_bounds__(kFrameMaxEdges) frames_adjoint_kernel(const RodInfo* rods, const float4* X0,
                                                                       const float4* gtb0, const float4* gd1b0,
                                                                       float4* gx0) {
    __shared__ D3 T[kFrameMaxEdges], A[kFrameMaxEdges], D[kFrameMaxEdges];   // tangents, axes, directors
    __shared__ Turn wsum[kFrameMaxWarps];
    __shared__ double red[kFrameMaxWarps];
    const int rod = blockIdx.x, j = threadIdx.x, lane = j & 31, w = j >> 5;
    const RodInfo R = rods[rod];
    const int nv = R.nv, ne = R.ne, v0 = R.v0, e0 = R.e0, nw = (int)blockDim.x >> 5;
    const bool closed = R.flags & ROD_CLOSED, on = j < ne;
    D3 t{0.0, 0.0, 1.0};
    double il = 0.0;
    if (on) {
        const D3 e = ld(X0[v0 + (j + 1 == nv ? 0 : j + 1)]) - ld(X0[v0 + j]);
        il = rsqrt(dot(e, e));
        t = il * e;
    }
    const D3 d = transported_director(t, false, ne, T, A, wsum);
    const D3 td = cross(t, d);
    if (on) D[j] = d;
    __syncthreads();   // D is complete; A is free and takes the tangents' cotangents below
    // cotangents of this edge's tangent (lt) and uncorrected director (ld1)
    D3 lt{0.0, 0.0, 0.0}, ld1 = lt;
    if (on) {
        lt = ld(gtb0[e0 + j]);
        ld1 = ld(gd1b0[e0 + j]);
    }
    const D3 a_first = A[0];
    if (closed) {   // the frames were turned by -psi j / ne, psi the holonomy
        const Turn z = transport_turn(T[ne - 1], D[ne - 1], T[0], a_first);
        const double phi = -atan2(z.s, z.c) * (double)j / (double)ne;
        double lpsi = 0.0;
        if (on) {
            const double cph = cos(phi), sph = sin(phi);
            const D3 l1 = ld1;
            ld1 = cph * l1 + sph * cross(l1, t);
            lt += sph * cross(d, l1);
            lpsi = -(double)j / (double)ne * dot(l1, cph * td - sph * d);
        }
        lpsi = warp_sum_d(lpsi);
        if (lane == 0) red[w] = lpsi;
        __syncthreads();
        lpsi = 0.0;
        for (int k = 0; k < nw; ++k) lpsi += red[k];
        __syncthreads();
        // psi is the angle from d_0 to u, the unit projection of the last director carried over
        if (j == 0 || j == ne - 1) {
            const D3 t0 = T[0], d0 = a_first;
            const D3 wl = transport_d(T[ne - 1], t0, D[ne - 1]);
            const D3 u = unit_d(wl - dot(wl, t0) * t0);
            const double y = dot(cross(d0, u), t0), x = dot(d0, u), r2 = x * x + y * y;
            const double ly = lpsi * x / r2, lx = -lpsi * y / r2;
            D3 lt0{0.0, 0.0, 0.0}, ltl = lt0;
            const D3 lw = adapt_rev(wl, t0, ly * cross(t0, d0) + lx * d0, lt0);
            const D3 ldl = transport_rev(T[ne - 1], t0, D[ne - 1], lw, ltl, lt0);
            if (j == 0) {
                ld1 += ly * cross(u, t0) + lx * u;
                lt += lt0 + ly * cross(d0, u);
            } else {
                lt += ltl;
                ld1 += ldl;
            }
        }
    }
    // W_j: suffix sum of the cotangents' parts along t x d
    double W = on ? dot(ld1, td) : 0.0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double p = __shfl_down_sync(0xffffffffu, W, o);
        if (lane + o < 32) W += p;
    }
    if (lane == 0) red[w] = W;
    __syncthreads();
    for (int k = nw - 1; k > w; --k) W += red[k];
    D3 lprev{0.0, 0.0, 0.0};   // cotangent of the previous edge's tangent
    if (on) {
        if (j == 0) {
            // the first director is the projection of a fixed axis; later edges' turns reach it as W_1 t x d
            adapt_rev(axis_of(t), t, ld1 + (W - dot(ld1, td)) * td, lt);
        } else {
            lt -= dot(ld1, t) * d;
            transport_rev(T[j - 1], t, D[j - 1], W * td, lprev, lt);
        }
    }
    __syncthreads();
    if (on && j > 0) A[j - 1] = lprev;   // from edge j to edge j - 1
    __syncthreads();
    float lex = 0.f, ley = 0.f, lez = 0.f;
    if (on) {
        if (j + 1 < ne) lt += A[j];
        const D3 le = il * (lt - dot(lt, t) * t);
        lex = (float)le.x;
        ley = (float)le.y;
        lez = (float)le.z;
    }
    if (on) D[j] = D3{(double)lex, (double)ley, (double)lez};
    __syncthreads();
    if (j < nv) {   // vertex j ends edge j - 1 and starts edge j
        float4 g = gx0[v0 + j];
        if (closed && j == 0) {
            g = make_float4(g.x - lex, g.y - ley, g.z - lez, g.w);
            const D3 p = D[ne - 1];
            g = make_float4(g.x + (float)p.x, g.y + (float)p.y, g.z + (float)p.z, g.w);
        } else {
            if (j > 0) {
                const D3 p = D[j - 1];
                g = make_float4(g.x + (float)p.x, g.y + (float)p.y, g.z + (float)p.z, g.w);
            }
            if (on) g = make_float4(g.x - lex, g.y - ley, g.z - lez, g.w);
        }
        gx0[v0 + j] = g;
    }
}

cudaError_t launch_rec(const BwdParams& P, int nv, bool c, int grid, int warps, cudaStream_t st) {
    switch (nv) {
        case 32: return launch_rec_nv32(P, c, grid, warps, st);
        case 64: return launch_rec_nv64(P, c, grid, warps, st);
        case 128: return launch_rec_nv128(P, c, grid, warps, st);
        case 192: return launch_rec_nv192(P, c, grid, warps, st);
        case 224: return launch_rec_nv224(P, c, grid, warps, st);
        case 256: return launch_rec_nv256(P, c, grid, warps, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_rev(const BwdParams& P, int nv, bool c, int grid, int warps, cudaStream_t st) {
    switch (nv) {
        case 32: return launch_rev_nv32(P, c, grid, warps, st);
        case 64: return launch_rev_nv64(P, c, grid, warps, st);
        case 128: return launch_rev_nv128(P, c, grid, warps, st);
        case 192: return launch_rev_nv192(P, c, grid, warps, st);
        case 224: return launch_rev_nv224(P, c, grid, warps, st);
        case 256: return launch_rev_nv256(P, c, grid, warps, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_frames_adjoint(const RodInfo* rods, int B, int nv_max, const float4* X0, const float4* gtb0,
                                  const float4* gd1b0, float4* gx0, cudaStream_t st) {
    frames_adjoint_kernel<<<B, nv_max, 0, st>>>(rods, X0, gtb0, gd1b0, gx0);
    return cudaGetLastError();
}

int rec_blocks_per_sm(int nv, bool c, int warps) {
    switch (nv) {
        case 32: return rec_occ_nv32(c, warps);
        case 64: return rec_occ_nv64(c, warps);
        case 128: return rec_occ_nv128(c, warps);
        case 192: return rec_occ_nv192(c, warps);
        case 224: return rec_occ_nv224(c, warps);
        case 256: return rec_occ_nv256(c, warps);
    }
    return 0;
}

int rev_blocks_per_sm(int nv, bool c, int warps) {
    switch (nv) {
        case 32: return rev_occ_nv32(c, warps);
        case 64: return rev_occ_nv64(c, warps);
        case 128: return rev_occ_nv128(c, warps);
        case 192: return rev_occ_nv192(c, warps);
        case 224: return rev_occ_nv224(c, warps);
        case 256: return rev_occ_nv256(c, warps);
    }
    return 0;
}

}  // namespace dlo

using namespace dlo;

namespace {

// record sizes (float4) of one rod of the class: cf. sub_rec / frame_rec / seg_state / cot_state
size_t frame_rec_h(int NV, int n_iter, int nsub) {
    return (size_t)(8 + NV) + (size_t)nsub * (size_t)(7 + 2 * n_iter + 2 * kPairsPerVertex) * NV;
}

// Rods per CTA and CTAs per SM that keep the most rods resident, with the fewest rods per CTA
// (a batch smaller than the device then spreads over all SMs: 304 rods of 128 vertices in CTAs of
// four filled half of them).
void best_shape(int nv, bool contact, bool rec, int& w, int& nb) {
    w = 0;
    nb = 0;
    for (int rpc = 1; rpc <= 16; ++rpc) {
        const int b = rec ? rec_blocks_per_sm(nv, contact, rpc) : rev_blocks_per_sm(nv, contact, rpc);
        if (b >= 1 && rpc * b > w * nb) {
            w = rpc;
            nb = b;
        }
    }
}

}  // namespace

void backward_shapes(dlo_ctx* c) {
    for (Bucket& bk : c->buckets) {
        best_shape(bk.nv_max, bk.contact, true, bk.rec_w, bk.rec_nb);
        best_shape(bk.nv_max, bk.contact, false, bk.rev_w, bk.rev_nb);
    }
}

// Plan of the chunked backward for checkpoint interval K: frames per chunk C (the records of
// one chunk of every rod within rec_budget, at most 64 frames), per-rod buffer sizes and the
// workspace of all rods at once.
dlo_status bwd_plan(dlo_ctx* c, int force, int K, BwdPlan& out, size_t rec_budget, int frames) {
    const size_t nb_ = c->buckets.size();
    if (!rec_budget) {
        const size_t budget = c->opt.hbm_budget ? c->opt.hbm_budget : ((size_t)80 << 30);
        rec_budget = std::min<size_t>((size_t)8 << 30, budget / 8);
    }
    out.nsmax.assign(nb_, 0);
    out.C.assign(nb_, 1);
    out.r3_rod.assign(nb_, 0);
    out.l2_rod.assign(nb_, 0);
    out.cs_rod.assign(nb_, 0);
    out.offset.assign(nb_, 0);
    size_t per_frame = 0;
    for (size_t k = 0; k < nb_; ++k) {
        const Bucket& bk = c->buckets[k];
        if (bk.rev_w < 1) return set_err(c, DLO_ERR_INVALID_ARG, "rod too large for the backward kernel's shared memory");
        if (bk.rec_w < 1) return set_err(c, DLO_ERR_INVALID_ARG, "rod too large for the recompute kernel's shared memory");
        int ns = force;
        if (!ns)
            for (int b = 0; b < c->B; ++b)
                if (size_class(c->rods_h[b].nv) == bk.nv_max) ns = std::max(ns, c->nsub[b]);
        out.nsmax[k] = ns;
        per_frame += 16 * (size_t)bk.n * frame_rec_h(bk.nv_max, c->opt.n_iter_pbd, ns);
    }
    int C = (int)std::max<size_t>(1, std::min<size_t>(64, rec_budget / std::max<size_t>(per_frame, 1)));
    if (frames > 0) C = std::min(C, (frames + K - 1) / K * K);
    if (C >= K) C = (C / K) * K;   // chunks start at checkpoints
    size_t need = 0;
    for (size_t k = 0; k < nb_; ++k) {
        const Bucket& bk = c->buckets[k];
        const int NV = bk.nv_max;
        out.C[k] = C;
        out.r3_rod[k] = (size_t)C * frame_rec_h(NV, c->opt.n_iter_pbd, out.nsmax[k]);
        out.l2_rod[k] = C < K ? (size_t)K * (5 * (size_t)NV + 6) : 0;
        out.cs_rod[k] = 5 * (size_t)NV + 6;
        out.offset[k] = need;   // each class has its own region: the classes run concurrently
        need += (16 * (size_t)bk.n * (out.r3_rod[k] + out.l2_rod[k] + out.cs_rod[k]) + 255) & ~(size_t)255;
    }
    out.fixed = (2 * 16 * (size_t)c->Et + 255) & ~(size_t)255;
    out.bytes = out.fixed + need;
    return DLO_OK;
}

dlo_status grow_workspace(dlo_ctx* c, size_t bytes, const char* what) {
    if (bytes <= c->bw_bytes) return DLO_OK;
    if (c->bw_mem) {
        const cudaError_t e = cudaStreamSynchronize(c->stream);
        if (e != cudaSuccess) return cuda_err(c, e, "stream");
        dev_free(c, c->bw_mem);
    }
    c->bw_mem = dev_alloc(c, bytes);
    c->bw_bytes = c->bw_mem ? bytes : 0;
    return c->bw_mem ? DLO_OK : set_err(c, DLO_ERR_OOM, what);
}

bool records_fit(const dlo_ctx* c, const BwdPlan& plan) {
    for (int C : plan.C)
        if (C < c->rec_frames) return false;
    return plan.bytes <= c->bw_bytes;
}

dlo_status enqueue_backward_class(dlo_ctx* c, const BwdPlan& plan, size_t k, cudaStream_t st, int item0, int n,
                                  float4* R3, float4* L2, float4* CS, int C, const BwdParams& common, bool stored) {
    const Bucket& bk = c->buckets[k];
    BwdParams P = common;
    P.order = bk.d_order;
    P.item0 = item0;
    P.n_items = n;
    P.counter = c->d_counters + kNumSizeClasses + k;
    P.nsub_max = plan.nsmax[k];
    P.R3 = R3;
    P.L2 = L2;
    P.CS = CS;
    backward_rod_f4(c, plan, k, C, P.r3_rod, P.l2_rod, P.cs_rod);
    const int rec_w = bk.rec_w, rev_w = bk.rev_w;
    const int rec_grid = (int)std::min<long long>((long long)bk.rec_nb * c->sm_count, (n + rec_w - 1) / rec_w);
    const int rev_grid = (int)std::min<long long>((long long)bk.rev_nb * c->sm_count, (n + rev_w - 1) / rev_w);
    const int K = c->ck_every, F = c->rec_frames;
    // the chunks, first to last: from every checkpoint when C >= K (C a multiple of K), else
    // within each segment
    std::vector<std::pair<int, int>> chunks;
    if (C >= K) {
        for (int fa = 0; fa < F; fa += C) chunks.push_back({fa, std::min(fa + C, F)});
    } else {
        for (int f0 = 0; f0 < F; f0 += K) {
            const int f1 = std::min(f0 + K, F);
            for (int fa = f0; fa < f1; fa += C) chunks.push_back({fa, std::min(fa + C, f1)});
        }
    }
    for (size_t q = chunks.size(); q-- > 0;) {
        const int fa = chunks[q].first, fb = chunks[q].second;
        const int f0 = (fa / K) * K;
        cudaError_t e = cudaSuccess;
        if (C < K && fb == std::min(f0 + K, F)) {   // entering a segment: its frame-start states
            P.mode = 0;
            P.fa = f0;
            P.fb = f0;
            e = cudaMemsetAsync(P.counter, 0, sizeof(int), st);
            if (e == cudaSuccess) e = launch_rec(P, bk.nv_max, bk.contact, rec_grid, rec_w, st);
            c->launches++;
        }
        P.mode = 1;
        P.fa = fa;
        P.fb = fb;
        if (!stored) {
            if (e == cudaSuccess) e = cudaMemsetAsync(P.counter, 0, sizeof(int), st);
            if (e == cudaSuccess) e = launch_rec(P, bk.nv_max, bk.contact, rec_grid, rec_w, st);
            c->launches++;
        }
        P.first_chunk = fb == F;
        P.last_chunk = fa == 0;
        if (e == cudaSuccess) e = cudaMemsetAsync(P.counter, 0, sizeof(int), st);
        if (e == cudaSuccess) e = launch_rev(P, bk.nv_max, bk.contact, rev_grid, rev_w, st);
        c->launches++;
        if (e != cudaSuccess) return cuda_err(c, e, "backward launch");
    }
    return DLO_OK;
}

void backward_rod_f4(dlo_ctx* c, const BwdPlan& plan, size_t k, int C, size_t& r3, size_t& l2, size_t& cs) {
    const int NV = c->buckets[k].nv_max, K = c->ck_every;
    r3 = (size_t)C * frame_rec_h(NV, c->opt.n_iter_pbd, plan.nsmax[k]);
    l2 = C < K ? (size_t)K * (5 * (size_t)NV + 6) : 0;
    cs = plan.cs_rod[k];
}

int backward_resident_rods(dlo_ctx* c, size_t k) {
    return c->buckets[k].rev_w * c->buckets[k].rev_nb * c->sm_count;
}

// the inputs and outputs shared by every launch of one backward
BwdParams backward_common(dlo_ctx* c, int force, const float* dL_dx_T, const float* dL_dv_T, const float* dL_dtheta_T,
                          float* dL_dactions, float* dL_dmaterial, float* dL_dx0, float* dL_dv0, float* dL_dtheta0,
                          float4* gtb0, float4* gd1b0) {
    BwdParams P{};
    P.rods = c->d_rods;
    P.ck = c->ck;
    P.ck_strideV = c->V;
    P.ck_strideE = c->Et;
    P.ck_strideB = 24LL * c->B;
    P.ck_every = c->ck_every;
    P.ck_count = c->ck_count;
    P.KIN = c->d_kin;
    P.ES = c->d_es;
    P.actions = c->rec_actions;
    P.frames = c->rec_frames;
    P.B = c->B;
    P.force_nsub = force;
    P.dLdx = reinterpret_cast<const float4*>(dL_dx_T);
    P.dLdv = reinterpret_cast<const float4*>(dL_dv_T);
    P.dLdth = dL_dtheta_T;
    P.gact = dL_dactions;
    P.gmat = dL_dmaterial;
    P.gx0 = reinterpret_cast<float4*>(dL_dx0);
    P.gv0 = reinterpret_cast<float4*>(dL_dv0);
    P.gth0 = dL_dtheta0;
    P.gtb0 = gtb0;
    P.gd1b0 = gd1b0;
    P.status = c->d_status;
    P.scene = c->scene;
    return P;
}

extern "C" dlo_status dlo_backward(dlo_ctx* c, const float* dL_dx_T, const float* dL_dv_T, const float* dL_dtheta_T,
                                   float* dL_dactions, float* dL_dmaterial, float* dL_dx0, float* dL_dv0,
                                   float* dL_dtheta0) {
    if (!c) return DLO_ERR_INVALID_ARG;
    if (!c->rec_active || c->rec_done != c->rec_frames || c->rec_frames == 0)
        return set_err(c, DLO_ERR_STATE, "dlo_backward needs a completed rollout armed by dlo_begin_rollout");
    for (const void* p : {(const void*)dL_dx_T, (const void*)dL_dv_T, (const void*)dL_dx0, (const void*)dL_dv0})
        if (p && ((uintptr_t)p & 15u)) return set_err(c, DLO_ERR_INVALID_ARG, "float4 arrays must be 16-byte aligned");
    if (c->opt.self_contact && c->opt.n_iter_pbd < 1)
        return set_err(c, DLO_ERR_INVALID_ARG, "self-contact gradients need at least one projection iteration");
    const int force = c->rec_nsub > 0 ? c->rec_nsub : 0;
    BwdPlan plan;
    dlo_status pst = bwd_plan(c, force, c->ck_every, plan, c->rec_budget, c->rec_frames);
    if (pst != DLO_OK) return pst;
    const bool stored = c->rec_stored && records_fit(c, plan);
    c->rec_wanted = true;
    pst = grow_workspace(c, plan.bytes, "backward workspace allocation failed");
    if (pst != DLO_OK) return pst;
    char* p = reinterpret_cast<char*>(c->bw_mem);
    float4* gtb0 = reinterpret_cast<float4*>(p);
    float4* gd1b0 = gtb0 + c->Et;
    char* region = p + plan.fixed;
    const BwdParams common = backward_common(c, force, dL_dx_T, dL_dv_T, dL_dtheta_T, dL_dactions, dL_dmaterial,
                                             dL_dx0, dL_dv0, dL_dtheta0, gtb0, gd1b0);
    {
        cudaError_t fe = fork_classes(c);
        if (fe != cudaSuccess) return cuda_err(c, fe, "fork");
    }
    for (size_t k = c->buckets.size(); k-- > 0;) {   // the longest rods first, as in the forward
        const int n = c->buckets[k].n;
        float4* R3 = reinterpret_cast<float4*>(region + plan.offset[k]);
        float4* L2 = R3 + (size_t)n * plan.r3_rod[k];
        float4* CS = L2 + (size_t)n * plan.l2_rod[k];
        dlo_status st = enqueue_backward_class(c, plan, k, class_stream(c, k), 0, n, R3, L2, CS, plan.C[k], common,
                                               stored);
        if (st != DLO_OK) return st;
    }
    {
        cudaError_t je = join_classes(c);
        if (je != cudaSuccess) return cuda_err(c, je, "join");
    }
    if (c->rec_from_set && dL_dx0) {
        cudaError_t e = launch_frames_adjoint(c->d_rods, c->B, c->buckets.back().nv_max, c->ck.X, gtb0, gd1b0,
                                              reinterpret_cast<float4*>(dL_dx0), c->stream);
        c->launches++;
        if (e != cudaSuccess) return cuda_err(c, e, "frames adjoint launch");
    }
    return check_status(c);
}
