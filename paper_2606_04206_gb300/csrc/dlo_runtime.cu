// dlo_runtime.cu -- device allocation, size-class buckets, the step launch and rollout recording
// (gradient checkpointing, DLO-Lab Sec. 3.3: one state snapshot per segment, kept in HBM).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "dlo_kernels.h"
#include "dlo_runtime.h"

using namespace dlo;


template <class T>
static T* alloc_up(dlo_ctx* c, const std::vector<T>& h, dlo_status& st) {
    if (st != DLO_OK) return nullptr;
    T* d = reinterpret_cast<T*>(dev_alloc(c, sizeof(T) * std::max<size_t>(h.size(), 1)));
    if (!d) {
        st = set_err(c, DLO_ERR_OOM, "device allocation failed");
        return nullptr;
    }
    if (!h.empty()) {
        cudaError_t e = cudaMemcpyAsync(d, h.data(), sizeof(T) * h.size(), cudaMemcpyHostToDevice, c->stream);
        if (e != cudaSuccess) st = cuda_err(c, e, "upload");
    }
    return d;
}

static void* alloc_zero(dlo_ctx* c, size_t bytes, dlo_status& st) {
    if (st != DLO_OK) return nullptr;
    void* d = dev_alloc(c, bytes);
    if (!d) {
        st = set_err(c, DLO_ERR_OOM, "device allocation failed");
        return nullptr;
    }
    cudaError_t e = cudaMemsetAsync(d, 0, bytes, c->stream);
    if (e != cudaSuccess) st = cuda_err(c, e, "memset");
    return d;
}

// Forward launch of one size class over `frames` frames without actions or recording.
static cudaError_t launch_bucket(dlo_ctx* c, size_t k, int warps, int grid, int frames) {
    const Bucket& bk = c->buckets[k];
    FwdParams P{};
    P.rods = c->d_rods;
    P.order = bk.d_order;
    P.n_order = bk.n;
    P.counter = c->d_counters + k;
    P.S = c->S;
    P.KIN = c->d_kin;
    P.ES = c->d_es;
    P.frames = frames;
    P.B = c->B;
    P.nvert_total = c->V;
    P.status = c->d_status;
    P.residual = c->d_residual;
    P.npairs = c->d_npairs;
    P.scene = c->scene;
    cudaError_t e = cudaMemsetAsync(P.counter, 0, sizeof(int), c->stream);
    if (e == cudaSuccess) e = launch_forward(P, bk.nv_max, bk.contact, grid, warps, c->stream);
    c->launches++;
    return e;
}

// The rods per CTA run for a requested count (0: refused).  A request is accepted when the
// rods would fit a CTA of 512 threads at up to 128 threads and 227 KB of shared memory for all
// (the rule callers know); a CTA of rods above 128 vertices, which take a thread per vertex, then
// holds as many of them as it can.
static int forced_rods_per_cta(int nv_max, bool contact, int want) {
    if (want * std::min(nv_max, 128) > 512 || want * (warp_smem_bytes(nv_max, contact) + 16 * nv_max + 768) > 227 * 1024) return 0;
    while (want > 1 && forward_blocks_per_sm(nv_max, contact, want) < 1) --want;
    return want;
}

// Rods per CTA by measurement (the autotuner): every count whose occupancy keeps at least
// half of the most resident rods is timed on two frames from the rest state, after one
// warm-up launch, and the fastest is kept.  The caller resets the state afterwards.
static dlo_status autotune_rods_per_cta(dlo_ctx* c) {
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return cuda_err(c, cudaGetLastError(), "event");
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return cuda_err(c, cudaGetLastError(), "event");
    }
    dlo_status st = DLO_OK;
    for (size_t k = 0; k < c->buckets.size() && st == DLO_OK; ++k) {
        Bucket& bk = c->buckets[k];
        int most = 0;
        for (int rpc = 1; rpc <= 16; ++rpc) most = std::max(most, rpc * forward_blocks_per_sm(bk.nv_max, bk.contact, rpc));
        float best_ms = 1e30f;
        int best_w = bk.warps, best_g = bk.grid;
        cudaError_t e = launch_bucket(c, k, bk.warps, bk.grid, 1);   // warm-up (module load, clocks)
        for (int rpc = 1; rpc <= 16 && e == cudaSuccess; ++rpc) {
            const int nb = forward_blocks_per_sm(bk.nv_max, bk.contact, rpc);
            if (nb < 1 || 2 * rpc * nb < most) continue;
            const int grid = (int)std::min<long long>((long long)nb * c->sm_count, (bk.n + rpc - 1) / rpc);
            e = cudaEventRecord(e0, c->stream);
            if (e == cudaSuccess) e = launch_bucket(c, k, rpc, grid, 2);
            if (e == cudaSuccess) e = cudaEventRecord(e1, c->stream);
            if (e == cudaSuccess) e = cudaEventSynchronize(e1);
            float ms = 0.f;
            if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
            if (e == cudaSuccess && ms < best_ms) {
                best_ms = ms;
                best_w = rpc;
                best_g = grid;
            }
        }
        if (e != cudaSuccess) st = cuda_err(c, e, "autotune");
        bk.warps = best_w;
        bk.grid = best_g;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return st;
}

// From this many rods of up to 32 vertices on they are packed into warps, when that saves warps: if none
// has more than 16 vertices, or if longer rods in the batch would give each a longer rod's block.
// dlo_set_state, a block per rod and packed: 1024 rods x 4 14.5 and 10.8 us, 65536 x 4 486 and
// 64 us, 65536 x 16 484 and 240 us, 65536 x 32 483 and 482 us.
static constexpr int kPackRods = 1024;

cudaError_t init_rods(dlo_ctx* c, InitParams& P) {
    const Bucket& bk = c->buckets.front();
    const bool pack = bk.nv_max <= 32 && bk.n >= kPackRods && (bk.nv_top <= 16 || bk.n < c->B);
    P.small = bk.d_order;
    P.n_small = pack ? bk.n : 0;
    P.nv_small = bk.nv_top;
    c->launches += pack && bk.n < c->B ? 2 : 1;
    return launch_init(P, c->buckets.back().nv_max, c->stream);
}

dlo_status runtime_allocate(dlo_ctx* c, const std::vector<RodInfo>& rods, const std::vector<float4>& kin,
                            const std::vector<float2>& mass, const std::vector<float2>& es,
                            const std::vector<float4>& rest, const std::vector<float>& gp0,
                            const std::vector<float4>& xr4) {
    dlo_status st = DLO_OK;
    c->d_rods = alloc_up(c, rods, st);
    c->d_kin = alloc_up(c, kin, st);
    c->d_mass = alloc_up(c, mass, st);
    c->d_es = alloc_up(c, es, st);
    c->d_rest = alloc_up(c, rest, st);
    c->d_gp0 = alloc_up(c, gp0, st);
    c->S.X = alloc_up(c, xr4, st);
    c->S.Vl = reinterpret_cast<float4*>(alloc_zero(c, 16 * c->V, st));
    c->S.HG = reinterpret_cast<float4*>(alloc_zero(c, 16 * c->V, st));
    c->S.ED = reinterpret_cast<float4*>(alloc_zero(c, 16 * c->Et, st));
    c->S.ET = reinterpret_cast<float4*>(alloc_zero(c, 16 * c->Et, st));
    c->S.GP = reinterpret_cast<float*>(alloc_zero(c, sizeof(float) * 24 * c->B, st));
    c->d_status = reinterpret_cast<unsigned*>(alloc_zero(c, sizeof(unsigned) * c->B, st));
    c->d_residual = reinterpret_cast<double*>(alloc_zero(c, sizeof(double) * c->B, st));
    c->d_npairs = reinterpret_cast<int*>(alloc_zero(c, sizeof(int) * c->B, st));
    if (c->opt.reaction) c->d_reaction = reinterpret_cast<float4*>(alloc_zero(c, 64 * c->V, st));
    if (c->opt.self_contact)
        c->d_pair_list = reinterpret_cast<uint32_t*>(
            alloc_zero(c, sizeof(uint32_t) * (1 + (size_t)kPairListStride) * c->B, st));
    if (st != DLO_OK) return st;
    // Size classes; rods of a class in decreasing cost, so that the longest do not start last, and
    // rods of one kind (elastic, with torsion, with length projections) side by side: rods on one SM
    // that take the same path take it together, and mixed ones keep fetching each other's code.
    // 4096 rods x 128, a third cables, 16 frames: with the kinds taking turns the forward takes
    // 4.6 ms and the reverse 8.6 ms, sorted 4.3 and 6.4 ms.  The cost in tenths of an elastic rod's
    // reverse, from batches of one kind.
    auto cost = [&](int b) {
        const RodInfo& R = rods[b];
        const int kind = 10 + (R.beta != 0.f ? 2 : 0) + (R.flags & (ROD_INEXT | ROD_SLIMIT) ? (6 * c->opt.n_iter_pbd + 9) / 10 : 0);
        return (long long)R.nv * R.nsub * kind;
    };
    std::vector<std::vector<int>> cls(kNumSizeClasses);
    for (int b = 0; b < c->B; ++b)
        for (int k = 0; k < kNumSizeClasses; ++k)
            if (size_class_at(k) == size_class(rods[b].nv)) cls[k].push_back(b);
    for (int k = 0; k < kNumSizeClasses; ++k) {
        if (cls[k].empty()) continue;
        std::vector<int>& ids = cls[k];
        std::stable_sort(ids.begin(), ids.end(), [&](int a, int b) {
            return cost(a) > cost(b);
        });
        Bucket bk;
        bk.nv_max = size_class_at(k);
        bk.contact = c->opt.self_contact != 0;
        bk.n = (int)ids.size();
        for (int b : ids) bk.nv_top = std::max(bk.nv_top, rods[b].nv);
        bk.d_order = alloc_up(c, ids, st);
        if (st != DLO_OK) return st;
        // rods per CTA: the count (within the thread budget) that keeps the most rods resident;
        // the measured autotune below may pick another
        int best = 0, best_nb = 0;
        const int forced = c->opt.warps_per_cta;
        const int cap = forced > 0 ? forced_rods_per_cta(bk.nv_max, bk.contact, forced) : 16;
        for (int rpc = forced > 0 ? std::max(cap, 1) : 1; rpc <= cap; ++rpc) {
            const int nb = forward_blocks_per_sm(bk.nv_max, bk.contact, rpc);
            if (nb >= 1 && rpc * nb >= best * best_nb) {
                best = rpc;
                best_nb = nb;
            }
        }
        if (best < 1) return set_err(c, DLO_ERR_INVALID_ARG, "rod too large for shared memory");
        bk.warps = best;
        long long want = (bk.n + best - 1) / best;
        bk.grid = (int)std::min<long long>((long long)best_nb * c->sm_count, want);
        c->buckets.push_back(bk);
    }
    backward_shapes(c);
    if (c->buckets.size() > 1) {   // one stream per size class (see dlo_ctx::side)
        c->side.resize(c->buckets.size(), nullptr);
        c->joins.resize(c->buckets.size(), nullptr);
        cudaError_t e = cudaEventCreateWithFlags(&c->fork, cudaEventDisableTiming);
        for (size_t k = 0; k < c->buckets.size() && e == cudaSuccess; ++k) {
            e = cudaStreamCreateWithFlags(&c->side[k], cudaStreamNonBlocking);
            if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->joins[k], cudaEventDisableTiming);
        }
        if (e != cudaSuccess) return cuda_err(c, e, "size-class streams");
    }
    // work-queue heads: one per size class for the forward, one per class for the backward
    c->d_counters = reinterpret_cast<int*>(alloc_zero(c, sizeof(int) * 2 * kNumSizeClasses, st));
    if (st != DLO_OK) return st;
    // rest twist from the rest frames, then the rest state
    InitParams P{};
    P.rods = c->d_rods;
    P.B = c->B;
    P.xin = c->S.X;
    P.mass = c->d_mass;
    P.ES = c->d_es;
    P.rest = c->d_rest;
    P.S = c->S;
    P.GP0 = c->d_gp0;
    P.rest_mode = 1;
    st = cuda_err(c, init_rods(c, P), "rest init");
    if (st != DLO_OK) return st;
    P.rest_mode = 0;
    st = cuda_err(c, init_rods(c, P), "state init");
    if (st == DLO_OK && c->opt.warps_per_cta == 0) {
        // measured autotune of rods per CTA; then the rest state is set again (positions
        // re-uploaded, frames, velocities and poses re-initialised, status cleared)
        st = autotune_rods_per_cta(c);
        if (st == DLO_OK)
            st = cuda_err(c, cudaMemcpyAsync(c->S.X, xr4.data(), sizeof(float4) * xr4.size(), cudaMemcpyHostToDevice,
                                             c->stream), "rest positions");
        if (st == DLO_OK)
            st = cuda_err(c, cudaMemsetAsync(c->d_status, 0, sizeof(unsigned) * c->B, c->stream), "status reset");
        if (st == DLO_OK) st = cuda_err(c, init_rods(c, P), "state init");
    }
    c->from_set_state = true;
    if (st == DLO_OK) st = cuda_err(c, cudaStreamSynchronize(c->stream), "create");
    return st;
}

void runtime_release(dlo_ctx* c) {
    for (cudaStream_t s : c->side) cudaStreamDestroy(s);
    for (cudaEvent_t e : c->joins) cudaEventDestroy(e);
    if (c->fork) cudaEventDestroy(c->fork);
    c->side.clear();
    c->joins.clear();
    c->fork = nullptr;
}

cudaStream_t class_stream(dlo_ctx* c, size_t k) { return c->side.empty() ? c->stream : c->side[k]; }

cudaError_t fork_classes(dlo_ctx* c) {
    if (c->side.empty()) return cudaSuccess;
    cudaError_t e = cudaEventRecord(c->fork, c->stream);
    for (size_t k = 0; k < c->side.size() && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(c->side[k], c->fork, 0);
    return e;
}

cudaError_t join_classes(dlo_ctx* c) {
    cudaError_t e = cudaSuccess;
    for (size_t k = 0; k < c->side.size() && e == cudaSuccess; ++k) {
        e = cudaEventRecord(c->joins[k], c->side[k]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(c->stream, c->joins[k], 0);
    }
    return e;
}

// ------------------------------------------------------------------ rollout recording
extern "C" dlo_status dlo_begin_rollout(dlo_ctx* c, int n_frames) {
    if (!c) return DLO_ERR_INVALID_ARG;
    if (n_frames <= 0) return set_err(c, DLO_ERR_INVALID_ARG, "n_frames must be positive");
    const size_t per = 16 * (3 * (size_t)c->V + 2 * (size_t)c->Et) + sizeof(float) * 24 * (size_t)c->B;
    const size_t abytes = sizeof(float) * 12 * (size_t)c->B * n_frames;
    int K = std::min(c->opt.checkpoint_every, n_frames);
    const size_t budget = c->opt.hbm_budget ? c->opt.hbm_budget : ((size_t)80 << 30);
    if (K <= 0) {
        // autotune: the shortest interval (the least recomputation in the backward) whose
        // checkpoint ring, action record and backward workspace fit the HBM budget; the
        // backward reruns at most K - 1 frames per segment to rebuild the frame-start states
        K = n_frames;
        for (int k = 1; k <= n_frames; ++k) {
            BwdPlan plan;
            if (bwd_plan(c, 0, k, plan) != DLO_OK) return DLO_ERR_INVALID_ARG;
            const size_t total = per * (size_t)((n_frames + k - 1) / k) + abytes + plan.bytes;
            if (total <= budget) {
                K = k;
                break;
            }
        }
    }
    const int count = (n_frames + K - 1) / K;
    // Frames per backward launch pair: the chunk records may take half of what the ring and the
    // action record leave of the budget (at most 24 GiB), and never less than the default the
    // interval was chosen with.  Longer chunks mean fewer launch pairs, each with its own tail.
    {
        const size_t used = per * (size_t)count + abytes;
        const size_t spare = budget > used ? budget - used : 0;
        const size_t dflt = std::min<size_t>((size_t)8 << 30, budget / 8);
        c->rec_budget = std::max(dflt, std::min<size_t>((size_t)24 << 30, spare / 2));
    }
    const size_t need = per * count + 256 * 8;
    if (need > c->ck_bytes) {
        dev_free(c, c->ck_mem);
        c->ck_mem = dev_alloc(c, need);
        c->ck_bytes = c->ck_mem ? need : 0;
        if (!c->ck_mem) return set_err(c, DLO_ERR_OOM, "checkpoint ring allocation failed");
    }
    char* p = reinterpret_cast<char*>(c->ck_mem);
    auto take = [&](size_t bytes) {
        char* q = p;
        p += (bytes + 255) & ~(size_t)255;
        return q;
    };
    c->ck.X = reinterpret_cast<float4*>(take(16 * c->V * count));
    c->ck.Vl = reinterpret_cast<float4*>(take(16 * c->V * count));
    c->ck.HG = reinterpret_cast<float4*>(take(16 * c->V * count));
    c->ck.ED = reinterpret_cast<float4*>(take(16 * c->Et * count));
    c->ck.ET = reinterpret_cast<float4*>(take(16 * c->Et * count));
    c->ck.GP = reinterpret_cast<float*>(take(sizeof(float) * 24 * c->B * count));
    if (abytes > c->rec_bytes) {
        dev_free(c, c->rec_actions);
        c->rec_actions = reinterpret_cast<float*>(dev_alloc(c, abytes));
        c->rec_bytes = c->rec_actions ? abytes : 0;
        if (!c->rec_actions) return set_err(c, DLO_ERR_OOM, "action record allocation failed");
    }
    c->ck_every = K;
    c->ck_count = count;
    c->rec_frames = n_frames;
    c->rec_done = 0;
    c->rec_active = true;
    // if they fit: the first step, which knows the substeps, finds out
    c->rec_stored = c->rec_wanted && !c->rec_captured;
    c->rec_from_set = c->from_set_state;
    c->rec_nsub = -1;
    return DLO_OK;
}

// ------------------------------------------------------------------ step
dlo_status note_capture(dlo_ctx* c) {
    if (c->rec_captured) return DLO_OK;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(c->stream, &cap);
    if (e != cudaSuccess) return cuda_err(c, e, "capture status");
    if (cap != cudaStreamCaptureStatusNone) {
        c->rec_captured = true;
        c->rec_stored = false;
    }
    return DLO_OK;
}

dlo_status launch_step(dlo_ctx* c, const float* actions, int frames, int substeps, float* x_frames, int frame0,
                       bool record) {
    // When the workspace of an earlier dlo_backward has room for the substep records of the whole
    // rollout, the forward stores them there as it steps and the backward does not step again to
    // get them.  Nothing is allocated for it: the first dlo_backward of a context recomputes, and
    // a caller of dlo_backward_noalloc or dlo_backward_plain, which read no such records, neither
    // holds memory for them nor writes them.  4096 rods x 128 vertices, 16 frames (19 GB of
    // records), forward and backward: 14.0 ms recomputed, 10.9 ms stored; one rod x 128, 10 frames:
    // 1.54 and 1.07 ms.
    if (record && c->rec_stored && c->rec_done == 0)
        c->rec_stored = bwd_plan(c, substeps, c->ck_every, c->rec_plan, c->rec_budget, c->rec_frames) == DLO_OK &&
                        records_fit(c, c->rec_plan);
    cudaError_t fe = cudaMemsetAsync(c->d_counters, 0, sizeof(int) * c->buckets.size(), c->stream);
    if (fe == cudaSuccess) fe = fork_classes(c);
    if (fe != cudaSuccess) return cuda_err(c, fe, "fork");
    // The longest rods first: they share the SMs with the other classes' and end last.
    // (1024 rods of 16-256 vertices: 1.73 -> 1.66 ms.)
    for (size_t k = c->buckets.size(); k-- > 0;) {
        const Bucket& bk = c->buckets[k];
        FwdParams P{};
        P.rods = c->d_rods;
        P.order = bk.d_order;
        P.n_order = bk.n;
        P.counter = c->d_counters + k;
        P.S = c->S;
        P.KIN = c->d_kin;
        P.ES = c->d_es;
        P.actions = actions;
        P.xframes = x_frames;
        P.frames = frames;
        P.B = c->B;
        P.force_nsub = substeps;
        P.frame0 = frame0;
        P.nvert_total = c->V;
        if (record) {
            P.ck = c->ck;
            P.ck_strideV = c->V;
            P.ck_strideE = c->Et;
            P.ck_strideB = 24LL * c->B;
            P.ck_every = c->ck_every;
            P.ck_count = c->ck_count;
            if (c->rec_stored) {
                const BwdPlan& plan = c->rec_plan;
                P.R3 = reinterpret_cast<float4*>(reinterpret_cast<char*>(c->bw_mem) + plan.fixed + plan.offset[k]);
                P.r3_rod = plan.r3_rod[k];
                P.nsub_max = plan.nsmax[k];
            }
        }
        P.status = c->d_status;
        P.residual = c->d_residual;
        P.npairs = c->d_npairs;
        P.reaction = c->d_reaction;
        P.pair_list = c->d_pair_list;
        P.scene = c->scene;
        cudaStream_t sk = class_stream(c, k);
        const cudaError_t e = launch_forward(P, bk.nv_max, bk.contact, bk.grid, bk.warps, sk);
        c->launches++;
        if (e != cudaSuccess) return cuda_err(c, e, "forward launch");
    }
    fe = join_classes(c);
    if (fe != cudaSuccess) return cuda_err(c, fe, "join");
    return DLO_OK;
}

extern "C" dlo_status dlo_step(dlo_ctx* c, const float* actions, int frames, int substeps, float* x_frames) {
    if (!c) return DLO_ERR_INVALID_ARG;
    if (frames < 0 || substeps < 0 || substeps > 100000) return set_err(c, DLO_ERR_INVALID_ARG, "bad frames/substeps");
    if (x_frames && ((uintptr_t)x_frames & 15u)) return set_err(c, DLO_ERR_INVALID_ARG, "x_frames must be 16-byte aligned");
    if (frames == 0) return DLO_OK;
    const bool rec = c->rec_active && c->rec_done < c->rec_frames;
    int frame0 = 0;
    const float* acts = actions;
    if (rec) {
        if (c->rec_done + frames > c->rec_frames)
            return set_err(c, DLO_ERR_STATE, "step runs past the frames armed by dlo_begin_rollout");
        if (c->rec_nsub >= 0 && c->rec_nsub != substeps)
            return set_err(c, DLO_ERR_STATE, "substeps changed inside a recorded rollout");
        dlo_status cs = note_capture(c);
        if (cs != DLO_OK) return cs;
        c->rec_nsub = substeps;
        float* dst = c->rec_actions + (size_t)12 * c->B * c->rec_done;
        cudaError_t e = actions ? cudaMemcpyAsync(dst, actions, sizeof(float) * 12 * c->B * frames,
                                                  cudaMemcpyDeviceToDevice, c->stream)
                                : cudaMemsetAsync(dst, 0, sizeof(float) * 12 * c->B * frames, c->stream);
        if (e != cudaSuccess) return cuda_err(c, e, "record actions");
        frame0 = c->rec_done;
        acts = dst;
    } else {
        c->rec_active = false;
    }
    dlo_status st = launch_step(c, acts, frames, substeps, x_frames, frame0, rec);
    if (st != DLO_OK) return st;
    if (rec) c->rec_done += frames;
    c->from_set_state = false;
    return DLO_OK;
}
