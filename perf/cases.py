"""Performance cases of the rod stepper: what its users have it do, through the public binding.

A case is a dict of plain values.  ``prepare`` draws the rods, their state and the gripper
actions from the seed and creates the context that a program keeps; ``run`` is one pass of the
program's inner loop (set the state, step, score, differentiate); ``exact`` evaluates the same
definitions (DLO-Lab, arXiv 2606.04206, Sec. 3 and App. A.1, with the library's documented
conventions) in 64 bits with torch alone.

Scenes, after the package's workloads (``inputs.py``):

* ``hang``    straight rods held at one end, released from horizontal (one rod, config "plain")
* ``table``   ropes lying on the ground, two grippers; thirds of inextensible cable, elastic
              rope and plastic wire (trajectory optimisation), self-contact on
* ``diff``    the same without cables, halves of rope and plastic wire, no self-contact
* ``ragged``  rods of 16 to 256 vertices, moduli over four decades, per-rod substeps (batching)
* ``bands``   closed knotted bands on a box, crossings in contact (self-contact)
* ``knot``    copies of one knotted rope, each with its own gripper trajectory (one CMA-ES
              generation of Unknotting), crossings in contact
* ``pair``    two tangled ropes per environment as strands of one record (Separation)

Rollouts start from a state in motion (rods swept across the table, crossings pressed together),
as in the middle of a manipulation, because a pass of a few frames from rest would never reach the contact that
most of a long rollout spends its time in.
"""
import math

import numpy as np
import torch

from paper_2606_04206_gb300 import dlo, inputs

RADIUS, DT, MU_SELF, MU_RIGID, GRAVITY, EPS, MARGIN, N_ITER = 0.002, 1e-3, 0.3, 0.5, 9.81, 0.5, 1.0, 10
GRIP_R, GRIP_HL = 0.01, 0.02
SIL_TAU = 0.5
KINDS = ("hang", "table", "diff", "ragged", "bands", "knot", "pair")


def listed():
    return [
        # the smallest call: one cantilevered rod, the library's first workload; all latency
        case("hang_1x32", "hang", "step", 1, 32, 20),
        # model-predictive control of a handful of environments: one frame per call, state read back
        case("control_16x64", "table", "step", 16, 64, 1),
        # one gradient through a short rollout of one rope: an interactive planner's inner step
        case("plan_1x128", "table", "grad", 1, 128, 10),
        # one CMA-ES generation of Unknotting, scored on the device (forward only, self-contact)
        case("cmaes_400x128", "knot", "score", 400, 128, 20),
        # a batch of uneven rods, stiffness over four decades: per-rod substeps, six size classes
        case("ragged_1024", "ragged", "step", 1024, 256, 1),
        # the same, differentiated (fewer rods of odd sizes)
        case("ragged_grad_203", "ragged", "grad", 203, 181, 1),
        # differentiation config: 256 rods x 64 vertices through the autograd function
        case("diff_256x64", "diff", "autograd", 256, 64, 16),
        # system identification: two 256 x 256 cameras' silhouette loss, gradient to the start and material
        case("sysid_64x64", "diff", "sysid", 64, 64, 8, pixels=256),
        # Separation: tangled pairs of 30-vertex ropes, contact between the strands of a record
        case("pair_1024x60", "pair", "step", 1024, 60, 10),
        # closed bands in self-contact, differentiated
        case("bands_512x200", "bands", "grad", 512, 200, 4),
        # the flagship: trajectory optimisation of 4096 ropes x 128 vertices
        case("trajopt_4096x128", "table", "grad", 4096, 128, 16),
        # task losses of a batch of final states with their gradients
        case("losses_2048x128", "table", "losses", 2048, 128, 0, points=256),
    ]


def case(name, scene, mode, rods, verts, frames, **more):
    return dict(name=name, scene=scene, mode=mode, rods=rods, verts=verts, frames=frames, **more)


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("step", "step", "grad", "grad", "score", "autograd", "sysid", "losses"))
    verts = rng.randint(24, 256)
    if kind == "step":
        scene = rng.choice(("hang", "table", "ragged", "pair"))
        rods = log_int(1, 512 if scene == "ragged" else 4096)
        frames = 1 if scene == "ragged" else rng.randint(1, 20)
        if scene == "pair":
            rods, verts = log_int(8, 2048), 2 * rng.randint(24, 45)
        return pure(case("", scene, kind, rods, verts, frames))
    if kind == "grad":
        scene = rng.choice(("table", "table", "bands"))
        rods = log_int(1, 512 if scene == "bands" else 1500)
        return pure(case("", scene, kind, rods, max(verts, 96) if scene == "bands" else verts, rng.randint(2, 8)))
    if kind == "score":
        return pure(case("", "knot", kind, log_int(16, 800), rng.randint(96, 200), rng.randint(4, 20)))
    if kind == "autograd":
        return pure(case("", "diff", kind, log_int(4, 1024), rng.randint(24, 128), rng.randint(2, 16)))
    if kind == "sysid":
        return pure(case("", "diff", kind, log_int(2, 64), rng.randint(32, 96), rng.randint(2, 8),
                         pixels=rng.choice((64, 120, 200, 256))))
    return pure(case("", "table", kind, log_int(16, 2048), verts, 0, points=log_int(16, 512)))


def pure(c):
    return {k: v for k, v in c.items() if k != "name"}


# ------------------------------------------------------------------ inputs


def f32(a):
    return np.asarray(a, np.float32).astype(np.float64)


def offsets(n):
    return np.concatenate([[0], np.cumsum(n)]).astype(np.int64)


def open_curves(rng, nv, length):
    """One smooth nearly horizontal curve per rod, packed: unit tangents around a random heading
    with three sine modes, too weak to turn it back (so no curve crosses itself).  A small
    random bow in z, lowest point 2.2 mm above the ground (in soft contact with it)."""
    n, B = int(nv.max()), len(nv)
    s = np.arange(n - 1)[None, :] / (np.maximum(nv, 2) - 1)[:, None]
    head = rng.uniform(0, 2 * np.pi, B)
    amp = np.minimum(1.0, length)[:, None]
    lat = np.zeros((B, n - 1))
    for k in (1, 2, 3):
        a = rng.uniform(-1, 1, (B, 2)) * 0.15 / k
        lat += amp * (a[:, :1] * np.sin(2 * np.pi * k * s) + a[:, 1:] * np.cos(2 * np.pi * k * s))
    t = np.stack([np.cos(head)[:, None] - lat * np.sin(head)[:, None],
                  np.sin(head)[:, None] + lat * np.cos(head)[:, None], np.zeros((B, n - 1))], -1)
    t /= np.linalg.norm(t, axis=-1, keepdims=True)
    step = t * (length / (nv - 1))[:, None, None]
    x = np.concatenate([np.zeros((B, 1, 3)), np.cumsum(step, 1)], 1)
    keep = np.arange(n)[None, :] < nv[:, None]
    mean = (x * keep[..., None]).sum(1) / nv[:, None]
    x[..., :2] += (rng.uniform(-0.1, 0.1, (B, 2)) - mean[:, :2])[:, None]
    x[..., 2] = 0.0022 + 0.0004 * (1 + np.sin(2 * np.pi * np.arange(n)[None, :] / 40.0 + rng.uniform(0, 6, B)[:, None]))
    return x[keep]


def trefoil(s):
    return np.stack([np.sin(s) + 2 * np.sin(2 * s), np.cos(s) - 2 * np.cos(2 * s), -np.sin(3 * s)], -1)


def flat_knots(rng, B, n, drop, gap):
    """Trefoil-family curves of about 1 m lying flat: their three crossings' strands ``gap`` (of
    2r) apart in z.  drop > 0 opens the curve by that many vertices."""
    m = n + drop
    fine = trefoil(np.linspace(0, 2 * np.pi, 4097))
    arc = np.concatenate([[0.0], np.cumsum(np.linalg.norm(np.diff(fine[:, :2], axis=0), axis=1))])
    s = np.interp(np.linspace(0, arc[-1], m, endpoint=False), arc, np.linspace(0, 2 * np.pi, 4097))
    phase = rng.uniform(0, 2 * np.pi, B) if drop == 0 else np.full(B, 0.3)
    x = trefoil(s[None, :] + phase[:, None]) / arc[-1]
    # the strands of a crossing sit at z = +-zc: scale z so that they are gap * 2r apart
    p = trefoil(np.linspace(0, 2 * np.pi, 721)[:-1])
    d = np.linalg.norm(p[:, None, :2] - p[None, :, :2], axis=-1) + 9.0 * (np.abs(p[:, None, 2] - p[None, :, 2]) < 0.5)
    a, b = np.unravel_index(np.argmin(d), d.shape)
    x[..., 2] *= gap[:, None] * 2 * RADIUS * arc[-1] / abs(p[a, 2] - p[b, 2])
    ang = rng.uniform(0, 2 * np.pi, B)
    sc = rng.uniform(0.9, 1.1, (B, 2))
    xy = x[..., :2] * sc[:, None]
    c, sn = np.cos(ang)[:, None], np.sin(ang)[:, None]
    x[..., 0], x[..., 1] = c * xy[..., 0] - sn * xy[..., 1], sn * xy[..., 0] + c * xy[..., 1]
    return x[:, :n]


def tangled_pairs(rng, B, n, length):
    """Two ropes of n vertices side by side on the table, crossing over and under where sin = 0,
    there about 2r apart (in contact)."""
    s = np.linspace(0, 1, n)[None, :]
    th = 2 * np.pi * rng.uniform(1.2, 1.8, (B, 1)) * s + rng.uniform(0, 2 * np.pi, (B, 1))
    a, d = rng.uniform(0.03, 0.05, (B, 1)), RADIUS * rng.uniform(0.93, 1.15, (B, 1))
    y, z = a * np.sin(th), d * np.cos(th)
    wig = rng.uniform(-0.02, 0.02, (B, 1)) * np.sin(2 * np.pi * s + rng.uniform(0, 6, (B, 1)))
    along = (s - 0.5) * 0.85 * length + 0 * th
    ropes = [np.stack([along, wig + sg * y, 0.0026 + d + sg * z], -1) for sg in (1.0, -1.0)]
    x = np.concatenate(ropes, 1)
    ang = rng.uniform(0, 2 * np.pi, (B, 1))
    c, sn = np.cos(ang), np.sin(ang)
    x[..., 0], x[..., 1] = c * x[..., 0] - sn * x[..., 1], sn * x[..., 0] + c * x[..., 1]
    x[..., :2] += rng.uniform(-0.1, 0.1, (B, 1, 2))
    return x


def grip_frames(x, nv, k0, k1):
    """Gripper positions [B,2,3] at vertices (k0, k1) of each rod and capsule frames whose axis
    (column 2) is horizontal and normal to the rod."""
    vo, B = offsets(nv)[:-1], len(nv)
    pos, rot = np.zeros((B, 2, 3)), np.zeros((B, 2, 3, 3))
    for g, k in enumerate((k0, k1)):
        pos[:, g] = x[vo + k]
        t = x[vo + np.minimum(k + 1, nv - 1)] - x[vo + np.maximum(k - 1, 0)]
        ax = np.cross(t, [0.0, 0.0, 1.0])
        ax /= np.linalg.norm(ax, axis=1, keepdims=True)
        c0 = t / np.linalg.norm(t, axis=1, keepdims=True)
        rot[:, g] = np.stack([c0, np.cross(ax, c0), ax], -1)
    return pos, rot


def smooth_actions(rng, frames, B, amp_pos, amp_rot):
    """Per-frame increments [F,B,2,6] of poses that are sums of three sinusoids per degree of
    freedom, 0.2 to 2 Hz."""
    t = np.arange(frames + 1)[:, None, None, None] * DT
    out = np.zeros((frames + 1, B, 2, 6))
    scale = np.array([amp_pos] * 3 + [amp_rot] * 3) / 3.0
    for _ in range(3):
        w = 2 * np.pi * rng.uniform(0.2, 2.0, (B, 2, 6))
        out += rng.uniform(0, 1, (B, 2, 6)) * scale * np.sin(w * t + rng.uniform(0, 2 * np.pi, (B, 2, 6)))
    return np.diff(out, axis=0)


def problem(c, seed):
    """The workload of a case as an ``inputs.Problem`` (shapes, materials, scene, start state)."""
    rng = np.random.default_rng(seed)
    scene, B, n, F = c["scene"], c["rods"], c["verts"], max(1, c["frames"])
    nv = np.full(B, n, np.int64)
    idx = np.arange(B)
    mat = dict(K=np.full(B, 1e5), E=np.full(B, 1e4), G=np.zeros(B), plastic=np.zeros(B, bool), inext=np.zeros(B, bool),
               slim=np.zeros(B), sy=np.zeros(B), damping=np.ones(B))
    closed, grips, planes, boxes, pin, strand = False, 2, [[0.0, 0.0, 1.0, 0.0]], [], None, None
    rest = None
    if scene == "hang":
        x = np.zeros((B, n, 3))
        x[..., 0] = np.linspace(0.0, 1.0, n)
        x[..., 2] = 1.0
        x[..., :2] += rng.uniform(-0.2, 0.2, (B, 1, 2))
        x = x.reshape(-1, 3)
        mat.update(K=np.full(B, 1e6), E=10 ** rng.uniform(5.5, 6, B), G=np.full(B, 4e5), damping=np.zeros(B))
        grips, planes = 0, []
        pin = np.zeros(B * n, bool)
        pin[::n] = True
    elif scene == "ragged":
        nv = np.random.default_rng([B, n]).integers(16, n + 1, B)   # the batch's sizes belong to the case
        nv[: min(B, 2)] = (n, 16)[: min(B, 2)]
        # stiff rods are stepped, not differentiated: float32 positions do not resolve their strains' gradients
        E = 10 ** rng.uniform(4, 8 if c["mode"] == "step" else 6, B)
        x = open_curves(rng, nv, rng.uniform(0.3, 2.0, B))
        mat.update(K=E, E=E, G=0.4 * E, plastic=np.ones(B, bool), sy=rng.uniform(1, 20, B))
    elif scene == "table":
        x = open_curves(rng, nv, np.full(B, 1.0))
        k = idx % 3
        mat.update(K=np.where(k == 0, 0.0, 1e5), G=np.where(k == 0, 1e3, 0.0), inext=k == 0, plastic=k == 2,
                   sy=np.where(k == 2, 5.0, 0.0))
    elif scene == "diff":
        x = open_curves(rng, nv, np.full(B, 1.0))
        mat.update(plastic=idx >= B // 2, sy=np.where(idx >= B // 2, rng.uniform(1, 20, B), 0.0))
    elif scene == "bands":
        x = flat_knots(rng, B, n, 0, rng.uniform(0.9, 1.15, B))
        x[..., 2] += 0.1026 - x[..., 2].min(1, keepdims=True)
        rest = x.reshape(-1, 3)
        x = rest
        inext = idx % 2 == 0
        mat.update(K=np.where(inext, 0.0, 1e5), G=np.full(B, 1e3), inext=inext, slim=np.where(inext, 0.0, 0.2))
        closed, grips, boxes = True, 0, [[0.0, 0.0, 0.05, 0.15, 0.15, 0.05]]
    elif scene == "knot":
        one = flat_knots(rng, 1, n, 3, np.array([1.0]))
        one[..., 2] += 0.0026 - one[..., 2].min()
        x = np.repeat(one, B, 0).reshape(-1, 3)
    elif scene == "pair":
        x = tangled_pairs(rng, B, n // 2, 0.6).reshape(-1, 3)
        mat.update(K=np.zeros(B), E=np.full(B, 5e3), G=np.full(B, 1e3), inext=np.ones(B, bool))
        strand = np.zeros(B * n, bool)
        strand[n // 2::n] = True
    if scene == "pair":
        k0, k1 = np.full(B, n // 8), np.full(B, n - 1 - n // 8)
    else:
        k0, k1 = np.rint(0.25 * (nv - 1)).astype(int), np.rint(0.75 * (nv - 1)).astype(int)
    # rods with twist stiffness start twisted by up to a quarter turn along their length
    ne = nv - 1 + int(closed)
    along = (np.arange(ne.sum()) - np.repeat(offsets(ne)[:-1], ne)) / np.repeat(ne, ne)
    turn = rng.uniform(-1.5, 1.5, B) * (mat["G"] > 0)
    twist = np.repeat(turn, ne) * (np.sin(2 * np.pi * along) if closed else along)
    # in motion: every rod translating in the plane (hanging rods at rest), its grippers carrying
    # it along and lifting it
    d = rng.uniform(0, 2 * np.pi, B)
    u = np.stack([np.cos(d), np.sin(d), 0 * d], -1) * rng.uniform(0.3, 0.6, (B, 1)) * (scene != "hang")
    vel = np.repeat(u, nv, 0)
    pos, rot, acts = np.zeros((B, 2, 3)), np.tile(np.eye(3), (B, 2, 1, 1)), np.zeros((F, B, 2, 6))
    if grips:
        pos, rot = grip_frames(f32(x), nv, k0, k1)
        acts[..., :3] = DT * (u + np.array([0.0, 0.0, 1.0]) * rng.uniform(0.1, 0.2, (B, 1)))[None, :, None]
        acts += smooth_actions(rng, F, 1 if scene == "knot" else B, 0.005, 0.05)
        if scene == "knot":
            acts += smooth_actions(rng, F, B, 0.05, 0.05)
    return inputs.Problem(
        name=scene, n_verts=nv, closed=np.full(B, closed), x_rest=f32(x), density=np.full(B, 1000.0), radius=f32(np.full(B, RADIUS)),
        K=f32(mat["K"]), E=f32(mat["E"]), G=f32(mat["G"]), inextensible=mat["inext"], strain_limit=f32(mat["slim"]),
        plastic=mat["plastic"], yield_curv=f32(mat["sy"]), creep_rate=np.ones(B), damping=f32(mat["damping"]),
        pinned=np.zeros(len(x), bool) if pin is None else pin, n_grippers=np.full(B, grips), grip_pos=f32(pos),
        grip_rot=f32(rot), actions=f32(acts), frames=F, grip_radius=GRIP_R, grip_half_len=GRIP_HL,
        planes=np.array(planes).reshape(-1, 4), boxes=np.array(boxes).reshape(-1, 6), dt=DT, n_iter=N_ITER,
        mu_self=MU_SELF, mu_rigid=MU_RIGID, eps_soft=EPS, contact_margin=MARGIN, gravity=GRAVITY,
        self_contact=scene in ("table", "bands", "knot", "pair"), v0=f32(vel), strand_start=strand,
        theta0=f32(twist))


def extras(c, prob, seed):
    """Host arrays a case needs beside its rods: loss targets, point sets, cameras, masks."""
    rng = np.random.default_rng(seed + 777)
    B, V = prob.batch, len(prob.x_rest)
    out = {}
    if c["mode"] in ("grad", "autograd"):
        out["target"] = f32(prob.x_rest + rng.normal(size=(B, 3)).repeat(prob.n_verts, 0) * 0.05 + rng.normal(size=(V, 3)) * 0.01)
    if c["mode"] == "losses":
        m = c["points"]
        vo = offsets(prob.n_verts)
        pick = vo[:-1, None] + rng.integers(0, prob.n_verts[0], (B, m))
        out["points"] = f32(prob.x_rest[pick] + rng.normal(size=(B, m, 3)) * 0.02)
        out["post"] = f32(np.concatenate([rng.uniform(-0.3, 0.3, (B, 2)), np.zeros((B, 2))], 1))
        out["repel"] = f32(np.tile([0.05, 4.0, 0.0, 0.0], (B, 1)))
        out["weight"] = f32(rng.uniform(0.5, 1.5, B))
    if c["mode"] == "sysid":
        out["cams"] = cameras(c["pixels"])
        # binary masks of each rod's start curve moved sideways: pixels within 1.5 px of it
        out["masks"] = masks_of(prob, out["cams"], c["pixels"], rng.uniform(-0.03, 0.03, (B, 3)) * [1, 1, 0])
    return out


def cameras(px):
    """Two pinhole cameras over the table: from above (1.6 m) and from the side at 50 degrees."""
    f, c = px / 256.0, px / 2.0
    down = np.concatenate([[160 * f, 160 * f, c, c], np.diag([1.0, -1.0, -1.0]).reshape(9), [0.0, 0.0, 1.6]])
    a = math.radians(50.0)
    R = np.array([[1.0, 0.0, 0.0], [0.0, -math.sin(a), -math.cos(a)], [0.0, math.cos(a), -math.sin(a)]])
    eye = np.array([0.0, -math.cos(a), math.sin(a)]) * 1.8
    return f32(np.stack([down, np.concatenate([[150 * f, 150 * f, c, c], R.reshape(9), -R @ eye])]))


def masks_of(prob, cams, px, shift):
    B, n = prob.batch, int(prob.n_verts[0])
    x = prob.x_rest.reshape(B, n, 3) + shift[:, None]
    fine = np.concatenate([x[:, :-1] * (1 - w) + x[:, 1:] * w for w in (0.0, 0.25, 0.5, 0.75)], 1)
    out = np.zeros((B, len(cams), px, px), np.uint8)
    for k, cam in enumerate(cams):
        p = fine @ cam[4:13].reshape(3, 3).T + cam[13:16]
        u = np.floor(cam[0] * p[..., 0] / p[..., 2] + cam[2]).astype(int)
        v = np.floor(cam[1] * p[..., 1] / p[..., 2] + cam[3]).astype(int)
        ok = (u >= 0) & (u < px) & (v >= 0) & (v < px)
        b = np.broadcast_to(np.arange(B)[:, None], u.shape)
        out[b[ok], k, v[ok], u[ok]] = 1
    return out


def prepare(case, seed):
    c, prob = case, problem(case, seed)
    dev = torch.device("cuda")

    def up(a, dtype=torch.float32):
        return torch.as_tensor(np.ascontiguousarray(a), device=dev).to(dtype)

    def up4(a):
        return up(np.concatenate([a, np.zeros((*a.shape[:-1], 1))], -1))

    sim = dlo.DloSim(prob)
    ex = extras(c, prob, seed)
    st = dict(case=c, sim=sim, x0=up4(prob.x0), v0=up4(prob.v0), th0=up(prob.theta0), acts=up(prob.actions))
    st["ex"] = {k: up(v, torch.uint8) if k == "masks" else up4(v) if k in ("target", "points") else up(v) for k, v in ex.items()}
    if c["mode"] in ("step", "score"):
        st["traj"] = torch.empty(c["frames"], sim.V, 4, device=dev)
    if c["mode"] == "score":
        st["ex"]["repel"] = up(np.tile([0.05, 4.0, 0.0, 0.0], (prob.batch, 1)))
    return st


# ------------------------------------------------------------------ the passes


def run(st):
    c, sim, ex, F = st["case"], st["sim"], st["ex"], st["case"]["frames"]
    mode = c["mode"]
    if mode == "losses":
        out = {}
        for name, kind, aux in (("chamfer", dlo.LOSS_CHAMFER, ex["points"]), ("crossing", dlo.LOSS_CROSSING, None),
                                ("repulsion", dlo.LOSS_REPULSION, ex["repel"]), ("winding", dlo.LOSS_WINDING, ex["post"]),
                                ("mindist", dlo.LOSS_MINDIST, ex["post"])):
            out[name] = list(sim.loss(kind, st["x0"], aux, ex["weight"]))
        return out
    if mode == "autograd":  # an optimiser's step through the differentiable rollout
        x0, acts = st["x0"].requires_grad_(True), st["acts"].requires_grad_(True)
        v0 = st["v0"].requires_grad_(True)
        x0.grad = v0.grad = acts.grad = None
        x, v, th = dlo.rollout(sim, x0, v0, st["th0"], acts)
        loss = ((x[:, :3] - ex["target"][:, :3]) ** 2).mean()
        loss.backward()
        return dict(loss=loss.detach(), x=x.detach(), x0=x0.grad, v0=v0.grad, actions=acts.grad)
    sim.set_state(st["x0"], st["v0"], st["th0"])
    if mode in ("step", "score"):
        sim.step(st["acts"], F, x_frames=st["traj"])
        if mode == "score":  # every candidate's trajectory and its two Unknotting terms
            x = st["traj"][F - 1]
            crossing = sim.loss(dlo.LOSS_CROSSING, x, grad=False)[0]
            return dict(traj=st["traj"], crossing=crossing, repulsion=sim.loss(dlo.LOSS_REPULSION, x, ex["repel"], grad=False)[0])
        x, v, th = sim.get_state()
        return dict(traj=st["traj"], x=x, theta=th)  # what planners and learners consume: the motion, frame by frame
    sim.begin_rollout(F)
    sim.step(st["acts"], F)
    x, v, th = sim.get_state()
    if mode == "grad":  # gradient of the mean squared distance to a target shape
        q, gx = sim.loss(dlo.LOSS_TARGET, x, ex["target"])
        g = sim.backward(gx, want=("actions", "x0", "v0"))
        return dict(x=x, loss=q, x0=g["x0"], v0=g["v0"], actions=g["actions"])
    # sysid: silhouettes of the final state in every camera against the observed masks
    q, gx, _ = sim.silhouette(x, ex["cams"], ex["masks"], SIL_TAU)
    g = sim.backward(gx, want=("material", "x0", "v0"))
    return dict(x=x, loss=q, gx=gx, x0=g["x0"], v0=g["v0"], material=g["material"])


# ------------------------------------------------------------------ what a pass cannot do without


def work(case):
    """Bytes: the state, actions and auxiliary inputs read once, the outputs written once.
    Operations per vertex and substep: the package's own counts of the element functions
    (tests/test_flop_count.py), 912 forward and 3650 for a backward with its recomputation; a
    loss pass counts its pairs."""
    c = case
    nv = c["verts"] if c["scene"] != "ragged" else (16 + c["verts"]) / 2
    V, F, B = c["rods"] * nv, c["frames"], c["rods"]
    sub = 5.0 if c["scene"] != "ragged" else 60.0
    if c["scene"] == "table":  # extensible rope of 1 m: 2 sqrt(K / rho) / l, two thirds of the rods
        sub = max(5.0, math.ceil(DT * 20.0 * (c["verts"] - 1)))
    if c["scene"] == "hang":  # 2 sqrt(K / rho) / l
        sub = max(5.0, math.ceil(DT * 63.3 * (c["verts"] - 1)))
    state = 16.0 * V * 3 + 4 * V
    acts = 48.0 * B * F * (c["scene"] not in ("hang", "bands"))
    if c["mode"] == "losses":
        m = c["points"]
        pairs = B * (2.0 * nv * m * 9 + nv * nv * (150 + 60))
        return dict(bytes=16.0 * B * (nv + m + 3) + 5 * 16.0 * V, flops=pairs)
    fwd = 912.0 * V * F * sub
    if c["mode"] in ("step", "score"):
        return dict(bytes=2 * state + acts + 16.0 * V * F, flops=fwd + (200.0 * B * nv * nv if c["mode"] == "score" else 0))
    px = c.get("pixels", 0)
    return dict(bytes=4 * state + 2 * acts + 2.0 * B * px * px, flops=fwd + 3650.0 * V * F * sub + 2.0 * B * px * px * 40)


# ------------------------------------------------------------------ the same in 64 bits


def dot(a, b):
    return (a * b).sum(-1)


def unit(a):
    return a / dot(a, a).sqrt()[..., None]


def cross(a, b):
    return torch.linalg.cross(a, b)


def transport(a, b, d):
    k = cross(a, b)
    return dot(a, b)[..., None] * d + cross(k, d) + (dot(k, d) / (1.0 + dot(a, b)))[..., None] * k


def adapt(d, t):
    return unit(d - dot(d, t)[..., None] * t)


def angle(u, w, axis):
    return torch.atan2(dot(cross(u, w), axis), dot(u, w))


def expm(p):
    t2 = dot(p, p)[..., None, None]
    t = torch.where(t2 > 1e-20, t2, torch.ones_like(t2)).sqrt()
    a = torch.where(t2 > 1e-20, torch.sin(t) / t, torch.ones_like(t))
    b = torch.where(t2 > 1e-20, (1 - torch.cos(t)) / (t * t), torch.full_like(t, 0.5))
    z = torch.zeros_like(p[..., 0])
    k = torch.stack([torch.stack([z, -p[..., 2], p[..., 1]], -1), torch.stack([p[..., 2], z, -p[..., 0]], -1),
                     torch.stack([-p[..., 1], p[..., 0], z], -1)], -2)
    return torch.eye(3, dtype=p.dtype, device=p.device) + a * k + b * (k @ k)


def closest(p1, q1, p2, q2):
    """Clamped closest points of two segments (Ericson, Real-Time Collision Detection, 5.1.9)."""
    d1, d2, r = q1 - p1, q2 - p2, p1 - p2
    a, e, f, c, b = dot(d1, d1), dot(d2, d2), dot(d2, r), dot(d1, r), dot(d1, d2)
    den = a * e - b * b
    par = den <= 1e-6 * a * e
    s = torch.where(par, torch.zeros_like(a), ((b * f - c * e) / torch.where(par, torch.ones_like(den), den)).clamp(0, 1))
    u = (b * s + f) / e
    s = torch.where(u < 0, (-c / a).clamp(0, 1), torch.where(u > 1, ((b - c) / a).clamp(0, 1), s))
    return s, u.clamp(0, 1)


class Rods:
    """The rods of a problem packed, in float64, and their motion (any device)."""

    def __init__(self, p, dev):
        self.p, self.dev = p, dev
        D = lambda a: torch.as_tensor(np.asarray(a, np.float64), device=dev)  # noqa: E731
        L = lambda a: torch.as_tensor(np.asarray(a, np.int64), device=dev)  # noqa: E731
        nv, B = p.n_verts.astype(np.int64), p.batch
        ne = p.n_edges.astype(np.int64)
        vo, eo = p.vert_off, p.edge_off
        er = np.repeat(np.arange(B), ne)
        ej = np.arange(eo[-1]) - eo[er]
        ea = vo[er] + ej
        eb = vo[er] + (ej + 1) % nv[er]
        real = ~(p.strand_start[eb] & (ej + 1 < nv[er]))
        # hinges: edge pairs (a, b) meeting at a vertex
        hb = np.arange(eo[-1])[(ej > 0) | p.closed[er]]
        ha = np.where(ej[hb] > 0, hb - 1, eo[er[hb]] + ne[er[hb]] - 1)
        ok = real[ha] & real[hb]
        ha, hb = ha[ok], hb[ok]
        self.V, self.E, self.B = int(vo[-1]), int(eo[-1]), B
        self.ea, self.eb, self.er, self.ej, self.vr = L(ea), L(eb), L(er), L(ej), L(np.repeat(np.arange(B), nv))
        self.ha, self.hb, self.hr = L(ha), L(hb), L(er[hb])
        self.real, self.ne, self.nv, self.eo, self.vo = torch.as_tensor(real, device=dev), ne, nv, eo, vo
        self.closed = torch.as_tensor(p.closed, device=dev)
        xr = p.x_rest
        bar = np.linalg.norm(xr[eb] - xr[ea], axis=1) * real
        r, rho = p.radius, p.density
        A = np.pi * r * r
        lv = np.zeros(self.V)
        np.add.at(lv, ea, 0.5 * bar)
        np.add.at(lv, eb, 0.5 * bar)
        mass = rho[np.repeat(np.arange(B), nv)] * A[np.repeat(np.arange(B), nv)] * lv
        kind, off = np.where(p.pinned, 1, 0), np.zeros((self.V, 3))
        if p.n_grippers.any():
            rid = np.repeat(np.arange(B), nv)
            for g in range(2):
                pos, rot = p.grip_pos[:, g], p.grip_rot[:, g]
                ax = rot[:, :, 2]
                d = xr - pos[rid]
                s = np.clip((d * ax[rid]).sum(1), -p.grip_half_len, p.grip_half_len)
                sd = np.linalg.norm(d - s[:, None] * ax[rid], axis=1) - p.grip_radius
                near = np.array([vo[b] + np.argmin(sd[vo[b]:vo[b + 1]]) for b in range(B)])
                grab = sd < r[rid]
                grab[near] = True
                grab &= kind == 0
                kind[grab] = 2 + g
                off[grab] = np.einsum("vi,vij->vj", d[grab], rot[rid[grab]])
        self.kind, self.off, self.w = L(kind), D(off), D(np.where(kind == 0, 1.0 / mass, 0.0))
        self.bar, self.A, self.r = D(bar), D(A), D(r)
        self.lbar = 0.5 * (self.bar[self.ha] + self.bar[self.hb])
        inertia = 0.5 * rho[er] * A[er] * r[er] ** 2 * np.where(real, bar, 1.0)
        self.invI = D(np.where(real & (p.G[er] > 0), 1.0 / inertia, 0.0))
        lmin = np.array([bar[eo[b]:eo[b + 1]][real[eo[b]:eo[b + 1]]].min() for b in range(B)])
        ws = np.where(p.inextensible, 0.0, 2 * np.sqrt(p.K / rho) / lmin)
        om = np.maximum(2 * r * np.sqrt(p.E / rho) / lmin**2, np.maximum(ws, 2 * np.sqrt(p.G / rho) / lmin))
        self.dt = float(np.float32(p.dt))
        self.nsub = np.maximum(p.substeps_min, np.ceil(self.dt * om)).astype(int)
        self.h = D(self.dt / self.nsub)
        self.excl = L(np.maximum(1, np.ceil(2 * r / lmin)))
        self.mats = dict(K=D(p.K), E=D(p.E), G=D(p.G), sy=D(p.yield_curv), cd=D(p.damping))
        self.inext, self.plastic = torch.as_tensor(p.inextensible, device=dev), torch.as_tensor(p.plastic, device=dev)
        self.slim = D(p.strain_limit)
        self.lenc = self.inext | (self.slim > 0)
        colour = np.where(p.closed[er] & (ne[er] % 2 == 1) & (ej == ne[er] - 1), 2, ej % 2)
        act = self.lenc.cpu().numpy()[er] & real
        self.colours = [L(np.nonzero(act & (colour == k))[0]) for k in range(3)]
        self.colours = [k for k in self.colours if len(k)]
        self.eps = float(np.float32(p.eps_soft)) * self.r
        f = lambda v: float(np.float32(v))  # noqa: E731
        self.mu_s, self.mu_r, self.g = f(p.mu_self), f(p.mu_rigid), f(p.gravity)
        self.gr, self.ghl = f(p.grip_radius), f(p.grip_half_len)
        self.gp, self.gR = D(p.grip_pos), D(p.grip_rot)
        self.kb_rest = torch.zeros(self.E, 2, dtype=torch.float64, device=dev)   # at each hinge's second edge
        self.kb_rest[:, 1] = torch.where(self.closed, 2 * torch.tan(math.pi / D(ne)), torch.zeros_like(self.r))[self.er]
        t, d1 = self.frames(D(xr))
        self.mbar = self.twist(t, d1)

    def edge(self, x):
        return x[self.eb] - x[self.ea]

    def frames(self, x):
        """Adapted reference frames by space-parallel transport (loops: holonomy spread)."""
        e = self.edge(x)
        e = torch.where(self.real[:, None], e, torch.tensor([0.0, 0, 1], dtype=e.dtype, device=e.device))
        t = unit(e)
        ez, ex = (torch.tensor(a, dtype=t.dtype, device=t.device).expand(t.shape) for a in ([0.0, 0, 1], [1.0, 0, 0]))
        fresh = adapt(torch.where((t[:, 2].abs() < 0.9)[:, None], ez, ex), torch.where(self.real[:, None], t, ez + ex))
        cols, last_d = [], None
        eo, ne = torch.as_tensor(self.eo[:-1], device=x.device), torch.as_tensor(self.ne, device=x.device)
        for j in range(int(self.ne.max())):
            rows = torch.nonzero(ne > j)[:, 0]
            k = eo[rows] + j
            dj = fresh[k]
            if j:
                dj = torch.where((self.real[k] & self.real[k - 1])[:, None], adapt(transport(t[k - 1], t[k], last_d[rows]), t[k]), dj)
                dj = torch.where(self.real[k][:, None], dj, ex[k])
            last_d = torch.zeros(self.B, 3, dtype=t.dtype, device=t.device).index_copy(0, rows, dj)
            cols.append((k, dj))
        k = torch.cat([c[0] for c in cols])
        d1 = torch.zeros_like(t).index_copy(0, k, torch.cat([c[1] for c in cols]))
        if bool(self.closed.any()):
            last = eo + ne - 1
            u = adapt(transport(t[last], t[eo], d1[last]), t[eo])
            psi = angle(d1[eo], u, t[eo]) * self.closed
            phi = -(psi / ne)[self.er] * self.ej
            d1 = torch.cos(phi)[:, None] * d1 + torch.sin(phi)[:, None] * cross(t, d1)
        return t, d1

    def twist(self, t, d1):
        a, b = self.ha, self.hb
        return torch.zeros(self.E, dtype=t.dtype, device=t.device).index_copy(0, b, angle(transport(t[a], t[b], d1[a]), d1[b], t[b]))

    def start(self, x0, v0, th0):
        """(x, v, theta, omega, base tangent, base director, rest curvature, reference twist, gripper p, R)"""
        t, d1 = self.frames(x0)
        z = torch.zeros_like(th0)
        return [x0, v0, th0, z, t, d1, self.kb_rest, self.twist(t, d1).detach(), self.gp, self.gR]

    def strains(self, x, th, tb, db, mref):
        """Tangents, reference directors, lengths, and each hinge's curvature and reference twist."""
        e = torch.where(self.real[:, None], self.edge(x), torch.ones_like(tb))
        ell = dot(e, e).sqrt()
        t = torch.where(self.real[:, None], e / ell[:, None], tb)
        d = torch.where(self.real[:, None], adapt(transport(tb, t, db), t), db)
        d2 = cross(t, d)
        c, s = torch.cos(th)[:, None], torch.sin(th)[:, None]
        m1, m2 = c * d + s * d2, c * d2 - s * d
        a, b = self.ha, self.hb
        kv = 2.0 * cross(t[a], t[b]) / (1.0 + dot(t[a], t[b]))[:, None]
        kap = 0.5 * torch.stack([dot(kv, m2[a] + m2[b]), dot(kv, m1[a] + m1[b])], -1)
        ang = angle(transport(t[a], t[b], d[a]), d[b], t[b])
        turns = torch.round((ang - mref[b]).detach() / (2 * math.pi))
        return t, d, ell, kap, ang - 2 * math.pi * turns

    def gradient(self, x, th, tb, db, kbn, mref, mats, graph):
        """(dU/dx, dU/dtheta) of the stretching, bending and twisting energies."""
        t, d, ell, kap, new = self.strains(x, th, tb, db, mref)
        A, r = self.A, self.r
        kA = torch.where(self.inext, torch.zeros_like(A), mats["K"] * A)[self.er] * self.real
        Bm, beta = (mats["E"] * A * r * r / 4)[self.hr], (mats["G"] * A * r * r / 2)[self.hr]
        bar = torch.where(self.real, self.bar, torch.ones_like(self.bar))
        m = th[self.hb] - th[self.ha] + new
        U = (0.5 * kA * (ell / bar - 1) ** 2 * bar).sum() + (0.5 * Bm / self.lbar * dot(kap - kbn, kap - kbn)).sum() \
            + (0.5 * beta / self.lbar * (m - self.mbar[self.hb]) ** 2).sum()
        return torch.autograd.grad(U, [x, th], create_graph=graph)

    def substep(self, S, act, mats, nsub, sb, live, pairs, graph):
        """One substep of the rods ``live`` ([B] bool; the others keep their state); ``graph``: its
        outputs can be differentiated with respect to S, act and mats."""
        x, v, th, om, tb, db, kb, mref, gp, gR = S
        R = self
        c0, c1 = sb / nsub, (sb + 1) / nsub
        with torch.enable_grad():
            if not graph:
                x, th = x.detach().requires_grad_(True), th.detach().requires_grad_(True)
            t, d, ell, kap, new = R.strains(x, th, tb, db, mref)
            el = kap - kb[R.hb]
            n = dot(el, el).clamp(min=1e-300).sqrt()
            yl = (R.plastic[R.hr] & (n > mats["sy"][R.hr] * R.lbar))[:, None]
            kbn = kb[R.hb] + torch.where(yl, (1 - mats["sy"][R.hr] * R.lbar / n)[:, None] * el, torch.zeros_like(el))
            # the force is the energy's gradient at a fixed rest curvature, taken on aliases of x
            # and theta that the rest curvature does not depend on
            gx, gth = R.gradient(x.view_as(x), th.view_as(th), tb, db, kbn if graph else kbn.detach(), mref, mats, graph)
        if not graph:
            x, th, t, d, new, kbn = (a.detach() for a in (x, th, t, d, new, kbn))
        h = R.h[R.vr][:, None]
        v1 = v + h * (-R.w[:, None] * gx + torch.tensor([0.0, 0, -R.g], dtype=x.dtype, device=x.device) - mats["cd"][R.vr][:, None] * v)
        v2 = R.rigid(x, v1, gp, gR, act, c0, self.dt)
        free = (R.kind == 0)[:, None]
        dd = torch.where(free, h * v2, torch.zeros_like(v2))
        target = None
        if bool((R.kind >= 2).any()):
            g = (R.kind - 2).clamp(min=0)
            p1 = gp + c1[:, None, None] * act[..., :3]
            R1 = expm(c1[:, None, None] * act[..., 3:]) @ gR
            target = p1[R.vr, g] + (R1[R.vr, g] @ R.off[..., None])[..., 0]
            dd = torch.where((R.kind >= 2)[:, None], target - x, dd)
        he = R.h[R.er]
        cde = mats["cd"][R.er]
        om1 = om + he * (-gth * R.invI - cde * om)
        th1 = th + he * om1
        first = None
        if R.colours or pairs is not None:
            lim = R.slim[R.er]
            for it in range(N_ITER):
                for k in R.colours:
                    a, b = R.ea[k], R.eb[k]
                    e = x[b] - x[a] + dd[b] - dd[a]
                    l = dot(e, e).sqrt()
                    lo, hi = (1 - lim[k]) * R.bar[k], (1 + lim[k]) * R.bar[k]
                    aim = torch.minimum(torch.maximum(l, lo), hi)
                    ws = R.w[a] + R.w[b]
                    lam = torch.where(ws > 0, (l - aim) / torch.where(ws > 0, ws, torch.ones_like(ws)), torch.zeros_like(l)) / l
                    dd = dd.index_add(0, a, (lam * R.w[a])[:, None] * e).index_add(0, b, (-lam * R.w[b])[:, None] * e)
                if pairs is not None:
                    dd, got = R.sweep(x, dd, pairs)
                    first = got if it == 0 else first
        vn = dd / h
        if first is not None:
            vn = R.friction(vn, pairs, first)
        xn = x + dd if target is None else torch.where((R.kind >= 2)[:, None], target, x + dd)
        kb1, mr1 = kb.index_copy(0, R.hb, kbn), mref.index_copy(0, R.hb, new)
        lv, le = live[R.vr][:, None], live[R.er]
        pick = lambda m, a, b: a if bool(live.all()) else torch.where(m, a, b)  # noqa: E731
        return [pick(lv, xn, x), pick(lv, vn, v), pick(le, th1, th), pick(le, om1, om), pick(le[:, None], t, tb), pick(le[:, None], d, db),
                pick(le[:, None], kb1, kb), pick(le, mr1, mref), gp, gR]

    def rigid(self, x, v, gp, gR, act, c0, dt):
        R, p = self, self.p
        r, eps = R.r[R.vr], R.eps[R.vr]

        def respond(v, sdf, n, vr):
            f = torch.exp(((r - sdf) / eps).clamp(max=0.0))
            on = (f > 0.1)[:, None]
            rel = v - vr
            vn = dot(rel, n)
            vt = rel - vn[:, None] * n
            vn2 = vn.clamp(min=0.0)
            s2 = dot(vt, vt)
            sp = torch.where(s2 > 1e-24, s2, torch.ones_like(s2)).sqrt()
            sc = torch.where(s2 > 1e-24, (1 - R.mu_r * (vn2 - vn) / sp).clamp(min=0.0), torch.ones_like(s2))
            return torch.where(on, v + f[:, None] * (vn2[:, None] * n + sc[:, None] * vt - rel), v)

        zero = torch.zeros_like(v)
        for pl in p.planes:
            n = torch.as_tensor(pl[:3], device=x.device).expand(x.shape)
            v = respond(v, dot(x, n) - pl[3], n, zero)
        for bx in p.boxes:
            c, hl = (torch.as_tensor(np.asarray(f32(a)), device=x.device) for a in (bx[:3], bx[3:]))
            q = (x - c).abs() - hl
            o = q.clamp(min=0.0)
            o2 = dot(o, o)
            out = o2 > 0
            ol = torch.where(out, o2, torch.ones_like(o2)).sqrt()
            sg = torch.where(x - c >= 0, 1.0, -1.0).to(x.dtype)
            k = torch.nn.functional.one_hot(q.argmax(-1), 3).to(x.dtype)
            v = respond(v, torch.where(out, ol, q.max(-1).values), sg * torch.where(out[:, None], o / ol[:, None], k), zero)
        if p.n_grippers.any():
            for g in range(2):
                pos = (gp[:, g] + c0[:, None] * act[:, g, :3])[R.vr]
                ax = (expm(c0[:, None] * act[:, g, 3:]) @ gR[:, g])[:, :, 2][R.vr]
                s = (dot(x - pos, ax) / dot(ax, ax)).clamp(-R.ghl, R.ghl)
                dv = x - pos - s[:, None] * ax
                d2 = dot(dv, dv)
                ok = d2 > 0
                d = torch.where(ok, d2, torch.ones_like(d2)).sqrt()
                vr = (act[:, g, :3] / dt)[R.vr] + cross((act[:, g, 3:] / dt)[R.vr], x - pos)
                v = respond(v, torch.where(ok, d - R.gr, torch.full_like(d, -R.gr)), torch.where(ok[:, None], dv / d[:, None], zero), vr)
        return v

    def candidates(self, x):
        """Edge pairs (a < b) of each rod outside the exclusion window and closer than the margin."""
        far = float(np.float32(2 * RADIUS + MARGIN * RADIUS))
        pa, pb = x[self.ea], x[self.eb]
        mid, half = 0.5 * (pa + pb), 0.5 * dot(pb - pa, pb - pa).sqrt()
        breaks = torch.cumsum((~self.real).long(), 0)
        A, Bq = [], []
        for n in np.unique(self.ne):
            rods = np.nonzero(self.ne == n)[0]
            for part in np.array_split(rods, max(1, len(rods) * n * n // 20_000_000)):
                k = torch.as_tensor(self.eo[part][:, None] + np.arange(n)[None, :], device=x.device)
                m, hf = mid[k], half[k]
                near = torch.cdist(m, m, compute_mode="donot_use_mm_for_euclid_dist") < far + hf[:, :, None] + hf[:, None, :]
                i, a, b = torch.nonzero(near.triu(1), as_tuple=True)
                A.append(k[i, a])
                Bq.append(k[i, b])
        a, b = torch.cat(A), torch.cat(Bq)
        sep = b - a
        ne = torch.as_tensor(self.ne, device=x.device)[self.er[a]]
        sep = torch.where(self.closed[self.er[a]], torch.minimum(sep, ne - sep), sep)
        ok = ((sep > self.excl[self.er[a]]) | (breaks[b] != breaks[a])) & self.real[a] & self.real[b]
        a, b = a[ok], b[ok]
        s, u = closest(pa[a], pb[a], pa[b], pb[b])
        dd = pa[a] + s[:, None] * (pb[a] - pa[a]) - pa[b] - u[:, None] * (pb[b] - pa[b])
        ok = dot(dd, dd).sqrt() < far
        a, b = a[ok], b[ok]
        if not len(a):
            return None
        return torch.stack([self.ea[a], self.eb[a], self.ea[b], self.eb[b]])

    def sweep(self, x, dd, pairs):
        P = x[pairs] + dd[pairs]
        w = self.w[pairs]
        s, u = closest(*P)
        wt = torch.stack([1 - s, s, 1 - u, u])
        sg = torch.tensor([1.0, 1, -1, -1], dtype=x.dtype, device=x.device)[:, None]
        dv = ((wt * sg)[..., None] * P).sum(0)
        W = (w * wt * wt).sum(0)
        d2 = dot(dv, dv)
        ok = (d2 > 1e-24) & (W > 0)
        dist = torch.where(ok, d2, torch.ones_like(d2)).sqrt()
        dep = 2 * self.r[self.vr[pairs[0]]] - dist
        on = ok & (dep > 0)
        n = dv / dist[:, None]
        k = torch.where(on, dep / torch.where(on, W, torch.ones_like(W)), torch.zeros_like(W))
        mv = (k * w * wt * sg)[..., None] * n
        return dd.index_add(0, pairs.reshape(-1), mv.reshape(-1, 3)), (on, n, dep, wt * sg, W)

    def friction(self, v, pairs, first):
        on, n, dep, ws, W = first
        rel = (ws[..., None] * v[pairs]).sum(0)
        vt = rel - dot(rel, n)[:, None] * n
        s2 = dot(vt, vt)
        on = on & (s2 > 1e-24)
        sp = torch.where(on, s2, torch.ones_like(s2)).sqrt()
        h = self.h[self.vr[pairs[0]]]
        k = torch.where(on, (self.mu_s * dep / (h * sp)).clamp(max=1.0) / torch.where(on, W, torch.ones_like(W)), torch.zeros_like(W))
        mv = -(k * self.w[pairs] * ws)[..., None] * vt
        return v.index_add(0, pairs.reshape(-1), mv.reshape(-1, 3))

    def advance(self, S, act):
        S = list(S)
        S[8] = S[8] + act[..., :3]
        S[9] = expm(act[..., 3:]) @ S[9]
        return S

    def plan(self):
        """(substep index, live rods) of one frame."""
        top = int(self.nsub.max())
        return [(k, torch.as_tensor(self.nsub > k, device=self.dev)) for k in range(top)]

    def rollout(self, S, acts, mats, keep=False):
        nsub = torch.as_tensor(self.nsub, dtype=torch.float64, device=self.dev)
        tape, traj = [], []
        for f in range(acts.shape[0]):
            pairs = self.candidates(S[0].detach()) if self.p.self_contact else None
            for sb, live in self.plan():
                if keep:
                    tape.append((S, f, sb, live, pairs))
                S = self.substep(S, acts[f], mats, nsub, sb, live, pairs, False)
            S = self.advance(S, acts[f])
            traj.append(S[0])
        return S, traj, tape

    def reverse(self, tape, acts, mats, gx):
        """Gradients of sum(gx * x_T): (the start state's, the actions', the material's)."""
        nsub = torch.as_tensor(self.nsub, dtype=torch.float64, device=self.dev)
        cot = [gx] + [None] * 9
        ga = torch.zeros_like(acts)
        gm = {k: torch.zeros_like(m) for k, m in mats.items()}
        last = max(int(self.nsub.max()) - 1, 0)
        for S, f, sb, live, pairs in reversed(tape):
            S = [a.detach().requires_grad_(True) for a in S]
            act = acts[f].detach().requires_grad_(True)
            ms = {k: m.detach().requires_grad_(True) for k, m in mats.items()}
            with torch.enable_grad():
                out = self.substep(S, act, ms, nsub, sb, live, pairs, True)
                if sb == last:
                    out = self.advance(out, act)
                got = [(o, c) for o, c in zip(out, cot) if c is not None and o.requires_grad]
                g = torch.autograd.grad([o for o, _ in got], S + [act] + list(ms.values()), [c for _, c in got], allow_unused=True)
            cot = [a if a is not None else torch.zeros_like(s) for a, s in zip(g[:10], S)]
            ga[f] += g[10] if g[10] is not None else 0.0
            for k, m in zip(gm, g[11:]):
                gm[k] += m if m is not None else 0.0
        return cot, ga, gm

    def reverse_start(self, x0, cot):
        """The start positions' gradient, the frames rebuilt from them included."""
        x = x0.detach().requires_grad_(True)
        with torch.enable_grad():
            t, d = self.frames(x)
            g = torch.autograd.grad([t, d], [x], [cot[4], cot[5]])[0]
        return cot[0] + g


def exact(case, seed):
    c = case
    B, n, F = c["rods"], c["verts"], c["frames"]
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    prob = problem(c, seed)
    ex = extras(c, prob, seed)
    D = lambda a: torch.as_tensor(np.asarray(a, np.float64), device=dev)  # noqa: E731
    four = lambda a: torch.cat([a, torch.zeros_like(a[..., :1])], -1)  # noqa: E731
    if c["mode"] == "losses":
        return exact_losses(prob, {k: D(v) for k, v in ex.items()}, D(prob.x0))
    R = Rods(prob, dev)
    subs = int(R.nsub.max()) * F
    grad = c["mode"] in ("grad", "autograd", "sysid")
    if subs * (60 if grad else 12) > 20_000:
        return None
    x0, acts = D(prob.x0), D(prob.actions)[:F]
    with torch.no_grad():
        S, traj, tape = R.rollout(R.start(x0, D(prob.v0), D(prob.theta0)), acts, R.mats, grad)
    x, th = S[0], S[2]
    xw = torch.cat([x, R.w[:, None]], -1)
    if not grad:
        tr = torch.stack([torch.cat([t, R.w[:, None]], -1) for t in traj])
        if c["mode"] == "score":
            q = [crossing(prob, x)[0], repulsion(prob, x, 0.05, 4)[0]]
            return dict(traj=tr, crossing=q[0], repulsion=q[1])
        return dict(traj=tr, x=xw, theta=th)
    xl = x.detach().requires_grad_(True)
    with torch.enable_grad():
        if c["mode"] == "sysid":
            q, gx = exact_silhouette(prob, D(ex["cams"]), torch.as_tensor(ex["masks"], device=dev), x)
        else:
            nvr = D(prob.n_verts)
            per = torch.zeros(B, dtype=torch.float64, device=dev).index_add(0, R.vr, dot(xl - D(ex["target"]), xl - D(ex["target"]))) / nvr
            L = per.sum() if c["mode"] == "grad" else ((xl - D(ex["target"])) ** 2).mean()
            gx = torch.autograd.grad(L, xl)[0]
            q = per.detach() if c["mode"] == "grad" else L.detach()
    cot, ga, gm = R.reverse(tape, acts, R.mats, gx)
    gx0 = R.reverse_start(x0, cot)
    gv = torch.cat([cot[1], torch.zeros_like(cot[1][:, :1])], -1)
    gv[R.ea, 3] = cot[3]
    out = dict(x=xw, loss=q, x0=four(gx0), v0=gv)
    if c["mode"] == "sysid":
        return dict(out, gx=four(gx), material=torch.stack([gm[k] for k in ("K", "E", "G", "sy", "cd")], 1))
    return dict(out, actions=ga)


def by_rods(fn, prob, x, per):
    """fn over parts of the rods ([b, n, 3] positions, rod slice), results concatenated."""
    B, n = prob.batch, int(prob.n_verts[0])
    xs = x.reshape(B, n, 3)
    got = [fn(xs[i:i + per], slice(i, min(B, i + per))) for i in range(0, B, per)]
    return [torch.cat([g[k] for g in got]) for k in range(len(got[0]))]


def with_grad(fn, prob, x, per):
    def one(xs, sl):
        xs = xs.detach().requires_grad_(True)
        with torch.enable_grad():
            q = fn(xs, sl)
            g = torch.autograd.grad(q.sum(), xs, allow_unused=True)[0]
        return q.detach(), (torch.zeros_like(xs) if g is None else g).reshape(-1, 3)
    return by_rods(one, prob, x, per)


def crossing(prob, x):
    """Sum over ordered pairs of non-adjacent edges of the Gauss double integral / (4 pi)."""
    def one(xs, sl):
        a, b = xs[:, :-1], xs[:, 1:]
        i, j = torch.triu_indices(a.shape[1], a.shape[1], 2, device=x.device)
        p1, p2, p3, p4 = a[:, i], b[:, i], a[:, j], b[:, j]
        r13, r14, r23, r24 = p3 - p1, p4 - p1, p3 - p2, p4 - p2
        l13, l14, l23, l24 = (dot(r, r).sqrt() for r in (r13, r14, r23, r24))
        m1 = l13 * l14 * l24 + dot(r13, r14) * l24 + dot(r13, r24) * l14 + dot(r14, r24) * l13
        m2 = l13 * l24 * l23 + dot(r13, r24) * l23 + dot(r13, r23) * l24 + dot(r24, r23) * l13
        om = -2 * (torch.atan2(dot(r13, cross(r14, r24)), m1) + torch.atan2(dot(r13, cross(r24, r23)), m2))
        return om.sum(1) / (2 * math.pi)
    return with_grad(one, prob, x, 128)


def repulsion(prob, x, delta, k):
    delta = float(np.float32(delta))

    def one(xs, sl):
        a, b = xs[:, :-1], xs[:, 1:]
        i, j = torch.triu_indices(a.shape[1], a.shape[1], k + 1, device=x.device)
        with torch.no_grad():
            s, u = closest(a[:, i], b[:, i], a[:, j], b[:, j])
        d = a[:, i] + s[..., None] * (b[:, i] - a[:, i]) - a[:, j] - u[..., None] * (b[:, j] - a[:, j])
        return ((delta - dot(d, d).sqrt()).clamp(min=0.0) ** 2).sum(1)
    return with_grad(one, prob, x, 128)


def exact_losses(prob, ex, x):
    w = ex["weight"]
    pts = ex["points"]

    def chamfer(xs, sl):
        d2 = ((xs[:, :, None] - pts[sl][:, None]) ** 2).sum(-1)
        return d2.min(2).values.mean(1) + d2.min(1).values.mean(1)

    def winding(xs, sl):
        d = xs[..., :2] - ex["post"][sl][:, None, :2]
        a, b = d[:, :-1], d[:, 1:]
        return torch.atan2(a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0], (a * b).sum(-1)).sum(1) / (2 * math.pi)

    def mindist(xs, sl):
        return dot(xs - ex["post"][sl][:, None, :3], xs - ex["post"][sl][:, None, :3]).sqrt().min(1).values

    got = dict(chamfer=with_grad(chamfer, prob, x, 64), crossing=crossing(prob, x), repulsion=repulsion(prob, x, 0.05, 4),
               winding=with_grad(winding, prob, x, 512), mindist=with_grad(mindist, prob, x, 512))
    out = {}
    for k, (q, g) in got.items():
        g = g * w.repeat_interleave(torch.as_tensor(prob.n_verts, device=g.device))[:, None]
        out[k] = [q, torch.cat([g, torch.zeros_like(g[:, :1])], -1)]
    return out


def exact_silhouette(prob, cams, masks, x):
    """Per rod the mean squared difference of soft silhouettes and masks, and dq/dx."""
    C, H, W = masks.shape[1:]
    py, px = torch.meshgrid(torch.arange(H, device=x.device) + 0.5, torch.arange(W, device=x.device) + 0.5, indexing="ij")
    pix = torch.stack([px, py], -1).reshape(-1, 2).double()
    r = float(prob.radius[0])

    def one(xs, sl):
        q = 0.0
        for k in range(C):
            cm = cams[k]
            P = xs[0] @ cm[4:13].reshape(3, 3).T + cm[13:16]
            uv = torch.stack([cm[0] * P[:, 0] / P[:, 2] + cm[2], cm[1] * P[:, 1] / P[:, 2] + cm[3]], -1)
            rho = cm[0] * r / P[:, 2]
            a, e, re = uv[:-1], uv[1:] - uv[:-1], 0.5 * (rho[1:] + rho[:-1])
            t = (((pix[:, None] - a) * e).sum(-1) / (e * e).sum(-1)).clamp(0, 1)
            dv = pix[:, None] - a - t[..., None] * e
            sd = (dv * dv).sum(-1).clamp(min=1e-300).sqrt() - re
            o = -torch.expm1(-torch.nn.functional.softplus(-sd / SIL_TAU).sum(1))
            q = q + ((o - masks[sl.start, k].reshape(-1).double()) ** 2).mean() / C
        return q[None]
    return with_grad(one, prob, x, 1)
