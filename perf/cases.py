"""What the library is used for, as cases that can be measured.

A case is a dict of plain values; `kind` names the public entry point:

  search     Context.search_so3: the docking search over orientation samples
  refine     Context.refine_se3: SE(3) refinement of the surviving candidates
  objective  autograd.objective, forward and backward, over a batch of twists
  register   Context.register: global search, local search, refinement
  batch      Context.register_batch: uneven registrations that arrive together
  object     Context.object_grid and the grid it exports: a new object model

Inputs are star-shaped objects and drop-to-contact trajectories like those of
`synth.make_workload`, with the contact points found on the GPU so that they
are made in a fraction of a second.  Lattice sides, probe sizes, trajectory
lengths, mesh sizes, sample counts and candidate counts are those of
`synth.CONFIGS`, of bench.py (the registration, its local stage of 5000
samples, the batched and the serving mix) and of the tests.
"""
import math

import numpy as np
import torch

from paper_2605_21398_gb300 import dock, synth
from paper_2605_21398_gb300.autograd import objective

THETA = math.radians(5.0)   # radius of the local search's ball
SIDES = (32, 64, 96, 128)
SAMPLERS = {"sf": dock.SAMPLER_SF, "hopf": dock.SAMPLER_HOPF, "geoball": dock.SAMPLER_GEOBALL}


def listed():
    return [
        # the smallest search: a coarse model, a short trajectory, few samples;
        # latency and launches count
        dict(name="search_n32", kind="search", N=32, h=0.5, degree=4, n_theta=24, n_phi=48, poses=200, radius=1.0,
             length=8.0, sampler="sf", rots=512, top_k=8, mode="plain"),
        # an ordinary global search: free-form object, 2000 noisy poses
        dict(name="search_n64", kind="search", N=64, h=0.25, degree=8, n_theta=72, n_phi=144, poses=2000, radius=0.8,
             length=12.0, sampler="sf", rots=4096, top_k=32, mode="plain"),
        # the label-aware score on the lattice side whose canvas is no power of
        # two, odd counts everywhere
        dict(name="search_n96_labels", kind="search", N=96, h=16.0 / 96, degree=8, n_theta=48, n_phi=96, poses=1501,
             radius=0.63, length=12.0, sampler="hopf", rots=1111, top_k=16, mode="labels"),
        # the largest search: the local stage of the 128^3 registration, and
        # (with other samples) a share of its global stage
        dict(name="search_n128", kind="search", N=128, h=0.15, degree=12, n_theta=128, n_phi=256, poses=5000,
             radius=0.8, length=12.0, sampler="geoball", rots=5000, top_k=64, mode="plain"),
        # the rotation mechanism as the paper prints it: the object rotated and
        # resampled, S fixed
        dict(name="search_n128_rotobj", kind="search", N=128, h=0.15, degree=12, n_theta=72, n_phi=144, poses=2000,
             radius=0.8, length=12.0, sampler="sf", rots=1000, top_k=64, mode="rotate_object"),
        # refining the few candidates of a small search
        dict(name="refine_small", kind="refine", N=32, h=0.5, degree=4, n_theta=24, n_phi=48, poses=200, radius=1.0,
             length=8.0, K=8, solver="gn"),
        # refining the 64 candidates of the 128^3 registration
        dict(name="refine_large", kind="refine", N=128, h=0.15, degree=12, n_theta=128, n_phi=256, poses=5000,
             radius=0.8, length=12.0, K=64, solver="gn"),
        # the solver the paper prints
        dict(name="refine_lbfgsb", kind="refine", N=64, h=0.25, degree=8, n_theta=72, n_phi=144, poses=2000,
             radius=0.8, length=12.0, K=32, solver="lbfgsb"),
        # the refinement objective inside a user's own torch program
        dict(name="objective_fwd_bwd", kind="objective", N=64, h=0.25, degree=8, n_theta=72, n_phi=144, poses=2000,
             radius=0.8, length=12.0, B=16),
        # one whole registration at the ordinary size
        dict(name="register_n64", kind="register", N=64, h=0.25, degree=8, n_theta=72, n_phi=144, poses=2000,
             radius=0.8, length=12.0, n_global=4096, n_local=1024, top_k=32),
        # registrations of all lattice sides that arrive together
        dict(name="batch_uneven", kind="batch", requests=8, objects=4, poses_lo=100, poses_hi=2000, rots_lo=500,
             rots_hi=2000, top_k=8, degree=8, n_theta=48, n_phi=96),
        # a new object: its grid, its spectrum and its search tree
        dict(name="object_n128", kind="object", N=128, h=0.15, degree=12, n_theta=128, n_phi=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search"] * 9 + ["refine"] * 4 + ["objective"] * 2 + ["register"] * 2 + ["batch"] + ["object"] * 2)
    N = rng.choice(SIDES)
    n_theta = _log_int(rng, 20, 128)
    c = dict(kind=kind, N=N, h=rng.uniform(16.0, 19.2) / N, degree=rng.randint(3, 12), n_theta=n_theta,
             n_phi=2 * n_theta)
    if kind == "object":
        return c
    if kind == "batch":
        lo = rng.randint(100, 400)
        return dict(kind=kind, requests=rng.randint(3, 8), objects=rng.randint(2, 4), poses_lo=lo,
                    poses_hi=rng.randint(lo, 2000), rots_lo=rng.randint(300, 600), rots_hi=rng.randint(600, 2000),
                    top_k=rng.randint(1, 16), degree=8, n_theta=48, n_phi=96)
    c.update(poses=_log_int(rng, 100, 5000), radius=rng.uniform(0.5, 1.5), length=rng.uniform(8.0, 12.0))
    if kind == "search":
        most = {32: 16384, 64: 8192, 96: 5000, 128: 3000}[N]
        c.update(sampler=rng.choice(sorted(SAMPLERS)), rots=_log_int(rng, 64, most), top_k=_log_int(rng, 1, 64),
                 mode=rng.choice(["plain", "plain", "plain", "labels", "rotate_object"]))
    elif kind == "refine":
        c.update(solver=rng.choice(["gn", "gn", "lbfgsb"]), poses=_log_int(rng, 100, 2500))
        c.update(K=_log_int(rng, 1, 64 if c["solver"] == "gn" else 16))
    elif kind == "objective":
        c.update(B=_log_int(rng, 1, 32))
    else:
        c["N"] = N = rng.choice([32, 64, 96])
        c["h"] = rng.uniform(16.0, 19.2) / N
        c.update(poses=_log_int(rng, 100, 2500), n_global=_log_int(rng, 500, 4096), n_local=_log_int(rng, 100, 1024), top_k=_log_int(rng, 1, 32))
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------


def _surface(verts, tris, sub):
    """Points on the triangles (barycentric grid of `sub` steps), FP64 on the GPU."""
    T = torch.as_tensor(verts, device="cuda")[torch.as_tensor(tris, device="cuda").long()]
    w = torch.tensor([(i / sub, j / sub, 1 - (i + j) / sub) for i in range(sub + 1) for j in range(sub + 1 - i)],
                     dtype=torch.float64, device="cuda")
    return torch.einsum("wk,tkc->twc", w, T).reshape(-1, 3)


def _trajectory(obj, n, radius, rng):
    """n poses of a flat-ended cylinder dropped along its axis onto the object:
    three segments of different tool axes, each a zig-zag raster of five lines
    over the part of the object below the tool; (n, 7), object frame."""
    edge = math.sqrt(4 * math.pi * 25.0 / len(obj.tris))
    pts = _surface(obj.verts, obj.tris, max(1, min(8, int(math.ceil(edge / 0.08)))))
    axes = synth.quat_to_mat(synth.random_quat(rng)).T
    poses = []
    for s in range(3):
        k = n // 3 + (1 if s < n % 3 else 0)
        if k == 0:
            continue
        a = axes[s] + rng.normal(size=3) * 0.15
        a /= np.linalg.norm(a)
        ref = np.eye(3)[int(np.argmin(np.abs(a)))]
        e1 = ref - a * (ref @ a)
        e1 /= np.linalg.norm(e1)
        e2 = np.cross(a, e1)
        i = np.arange(k)
        line = i * 5 // k
        tau = (i - np.ceil(line * k / 5.0)) / max(1.0, k / 5.0)
        v = 1.3 * (line - 2)
        half = np.sqrt(3.4 ** 2 - v ** 2)
        u = half * (2 * np.where(line % 2 == 0, tau, 1 - tau) - 1)
        P = pts @ torch.as_tensor(np.stack([e1, e2, a], axis=1), device="cuda")
        uv = torch.as_tensor(np.stack([u, v], axis=1), device="cuda")
        drop = []
        for q in uv.split(max(1, 60_000_000 // len(pts))):
            near = (P[None, :, 0] - q[:, :1]) ** 2 + (P[None, :, 1] - q[:, 1:]) ** 2 <= radius * radius
            drop.append(torch.where(near, P[None, :, 2], torch.full((), -1e9, dtype=P.dtype, device="cuda")).amax(1))
        z = torch.cat(drop).cpu().numpy()
        tip = u[:, None] * e1 + v[:, None] * e2 + z[:, None] * a
        q = synth.mat_to_quat(np.stack([e1, e2, a], axis=1))
        poses.append(np.concatenate([np.broadcast_to(q, (k, 4)), tip], axis=1))
    return np.concatenate(poses)


def _scene(c, seed):
    """Mesh, world poses, contact labels and planted object pose of a case."""
    obj = synth.star_mesh(c["degree"], 0.05, c["n_theta"], c["n_phi"], seed)
    rng = np.random.default_rng([seed, 1])
    poses = _trajectory(obj, c["poses"], c["radius"], rng)
    labels = np.ones(len(poses), dtype=np.uint8)
    if c.get("mode") == "labels":   # retreat arcs: a fifth of the poses lifted off the surface
        run = max(1, len(poses) // 25)
        for s in rng.choice(max(1, len(poses) - run), size=5, replace=False):
            axis = synth.quat_to_mat(poses[s:s + run, :4])[:, :, 2]
            m = len(axis)
            lift = rng.uniform(0.5, 2.0) * (0.25 + 0.75 * np.sin(np.pi * (np.arange(m) + 0.5) / m))
            poses[s:s + run, 4:] += lift[:, None] * axis
            labels[s:s + run] = 0
    gt_q, gt_t = synth.random_quat(rng), rng.uniform(-2.0, 2.0, size=3)
    world = synth.add_pose_noise(synth.transform_poses(gt_q, gt_t, poses), rng, 0.02, 0.0)
    return obj, np.ascontiguousarray(world), labels, gt_q, gt_t, rng


def _near(gt_q, gt_t, n, h, rng):
    """n candidate poses around the planted one, as a local search leaves them."""
    dq = synth.axis_angle_quat(rng.normal(0.0, math.radians(1.0), size=(n, 3)))
    q = synth.quat_mul(dq, np.broadcast_to(gt_q, (n, 4)))
    return q / np.linalg.norm(q, axis=1, keepdims=True), gt_t + rng.uniform(-0.5 * h, 0.5 * h, size=(n, 3))


_ctx = None


def _context():
    """The one context of the process, as a user's program keeps it."""
    global _ctx
    if _ctx is None:
        _ctx = dock.Context(0)
    return _ctx


def prepare(case, seed):
    c, ctx = case, _context()
    if c["kind"] == "object":
        obj = synth.star_mesh(c["degree"], 0.05, c["n_theta"], c["n_phi"], seed)
        return dict(case=c, ctx=ctx, verts=obj.verts, tris=obj.tris)
    if c["kind"] == "batch":
        rng = np.random.default_rng([seed, 2])
        pairs = []
        for k in range(c["objects"]):
            N = SIDES[k % 4]
            s = dict(c, N=N, h=16.0 / N, poses=int(rng.integers(c["poses_lo"], c["poses_hi"] + 1)),
                     radius=float(rng.uniform(0.5, 1.5)), length=12.0)
            obj, world, labels, _, _, _ = _scene(s, 100 * seed + k)
            pairs.append((ctx.object_grid(obj.verts, obj.tris, s["h"], N),
                          ctx.sweep_grid(world, s["radius"], s["length"], s["h"], N, contact=labels)))
        reqs = []
        for r in range(c["requests"]):
            n = int(rng.integers(c["rots_lo"], c["rots_hi"] + 1))
            reqs.append(pairs[r % len(pairs)] + (n, n // 4, THETA, c["top_k"]))
        return dict(case=c, ctx=ctx, reqs=reqs, pairs=pairs)
    obj, world, labels, gt_q, gt_t, rng = _scene(c, seed)
    st = dict(case=c, ctx=ctx, ob=ctx.object_grid(obj.verts, obj.tris, c["h"], c["N"]),
              sw=ctx.sweep_grid(world, c["radius"], c["length"], c["h"], c["N"], contact=labels))
    if c["kind"] == "search":
        st["sw"].set_label_aware(c["mode"] == "labels")
        st["sw"].set_rotate_object(c["mode"] == "rotate_object")
        # the local stage's centre: the best orientation of the global one
        st["q0"] = _near(gt_q, gt_t, 1, c["h"], rng)[0][0] if c["sampler"] == "geoball" else None
    elif c["kind"] == "refine":
        q, t = _near(gt_q, gt_t, c["K"], c["h"], rng)
        st["cands"] = [dict(q=q[i], t=t[i]) for i in range(c["K"])]
        st["params"] = dock.default_params()
        st["params"].solver = dock.SOLVER_LBFGSB if c["solver"] == "lbfgsb" else dock.SOLVER_GAUSS_NEWTON
    elif c["kind"] == "objective":
        q, t = _near(gt_q, gt_t, c["B"], c["h"], rng)
        st["base"] = np.concatenate([q, t], axis=1)
        xi = np.concatenate([rng.normal(0, 0.02, size=(c["B"], 3)), rng.normal(0, 0.004, size=(c["B"], 3))], axis=1)
        st["xi"] = torch.tensor(xi, dtype=torch.float32, device="cuda", requires_grad=True)
    return st


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------


def _candidates(cands):
    return dict(score=np.array([c["score"] for c in cands], dtype=np.float32), q=np.array([c["q"] for c in cands]),
                t=np.array([c["t"] for c in cands]), rot=np.array([c["rot"] for c in cands]),
                dk=np.array([c["dk"] for c in cands]), canvas_idx=np.array([c["canvas_idx"] for c in cands]))


def _results(rs):
    out = dict(q=np.array([r["q"] for r in rs]), t=np.array([r["t"] for r in rs]), J=np.array([r["J"] for r in rs]),
               best_cand=np.array([r["best_cand"] for r in rs]), n_evals=np.array([r["n_evals"] for r in rs]))
    out["best_search"] = _candidates([r["best_search"] for r in rs])
    return out


def run(st):
    c, ctx = st["case"], st["ctx"]
    kind = c["kind"]
    if kind == "search":
        return _candidates(ctx.search_so3(st["ob"], st["sw"], c["rots"], c["top_k"], sampler=SAMPLERS[c["sampler"]],
                                          q0=st["q0"], theta=THETA if c["sampler"] == "geoball" else 0.0))
    if kind == "refine":
        rs = ctx.refine_se3(st["ob"], st["sw"], st["cands"], st["params"])
        return dict(q=np.array([r["q"] for r in rs]), t=np.array([r["t"] for r in rs]),
                    xi=np.array([r["xi"] for r in rs]), J=np.array([r["J"] for r in rs]),
                    iters=np.array([r["iters"] for r in rs]))
    if kind == "objective":
        xi = st["xi"]
        xi.grad = None
        J = objective(xi, ctx, st["ob"], st["sw"], st["base"])
        J.sum().backward()
        return dict(J=J.detach(), grad=xi.grad)
    if kind == "register":
        return _results([ctx.register(st["ob"], st["sw"], c["n_global"], c["n_local"], THETA, c["top_k"])])
    if kind == "batch":
        return _results(ctx.register_batch(st["reqs"]))
    ob = ctx.object_grid(st["verts"], st["tris"], c["h"], c["N"])
    grid, origin = ob.export_grid()
    return dict(grid=grid, origin=origin)


# --------------------------------------------------------------------------
# the work of a pass
# --------------------------------------------------------------------------


def _fft_flops(N):
    """Forward and inverse real 3-D transforms of the (2N)^3 canvas and the product of their half spectra."""
    M = 2 * N
    return 2 * 2.5 * M ** 3 * 3 * math.log2(M) + 6 * M * M * (M // 2 + 1)


def _search_work(N, poses, rots):
    M = 2 * N
    return dict(bytes=8 * M * M * (M // 2 + 1) + 56 * poses + 8 * rots, flops=rots * _fft_flops(N))


def _refine_work(c, queries):
    mesh = 2 * c["n_phi"] * (c["n_theta"] - 1)
    # one point-to-probe distance per vertex of the triangle a query ends at, its score and derivatives
    return dict(bytes=24 * mesh + 56 * c["poses"], flops=150.0 * queries)


def work(case):
    c = case
    if c["kind"] == "search":
        w = _search_work(c["N"], c["poses"], c["rots"])
        if c["mode"] == "labels":
            w["flops"] += 0.5 * c["rots"] * _fft_flops(c["N"])   # the second forward transform
        return w
    if c["kind"] == "refine":
        return _refine_work(c, 21 * c["K"] * c["poses"])
    if c["kind"] == "objective":
        return _refine_work(c, 2 * c["B"] * c["poses"])
    if c["kind"] == "register":
        w, r = _search_work(c["N"], c["poses"], c["n_global"] + c["n_local"]), _refine_work(c, 21 * c["top_k"] * c["poses"])
        return dict(bytes=w["bytes"] + r["bytes"], flops=w["flops"] + r["flops"])
    if c["kind"] == "batch":
        n, p = (c["rots_lo"] + c["rots_hi"]) / 2 * 1.25, (c["poses_lo"] + c["poses_hi"]) / 2
        ws = [_search_work(SIDES[r % c["objects"] % 4], p, n) for r in range(c["requests"])]
        r = _refine_work(dict(c, poses=p), 21 * c["requests"] * c["top_k"] * p)
        return dict(bytes=sum(w["bytes"] for w in ws) + r["bytes"], flops=sum(w["flops"] for w in ws) + r["flops"])
    N, mesh = c["N"], 2 * c["n_phi"] * (c["n_theta"] - 1)
    return dict(bytes=24 * mesh + 4 * N ** 3 + 8 * 4 * N * N * (N + 1), flops=0.5 * _fft_flops(N))


# --------------------------------------------------------------------------
# the same in 64 bits
# --------------------------------------------------------------------------


def _rot64(q):
    w, x, y, z = torch.as_tensor(np.asarray(q), dtype=torch.float64, device="cuda").unbind(-1)
    m = [1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
         1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
         1 - 2 * (x * x + y * y)]
    return torch.stack(m, -1).reshape(w.shape + (3, 3))


def _tri_dist2(p, a, b, c):
    """Squared distance from points to triangles, pair by pair."""
    dot = lambda u, v: (u * v).sum(-1)  # noqa: E731

    def seg(o, e):
        t = (dot(p - o, e) / dot(e, e)).clamp(0, 1)
        d = p - o - t[..., None] * e
        return dot(d, d)

    ab, ac, ap = b - a, c - a, p - a
    n = torch.linalg.cross(ab, ac)
    nn = dot(n, n)
    v = dot(torch.linalg.cross(ap, ac), n) / nn
    w = dot(torch.linalg.cross(ab, ap), n) / nn
    inside = (v >= 0) & (w >= 0) & (v + w <= 1)
    edge = torch.minimum(torch.minimum(seg(a, ab), seg(a, ac)), seg(b, c - b))
    return torch.where(inside, dot(ap, n) ** 2 / nn, edge)


def _grid64(verts, tris, h, N, tau_out=0.5, tau_in=0.2, deep=-50.0):
    """min(O_t, O_m) of the signed distance on the object's lattice, and its origin."""
    V = torch.as_tensor(verts, device="cuda")
    T = torch.as_tensor(tris, device="cuda").long()
    mid = (V.amin(0) + V.amax(0)) * 0.5
    o = h * torch.round(mid / h) - (N // 2) * h
    best = torch.full((N ** 3,), float("inf"), dtype=torch.float64, device="cuda")
    for t in T.split(8192):
        tv = V[t]
        lo = torch.ceil((tv.amin(1) - tau_out - o) / h).long().clamp(0, N - 1)
        hi = torch.floor((tv.amax(1) + tau_out - o) / h).long().clamp(0, N - 1)
        n = (hi - lo + 1).amax(0).tolist()
        off = torch.cartesian_prod(*[torch.arange(k, device="cuda") for k in n])
        for part in range(0, len(t), max(1, 4_000_000 // len(off))):
            s = slice(part, part + max(1, 4_000_000 // len(off)))
            k = lo[s, None, :] + off
            ok = (k <= hi[s, None, :]).all(-1)
            i, _ = ok.nonzero(as_tuple=True)
            k = k[ok]
            a, b, c = tv[s][i].unbind(1)
            d2 = _tri_dist2(k.double() * h + o, a, b, c)
            best.scatter_reduce_(0, (k[:, 2] * N + k[:, 1]) * N + k[:, 0], d2, "amin")
    # crossings of every lattice row with the mesh beyond each voxel
    beyond = torch.zeros((N * N, N + 1), dtype=torch.long, device="cuda")
    for t in T.split(65536):
        tv = V[t]
        lo = torch.ceil((tv.amin(1) - o) / h).long()[:, 1:]
        hi = torch.floor((tv.amax(1) - o) / h).long()[:, 1:]
        ny, nz = (hi - lo + 1).amax(0).clamp(min=1).tolist()
        k = lo[:, None, :] + torch.cartesian_prod(torch.arange(ny, device="cuda"), torch.arange(nz, device="cuda"))
        ok = (k <= hi[:, None, :]).all(-1)
        i, _ = ok.nonzero(as_tuple=True)
        k = k[ok]
        a, b, c = tv[i].unbind(1)
        p = k.double() * h + o[1:]
        side = lambda u, v: (v[:, 1] - u[:, 1]) * (p[:, 1] - u[:, 2]) - (v[:, 2] - u[:, 2]) * (p[:, 0] - u[:, 1])  # noqa: E731
        ea, eb, ec = side(b, c), side(c, a), side(a, b)

        def sign(e, u, v):   # a row through an edge or a vertex is taken a little towards +y, less so towards +z
            dy, dz = v[:, 1] - u[:, 1], v[:, 2] - u[:, 2]
            return torch.sign(torch.where(e != 0, e, torch.where(dz != 0, -dz, dy)))

        sa, sb, sc = sign(ea, b, c), sign(eb, c, a), sign(ec, a, b)
        hit = (sa == sb) & (sb == sc) & (sa != 0) & (ea + eb + ec != 0)
        x = ((ea * a[:, 0] + eb * b[:, 0] + ec * c[:, 0]) / (ea + eb + ec))[hit]
        below = torch.ceil((x - o[0]) / h).long().clamp(0, N)   # voxels kx < below lie before the crossing
        beyond.index_put_((k[hit, 1] * N + k[hit, 0], below), torch.ones_like(below), accumulate=True)
    inside = (beyond.flip(1).cumsum(1).flip(1)[:, 1:] % 2 == 1).reshape(-1)
    D = torch.where(best < tau_out ** 2, best.sqrt(), torch.full_like(best, float("inf")))
    f = torch.where(inside, -D, D)
    Ot = torch.where((f >= 0) & (f < tau_out), 1 - f / tau_out, torch.zeros_like(f))
    Ot = torch.where((f > -tau_in) & (f < 0), 1 + f / tau_in, Ot)
    Ot = torch.where(f <= -tau_in, torch.full_like(f, deep), Ot)
    return torch.minimum(Ot, (1 - D / tau_out).clamp(min=0)).reshape(N, N, N), o


def _scores64(c, obj, world):
    """The top_k largest correlation peaks over the Super-Fibonacci samples."""
    N, h, M = c["N"], c["h"], 2 * c["N"]
    O, _ = _grid64(obj.verts, obj.tris, h, N)
    F = torch.fft.rfftn(O, s=(M, M, M)).conj()
    i = np.arange(c["rots"]) + 0.5
    t = i / c["rots"]
    al, be = 2 * np.pi * i / math.sqrt(2.0), 2 * np.pi * i / 1.533751168755204288118041
    Rs = _rot64(np.stack([np.sqrt(t) * np.sin(al), np.sqrt(t) * np.cos(al), np.sqrt(1 - t) * np.sin(be),
                          np.sqrt(1 - t) * np.cos(be)], axis=1))
    Rp = _rot64(world[:, :4])
    tp = torch.as_tensor(world[:, 4:], device="cuda")
    cs = tp.mean(0)
    k = torch.arange(N, device="cuda", dtype=torch.float64)
    grid = torch.stack(torch.meshgrid(k, k, k, indexing="ij"), -1).flip(-1).reshape(-1, 3)   # (x, y, z), x fastest
    peaks = []
    for R in Rs:
        o = h * torch.round(R.T @ cs / h) - (N // 2) * h
        x = (grid * h + o) @ R.T
        S = torch.zeros(len(x), dtype=torch.bool, device="cuda")
        for a, b in zip(Rp.split(64), tp.split(64)):
            l = torch.einsum("vpc,pck->vpk", x[:, None, :] - b, a)
            S |= ((l[..., 0] ** 2 + l[..., 1] ** 2 <= c["radius"] ** 2) & (l[..., 2] >= 0) & (l[..., 2] <= c["length"])).any(1)
        C = torch.fft.irfftn(torch.fft.rfftn(S.reshape(N, N, N).double(), s=(M, M, M)) * F, s=(M, M, M))
        peaks.append(C.max())
    return torch.stack(peaks).sort(descending=True).values[: c["top_k"]]


def _probe_sdf(x, r, L):
    dr = x[..., :2].norm(dim=-1) - r
    dz = torch.maximum(-x[..., 2], x[..., 2] - L)
    return torch.where((dr > 0) & (dz > 0), torch.sqrt(dr.clamp(min=0) ** 2 + dz.clamp(min=0) ** 2), torch.maximum(dr, dz))


def _tri_min64(v0, v1, v2, r, L):
    """Minimum of the (convex) probe distance over triangles: golden sections
    over one barycentric coordinate, of golden sections over the other."""
    g = (math.sqrt(5.0) - 1) / 2
    e1, e2 = v1 - v0, v2 - v0

    def golden(f, hi, steps):
        lo = torch.zeros_like(hi)
        c, d = hi - g * (hi - lo), lo + g * (hi - lo)
        fc, fd = f(c), f(d)
        for _ in range(steps):
            left = fc <= fd
            lo, hi = torch.where(left, lo, c), torch.where(left, d, hi)
            x = torch.where(left, hi - g * (hi - lo), lo + g * (hi - lo))
            fx = f(x)
            c, d = torch.where(left, x, d), torch.where(left, c, x)
            fc, fd = torch.where(left, fx, fd), torch.where(left, fc, fx)
        return torch.minimum(torch.minimum(fc, fd), f(0.5 * (lo + hi)))

    def inner(u):
        base = v0 + u[:, None] * e1
        vmax = 1 - u
        at = lambda v: _probe_sdf(base + v[:, None] * e2, r, L)  # noqa: E731
        return torch.minimum(golden(at, vmax, 46), torch.minimum(at(torch.zeros_like(u)), at(vmax)))

    one = torch.ones(len(v0), dtype=torch.float64, device=v0.device)
    return torch.minimum(golden(inner, one, 46), torch.minimum(inner(torch.zeros_like(one)), inner(one)))


def _objective64(c, obj, world, base, xi, tau_out=0.2, tau_in=0.03, k=15.0, lam=1e-3):
    """J and its gradient (central differences of every distance) for twists xi about base poses."""
    V = torch.as_tensor(obj.verts, device="cuda")
    T = torch.as_tensor(obj.tris, device="cuda").long()
    anchor = (V.amin(0) + V.amax(0)) * 0.5
    Rp, tp = _rot64(world[:, :4]), torch.as_tensor(world[:, 4:], device="cuda")
    r, L = c["radius"], c["length"]

    def frames(b, x):
        u, w = x[:3], x[3:]
        K = torch.zeros(3, 3, dtype=torch.float64, device="cuda")
        K[0, 1], K[0, 2], K[1, 0], K[1, 2], K[2, 0], K[2, 1] = -w[2], w[1], w[2], -w[0], -w[1], w[0]
        th = float(w.norm())
        a, bb, s = ((1 - math.cos(th)) / th ** 2, (th - math.sin(th)) / th ** 3, math.sin(th) / th) if th > 1e-4 else (0.5, 1 / 6, 1.0)
        eye = torch.eye(3, dtype=torch.float64, device="cuda")
        dR, Vw = eye + s * K + a * K @ K, eye + a * K + bb * K @ K
        R0, p0 = _rot64(b[:4]), torch.as_tensor(b[4:], device="cuda")
        R = dR @ R0
        p = p0 + Vw @ u + R0 @ anchor - dR @ (R0 @ anchor)
        return R.T @ Rp, (tp - p) @ R   # probe frames in the object frame

    def local(A, b, idx, tri):
        q = V[T[tri]] - b[idx][:, None, :]
        return torch.einsum("nmc,nck->nmk", q, A[idx])

    # every (twist, pose) query with the triangles that can hold its minimum
    xs = torch.as_tensor(np.asarray(xi, dtype=np.float64), device="cuda")
    B, n = len(xs), len(Rp)
    cen = V[T].mean(1)
    rad = (V[T] - cen[:, None, :]).norm(dim=-1).amax(1)
    idx, tri, verts = [], [], []
    for j, (b, x) in enumerate(zip(np.asarray(base), xs)):
        A, bv = frames(b, x)
        for s in range(0, n, 256):
            f = _probe_sdf(torch.einsum("ptc,pck->ptk", cen[None] - bv[s:s + 256, None], A[s:s + 256]), r, L)
            lim = (f + rad).amin(1).clamp(max=tau_out + 1e-3)
            i, t = (f - rad <= lim[:, None]).nonzero(as_tuple=True)
            idx.append(j * n + s + i)
            tri.append(t)
            verts.append(local(A, bv, s + i, t))
    idx, tri = torch.cat(idx), torch.cat(tri)
    d = _tri_min64(*torch.cat(verts).unbind(1), r, L)
    far = torch.full((B * n,), float("inf"), dtype=torch.float64, device="cuda")
    dmin = far.scatter_reduce(0, idx, d, "amin")
    near = (d <= dmin[idx] + 2e-4) & (d < tau_out + 1e-3)
    idx, tri = idx[near], tri[near]
    # central differences of each distance along the six twist coordinates
    step, verts = 1e-5, []
    for j, (b, x) in enumerate(zip(np.asarray(base), xs)):
        mine = (idx // n) == j
        for k6 in range(6):
            e = torch.zeros(6, dtype=torch.float64, device="cuda")
            e[k6] = step
            for sg in (1.0, -1.0):
                verts.append(local(*frames(b, x + sg * e), idx[mine] % n, tri[mine]))
    counts = [len(v) for v in verts]
    ds = _tri_min64(*torch.cat(verts).unbind(1), r, L).split(counts)
    J, G = [], []
    for j, x in enumerate(xs):
        own = idx[(idx // n) == j] % n
        two = [torch.full((n,), float("inf"), dtype=torch.float64, device="cuda").scatter_reduce(0, own, m, "amin")
               for m in ds[12 * j:12 * j + 12]]
        dd = [torch.where(torch.isfinite(p), (p - m) / (2 * step), torch.zeros_like(p))
              for p, m in zip(two[0::2], two[1::2])]
        t = dmin[j * n:(j + 1) * n] / tau_out
        rr = tau_in / tau_out
        a3, a2 = k / rr ** 2 - 2 / rr ** 3, k / rr - 3 / rr ** 2
        tc = t.clamp(max=2.0)
        s = torch.where(t > 1, 0 * tc, torch.where(t > 0, torch.cos(0.5 * math.pi * tc) ** 2,
                                                   torch.where(t > -rr, a3 * tc ** 3 + a2 * tc ** 2 + 1, k * (tc + rr))))
        s1 = torch.where(t > 1, 0 * tc, torch.where(t > 0, -0.5 * math.pi * torch.sin(math.pi * tc),
                                                    torch.where(t > -rr, 3 * a3 * tc ** 2 + 2 * a2 * tc, k + 0 * tc))) / tau_out
        J.append(-s.sum() + lam * (x * x).sum())
        G.append(torch.stack([-(s1 * g).sum() for g in dd]) + 2 * lam * x)
    return torch.stack(J), torch.stack(G)


def exact(case, seed):
    c = case
    if c["kind"] == "object":
        obj = synth.star_mesh(c["degree"], 0.05, c["n_theta"], c["n_phi"], seed)
        grid, o = _grid64(obj.verts, obj.tris, c["h"], c["N"])
        return dict(grid=grid.cpu().numpy(), origin=o.cpu().numpy())
    if c["kind"] == "search" and c["mode"] == "plain" and c["sampler"] == "sf" and c["rots"] * c["poses"] * c["N"] ** 3 < 5e9:
        obj, world, _, _, _, _ = _scene(c, seed)
        # the peaks' scores; their order among equals, and with it the poses, is left to the search
        return dict(score=_scores64(c, obj, world).cpu().numpy(), q=None, t=None, rot=None, dk=None, canvas_idx=None)
    if c["kind"] == "objective" and c["B"] * c["poses"] <= 40000:
        obj, world, _, gt_q, gt_t, rng = _scene(c, seed)
        q, t = _near(gt_q, gt_t, c["B"], c["h"], rng)
        xi = np.concatenate([rng.normal(0, 0.02, size=(c["B"], 3)), rng.normal(0, 0.004, size=(c["B"], 3))], axis=1)
        J, G = _objective64(c, obj, world, np.concatenate([q, t], axis=1), xi.astype(np.float32))
        return dict(J=J.cpu().numpy(), grad=G.cpu().numpy())
    return None
