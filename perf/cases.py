"""Performance cases: the calls that programs built on this library make, at the sizes of its scenes, tests and benchmark.

A simulation keeps one context and calls one frame after another (state evolves from pass to pass, and every pass reads the
new state into device buffers, as a renderer does); a differentiable program calls the functional forms on tensors of its
own; a scene is seeded by the volume sampler from host arrays.  Every case is a dict of plain values; ``kind`` picks the call.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2308_01629_gb300 as gs
import scenes
from paper_2308_01629_gb300 import diff

R_BED = 0.0089        # r_LR of the digging bed


def listed():
    return [
        # the smallest scene: 1,000 LR / 8,000 HR, where launches and latency are the frame
        dict(name="frame_cube", kind="frame", scene="cube", n_side=10, ratio=8, n_sub=4, iters=4),
        # the funnel: 20,000 LR / 500,000 HR on a cone shell (ordinary size, sparse grid, curved boundary)
        dict(name="frame_funnel", kind="frame", scene="funnel", n_low=20000, ratio=25, n_sub=4, iters=6),
        # the benchmark's workload: the digging bed, 50,527 LR / 2,021,080 HR, a bucket SDF whose pose is set every frame
        dict(name="frame_digging", kind="frame", scene="digging", size=1.0, ratio=40, n_sub=4, iters=8),
        # the same bed of 2 x 2 m: about 202,000 LR / 8.1 M HR (the largest)
        dict(name="frame_bed_2m", kind="frame", scene="digging", size=2.0, ratio=40, n_sub=4, iters=8),
        # the bed with the bucket sampled as particles of infinite mass: the gather's second form
        dict(name="frame_particle_bucket", kind="frame", scene="bucket", size=0.7, ratio=25, n_sub=4, iters=8),
        # many small scenes served by one batched context (500 to 8,000 LR each)
        dict(name="frame_batch", kind="batch", n_scenes=64, n_sub=4, iters=4),
        # CFL-limited substeps on the column that falls and spreads: 4,000 LR / 64,000 HR
        dict(name="frame_adaptive", kind="adaptive", scene="column", n_low=4000, ratio=16, iters=4),
        # one HR frame as a function of the caller's tensors: 500,000 HR
        dict(name="upsample", kind="upsample", scene="funnel", n_low=20000, ratio=25),
        # the HR frame forward and backward, at the size of the differentiable pattern
        dict(name="upsample_grad", kind="upsample_grad", scene="column", n_low=4000, ratio=16),
        # one LR step forward and backward
        dict(name="step_grad", kind="step_grad", n_low=4000, iters=4),
        # the differentiable pattern whole: a checkpointed 30-step rollout and its reverse
        dict(name="rollout_grad", kind="rollout", n_low=4000, ratio=16, frames=30, every=5, iters=4),
        # seeding HR particles from the castle's mesh: about a million candidates, host arrays in and out
        dict(name="sample_castle", kind="sample", size=0.6, height=0.2, r=0.0075, per_cell=4.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "batch", "adaptive", "upsample", "upsample", "upsample_grad",
                       "step_grad", "rollout", "sample"])
    if kind == "frame":
        scene = rng.choice(["cube", "funnel", "digging", "digging", "bucket", "boulder", "materials"])
        c = dict(kind=kind, scene=scene, n_sub=rng.randint(2, 5), iters=rng.randint(4, 8))
        if scene == "cube":
            c.update(n_side=rng.randint(5, 15), ratio=rng.randint(4, 24))
        elif scene == "funnel":
            c.update(n_low=int(_log(rng, 1500, 20000)), ratio=rng.randint(8, 25))
        elif scene == "digging":
            c.update(size=round(_log(rng, 0.3, 1.7), 3), ratio=rng.randint(8, 40))
        else:
            c.update(size=round(_log(rng, 0.65, 1.0), 3), ratio=rng.randint(8, 40))
        return c
    if kind == "batch":
        return dict(kind=kind, n_scenes=int(_log(rng, 4, 96)), n_sub=rng.randint(2, 4), iters=rng.randint(3, 6))
    if kind == "sample":
        return dict(kind=kind, size=round(rng.uniform(0.3, 0.7), 3), height=round(rng.uniform(0.1, 0.25), 3),
                    r=round(_log(rng, 0.008, 0.03), 5), per_cell=round(rng.uniform(2.0, 5.0), 2))
    if kind == "upsample" and rng.random() < 0.6:
        return dict(kind=kind, scene="funnel", n_low=int(_log(rng, 1500, 20000)), ratio=rng.randint(8, 25))
    c = dict(kind=kind, n_low=int(_log(rng, 150, 5000)))
    if kind != "step_grad":
        c.update(ratio=rng.randint(6, 24))
    if kind != "upsample" and kind != "upsample_grad":
        c.update(iters=rng.randint(3, 8))
    if kind in ("upsample", "upsample_grad", "adaptive"):
        c.update(scene="column")
    if kind == "rollout":
        c.update(frames=rng.randint(4, 30), every=rng.randint(3, 6))
    return c


# ------------------------------------------------------------------ scenes ---
def _scene(c, seed):
    """The case's scene.  The beds and the batch keep one geometry per size (their particle counts follow it) and take
    their state from the seed; ``stir`` (in ``prepare``) gives the functional calls an LR velocity field and HR particles
    in every blend case."""
    k, base = c.get("scene", "column"), scenes.SEED_BASE + 1000 + int(seed)
    if k == "cube":
        return scenes.cube(seed=base, n_side=c["n_side"], ratio=c["ratio"])
    if k == "funnel":
        return scenes.funnel(seed=base, n_low=c["n_low"], ratio=c["ratio"])
    if k == "column":
        return scenes.column(seed=base, n_low=c["n_low"], ratio=c.get("ratio", 1), z0=0.02)
    bed = dict(r_low=R_BED, ratio=c["ratio"], size=c["size"])
    if k == "bucket":
        s = _moving(scenes.digging_particle_bucket(t=0.1, **bed), base)
        s["lr_vel"][s["lr_pos"][:, 3] == 0.0] = 0.0          # the particle bucket rests on the bed
        return s
    if k == "boulder":
        return _moving(scenes.digging_with_boulder(**bed), base)
    return _moving(scenes.digging(**bed), base)


def _moving(sc, seed):
    """Seeded small motions: LR velocities of 5 cm/s, particles off their places by a fraction of their radius."""
    rng = np.random.default_rng(seed)
    n, m, r = len(sc["lr_pos"]), len(sc["hr_pos"]), sc["r_low"]
    sc["lr_vel"][:, :3] += rng.normal(0.0, 0.05, (n, 3)).astype(np.float32)
    free = sc["lr_pos"][:, 3:] > 0
    sc["lr_pos"][:, :3] += np.where(free, rng.uniform(-0.05 * r, 0.05 * r, (n, 3)), 0.0).astype(np.float32)
    sc["hr_pos"][:, :3] += rng.uniform(-0.1 * r, 0.1 * r, (m, 3)).astype(np.float32)
    return sc


def _context(sc, stream, **kw):
    with torch.cuda.stream(stream):
        ctx = gs.Context(sc, stream="torch", **kw)
    ctx.set_graphs(True)
    return ctx


def _state_buffers(ctx):
    new = lambda n: torch.zeros((n, 4), dtype=torch.float32, device="cuda")  # noqa: E731
    return [(gs.GS_FIELD_HR_POS, new(ctx.n_high)), (gs.GS_FIELD_HR_VEL, new(ctx.n_high)),
            (gs.GS_FIELD_LR_POS, new(ctx.n_low)), (gs.GS_FIELD_LR_VEL, new(ctx.n_low))]


def _randn(seed, n):
    g = torch.Generator(device="cpu").manual_seed(int(seed))
    t = torch.randn((n, 4), generator=g, dtype=torch.float32)
    t[:, 3] = 0.0
    return t.cuda()


def _sample_inputs(c, seed):
    V, T = scenes.castle_mesh(base=(0.5, 0.5, 0.0), size=c["size"], height=c["height"])
    return V, T, scenes.volume_candidates(V, c["r"], c["per_cell"], seed=scenes.SEED_BASE + 1000 + int(seed))


def _tensors(sc):
    return [torch.from_numpy(sc[k]).cuda() for k in ("lr_pos", "lr_vel", "hr_pos", "hr_vel")]


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "sample":
        V, T, cand = _sample_inputs(c, seed)
        return dict(case=c, V=V, T=T, cand=cand, out=np.empty(len(cand), np.int64))
    stream = torch.cuda.Stream()
    st = dict(case=c, stream=stream, frame=0)
    if c["kind"] == "batch":
        sl = [_moving(s, int(seed) * 1000 + i) for i, s in enumerate(scenes.batch(n_scenes=c["n_scenes"]))]
        st["ctx"] = _context(sl, stream)
        st["out"] = _state_buffers(st["ctx"])
        return st
    sc = _scene(c, seed)
    if c["kind"] in ("frame", "adaptive"):
        st["ctx"] = _context(sc, stream)
        if c["scene"] == "materials":
            mu, ids = scenes.materials(sc, seed, "layers")
            st["ctx"].set_materials(mu, ids)
        st["bucket"] = sc.get("bucket_index")
        st["out"] = _state_buffers(st["ctx"])
        return st
    sc = scenes.stir(sc, seed=int(seed) + 5, v_scale=0.2)
    st["ctx"] = _context(sc, stream)
    st["in"] = _tensors(sc)
    n, m = len(sc["lr_pos"]), len(sc["hr_pos"])
    if c["kind"] == "upsample_grad":
        st["g"] = [_randn(seed + 1, m), _randn(seed + 2, m)]
    elif c["kind"] == "step_grad":
        st["g"] = [_randn(seed + 1, n), _randn(seed + 2, n)]
    elif c["kind"] == "rollout":
        st["g"] = [_randn(seed + 1, m)]   # the loss is on the final HR positions
    torch.cuda.synchronize()
    return st


DT_HR, DT_LR = 1.0 / 60.0, 1.0 / 240.0


def run(state):
    c = state["case"]
    k = c["kind"]
    if k == "sample":
        rc, sel, inside = gs.gs_sample_volume(state["V"], state["T"], state["cand"], c["r"])
        if rc != gs.GS_OK:
            raise gs.GsError(rc, "gs_sample_volume")
        out = state["out"]                                    # the chosen indices, then -1
        out[:len(sel)], out[len(sel):] = sel, -1
        return dict(selected=out, inside=inside.view(np.uint8))
    ctx = state["ctx"]
    with torch.cuda.stream(state["stream"]):
        if k in ("frame", "batch", "adaptive"):
            if k == "adaptive":
                ctx.frame_adaptive(DT_HR, c["iters"])
            else:
                if state.get("bucket") is not None:
                    ctx.set_sdf(state["bucket"], scenes.bucket_sdf(state["frame"] * DT_HR))
                ctx.frame(DT_HR, c["n_sub"], c["iters"])
            state["frame"] += 1
            for f, buf in state["out"]:
                ctx.read(f, buf)
            return [buf for _, buf in state["out"]]
        if k == "upsample":
            return list(diff.UpsampleFn.apply(ctx, DT_HR, *state["in"]))
        ins = [t.detach().requires_grad_(True) for t in state["in"]]
        if k == "upsample_grad":
            outs = diff.UpsampleFn.apply(ctx, DT_HR, *ins)
        elif k == "step_grad":
            ins = ins[:2]
            outs = diff.StepLowFn.apply(ctx, DT_LR, c["iters"], *ins)
        else:
            outs = diff.rollout(ctx, *ins, DT_LR, c["frames"], n_sub=1, iters=c["iters"], checkpoint_every=c["every"])
        on = outs if k != "rollout" else outs[2:3]
        grads = torch.autograd.grad(on, ins, state["g"])
        return [t.detach() for t in outs] + list(grads)


# -------------------------------------------------------------------- work ---
def _sizes(c):
    if c["kind"] == "batch":
        return 4250 * c["n_scenes"], 4250 * 18 * c["n_scenes"]     # the means of the counts and ratios drawn
    k = c.get("scene", "column")
    if k in ("digging", "bucket", "boulder", "materials"):
        n = int(c["size"] ** 2 * 50527)
    elif k == "cube":
        n = c["n_side"] ** 3
    else:
        n = c["n_low"]
    return n, n * c.get("ratio", 0)


def work(case):
    """Bytes: each state record in and out once (position and velocity, 32 bytes each way), and the copy that a frame's
    caller reads.  Operations: about 14 LR particles within reach of an HR particle, 20 operations each; about 17 partners
    within 3 r_LR of an LR particle, of which 4 touch, in every Jacobi pass; the reverse modes about twice that again."""
    c = dict(case)
    if c["kind"] == "sample":
        V, T, cand = _sample_inputs(c, 0)
        return {"bytes": 24.0 * len(cand) + 24 * len(V) + 12 * len(T) + len(cand), "flops": 70.0 * len(T) * len(cand)}
    n, m = _sizes(c)
    step, up = n * (17 * 8 + 4 * 60) * (2 + c.get("iters", 0)), m * 14 * 20
    k = c["kind"]
    if k in ("frame", "batch", "adaptive"):
        return {"bytes": 96.0 * (n + m), "flops": float(c.get("n_sub", 4) * step + up)}
    if k == "upsample":
        return {"bytes": 32.0 * n + 64.0 * m, "flops": float(up)}
    if k == "upsample_grad":
        return {"bytes": 32.0 * 2 * n + 32.0 * 4 * m, "flops": 3.0 * up}
    if k == "step_grad":
        return {"bytes": 32.0 * 4 * n, "flops": 3.0 * step}
    return {"bytes": 32.0 * 4 * (n + m) * c["frames"], "flops": 3.0 * c["frames"] * (step + up)}


# ------------------------------------------------------- 64-bit references ---
def _f32(v):
    return float(np.float32(v))


def _pairs(a, b, radius):
    """Index pairs (i, j) with |a_i - b_j| < radius, by a grid of cells of side `radius`."""
    lo = torch.minimum(a.min(0).values, b.min(0).values) - radius
    hi = torch.maximum(a.max(0).values, b.max(0).values) + radius
    dims = ((hi - lo) / radius).floor().long() + 1
    key = lambda q: (q[:, 2] * dims[1] + q[:, 1]) * dims[0] + q[:, 0]  # noqa: E731
    ca, cb = ((a - lo) / radius).floor().long(), ((b - lo) / radius).floor().long()
    kb, order = key(cb).sort()
    ids = torch.arange(len(a), device=a.device)
    out_i, out_j = [], []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                q = key(ca + torch.tensor([dx, dy, dz], device=a.device))
                s = torch.searchsorted(kb, q)
                e = torch.searchsorted(kb, q, right=True)
                for t in range(int((e - s).max()) if len(a) else 0):
                    has = s + t < e
                    i, j = ids[has], order[(s + t)[has]]
                    near = ((a[i] - b[j]) ** 2).sum(1) < radius * radius
                    out_i.append(i[near])
                    out_j.append(j[near])
    return torch.cat(out_i), torch.cat(out_j)


def _upsample64(sc, X, V, x, v):
    """One HR frame in 64 bits: LR positions and velocities X, V, HR x, v (n, 3)."""
    r, rh, dt = _f32(sc["r_low"]), _f32(sc["r_high"]), _f32(DT_HR)
    g = torch.tensor([_f32(a) for a in sc["gravity"]], dtype=torch.float64, device=x.device)
    c1, c2 = _f32(512.0 / 729.0), _f32(0.6)
    with torch.no_grad():
        i, j = _pairs(x, X, 3.0 * r)
    w = (1.0 - ((x[i] - X[j]) ** 2).sum(1) / (9.0 * r * r)).clamp_min(0.0) ** 3
    zero = torch.zeros(len(x), dtype=torch.float64, device=x.device)
    S = zero.index_add(0, i, w)
    VV = torch.zeros_like(x).index_add(0, i, w[:, None] * V[j])
    wmax = zero.scatter_reduce(0, i, w, "amax")
    has = S > 0
    vt = torch.where(has[:, None], VV / torch.where(has, S, torch.ones_like(S))[:, None], torch.zeros_like(VV))
    blend = (wmax <= c1) | (has & (wmax >= c2 * S))
    alpha = torch.where(blend, 1.0 - wmax, torch.zeros_like(wmax))[:, None]
    nv = (1.0 - alpha) * vt + alpha * (v + dt * g)
    nx = x + dt * nv
    for b in sc["sdfs"]:
        p, u = [_f32(a) for a in b["p"]], [_f32(a) for a in b["vel"]]
        if b["kind"] == scenes.SDF_BOX_INTERIOR:
            hits = []
            for a in range(3):
                n = torch.zeros(3, dtype=torch.float64, device=x.device)
                n[a] = 1.0
                hits += [(lambda y, a=a: y[:, a] - p[a], n), (lambda y, a=a: p[3 + a] - y[:, a], -n)]
        else:                                            # the cone shell
            hits = [(None, None)]
        for phi_of, n in hits:
            phi, n = (phi_of(nx), n[None, :]) if phi_of else _cone64(p, nx)
            on = phi < rh
            nx = nx + torch.where(on, rh - phi, torch.zeros_like(phi))[:, None] * n
            vn = ((nv - torch.tensor(u, dtype=torch.float64, device=x.device)) * n).sum(1)
            nv = nv - torch.where(on & (vn < 0), vn, torch.zeros_like(vn))[:, None] * n
    return nx, nv


def _cone64(p, x):
    d = x[:, :2] - torch.tensor(p[:2], dtype=torch.float64, device=x.device)
    rho = d.norm(dim=1)
    er, ez = p[5] - p[3], p[4] - p[2]
    qr, qz = rho - p[3], x[:, 2] - p[2]
    t = ((qr * er + qz * ez) / (er * er + ez * ez)).clamp(0.0, 1.0)
    a, b = qr - t * er, qz - t * ez
    dist = (a * a + b * b).sqrt()
    s = (dist > 0).double() / torch.where(dist > 0, dist, torch.ones_like(dist))
    rr = torch.where(rho > 0, rho, torch.ones_like(rho))
    return dist - p[6], torch.stack([a * s * d[:, 0] / rr, a * s * d[:, 1] / rr, b * s], 1)


def _step64(sc, x, v, winv, iters):
    """One LR step in 64 bits (2 stabilization and `iters` solver passes; box walls)."""
    r, dt, dev = _f32(sc["r_low"]), _f32(DT_LR), x.device
    d0, mu_s, mu_k = 2.0 * r, _f32(sc["mu_s"]), _f32(sc["mu_k"])
    g = torch.tensor([_f32(a) for a in sc["gravity"]], dtype=torch.float64, device=dev)
    box = sc["sdfs"][0]
    p = [_f32(a) for a in box["p"]]
    bs, bk = math.sqrt(mu_s * _f32(box["mu_s"])), math.sqrt(mu_k * _f32(box["mu_k"]))
    xt = x + dt * (v + dt * g)
    ws = winv * torch.exp(x[:, 2] - _f32(sc["box_lo"][2]))
    with torch.no_grad():
        i, j = _pairs(xt, xt, 3.0 * r)
        i, j = i[i != j], j[i != j]

    def slide(rel, L2, s, k):
        L = torch.where(L2 > 0, L2, torch.ones_like(L2)).sqrt()
        return torch.where((L2 > 0) & (L >= s) & (L > k), k / L, torch.ones_like(L))[:, None] * rel

    for it in range(2 + iters):
        stab = it < 2
        y = x if stab else xt
        with torch.no_grad():
            d2 = ((y[j] - y[i]) ** 2).sum(1)
            on = (d2 > 0) & (d2.sqrt() < d0)
        a, b = i[on], j[on]
        e = y[b] - y[a]
        d = e.norm(dim=1)
        m = (ws[a] / (ws[a] + ws[b]))[:, None]
        c = -m * ((d0 - d) / d)[:, None] * e
        if not stab:
            rel = (xt - x)[a] - (xt - x)[b]
            t = rel - ((rel * e).sum(1) / (d * d))[:, None] * e
            c = c - m * slide(t, (t * t).sum(1), d0 * mu_s, d0 * mu_k)
        D = torch.zeros_like(x).index_add(0, a, c)
        n = torch.zeros(len(x), dtype=torch.float64, device=dev).index_add(0, a, torch.ones_like(d))
        for k in range(6):
            ax, sg = k // 2, -1.0 if k & 1 else 1.0
            phi = (p[3 + ax] - y[:, ax]) if k & 1 else (y[:, ax] - p[ax])
            hit = phi < r
            nv = torch.zeros(3, dtype=torch.float64, device=dev)
            nv[ax] = sg
            f = (r - phi)[:, None] * nv
            if not stab:
                rel = xt - x
                t = rel - (rel * nv).sum(1)[:, None] * nv
                f = f - slide(t, (t * t).sum(1), d0 * bs, d0 * bk)
            D = D + torch.where(hit[:, None], f, torch.zeros_like(f))
            n = n + hit.double()
        delta = torch.where((n > 0)[:, None], D / n.clamp_min(1.0)[:, None], torch.zeros_like(D))
        xt = xt + delta
        if stab:
            x = x + delta
    return xt, (xt - x) / dt


def exact(case, seed):
    """The functional calls in 64 bits.  A simulated frame and a rollout have no such value: contacts that one rounding
    makes and another does not decide what follows."""
    c = dict(case)
    if c["kind"] not in ("upsample", "upsample_grad", "step_grad"):
        return None
    sc = scenes.stir(_scene(c, seed), seed=int(seed) + 5, v_scale=0.2)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    full = [torch.from_numpy(sc[k]).to(dev).double() for k in ("lr_pos", "lr_vel", "hr_pos", "hr_vel")]
    grad = c["kind"] != "upsample"
    ins = [t[:, :3].clone().requires_grad_(grad) for t in full]
    if c["kind"] == "step_grad":
        ins, kept = ins[:2], full[0][:, 3:]
        outs = _step64(sc, ins[0], ins[1], kept[:, 0], c["iters"])
    else:
        kept = full[2][:, 3:]
        outs = _upsample64(sc, *ins)
    four = lambda t, w: torch.cat([t.detach(), w], 1)  # noqa: E731
    res = [four(outs[0], kept), four(outs[1], torch.zeros_like(kept))]
    if grad:
        n = len(outs[0])
        g = [_randn(seed + k, n).to(dev).double()[:, :3] for k in (1, 2)]
        for t in torch.autograd.grad(outs, ins, g):
            res.append(four(t, torch.zeros_like(t[:, :1])))
    return res
