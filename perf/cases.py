"""What a user of the framework has it do, as measurable cases over the real range of sizes.

Every case goes through a public entry point (`Scene.smoothed_grad`, `SmoothedLoss`,
`Scene.smoothed_grad_host`, `Scene.render_batch`, resident jobs with `step_batch`) on the
repository's seeded workloads at its configurations' sizes and at odd ones. `exact` is an
independent path tracer in 64 bits over the documented random streams (plain torch).
"""
import math

import numpy as np
import torch

import workloads
from paper_2211_17263_gb300 import api
from paper_2211_17263_gb300.autograd import SmoothedLoss

SCENES = {
    "small": workloads.config_small, "occlusion": workloads.config_occlusion, "gi": workloads.config_gi_box,
    "caustic": workloads.config_caustic, "walls": workloads.config_gi_albedo,
    "albedo": workloads.config_small_albedo, "texture": workloads.config_texture,
}
# closest-hit rays and diffuse vertices per path, and the share of paths whose own rays a
# moved object can meet (the rest are the same in every render under common random numbers)
RAYS = {"small": 1.0, "occlusion": 2.4, "gi": 3.6, "caustic": 2.7, "walls": 3.6, "albedo": 1.0, "texture": 2.0}
DIFFUSE = {"small": 1.0, "occlusion": 2.0, "gi": 2.9, "caustic": 0.55, "walls": 2.9, "albedo": 1.0, "texture": 1.0}
OWN = {"small": 0.1, "occlusion": 0.05, "gi": 1.0, "caustic": 1.0, "walls": 1.0, "albedo": 1.0, "texture": 1.0}
TESTS = {0: 22, 1: 32, 2: 12}  # flops of a ray-sphere, ray-quad and ray-box test


def listed():
    return [
        # The paper's plain method at its smallest (64x64, depth 1, 8 renders): launches and latency.
        dict(name="small-64", call="grad", scene="small", width=64, height=64, spp=4, pairs=4),
        # The occlusion/shadow task as a differentiable loss of a training loop (forward and backward).
        dict(name="occlusion-256", call="autograd", scene="occlusion", width=256, height=256, spp=16, pairs=8),
        # Independent samples per render and no antithetic pairs, Gaussian draws (the ablations), odd size.
        dict(name="occlusion-independent", call="grad", scene="occlusion", width=301, height=173, spp=12, pairs=6,
             crn=0, antithetic=0, sampler=2),
        # Global illumination: light position and two walls' colours, the configuration's size.
        dict(name="gi-512", call="grad", scene="gi", width=512, height=512, spp=32, pairs=16),
        # The same task at an odd size with few renders that no power of two divides, per-dimension draws.
        dict(name="gi-odd", call="grad", scene="gi", width=333, height=217, spp=13, pairs=5, sampler=1),
        # Material parameters with the pathwise estimator (Eq. 9), the configuration's size.
        dict(name="walls-eq9-512", call="grad", scene="walls", width=512, height=512, spp=32, pairs=16, estimator=1),
        # The same parameters with the kernel-gradient estimator (Eq. 10), a preview's size.
        dict(name="walls-eq10-256", call="grad", scene="walls", width=256, height=256, spp=32, pairs=16, sampler=0),
        # The caustic task, the largest configuration, called with host buffers as a host program does.
        dict(name="caustic-512-host", call="host", scene="caustic", width=512, height=512, spp=64, pairs=32),
        # The caustic task small and odd, as in a coarse-to-fine schedule.
        dict(name="caustic-odd", call="grad", scene="caustic", width=237, height=141, spp=20, pairs=12),
        # 49,152 texture parameters.
        dict(name="texture-128", call="grad", scene="texture", res=128, width=256, height=256, spp=4, pairs=8),
        # Forward images: reference views of the box with their own random streams.
        dict(name="render-gi-512", call="render", scene="gi", width=512, height=512, spp=32, n=4, crn=0),
        # Serving: six resident jobs of three tasks, four packed optimisation steps, then their state is read.
        dict(name="serving-6", call="jobs", jobs=6, steps=4, mix=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "occlusion", "gi", "caustic", "walls", "albedo", "texture", "render", "jobs"])
    if kind == "jobs":
        return dict(call="jobs", jobs=rng.randint(1, 10), steps=rng.randint(1, 6), mix=rng.randrange(1 << 20))
    if kind == "texture":
        return dict(call="grad", scene="texture", res=_log_int(rng, 8, 160), width=_log_int(rng, 24, 512),
                    height=_log_int(rng, 24, 512), spp=_log_int(rng, 1, 8), pairs=_log_int(rng, 1, 12),
                    sampler=rng.choice([0, 0, 2]))
    while True:
        size = dict(width=_log_int(rng, 24, 512), height=_log_int(rng, 24, 512), spp=_log_int(rng, 1, 64))
        if kind == "render":
            case = dict(call="render", scene=rng.choice(["small", "occlusion", "gi", "caustic"]), **size,
                        n=_log_int(rng, 1, 16), crn=rng.choice([0, 1]))
        else:
            case = dict(call=rng.choice(["grad", "grad", "autograd", "host"]), scene=kind, **size,
                        pairs=_log_int(rng, 1, 40), sampler=rng.choice([0, 0, 0, 1, 2]), crn=rng.choice([1, 1, 1, 0]),
                        antithetic=rng.choice([1, 1, 1, 0]))
            if kind in ("walls", "albedo") and rng.random() < 0.5:
                case.update(estimator=1, sampler=2)
        paths = _renders(case) * case["width"] * case["height"] * case["spp"]
        if 5e4 < paths < (2.5e8 if case.get("crn", 1) and case["call"] != "render" else 3e7):
            return case


def _renders(case):
    return case["n"] if case["call"] == "render" else 2 * case["pairs"]


def _workload(case, seed):
    """The case's workload: the repository's scene with parameters, start and streams of `seed`."""
    rng = np.random.default_rng([seed, 7])
    kw = {"res": case["res"]} if case["scene"] == "texture" else {}
    wl = SCENES[case["scene"]](seed=seed % (1 << 31), **kw)
    wl = workloads.scaled(wl, width=case["width"], height=case["height"], spp=case["spp"],
                          pairs=case.get("pairs", 1), sampler=case.get("sampler", wl.sampler),
                          antithetic=case.get("antithetic", 1), crn=case.get("crn", 1),
                          estimator=case.get("estimator", 0))
    wl.seed = int(rng.integers(0, 2**31 - 1))
    spread = 0.02 if case["scene"] == "texture" else 0.1
    wl.theta0 = (wl.theta0 + rng.uniform(-spread, spread, size=wl.D)).astype(np.float32)
    return wl


def _jobs(case, seed):
    """The workloads of a serving case: sizes from the case, scenes and starts from `seed`."""
    sizes, out = np.random.default_rng([case["mix"], 3]), []
    for j in range(case["jobs"]):
        res = int(sizes.choice([96, 128, 192, 256]))
        sub = dict(scene=["small", "occlusion", "gi"][j % 3], width=res, height=res, spp=int(sizes.choice([4, 8, 16])),
                   pairs=int(sizes.choice([4, 8, 16])))
        wl = _workload(sub, seed * 16 + j)
        wl.lr, wl.steps = 1e-3, 1000  # late in a descent
        out.append(wl)
    return out


def _target(wl, seed):
    """A photograph-like target [H, W, 4]: smooth shading, one edge and grain, in the scenes' range."""
    rng = np.random.default_rng([seed, 11])
    y, x = np.mgrid[0:wl.height, 0:wl.width].astype(np.float32)
    x, y = x / wl.width, y / wl.height
    img = np.zeros((wl.height, wl.width, 4), np.float32)
    for c in range(3):
        a, b, p = rng.uniform(1, 6), rng.uniform(1, 6), rng.uniform(0, 6)
        img[..., c] = 0.35 + 0.2 * np.sin(a * x + b * y + p) + 0.2 * (x + 0.3 * y > rng.uniform(0.3, 0.9))
    img[..., :3] += rng.uniform(-0.03, 0.03, size=(wl.height, wl.width, 3)).astype(np.float32)
    return np.ascontiguousarray(np.clip(img, 0.0, 1.0), np.float32)


def _thetas(case, wl, seed):
    rng = np.random.default_rng([seed, 13])
    return (wl.theta_ref + rng.uniform(-0.1, 0.1, size=(case["n"], wl.D))).astype(np.float32)


_contexts = []


def _context():
    """The program's one context."""
    if not _contexts:
        _contexts.append(api.Context(0))
    return _contexts[0]


class _Jobs:
    """A server's resident jobs; they go when the state does."""

    def __init__(self, ctx, wls, seed):
        self.ctx = ctx
        self.jobs = [api.Job(ctx.upload_scene(wl.scene, wl.bindings), wl, _target(wl, seed * 16 + j))
                     for j, wl in enumerate(wls)]

    def __del__(self):
        for j in self.jobs:
            j.release()


def prepare(case, seed):
    ctx = _context()
    if case["call"] == "jobs":
        return dict(case=case, jobs=_Jobs(ctx, _jobs(case, seed), seed))
    wl = _workload(case, seed)
    state = dict(case=case, wl=wl, scene=ctx.upload_scene(wl.scene, wl.bindings))
    if case["call"] == "render":
        state["thetas"] = torch.as_tensor(_thetas(case, wl, seed), device="cuda")
        return state
    state["opts"] = state["scene"].grad_opts(wl, step=0)
    target = _target(wl, seed)
    if case["call"] == "host":
        state.update(theta=wl.theta0, sigma=wl.sigma, target=torch.as_tensor(target).pin_memory())
    else:
        theta = torch.as_tensor(wl.theta0, device="cuda").requires_grad_(case["call"] == "autograd")
        state.update(theta=theta, sigma=torch.as_tensor(wl.sigma, device="cuda"),
                     target=torch.as_tensor(target, device="cuda"))
    return state


def run(state):
    case = state["case"]
    if case["call"] == "jobs":
        held = state["jobs"]
        for _ in range(case["steps"]):
            api.step_batch(held.ctx, held.jobs)
        return [{k: v for k, v in j.read().items() if k != "steps"} for j in held.jobs]
    scene, wl = state["scene"], state["wl"]
    if case["call"] == "render":
        return scene.render_batch(state["thetas"], wl.width, wl.height, wl.spp, wl.depth, rr_start=wl.rr_start,
                                  seed=wl.seed, step=0, tag=3, crn=wl.crn)
    args = state["theta"], state["sigma"], state["target"], state["opts"]
    if case["call"] == "host":
        grad, losses = scene.smoothed_grad_host(*args)
    elif case["call"] == "autograd":
        loss = SmoothedLoss.apply(args[0], scene, *args[1:])
        (grad,) = torch.autograd.grad(loss, args[0])
        return {"loss": loss.detach(), "grad": grad}
    else:
        grad, losses = scene.smoothed_grad(*args)
    return {"grad": grad, "losses": losses}


def _work(name, wl, renders):
    pix = wl.width * wl.height
    paths = pix * wl.spp
    tests = sum(TESTS[int(t)] for t in wl.scene.prim_type)
    path = 27.0 + RAYS[name] * (tests + 120.0) + DIFFUSE[name] * tests
    if wl.crn:  # each path once, and each render's own estimates where they can differ
        flops = paths * path + OWN[name] * renders * paths * DIFFUSE[name] * 52.0
        if wl.estimator:
            flops += renders * paths * DIFFUSE[name] * 10.0 * wl.D
    else:
        flops = renders * paths * path
    return dict(bytes=16.0 * pix + 12.0 * wl.D + 4.0 * renders, flops=flops + 60.0 * wl.D * renders)


def work(case):
    if case["call"] == "jobs":
        each = [_work(["small", "occlusion", "gi"][j % 3], wl, wl.renders) for j, wl in enumerate(_jobs(case, 0))]
        return {k: case["steps"] * sum(w[k] for w in each) for k in ("bytes", "flops")}
    wl = _workload(case, 0)
    w = _work(case["scene"], wl, _renders(case))
    if case["call"] == "render":
        w["bytes"] = 16.0 * wl.width * wl.height * case["n"]
    return w


# ---------------------------------------------------------------------------
# The same results in 64 bits: plain torch over the documented streams and conventions
# ---------------------------------------------------------------------------
DEV = "cuda"
EPS = 1e-4  # ray start and surface offset
CHUNK = 1 << 21  # paths at a time
F64 = torch.float64


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 words; c0 and c1 int64 tensors, the others numbers."""
    m32 = 0xFFFFFFFF
    k0, k1 = seed & m32, (seed >> 32) & m32
    a, b = c0, c1
    c, d = torch.full_like(a, c2), torch.full_like(a, c3)
    for _ in range(10):
        p, q = a * 0xD2511F53, c * 0xCD9E8D57
        a, b, c, d = ((q >> 32) & m32) ^ b ^ k0, q & m32, ((p >> 32) & m32) ^ d ^ k1, p & m32
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return [((w >> 9) * 2 + 1).to(F64) / 2.0**24 for w in (a, b, c, d)]


def _draws(wl):
    """Perturbations and weights [2P, D] (Eq. 11): tau rounded to 32 bits as the renders get it."""
    D, anti, n = wl.D, wl.antithetic, (wl.pairs if wl.antithetic else 2 * wl.pairs)
    n_exp, extra = (D + 1) // 2, int(D % 2 == 0)
    count = {0: 2 if D == 1 else n_exp + D + extra + 1, 1: D, 2: D + 1}[wl.sampler]
    blocks = (count + 3) // 4
    c0 = torch.arange(n, device=DEV).repeat_interleave(blocks)
    c1 = torch.arange(blocks, device=DEV).repeat(n)
    u = torch.stack(_philox(c0, c1, 0, 1 << 28, wl.seed), 1).reshape(n, blocks * 4)

    def normals(base, k):
        a, b = u[:, base : base + 2 * ((k + 1) // 2) : 2], u[:, base + 1 : base + 2 * ((k + 1) // 2) : 2]
        r = torch.sqrt(-2.0 * torch.log(a))
        return torch.stack([r * torch.cos(2 * math.pi * b), r * torch.sin(2 * math.pi * b)], 2).reshape(n, -1)[:, :k]

    c_d = math.sqrt(2.0) * math.exp(math.lgamma((D + 1) / 2) - math.lgamma(D / 2))
    if wl.sampler == 0 and D == 1:
        sign = torch.where(u[:, 1:2] < 0.5, -1.0, 1.0)
        t, w = sign * torch.sqrt(-2.0 * torch.log(u[:, :1])), sign * c_d
    elif wl.sampler == 0:
        z = normals(n_exp, D + extra)
        radius = (-2.0 * torch.log(u[:, :n_exp])).sum(1) + (z[:, D:] ** 2).sum(1)
        direction = z[:, :D] / z[:, :D].norm(dim=1, keepdim=True)
        t, w = torch.sqrt(radius)[:, None] * direction, c_d * direction
    elif wl.sampler == 1:
        low = u[:, :D] < 0.5
        t = torch.sqrt(-2.0 * torch.log(2.0 * torch.where(low, u[:, :D], 1.0 - u[:, :D])))
        t, w = torch.where(low, -t, t), torch.where(low, -1.0, 1.0) * math.sqrt(2.0 / math.pi)
    else:
        t = w = normals(0, D)
    sigma = torch.as_tensor(wl.sigma, device=DEV).to(F64)
    t, w = t * sigma, w / sigma
    if anti:
        t, w = torch.stack([t, -t], 1).reshape(-1, D), torch.stack([w, -w], 1).reshape(-1, D)
    return t.to(torch.float32), w


def _bound_scene(wl, theta):
    """Primitives and materials (lists of Python numbers) at 32-bit parameters, and the texture if any."""
    sc = wl.scene
    geom, mats = sc.prim_geom.astype(np.float64), sc.mat_param.astype(np.float64)
    texture = None
    if int(wl.bindings[0, 0]) == workloads.BIND_TEXTURE:
        texture = theta.to(F64).clamp(0.0, 1.0).reshape(-1, 3)
    else:
        for (kind, i, c), v in zip(wl.bindings.tolist(), theta.tolist()):
            if kind == workloads.BIND_PRIM_POS:
                geom[i, c] = v
            elif kind == workloads.BIND_SPHERE_RADIUS:
                geom[i, 3] = abs(v)
            else:
                mats[i, c + (3 if kind == workloads.BIND_MAT_EMISSION else 0)] = v
    mats[:, :3] = np.clip(mats[:, :3], 0.0, 1.0)
    mats[:, 3:6] = np.maximum(mats[:, 3:6], 0.0)
    return geom, mats, texture


def _v(x):
    return torch.tensor([float(q) for q in x], dtype=F64, device=DEV)[:, None]


def _dot(a, b):
    return (a * b).sum(0)


def _unit(a):
    return a / torch.sqrt(_dot(a, a))


class _Tracer:
    """Path tracing of one bound scene for arrays of paths, vectors as [3, n]."""

    def __init__(self, wl, theta):
        self.wl = wl
        self.geom, self.mats, self.texture = _bound_scene(wl, theta)
        self.type, self.mat = wl.scene.prim_type.tolist(), wl.scene.prim_mat.tolist()
        self.mat_type = torch.as_tensor(wl.scene.mat_type, device=DEV).to(torch.int64)
        self.table = torch.as_tensor(self.mats, device=DEV)
        self.bg = _v(wl.scene.background)
        self.prims = []
        for t, g in zip(self.type, self.geom):
            if t == 0:
                self.prims.append((_v(g[:3]), float(g[3])))
            elif t == 1:
                u, v = g[3:6], g[6:9]
                n = np.cross(u, v)
                self.prims.append((_v(g[:3]), _v(n / np.linalg.norm(n)), _v(u), float(u @ u), _v(v), float(v @ v)))
            else:
                self.prims.append((_v(g[:3] - g[3:6]), _v(g[:3] + g[3:6])))
        self.lights = [i for i, m in enumerate(self.mat) if self.type[i] != 2 and self.mats[m, 3:6].max() > 0]
        cam = wl.scene.camera.astype(np.float64)
        f = cam[3:6] - cam[:3]
        f = f / np.linalg.norm(f)
        r = np.cross(f, cam[6:9])
        r = r / np.linalg.norm(r)
        self.camera = _v(cam[:3]), _v(f), _v(r), _v(np.cross(r, f)), math.tan(0.5 * math.radians(cam[9]))

    def hit(self, i, o, d):
        """Distance along the ray to primitive i (inf: missed)."""
        p, inf = self.prims[i], math.inf
        if self.type[i] == 0:
            oc = o - p[0]
            b = _dot(oc, d)
            l = oc - d * b
            disc = p[1] * p[1] - _dot(l, l)
            sq = torch.sqrt(disc.clamp(min=0.0))
            t = torch.where(-b - sq > EPS, -b - sq, -b + sq)
            return torch.where((disc > 0) & (t > EPS), t, inf)
        if self.type[i] == 1:
            den = _dot(p[1], d)
            co = p[0] - o
            t = _dot(p[1], co) / den
            q = d * t - co
            inside = (_dot(q, p[2]).abs() <= 0.5 * p[3]) & (_dot(q, p[4]).abs() <= 0.5 * p[5])
            return torch.where((den.abs() >= 1e-12) & (t > EPS) & inside, t, inf)
        a, b = (p[0] - o) / d, (p[1] - o) / d
        near, far = torch.minimum(a, b).amax(0), torch.maximum(a, b).amin(0)
        t = torch.where(near > EPS, near, far)
        return torch.where((near <= far) & (t > EPS), t, inf)

    def normal(self, i, pt, o, d):
        p = self.prims[i]
        if self.type[i] == 0:
            return (pt - p[0]) / p[1]
        if self.type[i] == 1:
            return p[1].expand_as(pt)
        a, b = (p[0] - o) / d, (p[1] - o) / d
        near, axis_n = torch.minimum(a, b).max(0)
        axis_f = torch.maximum(a, b).min(0).indices
        entering = near > EPS
        axis = torch.where(entering, axis_n, axis_f)[None]
        s = torch.where(d.gather(0, axis) > 0, 1.0, -1.0) * torch.where(entering, -1.0, 1.0)
        return torch.zeros_like(pt).scatter(0, axis, s.to(F64))

    def light_sample(self, po, ns, pick, lu, lv):
        """Direction and geometry term of the estimate at each vertex, zero where it is not visible."""
        g, w_all = torch.zeros_like(lu), torch.zeros_like(po)
        which = (pick * len(self.lights)).to(torch.int64).clamp(max=len(self.lights) - 1)
        for k, i in enumerate(self.lights):
            p = self.prims[i]
            if self.type[i] == 1:
                y = p[0] + p[2] * (lu - 0.5) + p[4] * (lv - 0.5)
                ny = p[1].expand_as(y)
                area = float(torch.linalg.cross(p[2][:, 0], p[4][:, 0]).norm())
            else:
                z = 1.0 - 2.0 * lu
                rr = torch.sqrt((1.0 - z * z).clamp(min=0.0))
                ny = torch.stack([rr * torch.cos(2 * math.pi * lv), rr * torch.sin(2 * math.pi * lv), z])
                y = p[0] + ny * p[1]
                area = 4.0 * math.pi * p[1] * p[1]
            dv = y - po
            dist = torch.sqrt(_dot(dv, dv))
            w = dv / dist
            cx, cl = _dot(ns, w), -_dot(ny, w)
            ok = (which == k) & (cx > 0) & (cl > 0)
            for q in range(len(self.prims)):
                if q != i:
                    ok &= ~(self.hit(q, po, w) < dist)
            g = torch.where(ok, cx * cl / (dist * dist) * area * len(self.lights) / math.pi, g)
        return g, which

    def paths(self, pixel, sample, field, tag, seed, diff):
        """Radiance [3, n] of the paths and, for diff = [(material, channel, emission?)], its tangents [K, n]."""
        wl, n = self.wl, pixel.numel()
        out, tout = torch.zeros(3, n, dtype=F64, device=DEV), torch.zeros(len(diff), n, dtype=F64, device=DEV)
        c3 = (tag << 28) | field

        def words(b, slot):
            return _philox(pixel, sample | (b << 16) | (slot << 24), 0, c3, seed)

        eye, f, r, up, th = self.camera
        j = words(0, 2)
        x, y = (pixel % wl.width).to(F64), (pixel // wl.width).to(F64)
        sx = (2 * x - wl.width + 2 * j[0]) / wl.width * th * wl.width / wl.height
        sy = (wl.height - 2 * y - 2 * j[1]) / wl.height * th
        o, d = eye.expand(3, n), _unit(f + r * sx + up * sy)
        beta, ident = torch.ones(3, n, dtype=F64, device=DEV), torch.arange(n, device=DEV)
        specular = torch.ones(n, dtype=torch.bool, device=DEV)
        db = torch.zeros_like(tout)
        for b in range(wl.depth):
            t = torch.full_like(beta[0], math.inf)
            which = torch.full_like(ident, -1)
            for i in range(len(self.prims)):
                ti = self.hit(i, o, d)
                which = torch.where(ti < t, i, which)
                t = torch.minimum(t, ti)
            gone = which < 0
            out[:, ident[gone]] += beta[:, gone] * self.bg
            for k, (_, c, _) in enumerate(diff):
                tout[k, ident[gone]] += db[k, gone] * self.bg[c]
            keep = ~gone
            o, d, t, beta, which, ident = o[:, keep], d[:, keep], t[keep], beta[:, keep], which[keep], ident[keep]
            pixel, sample, specular, db = pixel[keep], sample[keep], specular[keep], db[:, keep]
            if not ident.numel():
                break
            pt = o + d * t
            ng = torch.zeros_like(pt)
            mat = torch.zeros_like(ident)
            for i in range(len(self.prims)):
                at = which == i
                ng = torch.where(at, self.normal(i, pt, o, d), ng)
                mat = torch.where(at, self.mat[i], mat)
            par = self.table[mat].T
            albedo, emission = par[:3], par[3:6]
            if self.texture is not None:
                p = self.prims[0]
                T = int(self.wl.bindings[0, 2])
                s = ((_dot(pt - p[0], p[2]) / p[3] + 0.5) * T).floor().to(torch.int64).clamp(0, T - 1)
                v = ((_dot(pt - p[0], p[4]) / p[5] + 0.5) * T).floor().to(torch.int64).clamp(0, T - 1)
                albedo = self.texture[v * T + s].T
            seen = (specular & (emission.amax(0) > 0) & (_dot(d, ng) < 0)).to(F64)
            out[:, ident] += beta * emission * seen
            for k, (m, c, e) in enumerate(diff):
                own = beta[c] * self.clamped[k] * (mat == m) if e else 0.0
                tout[k, ident] += (db[k] * emission[c] + own) * seen
            last = b + 1 >= wl.depth
            u0, u1 = words(b, 0), words(b, 1)
            kind = self.mat_type[mat]
            diffuse = kind == 0
            cos = _dot(ng, d)
            ns = torch.where(cos < 0, ng, -ng)
            po = pt + ns * EPS
            if self.lights:
                g, li = self.light_sample(po, ns, u1[0], u0[0], u0[1])
                g = torch.where(diffuse, g, 0.0)
                lm = torch.as_tensor([self.mat[i] for i in self.lights], device=DEV)[li]
                le = self.table[lm].T[3:6]
                out[:, ident] += beta * albedo * le * g
                for k, (m, c, e) in enumerate(diff):
                    own = beta[c] * (albedo[c] * (lm == m) if e else le[c] * (mat == m)) * self.clamped[k]
                    tout[k, ident] += (db[k] * albedo[c] * le[c] + own) * g
            if last:
                break
            # scattered direction and start: diffuse (cosine), mirror, dielectric
            rad, phi = torch.sqrt(u0[2]), 2 * math.pi * u0[3]
            sg = torch.where(ns[2] >= 0, 1.0, -1.0)
            a = -1.0 / (sg + ns[2])
            t1 = torch.stack([1 + sg * ns[0] * ns[0] * a, sg * ns[0] * ns[1] * a, -sg * ns[0]])
            t2 = torch.stack([ns[0] * ns[1] * a, sg + ns[1] * ns[1] * a, -ns[1]])
            new = t1 * (rad * torch.cos(phi)) + t2 * (rad * torch.sin(phi)) + ns * torch.sqrt((1 - u0[2]).clamp(min=0))
            start = po
            if bool((kind == 1).any()):
                new = torch.where(kind == 1, d - ns * (2 * _dot(d, ns)), new)
            if bool((kind == 2).any()):
                ior, ci = par[6], -cos
                outside = ci > 0
                eta, ci = torch.where(outside, 1.0 / ior, ior), ci.abs()
                s2 = eta * eta * (1 - ci * ci)
                ct = torch.sqrt((1 - s2).clamp(min=0.0))
                rs, rp = (eta * ci - ct) / (eta * ci + ct), (ci - eta * ct) / (ci + eta * ct)
                mirror = u1[2] < torch.where(s2 >= 1, 1.0, 0.5 * (rs * rs + rp * rp))
                bent = torch.where(mirror, d + ns * (2 * ci), d * eta + ns * (eta * ci - ct))
                new = torch.where(kind == 2, bent, new)
                start = torch.where((kind == 2) & ~mirror, pt - ns * EPS, start)
            for k, (m, c, e) in enumerate(diff):
                db[k] = db[k] * albedo[c] + (0.0 if e else beta[c] * self.clamped[k] * (mat == m))
            beta, o, d, specular = beta * albedo, start, _unit(new), ~diffuse
            keep = beta.amax(0) > 0
            if wl.rr_start >= 0 and b >= wl.rr_start:
                q = beta.amax(0).clamp(max=0.95)
                keep &= u1[1] < q
                beta, db = beta / q, db / q
            o, d, beta, ident, pixel = o[:, keep], d[:, keep], beta[:, keep], ident[keep], pixel[keep]
            sample, specular, db = sample[keep], specular[keep], db[:, keep]
        return out, tout

    def image(self, field, tag, diff=(), theta=None):
        """Mean image [3, H W] and its tangents [K, H W]."""
        wl = self.wl
        if diff:
            at = theta.tolist()
            self.clamped = [float(v >= 0) if e else float(0 <= v <= 1) for v, (_, _, e) in zip(at, diff)]
        pix, step = wl.width * wl.height, max(1, CHUNK // wl.spp)
        img, tan = torch.empty(3, pix, dtype=F64, device=DEV), torch.empty(len(diff), pix, dtype=F64, device=DEV)
        for p0 in range(0, pix, step):
            p1 = min(pix, p0 + step)
            pixel = torch.arange(p0, p1, device=DEV).repeat_interleave(wl.spp)
            sample = torch.arange(wl.spp, device=DEV).repeat(p1 - p0)
            L, T = self.paths(pixel, sample, field, tag, wl.seed, diff)
            img[:, p0:p1] = L.reshape(3, p1 - p0, wl.spp).mean(2)
            tan[:, p0:p1] = T.reshape(len(diff), p1 - p0, wl.spp).mean(2)
        return img, tan


def _estimate(wl, theta, target, step=0):
    """Gradient [D] and losses [2P] at 32-bit theta."""
    tau, w = _draws(wl)
    target = torch.as_tensor(target, device=DEV).to(F64).reshape(-1, 4)[:, :3].T
    diff = [(m, c, kind == workloads.BIND_MAT_EMISSION) for kind, m, c in wl.bindings.tolist()] if wl.estimator else []
    losses, grads = [], []
    for r in range(2 * wl.pairs):
        at = theta + tau[r]
        img, tan = _Tracer(wl, at).image(0 if wl.crn else r + 1, 2, diff, at)
        e = img - target
        losses.append((e * e).mean())
        grads.append(torch.stack([2.0 / e.numel() * (e[c] * tan[k]).sum() for k, (_, c, _) in enumerate(diff)])
                     if diff else None)
    losses = torch.stack(losses)
    if diff:
        return torch.stack(grads).mean(0), losses
    if wl.antithetic:
        return (w[::2] * (losses[::2] - losses[1::2])[:, None]).sum(0) / (2 * wl.pairs), losses
    return (w * losses[:, None]).mean(0), losses


def exact(case, seed):
    if case["call"] == "jobs":
        return None  # several steps of several jobs: each step's start depends on the last one's rounding
    wl = _workload(case, seed)
    rays = _renders(case) * wl.width * wl.height * wl.spp * RAYS[case["scene"]] * len(wl.scene.prim_type)
    if rays > 9e8:  # beyond about 20 seconds
        return None
    if case["call"] == "render":
        thetas = torch.as_tensor(_thetas(case, wl, seed), device=DEV)
        img = [_Tracer(wl, t).image(0 if wl.crn else i, 3)[0] for i, t in enumerate(thetas)]
        img = torch.stack(img).reshape(case["n"], 3, wl.height, wl.width).permute(0, 2, 3, 1)
        return torch.nn.functional.pad(img, (0, 1))
    grad, losses = _estimate(wl, torch.as_tensor(wl.theta0, device=DEV), _target(wl, seed))
    if case["call"] == "autograd":
        return {"loss": losses.mean(), "grad": grad}
    return {"grad": grad, "losses": losses}
