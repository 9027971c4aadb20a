"""The work a user of this library has it do, as measurable cases.

Every case runs the public entry points (paper_2509_18497_gb300.rgs / .api) on seeded
scenes of the kinds the library ships generators for (scenes.py): the small box, the fruit
bowl, many lights, the environment map, uneven scene batches, the textured room.  A case is
a dict of plain values; `kind` says which calls `run` makes:

  forward   build, trace, solve                                (previewing a scene)
  step      build, trace, solve, adjoint                       (one step of a fit, handles kept)
  autograd  api.radiosity and its backward                     (a fit in plain PyTorch)
  geometry  api.radiosity_geometry and its backward            (a fit of the geometry as well)
  batch     build + trace per scene, one batched solve, adjoint per scene
  pairs     build, center-to-center trace, solve, adjoint with the lambda gradient
  shooting  progressive refinement on a traced center-to-center transport
  render, render_adjoint   an image of a solved scene, and dL/dB from dL/dimage

`exact` is the same mathematics written plainly in 64 bits with torch: brute-force hit
lists, dense compositing, gradients by torch's autograd.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2509_18497_gb300 import api, rgs, scenes



def _case(name, kind, scene, n, L, nd, nb, lights, **more):
    return dict(name=name, kind=kind, scene=scene, n=n, L=L, nd=nd, nb=nb, lights=lights, **more)


def listed():
    return [
        # the smallest call: preview of a small enclosed scene, where launches and latency count
        _case("box_forward", "forward", "box", 2000, 2, 64, 3, 1),
        # one training iteration written in PyTorch: a small object, handles made per call
        _case("bowl_autograd", "autograd", "bowl", 3001, 3, 128, 3, 2),
        # the object-in-scene reconstruction step at its full size, FP32
        _case("bowl_step", "step", "bowl", 50000, 3, 256, 4, 1, precision="fp32"),
        # many lights as right-hand sides (light-stage capture), batched precision
        _case("many_lights", "step", "bowl", 16000, 3, 256, 4, 100, precision="rescorr"),
        # relighting under the 16 x 32 environment map, 512 distant lights
        _case("env_map", "step", "bowl", 3000, 3, 128, 3, 512, precision="rescorr", env=True),
        # several scenes of uneven size solved in one launch
        _case("uneven_batch", "batch", "uneven", 0, 0, 0, 0, 8, precision="rescorr", count=8, scale=0.1),
        # a large interior with a moderate light count, automatic checkpointing
        _case("room_step", "step", "room", 60000, 3, 128, 4, 16, precision="rescorr", checkpoint=-1),
        # the approximated transport with its learned scale lambda
        _case("pairs_step", "pairs", "bowl", 4000, 3, 0, 3, 1, precision="fp32"),
        # fitting positions, scales and rotations as well
        _case("geometry", "geometry", "bowl", 8000, 3, 128, 3, 1),
        # a full-HD view of a solved scene, and the transpose that a loss on a view needs
        _case("render_hd", "render", "bowl", 50000, 3, 32, 1, 1, width=1920, height=1080),
        _case("render_adjoint", "render_adjoint", "bowl", 20000, 3, 32, 1, 4, width=960, height=540),
        # the shooting phase of the hybrid solver
        _case("shooting", "shooting", "bowl", 2500, 2, 0, 0, 1, shots=400),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "step", "many", "env", "room", "autograd", "geometry", "batch", "pairs", "shooting",
                       "render", "render_adjoint"])
    L = rng.choice([1, 2, 3, 3])
    prec = rng.choice(["fp32", "rescorr"])
    model = rng.choice(["gauss", "gauss", "gfsgs"])
    nd = rng.choice([32, 64, 96, 128, 160, 256])
    nb = rng.randint(2, 5)
    if kind == "forward":
        return dict(kind="forward", scene=rng.choice(["box", "bowl"]), n=_log_int(rng, 500, 20000), L=L, nd=nd, nb=nb,
                    lights=1, model=model)
    if kind == "step":
        return dict(kind="step", scene="bowl", n=_log_int(rng, 500, 40000), L=L, nd=nd, nb=nb,
                    lights=rng.randint(1, 4), precision=prec, model=model)
    if kind == "many":
        nl = _log_int(rng, 24, 120)
        n = min(_log_int(rng, 1000, 16000), int(3.2e8 / (nl * nd)))
        return dict(kind="step", scene="bowl", n=n, L=3, nd=nd, nb=rng.randint(2, 4), lights=nl, precision="rescorr")
    if kind == "env":
        return dict(kind="step", scene="bowl", n=_log_int(rng, 800, 3000), L=3, nd=rng.choice([64, 96, 128]), nb=3,
                    lights=16 * rng.choice([8, 16, 24, 32]), precision="rescorr", env=True)
    if kind == "room":
        return dict(kind="step", scene="room", n=_log_int(rng, 10000, 50000), L=L, nd=rng.choice([64, 96, 128]),
                    nb=rng.randint(2, 4), lights=rng.randint(4, 16), precision=prec, checkpoint=rng.choice([0, -1, 2]))
    if kind == "autograd":
        return dict(kind="autograd", scene="bowl", n=_log_int(rng, 500, 10000), L=L, nd=nd, nb=nb,
                    lights=rng.randint(1, 3), model=model)
    if kind == "geometry":
        return dict(kind="geometry", scene="bowl", n=_log_int(rng, 500, 8000), L=L, nd=rng.choice([32, 64, 96, 128]),
                    nb=rng.randint(2, 3), lights=rng.randint(1, 2), model=model)
    if kind == "batch":
        return dict(kind="batch", scene="uneven", n=0, L=0, nd=0, nb=0, lights=rng.randint(1, 8),
                    precision=prec, count=rng.randint(2, 8), scale=round(rng.uniform(0.02, 0.09), 3))
    if kind == "pairs":
        return dict(kind="pairs", scene="bowl", n=_log_int(rng, 500, 4000), L=L, nd=0, nb=rng.randint(1, 3),
                    lights=rng.randint(1, 2), precision=prec, model=model)
    if kind == "shooting":
        return dict(kind="shooting", scene="bowl", n=_log_int(rng, 500, 3000), L=L, nd=0, nb=0, lights=1,
                    shots=_log_int(rng, 50, 400))
    return dict(kind=kind, scene="bowl", n=_log_int(rng, 2000, 50000), L=L, nd=32, nb=1, lights=rng.randint(1, 4),
                width=_log_int(rng, 200, 1280), height=_log_int(rng, 150, 720), model=model)


# ------------------------------------------------------------------ inputs
MODELS = {"gauss": rgs.RGS_ALPHA_GAUSS, "gfsgs": rgs.RGS_ALPHA_GFSGS}
PRECISIONS = {"fp32": rgs.RGS_FP32, "rescorr": rgs.RGS_BF16_FP32ACC_RESCORR}
FOV = 0.7


def _batch_shapes(case):
    out = []
    for q in range(case["count"]):
        rng = np.random.default_rng(1000 + q)
        n = int(round(math.exp(rng.uniform(math.log(5e3), math.log(3e5))) * case["scale"]))
        out.append((n, int(rng.choice([2, 3])), int(rng.choice([128, 192, 256])), int(rng.choice([3, 4, 5]))))
    return out


def _placed(make, seed, **kw):
    """make(seed=seed, ...); the bowl generator cannot place its twelve fruits for a few seeds
    in a thousand: the next seed of a fixed sequence stands in."""
    while True:
        try:
            return make(seed=seed, **kw)
        except RuntimeError:
            seed = (seed + 104729) & 0x7FFFFFFF


def _scenes(case, seed):
    """The numpy scene dicts of a case (one, or one per scene of a batch), from the seed alone."""
    seed = int(seed) & 0x7FFFFFFF
    if case["kind"] == "batch":
        # the shapes of scenes.uneven_batch (its draw from seed 1000 on), the contents from this seed
        out = []
        for q, (n, L, nd, nb) in enumerate(_batch_shapes(case)):
            out.append(_placed(scenes.fruit_bowl, seed + 7919 * q, n=n, L=L, nd=nd, nb=nb, n_lights=case["lights"]))
    else:
        kw = dict(n=case["n"], L=case["L"], nd=max(case["nd"], 32), nb=case["nb"])
        if case["scene"] == "box":
            sc = scenes.box_scene(seed=seed, **kw)
        elif case["scene"] == "room":
            sc = _placed(scenes.large_scene, seed, n_lights=case["lights"], **kw)
        else:
            sc = _placed(scenes.fruit_bowl, seed, n_lights=1 if case.get("env") else case["lights"], **kw)
        if case.get("env"):
            sc = scenes.with_env_map(sc, 16, case["lights"] // 16, seed=seed)
        out = [sc]
    rng = np.random.default_rng(seed + 1)
    if case["kind"] == "pairs":
        out[0]["lam"] = rng.uniform(0.5, 1.5, size=case["n"])
    # a fit starts from some emission: small, in every coefficient
    for sc in out:
        nc = (sc["L"] + 1) ** 2
        sc["E"] = (rng.uniform(0.0, 0.1, size=(sc["n"], nc, 3)) * np.where(np.arange(nc) == 0, 1.0, 0.2)[:, None]).astype(
            np.float32)
    return out


def _normal(shape, seed, device):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return torch.randn(shape, generator=g, device=device, dtype=torch.float32)


def _camera(seed):
    a = 0.3 + 0.1 * (int(seed) % 60)
    eye = np.array([4.4 * math.sin(a), 2.6, 4.4 * math.cos(a)])
    f = np.array([0.0, 0.5, 0.0]) - eye
    return [float(np.float32(v)) for v in (*eye, *(f / np.linalg.norm(f)), 0.0, 1.0, 0.0)]


def _solved_B(sc, C, seed, device):
    """Radiance of plausible shape for the image cases: a positive mean and small higher bands."""
    nc = (sc["L"] + 1) ** 2
    B = 0.05 * _normal((sc["n"], nc, C), seed + 5, device)
    B[:, 0] = B[:, 0].abs() * 10.0 + 0.2
    return B


def prepare(case, seed):
    scs = _scenes(case, seed)
    data = [api.upload(sc) for sc in scs]
    cols = [3 * max(int(d["light_pos"].shape[0]), 1) for d in data]
    pipes = [api.Pipeline(MODELS[case.get("model", "gauss")], PRECISIONS[case.get("precision", "fp32")],
                          checkpoint=case.get("checkpoint", 0), pairs=case["kind"] in ("pairs", "shooting"))
             for _ in data]
    st = dict(kind=case["kind"], case=dict(case), data=data, pipes=pipes)
    kind = case["kind"]
    if kind in ("step", "batch", "pairs", "autograd", "geometry"):
        st["grad"] = [_normal((d["n"], (d["L"] + 1) ** 2, c), seed + 3, "cuda") for d, c in zip(data, cols)]
    if kind == "batch":
        st["B"] = [torch.empty_like(g) for g in st["grad"]]
    if kind in ("autograd", "geometry"):
        d = data[0]
        keys = ("E", "ad", "o") + (("p", "s", "tu", "tv") if kind == "geometry" else ())
        st["leaves"] = [d[k].clone().requires_grad_(True) for k in keys]
    if kind in ("render", "render_adjoint", "shooting"):
        pipes[0].build(data[0])
        pipes[0].trace(data[0])
        st["cam"] = _camera(seed)
        if kind == "render":
            st["B"] = _solved_B(scs[0], cols[0], seed, "cuda")
        elif kind == "render_adjoint":
            st["dimg"] = _normal((case["height"], case["width"], cols[0]), seed + 4, "cuda")
    return st


def run(state):
    kind, case = state["kind"], state["case"]
    d, pipe = state["data"][0], state["pipes"][0]
    if kind == "forward":
        pipe.build(d)
        pipe.trace(d)
        return pipe.solve(d["E"], d["nb"])[0]
    if kind == "step":
        B, grads = pipe.step(d, state["grad"][0])
        return [B, *grads]
    if kind == "pairs":
        pipe.build(d)
        pipe.trace(d)
        B, _ = pipe.solve(d["E"], d["nb"])
        return [B, *pipe.adjoint_pairs(state["grad"][0])]
    if kind == "batch":
        for p, x in zip(state["pipes"], state["data"]):
            p.build(x)
            p.trace(x)
        rgs.rgs_solve_batched([p.transport for p in state["pipes"]], [x["E"] for x in state["data"]],
                              [x["nb"] for x in state["data"]], precision=pipe.precision, B_outs=state["B"])
        grads = [p.adjoint(g) for p, g in zip(state["pipes"], state["grad"])]
        return [[B, *g] for B, g in zip(state["B"], grads)]
    if kind in ("autograd", "geometry"):
        fn = api.radiosity if kind == "autograd" else api.radiosity_geometry
        B = fn(*state["leaves"], d, d["nb"], pipe.alpha_model)
        return [B.detach(), *torch.autograd.grad(B, state["leaves"], state["grad"][0])]
    if kind == "render":
        return rgs.rgs_render(pipe.transport, state["B"], state["cam"], case["width"], case["height"], FOV)
    if kind == "render_adjoint":
        return rgs.rgs_render_adjoint(pipe.transport, state["dimg"], state["cam"], case["width"], case["height"], FOV)
    return rgs.rgs_prog_refine(pipe.transport, case["shots"], E=d["E"])


# ------------------------------------------------------------------ what a pass cannot do without
HITS_PER_RAY = 19.0  # stored hits of a hemisphere or pixel ray on these scenes (16 - 21)


def _sizes(case):
    return _batch_shapes(case) if case["kind"] == "batch" else [(case["n"], case["L"], case["nd"], case["nb"])]


def work(case):
    kind, C = case["kind"], 3 * case["lights"]
    by = fl = 0.0
    for n, L, nd, nb in _sizes(case):
        nc = (L + 1) ** 2
        by += n * (19 + 3 * nc) * 4.0 + n * nc * C * 4.0  # surfels and emission in, B (or dL/dB) out
        if kind in ("step", "batch", "pairs", "autograd", "geometry"):
            by += n * nc * C * 4.0 + n * (3 * nc + 4) * 4.0  # dL/dB in; dL/dE, dL/da^d, dL/do out
        if kind == "geometry":
            by += n * 11 * 4.0
        # per hit and column: the source row's dot product, forward, transposed and for the weights
        per_hit = 2.0 * nc * C
        passes = nb if kind == "forward" else 3 * nb
        if kind in ("pairs", "shooting"):
            hits = 0.5 * n * n if kind == "pairs" else 0.5 * n * case["shots"]
            fl += hits * per_hit * (3 * max(nb, 1) if kind == "pairs" else 2)
        elif kind in ("render", "render_adjoint"):
            px = case["width"] * case["height"]
            by += px * C * 4.0
            fl += px * HITS_PER_RAY * per_hit
        else:
            fl += n * nd * HITS_PER_RAY * per_hit * passes
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------ 64-bit values
CHUNK = 1 << 26  # (ray, surfel) tests at a time
MAX_TESTS = 1.6e11
MAX_VALUES = 6.0e11  # hits x columns x coefficients over all bounces


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _sh(L, v):
    """Real orthonormal SH to degree L with the Condon-Shortley phase, [..., (L+1)^2]."""
    x, y, z = v.unbind(-1)
    s = math.sqrt
    Y = [torch.full_like(x, s(1 / (4 * math.pi)))]
    if L >= 1:
        c = s(3 / (4 * math.pi))
        Y += [-c * y, c * z, -c * x]
    if L >= 2:
        c, c0 = s(15 / math.pi) / 2, s(5 / math.pi) / 4
        Y += [c * x * y, -c * y * z, c0 * (3 * z * z - 1), -c * x * z, c / 2 * (x * x - y * y)]
    if L >= 3:
        c3, c2, c1, c0 = s(35 / (2 * math.pi)) / 4, s(105 / math.pi) / 2, s(21 / (2 * math.pi)) / 4, s(7 / math.pi) / 4
        Y += [-c3 * y * (3 * x * x - y * y), c2 * x * y * z, -c1 * y * (5 * z * z - 1), c0 * z * (5 * z * z - 3),
              -c1 * x * (5 * z * z - 1), c2 / 2 * z * (x * x - y * y), -c3 * x * (x * x - 3 * y * y)]
    return torch.stack(Y, -1)


def _mix64(x):
    """SplitMix64's output function on a uint64 array."""
    with np.errstate(over="ignore"):
        z = x + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


class _Exact:
    """A scene in 64 bits on the GPU; `grads` names the inputs that gradients are wanted for."""

    def __init__(self, sc, model, grads=()):
        put = lambda v: torch.as_tensor(np.asarray(v, np.float32).astype(np.float64), device="cuda")
        self.sc, self.model, self.L, self.n = sc, model, sc["L"], sc["n"]
        self.x = {k: put(sc[k]) for k in (*api.SURFEL_KEYS, "E")}
        self.x["lam"] = put(sc["lam"]) if sc.get("lam") is not None else torch.ones(sc["n"], dtype=torch.float64, device="cuda")
        self.lpos, self.lint = put(sc["light_pos"]).reshape(-1, 3), put(sc["light_I"]).reshape(-1, 3)
        self.nl, self.far = self.lpos.shape[0], bool(sc.get("light_dir", False))
        self.C = 3 * max(self.nl, 1)
        for k in grads:
            self.x[k].requires_grad_(True)
        x = self.x
        a = _unit(x["tu"])
        b = _unit(x["tv"] - (a * x["tv"]).sum(-1, keepdim=True) * a)
        self.U, self.V, self.N = a, b, torch.linalg.cross(a, b)
        ext = x["p"].detach().amax(0) - x["p"].detach().amin(0)
        self.eps = 1e-5 * float(ext.norm())
        s, k = x["shin"], x["k"][:, None]
        rho = [torch.ones_like(s), (s + 1) / (s + 2), s / (s + 3), (s + 1) * (s - 1) / ((s + 2) * (s + 4))]
        band = [4 * k * x["ad"] + (1 - k) * x["as_"]] + [(1 - k) * x["as_"] * r[:, None] for r in rho[1:]]
        self.c = torch.stack([band[l] for l in range(self.L + 1) for _ in range(2 * l + 1)], 1)  # [n, nc, 3]
        self.ch = torch.arange(self.C, device="cuda") % 3

    def alpha(self, o, q2):
        G = torch.exp(-0.5 * q2)
        return o * G if self.model == "gauss" else 1 - torch.exp(-0.03279 * (o * G) ** 3.4)

    def alpha0(self):
        return self.alpha(self.x["o"], torch.zeros_like(self.x["o"]))

    def reflect(self, n, d):
        return 2 * (n * d).sum(-1, keepdim=True) * n - d

    @torch.no_grad()
    def find(self, o, d, own, tmax=None, other=None):
        """(ray, surfel) of every hit, by testing every surfel: o, d [R, 3], own [R] (-1: none);
        other [R]: the segment's end, whose plane rule holds too."""
        p, U, V, N = (v.detach() for v in (self.x["p"], self.U, self.V, self.N))
        su, sv = self.x["s"].detach().unbind(-1)
        rays, surf, step = [], [], max(1, CHUNK // self.n)
        Np, Up, Vp = (N * p).sum(-1), (U * p).sum(-1), (V * p).sum(-1)
        for r0 in range(0, o.shape[0], step):
            oc, dc, ow = o[r0:r0 + step], d[r0:r0 + step], own[r0:r0 + step]
            h = Np - oc @ N.T
            t = h / (dc @ N.T)
            ok = (h.abs() > self.eps) & (t > 0)
            if tmax is not None:
                ok &= t < tmax[r0:r0 + step, None]
            u = (oc @ U.T - Up + t * (dc @ U.T)) / su
            v = (oc @ V.T - Vp + t * (dc @ V.T)) / sv
            ok &= u * u + v * v <= 9.0
            has = (ow >= 0).nonzero()[:, 0]
            ok[has, ow[has]] = False
            if other is not None:
                ot = other[r0:r0 + step]
                ok &= (p[ot] @ N.T - Np).abs() > self.eps
                ok[torch.arange(ok.shape[0], device=ok.device), ot] = False
            r, j = ok.nonzero(as_tuple=True)
            rays.append(r + r0)
            surf.append(j)
        return torch.cat(rays), torch.cat(surf)

    def cross(self, o, d, j):
        """t and u^2 + v^2 where the rays (o, d) meet the planes of surfels j."""
        p, n = self.x["p"][j], self.N[j]
        t = (n * (p - o)).sum(-1) / (n * d).sum(-1)
        q = o + t[:, None] * d - p
        s = self.x["s"][j]
        return t, ((q * self.U[j]).sum(-1) / s[:, 0]) ** 2 + ((q * self.V[j]).sum(-1) / s[:, 1]) ** 2

    def composite(self, o, d, own):
        """(ray, surfel, weight) of the hits of the rays, nearest first, equal depths by index."""
        R = o.shape[0]
        with torch.no_grad():
            ray, j = self.find(o.detach(), d.detach(), own)
            t, _ = self.cross(o[ray], d[ray], j)
            by = torch.argsort(t, stable=True)
            by = by[torch.argsort(ray[by], stable=True)]
            ray, j, t = ray[by], j[by], t[by]
            new = torch.ones_like(ray, dtype=torch.bool)
            new[1:] = (ray[1:] != ray[:-1]) | (t[1:] - t[:-1] > 1e-6 * t[:-1].clamp(min=1.0))
            by = torch.argsort(torch.cumsum(new, 0) * self.n + j)
            ray, j = ray[by], j[by]
            cnt = torch.bincount(ray, minlength=R)
            pos = torch.arange(ray.shape[0], device=ray.device) - (torch.cumsum(cnt, 0) - cnt)[ray]
        _, q2 = self.cross(o[ray], d[ray], j)
        al = self.alpha(self.x["o"][j], q2)
        # transmittance in front of every hit: products down the rays, a block of rays at a time
        T = torch.ones_like(al)
        width = int(cnt.max()) + 1 if ray.numel() else 1
        parts, step = [], max(1, (1 << 27) // width)
        for r0 in range(0, R, step):
            at = torch.searchsorted(ray, torch.tensor([r0, min(r0 + step, R)], device=ray.device))
            a, b = int(at[0]), int(at[1])
            om = torch.ones((min(step, R - r0), width), dtype=torch.float64, device=ray.device)
            om = om.index_put((ray[a:b] - r0, pos[a:b] + 1), 1 - al[a:b]) if b > a else om
            parts.append(torch.cumprod(om, 1)[ray[a:b] - r0, pos[a:b]])
        T = torch.cat(parts) if parts else T
        keep = (T.detach() >= 1e-6).nonzero()[:, 0]
        return ray[keep], j[keep], (al * T)[keep]

    def direct(self):
        """D [n, nc, C]: shadow rays to every light."""
        n, L, nc = self.n, self.L, (self.L + 1) ** 2
        if self.nl == 0:
            return torch.zeros((n, nc, 3), dtype=torch.float64, device="cuda")
        p, cols = self.x["p"], []
        for lt in range(self.nl):
            l = self.lpos[lt].expand(n, 3) if self.far else self.lpos[lt] - p
            r = l.norm(dim=-1)
            w, fall = l / r[:, None], torch.ones_like(r) if self.far else 1 / (r * r)
            cs = (self.N * w).sum(-1)
            lit = (cs.detach() > 0).nonzero()[:, 0]
            k, j = self.find(p.detach()[lit], w.detach()[lit], lit, None if self.far else r.detach()[lit])
            _, q2 = self.cross(p[lit][k], w[lit][k], j)
            om = 1 - self.alpha(self.x["o"][j], q2)
            T = torch.ones_like(cs).index_reduce(0, lit[k], om, "prod")
            Y = _sh(L, self.reflect(self.N, w))
            f = torch.where(cs > 0, self.alpha0() * cs * fall * T, torch.zeros_like(cs))
            cols.append((f[:, None] * Y)[:, :, None] * self.c * self.lint[lt])
        return torch.cat(cols, 2)

    def rays(self):
        """Origins and directions of the stratified hemisphere rays, [n * nd, 3]."""
        n, nd = self.n, self.sc["nd"]
        na = 1
        while (2 * na) ** 2 <= nd:
            na *= 2
        nbs = nd // na
        with np.errstate(over="ignore"):
            i, q = (v.reshape(-1) for v in np.meshgrid(np.arange(n), np.arange(nd), indexing="ij"))
            key = ((np.uint64(self.sc["seed"]) << np.uint64(32)) + i.astype(np.uint64) << np.uint64(12)) + q.astype(np.uint64)
            jit = [(_mix64(key * np.uint64(2) + np.uint64(dim)) >> np.uint64(40)).astype(np.float64) * 2.0 ** -24
                   for dim in (0, 1)]
        u1, u2 = (q // nbs + jit[0]) / na, (q % nbs + jit[1]) / nbs
        put = lambda v: torch.as_tensor(v, device="cuda")[:, None]
        rr, cz, ph = put(np.sqrt(u1)), put(np.sqrt(np.maximum(0.0, 1 - u1))), put(2 * math.pi * u2)
        i = torch.as_tensor(i, device="cuda")
        d = rr * torch.cos(ph) * self.U[i] + rr * torch.sin(ph) * self.V[i] + cz * self.N[i]
        return i, self.x["p"][i], d

    def hemisphere(self, nb):
        """B after nb bounces of the hemisphere-ray transport, [n, nc, C]."""
        own, o, d = self.rays()
        ray, j, a = self.composite(o, d, own)
        Yo, Yi = _sh(self.L, -d), _sh(self.L, self.reflect(self.N[own], d)) * (math.pi / self.sc["nd"])
        return self.bounces(nb, own, ray, j, a, Yo, Yi)

    def bounces(self, nb, own, ray, j, a, Yo, Yi):
        """Bounces over weighted (ray, source) records, ray r belonging to receiver own[r]."""
        S = self.x["E"][:, :, self.ch] + self.direct()
        f = self.alpha0()[:, None, None] * self.c[:, :, self.ch]
        nc, R = S.shape[1], own.shape[0]
        step = max(1, (1 << 28) // (nc * self.C))
        cuts = torch.searchsorted(ray, torch.arange(0, R + 1, max(1, R * step // max(ray.numel(), 1)), device="cuda")).tolist()
        cuts = sorted(set(cuts + [ray.numel()]))

        def part(B, a, Yo, Yi, h0, h1):
            rr, r0 = ray[h0:h1], int(ray[h0])
            x = (torch.einsum("hk,hkc->hc", Yo[rr], B[j[h0:h1]])) * a[h0:h1, None]
            X = torch.zeros((int(ray[h1 - 1]) - r0 + 1, self.C), dtype=torch.float64, device="cuda").index_add(0, rr - r0, x)
            i0 = int(own[r0])
            rows = own[r0:r0 + X.shape[0]]
            q = Yi[r0:r0 + X.shape[0], :, None] * X[:, None]
            return i0, torch.zeros((int(rows[-1]) - i0 + 1, nc, self.C), dtype=torch.float64, device="cuda").index_add(0, rows - i0, q)

        B, grad = S, any(v.requires_grad for v in self.x.values())
        for _ in range(nb):
            Q = torch.zeros_like(S)
            for h0, h1 in zip(cuts[:-1], cuts[1:]):
                i0, q = checkpoint(part, B, a, Yo, Yi, h0, h1, use_reentrant=False) if grad else part(B, a, Yo, Yi, h0, h1)
                Q = Q.index_add(0, torch.arange(i0, i0 + q.shape[0], device="cuda"), q)
            B = S + f * Q
        return B

    def segments(self):
        """Center-to-center pairs: (receiver, source, direction, V)."""
        p = self.x["p"]
        with torch.no_grad():
            front = (self.N @ p.T - (self.N * p).sum(-1, keepdim=True)) > self.eps
            front.fill_diagonal_(False)
            i, j = front.nonzero(as_tuple=True)
        dv = p[j] - p[i]
        r = dv.norm(dim=-1)
        d = dv / r[:, None]
        k, m = self.find(p.detach()[i], d.detach(), i, r.detach(), j)
        _, q2 = self.cross(p[i][k], d[k], m)
        T = torch.ones_like(r).index_reduce(0, k, 1 - self.alpha(self.x["o"][m], q2), "prod")
        s2, o = self.x["s"].prod(-1), self.x["o"]
        if self.model == "gauss":
            A = 2 * math.pi * s2 * o * (1 - math.exp(-4.5))
        else:
            A = 2 * math.pi / 3.4 * s2 * _ein(0.03279 * o ** 3.4)
        geo = (self.N[i] * d).sum(-1).abs() * (self.N[j] * d).sum(-1).abs() / r ** 2
        return i, j, d, self.x["lam"][j] * A[j] * T * geo

    def center(self, nb):
        i, j, d, V = self.segments()
        Yo, Yi = _sh(self.L, -d), _sh(self.L, self.reflect(self.N[i], d))
        return self.bounces(nb, i, torch.arange(i.shape[0], device="cuda"), j, V, Yo, Yi)

    @torch.no_grad()
    def shooting(self, shots):
        i, j, d, V = self.segments()
        W = torch.zeros((self.n, self.n), dtype=torch.float64, device="cuda")
        W[i, j] = V
        p, f = self.x["p"], self.alpha0()[:, None, None] * self.c[:, :, self.ch]
        lum = torch.tensor([0.2126, 0.7152, 0.0722], dtype=torch.float64, device="cuda")[self.ch]
        Bh = self.x["E"][:, :, self.ch] + self.direct()
        dB = Bh.clone()
        for _ in range(shots):
            b = int((dB.abs() * lum).sum((1, 2)).argmax())
            shot = dB[b].clone()
            dB[b] = 0
            to = (W[:, b] > 0).nonzero()[:, 0]
            d = _unit(p[b] - p[to])
            x = torch.einsum("ak,kc->ac", _sh(self.L, -d), shot) * W[to, b, None]
            add = f[to] * _sh(self.L, self.reflect(self.N[to], d))[:, :, None] * x[:, None]
            dB[to] += add
            Bh[to] += add
        return Bh, dB

    @torch.no_grad()
    def pixels(self, cam, W, H):
        """Hit records of the image's rays, a band of rows at a time: (first pixel, ray, surfel, weight, Y(-d))."""
        cam = torch.tensor(cam, dtype=torch.float64, device="cuda")
        f = _unit(cam[3:6])
        r = _unit(torch.linalg.cross(f, cam[6:9]))
        u = torch.linalg.cross(r, f)
        th = math.tan(0.5 * float(np.float32(FOV)))
        for y0 in range(0, H, 64):
            y, x = torch.meshgrid(torch.arange(y0, min(y0 + 64, H), device="cuda"), torch.arange(W, device="cuda"), indexing="ij")
            sx, sy = (2 * (x + 0.5) / W - 1) * th * W / H, (1 - 2 * (y + 0.5) / H) * th
            d = _unit(f + sx.reshape(-1, 1).double() * r + sy.reshape(-1, 1).double() * u)
            ray, j, a = self.composite(cam[:3].expand_as(d), d, torch.full((d.shape[0],), -1, device="cuda"))
            yield y0 * W, d.shape[0], ray, j, a, _sh(self.L, -d)


def _ein(x):
    """Ein(x) = int_0^x (1 - e^-y)/y dy by Gauss-Legendre quadrature on 64 nodes."""
    t, w = (torch.as_tensor(v, device=x.device) for v in np.polynomial.legendre.leggauss(64))
    y = 0.5 * x[..., None] * (t + 1)
    return (0.5 * x[..., None] * w * -torch.expm1(-y) / y).sum(-1)


def _affordable(case, scs):
    for sc in scs:
        n, C, nc = sc["n"], 3 * max(len(sc["light_pos"]), 1), (sc["L"] + 1) ** 2
        kind = case["kind"]
        if kind in ("render", "render_adjoint"):
            tests, hits = case["width"] * case["height"] * n, 0
        elif kind in ("pairs", "shooting"):
            tests, hits = 0.5 * n ** 3, 0.5 * n * n
        else:
            tests, hits = float(n) * n * (sc["nd"] + C / 3), n * sc["nd"] * HITS_PER_RAY
        if tests > MAX_TESTS or hits * C * nc * max(sc["nb"], 1) > MAX_VALUES:
            return False
    return True


def exact(case, seed):
    kind, model = case["kind"], case.get("model", "gauss")
    if kind == "batch":  # minutes of hit lists
        return None
    sc = _scenes(case, seed)[0]
    if not _affordable(case, [sc]):
        return None
    C = 3 * max(len(sc["light_pos"]), 1)
    names = {"step": ("E", "ad", "o"), "autograd": ("E", "ad", "o"), "pairs": ("E", "ad", "o", "lam"),
             "geometry": ("E", "ad", "o", "p", "s", "tu", "tv")}.get(kind, ())
    if kind == "shooting":
        return list(_Exact(sc, model).shooting(case["shots"]))
    if kind == "render":
        ex, B = _Exact(sc, model), _solved_B(sc, C, seed, "cuda").double()
        img = torch.zeros((case["height"] * case["width"], C), dtype=torch.float64, device="cuda")
        for p0, m, ray, j, a, Y in ex.pixels(_camera(seed), case["width"], case["height"]):
            img[p0:p0 + m].index_add_(0, ray, torch.einsum("hk,hkc->hc", Y[ray], B[j]) * a[:, None])
        return img.reshape(case["height"], case["width"], C)
    if kind == "render_adjoint":
        ex, g = _Exact(sc, model), _normal((case["height"], case["width"], C), seed + 4, "cuda").double().reshape(-1, C)
        dB = torch.zeros((sc["n"], (sc["L"] + 1) ** 2, C), dtype=torch.float64, device="cuda")
        for p0, m, ray, j, a, Y in ex.pixels(_camera(seed), case["width"], case["height"]):
            dB.index_add_(0, j, Y[ray][:, :, None] * (a[:, None] * g[p0:p0 + m][ray])[:, None])
        return dB
    ex = _Exact(sc, model, names)
    B = ex.center(case["nb"]) if kind == "pairs" else ex.hemisphere(case["nb"])
    if not names:
        return B.detach()
    W = _normal(tuple(B.shape), seed + 3, "cuda").double()
    grads = torch.autograd.grad(B, [ex.x[k] for k in names], W)
    return [B.detach(), *grads]
