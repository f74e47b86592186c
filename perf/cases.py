"""The work that users of this library have it do, as cases that can be timed.

A case is a dict of plain values. `prepare` makes what a program holds before
the call (context, loaded objects, rays, result buffers), `run` makes one pass
through the public entry points, `exact` computes the same outputs in 64-bit
floats with torch alone, and `work` counts the bytes and operations a pass
cannot do without.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2504_21627_gb300 import inputs as I
from paper_2504_21627_gb300 import lsnif

DEV = "cuda"
PRECISION = {"fp32": lsnif.FP32_PLAIN, "bf16": lsnif.BF16_FUSED, "fp16": lsnif.FP16_FUSED}


# --------------------------------------------------------------------------
# objects: the repository's own configurations
# --------------------------------------------------------------------------

def _config(name: str) -> I.Config:
    if name == "icosphere":      # 8 levels, 3 x 64: the smallest configuration in use
        return I.cfg_icosphere_small()
    if name == "torus":          # 16 levels of 2^19 entries, 4 x 64: the benchmark's
        return I.cfg_torus_4m()
    if name == "paper":          # 2 levels of 2^17 entries, 2 x 128: the parameter study's base
        return I.Config(V=32, H=18, L=2, F=4, log2_T=17, N_min=64, N_max=128, n_hidden=2, width=128, n_mat=4)
    if name.startswith("stress"):  # 16 levels x 4 features, 4 x 128: the instanced scene's
        return I.cfg_stress_object(log2_T=18)
    i = int(name[len("mixed"):])  # the many-object batch: V 64 or 128, tables of 2^16..2^18 entries
    V = (64, 128)[i % 2]
    return I.Config(V=V, H=18, L=16, F=2, log2_T=16 + i % 3, N_min=16, N_max=8 * V, n_hidden=4, width=64, n_mat=4)


@functools.lru_cache(maxsize=None)
def _mesh(name: str) -> I.Mesh:
    if name == "icosphere":
        return I.icosphere(3)
    if name == "torus":
        return I.noise_torus(seed=2)
    if name == "paper":
        return I.noise_torus_tris(11, 50000, amplitude=0.08, n_mat=4)
    i = int(name[-1])
    tris = 50000 if name.startswith("stress") else (5000, 20000, 50000)[i % 3]
    return I.noise_icosphere(200 + i, tris, n_mat=4) if i % 2 == 0 else I.noise_torus_tris(200 + i, tris, n_mat=4)


@functools.lru_cache(maxsize=None)
def _params(name: str) -> I.Params:
    p = I.random_params(_config(name), seed=5 + len(name) + ord(name[-1]), table_range=0.05, bias_range=0.1)
    if name.startswith("stress"):
        p.weights[-1][1][0] = 1.0  # occlusion biased towards hits, so that most bounces continue
    return p


def _load(ctx: lsnif.Context, name: str) -> int:
    p = _params(name)
    return ctx.load_object(_mesh(name), _config(name), tables=p.tables, mlp=p.packed_mlp())


def _box(name: str) -> tuple[np.ndarray, np.ndarray]:
    v = _mesh(name).verts.astype(np.float64)
    return v.min(0), v.max(0)


# --------------------------------------------------------------------------
# rays, from a seed, on the GPU: (8, n) float32 rows ox oy oz dx dy dz tmin tmax
# --------------------------------------------------------------------------

def _gen(seed: int) -> torch.Generator:
    return torch.Generator(DEV).manual_seed(int(seed))


def _t(a) -> torch.Tensor:
    return torch.as_tensor(np.asarray(a, np.float64), device=DEV)


def _unit(v: torch.Tensor) -> torch.Tensor:
    return v / v.norm(dim=-1, keepdim=True)


def _pack(o: torch.Tensor, d: torch.Tensor) -> torch.Tensor:
    r = torch.zeros((8, o.shape[0]), dtype=torch.float32, device=DEV)
    r[0:3] = o.T
    r[3:6] = d.T
    r[7] = math.inf
    return r


def _camera_rays(seed: int, width: int, height: int, radius: float, spp: int = 1) -> torch.Tensor:
    """Pixel-order rays of a pinhole camera near the benchmark's view; jittered within the pixel for spp > 1."""
    g = I.rng(seed)
    eye = I.seeded_camera(2, radius=1.0).eye + 0.15 * g.normal(size=3)
    eye *= radius / np.linalg.norm(eye)
    fwd = -eye / np.linalg.norm(eye)
    right = np.cross(fwd, [0.0, 0.0, 1.0])
    right /= np.linalg.norm(right)
    up = np.cross(right, fwd)
    n = width * height * spp
    p = torch.arange(n, device=DEV) // spp
    j = torch.rand((2, n), generator=_gen(seed), device=DEV, dtype=torch.float64) if spp > 1 else torch.full(
        (2, n), 0.5, device=DEV, dtype=torch.float64)
    th = math.tan(math.radians(45.0) / 2)
    x = ((p % width + j[0]) / width * 2 - 1) * th * width / height
    y = (1 - (p // width + j[1]) / height * 2) * th
    d = _unit(_t(fwd) + x[:, None] * _t(right) + y[:, None] * _t(up))
    return _pack(_t(eye).expand(n, 3), d)


def _sphere_rays(seed: int, n: int, name: str) -> torch.Tensor:
    """Origins on a sphere about the object, each aimed at a point of its box, in no order."""
    g = _gen(seed)
    lo, hi = map(_t, _box(name))
    o = 3.0 * _unit(torch.randn((n, 3), generator=g, device=DEV, dtype=torch.float64))
    to = lo + (hi - lo) * torch.rand((n, 3), generator=g, device=DEV, dtype=torch.float64)
    return _pack(o, _unit(to - o))


def _cosine(nrm: torch.Tensor, g: torch.Generator) -> torch.Tensor:
    """Cosine-weighted unit directions about unit normals."""
    return _unit(nrm + 0.999 * _unit(torch.randn(nrm.shape, generator=g, device=DEV, dtype=torch.float64)))


def _surface_rays(seed: int, n: int, name: str) -> torch.Tensor:
    """Secondary rays: from points of the surface into the cosine lobe of the normal, in no order."""
    g = _gen(seed)
    m = _mesh(name)
    v = _t(m.verts)[torch.as_tensor(m.tris, device=DEV).long()]
    c = torch.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0], dim=1)
    cum = c.norm(dim=1).cumsum(0)
    tri = torch.searchsorted(cum, torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * cum[-1]).clamp_(max=len(cum) - 1)
    u = torch.rand((n, 2), generator=g, device=DEV, dtype=torch.float64)
    s = u[:, :1].sqrt()
    p = (1 - s) * v[tri, 0] + s * (1 - u[:, 1:]) * v[tri, 1] + s * u[:, 1:] * v[tri, 2]
    nrm = _unit(c[tri])
    lo, hi = _box(name)
    return _pack(p + 1e-4 * float(np.linalg.norm(hi - lo)) * nrm, _cosine(nrm, g))


def _outside_rays(seed: int, n: int, name: str) -> torch.Tensor:
    """Training rays from outside: on the sphere about the box, into the cosine lobe of its centre."""
    g = _gen(seed)
    lo, hi = map(_t, _box(name))
    out = _unit(torch.randn((n, 3), generator=g, device=DEV, dtype=torch.float64))
    return _pack(0.5 * (lo + hi) + 1.05 * 0.5 * (hi - lo).norm() * out, _cosine(-out, g))


def _case_rays(case: dict, seed: int) -> torch.Tensor:
    if case["rays"] == "camera":
        return _camera_rays(seed, case["width"], case["height"], 4.0)
    if case["rays"] == "sphere":
        return _sphere_rays(seed, case["n"], case["object"])
    return _surface_rays(seed, case["n"], case["object"])


def _mixed_batch(case: dict, seed: int) -> tuple[torch.Tensor, torch.Tensor]:
    """Rays of several objects shuffled together: (rays, object number of each), uneven shares."""
    k, n = case["objects"], case["n"]
    share = np.array([1.0 / (1 + i) for i in range(k)])
    ends = np.round(np.cumsum(share / share.sum()) * n).astype(int)
    cnt = np.diff(np.concatenate([[0], ends]))
    rays = torch.cat([_sphere_rays(seed * 64 + i, int(c), f"mixed{i}") for i, c in enumerate(cnt)], 1)
    who = torch.repeat_interleave(torch.arange(k, device=DEV), torch.as_tensor(cnt, device=DEV))
    perm = torch.randperm(n, generator=_gen(seed), device=DEV)
    return rays[:, perm].contiguous(), who[perm]


def _training_batch(case: dict, seed: int) -> tuple[torch.Tensor, dict]:
    """Rays that reach the network, half of them from outside and half from the surface, and labels as a ray
    caster gives them (the step reads them as plain numbers, so theirs are drawn)."""
    n, name = case["n"], case["object"]
    part = []
    for make, want, s in ((_outside_rays, n // 2, 1), (_surface_rays, n - n // 2, 2)):
        got = []
        while sum(r.shape[1] for r in got) < want:
            r = make(seed * 64 + s, want, name)
            got.append(r[:, _Solid(name).walk(r)[0] > 0])
            s += 2
        part.append(torch.cat(got, 1)[:, :want])
    g = _gen(seed)
    rays = torch.cat(part, 1)[:, torch.randperm(n, generator=g, device=DEV)].contiguous()
    m = _mesh(name)
    occ = (torch.rand(n, generator=g, device=DEV) < 0.7).float()
    mat = torch.randint(0, m.n_mat, (n,), generator=g, device=DEV, dtype=torch.int32)
    nrm = _unit(torch.randn((n, 3), generator=g, device=DEV))
    return rays, {"occ": occ, "t_local": torch.rand(n, generator=g, device=DEV) * occ,
                  "normal": (nrm * occ[:, None]).contiguous(), "mat": mat * occ.int(),
                  "albedo": (torch.as_tensor(m.albedo, device=DEV)[mat.long()] * occ[:, None]).contiguous()}


def _instances(case: dict) -> list:
    return I.seeded_instances(case["instances"], case["objects"], seed=9, spread=6.0)


def _scene_rays(case: dict, seed: int) -> tuple[torch.Tensor, torch.Tensor]:
    rays = _camera_rays(seed, case["width"], case["height"], 9.0, spp=case["spp"])
    return rays, torch.rand((rays.shape[1], 2), generator=_gen(seed + 1), device=DEV)


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

def listed() -> list[dict]:
    return [
        # one small interactive request on the smallest network: launches and latency
        {"name": "icosphere_4k_bf16", "kind": "query", "object": "icosphere", "rays": "sphere", "n": 4096,
         "precision": "bf16"},
        # the same object through the reference arithmetic, an odd number of rays
        {"name": "icosphere_4k_fp32", "kind": "query", "object": "icosphere", "rays": "sphere", "n": 4099,
         "precision": "fp32"},
        # a served request of the usual size for picking and shadow probes on the large object
        {"name": "torus_20k_fp16", "kind": "query", "object": "torus", "rays": "surface", "n": 20001,
         "precision": "fp16"},
        # the headline workload: every pixel's primary ray of a 2048 x 2048 frame, shape chosen by the autotuner
        {"name": "torus_frame_bf16", "kind": "query", "object": "torus", "rays": "camera", "width": 2048,
         "height": 2048, "precision": "bf16", "tuned": True},
        # a frame whose sides are multiples of nothing, with the context as it is created
        {"name": "torus_frame_fp16", "kind": "query", "object": "torus", "rays": "camera", "width": 1365,
         "height": 767, "precision": "fp16"},
        # the reference arithmetic over a whole frame, as a renderer checks its fast path
        {"name": "torus_frame_fp32", "kind": "query", "object": "torus", "rays": "camera", "width": 1000,
         "height": 1000, "precision": "fp32"},
        # secondary rays of a path tracer: in no order, almost all of them alive
        {"name": "torus_bounce_bf16", "kind": "query", "object": "torus", "rays": "surface", "n": 1 << 20,
         "precision": "bf16", "sorted": True},
        # the end-to-end call: page-locked host rays in, host results out
        {"name": "torus_host_bf16", "kind": "query", "object": "torus", "rays": "camera", "width": 1500,
         "height": 1400, "precision": "bf16", "host": True},
        # a batch that mixes objects of several sizes, one handle a ray
        {"name": "mixed_bf16", "kind": "mixed", "objects": 6, "n": 400003, "precision": "bf16"},
        # one bounce of an instanced scene with the large network, and the rays of the next
        {"name": "scene_fp16", "kind": "scene", "objects": 2, "instances": 8, "width": 480, "height": 270, "spp": 4,
         "precision": "fp16"},
        # one step of training at the batch that the paper and the benchmark train with
        {"name": "train_torus_256k", "kind": "train", "object": "torus", "n": 1 << 18},
        # one step of the parameter study's training
        {"name": "train_paper_16k", "kind": "train", "object": "paper", "n": 1 << 14},
    ]


def draw(rng) -> dict:
    def size(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))

    kind = rng.choice(["query", "query", "query", "train", "mixed", "scene"])
    if kind == "train":
        name = rng.choice(["torus", "paper", "icosphere"])
        return {"kind": kind, "object": name, "n": size(1 << 12, 1 << 18)}
    if kind == "mixed":
        return {"kind": kind, "objects": rng.randint(2, 6), "n": size(1 << 14, 1 << 19), "precision": rng.choice(["bf16", "fp16"])}
    if kind == "scene":
        w = size(64, 480)
        return {"kind": kind, "objects": 2, "instances": rng.randint(2, 8), "width": w, "height": max(36, w * 9 // 16),
                "spp": rng.choice([1, 4]), "precision": "fp16"}
    precision = rng.choice(["bf16", "fp16", "fp32"])
    n = size(256, 1 << 20 if precision == "fp32" else 1 << 22)
    case = {"kind": kind, "object": rng.choice(["icosphere", "torus", "torus"]), "precision": precision,
            "rays": rng.choice(["camera", "sphere", "surface"])}
    if case["rays"] == "camera":
        w = max(16, int(math.sqrt(n * rng.uniform(1.0, 2.0))))
        case |= {"width": w, "height": max(16, n // w)}
    else:
        case["n"] = n
        case["sorted"] = n > 1 << 18
    return case


class State:
    pass


def _results(n: int, host: bool = False, n_out: int = 0) -> lsnif.QueryResult:
    kw = {"pin_memory": True} if host else {"device": DEV}
    f = {"dtype": torch.float32, **kw}
    return lsnif.QueryResult(torch.zeros(n, dtype=torch.uint8, **kw), torch.zeros(n, **f), torch.zeros((3, n), **f),
                             torch.zeros(n, dtype=torch.int32, **kw), torch.zeros((3, n), **f),
                             torch.zeros((n, n_out), **f) if n_out else None)


def prepare(case: dict, seed: int) -> State:
    s = State()
    s.case = case
    s.ctx = ctx = lsnif.Context(0)
    kind = case["kind"]
    if kind == "train":
        s.rays, s.labels = _training_batch(case, seed)
        s.obj = _load(ctx, case["object"])
        # page-locked copies of the gradients and the updated network
        cfg = _config(case["object"])
        n_mlp = int(ctx.object_info(s.obj).n_params_mlp)
        s.grad_tables = torch.zeros((cfg.L, cfg.T, cfg.F), pin_memory=True)
        s.grad_mlp = torch.zeros(n_mlp, pin_memory=True)
        s.mlp = torch.zeros(n_mlp, pin_memory=True)
        return s
    if kind == "scene":
        handles = [_load(ctx, f"stress{i}") for i in range(case["objects"])]
        s.instances = [(handles[o], A, b) for o, A, b in _instances(case)]
        s.rays, s.u = _scene_rays(case, seed)
        ctx.set_trace_mode(2)   # pairs mix objects and bounces have no order
        ctx.set_group_mode(2)
        return s
    if kind == "mixed":
        handles = torch.tensor([_load(ctx, f"mixed{i}") for i in range(case["objects"])], device=DEV, dtype=torch.int32)
        s.rays, who = _mixed_batch(case, seed)
        s.handles = handles[who].contiguous()
        s.out = _results(s.rays.shape[1])
        ctx.set_trace_mode(2)
        ctx.set_group_mode(2)
        return s
    s.obj = _load(ctx, case["object"])
    s.rays = _case_rays(case, seed)
    if case.get("tuned"):
        ctx.autotune(s.rays, obj=s.obj, reps=3)
    if case.get("sorted"):
        ctx.set_group_mode(2)
    n = s.rays.shape[1]
    if case.get("host"):
        s.rays = s.rays.cpu().pin_memory()
    # small calls read the raw outputs too
    s.out = _results(n, bool(case.get("host")), _config(case["object"]).n_out if _logits(case) else 0)
    return s


def _logits(case: dict) -> bool:
    return case["kind"] == "query" and case.get("n", 1 << 30) < 1 << 16


def _fields(r: lsnif.QueryResult) -> dict:
    out = {"hit": r.hit, "t": r.t, "normal": r.normal, "mat": r.mat, "albedo": r.albedo}
    return out if r.logits is None else out | {"logits": r.logits}


def _read(ctx: lsnif.Context, obj: int, which: int, to: torch.Tensor) -> torch.Tensor:
    rc = ctx.lib.lsnif_read_params(ctx.h, obj, which, to.data_ptr(), to.numel() * 4)
    if rc < 0:
        raise lsnif.LsnifError(rc, lsnif.last_error())
    return to


def run(s: State):
    ctx, case = s.ctx, s.case
    if case["kind"] == "train":
        # the learning rate keeps repeated passes on one state alike; every kernel of the step runs
        st = ctx.train_step(s.rays, s.labels, s.obj, lr=1e-6)
        return {"loss": [st.total, st.occ, st.t, st.normal, st.albedo, st.mat],
                "grad_tables": _read(ctx, s.obj, lsnif.PARAM_GRAD_TABLES, s.grad_tables),
                "grad_mlp": _read(ctx, s.obj, lsnif.PARAM_GRAD_MLP, s.grad_mlp),
                "mlp": _read(ctx, s.obj, lsnif.PARAM_MLP, s.mlp)}
    precision = PRECISION[case["precision"]]
    if case["kind"] == "scene":
        res, inst = ctx.query_scene(s.rays, s.instances, precision=precision)
        return _fields(res) | {"instance": inst, "bounce": ctx.bounce_rays(s.rays, res, s.u, 1e-3)}
    if case["kind"] == "mixed":
        return _fields(ctx.query_rays(s.rays, obj_per_ray=s.handles, precision=precision, out=s.out))
    if case.get("host"):
        return _fields(ctx.query_rays_host(s.rays, obj=s.obj, precision=precision, out=s.out))
    return _fields(ctx.query_rays(s.rays, obj=s.obj, precision=precision, out=s.out))


# share of the rays that reach the network, and boundary points of such a ray
_LIVE = {"camera": (0.35, 16.0), "sphere": (0.8, 15.0), "surface": (1.0, 6.3)}


def _network(cfg: I.Config) -> int:
    return sum(a * b for a, b in cfg.layer_dims())


def work(case: dict) -> dict:
    if case["kind"] == "train":
        cfg, n = _config(case["object"]), case["n"]
        points = 11.0 * n
        tables = min(cfg.L * cfg.T, points * cfg.L * 8) * cfg.F * 4
        state = cfg.L * cfg.T * cfg.F * 4
        # rays and labels; corners read and their gradients written; Adam on every parameter (gradient, two
        # moments and value read, the last three written); the half-precision copies; gradients to the host
        return {"bytes": n * (32 + 36) + 2 * tables + 7 * state + state // 2 + state,
                "flops": n * (6.0 * _network(cfg)) + 4 * points * cfg.L * 8 * cfg.F}
    if case["kind"] == "scene":
        n = case["width"] * case["height"] * case["spp"]
        cfg, (live, points), k = _config("stress0"), (0.5, 13.0), case["objects"]
    elif case["kind"] == "mixed":
        n, cfg, (live, points), k = case["n"], _config("mixed1"), _LIVE["sphere"], case["objects"]
    else:
        n = case["n"] if "n" in case else case["width"] * case["height"]
        cfg, (live, points), k = _config(case["object"]), _LIVE[case["rays"]], 1
    size = 4 if case["precision"] == "fp32" else 2
    corners = live * n * points * cfg.L * 8
    out = 33 + (4 * cfg.n_out if _logits(case) else 0) + (36 if case["kind"] == "scene" else 0)
    return {"bytes": n * (32 + out) + min(k * cfg.L * cfg.T, corners) * cfg.F * size + k * _network(cfg) * size,
            "flops": live * n * 2.0 * _network(cfg) + corners * 2 * cfg.F}


# --------------------------------------------------------------------------
# the same outputs in 64 bits, torch alone
# --------------------------------------------------------------------------

class _Solid:
    """One object in 64 bits: its box, its occupied voxels, its lattices and its network."""

    def __new__(cls, name: str):
        return _solid(name)

    def build(self, name: str) -> "_Solid":
        self.cfg = cfg = _config(name)
        lo, hi = _box(name)
        thin = np.linalg.norm(hi - lo) / 8
        mid, half = 0.5 * (lo + hi), np.maximum(hi - lo, thin) / 2
        lo, hi = np.where(hi - lo < thin, mid - half, lo), np.where(hi - lo < thin, mid + half, hi)
        f = np.float32
        l32, h32 = lo.astype(f), hi.astype(f)   # the box in 32 bits, rounded outward
        l32 = np.where(l32 > lo, np.nextafter(l32, f(-np.inf)), l32)
        h32 = np.where(h32 < hi, np.nextafter(h32, f(np.inf)), h32)
        self.lo, self.ext = _t(l32), _t(h32) - _t(l32)
        self.occ = self.voxels(_mesh(name))
        growth = (cfg.N_max / cfg.N_min) ** (1 / max(cfg.L - 1, 1))
        self.res = [int(math.floor(cfg.N_min * growth ** i + 0.5)) for i in range(cfg.L)]
        p = _params(name)
        self.tables = torch.as_tensor(p.tables, device=DEV)
        self.net = [(_t(W), _t(b)) for W, b in p.weights]
        return self

    def voxels(self, m: I.Mesh) -> torch.Tensor:
        """Voxels that a triangle touches (separating axes: box, triangle plane, edges), flat x + V (y + V z)."""
        V = self.cfg.V
        g = ((_t(m.verts) - self.lo) * V / self.ext)[torch.as_tensor(m.tris, device=DEV).long()]
        lo = (g.min(1).values.ceil() - 1).clamp_(min=0)
        span = (g.max(1).values.floor().clamp_(max=V - 1) - lo).max(0).values.long().tolist()
        e = torch.stack([g[:, 1] - g[:, 0], g[:, 2] - g[:, 1], g[:, 0] - g[:, 2]], 1)
        nrm = torch.cross(e[:, 0], e[:, 1], dim=1)
        occ = torch.zeros(V ** 3, dtype=torch.bool, device=DEV)
        for dz in range(span[2] + 1):
            for dy in range(span[1] + 1):
                for dx in range(span[0] + 1):
                    c = lo + torch.tensor([dx, dy, dz], device=DEV, dtype=torch.float64)
                    a = g - c[:, None] - 0.5
                    ok = (c <= V - 1).all(1) & ((a.min(1).values <= 0.5) & (a.max(1).values >= -0.5)).all(1)
                    ok &= (nrm * a[:, 0]).sum(1).abs() <= 0.5 * nrm.abs().sum(1)
                    for i in range(3):
                        for j in range(3):
                            unit = torch.zeros_like(e[:, i])
                            unit[:, j] = 1
                            ax = torch.cross(unit, e[:, i], dim=1)
                            p, r = (a * ax[:, None]).sum(2), 0.5 * ax.abs().sum(1)
                            ok &= (p.min(1).values <= r) & (p.max(1).values >= -r)
                    q = c[ok].long()
                    occ[q[:, 0] + V * (q[:, 1] + V * q[:, 2])] = True
        return occ

    def walk(self, rays: torch.Tensor):
        """(k, t01, points): occupied voxels met (at most H / 2), clipped interval, their entry and exit points."""
        cfg, n = self.cfg, rays.shape[1]
        V, H = cfg.V, cfg.H
        r = rays.double()
        o, d = (r[0:3].T - self.lo) / self.ext, r[3:6].T / self.ext
        zero = d == 0
        ta, tb = (0 - o) / d, (1 - o) / d
        inside = ((o >= 0) & (o <= 1)) | ~zero
        near = torch.where(zero, -math.inf, torch.minimum(ta, tb))
        far = torch.where(zero, math.inf, torch.maximum(ta, tb)).min(1).values
        tn, axis = near.max(1)
        t0 = torch.maximum(tn, r[6])
        axis = torch.where(tn >= r[6], axis, -1)
        k_all = torch.zeros(n, dtype=torch.long, device=DEV)
        pts = torch.zeros((n, H, 3), dtype=torch.float64, device=DEV)
        live = ((far > t0) & inside.all(1) & ~zero.all(1)).nonzero()[:, 0]
        t01 = torch.stack([t0, far], 1)
        o, d, tc, t1, ain = o[live], d[live], t0[live], far[live], axis[live]
        step = torch.sign(d).long()
        ix = ((o + tc[:, None] * d) * V).floor().long().clamp_(0, V - 1)
        first = torch.where(step > 0, 0, V - 1)
        entered = ain[:, None] == torch.arange(3, device=DEV)
        ix = torch.where(entered, first, ix)
        fin = torch.where(step.gather(1, ain.clamp(min=0)[:, None])[:, 0] > 0, 0.0, 1.0).double()
        k = torch.zeros(live.shape[0], dtype=torch.long, device=DEV)
        for it in range(3 * V + 3):
            if it % 16 == 0:   # rays that have ended leave
                go = (k >= 0).nonzero()[:, 0]
                if not go.numel():
                    break
                if go.numel() < k.numel():
                    live, o, d, tc, t1, ain, fin, step, ix, k = (x[go] for x in (live, o, d, tc, t1, ain, fin, step, ix, k))
            face = (ix + (step > 0)).double() / V
            te = torch.where(step != 0, (face - o) / d, math.inf)
            a = torch.where(te[:, 0] <= te[:, 1], torch.where(te[:, 0] <= te[:, 2], 0, 2), torch.where(te[:, 1] <= te[:, 2], 1, 2))
            a1 = a[:, None]
            tx, f = te.gather(1, a1)[:, 0], face.gather(1, a1)[:, 0]
            end = torch.minimum(tx, t1)
            run_ = k >= 0
            ixc = ix.clamp(0, V - 1)
            seen = run_ & (end > tc) & self.occ[ixc[:, 0] + V * (ixc[:, 1] + V * ixc[:, 2])]
            w = seen.nonzero()[:, 0]
            if w.numel():
                for slot, tt, ax, fc in ((0, tc, ain, fin), (1, end, a, f)):
                    p = o[w] + tt[w][:, None] * d[w]
                    p = torch.where(ax[w][:, None] == torch.arange(3, device=DEV), fc[w][:, None], p)
                    pts[live[w], 2 * k[w] + slot] = p
                k[w] += 1
                k_all[live[w]] = k[w]
            moved = ix.scatter_add(1, a1, step.gather(1, a1))
            m = moved.gather(1, a1)[:, 0]
            stop = run_ & ((k >= H // 2) | (tx >= t1) | (m < 0) | (m >= V))
            ix = moved.clamp(-1, V)
            tc, ain, fin = torch.where(run_, tx, tc), a, f
            k = torch.where(stop, -1, k)
        return k_all, t01, pts

    def corners(self, p: torch.Tensor, level: int):
        """(table index, weight) of the 8 lattice corners of each point, one after another."""
        x = p * self.res[level]
        c = x.floor()
        w, c = x - c, c.long()
        for i in range(8):
            q = [c[:, a] + (i >> a & 1) for a in range(3)]
            h = q[0] ^ (q[1] * 2654435761 & 0xFFFFFFFF) ^ (q[2] * 805459861 & 0xFFFFFFFF)
            ww = [w[:, a] if i >> a & 1 else 1 - w[:, a] for a in range(3)]
            yield h & (self.cfg.T - 1), ww[0] * ww[1] * ww[2]

    def features(self, k: torch.Tensor, pts: torch.Tensor) -> torch.Tensor:
        cfg = self.cfg
        x = torch.zeros((pts.shape[0], cfg.H, cfg.L, cfg.F), dtype=torch.float64, device=DEV)
        on = torch.arange(cfg.H, device=DEV) < 2 * k[:, None]
        p = pts[on]
        for level in range(cfg.L):
            f = torch.zeros((p.shape[0], cfg.F), dtype=torch.float64, device=DEV)
            for idx, w in self.corners(p, level):
                f += w[:, None] * self.tables[level][idx].double()
            x[:, :, level][on] = f
        return x.flatten(1)

    def network(self, x: torch.Tensor, net=None) -> torch.Tensor:
        net = net or self.net
        for i, (W, b) in enumerate(net):
            x = x @ W.T + b
            if i + 1 < len(net):
                x = torch.where(x > 0, x, 0.01 * x) if self.cfg.activation else torch.relu(x)
        return x

    def query(self, rays: torch.Tensor) -> dict:
        n, step = rays.shape[1], 1 << 18
        out = {"hit": torch.zeros(n, dtype=torch.bool, device=DEV)}
        f = {"dtype": torch.float64, "device": DEV}
        out |= {"t": torch.full((n,), math.inf, **f), "normal": torch.zeros((3, n), **f),
                "albedo": torch.zeros((3, n), **f), "logits": torch.full((n, self.cfg.n_out), math.nan, **f)}
        for i in range(0, n, step):
            r = rays[:, i:i + step]
            k, t01, pts = self.walk(r)
            g = (k > 0).nonzero()[:, 0]
            z = self.network(self.features(k[g], pts[g]))
            t = t01[g, 0] + torch.sigmoid(z[:, 1]) * (t01[g, 1] - t01[g, 0])
            at = g + i
            out["hit"][at] = (z[:, 0] > 0) & (t >= r[6, g]) & (t <= r[7, g])
            out["t"][at] = t
            out["normal"][:, at] = _unit(z[:, 2:5]).T
            out["albedo"][:, at] = torch.sigmoid(z[:, 5:8]).T
            out["logits"][at] = z
        return out


@functools.lru_cache(maxsize=4)
def _solid(name: str) -> _Solid:
    return object.__new__(_Solid).build(name)


def _exact_train(case: dict, seed: int) -> dict:
    s = _Solid(case["object"])
    cfg = s.cfg
    rays, lab = _training_batch(case, seed)
    k, _, pts = s.walk(rays)
    live = (k > 0).double()
    x = s.features(k, pts).requires_grad_()
    net = [(W.clone().requires_grad_(), b.clone().requires_grad_()) for W, b in s.net]
    z = s.network(x, net)
    y = lab["occ"].double()
    F = torch.nn.functional
    sa = torch.sigmoid(z[:, 5:8])
    # the relative L2's denominator is a weight, not differentiated
    terms = [F.softplus(-z[:, 0].abs()) + z[:, 0].clamp(min=0) - z[:, 0] * y,
             y * (torch.sigmoid(z[:, 1]) - lab["t_local"].double()).abs(),
             y * (1 - (z[:, 2:5] * lab["normal"].double()).sum(1) / z[:, 2:5].norm(dim=1)),
             y * ((sa - lab["albedo"].double()) ** 2 / (sa.detach() ** 2 + 0.01)).mean(1),
             y * F.cross_entropy(z[:, 8:], lab["mat"].long(), reduction="none")]
    terms = [(t * live).sum() / live.sum() for t in terms]
    sum(terms).backward()
    grad = torch.zeros((cfg.L, cfg.T, cfg.F), dtype=torch.float64, device=DEV)
    on = torch.arange(cfg.H, device=DEV) < 2 * k[:, None]
    p, dx = pts[on], x.grad.view(-1, cfg.H, cfg.L, cfg.F)[on]
    for level in range(cfg.L):
        for idx, w in s.corners(p, level):
            grad[level].index_add_(0, idx, w[:, None] * dx[:, level])
    flat = torch.cat([torch.cat([W.grad.flatten(), b.grad]) for W, b in net])
    vals = [float(t.detach()) for t in terms]
    return {"loss": [sum(vals)] + vals, "grad_tables": grad, "grad_mlp": flat, "mlp": None}


def _exact_scene(case: dict, seed: int) -> dict:
    rays, u = _scene_rays(case, seed)
    n = rays.shape[1]
    f = {"dtype": torch.float64, "device": DEV}
    best = torch.full((n,), math.inf, **f)
    nrm, alb = torch.zeros((3, n), **f), torch.zeros((3, n), **f)
    for o, A, b in _instances(case):
        A, b = _t(np.asarray(A, np.float32)), _t(np.asarray(b, np.float32))
        r = rays.double()
        r[0:3], r[3:6] = A @ r[0:3] + b[:, None], A @ r[3:6]
        q = _Solid(f"stress{o}").query(r)
        win = q["hit"] & (q["t"] < best)
        best = torch.where(win, q["t"], best)
        nrm = torch.where(win, _unit((A.T @ q["normal"]).T).T, nrm)
        alb = torch.where(win, q["albedo"], alb)
    return {"hit": None, "t": best, "normal": nrm, "mat": None, "albedo": alb, "instance": None, "bounce": None}


def exact(case: dict, seed: int):
    with torch.no_grad():
        if case["kind"] == "scene":
            return _exact_scene(case, seed)
        if case["kind"] == "mixed":
            rays, who = _mixed_batch(case, seed)
            out = {"hit": None, "t": torch.zeros(rays.shape[1], dtype=torch.float64, device=DEV), "mat": None}
            out |= {f: torch.zeros((3, rays.shape[1]), dtype=torch.float64, device=DEV) for f in ("normal", "albedo")}
            for i in range(case["objects"]):
                at = (who == i).nonzero()[:, 0]
                q = _Solid(f"mixed{i}").query(rays[:, at])
                out["t"][at], out["normal"][:, at], out["albedo"][:, at] = q["t"], q["normal"], q["albedo"]
            return out
        if case["kind"] == "query":
            q = _Solid(case["object"]).query(_case_rays(case, seed))
            out = {"hit": None, "t": q["t"], "normal": q["normal"], "mat": None, "albedo": q["albedo"]}
            return out | {"logits": q["logits"]} if _logits(case) else out
    return _exact_train(case, seed)
