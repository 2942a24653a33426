"""Workloads of the light tracer whose time is followed, through its public entry points.

A case names a scene of the synthetic generators (`scene`, film side `res`, height-field side
`hm`), how many light paths of which depth are traced, and the method that turns them into an
image and gradients.  One pass is one call or one optimisation step as a program makes it:

    lrb3     refit, primal, film loss, LRB-3-pass backward with its state kept between steps
    reslrb, naive, lrb2   `render` and its backward through autograd, by that method
    learned  ResLRB primal and backward with the learned reservoir target
    primal   refit and a forward render only
    bidir    bidirectional image and its gradient
    batch    primal and LRB-3 pass of many uneven scenes in persistent launches
    mlp      one training epoch of the learned target's network on collected pairs
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2609_32920_gb300 import inputs as I
from paper_2609_32920_gb300 import lt
from paper_2609_32920_gb300.autograd import render

DEV = "cuda"


def listed():
    def c(name, method, scene, res, hm, paths, depth, attached, filter=0, rr_depth=0, rr_prob=1.0, extra=0):
        return dict(name=name, method=method, scene=scene, res=res, hm=hm, paths=paths, depth=depth,
                    attached=attached, filter=filter, rr_depth=rr_depth, rr_prob=rr_prob, extra=extra)
    return [
        # the smallest optimisation step: the textured box at 64 x 64, albedo only, where the
        # launches and the longest single path count
        c("box_small_step", "lrb3", "box", 64, 0, 1 << 14, 4, 0),
        # a step of a geometry optimisation at interactive size, ragged in every size: a
        # 45 x 45 dielectric height field, odd film and path counts
        c("caustic_ragged_step", "lrb3", "slab", 101, 45, 65537, 13, 1),
        # the interior workload: high connectivity, 16 bounces, albedo, radiance and heights
        c("box_step", "lrb3", "box", 256, 32, 1 << 22, 16, 1),
        # the caustic workload the benchmark quotes: few connections, specular chains
        c("caustic_step", "lrb3", "slab", 512, 128, 1 << 24, 8, 1),
        # ResLRB through autograd on the interior
        c("box_reslrb", "reslrb", "box", 256, 32, 1 << 20, 16, 1),
        # ResLRB with the learned target on refraction inside a closed interior
        c("slabbox_learned", "learned", "slabbox", 256, 64, 1 << 20, 32, 1),
        # the buffered two-pass method through autograd
        c("box_lrb2", "lrb2", "box", 256, 32, 1 << 20, 16, 1),
        # tape differentiation through autograd, the method others are compared with
        c("caustic_naive", "naive", "slab", 256, 64, 1 << 20, 8, 1),
        # a forward render: deep paths under Russian roulette, the wider film filter
        c("box_render", "primal", "box", 256, 32, 1500007, 64, 0, filter=1, rr_depth=4, rr_prob=0.8),
        # the bidirectional estimator, light paths and camera samples (extra)
        c("box_bidir", "bidir", "box", 256, 0, 1 << 21, 6, 0, extra=1 << 19),
        # uneven scenes (extra of them) in one persistent launch per pass; paths: the most of one
        c("batch_step", "batch", "mixed", 128, 96, 1 << 19, 24, 1, extra=8),
        # training the learned target on the pairs of one collection (paths: pairs)
        c("mlp_epoch", "mlp", "pairs", 0, 0, 1 << 17, 0, 0, extra=4096),
    ]


def draw(rng):
    def lg(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    method = rng.choice(["lrb3", "lrb3", "lrb3", "reslrb", "learned", "lrb2", "naive", "primal", "bidir", "batch", "mlp"])
    c = dict(method=method, scene=rng.choice(["box", "slab", "slabbox"]), res=lg(48, 512), hm=lg(8, 128),
             paths=lg(1 << 14, 1 << 22), depth=lg(2, 32), attached=rng.randint(0, 1), filter=int(rng.random() < 0.25),
             rr_depth=0, rr_prob=1.0, extra=0)
    if rng.random() < 0.25:
        c.update(rr_depth=rng.randint(2, 6), rr_prob=round(rng.uniform(0.6, 0.95), 2))
    if method == "lrb3" and c["scene"] == "slab":
        c["paths"] = lg(1 << 14, 1 << 24)
        c["depth"] = min(c["depth"], 8)
    if method in ("naive", "lrb2") or c["scene"] == "slabbox":
        c["paths"] = lg(1 << 14, 1 << 20)
    if c["scene"] == "box" and rng.random() < 0.3:
        c["hm"] = 0
    if method == "bidir":
        c.update(scene="box", attached=0, rr_depth=0, rr_prob=1.0, paths=lg(1 << 14, 1 << 21), depth=lg(2, 12))
        c["extra"] = c["paths"] // rng.randint(2, 8)
    elif method == "batch":
        c.update(scene="mixed", res=lg(48, 128), hm=lg(24, 128), paths=lg(1 << 15, 1 << 19), depth=lg(4, 32),
                 attached=1, filter=0, rr_depth=0, rr_prob=1.0, extra=rng.randint(2, 8))
    elif method == "mlp":
        c.update(scene="pairs", res=0, hm=0, paths=lg(1 << 13, 1 << 18), depth=0, attached=0, filter=0, rr_depth=0,
                 rr_prob=1.0, extra=rng.choice([1000, 2048, 4096, 8192]))
    return c


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=32)
def _topology(scene, res, hm):
    if scene == "box":
        return I.box_scene(res, heightmap=hm)
    return I.slab_scene(res, n=hm) if scene == "slab" else I.slab_in_box(res, n=hm)


def _scene(scene, res, hm, seed):
    """The scene with the textures and heights of one seed, as its generator distributes them."""
    sc = _topology(scene, res, hm)
    g = np.random.default_rng([seed, 1])
    alb = g.uniform(0.2, 0.8, sc.albedo.size) if sc.albedo.size > 64 else sc.albedo
    h = sc.heights
    if h.size:
        h = 0.02 * g.standard_normal(h.size) if scene == "box" else I.gaussian_bumps(
            hm, 1.0 if scene == "slab" else 0.5, seed + 100, amp_std=0.01 if scene == "slab" else 0.005)
    return sc.with_params(albedo=alb, heights=h)


def _film(sc, seed):
    """A target image near the scene's own brightness, with smooth and per-pixel differences."""
    d = I.smooth_adjoint(sc.W, sc.H, seed + 7) * (sc.W * sc.H)
    return torch.tensor(np.maximum(0.0, 0.3 * (1.0 + d)), dtype=torch.float32, device=DEV)


def _adjoint(sc, seed):
    return torch.tensor(I.smooth_adjoint(sc.W, sc.H, seed + 7), dtype=torch.float32, device=DEV)


def _opts(case, seed):
    return dict(seed=seed + 1, n_paths=case["paths"], max_depth=case["depth"], filter=case["filter"],
                rr_depth=case["rr_depth"], rr_prob=case["rr_prob"])


def _pairs(n, seed):
    """Feature rows and targets with the ranges that connections have in a unit box."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    f = torch.randn((n, 16), generator=g, device=DEV)
    f[:, 0:3] = 0.5 + 0.3 * f[:, 0:3]
    f[:, 9:12] = 1.0 + f[:, 9:12]
    f[:, 12:15] = torch.rand((n, 3), generator=g, device=DEV)
    f[:, 15] = f[:, 15] - 3.0
    t = torch.sin(3.0 * f[:, 0]) + f[:, 3] * f[:, 6] - 0.5 * f[:, 12] - 9.0
    return f, t + 0.3 * torch.randn(n, generator=g, device=DEV)


def _network(seed):
    """Network weights with the standardisation of such features."""
    P = lt.mlp_init(seed, DEV)
    mean = torch.tensor([0.5] * 3 + [0.0] * 6 + [1.0] * 3 + [0.5] * 3 + [-14.0], device=DEV)
    std = torch.tensor([0.3] * 3 + [0.6] * 6 + [1.0] * 3 + [0.3] * 3 + [1.5], device=DEV)
    P[5313:5329], P[5329:5345] = mean, 1.0 / std
    return P


def _batch_specs(case):
    """Heights sides, depths and path counts of the batch, uneven as the batched set's are."""
    g = np.random.default_rng([case["extra"], case["paths"]])
    for k in range(case["extra"]):
        yield dict(scene="slab" if k % 2 == 0 else "box", hm=int(max(8, round(case["hm"] * 2 ** g.uniform(-2, 0)))),
                   paths=int(round(case["paths"] * 2 ** g.uniform(-5, 0))), depth=int(g.integers(4, max(5, case["depth"] + 1))))


def prepare(case, seed):
    m = case["method"]
    if m == "mlp":
        f, t = _pairs(case["paths"], seed)
        return dict(case=case, P0=lt.mlp_init(seed, DEV), f=f, t=t)
    if m == "batch":
        items = []
        for k, s in enumerate(_batch_specs(case)):
            sc = _scene(s["scene"], case["res"], s["hm"], seed + k)
            S = lt.Scene(sc)
            items.append(dict(scene=S, n_paths=s["paths"], max_depth=s["depth"], attached=1, seed=seed + k,
                              lrb3_state=True, heights=S.heights.clone(), d_image=_adjoint(sc, seed + k)))
        return dict(case=case, items=items, batch=lt.Batch(items))
    sc = _scene(case["scene"], case["res"], case["hm"], seed)
    S = lt.Scene(sc)
    st = dict(case=case, S=S, heights=S.heights.clone(), kw=_opts(case, seed))
    if m == "lrb3":
        state = S.new_lrb3_state(case["paths"])
        st.update(primal=S.opts(lrb3_state=state, **st["kw"]), target=_film(sc, seed), image=S.new_image(),
                  backward=S.opts(lrb3_state=state, lrb3_mask_ready=1, attached=case["attached"], **st["kw"]),
                  dI=S.new_image(), loss=torch.empty(1, device=DEV), grads=S.new_grads())
    elif m in ("reslrb", "naive", "lrb2"):
        st["params"] = [x.clone().requires_grad_() for x in (S.albedo, S.Le, S.heights)]
        st["dI"] = _adjoint(sc, seed)
    elif m == "learned":
        st.update(opts=S.opts(attached=case["attached"], target=lt.TARGET_MLP, mlp=_network(seed), **st["kw"]),
                  records=torch.zeros((case["paths"], 8), device=DEV), dI=_adjoint(sc, seed), image=S.new_image(),
                  grads=S.new_grads())
    elif m == "primal":
        st.update(opts=S.opts(**st["kw"]), image=S.new_image())
    else:
        st.update(opts=S.opts(**st["kw"]), bidir=S.bidir_opts(case["extra"]), dI=_adjoint(sc, seed),
                  image=S.new_image(), grads=S.new_grads())
    return st


def run(st):
    case = st["case"]
    m = case["method"]
    if m == "mlp":
        P = st["P0"].clone()
        losses = lt.mlp_train(P, st["f"], st["t"], epochs=1, batch=case["extra"])
        return dict(P=P, losses=losses)
    if m == "batch":
        st["batch"].run(lt.PASS_PRIMAL)
        st["batch"].run(lt.PASS_LRB3)
        return [dict(image=it["image"], grads=it["grads"]) for it in st["items"]]
    S = st["S"]
    if m in ("reslrb", "naive", "lrb2"):
        for x in st["params"]:
            x.grad = None
        img = render(S, *st["params"], method=m, attached=bool(case["attached"]), **st["kw"])
        img.backward(st["dI"])
        return dict(image=img.detach(), grads=[x.grad for x in st["params"]])
    if S.n_heights:
        S.refit(st["heights"])
    if m == "lrb3":
        S.primal(st["primal"], image=st["image"])
        lt.film_l2(st["image"], st["target"], d_image=st["dI"], loss=st["loss"])
        S.backward_lrb3(st["backward"], st["dI"], grads=st["grads"])
        return dict(image=st["image"], loss=st["loss"], dI=st["dI"], grads=st["grads"])
    if m == "primal":
        return S.primal(st["opts"], image=st["image"])
    if m == "learned":
        S.primal(st["opts"], estimator=lt.EST_RESLRB, image=st["image"], aux=st["records"])
        S.backward_reslrb(st["opts"], st["dI"], st["records"], grads=st["grads"])
        return dict(image=st["image"], records=st["records"], grads=st["grads"])
    S.bidir_primal(st["opts"], st["bidir"], image=st["image"])
    S.bidir_backward(st["opts"], st["bidir"], st["dI"], grads=st["grads"])
    return dict(image=st["image"], grads=st["grads"])


# ------------------------------------------------------------------ work
def _path_work(scene, hm, paths, depth, q=1.0, d0=64):
    """(vertices, connections) of the primal's paths.  In the open box a path goes on from a
    vertex with probability 0.72; of the caustic's paths a quarter meets the slab or the
    receiver, a third of those by way of two or more specular vertices."""
    if scene == "slab":
        return paths * min(depth, 3) * 0.2, paths * 0.11
    live, n = 1.0, 0.0
    for k in range(depth):
        n += live
        live *= 0.72 * (q if k + 1 >= d0 else 1.0)
    return paths * n, paths * n * (0.6 if scene == "box" else 0.4)


def _trace_flops(scene, res, hm, paths, depth, rays, rr=(0, 1.0)):
    """One walk over the paths: `rays` rays a vertex, each through a 4-ary tree (24 a box, 30
    a primitive) and the few large walls, and 150 for the vertex itself."""
    v, c = _path_work(scene, hm, paths, depth, rr[1], rr[0] if rr[0] else 64)
    per_ray = 30 * (6 if scene != "slab" else 2) + (24 * 4 * max(1.0, math.log(2 * hm * hm, 4)) / 2 + 60 if hm else 0)
    return v * (rays * per_ray + 150) + c * 100 + paths * 150


def _scene_bytes(scene, res, hm):
    return 52 * (2 * hm * hm + 8) + 4 * hm * hm * 2 + 4 * 3840 * 2 + 12 * res * res


def work(case):
    m, sc, res, hm, n, D = (case[k] for k in ("method", "scene", "res", "hm", "paths", "depth"))
    rr = (case["rr_depth"], case["rr_prob"])
    if m == "mlp":
        return {"bytes": 3 * 68 * n, "flops": 3 * 2 * 5184 * n}
    if m == "batch":
        b = f = 0
        for s in _batch_specs(case):
            w = work(dict(case, method="lrb3", scene=s["scene"], hm=s["hm"], paths=s["paths"], depth=s["depth"]))
            b, f = b + w["bytes"], f + w["flops"]
        return {"bytes": b, "flops": f}
    forward = _trace_flops(sc, res, hm, n, D, 2, rr)
    image = 12 * res * res
    b = _scene_bytes(sc, res, hm) + image
    if m == "primal":
        return {"bytes": b, "flops": forward}
    # a backward meets again the vertices up to a path's last connection, without visibility
    back = _trace_flops(sc, res, hm, n * (0.12 if sc == "slab" else 0.8), D, 1, rr)
    if m == "bidir":
        return {"bytes": 2 * b + image, "flops": (1 + 0.25 * 2) * forward + back}
    if m in ("reslrb", "learned"):
        return {"bytes": 2 * b + 64 * n, "flops": forward + 0.6 * back}
    if m == "naive":  # a tape record a vertex, written and read
        return {"bytes": 2 * b + 64 * _path_work(sc, hm, n, D)[0], "flops": forward + 150 * _path_work(sc, hm, n, D)[0]}
    if m == "lrb2":
        return {"bytes": 2 * b + 40 * _path_work(sc, hm, n, D)[0], "flops": forward + back}
    return {"bytes": 2 * b + 2 * image, "flops": forward + 2 * back}


# ------------------------------------------------------------------ exact values
# A light tracer in 64 bits on plain tensors: every ray against every primitive, the path's
# decisions taken on detached values, image and gradients by autograd through the frozen
# paths (a vertex after a specular one slides along its primitive's plane, any other keeps its
# surface coordinates and weighs its segment).
def _philox(seed, n, d, s):
    M = 0xFFFFFFFF
    c = [n & M, n >> 32, torch.full_like(n, d), torch.full_like(n, s)]
    k0, k1 = seed & M, (seed >> 32) & M
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [((p1 >> 32) & M) ^ c[1] ^ k0, p1 & M, ((p0 >> 32) & M) ^ c[3] ^ k1, p0 & M]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return [(x >> 8).double() / 16777216.0 for x in c]


def _dot(a, b):
    return (a * b).sum(-1, keepdim=True)


def _unit(a):
    return a / _dot(a, a).sqrt()


def _cosine(n, u0, u1):
    sign = torch.where(n[:, 2:] < 0, -1.0, 1.0).double()
    a = -1.0 / (sign + n[:, 2:])
    x, y = n[:, 0:1], n[:, 1:2]
    t = torch.cat([1 + sign * x * x * a, sign * x * y * a, -sign * x], 1)
    b = torch.cat([x * y * a, sign + y * y * a, -y], 1)
    r, ph, u0 = u0.sqrt()[:, None], 2 * math.pi * u1[:, None], u0[:, None]
    return t * r * ph.cos() + b * r * ph.sin() + n * (1 - u0).clamp(min=0).sqrt()


class _Exact:
    def __init__(self, sc, case):
        def t(a, dt=torch.float64):
            return torch.tensor(np.asarray(a), dtype=dt, device=DEV)
        f32 = np.float32  # the library holds its geometry and parameters in 32 bits
        self.sc, self.case = sc, case
        self.quads = t(sc.quads.astype(f32))
        self.verts, self.vert_h = t(sc.verts.astype(f32).reshape(-1, 3)), t(sc.vert_h.reshape(-1), torch.int64)
        self.tris, self.mat = t(sc.tris.reshape(-1, 3), torch.int64), t(sc.prim_mat, torch.int64)
        self.kind, self.ior = t(sc.mat_type, torch.int64), t(sc.mat_ior.astype(f32))
        self.off, self.tw, self.th = (t(a, torch.int64) for a in (sc.mat_tex_off, sc.mat_tex_w, sc.mat_tex_h))
        self.albedo, self.Le = t(sc.albedo.astype(f32)), t(sc.Le.astype(f32))
        self.heights = t(sc.heights.astype(f32)) if sc.heights.size else t([0.0])
        pos, look, up = (t(a.astype(f32)) for a in (sc.cam_pos, sc.cam_look, sc.cam_up))
        self.cpos, self.cf = pos, _unit(look - pos)
        self.cr = _unit(torch.linalg.cross(self.cf, up))
        self.cu = torch.linalg.cross(self.cr, self.cf)
        self.ty = math.tan(math.radians(sc.fov_y_deg) / 2)
        self.tx = self.ty * sc.W / sc.H
        self.K0 = sc.W * sc.H / (4 * self.tx * self.ty * math.pi)

    def geometry(self, h):
        o, e1, e2 = self.quads[:, 0:3], self.quads[:, 3:6], self.quads[:, 6:9]
        if self.tris.numel():
            hv = torch.where(self.vert_h >= 0, h[self.vert_h.clamp(min=0)], torch.zeros((), dtype=h.dtype, device=DEV))
            v = self.verts + torch.stack([0 * hv, hv, 0 * hv], 1)
            a, b, c = v[self.tris[:, 0]], v[self.tris[:, 1]], v[self.tris[:, 2]]
            o, e1, e2 = torch.cat([o, a]), torch.cat([e1, b - a]), torch.cat([e2, c - a])
        return o, e1, e2

    def hits(self, G, org, d, skip, tmax=None):
        """Closest primitive and its (t, u, v) for each ray; with tmax, whether any lies before it."""
        o, e1, e2 = (g.detach() for g in G)
        nq, P, n = self.quads.shape[0], o.shape[0], org.shape[0]
        out = [torch.empty(n, dtype=torch.float64, device=DEV) for _ in range(3)]
        prim = torch.empty(n, dtype=torch.int64, device=DEV)
        tri = torch.arange(P, device=DEV) >= nq
        step = max(1, 24_000_000 // P)
        m = torch.linalg.cross(e1, e2)
        for i in range(0, n, step):
            s = slice(i, i + step)
            # with q = (org - o): det = -d.m, t = q.m / det, u = (q x d).e2 / det, v = -(q x d).e1 / det
            det = -(d[s] @ m.T)
            qd = torch.linalg.cross(org[s], d[s])
            od_e2 = d[s] @ torch.linalg.cross(e2, o).T   # (o x d) . e2 = d . (e2 x o)
            od_e1 = d[s] @ torch.linalg.cross(e1, o).T
            t = (org[s] @ m.T - (o * m).sum(1)) / det
            u, v = (qd @ e2.T - od_e2) / det, -(qd @ e1.T - od_e1) / det
            ok = (det != 0) & (t > 1e-5) & (u >= 0) & (v >= 0) & torch.where(tri, u + v <= 1, (u <= 1) & (v <= 1))
            ok &= torch.arange(P, device=DEV) != skip[s, None]
            t = torch.where(ok, t, math.inf)
            best, j = t.min(1)
            prim[s] = torch.where(best < math.inf, j, -1)
            for dst, x in zip(out, (best, u.gather(1, j[:, None])[:, 0], v.gather(1, j[:, None])[:, 0])):
                dst[s] = x
        return (prim >= 0) & (out[0] < tmax) if tmax is not None else (prim, *out)

    def film(self, x):
        d = x - self.cpos
        z = d @ self.cf
        return (0.5 * self.sc.W * (1 + (d @ self.cr) / z / self.tx), 0.5 * self.sc.H * (1 - (d @ self.cu) / z / self.ty), z)

    def splat(self, img, ux, uy, L):
        W, H = self.sc.W, self.sc.H
        if self.case["filter"]:
            cut = math.exp(-4.5)
            C = math.sqrt(math.pi / 2) * math.erf(1.5 * math.sqrt(2)) - 3 * cut
            taps = [-1, 0, 1, 2]

            def w(u, X):
                e = u - (X + 0.5)
                return torch.where(e.abs() < 1.5, ((-2 * e * e).exp() - cut) / C, 0.0)
        else:
            taps = [0, 1]

            def w(u, X):
                return (1 - (u - (X + 0.5)).abs()).clamp(min=0)
        x0, y0 = (ux.detach() - 0.5).floor(), (uy.detach() - 0.5).floor()
        for j in taps:
            for i in taps:
                X, Y = x0 + i, y0 + j
                on = (X >= 0) & (X < W) & (Y >= 0) & (Y < H)
                at = (Y * W + X).long()[on]
                img = img.index_add(0, at, (w(ux, X) * w(uy, Y))[on, None] * L[on])
        return img

    def texture(self, albedo, mat, s, t):
        tw, th, off = self.tw[mat], self.th[mat], self.off[mat]
        x, y = s * tw - 0.5, t * th - 0.5
        x0, y0 = x.detach().floor(), y.detach().floor()
        fx, fy = (x - x0)[:, None], (y - y0)[:, None]
        xs = [torch.minimum((x0 + i).clamp(min=0), tw - 1).long() for i in (0, 1)]
        ys = [torch.minimum((y0 + i).clamp(min=0), th - 1).long() for i in (0, 1)]

        def at(j, i):
            k = off + 3 * (ys[j] * tw + xs[i])
            return albedo[k[:, None] + torch.arange(3, device=DEV)]
        return (at(0, 0) * (1 - fx) + at(0, 1) * fx) * (1 - fy) + (at(1, 0) * (1 - fx) + at(1, 1) * fx) * fy

    def image(self, n, albedo, Le, heights, seed, inv_n):
        """Image of the paths `n`, differentiable in its parameters (heights where they ask for it)."""
        sc, case = self.sc, self.case
        G = self.geometry(heights)
        att = heights.requires_grad
        img = torch.zeros((sc.W * sc.H, 3), dtype=torch.float64, device=DEV)
        q = self.quads[sc.emitter_quad]
        le1, le2 = q[3:6], q[6:9]
        ln = torch.linalg.cross(le1, le2)
        area = ln.norm()
        ln = (ln / area).expand(n.numel(), 3)
        r = _philox(seed, n, 0, 0)
        x = q[0:3] + r[0][:, None] * le1 + r[1][:, None] * le2
        d = _cosine(ln, r[2], r[3])
        nr = ln                                  # the previous vertex's unnormalised normal
        skip = torch.full_like(n, sc.emitter_quad)
        beta = (Le * area * math.pi).expand(n.numel(), 3)
        spec = torch.zeros(n.numel(), dtype=torch.bool, device=DEV)
        for k in range(case["depth"]):
            prim, _, u, v = self.hits(G, x.detach(), d.detach(), skip)
            live = prim >= 0
            live &= self.kind[self.mat[prim.clamp(min=0)]] != 2
            n, x, d, nr, beta, spec, prim, u, v = (a[live] for a in (n, x, d, nr, beta, spec, prim, u, v))
            if not n.numel():
                break
            o, e1, e2 = (g[prim] for g in G)
            m = torch.linalg.cross(e1, e2)
            y = o + u[:, None] * e1 + v[:, None] * e2
            slid = x + d * (_dot(o - x, m) / _dot(d, m))
            y = torch.where(spec[:, None], slid, y)
            w = y - x
            if att:
                g = (_dot(nr, w) * _dot(m, w)).abs() / (_dot(nr, nr).sqrt() * _dot(w, w) ** 2)
                beta = beta * torch.where(spec[:, None], torch.ones_like(g), g / g.detach())
                d = torch.where(spec[:, None], d, _unit(w))
            mat = self.mat[prim]
            ior = self.ior[mat][:, None]
            diff = self.kind[mat] == 0
            nn = _unit(m)
            ns = torch.where(_dot(nn, d) < 0, nn, -nn)
            r = _philox(seed, n, k + 1, 0)
            if diff.any():
                q2, mm = y - o, _dot(m, m)       # surface coordinates of a sliding vertex follow it
                ts = torch.where(spec, (_dot(torch.linalg.cross(q2, e2), m) / mm)[:, 0], u)
                tt = torch.where(spec, (_dot(torch.linalg.cross(e1, q2), m) / mm)[:, 0], v)
                rho = self.texture(albedo, torch.where(diff, mat, mat[diff][0]), ts, tt)
                cv = self.cpos - y
                dist = _dot(cv, cv).sqrt()
                cosc = _dot(ns, cv / dist)
                ux, uy, z = self.film(y)
                c = diff & (cosc[:, 0] > 0) & (z > 0) & (ux >= 0) & (ux < sc.W) & (uy >= 0) & (uy < sc.H)
                i = c.nonzero()[:, 0]
                if i.numel():
                    occ = self.hits(G, y[i].detach(), (cv / dist)[i].detach(), prim[i], dist[i, 0].detach() - 1e-5)
                    i = i[~occ]
                    geo = cosc * self.K0 / (dist * dist * (z[:, None] / dist) ** 3)
                    img = self.splat(img, ux[i], uy[i], (beta * rho * geo * inv_n)[i])
                beta = torch.where(diff[:, None], beta * rho, beta)
            # dielectric branch
            into = _dot(d, nn) < 0
            eta = torch.where(into, 1 / ior, ior)
            ci = -_dot(d, ns)
            s2 = eta * eta * (1 - ci * ci)
            tir = s2 >= 1
            ct = (1 - torch.where(tir, torch.zeros_like(s2), s2)).sqrt()
            F = 0.5 * (((eta * ci - ct) / (eta * ci + ct)) ** 2 + ((ci - eta * ct) / (ci + eta * ct)) ** 2)
            back = tir | (r[2][:, None] < F)
            dout = torch.where(back, d + 2 * ci * ns, eta * d + (eta * ci - ct) * ns)
            if att:
                keep = torch.where(back, F, 1 - F)
                ratio = torch.where(tir, torch.ones_like(keep), keep / keep.detach())
                beta = torch.where(diff[:, None], beta, beta * ratio)
            d = torch.where(diff[:, None], _cosine(ns.detach(), r[0], r[1]), dout)
            spec, x, nr, skip = ~diff, y, m, prim
            if case["rr_depth"] and k + 1 >= case["rr_depth"]:
                on = _philox(seed, n, k + 1, 2)[0] < float(np.float32(case["rr_prob"]))
                n, x, d, nr, beta, spec, skip = (a[on] for a in (n, x, d, nr, beta / case["rr_prob"], spec, skip))
        return img.view(sc.H, sc.W, 3)


def exact(case, seed):
    m = case["method"]
    if m == "mlp":
        return _exact_epoch(case, seed)
    if m not in ("lrb3", "lrb2", "naive", "primal"):
        return None  # decided by sampled weights or of many scenes: held to the start's outputs
    sc = _scene(case["scene"], case["res"], case["hm"], seed)
    steps = case["paths"] * sc.n_prims * max(1.0, _path_work(case["scene"], 0, 1, case["depth"])[0])
    if steps * (1 if m == "primal" else 3) > 3e10:
        return None
    E = _Exact(sc, case)
    n = torch.arange(case["paths"], device=DEV)
    parts = n.split(1 << 16)
    args = (seed + 1, 1.0 / case["paths"])
    with torch.no_grad():
        img = sum(E.image(p, E.albedo, E.Le, E.heights, *args) for p in parts)
    if m == "primal":
        return img
    out = {}
    if m == "lrb3":
        e = img - _film(sc, seed).double()
        dI = 2 * e / e.numel()
        out = dict(loss=(e * e).mean().view(1), dI=dI)
    else:
        dI = _adjoint(sc, seed).double()
    par = [E.albedo.clone().requires_grad_(), E.Le.clone().requires_grad_(), E.heights.clone()]
    par[2].requires_grad_(bool(case["attached"] and sc.heights.size))
    for p in parts:
        value = (E.image(p, *par, *args) * dI).sum()
        if value.requires_grad:  # a few paths may all miss the film
            value.backward()
    grads = [torch.zeros_like(x) if x.grad is None else x.grad for x in par]
    return dict(image=img, grads=grads, **out)


def _exact_epoch(case, seed):
    """One epoch of Adam on the standardised squared error, in 64 bits."""
    f, t = (a.double() for a in _pairs(case["paths"], seed))
    P = lt.mlp_init(seed, DEV).double()
    P[5313:5329], P[5329:5345] = f.mean(0), 1.0 / f.var(0, unbiased=False).sqrt()
    P[5345], P[5346] = t.var(unbiased=False).sqrt(), t.mean()
    x, y = (f - P[5313:5329]) * P[5329:5345], (t - P[5346]) / P[5345]
    perm = torch.randperm(case["paths"], generator=torch.Generator().manual_seed(0)).to(DEV)
    x, y = x[perm], y[perm]
    w = P[:5313].clone().requires_grad_()
    mom, var, total, nb = torch.zeros(5313, device=DEV).double(), torch.zeros(5313, device=DEV).double(), 0.0, 0
    for b in range(0, case["paths"], case["extra"]):
        W1, b1, W2, b2, W3, b3 = (w[a:z] for a, z in ((0, 1024), (1024, 1088), (1088, 5184), (5184, 5248), (5248, 5312), (5312, 5313)))
        h = (x[b:b + case["extra"]] @ W1.view(16, 64) + b1).relu()
        h = (h @ W2.view(64, 64) + b2).relu()
        loss = ((h @ W3 + b3 - y[b:b + case["extra"]]) ** 2).mean()
        g, = torch.autograd.grad(loss, w)
        nb += 1
        mom, var = 0.9 * mom + 0.1 * g, 0.999 * var + 0.001 * g * g
        with torch.no_grad():
            w -= 1e-3 * (mom / (1 - 0.9 ** nb)) / ((var / (1 - 0.999 ** nb)).sqrt() + 1e-8)
        total += float(loss)
    P[:5313] = w.detach()
    return dict(P=P, losses=[total / nb])
