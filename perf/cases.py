"""Workloads of the 3DGS^2-TR hot path for timing and comparison.

`listed()` names the workloads, `draw(rng)` gives further ones of the same
ranges, `prepare(case, seed)` makes what a training or serving program holds
before the call, `run(state)` makes one pass through the public entry points
(`engine.TRStep`, `engine.BatchStep`, `autograd.render`, the C-ABI binding) and
`exact(case, seed)` evaluates the same definition in FP64 with plain PyTorch.
"""
from __future__ import annotations

import math
import random
from dataclasses import dataclass

import numpy as np
import torch

from paper_2602_00395_gb300 import gs3dtr as G
from paper_2602_00395_gb300 import synth
from paper_2602_00395_gb300.autograd import render
from paper_2602_00395_gb300.engine import BatchEntry, BatchStep, TRConfig, TRStep

DEV = "cuda"
PROBE_SEED = 42
EPS = 1e-6
GN_FLOOR = 1e-3
LAMBDA = 0.2


# ------------------------------------------------------------------ the cases
def _case(name, kind, n, deg, views, w, h, nu, scene):
    c = dict(kind=kind, n=n, deg=deg, views=views, w=w, h=h, nu=nu, scene=scene)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the tiny plain step: 1,000 Gaussians, 128x128, one probe; launches and latency count
        _case("step 1k 128x128", "step", 1000, 0, 1, 128, 128, 1, "unit"),
        # a served render (no probes) of a small scene, its count and image not multiples of anything
        _case("render 61k 800x600", "render", 61325, 3, 1, 800, 600, 0, "cube"),
        # a served batch of training steps: four scenes of 256x256 in shared launches
        _case("served batch 4x301k 256x256", "batch", 301056, 3, 4, 256, 256, 1, "cube"),
        # the reverse pass of plain single-view training (100k, 1297x840, one probe)
        _case("reverse 100k 1297x840", "reverse", 100000, 3, 1, 1297, 840, 1, "cube"),
        # the calls of the batched multi-view step (1M Gaussians, 8 views of 1080p, two probes), one by one
        _case("project 1M x8 nu2", "project", 1000000, 3, 8, 1920, 1080, 2, "clusters"),
        _case("sort 1M x8", "sort", 1000000, 3, 8, 1920, 1080, 2, "clusters"),
        _case("forward 1M x8 nu2", "forward", 1000000, 3, 8, 1920, 1080, 2, "clusters"),
        _case("reverse 1M x8 nu2", "reverse", 1000000, 3, 8, 1920, 1080, 2, "clusters"),
        _case("update 1M", "update", 1000000, 3, 1, 64, 64, 1, "clusters"),
        # the D-SSIM pixel loss of the same frame: gradient and both curvature cotangents
        _case("dssim x8 1080p nu2", "dssim", 1024, 0, 8, 1920, 1080, 2, "unit"),
        # the large scene through torch.autograd: a 6M render and its backward pass
        _case("autograd 6M 1080p", "autograd", 6000000, 3, 1, 1920, 1080, 0, "clusters"),
        # the whole batched multi-view step, replayed from its captured CUDA graph
        _case("graph step 1M x8 nu2", "graph", 1000000, 3, 8, 1920, 1080, 2, "clusters"),
    ]


def draw(rng):
    kind = rng.choice(["step", "render", "batch", "reverse", "reverse", "project", "sort", "forward", "update",
                       "dssim", "autograd", "graph"])
    logu = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))
    if kind == "batch":
        w, h = rng.choice([(256, 256), (800, 600), (logu(65, 640), logu(65, 480))])
        return _case(None, kind, logu(50000, 500000), 3, rng.randint(2, 5), w, h, 1, "cube")
    scene = rng.choice(["unit", "cube", "clusters", "clusters"])
    views = 1 if kind == "autograd" else rng.choice([1, 1, 2, 3, 5, 8])
    n = logu(300, 20000) if scene == "unit" else logu(50000, 2000000 // views)
    w, h = rng.choice([(256, 256), (800, 600), (1297, 840), (1920, 1080), (logu(65, 1920), logu(49, 1080))])
    if scene == "unit":
        w, h = logu(33, 400), logu(33, 400)
    nu = 0 if kind in ("render", "autograd") else rng.choice([0, 1, 2, 2])
    if kind in ("step", "update", "graph"):
        nu = max(nu, 1)
    return _case(None, kind, n, rng.choice([0, 1, 2, 3, 3, 3]), views, w, h, nu, scene)


# ------------------------------------------------------------------ the inputs
@dataclass
class Cam:
    viewmat: np.ndarray
    fx: float
    fy: float
    cx: float
    cy: float
    near: float
    width: int
    height: int


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _params(c, seed):
    """Parameter matrix rows x n: the seeded scene distributions of the configurations."""
    g, n, K = _gen(seed), c["n"], (c["deg"] + 1) ** 2
    nrm = lambda *s: torch.randn(*s, generator=g, device=DEV)
    if c["scene"] == "clusters":  # 20 clusters of sigma 0.3 in a radius-10 ball
        d = nrm(3, 20)
        ctr = d / d.norm(dim=0) * 10.0 * torch.rand(20, generator=g, device=DEV) ** (1.0 / 3.0)
        mu = ctr[:, torch.randint(20, (n,), generator=g, device=DEV)] + 0.3 * nrm(3, n)
        shift = 0.0
    else:  # a uniform cube; scales as in the served scenes, so that the pairs per Gaussian stay comparable
        ext = 1.0 if c["scene"] == "unit" else 5.0
        mu = ext * (2.0 * torch.rand(3, n, generator=g, device=DEV) - 1.0)
        shift = 0.0 if c["scene"] == "unit" else math.log(ext) + math.log(1e5 / n) / 3.0
    q = nrm(4, n)
    sh = nrm(K, 3, n) * 0.1
    sh[0] = nrm(3, n) * 0.709
    return torch.cat([mu, nrm(3, n) * 0.5 - 3.0 + shift, q / q.norm(dim=0), nrm(1, n), sh.view(3 * K, n)])


def _cams(c, seed, count=None):
    """Cameras on a jittered ring around the scene, looking at its centre; 60 degrees of field of view."""
    r = random.Random(seed + 7)
    R = {"unit": 4.0, "cube": 12.0, "clusters": 24.0}[c["scene"]]
    fx, az0, out = 0.5 * c["w"] / math.tan(math.radians(30)), r.uniform(0, 2 * math.pi), []
    for v in range(count or c["views"]):
        az, el = az0 + 2 * math.pi * v / c["views"], math.radians(r.uniform(-15, 15))
        pos = R * np.array([math.cos(el) * math.cos(az), math.cos(el) * math.sin(az), math.sin(el)])
        vm = synth.look_at(pos + R / 120.0 * np.array([r.gauss(0, 1) for _ in range(3)]))
        out.append(Cam(vm.astype(np.float32), *(float(np.float32(x)) for x in (fx, fx, c["w"] / 2, c["h"] / 2, 0.2)),
                       c["w"], c["h"]))
    return out


def _target(c, seed, views=None):
    """Smooth target images in [0, 1], V x 3 x H x W."""
    g, V = _gen(seed + 1), views or c["views"]
    y = torch.linspace(0, 2 * math.pi, c["h"], device=DEV)[:, None]
    x = torch.linspace(0, 2 * math.pi, c["w"], device=DEV)[None, :]
    k = 0.5 + 3.5 * torch.rand(V, 3, 3, 2, generator=g, device=DEV)
    ph = 2 * math.pi * torch.rand(V, 3, 3, generator=g, device=DEV)
    img = torch.full((V, 3, c["h"], c["w"]), 0.5, device=DEV)
    for v in range(V):
        for ch in range(3):
            for j in range(3):
                img[v, ch] += 0.15 * torch.sin(k[v, ch, j, 0] * x + k[v, ch, j, 1] * y + ph[v, ch, j])
    return img.clamp_(0, 1)


def _engine(c, seed):
    e = TRStep(c["n"], c["deg"], c["views"], c["w"], c["h"], nu=c["nu"], cfg=TRConfig(l=1), probe_seed=PROBE_SEED)
    e.set_cameras(_cams(c, seed))
    e.set_params(_params(c, seed))
    return e


def _update_state(c, seed):
    """Gradient, curvature and EMAs of the sizes that the reverse passes leave them in."""
    g, s = _gen(seed + 2), (synth.n_rows(c["deg"]), c["n"])
    nrm = lambda: torch.randn(*s, generator=g, device=DEV)
    return 1e-6 * nrm(), 1e-9 * nrm().square(), 1e-6 * nrm(), 1e-9 * nrm().square()


def _dssim_inputs(c, seed):
    g = _gen(seed + 3)
    tgt = _target(c, seed)
    img = (tgt + 0.05 * torch.randn(tgt.shape, generator=g, device=DEV)).clamp_(0, 1)
    tan = 0.1 * torch.randn(max(c["nu"], 1), *tgt.shape, generator=g, device=DEV)
    return img, tgt, tan


def prepare(case, seed):
    c, kind = case, case["kind"]
    st = dict(c=c, t=0)
    if kind == "batch":
        st["scenes"] = _batch_scenes(c, seed)
        st["pool"] = {}
        entries = _entries(st, 1)
        need = 0
        for e in entries:  # the scenes' pair counts, as a server takes them when it loads a scene
            s = TRStep(e.n, c["deg"], 1, c["w"], c["h"], nu=c["nu"], state=(e.x, e.g_ema, e.d_ema), zero_init=False)
            s.cams = e.cam
            need += s.ensure_capacity()
        st["capacity"] = int(need * 1.25) + 1024
        return st
    if kind == "dssim":
        img, tgt, tan = _dssim_inputs(c, seed)
        fr = G.frame_struct(c["views"], c["w"], c["h"])
        ws = torch.empty(G.gs_dssim_workspace_size(fr, c["nu"]), dtype=torch.uint8, device=DEV)
        cot = torch.empty((1 + c["nu"], *tgt.shape), device=DEV)
        st.update(img=img, tgt=tgt, tan=tan, fr=fr, ws=ws, cot=cot, loss=torch.zeros(1, device=DEV))
        return st
    e = st["e"] = _engine(c, seed)
    e.ensure_capacity()
    if kind in ("step", "reverse", "graph"):
        e.set_target(_target(c, seed))
    if kind == "update":
        for dst, src in zip((e.grad, e.hz, e.g_ema, e.d_ema), _update_state(c, seed)):
            dst[:, : c["n"]].copy_(src)
    if kind == "sort":
        e.keys.zero_()  # the places past the pairs in use are the caller's, and stay
        e.vals.zero_()
    if kind in ("sort", "forward", "reverse"):
        e.project(1)
        if kind != "sort":
            e.bin_sort()
        if kind == "reverse":
            e.raster_fwd(1)
    if kind == "autograd":
        st["x"] = e.x.clone().requires_grad_(True)
        st["cot"] = (_target(c, seed) - 0.5) / (3 * c["w"] * c["h"] * c["views"])
    if kind == "graph":
        e.step(1, EPS)  # sets the kernels' attributes before the capture
        e.set_params(_params(c, seed))
        e.g_ema.zero_()
        e.d_ema.zero_()
        st["graph"] = e.capture_step(True, G.gs_eps_schedule(EPS, 1e-8, 30000))
    return st


def _batch_scenes(c, seed):
    """One scene per request, of sizes within a factor of two: parameters, state, camera and target."""
    out = []
    for b in range(c["views"]):
        sc = dict(c, n=int(c["n"] * 2 ** (b / c["views"] - 0.5)), views=1)
        p = _params(sc, seed + 100 * b)
        x = torch.zeros(p.shape[0], synth.pad_count(sc["n"]), device=DEV)
        x[:, : sc["n"]] = p
        cam = _cams(sc, seed + 100 * b)
        out.append(dict(c=sc, x=x, ge=torch.zeros_like(x), de=torch.zeros_like(x), cams=cam,
                        cam=torch.from_numpy(G.camera_bytes(cam)).to(DEV), tgt=_target(sc, seed + 100 * b).view(-1)))
    return out


def _entries(st, t):
    return [BatchEntry(s["x"], s["ge"], s["de"], s["c"]["n"], s["cam"], s["tgt"], t, EPS) for s in st["scenes"]]


# ------------------------------------------------------------------ one pass
def run(st):
    c, kind, e = st["c"], st["c"]["kind"], st.get("e")
    V, n, w, h, nu = c["views"], c["n"], c["w"], c["h"], c["nu"]
    if kind == "project":
        e.project(1)
        rec = e.rec.view(V, e.n_pad, 12)[:, :n]
        out = dict(rec=rec[..., :10], radius=rec.view(torch.int32)[..., 10], extents=rec.view(torch.int32)[..., 11])
        if nu:
            out["tan"] = e.tan.view(V, e.n_pad, 1 + nu, 12)[:, :n, 1:, :9]
        return out
    if kind == "sort":
        e.bin_sort()
        return dict(keys=e.keys, vals=e.vals, ranges=e.ranges, n_pairs=e.n_pairs)
    if kind in ("forward", "render"):
        e.raster_fwd(1) if kind == "forward" else e.render()
        out = dict(image=e.image.view(V, 3, h, w), T=e.final_T.view(V, h, w), n_contrib=e.n_contrib)
        if nu:
            out["tan"] = e.image_tan.view(nu, V, 3, h, w)
        return out
    if kind == "reverse":
        e.loss_val.zero_()
        e.raster_bwd(1)
        return dict(grad=e.grad[:, :n], loss=e.loss_val, **(dict(hz=e.hz[:, :n]) if nu else {}))
    if kind == "update":
        e.update(1, EPS)
        return dict(x=e.x[:, :n], g=e.g_ema[:, :n], d=e.d_ema[:, :n])
    if kind == "dssim":
        st["loss"].zero_()
        G.gs_dssim_cotangents(st["fr"], st["img"], st["tgt"], st["tan"] if nu else None, nu, LAMBDA, GN_FLOOR, True,
                              st["cot"], st["loss"], st["ws"])
        return dict(cot=st["cot"], loss=st["loss"])
    if kind == "autograd":
        img = render(st["x"], e)
        (grad,) = torch.autograd.grad(img, st["x"], st["cot"])
        return dict(image=img.detach(), grad=grad[:, :n])
    st["t"] += 1
    if kind == "batch":
        b = BatchStep(_entries(st, st["t"]), w, h, sh_degree=c["deg"], nu=nu, capacity=st["capacity"],
                      cfg=TRConfig(l=1), probe_seed=PROBE_SEED, pool=st["pool"])
        b.run()
        ns = [s["c"]["n"] for s in st["scenes"]]
        return dict(image=b.images(), loss=b.loss_val, grad=[g[:, :m] for g, m in zip(b.grads, ns)],
                    hz=[g[:, :m] for g, m in zip(b.hzs, ns)], x=[s["x"][:, :m] for s, m in zip(st["scenes"], ns)])
    if kind == "graph":
        st["graph"].replay()
    else:
        e.step(st["t"], EPS)
    return dict(image=e.image.view(V, 3, h, w), loss=e.loss_val, grad=e.grad[:, :n], hz=e.hz[:, :n], x=e.x[:, :n],
                g=e.g_ema[:, :n], d=e.d_ema[:, :n])


# ------------------------------------------------------------------ the work
def work(case):
    """Bytes and FP32 operations of one pass: inputs read once, outputs written
    once; the blends' operations per (pixel, splat) blended, with the typical
    numbers of tiles a splat reaches and of splats a pixel blends."""
    c = case
    V, n, nu, px = c["views"], c["n"], c["nu"], c["views"] * c["w"] * c["h"]
    prm = 4.0 * (11 + 3 * (c["deg"] + 1) ** 2) * n
    recs = 48.0 * n * V
    # 3-sigma width of a typical splat in pixels, and the 16 x 16 tiles that it meets
    dist, scale = {"unit": (4.0, 1.0), "cube": (12.0, 5.0 * (1e5 / n) ** (1 / 3)), "clusters": (24.0, 1.0)}[c["scene"]]
    wide = 6 * scale * math.exp(-3) * (0.5 * c["w"] / math.tan(math.radians(30))) / dist
    pairs = n * V * (wide / 16 + 1) ** 2
    blends = px * {"unit": 20, "cube": 25, "clusters": 13}[c["scene"]]
    if c["kind"] == "batch":
        prm *= V
        recs = 48.0 * n * V
    project = (prm + recs * (1 + (1 + nu if nu else 0)), n * V * 400.0 * (1 + nu))
    sort = (recs + 8.0 * pairs, 0.0)
    fwd = (recs * (1 + nu) + 4.0 * pairs + px * (20.0 + 12.0 * nu), blends * (20.0 + 25.0 * nu))
    rev = (recs + 4.0 * pairs + px * (32.0 + 12.0 * nu) + prm * (2 + (nu > 0)), blends * 50.0 * (1 + nu))
    upd = (8.0 * prm, 0.0)
    ssim = (px * 12.0 * (3 + 2 * nu), px * 3.0 * 22 * 2 * (5 + 3 + 6 * nu))
    parts = dict(project=[project], sort=[sort], forward=[fwd], render=[project, sort, fwd], reverse=[rev],
                 update=[upd], dssim=[ssim], autograd=[project, sort, fwd, rev])
    todo = parts.get(c["kind"], [project, sort, fwd, rev, upd])
    return dict(bytes=sum(p[0] for p in todo), flops=sum(p[1] for p in todo))


# ------------------------------------------------------------------ in 64 bits
def _basis(d, deg):
    x, y, z = d
    Y = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    if deg >= 1:
        k = math.sqrt(3 / (4 * math.pi))
        Y += [-k * y, k * z, -k * x]
    if deg >= 2:
        k = math.sqrt(15 / math.pi) / 2
        Y += [k * x * y, -k * y * z, math.sqrt(5 / math.pi) / 4 * (2 * z * z - x * x - y * y), -k * x * z,
              k / 2 * (x * x - y * y)]
    if deg >= 3:
        a, b, e, f = (math.sqrt(35 / (2 * math.pi)) / 4, math.sqrt(105 / math.pi) / 2,
                      math.sqrt(21 / (2 * math.pi)) / 4, math.sqrt(7 / math.pi) / 4)
        Y += [-a * y * (3 * x * x - y * y), b * x * y * z, -e * y * (4 * z * z - x * x - y * y),
              f * z * (2 * z * z - 3 * x * x - 3 * y * y), -e * x * (4 * z * z - x * x - y * y),
              b / 2 * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(Y)


def _rotation(q):
    x, y, z, w = q / q.norm(dim=0)
    return torch.stack([torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)]),
                        torch.stack([2 * (x * y + w * z), 1 - 2 * (z * z + x * x), 2 * (y * z - w * x)]),
                        torch.stack([2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)])])


def _fields(P, cam, deg):
    """(mx, my, A, B, C, opacity, r, g, b) x n of the splats, their depth and 3-sigma radius (0: culled)."""
    vm = torch.tensor(np.asarray(cam.viewmat, np.float64), device=DEV)
    Rc, tc = vm[:3, :3], vm[:3, 3]
    t = Rc @ P[:3] + tc[:, None]
    seen = t[2] > cam.near
    tz = torch.where(seen, t[2], torch.ones_like(t[2]))
    M = _rotation(P[6:10]) * torch.exp(P[3:6])[None]
    M = torch.einsum("ab,bcn->acn", Rc, M)
    Sc = torch.einsum("acn,bcn->abn", M, M)
    u, v = t[0] / tz, t[1] / tz
    limx, limy = 0.65 * cam.width / cam.fx, 0.65 * cam.height / cam.fy
    uc, vc = u.clamp(-limx, limx), v.clamp(-limy, limy)
    zero = torch.zeros_like(tz)
    J = torch.stack([torch.stack([cam.fx / tz, zero, -cam.fx * uc / tz]),
                     torch.stack([zero, cam.fy / tz, -cam.fy * vc / tz])])
    S2 = torch.einsum("ian,abn,jbn->ijn", J, Sc, J)
    a, b, d = S2[0, 0] + 0.3, S2[0, 1], S2[1, 1] + 0.3
    det = a * d - b * b
    mid = 0.5 * (a + d)
    rad = torch.ceil(3 * torch.sqrt(mid + torch.sqrt(torch.clamp(mid * mid - det, min=0.1))))
    dr = P[:3] + (Rc.T @ tc)[:, None]
    Y = _basis(dr / dr.norm(dim=0), deg)
    rgb = torch.clamp(0.5 + torch.einsum("kn,kcn->cn", Y, P[11:].view(-1, 3, P.shape[1])), min=0)
    F = torch.cat([torch.stack([cam.fx * u + cam.cx, cam.fy * v + cam.cy, d / det, -b / det, a / det,
                                torch.sigmoid(P[10])]), rgb])
    return torch.where(seen, F, torch.zeros_like(F)), (t[2] * seen).detach(), (rad * seen).detach()


def _probes(n, rows, t, k):
    """The Rademacher probe k of step t, rows x n: bits of SplitMix64."""
    with np.errstate(over="ignore"):
        U = np.uint64
        word = np.arange((n * rows + 63) // 64, dtype=U)
        key = U(PROBE_SEED) ^ (U(t) * U(0x9E3779B97F4A7C15)) ^ (U(k) << U(56))
        s = (key ^ word) + U(0x9E3779B97F4A7C15)
        s = (s ^ (s >> U(30))) * U(0xBF58476D1CE4E5B9)
        s = (s ^ (s >> U(27))) * U(0x94D049BB133111EB)
        s = s ^ (s >> U(31))
    bits = np.unpackbits(s.astype("<u8").view(np.uint8), bitorder="little")[: n * rows].reshape(n, rows)
    return torch.from_numpy(1.0 - 2.0 * bits.astype(np.float64)).to(DEV).T


def _tile_lists(F, depth, rad, w, h):
    """Splat index of every (tile, splat) pair of the splats' 3-sigma tile squares, by tile and depth."""
    Tx, Ty = -(-w // 16), -(-h // 16)
    lo = lambda m, T: torch.floor((m - rad) / 16).clamp(0, T).long()
    hi = lambda m, T: torch.floor((m + rad + 15) / 16).clamp(0, T).long()
    order = torch.argsort(depth, stable=True)
    x0, x1, y0, y1 = (v[order] for v in (lo(F[0], Tx), hi(F[0], Tx), lo(F[1], Ty), hi(F[1], Ty)))
    cnt = (x1 - x0).clamp(min=0) * (y1 - y0).clamp(min=0) * (rad[order] > 0)
    own = torch.repeat_interleave(torch.arange(len(cnt), device=DEV), cnt)
    q = torch.arange(len(own), device=DEV) - (torch.cumsum(cnt, 0) - cnt)[own]
    nx = (x1 - x0)[own]
    tile, at = torch.sort((y0[own] + q // nx) * Tx + x0[own] + q % nx, stable=True)
    return order[own[at]], torch.bincount(tile, minlength=Tx * Ty), Tx


def _blend(F, tans, depth, rad, w, h, cot_of, n_streams):
    """Front-to-back blend of one view: image, final T, tangent images, and the
    sums over pixels of each cotangent stream's derivative by the splat fields.
    cot_of(image, tangents, pixels) gives the streams' dL/dC at the pixels."""
    n, nu = F.shape[1], len(tans)
    idx, cnt, Tx = _tile_lists(F, depth, rad, w, h)
    start = torch.cumsum(cnt, 0) - cnt
    F1 = torch.cat([F, torch.zeros(9, 1, dtype=F.dtype, device=DEV)], 1)
    D1 = [torch.cat([d, torch.zeros(9, 1, dtype=F.dtype, device=DEV)], 1) for d in tans]
    img = torch.zeros(3, h * w, dtype=F.dtype, device=DEV)
    Tf = torch.ones(h * w, dtype=F.dtype, device=DEV)
    dimg = torch.zeros(nu, 3, h * w, dtype=F.dtype, device=DEV)
    sums = torch.zeros(n_streams, n + 1, 9, dtype=F.dtype, device=DEV)
    tiles = torch.argsort(cnt, descending=True)
    lens = cnt[tiles].tolist()
    sub = torch.arange(256, device=DEV)
    idx = torch.cat([idx, torch.full((1,), n, device=DEV)])
    a0 = 0
    while a0 < len(lens):  # all tiles: a pixel without splats still has a cotangent to report
        K = max(lens[a0], 1)
        a1 = min(len(lens), a0 + max(1, (12 << 20) // (256 * K)))
        tl = tiles[a0:a1]
        a0 = a1
        ks = torch.arange(K, device=DEV)[None]
        g = idx[torch.where(ks < cnt[tl][:, None], start[tl][:, None] + ks, torch.full_like(ks, len(idx) - 1))]
        X, Yp = (tl % Tx * 16)[:, None] + sub % 16, (tl // Tx * 16)[:, None] + sub // 16
        inside = (X < w) & (Yp < h)
        at = (Yp * w + X)[inside]
        f = F1[:, g][..., None]
        dx, dy = f[0] - (X + 0.5)[:, None], f[1] - (Yp + 0.5)[:, None]
        power = -0.5 * (f[2] * dx * dx + f[4] * dy * dy) - f[3] * dx * dy
        Gs = torch.exp(power)
        oG = f[5] * Gs
        al = oG.clamp(max=0.99)
        keep = (power <= 0) & (al >= 1 / 255)
        Ta = torch.cumprod(torch.where(keep, 1 - al, torch.ones_like(al)), 1)
        keep &= Ta >= 1e-4
        al = torch.where(keep, al, torch.zeros_like(al))
        om = 1 - al
        Ta = torch.cumprod(om, 1)
        Tb = Ta / om
        free = keep & (oG <= 0.99)
        wgt = al * Tb
        C = [(wgt * f[6 + q]).sum(1) for q in range(3)]
        da = [f[6 + q] * Tb - (C[q][:, None] - torch.cumsum(wgt * f[6 + q], 1)) / om for q in range(3)]
        for q in range(3):
            img[q, at] = C[q][inside]
        Tf[at] = Ta[:, -1][inside]
        dC = []
        for k in range(nu):
            d = D1[k][:, g][..., None]
            dp = (-0.5 * (d[2] * dx * dx + d[4] * dy * dy) - d[3] * dx * dy - (f[2] * dx + f[3] * dy) * d[0]
                  - (f[4] * dy + f[3] * dx) * d[1])
            dal = torch.where(free, d[5] * Gs + al * dp, torch.zeros_like(al))
            dC.append([(dal * da[q] + wgt * d[6 + q]).sum(1) for q in range(3)])
            for q in range(3):
                dimg[k, q, at] = dC[k][q][inside]
        if not n_streams:
            continue
        pix = torch.where(inside, Yp * w + X, torch.zeros_like(X))
        W = cot_of(torch.stack(C), torch.stack([torch.stack(v) for v in dC]) if nu else None, pix)
        for s in range(n_streams):
            Ws = W[s] * inside
            ga = sum(Ws[q][:, None] * da[q] for q in range(3)) * free
            gp = ga * al
            rows = [(-(f[2] * dx + f[3] * dy) * gp).sum(2), (-(f[4] * dy + f[3] * dx) * gp).sum(2),
                    -0.5 * (dx * dx * gp).sum(2), -(dx * dy * gp).sum(2), -0.5 * (dy * dy * gp).sum(2),
                    (ga * Gs).sum(2)] + [(wgt * Ws[q][:, None]).sum(2) for q in range(3)]
            sums[s].index_add_(0, g.reshape(-1), torch.stack(rows, -1).reshape(-1, 9))
    return img, Tf, dimg, sums[:, :n].transpose(1, 2)


def _passes(c, seed, P32, cams, target, nu, t, cot=None):
    """The whole path over the views: images, T, tangents, loss, gradient and Hutchinson diagonal."""
    P, V, w, h, n = P32.double(), len(cams), c["w"], c["h"], P32.shape[1]
    m = 3.0 * w * h * V
    zs = [_probes(n, P.shape[0], t, k) for k in range(nu)]
    imgs, Ts, dimgs, loss = [], [], [], 0.0
    grad, hz = torch.zeros_like(P), torch.zeros_like(P)
    for v, cam in enumerate(cams):
        fn = lambda p: _fields(p, cam, c["deg"])
        tans = [torch.func.jvp(lambda p: fn(p)[0], (P,), (z,))[1] for z in zs]
        Q = P.clone().requires_grad_(True)
        F, depth, rad = fn(Q)
        tgt = None if target is None else target[v].double().reshape(3, -1)

        def cot_of(C, dC, pix):
            if cot is not None:
                return [cot[v].double().reshape(3, -1)[:, pix]]
            r = C - tgt[:, pix]
            return [torch.sign(r) / (2 * m)] + [dC[k] / (4 * r.abs().clamp(min=GN_FLOOR)) / m for k in range(nu)]
        ns = 0 if tgt is None and cot is None else 1 + nu
        img, T, dimg, sums = _blend(F.detach(), tans, depth, rad, w, h, cot_of, ns)
        imgs.append(img.view(3, h, w))
        Ts.append(T.view(h, w))
        dimgs.append(dimg.view(nu, 3, h, w))
        if tgt is not None:
            loss += float((img - tgt).abs().sum()) / (2 * m)
        for s in range(ns):
            (gq,) = torch.autograd.grad(F, Q, sums[s], retain_graph=True)
            if s == 0:
                grad += gq
            else:
                hz += zs[s - 1] * gq / nu
        del F, Q
    return dict(image=torch.stack(imgs), T=torch.stack(Ts), tan=torch.stack(dimgs, 1), loss=torch.tensor([loss], dtype=torch.float64),
                grad=grad, hz=hz)


def _update(P32, grad, hz, g0, d0):
    """Algorithm 1 for one step: new x, g_ema, d_ema."""
    x = P32.double()
    g, d = 0.9 * g0.double() + 0.1 * grad, 0.999 * d0.double() + (1 - 0.999) * hz
    eps = float(np.float32(EPS))
    al, s, q = torch.sigmoid(x[10]), torch.exp(x[3:6]), x[6:10]
    R, L = _rotation(q), torch.log1p(-eps / al)
    eta = torch.full_like(x, math.inf)
    eta[:3] = torch.sqrt(-8 * L * torch.einsum("abn,bn->an", R * R, s * s))
    eta[3:6] = torch.sqrt(2 * eps / al)
    ln = q.norm(dim=0)
    X, Y, Z, W = q / ln
    om = torch.stack([torch.stack([W, -Z, Y]), torch.stack([Z, W, -X]), torch.stack([-Y, X, W]),
                      torch.stack([-X, -Y, -Z])]) * (2 / ln)
    r = torch.stack([s[1] / s[2] - s[2] / s[1], s[0] / s[2] - s[2] / s[0], s[0] / s[1] - s[1] / s[0]])
    eta[6:10] = torch.sqrt(-8 * L / (2 * (om * r[None]).square().sum(1)))
    eta[10] = torch.sqrt(4 * al * eps) / (al * (1 - al))
    Cc = (0.5 / math.sqrt(math.pi) * x[11:14] + 0.5).clamp(min=1e-2)
    top = {0: 1.0, 1: 1.0, 2: 1.0, 3: 1.0, 4: 0.5, 5: 0.5, 6: 2.0, 7: 0.5, 8: 1.0, 9: 1.0, 10: 3 ** -1.5,
           11: 16 / math.sqrt(135), 12: 2.0, 13: 16 / math.sqrt(135), 14: 2 / (3 * math.sqrt(3)), 15: 1.0}
    k1, k2, k35, k105 = (math.sqrt(v / math.pi) for v in (3 / 4, 15 / 4, 35 / 32, 105 / 4))
    amp = [0.5 / math.sqrt(math.pi), k1, k1, k1, k2, k2, math.sqrt(5 / math.pi) / 4, k2, k2 / 2, k35, k105,
           math.sqrt(21 / (2 * math.pi)) / 4, math.sqrt(7 / math.pi) / 4, math.sqrt(21 / (2 * math.pi)) / 4,
           k105 / 2, k35]
    for k in range((x.shape[0] - 11) // 3):
        eta[11 + 3 * k: 14 + 3 * k] = torch.sqrt(4 * Cc * eps / al) / (amp[k] * top[k])
    step = -g / d.clamp(min=float(np.float32(1e-12)))
    return x + torch.minimum(torch.maximum(step, -eta), eta), g, d


def _dssim(c, seed):
    img, tgt, tan = (v.double() for v in _dssim_inputs(c, seed))
    k = torch.exp(-torch.arange(-5, 6, dtype=torch.float64, device=DEV) ** 2 / 4.5)
    k = k / k.sum()

    def filt(a):
        b = a.reshape(-1, 1, *a.shape[-2:])
        b = torch.nn.functional.conv2d(b, k.view(1, 1, 11, 1), padding=(5, 0))
        return torch.nn.functional.conv2d(b, k.view(1, 1, 1, 11), padding=(0, 5)).reshape(a.shape)
    mx, my, ex, ey, exy = filt(img), filt(tgt), filt(img * img), filt(tgt * tgt), filt(img * tgt)
    A1, A2 = 2 * mx * my + 1e-4, 2 * (exy - mx * my) + 9e-4
    B1, B2 = mx * mx + my * my + 1e-4, ex - mx * mx + ey - my * my + 9e-4
    S = A1 * A2 / (B1 * B2)
    p2, p3 = -S / B2, 2 * A1 / (B1 * B2)
    p1 = 2 * A2 / (B1 * B2) * (my - mx * A1 / B1) - 2 * mx * p2 - my * p3
    adj = lambda a: filt(a * p1) + 2 * img * filt(a * p2) + tgt * filt(a * p3)
    r, m = img - tgt, 6.0 * c["w"] * c["h"] * c["views"]
    out = [((1 - LAMBDA) * torch.sign(r) - LAMBDA * adj(torch.ones_like(img))) / (2 * m)]
    for q in range(c["nu"]):
        d = tan[q]
        dS = p1 * filt(d) + p2 * filt(2 * img * d) + p3 * filt(tgt * d)
        a = LAMBDA / (4 * (1 - S).clamp(min=GN_FLOOR)) / m * dS
        out.append((1 - LAMBDA) / (4 * r.abs().clamp(min=GN_FLOOR)) / m * d + adj(a))
    loss = (((1 - LAMBDA) * r.abs() + LAMBDA * (1 - S)) / (2 * m)).sum()
    return dict(cot=torch.stack(out), loss=loss.view(1))


def exact(case, seed):
    c, kind, nu = case, case["kind"], case["nu"]
    if kind == "sort":
        return None
    if kind == "dssim":
        return _dssim(c, seed)
    if kind == "update":
        P = _params(c, seed)
        gr, hz, ge, de = (v.double() for v in _update_state(c, seed))
        x, g, d = _update(P, gr, hz, ge, de)
        return dict(x=x, g=g, d=d)
    if kind == "batch":
        if c["n"] * c["views"] > 1300000:
            return None
        out = dict(image=[], loss=[], grad=[], hz=[], x=[])
        for s in _batch_scenes(c, seed):
            P = s["x"][:, : s["c"]["n"]]
            p = _passes(s["c"], seed, P, s["cams"], s["tgt"].view(1, 3, c["h"], c["w"]), nu, 1)
            for q in ("image", "loss", "grad", "hz"):
                out[q].append(p[q][0] if q in ("image", "loss") else p[q])
            out["x"].append(_update(P, p["grad"], p["hz"], 0 * p["grad"], 0 * p["hz"])[0])
        return dict(out, image=torch.stack(out["image"]), loss=torch.stack(out["loss"]))
    P, cams = _params(c, seed), _cams(c, seed)
    if kind == "project":
        recs, tans = [], []
        zs = [_probes(c["n"], P.shape[0], 1, k) for k in range(nu)]
        for cam in cams:
            F, depth, _ = _fields(P.double(), cam, c["deg"])
            recs.append(torch.cat([F, depth[None]]).T)
            tans.append([torch.func.jvp(lambda p: _fields(p, cam, c["deg"])[0], (P.double(),), (z,))[1].T for z in zs])
        out = dict(rec=torch.stack(recs), radius=None, extents=None)
        if nu:
            out["tan"] = torch.stack([torch.stack(v, 1) for v in tans])
        return out
    if c["n"] * c["views"] > 400000:
        return None
    if kind == "autograd":
        cot = (_target(c, seed) - 0.5) / (3 * c["w"] * c["h"] * c["views"])
        p = _passes(c, seed, P, cams, None, 0, 1, cot)
        return dict(image=p["image"], grad=p["grad"])
    if kind in ("forward", "render"):
        p = _passes(c, seed, P, cams, None, nu, 1)
        return dict(image=p["image"], T=p["T"], n_contrib=None, **(dict(tan=p["tan"]) if nu else {}))
    p = _passes(c, seed, P, cams, _target(c, seed), nu, 1)
    out = dict(grad=p["grad"], loss=p["loss"], **(dict(hz=p["hz"]) if nu else {}))
    if kind == "reverse":
        return out
    x, g, d = _update(P, p["grad"], p["hz"], 0 * p["grad"], 0 * p["hz"])
    return dict(out, image=p["image"], x=x, g=g, d=d)
