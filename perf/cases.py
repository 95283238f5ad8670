"""The performance cases of this library: what a user has it do, through its public entry points.

A case is a plain dict; `kind` says which calls it makes.  The scenes, cell sizes and kernel scales are those of
paper_2603_29227_gb300/scenes.py (the room, the large scene, the 2D plane, the city block with its scanner), redrawn
here on the GPU from a seed so that making inputs takes no time to speak of.

  lookup   a fitted map answers a few points (sdf, grad): latency
  plan     one planner iteration: sdf and grad of the collision spheres of some trajectories, and the adjoint
  align    scan-to-map alignment: sdf, grad and var_sdf of points near the surface, adjoint of sdf and grad
  field    a fitted map answers many points with every real-valued output
  vargrad  the same with the SDF-gradient variance
  plane64  2D: fit, then the plain FP64 query of a grid
  mesh     fit of a large map, a dense grid of queries and the adjoint (the library's headline step)
  matern   the Matern 3/2 kernel: fit and query
  dense    densely scanned room: fit and query with cells of up to 512 samples
  stream   one frame of the city stream: the last scan's samples are replaced by a new scan's, then a query
  bhm      the occupancy front-end: one scan's update, then a prediction at many points
"""
import math

import numpy as np
import torch

from paper_2603_29227_gb300 import bhm, ksdf, scenes

OUT_REAL = ksdf.OUT_SDF | ksdf.OUT_GRAD | ksdf.OUT_VAR_SDF | ksdf.OUT_VAR_F


def listed():
    return [
        # a robot asks for the clearance of a few points of its body
        {"name": "lookup_37", "kind": "lookup", "samples": 200_000, "queries": 37},
        # one trajectory of 64 waypoints x 8 collision spheres, distance and its gradient for one optimiser step
        {"name": "plan_1", "kind": "plan", "samples": 200_000, "queries": 512},
        # 4,096 trajectories at once (batched trajectory optimisation)
        {"name": "plan_4096", "kind": "plan", "samples": 200_000, "queries": 2_097_152},
        # a LiDAR scan registered against the map
        {"name": "align_scan", "kind": "align", "samples": 200_000, "queries": 125_003},
        # a volume of points with every output, as for exploration or uncertainty-aware planning
        {"name": "field_1m", "kind": "field", "samples": 200_000, "queries": 1_000_000},
        # with the variance of the gradient
        {"name": "vargrad_262k", "kind": "vargrad", "samples": 200_000, "queries": 262_147},
        # a 2D occupancy-grid robot's map, all in FP64
        {"name": "plane2d_f64", "kind": "plane64", "samples": 2_000, "grid": 128},
        # a building-sized map built, meshed on a 256^3 grid and differentiated
        {"name": "mesh_256", "kind": "mesh", "samples": 2_000_000, "grid": 256},
        # the other kernel
        {"name": "matern_room", "kind": "matern", "samples": 200_000, "queries": 500_009},
        # a small room scanned densely: cells of several hundred samples
        {"name": "dense_room", "kind": "dense", "samples": 150_000, "queries": 300_007},
        # one frame of the streaming map
        {"name": "stream_frame", "kind": "stream", "frames": 3, "queries": 1_000_000},
        # one frame of the occupancy front-end
        {"name": "bhm_frame", "kind": "bhm", "frames": 2, "queries": 1_000_000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lookup", "plan", "align", "field", "vargrad", "plane64", "mesh", "matern", "dense", "stream",
                       "bhm"])
    s = _log(rng, 20_000, 400_000)
    if kind == "lookup":
        return {"kind": kind, "samples": s, "queries": _log(rng, 1, 400)}
    if kind == "plan":
        return {"kind": kind, "samples": s, "queries": 512 * _log(rng, 1, 4096)}
    if kind == "align":
        return {"kind": kind, "samples": s, "queries": _log(rng, 1_000, 131_072)}
    if kind in ("field", "matern"):
        return {"kind": kind, "samples": s, "queries": _log(rng, 1_000, 1_500_000)}
    if kind == "vargrad":
        return {"kind": kind, "samples": s, "queries": _log(rng, 1_000, 500_000)}
    if kind == "plane64":
        return {"kind": kind, "samples": _log(rng, 500, 8_000), "grid": _log(rng, 16, 160)}
    if kind == "mesh":
        return {"kind": kind, "samples": _log(rng, 100_000, 2_000_000), "grid": _log(rng, 40, 250)}
    if kind == "dense":
        return {"kind": kind, "samples": _log(rng, 60_000, 160_000), "queries": _log(rng, 10_000, 400_000)}
    return {"kind": kind, "frames": rng.randint(1, 4), "queries": _log(rng, 10_000, 1_000_000)}


# ---------------------------------------------------------------------------------------------------------
# inputs

_GPU = "cuda"


class _Scene:
    """Free box `hi` (lower corner 0) minus spheres and axis-aligned boxes, drawn on the GPU."""

    def __init__(self, gen, hi, n_prims):
        self.gen, self.dim = gen, len(hi)
        self.hi = torch.tensor(hi, dtype=torch.float64, device=_GPU)
        n_ball = n_prims if self.dim == 2 else n_prims // 2
        n_box = n_prims - n_ball
        if self.dim == 2:  # circles may cross the border
            self.r = 0.2 + 0.8 * self._u(n_ball)
            self.c = self._u(n_ball, self.dim) * self.hi
        else:
            self.r = 0.5 * (0.2 + 1.8 * self._u(n_ball))
            self.c = self.r[:, None] + self._u(n_ball, self.dim) * (self.hi - 2 * self.r[:, None])
        e = 0.2 + 1.8 * self._u(n_box, self.dim)
        self.lo_b = self._u(n_box, self.dim) * (self.hi - e)
        self.hi_b = self.lo_b + e
        self.host = [t.cpu().numpy() for t in (self.c, self.r, self.lo_b, self.hi_b)]

    def _u(self, *shape):
        return torch.rand(*shape, dtype=torch.float64, device=_GPU, generator=self.gen)

    def inside(self, x, tol):
        out = ((x < -tol) | (x > self.hi + tol)).any(1)
        c, r, lo, hi = self.host
        ax = [x[:, j].contiguous() for j in range(self.dim)]
        for i in range(len(r)):
            d = (ax[0] - float(c[i, 0])) ** 2
            for j in range(1, self.dim):
                d += (ax[j] - float(c[i, j])) ** 2
            out |= d < (float(r[i]) - tol) ** 2
        for i in range(len(lo)):
            m = (ax[0] > float(lo[i, 0]) + tol) & (ax[0] < float(hi[i, 0]) - tol)
            for j in range(1, self.dim):
                m &= (ax[j] > float(lo[i, j]) + tol) & (ax[j] < float(hi[i, j]) - tol)
            out |= m
        return out

    def surface(self, n, noise):
        """n noisy surface samples in random order: (x, var, normals)."""
        dim = self.dim
        area = lambda e: torch.stack([torch.prod(e[:, [k for k in range(dim) if k != j]], 1)  # noqa: E731
                                      for j in range(dim)], 1)
        blo = torch.cat([torch.zeros(1, dim, dtype=torch.float64, device=_GPU), self.lo_b])  # the room, the boxes
        bhi = torch.cat([self.hi[None], self.hi_b])
        w_box = area(bhi - blo).repeat_interleave(2, 1).reshape(-1)
        w_ball = 4 * math.pi * self.r ** 2 if dim == 3 else 2 * math.pi * self.r
        w = torch.cat([w_box, w_ball])
        cdf = torch.cumsum(w, 0)
        xs, ns, have = [], [], 0
        while have < n:
            m = int(1.4 * (n - have)) + 1024
            k = torch.searchsorted(cdf, self._u(m) * cdf[-1]).clamp(max=len(w) - 1)
            kb = k.clamp(max=len(w_box) - 1)
            box, ax, side = kb // (2 * dim), (kb // 2) % dim, kb % 2
            x = blo[box] + self._u(m, dim) * (bhi - blo)[box]
            face = torch.where(side == 0, blo[box, ax], bhi[box, ax])
            x.scatter_(1, ax[:, None], face[:, None])
            nrm = torch.zeros_like(x)
            out = torch.where(side == 0, -1.0, 1.0) * torch.where(box == 0, -1.0, 1.0)  # into free space
            nrm.scatter_(1, ax[:, None], out[:, None].to(nrm.dtype))
            ball = k >= len(w_box)
            v = torch.randn(m, dim, dtype=torch.float64, device=_GPU, generator=self.gen)
            v /= v.norm(dim=1, keepdim=True)
            b = (k - len(w_box)).clamp(min=0)
            x = torch.where(ball[:, None], self.c[b] + self.r[b, None] * v, x)
            nrm = torch.where(ball[:, None], v, nrm)
            keep = ~self.inside(x, 1e-9)
            xs.append(x[keep])
            ns.append(nrm[keep])
            have += int(keep.sum())
        x, nrm = torch.cat(xs)[:n], torch.cat(ns)[:n].float()
        x = x + noise * torch.randn(n, dim, dtype=torch.float64, device=_GPU, generator=self.gen)
        var = ((noise * (0.5 + 1.5 * self._u(n))) ** 2).float()
        return x.contiguous(), var, nrm.contiguous()

    def sign(self, xq):
        return torch.where(self.inside(xq.double(), 0.0), -1, 1).to(torch.int8)

    def grid(self, n):
        """Cell centres of an n^dim grid (x fastest) and their signs."""
        ax = [((torch.arange(n, dtype=torch.float64, device=_GPU) + 0.5) * (float(h) / n)) for h in self.hi]
        mesh = torch.meshgrid(*reversed(ax), indexing="ij")
        xq = torch.stack([m.reshape(-1) for m in reversed(mesh)], 1).float().contiguous()
        sg = torch.ones((n,) * self.dim, dtype=torch.int8, device=_GPU)
        c, r, lo, hi = self.host
        box = [(c[i] - r[i], c[i] + r[i], i) for i in range(len(r))] + [(lo[i], hi[i], -1) for i in range(len(lo))]
        side = self.hi.cpu().numpy()
        for a, b, ball in box:  # each primitive touches a slice of the grid
            i0 = [max(0, int(math.ceil(a[j] * n / side[j] - 0.5))) for j in range(self.dim)]
            i1 = [min(n, int(math.floor(b[j] * n / side[j] - 0.5)) + 1) for j in range(self.dim)]
            if any(p >= q for p, q in zip(i0, i1)):
                continue
            sl = tuple(slice(i0[j], i1[j]) for j in reversed(range(self.dim)))
            if ball < 0:
                sg[sl] = -1
                continue
            d = 0
            for j in range(self.dim):
                shape = [1] * self.dim
                shape[self.dim - 1 - j] = -1
                d = d + ((ax[j][i0[j]:i1[j]] - float(c[ball, j])) ** 2).reshape(shape)
            sg[sl] = torch.where(d < float(r[ball]) ** 2, -1, sg[sl])
        return xq, sg.reshape(-1).contiguous()


def _trajectories(gen, hi, n):
    """n points: cubic Bezier trajectories x 64 waypoints x the 8 corners of a 0.3 m cube."""
    nt = n // 512
    u = lambda *s: torch.rand(*s, dtype=torch.float64, device=_GPU, generator=gen)  # noqa: E731
    P = 0.3 + u(nt, 4, 3) * (hi - 0.6)
    t = (torch.arange(64, dtype=torch.float64, device=_GPU) + 0.5) / 64
    B = torch.stack([(1 - t) ** 3, 3 * (1 - t) ** 2 * t, 3 * (1 - t) * t ** 2, t ** 3], 1)
    way = torch.einsum("wk,tkj->twj", B, P).reshape(-1, 1, 3)
    off = torch.tensor([[x, y, z] for z in (-1, 1) for y in (-1, 1) for x in (-1, 1)], dtype=torch.float64,
                       device=_GPU) * 0.15
    return (way + off).reshape(-1, 3).float().contiguous()


def _scan(gen, city, f):
    """Hits of a 64 x 2048 scan of the city from pose f: (x, var, normals), 0.02 m range noise."""
    o = torch.tensor(city.poses[f % len(city.poses)], dtype=torch.float64, device=_GPU)
    el = torch.deg2rad(torch.linspace(-25.0, 15.0, city.n_beams, dtype=torch.float64, device=_GPU))
    az = (torch.arange(city.n_az, dtype=torch.float64, device=_GPU) +
          torch.rand(1, dtype=torch.float64, device=_GPU, generator=gen)) * (2 * math.pi / city.n_az)
    ce, se = torch.cos(el)[:, None], torch.sin(el)[:, None]
    d = torch.stack([(ce * torch.cos(az)).reshape(-1), (ce * torch.sin(az)).reshape(-1),
                     se.expand(-1, city.n_az).reshape(-1)], 1)
    inf = torch.full((len(d),), math.inf, dtype=torch.float64, device=_GPU)
    t = torch.where(d[:, 2] < 0, -o[2] / d[:, 2].clamp(max=-1e-12), inf)
    nrm = torch.zeros_like(d)
    nrm[:, 2] = 1.0
    inv = 1.0 / torch.where(d.abs() < 1e-12, torch.full_like(d, 1e-12), d)
    for lo, hi in zip(city.box_lo, city.box_hi):
        a = (torch.tensor(lo, dtype=torch.float64, device=_GPU) - o) * inv
        b = (torch.tensor(hi, dtype=torch.float64, device=_GPU) - o) * inv
        near3, far = torch.minimum(a, b), torch.maximum(a, b).amin(1)
        near, ax = near3.max(1)
        hit = (near <= far) & (near > 1e-6) & (near < t)
        nb = torch.zeros_like(d).scatter_(1, ax[:, None], -torch.sign(d.gather(1, ax[:, None])))
        t = torch.where(hit, near, t)
        nrm = torch.where(hit[:, None], nb, nrm)
    ok = t < city.max_range
    t = t[ok] + city.sigma * torch.randn(int(ok.sum()), dtype=torch.float64, device=_GPU, generator=gen)
    x = (o + t[:, None] * d[ok]).contiguous()
    return x, torch.full((len(x),), city.sigma ** 2, dtype=torch.float32, device=_GPU), nrm[ok].float().contiguous()


def _params(kind):
    if kind == "plane64":
        return dict(dim=2, origin=(0.0, 0.0, 0.0), cell=1.0, margin=0.1, n_max=64, k_cand=4, **{"lambda": 500.0},
                    softmin_alpha=500.0, sign_mode=0)
    p = dict(dim=3, origin=(0.0, 0.0, 0.0), cell=0.5, margin=0.1, n_max=256, k_cand=8, **{"lambda": 300.0},
             softmin_alpha=300.0, sign_mode=1 if kind == "stream" else 0)
    if kind in ("mesh", "dense"):
        p["n_max"] = 512
    if kind == "matern":
        p["kernel"] = "matern32"
        p["lambda"] = 100.0  # scale sqrt(3) / lambda = 0.017 m
        p["softmin_alpha"] = 100.0
    return p


def _inputs(case, seed):
    """The tensors of a case, from the seed alone."""
    kind = case["kind"]
    gen = torch.Generator(device=_GPU).manual_seed(int(seed) * 7919 + 13)
    rand = lambda *s: torch.randn(*s, device=_GPU, generator=gen)  # noqa: E731
    i = {"params": _params(kind)}
    if kind in ("stream", "bhm"):
        city = scenes.make_city()
        f0 = 7 * (int(seed) % 97)
        i["scans"] = [_scan(gen, city, f0 + k) for k in range(case["frames"] + 1)]
        i["poses"] = [city.poses[(f0 + k) % len(city.poses)] for k in range(case["frames"] + 1)]
        o = torch.tensor(i["poses"][-1], device=_GPU)
        u = torch.rand(case["queries"], 3, dtype=torch.float64, device=_GPU, generator=gen)
        lo = torch.stack([o[0] - 20.0, o[1] - 20.0, torch.zeros_like(o[0])])
        i["xq"] = (lo + u * torch.tensor([40.0, 40.0, 6.0], dtype=torch.float64, device=_GPU)).float().contiguous()
        return i
    if kind == "plane64":
        sc = _Scene(gen, (10.0, 10.0), 20)
    elif kind == "mesh":
        sc = _Scene(gen, (50.0, 50.0, 10.0), 1000)
    elif kind == "dense":
        sc = _Scene(gen, (5.0, 5.0, 2.5), 6)
    else:
        sc = _Scene(gen, (20.0, 20.0, 5.0), 50)
    i["x"], i["var"], i["nrm"] = sc.surface(case["samples"], 0.01)
    if "grid" in case:
        i["xq"], i["sign"] = sc.grid(case["grid"])
        if kind == "plane64":
            i["xq"] = i["xq"].double()
    else:
        n = case["queries"]
        if kind == "plan":
            xq = _trajectories(gen, sc.hi, n)
        elif kind == "align":  # scan points: the surface again, with the registration's and the scanner's error
            x2, _, _ = sc.surface(n, 0.02)
            xq = x2.float().contiguous()
        else:
            u = torch.rand(n, 3, dtype=torch.float64, device=_GPU, generator=gen)
            xq = (u * sc.hi).float().contiguous()
        i["xq"], i["sign"] = xq, sc.sign(xq)
    n = len(i["xq"])
    if kind in ("plan", "align", "mesh"):
        i["d_sdf"] = rand(n)
    if kind == "align":
        i["d_grad"] = rand(n, 3)
    return i


# ---------------------------------------------------------------------------------------------------------
# the calls

_MASK = {"lookup": ksdf.OUT_SDF | ksdf.OUT_GRAD, "plan": ksdf.OUT_SDF | ksdf.OUT_GRAD | ksdf.OUT_WINNER,
         "align": ksdf.OUT_SDF | ksdf.OUT_GRAD | ksdf.OUT_VAR_SDF | ksdf.OUT_WINNER, "field": OUT_REAL,
         "vargrad": OUT_REAL | ksdf.OUT_VAR_GRAD, "plane64": OUT_REAL, "mesh": OUT_REAL | ksdf.OUT_WINNER,
         "matern": OUT_REAL, "dense": OUT_REAL, "stream": ksdf.OUT_SDF | ksdf.OUT_GRAD | ksdf.OUT_VAR_SDF}
_FITS = ("plane64", "mesh", "matern", "dense")  # the fit is part of the pass
_BHM_MASK = bhm.BHM_LOGODDS | bhm.BHM_GRAD | bhm.BHM_PROB


def prepare(case, seed):
    s = _inputs(case, seed)
    s["kind"] = kind = case["kind"]
    if kind == "bhm":  # a map that has seen some frames
        s["map"] = bhm.BHMap(scenes.CITY_BHM, max_blocks=1 << 16)
        for (x, _, _), p in zip(s["scans"][:-1], s["poses"][:-1]):
            s["map"].update(p, x)
        return s
    s["model"] = ksdf.KernelSDF(s["params"])
    if kind == "stream":  # a map of some frames; the newest one's samples are replaced on each pass
        old, (x, v, nr) = s["scans"][:-1], s["scans"][-1]
        s["model"].fit(*[torch.cat([o[k] for o in old] + [(x, v, nr)[k]]) for k in range(3)])
        s["drop"] = torch.zeros(s["model"].S, dtype=torch.uint8, device=_GPU)
        s["drop"][-len(x):] = 1
    elif kind in _FITS:
        s["model"].reserve(len(s["x"]), len(s["xq"]))
    else:
        s["model"].fit(s["x"], s["var"], s["nrm"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "bhm":
        s["map"].update(s["poses"][-1], s["scans"][-1][0])
        o = s["map"].query(s["xq"], _BHM_MASK)
        return {k: o[k] for k in ("logodds", "grad", "prob")}
    m = s["model"]
    if kind == "stream":
        m.update_replace(s["drop"], *s["scans"][-1])
    elif kind in _FITS:
        m.fit(s["x"], s["var"], s["nrm"])
    o = m.query(s["xq"], s.get("sign"), _MASK[kind], f64=kind == "plane64")
    out = {k: v for k, v in o.items() if v is not None and k != "winner"}
    if "d_sdf" in s:
        out["d_xq"], out["d_x"] = m.backward(s["xq"], o["winner"], s["d_sdf"], s.get("d_grad"), s["sign"])
    return out


# mean training-set size, and the nearest cells' samples a query meets, per 1,000 samples of the scene (measured)
_MEAN_N = {"plane64": 0.0135, "mesh": 4.0e-5, "dense": 1.4e-3}


def work(case):
    """Bytes: every input and output once, and the model's records; flops: per query 9 per candidate sample (the
    posterior means) and 18 per winner sample (gradient, variances), N^2 for V[f] where it is asked for; N^3 / 3 per
    fitted cell; the adjoint 25 per winner sample and 4 N^2 per cell."""
    kind = case["kind"]
    if kind == "bhm":
        hits, q = 125_000, case["queries"]
        samples = 24 * hits  # free samples along the rays
        return {"bytes": 24 * hits + q * (12 + 4 + 12 + 4), "flops": 2 * samples * 53 * 8 + q * 53 * 14}
    dim = 2 if kind == "plane64" else 3
    q = case["grid"] ** dim if "grid" in case else case["queries"]
    s = 125_000 * (case["frames"] + 1) if kind == "stream" else case["samples"]
    word = 8 if kind == "plane64" else 4
    n = min(_params(kind)["n_max"], max(4.0, s * _MEAN_N.get(kind, 3.4e-4)))
    if kind == "stream":
        n = 40.0
    cells = s * (1.2 if dim == 2 else 1.96) / n
    k = _params(kind)["k_cand"]
    mask = _MASK[kind]
    width = sum(w for b, w in ((ksdf.OUT_SDF, 1), (ksdf.OUT_GRAD, dim), (ksdf.OUT_VAR_SDF, 1), (ksdf.OUT_VAR_F, 1),
                               (ksdf.OUT_VAR_GRAD, dim)) if mask & b)
    touched = min(cells, q / 4.0)
    nbytes = q * (word * (dim + width) + 1) + touched * n * 20
    flops = q * n * (9 * k + 18) + (q * n * n if mask & ksdf.OUT_VAR_F else 0) + (40 * q * n if kind == "vargrad" else 0)
    if kind in _FITS or kind == "stream":
        fitted = cells if kind in _FITS else 125_000 * 1.96 / n
        nbytes += s * (8 * dim + 4 + 4 * dim) + cells * n * 36 + fitted * (8 + 4) * n * n / 2
        flops += fitted * n ** 3 / 3
    if kind in ("plan", "align", "mesh"):
        nbytes += q * 4 * (dim + 1 + (dim if kind == "align" else 0)) + s * 4 * dim
        flops += 25 * q * n + touched * (4 * n * n + 10 * n * n)
    return {"bytes": float(nbytes), "flops": float(flops)}


# ---------------------------------------------------------------------------------------------------------
# the same results in 64 bits, in plain torch

def _cells(x, p):
    """Cell coordinates (G x dim, ascending (z, y, x)) and padded training sets (G x N ids, -1 padded)."""
    dim, h, mu = p["dim"], p["cell"], p["margin"]
    off = 1 << 20
    key = lambda c: sum((c[..., j] + off) << (21 * j) for j in range(dim))  # noqa: E731
    c = torch.floor(x / h).long()
    keys = torch.unique(key(c))
    cc = torch.stack([((keys >> (21 * j)) & 0x1FFFFF) - off for j in range(dim)], 1)
    pairs = []
    ids = torch.arange(len(x), device=x.device)
    for o in np.ndindex(*(3,) * dim):
        n = c + torch.tensor(o, device=x.device) - 1
        inside = ((x >= n.double() * h - mu) & (x < (n.double() + 1) * h + mu)).all(1)
        k = key(n)
        g = torch.searchsorted(keys, k).clamp(max=len(keys) - 1)
        ok = inside & (keys[g] == k)
        pairs.append(g[ok] * (1 << 32) + ids[ok])
    pairs = torch.sort(torch.cat(pairs))[0]
    g, i = pairs >> 32, pairs & 0xFFFFFFFF
    cnt = torch.bincount(g, minlength=len(keys))
    start = torch.cumsum(cnt, 0) - cnt
    keep = cnt.clamp(max=p["n_max"])
    j = torch.arange(int(keep.max()), device=x.device)[None]
    rank = torch.where((cnt > p["n_max"])[:, None], j * cnt[:, None] // p["n_max"], j)
    src = (start[:, None] + rank).clamp(max=len(i) - 1)
    return keys, cc, torch.where(j < keep[:, None], i[src], torch.full_like(src, -1))


def _kernel(r2, p):
    if p.get("kernel") == "matern32":
        z = p["lambda"] * torch.sqrt(r2.clamp(min=1e-300))
        return (1 + z) * torch.exp(-z)
    return torch.exp(-p["lambda"] * r2)


def _chol(pos, var, live, p):
    """Cholesky factors of the padded cells (identity on the padding) in 64 bits."""
    d = pos[:, :, None, :] - pos[:, None, :, :]
    both = live[:, :, None] & live[:, None, :]
    A = torch.where(both, _kernel((d * d).sum(-1), p), torch.zeros((), dtype=torch.float64, device=pos.device))
    return torch.linalg.cholesky(A * (1 - torch.eye(A.shape[1], dtype=A.dtype, device=A.device)) +
                                 torch.diag_embed(torch.where(live, 1 + var, torch.ones_like(var))))


def _mean(xq, pos, al, live, p):
    """f' (scaled by the nearest sample's factor), offsets, kernel values, gradient weights, nearest distance, r."""
    lam = p["lambda"]
    r = xq[:, None, :] - pos
    inf = torch.full((), math.inf, dtype=torch.float64, device=xq.device)
    r2 = (r * r).sum(-1)
    m = torch.where(live, r2, inf).amin(1).detach()
    if p.get("kernel") == "matern32":
        z = torch.sqrt(r2.clamp(min=1e-300))
        w = torch.exp(-lam * (z - torch.sqrt(m)[:, None]))
        k = (1 + lam * z) * w
    else:
        w = k = torch.exp(-lam * (r2 - m[:, None]))
    zero = torch.zeros((), dtype=torch.float64, device=xq.device)
    k, w = torch.where(live, k, zero), torch.where(live, w, zero)
    f = (al * k).sum(1)
    d = torch.sqrt(m)
    safe = torch.where(f > 0, f, torch.ones_like(f))
    if p.get("kernel") == "matern32":
        u = (-torch.log(safe) / lam + d).clamp(min=0)
    else:
        u2 = -torch.log(safe) / lam + m
        u = torch.where(u2 > 0, torch.sqrt(torch.where(u2 > 0, u2, torch.ones_like(u2))), torch.zeros_like(u2))
    fall = torch.sqrt(r2.clamp(min=1e-300))
    near = torch.where(live, r2, inf).argmin(1)
    u = torch.where(f > 0, u, fall.gather(1, near[:, None])[:, 0])
    return u, r, k, w, m, r2


def exact(case, seed):
    kind = case["kind"]
    if kind in ("mesh", "stream", "bhm"):
        return None  # too long in 64 bits (mesh); state carried from pass to pass (stream, bhm)
    i = _inputs(case, seed)
    p, x, xq = i["params"], i["x"], i["xq"].double()
    dim, K, lam, al_s = p["dim"], p["k_cand"], p["lambda"], p["softmin_alpha"]
    keys, cc, mem = _cells(x, p)
    G, N = mem.shape
    live = mem >= 0
    pos = x[mem.clamp(min=0)]
    var = i["var"].double()[mem.clamp(min=0)] * live
    one = torch.where(live, 1.0, 0.0).double()
    L = torch.empty(G, N, N, dtype=torch.float64, device=x.device)
    alpha = torch.empty(G, N, dtype=torch.float64, device=x.device)
    step = max(1, int(2e8 // (N * N)))
    for a in range(0, G, step):
        sl = slice(a, a + step)
        L[sl] = _chol(pos[sl], var[sl], live[sl], p)
        alpha[sl] = torch.cholesky_solve(one[sl, :, None], L[sl])[:, :, 0]
    # candidates per query bin, min-fusion
    c = torch.floor(xq / p["cell"]).long()
    bins, back = torch.unique(c, dim=0, return_inverse=True)
    cand = torch.empty(len(bins), min(K, G), dtype=torch.long, device=x.device)
    for a in range(0, len(bins), 2048):
        D = ((bins[a:a + 2048, None, :] - cc[None]) ** 2).sum(-1) * G + torch.arange(G, device=x.device)[None]
        cand[a:a + 2048] = torch.topk(D, cand.shape[1], dim=1, largest=False)[1]
    Q = len(xq)
    u = torch.full((Q,), math.inf, dtype=torch.float64, device=x.device)
    win = torch.zeros(Q, dtype=torch.long, device=x.device)
    step = max(1, int(4e7 // N))
    for a in range(0, Q, step):
        sl = slice(a, a + step)
        for k in range(cand.shape[1]):
            g = cand[back[sl], k]
            v = _mean(xq[sl], pos[g], alpha[g], live[g], p)[0]
            better = v < u[sl]
            u[sl] = torch.where(better, v, u[sl])
            win[sl] = torch.where(better, g, win[sl])
    # the winner's outputs
    sg = i["sign"].double()
    o = {"sdf": sg * u}
    names = {"grad": ksdf.OUT_GRAD, "var_sdf": ksdf.OUT_VAR_SDF, "var_f": ksdf.OUT_VAR_F, "var_grad": ksdf.OUT_VAR_GRAD}
    for k, bit in names.items():
        if _MASK[kind] & bit:
            o[k] = torch.zeros(Q, dim, dtype=torch.float64, device=x.device) if "grad" in k else torch.zeros_like(u)
    order = torch.argsort(win)
    step = max(1, int(2e7 // N))
    for a in range(0, Q, step):
        q = order[a:a + step]
        g = win[q]
        _, r, k, w, m, r2 = _mean(xq[q], pos[g], alpha[g], live[g], p)
        Gv = ((alpha[g] * w)[..., None] * r).sum(1)
        gn = Gv.norm(dim=1, keepdim=True)
        o["grad"][q] = torch.where(gn > 0, sg[q, None] * Gv / gn, torch.zeros_like(Gv))
        z = torch.sqrt(r2)
        e = torch.where(live[g], torch.exp(-al_s * (z - torch.sqrt(m)[:, None])), torch.zeros_like(z))
        s = e / e.sum(1, keepdim=True)
        h = (s * torch.where(live[g], z, torch.zeros_like(z))).sum(1, keepdim=True)
        t = al_s * (h - z) + 1
        if "var_sdf" in o:
            o["var_sdf"][q] = (s * s * t * t * var[g]).sum(1)
        if "var_f" in o:
            gs, cnt = torch.unique_consecutive(g, return_counts=True)
            b, sc = 0, torch.exp(-2 * lam * (torch.sqrt(m) if p.get("kernel") == "matern32" else m))
            for gi, n in zip(gs.tolist(), cnt.tolist()):
                y = torch.linalg.solve_triangular(L[gi], k[b:b + n].T, upper=False)
                o["var_f"][q[b:b + n]] = (1 - sc[b:b + n] * (y * y).sum(0)).clamp(min=0)
                b += n
        if "var_grad" in o:
            v = torch.where(live[g][..., None], r / z.clamp(min=1e-300)[..., None], torch.zeros_like(r))
            li = s * t
            Vs, gg = (s[..., None] * v).sum(1, keepdim=True), (li[..., None] * v).sum(1, keepdim=True)
            wk = li[..., None] * (v - Vs) + s[..., None] * (v - gg)
            ci = torch.where(live[g], li / z.clamp(min=1e-300), torch.zeros_like(li))[..., None]
            o["var_grad"][q] = (var[g][..., None] * (al_s ** 2 * wk * wk + ci * ci * (1 - v * v))).sum(1)
    if "d_sdf" not in i:
        return o
    # the adjoint: autograd over the winners, the sample gradient in two stages (queries, then the fit)
    touched, tq = torch.unique(win, return_inverse=True)
    apos, aal = pos[touched].clone().requires_grad_(True), alpha[touched].clone().requires_grad_(True)
    o["d_xq"] = torch.zeros(Q, dim, dtype=torch.float64, device=x.device)
    for a in range(0, Q, step):
        q = order[a:a + step]
        t = tq[q]
        xl = xq[q].clone().requires_grad_(True)
        uq, r, k, w, m, _ = _mean(xl, apos[t], aal[t], live[touched][t], p)
        loss = (uq * sg[q] * i["d_sdf"][q].double()).sum()
        if "d_grad" in i:
            Gv = ((aal[t] * w)[..., None] * r).sum(1)
            loss = loss + (sg[q, None] * Gv / Gv.norm(dim=1, keepdim=True) * i["d_grad"][q].double()).sum()
        loss.backward()
        o["d_xq"][q] = xl.grad
    d_x = torch.zeros_like(x)
    step = max(1, int(4e7 // (N * N)))
    for a in range(0, len(touched), step):
        sl = slice(a, a + step)
        t = touched[sl]
        pl = pos[t].clone().requires_grad_(True)
        al = torch.cholesky_solve(one[t, :, None], _chol(pl, var[t], live[t], p))[:, :, 0]
        al.backward(aal.grad[sl])
        d = (pl.grad + apos.grad[sl])[live[t]]
        d_x.index_add_(0, mem[t][live[t]], d)
    o["d_x"] = d_x
    return o
