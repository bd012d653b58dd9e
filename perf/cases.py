"""Workloads of the registration library, through its public entry points.

A case names an entry point, an image size and spacing, a node grid, the image type and the terms of the objective
(weights as in the benchmark: eta = 10, alpha = 1, gamma = 0.001 where the volume term is on).  Inputs are seeded
lung-like pairs after ``phantom.py``'s recipe (body and lung ellipsoids, vessels, density change, 15 HU noise, sums
of Gaussian motions), made with torch on the device; vessels are straight tubes.  ``exact`` evaluates the same
quantities in FP64 with plain torch; the sample cell of a voxel is decided in FP32, as include/ngfreg.h defines it.
"""
import math

import torch
import torch.nn.functional as F

from paper_1807_00467_gb300 import api, autograd, batch, discrete

FOV = (358.4, 358.4, 320.0)     # mm, a thorax scan (the batching workload's field of view)
ETA, ALPHA = 10.0, 1.0
LABELS = 35937
KP_MAX = 20000         # keypoints a detector call has room for


def _case(name, kind, n, h, rho, half=False, gamma=0.001, nk=0, delta=0.0, iters=0, pairs=1):
    return {"name": name, "kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "hx": h[0], "hy": h[1], "hz": h[2],
            "rx": rho[0], "ry": rho[1], "rz": rho[2], "half": half, "gamma": gamma, "nk": nk, "delta": delta,
            "iters": iters, "pairs": pairs}


def listed():
    full, mid, tiny = (512, 512, 128), (256, 256, 64), (64, 64, 48)
    hf, hm, ht = (0.7, 0.7, 2.5), (1.4, 1.4, 5.0), (1.0, 1.0, 2.5)
    iso = (1.0, 1.0, 1.0)
    return [
        # one objective + gradient evaluation of the smallest configured problem: launches and latency
        _case("gradient_tiny", "gradient", tiny, ht, (4, 4, 4), gamma=0.0),
        # one Gauss-Newton iteration of the same problem, as its solve runs five of
        _case("step_tiny", "step", tiny, ht, (4, 4, 4), gamma=0.0, iters=30),
        # an odd-sized, ragged half-resolution crop with FP16 images: a Hessian-vector product at a new iterate
        _case("hvp_odd_f16", "hvp", (182, 150, 94), (1.9, 1.9, 3.3), (2, 2, 2), half=True),
        # the differentiation workload: forward and backward through autograd with 3000 vessel keypoints
        _case("autograd_mid_kp", "autograd", mid, hm, (4, 4, 2), nk=3000, delta=10.0),
        # the linear solve of one Gauss-Newton step at the middle pyramid level
        _case("pcg_mid", "pcg", mid, hm, (4, 4, 2), iters=30),
        # a batch of uneven FP16 pairs advanced by one Gauss-Newton iteration each through one graph
        _case("batch_f16", "batch", (512, 512, 128), (0.7, 0.7, 2.5), (4, 4, 4), half=True, iters=30, pairs=8),
        # full resolution: the line search's objective with FP16 images ...
        _case("objective_full_f16", "objective", full, hf, (4, 4, 2), half=True),
        # ... the gradient with the stored linearisation, FP32 images ...
        _case("linearize_full", "linearize", full, hf, (4, 4, 2)),
        # ... one product with the stored Gauss-Newton matrix (30 of these per step) ...
        _case("matvec_full", "matvec", full, hf, (4, 4, 2)),
        # ... and a whole Gauss-Newton iteration, the benchmark's step
        _case("step_full", "step", full, hf, (4, 4, 2), iters=30),
        # the discrete stage at 1 mm: symmetric match of 3000 vessel keypoints
        _case("match_3000", "match", (224, 192, 192), iso, (4, 4, 4), nk=3000),
        # its keypoint detector on the same volume
        _case("forstner", "forstner", (224, 192, 192), iso, (4, 4, 4)),
    ]


def draw(rng):
    top = {k: max(work(c)[k] for c in listed()) for k in ("bytes", "flops")}
    while True:
        c = _draw(rng)
        w = work(c)
        if w["bytes"] <= top["bytes"] and w["flops"] <= top["flops"]:
            return c


def _draw(rng):
    kind = rng.choice(["gradient", "objective", "linearize", "hvp", "matvec", "matvec", "autograd", "pcg", "pcg", "step",
                       "batch", "match", "forstner"])
    if kind in ("match", "forstner"):
        n = tuple(rng.randrange(72, 225) for _ in range(3))
        nk = int(math.exp(rng.uniform(math.log(40), math.log(3000)))) if kind == "match" else 0
        return _drawn(kind, n, (1.0, 1.0, 1.0), (4, 4, 4), nk=nk)
    # voxels log-uniform between the smallest and the largest configured volume, z extent with the cube root
    v0, v1 = 64 * 64 * 48, 512 * 512 * 128
    v = math.exp(rng.uniform(math.log(v0), math.log(v1)))
    rho = tuple(rng.choice([1, 2, 2, 4, 4, 4, 8]) if a == 2 else rng.choice([2, 4, 4, 4, 8]) for a in range(3))
    nz = min(128.0, 48.0 * (v / v0) ** (1.0 / 3.0) * rng.uniform(0.7, 1.3))
    aspect = rng.uniform(0.8, 1.25)
    nx = min(512.0, math.sqrt(v / nz) * aspect)
    ny = min(512.0, math.sqrt(v / nz) / aspect)
    n = tuple(max(rho[a], int(x) // rho[a] * rho[a]) for a, x in enumerate((nx, ny, nz)))
    if kind == "batch":     # (pyramid-sized grids of one node per four voxels; the batch's largest pair)
        n, rho = tuple(max(64, int(x) // 16 * 16) for x in (nx, ny, nz)), (4, 4, 4)
    h = tuple(round(FOV[a] / n[a], 3) for a in range(3))
    nk = rng.randrange(100, 3001) if kind != "batch" and rng.random() < 0.3 else 0
    return _drawn(kind, n, h, rho, half=kind == "batch" or rng.random() < 0.4, gamma=rng.choice([0.0, 0.001]), nk=nk,
                  delta=10.0 if nk else 0.0, iters=rng.randrange(5, 31), pairs=rng.randrange(2, 9) if kind == "batch" else 1)


def _drawn(*args, **kw):
    c = _case("", *args, **kw)
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs

def _dims(c):
    n = (c["nx"], c["ny"], c["nz"])
    m = tuple(n[a] // (c["rx"], c["ry"], c["rz"])[a] + 1 for a in range(3))
    return n, (c["hx"], c["hy"], c["hz"]), m


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _axes(n, h, dev="cuda"):
    ax = [(torch.arange(n[a], device=dev, dtype=torch.float32) + 0.5) * h[a] for a in range(3)]
    return ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]


def _ellipsoid(p, centre, semi):
    return sum(((p[a] - centre[a]) / semi[a]) ** 2 for a in range(3)) <= 1.0


def _density(p, fov, vessels, parenchyma):
    """Density at the points p (x, y, z tensors), the recipe's values in HU; vessels: (ends, radius) per tube."""
    c0 = [f / 2 for f in fov]
    dens = torch.where(_ellipsoid(p, c0, [0.46 * fov[0], 0.40 * fov[1], 0.48 * fov[2]]), 40.0, -1000.0)
    semi = [0.17 * fov[0], 0.26 * fov[1], 0.42 * fov[2]]
    lung = (_ellipsoid(p, [c0[0] - 0.2 * fov[0], c0[1], c0[2]], semi)
            | _ellipsoid(p, [c0[0] + 0.2 * fov[0], c0[1], c0[2]], semi))
    prof = torch.zeros_like(dens)
    for a, b, r in vessels:
        d = [b[k] - a[k] for k in range(3)]
        t = (sum((p[k] - a[k]) * d[k] for k in range(3)) / sum(x * x for x in d)).clamp(0.0, 1.0)
        d2 = sum((p[k] - a[k] - t * d[k]) ** 2 for k in range(3))
        prof = torch.maximum(prof, torch.exp(d2 / (-2.0 * r * r)))
    return torch.where(lung, parenchyma + (40.0 - parenchyma) * prof, dens)


def _motion(p, amps, centres):
    u = [0.0, 0.0, 0.0]
    for A, c in zip(amps, centres):
        e = torch.exp(sum((p[k] - c[k]) ** 2 for k in range(3)) / (-2.0 * 15.0 ** 2))
        u = [u[k] + A[k] * e for k in range(3)]
    return torch.stack(u)


def _min_max_det(u, g):
    d = [torch.stack([torch.diff(u[k], dim=2 - a)[:-1 if a != 2 else None, :-1 if a != 1 else None,
                                                  :-1 if a != 0 else None] / g[a] + (1.0 if a == k else 0.0)
                      for k in range(3)]) for a in range(3)]
    det = (d[0] * torch.linalg.cross(d[1], d[2], dim=0)).sum(0)
    return float(det.min()), float(det.max())


def _pair(n, h, m, seed, large):
    """R, T (HU, float32), the motion on the m-node grid, and the vessels."""
    g = _gen(seed)
    fov = [n[a] * h[a] for a in range(3)]
    r = torch.rand(400, generator=g, device="cuda").tolist()
    vessels = []
    for v in range(30):
        q = r[v * 8:v * 8 + 8]
        cx = fov[0] * (0.3 if v % 2 else 0.7)
        ends = [[cx + (q[3 * e] - 0.5) * 0.18 * fov[0], fov[1] * (0.5 + (q[3 * e + 1] - 0.5) * 0.28),
                 fov[2] * (0.5 + (q[3 * e + 2] - 0.5) * 0.45)] for e in range(2)]
        vessels.append((ends[0], ends[1], (1.0 + 2.0 * q[6]) * h[0]))
    amps, centres = [], []
    for j in range(8):
        q = r[240 + j * 8:248 + j * 8]
        centres.append([fov[0] * (0.13 + 0.74 * q[0]), fov[1] * (0.24 + 0.52 * q[1]), fov[2] * (0.08 + 0.84 * q[2])])
        a = 5.0 + 15.0 * q[3]
        amps.append([a * (0.5 * q[4] - 0.25), a * (0.5 * q[5] - 0.25), a] if large
                    else [(2.0 * q[4 + k] - 1.0) * 3.4 for k in range(3)])
    nodes = [torch.linspace(0.0, fov[a], m[a], device="cuda") for a in range(3)]
    p = nodes[0][None, None, :], nodes[1][None, :, None], nodes[2][:, None, None]
    while True:
        u = _motion(p, amps, centres)
        lo, hi = _min_max_det(u, [fov[a] / (m[a] - 1) for a in range(3)])
        if lo >= 0.3 and hi <= 3.5:
            break
        amps = [[0.8 * x for x in A] for A in amps]
    q = [p[k] for k in range(3)]        # pre-images of the nodes under x + u(x)
    for _ in range(12):
        w = _motion(q, amps, centres)
        q = [p[k] - w[k] for k in range(3)]
    w = F.interpolate(w[None], size=(n[2], n[1], n[0]), mode="trilinear")[0]
    x = _axes(n, h)
    R = _density(x, fov, vessels, -850.0)
    T = _density([x[k] - w[k] for k in range(3)], fov, vessels, -765.0)
    del w
    R += 15.0 * torch.randn(R.shape, generator=g, device="cuda")
    T += 15.0 * torch.randn(T.shape, generator=g, device="cuda")
    return R, T, u.contiguous(), vessels, (amps, centres)


def _stored(x, half):
    """As the library stores it: float32 HU, or half of HU + 1024."""
    return (x + 1024.0).half() if half else x


def _vessel_points(vessels, nk, g):
    t = torch.rand(nk, generator=g, device="cuda")
    which = torch.randint(0, len(vessels), (nk,), generator=g, device="cuda")
    a = torch.tensor([v[0] for v in vessels], device="cuda")[which]
    b = torch.tensor([v[1] for v in vessels], device="cuda")[which]
    return a + t[:, None] * (b - a)


def _vessel_voxels(vessels, nk, n, g):
    """nk distinct voxels (x, y, z) within two voxels of a centre line, at 1 mm."""
    p = _vessel_points(vessels, 20 * nk, g).int() + torch.randint(-2, 3, (20 * nk, 3), generator=g, device="cuda").int()
    p = torch.unique(p.clamp(min=torch.zeros(3, device="cuda").int(), max=torch.tensor(n, device="cuda").int() - 1), dim=0)
    return p[torch.randperm(p.shape[0], generator=g, device="cuda")[:nk]].contiguous()


def _batch_geometry(c):
    """Sizes of a batch's pairs, log-spaced from 96 x 96 x 64 to the case's own."""
    lo, out = (min(96, c["nx"]), min(96, c["ny"]), min(64, c["nz"])), []
    for i in range(c["pairs"]):
        s = i / max(1, c["pairs"] - 1)
        n = tuple(max(16, int(round(lo[a] * (hi / lo[a]) ** s / 16)) * 16) for a, hi in enumerate((c["nx"], c["ny"], c["nz"])))
        out.append((n, tuple(FOV[a] / n[a] for a in range(3)), tuple(k // 4 + 1 for k in n)))
    return out


def _problem(c, seed):
    n, h, m = _dims(c)
    R, T, u, vessels, mot = _pair(n, h, m, seed, large=min(n[a] * h[a] for a in range(3)) > 150.0)
    kx = ky = None
    g = _gen(seed + 7919)
    if c["nk"]:
        kx = _vessel_points(vessels, c["nk"], g)
        ky = (kx + _motion(kx.unbind(1), *mot).T + torch.randn(kx.shape, generator=g, device="cuda")).contiguous()
    v = torch.randn(u.shape, generator=g, device="cuda")
    return R, T, 0.5 * u, v, kx, ky


def _params(c):
    return api.make_params(eta=ETA, alpha=ALPHA, gamma=c["gamma"], delta=c["delta"])


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c, "kind": kind}
    if kind == "batch":
        s["pairs"] = []
        for i, (n, h, m) in enumerate(_batch_geometry(c)):
            R, T = _pair(n, h, m, seed + 31 * i, large=True)[:2]
            s["pairs"].append((_stored(R, True), _stored(T, True), h, m))
        return s
    n, h, m = _dims(c)
    if kind in ("match", "forstner"):
        R, T, u, vessels, _ = _pair(n, h, m, seed, large=True)
        if kind == "match":
            kps = _vessel_voxels(vessels, c["nk"], n, _gen(seed + 7919))
            s.update(F=R, M=T, kps=kps, matcher=discrete.Matcher(tuple(R.shape), kps.shape[0], alpha=0.2))
        else:
            fov = [n[a] * h[a] for a in range(3)]
            semi = [0.17 * fov[0], 0.26 * fov[1], 0.42 * fov[2]]
            lung = (_ellipsoid(_axes(n, h), [0.3 * fov[0], 0.5 * fov[1], 0.5 * fov[2]], semi)
                    | _ellipsoid(_axes(n, h), [0.7 * fov[0], 0.5 * fov[1], 0.5 * fov[2]], semi))
            s.update(F=R, mask=lung.to(torch.uint8))
        return s
    R, T, u, v, kx, ky = _problem(c, seed)
    ctx = api.Context(_stored(R, c["half"]), _stored(T, c["half"]), h, m, _params(c), nk_max=c["nk"], pcg_max=max(1, c["iters"]))
    if kx is not None:
        ctx.set_keypoints(kx, ky)
    s.update(ctx=ctx, u=u, v=v)
    if kind in ("matvec", "pcg"):       # products and solves at a linearisation that the caller has made
        s["g"] = ctx.gn_linearize(u)[1]
    return s


def run(state):
    kind = state["kind"]
    if kind == "batch":
        us, _, _, code = batch.register_batch_graph(state["pairs"], _params(state["case"]), levels=1, gn_iters=1,
                                                    pcg_iters=state["case"]["iters"])
        return {"u": us, "code": code}
    if kind == "match":
        disp, E = state["matcher"].match(state["F"], state["M"], state["kps"], symmetric=True, marginals=True)
        nk = state["kps"].shape[0]
        return {"disp": disp, "forward": E[:nk], "backward": E[nk:]}
    if kind == "forstner":
        kps, resp = discrete.forstner(state["F"], state["mask"], max_kp=KP_MAX, response=True)
        return {"count": kps.shape[0], "kps": F.pad(kps, (0, 0, 0, KP_MAX - kps.shape[0])), "response": resp}
    ctx, u, v = state["ctx"], state["u"], state["v"]
    if kind == "objective":
        return {"terms": ctx.ngf_objective(u)}
    if kind == "gradient":
        terms, grad = ctx.ngf_gradient(u)
        return {"terms": terms, "grad": grad}
    if kind == "linearize":
        terms, grad = ctx.gn_linearize(u)
        return {"terms": terms, "grad": grad}
    if kind == "hvp":
        return {"Hv": autograd.gn_hvp(ctx, u, v)}
    if kind == "matvec":
        return {"Hv": ctx.gn_matvec(v)}
    if kind == "autograd":
        w = u.detach().requires_grad_(True)
        J = autograd.objective(ctx, w)
        J.backward()
        return {"J": J.detach(), "grad": w.grad}
    if kind == "pcg":
        p, stats = ctx.gn_pcg_solve(state["g"], state["case"]["iters"])
        return {"p": p}
    w = u.clone()                       # step: the schedule updates its field in place
    code, _ = ctx.gn_solve(w, gn_iters=1, pcg_iters=state["case"]["iters"])
    return {"u": w, "code": code}


# ---------------------------------------------------------------- the work of one pass

def _gn_work(c, n, m, kind):
    N, M = math.prod(n), math.prod(m)
    img, vcc = (4 if c["half"] else 8) * N, (64 * 40 * M if c["gamma"] else 0)
    lin = {"bytes": img + 24 * M, "flops": 260 * N + vcc}
    mv = {"bytes": 24 * N + 24 * M + (12 * M if c["gamma"] else 0), "flops": 80 * N + vcc}
    obj = {"bytes": img + 12 * M, "flops": 160 * N + vcc // 2}
    if kind == "objective":
        return obj
    if kind in ("gradient", "linearize"):
        return lin
    if kind == "matvec":
        return mv
    if kind == "hvp":
        return {"bytes": img + 36 * M, "flops": lin["flops"] + mv["flops"]}
    if kind == "autograd":
        return {"bytes": 2 * img + 36 * M, "flops": lin["flops"] + obj["flops"]}
    # k products and vector updates: step k reads its k + 1 earlier residuals once
    k = c["iters"]
    hist = sum(12 * M * (j + 1) for j in range(k))
    pcg = {"bytes": k * (mv["bytes"] + 10 * 12 * M) + hist, "flops": k * (mv["flops"] + 20 * M) + hist}
    if kind == "pcg":
        return pcg
    return {"bytes": lin["bytes"] + 24 * N + pcg["bytes"] + obj["bytes"], "flops": lin["flops"] + pcg["flops"] + obj["flops"]}


def work(case):
    c, kind = case, case["kind"]
    n, _, m = _dims(c)
    N = math.prod(n)
    if kind == "batch":
        parts = [_gn_work(c, n, m, "step") for n, _, m in _batch_geometry(c)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "match":     # per direction: 64 patch points of 10 operations per label, two messages of 3 x 33 x 3 per edge
        return {"bytes": 8 * N + 2 * 4 * LABELS * c["nk"],
                "flops": 2 * c["nk"] * LABELS * (64 * 10 + 2 * 3 * 33 * 3)}
    if kind == "forstner":  # six products through three 11-tap passes
        return {"bytes": 5 * N + 8 * N, "flops": N * (6 * 3 * 22 + 40)}
    return _gn_work(c, n, m, kind)


# ---------------------------------------------------------------- the same quantities in FP64

class _Exact:
    """Objective, gradient and Gauss-Newton products of one problem in FP64."""

    def __init__(self, R, T, h, m, gamma, delta, kx=None, ky=None):
        self.R, self.T, self.h, self.m = R.double(), T.double(), h, m
        self.n = (R.shape[2], R.shape[1], R.shape[0])
        self.rho = [self.n[a] // (m[a] - 1) for a in range(3)]
        self.g = [self.n[a] * h[a] / (m[a] - 1) for a in range(3)]
        self.hbar, self.ghat = math.prod(h), math.prod(self.g)
        self.gamma, self.delta = gamma, delta
        self.P = []
        for a in range(3):
            t = (torch.arange(self.n[a], device="cuda", dtype=torch.float64) + 0.5) / self.rho[a]
            self.P.append((1.0 - (t[:, None] - torch.arange(m[a], device="cuda")).abs()).clamp(min=0.0))
        self.kp = None
        if kx is not None and kx.shape[0]:
            x, M = kx.double(), math.prod(m)
            cell = [(x[:, a] / self.g[a]).floor().clamp(0, m[a] - 2) for a in range(3)]
            idx, wgt = [], []
            for o in range(8):
                b = [o & 1, o >> 1 & 1, o >> 2]
                k = [(cell[a] + b[a]).long() for a in range(3)]
                idx.append((k[2] * m[1] + k[1]) * m[0] + k[0])
                wgt.append(math.prod((x[:, a] / self.g[a] - cell[a]) if b[a] else 1.0 - (x[:, a] / self.g[a] - cell[a])
                                     for a in range(3)))
            self.kp = torch.stack(idx), torch.stack(wgt), (x - ky.double()).T, M

    # prolongation and its transpose
    def prolong(self, u):
        u = torch.einsum("zc,kcba->kzba", self.P[2], u)
        u = torch.einsum("yb,kzba->kzya", self.P[1], u)
        return torch.einsum("xa,kzya->kzyx", self.P[0], u)

    def prolong_t(self, z, square=False):
        P = [p * p for p in self.P] if square else self.P
        z = torch.einsum("xa,kzyx->kzya", P[0], z)
        z = torch.einsum("yb,kzya->kzba", P[1], z)
        return torch.einsum("zc,kzba->kcba", P[2], z)

    def cells(self, u32):
        """Sample cell offsets and FP32 fractions per component: x, then y, then z, each step fma(w1, b, w0 a)."""
        out = []
        for k in range(3):
            v = u32[k]
            for a in range(3):
                dim = 2 - a
                t = (torch.arange(self.n[a], device="cuda", dtype=torch.float64) + 0.5) / self.rho[a]
                # cells inside [0, m - 2]; dyadic weights, exact in FP32
                c = t.floor().clamp(max=self.m[a] - 2)
                shape = [1, 1, 1]
                shape[dim] = self.n[a]
                w1 = (t - c).reshape(shape)
                p = v.index_select(dim, c.long())
                q = v.index_select(dim, c.long() + 1)
                low = ((1.0 - w1).float() * p).double()
                v = (w1 * q.double() + low).float()
            q = v * torch.tensor(1.0 / self.h[k], dtype=torch.float64).float().item()
            fl = q.floor()
            out.append((fl.long(), q - fl))
        return out

    def warp(self, u):
        """T(y) and dT/dy at the voxels, the displacement interpolated in FP64."""
        d = self.prolong(u)
        cells = self.cells(u.float())
        lo, fr, inside = [], [], []
        for a in range(3):
            n = self.n[a]
            shape = [1, 1, 1]
            shape[2 - a] = n
            i = torch.arange(n, device="cuda").reshape(shape)
            k = i + cells[a][0]
            s = i + d[a] / self.h[a]
            above = (k > n - 1) | ((k == n - 1) & (cells[a][1] > 0))
            below = k < 0
            c = k.clamp(0, n - 2)
            f = torch.where(below, 0.0, torch.where(above, 1.0, s - c))
            lo.append(c)
            fr.append(f)
            inside.append(~(above | below))
        del d, cells
        val, der = 0.0, [0.0, 0.0, 0.0]
        flat = self.T.reshape(-1)
        for o in range(8):
            b = [o & 1, o >> 1 & 1, o >> 2]
            t = flat[((lo[2] + b[2]) * self.n[1] + lo[1] + b[1]) * self.n[0] + lo[0] + b[0]]
            w = [fr[a] if b[a] else 1.0 - fr[a] for a in range(3)]
            val = val + w[0] * w[1] * w[2] * t
            for a in range(3):
                der[a] = der[a] + (1.0 if b[a] else -1.0) * w[(a + 1) % 3] * w[(a + 2) % 3] * t
        return val, torch.stack([torch.where(inside[a], der[a] / self.h[a], 0.0) for a in range(3)])

    def grad_image(self, I):
        """Central differences at the interior voxels, zero elsewhere."""
        out = torch.zeros((3,) + I.shape, dtype=I.dtype, device=I.device)
        inner = (slice(1, -1),) * 3
        for a in range(3):
            dim = 2 - a
            hi = tuple(slice(2, None) if k == dim else slice(1, -1) for k in range(3))
            lo = tuple(slice(None, -2) if k == dim else slice(1, -1) for k in range(3))
            out[a][inner] = (I[hi] - I[lo]) / (2.0 * self.h[a])
        return out

    def grad_image_t(self, c):
        """Its transpose; c is zero off the interior."""
        out = torch.zeros_like(c[0])
        for a in range(3):
            dim, k = 2 - a, c[a] / (2.0 * self.h[a])
            out.narrow(dim, 1, c[a].shape[dim] - 1).add_(k.narrow(dim, 0, k.shape[dim] - 1))
            out.narrow(dim, 0, c[a].shape[dim] - 1).sub_(k.narrow(dim, 1, k.shape[dim] - 1))
        return out

    def ngf(self, u):
        """D, and r, dr/dg, dT/dy per voxel."""
        Tw, dT = self.warp(u)
        f, g = self.grad_image(self.R), self.grad_image(Tw)
        ff, gg, fg = (ETA * ETA + (p * q).sum(0) for p, q in ((f, f), (g, g), (f, g)))
        nf, ng = ff.sqrt(), gg.sqrt()
        r = fg / (nf * ng)
        cr = torch.linalg.cross(f, g, dim=0)
        one_minus = ((cr * cr).sum(0) + ETA * ETA * ((f - g) ** 2).sum(0)) / (ff * gg)
        a = f / (nf * ng) - r * g / gg
        keep = torch.zeros_like(r)
        keep[1:-1, 1:-1, 1:-1] = 1.0
        return self.hbar * float((one_minus * keep).sum()), r * keep, a * keep, dT

    # curvature
    def L(self, u, transpose=False):
        out = torch.zeros_like(u)
        for a in range(3):
            dim, m = 3 - a, self.m[a]
            if m < 3:
                continue
            part = lambda x, s: x.narrow(dim, s, m - 2)  # noqa: E731
            if transpose:
                w = part(u, 1) / self.g[a] ** 2
                for s, f in ((0, 1.0), (1, -2.0), (2, 1.0)):
                    part(out, s).add_(f * w)
            else:
                part(out, 1).add_((part(u, 0) - 2.0 * part(u, 1) + part(u, 2)) / self.g[a] ** 2)
        return out

    # volume change: corner values [8, 3, cells] and the 64 bounds of each cell
    def corners(self, u):
        m = self.m
        return torch.stack([u[:, o >> 2:m[2] - 1 + (o >> 2), o >> 1 & 1:m[1] - 1 + (o >> 1 & 1), o & 1:m[0] - 1 + (o & 1)]
                            .reshape(3, -1) for o in range(8)])

    def corners_t(self, U):
        m = self.m
        out = torch.zeros((3, m[2], m[1], m[0]), dtype=U.dtype, device=U.device)
        for o in range(8):
            out[:, o >> 2:m[2] - 1 + (o >> 2), o >> 1 & 1:m[1] - 1 + (o >> 1 & 1), o & 1:m[0] - 1 + (o & 1)] += \
                U[o].reshape(3, m[2] - 1, m[1] - 1, m[0] - 1)
        return out

    def edges(self, U, unit):
        E = []
        for a in range(3):
            lo = [o for o in range(8) if not o >> a & 1]
            e = torch.stack([(U[o + (1 << a)] - U[o]) / self.g[a] for o in lo], 1)     # [3, 4, cells]
            if unit:
                e = e + torch.eye(3, device=U.device, dtype=U.dtype)[a][:, None, None]
            E.append(e)
        return E

    @staticmethod
    def cross(p, q):
        return torch.stack([p[1] * q[2] - p[2] * q[1], p[2] * q[0] - p[0] * q[2], p[0] * q[1] - p[1] * q[0]])

    def bounds(self, U, V=None):
        """d [4, 4, 4, cells] (a, b, c), its derivative along V, and the edges' cofactors."""
        e1, e2, e3 = self.edges(U, True)
        A, B, C = e1[:, :, None, None], e2[:, None, :, None], e3[:, None, None, :]
        x23, x31, x12 = self.cross(B, C), self.cross(C, A), self.cross(A, B)
        d = (A * x23).sum(0)
        dv = None
        if V is not None:
            v1, v2, v3 = self.edges(V, False)
            dv = ((v1[:, :, None, None] * x23).sum(0) + (v2[:, None, :, None] * x31).sum(0)
                  + (v3[:, None, None, :] * x12).sum(0))
        return d, dv, (x23, x31, x12)

    def spread(self, w, X):
        """sum of w dd/du over the bounds, per corner [8, 3, cells]."""
        G = [(w * X[0]).sum((2, 3)), (w * X[1]).sum((1, 3)), (w * X[2]).sum((1, 2))]
        out = [0.0] * 8
        for a in range(3):
            for i, o in enumerate(o for o in range(8) if not o >> a & 1):
                out[o + (1 << a)] = out[o + (1 << a)] + G[a][:, i] / self.g[a]
                out[o] = out[o] - G[a][:, i] / self.g[a]
        return torch.stack(out)

    def vcc(self, u, v=None, diag=False):
        """(energy, gradient), or the Gauss-Newton product with v, or the diagonal; slices of cells bound the memory."""
        U, V = self.corners(u), None if v is None else self.corners(v)
        e, parts = 0.0, []
        for i in range(0, U.shape[2], 1 << 17):
            s = slice(i, i + (1 << 17))
            d, dv, X = self.bounds(U[:, :, s], None if V is None else V[:, :, s])
            if diag:
                out = torch.zeros_like(U[:, :, s])
                for o in range(8):
                    for k in range(3):
                        one = torch.zeros_like(out)
                        one[o, k] = 1.0
                        out[o, k] = (self.ghat * 2.0 / d ** 3 * self.bounds(U[:, :, s], one)[1] ** 2).sum((0, 1, 2))
                parts.append(out)
                continue
            if bool((d <= 0).any()):
                e = math.inf
            e += self.ghat * float(((d - 1.0) ** 2 / d).sum())
            parts.append(self.spread(self.ghat * (1.0 - 1.0 / (d * d)) if v is None else self.ghat * 2.0 / d ** 3 * dv, X))
        out = self.corners_t(torch.cat(parts, 2))
        return (e, out) if v is None and not diag else out

    # keypoints
    def kp_at(self, u):
        idx, w, _, _ = self.kp
        return (u.reshape(3, -1)[:, idx] * w).sum(1)

    def kp_t(self, r, square=False):
        idx, w, _, M = self.kp
        out = torch.zeros((3, M), dtype=torch.float64, device="cuda")
        for o in range(8):
            out.index_add_(1, idx[o], r * (w[o] * w[o] if square else w[o]))
        return out.reshape(3, self.m[2], self.m[1], self.m[0])

    # the whole objective
    def gradient(self, u, want=True):
        D, r, a, dT = self.ngf(u)
        self.a, self.dT, self.u = a, dT, u
        Lu = self.L(u)
        Rc = 0.5 * self.ghat * float((Lu * Lu).sum())
        V, gV = self.vcc(u) if self.gamma else (0.0, 0.0)
        K, gK = 0.0, 0.0
        if self.kp is not None:
            res = self.kp[2] + self.kp_at(u)
            K, gK = float((res * res).sum()), 2.0 * self.kp_t(res)
        J = D + ALPHA * Rc + self.gamma * V + self.delta * K
        terms = torch.tensor([D, Rc, V, K, J], dtype=torch.float64)
        if not want:
            return terms, None
        g = self.prolong_t(self.grad_image_t(-2.0 * self.hbar * r * a) * dT)
        return terms, g + ALPHA * self.ghat * self.L(Lu, True) + self.gamma * gV + self.delta * gK

    def product(self, v):
        t = (self.dT * self.prolong(v)).sum(0)
        c = 2.0 * self.hbar * (self.a * self.grad_image(t)).sum(0) * self.a
        out = self.prolong_t(self.grad_image_t(c) * self.dT) + ALPHA * self.ghat * self.L(self.L(v), True)
        if self.gamma:
            out = out + self.gamma * self.vcc(self.u, v)
        if self.kp is not None:
            out = out + self.delta * 2.0 * self.kp_t(self.kp_at(v))
        return out

    def diagonal(self):
        """Jacobi diagonal, the NGF part without the adjoint's cross terms; entries <= 0 use 1."""
        beta = torch.zeros_like(self.a[0])
        for a in range(3):
            dim, q = 2 - a, self.a[a] ** 2 / (4.0 * self.h[a] ** 2)
            beta.narrow(dim, 1, q.shape[dim] - 1).add_(q.narrow(dim, 0, q.shape[dim] - 1))
            beta.narrow(dim, 0, q.shape[dim] - 1).add_(q.narrow(dim, 1, q.shape[dim] - 1))
        out = 2.0 * self.hbar * self.prolong_t(self.dT ** 2 * beta, square=True)
        # diag(L^T L): squared stencil entries, summed per row by probing with one axis' entries at a time
        lap = torch.zeros(self.m[::-1], dtype=torch.float64, device="cuda")
        centre = torch.zeros_like(lap)
        for a in range(3):
            if self.m[a] < 3:
                continue
            dim = 2 - a
            centre.narrow(dim, 1, self.m[a] - 2).add_(-2.0 / self.g[a] ** 2)
            for s in (0, 2):
                lap.narrow(dim, s, self.m[a] - 2).add_(1.0 / self.g[a] ** 4)
        out = out + ALPHA * self.ghat * (lap + centre ** 2)
        if self.gamma:
            out = out + self.gamma * self.vcc(self.u, diag=True)
        if self.kp is not None:
            out = out + self.delta * 2.0 * self.kp_t(torch.ones_like(self.kp[2]), square=True)
        return torch.where(out > 0, out, 1.0)

    def pcg(self, g, iters):
        """Fixed-length preconditioned CG on H p = -g, residuals reorthogonalised against all earlier ones."""
        Mi = 1.0 / self.diagonal()
        r = -g
        p, d, old = torch.zeros_like(r), Mi * r, []
        rz = float((r * d).sum())
        for _ in range(iters):
            q = self.product(d)
            dq = float((d * q).sum())
            if not (rz > 0 and dq > 0):
                break
            old.append((r, Mi * r, rz))
            p = p + rz / dq * d
            r = r - rz / dq * q
            co = [float((r * z).sum()) / s for _, z, s in old]
            for f, (x, _, _) in zip(co, old):
                r = r - f * x
            z = Mi * r
            new = float((r * z).sum())
            d, rz = z + new / rz * d, new
        return p

    def step(self, u, iters):
        """One Gauss-Newton iteration: solve, then Armijo backtracking t = 1, 1/2, ..., 2^-10."""
        terms, g = self.gradient(u)
        p = self.pcg(g, iters)
        slope, t = float((g * p).sum()), 1.0
        for _ in range(11):
            new = self.gradient(u + t * p, want=False)[0][4]
            if bool(torch.isfinite(new)) and float(new) <= float(terms[4]) + 1e-4 * t * slope:
                return u + t * p
            t *= 0.5
        return u


def _exact_marginals(F_, M_, kps, alpha=0.2, sigma=150.0):
    """FP64 min-marginals of the patch costs on the minimum spanning tree (edge weights compared in FP32)."""
    nk, n = kps.shape[0], F_.shape

    def features(I):
        pad = F.pad(I[None, None].double(), (1,) * 6, mode="replicate")[0, 0]
        g = [(pad[tuple(slice(2, None) if k == d else slice(1, -1) for k in range(3))]
              - pad[tuple(slice(None, -2) if k == d else slice(1, -1) for k in range(3))]) / 2.0 for d in (2, 1, 0)]
        f = torch.stack(g + [torch.full_like(g[0], ETA)], -1)
        return f / f.norm(dim=-1, keepdim=True)

    def at(f, p):
        q = [p[..., a].clamp(0, n[2 - a] - 1) for a in range(3)]
        return f[q[2], q[1], q[0]]

    ff, fm = features(F_), features(M_)
    off = torch.tensor([(x, y, z) for z in (-3, -1, 1, 3) for y in (-3, -1, 1, 3) for x in (-3, -1, 1, 3)], device="cuda")
    lab = 2 * (torch.arange(33, device="cuda") - 16)
    ax = torch.stack(torch.meshgrid(lab, lab, lab, indexing="ij"), -1).flip(-1).reshape(-1, 3)      # x fastest
    D = torch.zeros((nk, LABELS), dtype=torch.float64, device="cuda")
    for k in range(nk):
        base = kps[k].long() + off
        fk = at(ff, base)
        for s in range(0, LABELS, 12000):
            r = (at(fm, base[None] + ax[s:s + 12000, None]) * fk[None]).sum(-1)
            D[k, s:s + 12000] = (1.0 - r * r).mean(1)
    # Prim's tree of the complete graph, from keypoint 0
    p, inten = kps.float(), F_[kps[:, 2].long(), kps[:, 1].long(), kps[:, 0].long()]
    seen, best, parent, order = torch.zeros(nk, dtype=torch.bool, device="cuda"), None, torch.zeros(nk, dtype=torch.long), [0]
    best = torch.full((nk,), math.inf, device="cuda")
    par, last, wts = torch.zeros(nk, dtype=torch.long, device="cuda"), 0, [0.0] * nk
    for _ in range(nk - 1):
        seen[last] = True
        w = ((p - p[last]) ** 2).sum(1).sqrt() + (inten - inten[last]).abs() / sigma
        closer = (w < best) & ~seen
        best = torch.where(closer, w, best)
        par = torch.where(closer, last, par)
        last = int(torch.where(seen, math.inf, best).argmin())
        order.append(last)
    parent = par.tolist()
    pd, it = kps.double(), inten.double()
    for k in order[1:]:
        q = parent[k]
        wts[k] = float((pd[k] - pd[q]).norm() + (it[k] - it[q]).abs() / sigma)
    sq = (lab.double()[:, None] - lab.double()[None]) ** 2

    def message(H, lam):
        H = H.reshape(33, 33, 33)
        for d in range(3):
            c = H.movedim(d, -1)
            H = (c[..., None, :] + lam * sq).amin(-1).movedim(-1, d)
        return H.reshape(-1)

    up, total = [None] * nk, D.clone()
    for k in reversed(order[1:]):
        up[k] = message(total[k], alpha / wts[k])
        total[parent[k]] += up[k]
    for k in order[1:]:
        total[k] += message(total[parent[k]] - up[k], alpha / wts[k])
    return total


def _exact_forstner(F_, sigma=1.4):
    I = F_.double()
    pad = F.pad(I[None, None], (1,) * 6, mode="replicate")[0, 0]
    g = [(pad[tuple(slice(2, None) if k == d else slice(1, -1) for k in range(3))]
          - pad[tuple(slice(None, -2) if k == d else slice(1, -1) for k in range(3))]) / 2.0 for d in (2, 1, 0)]
    w = torch.exp(-torch.arange(-5, 6, device="cuda", dtype=torch.float64) ** 2 / (2.0 * sigma * sigma))
    w = w / w.sum()

    def smooth(x):
        for d in range(3):
            idx = torch.arange(x.shape[d], device="cuda")
            x = sum(w[i + 5] * x.index_select(d, (idx + i).clamp(0, x.shape[d] - 1)) for i in range(-5, 6))
        return x

    a, b, c = smooth(g[0] * g[0]), smooth(g[1] * g[1]), smooth(g[2] * g[2])
    d, e, f = smooth(g[0] * g[1]), smooth(g[0] * g[2]), smooth(g[1] * g[2])
    det = a * (b * c - f * f) - d * (d * c - f * e) + e * (d * f - b * e)
    minors = (b * c - f * f) + (a * c - e * e) + (a * b - d * d)
    return torch.where(minors > 0, det / minors, 0.0)


def exact(case, seed):
    c, kind = case, case["kind"]
    n, h, m = _dims(c)
    if kind == "match":
        if c["nk"] > 400:
            return None         # the FP64 costs of 3000 keypoints take minutes
        R, T, _, vessels, _ = _pair(n, h, m, seed, large=True)
        kps = _vessel_voxels(vessels, c["nk"], n, _gen(seed + 7919))
        return {"disp": None, "forward": _exact_marginals(R, T, kps), "backward": None}
    if kind == "forstner":
        return {"count": None, "kps": None, "response": _exact_forstner(_pair(n, h, m, seed, large=True)[0])}
    if kind == "batch":
        us = []
        for i, (n, h, m) in enumerate(_batch_geometry(c)):
            if math.prod(n) > 4 << 20:
                us.append(None)
                continue
            R, T = (_stored(x, True).double() - 1024.0 for x in _pair(n, h, m, seed + 31 * i, large=True)[:2])
            u = torch.zeros((3, m[2], m[1], m[0]), dtype=torch.float64, device="cuda")
            us.append(_Exact(R, T, h, m, c["gamma"], 0.0).step(u, c["iters"]))
        return {"u": us, "code": None}
    if kind in ("pcg", "step") and math.prod(n) > 8 << 20:
        return None
    R, T, u, v, kx, ky = _problem(c, seed)
    if c["half"]:
        R, T = (_stored(x, True).double() - 1024.0 for x in (R, T))
    P = _Exact(R, T, h, m, c["gamma"], c["delta"], kx, ky)
    u, v = u.double(), v.double()
    terms, g = P.gradient(u)
    if kind == "objective":
        return {"terms": terms}
    if kind in ("gradient", "linearize"):
        return {"terms": terms, "grad": g}
    if kind in ("hvp", "matvec"):
        return {"Hv": P.product(v)}
    if kind == "autograd":
        return {"J": terms[4], "grad": g}
    if kind == "pcg":
        return {"p": P.pcg(g, c["iters"])}
    return {"u": P.step(u, c["iters"]), "code": None}
