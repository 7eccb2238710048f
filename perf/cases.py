"""Cases of the performance measurement: the calls that users of this package
make, at the sizes they make them.

A scanner's program builds one ``Plan`` per geometry and keeps it; per slice
(or batch of slices) it runs the ADM-TV reconstruction and the PLS
decomposition.  Programs with their own iteration call the projector pair
directly, an analytic preview is an FBP, volumes go through the cone-beam
operators, and the warm-start network is trained on pairs the method makes.

Geometries keep the proportions of this repository's configurations (pitch
1.2 pixels at twice the magnification, 1.44 to 1.5 bins per pixel column,
SOD 500 mm, SDD 1000 mm).  The ADM runs a fixed number of iterations, as its
configurations of 100, 200 and 300 iterations do: the iteration at which the
relative-objective rule stops turns on rounding.
"""
import math
import types

import numpy as np
import torch

import paper_1607_01650_gb300 as dect

# attenuation (1/mm) of the water-like and the bone-like material at (high, low) energy
ETA = ((0.0184, 0.0227), (0.0342, 0.0573))
MU, RHO, BETA = 4.0, 256.0, (1.0, 0.6)
GAMMA, TAU, EPS = 0.1, 0.2, 0.05
SCALE = 0.02  # input scale of the warm-start network, 1/mm
DEV = "cuda"


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def _adm(name, n, nv, nb, slices, iters, fov=256.0, **more):
    return dict(name=name, path="adm", n=n, nv=nv, nb=nb, fov=fov, slices=slices, iters=iters,
                joint=False, nonneg=False, **more)


def listed():
    return [
        # the smallest configuration: one 128^2 slice, 100 iterations; launches and host work count
        _adm("adm_small", 128, 60, 192, 1, 100, fov=128.0),
        # one paper-sized slice, as a scanner's console asks for it
        _adm("adm_slice", 512, 60, 736, 1, 60),
        # the headline's batch: 32 slices that share the plan
        _adm("adm_batch", 512, 60, 736, 32, 100),
        # slices of uneven size and view count (odd sizes too), each its own plan, joint TV
        dict(name="adm_uneven", path="groups", entry="groups", ns="256,320,384,448,512,331", nvs="45,180,97,60,31,120",
             slices=1, iters=40, joint=True, nonneg=False),
        # the dense configuration: 1024^2, 360 views, a small batch
        _adm("adm_dense", 1024, 360, 1472, 8, 10),
        # a user's own iteration on one dual-energy slice: A x, then A^T of the residual
        dict(name="operators_pair", path="operators", n=512, nv=60, nb=736, fov=256.0, batch=2),
        # the same pair over a whole series
        dict(name="operators_series", path="operators", n=512, nv=60, nb=736, fov=256.0, batch=64),
        # analytic preview of a series: 32 slices, both energies
        dict(name="fbp_series", path="fbp", n=512, nv=60, nb=736, fov=256.0, batch=64),
        # the decomposition of one slice, and of a series
        dict(name="pls_slice", path="pls", n=512, batch=1),
        dict(name="pls_series", path="pls", n=512, batch=32),
        # cone-beam operators on one dual-energy volume
        dict(name="cone_pair", path="cone", n=256, nz=64, nv=60, nr=64, nc=368, batch=2),
        # one training step of the warm-start network
        dict(name="cnn_train", path="cnn", train=True, h=256, w=256, batch=16),
    ]


def _bins(n, nb):
    # an odd number of bins has a ray along the axis, which is a grid line where n is even: those go with odd n
    return nb + 1 if n % 2 == 0 and nb % 2 else nb


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["adm", "adm", "adm", "groups", "operators", "operators", "fbp", "pls", "pls", "cone", "cnn"])
    fov = rng.choice([128.0, 200.0, 256.0])
    if path == "adm":
        n = _log_int(rng, 96, 640)
        nv = _log_int(rng, 30, 180)
        c = dict(path=path, n=n, nv=nv, nb=_bins(n, int(n * rng.uniform(1.43, 1.5))), fov=fov, slices=_log_int(rng, 1, 40),
                 iters=rng.randrange(10, 101), joint=rng.random() < 0.3, nonneg=rng.random() < 0.2)
        cap = 0.9 * 512 * 736 * 60 * 32 * 100
        cost = lambda: c["n"] * c["nb"] * c["nv"] * c["slices"] * c["iters"]  # noqa: E731
        while cost() > cap:
            c["slices"] = max(1, c["slices"] // 2)
            c["iters"] = max(10, c["iters"] // 2)
        return c
    if path == "groups":
        k = rng.randrange(2, 7)
        ns = [_log_int(rng, 200, 512) for _ in range(k)]
        nvs = [_log_int(rng, 30, 180) for _ in range(k)]
        return dict(path=path, entry=rng.choice(["groups", "groups", "table", "otf"]), ns=",".join(map(str, ns)),
                    nvs=",".join(map(str, nvs)), slices=rng.randrange(1, 3), iters=rng.randrange(10, 41),
                    joint=rng.random() < 0.5, nonneg=rng.random() < 0.2)
    if path in ("operators", "fbp"):
        n = _log_int(rng, 96, 640)
        return dict(path=path, n=n, nv=_log_int(rng, 30, 180), nb=_bins(n, int(n * rng.uniform(1.43, 1.5))), fov=fov,
                    batch=_log_int(rng, 1, 70))
    if path == "pls":
        return dict(path=path, n=_log_int(rng, 96, 700), batch=_log_int(rng, 1, 40))
    if path == "cone":
        n = _log_int(rng, 64, 256)
        nz = rng.randrange(12, 65)
        return dict(path=path, n=n, nz=nz, nv=rng.randrange(24, 61), nr=nz, nc=_bins(n, int(1.44 * n)), batch=rng.randrange(1, 5))
    return dict(path=path, train=rng.random() < 0.3, h=4 * _log_int(rng, 16, 64), w=4 * _log_int(rng, 16, 64),
                batch=_log_int(rng, 1, 16))


# ---------------------------------------------------------------------------
# Inputs: seeded head-like phantoms (sums of ellipses), their exact line
# integrals with Poisson noise, and their images
# ---------------------------------------------------------------------------
def _phantom(rng, half):
    """Rows (cx, cy, a, b, phi, water, bone): scalp, skull, brain and 6-12 inserts, inside a disk of radius `half` mm."""
    s = 0.8 * half / 105.0
    tilt, skull = rng.uniform(-0.1, 0.1), rng.uniform(4.0, 7.0)
    A, B = 90.0, 105.0
    rows = [(0, 0, A, B, tilt, 1, 0), (0, 0, A - 3, B - 3, tilt, -1, 1),
            (0, 0, A - 3 - skull, B - 3 - skull, tilt, 1, -1)]
    for _ in range(int(rng.integers(6, 13))):
        d, r, t = rng.uniform(2.0, 12.0), 0.75 * math.sqrt(rng.uniform()), rng.uniform(0, 2 * math.pi)
        dw, db = ((-0.5, 0.5), (-1.0, 1.0), (0.3, 0.0))[int(rng.integers(0, 3))]
        rows.append((r * (A - 10) * math.cos(t), r * (B - 10) * math.sin(t), d / 2, d * rng.uniform(0.6, 1.0) / 2,
                     rng.uniform(0, math.pi), dw, db))
    e = np.array(rows, dtype=np.float64)
    e[:, :4] *= s
    return e


def _geometry(c):
    px = c["fov"] / c["n"]
    return dect.Geometry(n=c["n"], px=px, nv=c["nv"], nb=c["nb"], pitch=1.2 * px, sod=500.0, sdd=1000.0)


def _ends(g):
    """Ray end points [nv, nb, 2] (float64)."""
    th = g.start + torch.arange(g.nv, dtype=torch.float64, device=DEV) * (g.arc / g.nv)
    c, s = torch.cos(th)[:, None], torch.sin(th)[:, None]
    u = (torch.arange(g.nb, dtype=torch.float64, device=DEV) - 0.5 * (g.nb - 1)) * g.pitch + g.det_offset
    S = torch.stack([(g.sod * c).expand(g.nv, g.nb), (g.sod * s).expand(g.nv, g.nb)], -1)
    D = torch.stack([(g.sod - g.sdd) * c - u * s, (g.sod - g.sdd) * s + u * c], -1)
    return S, D


def _fov_radius(g):
    half = 0.5 * g.nb * g.pitch
    return min(0.5 * g.n * g.px, half * g.sod / math.hypot(g.sdd, half))


def _sinograms(g, seed, slices, i0=2e5):
    """Measured line integrals m [slices, 2, nv, nb] float32."""
    rng = np.random.default_rng(seed)
    S, D = _ends(g)
    d = D - S
    d = d / d.norm(dim=-1, keepdim=True)
    p = torch.empty((slices, 2, g.nv, g.nb), dtype=torch.float64, device=DEV)
    for k in range(slices):
        water, bone = torch.zeros_like(d[..., 0]), torch.zeros_like(d[..., 0])
        for cx, cy, a, b, phi, fw, fb in _phantom(rng, 0.95 * _fov_radius(g)).tolist():
            co, si = math.cos(phi), math.sin(phi)
            px, py = S[..., 0] - cx, S[..., 1] - cy
            ox, oy = (co * px + si * py) / a, (co * py - si * px) / b
            dx, dy = (co * d[..., 0] + si * d[..., 1]) / a, (co * d[..., 1] - si * d[..., 0]) / b
            qa, qb, qc = dx * dx + dy * dy, 2 * (ox * dx + oy * dy), ox * ox + oy * oy - 1
            chord = (qb * qb - 4 * qa * qc).clamp_min(0).sqrt() / qa
            water += fw * chord
            bone += fb * chord
        for e in range(2):
            p[k, e] = ETA[0][e] * water + ETA[1][e] * bone
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) + 1)
    counts = torch.poisson(i0 * torch.exp(-p), generator=gen)
    return (-torch.log(counts.clamp_min(1) / i0)).float().contiguous()


def _images(n, seed, slices, noise=0.02, nz=0):
    """Attenuation images [slices, 2, (nz,) n, n] float32 of phantoms, with reconstruction-like noise."""
    rng = np.random.default_rng(seed)
    t = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) * (256.0 / n) - 128.0
    X, Y = t[None, :], t[:, None]
    out = torch.empty((slices, 2) + ((nz,) if nz else ()) + (n, n), dtype=torch.float32, device=DEV)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) + 2)
    for k in range(slices):
        u = torch.zeros((2, n, n), dtype=torch.float64, device=DEV)
        for cx, cy, a, b, phi, fw, fb in _phantom(rng, 120.0).tolist():
            co, si = math.cos(phi), math.sin(phi)
            q = ((co * (X - cx) + si * (Y - cy)) / a) ** 2 + ((co * (Y - cy) - si * (X - cx)) / b) ** 2
            inside = ((1 - q) * (0.5 * min(a, b) * n / 256.0) + 0.5).clamp(0, 1)  # soft over about a pixel
            u[0] += fw * inside
            u[1] += fb * inside
        for e in range(2):
            x = ETA[0][e] * u[0] + ETA[1][e] * u[1]
            if nz:
                x = x[None] * torch.linspace(0.8, 1.1, nz, dtype=torch.float64, device=DEV)[:, None, None]
            z = torch.randn(x.shape, generator=gen, device=DEV, dtype=torch.float64)
            out[k, e] = (x + noise * SCALE * z).float()
    return out


def _pls_params():
    return dect.PlsParams(eta=ETA, gamma=GAMMA, edge_tau=TAU, edge_eps=EPS, max_iter=500, tol=1e-6)


def _adm_params(c):
    return dect.AdmParams(mu=MU, rho=RHO, beta=BETA, max_iter=c["iters"], joint=c["joint"], nonneg=c["nonneg"])


def _group_geometries(c):
    """The uneven workload's geometries: 0.5 mm pixels, 0.6 mm pitch, bins scaled with n."""
    out = []
    for n, nv in zip(map(int, c["ns"].split(",")), map(int, c["nvs"].split(","))):
        out.append(dect.Geometry(n=n, px=0.5, nv=nv, nb=368 + 2 * int(round((n - 256) / 256.0 * 184)), pitch=0.6,
                                 sod=500.0, sdd=1000.0))
    return out


def _cone_geometry(c):
    s = 256.0 / c["n"]
    return types.SimpleNamespace(n=c["n"], nz=c["nz"], px=0.5 * s, pz=0.5 * s, nv=c["nv"], nr=c["nr"], nc=c["nc"],
                                 pu=0.6 * s, pv=0.6 * s, sod=500.0, sdd=1000.0, start=0.0, arc=2.0 * math.pi,
                                 off_u=0.0, off_v=0.0)


_CNN = [(1, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128), (192, 64), (64, 64), (96, 32), (32, 32)]


def _cnn_weights(seed):
    rng = np.random.default_rng(seed)
    parts = []
    for ci, co in _CNN:
        parts += [rng.standard_normal(co * ci * 9) * math.sqrt(2.0 / (9 * ci)), 0.01 * rng.standard_normal(co)]
    parts += [0.1 * rng.standard_normal(32), np.zeros(1)]  # a head as it is some steps into the training
    return np.concatenate(parts).astype(np.float32)


def _cnn_pairs(c, seed):
    n = max(c["h"], c["w"])
    k = (c["batch"] + 1) // 2
    t = _images(n, seed, k, noise=0.0).reshape(2 * k, n, n)[:c["batch"], :c["h"], :c["w"]].contiguous()
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) + 3)
    x = t + 0.05 * SCALE * torch.randn(t.shape, generator=gen, device=DEV)
    return x.contiguous(), t


def prepare(case, seed):
    c, path = case, case["path"]
    if path == "adm":
        g = _geometry(c)
        return dict(path=path, plan=dect.Plan(g), m=_sinograms(g, seed, c["slices"]), params=_adm_params(c))
    if path == "groups":
        gs = _group_geometries(c)
        return dict(path=path, entry=c["entry"], plans=[dect.Plan(g) for g in gs], params=_adm_params(c),
                    ms=[_sinograms(g, seed + 31 * k, c["slices"]) for k, g in enumerate(gs)])
    if path == "operators":
        g = _geometry(c)
        x = _images(c["n"], seed, (c["batch"] + 1) // 2).reshape(-1, c["n"], c["n"])[:c["batch"]].contiguous()
        m = _sinograms(g, seed + 5, 1)[0, 0]
        return dict(path=path, plan=dect.Plan(g), x=x, m=m.expand(c["batch"], -1, -1).contiguous())
    if path == "fbp":
        g = _geometry(c)
        m = _sinograms(g, seed, (c["batch"] + 1) // 2).reshape(-1, c["nv"], c["nb"])[:c["batch"]].contiguous()
        return dict(path=path, plan=dect.Plan(g), m=m)
    if path == "pls":
        return dict(path=path, x=_images(c["n"], seed, c["batch"]), params=_pls_params())
    if path == "cone":
        x = _images(c["n"], seed, (c["batch"] + 1) // 2, nz=c["nz"])
        x = x.reshape(-1, c["nz"], c["n"], c["n"])[:c["batch"]].contiguous()
        return dict(path=path, plan=dect.ConePlan(_cone_geometry(c)), x=x)
    net = dect.Cnn(max_pixels=c["batch"] * c["h"] * c["w"])
    net.set_params(_cnn_weights(seed))
    x, t = _cnn_pairs(c, seed)
    return dict(path=path, train=c["train"], net=net, x=x, t=t)


def _reports(reps):
    return {"iters": np.array([r.iters for r in reps], dtype=np.int64),
            "objective": np.array([r.objective for r in reps], dtype=np.float32)}


def run(state):
    s, path = state, state["path"]
    if path == "adm":
        x, reps = dect.adm_tv(s["plan"], s["m"], s["params"])
        return {"x": x, **_reports(reps)}
    if path == "groups":
        groups = [(p, m, None) for p, m in zip(s["plans"], s["ms"])]
        got = dect.adm_tv_groups(groups, s["params"]) if s["entry"] == "groups" else \
            dect.adm_tv_batch(groups, s["params"], projector=s["entry"])
        return [{"x": x, **_reports(reps)} for x, reps in got]
    if path == "operators":
        y = dect.project(s["plan"], s["x"])
        return {"y": y, "g": dect.backproject(s["plan"], s["m"] - y)}
    if path == "fbp":
        return dect.fbp(s["plan"], s["m"])
    if path == "pls":
        u, reps = dect.pls_decompose(s["x"], s["params"])
        return {"u": u, "iters": np.array([r[0] for r in reps], dtype=np.int64)}
    if path == "cone":
        y = dect.project_cone(s["plan"], s["x"])
        return {"y": y, "g": dect.backproject_cone(s["plan"], y)}
    if not s["train"]:
        return s["net"].forward(s["x"], SCALE)
    loss, grad = s["net"].loss_grad(s["x"], s["t"], SCALE, want_grad=True)
    s["net"].adam_step(3e-4)
    return {"loss": loss, "grad": grad}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _nnz(n, nv, nb):
    # a ray meets about 1.27 pixels per row it crosses, and crosses about all n rows
    return 1.27 * n * nv * nb


def work(case):
    c, path = case, case["path"]
    if path in ("adm", "groups"):
        shapes = [(c["n"], c["nv"], c["nb"])] if path == "adm" else [(g.n, g.nv, g.nb) for g in _group_geometries(c)]
        by, fl = 0.0, 0.0
        for n, nv, nb in shapes:
            ch = 2 * c["slices"]
            by += 4.0 * ch * (nv * nb + n * n)
            # per iteration and channel: A, A^T (2 operations per element each) and the TV step
            fl += ch * c["iters"] * (4.0 * _nnz(n, nv, nb) * (1.5 if c["nonneg"] else 1.0) + 40.0 * n * n)
        return {"bytes": by, "flops": fl}
    if path == "operators":
        N, M = c["n"] ** 2, c["nv"] * c["nb"]
        return {"bytes": 4.0 * c["batch"] * (2 * N + 4 * M), "flops": 4.0 * c["batch"] * _nnz(c["n"], c["nv"], c["nb"])}
    if path == "fbp":
        N, M = c["n"] ** 2, c["nv"] * c["nb"]
        return {"bytes": 4.0 * c["batch"] * (N + M), "flops": c["batch"] * (5.0 * N * c["nv"] + 40.0 * M)}
    if path == "pls":
        N = c["n"] ** 2
        return {"bytes": 16.0 * c["batch"] * N, "flops": c["batch"] * N * (40.0 + 2 * 5 * 30.0)}
    if path == "cone":
        N, M = c["n"] ** 2 * c["nz"], c["nv"] * c["nr"] * c["nc"]
        return {"bytes": 4.0 * c["batch"] * (2 * N + 2 * M), "flops": 4.0 * c["batch"] * 1.3 * c["n"] * M}
    px = float(c["batch"] * c["h"] * c["w"])
    macs = sum(ci * co * 9 / f for (ci, co), f in zip(_CNN, (1, 1, 4, 4, 16, 16, 4, 4, 1, 1)))
    w = sum(ci * co * 9 + co for ci, co in _CNN) + 33
    if c["train"]:
        return {"bytes": 4.0 * (2 * px + 9 * w), "flops": 6.0 * macs * px}
    return {"bytes": 4.0 * (2 * px + w), "flops": 2.0 * macs * px}


# ---------------------------------------------------------------------------
# The same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _crossings(S, D, axes):
    """Siddon pieces of the rays S -> D [R, dim]: (index [R, K], length [R, K]); axes: (lo, step, count) per axis,
    the first axis the fastest index."""
    d = D - S
    L = d.norm(dim=-1, keepdim=True)
    R = S.shape[0]
    amin, amax = torch.zeros((R, 1), device=DEV, dtype=torch.float64), torch.ones((R, 1), device=DEV, dtype=torch.float64)
    cuts = []
    for a, (lo, step, cnt) in enumerate(axes):
        lines = lo + step * torch.arange(cnt + 1, device=DEV, dtype=torch.float64)
        t = (lines[None, :] - S[:, a:a + 1]) / d[:, a:a + 1]
        t = torch.where(torch.isfinite(t), t, torch.full_like(t, -1.0))
        flat = d[:, a:a + 1].abs() == 0
        inside = (S[:, a:a + 1] >= lo) & (S[:, a:a + 1] < lo + step * cnt)
        t0, t1 = torch.minimum(t[:, :1], t[:, -1:]), torch.maximum(t[:, :1], t[:, -1:])
        amin = torch.where(flat, torch.where(inside, amin, torch.full_like(amin, 2.0)), torch.maximum(amin, t0))
        amax = torch.where(flat, amax, torch.minimum(amax, t1))
        cuts.append(t)
    amax = torch.maximum(amax, amin)
    t = torch.cat(cuts + [amin, amax], 1)
    t = torch.minimum(torch.maximum(t, amin), amax).sort(dim=1).values
    mid, seg = 0.5 * (t[:, 1:] + t[:, :-1]), (t[:, 1:] - t[:, :-1]) * L
    idx = torch.zeros_like(mid, dtype=torch.int64)
    stride = 1
    for a, (lo, step, cnt) in enumerate(axes):
        k = torch.floor((S[:, a:a + 1] + mid * d[:, a:a + 1] - lo) / step).to(torch.int64)
        seg = torch.where((k >= 0) & (k < cnt), seg, torch.zeros_like(seg))
        idx += k.clamp(0, cnt - 1) * stride
        stride *= cnt
    return idx, seg


class _Matrix:
    """A and its transpose as sparse float64 matrices."""

    def __init__(self, g):
        S, D = _ends(g)
        S, D = S.reshape(-1, 2), D.reshape(-1, 2)
        M, N = g.nv * g.nb, g.n * g.n
        axes = [(-0.5 * g.n * g.px, g.px, g.n)] * 2
        rows, cols, vals = [], [], []
        step = max(1, 30_000_000 // (2 * g.n))
        for r in range(0, M, step):
            idx, seg = _crossings(S[r:r + step], D[r:r + step], axes)
            keep = seg > 0
            rows.append(keep.sum(1))
            cols.append(idx[keep].to(torch.int32))
            vals.append(seg[keep])
        cnt, cols, vals = torch.cat(rows), torch.cat(cols), torch.cat(vals)
        z = torch.zeros(1, dtype=torch.int64, device=DEV)
        ptr = torch.cat([z, cnt.cumsum(0)]).to(torch.int32)
        ray = torch.repeat_interleave(torch.arange(M, device=DEV, dtype=torch.int32), cnt)
        order = torch.argsort(cols, stable=True)
        tptr = torch.cat([z, torch.bincount(cols, minlength=N).cumsum(0)]).to(torch.int32)
        self.A = torch.sparse_csr_tensor(ptr, cols, vals, size=(M, N))
        self.T = torch.sparse_csr_tensor(tptr, ray[order], vals[order], size=(N, M))

    def fwd(self, x):  # [N, C] -> [M, C]
        return torch.sparse.mm(self.A, x)

    def adj(self, y):
        return torch.sparse.mm(self.T, y)


def _grad(f):  # [n, n, C] -> backward differences along rows and columns
    d0, d1 = torch.zeros_like(f), torch.zeros_like(f)
    d0[1:] = f[1:] - f[:-1]
    d1[:, 1:] = f[:, 1:] - f[:, :-1]
    return d0, d1


def _grad_t(p0, p1):
    g = p0.clone()
    g[0] = 0
    g[:-1] -= p0[1:]
    g[:, 1:] += p1[:, 1:]
    g[:, :-1] -= p1[:, 1:]
    return g


def _adm_exact(g, m, c):
    n, C = g.n, 2 * m.shape[0]
    A = _Matrix(g)
    beta = torch.tensor(BETA, dtype=torch.float64, device=DEV).repeat(m.shape[0])
    meas = beta[None, :] * m.double().reshape(C, -1).t().contiguous()

    def pair(v):  # joint TV: sums over both energies of a slice
        return v.reshape(v.shape[:-1] + (C // 2, 2)).sum(-1).repeat_interleave(2, dim=-1) if c["joint"] else v

    f = torch.zeros((n, n, C), dtype=torch.float64, device=DEV)
    l0, l1 = torch.zeros_like(f), torch.zeros_like(f)
    for _ in range(c["iters"]):
        r = A.fwd(f.reshape(-1, C)) - meas
        d0, d1 = _grad(f)
        w0, w1 = d0 - l0 / RHO, d1 - l1 / RHO
        nrm = pair(w0 * w0 + w1 * w1).sqrt()
        k = torch.where(nrm > 1 / RHO, (nrm - 1 / RHO) / nrm.clamp_min(1e-300), torch.zeros_like(nrm))
        z0, z1 = k * w0, k * w1
        G = MU * A.adj(r).reshape(n, n, C) + _grad_t(RHO * (d0 - z0) - l0, RHO * (d1 - z1) - l1)
        q = A.fwd(G.reshape(-1, C))
        e0, e1 = _grad(G)
        num, den = pair((G * G).sum((0, 1))), pair(MU * (q * q).sum(0) + RHO * (e0 * e0 + e1 * e1).sum((0, 1)))
        f = f - torch.where(den > 0, num / den.clamp_min(1e-300), torch.zeros_like(num)) * G
        if c["nonneg"]:
            f = f.clamp_min(0)
        d0, d1 = _grad(f)
        l0, l1 = l0 - RHO * (d0 - z0), l1 - RHO * (d1 - z1)
    r = A.fwd(f.reshape(-1, C)) - meas
    d0, d1 = _grad(f)
    tv = pair(d0 * d0 + d1 * d1).sqrt().sum((0, 1))
    obj = tv + 0.5 * MU * pair((r * r).sum(0))
    x = (f / beta).permute(2, 0, 1).reshape(C // 2, 2, n, n)
    return {"x": x, "iters": None, "objective": obj.cpu().numpy()}


def _fbp_exact(g, m):
    ds = g.pitch * g.sod / g.sdd
    s = ((torch.arange(g.nb, dtype=torch.float64, device=DEV) - 0.5 * (g.nb - 1)) * g.pitch + g.det_offset) * g.sod / g.sdd
    k = torch.arange(g.nb, device=DEV)[:, None] - torch.arange(g.nb, device=DEV)[None, :]
    h = torch.where(k % 2 != 0, -1.0 / (math.pi ** 2 * k.double() ** 2 * ds * ds).clamp_min(1e-300), torch.zeros_like(k, dtype=torch.float64))
    h = torch.where(k == 0, torch.full_like(h, 1.0 / (4 * ds * ds)), h)
    q = ds * ((m.double() * (g.sod / torch.sqrt(g.sod ** 2 + s * s))) @ h)
    t = (torch.arange(g.n, dtype=torch.float64, device=DEV) + 0.5 - 0.5 * g.n) * g.px
    X, Y = t[None, :].expand(g.n, g.n), t[:, None].expand(g.n, g.n)
    out = torch.zeros(m.shape[:-2] + (g.n, g.n), dtype=torch.float64, device=DEV)
    for v in range(g.nv):
        th = g.start + v * (g.arc / g.nv)
        co, si = math.cos(th), math.sin(th)
        r = g.sod / (g.sod - X * co - Y * si)
        b = ((Y * co - X * si) * r - s[0]) / ds
        ok = (b >= 0) & (b <= g.nb - 1)
        b0 = torch.floor(b).clamp(0, g.nb - 2).to(torch.int64)
        w = b - b0
        row = q[..., v, :]
        val = (1 - w) * row[..., b0] + w * row[..., b0 + 1]
        out += torch.where(ok, 0.5 * g.arc / g.nv * r * r, torch.zeros_like(r)) * val
    return out


def _prewitt(x):
    p = torch.nn.functional.pad(x, (1, 1, 1, 1), mode="replicate")
    gx = sum(p[..., a:a + x.shape[-2], 2:] - p[..., a:a + x.shape[-2], :-2] for a in range(3))
    gy = sum(p[..., 2:, a:a + x.shape[-1]] - p[..., :-2, a:a + x.shape[-1]] for a in range(3))
    return (gx * gx + gy * gy).sqrt()


def _pls_exact(x):
    x = x.double()
    (a, c), (b, e) = ETA
    det = a * e - b * c
    d = torch.stack([(e * x[:, 0] - b * x[:, 1]) / det, (a * x[:, 1] - c * x[:, 0]) / det], 1)
    mag = _prewitt(x)
    edge = (mag / mag.amax((2, 3), keepdim=True) > TAU).any(1, keepdim=True)
    w0 = torch.where(edge[:, :, 1:] | edge[:, :, :-1], EPS, 1.0).double()
    w1 = torch.where(edge[..., 1:] | edge[..., :-1], EPS, 1.0).double()

    def op(u):
        out = u.clone()
        t0, t1 = GAMMA * w0 * (u[:, :, 1:] - u[:, :, :-1]), GAMMA * w1 * (u[..., 1:] - u[..., :-1])
        out[:, :, 1:] += t0
        out[:, :, :-1] -= t0
        out[..., 1:] += t1
        out[..., :-1] -= t1
        return out

    def dot(p, q):
        return (p * q).sum((2, 3), keepdim=True)

    u = d.clone()
    r = d - op(u)
    p = r.clone()
    rr = dot(r, r)
    for _ in range(60):
        q = op(p)
        al = rr / dot(p, q).clamp_min(1e-300)
        u += al * p
        r -= al * q
        new = dot(r, r)
        p = r + new / rr.clamp_min(1e-300) * p
        rr = new
    return {"u": u, "iters": None}


def _cone_exact(c, x):
    g = _cone_geometry(c)
    th = g.start + torch.arange(g.nv, dtype=torch.float64, device=DEV) * (g.arc / g.nv)
    u = (torch.arange(g.nc, dtype=torch.float64, device=DEV) - 0.5 * (g.nc - 1)) * g.pu + g.off_u
    z = (torch.arange(g.nr, dtype=torch.float64, device=DEV) - 0.5 * (g.nr - 1)) * g.pv + g.off_v
    axes = [(-0.5 * g.n * g.px, g.px, g.n)] * 2 + [(-0.5 * g.nz * g.pz, g.pz, g.nz)]
    B = x.shape[0]
    xf = x.double().reshape(B, -1).t().contiguous()
    y = torch.empty((g.nv * g.nr * g.nc, B), dtype=torch.float64, device=DEV)
    bt = torch.zeros_like(xf)
    per = g.nr * g.nc
    for v in range(g.nv):
        co, si = torch.cos(th[v]), torch.sin(th[v])
        D = torch.stack([((g.sod - g.sdd) * co - u * si).expand(g.nr, g.nc), ((g.sod - g.sdd) * si + u * co).expand(g.nr, g.nc),
                         z[:, None].expand(g.nr, g.nc)], -1).reshape(-1, 3)
        S = torch.stack([g.sod * co, g.sod * si, torch.zeros_like(co)]).expand(per, 3)
        idx, seg = _crossings(S, D, axes)
        for k in range(B):
            yk = (seg * xf[:, k][idx]).sum(1)
            y[v * per:(v + 1) * per, k] = yk
            keep = seg > 0
            bt[:, k].index_add_(0, idx[keep], (seg * yk[:, None])[keep])
    return {"y": y.t().reshape(B, g.nv, g.nr, g.nc), "g": bt.t().reshape(x.shape)}


def _cnn_exact(c, seed):
    w = torch.tensor(_cnn_weights(seed), dtype=torch.float64, device=DEV).requires_grad_(c["train"])
    x, t = _cnn_pairs(c, seed)
    at, F = 0, torch.nn.functional
    layers = []
    for ci, co in _CNN:
        k, at = w[at:at + co * ci * 9].reshape(co, ci, 3, 3), at + co * ci * 9
        layers.append((k, w[at:at + co]))
        at += co
    head, hb = w[at:at + 32].reshape(1, 32, 1, 1), w[at + 32:at + 33]

    def conv(v, i):
        return F.relu(F.conv2d(v, layers[i][0], layers[i][1], padding=1))

    total, out = 0.0, []
    for b in range(c["batch"]):
        xb = x[b:b + 1, None].double()
        e1 = conv(conv(xb / SCALE, 0), 1)
        e2 = conv(conv(F.avg_pool2d(e1, 2), 2), 3)
        bt = conv(conv(F.avg_pool2d(e2, 2), 4), 5)
        d2 = conv(conv(torch.cat([F.interpolate(bt, scale_factor=2), e2], 1), 6), 7)
        d1 = conv(conv(torch.cat([F.interpolate(d2, scale_factor=2), e1], 1), 8), 9)
        y = xb + SCALE * F.conv2d(d1, head, hb)
        if c["train"]:
            loss = ((y[:, 0] - t[b:b + 1].double()) ** 2).sum() / x.numel()
            loss.backward()
            total += float(loss)
        else:
            out.append(y[:, 0])
    return {"loss": total, "grad": w.grad} if c["train"] else torch.cat(out)


def exact(case, seed):
    c, path = case, case["path"]
    if path == "adm":
        g = _geometry(c)
        if g.n * g.nv * g.nb > 60_000_000:  # the sparse matrix in 64 bits would take longer than the measurement waits
            return None
        return _adm_exact(g, _sinograms(g, seed, c["slices"]), c)
    if path == "groups":
        return [_adm_exact(g, _sinograms(g, seed + 31 * k, c["slices"]), c) for k, g in enumerate(_group_geometries(c))]
    if path == "operators":
        g = _geometry(c)
        A = _Matrix(g)
        x = _images(c["n"], seed, (c["batch"] + 1) // 2).reshape(-1, c["n"], c["n"])[:c["batch"]]
        m = _sinograms(g, seed + 5, 1)[0, 0].double()
        y = A.fwd(x.double().reshape(c["batch"], -1).t().contiguous())
        r = A.adj(m.reshape(-1, 1) - y)
        return {"y": y.t().reshape(c["batch"], g.nv, g.nb), "g": r.t().reshape(x.shape)}
    if path == "fbp":
        g = _geometry(c)
        m = _sinograms(g, seed, (c["batch"] + 1) // 2).reshape(-1, c["nv"], c["nb"])[:c["batch"]]
        return torch.cat([_fbp_exact(g, k) for k in m.split(8)])
    if path == "pls":
        return _pls_exact(_images(c["n"], seed, c["batch"]))
    if path == "cone":
        x = _images(c["n"], seed, (c["batch"] + 1) // 2, nz=c["nz"])
        return _cone_exact(c, x.reshape(-1, c["nz"], c["n"], c["n"])[:c["batch"]])
    return _cnn_exact(c, seed)
