"""The calls of this framework whose speed and accuracy are watched.

A case is one call, or one fitting step, through the public entry points of
paper_2401_12724_gb300.api, with inputs drawn on the GPU from a seed: hit
records with the distributions of the package's synthetic workloads (h, u, v
uniform, omega_i about the yarn normal, omega_o uniform on the sphere,
log-uniform footprints), materials over the same parameter ranges, and camera
rays over a plain-weave patch.

exact() evaluates the same model in float64 with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2401_12724_gb300 import api

DEV = "cuda"
F32 = np.float32
PI = math.pi

# Scalars of a material that the workloads leave at their defaults, as the
# float32 values the library receives.
DEFAULTS = dict(yarn_radius=1.0, eta=1.55, k_spec=1.0, body_B=0.5, body_r=0.5, sigma_t=0.5,
                shadow_density=1.0, packing=0.8, map_texels=256, trace_iters=5, k_max=16, flags=0)

EVAL_OPS = ("eval", "pdf", "sample", "fused")
FIT_OPS = ("fit", "fit_l2", "fit_directions")


# ------------------------------------------------------------------- cases --
def _case(name, op, n, materials, **over):
    c = dict(name=name, op=op, n=n, materials=materials, sorted=False, footprint=False,
             maps=1, stochastic=False, deterministic=False)
    c.update(over)
    return c


def listed():
    return [
        # one render bucket of an interactive preview: launch and latency
        _case("bucket", "fused", 1009, 8),
        # the near-field evaluation batch of a single-yarn preview
        _case("near_eval", "eval", 65536, 1),
        # one bounce of a wavefront path tracer: directions to continue with
        _case("bounce", "sample", 1000003, 8),
        # light sampling and continuation of a whole wavefront in one call
        _case("wavefront", "fused", 1 << 24, 8),
        # cloth seen from afar: footprints from a fraction of a yarn to many
        _case("multiscale", "fused", 1 << 22, 8, footprint=True),
        # the Monte Carlo estimators of the same records (a reference render)
        _case("stochastic", "eval", (1 << 20) + 7, 8, footprint=True, stochastic=True),
        # hairy yarns whose fibers migrate between the ply's surface and core
        _case("migrating", "eval", (1 << 21) - 1, 8, maps=2),
        # a scene of many yarn types, records binned by type, skewed counts
        _case("many_yarns", "fused", 1 << 26, 256, sorted=True),
        # one step of fitting 64 yarns to captured radiance (L2 loss)
        _case("fit_l2", "fit_l2", 1 << 24, 64, sorted=True),
        # a mini-batch fitting step under a loss of the caller's own
        _case("fit_batch", "fit", 200003, 8),
        # inverse rendering: the extended parameter set and both directions
        _case("fit_directions", "fit_directions", 1 << 21, 8),
        # camera rays with differentials over a woven patch
        dict(name="camera", op="trace", width=2048, height=2048, yarns=16, pieces=16,
             differentials=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["eval", "pdf", "sample", "fused", "fused", "fit", "fit_l2",
                     "fit_directions", "trace"])
    if op == "trace":
        return dict(op=op, width=_log_int(rng, 40, 2048), height=_log_int(rng, 40, 2048),
                    yarns=rng.randint(2, 32), pieces=rng.randint(4, 32),
                    differentials=rng.random() < 0.5)
    footprint = rng.random() < 0.35
    order = rng.random() < 0.4
    maps = rng.choice([1, 1, 1, 2])
    stochastic = op in ("eval", "fused") and rng.random() < 0.3
    top = {"fit": 1 << 23, "fit_l2": 1 << 23, "fit_directions": 1 << 21}.get(op, 1 << 25)
    if footprint:
        top >>= 3
    if stochastic:
        top = min(top, 1 << 21)
    c = dict(op=op, n=_log_int(rng, 1000, top),
             materials=rng.randint(1, 256) if order else rng.randint(1, 20 if maps == 1 else 9),
             sorted=order, footprint=footprint, maps=maps, stochastic=stochastic,
             deterministic=order and op in FIT_OPS and rng.random() < 0.5)
    return c


# ------------------------------------------------------------------ inputs --
def _f(x):
    return float(F32(x))


def _descs(case, seed):
    g = np.random.RandomState((seed * 9176 + 11) % (1 << 32))
    out = []
    for _ in range(case["materials"]):
        d = {k: (v if isinstance(v, int) else _f(v)) for k, v in DEFAULTS.items()}
        beta = _f(g.uniform(5.0, 20.0))
        d.update(n_plies=int(g.randint(2, 6)), fibers_per_ply=int(g.randint(32, 129)),
                 ply_twist_deg=_f(g.uniform(10.0, 45.0)),
                 fiber_twist_deg=_f(g.uniform(10.0, 45.0)), beta_deg=[beta, beta],
                 albedo=[_f(a) for a in g.uniform(0.1, 0.95, 3)])
        if case["maps"] > 1:
            d.update(migration_maps=case["maps"], migration_seed=int(g.randint(0, 1 << 16)),
                     migration_length=1.5, migration_blend=0.25)
        out.append(d)
    return out


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _planes(g, n, k, lo=0.0, hi=1.0):
    x = torch.rand((k, n) if k > 1 else (n,), generator=g, device=DEV, dtype=torch.float32)
    return x * (hi - lo) + lo if (lo, hi) != (0.0, 1.0) else x


def _sphere(g, n):
    z = 1.0 - 2.0 * _planes(g, n, 1)
    phi = (2.0 * PI) * _planes(g, n, 1)
    r = (1.0 - z * z).clamp_(min=0.0).sqrt_()
    return torch.stack([r * phi.cos(), r * phi.sin(), z])


def _about_normal(g, n, u):
    """Cosine-distributed directions about the yarn normal at azimuth u."""
    a, phi = _planes(g, n, 1), (2.0 * PI) * _planes(g, n, 1)
    lt, lb, ln = a.sqrt() * phi.cos(), a.sqrt() * phi.sin(), (1.0 - a).sqrt()
    return torch.stack([ln * u.cos() - lb * u.sin(), ln * u.sin() + lb * u.cos(), lt])


def _offsets(case, seed):
    """First record of each material: skewed (Zipf) counts in a drawn order."""
    m, n = case["materials"], case["n"]
    g = np.random.RandomState((seed * 7919 + 5) % (1 << 32))
    w = 1.0 / np.arange(1, m + 1) ** 1.1
    if case["op"] in FIT_OPS:
        w = np.ones(m)
    c = np.floor(g.permutation(w / w.sum()) * n).astype(np.int64)
    c[int(g.randint(0, m))] += n - int(c.sum())
    return np.concatenate([[0], np.cumsum(c)]).astype(np.int64)


def _records(case, seed):
    n, g = case["n"], _gen(seed)
    r = dict(h=_planes(g, n, 1, -1.0, 1.0), u=_planes(g, n, 1, 0.0, 2.0 * PI),
             # a captured stretch of yarn when fitting, a length of it otherwise
             v=_planes(g, n, 1, 0.0, 10.0 if case["op"] in FIT_OPS else 100.0))
    r["wi"] = _about_normal(g, n, r["u"])
    r["wo"] = _sphere(g, n)
    r["u0"], r["u1"] = _planes(g, n, 1), _planes(g, n, 1)
    if case["footprint"]:
        r["ratio"] = _planes(g, n, 1, math.log(0.01), math.log(100.0)).exp_()
    if case["sorted"]:
        offs = torch.from_numpy(_offsets(case, seed)).to(DEV)
        r["seg_offsets"] = offs
        r["mat_id"] = torch.repeat_interleave(
            torch.arange(case["materials"], device=DEV, dtype=torch.int32), offs.diff())
    else:
        r["mat_id"] = torch.randint(0, case["materials"], (n,), generator=g, device=DEV,
                                    dtype=torch.int32)
    if case["op"] == "fit_l2":
        r["target"] = _planes(g, n, 3)
    elif case["op"] in FIT_OPS:
        r["grad"] = _planes(g, n, 3, -1.0, 1.0)
    return r


def _scene(case, seed):
    """A plain weave of straight pieces, and camera rays over it."""
    g = np.random.RandomState((seed * 31 + 3) % (1 << 32))
    ny, npc, spacing = case["yarns"], case["pieces"], 2.5
    lift = g.uniform(0.5, 0.7)
    pieces = []
    for axis in (0, 1):
        for j in range(ny):
            mat, v0 = int(g.randint(0, 8)), 0.0
            for k in range(npc):
                p = np.zeros((2, 3))
                p[:, axis] = [k * spacing, (k + 1) * spacing]
                p[:, 1 - axis] = (j + 0.5) * spacing
                up = [lift if (i + j + axis) % 2 == 0 else -lift for i in (k, k + 1)]
                p[:, 2] = up
                d = p[1] - p[0]
                length = float(np.linalg.norm(d))
                t = d / length
                nr = np.array([0.0, 0.0, 1.0]) - t * t[2]
                nr /= np.linalg.norm(nr)
                pieces.append(dict(p0=p[0].tolist(), t=t.tolist(), n_ref=nr.tolist(),
                                   length=length, radius=1.0, v0=v0, mat_id=mat))
                v0 += length
    w, h = case["width"], case["height"]
    extent = max(ny, npc) * spacing
    tan_h = math.tan(math.radians(15.0))
    el = math.radians(55.0)
    c = np.array([npc, ny, 0.0]) * spacing / 2
    eye = c + 0.4 * extent / tan_h * np.array([0.0, -math.cos(el), math.sin(el)])
    fwd = (c - eye) / np.linalg.norm(c - eye)
    right = np.cross(fwd, [0.0, 0.0, 1.0])
    right /= np.linalg.norm(right)
    up = np.cross(right, fwd)
    gen = _gen(seed)
    px = torch.arange(w, device=DEV, dtype=torch.float64).repeat(h)
    py = torch.arange(h, device=DEV, dtype=torch.float64).repeat_interleave(w)
    px = px + _planes(gen, w * h, 1).double() - 0.5
    py = py + _planes(gen, w * h, 1).double() - 0.5

    def dirs(off):
        sx = ((px + 0.5 + off) / w * 2 - 1) * tan_h
        sy = (1 - (py + 0.5 + off) / h * 2) * tan_h * h / w
        d = torch.stack([fwd[i] + right[i] * sx + up[i] * sy for i in range(3)])
        return (d / d.norm(dim=0)).float()

    o = torch.from_numpy(eye).to(DEV).float()[:, None].expand(3, w * h).contiguous()
    rays = dict(o=o, d=dirs(0.0))
    if case["differentials"]:
        rays.update(o1=o, d1=dirs(0.5), o2=o, d2=dirs(-0.5))
    a = g.uniform(0.2, 1.2)
    light = [_f(math.cos(a) * 0.6), _f(math.sin(a) * 0.6), _f(0.8)]
    return pieces, rays, light


def _params(descs, columns):
    rows = []
    for d in descs:
        al = list(d["albedo"])
        r = al + [math.radians(d["beta_deg"][0]), math.radians(d["beta_deg"][1]),
                  math.radians(d["ply_twist_deg"]), math.radians(d["fiber_twist_deg"]),
                  d["shadow_density"]]
        rows.append((r + [d["body_r"]] + al + [d["sigma_t"], d["body_B"], d["k_spec"]])[:columns])
    return torch.tensor(rows, dtype=torch.float64).float().to(DEV)


# ------------------------------------------------------------ prepare, run --
def prepare(case, seed):
    op = case["op"]
    if op == "trace":
        pieces, rays, light = _scene(case, seed)
        return dict(case=case, yarns=api.yarns_to_device(pieces), rays=rays, light=light)
    descs = _descs(case, seed)
    rec = _records(case, seed)
    s = dict(case=case, mats=api.Materials(descs), seed=int(seed))
    if op in FIT_OPS:
        s["params"] = _params(descs, 15 if op == "fit_directions" else 8).requires_grad_()
        s["grad"], s["target"] = rec.pop("grad", None), rec.pop("target", None)
        del rec["u0"], rec["u1"]
        if op == "fit_directions":
            s["wi"] = rec["wi"].clone().requires_grad_()
            s["wo"] = rec["wo"].clone().requires_grad_()
    s["rec"] = rec
    return s


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "trace":
        return api.trace_yarns(s["yarns"], s["rays"], s["light"])
    mats, rec, det = s["mats"], s["rec"], case["deterministic"]
    if op == "eval":
        if case["stochastic"]:
            return api.eval_stochastic(mats, rec, s["seed"], 3)
        return api.eval(mats, rec)
    if op == "pdf":
        return api.pdf(mats, rec)
    if op == "sample":
        return api.sample(mats, rec)
    if op == "fused":
        if case["stochastic"]:
            return api.eval_sample_pdf_stochastic(mats, rec, s["seed"], 3)
        return api.eval_sample_pdf(mats, rec)
    p = s["params"]
    p.grad = None
    if op == "fit_l2":
        loss = api.bysdf_l2_loss(p, mats, rec, s["target"], deterministic=det)
        loss.backward()
        return dict(loss=loss.detach(), grad=p.grad, appearance=p.grad[:, :5])
    if op == "fit":
        f, st = api.bysdf(p, mats, rec, det)
        f.backward(s["grad"])
        return dict(f=f.detach(), status=st, grad=p.grad, appearance=p.grad[:, :5])
    s["wi"].grad = s["wo"].grad = None
    f, st = api.bysdf_ext(p, s["wi"], s["wo"], mats, rec, det)
    f.backward(s["grad"])
    return dict(f=f.detach(), status=st, grad=p.grad, appearance=p.grad[:, :5], wi=s["wi"].grad,
                wo=s["wo"].grad)


# -------------------------------------------------------------------- work --
# Arithmetic of one record (adds, multiplies, divisions, roots and
# transcendental calls of the model's formulas, averaged over the workloads):
# an evaluation, an evaluation with a sample, their share per footprint node,
# and a reverse sweep over the evaluation.
_FLOPS = dict(eval=550.0, pdf=530.0, sample=700.0, fused=790.0, fit=2500.0, fit_l2=2000.0,
              fit_directions=2500.0, trace=300.0)


def work(case):
    op = case["op"]
    if op == "trace":
        n = case["width"] * case["height"]
        return dict(bytes=n * ((72 if case["differentials"] else 24) + 56), flops=n * _FLOPS[op])
    n = case["n"]
    read = 4 * (3 + 3) + 4 * (not case["sorted"]) + 4 * case["footprint"]  # h u v wi id ratio
    read += {"eval": 12, "pdf": 12, "sample": 8, "fused": 20}.get(op, 24)  # wo, u0 u1, or wo + 3
    wrote = {"eval": 17, "pdf": 5, "sample": 29, "fused": 46, "fit_l2": 0, "fit": 13,
             "fit_directions": 37}[op]
    return dict(bytes=n * (read + wrote), flops=n * _FLOPS[op] * (5.0 if case["footprint"] else 1.0))


# ------------------------------------------------------- the model, float64 --
def _layout(d, k=0):
    """Ply and fiber layout; k: the ring of migration map k."""
    R = d["yarn_radius"]
    s = math.sin(PI / d["n_plies"])
    Rc, Rp = (R / (1 + s), R * s / (1 + s)) if d["n_plies"] > 1 else (0.0, R)
    rf = Rp * math.sqrt(d["packing"] / d["fibers_per_ply"])
    Rfc = Rp - rf - k * rf / d.get("migration_maps", 1)
    return Rp, Rc, rf, Rfc, math.ceil(PI / math.asin(rf / Rfc))


def _maps(d, k):
    """Fiber normal deviation and occluded share of the half-plane, T texels."""
    _, _, rf, Rfc, M = _layout(d, k)
    T = d["map_texels"]
    D = ((np.arange(T) + 0.5) / T - 0.5) * 2 * PI / M
    s = Rfc * np.sin(D)
    c = np.sqrt(np.maximum(rf * rf - s * s, 0.0))
    rho = Rfc * np.cos(D) + c
    px, py = rho * np.cos(D), rho * np.sin(D)
    phin = np.arctan2(py, px - Rfc)
    a = 2 * PI * np.arange(1, M) / M
    wx, wy = Rfc * np.cos(a)[None] - px[:, None], Rfc * np.sin(a)[None] - py[:, None]
    dist = np.hypot(wx, wy)
    half = np.where(dist > rf, np.arcsin(np.minimum(rf / dist, 1.0)), PI / 2)
    mid = np.remainder(np.arctan2(wy, wx) - phin[:, None] + PI, 2 * PI) - PI
    sh = 2 * PI * np.array([-1.0, 0.0, 1.0])
    lo = np.maximum((mid - half)[..., None] + sh, -PI / 2).reshape(T, -1)
    hi = np.minimum((mid + half)[..., None] + sh, PI / 2).reshape(T, -1)
    hi = np.maximum(hi, lo)
    order = np.argsort(lo, axis=1)
    lo, hi = np.take_along_axis(lo, order, 1), np.take_along_axis(hi, order, 1)
    reach = np.maximum.accumulate(np.concatenate([np.full((T, 1), -PI / 2), hi], 1), 1)[:, :-1]
    covered = np.maximum(hi - np.maximum(lo, reach), 0.0).sum(1)
    return np.arctan2(s, c), covered / PI


_M0, _M1 = 0xD2E7470EE14C6C93, 0xCA5A826395121157
_W0, _W1 = 0x9E3779B97F4A7C15, 0xBB67AE8584CAA73B


def _mulhi(a, b):
    """High 64 bits of a (Python int) times b (uint64 array)."""
    m = np.uint64(0xFFFFFFFF)
    s = np.uint64(32)
    al, ah = np.uint64(a & 0xFFFFFFFF), np.uint64(a >> 32)
    bl, bh = b & m, b >> s
    t = al * bl
    x = ah * bl + (t >> s)
    y = al * bh + (x & m)
    return ah * bh + (x >> s) + (y >> s)


def _philox(c0, c1, k0, k1):
    """Philox4x64-10 words of the counters (c0, c1, 0, 0) (Salmon et al. 2011)."""
    one = np.uint64(0xFFFFFFFFFFFFFFFF)
    x0 = np.asarray(c0, np.uint64)
    x1 = np.full_like(x0, c1)
    x2, x3 = np.zeros_like(x0), np.zeros_like(x0)
    with np.errstate(over="ignore"):
        for r in range(10):
            h0, l0 = _mulhi(_M0, x0), np.uint64(_M0) * x0
            h1, l1 = _mulhi(_M1, x2), np.uint64(_M1) * x2
            x0, x1, x2, x3 = (h1 ^ x1 ^ np.uint64((k0 + r * _W0) & int(one)), l1,
                              h0 ^ x3 ^ np.uint64((k1 + r * _W1) & int(one)), l0)
    return x0, x1, x2, x3


def _unit(w):
    return torch.from_numpy((w >> np.uint64(40)).astype(np.float64) * 2.0 ** -24).to(DEV)


def _tables(descs):
    """Per-material constants and maps as float64 tensors."""
    K = max(d.get("migration_maps", 1) for d in descs)
    t = {}
    col = lambda key: torch.tensor([float(d[key]) for d in descs], dtype=torch.float64).to(DEV)  # noqa: E731
    for key in ("yarn_radius", "eta", "n_plies"):
        t[key] = col(key)
    lay = [[_layout(d, k) for k in range(K)] for d in descs]
    t["Rp"] = torch.tensor([x[0][0] for x in lay], dtype=torch.float64).to(DEV)
    t["Rc"] = torch.tensor([x[0][1] for x in lay], dtype=torch.float64).to(DEV)
    t["Rfc"] = torch.tensor([[y[3] for y in x] for x in lay], dtype=torch.float64).to(DEV)
    t["M"] = torch.tensor([[float(y[4]) for y in x] for x in lay], dtype=torch.float64).to(DEV)
    m = np.array([[_maps(d, k) for k in range(K)] for d in descs])  # materials, K, 2, T
    t["maps"] = torch.from_numpy(m).to(DEV)
    if K > 1:
        pick = [(_philox(np.arange(256), 0, d["migration_seed"], 0xB15DF000F1BE0002)[0]
                 % np.uint64(K)).astype(np.int64) for d in descs]
        t["segments"] = torch.from_numpy(np.array(pick)).to(DEV)
        t["length"], t["blend"] = col("migration_length"), col("migration_blend")
    t["K"], t["plies"] = K, int(t["n_plies"].max())
    t["iters"], t["texels"] = descs[0]["trace_iters"], descs[0]["map_texels"]
    t["k_max"] = descs[0]["k_max"]
    return t


def _root(x, ok):
    """sqrt(x) where ok, with no infinite or undefined derivative elsewhere."""
    return torch.where(ok, x, torch.ones_like(x)).sqrt()


def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


def _cross(a, b):
    return (a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0])


def _scale(a, s):
    return tuple(x * s for x in a)


def _add(a, b):
    return tuple(x + y for x, y in zip(a, b))


def _pick(c, a, b):
    return tuple(torch.where(c, x, y) for x, y in zip(a, b))


def _node(t, m, P, q, X0, e, kappa, w2):
    """One footprint node: hit flag, ply count, hit point, fiber normal and
    tangent, and shadowing."""
    Rp, Rc, plies = t["Rp"][m], t["Rc"][m], t["n_plies"][m]
    omega_p = torch.tan(P[5]) / Rc
    ex, ey = e

    def update(k, tt, om, kap):
        psi = 2 * PI * k / plies + om * (q["v"] + kap * tt)
        cx, cy = Rc * psi.cos(), Rc * psi.sin()
        qx, qy = X0[0] - cx, X0[1] - cy
        b = qx * ex + qy * ey
        disc = b * b - (qx * qx + qy * qy - Rp * Rp)
        return psi, cx, cy, b, disc

    with torch.no_grad():
        best = torch.full_like(m, -1)
        best_t = torch.full_like(Rp, math.inf)
        count = torch.zeros_like(Rp)
        for k in range(t["plies"]):
            tt, hit = torch.zeros_like(Rp), plies > k
            for _ in range(t["iters"]):
                _, _, _, b, disc = update(k, tt, omega_p.detach(), kappa.detach())
                hit = hit & (disc >= 0)
                tt = (-b - disc.clamp(min=0).sqrt()).clamp(min=0)
            nearer = hit & (tt < best_t)
            best, best_t = torch.where(nearer, k, best), torch.where(nearer, tt, best_t)
            count = count + hit
        hit = best >= 0
        kf = best.clamp(min=0).double()
    tt = torch.zeros_like(Rp)
    for _ in range(t["iters"]):
        psi, cx, cy, b, disc = update(kf, tt, omega_p, kappa)
        tt = (-b - _root(disc, hit & (disc > 0))).clamp(min=0)
    xx, xy = X0[0] + tt * ex, X0[1] + tt * ey
    z = q["v"] + kappa * tt
    dx, dy = xx - cx, xy - cy
    dl = (dx * dx + dy * dy).sqrt()
    zero = torch.zeros_like(Rp)
    n_p = (dx / dl, dy / dl, zero)
    raw = (-omega_p * xy, omega_p * xx, torch.ones_like(Rp))
    raw = _add(raw, _scale(n_p, -_dot(raw, n_p)))
    t_p = _scale(raw, 1 / _dot(raw, raw).sqrt())
    e_p = _cross(t_p, n_p)
    cp, sp = psi.cos(), psi.sin()
    u_ply = torch.atan2(cp * n_p[1] - sp * n_p[0], cp * n_p[0] + sp * n_p[1])

    def lookup(k):
        M, Rfc = t["M"][m, k], t["Rfc"][m, k]
        w = (u_ply - torch.tan(P[6]) / Rfc * z) * (M / (2 * PI))
        a = w + 0.5 - (w.detach() + 0.5).floor()
        tau = a * t["texels"] - 0.5
        fl = tau.detach().floor()
        f = tau - fl
        i0 = fl.long() % t["texels"]
        i1 = (i0 + 1) % t["texels"]
        mp = t["maps"]
        return [(1 - f) * mp[m, k, c, i0] + f * mp[m, k, c, i1] for c in (0, 1)]

    if t["K"] == 1:
        delta, of = lookup(torch.zeros_like(m))
    else:
        y = z / t["length"][m]
        sf = y.detach().floor()
        a, bl, seg = y - sf, t["blend"][m], sf.long()
        low, high = a < bl, a > 1 - bl
        wgt = torch.where(low, 0.5 - a / (2 * bl),
                          torch.where(high, 0.5 - (1 - a) / (2 * bl), zero))
        nb = torch.where(low, seg - 1, torch.where(high, seg + 1, seg))
        d0, o0 = lookup(t["segments"][m, seg % 256])
        d1, o1 = lookup(t["segments"][m, nb % 256])
        delta, of = (1 - wgt) * d0 + wgt * d1, (1 - wgt) * o0 + wgt * o1
    t_f = _add(_scale(t_p, P[6].cos()), _scale(e_p, P[6].sin()))
    n_f = _add(_scale(n_p, delta.cos()), _scale(_cross(t_f, n_p), delta.sin()))
    occ = zero
    for j in range(1, t["plies"]):
        ps = psi + 2 * PI * j / plies
        qx, qy = xx - Rc * ps.cos(), xy - Rc * ps.sin()
        b = qx * w2[0] + qy * w2[1]
        disc = b * b - (qx * qx + qy * qy - Rp * Rp)
        sq = _root(disc, disc > 0)
        far = sq - b
        chord = far - (-b - sq).clamp(min=0)
        occ = occ + torch.where((disc > 0) & (far > 0) & (plies > j), chord, zero)
    return hit, count, (xx, xy, z), n_f, t_f, torch.exp(-P[7] * (occ / (2 * Rp) + of))


def _fresnel(c, eta):
    s2 = (1 - c * c) / (eta * eta)
    ok = s2 < 1
    ct = _root(1 - s2, ok)
    rs, rp = (c - eta * ct) / (c + eta * ct), (eta * c - ct) / (eta * c + ct)
    return torch.where(ok, 0.5 * (rs * rs + rp * rp), torch.ones_like(c))


def _ggx_d(h, at, ab):
    q = h[0] * h[0] / (at * at) + h[1] * h[1] / (ab * ab) + h[2] * h[2]
    q = torch.where(h[2] > 0, q, torch.ones_like(q))
    return torch.where(h[2] > 0, 1 / (PI * at * ab * q * q), torch.zeros_like(q))


def _ggx_g1(w, wm, at, ab):
    an = w[2].abs()
    on = wm * w[2] > 0
    r = _root(an * an + at * at * w[0] * w[0] + ab * ab * w[1] * w[1], on)
    return torch.where(on, 2 * an / (an + r), torch.zeros_like(r))


def _vndf(w, at, ab, u0, u1):
    """A GGX visible normal (Heitz 2018)."""
    V = (at * w[0], ab * w[1], w[2])
    V = _scale(V, 1 / _dot(V, V).sqrt())
    ls = V[0] * V[0] + V[1] * V[1]
    il = 1 / _root(ls, ls > 0)
    zero = torch.zeros_like(ls)
    T1 = _pick(ls > 0, (-V[1] * il, V[0] * il, zero), (zero + 1, zero, zero))
    T2 = _cross(V, T1)
    r, phi = u0.sqrt(), 2 * PI * u1
    t1, t2 = r * phi.cos(), r * phi.sin()
    s = 0.5 * (1 + V[2])
    t2 = (1 - s) * (1 - t1 * t1).sqrt() + s * t2
    tz = (1 - t1 * t1 - t2 * t2).clamp(min=0).sqrt()
    N = _add(_add(_scale(T1, t1), _scale(T2, t2)), _scale(V, tz))
    N = (at * N[0], ab * N[1], N[2].clamp(min=0))
    return _scale(N, 1 / _dot(N, N).sqrt())


def _local(w, t, b, n):
    return (_dot(w, t), _dot(w, b), _dot(w, n))


def _geometry(t, m, P, q, wi, jitter):
    h, u = q["h"], q["u"]
    zero = torch.zeros_like(h)
    g0 = torch.asin(h)
    e = (-(u - g0).cos(), -(u - g0).sin())
    l = (wi[0] * wi[0] + wi[1] * wi[1]).sqrt()
    ok = l >= 1e-7
    l = torch.where(ok, l, torch.ones_like(l))
    kappa, w2 = -wi[2] / l, (wi[0] / l, wi[1] / l)
    R = t["yarn_radius"][m]
    if "ratio" in q:
        # the node count is an integer that float32 arithmetic decides
        h32, r32 = h.float(), q["ratio"].float()
        h1 = (h32 - r32).clamp(min=-1.0)
        wd = (h32 + r32).clamp(max=1.0) - h1
        K = torch.ceil(wd * (0.5 * t["k_max"])).clamp(1, t["k_max"])
        h1, wd, K = h1.double(), wd.double(), K.double()
        top = int(K.max())
    else:
        h1, wd, K, top = h, zero, zero + 1, 1
    ns, ts, xs = [(zero, zero, zero)] * 3
    gs, nis, nhit = zero, zero, zero
    for j in range(top):
        x = 0.5 if jitter is None else jitter(j)
        uj = (u - g0) + torch.asin((h1 + (j + x) * wd / K).clamp(-1.0, 1.0))
        hit, ni, xp, nf, tf, g = _node(t, m, P, q, (R * uj.cos(), R * uj.sin()), e, kappa, w2)
        hit = hit & ok & (K > j)
        sel = lambda a, s: torch.where(hit, s + a, s)  # noqa: E731
        ns, ts, xs = [tuple(sel(a, s) for a, s in zip(v, w)) for v, w in
                      ((nf, ns), (tf, ts), (xp, xs))]
        gs, nis, nhit = sel(g, gs), sel(ni, nis), nhit + hit
    inv = 1 / nhit.clamp(min=1)
    nn = _dot(ns, ns)
    fine = (nhit > 0) & (nn.sqrt() > 1e-9 * nhit)
    n = _scale(ns, 1 / _root(nn, fine))
    tp = _add(ts, _scale(n, -_dot(ts, n)))
    tt = _dot(tp, tp)
    fine = fine & (tt.sqrt() > 1e-9 * nhit)
    return fine, n, _scale(tp, 1 / _root(tt, fine)), _scale(xs, inv), gs * inv, nis * inv, wd


def _model(t, m, P, q, wi, wo, sample, entry=None, jitter=None):
    """f, pdf and a sample of a batch; P: the 15 parameters per record."""
    hit, n, tn, x, G, ni, wd = _geometry(t, m, P, q, wi, jitter)
    eta, R = t["eta"][m], t["yarn_radius"][m]
    zero = torch.zeros_like(G)
    b = _cross(n, tn)
    flip = _dot(wi, n) < 0
    sg = torch.where(flip, -torch.ones_like(G), torch.ones_like(G))
    n, b = _scale(n, sg), _scale(b, sg)
    mui = _dot(wi, n)
    lit = hit & (mui > 0)
    mu = torch.where(lit, mui, torch.ones_like(mui))
    at, ab = (P[3] + wd / 2).clamp(1e-3, 1.5), (P[4] + wd / 2).clamp(1e-3, 1.5)
    B, r, ks = P[13], P[8], (1 - P[13]) * P[14]
    fr = _fresnel(mui, eta)
    # transmission path: refraction at x, exit at y
    mn, ci, Fe = n, mui, fr
    if entry is not None:
        ml = _vndf(_local(wi, tn, b, n), at, ab, *entry)
        mn = _add(_add(_scale(tn, ml[0]), _scale(b, ml[1])), _scale(n, ml[2]))
        ci = _dot(wi, mn)
        Fe = _fresnel(ci, eta)
    s2 = (1 - ci * ci) / (eta * eta)
    ok = lit & (ci > 0) & (s2 < 1)
    ct = _root(1 - s2, ok)
    din = _add(_scale(wi, -1 / eta), _scale(mn, ci / eta - ct))
    ok = ok & (_dot(din, n) < 0)
    a = din[0] * din[0] + din[1] * din[1]
    ok = ok & (a > 1e-12)
    a = torch.where(ok, a, torch.ones_like(a))
    bq = x[0] * din[0] + x[1] * din[1]
    disc = bq * bq - a * (x[0] * x[0] + x[1] * x[1] - R * R)
    sy = ((torch.where(disc > 0, _root(disc, ok & (disc > 0)), zero) - bq) / a).clamp(min=0)
    yx, yy = x[0] + din[0] * sy, x[1] + din[1] * sy
    il = 1 / _root(yx * yx + yy * yy, ok)
    ny = (yx * il, yy * il, zero)
    tz = (zero, zero, zero + 1)
    by = _cross(ny, tz)
    iy = _scale(din, -1.0)
    tau = torch.exp(-P[12] * ni * sy)

    def lobes(w):
        muo = _dot(w, n)
        up, dn = lit & (muo > 0), lit & (muo < 0)
        # reflection at x (Eq. 2) and the body lobe of its side (Eq. 5)
        h = _add(wi, w)
        hh = _dot(h, h)
        h = _scale(h, 1 / _root(hh, up & (hh > 0)))
        ih = _dot(wi, h)
        D = _ggx_d(_local(h, tn, b, n), at, ab)
        gi = _ggx_g1(_local(wi, tn, b, n), ih, at, ab)
        go = _ggx_g1(_local(w, tn, b, n), _dot(w, h), at, ab)
        base = gi * D / (4 * mu)
        F = _fresnel(torch.where(up, ih, torch.ones_like(ih)), eta)
        fR = torch.where(up, ks * F * go * base, zero)
        pR = torch.where(up, base, zero)
        al = 0.5 * (1 - mu * torch.log(1 + 1 / mu))
        mo = torch.where(up, muo, torch.ones_like(muo))
        br = (1 / (4 * PI * (mu + mo)) + 1 / PI) / (1 + al) * mo
        body_x = torch.where(up, r * B * G * br, zero)
        body_y = torch.where(dn, (1 - r) * B * G * (-muo) / PI, zero)
        # transmission (Eq. 3): the exit at y, times entry and tau^N
        ion, oon = _dot(iy, ny), _dot(w, ny)
        go_on = dn & ok & (ion < 0) & (oon > 0)
        ht = _scale(_add(_scale(iy, eta), w), -1.0)
        h2 = _dot(ht, ht)
        ht = _scale(ht, 1 / _root(h2, go_on & (h2 > 0)))
        sgn = torch.where(_dot(ht, ny) < 0, -torch.ones_like(G), torch.ones_like(G))
        ht = _scale(ht, sgn)
        ih, oh = _dot(iy, ht), _dot(w, ht)
        go_on = go_on & (ih < 0) & (oh > 0)
        one = torch.ones_like(G)
        ihs, ohs = torch.where(go_on, ih, -one), torch.where(go_on, oh, one)
        den = torch.where(go_on, eta * ihs + ohs, one)
        D = _ggx_d(_local(ht, tz, by, ny), at, ab)
        gi = _ggx_g1(_local(iy, tz, by, ny), ihs, at, ab)
        go = _ggx_g1(_local(w, tz, by, ny), ohs, at, ab)
        base = gi * -ihs * D * ohs / (torch.where(go_on, -ion, one) * den * den)
        Fy = _fresnel(-ihs, 1 / eta)
        fT = torch.where(go_on, ks * (1 - Fe) * tau * (1 - Fy) * go * base, zero)
        pT = torch.where(go_on, base, zero)
        f = [fR + fT + P[c] * body_x + P[9 + c] * body_y for c in range(3)]
        pdf = ((1 - B) * fr * pR + (1 - B) * (1 - fr) * pT
               + B * r * torch.where(up, muo / PI, zero)
               + B * (1 - r) * torch.where(dn, -muo / PI, zero))
        f = torch.stack([torch.where(hit, c, zero) for c in f])
        return f, torch.where(hit, pdf, zero)

    out = dict(hit=hit)
    if wo is not None:
        out["f"], out["pdf"] = lobes(wo)
    if not sample:
        return out
    u0, u1 = q["u0"], q["u1"]
    c = [(1 - B) * fr, (1 - B) * (1 - fr), B * r, B * (1 - r)]
    e0, e1, e2 = c[0], c[0] + c[1], c[0] + c[1] + c[2]
    lobe = (u0 >= e0).long() + (u0 >= e1) + (u0 >= e2)
    lo = torch.where(lobe == 0, zero, torch.where(lobe == 1, e0, torch.where(lobe == 2, e1, e2)))
    pk = torch.where(lobe == 0, c[0], torch.where(lobe == 1, c[1],
                                                 torch.where(lobe == 2, c[2], c[3])))
    ur = torch.where(pk > 0, (u0 - lo) / pk, zero).clamp(0.0, 1 - 1e-12)
    ml = _vndf(_local(wi, tn, b, n), at, ab, ur, u1)
    mw = _add(_add(_scale(tn, ml[0]), _scale(b, ml[1])), _scale(n, ml[2]))
    w0 = _add(_scale(mw, 2 * _dot(wi, mw)), _scale(wi, -1.0))
    N = _scale(ny, -1.0)
    Bn = _cross(N, tz)
    ml = _vndf(_local(iy, tz, Bn, N), at, ab, ur, u1)
    mw = _add(_add(_scale(tz, ml[0]), _scale(Bn, ml[1])), _scale(N, ml[2]))
    cc = _dot(iy, mw)
    s2 = eta * eta * (1 - cc * cc)
    ok1 = ok & (cc > 0) & (s2 < 1)
    w1 = _add(_scale(iy, -eta), _scale(mw, eta * cc - _root(1 - s2, ok1)))
    w1 = _scale(w1, 1 / _dot(w1, w1).sqrt())
    rr, phi = ur.sqrt(), 2 * PI * u1
    zc = (1 - ur).clamp(min=0).sqrt() * torch.where(lobe == 2, 1.0, -1.0)
    w2 = _add(_add(_scale(tn, rr * phi.cos()), _scale(b, rr * phi.sin())), _scale(n, zc))
    good = torch.where(lobe == 0, _dot(w0, n) > 0,
                       torch.where(lobe == 1, ok1 & (_dot(w1, ny) > 0) & (_dot(w1, n) < 0),
                                   torch.ones_like(ok)))
    w = _pick(lobe == 0, w0, _pick(lobe == 1, w1, w2))
    f, pdf = lobes(w)
    miss = ~hit
    good = good & hit
    live = good & (pdf > 0)
    pick = lambda a, none: torch.where(miss, none, torch.where(live, a, zero))  # noqa: E731
    ip = 1 / torch.where(live, pdf, torch.ones_like(pdf))
    out["wo"] = torch.stack([torch.where(miss, -wi[k], torch.where(good, w[k], zero))
                             for k in range(3)])
    out["weight"] = torch.stack([pick(f[k] * ip, zero + 1) for k in range(3)])
    out["pdf_s"] = pick(pdf, zero)
    return out


def _chunks(n, size):
    return [(a, min(a + size, n)) for a in range(0, n, size)]


def _rand(case, seed, a, b):
    """The stochastic estimators' numbers of records a .. b - 1."""
    idx = np.arange(a, b, dtype=np.uint64)
    blocks = {}

    def words(k):
        if k not in blocks:
            blocks[k] = [_unit(w) for w in _philox(idx, k, int(seed), 0xB15DF0005EED0001)]
        return blocks[k]

    jitter = (lambda j: words(j // 4)[j % 4]) if case["footprint"] else None
    return words(16)[:2], jitter


def _exact_trace(case, seed):
    pieces, rays, light = _scene(case, seed)
    dev = dict(device=DEV, dtype=torch.float64)
    w32 = lambda x: [float(F32(v)) for v in x]  # noqa: E731
    fr = []
    for y in pieces:
        t, nr = np.array(w32(y["t"])), np.array(w32(y["n_ref"]))
        t = t / np.linalg.norm(t)
        nr = nr - t * (nr @ t)
        nr /= np.linalg.norm(nr)
        fr.append([*w32(y["p0"]), *t, *nr, *np.cross(t, nr), float(F32(y["length"])),
                   float(F32(y["radius"])), float(F32(y["v0"]))])
    fr = np.array(fr)
    outs = []
    n = case["width"] * case["height"]
    L = torch.tensor(light, **dev)
    for a, b in _chunks(n, 1 << 22):
        o, d = rays["o"][:, a:b].double(), rays["d"][:, a:b].double()
        best = torch.full((b - a,), -1, device=DEV, dtype=torch.int64)
        sb = torch.full((b - a,), math.inf, **dev)
        for k, y in enumerate(fr):
            p0, t, length, R = y[0:3], y[3:6], y[12], y[13]
            q = [o[i] - p0[i] for i in range(3)]
            qt, dt = _dot(q, t), _dot(d, t)
            qp = [q[i] - qt * t[i] for i in range(3)]
            dp = [d[i] - dt * t[i] for i in range(3)]
            aa, bb, cc = _dot(dp, dp), _dot(qp, dp), _dot(qp, qp) - R * R
            disc = bb * bb - aa * cc
            s = (-bb - disc.clamp(min=0).sqrt()) / aa
            w = qt + s * dt
            ok = (aa > 1e-24) & (cc > 0) & (disc >= 0) & (s > 0) & (w >= 0) & (w <= length)
            ok &= s < sb
            best, sb = torch.where(ok, k, best), torch.where(ok, s, sb)
        hit = best >= 0
        y = torch.from_numpy(fr).to(DEV)[best.clamp(min=0)].T
        p0, t, nr, br, R, v0 = y[0:3], y[3:6], y[6:9], y[9:12], y[13], y[14]
        s = torch.where(hit, sb, torch.zeros_like(sb))
        x = [o[i] + d[i] * s - p0[i] for i in range(3)]
        u = torch.atan2(_dot(x, br), _dot(x, nr))
        u = torch.where(u < 0, u + 2 * PI, u)

        def offset(o, d):
            q = [o[i] - p0[i] for i in range(3)]
            qn, qb, dn, db = _dot(q, nr), _dot(q, br), _dot(d, nr), _dot(d, br)
            return (qn * db - qb * dn) / ((dn * dn + db * db).sqrt() * R)

        h = offset(o, d).clamp(-1, 1)
        keep = lambda v: torch.where(hit, v, torch.zeros_like(v))  # noqa: E731
        r = dict(h=keep(h), u=keep(u), v=keep(v0 + _dot(x, t)), t_hit=s,
                 wi=torch.stack([keep(-_dot(d, f)) for f in (nr, br, t)]),
                 wo=torch.stack([keep(_dot([L[0], L[1], L[2]], f)) for f in (nr, br, t)]))
        r["ratio"] = torch.zeros_like(s)
        if case["differentials"]:
            hs = [(offset(rays["o" + c][:, a:b].double(), rays["d" + c][:, a:b].double())
                   - h).abs() for c in ("1", "2")]
            r["ratio"] = keep(torch.maximum(*hs))
        outs.append(r)
    out = {k: torch.cat([r[k] for r in outs], dim=-1) for k in outs[0]}
    return dict(out, mat_id=None, yarn_id=None)


def exact(case, seed):
    op = case["op"]
    if op == "trace":
        return _exact_trace(case, seed)
    n, descs = case["n"], _descs(case, seed)
    t, rec = _tables(descs), _records(case, seed)
    fit = op in FIT_OPS
    cols = {"fit_directions": 15, "fit": 8, "fit_l2": 8}.get(op, 15)
    p = _params(descs, cols).double()
    if not fit:
        # the descriptors' own angles, not their float32 radians
        for c, key in ((5, "ply_twist_deg"), (6, "fiber_twist_deg")):
            p[:, c] = torch.tensor([math.radians(d[key]) for d in descs], dtype=torch.float64)
    rest = _params(descs, 15).double()
    grad = torch.zeros_like(p)
    loss = 0.0
    got = {}
    size = (1 << 18) if fit else (1 << 21)
    if case["footprint"]:
        size >>= 2
    for a, b in _chunks(n, size):
        m = rec["mat_id"][a:b].long()
        q = {k: rec[k][a:b].double() for k in ("h", "u", "v", "u0", "u1", "ratio") if k in rec}
        wi, wo = rec["wi"][:, a:b].double(), rec["wo"][:, a:b].double()
        leaf = p.clone().requires_grad_(fit)
        full = leaf
        if cols == 8:  # both body colours are the albedo
            full = torch.cat([leaf, rest[:, 8:9], leaf[:, 0:3], rest[:, 12:]], dim=1)
        P = full[m].T
        if op == "fit_directions":
            wi, wo = wi.requires_grad_(), wo.requires_grad_()
        if fit:
            r = _model(t, m, P, q, tuple(wi), tuple(wo), False)
            f, hit = r["f"], r["hit"]
            r = {}
            if op == "fit_l2":
                # the loss runs over the records with a ply hit
                part = ((f - rec["target"][:, a:b].double()) ** 2 * hit).sum()
                part.backward()
                loss += part.detach()
            else:
                (f * rec["grad"][:, a:b].double()).sum().backward()
                r["f"] = f.detach()
            grad += leaf.grad
            if op == "fit_directions":
                r["wi"], r["wo"] = wi.grad, wo.grad
        else:
            with torch.no_grad():
                e, j = _rand(case, seed, a, b) if case["stochastic"] else (None, None)
                r = _model(t, m, P, q, tuple(wi), None if op == "sample" else tuple(wo),
                           op in ("sample", "fused"), e, j)
        for k, x in r.items():
            got.setdefault(k, []).append(x)
    o = {k: torch.cat(v, dim=-1) for k, v in got.items()}
    if op == "eval":
        return o["f"], o["pdf"], None
    if op == "pdf":
        return o["pdf"], None
    if op == "sample":
        return o["wo"], o["weight"], o["pdf_s"], None
    if op == "fused":
        return dict(f=o["f"], pdf=o["pdf"], status=None, wo=o["wo"], weight=o["weight"],
                    pdf_s=o["pdf_s"], lobe_status=None)
    # The helix angles' sums and the derivatives in omega_i hang on the few
    # records on a cusp of the fiber maps (a whole fiber's slope in one texel),
    # whose side the last bits of the fiber phase decide: no value in 64 bits
    # stands for what 32 bits give there.  The other parameters have one.
    out = dict(grad=None, appearance=grad[:, :5])
    if op == "fit_l2":
        return dict(out, loss=loss)
    out.update(f=o["f"], status=None)
    return dict(out, wi=None, wo=o["wo"]) if op == "fit_directions" else out

