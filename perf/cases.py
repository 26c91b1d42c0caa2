"""Performance cases of the thin-wire S-NFC solver: what its users have it do, over the real range.

Every case goes through the public entry points (paper_2410_03060_gb300.swm) on wire clouds of the
statistics the repository's workloads use (wavelength 1, radius 1e-3, lengths U[0.3, 0.6] cut into
segments of at most 0.08, random directions; Gaussian, uniform or clustered centres whose density
stays that of the workload as the cloud grows or shrinks).  Clouds are device tensors, as a program
that draws or transforms its clouds with torch holds them; incidence and observation lists are host
arrays, as the entry points take them.

The complex64 path computes in single precision and hands its results out in float64 containers;
a program that asked for that path keeps them as float32 / complex64, and so do these cases (its
outputs carry no more digits: the product form is timed per system shape, and forms sum in
different orders).  Results of the complex128 path stay float64 / complex128.
"""
import math
import weakref

import numpy as np
import torch

from paper_2410_03060_gb300 import swm

K0 = 2.0 * math.pi
TOL = 1e-6
MEAN_M = 5.13  # unknowns per wire for lengths U[0.3, 0.6] and segments of at most 0.08


def listed():
    return [
        # One small cloud on the float64 path: the call whose cost is launches and latency.
        dict(name="small_c128", path="run", cloud="cube8", nw=200, r_c=3.0, precision="c128", solver="gmres",
             n_inc=1, n_obs=360, currents=False),
        # A chaff cloud's bistatic pattern at one incidence, the ordinary interactive call.
        dict(name="bistatic_c64", path="run", cloud="gauss", nw=10000, r_c=3.0, precision="c64", solver="gmres",
             n_inc=1, n_obs=720, currents=False),
        # Entire coupling (every block kept), the reference that sparsified runs are judged by.
        dict(name="dense_c64", path="run", cloud="gauss", nw=1000, r_c=0.0, precision="c64", solver="gmres",
             n_inc=1, n_obs=360, currents=True),
        # One snapshot of a drifting cloud, monostatic at 1-degree steps (the batching workload).
        dict(name="snapshot_c64", path="run", cloud="cube", nw=24535, r_c=3.0, precision="c64", solver="gmres",
             n_inc=181, n_obs=0, currents=False),
        # A million wires, a monostatic cut at 5-degree steps: the headline workload.
        dict(name="million_c64", path="run", cloud="clusters", nw=1000000, r_c=3.0, precision="c64",
             solver="bicgstab", n_inc=37, n_obs=0, currents=True),
        # A large cloud at one incidence (the paper's sweeps of 1e5 and 1e6 chaffs).
        dict(name="large_one_c64", path="run", cloud="clusters", nw=400001, r_c=3.0, precision="c64",
             solver="gmres", n_inc=1, n_obs=360, currents=True),
        # The float64 path with several incidences: the accuracy reference of the fast path.
        dict(name="plain_c128", path="run", cloud="clusters", nw=10007, r_c=3.0, precision="c128", solver="gmres",
             n_inc=19, n_obs=0, currents=True),
        # A frequency sweep with the paper's GCR solver on one kept pattern.
        dict(name="sweep_gcr_c64", path="sweep", cloud="cube", nw=5001, r_c=3.0, n_freq=6, n_obs=361),
        # The operator and preconditioner of a Krylov loop driven by the caller (a cloud split over ranks).
        dict(name="operator_c128", path="operator", cloud="clusters", nw=50000, r_c=3.0, n_rhs=7),
        # RCS of given currents at many angles, float64 (post-processing of stored solutions).
        dict(name="far_field_c128", path="far", cloud="gauss", nw=10000, n_rhs=2, n_obs=361),
        # One gradient of the warm-start network (forward and backward) on a cloud's wires.
        dict(name="train_f32", path="train", cloud="gauss", nw=10000, r_c=3.0, n_inc=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["bistatic", "bistatic", "dense", "snapshot", "snapshot", "clusters", "large_one", "plain",
                       "sweep", "operator", "far", "train"])
    if path == "bistatic":
        return dict(path="run", cloud="gauss", nw=_log_int(rng, 300, 60000), r_c=3.0,
                    precision=rng.choice(["c64", "c64", "c128"]), solver="gmres", n_inc=rng.randint(1, 4),
                    n_obs=rng.randint(90, 720), currents=rng.random() < 0.5)
    if path == "dense":
        return dict(path="run", cloud="gauss", nw=_log_int(rng, 100, 1500), r_c=0.0, precision="c64", solver="gmres",
                    n_inc=rng.randint(1, 3), n_obs=rng.randint(90, 720), currents=True)
    if path == "snapshot":
        return dict(path="run", cloud="cube", nw=_log_int(rng, 2000, 50000), r_c=3.0, precision="c64",
                    solver=rng.choice(["gmres", "bicgstab"]), n_inc=rng.choice([13, 37, 91, 181, rng.randint(9, 181)]),
                    n_obs=0, currents=rng.random() < 0.5)
    if path == "clusters":
        return dict(path="run", cloud="clusters", nw=_log_int(rng, 50000, 900000), r_c=3.0, precision="c64",
                    solver="bicgstab", n_inc=rng.randint(9, 37), n_obs=0, currents=rng.random() < 0.5)
    if path == "large_one":
        return dict(path="run", cloud="clusters", nw=_log_int(rng, 100000, 1000000), r_c=3.0, precision="c64",
                    solver="gmres", n_inc=rng.randint(1, 2), n_obs=rng.randint(90, 720), currents=True)
    if path == "plain":
        return dict(path="run", cloud="clusters", nw=_log_int(rng, 1000, 30000), r_c=3.0, precision="c128",
                    solver=rng.choice(["gmres", "bicgstab"]), n_inc=rng.randint(9, 37), n_obs=0, currents=True)
    if path == "sweep":
        return dict(path="sweep", cloud="cube", nw=_log_int(rng, 1000, 50000), r_c=3.0, n_freq=rng.randint(3, 9),
                    n_obs=rng.randint(90, 720))
    if path == "operator":
        return dict(path="operator", cloud="clusters", nw=_log_int(rng, 3000, 200000), r_c=3.0,
                    n_rhs=rng.randint(1, 24))
    if path == "far":
        return dict(path="far", cloud="gauss", nw=_log_int(rng, 500, 60000), n_rhs=rng.randint(1, 4),
                    n_obs=rng.randint(37, 720))
    return dict(path="train", cloud="gauss", nw=_log_int(rng, 1000, 30000), r_c=3.0, n_inc=rng.randint(1, 3))


# ------------------------------------------------------------------------------ inputs
def _cloud(case, g):
    """Centres, directions, lengths, radii and segment counts as device tensors."""
    nw, f64 = case["nw"], dict(dtype=torch.float64, device="cuda")
    if case["cloud"] == "gauss":
        c = 30.0 * (nw / 1e4) ** (1 / 3) * torch.randn(nw, 3, generator=g, **f64)
    elif case["cloud"] == "clusters":
        scale = (nw / 1e6) ** (1 / 3)
        cc = 180.0 * scale * (2 * torch.rand(8, 3, generator=g, **f64) - 1)
        which = torch.randint(0, 8, (nw,), generator=g, device="cuda")
        c = cc[which] + 40.0 * scale * torch.randn(nw, 3, generator=g, **f64)
    else:  # uniform cubes: 0.005 wires per cubic wavelength, 0.025 for the half-wave one
        side = (nw / (0.025 if case["cloud"] == "cube8" else 0.005)) ** (1 / 3)
        c = side * (torch.rand(nw, 3, generator=g, **f64) - 0.5)
    t = torch.randn(nw, 3, generator=g, **f64)
    t = t / torch.linalg.vector_norm(t, dim=1, keepdim=True)
    if case["cloud"] == "cube8":
        L = torch.full((nw,), 0.5, **f64)
        ns = torch.full((nw,), 8, dtype=torch.int32, device="cuda")
    else:
        # the quantiles of U[0.3, 0.6] in random order: the number of unknowns depends on nw alone
        L = 0.3 + 0.3 * (torch.randperm(nw, generator=g, device="cuda").double() + 0.5) / nw
        ns = torch.ceil(L / 0.08).to(torch.int32)
    return c.contiguous(), t.contiguous(), L, torch.full((nw,), 1e-3, **f64), ns


def _incidences(case):
    """One wave from +z, or a monostatic cut theta = 0..180 degrees (phi = 0, theta-polarised)."""
    n = case["n_inc"]
    th = np.linspace(0.0, math.pi, n) if n > 1 else np.zeros(1)
    return np.stack([th, np.zeros(n), np.zeros(n)], axis=1)


def _observations(n):
    ph = np.arange(n) * (2.0 * math.pi / n)
    return np.stack([np.full(n, math.pi / 2), ph], axis=1)


def _sweep_ks(case):
    return K0 * np.linspace(0.85, 1.0, case["n_freq"])


def _profiles(cloud, n, g):
    """Currents shaped as a solve's: three sine modes per wire with the wire's random phase."""
    _, _, _, _, ns = cloud
    m = ns.to(torch.int64) - 1
    wire = torch.repeat_interleave(torch.arange(len(m), device="cuda"), m)
    off = torch.cumsum(m, 0) - m
    i = torch.arange(len(wire), device="cuda") - off[wire] + 1
    out = torch.zeros(n, len(wire), dtype=torch.complex128, device="cuda")
    for mode, size in ((1, 1.0), (2, 0.3), (3, 0.1)):
        amp = size * torch.randn(n, len(m), 2, generator=g, dtype=torch.float64, device="cuda")
        out += torch.view_as_complex(amp)[:, wire] * torch.sin(mode * math.pi * (i / ns[wire].double()))
    return out


LAYERS = [(16, 128), (128, 128), (128, 18), (20, 256), (256, 256), (256, 6)]


def _net_params(seed):
    rng = np.random.default_rng(seed)
    parts = []
    for i, o in LAYERS:
        parts += [(rng.standard_normal((i, o)) / math.sqrt(i)).ravel() * (0.1 if o in (18, 6) else 1.0),
                  0.05 * rng.standard_normal(o)]
    return np.concatenate(parts).astype(np.float32)


class State:
    """What a program holds between calls: the inputs and its context (released with the state)."""

    def __init__(self, case):
        self.case = case


def _context(state):
    ctx = swm.swm_create(0)
    weakref.finalize(state, swm.swm_destroy, ctx)
    return ctx


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    s = State(case)
    s.cloud = _cloud(case, g)
    nw = case["nw"]
    if case["path"] == "far":
        c, t, L, _, ns = s.cloud
        s.off = torch.zeros(nw + 1, dtype=torch.int64, device="cuda")
        s.off[1:] = torch.cumsum(ns.to(torch.int64) - 1, 0)
        s.currents = _profiles(s.cloud, case["n_rhs"], g)
        s.obs = torch.from_numpy(_observations(case["n_obs"])).cuda()
        s.sigma = torch.empty(case["n_rhs"], case["n_obs"], 2, dtype=torch.float64, device="cuda")
        return s
    s.ctx = _context(s)
    if case["path"] == "run":
        s.inc = _incidences(case)
        s.obs = _observations(case["n_obs"]) if case["n_obs"] else None
        shape = (case["n_inc"], case["n_obs"], 2) if case["n_obs"] else (case["n_inc"], 2)
        s.sigma = torch.empty(shape, dtype=torch.float64, device="cuda")
        if case["currents"]:
            n = int((s.cloud[4].to(torch.int64) - 1).sum())
            s.currents = torch.empty(case["n_inc"], n, dtype=torch.complex128, device="cuda")
        swm.swm_set_solver(s.ctx, case["solver"])
    elif case["path"] == "sweep":
        s.obs = _observations(case["n_obs"])
        s.inc = np.zeros((1, 3))
        s.sigma = torch.empty(1, case["n_obs"], 2, dtype=torch.float64, device="cuda")
        swm.swm_set_solver(s.ctx, "gcr")
    elif case["path"] == "operator":
        swm.swm_set_cloud(s.ctx, *s.cloud)
        swm.swm_build(s.ctx, K0, case["r_c"], swm.SWM_C128)
        n = swm.swm_get_stats(s.ctx)["n"]
        x = torch.randn(case["n_rhs"], n, 2, generator=g, dtype=torch.float64, device="cuda")
        s.x = torch.view_as_complex(x)
        s.y, s.z = torch.empty_like(s.x), torch.empty_like(s.x)
    else:  # train
        s.inc = _incidences(case)
        swm.swm_set_cloud(s.ctx, *s.cloud)
        swm.swm_build(s.ctx, K0, case["r_c"], swm.SWM_C64)
        s.net = swm.swm_net_create(0)
        weakref.finalize(s, swm.swm_net_destroy, s.net)
        swm.swm_net_set_params(s.net, _net_params(seed))
        s.target = 0.1 * _profiles(s.cloud, case["n_inc"], g)
    return s


def run(s):
    case = s.case
    if case["path"] == "far":
        c, t, L, _, ns = s.cloud
        swm.swm_far_field(None, c, t, L, ns, s.off, K0, s.currents, s.obs, s.sigma)
        return {"sigma": s.sigma}
    if case["path"] == "operator":
        swm.swm_apply(s.ctx, s.x, s.y)
        swm.swm_precond_apply(s.ctx, s.y, s.z)
        return {"y": s.y, "z": s.z}
    if case["path"] == "train":
        loss, grad = swm.swm_net_train_step(s.net, s.ctx, s.inc, s.target, want_grad=True)
        return {"loss": np.float32(loss), "grad": grad}
    if case["path"] == "sweep":
        swm.swm_set_cloud(s.ctx, *s.cloud)
        out = []
        for k in _sweep_ks(case):
            swm.swm_build(s.ctx, k, case["r_c"], swm.SWM_C64)
            swm.swm_solve(s.ctx, s.inc, TOL)
            swm.swm_rcs_bistatic(s.ctx, s.obs, s.sigma)
            out.append(s.sigma.float())
        return {"sigma": out}
    single = case["precision"] == "c64"
    prec = swm.SWM_C64 if single else swm.SWM_C128
    if not case["currents"]:
        swm.swm_run(s.ctx, *s.cloud, K0, case["r_c"], prec, s.inc, s.obs, s.sigma, tol=TOL)
        return {"sigma": s.sigma.float() if single else s.sigma}
    swm.swm_set_cloud(s.ctx, *s.cloud)
    swm.swm_build(s.ctx, K0, case["r_c"], prec)
    swm.swm_solve(s.ctx, s.inc, TOL, currents_out=s.currents)
    if s.obs is None:
        swm.swm_rcs_monostatic(s.ctx, s.sigma)
    else:
        swm.swm_rcs_bistatic(s.ctx, s.obs, s.sigma)
    if single:
        return {"sigma": s.sigma.float(), "currents": s.currents.to(torch.complex64)}
    return {"sigma": s.sigma, "currents": s.currents}


# ------------------------------------------------------------------------------ work
def _partners(case):
    """Expected other wires within r_c of a wire."""
    nw, r = case["nw"], case["r_c"]
    if r <= 0:
        return nw - 1.0
    ball = 4.0 / 3.0 * math.pi * r ** 3
    if case["cloud"] == "gauss":
        s = 30.0 * (nw / 1e4) ** (1 / 3)
        return nw * ball / (4.0 * math.pi * s * s) ** 1.5
    if case["cloud"] == "clusters":
        s = 40.0 * (nw / 1e6) ** (1 / 3)
        return nw / 8 * ball / (4.0 * math.pi * s * s) ** 1.5
    return ball * (0.025 if case["cloud"] == "cube8" else 0.005)


def work(case):
    """Bytes: inputs, stored blocks written once, and per product E, its column map and the vectors
    once; outputs.  Operations: 29 per kernel evaluation, 8 per complex multiply-add; the number of
    products is what these densities take at 1e-6 (the sizes keep the density)."""
    nw, m = case["nw"], 7.0 if case["cloud"] == "cube8" else MEAN_M
    n = nw * m
    far = lambda r, o: r * o * nw * (8.0 * m + 40.0)  # noqa: E731
    if case["path"] == "far":
        r, o = case["n_rhs"], case["n_obs"]
        return dict(bytes=16.0 * n * r + 68.0 * nw + 16.0 * r * o, flops=far(r, o))
    q = _partners(case)
    nnz = nw * q * m * m
    single = case.get("precision", "c64") == "c64" and case["path"] != "operator"
    esz = 8.0 if single else 16.0
    evals = 0.5 * nw * q * 16.0 * (m + 1) ** 2 + nw * 32.0 * (m + 1)
    if case["path"] == "operator":
        r = case["n_rhs"]
        return dict(bytes=esz * (nnz + nw * m * m) + 4.0 * nw * q * m + 64.0 * r * n, flops=8.0 * r * (nnz + n * m))
    if case["path"] == "train":
        dense = 2.0 * sum(i * o for i, o in LAYERS[:3]) * min(q, 16.0) + 2.0 * sum(i * o for i, o in LAYERS[3:])
        return dict(bytes=nw * 100.0 + 32.0 * n * case["n_inc"], flops=3.0 * dense * nw * case["n_inc"])
    r = 1 if case["path"] == "sweep" else case["n_inc"]
    builds = case["n_freq"] if case["path"] == "sweep" else 1
    if case["r_c"] <= 0:
        products = 25
    elif case["cloud"] == "clusters":
        products = 94 if case.get("solver") == "bicgstab" else 54
    else:
        products = 22 if case.get("solver") == "bicgstab" else 11
    pairs = r * case["n_obs"] if case["n_obs"] else r
    return dict(bytes=68.0 * nw + builds * (esz * nnz + products * (esz * nnz + 4.0 * nw * q * m + 2 * esz * r * n))
                + 16.0 * pairs + 16.0 * r * n,
                flops=builds * (29.0 * evals + products * 8.0 * nnz * r + far(1, pairs)))


# ------------------------------------------------------------------------------ 64-bit values
EXACT_MAX = 4.0e7  # unknowns x incidences: above it a solve takes over about 20 seconds
# The method in plain torch, float64: the same discretisation and quadrature (segments, rooftops,
# Gauss points, reduced kernel), solved to 1e-12.
def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (x + 1.0), 0.5 * w


def _dev(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.float64, device="cuda")


def _pairs(c, r_c):
    """All p < q whose centres are at most r_c apart (every pair for r_c <= 0, none for None)."""
    n = len(c)
    if r_c is None:
        return torch.zeros(2, 0, dtype=torch.int64, device="cuda")
    if r_c <= 0:
        p, q = torch.triu_indices(n, n, 1, device="cuda")
        return p, q
    cell = torch.floor((c - c.amin(0)) / r_c).to(torch.int64) + 1
    dim = cell.amax(0) + 2
    key = (cell[:, 0] * dim[1] + cell[:, 1]) * dim[2] + cell[:, 2]
    skey, order = torch.sort(key)
    got = []
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dz in (-1, 0, 1):
                want = key + (dx * dim[1] + dy) * dim[2] + dz
                lo = torch.searchsorted(skey, want)
                cnt = torch.searchsorted(skey, want, right=True) - lo
                p = torch.repeat_interleave(torch.arange(n, device="cuda"), cnt)
                first = torch.cumsum(cnt, 0) - cnt
                q = order[lo[p] + torch.arange(len(p), device="cuda") - first[p]]
                d = c[p] - c[q]
                d = d * d
                keep = (q > p) & (d[:, 0] + d[:, 1] + d[:, 2] <= r_c * r_c)
                got.append(torch.stack([p[keep], q[keep]]))
    p, q = torch.cat(got, 1)
    return p, q


def _segment_distance(c, t, L, p, q):
    """Shortest distance between the wires of each pair, as line segments."""
    d = c[p] - c[q]
    dot = lambda a, b: (a * b).sum(1)  # noqa: E731
    b, dp, dq = dot(t[p], t[q]), dot(d, t[p]), dot(d, t[q])
    hp, hq = 0.5 * L[p], 0.5 * L[q]
    dist2 = lambda s, u: ((d + s[:, None] * t[p] - u[:, None] * t[q]) ** 2).sum(1)  # noqa: E731
    det = 1.0 - b * b
    safe = torch.where(det > 1e-12, det, torch.ones_like(det))
    s, u = (b * dq - dp) / safe, (dq - b * dp) / safe
    inside = (det > 1e-12) & (s.abs() <= hp) & (u.abs() <= hq)
    best = torch.where(inside, dist2(s, u), torch.full_like(s, math.inf))
    for e in (-hp, hp):
        best = torch.minimum(best, dist2(e, torch.minimum(torch.maximum(dq + b * e, -hq), hq)))
    for e in (-hq, hq):
        best = torch.minimum(best, dist2(torch.minimum(torch.maximum(b * e - dp, -hp), hp), e))
    return torch.sqrt(best)


def _assemble(rise_fall, total, tpq, dd, k):
    """Rooftop blocks from segment-pair integrals I[B, u, v, a, b] (a, b: 0 rising, 1 falling)."""
    i, s = rise_fall, total
    vec = i[:, :-1, :-1, 0, 0] + i[:, :-1, 1:, 0, 1] + i[:, 1:, :-1, 1, 0] + i[:, 1:, 1:, 1, 1]
    div = s[:, :-1, :-1] - s[:, :-1, 1:] - s[:, 1:, :-1] + s[:, 1:, 1:]
    return tpq[:, None, None] * vec - div / (dd * k * k)[:, None, None]


def _mutual(cloud, k, p, q, nsp, nsq, nq):
    c, t, L, a, _ = cloud
    x, w = _gauss(nq)
    sh = torch.complex(_dev(np.stack([x * w, (1 - x) * w])), torch.zeros(2, nq, dtype=torch.float64, device="cuda"))
    step = max(1, (1 << 24) // (nsp * nsq * nq * nq))
    out = []
    for b in range(0, len(p), step):
        i, j = p[b:b + step], q[b:b + step]

        def points(i, ns):
            s = (_dev(np.arange(ns)[:, None] + x[None, :]).reshape(-1)[None, :] / ns - 0.5) * L[i][:, None]
            return c[i][:, None, :] + s[..., None] * t[i][:, None, :]
        u, v = points(i, nsp), points(j, nsq)
        r2 = sum((u[:, :, None, d] - v[:, None, :, d]) ** 2 for d in range(3))
        r = torch.sqrt(r2 + 0.5 * (a[i] ** 2 + a[j] ** 2)[:, None, None])
        gr = torch.polar(1.0 / (4.0 * math.pi * r), -k * r).reshape(len(i), nsp, nq, nsq, nq)
        dd = (L[i] / nsp) * (L[j] / nsq)
        ints = torch.einsum("Buavh,bh->Buvab", torch.einsum("Bugvh,ag->Buavh", gr, sh), sh) * dd[:, None, None, None, None]
        out.append(_assemble(ints, ints.sum((3, 4)), (t[i] * t[j]).sum(1), dd, k))
    return torch.cat(out)


def _self(cloud, k, w, ns):
    """Self blocks of the wires w of ns segments: 1-D reduction against the convolution W_ab of the
    segment shapes, the static part of touching segments in closed form."""
    _, _, L, a, _ = cloud
    D, a = L[w] / ns, a[w]
    shape = (lambda x: x, lambda x: 1.0 - x)
    xg, wg = _gauss(8)
    x2, w2 = _gauss(4)
    al = a / D
    table = {}
    for delta in range(-(ns - 1), ns):
        val = torch.zeros(len(w), 2, 2, dtype=torch.complex128, device="cuda")
        for w0 in (-1.0, 0.0):
            def conv(fa, fb, v):  # int of phi_a(x) phi_b(x - v) over x, x - v in [0, 1]
                lo, hi = max(0.0, v), min(1.0, 1.0 + v)
                xx = lo + (hi - lo) * x2
                return (hi - lo) * float(np.sum(w2 * fa(xx) * fb(xx - v)))
            nodes = w0 + xg
            tt = _dev(nodes + delta)
            R = torch.sqrt((D[:, None] * tt[None, :]) ** 2 + (a * a)[:, None])
            kern = torch.polar(torch.ones_like(R), -k * R)
            near = abs(delta) <= 1
            kern = (kern - 1.0 if near else kern) / (4.0 * math.pi * R)
            if near:
                prim = []
                for e in (w0 + delta, w0 + 1.0 + delta):
                    r = torch.sqrt(e * e + al * al)
                    ash = torch.asinh(e / al)
                    prim.append([ash, r, 0.5 * (e * r - al * al * ash), (e * e - 2 * al * al) * r / 3.0])
                prim = [h - lo for lo, h in zip(*prim)]
            at = w0 + np.array([0.0, 1.0 / 3.0, 2.0 / 3.0, 1.0])
            vander = np.vander(at + delta, 4, increasing=True)
            for ia, fa in enumerate(shape):
                for ib, fb in enumerate(shape):
                    cw = _dev([conv(fa, fb, v) for v in nodes] * wg)
                    val[:, ia, ib] += (kern * cw).sum(1)
                    if near:
                        co = np.linalg.solve(vander, [conv(fa, fb, v) for v in at])
                        val[:, ia, ib] += sum(float(co[n]) * prim[n] for n in range(4)) / (4.0 * math.pi * D)
        table[delta] = val * (D * D)[:, None, None]
    ints = torch.stack([torch.stack([table[u - v] for v in range(ns)], 1) for u in range(ns)], 1)
    return _assemble(ints, ints.sum((3, 4)), torch.ones_like(D), D * D, k)


class _System:
    """Block-sparse Z and the inverses of its self blocks; vectors are [unknowns, right-hand sides]."""

    def __init__(self, cloud, k, r_c):
        c, t, L, a, ns = cloud
        ns = ns.to(torch.int64)
        self.cloud, self.k, self.ns, self.m = cloud, k, ns, ns - 1
        self.off = torch.cumsum(self.m, 0) - self.m
        self.n = int(self.m.sum())
        p, q = _pairs(c, r_c)
        near = _segment_distance(c, t, L, p, q) < torch.maximum(L[p] / ns[p], L[q] / ns[q])
        self.self_blocks, self.blocks = [], []
        sizes = [int(v) for v in torch.unique(ns)]
        for i in sizes:
            w = torch.nonzero(ns == i).flatten()
            z = _self(cloud, k, w, i)
            self.self_blocks.append((self._rows(w, i - 1), z, torch.linalg.inv(z)))
            for j in sizes:
                for nq in (4, 8):
                    at = torch.nonzero((ns[p] == i) & (ns[q] == j) & (near == (nq == 8))).flatten()
                    if len(at):
                        self.blocks.append((self._rows(p[at], i - 1), self._rows(q[at], j - 1),
                                            _mutual(cloud, k, p[at], q[at], i, j, nq)))

    def _rows(self, w, m):
        return self.off[w][:, None] + torch.arange(m, device="cuda")[None, :]

    def precond(self, y):
        x = torch.empty_like(y)
        for rows, _, inv in self.self_blocks:
            x[rows.reshape(-1)] = (inv @ y[rows]).reshape(-1, y.shape[1])
        return x

    def apply(self, x):
        """(Z M^-1) x"""
        v = self.precond(x)
        y = x.clone()  # Z_pp Z_pp^-1 x_p
        for pr, qr, z in self.blocks:
            step = max(1, (1 << 24) // (8 * x.shape[1]))
            for b in range(0, len(z), step):
                i, j, zz = pr[b:b + step], qr[b:b + step], z[b:b + step]
                y.index_add_(0, i.reshape(-1), (zz @ v[j]).reshape(-1, x.shape[1]))
                y.index_add_(0, j.reshape(-1), (zz.transpose(1, 2) @ v[i]).reshape(-1, x.shape[1]))
        return y

    def solve(self, b):
        """BiCGSTAB on (Z M^-1) y = b for every column, x = M^-1 y."""
        dot = lambda u, v: (u.conj() * v).sum(0)  # noqa: E731
        y = torch.zeros_like(b)
        r, bn = b.clone(), torch.linalg.vector_norm(b, dim=0)
        for _ in range(4):
            rh, p = r.clone(), r.clone()
            rho = dot(rh, r)
            for _ in range(200):
                v = self.apply(p)
                alpha = rho / dot(rh, v)
                s = r - alpha * v
                t = self.apply(s)
                omega = dot(t, s) / dot(t, t)
                y += alpha * p + omega * s
                r = s - omega * t
                if float((torch.linalg.vector_norm(r, dim=0) / bn).max()) < 1e-12:
                    break
                rho, old = dot(rh, r), rho
                p = r + (rho / old) * (alpha / omega) * (p - omega * v)
            r = b - self.apply(y)
            if float((torch.linalg.vector_norm(r, dim=0) / bn).max()) < 1e-11:
                break
        return self.precond(y)


def _frames(th, ph):
    th, ph = np.asarray(th), np.asarray(ph)
    u = np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], 1)
    e1 = np.stack([np.cos(th) * np.cos(ph), np.cos(th) * np.sin(ph), -np.sin(th)], 1)
    e2 = np.stack([-np.sin(ph), np.cos(ph), 0 * ph], 1)
    return _dev(u), _dev(e1), _dev(e2)


def _wave(cloud, k, dirs, rows_wire, rows_s, rows_D):
    """exp(+j k u . r) integrated against each rooftop, [unknowns, directions]."""
    c, t, _, _, _ = cloud
    kt = t @ dirs.T
    z = 0.5 * k * kt[rows_wire] * rows_D[:, None]
    sinc = torch.sinc(z / math.pi)
    ph = k * ((c @ dirs.T)[rows_wire] + rows_s[:, None] * kt[rows_wire])
    return torch.polar(rows_D[:, None] * sinc * sinc, ph)


def _rows_of(cloud):
    _, _, L, _, ns = cloud
    m = ns.to(torch.int64) - 1
    wire = torch.repeat_interleave(torch.arange(len(m), device="cuda"), m)
    i = torch.arange(len(wire), device="cuda") - (torch.cumsum(m, 0) - m)[wire] + 1
    D = (L / ns)[wire]
    return wire, -0.5 * L[wire] + i * D, D


def _rhs(cloud, k, inc):
    u, e1, e2 = _frames(inc[:, 0], inc[:, 1])
    e = _dev(np.cos(inc[:, 2]))[:, None] * e1 + _dev(np.sin(inc[:, 2]))[:, None] * e2
    wire, s, D = _rows_of(cloud)
    return _wave(cloud, k, u, wire, s, D) * (cloud[1] @ e.T)[wire]  # exp(-j k k_hat . r), k_hat = -u


def _rcs(cloud, k, x, obs, mono):
    """sigma[r, o, 2], or [r, 2] with each column observed along its own direction."""
    u, e1, e2 = _frames(obs[:, 0], obs[:, 1])
    wire, s, D = _rows_of(cloud)
    out = 0
    step = max(1, (1 << 24) // len(obs))
    for b in range(0, len(wire), step):
        w = wire[b:b + step]
        f = _wave(cloud, k, u, w, s[b:b + step], D[b:b + step])
        parts = []
        for e in (e1, e2):
            g = f * (cloud[1] @ e.T)[w]
            parts.append((g * x[b:b + step]).sum(0) if mono else x[b:b + step].T @ g)
        out = out + torch.stack(parts, -1)
    return (out.real ** 2 + out.imag ** 2) / (4.0 * math.pi)


def _exact_train(cloud, case, seed, target):
    k, r_c, inc = K0, case["r_c"], _incidences(case)
    c, t, L, _, ns = cloud
    nw, R = case["nw"], case["n_inc"]
    flat = _dev(_net_params(seed)).requires_grad_(True)
    W, o = [], 0
    for i, n in LAYERS:
        W.append((flat[o:o + i * n].reshape(i, n), flat[o + i * n:o + i * n + n]))
        o += i * n + n
    sysm = _System(cloud, k, None)  # self blocks only
    x_iso = sysm.precond(_rhs(cloud, k, inc))  # [n, R]
    u, e1, _ = _frames(inc[:, 0], inc[:, 1])
    kh = -u
    wire, s, _ = _rows_of(cloud)
    i = torch.arange(len(wire), device="cuda") - sysm.off[wire] + 1
    modes = torch.stack([torch.sin(q * math.pi * (i / ns[wire].double())) for q in (1, 2, 3)], 1)  # [n, 3]
    phase = torch.polar(torch.ones(nw, R, dtype=torch.float64, device="cuda"), k * (c @ kh.T))
    amp = torch.zeros(nw, R, 3, dtype=torch.complex128, device="cuda")
    amp.index_add_(0, wire, x_iso[:, :, None] * modes[:, None, :])
    amp = amp * (2.0 / ns.double())[:, None, None] * phase[:, :, None]
    p, q = _pairs(c, r_c)
    p, q = torch.cat([p, q]), torch.cat([q, p])
    d = c[q] - c[p]
    d2 = d * d
    d2 = d2[:, 0] + d2[:, 1] + d2[:, 2]
    order = torch.arange(len(p), device="cuda")
    for key in (q, d2, p):  # by wire, then distance, then index
        order = order[torch.sort(key[order], stable=True)[1]]
    p, q, d, d2 = p[order], q[order], d[order], d2[order]
    cnt = torch.bincount(p, minlength=nw)
    rank = torch.arange(len(p), device="cuda") - (torch.cumsum(cnt, 0) - cnt)[p]
    keep = rank < 16
    p, q, d, d2 = p[keep], q[keep], d[keep], d2[keep]
    cnt = torch.clamp(cnt, max=16)
    dist = torch.sqrt(d2)
    z = (d * t[p]).sum(1)
    rho = torch.sqrt(torch.clamp(d2 - z * z, min=0.0))
    silu = torch.nn.functional.silu
    h = torch.zeros(nw, R, 3, dtype=torch.complex128, device="cuda")
    parts = []
    for r in range(R):
        et, kt = t @ e1[r], t @ kh[r]
        ph = k * (d @ kh[r])
        one = torch.ones_like(ph)
        f = torch.stack([z / r_c, rho / r_c, (t[p] * t[q]).sum(1), (t[q] * d).sum(1) / r_c, L[q] * k / (2 * math.pi),
                         L[p] * k / (2 * math.pi), et[p], kt[p], et[q], kt[q], torch.cos(ph), torch.sin(ph),
                         torch.cos(k * dist), torch.sin(k * dist), 1.0 / (1.0 + k * dist), one], 1)
        g = silu(silu(f @ W[0][0] + W[0][1]) @ W[1][0] + W[1][1]) @ W[2][0] + W[2][1]
        cm = torch.complex(g[:, :9], g[:, 9:]).reshape(-1, 3, 3)
        rel = amp[q, r] * torch.polar(one, -ph)[:, None]
        hr = torch.zeros(nw, 3, dtype=torch.complex128, device="cuda").index_add(0, p, (cm @ rel[:, :, None])[:, :, 0])
        zero = torch.zeros_like(et)
        own = torch.stack([et, kt, L * k / (2 * math.pi), cnt / 16.0, et * kt, kt * kt, zero, zero], 1)
        a = amp[:, r]
        v = torch.cat([hr.real, hr.imag, own, a.real, a.imag], 1)
        v = silu(silu(v @ W[3][0] + W[3][1]) @ W[4][0] + W[4][1]) @ W[5][0] + W[5][1]
        cmode = hr + torch.complex(v[:, 0::2], v[:, 1::2])
        parts.append(x_iso[:, r] + phase.conj()[wire, r] * (cmode[wire] * modes).sum(1))
    err = torch.stack(parts) - target
    loss = (err.real ** 2 + err.imag ** 2).sum() / (target.real ** 2 + target.imag ** 2).sum()
    loss.backward()
    return {"loss": float(loss.detach()), "grad": flat.grad}


def exact(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    cloud = _cloud(case, g)
    if case["path"] == "far":
        x = _profiles(cloud, case["n_rhs"], g)
        return {"sigma": _rcs(cloud, K0, x.T.contiguous(), _observations(case["n_obs"]), False)}
    if case["path"] == "train":
        return _exact_train(cloud, case, seed, 0.1 * _profiles(cloud, case["n_inc"], g))
    if case["path"] == "operator":
        s = _System(cloud, K0, case["r_c"])
        x = torch.view_as_complex(torch.randn(case["n_rhs"], s.n, 2, generator=g, dtype=torch.float64, device="cuda"))
        y = s.apply(x.T.contiguous())
        return {"y": y.T.contiguous(), "z": s.precond(y).T.contiguous()}
    if case["path"] == "sweep":
        out, inc, obs = [], np.zeros((1, 3)), _observations(case["n_obs"])
        for k in _sweep_ks(case):
            s = _System(cloud, float(k), case["r_c"])
            out.append(_rcs(cloud, float(k), s.solve(_rhs(cloud, float(k), inc)), obs, False))
        return {"sigma": out}
    if case["nw"] * MEAN_M * case["n_inc"] > EXACT_MAX:
        return None
    s = _System(cloud, K0, case["r_c"])
    inc = _incidences(case)
    x = s.solve(_rhs(cloud, K0, inc))
    mono = not case["n_obs"]
    sigma = _rcs(cloud, K0, x, inc if mono else _observations(case["n_obs"]), mono)
    out = {"sigma": sigma}
    if case["currents"]:
        out["currents"] = x.T.contiguous()
    return out


