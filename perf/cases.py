"""What is measured: the calls a solver built on this framework makes, over their real range.

A solver makes a plan once and then, in every iteration, aggregates its currents into group
spectra, translates them between groups and disaggregates them; before the iterations it asks
for the excitations.  The cases are these calls through the public binding
(``paper_2103_05822_gb300.tfmm``), with the box grids, direction grids and ranks of the
repository's workloads:

* ``matvec``        tfmm_aggregate then tfmm_disaggregate on device buffers (``graph``: the same
                    two stages replayed from a captured CUDA graph);
* ``aggregate`` / ``disaggregate``   one of the two stages alone;
* ``host``          tfmm_matvec_host, from and to pinned host buffers;
* ``translate``     tfmm_translate, outgoing to incoming spectra of every group;
* ``planewave``     tfmm_planewave, the RWG-tested excitations of R incidences.

Factors of the first four are synthetic: groups as points of the workload's surface fall into
its boxes (so group sizes are as uneven as there), ranks that grow with the group size up to the
largest rank of the workload, orthonormal theta / phi factors and core slices that decay to the
Tucker tolerance.  They go through tfmm_plan_from_tucker.  Translation and excitations need the
geometry: a geodesic sphere through tfmm_plan_create.
"""
from __future__ import annotations

import functools
import json
import math

import numpy as np
import torch

from paper_2103_05822_gb300 import inputs, tfmm

# bandwidth L of a box edge (wavelengths) at 3 and 6 digits, and the largest (theta, phi, beta)
# ranks of a lambda/10 sphere at each Tucker tolerance
BANDWIDTH = {0.5: {3: 13, 6: 16}, 1.0: {3: 20, 6: 25}, 2.0: {3: 33, 6: 39}, 4.0: {3: 57, 6: 65}}
RANKS = {
    0.5: {3: (9, 13, 35), 4: (11, 15, 48), 6: (14, 19, 78)},
    1.0: {3: (13, 17, 65), 4: (15, 21, 87), 6: (19, 25, 137)},
    2.0: {3: (18, 26, 140), 4: (20, 30, 179), 6: (25, 36, 268)},
    4.0: {3: (27, 43, 318), 4: (31, 47, 388), 6: (36, 55, 541)},
}
TEMPLATES = 24          # distinct factor sets per component; groups of like size share one
MOST_RWG = 972_000      # the 30-lambda sphere
MOST_SPECTRA = 128 * 1034 * 6400


def _case(name, do, size, box, digits, gamma, rhs=1, engine=0, graph=False, beta=0.0, shape="sphere"):
    return {"name": name, "do": do, "shape": shape, "size": float(size), "box": float(box), "digits": digits,
            "gamma": gamma, "rhs": rhs, "engine": engine, "graph": graph, "beta": float(beta)}


def listed():
    return [
        # the smallest problem: a 2-lambda sphere in half-wavelength boxes, an iterative solver
        # replaying its captured matvec; latency and launches count
        _case("sphere2_graph", "matvec", 2, 0.5, 3, 4, graph=True),
        # the trihedral corner reflector: few groups, up to thousands of RWGs each, odd N_phi
        _case("corner6", "matvec", 6, 2, 5, 6, shape="corner"),
        # an ordinary problem, one right-hand side per iteration
        _case("sphere10", "matvec", 10, 1, 6, 6),
        # the same called from a program that keeps its vectors on the host
        _case("sphere10_host", "host", 10, 1, 6, 6),
        # the benchmark: 972,000 RWGs, one right-hand side
        _case("sphere30", "matvec", 30, 2, 6, 6),
        # a block solver's 16 columns on the tensor cores (3 terms), a middle-sized sphere
        _case("sphere20_rhs16", "matvec", 20, 2, 6, 6, rhs=16, engine=3),
        # many tiny groups, 16 columns, the default engine (FP32 on CUDA cores), 3 digits
        _case("sphere20_small_boxes", "matvec", 20, 0.5, 3, 3, rhs=16),
        # an odd block of columns, y holding the near-field product already (beta = 1)
        _case("sphere10_rhs37", "matvec", 10, 1, 6, 6, rhs=37, engine=3, beta=1.0),
        # the monostatic RCS sweep: 128 incidences at once, each stage on its own
        _case("sphere30_rhs128_agg", "aggregate", 30, 2, 6, 6, rhs=128, engine=3),
        _case("sphere30_rhs128_dis", "disaggregate", 30, 2, 6, 6, rhs=128, engine=3),
        # the stage between the two, once per iteration
        _case("sphere30_translate", "translate", 30, 2, 6, 6),
        # the right-hand sides of an RCS sweep
        _case("sphere10_planewave", "planewave", 10, 1, 6, 6, rhs=128),
    ]


def draw(rng):
    """One more case: kind, box and tolerance as the workloads combine them, sizes over the range."""
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    do = rng.choice(["matvec", "matvec", "matvec", "aggregate", "disaggregate", "host", "translate", "planewave"])
    digits, gamma = rng.choice([3, 6]), rng.choice([3, 4, 6])
    if do == "planewave":
        size, box, rhs = round(log(2, 10), 2), 1.0, int(round(log(1, 128)))
        return _pure(_case("", do, size, box, digits, gamma, rhs=max(rhs, 1)))
    if do == "translate":
        box = rng.choice([0.5, 1.0, 2.0])
        size = round(box * log(4, 16), 2)
        return _pure(_case("", do, size, box, digits, gamma, rhs=rng.choice([1, 1, 2, 3])))
    box = rng.choice([0.5, 1.0, 2.0, 4.0])
    size = round(log(max(2.0, 3 * box), min(30.0, 40 * box, 60 / box if box == 4 else 30.0)), 2)
    rhs = 1 if do == "host" or rng.random() < 0.45 else int(round(log(2, 128)))
    n = 1080 * size * size
    per_rhs = 4.6 * (size / box) ** 2 * 4 * (BANDWIDTH[box][digits] + 1) ** 2
    rhs = max(1, min(rhs, int(0.8 * 128 * MOST_RWG * 268 / (n * RANKS[box][gamma][2])), int(0.8 * MOST_SPECTRA / per_rhs)))
    engine = rng.choice([0, 3, 3]) if rhs > 1 else 0
    if engine == 0 and rhs > 1:  # the CUDA-core chain runs the smaller blocks
        rhs = max(2, min(rhs, 32))
    return _pure(_case("", do, size, box, digits, gamma, rhs=rhs, engine=engine,
                       graph=do == "matvec" and rng.random() < 0.3,
                       beta=rng.choice([0.0, 0.0, 1.0]) if do in ("matvec", "disaggregate") else 0.0))


def _pure(case):
    return {k: v for k, v in case.items() if k != "name"}


# ------------------------------------------------------------------ groups, ranks and factors
def _grid(case):
    """(n_theta, n_phi): the corner reflector runs the paper's 38 x 75 grid (L = 37, N_phi = 2L + 1)."""
    if case["shape"] == "corner":
        return 38, 75
    L = BANDWIDTH[case["box"]][case["digits"]]
    return L + 1, 2 * (L + 1)


def _weights(case):
    """Gauss-Legendre in cos(theta) times the uniform phi weight, theta fastest."""
    nt, npf = _grid(case)
    w = np.polynomial.legendre.leggauss(nt)[1]
    return np.tile(w * (2 * math.pi / npf), npf)


def _plan_key(case):
    return json.dumps({k: case[k] for k in ("do", "shape", "size", "box", "digits", "gamma", "rhs", "engine")}, sort_keys=True)


@functools.lru_cache(maxsize=2)
def _groups(shape, size, box):
    """RWG ids of every occupied box: the workload's RWG count, spread evenly over its surface."""
    rng = np.random.default_rng(7)
    if shape == "corner":
        n = int(round(1184.5 * size * size))  # 42,642 on 6-lambda plates
        p = rng.uniform(0, size, (n, 3))
        p[np.arange(n), rng.integers(0, 3, n)] = 0.0
    else:
        n = int(round(1080 * size * size))
        p = rng.standard_normal((n, 3))
        p *= 0.5 * size / np.linalg.norm(p, axis=1)[:, None]
    lo = p.min(0)
    K = np.maximum(1, np.ceil((p.max(0) - lo) / box)).astype(np.int64)
    i = np.minimum(((p - lo) / box).astype(np.int64), K - 1)
    b = i[:, 0] + K[0] * (i[:, 1] + K[1] * i[:, 2])
    order = np.argsort(b, kind="stable")
    cuts = np.flatnonzero(np.diff(b[order])) + 1
    return n, np.split(order, cuts)


@functools.lru_cache(maxsize=2)
def _layout(shape, size, box, digits, gamma):
    """Per group its template, and per (template, component) the ranks: r_beta follows the group size
    as on the 30-lambda sphere (about 180 at 940 RWGs of 268 at most)."""
    n_rwg, members = _groups(shape, size, box)
    nt, npf = (38, 75) if shape == "corner" else (BANDWIDTH[box][digits] + 1, 2 * (BANDWIDTH[box][digits] + 1))
    top = RANKS[box][gamma]
    sizes = np.array([len(m) for m in members])
    rng = np.random.default_rng(11)
    template = np.zeros(len(members), np.int64)
    ranks = []
    half = 1300.0 * (box / 2.0) ** 2
    for t, idx in enumerate(np.array_split(np.argsort(sizes, kind="stable"), min(TEMPLATES, len(members)))):
        template[idx] = t
        n = int(sizes[idx].min())
        big = 1972.0 * (box / 2.0) ** 2
        grow = min(1.0, (n / (n + half)) / (big / (big + half)))
        both = []
        for _ in range(2):
            rt = max(1, min(nt, n, int(round(top[0] * (0.75 + 0.25 * grow) * rng.uniform(0.9, 1.0)))))
            rp = max(1, min(npf, n, int(round(top[1] * (0.75 + 0.25 * grow) * rng.uniform(0.9, 1.0)))))
            rb = max(1, min(n, rt * rp, int(round(top[2] * grow * rng.uniform(0.92, 1.0)))))
            both.append((rt, rp, rb, n))
        ranks.append(both)
    return n_rwg, members, template, ranks


def _lay(case):
    return _layout(case["shape"], case["size"], case["box"], case["digits"], case["gamma"])


@functools.lru_cache(maxsize=1)
def _factor_sets(key):
    """[template][component] = (U_theta, U_phi, flat U_beta for the template's largest group, core)."""
    case = json.loads(key)
    nt, npf = _grid(case)
    _, members, template, ranks = _lay(case)
    sizes = np.array([len(m) for m in members])
    rng = np.random.default_rng(13)

    def cn(*shape):
        return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) * math.sqrt(0.5)

    out = []
    for t, both in enumerate(ranks):
        n_max = int(sizes[template == t].max())
        per = []
        for rt, rp, rb, n in both:
            decay = np.minimum(1.0, 10.0 ** (-case["gamma"] * (2.0 * np.arange(rb) / rb - 1.0)))
            core = cn(rt * rp, rb) * (decay / math.sqrt(rt * rp))
            per.append((np.asfortranarray(np.linalg.qr(cn(nt, rt))[0]), np.asfortranarray(np.linalg.qr(cn(npf, rp))[0]),
                        cn(n_max * rb) / math.sqrt(max(n, 1)),
                        np.asfortranarray(core).reshape(rt, rp, rb, order="F")))
        out.append(per)
    return out


def _factor_key(case):
    return json.dumps({k: case[k] for k in ("shape", "size", "box", "digits", "gamma")}, sort_keys=True)


def _sphere(case):
    """The geodesic sphere: lambda/10 edges for the excitations; for the translation, which sees only
    the boxes, edges of a quarter box keep the plan's setup short."""
    d = case["size"]
    nu = max(2, int(round(6 * d))) if case["do"] == "planewave" else max(4, int(round(2.4 * d / case["box"])))
    return inputs.icosphere(d, nu)


@functools.lru_cache(maxsize=1)
def _plan(key):
    """The plan a program keeps for all its calls."""
    case = json.loads(key)
    if case["do"] in ("translate", "planewave"):
        v, f = _sphere(case)
        prm = tfmm.tfmm_params_default(box=case["box"], digits=3.0, L_override=_grid(case)[0] - 1, tol=1e-3,
                                       max_rhs=case["rhs"])
        return tfmm.tfmm_plan_create(tfmm.tfmm_mesh_create(v, f), prm)
    nt, npf = _grid(case)
    n_rwg, members, template, _ = _lay(case)
    sets = _factor_sets(_factor_key(case))
    factors = []
    for g, m in enumerate(members):
        per = []
        for ut, up, ub, core in sets[template[g]]:
            rb = core.shape[2]
            per.append((ut, up, ub[:len(m) * rb].reshape(len(m), rb, order="F"), core))
        factors.append(per)
    return tfmm.tfmm_plan_from_tucker(n_rwg, nt, npf, members, factors, weights=_weights(case), max_rhs=case["rhs"],
                                      mrhs_precision=case["engine"])


def _randn(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    return torch.randn(shape, dtype=torch.complex64, device="cuda", generator=g)


def _incidences(case, seed):
    """R plane waves from random directions, polarised across them."""
    rng = np.random.default_rng(seed)
    k = rng.standard_normal((case["rhs"], 3))
    k /= np.linalg.norm(k, axis=1)[:, None]
    p = np.cross(k, rng.standard_normal((case["rhs"], 3)))
    return k, p / np.linalg.norm(p, axis=1)[:, None]


def _shapes(case, plan=None):
    nt, npf = _grid(case)
    if plan is not None:
        return plan.info["n_rwg"], plan.info["n_groups"], nt * npf
    n_rwg, members, _, _ = _lay(case)
    return n_rwg, len(members), nt * npf


def prepare(case, seed):
    plan = _plan(_plan_key(case))
    R, do = case["rhs"], case["do"]
    n, G, nd = _shapes(case, plan)
    s = {"case": case, "plan": plan}
    if do == "planewave":
        s["k"], s["p"] = _incidences(case, seed)
        s["V"] = torch.empty((R, n), dtype=torch.complex64, device="cuda")
        return s
    if do == "host":
        s["x"] = _randn((n,), seed).cpu().pin_memory()
        s["y"] = torch.empty(n, dtype=torch.complex64).pin_memory()
        return s
    if do == "translate":
        s["out"] = _randn((R, G, 2, nd), seed)
        s["in"] = torch.empty_like(s["out"])
        return s
    s["spec"] = _randn((R, G, 2, nd), seed) if do == "disaggregate" else torch.empty((R, G, 2, nd), dtype=torch.complex64, device="cuda")
    if do != "disaggregate":
        s["x"] = _randn((R, n), seed)
    if do != "aggregate":
        s["y"] = _randn((R, n), seed + 1000003) if case["beta"] else torch.empty((R, n), dtype=torch.complex64, device="cuda")
    if case["graph"]:
        y0 = s["y"].clone()
        s["graph"] = tfmm.tfmm_graph_capture(plan, 3, s["spec"], x=s["x"], y=s["y"], R=R, beta=case["beta"])
        s["y"].copy_(y0)  # the capture's own pass wrote it
    return s


def run(s):
    do, plan, beta = s["case"]["do"], s["plan"], s["case"]["beta"]
    if do == "planewave":
        tfmm.tfmm_planewave(plan, s["k"], s["p"], s["V"])
        return s["V"]
    if do == "host":
        tfmm.tfmm_matvec_host(plan, s["x"], s["y"])
        return s["y"]
    if do == "translate":
        tfmm.tfmm_translate(plan, s["out"], s["in"])
        return s["in"]
    if "graph" in s:
        s["graph"].launch()
        return {"spectra": s["spec"], "y": s["y"]}
    out = {}
    if do != "disaggregate":
        tfmm.tfmm_aggregate(plan, s["x"], s["spec"])
        out["spectra"] = s["spec"]
    if do != "aggregate":
        tfmm.tfmm_disaggregate(plan, s["spec"], s["y"], beta=beta)
        out["y"] = s["y"]
    return out


def work(case):
    """Each call reads its factors and inputs once and writes its outputs once; a matvec is two calls."""
    nt, npf = _grid(case)
    nd, R, do = nt * npf, case["rhs"], case["do"]
    if do == "planewave":
        v, f = _sphere(case)
        n = 3 * len(f) // 2
        # 2 triangles x 25 points: phase and amplitude (two dot products) and a complex exponential
        return {"bytes": n * 128 + 8 * n * R, "flops": 50 * 20 * n * R}
    if do == "translate":
        n, boxes = _boxes(case)
        G = len(boxes)
        grid = 1
        for K in boxes.max(0) + 1:
            grid *= 2 * int(K) - 1
        # spectra in and out, the translation operator over the grid of box differences; the
        # cost of a zero-padded FFT convolution of both components
        return {"bytes": 2 * R * G * 2 * nd * 8 + grid * nd * 8,
                "flops": R * 2 * nd * (2 * 5 * grid * math.log2(grid) + 6 * grid)}
    n_rwg, members, template, ranks = _lay(case)
    elems = flops = 0
    for g, m in enumerate(members):
        for rt, rp, rb, _ in ranks[template[g]]:
            big = len(m) * rb + rt * rp * rb
            elems += big + nt * rt + npf * rp
            flops += 8 * (big + npf * rt * rp + nt * npf * rt)
    stages = 1 if do in ("aggregate", "disaggregate") else 2
    spectra, vec = 8 * R * len(members) * 2 * nd, 8 * R * n_rwg
    extra = vec if case["beta"] else 0
    return {"bytes": stages * (8 * elems + spectra + vec) + extra, "flops": stages * R * flops}


# ------------------------------------------------------------------------ 64-bit references
def _boxes(case):
    """Box index of every group, from the mesh's edge midpoints (every edge of the closed mesh carries
    one RWG): boxes anchored at the lowest midpoint, groups in ascending x-fastest order."""
    v, f = _sphere(case)
    e = np.unique(np.sort(np.concatenate([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]]).astype(np.int64), axis=1), axis=0)
    mid = 0.5 * (v[e[:, 0]] + v[e[:, 1]])
    lo = mid.min(0)
    K = np.maximum(1, np.ceil((mid.max(0) - lo) / case["box"])).astype(np.int64)
    i = np.minimum(((mid - lo) / case["box"]).astype(np.int64), K - 1)
    b = np.unique(i[:, 0] + K[0] * (i[:, 1] + K[1] * i[:, 2]))
    return len(e), np.stack([b % K[0], b // K[0] % K[1], b // (K[0] * K[1])], axis=1)


def _exact_translate(case, seed):
    """Direct sums of the addition theorem over far box pairs."""
    nt, npf = _grid(case)
    L, k, a = nt - 1, 2 * math.pi, case["box"]
    _, boxes = _boxes(case)
    G = len(boxes)
    K = torch.tensor(boxes.max(0) + 1)
    dev = torch.device("cuda")
    F = _randn((case["rhs"], G, 2, nt * npf), seed).to(torch.complex128)
    bx = torch.tensor(boxes, device=dev)
    W = [2 * int(c) - 1 for c in K]
    diff = bx[:, None, :] - bx[None, :, :] + (K.to(dev) - 1)
    idx = diff[..., 0] + W[0] * (diff[..., 1] + W[1] * diff[..., 2])
    lin = torch.arange(W[0] * W[1] * W[2], device=dev)
    d = torch.stack([lin % W[0], lin // W[0] % W[1], lin // (W[0] * W[1])], 1) - (K.to(dev) - 1)
    far = d.abs().max(1).values >= 2
    X = d[far].to(torch.float64) * a
    r = X.norm(dim=1)
    x = k * r
    h = [torch.complex(torch.sin(x) / x, torch.cos(x) / x)]
    h.append(torch.complex(torch.sin(x) / x ** 2 - torch.cos(x) / x, torch.cos(x) / x ** 2 + torch.sin(x) / x))
    for l in range(1, L):
        h.append((2 * l + 1) / x * h[l] - h[l - 1])
    theta = np.arccos(np.polynomial.legendre.leggauss(nt)[0])[::-1]
    phi = 2 * math.pi * np.arange(npf) / npf
    kh = np.stack([np.outer(np.cos(phi), np.sin(theta)), np.outer(np.sin(phi), np.sin(theta)),
                   np.outer(np.ones(npf), np.cos(theta))], -1).reshape(-1, 3)
    kh = torch.tensor(kh, device=dev)
    xh = X / r[:, None]
    out = torch.empty_like(F)
    step = max(1, min(64, int(2e8 // max(G * G, len(lin)))))
    for i0 in range(0, nt * npf, step):
        ct = xh @ kh[i0:i0 + step].T
        p0, p1 = torch.ones_like(ct), ct
        acc = h[0][:, None] * p0
        for l in range(1, L + 1):
            acc = acc + ((-1j) ** l * (2 * l + 1)) * h[l][:, None] * p1
            p0, p1 = p1, ((2 * l + 1) * ct * p1 - l * p0) / (l + 1)
        T = torch.zeros((len(lin), ct.shape[1]), dtype=torch.complex128, device=dev)
        T[far] = (-1j * k / (16 * math.pi ** 2)) * acc
        M = T.T[:, idx]  # directions x G x G
        f = F[..., i0:i0 + step].permute(3, 1, 0, 2).reshape(ct.shape[1], G, -1)
        out[..., i0:i0 + step] = (M @ f).reshape(ct.shape[1], G, case["rhs"], 2).permute(2, 1, 3, 0)
    return out


def _exact_planewave(case, seed):
    """Collapsed Gauss-Legendre on both triangles of every RWG, order 6."""
    v, f = _sphere(case)
    f = f.astype(np.int64)
    nf = len(f)
    e = np.sort(np.concatenate([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]]), axis=1)
    opposite = np.concatenate([f[:, 2], f[:, 0], f[:, 1]])
    tri = np.tile(np.arange(nf), 3)
    order = np.lexsort((tri, e[:, 1], e[:, 0]))  # pairs (T+, T-), T+ the lower triangle
    e, opposite = e[order].reshape(-1, 2, 2)[:, 0], opposite[order].reshape(-1, 2)
    x, w = np.polynomial.legendre.leggauss(6)
    u, w = 0.5 * (x + 1), 0.5 * w
    dev = torch.device("cuda")
    P = lambda i: torch.tensor(v[i], device=dev)  # noqa: E731
    q1, q2 = P(e[:, 0]), P(e[:, 1])
    length = (q1 - q2).norm(dim=1)
    kh, pol = (torch.tensor(c, device=dev) for c in _incidences(case, seed))
    V = torch.zeros((case["rhs"], len(e)), dtype=torch.complex128, device=dev)
    for side, sign in ((0, 1.0), (1, -1.0)):
        p = P(opposite[:, side])
        for a in range(6):
            for b in range(6):
                rho = u[a] * (q1 - p) + u[b] * (1 - u[a]) * (q2 - p)
                amp = (sign * w[a] * w[b] * (1 - u[a])) * length[:, None] * rho
                V -= (pol @ amp.T) * torch.exp(-2j * math.pi * (kh @ (p + rho).T))
    return V


def exact(case, seed):
    if case["do"] == "translate":
        return _exact_translate(case, seed)
    if case["do"] == "planewave":
        return _exact_planewave(case, seed)
    nt, npf = _grid(case)
    n_rwg, members, template, ranks = _lay(case)
    R, do, G, nd = case["rhs"], case["do"], len(members), nt * npf
    dev = torch.device("cuda")
    sets = [[tuple(torch.tensor(c, device=dev) for c in (ut, up, ub, core.reshape(-1, core.shape[2], order="F")))
             for ut, up, ub, core in per] for per in _factor_sets(_factor_key(case))]
    ids = [torch.tensor(m, device=dev) for m in members]
    x = spec = None
    if do == "disaggregate":
        spec = _randn((R, G, 2, nd), seed).to(torch.complex128)
    else:
        x = _randn((n_rwg,) if do == "host" else (R, n_rwg), seed).reshape(R, n_rwg).to(torch.complex128)
        spec = torch.empty((R, G, 2, nd), dtype=torch.complex128, device=dev)
        for g in range(G):
            xg = x[:, ids[g]].T
            for al in range(2):
                ut, up, ub, core = sets[template[g]][al]
                rt, rp, rb, _ = ranks[template[g]][al]
                t = ub[:len(ids[g]) * rb].reshape(rb, len(ids[g])) @ xg
                M = (core @ t).reshape(rp, rt, R)  # element a + rt b
                spec[:, g, al] = torch.einsum("pb,bar,ta->rpt", up, M, ut).reshape(R, nd)
    if do == "aggregate":
        return {"spectra": spec}
    beta = case["beta"]
    y = _randn((R, n_rwg), seed + 1000003).to(torch.complex128) if beta else torch.zeros((R, n_rwg), dtype=torch.complex128, device=dev)
    y *= beta
    w = torch.tensor(_weights(case).astype(np.float32), device=dev).to(torch.float64)
    for g in range(G):
        for al in range(2):
            ut, up, ub, core = sets[template[g]][al]
            rt, rp, rb, _ = ranks[template[g]][al]
            gw = (spec[:, g, al] * w).conj().reshape(R, npf, nt)
            H = torch.einsum("ta,rpt,pb->bar", ut, gw, up).reshape(rp * rt, R)
            yg = ub[:len(ids[g]) * rb].reshape(rb, len(ids[g])).T @ (core.T @ H)
            y[:, ids[g]] += yg.conj().T
    if do == "host":
        return y.reshape(n_rwg).cpu()
    return {"spectra": spec, "y": y} if do == "matvec" else {"y": y}
