"""What a user of this framework has it do, as timed cases.

The framework solves acoustic scattering by many bodies in a layered medium with an FMM-accelerated
boundary integral equation.  Its users build a geometry, then mostly multiply by the operator: directly,
with blocks of incidence angles, over several geometries at once, or inside GMRES; they also evaluate
fields and run whole requests.  Every case goes through ``paper_2511_12450_gb300.lfmm``.

``listed`` gives the fixed cases, ``draw`` more of the same ranges, ``prepare`` what a program holds
before the call, ``run`` one pass, ``work`` what it cannot do without, ``exact`` its outputs from dense
64-bit sums: free space by Hankel functions, the layers' reflections by a contour integral over plane
waves with one interface system per wave.
"""

import math

import numpy as np
import torch

from paper_2511_12450_gb300 import lfmm

# Layered media of the framework's own configurations: interface heights, wavenumbers, densities.
MEDIA = {
    "half": ([0.0], [2.0, 4.0], [1.0, 2.0]),
    "three": ([0.0, -2.0], [4.0, 6.0, 8.0], [1.0, 2.0, 3.0]),
    "four": ([0.0, -2.0, -4.0], [6.0, 10.0, 8.0, 12.0], [1.0, 2.0, 3.0, 4.0]),
    "deep": ([0.0, -6.0, -12.0], [6.0, 10.0, 8.0, 12.0], [1.0, 2.0, 3.0, 4.0]),
    "six": ([0.0, -1.0, -2.0, -3.0, -4.0], [2.0, 3.0, 6.0, 5.0, 8.0, 10.0], [1.0, 2.0, 3.0, 4.0, 5.0, 6.0]),
}


def listed():
    return [
        # one small scatterer above a half space: the smallest call, where launches and latency count,
        # as in a parameter study over many tiny problems
        {"name": "matvec_tiny", "kind": "matvec", "medium": "half", "bodies": 1, "nodes": 256, "cross": False,
         "leaf": 64, "cols": 1, "mixed": False, "combined": False},
        # a few ragged bodies between three layers: ordinary interactive work
        {"name": "matvec_small", "kind": "matvec", "medium": "three", "bodies": 7, "nodes": 487, "cross": False,
         "leaf": 64, "cols": 1, "mixed": False, "combined": False},
        # the benchmark's configuration: 64 bodies x 1024 nodes in three layers, bodies across interfaces
        {"name": "matvec_c2", "kind": "matvec", "medium": "three", "bodies": 64, "nodes": 1024, "cross": True,
         "leaf": 64, "cols": 1, "mixed": False, "combined": False},
        # the same size in the precision form with single-precision vectors (sweeps that need six digits)
        {"name": "matvec_mixed", "kind": "matvec", "medium": "three", "bodies": 64, "nodes": 1024, "cross": False,
         "leaf": 64, "cols": 1, "mixed": True, "combined": False},
        # the large end: a quarter of a million points in four layers, coarse levels many wavelengths wide
        {"name": "matvec_large", "kind": "matvec", "medium": "deep", "bodies": 256, "nodes": 1024, "cross": True,
         "leaf": 64, "cols": 1, "mixed": False, "combined": False},
        # the second-kind operator users take for fast GMRES convergence, odd sizes
        {"name": "matvec_combined", "kind": "matvec", "medium": "half", "bodies": 31, "nodes": 641, "cross": False,
         "leaf": 64, "cols": 1, "mixed": False, "combined": True},
        # a few incidence angles at once in FP64 (block products of a multi-angle solve)
        {"name": "block_fp64", "kind": "matvec", "medium": "four", "bodies": 11, "nodes": 1117, "cross": False,
         "leaf": 64, "cols": 5, "mixed": False, "combined": False},
        # 32 incidence angles as one block in the precision form (an angle sweep)
        {"name": "block_mixed", "kind": "matvec", "medium": "three", "bodies": 40, "nodes": 1030, "cross": False,
         "leaf": 64, "cols": 32, "mixed": True, "combined": False},
        # several uneven geometries multiplied in shared launches (batched serving)
        {"name": "batch", "kind": "batch", "geometries": 5, "bodies": 4, "nodes": 1024, "growth": 1.6, "cols": 1},
        # a preconditioned GMRES solve to 1e-8, six layers, flower-shaped scatterers across the interfaces
        {"name": "solve", "kind": "solve", "nodes": 12000, "tol": 1e-8},
        # the scattered field of a known density on a grid of points (pictures, far-field maps)
        {"name": "field", "kind": "field", "medium": "three", "bodies": 16, "nodes": 1024, "targets": 6007},
        # a whole cold request: geometry set-up, right-hand side, solve (the serving path of one user)
        {"name": "request", "kind": "request", "medium": "half", "bodies": 9, "nodes": 911, "tol": 1e-8},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["matvec", "matvec", "matvec", "block", "batch", "solve", "field", "request"])
    if kind in ("matvec", "block"):
        n = _log(rng, 256, 131072) if kind == "matvec" else _log(rng, 2000, 41000)
        bodies = max(1, min(128, round(n / _log(rng, 200, 1100))))
        return {"kind": "matvec", "medium": rng.choice(["half", "three", "four", "deep"]), "bodies": bodies,
                "nodes": max(60, round(n / bodies)), "cross": rng.random() < 0.5, "leaf": rng.choice([32, 64, 64]),
                "cols": 1 if kind == "matvec" else rng.randint(2, 32), "mixed": rng.random() < 0.35,
                "combined": rng.random() < 0.2}
    if kind == "batch":
        return {"kind": "batch", "geometries": rng.randint(2, 6), "bodies": rng.randint(1, 5),
                "nodes": round(_log(rng, 300, 1100)), "growth": rng.uniform(1.0, 1.6), "cols": rng.randint(1, 3)}
    if kind == "solve":
        return {"kind": "solve", "nodes": 5 * round(_log(rng, 600, 4000)), "tol": 1e-8}
    if kind == "field":
        return {"kind": "field", "medium": rng.choice(["half", "three", "four"]), "bodies": rng.randint(3, 20),
                "nodes": round(_log(rng, 300, 1100)), "targets": round(_log(rng, 300, 9000))}
    return {"kind": "request", "medium": rng.choice(["half", "three"]), "bodies": rng.randint(2, 10),
            "nodes": round(_log(rng, 300, 1100)), "tol": 1e-8}


# ---------------------------------------------------------------------------------------- inputs

def _bodies(rng, medium, count, nodes, cross, gap=0.05, margin=0.1):
    """Circles and ellipses (half each) in a field as wide as the count asks for; with cross=False each keeps
    ``margin`` from the interfaces, with cross=True only its vertices and midpoints keep off them."""
    yint = np.asarray(MEDIA[medium][0])
    deep = medium == "deep"
    ylo, yhi = float(yint[-1]) - (3.0 if deep else 2.0), 3.0 if deep else 2.0
    half = max(2.0, 0.9 * count / (yhi - ylo))
    centres, radii, out = [], [], []
    while len(out) < count:
        cx, cy = rng.uniform(-half, half), rng.uniform(ylo, yhi)
        a, b = rng.uniform(0.2, 0.6, 2)
        rot = rng.uniform(0.0, math.pi)
        if rng.random() < 0.5:
            b = a
        r = max(a, b)
        if not cross and np.min(np.abs(cy - yint)) < r + margin:
            half *= 1.0005
            continue
        if centres and np.any(np.hypot(np.asarray(centres)[:, 0] - cx, np.asarray(centres)[:, 1] - cy) < np.asarray(radii) + r + gap):
            half *= 1.0005   # the field widens slowly, so that every count finds room
            continue
        t = 2.0 * np.pi * np.arange(nodes) / nodes
        ex, ey = a * np.cos(t), b * np.sin(t)
        v = np.stack([cx + math.cos(rot) * ex - math.sin(rot) * ey, cy + math.sin(rot) * ex + math.cos(rot) * ey], axis=1)
        ys = np.concatenate([v[:, 1], 0.5 * (v[:, 1] + np.roll(v[:, 1], -1))])
        if np.min(np.abs(ys[:, None] - yint[None, :])) < 1e-5:
            continue
        centres.append((cx, cy))
        radii.append(r)
        out.append(v)
    return out


def _flowers(rng, nodes):
    """The five flower scatterers of the paper's third example, turned at random."""
    per = nodes // 5
    t = 2.0 * np.pi * np.arange(per) / per
    out = []
    for cx, cy in [(-1.5, 0.0), (1.5, 0.0), (0.0, -2.0), (-1.5, -4.0), (1.5, 4.0)]:
        r = 0.7 + 0.2 * np.sin(5.0 * (t - rng.uniform(0.0, 2.0 * np.pi)))
        out.append(np.stack([cx + r * np.cos(t), cy + 1e-3 * rng.uniform(0.1, 1.0) + r * np.sin(t)], axis=1))
    return out


def _elements(bodies):
    """Chord midpoints, lengths and outward normals."""
    pts, w, nrm = [], [], []
    for v in bodies:
        d = np.roll(v, -1, axis=0) - v
        ln = np.hypot(d[:, 0], d[:, 1])
        pts.append(0.5 * (v + np.roll(v, -1, axis=0)))
        w.append(ln)
        nrm.append(np.stack([d[:, 1], -d[:, 0]], axis=1) / ln[:, None])
    return np.concatenate(pts), np.concatenate(w), np.concatenate(nrm)


def _columns(rng, n, cols, dtype):
    v = rng.standard_normal((cols, n)) + 1j * rng.standard_normal((cols, n))
    v = torch.from_numpy(v if cols > 1 else v[0]).to("cuda")
    return v.to(dtype)


def _batch_sizes(case):
    media = ["half", "three", "four"]
    return [(media[i % 3], max(1, round(case["bodies"] * case["growth"] ** i)), case["nodes"] - 17 * i)
            for i in range(case["geometries"])]


def _inputs(case, seed):
    """The host side of a case, from the seed alone: (medium name, points, weights, normals) per geometry, and rng."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "batch":
        return [(m, *_elements(_bodies(rng, m, b, n, False))) for m, b, n in _batch_sizes(case)], rng
    if kind == "solve":
        return [("six", *_elements(_flowers(rng, case["nodes"])))], rng
    return [(case["medium"], *_elements(_bodies(rng, case["medium"], case["bodies"], case["nodes"], case.get("cross", False))))], rng


def _targets(rng, case, pts):
    """Points of a picture around the bodies, off the boundaries and the interfaces."""
    yint = np.asarray(MEDIA[case["medium"]][0])
    lo, hi = pts.min(axis=0) - 1.0, pts.max(axis=0) + 1.0
    out = np.empty((0, 2))
    while out.shape[0] < case["targets"]:
        t = rng.uniform(lo, hi, (2 * case["targets"], 2))
        t = t[np.min(np.abs(t[:, 1:2] - yint[None, :]), axis=1) > 0.1]
        d = np.full(t.shape[0], np.inf)
        for i in range(0, pts.shape[0], 256):
            d = np.minimum(d, np.min(np.hypot(t[:, None, 0] - pts[None, i:i + 256:16, 0], t[:, None, 1] - pts[None, i:i + 256:16, 1]), axis=1))
        out = np.concatenate([out, t[d > 0.06]])
    return out[:case["targets"]]


def _dtype(case):
    return torch.complex64 if case.get("mixed") else torch.complex128


def prepare(case, seed):
    geos, rng = _inputs(case, seed)
    kind = case["kind"]
    if kind == "request":
        m, pts, w, nrm = geos[0]
        return {"case": case, "medium": m, "pts": pts, "w": w, "nrm": nrm, "angle": float(rng.uniform(0.1, 3.0))}
    built = []
    for m, pts, w, nrm in geos:
        M = lfmm.medium_create(*MEDIA[m])
        combined = bool(case.get("combined"))
        built.append(lfmm.geometry_build(M, pts, w, nrm if combined else None, p=20, leaf_size=case.get("leaf", 64),
                                         combined=combined))
    s = {"case": case, "G": built}
    if kind == "solve":
        s["b"] = lfmm.rhs_plane_wave(built[0], [float(rng.uniform(0.4, 2.7))], device=True)
        return s
    if kind == "field":
        s["targets"] = _targets(rng, case, geos[0][1])
        s["x"] = [_columns(rng, built[0].n, 1, torch.complex128)]
        return s
    s["x"] = [_columns(rng, G.n, case["cols"], _dtype(case)) for G in built]
    if case.get("mixed"):
        lfmm.matvec(built[0], s["x"][0], mixed=True)   # a program keeps the precision form's tables, built on first use
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "matvec":
        return lfmm.matvec(state["G"][0], state["x"][0], mixed=case["mixed"])
    if kind == "batch":
        return lfmm.matvec_batch(state["G"], state["x"])
    if kind == "solve":
        x, _ = lfmm.gmres_solve(state["G"][0], state["b"], tol=case["tol"])
        return x
    if kind == "field":
        return lfmm.eval_field(state["G"][0], state["x"][0], state["targets"])
    M = lfmm.medium_create(*MEDIA[state["medium"]])
    G = lfmm.geometry_build(M, state["pts"], state["w"])
    b = lfmm.rhs_plane_wave(G, [state["angle"]])
    x, _ = lfmm.gmres_solve(G, b, tol=case["tol"])
    G.destroy()
    return {"rhs": b, "phi": x}


# ---------------------------------------------------------------------------------------- work

def _points(case):
    kind = case["kind"]
    if kind == "batch":
        return sum(b * n for _, b, n in _batch_sizes(case))
    if kind == "solve":
        return case["nodes"]
    return case["bodies"] * case["nodes"]


def work(case):
    """Vectors and elements read and written once; a product's operations from the method: the leaf expansions
    and stored near rows per point, and about 16 thousand for its share of the translations, or the dense sum
    where that is less.  A solve is some 70 products and preconditioner steps, a request a solve and a set-up."""
    n, cols = _points(case), case.get("cols", 1)
    m = case.get("targets", 0)
    item = 8 if case.get("mixed") else 16
    product = min(8.0 * (n + m) * n, 1.8e4 * (n + m))
    times = {"solve": 70, "request": 75}.get(case["kind"], 1)
    return {"bytes": float((n * cols + max(m, n * cols if not m else 0)) * item + 24 * n + 16 * m), "flops": product * cols * times}


# ---------------------------------------------------------------------------------------- 64-bit reference

def _ky(k, lam):
    s = torch.sqrt((k * k - lam * lam).to(torch.complex128))
    return torch.where(s.imag < 0, -s, s)


def _bessel(z):
    """J0, Y0, J1, Y1 of z > 0 in 64 bits (torch's own are good to about 1e-7): ascending series below 3, downward
    recurrence with Neumann's series for Y up to 25, Hankel's asymptotic series beyond."""
    out = [torch.empty_like(z) for _ in range(4)]
    eg = 0.57721566490153286061
    for lo, hi in ((0.0, 3.0), (3.0, 25.0), (25.0, math.inf)):
        at = (z >= lo) & (z < hi)
        x = z[at]
        if not x.numel():
            continue
        if hi == 3.0:
            q, a, b, h = -0.25 * x * x, torch.ones_like(x), torch.ones_like(x), 0.0
            j0, j1, s0, s1 = a.clone(), b.clone(), torch.zeros_like(x), (1.0 - 2.0 * eg) * b
            for n in range(1, 20):
                a, b, h = a * q / (n * n), b * q / (n * (n + 1)), h + 1.0 / n
                j0, j1, s0, s1 = j0 + a, j1 + b, s0 - h * a, s1 + (2.0 * h + 1.0 / (n + 1) - 2.0 * eg) * b
            j1, s1, ln = 0.5 * x * j1, 0.5 * x * s1, torch.log(0.5 * x)
            v = [j0, (2.0 / math.pi) * ((ln + eg) * j0 + s0), j1, (2.0 / math.pi) * (ln * j1 - 1.0 / x) - s1 / math.pi]
        elif hi == 25.0:
            up, cur = torch.zeros_like(x), torch.full_like(x, 1e-150)
            norm, s0, s1 = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(x)
            for n in range(64, 0, -1):   # cur = J_n up to a factor
                if n % 2 == 0:
                    norm, s0 = norm + 2.0 * cur, s0 + ((-1) ** (n // 2) / (n // 2)) * cur
                elif n > 1:
                    i = n // 2
                    s1 = s1 + ((-1) ** i * n / (i * (i + 1.0))) * cur
                else:
                    j1 = cur
                up, cur = cur, (2.0 * n / x) * cur - up
            norm, ln = norm + cur, torch.log(0.5 * x) + eg
            j0, j1, s0, s1 = cur / norm, j1 / norm, s0 / norm, s1 / norm
            v = [j0, (2.0 / math.pi) * (ln * j0 - 2.0 * s0), j1,
                 (2.0 / math.pi) * ((ln - 1.0) * j1 - j0 / x - s1)]
        else:
            v = []
            for nu in (0, 1):
                p, q, t = torch.ones_like(x), torch.zeros_like(x), torch.ones_like(x)
                for n in range(1, 24):
                    t = t * ((4.0 * nu * nu - (2 * n - 1) ** 2) / (8.0 * n)) / x
                    if n % 2:
                        q = q + (-1) ** (n // 2) * t
                    else:
                        p = p + (-1) ** (n // 2) * t
                c, f = torch.cos(x - (0.5 * nu + 0.25) * math.pi), torch.sqrt(2.0 / (math.pi * x))
                d = torch.sin(x - (0.5 * nu + 0.25) * math.pi)
                v += [f * (p * c - q * d), f * (p * d + q * c)]
        for o, w in zip(out, v):
            o[at] = w
    return out


def _free(k, pt, ps, s, nrm_s, coupling):
    """sum_e s_e (i/4) H_0(k |r - c_e|) for the columns of s, coincident points left out; with normals the
    dipole along them minus i k times that."""
    out = torch.zeros((pt.shape[0], s.shape[1]), dtype=torch.complex128, device="cuda")
    step = max(1, (1 << 24) // max(1, ps.shape[0]))
    for i in range(0, pt.shape[0], step):
        d = ps[None, :, :] - pt[i:i + step, None, :]
        r = torch.hypot(d[..., 0], d[..., 1])
        zero = r == 0
        z = k * torch.where(zero, torch.ones_like(r), r)
        j0, y0, j1, y1 = _bessel(z)
        g = 0.25j * torch.complex(j0, y0)
        if nrm_s is not None:
            h1 = torch.complex(j1, y1)
            cosn = (d * nrm_s[None, :, :]).sum(-1) * k / z
            g = -0.25j * k * h1 * cosn - 1j * coupling * g
        g = torch.where(zero, torch.zeros_like(g), g)
        out[i:i + step] = g @ s
    return out


def _contour(kmax, X, hmin):
    """Nodes and weights (with the 1/2pi) of a path from -Lambda to Lambda below the positive singularities."""
    gx, gw = np.polynomial.legendre.leggauss(16)
    T, h = kmax + 2.0, min(0.3, 1.0 / max(X, 1.0))
    end = T + kmax + 40.0 / hmin
    e1 = np.linspace(0.0, T, 2 + int(T / (0.5 * h)))
    e2 = np.linspace(T, end, 2 + int((end - T) / min(1.0, 9.0 / max(X, 1.0))))
    lam, wt = [], []
    for e, bent in ((e1, True), (e2, False)):
        mid, hw = 0.5 * (e[1:] + e[:-1]), 0.5 * (e[1:] - e[:-1])
        t = (mid[:, None] + hw[:, None] * gx[None, :]).reshape(-1)
        w = (hw[:, None] * gw[None, :]).reshape(-1)
        lam.append(t - 1j * h * np.sin(np.pi * t / T) if bent else t + 0j)
        wt.append(w * (1.0 - 1j * h * np.pi / T * np.cos(np.pi * t / T)) if bent else w + 0j)
    lam, wt = np.concatenate(lam), np.concatenate(wt) / (2.0 * np.pi)
    return np.concatenate([-lam[::-1], lam]), np.concatenate([wt[::-1], wt])


def _product(medium, pts, w, nrm, X, targets):
    """K X (targets None) or the scattered field at the targets, columns of X, or None where it costs too much."""
    yint, k, eta = (np.asarray(v, dtype=np.float64) for v in MEDIA[medium])
    L = yint.size
    dev = "cuda"
    tp = pts if targets is None else targets
    hs, ht = np.abs(pts[:, 1:2] - yint[None, :]), np.abs(tp[:, 1:2] - yint[None, :])
    hmin = float(np.min(hs.min(axis=0) + ht.min(axis=0)))
    both = np.concatenate([pts, tp])
    lam, wt = _contour(k.max(), float(np.ptp(both[:, 0])), hmin)
    cost = 4.0 * lam.size * (pts.shape[0] + tp.shape[0]) + float(pts.shape[0]) * tp.shape[0]
    if hmin < 1e-3 or cost > 5e10:
        return None
    lay_s, lay_t = (np.sum(p[:, 1:2] < yint[None, :], axis=1) for p in (pts, tp))
    P, Q = torch.from_numpy(pts).to(dev), torch.from_numpy(np.ascontiguousarray(tp)).to(dev)
    ls, lt = torch.from_numpy(lay_s).to(dev), torch.from_numpy(lay_t).to(dev)
    kt, et, wd = (torch.from_numpy(v).to(dev) for v in (k, eta, w))
    N = torch.from_numpy(nrm).to(dev) if nrm is not None else None
    S = X * (wd / et[ls])[:, None]      # strengths of the physical sources, by reciprocity
    U = torch.zeros((tp.shape[0], X.shape[1]), dtype=torch.complex128, device=dev)
    for m in range(L + 1):
        si, ti = (ls == m).nonzero()[:, 0], (lt == m).nonzero()[:, 0]
        if si.numel() and ti.numel():
            U[ti] += _free(float(k[m]), Q[ti], P[si], S[si], None if N is None else N[si], float(k[m]))
    lamt, wtt = torch.from_numpy(lam).to(dev), torch.from_numpy(wt).to(dev)
    step = max(64, (1 << 27) // (16 * max(pts.shape[0], tp.shape[0])))
    for a in range(0, lam.size, step):
        la, wa = lamt[a:a + step], wtt[a:a + step]
        q, c = la.numel(), X.shape[1]
        ky = torch.stack([_ky(float(kk), la) for kk in k])                       # [L+1, q]
        A = torch.zeros((q, 2 * L, 2 * L), dtype=torch.complex128, device=dev)   # up-going 0..L-1, down-going L..2L-1
        R = torch.zeros((q, 2 * L, c), dtype=torch.complex128, device=dev)
        for j in range(L):
            up, lo = j, j + 1
            A[:, 2 * j, up] += 1.0
            A[:, 2 * j + 1, up] += 1j * eta[up] * ky[up]
            if up >= 1:
                e = torch.exp(1j * ky[up] * float(yint[up - 1] - yint[up]))
                A[:, 2 * j, L + up - 1] += e
                A[:, 2 * j + 1, L + up - 1] += -1j * eta[up] * ky[up] * e
            if lo <= L - 1:
                e = torch.exp(1j * ky[lo] * float(yint[lo - 1] - yint[lo]))
                A[:, 2 * j, lo] -= e
                A[:, 2 * j + 1, lo] -= 1j * eta[lo] * ky[lo] * e
            A[:, 2 * j, L + lo - 1] -= 1.0
            A[:, 2 * j + 1, L + lo - 1] += 1j * eta[lo] * ky[lo]
            for layer, sgn in ((up, 1.0), (lo, -1.0)):   # direct waves: down from the layer above, up from the one below
                si = (ls == layer).nonzero()[:, 0]
                if not si.numel():
                    continue
                p = P[si]
                ex = torch.exp(1j * (ky[layer][:, None] * (sgn * (p[:, 1] - float(yint[j])))[None, :] - la[:, None] * p[None, :, 0]))
                if N is not None:   # normal derivative at the source, minus i k
                    n2 = N[si]
                    ex = ex * (1j * (sgn * ky[layer][:, None] * n2[None, :, 1] - la[:, None] * n2[None, :, 0]) - 1j * float(k[layer]))
                v = (ex @ S[si]) * (0.5j / ky[layer])[:, None]
                R[:, 2 * j] -= sgn * v
                R[:, 2 * j + 1] += 1j * eta[layer] * ky[layer][:, None] * v
        sol = torch.linalg.solve(A, R) * wa[:, None, None]
        for m in range(L + 1):
            ti = (lt == m).nonzero()[:, 0]
            if not ti.numel():
                continue
            t = Q[ti]
            for amp, h in ((m if m <= L - 1 else -1, None), (L + m - 1 if m >= 1 else -1, 1)):
                if amp < 0:
                    continue
                hh = t[:, 1] - float(yint[m]) if h is None else float(yint[m - 1]) - t[:, 1]
                U[ti] += torch.exp(1j * (ky[m][None, :] * hh[:, None] + la[None, :] * t[:, 0:1])) @ sol[:, amp]
    if targets is not None:
        return U
    U *= et[lt][:, None]
    ks = kt[ls]
    self_term = (0.25j - (0.57721566490153286 + torch.log(ks * wd / 4.0) - 1.0) / (2.0 * math.pi)) * wd
    if N is not None:
        self_term = 0.5 - 1j * ks * self_term
    return U + self_term[:, None] * X


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "request"):
        return None
    geos, rng = _inputs(case, seed)
    targets = _targets(rng, case, geos[0][1]) if kind == "field" else None
    out = []
    for m, pts, w, nrm in geos:
        X = _columns(rng, pts.shape[0], case.get("cols", 1), _dtype(case)).to(torch.complex128)
        X = X.reshape(-1, pts.shape[0]).T.contiguous()
        y = _product(m, pts, w, nrm if case.get("combined") else None, X, targets)
        if y is None:
            out.append(None)
        elif kind == "field":
            out.append(y[:, 0].cpu().numpy())
        else:
            out.append(y.T.contiguous() if case["cols"] > 1 else y[:, 0].contiguous())
    if kind == "batch":
        return out
    return out[0]
