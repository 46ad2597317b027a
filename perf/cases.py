"""What the performance of this framework is measured on: the calls a user makes, from the smallest surface to the
5,000-atom size, through the public entry points of ``paper_2108_10481_gb300``.

Surfaces: a geodesic sphere of frequency f (20 f^2 triangles, 10 f^2 + 2 vertices) at about four vertices per square
Angstrom, deformed by seeded bumps and dents, its vertices moved about within the surface, and its triangles listed
slab by slab as a level-set extraction lists them. f = 4 is about the smallest sphere of the tests, f = 8 the
closed-form sphere of 1,280 triangles, f = 32 the 20-charge sphere of 20,480, f = 44 the size of the 500-atom molecule
and f = 105 that of the 5,000-atom one. Charges: one atom for about 80 triangles, away from the surface. Physics as in
the benchmark (permittivities 4 and 80, inverse Debye length 0.125 per Angstrom).

Plans: "reference" is the 6-point far rule with 4 singular Gauss points, "band" the benchmark's autotuned kind of plan
(3-point rule beyond three radii, 6-point rule inside, 3 Gauss points on coincident pairs).

Calls that compute in single precision (PB_F32, PB_F32_ACCURATE, PB_MIXED) hand their results back in float64 storage;
a pass keeps them as float32, which is the precision that they carry. PB_F64 results stay float64.
"""
import math

import numpy as np
import torch

import paper_2108_10481_gb300 as pb

PARAMS = (4.0, 80.0, 0.125)
PLANS = {"reference": {"far_q": 6, "n_ss": 4},
         "band": {"far_q": 3, "n_ss": 4, "band_eta": 3.0, "band_q": 6, "n_ss_coin": 3}}
PREC = {"f64": pb.PB_F64, "f32": pb.PB_F32, "split": pb.PB_F32_ACCURATE, "mixed": pb.PB_MIXED}


def listed():
    return [
        # one FP64 application on the smallest sphere of the tests: launches and latency
        {"name": "apply_f64_small", "do": "apply", "f": 4, "plan": "reference", "form": "direct_int", "prec": "f64"},
        # one FP64 application of the V/K + D/T form on the closed-form sphere: what every default (FP64) solve repeats
        {"name": "apply_f64", "do": "apply", "f": 8, "plan": "reference", "form": "juffer", "prec": "f64"},
        # one FP32 application below the treecode's size: direct pair sums, a served small molecule's inner iteration
        {"name": "apply_f32_direct", "do": "apply", "f": 16, "plan": "reference", "form": "lu", "prec": "f32"},
        # one FP32 treecode application, V/K rows, 500-atom size: an inner iteration of Case 2
        {"name": "apply_f32_tree", "do": "apply", "f": 44, "plan": "band", "form": "direct_int", "prec": "f32"},
        # the same for V/K + D/T rows at the 5,000-atom size: an inner iteration of the benchmark's Case 10
        {"name": "apply_f32_tree_large", "do": "apply", "f": 105, "plan": "band", "form": "juffer", "prec": "f32"},
        # the exact outer residual of a mixed solve on the 20-charge sphere's size
        {"name": "residual_split", "do": "apply", "f": 32, "plan": "band", "form": "juffer", "prec": "split"},
        # near-field set-up with the reference plan on a small surface, then the block-diagonal preconditioner
        # and a first application with it
        {"name": "near_reference", "do": "near", "f": 10, "plan": "reference", "form": "direct_int"},
        # the same with the band plan at the 500-atom size
        {"name": "near_band", "do": "near", "f": 44, "plan": "band", "form": "juffer"},
        # right-hand side and reaction potential of the 500-atom size, as the mixed path computes them
        {"name": "charges_split", "do": "charges", "f": 44, "plan": "band", "form": "juffer", "prec": "split"},
        # the mass preconditioner in FP64 on the 20-charge sphere's size: the norm of every outer residual
        {"name": "mass_f64", "do": "precond", "f": 32, "plan": "band", "form": "juffer", "precond": "scaled_mass",
         "prec": "f64"},
        # a whole default solve of a small surface: load, near field, charges, FP64 Calderon GMRES, energy (Case 23)
        {"name": "whole_f64", "do": "whole", "f": 5, "plan": "reference", "form": "pmchwt_int",
         "precond": "scaled_calderon_int", "prec": "f64"},
        # the benchmark's step on the 500-atom size: the same in mixed precision (Case 10)
        {"name": "whole_mixed", "do": "whole", "f": 44, "plan": "band", "form": "juffer", "precond": "scaled_mass",
         "prec": "mixed"},
    ]


SYSTEMS = [("direct_int", "block_diag"), ("juffer", "scaled_mass"), ("lu", "mass"),
           ("pmchwt_int", "scaled_calderon_int")]  # the served cases 2, 10, 12 and 23


def draw(rng):
    """One more case of the same kinds, its size spread over the logarithm of the kind's range."""
    def freq(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    do = rng.choice(["apply", "apply", "apply", "near", "charges", "precond", "whole"])
    form, precond = rng.choice(SYSTEMS)
    plan = rng.choice(["reference", "band"])
    if do == "apply":
        prec = rng.choice(["f64", "f32", "f32", "split"])
        top = {"f64": 9, "f32": 105, "split": 44}[prec]
        f = freq(2 if prec == "f64" else 5, top)
        return {"do": do, "f": f, "plan": "band" if f > 22 else plan, "form": form, "prec": prec}
    if do == "near":
        return {"do": do, "f": freq(2, 44), "plan": plan, "form": rng.choice(["direct_int", "juffer", "lu"])}
    if do == "charges":
        prec = rng.choice(["f64", "split"])
        return {"do": do, "f": freq(3, 30 if prec == "f64" else 80), "plan": plan, "form": form, "prec": prec}
    if do == "precond":
        form, precond = rng.choice([("juffer", "scaled_mass"), ("lu", "mass"), ("muller_int", "mass")])
        return {"do": do, "f": freq(3, 80), "plan": "band", "form": form, "precond": precond,
                "prec": rng.choice(["f64", "f32"])}
    prec = rng.choice(["f64", "mixed"])
    if prec == "f64":
        return {"do": do, "f": freq(2, 7), "plan": "reference", "form": form, "precond": precond, "prec": prec}
    # Case 23 on band plans stalls above 1e-6 in mixed precision, so the mixed solves are the other three
    form, precond = rng.choice(SYSTEMS[:3])
    return {"do": do, "f": freq(8, 44), "plan": "band", "form": form, "precond": precond, "prec": prec}


# ------------------------------------------------------------------ surfaces
def _geodesic(f):
    """(unit vertices, triangles, outward) of the icosahedron with every face split into f^2."""
    g = (1.0 + 5.0 ** 0.5) / 2.0
    corners = np.array([[s * a, t * b, 0.0] for a, b in ((1.0, g),) for s in (1, -1) for t in (1, -1)])
    corners = np.concatenate([np.roll(corners, k, axis=1) for k in range(3)])
    d = np.linalg.norm(corners[:, None] - corners[None], axis=2)
    near = (d > 0) & (d < 2.01)
    faces = [(i, j, k) for i in range(12) for j in range(i + 1, 12) for k in range(j + 1, 12)
             if near[i, j] and near[j, k] and near[i, k]]
    points, tris, base = [], [], 0
    index = -np.ones((f + 1, f + 1), dtype=np.int64)
    ii, jj = np.array([(i, j) for i in range(f + 1) for j in range(f + 1 - i)]).T
    index[ii, jj] = np.arange(len(ii))
    up = np.array([(index[i, j], index[i + 1, j], index[i, j + 1]) for i in range(f) for j in range(f - i)])
    down = np.array([(index[i + 1, j], index[i + 1, j + 1], index[i, j + 1])
                     for i in range(f) for j in range(f - i - 1)], dtype=np.int64).reshape(-1, 3)
    for a, b, c in faces:
        a, b, c = corners[a], corners[b], corners[c]
        p = ((f - ii - jj)[:, None] * a + ii[:, None] * b + jj[:, None] * c) / f
        t = np.concatenate([up, down])
        if np.dot(np.cross(b - a, c - a), a + b + c) < 0:
            t = t[:, ::-1]
        points.append(p)
        tris.append(t + base)
        base += len(p)
    p = np.concatenate(points)
    key = np.round(p * 1e7).astype(np.int64)  # points on shared edges are one vertex
    _, first, inv = np.unique(key, axis=0, return_index=True, return_inverse=True)
    v = p[first]
    return v / np.linalg.norm(v, axis=1, keepdims=True), inv.reshape(-1)[np.concatenate(tris)]


def _surface(f, seed):
    """(vertices float64, triangles int32, charge positions, charges), numpy."""
    rng = np.random.default_rng([seed, f])
    u, t = _geodesic(f)
    radius = math.sqrt(len(u) / (16.0 * math.pi))  # four vertices per square Angstrom
    edge = 1.1 / f
    u = u + rng.uniform(-0.12, 0.12, u.shape) * edge  # irregular triangles
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    n_bumps = 24
    c = rng.standard_normal((n_bumps, 3))
    c /= np.linalg.norm(c, axis=1, keepdims=True)
    amp = rng.uniform(-0.12, 0.12, n_bumps)
    r = radius * (1.0 + np.exp(12.0 * (u @ c.T - 1.0)) @ amp)
    v = u * r[:, None]
    mid = v[t].mean(axis=1)
    cell = np.floor(mid / (1.5 * edge * radius))
    t = t[np.lexsort((cell[:, 2], cell[:, 1], cell[:, 0]))]  # slab by slab
    n_q = max(1, len(t) // 80)
    p = rng.standard_normal((n_q, 3))
    p *= (rng.uniform(0.0, 1.0, n_q) ** (1 / 3) * max(0.5 * r.min(), r.min() - 2.2) /
          np.linalg.norm(p, axis=1))[:, None]
    q = rng.uniform(-0.8, 0.8, n_q)
    return (np.ascontiguousarray(v), np.ascontiguousarray(t, dtype=np.int32), np.ascontiguousarray(p),
            np.ascontiguousarray(q))


def _vector(v, xq, q, seed):
    """[u; v] as an iteration meets it: the charges' potential at the vertices and rough parts, of norm one."""
    rng = np.random.default_rng([seed, 77])
    k = slice(0, min(len(q), 64))
    phi = (q[k] / np.linalg.norm(v[:, None] - xq[None, k], axis=2)).sum(axis=1)
    x = np.concatenate([phi, phi])
    x = x / np.linalg.norm(x) + 0.3 * rng.standard_normal(len(x)) / math.sqrt(len(x))
    return x / np.linalg.norm(x)


# ------------------------------------------------------------------- the calls
_context = []


def _ctx():
    if not _context:
        _context.append(pb.pb_init(torch.cuda.current_device()))
    return _context[0]


def prepare(case, seed):
    ctx = _ctx()
    v, t, xq, q = _surface(case["f"], seed)
    s = {"case": case, "ctx": ctx, "params": pb.Params(*PARAMS), "plan": PLANS[case["plan"]],
         "xq": torch.as_tensor(xq, device="cuda"), "q": torch.as_tensor(q, device="cuda")}
    if case["do"] == "whole":
        s |= {"verts": torch.as_tensor(v, device="cuda"), "tris": torch.as_tensor(t, device="cuda"),
              "opts": pb.solve_opts(tol=1e-6, max_it=400, precision=PREC[case["prec"]])}
        return s
    s["x"] = torch.as_tensor(_vector(v, xq, q, seed), device="cuda")
    s["mesh"] = pb.pb_mesh_load(ctx, v, t, **s["plan"])
    if case["do"] in ("apply", "precond"):
        s["near"] = pb.pb_near_build(ctx, s["mesh"], PARAMS[2])
    return s


def run(s):
    case, ctx, p = s["case"], s["ctx"], s["params"]
    form = case["form"]
    prec = PREC[case["prec"]] if "prec" in case else None

    def kept(x):
        return x if prec == pb.PB_F64 else x.float()

    if case["do"] == "apply":
        return kept(pb.pb_system_apply(ctx, s["mesh"], s["near"], p, form, s["x"], prec=prec))
    if case["do"] == "precond":
        return kept(pb.pb_precond_apply(ctx, s["mesh"], s["near"], p, form, case["precond"], s["x"], prec=prec))
    if case["do"] == "near":
        near = pb.pb_near_build(ctx, s["mesh"], p.kappa)
        diag = pb.pb_precond_apply(ctx, s["mesh"], near, p, form, "block_diag", s["x"])
        y = pb.pb_system_apply(ctx, s["mesh"], near, p, form, s["x"], prec=pb.PB_F32)
        near.free()
        return {"diag": diag, "y": y.float()}
    phi = torch.empty_like(s["q"])
    if case["do"] == "charges":
        rhs = pb.pb_rhs_charges(ctx, s["mesh"], s["xq"], s["q"], p, form, prec=prec)
        dg, _ = pb.pb_energy(ctx, s["mesh"], s["x"], form, s["xq"], s["q"], p, phi=phi, prec=prec)
        return {"rhs": kept(rhs), "phi": kept(phi), "dG": dg}
    charges = pb.PB_F32_ACCURATE if prec == pb.PB_MIXED else pb.PB_F64
    mesh = pb.pb_mesh_load(ctx, s["verts"], s["tris"], **s["plan"])
    near = pb.pb_near_build(ctx, mesh, p.kappa)
    rhs = pb.pb_rhs_charges(ctx, mesh, s["xq"], s["q"], p, form, prec=charges)
    x, _ = pb.pb_solve(ctx, mesh, near, p, form, case["precond"], rhs, opts=s["opts"])
    dg, _ = pb.pb_energy(ctx, mesh, x, form, s["xq"], s["q"], p, phi=phi, prec=charges)
    near.free()
    mesh.free()
    return {"rhs": kept(rhs), "x": kept(x), "phi": kept(phi), "dG": dg}


# --------------------------------------------------------------- floors
def _sizes(case):
    f, band = case["f"], case["plan"] == "band"
    nt, nv = 20 * f * f, 10 * f * f + 2
    q = 3 if band else 6
    nnz = nv * (147 if band else 19)  # columns of a vertex: within three radii, or its triangles' neighbours
    return {"nt": nt, "nv": nv, "np": q * nt, "np_ref": 6 * nt, "nnz": nnz, "nq": max(1, nt // 80),
            "pairs": nt * (72 if band else 0)}


def _apply_work(case, s, prec):
    """A pair of points: 25 operations (V/K rows) or 36 (V/K + D/T rows). Single precision from 50,000 points on needs
    not all pairs: about 1,200 interactions a point and doubling, from trees that reach the same accuracy."""
    per = 25.0 if case["form"] == "direct_int" else 36.0
    pairs = float(s["np"]) ** 2
    if prec == "f32" and s["np"] >= 50000:
        pairs = min(pairs, s["np"] * 1200.0 * math.log2(s["np"]))
    value = 4 if prec == "f32" else 8
    # the near matrix's seven values, its columns, and x and y; positions, weights and geometry
    return {"bytes": s["nnz"] * (7 * value + 4) + 32.0 * s["nv"] + 32.0 * s["np"] + 128.0 * s["nt"], "flops": per * pairs}


def _near_work(case, s):
    """Quadrature points of the pairs that share an edge (1.5 a triangle), a vertex (4.5) or all (1), and of the band."""
    coin = 3 if case["plan"] == "band" else 4
    points = s["nt"] * (1.5 * 6 * 256 + 4.5 * 2 * 256 + 3 * coin ** 4) + s["pairs"] * 45.0
    return {"bytes": 56.0 * s["nnz"] + 152.0 * s["nt"] + 24.0 * s["nv"], "flops": 60.0 * points}


def _charge_work(s):
    pairs = float(s["np_ref"]) * s["nq"]
    return {"bytes": 2 * 128.0 * s["nt"] + 64.0 * s["nv"] + 64.0 * s["nq"], "flops": 2 * 20.0 * pairs}


def work(case):
    s = _sizes(case)
    total = {"bytes": 0.0, "flops": 0.0}

    def add(w, n=1.0):
        for k in total:
            total[k] += n * w[k]

    mass = {"bytes": 16.0 * 7 * s["nv"] + 32.0 * s["nv"], "flops": 4.0 * 7 * s["nv"] * 16}
    if case["do"] == "apply":
        add(_apply_work(case, s, case["prec"]))
    elif case["do"] == "precond":
        add(mass)
    elif case["do"] == "near":
        add(_near_work(case, s))
        add(_apply_work(case, s, "f32"))
    elif case["do"] == "charges":
        add(_charge_work(s))
    else:
        steps = 20.0 if case["prec"] == "mixed" else 15.0
        add(_near_work(case, s))
        add(_charge_work(s))
        add(_apply_work(case, s, "f32" if case["prec"] == "mixed" else "f64"), steps)
        if case["prec"] == "mixed":
            add(_apply_work(case, s, "split"))
        add(mass, steps)
    return total


# --------------------------------------- the same in 64 bits, in plain torch
def _rule(q):
    if q == 6:
        a = (0.445948490915965, 0.091576213509771)
        w = (0.223381589678011, 0.109951743655322)
    else:
        a, w = (1.0 / 6.0,), (1.0 / 3.0,)
    lam, wt = [], []
    for ao, wo in zip(a, w):
        for k in range(3):
            lam.append([1.0 - 2.0 * ao if c == k else ao for c in range(3)])
            wt.append(wo)
    return torch.tensor(lam, dtype=torch.float64), torch.tensor(wt, dtype=torch.float64)


def _cube_rule(kind, n):
    """Points (s, t) and (s', t') of 0 <= t <= s <= 1 in both triangles and their weights: the n^4 Gauss rule on the
    regularising maps of a coincident ("same"), edge- or vertex-sharing pair (Sauter and Schwab's regions; the edge
    map splits on the larger edge coordinate, then on the largest of the three vanishing coordinates)."""
    x, w = np.polynomial.legendre.leggauss(n)
    x, w = 0.5 * (x + 1.0), 0.5 * w
    k, a, b, c = (m.reshape(-1) for m in np.meshgrid(x, x, x, x, indexing="ij"))
    wt = np.prod(np.meshgrid(w, w, w, w, indexing="ij"), axis=0).reshape(-1)
    out = []
    if kind == "vertex":
        out.append((k, k * a, k * b, k * b * c, k ** 3 * b))
    elif kind == "edge":
        for which in range(3):
            h, w1, w2 = [(a, a * b, a * c), (a * b, a, a * c), (a * b, a * c, a)][which]
            out.append((k, k * w1, k * (1 - h), k * (1 - h) * w2, k ** 3 * (1 - h) * a ** 2))
    else:
        j = k ** 3 * a ** 2 * b
        out.append((k, k * (1 - a + a * b), k * (1 - a * b * c), k * (1 - a), j))
        out.append((k, k * a * (1 - b + b * c), k * (1 - a * b), k * a * (1 - b), j))
        out.append((k * (1 - a * b * c), k * a * (1 - b * c), k, k * a * (1 - b), j))
    out += [(s2, t2, s1, t1, j) for s1, t1, s2, t2, j in out]
    cols = [np.concatenate([r[i] for r in out]) for i in range(4)]
    return [torch.tensor(m) for m in cols] + [torch.tensor(np.concatenate([r[4] * wt for r in out]))]


class _Exact:
    """The discrete operators of a surface and a plan on vectors, in float64."""

    def __init__(self, case, v, t):
        plan = PLANS[case["plan"]]
        dev = "cuda"
        self.kappa = PARAMS[2]
        self.v, self.t = torch.as_tensor(v, device=dev), torch.as_tensor(t, device=dev).long()
        self.nv, self.nt = len(v), len(t)
        p = self.v[self.t]
        n = torch.linalg.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0])
        length = n.norm(dim=1)
        self.corner, self.area, self.n = p, 0.5 * length, n / length[:, None]
        edges = torch.stack([p[:, 2] - p[:, 1], p[:, 0] - p[:, 2], p[:, 1] - p[:, 0]], dim=1)
        self.curl = -edges / length[:, None, None]  # of the basis function of each corner
        self.lam, self.w = (m.to(dev) for m in _rule(plan["far_q"]))
        self.lam_ref, self.w_ref = (m.to(dev) for m in _rule(plan.get("band_q", plan["far_q"])))
        self.pairs = self._adjacent(plan)
        if plan.get("band_eta"):
            self.pairs.append(self._band(plan))

    def _adjacent(self, plan):
        """[(triangles, partners, point rule)] by class; corners listed so that the shared ones come first."""
        t, nt = self.t.cpu().numpy(), self.nt
        order = np.argsort(t.reshape(-1), kind="stable")
        owner, vert = order // 3, t.reshape(-1)[order]
        start = np.searchsorted(vert, np.arange(self.nv + 1))
        count = np.diff(start)
        code = []
        for d in np.unique(count):
            tri = owner[start[:-1][count == d][:, None] + np.arange(d)]
            code.append((tri[:, :, None] * nt + tri[:, None, :]).reshape(-1))
        code = np.unique(np.concatenate(code))
        a, b = code // nt, code % nt
        same = t[a][:, :, None] == t[b][:, None, :]
        shared = same.any(axis=2).sum(axis=1)
        out = []
        n_coin = plan.get("n_ss_coin") or plan["n_ss"]
        for kind, k, n in (("same", 3, n_coin), ("edge", 2, plan["n_ss"]), ("vertex", 1, plan["n_ss"])):
            sel = np.nonzero(shared == k)[0]
            ta, tb = t[a[sel]], t[b[sel]]
            eq = same[sel]
            if kind == "same":
                pa = pb_ = np.tile(np.arange(3), (len(sel), 1))
            elif kind == "edge":  # the shared edge from its lower to its higher vertex, then the third corner
                fa, fb = ~eq.any(axis=2), ~eq.any(axis=1)

                def perm(tri, free):
                    third = free.argmax(axis=1)
                    rest = np.stack([(third + 1) % 3, (third + 2) % 3], 1)
                    g = np.take_along_axis(tri, rest, 1)
                    rest = np.where((g[:, 0] < g[:, 1])[:, None], rest, rest[:, ::-1])
                    return np.concatenate([rest, third[:, None]], 1)

                pa, pb_ = perm(ta, fa), perm(tb, fb)
            else:
                pa = (eq.any(axis=2).argmax(axis=1)[:, None] + np.arange(3)) % 3
                pb_ = (eq.any(axis=1).argmax(axis=1)[:, None] + np.arange(3)) % 3
            s1, t1, s2, t2, w = (m.cuda() for m in _cube_rule(kind, n))
            la = torch.stack([1 - s1, s1 - t1, t1], 1)
            lb = torch.stack([1 - s2, s2 - t2, t2], 1)
            out.append({"a": torch.as_tensor(a[sel]).cuda(), "b": torch.as_tensor(b[sel]).cuda(),
                        "pa": torch.as_tensor(pa).cuda(), "pb": torch.as_tensor(pb_).cuda(),
                        "la": la, "lb": lb, "w": 4.0 * w, "full": True})
        return out

    def _band(self, plan):
        p, eta = self.corner, plan["band_eta"]
        c = (p[:, 0] + p[:, 1] + p[:, 2]) / 3.0
        e = p - c[:, None]
        r = (e[..., 0] * e[..., 0] + e[..., 1] * e[..., 1] + e[..., 2] * e[..., 2]).max(dim=1).values.sqrt()
        a, b = [], []
        for i0 in range(0, self.nt, 2048):
            i1 = min(self.nt, i0 + 2048)
            d = [c[i0:i1, None, k] - c[None, :, k] for k in range(3)]
            lim = eta * (r[i0:i1, None] + r[None])
            hit = (d[0] * d[0] + d[1] * d[1]) + d[2] * d[2] < lim * lim
            ia, ib = hit.nonzero(as_tuple=True)
            ia = ia + i0
            keep = ~(self.t[ia][:, :, None] == self.t[ib][:, None]).any(dim=2).any(dim=1)
            a.append(ia[keep])
            b.append(ib[keep])
        q = len(self.w_ref)
        ids = torch.arange(3, device="cuda").expand(sum(len(x) for x in a), 3)
        return {"a": torch.cat(a), "b": torch.cat(b), "pa": ids, "pb": ids, "full": False,
                "la": self.lam_ref.repeat_interleave(q, 0), "lb": self.lam_ref.repeat(q, 1),
                "w": (self.w_ref[:, None] * self.w_ref[None]).reshape(-1)}

    def _blocks(self, g, lo, hi, la, lb, w):
        """Local 3x3 blocks (in the triangles' own corner order) of V, K and D, Laplace and Yukawa, of the pairs
        lo..hi of a class under one point rule; points that coincide are left out."""
        a, b, pa, pb_ = (g[k][lo:hi] for k in ("a", "b", "pa", "pb"))
        m = hi - lo
        ca = torch.gather(self.corner[a], 1, pa[:, :, None].expand(m, 3, 3))
        cb = torch.gather(self.corner[b], 1, pb_[:, :, None].expand(m, 3, 3))
        d = torch.matmul(la, ca) - torch.matmul(lb, cb)
        r2 = (d * d).sum(dim=2)
        rinv = torch.where(r2 > 0, r2, 1.0).rsqrt() * (r2 > 0)
        gl = rinv * (w / (4.0 * math.pi)) * (self.area[a] * self.area[b])[:, None]
        kr = self.kappa * r2 * rinv
        ex = torch.exp(-kr)
        kl = gl * rinv * rinv * (d * self.n[b][:, None]).sum(dim=2)
        out = {}
        inv_a, inv_b = pa.argsort(dim=1), pb_.argsort(dim=1)
        ll = (la[:, :, None] * lb[:, None, :]).reshape(len(w), 9)
        for name, val in (("VL", gl), ("VY", gl * ex), ("KL", kl), ("KY", kl * ex * (1.0 + kr))):
            blk = (val @ ll).reshape(m, 3, 3)
            blk = torch.gather(blk, 1, inv_a[:, :, None].expand(m, 3, 3))
            out[name] = torch.gather(blk, 2, inv_b[:, None, :].expand(m, 3, 3))
        cc = torch.matmul(self.curl[a], self.curl[b].transpose(1, 2))
        nn = (self.n[a] * self.n[b]).sum(dim=1)[:, None, None]
        out["DL"] = cc * out["VL"].sum(dim=(1, 2), keepdim=True)
        out["DY"] = cc * out["VY"].sum(dim=(1, 2), keepdim=True) + self.kappa ** 2 * nn * out["VY"]
        return out

    def _near(self):
        """(triangles, partners, near blocks, full blocks or None), chunk by chunk."""
        q = len(self.w)
        far = (self.lam.repeat_interleave(q, 0), self.lam.repeat(q, 1), (self.w[:, None] * self.w[None]).reshape(-1))
        for g in self.pairs:
            step = max(1, int(6e7) // len(g["w"]))
            own = {**g, "pa": torch.arange(3, device="cuda").expand(len(g["a"]), 3)}
            own["pb"] = own["pa"]
            for lo in range(0, len(g["a"]), step):
                hi = min(len(g["a"]), lo + step)
                full = self._blocks(g, lo, hi, g["la"], g["lb"], g["w"])
                coarse = self._blocks(own, lo, hi, *far)
                yield g["a"][lo:hi], g["b"][lo:hi], {k: full[k] - coarse[k] for k in full}, full if g["full"] else None

    def mass(self):
        loc = (torch.ones(3, 3, device="cuda", dtype=torch.float64) + torch.eye(3, device="cuda", dtype=torch.float64))
        val = self.area[:, None, None] * loc / 12.0
        i = self.t[:, :, None].expand(-1, 3, 3).reshape(-1)
        j = self.t[:, None, :].expand(-1, 3, 3).reshape(-1)
        return torch.sparse_coo_tensor(torch.stack([i, j]), val.reshape(-1), (self.nv, self.nv)).coalesce()

    def system(self, form):
        """{operator: coefficient} of the four blocks (row, column) of a formulation (the paper's equations)."""
        ei, ee, _ = PARAMS
        r = ei / ee
        int_int = [{"M": 0.5, "KL": 1.0}, {"VL": -1.0}, {"DL": -1.0}, {"M": 0.5, "TL": -1.0}]
        ext_int = [{"M": 0.5, "KY": -1.0}, {"VY": r}, {"DY": 1.0 / r}, {"M": 0.5, "TY": 1.0}]
        ext_ext = [{"M": 0.5, "KY": -1.0}, {"VY": 1.0}, {"DY": 1.0}, {"M": 0.5, "TY": 1.0}]
        int_ext = [{"M": 0.5, "KL": 1.0}, {"VL": -1.0 / r}, {"DL": -r}, {"M": 0.5, "TL": -1.0}]
        if form == "direct_int":
            return int_int[:2] + ext_int[:2]
        first, second, alpha, beta, scale = {
            "juffer": (int_int, ext_int, 1.0 / r, r, (1.0, 1.0)),
            "muller_int": (int_int, ext_int, 1.0, 1.0, (1.0, 1.0)),
            "pmchwt_int": (int_int, ext_int, -1.0, -1.0, (-1.0, -1.0)),
            "lu": (ext_ext, int_ext, r, 1.0 / r, (1.0, r))}[form]
        out = []
        for k in range(4):
            f, s = (alpha, scale[0]) if k < 2 else (beta, scale[1])
            both = {o: s * c for o, c in first[k].items()}
            for o, c in second[k].items():
                both[o] = both.get(o, 0.0) + s * f * c
            out.append(both)
        return out

    def apply(self, blocks, x):
        """A x for the columns of x [2 nv, k]."""
        nv, kap = self.nv, self.kappa
        y = torch.zeros_like(x)
        xs = (x[:nv], x[nv:])
        k = x.shape[1]
        mass = self.mass()
        for n, blk in enumerate(blocks):
            if "M" in blk:
                y[(n // 2) * nv:(n // 2 + 1) * nv] += blk["M"] * torch.sparse.mm(mass, xs[n % 2])
        # near blocks; T is the transpose of the reversed pair's K
        for a, b, near, _ in self._near():
            ra, cb = self.t[a], self.t[b]
            for n, blk in enumerate(blocks):
                val = 0.0
                tra = 0.0
                for o, c in blk.items():
                    if o[0] == "T":
                        tra = tra + c * near["K" + o[1]]
                    elif o != "M":
                        val = val + c * near[o]
                row = y[(n // 2) * nv:(n // 2 + 1) * nv]
                if torch.is_tensor(val):
                    row.index_add_(0, ra.reshape(-1), torch.matmul(val, xs[n % 2][cb]).reshape(-1, k))
                if torch.is_tensor(tra):
                    row.index_add_(0, cb.reshape(-1), torch.matmul(tra.transpose(1, 2), xs[n % 2][ra]).reshape(-1, k))
        # the far rule on all pairs of points
        pts = torch.matmul(self.lam, self.corner).reshape(-1, 3)
        q = len(self.w)
        wt = (self.area[:, None] * self.w).reshape(-1)
        nrm = self.n.repeat_interleave(q, 0)
        dens = [torch.matmul(self.lam, z[self.t]).reshape(-1, k) * wt[:, None] for z in xs]
        curl = (self.curl[:, :, None, :] * xs[0][self.t][:, :, :, None]).sum(dim=1)  # [nt, k, 3]
        curl = curl.repeat_interleave(q, 0) * wt[:, None, None]
        need = {o for blk in blocks for o in blk if o != "M"}
        step = max(1, int(2.5e8) // len(pts))
        for lo in range(0, len(pts), step):
            hi = min(len(pts), lo + step)
            d = [pts[lo:hi, None, c] - pts[None, :, c] for c in range(3)]
            r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
            rinv = torch.where(r2 > 0, r2, 1.0).rsqrt_() * (r2 > 0)
            kr = kap * r2 * rinv
            gl = rinv / (4.0 * math.pi)
            ex = torch.exp(-kr)
            kern = {"L": (gl, gl * rinv * rinv)}
            if any(o[1] == "Y" for o in need):
                kern["Y"] = (gl * ex, kern["L"][1] * ex * (1.0 + kr))
            del r2, kr
            dn = sum(d[c] * nrm[None, :, c] for c in range(3)) if any(o[0] == "K" for o in need) else None
            dx = sum(d[c] * nrm[lo:hi, None, c] for c in range(3)) if any(o[0] == "T" for o in need) else None
            val = {}
            for o in need:
                g, g3 = kern[o[1]]
                if o[0] == "V":
                    val[o] = g @ dens[1]
                elif o[0] == "K":
                    val[o] = (g3 * dn) @ dens[0]
                elif o[0] == "T":
                    val[o] = -(g3 * dx) @ dens[1]
                else:
                    val[o] = torch.stack([g @ curl[:, :, c] for c in range(3)], 2)
                    if o[1] == "Y":
                        val["N"] = sum(nrm[lo:hi, None, c] * (g @ (dens[0] * nrm[:, c, None])) for c in range(3))
            tri = torch.arange(lo, hi, device="cuda") // q
            lam = self.lam[torch.arange(lo, hi, device="cuda") % q]
            wl = wt[lo:hi, None] * lam
            for n, blk in enumerate(blocks):
                row = y[(n // 2) * nv:(n // 2 + 1) * nv]
                for o, c in blk.items():
                    if o == "M":
                        continue
                    if o[0] == "D":
                        loc = torch.einsum("pac,pkc->pak", self.curl[tri] * wt[lo:hi, None, None], val[o])
                        if o[1] == "Y":
                            loc = loc + kap ** 2 * wl[:, :, None] * val["N"][:, None]
                    else:
                        loc = wl[:, :, None] * val[o][:, None]
                    row.index_add_(0, self.t[tri].reshape(-1), c * loc.reshape(-1, k))
        return y

    def diagonal(self, blocks):
        """[nv, 2, 2]: each vertex's own entries of the four blocks."""
        out = torch.zeros(self.nv, 4, device="cuda", dtype=torch.float64)
        mass = self.mass()
        i, j = mass.indices()
        own = torch.zeros(self.nv, device="cuda", dtype=torch.float64)
        own.index_add_(0, i[i == j], mass.values()[i == j])
        for n, blk in enumerate(blocks):
            out[:, n] += blk.get("M", 0.0) * own
        for a, b, _, full in self._near():
            if full is None:
                continue
            p, ca, cb = (self.t[a][:, :, None] == self.t[b][:, None]).nonzero(as_tuple=True)
            at = self.t[a][p, ca]
            for n, blk in enumerate(blocks):
                for o, c in blk.items():
                    if o != "M":
                        out[:, n].index_add_(0, at, c * full["K" + o[1] if o[0] == "T" else o][p, ca, cb])
        return out.reshape(-1, 2, 2)

    def _tested(self):
        pts = torch.matmul(self.lam_ref, self.corner).reshape(-1, 3)
        q = len(self.w_ref)
        return pts, (self.area[:, None] * self.w_ref).reshape(-1), self.n.repeat_interleave(q, 0), q

    def rhs(self, form, xq, q):
        ei, ee, _ = PARAMS
        pts, wt, nrm, nq = self._tested()
        phi = torch.zeros(2, len(pts), device="cuda", dtype=torch.float64)
        for lo in range(0, len(pts), 65536):
            d = pts[lo:lo + 65536, None] - xq[None]
            rinv = d.norm(dim=2).reciprocal()
            phi[0, lo:lo + 65536] = rinv @ q
            phi[1, lo:lo + 65536] = -((d * nrm[lo:lo + 65536, None]).sum(dim=2) * rinv ** 3) @ q
        out = []
        for k in range(2):
            loc = (phi[k] * wt / (4.0 * math.pi * ei)).reshape(-1, nq) @ self.lam_ref
            out.append(torch.zeros(self.nv, device="cuda", dtype=torch.float64).index_add_(
                0, self.t.reshape(-1), loc.reshape(-1)))
        d, n = out
        r = ei / ee
        zero = torch.zeros_like(d)
        return {"direct_int": [d, zero], "juffer": [d, n], "muller_int": [d, n], "pmchwt_int": [-d, -n],
                "lu": [r * d, r * n]}[form]  # Lu: diag(alpha, r beta) = (r, 1), its second row times r

    def reaction(self, form, x, xq):
        ei, ee, _ = PARAMS
        pts, wt, nrm, nq = self._tested()
        u, v = x[:self.nv], x[self.nv:] * (ee / ei if form == "lu" else 1.0)
        uu = (u[self.t] @ self.lam_ref.T).reshape(-1) * wt
        vv = (v[self.t] @ self.lam_ref.T).reshape(-1) * wt
        out = []
        for lo in range(0, len(xq), 64):
            d = xq[lo:lo + 64, None] - pts[None]
            rinv = d.norm(dim=2).reciprocal()
            out.append((rinv @ vv - ((d * nrm[None]).sum(dim=2) * rinv ** 3) @ uu) / (4.0 * math.pi))
        return torch.cat(out)


def _mass_inverse(mass, b):
    """Conjugate gradients with the diagonal, to rounding (its scaled spectrum lies in [1/2, 2])."""
    i, j = mass.indices()
    d = torch.zeros_like(b[:, 0]).index_add_(0, i[i == j], mass.values()[i == j])[:, None]
    x = torch.zeros_like(b)
    r = b.clone()
    z = r / d
    p = z.clone()
    rz = (r * z).sum(dim=0)
    for _ in range(60):
        ap = torch.sparse.mm(mass, p)
        alpha = rz / (p * ap).sum(dim=0)
        x += alpha * p
        r -= alpha * ap
        z = r / d
        new = (r * z).sum(dim=0)
        if float(new.abs().max()) < 1e-34 * float((b * b / d).sum()):
            break
        p = z + new / rz * p
        rz = new
    return x


def exact(case, seed):
    s = _sizes(case)
    if case["do"] in ("apply", "near") and s["np"] > 160000:
        return None  # the pair sums alone would take a minute in 64 bits
    if case["do"] == "whole" and (case["prec"] == "mixed" or case["f"] > 8):
        return None  # the dense system of a mixed solve's sizes takes minutes
    v, t, xq, q = _surface(case["f"], seed)
    e = _Exact(case, v, t)
    form = case["form"]
    dxq, dq = torch.as_tensor(xq, device="cuda"), torch.as_tensor(q, device="cuda")
    blocks = e.system(form)
    ei, ee, _ = PARAMS
    if case["do"] == "whole":
        nv = e.nv
        a = e.apply(blocks, torch.eye(2 * nv, device="cuda", dtype=torch.float64))
        b = torch.cat(e.rhs(form, dxq, dq))
        x = torch.linalg.solve(a, b)
        phi = e.reaction(form, x, dxq)
        return {"rhs": b, "x": x, "phi": phi, "dG": float(0.5 * (dq * phi).sum())}
    x = torch.as_tensor(_vector(v, xq, q, seed), device="cuda")
    if case["do"] == "apply":
        return e.apply(blocks, x[:, None])[:, 0]
    if case["do"] == "near":
        inv = torch.linalg.inv(e.diagonal(blocks))
        z = torch.matmul(inv, torch.stack([x[:e.nv], x[e.nv:]], 1)[:, :, None])[:, :, 0]
        return {"diag": torch.cat([z[:, 0], z[:, 1]]), "y": e.apply(blocks, x[:, None])[:, 0]}
    if case["do"] == "precond":
        z = _mass_inverse(e.mass(), torch.stack([x[:e.nv], x[e.nv:]], 1))
        sa, sb = (1.0 + ee / ei, 1.0 + ei / ee) if case["precond"] == "scaled_mass" else (1.0, 1.0)
        return torch.cat([z[:, 0] / sa, z[:, 1] / sb])
    phi = e.reaction(form, x, dxq)
    return {"rhs": torch.cat(e.rhs(form, dxq, dq)), "phi": phi, "dG": float(0.5 * (dq * phi).sum())}
