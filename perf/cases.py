"""Measured cases of the isogeometric boundary element library: what a program that uses it has it do.

Each case is one call, or one short sequence of calls, through the public entry points
(paper_2306_11324_gb300.binding, the C ABI of include/igabem.h):

  product    y = A x with a resident problem (igabem_matvec): the step of every iterative solve
  operator   a problem set up and applied once (igabem_problem_create, igabem_matvec, destroy): the
             near-field quadrature, the tree and the tables of a new wavenumber or geometry
  request    one scattering request from geometry to result (set-up, GMRES, far field, destroy): a step
             of a frequency sweep, or what the serving loop runs for each request
  solve      GMRES on a resident problem for new incident directions (igabem_solve)
  farfield   the far field of given densities at many directions (igabem_farfield)
  potential  the scattered field of given densities at many points (igabem_potential)

Geometries, discretisations, wavenumbers and column counts are those of the repository's benchmark
workloads and tests (degree 1 to 3, 4 x 4 to 128 x 128 elements per patch, at least 8 unknowns per
wavelength, 1 to 64 columns, each precision, coupling blocks on the fly or stored).  The mixed
precisions compute in FP32: a program that chooses them holds their results in complex64, so run()
returns that type for them, and complex128 for FP64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2306_11324_gb300 import binding as B
from paper_2306_11324_gb300 import inputs

# elements per patch are 2^m x 2^m; defaults of every case (leaf clusters of 2^b x 2^b elements)
BASE = dict(geometry="deformed", hard=False, m=5, p=2, b=2, q=7, q_max=0, cap=0.0, precision="fp64", stored=False,
            precond=False, columns=1)
PRECISION = {"fp64": B.FP64, "mixed": B.MIXED_FP32, "tc": B.MIXED_TC}
PATCHES = {"sphere": 6, "deformed": 6, "torus": 16}


def listed():
    def case(name, kind, **kw):
        return {"name": name, "kind": kind, **BASE, **kw}

    return [
        # the smallest problem (degree 1, 96 elements): one product is launches and latency
        case("product_sphere_soft_4x4_p1_fp64", "product", geometry="sphere", m=2, p=1, b=0, kappa=1.0),
        # one product of a plain FP64 GMRES, 6936 unknowns, coupling samples generated on the fly
        case("product_sphere_soft_32x32_fp64", "product", geometry="sphere", m=5, kappa=8.0),
        # the product of a sound-hard request of the serving stream: stored blocks, an odd column count
        case("product_hard_32x32_stored_r5", "product", hard=True, m=5, kappa=11.0, cap=6.0, precision="mixed",
             stored=True, columns=5),
        # the product of the 64-direction sound-hard solve: the multi-column M2L on the tensor cores
        case("product_hard_64x64_tc_r64", "product", hard=True, m=6, kappa=20.0, cap=6.0, precision="tc", columns=64),
        # the product of a large scatterer's frequency sweep: stored blocks, level-adaptive q, 8 directions
        case("product_soft_128x128_stored_r8", "product", m=7, kappa=27.0, cap=6.0, q_max=12, precision="mixed",
             stored=True, columns=8),
        # a sound-hard operator set up for a new wavenumber and applied once
        case("operator_hard_32x32_mixed", "operator", hard=True, m=5, kappa=13.0, cap=6.0, precision="mixed"),
        # the smallest request of the serving stream: one plane wave on the sphere
        case("request_sphere_soft_16x16_mixed", "request", geometry="sphere", m=4, kappa=6.0, precision="mixed",
             precond=True, tol=1e-6, directions=100),
        # a step of a frequency sweep: set-up, 8 directions, far field at 2048 directions
        case("request_soft_64x64_stored_r8", "request", m=6, kappa=27.0, cap=6.0, q_max=12, precision="mixed",
             stored=True, precond=True, columns=8, tol=1e-6, directions=2048),
        # a request with everything in FP64, on the torus
        case("request_torus_soft_8x8_fp64_r2", "request", geometry="torus", m=3, b=1, kappa=2.0, stored=True,
             precond=True, columns=2, tol=1e-8, directions=100),
        # a resident sound-hard problem solved for three new directions (long Krylov cycles)
        case("solve_sphere_hard_16x16_fp64_r3", "solve", geometry="sphere", hard=True, m=4, kappa=3.0, precond=True,
             columns=3, tol=1e-10),
        # the sweep's far field for 8 densities
        case("farfield_soft_64x64_2048dirs_r8", "farfield", m=6, kappa=27.0, precision="mixed", columns=8,
             directions=2048),
        # the scattered field on a point cloud around the scatterer
        case("potential_soft_8x8_4001pts", "potential", m=3, kappa=3.0, precision="mixed", points=4001),
    ]


def draw(rng):
    """One more case of these ranges."""
    kind = rng.choice(["product", "product", "product", "operator", "request", "solve", "farfield", "potential"])
    c = {"kind": kind, **BASE}
    c["geometry"] = rng.choice(["sphere", "deformed", "deformed", "torus"])
    c["hard"] = rng.random() < 0.4
    c["p"] = rng.choice([1, 2, 2, 2, 3])
    c["precision"] = rng.choice(["fp64", "mixed"])
    c["q"] = rng.choice([6, 7, 7])
    top = {"sphere": 5, "deformed": 5, "torus": 4}[c["geometry"]]

    def log_int(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    def wavenumber(m, part):  # at most 8 unknowns per wavelength, a part of that range
        return round(rng.uniform(0.3, part) * (2 ** m + 2) / 2 * (0.5 if c["geometry"] == "torus" else 1.0), 3)

    if kind == "product":
        c["m"] = rng.randint(3, 6 if c["geometry"] != "torus" and c["p"] <= 2 else top)
        c["stored"] = rng.random() < 0.5 and (c["precision"] == "mixed" or c["m"] <= 4)
        c["columns"] = log_int(1, 24 if c["precision"] == "mixed" else 6)
        if c["precision"] == "mixed" and not c["stored"] and rng.random() < 0.4:
            c["precision"], c["columns"] = "tc", 16 * rng.randint(1, 4)
        if c["m"] == 6:  # the largest meshes in the mixed precisions, few columns
            c["precision"] = "mixed" if c["precision"] == "fp64" else c["precision"]
            c["columns"] = min(c["columns"], 16)
        c["cap"] = 6.0
        c["kappa"] = wavenumber(c["m"], 0.9)
    elif kind == "operator":
        c["m"] = rng.randint(3, 4 if c["precision"] == "fp64" or c["p"] == 3 else 5 if c["geometry"] != "torus" else 4)
        c["columns"] = rng.randint(1, 4)
        c["stored"] = rng.random() < 0.5
        c["cap"] = 6.0
        c["kappa"] = wavenumber(c["m"], 0.9)
    elif kind == "request":
        c["hard"] = False
        c["p"] = rng.choice([1, 2, 2])
        c["m"] = rng.randint(3, 3 if c["precision"] == "fp64" else top)
        c["columns"] = rng.randint(1, 9 if c["precision"] == "mixed" else 3)
        c["stored"] = c["precision"] == "fp64" or rng.random() < 0.7
        c["cap"], c["precond"] = 6.0, True
        c["tol"] = 1e-6 if c["precision"] == "mixed" else 1e-8
        c["directions"] = log_int(50, 2500)
        c["kappa"] = wavenumber(c["m"], 0.7)
    elif kind == "solve":
        c["precision"], c["p"] = "fp64", rng.choice([1, 2])
        c["m"] = rng.randint(2, 2 if c["geometry"] == "torus" else 3 if c["hard"] else 4)
        c["columns"] = rng.randint(1, 4)
        c["precond"], c["tol"], c["cap"] = True, 1e-10, 6.0
        c["kappa"] = wavenumber(c["m"], 0.4)
    elif kind == "farfield":
        c["m"] = rng.randint(3, 6 if c["precision"] == "mixed" and c["geometry"] != "torus" else 4)
        c["columns"] = log_int(1, 24 if c["precision"] == "mixed" else 4)
        c["directions"] = log_int(40, 3000 if c["precision"] == "mixed" else 600)
        c["kappa"] = wavenumber(c["m"], 0.9)
    else:
        c["geometry"] = rng.choice(["sphere", "deformed"])
        c["m"] = rng.randint(2, 3)
        c["columns"] = rng.randint(1, 2)
        c["points"] = log_int(300, 4000 if c["precision"] == "mixed" else 1200)
        c["kappa"] = wavenumber(c["m"], 0.6)
    c["b"] = rng.randint(1, 2) if c["m"] <= 4 else 2
    if c["p"] == 3 or (c["hard"] and c["geometry"] == "torus"):
        c["b"] = 1
    if c["hard"]:
        c["p"] = max(1, c["p"])
    if c["precision"] != "fp64" and c["cap"] > 0 and not c["hard"] and c["precision"] != "tc" and rng.random() < 0.3:
        c["q_max"] = rng.randint(c["q"] + 1, 12)
    return c


# ---------------------------------------------------------------------------------------------------
# the user's program

_CONTEXT = None


def _context():
    """One library context on a CUDA stream that PyTorch works on too (a program makes one and keeps it)."""
    global _CONTEXT
    if _CONTEXT is None:
        stream = torch.cuda.Stream()
        _CONTEXT = (B.igabem_create(torch.cuda.current_device(), stream.cuda_stream), stream)
    return _CONTEXT


class _Handle:
    """Owns the geometry and, where the case keeps one, the problem."""

    def __init__(self, geom):
        self.geom, self.prob = geom, None

    def __del__(self):
        if self.prob is not None:
            B.igabem_problem_destroy(self.prob)
        B.igabem_geometry_destroy(self.geom)


def _patches(case, seed):
    if case["geometry"] == "sphere":
        return inputs.unit_sphere_patches()
    if case["geometry"] == "torus":
        return inputs.torus_patches()
    return inputs.deformed_sphere_patches(spans=4, seed=1 + seed % 1000003)


def _options(case):
    # sound-soft systems couple with eta = kappa, sound-hard ones with 1 / kappa
    eta = 1.0 / case["kappa"] if case["hard"] else case["kappa"]
    return B.igabem_default_options(
        degree_p=case["p"], level_m=case["m"], kappa=case["kappa"], eta_cfie=eta, bc=int(case["hard"]),
        cheb_q=case["q"], q_max=case["q_max"], leaf_offset=case["b"], kappa_cap=case["cap"],
        precision=PRECISION[case["precision"]], m2l_stored=int(case["stored"]), precond=int(case["precond"]),
        gmres_restart=300 if case["hard"] else 30, max_iter=2000, tol=case.get("tol", 1e-6))


def _n_dofs(case):
    """Dimension of the ansatz space: patch-wise splines (soft), glued across the patches (hard)."""
    n, nb = PATCHES[case["geometry"]], 2 ** case["m"] + case["p"]
    if not case["hard"]:
        return n * nb * nb
    edges, corners = {"sphere": (12, 8), "deformed": (12, 8), "torus": (32, 16)}[case["geometry"]]
    return n * (nb - 2) ** 2 + edges * (nb - 2) + corners


def _directions(n, seed, k):
    """n seeded unit vectors."""
    v = np.random.default_rng([seed, k]).standard_normal((n, 3))
    return v / np.linalg.norm(v, axis=1, keepdims=True)


def _vectors(case, seed):
    """The seeded complex vector(s) [N][columns] of a case, entries (N(0,1) + i N(0,1)) / sqrt 2."""
    return inputs.random_complex(_n_dofs(case), seed=seed, cols=case["columns"])


def _points(case, seed):
    """Seeded evaluation points around the scatterer, 1.6 to 4 radii from its centre."""
    r = np.random.default_rng([seed, 7]).uniform(1.6, 4.0, (case["points"], 1))
    return r * _directions(case["points"], seed, 8)


def prepare(case, seed):
    ctx, stream = _context()
    h = _Handle(B.igabem_geometry_create(ctx, _patches(case, seed)))
    kind, n, cols = case["kind"], _n_dofs(case), case["columns"]
    s = {"case": case, "handle": h, "options": _options(case), "stream": stream}
    if kind in ("product", "solve", "farfield", "potential"):
        h.prob = B.igabem_problem_create(h.geom, s["options"])
        assert B.igabem_problem_info(h.prob)["n_dofs"] == n
    if kind in ("product", "operator"):
        s["x"] = torch.from_numpy(_vectors(case, seed)).cuda()
        s["y"] = torch.empty_like(s["x"])
    if kind in ("farfield", "potential"):
        s["density"] = torch.from_numpy(_vectors(case, seed)).cuda()
    if kind in ("request", "solve"):
        s["incident"] = _directions(cols, seed, 1)
        s["density"] = torch.empty((n, cols), dtype=torch.complex128, device="cuda")
    if kind in ("request", "farfield"):
        s["xhat"] = _directions(case["directions"], seed, 2)
        s["uinf"] = torch.empty((case["directions"], cols), dtype=torch.complex128, device="cuda")
    if kind == "potential":
        s["points"] = torch.from_numpy(_points(case, seed)).cuda()
        s["u"] = torch.empty((case["points"], cols), dtype=torch.complex128, device="cuda")
    return s


def run(s):
    case, h = s["case"], s["handle"]
    kind = case["kind"]
    if kind in ("operator", "request"):
        prob = B.igabem_problem_create(h.geom, s["options"])
    else:
        prob = h.prob
    try:
        if kind in ("product", "operator"):
            out = {"y": B.igabem_matvec(prob, s["x"], s["y"])}
        elif kind == "solve":
            out = {"density": B.igabem_solve(prob, s["incident"], _n_dofs(case), s["density"])[0]}
        elif kind == "request":
            density, _ = B.igabem_solve(prob, s["incident"], _n_dofs(case), s["density"])
            out = {"density": density, "uinf": B.igabem_farfield(prob, density, s["xhat"], s["uinf"])}
        elif kind == "farfield":
            out = {"uinf": B.igabem_farfield(prob, s["density"], s["xhat"], s["uinf"])}
        else:
            out = {"u": B.igabem_potential(prob, s["density"], s["points"], s["u"])}
    finally:
        if kind in ("operator", "request"):
            B.igabem_problem_destroy(prob)
    # results in the type the precision carries, on the library's stream
    dtype = torch.complex128 if case["precision"] == "fp64" else torch.complex64
    with torch.cuda.stream(s["stream"]):
        return {k: v.to(dtype, copy=True) for k, v in out.items()}


# ---------------------------------------------------------------------------------------------------
# what a pass cannot do without

def work(case):
    """Bytes: vectors, results and, with a resident problem, its stored operator, each once.  Flops: kernel
    samples (40 each) and complex multiply-adds (8).  A leaf of these trees has about 62 near and 250
    admissible pairs (all levels, counted at the leaf's q)."""
    kind, cols, hard = case["kind"], case["columns"], case["hard"]
    n, real = _n_dofs(case), 8 if case["precision"] == "fp64" else 4
    elements = PATCHES[case["geometry"]] * 4 ** case["m"]
    leaves = elements / 4 ** case["b"]
    near = 62 * leaves * (2 ** case["b"] + case["p"]) ** 4            # entries of the near-field blocks
    far = 250 * leaves * case["q"] ** 4 * (2 if hard else 1)          # entries of the coupling blocks
    vector = 16.0 * n * cols
    gauss = 16 * elements
    # the product: both operands, the near field read once, the far field read once or sampled
    product = {"bytes": 2 * vector + 2 * real * near + (2 * real * far if case["stored"] else 0),
               "flops": 8 * cols * near + 8 * cols * far * (3.5 if hard else 1) + (0 if case["stored"] else 40 * far)}
    # the set-up: 256 samples and two contractions per regular near element pair, about 15000 points of the
    # singular rules per element, the near-field blocks written
    funcs = (case["p"] + 1) ** 2
    setup = {"bytes": 2 * real * near + 8.0 * 100 * elements,
             "flops": 62 * leaves * 16 ** case["b"] * (256 * 60 + 8 * 16 * funcs * (16 + funcs)) + elements * 15000 * 250.0}
    solve = 20                                                        # products of a preconditioned solve
    if kind == "product":
        return product
    if kind == "operator":
        return {k: setup[k] + product[k] for k in setup}
    if kind == "solve":
        return {"bytes": vector + solve * product["bytes"], "flops": solve * product["flops"]}
    if kind in ("request", "farfield"):
        d = case["directions"]
        far_field = {"bytes": vector + 16.0 * d * cols + 8.0 * 7 * gauss, "flops": d * gauss * (20.0 + 8 * cols)}
        if kind == "farfield":
            return far_field
        return {k: setup[k] + solve * product[k] + far_field[k] for k in setup}
    # the tree code: every point against its 27 boxes of 64 sources nearby and the expansion of its own box
    pts = case["points"]
    return {"bytes": vector + (24.0 + 16 * cols) * pts + 8.0 * 7 * gauss,
            "flops": pts * (27 * 64 * 40.0 + 8.0 * cols * case["q"] ** 3) + gauss * 8.0 * cols * case["q"] ** 3}


# ---------------------------------------------------------------------------------------------------
# the defining sums in 64 bits

def _spline_rows(knots, degree, count, x):
    """Values [len(x)][count] and derivatives of the B-splines of a degree at points inside [0, 1)."""
    def cox(d):
        if d == 0:
            return [((knots[i] <= x) & (x < knots[i + 1])).astype(float) for i in range(len(knots) - 1)]
        low, out = cox(d - 1), []
        for i in range(len(knots) - 1 - d):
            v = np.zeros_like(x)
            if knots[i + d] > knots[i]:
                v = v + (x - knots[i]) / (knots[i + d] - knots[i]) * low[i]
            if knots[i + d + 1] > knots[i + 1]:
                v = v + (knots[i + d + 1] - x) / (knots[i + d + 1] - knots[i + 1]) * low[i + 1]
            out.append(v)
        return out

    val, low = cox(degree), cox(degree - 1)
    der = []
    for i in range(count):
        v = np.zeros_like(x)
        if knots[i + degree] > knots[i]:
            v = v + degree / (knots[i + degree] - knots[i]) * low[i]
        if knots[i + degree + 1] > knots[i + 1]:
            v = v - degree / (knots[i + degree + 1] - knots[i + 1]) * low[i + 1]
        der.append(v)
    return np.stack(val[:count], 1), np.stack(der, 1)


def _surface(patch, s, t):
    """Points and normals n~ = F_s x F_t of a NURBS patch on the grid s x t."""
    Hw = np.concatenate([patch.ctrl * patch.weights[..., None], patch.weights[..., None]], axis=-1)
    N1, D1 = _spline_rows(patch.knots1, patch.p1, Hw.shape[0], s)
    N2, D2 = _spline_rows(patch.knots2, patch.p2, Hw.shape[1], t)
    h, hs, ht = (np.einsum("ai,bj,ijc->abc", a, b, Hw) for a, b in ((N1, N2), (D1, N2), (N1, D2)))
    F = h[..., :3] / h[..., 3:]
    Fs = (hs[..., :3] - F * hs[..., 3:]) / h[..., 3:]
    Ft = (ht[..., :3] - F * ht[..., 3:]) / h[..., 3:]
    return F, np.cross(Fs, Ft)


def _weighted_density(case, seed):
    """Gauss points [G][3], normals n~ [G][3] and the density times the Gauss weights [G][columns]."""
    n1, p = 2 ** case["m"], case["p"]
    nb = n1 + p
    g, w = np.polynomial.legendre.leggauss(4)
    s = ((np.arange(n1)[:, None] + 0.5 * (g + 1.0)) / n1).reshape(-1)
    ws = np.tile(0.5 * w, n1) / n1
    knots = np.concatenate([np.zeros(p), np.arange(n1 + 1) / n1, np.ones(p)])
    phi = _spline_rows(knots, p, nb, s)[0]
    patches = _patches(case, seed)
    x = _vectors(case, seed)
    if case["hard"]:  # coefficients of the functions glued across the patches: coinciding Greville anchors
        grev = np.array([knots[i + 1:i + p + 1].mean() for i in range(nb)]).clip(0.0, 1.0 - 1e-15)
        anchors = np.concatenate([_surface(q, grev, grev)[0].reshape(-1, 3) for q in patches])
        key, number, index = {}, 0, np.zeros(len(anchors), int)
        for i, a in enumerate(np.round(anchors * 1e6).astype(int)):
            near = [(a[0] + i0, a[1] + i1, a[2] + i2) for i0 in (0, -1, 1) for i1 in (0, -1, 1) for i2 in (0, -1, 1)]
            hit = next((key[k] for k in near if k in key), None)
            if hit is None:
                hit = key[near[0]] = number
                number += 1
            index[i] = hit
        x = x[index]
    x = x.reshape(len(patches), nb, nb, -1)
    X, nn, rho = [], [], []
    for j, patch in enumerate(patches):
        F, n = _surface(patch, s, s)
        X.append(F.reshape(-1, 3))
        nn.append(n.reshape(-1, 3))
        r = np.einsum("ai,bj,ijr->abr", phi, phi, x[j]) * (ws[:, None] * ws[None, :])[..., None]
        rho.append(r.reshape(-1, r.shape[-1]))
    return np.concatenate(X), np.concatenate(nn), np.concatenate(rho)


def _mie_soft(kappa, cosine):
    """Far field of a plane wave on the sound-soft unit sphere: (i / kappa) sum (2n+1) j_n / h_n P_n."""
    top = int(kappa + 4 * kappa ** (1 / 3) + 20)
    # j_n by Miller's downward recurrence, y_n by the upward one
    j = np.zeros(top + 42)
    j[-2] = 1e-280
    for k in range(top + 39, -1, -1):
        j[k] = (2 * k + 3) / kappa * j[k + 1] - j[k + 2]
        if abs(j[k]) > 1e200:
            j *= 1e-200
    lead = 0 if abs(math.sin(kappa)) > 0.3 else 1
    true = math.sin(kappa) / kappa if lead == 0 else math.sin(kappa) / kappa ** 2 - math.cos(kappa) / kappa
    j *= true / j[lead]
    y = [-math.cos(kappa) / kappa, -math.cos(kappa) / kappa ** 2 - math.sin(kappa) / kappa]
    p0, p1, out = np.ones_like(cosine), cosine, 0.0
    for k in range(top + 1):
        if k >= 2:
            y.append((2 * k - 1) / kappa * y[-1] - y[-2])
            p0, p1 = p1, ((2 * k - 1) * cosine * p1 - (k - 1) * p0) / k
        out = out + (2 * k + 1) * j[k] / (j[k] + 1j * y[k]) * (p0 if k == 0 else p1)
    return 1j / kappa * out


def exact(case, seed):
    """Far fields and potentials: the sums over the Gauss points.  Requests on the sphere: the Mie series of the
    far field.  Products, operators, solves and the other requests have no value here: they are the
    Galerkin matrix with the interpolated kernel, whose rows take minutes in plain 64-bit arrays."""
    kind, kappa = case["kind"], case["kappa"]
    if kind == "request" and case["geometry"] == "sphere" and not case["hard"]:
        cosine = _directions(case["directions"], seed, 2) @ _directions(case["columns"], seed, 1).T
        return {"density": None, "uinf": _mie_soft(kappa, cosine)}
    if kind not in ("farfield", "potential"):
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    X, nn, rho = (torch.from_numpy(a).to(dev) for a in _weighted_density(case, seed))
    area, out = nn.norm(dim=1), []
    to = torch.from_numpy(_directions(case["directions"], seed, 2) if kind == "farfield" else _points(case, seed)).to(dev)
    step = max(1, 2 ** 25 // len(X))
    for i in range(0, len(to), step):
        v = to[i:i + step]
        if kind == "farfield":
            phase = -kappa * (v @ X.T)
            kernel = torch.complex(phase.cos(), phase.sin())
            kernel = kernel * (-1j * kappa * (v @ nn.T)) if case["hard"] else kernel * -area
            out.append(kernel @ rho / (4 * math.pi))
        else:
            d = X[None] - v[:, None]
            r = d.norm(dim=2)
            G = torch.complex((kappa * r).cos(), (kappa * r).sin()) / (4 * math.pi * r)
            if case["hard"]:
                G = G * torch.complex(-torch.ones_like(r), kappa * r) * ((d * nn[None]).sum(2) / r ** 2)
            else:
                G = G * -area
            out.append(G @ rho)
    return {"uinf" if kind == "farfield" else "u": torch.cat(out)}
