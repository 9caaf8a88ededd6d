"""The work that users of this library have it do, as a list of cases: one
preconditioner application in a caller's own Krylov loop (one vector or a
batch), a solve on a handle that is kept, a whole setup and solve on a new
problem, and a gradient step, over the meshes, degrees, precisions and
schedules of the tests and the benchmark.

A case is a dict:
  kind       "vcycle", "vcycle_batched", "solve", "solve_batched" (the handle
             is the user's and kept), "setup_solve" (handle, solve, release),
             "fbf" (the same through FBF(phMG)), "grad" (autograd forward and
             backward with one viscosity per cell)
  mesh, n    coarse mesh: "square" (n x n, cut along the diagonal), "cube"
             (n^3, Kuhn) or "disk" (Delaunay, spacing 1 / n)
  refine, alfeld, family, k, schedule, precision, relax, nrhs
Solves of uniform viscosity take a random polynomial flow of the degree that
the elements hold (volume force and boundary velocity), whose discrete
solution is the polynomial itself.
"""
import functools

import numpy as np
import torch

import paper_2407_07253_gb300 as P
import workloads as W
from paper_2407_07253_gb300 import autograd

# the benchmark's relaxation and the library's defaults
RELAX = {"v22": dict(nu_p=2, nu_h=2, cheb_lo=0.5, cheb_hi=2.0, eig_steps=8), "default": {}}
# the autograd wrappers' default: the pressure keeps six digits or more
TOL = 1e-10


def _case(kind, mesh, n, refine, family, k, schedule, precision="mixed", relax="v22", nrhs=1):
    return dict(kind=kind, mesh=mesh, n=n, refine=refine, alfeld=family == "SV", family=family, k=k, schedule=schedule,
                precision=precision, relax=relax, nrhs=nrhs)


def listed():
    return [
        # a small problem's preconditioner: latency and launches (the smoke test's problem, library defaults)
        dict(_case("vcycle", "square", 2, 2, "TH", 2, "2", "fp64", "default"), name="vcycle_th_p2_8x8_fp64"),
        # the benchmark's hierarchy as a preconditioner inside the user's own Krylov method
        dict(_case("vcycle", "square", 8, 3, "TH", 4, "4,2"), name="vcycle_th_p4_64x64"),
        # the same in three dimensions: large stars, many more entries per row
        dict(_case("vcycle", "cube", 4, 2, "TH", 3, "3,2"), name="vcycle_th_p3_cube16"),
        # the widest batch: a block method's 64 directions at once, FP32 accuracy
        dict(_case("vcycle_batched", "cube", 4, 2, "TH", 3, "3,2", nrhs=64), name="vcycle_b64_th_p3_cube16"),
        # the paper's size: one more load case on an operator that is set up
        dict(_case("solve", "square", 8, 5, "TH", 4, "4,2"), name="solve_th_p4_256x256"),
        # a parameter study: 32 load cases of one operator in lockstep
        dict(_case("solve_batched", "square", 8, 4, "TH", 3, "3,2", nrhs=32), name="solve_b32_th_p3_128x128"),
        # the benchmark: time to solution of a new problem
        dict(_case("setup_solve", "square", 8, 3, "TH", 4, "4,2"), name="setup_solve_th_p4_64x64"),
        # Scott-Vogelius on the unstructured disk: patches of very different sizes
        dict(_case("setup_solve", "disk", 6.25, 2, "SV", 4, "4,2"), name="setup_solve_sv_p4_disk"),
        # the same system through the block factorisation preconditioner
        dict(_case("fbf", "disk", 6.25, 2, "SV", 4, "4,2"), name="fbf_sv_p4_disk"),
        # high order with the gradual schedule; FP64 throughout
        dict(_case("setup_solve", "square", 8, 2, "TH", 6, "6,4,2", "fp64"), name="setup_solve_th_p6_32x32_fp64"),
        # the highest order of the benchmark: few, large patches
        dict(_case("setup_solve", "square", 8, 2, "TH", 8, "8,5,2"), name="setup_solve_th_p8_32x32"),
        # one step of an inverse problem: forward, adjoint and both gradients (half the benchmark's 128 x 128)
        dict(_case("grad", "square", 8, 3, "TH", 3, "3,2"), name="grad_th_p3_64x64_nu"),
    ]


# degrees of the hierarchies that the paper and the tests use
SCHEDULES = {2: ["2"], 3: ["3,2"], 4: ["4,2"], 5: ["5,2"], 6: ["6,4,2", "6,2"], 7: ["7,4,2"], 8: ["8,5,2"]}


def draw(rng):
    kind = rng.choice(["vcycle", "vcycle", "vcycle_batched", "solve", "solve_batched", "setup_solve", "setup_solve", "fbf", "grad"])
    fbf = kind == "fbf"
    batched = kind in ("vcycle_batched", "solve_batched")
    mixed = batched or rng.random() < 0.75
    nrhs = int(round(2 ** rng.uniform(0.6, 6))) if batched else 1
    sv = fbf or (not batched and kind != "grad" and rng.random() < 0.2)
    cube = not sv and kind != "grad" and rng.random() < 0.25
    top = {"solve": 1.5e6, "vcycle": 6e5, "vcycle_batched": 1.2e5, "solve_batched": 1.2e5}.get(kind, 1.5e5)
    dofs = 10 ** rng.uniform(2.8, np.log10(top))
    if cube:
        k = rng.choice([2, 3])
        cells = max(3.0, min(16.0, (dofs / (3 * k**3 + (k - 1) ** 3)) ** (1 / 3)))
    elif sv:
        k = rng.choice([3, 4])
        cells = max(4.0, (dofs / (3 * k * k + 3 * k * (k + 1))) ** 0.5)
    else:
        k = rng.choice([2, 3, 4, 5, 6] if batched else [2, 3, 4, 5, 6, 7, 8])
        cells = max(4.0, (dofs / (2 * k * k + (k - 1) ** 2)) ** 0.5)
    # the coarse mesh has 2 to 4 (cube) or 3 to 9 cells a side
    refine = 1
    while cells / 2**refine > (4 if cube else 9):
        refine += 1
    n = max(2 if cube else 3, int(round(cells / 2**refine)))
    mesh = "cube" if cube else "square"
    if sv and rng.random() < 0.5:
        mesh, n = "disk", 0.5 * max(n, 5)
    return _case(kind, mesh, n, refine, "SV" if sv else "TH", k, rng.choice(SCHEDULES[k]), "mixed" if mixed else "fp64",
                 "v22", nrhs)


# ------------------------------------------------------------- the problem
@functools.lru_cache(maxsize=None)
def _mesh(mesh, n):
    if mesh == "square":
        return W.unit_square_mesh(int(n))
    return W.kuhn_cube_mesh(int(n)) if mesh == "cube" else W.delaunay_disk_mesh(0, h=1.0 / n)


def _args(case):
    """Positional and keyword arguments of StokesMG for this case."""
    v, c = _mesh(case["mesh"], case["n"])
    kw = dict(barycentric=case["alfeld"], hierarchy=P.HIER_EXPLICIT, schedule=[int(x) for x in case["schedule"].split(",")],
              precision=P.MIXED if case["precision"] == "mixed" else P.FP64, **RELAX[case["relax"]])
    if case["kind"] == "fbf":
        kw["fbf"] = True
    return (v, c, case["refine"], P.SV if case["family"] == "SV" else P.TH, case["k"]), kw


@functools.lru_cache(maxsize=2)
def _host(key):
    """The problem's host-side hierarchy alone (node coordinates, sizes)."""
    case = dict(key)
    a, kw = _args(dict(case, kind="solve"))
    return P.StokesMG(*a, host_only=1, **kw)


def _host_of(case):
    return _host(tuple((x, case[x]) for x in ("mesh", "n", "refine", "alfeld", "family", "k", "schedule", "precision", "relax")))


def _flow(case, seed, q=0):
    """Coefficient arrays of a random divergence-free velocity of degree k
    (the curl of a random potential) and of a pressure of degree k - 1, of the
    size of the viscous stress."""
    d, k = (3 if case["mesh"] == "cube" else 2), case["k"]
    rng = np.random.default_rng([seed, q])
    der = np.polynomial.polynomial.polyder

    def poly(deg):
        c = rng.standard_normal((deg + 1,) * d)
        return np.where(sum(np.indices(c.shape)) <= deg, c, 0.0)

    def add(a, b):
        s = np.zeros([max(x, y) for x, y in zip(a.shape, b.shape)])
        s[tuple(slice(x) for x in a.shape)] += a
        s[tuple(slice(x) for x in b.shape)] += b
        return s

    if d == 2:
        s = poly(k + 1)
        u = [der(s, axis=1), -der(s, axis=0)]
    else:
        A = [poly(k + 1) for _ in range(3)]
        u = [add(der(A[(c + 2) % 3], axis=(c + 1) % 3), -der(A[(c + 1) % 3], axis=(c + 2) % 3)) for c in range(3)]
    p = k * (k + 1) * poly(k - 1)
    f = []
    for c in range(d):
        t = der(p, axis=c)
        for a in range(d):
            t = add(t, -der(u[c], 2, axis=a))
        f.append(t)
    return u, p, f


def _at(c, x):
    ev = np.polynomial.polynomial
    return (ev.polyval2d if c.ndim == 2 else ev.polyval3d)(*x.T, c)


def _mean(case, p):
    """Mean of a polynomial over the domain: collapsed Gauss quadrature on the coarse cells."""
    v, c = _mesh(case["mesh"], case["n"])
    d = v.shape[1]
    t, w = np.polynomial.legendre.leggauss(case["k"] + 2)
    t, w = 0.5 * (t + 1), 0.5 * w
    g = np.stack(np.meshgrid(*[t] * d, indexing="ij"), -1).reshape(-1, d)
    wt = functools.reduce(np.multiply.outer, [w] * d).ravel()
    lam, left = np.empty_like(g), np.ones(len(g))
    for a in range(d):
        lam[:, a] = left * g[:, a]
        wt = wt * left ** (1 if a else 0)
        left = left * (1 - g[:, a])
    J = v[c[:, 1:]] - v[c[:, :1]]
    vol = np.abs(np.linalg.det(J))
    x = v[c[:, 0]][:, None, :] + np.einsum("qa,eac->eqc", lam, J)
    return float((vol[:, None] * wt * _at(p, x.reshape(-1, d)).reshape(len(c), -1)).sum() / (vol.sum() * wt.sum()))


def _data(case, seed, nodes):
    """Nodal force and boundary velocity of every load case, [nrhs, d * nodes] on the GPU."""
    f, g = [], []
    for q in range(case["nrhs"]):
        u, _, ff = _flow(case, seed, q)
        f.append(np.concatenate([_at(c, nodes) for c in ff]))
        g.append(np.concatenate([_at(c, nodes) for c in u]))
    return torch.tensor(np.stack(f), device="cuda"), torch.tensor(np.stack(g), device="cuda")


# ------------------------------------------------------------ the measured
def prepare(case, seed):
    a, kw = _args(case)
    s = {"case": case, "args": a, "kw": kw}
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind in ("setup_solve", "fbf"):
        s["f"], s["g"] = (t[0] for t in _data(case, seed, _host_of(case).nodes()[0]))
    elif kind == "grad":
        i = _host_of(case).info()
        dim, nV, nQ = i["dim"], i["n_vel_nodes"], i["n_pres_nodes"]
        s["f"] = torch.tensor(W.nodal_forcing(nV, dim, seed), device="cuda", requires_grad=True)
        s["nu"] = torch.tensor(W.cell_viscosity(_host_of(case).n_cells(), seed), requires_grad=True)
        s["gu"] = torch.tensor(rng.standard_normal((dim, nV)), device="cuda")
        s["gp"] = torch.tensor(rng.standard_normal(nQ), device="cuda")
    else:
        s["h"] = P.StokesMG(*a, **kw)
        if kind in ("vcycle", "vcycle_batched"):
            # a residual: every DoF excited
            n = s["h"].info()["n_free"][0]
            g = torch.Generator(device="cuda").manual_seed(seed)
            s["r"] = torch.randn(*([case["nrhs"], n] if kind == "vcycle_batched" else [n]), dtype=torch.float64, device="cuda",
                                 generator=g)
        else:
            f, g = _data(case, seed, s["h"].nodes()[0])
            s["f"], s["g"] = (f, g) if kind == "solve_batched" else (f[0], g[0])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "vcycle":
        z = s["h"].vcycle(s["r"])
        # a mixed cycle's result is an FP32 vector, widened for the caller: narrowing it again loses nothing
        return {"z": z.float() if case["precision"] == "mixed" else z}
    if kind == "vcycle_batched":
        return {"z": s["h"].vcycle_batched(s["r"], P.BATCH_3XTF32).float()}
    if kind == "solve":
        u, p, _, _ = s["h"].solve(s["f"], s["g"], tol=TOL)
        return {"u": u, "p": p}
    if kind == "solve_batched":
        u, p, _, _ = s["h"].solve_batched(s["f"], s["g"], tol=TOL)
        return {"u": u, "p": p}
    if kind == "grad":
        f, nu = s["f"].detach().requires_grad_(), s["nu"].detach().requires_grad_()
        u, p = autograd.solve(*s["args"], f, nu, tol=TOL, **s["kw"])
        gf, gnu = torch.autograd.grad((u, p), (f, nu), (s["gu"], s["gp"]))
        return {"u": u.detach(), "p": p.detach(), "grad_f": gf, "grad_nu": gnu}
    h = P.StokesMG(*s["args"], **s["kw"])
    u, p, _, _ = h.solve(s["f"], s["g"], tol=TOL)
    h.close()
    return {"u": u, "p": p}


@functools.lru_cache(maxsize=None)
def _counts(key):
    """Per level of the hierarchy: free DoFs, entries of K, and over the
    patches the sums of entries of the factored inverse, of the cubes of the
    velocity and pressure blocks, and of DoFs."""
    case = dict(key)
    h = _host_of(case)
    i = h.info()
    out = []
    for l in range(len(i["n_free"]) - 1):
        off, dofs = h.patches(l)
        _, comp, _ = h.level_dofs(l)
        np_ = np.add.reduceat(np.append(comp[dofs] == i["dim"], 0).astype(np.int64), off[:-1])
        nv = (np.diff(off) - np_) // i["dim"]
        out.append((i["n_free"][l], i["nnz"][l], float((nv * (nv + 1) / 2 + i["dim"] * nv * np_ + np_ * (np_ + 1) / 2).sum()),
                    float((nv.astype(float) ** 3 + np_.astype(float) ** 3 + 2.0 * i["dim"] * nv * nv * np_).sum()),
                    float(i["dim"] * 2.0 * (nv.astype(float) ** 2 + 2 * nv * np_).sum()), len(dofs)))
    return i["dim"], i["n_vel_nodes"], i["n_pres_nodes"], out


def work(case):
    """A cycle reads every level's operator and factored patch inverses once
    for each of its two smoothing passes and touches its vectors once; a
    solve is ten cycles and ten FP64 products with the finest operator
    (what the problems here take); a setup makes every patch inverse."""
    key = tuple((x, case[x]) for x in ("mesh", "n", "refine", "alfeld", "family", "k", "schedule", "precision", "relax", "kind"))
    d, nV, nQ, lv = _counts(key)
    m, e = case["nrhs"], 4 if case["precision"] == "mixed" else 8
    steps = 2 if case["relax"] == "v22" else 1
    cb = sum(2 * (e * fac + (e + 4) * nnz) + 4 * e * m * n for n, nnz, fac, _, _, _ in lv)
    cf = sum(2 * m * steps * (ap + 2 * nnz) for n, nnz, _, _, ap, _ in lv)
    vec = 8 * m * (d * nV + nQ)
    if case["kind"] in ("vcycle", "vcycle_batched"):
        return {"bytes": cb + vec, "flops": cf}
    n0, nnz0 = lv[0][:2]
    sb, sf = 10 * (cb + 12 * nnz0 + 24 * m * n0) + 4 * vec, 10 * (cf + 2 * m * nnz0 + 44 * m * n0)
    if case["kind"] in ("solve", "solve_batched"):
        return {"bytes": sb, "flops": sf}
    ib, inv = sum(e * fac + 16 * nnz for _, nnz, fac, _, _, _ in lv), sum(x[3] for x in lv)
    two = 2 if case["kind"] == "grad" else 1
    return {"bytes": ib + two * sb, "flops": inv + two * sf}


# ------------------------------------------------------- the same in 64 bits
def exact(case, seed):
    kind = case["kind"]
    if kind == "grad":
        return None           # no closed form with a random viscosity per cell
    if kind in ("vcycle", "vcycle_batched"):
        s = prepare(case, seed)
        z = _plain_vcycle(s["h"], case, s["r"].reshape(case["nrhs"], -1).T.contiguous())
        return {"z": z.T.reshape(s["r"].shape)}
    vx, px, _ = _host_of(case).nodes()
    U, Q = [], []
    for q in range(case["nrhs"]):
        u, p, _ = _flow(case, seed, q)
        U.append(np.concatenate([_at(c, vx) for c in u]))
        Q.append(_at(p, px) - _mean(case, p))
    if kind != "solve_batched":
        U, Q = U[0], Q[0]
    return {"u": np.array(U), "p": np.array(Q)}


def _plain_vcycle(h, case, r):
    """The V-cycle on the exported operators in FP64 torch: Chebyshev around
    the additive patch solves, each patch block inverted densely."""
    o = RELAX[case["relax"]]
    nu, lo, hi = o.get("nu_p", 1), o.get("cheb_lo", 0.1), o.get("cheb_hi", 1.1)
    i = h.info()
    n = i["n_free"]

    def csr(level, which):
        a = h.get_csr(level, which)
        t = [torch.tensor(x, device="cuda") for x in (a.indptr.astype(np.int64), a.indices.astype(np.int64), a.data)]
        return torch.sparse_csr_tensor(*t, size=a.shape)

    K = [csr(l, 0) for l in range(len(n))]
    R, Pr = [csr(l, 2) for l in range(len(n) - 1)], [csr(l, 1) for l in range(len(n) - 1)]
    solves = []
    for l in range(len(n) - 1):
        off, dofs = (torch.tensor(x.astype(np.int64), device="cuda") for x in h.patches(l))
        size = off.diff()
        rows = torch.repeat_interleave(torch.arange(n[l], device="cuda"), K[l].crow_indices().diff())
        keys, order = (rows * n[l] + K[l].col_indices()).sort()
        vals = K[l].values()[order]
        groups = []
        for m in size.unique().tolist():
            for first in (off[:-1][size == m]).split(max(1, 40_000_000 // (m * m))):
                idx = dofs[first[:, None] + torch.arange(m, device="cuda")]
                want = (idx[:, :, None] * n[l] + idx[:, None, :]).reshape(-1)
                at = torch.searchsorted(keys, want).clamp_(max=len(keys) - 1)
                block = torch.where(keys[at] == want, vals[at], 0.0).reshape(len(first), m, m)
                groups.append((idx, torch.linalg.inv(block)))
        solves.append((groups, 1.0 / torch.bincount(dofs, minlength=n[l]).double()))

    def smooth(l, b, x):
        a, c = lo * i["lmax"][l], hi * i["lmax"][l]
        theta, delta = 0.5 * (c + a), 0.5 * (c - a)
        groups, w = solves[l]

        def asm(v):
            z = torch.zeros_like(v)
            for idx, inv in groups:
                z.index_add_(0, idx.reshape(-1), (inv @ v[idx]).reshape(-1, v.shape[1]))
            return z * w[:, None]

        rho, res = delta / theta, b - K[l] @ x
        step = asm(res) / theta
        x = x + step
        for _ in range(1, nu):
            res = res - K[l] @ step
            new = 1.0 / (2.0 * theta / delta - rho)
            step = 2.0 * new / delta * asm(res) + new * rho * step
            x, rho = x + step, new
        return x

    # the coarsest system, bordered with the integrals of the linear pressure basis
    v, c = _mesh(case["mesh"], case["n"])
    vol = np.abs(np.linalg.det(v[c[:, 1:]] - v[c[:, :1]]))
    share = np.zeros(len(v))
    np.add.at(share, c, vol[:, None])
    xyz, comp, _ = h.level_dofs(len(n) - 1)
    at = ((xyz[comp == i["dim"]][:, None] - v[None]) ** 2).sum(-1).argmin(1)
    border = np.zeros(n[-1])
    border[comp == i["dim"]] = share[at]
    A = torch.zeros(n[-1] + 1, n[-1] + 1, dtype=torch.float64, device="cuda")
    A[:-1, :-1] = K[-1].to_dense()
    A[:-1, -1] = A[-1, :-1] = torch.tensor(border, device="cuda")

    def cycle(l, b):
        if l == len(n) - 1:
            return torch.linalg.solve(A, torch.cat([b, torch.zeros_like(b[:1])]))[:-1]
        x = smooth(l, b, torch.zeros_like(b))
        x = x + Pr[l] @ cycle(l + 1, R[l] @ (b - K[l] @ x))
        return smooth(l, b, x)

    return cycle(0, r)
