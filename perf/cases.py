"""Performance cases of the library: calls a program makes through the Python
binding, on the meshes of this repository's workloads, tests and benchmark.

A case names an operation (``op``), a mesh (molecule, box, coarse cells per
axis, degree, refinement levels), an orbital count ``n``, a precision and what
the operation needs beside them.  ``listed()`` gives the fixed cases,
``draw(rng)`` others of the same ranges; ``prepare`` makes what a program holds
before the call, ``run`` is one pass, ``work`` what the pass cannot do
without, and ``exact`` the same result in 64 bits from the plain finite-element
definitions (class ``Space`` below, torch only; of the library it uses nothing
but the coordinates of the unknowns, which say in what order results are laid
out).
"""
import functools
import itertools
import math

import numpy as np
import torch

import paper_2301_02387_gb300 as pkg
from paper_2301_02387_gb300 import adjoint

BATCH_BOX = 30.0
C3 = 3.0 * math.log(2.0 + math.sqrt(3.0)) - math.pi / 2.0   # mean of 1/|r| over a unit cube
LMAX = 12                                                   # multipole surface data of the mean fields
KEY = 512                                                   # key units per smallest cell side


# ------------------------------------------------------------------ the cases
def listed():
    hyd = dict(mol="h", box=20.0, nc=8, p=2, levels=3)
    h2 = dict(mol="h2", box=40.0, nc=20, p=4, levels=5)
    small = dict(mol="h2", box=8.0, nc=4, p=4, levels=2)
    odd = dict(mol="h2", box=30.0, nc=13, p=3, levels=3)
    water = dict(mol="water", box=50.0, nc=32, p=4, levels=6)
    return [
        # the smallest call: one orbital of the hydrogen workload, latency counts
        dict(name="h1 fp64 hydrogen", op="h1", n=1, mixed=False, **hyd),
        # the one-body operator on the benchmark's four orbitals (observables, initial-state work)
        dict(name="h1 c64 h2", op="h1", n=4, mixed=True, **h2),
        # the stiffness on all 64 pair densities of the water workload: the largest operator call
        dict(name="stiff f32 water", op="stiff", n=8, mixed=True, **water),
        # the batching form: one operator application on uneven molecules at once
        dict(name="batch h1 c64", op="batch", count=8, lo_dofs=2.0e4, hi_dofs=4.0e5),
        # the mean fields of a time step of the benchmark, from the previous step's fields
        dict(name="poisson mixed h2", op="poisson", n=4, mixed=True, mg=True, warm=True, **h2),
        # the mean fields of a first step on a degree-3 mesh, odd orbital count, default solver
        dict(name="poisson fp64 odd", op="poisson", n=3, mixed=False, mg=False, warm=False, **odd),
        # the two-electron integrals of eight orbitals
        dict(name="integrals mixed water", op="integrals", n=8, mixed=True, **water),
        # the orbital propagation of a (short) time step of the benchmark: the main path
        dict(name="propagate mixed h2", op="propagate", n=4, mixed=True, m=10, z=24.0, rule="ladder", **h2),
        # the same in plain FP64 on an odd count and degree
        dict(name="propagate fp64 odd", op="propagate", n=3, mixed=False, m=12, z=60.0, rule="ladder", **odd),
        # whole time steps: the benchmark's own, and the FP64 form on a small molecule box
        dict(name="step mixed h2", op="step", n=4, mixed=True, m=10, dt=0.02, mg=True, warm=True, **h2),
        dict(name="step fp64 small", op="step", n=4, mixed=False, m=10, dt=0.02, mg=True, warm=True, **small),
        # a control-field gradient: dipole signal forward, adjoint sweep backward
        dict(name="gradient fp64 small", op="gradient", mixed=False, m=12, steps=4, dt=0.02, **small),
    ]


def draw(rng):
    """One more case: the same operations over degrees, sizes, orbital counts, precisions and rules."""
    op = rng.choice(["h1", "stiff", "batch", "poisson", "integrals", "propagate", "propagate", "step", "gradient"])
    if op == "batch":
        lo = 2.0e4 * 2.0 ** rng.uniform(0.0, 2.0)
        return dict(op=op, count=rng.randint(2, 12), lo_dofs=round(lo), hi_dofs=round(lo * 2.0 ** rng.uniform(0.5, 2.5)))
    p = rng.choice([2, 3, 4, 4])
    levels = rng.randint(1, 5)
    # unknowns before refinement, log-uniform; the iterative calls take the smaller part of the range
    top = {"h1": 1.6e6, "stiff": 1.6e6, "integrals": 8e5, "poisson": 4e5, "propagate": 4e5}.get(op, 6e4)
    target = math.exp(rng.uniform(math.log(8e3), math.log(top)))
    nc = max(3, round(target ** (1.0 / 3.0) / p))
    c = dict(op=op, mol=rng.choice(["h", "h2", "h2", "water"]), box=round(rng.uniform(8.0, 40.0), 2), nc=nc, p=p,
             levels=levels, mixed=rng.random() < 0.7)
    if op == "gradient":
        c.update(m=rng.randint(8, 14), steps=rng.randint(2, 5), dt=round(_dt(c, rng.uniform(5.0, 20.0)), 9))
        return c
    c["n"] = rng.randint(2, 4) if op == "step" else rng.randint(1, 8)
    if op in ("stiff", "poisson") and c["n"] == 7:
        c["n"] = 6   # 49 real columns at degree 4 are outside the launch limits of the float64 stiffness
    if op == "poisson":
        c.update(mg=rng.random() < 0.6, warm=rng.random() < 0.5)
    elif op == "propagate":
        c.update(m=rng.randint(6, 16), z=round(rng.uniform(5.0, 40.0), 2), rule=rng.choice(["ladder", "ladder", "fixed"]))
    elif op == "step":
        c.update(m=rng.randint(8, 14), dt=round(_dt(c, rng.uniform(5.0, 30.0)), 9), mg=rng.random() < 0.7, warm=rng.random() < 0.5)
    return c


def _nuclei(c):
    """((position), charge, refinement levels) as in the workloads."""
    L = c["levels"]
    if c["mol"] == "h":
        return [((0.0, 0.0, 0.0), 1.0, L)]
    if c["mol"] == "h2":
        return [((0.0, 0.0, 0.7), 1.0, L), ((0.0, 0.0, -0.7), 1.0, L)]
    return [((0.0, 0.0, 0.0), 8.0, L), ((1.4311, 1.1081, 0.0), 1.0, L - 1), ((-1.4311, 1.1081, 0.0), 1.0, L - 1)]


def _mesh_args(c):
    return -c["box"], c["box"], c["nc"], c["p"], _nuclei(c), 2.0


def _top_eigenvalue(c):
    """Size of the largest eigenvalue of H1~: about 844 (p/4)^4 / h_min^2."""
    return 844.0 * (c["p"] / 4.0) ** 4 / (2.0 * c["box"] / c["nc"] / 2 ** c["levels"]) ** 2


def _dt(c, z):
    """The propagation length that spans z in units of the inverse largest eigenvalue."""
    return z / _top_eigenvalue(c)


def _batch_instances(c):
    """Uneven instances of the batching form: log-uniform sizes, degrees 2..4, 1..8 orbitals."""
    rng = np.random.default_rng(2301 + c["count"])
    out = []
    for _ in range(c["count"]):
        target = math.exp(rng.uniform(math.log(c["lo_dofs"]), math.log(c["hi_dofs"])))
        p = int(rng.integers(2, 5))
        out.append(dict(mol=("h", "h2", "water")[int(rng.integers(0, 3))], box=BATCH_BOX, p=p, levels=2,
                        nc=max(2, round(target ** (1.0 / 3.0) / p)), n=int(rng.integers(1, 9))))
    return out


# ------------------------------------------------------- what a program holds
@functools.lru_cache(maxsize=32)
def _mesh(mol, box, nc, p, levels, mg):
    """One mesh handle per workload, as a program builds it once and keeps it."""
    c = dict(mol=mol, box=box, nc=nc, p=p, levels=levels)
    mesh = pkg.Mesh(*_mesh_args(c))
    if mg:
        pkg.mesh_set_option(mesh, pkg.OPT_POISSON_SOLVER, pkg.POISSON_MULTIGRID)
    X, ml, _ = mesh.tables()
    return mesh, torch.from_numpy(X).cuda(), torch.from_numpy(ml).cuda()


def _mesh_of(c):
    return _mesh(c["mol"], c["box"], c["nc"], c["p"], c["levels"], bool(c.get("mg", False)))


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _orbitals(c, X, ml, n_interior, n, seed):
    """n Gaussian orbitals on the nuclei with seeded exponents, displacements and
    momenta, orthonormal in the mass M_L, zero on the box surface."""
    rng = np.random.default_rng(seed)
    nuc = _nuclei(c)
    cols = []
    for j in range(n):
        d = X - torch.from_numpy(np.array(nuc[j % len(nuc)][0]) + 0.05 * rng.standard_normal(3)).to(X)
        a = d[:, j % 3] * (1.0 if j < 5 else d[:, (j + 1) % 3]) if j >= len(nuc) else torch.ones_like(d[:, 0])
        a = a * torch.exp(-(0.5 + 0.4 * j / n + 0.05 * rng.random()) * (d * d).sum(1))
        cols.append(torch.polar(torch.ones_like(a), X @ torch.from_numpy(0.2 * rng.standard_normal(3)).to(X)) * a)
    phi = torch.stack(cols, 1)
    phi[n_interior:] = 0
    S = phi.conj().T @ (ml[:, None] * phi)
    w, V = torch.linalg.eigh(S)
    return (phi @ (V * w.rsqrt().to(V.dtype)) @ V.conj().T).contiguous()


def _mean_field(X, n, seed):
    """Smooth seeded mean-field operator fields U_pq, nearly Hermitian, [N, n, n]."""
    rng = np.random.default_rng(seed + 1)
    U = torch.empty((len(X), n, n), dtype=torch.complex128, device="cuda")
    for q in range(n):
        for r in range(q, n):
            s = torch.from_numpy(0.4 * rng.standard_normal(3)).to(X)
            f = ((X - s) ** 2).sum(1).add_(1.0 + rng.random()).rsqrt()
            a = complex(0.3 * rng.standard_normal(), 0.3 * rng.standard_normal()) if r > q else 1.0 + 0.2 * rng.random()
            U[:, q, r] = a * f
            if r > q:
                U[:, r, q] = (0.9 * np.conj(a)) * f
    return U


def _fields(X, n, seed):
    """Smooth seeded pair potentials in the column layout of the Poisson batch, [N, n^2]."""
    rng = np.random.default_rng(seed + 2)
    W = torch.empty((len(X), n * n), dtype=torch.float64, device="cuda")
    for q in range(n * n):
        s = torch.from_numpy(0.5 * rng.standard_normal(3)).to(X)
        W[:, q] = (1.0 if q < n else 0.3 * rng.standard_normal()) * ((X - s) ** 2).sum(1).add_(0.5 + rng.random()).rsqrt()
    return W


def _field(seed, amp=0.05):
    e = np.random.default_rng(seed + 3).standard_normal(3)
    return tuple(float(v) for v in amp * e / np.linalg.norm(e))


def _ci(n, seed):
    """CI vector of one alpha and one beta electron: the lowest determinant and seeded others."""
    rng = np.random.default_rng(seed + 4)
    C = 0.1 * (rng.standard_normal(n * n) + 1j * rng.standard_normal(n * n))
    C[0] = 1.0
    return C / np.linalg.norm(C)


def _inputs(case, seed):
    """Everything made from the seed, without a library call that computes: shared by prepare and exact."""
    op = case["op"]
    mesh, X, ml = _mesh_of(case)
    n, g = case.get("n", 1), _generator(seed)
    if op == "h1":
        x = torch.randn((mesh.N, n), generator=g, dtype=torch.complex128, device="cuda")
        return dict(x=x.to(torch.complex64) if case["mixed"] else x, E=_field(seed))
    if op == "stiff":
        return dict(x=torch.randn((mesh.N, n * n), generator=g, dtype=torch.float32 if case["mixed"] else torch.float64, device="cuda"))
    phi = _orbitals(case, X, ml, mesh.n_interior, n, seed)
    s = dict(phi=phi, E=_field(seed))
    if op == "propagate":
        s.update(U=_mean_field(X, n, seed), dt=_dt(case, case["z"]))
    elif op == "integrals":
        s["W"] = _fields(X, n, seed)
    elif op == "step":
        s["C"] = torch.from_numpy(_ci(n, seed)).cuda()
    elif op == "gradient":
        rng = np.random.default_rng(seed + 5)
        s.update(phi=phi[:, 0].contiguous(), Ek=0.05 * rng.standard_normal(case["steps"]), g=rng.standard_normal(case["steps"] + 1))
    return s


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        parts = _batch_instances(case)
        meshes = [_mesh_of(c)[0] for c in parts]
        xs = _batch_inputs(parts, meshes, seed)
        return dict(case=case, batch=pkg.Batch(meshes), xs=xs, ys=[torch.empty_like(x) for x in xs],
                    E=[_field(seed + i) for i in range(len(parts))])
    mesh, X, ml = _mesh_of(case)
    s = dict(case=case, mesh=mesh, prec=pkg.PREC_MIXED if case["mixed"] else pkg.PREC_FP64, **_inputs(case, seed))
    n = case.get("n", 1)
    if op in ("h1", "stiff"):
        s["y"] = torch.empty_like(s["x"])
    elif op == "propagate":
        s["out"] = torch.empty_like(s["phi"])
    elif op in ("poisson", "step"):
        s["W"] = torch.empty((mesh.N, n * n), dtype=torch.float64, device="cuda")
        s["W0"] = torch.zeros_like(s["W"])
        if case["warm"]:   # the fields of slightly different orbitals, as the previous step leaves them
            prev = s["phi"] * (1.0 + 2e-3 * X[:, 2:].clamp(-4.0, 4.0))
            pkg.poisson_batch(mesh, prev.contiguous(), s["W0"], rtol=1e-8, precision=s["prec"])
        if op == "step":
            s["solver"] = pkg.MCTDHF(mesh, n, 1, 1, case["m"])
            s["solver"].set_precision(s["prec"])
            s["solver"].set_krylov_tol(1e-10)
            s["phi_t"], s["C_t"] = torch.empty_like(s["phi"]), torch.empty_like(s["C"])
    elif op == "integrals":
        s["eri"] = torch.empty((n * n, n * n), dtype=torch.complex128, device="cuda")
    return s


def _batch_inputs(parts, meshes, seed):
    return [torch.randn((m.N, c["n"]), generator=_generator(seed + i), dtype=torch.complex64, device="cuda")
            for i, (c, m) in enumerate(zip(parts, meshes))]


# -------------------------------------------------------------------- one pass
def run(s):
    case = s["case"]
    op = case["op"]
    if op == "batch":
        return s["batch"].apply(pkg.OP_H1_C64, s["xs"], s["ys"], E=s["E"])
    mesh, prec = s["mesh"], s["prec"]
    if op == "h1":
        return pkg.op_apply(mesh, pkg.OP_H1_C64 if case["mixed"] else pkg.OP_H1, s["x"], s["y"], E=s["E"])
    if op == "stiff":
        return pkg.op_apply(mesh, pkg.OP_STIFF_F32 if case["mixed"] else pkg.OP_STIFF, s["x"], s["y"])
    if op == "integrals":
        return pkg.two_electron_integrals(mesh, s["phi"], s["W"], eri=s["eri"], precision=prec)
    if op == "poisson":
        s["W"].copy_(s["W0"])
        pkg.poisson_batch(mesh, s["phi"], s["W"], rtol=1e-10, warm_start=case["warm"], precision=prec)
        return s["W"]
    if op == "propagate":
        if case["rule"] == "fixed":   # one Krylov step of dimension m over a short time
            return pkg.arnoldi_step(mesh, s["phi"], s["U"], case["m"], 0.1 * s["dt"], E=s["E"], out=s["out"], precision=prec)[0]
        return pkg.arnoldi_propagate(mesh, s["phi"], s["U"], case["m"], s["dt"], 1e-10, E=s["E"], out=s["out"], precision=prec)[0]
    if op == "gradient":
        d, _, ckpt = adjoint.tdse_forward(mesh, s["phi"], s["Ek"], case["dt"], krylov_m=case["m"], tol=1e-10, precision=prec, ckpt_every=2)
        grad, lam = adjoint.tdse_vjp(mesh, ckpt, 2, s["Ek"], s["g"], case["dt"], krylov_m=case["m"], tol=1e-10, precision=prec, want_lam0=True)
        return dict(signal=d, grad=grad, lam=lam)
    # a whole time step from the same state each pass (the step works in place)
    s["phi_t"].copy_(s["phi"])
    s["C_t"].copy_(s["C"])
    s["W"].copy_(s["W0"])
    info = s["solver"].step(s["phi_t"], s["C_t"], s["W"], s["E"], case["dt"])
    return dict(phi=s["phi_t"], C=s["C_t"], W=s["W"], energy=info["energy"], dipole=np.array(info["dipole"]))


# --------------------------------------------- what a pass cannot do without
def _unknowns(c):
    """Unknowns of the mesh, from its host description."""
    return _counts(c["mol"], c["box"], c["nc"], c["p"], c["levels"])


@functools.lru_cache(maxsize=64)
def _counts(mol, box, nc, p, levels):
    m = pkg.Mesh(*_mesh_args(dict(mol=mol, box=box, nc=nc, p=p, levels=levels)), host_only=True)
    return m.N, m.n_cells


def work(case):
    """Each input read and each output written once; the arithmetic of the
    definitions: 6 (p + 1) + 6 flops per cell node and real column of an
    operator, 8 per complex product of the Gram-Schmidt passes."""
    op = case["op"]
    if op == "batch":
        parts = [work(dict(c, op="h1", mixed=True)) for c in _batch_instances(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    N, cells = _unknowns(case)
    n, p1 = case.get("n", 1), case["p"] + 1
    cell = cells * p1 ** 3 * (6.0 * p1 + 6.0)          # one real column
    size = 8 if case["mixed"] else 16
    if op == "h1":
        return dict(bytes=2.0 * N * n * size, flops=2.0 * n * cell)
    if op == "stiff":
        return dict(bytes=N * n * n * size, flops=n * n * cell)
    if op == "integrals":
        return dict(bytes=N * (16.0 * n + 8.0 * n * n) + 16.0 * n ** 4, flops=4.0 * N * n ** 4)
    poisson = dict(bytes=N * (16.0 * n + 16.0 * n * n), flops=12.0 * n * n * cell)   # a dozen preconditioned sweeps
    if op == "poisson":
        return poisson
    # applications of G: about half the span of the spectrum times the length
    m = case["m"]
    if op == "gradient":
        z = case["steps"] * case["dt"] * _top_eigenvalue(case) * 4.0   # forward, recomputation, a pair backward
    elif op == "step":
        z = case["dt"] * _top_eigenvalue(case)
    else:
        z = case["z"] * (0.1 if case["rule"] == "fixed" else 1.0)
    apps = max(m, z * m / 4.0)
    flops = apps * (2.0 * n * cell + N * n * (8.0 * n + 8.0 * (m + 1)))
    if op == "gradient":
        return dict(bytes=3.0 * 16.0 * N, flops=flops)
    prop = dict(bytes=N * n * 16.0 * (2 + n), flops=flops)
    if op == "propagate":
        return prop
    return dict(bytes=2.0 * 16.0 * N * n + poisson["bytes"], flops=flops + poisson["flops"] + 4.0 * N * n ** 4)


# ------------------------------------------------------ the same in 64 bits
def _lagrange(xi, t):
    """Values of the Lagrange polynomials through xi at t: [..., p + 1]."""
    out = []
    for i in range(len(xi)):
        v = torch.ones_like(t)
        for j in range(len(xi)):
            if j != i:
                v = v * (t - xi[j]) / (xi[i] - xi[j])
        out.append(v)
    return torch.stack(out, -1)


def _gll(p):
    """Gauss-Lobatto points and weights on [0, 1] and the stiffness int L_i' L_j'."""
    P = np.polynomial.legendre.Legendre.basis(p)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real) if p > 1 else [], [1.0]])
    x = 0.5 * (x - x[::-1])
    w = 1.0 / (p * (p + 1) * P(x) ** 2)
    xi = 0.5 * (x + 1.0)
    D = np.zeros((p + 1, p + 1))   # D[i, j] = L_j'(xi_i)
    for j in range(p + 1):
        poly = np.poly1d([1.0])
        for k in range(p + 1):
            if k != j:
                poly *= np.poly1d([1.0, -xi[k]]) / (xi[j] - xi[k])
        D[:, j] = np.polyder(poly)(xi)
    return xi, w, D.T @ (w[:, None] * D)


class Space:
    """The finite-element space of a case in plain torch: octree, support points,
    hanging-point interpolation C, and the operators, all in 64 bits."""

    def __init__(self, c, X):
        dev = X.device
        nc, p, box = c["nc"], c["p"], c["box"]
        nuc = [(np.array(R), Z, L) for R, Z, L in _nuclei(c)]
        lo, h0, top = -box, 2.0 * box / nc, max(L for _, _, L in nuc)
        cells = self._octree(lo, h0, nc, nuc, top)
        hmin = h0 / 2 ** int(cells[:, 0].max())
        self.nuc, self.c = nuc, c
        xi, w, K = _gll(p)
        self.K, self.w = torch.from_numpy(K).to(dev), torch.from_numpy(w).to(dev)
        xi = torch.from_numpy(xi).to(dev)
        lev, ijk = torch.from_numpy(cells[:, 0]).to(dev), torch.from_numpy(cells[:, 1:]).to(dev)
        h = h0 / 2.0 ** lev.double()
        self.h = h
        p1 = p + 1
        loc = torch.stack(torch.meshgrid(xi, xi, xi, indexing="ij")[::-1], -1).reshape(-1, 3)   # x runs fastest
        pos = lo + (ijk[:, None, :] + loc[None]) * h[:, None, None]

        def keys(x):
            q = torch.round((x - lo) / hmin * KEY).long()
            return (q[..., 0] << 42) | (q[..., 1] << 21) | q[..., 2]
        uniq, self.cell = torch.unique(keys(pos), return_inverse=True)
        nf = len(uniq)
        self.X = torch.empty((nf, 3), dtype=torch.float64, device=dev)
        self.X[self.cell.reshape(-1)] = pos.reshape(-1, 3)
        # the coarsest leaf whose closure holds each point
        coarse, leaf = torch.full((nf,), 99, device=dev), torch.zeros(nf, dtype=torch.long, device=dev)
        order = {}
        for lv in torch.unique(lev).tolist():
            at = (lev == lv).nonzero()[:, 0]
            m = nc << lv
            kk = (ijk[at, 0] * m + ijk[at, 1]) * m + ijk[at, 2]
            kk, perm = kk.sort()
            order[lv] = (kk, at[perm], m)
        for sg in itertools.product((-1.0, 1.0), repeat=3):
            y = self.X + 1e-3 * hmin * torch.tensor(sg, dtype=torch.float64, device=dev)
            inside = ((y > lo) & (y < box)).all(1)
            for lv, (kk, at, m) in order.items():
                q = torch.floor((y - lo) / (h0 / 2 ** lv)).long().clamp(0, m - 1)
                k = (q[:, 0] * m + q[:, 1]) * m + q[:, 2]
                j = torch.searchsorted(kk, k).clamp(max=len(kk) - 1)
                hit = inside & (kk[j] == k) & (lv < coarse)
                coarse[hit], leaf[hit] = lv, at[j[hit]]
        t = (self.X - (lo + ijk[leaf] * h[leaf, None])) / h[leaf, None]
        master = ((t[..., None] - xi).abs().amin(-1) < 1e-7).all(1)
        # unknowns in the caller's order
        pk, porder = keys(X).sort()
        if int(master.sum()) != len(X) or not torch.equal(pk, uniq[master]):
            raise RuntimeError("the mesh of the definitions and the caller's unknowns differ")
        number = torch.full((nf,), -1, dtype=torch.long, device=dev)
        number[master] = porder
        hang = (~master).nonzero()[:, 0]
        L = _lagrange(xi, t[hang])
        wts = torch.einsum("hc,hb,ha->hcba", L[:, 2], L[:, 1], L[:, 0]).reshape(len(hang), -1)
        cols = number[self.cell[leaf[hang]]]
        keep = wts.abs() > 1e-9
        if int(cols[keep].min() if keep.any() else 0) < 0:
            raise RuntimeError("a hanging point depends on another")
        rows = hang[:, None].expand_as(cols)[keep]
        ij = torch.stack([torch.cat([master.nonzero()[:, 0], rows]), torch.cat([number[master], cols[keep]])])
        v = torch.cat([torch.ones(len(X), dtype=torch.float64, device=dev), wts[keep]])
        self.C = torch.sparse_coo_tensor(ij, v, (nf, len(X))).coalesce().to_sparse_csr()
        self.CT = torch.sparse_coo_tensor(ij.flip(0), v, (len(X), nf)).coalesce().to_sparse_csr()
        self.C2T = torch.sparse_coo_tensor(ij.flip(0), v * v, (len(X), nf)).coalesce().to_sparse_csr()
        w3 = torch.einsum("c,b,a->cba", self.w, self.w, self.w).reshape(-1)
        self.mf = self._add(h[:, None] ** 3 * w3)
        self.ml = (self.CT @ self.mf[:, None])[:, 0]
        self.inside = ((X.abs() < box - 1e-9 * box).all(1)).double()[:, None]
        self.V = torch.zeros(nf, dtype=torch.float64, device=dev)
        for R, Z, _ in nuc:
            d = (self.X - torch.from_numpy(R).to(dev)).norm(dim=1)
            self.V -= Z * torch.where(d < 1e-10, C3 / self.mf ** (1.0 / 3.0), 1.0 / d.clamp(min=1e-10))
        self.Xm = X

    @staticmethod
    def _octree(lo, h0, nc, nuc, top):
        grid = np.stack(np.meshgrid(*[np.arange(nc)] * 3, indexing="ij"), -1).reshape(-1, 3)
        kids = np.array(list(itertools.product((0, 1), repeat=3)))

        def children(q):
            return (2 * q[:, None, :] + kids).reshape(-1, 3)
        split, q = [], grid
        for lv in range(top):
            h = h0 / 2 ** lv
            a = lo + q * h
            hit = np.zeros(len(q), bool)
            for R, _, L in nuc:
                if lv < L:
                    d = np.maximum(np.maximum(a - R, R - (a + h)), 0.0)
                    hit |= (d * d).sum(1) <= (2.0 * h) ** 2
            split.append(q[hit])
            q = children(q[hit])
        around = np.array(list(itertools.product((-1, 0, 1), repeat=3)))
        for lv in range(top - 1, 0, -1):   # the neighbours of a split cell exist at its level
            nb = (split[lv][:, None, :] + around).reshape(-1, 3)
            nb = nb[((nb >= 0) & (nb < nc << lv)).all(1)] // 2
            split[lv - 1] = np.unique(np.concatenate([split[lv - 1], nb]), axis=0)
        out = []
        for lv in range(top + 1):
            q = grid if lv == 0 else children(split[lv - 1])
            if lv < top and len(split[lv]):
                m = nc << lv
                flat = [(v[:, 0] * m + v[:, 1]) * m + v[:, 2] for v in (q, split[lv])]
                q = q[~np.isin(flat[0], flat[1])]
            out.append(np.concatenate([np.full((len(q), 1), lv), q], 1))
        return np.concatenate(out).astype(np.int64)

    def _add(self, y):
        """Sum of cell-node values [cells, nodes, ...] at the support points."""
        out = torch.zeros((len(self.X),) + y.shape[2:], dtype=y.dtype, device=y.device)
        return out.index_add_(0, self.cell.reshape(-1), y.reshape((-1,) + y.shape[2:]))

    @staticmethod
    def _mm(S, x):
        if x.is_complex():
            k = x.shape[1]
            return torch.view_as_complex((S @ torch.view_as_real(x).reshape(len(x), 2 * k)).reshape(-1, k, 2))
        return S @ x

    def full(self, x):
        return self._mm(self.C, x)

    def back(self, y):
        return self._mm(self.CT, y)

    def stiff_full(self, u):
        """A_f u for real u [support points, k]."""
        p1, k = len(self.w), u.shape[1]
        out = torch.zeros_like(u)
        step = max(1, (1 << 27) // (p1 ** 3 * k))
        for a in range(0, len(self.h), step):
            at = self.cell[a:a + step]
            v = u[at].reshape(-1, p1, p1, p1, k)
            w, K = self.w, self.K
            y = torch.einsum("xi,czyik->czyxk", K, v) * (w[:, None] * w)[None, :, :, None, None]
            y += torch.einsum("yi,czixk->czyxk", K, v) * (w[:, None, None] * w)[None, :, :, :, None]
            y += torch.einsum("zi,ciyxk->czyxk", K, v) * (w[:, None] * w)[None, None, :, :, None]
            y *= self.h[a:a + step, None, None, None, None]
            out.index_add_(0, at.reshape(-1), y.reshape(-1, k))
        return out

    def stiff(self, x):
        if x.is_complex():
            k = x.shape[1]
            return torch.view_as_complex(self.stiff(torch.view_as_real(x).reshape(len(x), 2 * k)).reshape(-1, k, 2))
        return self.back(self.stiff_full(self.full(x)))

    def h1_matrix(self, x, E):
        """H1~ x without the inverse mass (surface entries of x are zero)."""
        f = self.mf * (self.V + self.X @ torch.tensor(E, dtype=torch.float64, device=x.device))
        return 0.5 * self.stiff(x) + self.back(f[:, None] * self.full(x))

    def h1(self, x, E):
        return self.inside * self.h1_matrix(self.inside * x, E) / self.ml[:, None]

    def spectrum(self):
        """An interval that holds the spectrum of H1~ and what is added to it."""
        r = torch.linalg.eigvalsh(self.K / (self.w[:, None] * self.w).sqrt()).max()
        return -60.0 - 2.0 * sum(Z for _, Z, _ in self.nuc) ** 2, float(1.4 * 1.5 * r / self.h.min() ** 2 + 60.0)

    def propagator(self, apply, v, dt, span=None):
        """exp(-i dt A) v by the Chebyshev series of the exponential on an interval around the spectrum."""
        a, b = span or self.spectrum()
        c, R = 0.5 * (a + b), 0.5 * (b - a)
        z = R * abs(dt)
        J = _bessel(z, int(z + 14.0 * z ** (1.0 / 3.0)) + 40)
        sg = -1j if dt > 0 else 1j
        t0, t1 = v, (apply(v) - c * v) / R
        out = J[0] * t0 + 2.0 * sg * J[1] * t1
        f = sg
        for k in range(2, len(J)):
            t0, t1 = t1, 2.0 * (apply(t1) - c * t1) / R - t0
            f = f * sg
            out = out + (2.0 * J[k] * f) * t1
        return out * complex(math.cos(c * dt), -math.sin(c * dt))

    def mean_fields(self, phi):
        """Columns of the pair potentials: multipole surface data, then the Dirichlet problem by CG."""
        n = phi.shape[1]
        pf = self.full(self.inside * phi)
        rho = [pf[:, r].abs() ** 2 for r in range(n)]
        for r in range(n):
            for q in range(r + 1, n):
                z = pf[:, r].conj() * pf[:, q]
                rho += [z.real, z.imag]
        src = self.mf[:, None] * torch.stack(rho, 1)
        W = torch.zeros((len(phi), n * n), dtype=torch.float64, device=phi.device)
        edge = self.inside[:, 0] == 0
        r2 = (self.Xm[edge] ** 2).sum(1)
        for (l, f), (_, e) in zip(_harmonics(self.X), _harmonics(self.Xm[edge])):
            W[edge] += (4.0 * math.pi / (2 * l + 1)) * (e / r2 ** (l + 0.5))[:, None] * (f @ src)[None]
        b = self.inside * (4.0 * math.pi * self.back(src) - self.stiff(W))
        w3 = torch.einsum("c,b,a->cba", self.w, self.w, self.w)
        kd = self.K.diagonal() / self.w
        diag = self._add((self.h[:, None] * (w3 * (kd[:, None, None] + kd[:, None] + kd)).reshape(-1)))
        dinv = self.inside / (self.C2T @ diag[:, None])
        x, r = torch.zeros_like(b), b.clone()
        z = dinv * r
        q, rz, bb = z.clone(), (r * z).sum(0), (b * b).sum(0)
        for it in range(20000):
            Aq = self.inside * self.stiff(q)
            al = torch.nan_to_num(rz / (q * Aq).sum(0), 0.0, 0.0, 0.0)
            x += al * q
            r -= al * Aq
            z = dinv * r
            new = (r * z).sum(0)
            if it % 20 == 0 and bool(((r * r).sum(0) <= 1e-27 * bb).all()):
                break
            q = z + torch.nan_to_num(new / rz, 0.0, 0.0, 0.0) * q
            rz = new
        return W + x

    def integrals(self, phi, W):
        """(pq|rs), [n^2, n^2], from orbitals and the columns of their pair potentials."""
        n = phi.shape[1]
        pf, Wf = self.full(self.inside * phi), self.full(_pairs(W, n))
        d = (pf.conj()[:, :, None] * pf[:, None, :]).reshape(-1, n * n)
        return sum(a.T @ (m[:, None] * b) for a, m, b in zip(d.split(1 << 18), self.mf.split(1 << 18), Wf.split(1 << 18)))

    def packed(self, phi, U, E):
        """v -> G v with the projector on phi and the mean-field operator U [N, n, n]."""
        n = phi.shape[1]
        Uf = (self.mf[:, None] * self.full(U.reshape(len(phi), n * n))).reshape(-1, n, n)
        phi = self.inside * phi

        def apply(v):
            v = self.inside * v
            z = self.inside * (self.h1_matrix(v, E) + self.back((Uf * self.full(v)[:, None, :]).sum(2)))
            return z / self.ml[:, None] - phi @ (phi.conj().T @ z)
        return apply

    def step(self, phi, C, E, dt):
        n = phi.shape[1]
        W = self.mean_fields(phi)
        x = self.inside * phi
        h = x.conj().T @ self.h1_matrix(x, E)
        eri = self.integrals(phi, W).reshape(n, n, n, n)
        Ex = [[_excitation(n, p, q).to(phi.device) for q in range(n)] for p in range(n)]
        H = sum(h[p, q] * Ex[p][q] for p in range(n) for q in range(n))
        g1 = torch.empty((n, n), dtype=phi.dtype, device=phi.device)
        g2 = torch.empty((n,) * 4, dtype=phi.dtype, device=phi.device)
        for p, q in itertools.product(range(n), repeat=2):
            g1[p, q] = torch.vdot(C, Ex[p][q] @ C)
        for p, q, r, s in itertools.product(range(n), repeat=4):
            T = Ex[p][q] @ Ex[r][s] - (Ex[p][s] if q == r else 0.0)
            H = H + 0.5 * eri[p, q, r, s] * T
            g2[p, q, r, s] = torch.vdot(C, T @ C)
        lam, B = torch.linalg.eigh(0.5 * (H + H.conj().T))
        Cn = B @ (torch.polar(torch.ones_like(lam), -dt * lam) * (B.conj().T @ C))
        G = torch.einsum("po,oqrs->pqrs", torch.linalg.inv(g1), g2).reshape(n * n, n * n)
        U = (_pairs(W, n) @ G.T).reshape(-1, n, n)
        energy = float((h * g1).sum().real + 0.5 * (eri * g2).sum().real)
        pf = self.full(x)
        dip = [float((g1 * (pf.conj().T @ ((self.mf * self.X[:, d])[:, None] * pf))).sum().real) for d in range(3)]
        new = self.propagator(self.packed(phi, U, E), phi, dt)
        return dict(phi=new, C=Cn, W=W, energy=energy, dipole=np.array(dip))

    def gradient(self, phi, Ek, g, dt):
        """Signal <phi_k, z phi_k> of a field along z, its gradient by the adjoint recursion, and lambda_0."""
        zf = self.mf * self.X[:, 2]

        def pos(x):
            return self.inside * self.back(zf[:, None] * self.full(self.inside * x)) / self.ml[:, None]

        def dot(u, v):
            return torch.vdot(u[:, 0], self.ml * v[:, 0])
        traj = [phi[:, None]]
        for e in Ek:
            traj.append(self.propagator(lambda v, e=e: self.h1(v, (0.0, 0.0, e)), traj[-1], dt))
        d = np.array([float(dot(x, pos(x)).real) for x in traj])
        lam, grad = g[-1] * pos(traj[-1]), np.zeros(len(Ek))
        for k in range(len(Ek) - 1, -1, -1):
            E = (0.0, 0.0, float(Ek[k]))

            def block(v, E=E):
                y = self.h1(v, E)
                return torch.cat([y[:, :1], y[:, 1:] + pos(v[:, :1])], 1)
            out = self.propagator(block, torch.cat([lam, torch.zeros_like(lam)], 1), -dt)
            grad[k] = 2.0 * float(dot(out[:, 1:], traj[k]).real)
            lam = out[:, :1] + g[k] * pos(traj[k])
        return dict(signal=d, grad=grad, lam=lam[:, 0])


def _bessel(z, top):
    """J_0(z)..J_top(z) by downward recurrence, normalised with J_0 + 2 sum J_2k = 1."""
    start = max(top, int(z)) + 60
    J = [0.0] * (start + 2)
    J[start] = 1e-280
    for k in range(start, 0, -1):
        J[k - 1] = 2.0 * k / z * J[k] - J[k + 1]
        if abs(J[k - 1]) > 1e200:
            J = [v * 1e-200 for v in J]
    s = J[0] + 2.0 * sum(J[2::2])
    return [v / s for v in J[:top + 1]]


def _harmonics(X):
    """(l, r^l Y_lm(X)) for l <= LMAX, real and orthonormal, from the recurrences in m and l."""
    x, y, z = X.unbind(1)
    r2 = (X * X).sum(1)
    cm, sm = torch.ones_like(x), torch.zeros_like(x)
    for m in range(LMAX + 1):
        for part in ((cm, sm) if m else (cm,)):
            prev, cur = torch.zeros_like(x), part
            for l in range(m, LMAX + 1):
                norm = math.sqrt((2 * l + 1) / (4.0 * math.pi) * math.factorial(l - m) / math.factorial(l + m) * (2 if m else 1))
                yield l, norm * cur
                prev, cur = cur, ((2 * l + 1) * z * cur - (l + m) * r2 * prev) / (l + 1 - m)
        cm, sm = (2 * m + 1) * (x * cm - y * sm), (2 * m + 1) * (x * sm + y * cm)


def _pairs(W, n):
    """Complex W_rs [N, n^2] from the real columns of the Poisson batch."""
    out = torch.zeros((len(W), n, n), dtype=torch.complex128, device=W.device)
    for r in range(n):
        out[:, r, r] = W[:, r].to(out.dtype)
    c = n
    for r in range(n):
        for s in range(r + 1, n):
            out[:, r, s] = torch.complex(W[:, c], W[:, c + 1])
            out[:, s, r] = out[:, r, s].conj()
            c += 2
    return out.reshape(len(W), n * n)


def _excitation(n, p, q):
    """E_pq on the determinants (alpha orbital, beta orbital) of one electron each."""
    e = torch.zeros((n, n), dtype=torch.complex128)
    e[p, q] = 1.0
    one = torch.eye(n, dtype=torch.complex128)
    return torch.kron(e, one) + torch.kron(one, e)


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        parts = _batch_instances(case)
        xs = _batch_inputs(parts, [_mesh_of(c)[0] for c in parts], seed)
        return [Space(c, _mesh_of(c)[1]).h1(x.to(torch.complex128), _field(seed + i)) for i, (c, x) in enumerate(zip(parts, xs))]
    s = _inputs(case, seed)
    sp = Space(case, _mesh_of(case)[1])
    if op == "h1":
        return sp.h1(s["x"].to(torch.complex128), s["E"])
    if op == "stiff":
        return sp.stiff(s["x"].double())
    if op == "integrals":
        return sp.integrals(s["phi"], s["W"])
    if op == "poisson":
        return sp.mean_fields(s["phi"])
    if op == "propagate":
        dt = s["dt"] * (0.1 if case["rule"] == "fixed" else 1.0)
        return sp.propagator(sp.packed(s["phi"], s["U"], s["E"]), s["phi"], dt)
    if op == "gradient":
        return sp.gradient(s["phi"], s["Ek"], s["g"], case["dt"])
    return sp.step(s["phi"], s["C"], s["E"], case["dt"])
