"""The work a program has this library do, as cases for timing it.

Every case builds one boundary-value problem on the host (what a program has
in hand), creates its solver, and times one call of a public entry point on
it: a linear solve, a block solve of several load cases, one application of
the dual operator and the preconditioner, a load step of the hyperelastic
model, or the element matrices alone.  The seed draws the node positions, the
material, the loads and the vectors; the mesh topology and its partition
belong to the case.

Sizes are those of the repository's own workloads: the 8-subdomain cube, the
64-subdomain tube, the 128- and 1024-subdomain jittered tubes, the quadratic
Kelvin cube and the hyperelastic tube.
"""
from __future__ import annotations

import dataclasses
import functools
import math

import numpy as np
import torch

from feti_inputs import mesh
from paper_1508_02599_gb300 import FetiSolver

TOL = 1e-10          # the solver's own default


def listed():
    tube16 = {"mesh": "tube", "nr": 16, "nt": 64, "nz": 32, "pr": 4, "pt": 8, "pz": 2}
    jtube16 = {"mesh": "jtube", "nr": 16, "nt": 64, "nz": 32, "parts": 128}
    jtube32 = {"mesh": "jtube", "nr": 32, "nt": 128, "nz": 64, "parts": 1024}
    cube12 = {"mesh": "cube", "n": 12, "p": 2}
    return [
        # the smallest complete solve: classical FETI on the clamped cube (8 sub-cubes, H/h = 6)
        {"name": "cube_solve", "kind": "solve", **cube12, "method": "classical", "precond": "dirichlet",
         "precision": "fp64"},
        # one operator apply of a program's own Krylov loop at the smallest size: launches and latency
        {"name": "cube_apply", "kind": "apply", **cube12, "precision": "fp64"},
        # an ordinary solve in the default precision: the 64-subdomain tube
        {"name": "tube_solve", "kind": "solve", **tube16, "method": "af", "precond": "dirichlet", "precision": "fp64"},
        # uneven subdomains, the preconditioner of the scaling studies, FP32 operators in the iteration
        {"name": "jtube_lumped", "kind": "solve", **jtube16, "method": "af", "precond": "lumped",
         "precision": "mixed"},
        # eight load cases solved as one block
        {"name": "jtube_block", "kind": "multi", **jtube16, "precision": "mixed", "nrhs": 8},
        # the quadratic cube study with Kelvin's solution as boundary data
        {"name": "p2_solve", "kind": "solve", "mesh": "kelvin_p2", "n": 12, "p": 4, "method": "classical",
         "precond": "dirichlet", "precision": "fp64"},
        # the headline solve: 1024 uneven subdomains, FP32 operators from FP64 factors
        {"name": "jtube32_mixed", "kind": "solve", **jtube32, "method": "af", "precond": "dirichlet",
         "precision": "mixed"},
        # the same with FP32 factors and refined K^+, the fastest form of one solve
        {"name": "jtube32_f32factor", "kind": "solve", **jtube32, "method": "af", "precond": "dirichlet",
         "precision": "mixed_f32factor"},
        # the inner step of every iteration at that size, in both precisions
        {"name": "jtube32_apply_mixed", "kind": "apply", **jtube32, "precision": "mixed"},
        {"name": "jtube32_apply_fp64", "kind": "apply", **jtube32, "precision": "fp64"},
        # element tangents and forces of the two-fibre tube, for a program with its own assembly
        {"name": "hgo_elements", "kind": "elements", "mesh": "hgo", "nr": 24, "nt": 96, "nz": 48, "pr": 4, "pt": 16,
         "pz": 4},
        # one load step (1 mmHg) of the artery model: Newton with a FETI solve per increment
        {"name": "hgo_newton", "kind": "newton", "mesh": "hgo", "nr": 8, "nt": 32, "nz": 16, "pr": 2, "pt": 8,
         "pz": 2, "method": "af"},
    ]


def _draw_tube(rng, lo, hi):
    """Cells of a jittered tube with between lo and hi cells in all, and its number of parts."""
    cells = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    nr = max(3, round((cells / 8) ** (1 / 3) * rng.uniform(0.8, 1.25)))
    nt = 4 * max(3, round((cells / 8) ** (1 / 3) * rng.uniform(0.8, 1.25)))
    nz = max(4, round(cells / (nr * nt)))
    parts = max(2, round(nr * nt * nz / rng.uniform(180, 500)))
    return {"mesh": "jtube", "nr": nr, "nt": nt, "nz": nz, "parts": parts}


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "apply", "apply", "multi", "p2", "elements", "newton"])
    precision = rng.choice(["fp64", "mixed", "mixed_f32factor"])
    if kind == "solve":
        return {"kind": "solve", **_draw_tube(rng, 2e3, 1e5), "method": rng.choice(["af", "af", "classical"]),
                "precond": rng.choice(["dirichlet", "dirichlet", "lumped"]), "precision": precision}
    if kind == "apply":
        return {"kind": "apply", **_draw_tube(rng, 1e3, 2e5), "precision": rng.choice(["fp64", "mixed"])}
    if kind == "multi":
        return {"kind": "multi", **_draw_tube(rng, 2e3, 5e4), "precision": precision, "nrhs": rng.randint(2, 16)}
    if kind == "p2":
        p = rng.randint(2, 4)
        return {"kind": "solve", "mesh": "kelvin_p2", "n": p * rng.randint(2, 3), "p": p,
                "method": rng.choice(["af", "classical"]), "precond": rng.choice(["dirichlet", "lumped"]),
                "precision": precision}
    n = 1 if kind == "newton" else rng.randint(1, 5)
    pr, pt, pz = rng.randint(1, 2) * n, 4 * rng.randint(1, 3), rng.randint(1, 3)
    return {"kind": kind, "mesh": "hgo", "nr": 3 * pr, "nt": pt * rng.randint(3, 5), "nz": pz * rng.randint(3, 6) * n,
            "pr": pr, "pt": pt, "pz": pz, "method": "af"}


@functools.lru_cache(maxsize=4)
def _topology(kind, *size):
    """Mesh, partition and boundary sets of a case before the seed moves anything; and its smallest cell."""
    if kind == "cube":
        n, p = size
        return mesh.cube_problem(n, (p, p, p)), 1.0 / n
    if kind == "kelvin_p2":
        n, p = size
        return mesh.kelvin_cube_problem_p2(n, (p, p, p)), 1.0 / n
    if kind == "jtube":
        nr, nt, nz, parts = size
        return mesh.jittered_cylinder_problem(nr, nt, nz, parts, 1508, 2599), min(0.5 / nr, 2.0 / nz, 2 * math.pi / nt)
    nr, nt, nz, pr, pt, pz = size
    h = min(0.5 / nr, 2.0 / nz, 2 * math.pi / nt)
    if kind == "tube":
        return mesh.cylinder_problem(nr, nt, nz, (pr, pt, pz)), h
    # 1 mmHg in kPa, bulk modulus 100 kPa as in the paper's scaling studies
    return mesh.cylinder_problem(nr, nt, nz, (pr, pt, pz), material=mesh.hgo_material(kappa=100.0),
                                 pressure=0.13332), h


_SIZE = {"cube": ("n", "p"), "kelvin_p2": ("n", "p"), "jtube": ("nr", "nt", "nz", "parts"),
         "tube": ("nr", "nt", "nz", "pr", "pt", "pz"), "hgo": ("nr", "nt", "nz", "pr", "pt", "pz")}


def _base(case):
    return _topology(case["mesh"], *(case[k] for k in _SIZE[case["mesh"]]))


def _problem(case, seed):
    """The case's problem with the seed's node positions (moved by up to 5 % of
    a cell), material and loads."""
    base, h = _base(case)
    rng = np.random.default_rng([seed, 1])
    t = base.tets
    corners = int(t[:, :4].max()) + 1            # 10-node meshes number the vertices first
    x = base.coords.copy()
    x[:corners] += rng.uniform(-0.05 * h, 0.05 * h, size=(corners, 3))
    while True:                                  # nodes that would invert an element of a jittered mesh stay
        e = x[t[:, 1:4]] - x[t[:, :1]]
        bad = np.nonzero(np.einsum("ei,ei->e", e[:, 0], np.cross(e[:, 1], e[:, 2])) <= 1e-3 * h ** 3)[0]
        stay = np.unique(t[bad, :4])
        if np.array_equal(x[stay], base.coords[stay]):
            break
        x[stay] = base.coords[stay]
    if t.shape[1] == 10:                         # straight edges: midpoints follow their vertices
        for k, (a, b) in enumerate(mesh.P2_EDGES):
            x[t[:, 4 + k]] = 0.5 * (x[t[:, a]] + x[t[:, b]])
    load = rng.uniform(0.8, 1.2)
    mat = dict(base.material)
    if mat["kind"] == mesh.HGO_TWO_FIBRE:
        mat["c"] *= rng.uniform(0.9, 1.1)
    else:
        mat["E"] *= rng.uniform(0.8, 1.2)
        mat["nu"] = min(0.47, mat["nu"] * rng.uniform(0.9, 1.1))
    return dataclasses.replace(base, coords=x, material=mat, pressure=base.pressure * load,
                               traction=base.traction * load, dir_val=base.dir_val * load)


def _scales(case, seed):
    return np.random.default_rng([seed, 2]).uniform(8.0, 16.0, size=case["nrhs"])


def _displacement(case, seed, prob):
    """A state of the artery under load: radial expansion with local variation, [3 N]."""
    rng = np.random.default_rng([seed, 3])
    x = prob.coords
    u = 0.05 * x * np.array([1.0, 1.0, 0.0]) + rng.uniform(-0.02, 0.02, size=x.shape) * _base(case)[1]
    return u.ravel()


def _vector(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(n, dtype=torch.float64, device="cuda", generator=g)


def prepare(case, seed):
    prob = _problem(case, seed)
    kind = case["kind"]
    opt = {"method": case.get("method", "af"), "precond": case.get("precond", "dirichlet"),
           "precision": case.get("precision", "fp64"), "tol": TOL, "maxit": 3000}
    if kind == "newton":
        opt |= {"n_load_steps": 1, "newton_tol": 1e-10}
    s = FetiSolver(prob, **opt)
    state = {"kind": kind, "solver": s}
    if kind in ("solve", "newton"):
        state["u"] = torch.empty(3 * prob.n_nodes, dtype=torch.float64, device="cuda")
    elif kind == "multi":
        state["scales"] = _scales(case, seed)
        state["u"] = torch.empty((case["nrhs"], 3 * prob.n_nodes), dtype=torch.float64, device="cuda")
    elif kind == "apply":
        s.prepare()
        n = s.sizes()["n_lambda"]
        state |= {"v": _vector(n, seed), "q": torch.empty(n, dtype=torch.float64, device="cuda"),
                  "z": torch.empty(n, dtype=torch.float64, device="cuda"), "f32": case["precision"] != "fp64"}
    elif kind == "elements":
        E = prob.n_tets
        state |= {"U": torch.from_numpy(_displacement(case, seed, prob)).cuda(),
                  "Ke": torch.empty((E, 12, 12), dtype=torch.float64, device="cuda"),
                  "fe": torch.empty((E, 12), dtype=torch.float64, device="cuda")}
    torch.cuda.synchronize()                     # the solver runs on its own stream
    return state


def run(state):
    s, kind = state["solver"], state["kind"]
    if kind == "solve":
        return s.solve(out=state["u"])[0]
    if kind == "multi":
        return s.solve_multi(state["scales"], out=state["u"])[0]
    if kind == "newton":
        return s.newton(out=state["u"])[0]
    if kind == "elements":
        Ke, fe = s.elements(state["U"], out=(state["Ke"], state["fe"]))
        return {"Ke": Ke, "fe": fe}
    s.dual_apply(state["v"], state["q"], state["z"], 1)
    if state["f32"]:                             # products with FP32 operators: what they are worth
        return {"q": state["q"].float(), "z": state["z"].float()}
    return {"q": state["q"], "z": state["z"]}


# ---- work -------------------------------------------------------------------

def _sub_sizes(case):
    """Free and boundary DOFs of every subdomain (Dirichlet DOFs are boundary DOFs when all subdomains float)."""
    prob, _ = _base(case)
    npe = prob.tets.shape[1]
    pair = np.unique(np.repeat(prob.part.astype(np.int64), npe) * prob.n_nodes + prob.tets.ravel())
    sub, node = pair // prob.n_nodes, pair % prob.n_nodes
    shared = np.bincount(node, minlength=prob.n_nodes) > 1
    is_dir = np.zeros(3 * prob.n_nodes, bool)
    is_dir[prob.dir_dof] = True
    d = is_dir.reshape(-1, 3).sum(axis=1)
    if case.get("method", "af") == "af":
        n, b = np.full(prob.n_nodes, 3), np.where(shared, 3, d)
    else:
        n, b = 3 - d, np.where(shared, 3 - d, 0)
    count = lambda w: np.bincount(sub, weights=w[node], minlength=prob.n_parts)  # noqa: E731
    return count(n), count(b)


def work(case):
    prob, _ = _base(case)
    E, N = prob.n_tets, prob.n_nodes
    mesh_bytes = 24.0 * N + 4.0 * prob.tets.size + 4.0 * E
    if case["kind"] == "elements":
        return {"bytes": E * (16 + 48 + 156 * 8.0) + 48.0 * N, "flops": 1100.0 * E}
    n, b = _sub_sizes(case)
    ops = 2.0 * float((b * b).sum())                        # flops of one dense local apply
    nl = float(b.sum()) / 2
    if case["kind"] == "apply":
        entry = 8.0 if case["precision"] == "fp64" else 4.0
        return {"bytes": entry * float((b * (b + 1)).sum()) + 24.0 * nl, "flops": 2 * ops}
    factor = float((n ** 3 / 3 + 2 * b ** 3 / 3).sum())     # K_rr, S and its inverse
    rounds = case.get("nrhs", 1)
    if case["kind"] == "newton":
        return {"bytes": mesh_bytes + 48.0 * E + 24.0 * N, "flops": 4 * (factor + 40 * 2 * ops)}
    its = 70 if case.get("precond") == "lumped" else 40     # about what these meshes take to TOL
    return {"bytes": mesh_bytes + 24.0 * N * rounds, "flops": factor + its * rounds * 2 * ops}


# ---- the same results in 64 bits from plain torch ----------------------------

def _dev(a, dtype=None):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda", dtype=dtype)


def _gradients(X):
    """Gradients [E, 4, 3] of the barycentric coordinates and volumes [E] of tetrahedra with vertices X [E, 4, 3]."""
    J = X[:, 1:] - X[:, :1]
    g = torch.linalg.inv(J).transpose(1, 2)                 # rows: gradients of coordinates 1..3
    return torch.cat([-g.sum(dim=1, keepdim=True), g], dim=1), torch.linalg.det(J) / 6.0


def _hooke(G, lam, mu):
    """Element matrix of Hooke's law for shape gradients G [E, a, 3]: [E, 3a, 3a] per unit volume."""
    a = G.shape[1]
    dot = torch.einsum("eak,ebk->eab", G, G)
    K = mu * torch.einsum("eab,ij->eaibj", dot, torch.eye(3, dtype=G.dtype, device=G.device))
    K = K + mu * torch.einsum("eaj,ebi->eaibj", G, G) + lam * torch.einsum("eai,ebj->eaibj", G, G)
    return K.reshape(-1, 3 * a, 3 * a)


def _linear_elements(prob, tets):
    m = prob.material
    lam = m["E"] * m["nu"] / ((1 + m["nu"]) * (1 - 2 * m["nu"]))
    mu = m["E"] / (2 * (1 + m["nu"]))
    x = _dev(prob.coords)
    g, V = _gradients(x[tets[:, :4]])
    if tets.shape[1] == 4:
        return _hooke(g, lam, mu) * V[:, None, None]
    a, b = (5 + 3 * math.sqrt(5)) / 20, (5 - math.sqrt(5)) / 20      # four points, exact for quadratics
    K = 0.0
    for q in range(4):
        L = [a if i == q else b for i in range(4)]
        G = [(4 * L[i] - 1) * g[:, i] for i in range(4)]
        G += [4 * (L[i] * g[:, j] + L[j] * g[:, i]) for i, j in mesh.P2_EDGES]
        K = K + 0.25 * _hooke(torch.stack(G, dim=1), lam, mu)
    return K * V[:, None, None]


def _hgo_energy(u, g, V, a1, a2, c, k1, k2, kappa):
    """Strain energy of one element at its nodal displacements u [12]."""
    F = torch.eye(3, dtype=u.dtype, device=u.device) + u.reshape(4, 3).T @ g
    C = F.T @ F
    J = F[0] @ torch.linalg.cross(F[1], F[2])
    J23 = J ** (-2.0 / 3.0)
    psi = 0.5 * kappa * (J - 1) ** 2 + 0.5 * c * (J23 * torch.trace(C) - 3)
    for a in (a1, a2):
        I4 = J23 * (a @ (C @ a)) - 1
        psi = psi + torch.where(I4 > 1e-12, k1 / (2 * k2) * torch.expm1(k2 * I4 * I4), torch.zeros_like(I4))
    return V * psi


def _hgo_elements(prob, tets, U):
    """Tangents [E, 12, 12] and forces [E, 12] by differentiating the energy."""
    m = prob.material
    g, V = _gradients(_dev(prob.coords)[tets])
    fib = _dev(prob.fibres)
    u = U.reshape(-1, 3)[tets].reshape(-1, 12)
    f = functools.partial(_hgo_energy, c=m["c"], k1=m["k1"], k2=m["k2"], kappa=m["kappa"])
    grad = torch.func.vmap(torch.func.grad(f))
    hess = torch.func.vmap(torch.func.jacfwd(torch.func.grad(f)))
    Ke, fe = [], []
    for s in range(0, tets.shape[0], 1 << 16):
        arg = [t[s:s + (1 << 16)] for t in (u, g, V, fib[:, :3], fib[:, 3:])]
        Ke.append(hess(*arg))
        fe.append(grad(*arg))
    return torch.cat(Ke), torch.cat(fe)


def _loads(prob, U=None):
    """Consistent nodal loads of the pressure (on the moved surface) and traction faces, [3 N]."""
    x = _dev(prob.coords) + (0 if U is None else U.reshape(-1, 3))
    f = torch.zeros((prob.n_nodes, 3), dtype=torch.float64, device="cuda")
    for tri, pressure in ((prob.press_tri, True), (prob.trac_tri, False)):
        if tri.shape[0] == 0:
            continue
        t = _dev(tri, torch.int64)
        X = x if pressure else _dev(prob.coords)
        area = 0.5 * torch.linalg.cross(X[t[:, 1]] - X[t[:, 0]], X[t[:, 2]] - X[t[:, 0]])
        w = prob.pressure * area if pressure else torch.linalg.norm(area, dim=1, keepdim=True) * _dev(prob.traction)
        for v in (range(3, 6) if t.shape[1] == 6 else range(3)):
            f.index_add_(0, t[:, v], w / 3.0)
    return f.ravel()


def _assembled(tets, Ke, n):
    """Sparse CSR matrix [n, n] of the element matrices."""
    nd = Ke.shape[1]
    dof = (3 * tets[:, :, None] + torch.arange(3, device="cuda")).reshape(-1, nd)
    key = (dof[:, :, None] * n + dof[:, None, :]).ravel()
    key, order = torch.sort(key)
    val = Ke.ravel()[order]
    del order
    key, count = torch.unique_consecutive(key, return_counts=True)
    val = torch.segment_reduce(val, "sum", lengths=count)
    row = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    return torch.sparse_csr_tensor(row, key % n, val, (n, n))


def _cg(K, f, free, diag, rounds=4, to=1e-14):
    """K x = f on the free DOFs (x = 0 elsewhere): conjugate gradients, restarted from the true residual."""
    x = torch.zeros_like(f)
    d = torch.where(free, 1.0 / diag, torch.zeros_like(diag))
    goal = to * float(torch.linalg.norm(f * free))
    for _ in range(rounds):
        r = (f - K @ x) * free
        if float(torch.linalg.norm(r)) <= goal:
            break
        z = d * r
        p, rz, dx = z.clone(), r @ z, torch.zeros_like(x)
        for it in range(12000):
            q = (K @ p) * free
            a = rz / (p @ q)
            dx += a * p
            r -= a * q
            z = d * r
            new = r @ z
            if it % 50 == 49 and float(torch.linalg.norm(r)) <= goal:
                break
            p = z + (new / rz) * p
            rz = new
        x = x + dx
    return x


def _diagonal(tets, Ke, n):
    dof = (3 * tets[:, :, None] + torch.arange(3, device="cuda")).reshape(-1)
    return torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(
        0, dof, torch.diagonal(Ke, dim1=1, dim2=2).reshape(-1))


def _exact_solve(prob):
    n = 3 * prob.n_nodes
    tets = _dev(prob.tets, torch.int64)
    Ke = _linear_elements(prob, tets)
    diag = _diagonal(tets, Ke, n)
    K = _assembled(tets, Ke, n)
    del Ke
    free = torch.ones(n, dtype=torch.float64, device="cuda")
    uD = torch.zeros(n, dtype=torch.float64, device="cuda")
    dof = _dev(prob.dir_dof, torch.int64)
    free[dof] = 0.0
    uD[dof] = _dev(prob.dir_val)
    return uD + _cg(K, _loads(prob) - K @ uD, free > 0, diag)


def _exact_newton(prob):
    n = 3 * prob.n_nodes
    tets = _dev(prob.tets, torch.int64)
    dof12 = (3 * tets[:, :, None] + torch.arange(3, device="cuda")).reshape(-1)
    free = torch.ones(n, dtype=torch.bool, device="cuda")
    free[_dev(prob.dir_dof, torch.int64)] = False
    U = torch.zeros(n, dtype=torch.float64, device="cuda")
    for _ in range(40):
        Ke, fe = _hgo_elements(prob, tets, U)
        f = _loads(prob, U)
        r = (f - torch.zeros_like(U).index_add_(0, dof12, fe.ravel())) * free
        if float(torch.linalg.norm(r)) <= 5e-13 * float(torch.linalg.norm(f * free)):
            break
        U = U + _cg(_assembled(tets, Ke, n), r, free, _diagonal(tets, Ke, n), rounds=1, to=1e-8)
    return U


def _exact_apply(prob, seed):
    """q = sum B K^+ B^T v and z = sum W B S B^T W q, all subdomains floating.

    Multipliers: per shared node and component one for every pair of its
    subdomains (lower number first, +1 / -1), in that order, then one for
    every prescribed DOF and subdomain.  Weights: 1 / (number of subdomains)
    on the former (0 on a prescribed DOF), 1 on the latter.  K^+ is zero on
    six boundary DOFs per subdomain, taken by pivoted Gram-Schmidt on the
    rigid modes about the mean node.
    """
    N, P = prob.n_nodes, prob.n_parts
    pair = np.unique(np.repeat(prob.part.astype(np.int64), 4) * N + prob.tets.ravel())
    sub, node = pair // N, pair % N                          # local nodes, subdomain by subdomain, ascending
    first = np.searchsorted(sub, np.arange(P + 1))
    is_dir = np.zeros(3 * N, bool)
    is_dir[prob.dir_dof] = True
    order = np.lexsort((sub, node))                          # copies of each node by subdomain
    ptr = np.searchsorted(node[order], np.arange(N + 1))
    mult = np.diff(ptr)
    rows = []                                                # (node, +1 copy, -1 copy) before components
    for m in range(2, int(mult.max()) + 1):
        nodes = np.nonzero(mult == m)[0]
        k = 0
        for a in range(m):
            for b in range(a + 1, m):
                rows.append(np.stack([nodes, np.full(nodes.size, k), order[ptr[nodes] + a], order[ptr[nodes] + b]], 1))
                k += 1
    rows = np.concatenate(rows)
    rep = np.repeat(rows, 3, axis=0)
    comp = np.tile(np.arange(3), rows.shape[0])
    rank = np.lexsort((rep[:, 1], comp, rep[:, 0]))
    rep, comp = rep[rank], comp[rank]
    w_int = np.where(is_dir[3 * rep[:, 0] + comp], 0.0, 1.0 / mult[rep[:, 0]])
    dnode, dcomp = prob.dir_dof // 3, prob.dir_dof % 3
    reps = mult[dnode]
    start = np.repeat(ptr[dnode], reps) + np.arange(reps.sum()) - np.repeat(np.cumsum(reps) - reps, reps)
    plus = _dev(np.concatenate([3 * rep[:, 2] + comp, 3 * order[start] + np.repeat(dcomp, reps)]), torch.int64)
    minus = _dev(3 * rep[:, 3] + comp, torch.int64)
    n_int, n_all = minus.numel(), 3 * pair.size
    w = _dev(np.concatenate([w_int, np.ones(start.size)]))

    def transpose(x):
        y = torch.zeros(n_all, dtype=torch.float64, device="cuda").index_add_(0, plus, x)
        return y.index_add_(0, minus, -x[:n_int])

    def jump(y):
        q = y[plus]
        q[:n_int] -= y[minus]
        return q

    v = _vector(w.numel(), seed)
    touched = torch.zeros(n_all, dtype=torch.bool, device="cuda")
    touched[plus] = True
    touched[minus] = True
    tets = _dev(prob.tets, torch.int64)
    Ke = _linear_elements(prob, tets)
    by_part = np.argsort(prob.part, kind="stable")
    eptr = np.searchsorted(prob.part[by_part], np.arange(P + 1))
    local = np.searchsorted(pair, prob.part.astype(np.int64)[:, None] * N + prob.tets)
    local, by_part = _dev(local, torch.int64), _dev(by_part, torch.int64)
    touched_h = touched.cpu().numpy()

    def matrix(s):
        e = by_part[eptr[s]:eptr[s + 1]]
        n = 3 * int(first[s + 1] - first[s])
        d = (3 * (local[e] - int(first[s]))[:, :, None] + torch.arange(3, device="cuda")).reshape(-1, 12)
        K = torch.zeros(n * n, dtype=torch.float64, device="cuda")
        K.index_add_(0, (d[:, :, None] * n + d[:, None, :]).ravel(), Ke[e].ravel())
        return K.reshape(n, n)

    g, y = transpose(v), torch.zeros(n_all, dtype=torch.float64, device="cuda")
    for s in range(P):
        lo, hi = 3 * int(first[s]), 3 * int(first[s + 1])
        x = prob.coords[node[first[s]:first[s + 1]]]
        d = x - x.mean(axis=0)
        R = np.zeros((d.shape[0], 3, 6))
        R[:, 0, 0] = R[:, 1, 1] = R[:, 2, 2] = 1.0
        R[:, 0, 3], R[:, 1, 3] = -d[:, 1], d[:, 0]
        R[:, 1, 4], R[:, 2, 4] = -d[:, 2], d[:, 1]
        R[:, 2, 5], R[:, 0, 5] = -d[:, 0], d[:, 2]
        bnd = np.nonzero(touched_h[lo:hi])[0]
        W, fix = R.reshape(-1, 6)[bnd], []
        for _ in range(6):
            nrm = np.einsum("ij,ij->i", W, W)
            nrm[fix] = -1.0
            j = int(np.nonzero(nrm >= nrm.max() * (1 - 1e-10))[0].min())
            fix.append(j)
            W = W - np.outer(W @ W[j], W[j]) / nrm[j]
        keep = np.ones(hi - lo, bool)
        keep[bnd[fix]] = False
        r = _dev(np.nonzero(keep)[0])
        L = torch.linalg.cholesky(matrix(s)[r][:, r])
        y[lo + r] = torch.cholesky_solve(g[lo + r][:, None], L)[:, 0]
    q = jump(y)
    g = transpose(w * q)
    y.zero_()
    for s in range(P):
        lo, hi = 3 * int(first[s]), 3 * int(first[s + 1])
        K = matrix(s)
        b, i = torch.nonzero(touched[lo:hi])[:, 0], torch.nonzero(~touched[lo:hi])[:, 0]
        gb = g[lo + b]
        t = K[b][:, b] @ gb
        if i.numel():
            KIb = K[i][:, b]
            L = torch.linalg.cholesky(K[i][:, i])
            t = t - KIb.T @ torch.cholesky_solve((KIb @ gb)[:, None], L)[:, 0]
        y[lo + b] = t
    return {"q": q, "z": w * jump(y)}


def exact(case, seed):
    prob = _problem(case, seed)
    kind = case["kind"]
    if kind == "solve":
        return _exact_solve(prob)
    if kind == "multi":
        return _dev(_scales(case, seed))[:, None] * _exact_solve(prob)
    if kind == "newton":
        return _exact_newton(prob)
    if kind == "elements":
        Ke, fe = _hgo_elements(prob, _dev(prob.tets, torch.int64), _dev(_displacement(case, seed, prob)))
        return {"Ke": Ke, "fe": fe}
    return _exact_apply(prob, seed)
