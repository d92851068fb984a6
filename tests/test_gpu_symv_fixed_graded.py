"""The fixed-point applies entry by entry, on vectors that fall across a subdomain.

Against the FP64 rows of the same operators, relative to |M| |v| of each
multiplier (|M| from the oracle's dense matrices).  Bound: a row that the
fixed-point form keeps is off by (1.3 m + 80) 2^-56 2^e w and has |M| |v| of at
least 2^-8 2^e w, so by (1.3 m + 80) 2^-48 of |M| |v|; an FP64 sum of m terms by
m 2^-53, in either form and in the other rows.  Without the rows taken in FP64 the
vector that falls by 1e-16 is off by a hundredth of |S| |v|.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from feti_inputs import mesh  # noqa: E402
from oracle import feti  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    prob = mesh.jittered_cylinder_problem(8, 32, 16, 9, 77, 78)
    o = feti.FetiOracle(prob, "af", "dirichlet")
    o.assemble()
    o.factorize()
    # |F_i| and |S_i| between the multipliers of a subdomain, and the coordinate each sits at
    ops = []
    height = np.zeros(o.n_lambda)
    for sd in o.subs:
        bnd = sd.bnd
        keep = ~np.isin(sd.free[bnd], sd.fix)
        F = np.zeros((bnd.size, bnd.size))
        cols = np.zeros((sd.free.size, bnd.size))
        cols[bnd, np.arange(bnd.size)] = 1.0
        F[:, keep] = o.kplus(sd, cols[:, keep])[bnd]
        B = sd.B[:, bnd]
        ops.append((B, np.abs(F), np.abs(sd.Y)))
        z = prob.coords[sd.nodes[sd.free[bnd] // 3], 2]
        rows, c = B.nonzero()
        height[rows] = z[c]
    return prob, o, ops, height / height.max()


VECTORS = {
    "random": lambda g, h: g,
    "falls by 1e-8": lambda g, h: g * 10.0 ** (-8 * h),
    "falls by 1e-16": lambda g, h: g * 10.0 ** (-16 * h),
    "falls by 1e-300": lambda g, h: g * 10.0 ** (-300 * h),
    "one entry": lambda g, h: np.where(np.arange(g.size) == g.size // 2, g, 0.0),
    "one component": lambda g, h: np.where(np.arange(g.size) % 3 == 0, g, 0.0),
    "subnormal": lambda g, h: g * 2.0 ** -1030,
    "almost subnormal": lambda g, h: g * 2.0 ** -1015,
}


@pytest.mark.parametrize("name", VECTORS)
def test_entries_match_the_rows(case, name):
    from paper_1508_02599_gb300 import FetiSolver
    prob, o, ops, height = case
    v = VECTORS[name](np.random.default_rng(5).normal(size=o.n_lambda), height)
    out = {}
    for sym in ("off", "force"):
        with FetiSolver(prob, method="af", precond="dirichlet", symmetric=sym) as s:
            s.prepare()
            assert (s.schedule()["fp64_F"][0] < -400) == (sym == "force")
            assert (s.schedule()["fp64_M"][0] < -400) == (sym == "force")
            d = torch.tensor(v, device="cuda")
            q, z = torch.empty_like(d), torch.empty_like(d)
            s.dual_apply(d, q, z, 1)
            torch.cuda.synchronize()
            out[sym] = q.cpu().numpy(), z.cpu().numpy()
    m = max(B.shape[1] for B, _, _ in ops)
    unit = (1.3 * m + 80) * 2.0 ** -48 + 2 * m * 2.0 ** -53
    tiny = 2 * m * 2.0 ** -1074                      # rounding of subnormal products and sums
    W = o.maps.weight
    dq = sum(abs(B) @ (F @ np.abs(B.T @ v)) for B, F, _ in ops) * unit + tiny
    assert (np.abs(out["force"][0] - out["off"][0]) <= dq).all()
    q = out["off"][0]
    dz = sum(W * (abs(B) @ (S @ (unit * np.abs(B.T @ (W * q)) + abs(B.T) @ (W * dq)))) for B, _, S in ops) + tiny
    assert (np.abs(out["force"][1] - out["off"][1]) <= dz).all()
