"""The batched elimination at the edges of its 64-column panels and 128 x 64 tiles.

One dual apply (q = F v, z = M^-1 q) against the oracle's dense LAPACK route,
on subdomains from a few DOFs (no interior, one partial panel) to several
tiles with remainders in both phases.  Tolerances: FP64 -- an update is exact
down to 2^-54 of its two row maxima, so about n of them leave
n 2^-54 < 1e-13 relative to the matrix, times the local condition number
(below 100 for these blocks): 1e-11.  FP32 -- 2^-24 rounding of the factor
amplified by the local condition of K_rr: 1e-3, as for any FP32
factorization of these operators.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from feti_inputs import mesh  # noqa: E402
from oracle import feti  # noqa: E402

pytestmark = pytest.mark.gpu

MESHES = {
    "18 nodes": lambda: mesh.cube_problem(2, (2, 1, 1)),
    "27 nodes": lambda: mesh.cube_problem(2, (1, 1, 1)),
    "64 nodes": lambda: mesh.cube_problem(3, (1, 1, 1)),
    "125 nodes": lambda: mesh.cube_problem(4, (1, 1, 1)),
    "343 nodes": lambda: mesh.cube_problem(6, (1, 1, 1)),
    "75 nodes": lambda: mesh.cube_problem(4, (2, 1, 1)),
    "uneven": lambda: mesh.jittered_cylinder_problem(6, 24, 12, 13, mesh_seed=7, part_seed=8),
}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("mixed_f32factor", 1e-3)])
@pytest.mark.parametrize("name", MESHES)
def test_operators_match_oracle(name, precision, tol):
    from paper_1508_02599_gb300 import FetiSolver
    prob = MESHES[name]()
    o = feti.FetiOracle(prob, "af", "dirichlet")
    o.assemble()
    o.factorize()
    v = np.random.default_rng(17).normal(size=o.n_lambda)
    q_ref = o.apply_F(v)
    z_ref = o.apply_prec(q_ref)
    with FetiSolver(prob, method="af", precond="dirichlet", precision=precision) as s:
        s.prepare()
        dv = torch.tensor(v, device="cuda", dtype=torch.float64)
        q, z = torch.empty_like(dv), torch.empty_like(dv)
        s.dual_apply(dv, q, z, 1)
        torch.cuda.synchronize()
    assert np.linalg.norm(q.cpu().numpy() - q_ref) <= tol * np.linalg.norm(q_ref)
    assert np.linalg.norm(z.cpu().numpy() - z_ref) <= tol * np.linalg.norm(z_ref)
