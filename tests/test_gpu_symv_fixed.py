"""FP64 local applies from the fixed-point panels against the FP64 rows.

symmetric="force" applies F_i and S_i from their 56-bit fixed-point lower block
triangles, "off" from the full FP64 rows.  Both round: the rows in a sum of n
FP64 terms (n <= 1400 here: below n 2^-53 = 1.6e-13 of |M| |v|), the fixed-point
form in its operands (2^-57 of the row's and the vector's largest entries) --
1e-12 between the two.  Sizes around the 16-row panels, 64-column tiles and
the split over CTAs; a scaled vector gives the scaled result bit for bit; an
infinite entry or a NaN is not lost.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from feti_inputs import mesh  # noqa: E402

pytestmark = pytest.mark.gpu

MESHES = {
    "18 nodes": lambda: mesh.cube_problem(2, (2, 1, 1)),
    "27 nodes": lambda: mesh.cube_problem(2, (1, 1, 1)),
    "cube8": lambda: mesh.cube_problem(8, (2, 2, 2)),
    "uneven": lambda: mesh.jittered_cylinder_problem(8, 32, 16, 9, 77, 78),
    "many": lambda: mesh.jittered_cylinder_problem(8, 48, 32, 160, 77, 78),
}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _apply(s, v):
    q, z = torch.empty_like(v), torch.empty_like(v)
    s.dual_apply(v, q, z, 1)
    torch.cuda.synchronize()
    return q, z


@pytest.mark.parametrize("name", MESHES)
def test_fixed_point_apply_matches_rows(name):
    from paper_1508_02599_gb300 import FetiSolver
    prob = MESHES[name]()
    out, lost = {}, {}
    for sym in ("off", "force"):
        with FetiSolver(prob, method="af", precond="dirichlet", symmetric=sym) as s:
            s.prepare()
            assert (s.schedule()["fp64_F"][0] < -400) == (sym == "force"), s.schedule()
            n = s.sizes()["n_lambda"]
            v = torch.tensor(np.random.default_rng(23).normal(size=n), device="cuda")
            out[sym] = _apply(s, v)
            if sym == "force":
                q, z = _apply(s, v * 2.0 ** 300)
                assert torch.equal(q, out[sym][0] * 2.0 ** 300) and torch.equal(z, out[sym][1] * 2.0 ** 300)
                q, z = _apply(s, torch.zeros_like(v))
                assert not q.any() and not z.any()
            lost[sym] = []
            for bad in (float("nan"), float("inf")):
                w = v.clone()
                w[n // 3::n // 3] = bad
                lost[sym] += [torch.isfinite(x) for x in _apply(s, w)]
    assert all(torch.equal(a, b) for a, b in zip(*lost.values()))   # the same entries, whichever form
    for a, b in zip(*out.values()):
        assert float(torch.linalg.norm(a - b)) <= 1e-12 * float(torch.linalg.norm(a))
