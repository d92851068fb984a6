"""The projection with one chunk per subdomain (more than 304 of them, several
positions per thread) and with chunks of 256 positions, single-vector kernels
against those of the block iteration.

Both solve to a relative dual residual of 1e-10; with the Dirichlet
preconditioner the condition number is below 1e3, so the displacements agree to
1e-7 of the largest, here bounded by 1e-6.
"""
import numpy as np
import pytest

from feti_inputs import mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells,parts", [((8, 160, 16), (2, 40, 4)),    # 320 chunks of 282..294 positions
                                         ((3, 30, 3), (1, 10, 1))])     # 10 subdomains, chunks of 256
def test_projection_chunks(cells, parts):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1508_02599_gb300 import FetiSolver
    prob = mesh.cylinder_problem(*cells, parts, pressure=0.1)
    with FetiSolver(prob, method="af", precond="dirichlet", tol=1e-10, maxit=2000) as s:
        u, _ = s.solve()
        v, _ = s.solve_multi(np.array([1.0, 2.0]))
    scale = np.abs(u).max()
    assert scale > 0
    assert np.abs(v[0] - u).max() <= 1e-6 * scale
    assert np.abs(v[1] - 2 * u).max() <= 2e-6 * scale
