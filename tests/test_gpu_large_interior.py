"""Subdomains whose interior vector fills most of a CTA's shared memory.

The backward sweep of K^+ holds the interior vector once where five of them do
not fit: 17,457 interior DOFs are 140 KB in FP64 (twice that does not fit
either) and 70 KB in FP32.  The displacement against conjugate gradients on the
assembled matrix, refined down to the rounding of its residual (1e-16 times the
condition number, about 1e4).  Tolerance: PCG stops at 1e-12 relative, times that
condition number: 1e-8.
"""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

torch = pytest.importorskip("torch")

from feti_inputs import mesh  # noqa: E402
from oracle import fem  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


@pytest.fixture(scope="module")
def case():
    prob = mesh.cube_problem(22, (2, 1, 1))
    Ke, _ = fem.element_matrices(prob)
    K = fem.assemble_global(prob, Ke)
    free = np.setdiff1d(np.arange(K.shape[0]), prob.dir_dof)     # clamped to zero
    A, b = K[free][:, free], fem.load_vector(prob)[free]
    inv_diag = 1.0 / A.diagonal()
    M = spla.LinearOperator(A.shape, lambda v: inv_diag * v)
    x = np.zeros_like(b)
    for _ in range(3):
        x += spla.cg(A, b - A @ x, rtol=1e-10, maxiter=5000, M=M)[0]
    assert np.linalg.norm(b - A @ x) <= 1e-11 * np.linalg.norm(b)
    ref = np.zeros(K.shape[0])
    ref[free] = x
    return prob, ref


@pytest.mark.parametrize("precision", ["fp64", "mixed_f32factor"])
def test_displacement(case, precision):
    from paper_1508_02599_gb300 import FetiSolver
    prob, ref = case
    with FetiSolver(prob, method="classical", precision=precision, tol=1e-12) as s:
        U, rep = s.solve()
    assert rep["converged"] == 1
    assert np.linalg.norm(U - ref) <= 1e-8 * np.linalg.norm(ref)
