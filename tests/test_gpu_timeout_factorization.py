"""The waits of the local factorizations that run out: FETI_ERR_TIMEOUT, then a usable context.

With a budget of one nanosecond the panel solve and the trailing update give up
waiting for their copies and tensor-core products at the first check, wait for
what they have in flight (a budget of its own), release tensor memory and flag
the set-up.  The operators are then not there; with the default budget the
solve sets them up and matches the FP64 oracle.  A zero budget is for the
pipelines of the solve and leaves the factorizations alone.
"""
import numpy as np
import pytest

from feti_inputs import mesh
from oracle import feti

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


@pytest.fixture(scope="module")
def case():
    prob = mesh.cylinder_problem(4, 16, 8, (2, 8, 2))
    return prob, feti.FetiOracle(prob, feti.ALL_FLOATING, "dirichlet").solve(tol=1e-12)[0]


@pytest.mark.parametrize("first", ["never set up", "set up before"])
@pytest.mark.parametrize("precision", ["fp64", "mixed_f32factor"])
def test_factorization_times_out_then_recovers(case, precision, first):
    from paper_1508_02599_gb300 import FetiError, FetiSolver
    prob, ref = case
    with FetiSolver(prob, method="af", precision=precision, tol=1e-10,
                    spin_timeout_ns=1 if first == "never set up" else 0) as s:
        if first == "set up before":
            s.set_spin_timeout(0)
            s.prepare()
            s.set_spin_timeout(1)
        with pytest.raises(FetiError) as ei:
            s.prepare()
        assert ei.value.status == 9 and "bounded wait" in str(ei.value)
        v = torch.ones(s.sizes()["n_lambda"], dtype=torch.float64, device="cuda")
        with pytest.raises(FetiError) as ei:
            s.dual_apply(v, torch.empty_like(v), torch.empty_like(v), 1)
        assert ei.value.status == 12
        s.set_spin_timeout(100_000_000)
        U, rep = s.solve()
    assert rep["converged"] == 1
    assert np.linalg.norm(U - ref) <= 1e-8 * np.linalg.norm(ref)
