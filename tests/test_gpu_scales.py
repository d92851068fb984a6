"""Linear problems in units near the ends of the FP64 range.

Young's modulus and the pressure times 2^k leave the displacement as it is.  At
k = 1010 the entries of F_i are near 2^-1010 and what the elimination subtracts from
them is partly subnormal; at k = -970 the entries of K_i are.  A number of 2^-1010
is rounded to 2^-64 of itself, one of 2^-970 to less, and PCG stops at 1e-10: 1e-10.
"""
import dataclasses
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from feti_inputs import mesh  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    prob = mesh.jittered_cylinder_problem(6, 24, 12, 13, 7, 8)
    return prob, _solve(prob, 0)


def _solve(prob, k):
    from paper_1508_02599_gb300 import FetiSolver
    p = dataclasses.replace(prob, material=dict(prob.material, E=math.ldexp(prob.material["E"], k)),
                            pressure=math.ldexp(prob.pressure, k))
    with FetiSolver(p, method="af", tol=1e-10) as s:
        U, rep = s.solve()
    return U, rep["iterations"]


@pytest.mark.parametrize("k", [-970, -900, 900, 1000, 1010])
def test_displacement_does_not_depend_on_the_unit(case, k):
    prob, (ref, its) = case
    U, n = _solve(prob, k)
    assert abs(n - its) <= 1
    assert np.linalg.norm(U - ref) <= 1e-10 * np.linalg.norm(ref)
