"""feti_elements on an inverted element: an error, and the caller's arrays as they were.

The two-fibre matrices of an array aligned to 32 bytes are written in place, the
others expanded from packed ones; both refuse the same elements.  One node is
moved towards and through the opposite faces of its elements, up to 1e-16 of the
way on either side of the first face it meets.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from feti_inputs import mesh  # noqa: E402

pytestmark = pytest.mark.gpu

STEPS = [0.0, 0.5, 0.99, 1 - 1e-4, 1 - 1e-8, 1 - 1e-12, 1 - 1e-15, 1 - 1e-16, 1.0, 1 + 4e-16, 1 + 1e-12, 1.01, 3.0, np.nan]


@pytest.fixture(scope="module")
def case():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    prob = mesh.cylinder_problem(2, 14, 3, (1, 2, 1), material=mesh.hgo_material(), pressure=0.1)
    node = int(prob.tets[100, 0])
    x = prob.coords
    way = np.array([1.0, 0.3, 0.2])                 # of the node
    first = np.inf                                  # where the first of its elements has no volume left
    for t in prob.tets:
        if node in t:
            a, b, c = x[[n for n in t if n != node]]
            nrm = np.cross(b - a, c - a)
            s = nrm @ (a - x[node]) / (nrm @ way)
            first = min(first, s) if s > 0 else first
    return prob, node, first * way


def _run(s, E, U, offset):
    flat = torch.full((E * 144 + 8,), 7.0, dtype=torch.float64, device="cuda")
    K, f = flat[offset:offset + E * 144].view(E, 12, 12), torch.full((E, 12), 7.0, dtype=torch.float64, device="cuda")
    from paper_1508_02599_gb300 import FetiError
    try:
        s.elements(torch.tensor(U.ravel(), device="cuda"), out=(K, f))
        status = 0
    except FetiError as e:
        status = e.status
    torch.cuda.synchronize()
    if status:
        assert status == 3 and (flat == 7.0).all() and (f == 7.0).all()
    return status


@pytest.mark.parametrize("scale", [1.0, 1e-12, 1e12])
def test_inverted_element_leaves_the_arrays(case, scale):
    import dataclasses
    from paper_1508_02599_gb300 import FetiSolver
    prob, node, way = case
    E = prob.tets.shape[0]
    with FetiSolver(dataclasses.replace(prob, coords=prob.coords * scale), method="classical") as s:
        seen = []
        for t in STEPS:
            U = np.zeros_like(prob.coords)
            U[node] = scale * t * way
            direct, packed = _run(s, E, U, 0), _run(s, E, U, 1)
            assert direct == packed
            seen.append(direct)
    assert seen[:4] == [0] * 4 and seen[-4:] == [3] * 4
