"""Two-fibre element matrices for a device array: written in place where the
array is aligned to 32 bytes, expanded from the packed form where it is not.

Both forms evaluate the same expressions, so they agree to rounding: 1e-14 of
the element's largest entry (45 units in the last place).  The element counts
leave a partial last block of threads.
"""
import numpy as np
import pytest

from feti_inputs import mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells", [(1, 6, 1), (2, 14, 3)])
@pytest.mark.parametrize("offset", [0, 1, 2, 4])
def test_direct_and_expanded_matrices_agree(cells, offset):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1508_02599_gb300 import FetiSolver
    prob = mesh.cylinder_problem(*cells, (1, 2, 1), material=mesh.hgo_material(), pressure=0.1)
    E = prob.tets.shape[0]
    U = 0.05 * prob.coords * np.array([1.0, 1.0, 0.0]) + 1e-3 * np.random.default_rng(5).normal(size=prob.coords.shape)
    flat = torch.full((E * 144 + 8,), 7.0, dtype=torch.float64, device="cuda")
    Kd = flat[offset:offset + E * 144].view(E, 12, 12)
    fd = torch.empty((E, 12), dtype=torch.float64, device="cuda")
    with FetiSolver(prob, method="classical") as s:
        Kh, fh = s.elements(U)
        s.elements(torch.tensor(U.ravel(), device="cuda"), out=(Kd, fd))
    scale = np.abs(Kh).reshape(E, -1).max(axis=1)[:, None, None]
    K = Kd.cpu().numpy()
    assert (np.abs(K - Kh) <= 1e-14 * scale).all()
    assert (K == K.transpose(0, 2, 1)).all()
    assert (np.abs(fd.cpu().numpy() - fh) <= 1e-14 * np.abs(fh).max()).all()
    rest = torch.cat([flat[:offset], flat[offset + E * 144:]])
    assert (rest == 7.0).all()
