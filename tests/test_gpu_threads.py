"""Independent contexts in two threads, with subdomains of different sizes.

The fixed-point applies and the K^+ sweeps of the two contexts need different
amounts of shared memory (about 100 and 16 KB); each thread solves again and
again while the other does, and gets the bits that it gets alone.
"""
import threading

import pytest

torch = pytest.importorskip("torch")

from feti_inputs import mesh  # noqa: E402

pytestmark = pytest.mark.gpu

SOLVES = 40


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def test_two_contexts_of_different_sizes():
    from paper_1508_02599_gb300 import FetiSolver
    probs = [mesh.jittered_cylinder_problem(10, 44, 15, 17, 7, 8), mesh.cube_problem(6, (2, 2, 2))]
    alone, wrong = [], []
    for p in probs:
        with FetiSolver(p, method="af", symmetric="force") as s:
            alone.append(s.solve()[0].copy())
    start = threading.Barrier(len(probs))

    def work(k):
        try:
            with FetiSolver(probs[k], method="af", symmetric="force") as s:
                start.wait()
                for _ in range(SOLVES):
                    if not (s.solve()[0] == alone[k]).all():
                        wrong.append((k, "other bits"))
        except Exception as e:  # noqa: BLE001 - reported below, from the main thread
            wrong.append((k, repr(e)))
            start.abort()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(probs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong[:3]
