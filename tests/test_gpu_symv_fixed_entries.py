"""The fixed-point apply of one matrix, entry by entry, against extended precision.

Matrices like a local Schur complement: couplings that fall with the distance of
their rows, between rows of one size and of sizes 1e-6 to 1e6.  Bound, relative to
|M| |v|: (1.3 m + 80) 2^-48 for a row that the copy serves and m 2^-53 for one
summed in FP64; the larger one holds for all.  A vector that falls by 1e-8 or
1e-16 exceeds it by far where every row is served by the copy.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def apply(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1508_02599_gb300 import build, library_path
    so = str(tmp_path_factory.mktemp("probe") / "probe.so")
    subprocess.run([build.nvcc(), "-shared", "-Xcompiler", "-fPIC", "-std=c++17", *build.ARCH, "-I", build.CSRC,
                    "-I", build.INCLUDE, os.path.join(HERE, "symv_fixed_probe.cu"), library_path(), "-o", so,
                    "-lcudart", "-Xlinker", "-rpath=" + os.path.dirname(library_path())], check=True)
    probe = C.CDLL(so).symv_fixed_probe

    def run(M, v, ctas):
        y = np.empty_like(v)
        a = [x.ctypes.data_as(C.POINTER(C.c_double)) for x in (M, v, y)]
        assert probe(v.size, ctas, *a) == 0
        return y
    return run


def _matrix(m, sizes):
    i = np.arange(m)
    x = np.random.default_rng(3).uniform(0.9, 1.1, size=(m, m))
    M = np.exp(-np.abs(i[:, None] - i[None, :]) / 12.0) * (x + x.T) / 2 * np.where((i[:, None] + i[None, :]) % 3, -1, 1)
    np.fill_diagonal(M, 1.5)
    d = np.ones(m) if sizes == "one size" else 10.0 ** np.random.default_rng(4).uniform(-6, 6, size=m)
    return np.ascontiguousarray(M * d[:, None] * d[None, :]), d


VECTORS = {
    "random": lambda g, s: g,
    "falls by 1e-8": lambda g, s: g * 10.0 ** (-8 * s),
    "falls by 1e-16": lambda g, s: g * 10.0 ** (-16 * s),
    "falls by 1e-300": lambda g, s: g * 10.0 ** (-300 * s),
    "first entry": lambda g, s: np.where(s == 0, g, 0.0),
    "every third": lambda g, s: np.where(np.arange(g.size) % 3 == 0, g, 0.0),
    "subnormal": lambda g, s: g * 2.0 ** -1030,
    "zero": lambda g, s: 0.0 * g,
}


@pytest.mark.parametrize("sizes", ["one size", "1e-6 to 1e6"])
@pytest.mark.parametrize("m,ctas", [(1, 1), (17, 1), (64, 2), (330, 4), (858, 1), (1605, 8)])
def test_entries(apply, m, ctas, sizes):
    M, d = _matrix(m, sizes)
    g = np.random.default_rng(5).normal(size=m) / d
    s = np.arange(m) / max(m - 1, 1)
    wide = np.longdouble
    tol = max((1.3 * m + 80) * 2.0 ** -48, m * 2.0 ** -53)
    for name, f in VECTORS.items():
        v = f(g, s)
        y = apply(M, v, ctas)
        prod = M.astype(wide) * v.astype(wide)[None, :]
        bound = tol * np.abs(prod).sum(axis=1) + m * wide(2.0) ** -1074
        assert (np.abs(y - prod.sum(axis=1)) <= bound).all(), name


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_entries_that_are_not_finite(apply, bad):
    M, d = _matrix(330, "one size")
    v = np.random.default_rng(5).normal(size=330)
    v[7] = bad
    with np.errstate(all="ignore"):
        want = M @ v
    y = apply(M, v, 2)
    assert (np.isnan(y) == np.isnan(want)).all() and (y[~np.isnan(want)] == want[~np.isnan(want)]).all()
    v[7] = 1.0
    M[3, 9] = M[9, 3] = bad
    y = apply(M, v, 2)
    assert (np.isfinite(y) == np.isfinite(M @ v)).all()
