"""Failing runtime calls in the host driver, on a runtime without a device.

The launches do nothing here, so only statuses, graphs and allocations are
looked at.
"""
import numpy as np
import pytest

import fake_cuda
from feti_inputs import mesh
from paper_1508_02599_gb300 import FetiError

OOM, CUDA = 10, 11                      # statuses
GRAPHS, FIXED = 0, 2                    # counters of the fake


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fake_cuda.load(fake_cuda.build(str(tmp_path_factory.mktemp("fake_cuda"))))


def _prob():
    return mesh.cube_problem(4, (2, 2, 2))


@pytest.mark.parametrize("call", ["solve", "solve_multi", "dual_apply", "dual_apply_multi"])
def test_refused_launch_in_a_capture_leaves_no_graph(lib, monkeypatch, call):
    with fake_cuda.solver(lib, monkeypatch, _prob(), method="af", symmetric="force", maxit=20) as s:
        s.prepare()
        n = s.sizes()["n_lambda"]
        v, q, z = (np.zeros((n, 2)) for _ in range(3))
        run = {"solve": s.solve, "solve_multi": lambda: s.solve_multi([1.0, 2.0]),
               "dual_apply": lambda: fake_cuda.dual_apply(lib, s, v, q, z),
               "dual_apply_multi": lambda: fake_cuda.dual_apply(lib, s, v, q, z, 2)}[call]
        lib.fake_refuse_in_capture(1)
        launched, graphs = lib.fake_count(FIXED), lib.fake_count(GRAPHS)
        with pytest.raises(FetiError) as ei:
            run()
        assert ei.value.status == CUDA and "launch in a captured graph" in str(ei.value)
        assert lib.fake_count(FIXED) > launched and lib.fake_count(GRAPHS) == graphs
        lib.fake_refuse_in_capture(0)
        run()                            # captured anew, not replayed
        assert lib.fake_count(GRAPHS) > graphs


def _prepared_bytes(lib, monkeypatch, symmetric, **opt):
    with fake_cuda.solver(lib, monkeypatch, _prob(), method="af", symmetric=symmetric, maxit=20, **opt) as s:
        s.prepare()
        return lib.fake_live_bytes()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_fixed_point_copies_the_tuner_rejects_are_given_back(lib, monkeypatch, precision):
    """Every launch takes as long here: the rows are kept."""
    rows = _prepared_bytes(lib, monkeypatch, "off", precision=precision)
    with fake_cuda.solver(lib, monkeypatch, _prob(), method="af", precision=precision, maxit=20) as s:
        s.prepare()
        assert s.schedule()["fp64_F"][0] > 0
        auto = lib.fake_live_bytes()
    if precision == "fp64":                # the FP32 forms have further copies beside the full rows
        assert auto == rows
        assert _prepared_bytes(lib, monkeypatch, "force") > rows
    assert _prepared_bytes(lib, monkeypatch, "auto", precision=precision) == auto   # the remembered pick


@pytest.mark.parametrize("symmetric", ["auto", "force"])
def test_memory_for_the_rows_alone_suffices(lib, monkeypatch, symmetric):
    _prepared_bytes(lib, monkeypatch, "off", workspace_mb=1)
    need = lib.fake_peak_bytes()
    with fake_cuda.solver(lib, monkeypatch, _prob(), method="af", symmetric=symmetric, workspace_mb=1,
                          maxit=20) as s:
        lib.fake_capacity(need)
        s.prepare()
        assert s.schedule()["fp64_F"][0] > 0 and s.schedule()["fp64_M"][0] > 0
        launched = lib.fake_count(FIXED)
        s.solve()
        assert lib.fake_count(FIXED) == launched


def test_later_allocations_come_before_the_copies(lib, monkeypatch):
    with fake_cuda.solver(lib, monkeypatch, _prob(), method="af", symmetric="force", maxit=20) as s:
        s.solve()
        assert s.schedule()["fp64_F"][0] < -400
        lib.fake_capacity(lib.fake_live_bytes())
        launched, graphs = lib.fake_count(FIXED), lib.fake_count(GRAPHS)
        s.solve_multi([1.0, 2.0])          # its vectors fit where the copies were
        assert s.schedule()["fp64_F"][0] > 0
        s.solve()                          # not from the graph that names the copies
        assert lib.fake_count(GRAPHS) >= graphs + 2
        after = lib.fake_count(FIXED)
        s.solve()
        assert lib.fake_count(FIXED) == after and after >= launched


def test_set_up_that_ran_out_of_memory_is_completed_by_the_next(lib, monkeypatch):
    """No kernel gets an array that the failed set-up did not reach."""
    full = _prepared_bytes(lib, monkeypatch, "off")
    with fake_cuda.solver(lib, monkeypatch, _prob(), method="af", symmetric="off", maxit=20) as s:
        base = lib.fake_live_bytes()
        for part in (0.2, 0.5, 0.8):
            lib.fake_capacity(int(base + part * (full - base)))
            with pytest.raises(FetiError) as ei:
                s.prepare()
            assert ei.value.status == OOM
        lib.fake_capacity(2 ** 62)
        s.prepare()
        assert lib.fake_live_bytes() == full


@pytest.mark.parametrize("symmetric,block,columns", [("auto", 3.0, False), ("auto", 6.0, True), ("force", 3.0, True)])
def test_block_products_take_the_faster_form(lib, monkeypatch, symmetric, block, columns):
    """Two columns of cost 2 through the fixed-point copy, or one block launch."""
    prob = mesh.cube_problem(4, (2, 2, 1))                      # the picks of _prob() are known by now
    with fake_cuda.solver(lib, monkeypatch, prob, method="af", symmetric=symmetric, maxit=20) as s:
        lib.fake_cost(2.0, 9.0, block)
        s.prepare()
        assert s.schedule()["fp64_M"][0] <= -400               # the tuner's pick for one vector
        v, q, z = (np.zeros((s.sizes()["n_lambda"], 2)) for _ in range(3))
        fake_cuda.dual_apply(lib, s, v, q, z, 2)               # tunes the block form
        launched = lib.fake_count(FIXED)
        fake_cuda.dual_apply(lib, s, v, z, q, 2)               # captured anew: F v as a block, then the preconditioner
        assert lib.fake_count(FIXED) - launched == (2 if columns else 0)


def test_bytes_of_an_apply_are_those_stored(lib, monkeypatch):
    """An entry takes 8 bytes in the FP64 rows and in the fixed-point copy."""
    moved = []
    for symmetric in ("off", "force"):
        with fake_cuda.solver(lib, monkeypatch, _prob(), method="af", symmetric=symmetric, maxit=20) as s:
            s.prepare()
            n = s.sizes()["n_lambda"]
            fake_cuda.dual_apply(lib, s, *(np.zeros(n) for _ in range(3)))
            moved.append(s.kernel_stats()["gemv_bytes"])
    assert moved[0] == moved[1] > 0
