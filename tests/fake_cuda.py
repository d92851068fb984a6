"""libfeti's host driver on a CUDA runtime without a device.

build() compiles the driver's C++ sources with fake_cudart.cpp (device memory
is host memory, launches do nothing) into a library with the C ABI of
libfeti.so; `solver` makes contexts on it.  For the paths that only a failing
runtime call reaches: nothing computed here means anything.
"""
import contextlib
import ctypes as C
import os
import shutil
import subprocess

from paper_1508_02599_gb300 import _lib, api

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_1508_02599_gb300", "csrc")
SOURCES = ["feti_host.cpp", "feti_coarse_plan.cpp", "feti_checkpoint.cpp"]


def cuda_include():
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")


def build(folder):
    """The library's path; every undefined launcher returns zero, the local products ask the fake."""
    inc = ["-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I", cuda_include(),
           "-I", "/usr/local/cuda/include"]
    jobs, objs = [], []
    for src in [os.path.join(CSRC, s) for s in SOURCES] + [os.path.join(HERE, "fake_cudart.cpp")]:
        objs.append(os.path.join(folder, os.path.basename(src) + ".o"))
        jobs.append(subprocess.Popen(["g++", "-std=c++17", "-O1", "-fPIC", "-c", src, "-o", objs[-1], *inc]))
    assert not any(j.wait() for j in jobs)

    def names(flag):
        out = subprocess.run(["nm", flag, *objs], check=True, capture_output=True, text=True).stdout
        return {line.split()[-1] for line in out.splitlines() if line.split() and "4feti" in line}

    stub = os.path.join(folder, "stubs.c")
    with open(stub, "w") as f:
        fakes = {"launch_symv_fixed": "fixed", "launch_gemv_loc": "rows", "launch_gemm_loc": "block"}
        f.write("".join(f"long fake_{v}_launch(void);\n" for v in fakes.values()))
        for k, name in enumerate(sorted(names("--undefined-only") - names("--defined-only"))):
            body = next((f"fake_{v}_launch()" for n, v in fakes.items() if n in name), "0")
            f.write(f'long stub{k}(void) __asm__("{name}");\nlong stub{k}(void) {{ return {body}; }}\n')
    lib = os.path.join(folder, "libfeti_fake.so")
    subprocess.run(["gcc", "-fPIC", "-O1", "-c", stub, "-o", stub + ".o"], check=True)
    subprocess.run(["g++", "-shared", "-Wl,--no-undefined,-Bsymbolic", "-o", lib, *objs, stub + ".o", "-pthread"], check=True)
    return lib


def load(path):
    """The library bound like the real one."""
    real, _lib._lib = _lib._lib, None
    try:
        lib = _lib.load(path)
    finally:
        _lib._lib = real
    lib.fake_live_bytes.restype = lib.fake_peak_bytes.restype = C.c_size_t
    lib.fake_capacity.argtypes = [C.c_size_t]
    lib.fake_cost.argtypes = [C.c_float] * 3
    return lib


@contextlib.contextmanager
def solver(lib, monkeypatch, prob, **opt):
    monkeypatch.setattr(_lib, "_lib", lib)
    lib.fake_reset()
    with api.FetiSolver(prob, **opt) as s:
        yield s


def dual_apply(lib, s, v, q, z, nrhs=1):
    """feti_dual_apply or feti_dual_apply_multi on host arrays, which are device arrays here."""
    a = [C.c_void_p(x.ctypes.data) for x in (v, q, z)]
    if nrhs == 1:
        s._check(lib.feti_dual_apply(s._ctx, *a, 1, None))
    else:
        s._check(lib.feti_dual_apply_multi(s._ctx, *a, nrhs, 1, None))
