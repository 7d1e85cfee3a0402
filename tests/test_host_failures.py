"""Failures on the host side of the exact coarsest solve: allocations that fail in the middle of a plan. The library's objects run against a CUDA runtime
whose memory is host memory and whose launches do nothing (fake_cudart.cpp), so no device is involved."""
import ctypes
import glob
import os
import subprocess

import numpy as np
import pytest

from paper_0707_4018_gb300 import binding, build

HERE = os.path.dirname(os.path.abspath(__file__))
OOM, NOT_CONVERGED = 3, 4
DIMS = (16, 12)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    build.build()
    objs = [os.path.join(build.BUILD, os.path.basename(s) + ".o") for s in build.sources()]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    out = str(tmp_path_factory.mktemp("fake") / "libmg_fake.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I" + inc, "-Wl,-Bsymbolic", "-o", out,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs], check=True)
    so = ctypes.CDLL(out)
    so.fake_fail_at.argtypes = [ctypes.c_long]
    so.mg_last_error.restype = ctypes.c_char_p
    return so


class Ctx:
    def __init__(self, lib, max_rhs):
        self.lib, self.p = lib, ctypes.c_void_p()
        p = binding.mg_params()
        lib.mg_default_params(ctypes.byref(p))
        p.block[0][0] = p.block[0][1] = 2
        p.Nv[0], p.n_pass, p.max_rhs, p.max_iter = 4, 1, max_rhs, 2
        self.U = np.zeros((DIMS[0] * DIMS[1], 2), dtype=np.complex128)
        self.v = np.zeros((4, DIMS[0] * DIMS[1], 2), dtype=np.complex128)
        rc = lib.mg_setup(ctypes.byref(self.p), ctypes.byref(binding.make_geom(DIMS)), self._at(self.U),
                          ctypes.c_double(0.1), ctypes.byref(p), None)
        assert rc == 0, lib.mg_last_error()

    @staticmethod
    def _at(a):
        return ctypes.c_void_p(a.ctypes.data)

    def batch(self, *masses):
        m = (ctypes.c_double * len(masses))(*masses)
        return self.lib.mg_solve_batch(self.p, len(masses), self._at(self.v), self._at(self.v[2:]), m,
                                       ctypes.c_double(1e-10), None)

    def close(self):
        self.lib.mg_destroy(self.p)


@pytest.fixture(autouse=True)
def _reset(lib):
    yield
    lib.fake_fail_at(0)
    lib.fake_factor(0, 0)


@pytest.mark.parametrize("reject", [0, 1])  # the cyclic reduction's plan, and the dense factors behind it too
@pytest.mark.parametrize("max_rhs", [2])
def test_a_failed_allocation_leaves_nothing_half_made(lib, max_rhs, reject):
    nth, failures = 0, 0
    while True:
        nth += 1
        ctx = Ctx(lib, max_rhs)
        lib.fake_factor(reject, 0)
        masses = [0.2, 0.3][:max_rhs]
        lib.fake_fail_at(nth)
        rc = ctx.batch(*masses)
        lib.fake_fail_at(0)
        if rc == OOM:
            failures += 1
            assert ctx.batch(*masses) in (0, NOT_CONVERGED), (nth, lib.mg_last_error())
        ctx.close()
        lib.fake_factor(0, 0)
        assert lib.fake_nulls() == 0, nth
        if rc != OOM:
            break
    assert failures >= 7  # mem, tmp, pinv, chk, berr, info and the job list of one slot at least
