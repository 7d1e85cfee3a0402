"""Failures on the host side: allocations that fail in the middle of a plan or of the buffers that a first call makes,
factorisations that fail, and captured V-cycles when the kind of factors changes. The library's objects run against a CUDA runtime
whose memory is host memory and whose launches do nothing (fake_cudart.cpp), so no device is involved."""
import ctypes
import glob
import os
import subprocess

import numpy as np
import pytest

from paper_0707_4018_gb300 import binding, build

HERE = os.path.dirname(os.path.abspath(__file__))
FAILED = (2, 3)  # pinned host memory, device memory
NOT_CONVERGED, NAN, STATE = 4, 5, 7
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


def _at(a):
    return ctypes.c_void_p(a.ctypes.data)


class Ctx:
    def __init__(self, lib, max_rhs, dims=DIMS, **params):
        self.lib, self.p = lib, ctypes.c_void_p()
        p = binding.mg_params()
        lib.mg_default_params(ctypes.byref(p))
        p.block[0][0] = p.block[0][1] = 2
        p.Nv[0], p.n_pass, p.max_rhs, p.max_iter = 4, 1, max_rhs, 2
        for k, v in params.items():
            setattr(p, k, v)
        self.U = np.zeros((dims[0] * dims[1], 2), dtype=np.complex128)
        self.v = np.zeros((4, dims[0] * dims[1], 2), dtype=np.complex128)
        rc = lib.mg_setup(ctypes.byref(self.p), ctypes.byref(binding.make_geom(dims)), _at(self.U),
                          ctypes.c_double(0.1), ctypes.byref(p), None)
        assert rc == 0, lib.mg_last_error()

    def batch(self, *masses):
        m = (ctypes.c_double * len(masses))(*masses)
        return self.lib.mg_solve_batch(self.p, len(masses), _at(self.v), _at(self.v[2:]), m,
                                       ctypes.c_double(1e-10), None)

    def vcycle(self):
        return self.lib.mg_vcycle(self.p, _at(self.v), _at(self.v[2:]))

    def update_mass(self, m):
        return self.lib.mg_update_mass(self.p, ctypes.c_double(m))

    def close(self):
        self.lib.mg_destroy(self.p)


@pytest.fixture(autouse=True)
def _reset(lib):
    yield
    lib.fake_fail_at(0)
    lib.fake_factor(0, 0)


@pytest.mark.parametrize("reject", [0, 1])  # the cyclic reduction's plan, and the dense factors behind it too
@pytest.mark.parametrize("max_rhs", [1, 2])  # a limit of one: the buffers of batches are made by the first batch
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
        if rc in FAILED:
            failures += 1
            assert ctx.batch(*masses) in (0, NOT_CONVERGED), (nth, lib.mg_last_error())
        ctx.close()
        lib.fake_factor(0, 0)
        assert lib.fake_nulls() == 0, nth
        if rc not in FAILED:
            break
    assert failures >= 7  # mem, tmp, pinv, chk, berr, info and the job list of one slot at least


def test_a_failed_allocation_of_a_4d_batch_is_made_up_for(lib):
    dims = (4, 4, 4, 4)
    U, v = np.zeros((256, 4, 3, 3), dtype=np.complex128), np.zeros((4, 256, 4, 3), dtype=np.complex128)
    p = binding.mg_params()
    lib.mg_default_params(ctypes.byref(p))
    for i in range(4):
        p.block[0][i] = 2
    p.Nv[0], p.n_pass, p.nu_setup, p.chiral_split, p.max_iter, p.coarsest_max_iter = 2, 1, 1, 1, 2, 2
    nth, rc = 0, FAILED[0]
    while rc in FAILED:
        nth += 1
        ctx = ctypes.c_void_p()
        assert lib.mg_setup(ctypes.byref(ctx), ctypes.byref(binding.make_geom(dims, 3)), _at(U), ctypes.c_double(0.1),
                            ctypes.byref(p), None) == 0, lib.mg_last_error()
        solve = lambda: lib.mg_solve_batch(ctx, 1, _at(v), _at(v[2:]), None, ctypes.c_double(1e-10), None)
        lib.fake_fail_at(nth)
        rc = solve()
        lib.fake_fail_at(0)
        if rc in FAILED:
            assert solve() in (0, NOT_CONVERGED), (nth, lib.mg_last_error())
        lib.mg_destroy(ctx)
        assert lib.fake_nulls() == 0, nth
    assert nth > 20


def test_a_failed_growth_of_the_network_buffers_is_made_up_for(lib):
    dims, block = (8, 8), (ctypes.c_int * 2)(4, 4)
    U, tgt = np.zeros((2, 64, 2), dtype=np.complex128), np.zeros((2, 2, 64, 2), dtype=np.complex128)
    nth, rc = 0, FAILED[0]
    while rc in FAILED:
        nth += 1
        net = ctypes.c_void_p()
        assert lib.mg_nullnet_create(ctypes.byref(net), 2, 2, 2, ctypes.c_uint64(1)) == 0

        def gradient(fields):
            seeds = (ctypes.c_uint64 * fields)(*range(fields))
            loss = ctypes.c_double()
            return lib.mg_nullnet_gradient(net, ctypes.byref(binding.make_geom(dims)), fields, _at(U), seeds, _at(tgt),
                                           block, ctypes.byref(loss), None, None)
        assert gradient(1) == 0
        lib.fake_fail_at(nth)
        rc = gradient(2)
        lib.fake_fail_at(0)
        if rc in FAILED:
            assert gradient(1) == 0, (nth, lib.mg_last_error())
        lib.mg_nullnet_destroy(net)
        assert lib.fake_nulls() == 0, nth
    assert nth > 10


def test_a_failed_mass_update_does_not_leave_missing_factors_in_use(lib):
    ctx = Ctx(lib, 1)
    assert ctx.vcycle() == 0
    lib.fake_factor(1, 0)
    lib.fake_fail_at(1)  # the dense factors
    assert ctx.update_mass(0.2) in FAILED
    assert ctx.vcycle() == STATE
    assert ctx.update_mass(0.2) == 0 and ctx.vcycle() == 0
    lib.fake_factor(0, 0)
    assert ctx.update_mass(0.3) == 0 and ctx.vcycle() == 0
    assert lib.fake_nulls() == 0
    ctx.close()


def test_a_failed_factorisation_drops_captured_cycles_of_the_other_kind(lib):
    ctx = Ctx(lib, 2)
    assert ctx.batch(0.2, 0.3) == NOT_CONVERGED
    captured = lib.fake_graphs()
    assert ctx.batch(0.2, 0.3) == NOT_CONVERGED and lib.fake_graphs() == captured  # replayed
    lib.fake_factor(1, 1)
    assert ctx.batch(0.4, 0.3) == NAN
    lib.fake_factor(1, 0)
    assert ctx.batch(0.4, 0.3) == NOT_CONVERGED
    assert lib.fake_graphs() > captured  # the captured cycle held the reduction's launches
    ctx.close()


def test_a_failed_factorisation_is_not_taken_for_the_one_before(lib):
    ctx = Ctx(lib, 2)
    assert ctx.batch(0.2, 0.3) == NOT_CONVERGED
    lib.fake_factor(1, 1)
    assert ctx.batch(0.4, 0.3) == NAN
    lib.fake_factor(0, 0)
    checks = lib.fake_checks()
    assert ctx.batch(0.2, 0.3) == NOT_CONVERGED
    assert lib.fake_checks() == checks + 1  # the first slot's factors were overwritten, the second's were not
    ctx.close()


def test_a_ring_of_more_lines_than_a_grid_has_rows(lib):
    # a coarse lattice of 1 x 70000 sites: more lines, and products of them, than the second extent of a grid takes
    ctx = Ctx(lib, 1, dims=(2, 140000), nu_setup=1, nu_pre=1, nu_post=1, coarsest_lu_max=300000)
    assert ctx.vcycle() == 0
    ctx.close()
