"""A context whose device arrays could not all be made must not be used: every call of bind_qps and macro_create that
can fail is made to fail in turn, after a successful one of another size, and the solves that follow have to be refused
(with the arrays half replaced, their kernels would read and write out of range).  The library's host code on the CPU:
its objects linked to a stand-in for the CUDA runtime (fake_cudart.cpp) that runs no kernel."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1908_08292_gb300 import _SIGS, Options, build

STATE, CUDA, OOM = -4, -2, -3
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def L(tmp_path_factory):
    objs = [os.path.join(build.BUILD, os.path.splitext(s)[0] + ".o") for s in build.SOURCES]
    build.build(force=not all(map(os.path.exists, objs)))
    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I" + inc, "-Wl,-Bsymbolic", "-o", so,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs], check=True)
    lib = ctypes.CDLL(so)
    for name, (res, args) in _SIGS.items():
        getattr(lib, name).restype, getattr(lib, name).argtypes = res, args
    return lib


def context(L, dim, precision, sizes):
    opt, h = Options(), ctypes.c_void_p()
    assert L.fehmm_default_options(ctypes.byref(opt), dim, precision) == 0
    assert L.fehmm_create(ctypes.byref(h), ctypes.byref(opt)) == 0
    grid = np.array(sizes, dtype=np.int32)
    phase = np.zeros(sum(n ** dim for n in sizes), dtype=np.uint8)
    E, nu, first = np.ones(len(sizes)), np.full(len(sizes), 0.3), ctypes.c_int()
    assert L.fehmm_add_rves(h, len(sizes), grid.ctypes.data, phase.ctypes.data, E.ctypes.data, nu.ctypes.data, 1,
                            ctypes.byref(first)) == 0
    return h


@pytest.mark.parametrize("dim,precision", [(2, 0), (2, 1), (3, 1)])
def test_bind_qps(L, dim, precision):
    before = L.fake_blocks()
    h = context(L, dim, precision, [2, 4, 6])
    some, more = np.array([0, 1, 0], dtype=np.int32), np.array([2, 0, 1, 2, 2, 1, 0, 2], dtype=np.int32)
    p = ctypes.c_void_p(16)  # never dereferenced: no kernel runs
    solve = lambda: L.fehmm_rve_solve(h, p, p, p, None, p, None, 0, None)  # noqa: E731
    bind = lambda q: L.fehmm_bind_qps(h, q.size, q.ctypes.data)  # noqa: E731
    assert solve() == STATE
    for k in range(1, 1000):
        assert bind(some) == 0 and solve() == 0
        L.fake_fail(k)
        rc = bind(more)
        if rc == 0:
            break
        assert rc in (CUDA, OOM)
        assert solve() == STATE, k
        assert L.fehmm_commit(h, None) == STATE and L.fehmm_rollback(h, None) == STATE
        L.fake_fail(0)
        assert bind(more) == 0 and solve() == 0  # usable again
    assert k > 10
    L.fake_fail(0)
    bad = np.array([0, 9], dtype=np.int32)  # refused before anything is touched: the binding stays
    assert bind(bad) == -1 and solve() == 0
    assert L.fehmm_destroy(h) == 0 and L.fake_blocks() == before


@pytest.mark.parametrize("n_el", [(3, 2), (9, 9), (3, 2, 1), (6, 6, 6)])  # one block, several
def test_macro_create(L, n_el):
    before = L.fake_blocks()
    h = context(L, len(n_el), 0, [2])
    small, big = np.ones(3, dtype=np.int32), np.array(n_el, dtype=np.int32)
    p = ctypes.c_void_p(16)
    calls = [lambda: L.fehmm_macro_solve(h, p, p, p, p, 1e-10, 10, None), lambda: L.fehmm_macro_qp_F(h, p, p, None),
             lambda: L.fehmm_macro_set_dirichlet(h, 0, None, None), lambda: L.fehmm_macro_update(h, p, p, None)]
    for k in range(1, 1000):
        assert L.fehmm_macro_create(h, small.ctypes.data) == 0 and all(c() == 0 for c in calls)
        L.fake_fail(k)
        rc = L.fehmm_macro_create(h, big.ctypes.data)
        if rc == 0:
            break
        assert rc in (CUDA, OOM)
        assert all(c() == STATE for c in calls), k
        L.fake_fail(0)
        assert L.fehmm_macro_create(h, big.ctypes.data) == 0 and all(c() == 0 for c in calls)
    assert k > 10
    L.fake_fail(0)
    bad = np.zeros(3, dtype=np.int32)
    assert L.fehmm_macro_create(h, bad.ctypes.data) == -1 and all(c() == 0 for c in calls)
    assert L.fehmm_destroy(h) == 0 and L.fake_blocks() == before
