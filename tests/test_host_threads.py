"""Threads of the host eigensolvers (csrc/host_threads.h): bounded over all callers together, and
the eigenvectors the same bits however many are granted.  Plain C++, compiled with g++."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_06316_gb300", "csrc")

DRIVER = r"""
#include "host_threads.h"
#include "symeig.h"
extern "C" void *take(int want, int *got) {
  auto *t = new afmpb::HostThreads(want);
  *got = t->count();
  return t;
}
extern "C" void give(void *t) { delete (afmpb::HostThreads *)t; }
extern "C" int cores() { return (int)std::max(1u, std::thread::hardware_concurrency()); }
extern "C" int eig(int n, double *a, double *w, double *zt) { return afmpb::sym_eig_desc(n, a, w, zt); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_threads")
    (d / "driver.cpp").write_text(DRIVER)
    so = d / "libthreads.so"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-pthread", "-fPIC", "-shared", "-I", CSRC, str(d / "driver.cpp"),
                           "-x", "c++", os.path.join(CSRC, "symeig.cu"), "-o", str(so)])
    L = ctypes.CDLL(str(so))
    L.take.restype = ctypes.c_void_p
    L.give.argtypes = [ctypes.c_void_p]
    return L


def take(lib, want):
    got = ctypes.c_int()
    return lib.take(want, ctypes.byref(got)), got.value


def test_threads_are_granted_up_to_two_per_core_and_given_back(lib):
    limit = 2 * lib.cores()
    a, na = take(lib, 1)
    b, nb = take(lib, 10 ** 6)
    c, nc = take(lib, 3)
    assert (na, nb, nc) == (1, limit - 1, 0)
    lib.give(b)
    d, nd = take(lib, limit)
    assert nd == limit - 1
    for t in (a, c, d):
        lib.give(t)
    e, ne = take(lib, limit)
    lib.give(e)
    assert ne == limit


@pytest.mark.parametrize("n", [127, 128, 216])
def test_eigenvectors_without_a_thread_to_be_had(lib, n):
    rng = np.random.default_rng(n)
    a = rng.standard_normal((n, n))
    a = a + a.T
    p = lambda v: v.ctypes.data_as(ctypes.c_void_p)
    out = []
    for want in (0, 10 ** 6):                       # all threads free, none free
        t, _ = take(lib, want)
        keep, w, zt = a.copy(), np.zeros(n), np.zeros((n, n))
        assert lib.eig(n, p(keep), p(w), p(zt)) == 0
        lib.give(t)
        out.append((w, zt))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
