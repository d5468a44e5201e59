"""Single cells of the auxiliary grid, built on the CPU from the library's own
headers (tests/grid_host.cpp), against the oracle: factors whose Gaussian parts
are much tighter than the exponents of a basis, decaying and growing long
ranges, orders up to 14, and what the library's check of a cell accepts."""
import ctypes
import os
import shutil
import subprocess
from concurrent.futures import ThreadPoolExecutor
from math import factorial

import numpy as np
import pytest

from oracle import oracle as O

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1412_5070_gb300", "csrc")
SRC = [os.path.join(HERE, "grid_host.cpp"), os.path.join(CSRC, "termlist.cpp")]
DEPS = SRC + [os.path.join(CSRC, f) for f in ("aux.cuh", "auxtab.h", "auxgrid.cuh", "gridtab.h", "termlist.h")]
LIB = os.path.join(HERE, "_build", "libgridhost.so")
dp = ctypes.POINTER(ctypes.c_double)


@pytest.fixture(scope="module")
def lib():
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    os.makedirs(os.path.dirname(LIB), exist_ok=True)
    if not os.path.exists(LIB) or any(os.path.getmtime(d) > os.path.getmtime(LIB) for d in DEPS):
        tmp = LIB + ".tmp%d" % os.getpid()
        subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-pthread", "-o", tmp,
                        *SRC], check=True)
        os.replace(tmp, LIB)
    L = ctypes.CDLL(LIB)
    L.grid_host_new.argtypes = [dp, ctypes.c_int, dp, ctypes.c_int, ctypes.c_int]
    L.grid_host_new.restype = ctypes.c_void_p
    L.grid_host_free.argtypes = [ctypes.c_void_p]
    L.grid_host_ok.argtypes = [ctypes.c_void_p, ctypes.c_double, ctypes.c_double]
    L.grid_host_eval.argtypes = [ctypes.c_void_p, ctypes.c_double, ctypes.c_double, ctypes.c_int, dp]
    return L


def rs12(mu=1.0, B=0.5, c0=0.5, rho=-0.5, n=0):
    """The terms of (1 + r/2) e^{-mu r^2} + c0 r^rho e^{Br} (1 - e^{-mu r^2} sum_k (mu r^2)^k/k!)."""
    return ([(1.0, 0, 0, mu), (0.5, 1, 0, mu), (c0, rho, B, 0)]
            + [(-c0 * mu ** k / factorial(k), rho + 2 * k, B, mu) for k in range(n + 1)])


class Grid:
    def __init__(self, lib, terms, cls):
        t = np.ascontiguousarray(terms, dtype=np.float64)
        self.lib, self.p = lib, lib.grid_host_new(t.ctypes.data_as(dp), len(t), t.ctypes.data_as(dp), len(t), cls)
        if not self.p:
            pytest.skip("not served by the grid")

    def __del__(self):
        if getattr(self, "p", None):
            self.lib.grid_host_free(self.p)

    def ok(self, xi, D):
        return self.lib.grid_host_ok(self.p, xi, D)

    def eval(self, xi, D, L):
        out = np.zeros(L + 1)
        assert self.lib.grid_host_eval(self.p, xi, D, L, out.ctypes.data_as(dp)) == 0
        return out


def reference(kern, cls, pts):
    with ThreadPoolExecutor(max_workers=min(16, os.cpu_count() or 1)) as ex:
        return np.array(list(ex.map(lambda p: O.radial(kern, cls, p[0], p[1], 15), pts)))


def errors(grid, ref, pts, L):
    """Relative error of every order at every point; an order that passes
    through zero is measured against a twentieth of the next over the local
    width, as in the GPU test of the grid."""
    got = np.array([grid.eval(x, d, L) for x, d in pts])
    w = np.array([min(d * d + 1e-300, 1.0 / x) for x, d in pts])
    return np.abs(got - ref[:, :L + 1]) / (np.abs(ref[:, :L + 1]) + 0.05 * np.abs(ref[:, 1:L + 2]) * w[:, None])


TIGHT = {
    "mu=1": rs12(1.0),
    "mu=50": rs12(50.0),
    "mu=400": rs12(400.0),
    "mu=2000": rs12(2000.0),
    "mu=20000": rs12(20000.0),
    "B=-0.5 mu=2000": rs12(2000.0, B=-0.5),
    "n=2 mu=400": rs12(400.0, n=2),
    "long range and g=1000": [(0.5, 0.5, 0.5, 0), (0.8, 0, 0, 1000.0)],
}


@pytest.mark.parametrize("name", list(TIGHT))
@pytest.mark.parametrize("cls", [2, 3, 4, 6])
def test_tight_gaussians(lib, name, cls):
    """The quadrature resolves the long range's branch point at r = 0 past the
    reach of a tight Gaussian.  Every point lies where the library uses the grid
    (exponents of an ordinary basis, a molecule's distances).  1e-10: what the
    auxiliary stage holds for the orders of its general classes."""
    g = Grid(lib, TIGHT[name], cls)
    pts = [(0.112, 0.0), (0.112, 3.1), (0.7, 0.02), (3.3, 1.1), (21.0, 0.0), (150.0, 0.6)]
    ref = reference(O.factor_kernel_terms(TIGHT[name]), cls, pts)
    for L in (8, 14):
        e = errors(g, ref, pts, L)
        assert e.max() < 1e-10, (L, e.max(1))


def test_rounding_of_the_quadrature(lib):
    """The cells carry the rounding of a few operations, not of the quadrature's
    nodes and sums: 3 u root mean square for f over a molecule's exponents and
    distances (nodes and weights as rounded doubles, summed one by one: 5 u).
    The point itself, the cell's polynomials and its Taylor sum account for 1 to
    2 u."""
    g = Grid(lib, rs12(), 3)
    kern = O.factor_kernel_terms(rs12())
    rng = np.random.default_rng(3)
    pts = [(float(np.exp(rng.uniform(np.log(0.06), np.log(6.0)))), float(rng.uniform(0.0, 7.0))) for _ in range(40)]
    with ThreadPoolExecutor(max_workers=min(16, os.cpu_count() or 1)) as ex:
        ref = np.array(list(ex.map(lambda p: O.radial(kern, 3, p[0], p[1], 0)[0], pts)))
    e = np.array([g.eval(x, d, 0)[0] for x, d in pts]) / ref - 1.0
    assert np.sqrt(np.mean(e * e)) < 3.0 * 2.0 ** -53


ACCEPT = {
    "default": rs12(),
    "B=2": rs12(B=2.0),
    "B=-0.5": rs12(B=-0.5),
    "B=-1.3": rs12(B=-1.3),
    "B=-4": rs12(B=-4.0),
    "mu=2000": rs12(2000.0),
    "long range and g=1000": [(0.5, 0.5, 0.5, 0), (0.8, 0, 0, 1000.0)],
}


@pytest.mark.parametrize("name", list(ACCEPT))
@pytest.mark.parametrize("cls", [2, 3, 4, 6])
def test_accepted_cells(lib, name, cls):
    """In both regions, out to where the exponents are diffuse and the kernels
    have grown or decayed, a cell that the check accepts holds every form that
    the kernels take to 1e-10 anywhere inside, not at the check's point alone
    (the check asks 1e-12 of one corner, 5e-11 of orders past 8).  Points with next to no refusals as
    well, so that a check that refuses everything fails."""
    g = Grid(lib, ACCEPT[name], cls)
    pts = [(0.0088, 0.0), (0.0102, 2.2), (0.0213, 1.0), (0.05, 9.3), (0.105, 0.0), (0.12, 20.2), (0.47, 6.9), (2.2, 14.3),
           (3.0, 0.7), (22.0, 9.1), (112.0, 3.1), (112.0, 7.9), (300.0, 1.9)]
    good = [p for p in pts if g.ok(*p) == 1]
    assert (0.47, 6.9) in good and (3.0, 0.7) in good and (112.0, 3.1) in good
    ref = reference(O.factor_kernel_terms(ACCEPT[name]), cls, good)
    for L in (0, 4, 8, 14):
        e = errors(g, ref, good, L)
        assert e.max() < 1e-10, (L, good[int(e.max(1).argmax())], e.max())


def test_default_factor_stays_on_the_grid(lib):
    """The default factor and its decaying form over the exponents and
    distances of the repository's molecules: nothing is refused."""
    for terms in (rs12(), rs12(B=-0.5)):
        for cls in (3, 4, 6):
            g = Grid(lib, terms, cls)
            assert all(g.ok(xi, D) == 1 for xi in (0.02, 0.0305, 4.1, 500.0) for D in (0.0, 8.0, 20.0))
            # (high orders pass through zero here)
            assert all(g.ok(xi, np.sqrt(T / xi)) == 1 for xi in (0.133, 0.266, 0.53) for T in (0.3, 0.4, 0.9))


def test_steep_decay_has_both_quadratures(lib):
    """The check's narrower panels are not what a factor is refused for: a decay of
    e^{-60 r} takes 337 panels in the lowest octave, 421 for the check."""
    g = Grid(lib, rs12(B=-60.0), 3)
    assert g.ok(0.0081, 0.3) != -1
