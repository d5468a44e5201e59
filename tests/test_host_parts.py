"""Host-side parts of the library that need no GPU, compiled from its headers
(tests/host_parts.cpp)."""
import ctypes
import glob
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1412_5070_gb300", "csrc")
SRC = os.path.join(HERE, "host_parts.cpp")
LIB = os.path.join(HERE, "_build", "libhostparts.so")


@pytest.fixture(scope="module")
def lib():
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    os.makedirs(os.path.dirname(LIB), exist_ok=True)
    deps = [SRC] + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    if not os.path.exists(LIB) or any(os.path.getmtime(d) > os.path.getmtime(LIB) for d in deps):
        tmp = LIB + ".tmp%d" % os.getpid()
        subprocess.run([gxx, "-O1", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-pthread", "-o", tmp, SRC], check=True)
        os.replace(tmp, LIB)
    return ctypes.CDLL(LIB)


def test_a_batch_is_running_until_its_last_launch(lib):
    """A ticket whose batch is being launched is not in flight yet; its staging
    buffer's event is an earlier batch's, complete or never recorded."""
    idle = lib.host_tickets_idle
    assert idle(0, -1, 0, 1) == 0                          # queued
    assert idle(0, 0, 0, 1) == 0 and idle(0, 1, 0, 1) == 0  # between the passes of its batch
    assert idle(0, 0, 1, 0) == 0                           # in flight
    assert idle(0, 0, 1, 1) == 1                           # finished, not yet reported
    assert idle(1, -1, 0, 1) == 1                          # done


def test_least_rows_hold_an_outer_pair_of_any_admitted_quartet(lib):
    """Sides of a and b primitive pairs, a b <= items: the inner side is either
    one up to 256 pairs, the smaller one past that; 680 doubles a row at the
    highest order.  And no more than is needed for small limits (a context
    with a tight budget)."""
    lib.host_rows_least.restype = ctypes.c_int64
    lib.host_rows_least.argtypes = [ctypes.c_int64]
    for items in (1, 36, 255, 256, 257, 4096, 65536, 65537, 10 ** 6, 1 << 26):
        least = lib.host_rows_least(items)
        for a in sorted({1, 2, 17, 255, 256, 257, 300, int(items ** 0.5), items}):
            b = items // a
            if b < 1:
                continue
            inner = min(a, b) if max(a, b) > 256 else max(a, b)
            assert 680 * inner <= least, (items, a, b)
    assert lib.host_rows_least(100) == 68000


def test_tables_are_filled_once_per_device(lib):
    """The constant tables and their addresses belong to a device: a context on
    another device of the process fills its own, and a fill that failed is
    tried again."""
    dev = (ctypes.c_int * 6)(0, 1, 0, 3, 3, 1)
    val, st = (ctypes.c_int * 6)(*[-1] * 6), (ctypes.c_int * 6)()
    assert lib.host_per_device(dev, 6, 3, val, st) == 4
    assert list(st) == [0, 0, 0, -6, 0, 0]
    assert list(val) == [100, 101, 100, -1, 103, 101]


def test_static_staging_never_locks_pages(lib):
    """The staging of the static call stays in plain memory whatever the list's
    length (locking pages waits for other streams); the allocating call's is
    page-locked from 256 KB on, and freed as it was allocated."""
    sizes = (ctypes.c_int64 * 5)(1000, 100_000, 400_000, 3_000_000, 200_000_000)
    locks = (ctypes.c_int * 2)()
    assert lib.host_stage(0, sizes, 5, locks) == 1 and list(locks) == [0, 0]
    assert lib.host_stage(1, sizes, 5, locks) == 1 and list(locks) == [2, 2]


def test_the_static_call_uses_that_staging():
    src = open(os.path.join(CSRC, "f12int.cu")).read()
    body = src[src.index('extern "C" int f12int_compute_class_static('):]
    assert "ctx->static_stage" in body and "ctx->stage" not in body
    assert "HostStage static_stage{false};" in src


def test_uploads_are_ordered_with_the_kernels_streams():
    """A plain cudaMemcpy from pageable memory, or a cudaMemset, may return before
    its last part has arrived, on a stream that non-blocking streams do not wait
    for: every upload names its stream."""
    for path in glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        assert not re.search(r"\bcudaMemset\(", src), path
        assert not re.search(r"\bcudaMemcpy\([^;]*cudaMemcpyHostToDevice\)", src), path


@pytest.mark.parametrize("direct", [0, 1])
def test_a_static_list_that_is_accepted_runs_in_its_scratch(lib, direct):
    """Whatever room the list leaves, an accepted one has the items and the rows of
    one outer pair of any general quartet, the items of any thin one, and stays
    inside the room: nothing is refused once work is queued.  Refused is what
    lacks the items of a quartet, or the rows of one outer pair."""
    cut = lib.host_scratch_cut
    cut.argtypes = [ctypes.c_int64, ctypes.c_int] + [ctypes.c_int64] * 4 + [ctypes.POINTER(ctypes.c_int64)]
    c = (ctypes.c_int64 * 4)()
    for nf in (1, 5, 12):
        for pq, inner in ((1, 1), (36, 6), (36, 36), (6561, 81), (4, 0), (70000, 256)):
            for pitch in (36, 288, 680):
                need = pq * nf * 136
                tight = need + (inner * pitch * 8 if inner else 0)
                for room in sorted({need - 1, need, need + 64, inner * (nf * 136 + pitch * 8 + 64), tight, tight + 136,
                                    tight + 300, 2 * tight + 4096, 60_000_000}):
                    ok = cut(room, direct, nf, pq, inner, pitch, c)
                    keys, thin, part, rows = list(c)
                    if room < need:
                        assert not ok
                    if room >= 2 * tight + 4096:
                        assert ok
                    if not ok:
                        continue
                    if direct:
                        assert keys >= inner and rows >= inner * pitch and 4 * keys + 8 * rows <= room
                        continue
                    assert 8 * keys + 8 * thin <= room and thin >= pq * nf * 16
                    if inner:
                        assert part >= inner * nf * 16 and rows >= inner * pitch and part + rows <= thin
                        assert part % 16 == 0


def test_growth_table_index_stays_in_the_table(lib):
    """Distances to 1e38 bohr and past single precision's range (atoms that far
    apart are accepted input) take the last entry."""
    idx = lib.host_grow_index
    idx.argtypes = [ctypes.c_float, ctypes.c_int]
    n = 2401
    for x in (0.0, 0.5, 1.0, 17.3, 2398.5, 2399.0, 2399.9, 2400.0, 2401.0, 1e6, 2.2e9, 4.3e9, 1e20, 3e38, float("inf"),
              float("nan")):
        assert idx(x, n) == (min(n - 1, int(x) + 1) if x < 1e9 else n - 1), x


@pytest.mark.parametrize("rate", [0.02, 0.5, 1.0, 4.0, 9.0])
def test_primitive_screen_decides_as_in_double_precision(lib, rate):
    """Weighed in single precision first, every candidate is decided as the weighing
    in double precision alone decides it: kernels that grow like e^{rate r}
    (the last two past single precision's range), distances from one centre to
    past the table, products spread around the threshold and on it."""
    rng = np.random.default_rng(int(100 * rate))
    r = np.arange(2401) * 0.05
    with np.errstate(over="ignore"):
        g = np.maximum(1.0, np.exp(rate * r) / np.exp(1.5 * rate))
    n = 200_000
    R = np.where(rng.random(n) < 0.1, 0.0, rng.uniform(0.0, 130.0, n))
    R[::7] = 0.05 * np.round(R[::7] / 0.05)            # on the table's entries
    iv = np.exp(rng.uniform(np.log(1e-3), np.log(60.0), n))
    gam = np.interp(R, r, np.log(g))                   # about ln Gamma
    v = 1e-26 * np.exp(-gam + rng.normal(0.0, np.where(rng.random(n) < 0.5, 1.0, 0.01) * (1 + 2 * rate)))
    v[::11] = 0.0
    v = np.minimum(v, 0.999e-26)
    dp, ip = ctypes.POINTER(ctypes.c_double), ctypes.POINTER(ctypes.c_int)
    u = R * R
    got, want = np.zeros(n, np.int32), np.zeros(n, np.int32)
    f = lib.host_screen
    f.argtypes = [dp, ctypes.c_int, ctypes.c_double, dp, dp, dp, ctypes.c_int, ip, ip]
    f(g.ctypes.data_as(dp), len(g), 1e-26, v.ctypes.data_as(dp), u.ctypes.data_as(dp), iv.ctypes.data_as(dp), n,
      got.ctypes.data_as(ip), want.ctypes.data_as(ip))
    assert np.array_equal(got, want)
    assert 0 < want.sum() < n
    # candidates as they come, over thirty orders of magnitude: few take both weighings
    v = np.minimum(1e-26 * np.exp(-gam + rng.uniform(-35.0, 35.0, n)), 0.999e-26)
    both = f(g.ctypes.data_as(dp), len(g), 1e-26, v.ctypes.data_as(dp), u.ctypes.data_as(dp), iv.ctypes.data_as(dp), n,
             got.ctypes.data_as(ip), want.ctypes.data_as(ip))
    assert np.array_equal(got, want)
    assert rate > 0.6 or both < n // 10   # (past that the table leaves single precision within the distances)
