"""State of the batch engine and its context on the GPU: what is refused while a
batch runs, what a small budget leaves usable, and calls after an error."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1412_5070_gb300 import build as B
from paper_1412_5070_gb300 import f12int as F
from paper_1412_5070_gb300 import molecules as M

from test_gpu_batch import layout, per_call, sample


def make(budget=0):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    return F.f12int_create(0, budget, None)


def finish(ctx, t, limit_s=120.0):
    t0 = time.time()
    while not F.f12int_poll(ctx, t, 100_000):
        assert time.time() - t0 < limit_s, "request did not finish"


def test_settings_are_refused_between_the_passes_of_a_batch():
    """A batch whose Hermite rows exceed the class's buffer runs in passes.  Until
    the last one is launched and done, calls that change what it reads are
    refused (the series cap here, set to what it is)."""
    ctx = make()
    try:
        F.f12int_set_factor(ctx, M.P0)
        F.f12int_batch_limits(ctx, 4096, 1 << 18)
        basis = M.random_molecule(5, 4, 8.0, 1.8, (1, 1, 2, 2), (2, 3), (0.1, 60.0))
        bid = F.f12int_set_basis(ctx, basis)
        q = sample(basis, 3, 2000, 4)
        q = q[np.argsort(-basis.l[q].sum(axis=1))][:400]
        pq = np.prod(basis.nprim[q], axis=1)
        q = q[np.cumsum(pq) * 5 < (1 << 18)]      # five families at most: one request
        off, tot = layout(basis, q, (3,))
        out = torch.zeros(tot, dtype=torch.float64, device="cuda")
        finish(ctx, F.f12int_submit(ctx, bid, q, (3,), out, off))   # bounds, buffers, graph
        refused = 0
        for _ in range(5):
            t = F.f12int_submit(ctx, bid, q, (3,), out, off)
            done = False
            while not done:
                try:
                    F.f12int_set_series_cap(ctx, 0)
                    accepted = True
                except F.F12IntError as e:
                    assert e.status == F.EINVAL
                    accepted = False
                    refused += 1
                done = F.f12int_poll(ctx, t, 0)
                assert done or not accepted
        assert refused > 0
        ref = per_call(ctx, bid, 3, q, basis)
        tol = 1e-13 * np.abs(ref) + 1e-15 * np.max(np.abs(ref))
        assert np.all(np.abs(out.cpu().numpy() - ref) <= tol)
    finally:
        F.f12int_destroy(ctx)


GEMINAL = [(0.35, 0, 0, 0.4), (0.3, 0, 0, 1.3), (0.2, 0, 0, 4.5)]   # not on the grid: family by family


def test_family_batch_under_a_tight_budget():
    """A request that submit admits is not refused by the worker for want of
    memory: the Hermite rows of the family path come with the engine's other
    buffers (at least what one outer pair of a request's largest quartet takes).
    50 MB hold the engine's 20 MB and the bounds of a few shells."""
    basis = M.random_molecule(8, 2, 6.0, 1.8, (1, 1, 1, 1), (1, 3), (0.2, 30.0))
    q = M.canonical_quartets(basis, 3)[::3]
    off, tot = layout(basis, q, (3, 5))
    ctx = make(50 << 20)
    try:
        F.f12int_set_factor_terms(ctx, GEMINAL)
        F.f12int_batch_limits(ctx, 1024, 1 << 14)
        bid = F.f12int_set_basis(ctx, basis)
        out = torch.full((tot,), float("nan"), dtype=torch.float64, device="cuda")
        finish(ctx, F.f12int_submit(ctx, bid, q, (3, 5), out, off))
        got = out.cpu().numpy()
    finally:
        F.f12int_destroy(ctx)
    ctx = make()
    try:
        F.f12int_set_factor_terms(ctx, GEMINAL)
        bid = F.f12int_set_basis(ctx, basis)
        for k, cls in enumerate((3, 5)):
            ref = per_call(ctx, bid, cls, q, basis)
            mine = got[off[k, 0]:off[k, 0] + len(ref)]
            assert np.all(np.abs(mine - ref) <= 1e-13 * np.abs(ref) + 1e-15 * np.max(np.abs(ref)))
    finally:
        F.f12int_destroy(ctx)


def test_worker_allocates_nothing():
    """The first batch of a factor that goes family by family takes no device
    memory of its own (64 MB leave room for the instantiated graph)."""
    ctx = make()
    try:
        basis = M.random_molecule(8, 2, 6.0, 1.8, (1, 1, 1, 1), (1, 3), (0.2, 30.0))
        q = M.canonical_quartets(basis, 3)[::3]
        off, tot = layout(basis, q, (3,))
        out = torch.zeros(tot, dtype=torch.float64, device="cuda")
        F.f12int_set_factor(ctx, M.P0)
        F.f12int_batch_limits(ctx, 4096, 1 << 18)
        bid = F.f12int_set_basis(ctx, basis)
        finish(ctx, F.f12int_submit(ctx, bid, q, (3,), out, off))
        F.f12int_set_factor_terms(ctx, GEMINAL)
        per_call(ctx, bid, 3, q, basis)
        torch.cuda.synchronize()
        free0 = torch.cuda.mem_get_info()[0]
        finish(ctx, F.f12int_submit(ctx, bid, q, (3,), out, off))
        assert free0 - torch.cuda.mem_get_info()[0] < 64 << 20
    finally:
        F.f12int_destroy(ctx)


def test_no_factor_after_a_set_factor_that_failed():
    """set_factor replaces the tables one by one; when one of them exceeds the
    budget the context has no factor left (neither freed tables nor the former
    grid are read), and takes the next one."""
    one = [(1.0, 0, 0, 0.7)]
    xi, D = torch.tensor([0.4, 3.0], dtype=torch.float64).cuda(), torch.tensor([1.0, 0.2], dtype=torch.float64).cuda()
    for budget in (1 << k for k in range(16, 24)):   # the least of these that holds the tables of one Gaussian
        ctx = make(budget)
        try:
            F.f12int_set_factor_terms(ctx, one)
        except F.F12IntError as e:
            assert e.status == F.ENOMEM
            F.f12int_destroy(ctx)
            continue
        break
    try:
        out = torch.zeros((2, 3), dtype=torch.float64, device="cuda")
        F.f12int_aux(ctx, 3, xi, D, 2, out)
        torch.cuda.synchronize()
        want = out.cpu().numpy().copy()
        with pytest.raises(F.F12IntError) as e:      # the start-value tables of its growing families alone take more
            F.f12int_set_factor(ctx, M.P0)
        assert e.value.status == F.ENOMEM
        with pytest.raises(F.F12IntError) as e:
            F.f12int_aux(ctx, 3, xi, D, 2, out)
        assert e.value.status == F.ENOTREADY
        F.f12int_set_factor_terms(ctx, one)
        out.zero_()
        F.f12int_aux(ctx, 3, xi, D, 2, out)
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), want)
    finally:
        F.f12int_destroy(ctx)


def test_calls_after_an_allocation_that_failed():
    """An engine whose buffers do not fit the device (2^46 items) is refused with
    F12INT_ENOMEM; the calls after it do not report that error again."""
    ctx = make()
    try:
        F.f12int_set_factor(ctx, M.P0)
        basis = M.two_centre_sp()
        bid = F.f12int_set_basis(ctx, basis)
        q = M.canonical_quartets(basis, 3)[:12]
        want = per_call(ctx, bid, 3, q, basis)
        F.f12int_batch_limits(ctx, 16, 1 << 46)
        off, tot = layout(basis, q, (3,))
        out = torch.zeros(tot, dtype=torch.float64, device="cuda")
        with pytest.raises(F.F12IntError) as e:
            F.f12int_submit(ctx, bid, q, (3,), out, off)
        assert e.value.status == F.ENOMEM
        assert np.array_equal(per_call(ctx, bid, 3, q, basis), want)
    finally:
        F.f12int_destroy(ctx)
