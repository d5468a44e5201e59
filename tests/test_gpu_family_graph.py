"""Calls that go family by family: a factor of Gaussians alone, and a factor with
b < 0 families (a second evaluation launch) on a basis whose exponents the grid
of auxiliary functions does not hold.  Every entry point -- plain, static, mixed
and batched (the engine's second graph, its passes, and a quartet larger than
its row buffer) -- against the oracle or the plain call."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O
from paper_1412_5070_gb300 import build as B
from paper_1412_5070_gb300 import f12int as F
from paper_1412_5070_gb300 import molecules as M

from test_gpu_batch import layout, per_call, sample
from test_gpu_contract import shells
from test_gpu_parity import close, report

GEMINAL = [(0.35, 0, 0, 0.4), (0.3, 0, 0, 1.3), (0.2, 0, 0, 4.5)]
DECAYING = dict(c0=0.5, rho=-0.5, B=-0.8, mu=1.0, n=0)
TIGHT = 2.0e4          # an exponent past the grid's range of xi (2^13)


def context(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    c = F.f12int_create(0, 0, None)
    if name == "geminal":
        F.f12int_set_factor_terms(c, GEMINAL)
        return c, O.factor_kernel_terms(GEMINAL)
    assert all(F.f12int_factor_classes(DECAYING)[k] == 3 for k in (2, 3, 4, 6))   # the quadrature launch
    F.f12int_set_factor(c, DECAYING)
    return c, O.factor_kernel(DECAYING)


def molecule():
    b = M.random_molecule(21, 2, 5.0, 1.8, (2, 1, 1, 1), (1, 2), (0.2, 20.0))
    b.exps[0] = TIGHT
    return b


def finish(ctx, t, limit_s=120.0):
    t0 = time.time()
    while not F.f12int_poll(ctx, t, 100_000):
        assert time.time() - t0 < limit_s, "request did not finish"


@pytest.mark.parametrize("name", ["geminal", "decaying"])
def test_request_against_oracle(name):
    """One request for every class through the engine's family graph."""
    ctx, kern = context(name)
    try:
        basis = molecule()
        bid = F.f12int_set_basis(ctx, basis)
        classes = (2, 3, 4, 5, 6)
        q = sample(basis, 5, 60, 12)
        off, tot = layout(basis, q, classes)
        out = torch.full((tot,), float("nan"), dtype=torch.float64, device="cuda")
        finish(ctx, F.f12int_submit(ctx, bid, q, classes, out, off))
        got = out.cpu().numpy()
        for k, cls in enumerate(classes):
            ref, _, mag = O.shell_blocks(kern, cls, basis, q, with_mag=True)
            mine = got[off[k, 0]:off[k, 0] + len(ref)]
            bad = close(mine, ref, mag, "I%d %s" % (cls, name))
            assert not np.isnan(mine).any()
            assert not bad.any(), report(mine, ref, mag, bad)
    finally:
        F.f12int_destroy(ctx)


@pytest.mark.parametrize("name", ["geminal", "decaying"])
@pytest.mark.parametrize("cls", [3, 5, 6])
def test_plain_static_and_mixed_calls(name, cls):
    """The plain call against the oracle, the static one bitwise against it, and the
    mixed one as its own tests hold it: FP64 quartets bitwise, the others within
    1e-10 at the default bound."""
    ctx, kern = context(name)
    try:
        basis = molecule()
        bid = F.f12int_set_basis(ctx, basis)
        q = np.ascontiguousarray(sample(basis, cls, 60, 30 + cls))
        want = per_call(ctx, bid, cls, q, basis)
        ref, _, mag = O.shell_blocks(kern, cls, basis, q, with_mag=True)
        bad = close(want, ref, mag, "I%d %s" % (cls, name))
        assert not bad.any(), report(want, ref, mag, bad)
        off = M.block_offsets(basis, q)
        dq, doff = torch.from_numpy(q).cuda(), torch.from_numpy(off[:-1].copy()).cuda()
        out = torch.full((int(off[-1]),), float("nan"), dtype=torch.float64, device="cuda")
        F.f12int_compute_class_static(ctx, bid, cls, dq, out, doff)
        torch.cuda.synchronize()
        F.f12int_device_status(ctx)
        assert np.array_equal(out.cpu().numpy(), want)
        est = F.f12int_quartet_estimates(ctx, bid, cls, q)
        below = 1e-5
        out.fill_(float("nan"))
        F.f12int_compute_class_mixed(ctx, bid, cls, dq, out, doff, below)
        torch.cuda.synchronize()
        got = out.cpu().numpy()
        f32 = np.repeat(est < below, np.diff(off))
        assert f32.any() and not f32.all()
        assert np.array_equal(got[~f32], want[~f32])
        assert np.abs(got - ref)[f32].max() <= 1e-10
    finally:
        F.f12int_destroy(ctx)


@pytest.mark.parametrize("name", ["geminal", "decaying"])
@pytest.mark.parametrize("cls", [3, 5])
def test_quartet_larger_than_the_row_buffer(name, cls):
    """(ff|ff) of 12^4 primitive quartets, 76 MB of rows (113 MB for I5), in an engine
    whose family graph holds 36 MB a class: outer pair by outer pair, with two
    ordinary quartets in passes of their own.  Tolerance as in the general
    contraction's test of the same on the grid."""
    ctx, _ = context(name)
    try:
        F.f12int_batch_limits(ctx, 1024, 1 << 18)
        basis = shells([(3, 12), (3, 12), (0, 2), (2, 2)], 9)
        basis.exps[0] = TIGHT
        bid = F.f12int_set_basis(ctx, basis)
        q = np.array([[0, 1, 0, 1], [3, 2, 3, 2], [0, 2, 3, 2], [2, 3, 0, 2]], dtype=np.int32)
        want = per_call(ctx, bid, cls, q, basis)
        off, tot = layout(basis, q, (cls,))
        out = torch.full((tot,), float("nan"), dtype=torch.float64, device="cuda")
        finish(ctx, F.f12int_submit(ctx, bid, q, (cls,), out, off))
        got = out.cpu().numpy()
        ends = np.append(off[0], tot)
        for a, b in zip(ends[:-1], ends[1:]):
            assert np.abs(got[a:b] - want[a:b]).max() <= 1e-11 * np.abs(want[a:b]).max()
    finally:
        F.f12int_destroy(ctx)


@pytest.mark.parametrize("name", ["geminal", "decaying"])
def test_batch_in_passes(name):
    """A batch whose rows exceed the family graph's buffer several times over."""
    ctx, _ = context(name)
    try:
        F.f12int_batch_limits(ctx, 4096, 1 << 18)
        basis = M.random_molecule(5, 4, 8.0, 1.8, (1, 1, 2, 2), (2, 3), (0.1, 60.0))
        basis.exps[0] = TIGHT
        bid = F.f12int_set_basis(ctx, basis)
        q = sample(basis, 3, 2000, 4)
        q = q[np.argsort(-basis.l[q].sum(axis=1))][:400]
        q = q[np.cumsum(np.prod(basis.nprim[q], axis=1)) * 5 < (1 << 18)]
        off, tot = layout(basis, q, (3,))
        out = torch.full((tot,), float("nan"), dtype=torch.float64, device="cuda")
        finish(ctx, F.f12int_submit(ctx, bid, q, (3,), out, off))
        ref, got = per_call(ctx, bid, 3, q, basis), out.cpu().numpy()
        assert np.all(np.abs(got - ref) <= 1e-13 * np.abs(ref) + 1e-15 * np.max(np.abs(ref)))
    finally:
        F.f12int_destroy(ctx)


def test_requests_of_both_sorts():
    """Requests on a basis inside the grid and on one past it, in flight at once: a
    batch holds one sort, and every request is its plain call."""
    ctx, _ = context("decaying")
    try:
        inside, past = M.random_molecule(21, 2, 5.0, 1.8, (2, 1, 1, 1), (1, 2), (0.2, 20.0)), molecule()
        reqs = []
        for k in range(6):
            basis = (inside, past)[k % 2]
            bid = F.f12int_set_basis(ctx, basis)
            q = sample(basis, 3, 80, 50 + k)
            off, tot = layout(basis, q, (3, 6))
            out = torch.full((tot,), float("nan"), dtype=torch.float64, device="cuda")
            reqs.append((basis, bid, q, off, out, F.f12int_submit(ctx, bid, q, (3, 6), out, off)))
        for r in reqs:
            finish(ctx, r[-1])
        for basis, bid, q, off, out, _ in reqs:
            got = out.cpu().numpy()
            for k, cls in enumerate((3, 6)):
                ref = per_call(ctx, bid, cls, q, basis)
                mine = got[off[k, 0]:off[k, 0] + len(ref)]
                assert np.all(np.abs(mine - ref) <= 1e-13 * np.abs(ref) + 1e-15 * np.max(np.abs(ref)))
    finally:
        F.f12int_destroy(ctx)
