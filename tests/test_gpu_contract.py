"""The general contraction of the CUDA library at the sizes where its variants
meet: inner primitive pairs around the number that is staged at once (15, 16,
17, 36), both orientations of a quartet (bra or ket summed first), component
ranges, orders on both sides of the register/local-memory recursion, and rows
that exceed the scratch of the static call and of the batch engine (outer pairs
in several launches).  Against the oracle, and against each other."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O
from paper_1412_5070_gb300 import build as B
from paper_1412_5070_gb300 import f12int as F
from paper_1412_5070_gb300 import molecules as M
from test_gpu_parity import close, gpu_blocks, report


@pytest.fixture()
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    c = F.f12int_create(0, 0, None)
    F.f12int_set_factor(c, M.P0)
    yield c
    F.f12int_destroy(c)


def shells(spec, seed):
    """A basis of the shells (l, primitives), each on a centre of its own."""
    rng = np.random.default_rng(seed)
    n = np.array([k for _, k in spec], dtype=np.int32)
    return M.Basis(centers=rng.uniform(0.0, 4.0, size=(len(spec), 3)), l=np.array([l for l, _ in spec], dtype=np.int32),
                   nprim=n, exps=np.exp(rng.uniform(np.log(0.1), np.log(8.0), size=int(n.sum()))),
                   coefs=rng.uniform(0.1, 1.0, size=int(n.sum())), name="edge shells")


# s3 s5 s17 s4 s4 s6 s6 | p1 p1 d1 d1 f1 f1
EDGE = [(0, 3), (0, 5), (0, 17), (0, 4), (0, 4), (0, 6), (0, 6), (1, 1), (1, 1), (2, 1), (2, 1), (3, 1), (3, 1)]
PAIRS_S = [(0, 1), (3, 4), (2, 7), (5, 6)]              # 15, 16, 17 and 36 primitive pairs
PAIRS_L = [(8, 10), (9, 10), (9, 11), (11, 12)]         # pd, dd, df, ff


@pytest.mark.parametrize("cls", [1, 3, 5, 6])
def test_staging_edges_and_orientations(ctx, cls):
    """(few functions, many pairs | many functions, one pair) and its mirror:
    whichever pair is summed first, the staged count is met from both sides; 289 pairs, past the bound on the inner pair, as well."""
    basis = shells(EDGE, 5)
    q = np.array([[*a, *b] for a in PAIRS_S for b in PAIRS_L] + [[*b, *a] for a in PAIRS_S for b in PAIRS_L] +
                 [[11, 12, 11, 12], [9, 10, 11, 12], [2, 2, 9, 10], [9, 10, 2, 2]], dtype=np.int32)
    bid = F.f12int_set_basis(ctx, basis)
    got, _ = gpu_blocks(ctx, bid, cls, basis, q)
    ref, _, mag = O.shell_blocks(O.factor_kernel(M.P0), cls, basis, q, with_mag=True)
    bad = close(got, ref, mag, "I%d %s" % (cls, basis.name))
    assert not np.isnan(got).any()
    assert not bad.any(), report(got, ref, mag, bad)


@pytest.mark.parametrize("cls", [3, 5])
def test_rows_beyond_the_scratch(ctx, cls):
    """(ff|ff) of 12^4 primitive quartets: 76 MB of rows, 113 MB for I5.  The
    static call (64 MB of scratch) and an engine with 32 MB row buffers take its outer pairs in several launches.  Every element is summed in
    the same order: the static call (the same kernel) equals the allocating one
    bitwise.  The engine's instance of the kernel may contract its products into
    multiply-adds differently: 2e4 primitive quartets of at most 1e3 products,
    rounded at random, move an element by sqrt(2e7) u = 5e-13 of its terms, here
    taken as at most 20 times the largest element of its block."""
    F.f12int_batch_limits(ctx, 1024, 1 << 18)
    basis = shells([(3, 12), (3, 12), (0, 2), (2, 2)], 9)
    bid = F.f12int_set_basis(ctx, basis)
    q = np.array([[0, 1, 0, 1], [3, 2, 3, 2], [0, 2, 3, 2], [2, 3, 0, 2]], dtype=np.int32)
    want, off = gpu_blocks(ctx, bid, cls, basis, q)
    dq, doff = torch.from_numpy(q).cuda(), torch.from_numpy(off[:-1].copy()).cuda()
    out = torch.full((int(off[-1]),), float("nan"), dtype=torch.float64, device="cuda")
    F.f12int_compute_class_static(ctx, bid, cls, dq, out, doff)
    torch.cuda.synchronize()
    F.f12int_device_status(ctx)
    assert np.array_equal(out.cpu().numpy(), want)
    out.fill_(float("nan"))
    torch.cuda.synchronize()
    t = F.f12int_submit(ctx, bid, q, [cls], out, off[:-1].reshape(1, -1).copy())
    for _ in range(100):
        if F.f12int_poll(ctx, t, 1_000_000):
            break
    got = out.cpu().numpy()
    for k in range(len(q)):
        a, b = int(off[k]), int(off[k + 1])
        assert np.abs(got[a:b] - want[a:b]).max() <= 1e-11 * np.abs(want[a:b]).max()
