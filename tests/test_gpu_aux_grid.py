"""The auxiliary grid and the Boys path of the CUDA library where they can go
wrong: ends of cells in xi and in D^2, the seams between the regions, D = 0,
every order bucket, and points the grid does not hold (which take the family
path).  Against the oracle's radial integrals."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import oracle as O
from paper_1412_5070_gb300 import build as B
from paper_1412_5070_gb300 import f12int as F
from paper_1412_5070_gb300 import molecules as M

# relative to |g_l| + |g_{l+1}| times a twentieth of the local width (an order
# that passes through zero has no relative accuracy of its own): the cells'
# acceptance 3e-13 per order plus the rounding of the terms
TOL = 2e-12


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()
    c = F.f12int_create(0, 0, None)
    F.f12int_set_factor(c, M.P0)
    yield c
    F.f12int_destroy(c)


def edge_points():
    eps = 1e-13
    pts = []
    for xi0 in (2.0 ** -5, 2.0 ** -3, 0.140625, 1.0, 1.125, 6.5, 64.0, 300.0):   # cell ends in xi, octaves, the finer part
        for xi in (xi0 * (1 - eps), xi0 * (1 + eps), xi0 * 1.03):
            for T in (0.0, 1e-9, 0.25, 7.999, 8.001, 8.5, 31.99, 64.01, 99.9, 100.1, 479.0, 511.0, 513.0, 545.0):
                D = np.sqrt(T / xi)
                if D < 30.0:
                    pts.append((xi, D))
    for xi, D in ((500.0, 12.0), (8000.0, 3.0), (8000.0, 0.01), (0.009, 2.0), (0.5, 24.0), (40.0, 18.0)):
        pts.append((xi, D))
    return np.array(pts)


@pytest.mark.parametrize("cls", [1, 2, 3, 4, 6])
@pytest.mark.parametrize("nmax", [0, 4, 5, 8, 9])
def test_cell_edges_and_seams(ctx, cls, nmax):
    pts = edge_points()[nmax % 3::3]
    xi, D = pts[:, 0].copy(), pts[:, 1].copy()
    out = torch.full((len(xi), nmax + 1), float("nan"), dtype=torch.float64, device="cuda")
    F.f12int_aux(ctx, cls, torch.from_numpy(xi).cuda(), torch.from_numpy(D).cuda(), nmax, out)
    torch.cuda.synchronize()
    F.f12int_device_status(ctx)
    got = out.cpu().numpy()
    kern = O.factor_kernel(M.P0)
    ref = np.array([O.radial(kern, cls, x, d, nmax + 1) for x, d in zip(xi, D)])
    scale = np.abs(ref[:, :-1]) + 0.05 * np.abs(ref[:, 1:]) * np.minimum(D * D + 1e-300, 1.0 / xi)[:, None]
    err = np.abs(got - ref[:, :-1]) / scale
    assert np.isfinite(got).all() and err.max() <= TOL, (err.max(), pts[err.max(1).argmax()])


def test_points_outside_the_grid_take_the_family_path(ctx):
    xi, D = np.array([2.0e4, 0.005, 0.02]), np.array([0.4, 3.0, 140.0])
    out = torch.full((3, 3), float("nan"), dtype=torch.float64, device="cuda")
    F.f12int_aux(ctx, 3, torch.from_numpy(xi).cuda(), torch.from_numpy(D).cuda(), 2, out)
    torch.cuda.synchronize()
    kern = O.factor_kernel(M.P0)
    ref = np.array([O.radial(kern, 3, x, d, 2) for x, d in zip(xi, D)])
    assert np.all(np.abs(out.cpu().numpy() - ref) <= 1e-10 * np.abs(ref))


def test_basis_past_the_grid_equals_the_oracle(ctx):
    """A basis whose exponents leave the grid is evaluated family by family."""
    basis = M.random_molecule(3, 2, 6.0, 1.8, (2, 1, 0, 0), (1, 2), (0.05, 3.0e4))
    basis.exps[0] = 2.0e4
    bid = F.f12int_set_basis(ctx, basis)
    q = M.canonical_quartets(basis, 2)[::5]
    off = M.block_offsets(basis, q)
    out = torch.full((int(off[-1]),), float("nan"), dtype=torch.float64, device="cuda")
    F.f12int_compute_class(ctx, bid, 2, torch.from_numpy(np.ascontiguousarray(q)).cuda(), out,
                           torch.from_numpy(off[:-1].copy()).cuda())
    torch.cuda.synchronize()
    ref, _ = O.shell_blocks(O.factor_kernel(M.P0), 2, basis, q)
    got = out.cpu().numpy()
    big = np.abs(ref) > 1e-12
    assert np.all(np.abs(got - ref)[big] <= 1e-10 * np.abs(ref)[big]) and np.all(np.abs(got - ref)[~big] <= 1e-12)
