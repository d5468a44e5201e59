"""Timed cases of the integral library: what a user has it compute.

A case is one call (or one set of batched requests) on a seeded random
molecule of the kind the repository's configurations describe: s/p shells on
two centres, contracted s/p/d shells on a dozen atoms, and contracted shells
up to f; all integral classes, the plain, mixed-precision, static-scratch and
batched entry points, and the auxiliary stage alone.  ``prepare`` holds what a
program keeps between calls (a context with its factor and basis, the screened
quartet list and the output array on the device); ``run`` is one pass.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1412_5070_gb300 import f12int as F
from paper_1412_5070_gb300 import molecules as M

# Correlation factors: the default range-separated one, its decaying form
# (B < 0), and a Gaussian geminal given as a term list.
FACTORS = {
    "rs12": dict(c0=0.5, rho=-0.5, B=0.5, mu=1.0, n=0),
    "rs12_decay": dict(c0=0.5, rho=-0.5, B=-0.5, mu=1.0, n=0),
}
GEMINAL = ((0.35, 0.0, 0.0, 0.4), (0.3, 0.0, 0.0, 1.3), (0.2, 0.0, 0.0, 4.5))


def _case(name, kind, classes, atoms, shells, prims, exps, n, factor="rs12", box=12.0, mols=1):
    s, p, d, f = shells
    return {"name": name, "kind": kind, "classes": classes, "atoms": atoms, "s": s, "p": p, "d": d, "f": f,
            "prim_lo": prims[0], "prim_hi": prims[1], "exp_lo": exps[0], "exp_hi": exps[1], "n": n,
            "factor": factor, "box": box, "mols": mols}


SP = ((4, 2, 0, 0), (1, 1), (0.1, 2.7))        # the two-centre s/p system
SPD = ((3, 2, 1, 0), (3, 3), (0.05, 50.0))     # the 12-atom s/p/d benchmark
SPDF = ((4, 3, 2, 1), (1, 6), (0.03, 200.0))   # the batching and serving molecules
TZ = ((5, 4, 3, 2), (1, 8), (0.02, 500.0))     # the mixed-precision molecule's shells


def listed():
    return [
        # a handful of blocks, as an integral-direct program asks for them: launch and host latency
        _case("sp2_I3_16", "class", "3", 2, *SP, 16),
        # a diatomic's blocks with s and p shells
        _case("sp2_I6_600", "class", "6", 2, *SP, 600),
        # ordinary ERIs of a contracted basis, the reference class
        _case("spd12_I1_200k", "class", "1", 12, *SPD, 200000),
        # an F12 class of the same, odd number of blocks
        _case("spd12_I3_50001", "class", "3", 12, *SPD, 50001),
        _case("spd12_I4_200k", "class", "4", 12, *SPD, 200000),
        # the commutator class (orders L + 2, no bra-ket symmetry): the bulk of a whole F12 calculation
        _case("spd12_I5_600k", "class", "5", 12, *SPD, 600000),
        # shells up to f, uneven contraction lengths: one integral-block request through the plain call
        _case("spdf6_I2_3000", "class", "2", 6, *SPDF, 3000),
        # FP32 recursion for small blocks, triple-zeta-like shells
        _case("tz4_I4_mixed_2000", "mixed", "4", 4, *TZ, 2000, box=20.0),
        # a decaying long range (B < 0)
        _case("spd5_I3_decay_4000", "class", "3", 5, *SPD, 4000, factor="rs12_decay"),
        # a Gaussian geminal given as a term list, through the call that allocates nothing
        _case("spd8_I6_geminal_static_5000", "static", "6", 8, *SPD, 5000, factor="geminal"),
        # several molecules' requests for all five F12 classes, in flight at once
        _case("batch_spdf_4x600", "batch", "23456", 6, *SPDF, 600, mols=4),
        # the auxiliary functions alone, over the exponents and distances molecules give
        _case("aux_I4_5000", "aux", "4", 0, (0, 0, 0, 0), (1, 1), (0.02, 300.0), 5000),
    ]


def draw(rng):
    lu = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    kind = rng.choice(("class", "class", "class", "mixed", "static", "batch", "aux"))
    factor = rng.choice(("rs12", "rs12", "rs12", "rs12_decay", "geminal"))
    cls = rng.choice("123456")
    if kind == "aux":
        c = _case("", kind, cls, 0, (0, 0, 0, 0), (1, 1), (0.02, 300.0), lu(100, 100000), factor)
    elif kind == "batch":
        c = _case("", kind, "".join(k for k in "23456" if rng.random() < 0.7) or "3", rng.randint(2, 9), *SPDF,
                  lu(50, 800), "rs12", mols=rng.randint(1, 5))
    elif kind == "mixed":
        c = _case("", kind, cls, rng.randint(2, 4), *TZ, lu(100, 2500), "rs12", box=20.0)
    else:
        basis = rng.choice((SP, SPD, SPD, SPDF))
        atoms = 2 if basis is SP else rng.randint(3, 12) if basis is SPD else rng.randint(2, 8)
        hi = 2500 if basis is SP else 4000 if basis is SPDF else 200000 if factor == "rs12" else 8000
        if kind == "static":
            hi = min(hi, 4000)
        c = _case("", kind, cls, atoms, *basis, lu(8, hi), factor)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs --

class State:
    """A context with its factor, bases and device arrays; the context's
    device memory goes with the object."""

    def __init__(self, factor):
        self.ctx = F.f12int_create(0, 0, None)
        if factor == "geminal":
            F.f12int_set_factor_terms(self.ctx, GEMINAL)
        else:
            F.f12int_set_factor(self.ctx, FACTORS[factor])

    def __del__(self):
        if getattr(self, "ctx", None) is not None:
            torch.cuda.synchronize()
            F.f12int_destroy(self.ctx)
            self.ctx = None


def _molecule(case, seed):
    return M.random_molecule(seed, case["atoms"], case["box"], 1.8, (case["s"], case["p"], case["d"], case["f"]),
                             (case["prim_lo"], case["prim_hi"]), (case["exp_lo"], case["exp_hi"]))


def _shells(case):
    """Angular momentum of every shell, as random_molecule orders them."""
    return np.array([l for _ in range(case["atoms"]) for l, k in enumerate("spdf") for _ in range(case[k])])


def _canonical_sample(case):
    """n canonical shell quartets (as f12int_screen lists them), the same
    shells for every seed so that every molecule's blocks lie alike."""
    ns = len(_shells(case))
    a, b = np.tril_indices(ns)
    npair = len(a)
    total = npair * npair if case["classes"] == "5" else npair * (npair + 1) // 2
    rng = np.random.default_rng(case["n"])
    k = np.sort(rng.choice(total, size=min(case["n"], total), replace=False))
    if case["classes"] == "5":
        i, j = k // npair, k % npair
    else:
        i = ((np.sqrt(8.0 * k + 1.0) - 1.0) / 2.0).astype(np.int64)
        i += (i + 1) * (i + 2) // 2 <= k
        i -= i * (i + 1) // 2 > k
        j = k - i * (i + 1) // 2
    return np.stack([a[i], b[i], a[j], b[j]], axis=1).astype(np.int32)


def _screened_sample(case, rng, estimate):
    """The sample with every quartet below the 1e-12 screen replaced by a
    surviving one of the same angular momenta."""
    q = _canonical_sample(case)
    keep = estimate(q) >= 1e-12
    l = _shells(case)[q]
    key = ((l[:, 0] * 4 + l[:, 1]) * 4 + l[:, 2]) * 4 + l[:, 3]
    for k in np.unique(key[~keep]):
        good, bad = np.nonzero(keep & (key == k))[0], np.nonzero(~keep & (key == k))[0]
        if len(good):
            q[bad] = q[rng.choice(good, size=len(bad))]
    return np.ascontiguousarray(q)


def _geometric_block(case, rng, basis):
    """A block of nb bra x nk ket significant shell pairs (pair by pair, as
    requests ask for them); the pairs' angular momenta are the same for every
    seed."""
    n = case["n"]
    nb = max(1, int(math.sqrt(n)))
    nk = -(-n // nb)
    l = _shells(case)
    a, b = np.tril_indices(len(l))
    draw_types = np.random.default_rng(n)
    pick = draw_types.integers(0, len(a), size=nb + nk)
    sig = M.significant_pairs(basis)
    skey = l[sig[:, 0]] * 4 + l[sig[:, 1]]
    out = []
    for p in pick:
        rows = sig[skey == l[a[p]] * 4 + l[b[p]]]
        out.append(rows[rng.integers(len(rows))] if len(rows) else (a[p], b[p]))
    out = np.array(out)
    q = np.concatenate([np.repeat(out[:nb], nk, axis=0), np.tile(out[nb:], (nb, 1))], axis=1)
    return np.ascontiguousarray(q[:n], dtype=np.int32)


def _aux_points(case, seed):
    rng = np.random.default_rng(seed)
    lo, hi = math.log(case["exp_lo"]), math.log(case["exp_hi"])
    xi = np.exp(rng.uniform(lo, hi, size=case["n"]))
    # pairs of distributions on the same centre, nearby, and across a molecule
    D = np.where(rng.random(case["n"]) < 0.05, 0.0, rng.uniform(0.0, 12.0, size=case["n"]))
    return xi, D


AUX_NMAX = 6


def prepare(case, seed):
    st = State(case["factor"])
    st.kind = case["kind"]
    rng = np.random.default_rng(seed + 7919)
    if case["kind"] == "aux":
        xi, D = _aux_points(case, seed)
        st.cls = int(case["classes"])
        st.xi, st.D = torch.from_numpy(xi).cuda(), torch.from_numpy(D).cuda()
        st.out = torch.empty((case["n"], AUX_NMAX + 1), dtype=torch.float64, device="cuda")
        return st
    if case["kind"] == "batch":
        st.requests = []
        st.classes = tuple(int(c) for c in case["classes"])
        for m in range(case["mols"]):
            basis = _molecule(case, 1000 * seed + m)
            bid = F.f12int_set_basis(st.ctx, basis)
            q = _geometric_block(case, rng, basis)
            off1 = M.block_offsets(basis, q)
            off = np.stack([off1[:-1] + k * int(off1[-1]) for k in range(len(st.classes))])
            out = torch.empty(int(off1[-1]) * len(st.classes), dtype=torch.float64, device="cuda")
            st.requests.append((bid, q, off, out))
        return st
    basis = _molecule(case, seed)
    st.cls = int(case["classes"])
    st.bid = F.f12int_set_basis(st.ctx, basis)
    q = _quartets(case, seed, basis, lambda q: F.f12int_quartet_estimates(st.ctx, st.bid, st.cls, q))
    off = M.block_offsets(basis, q)
    st.q, st.off = torch.from_numpy(q).cuda(), torch.from_numpy(off[:-1].copy()).cuda()
    st.out = torch.empty(int(off[-1]), dtype=torch.float64, device="cuda")
    return st


def _quartets(case, seed, basis, estimate):
    rng = np.random.default_rng(seed + 7919)
    if case["f"]:
        return _geometric_block(case, rng, basis)
    if not case["d"]:   # a diatomic's whole list is significant
        return _canonical_sample(case)
    return _screened_sample(case, rng, estimate)


def run(state):
    st = state
    if st.kind == "aux":
        F.f12int_aux(st.ctx, st.cls, st.xi, st.D, AUX_NMAX, st.out)
        return st.out
    if st.kind == "batch":
        tickets = [F.f12int_submit(st.ctx, bid, q, st.classes, out, off) for bid, q, off, out in st.requests]
        for t in tickets:
            while not F.f12int_poll(st.ctx, t, 100000):
                pass
        return [r[3] for r in st.requests]
    if st.kind == "mixed":
        F.f12int_compute_class_mixed(st.ctx, st.bid, st.cls, st.q, st.out, st.off, 1e-5)
    elif st.kind == "static":
        F.f12int_compute_class_static(st.ctx, st.bid, st.cls, st.q, st.out, st.off)
    else:
        F.f12int_compute_class(st.ctx, st.bid, st.cls, st.q, st.out, st.off)
    return st.out


# -------------------------------------------------------------------- work --

def work(case):
    """Bytes of the lists, pair data and blocks; flops of the Hermite
    recursion and contraction of each primitive quartet (as the library counts
    them) and 16 multiply-adds per auxiliary function, at the mean over the
    basis's shell quartets."""
    if case["kind"] == "aux":
        return {"bytes": 8.0 * case["n"] * (AUX_NMAX + 3), "flops": 32.0 * case["n"] * (AUX_NMAX + 1)}
    nh = lambda l: (l + 1) * (l + 2) * (l + 3) // 6  # noqa: E731
    nc = lambda l: (l + 1) * (l + 2) // 2  # noqa: E731
    per = (case["s"], case["p"], case["d"], case["f"])
    tot = float(sum(per))
    mean_prim = 0.5 * (case["prim_lo"] + case["prim_hi"])
    flops = values = 0.0
    classes = [int(c) for c in case["classes"]]
    for la in range(4):
        for lb in range(4):
            for lc in range(4):
                for ld in range(4):
                    w = per[la] * per[lb] * per[lc] * per[ld] / tot ** 4
                    block = nc(la) * nc(lb) * nc(lc) * nc(ld)
                    values += w * block * len(classes)
                    for c in classes:
                        e = 2 if c == 5 else 0
                        L = la + lb + lc + ld + e
                        flops += w * (2.0 * (L + 1) * (L + 2) * (L + 3) * (L + 4) / 24 + 32.0 * (L + 1)
                                      + 2.0 * nh(la + lb + e) * nh(lc + ld) * nc(lc) * nc(ld)
                                      + 2.0 * block * nh(la + lb) * (4 if c == 5 else 1))
    nsh = case["atoms"] * tot
    pair_bytes = (nsh * mean_prim) ** 2 * 8.0 * 60
    n = case["n"] * case["mols"]
    return {"bytes": case["mols"] * pair_bytes + n * (24.0 + 8.0 * values), "flops": n * mean_prim ** 4 * flops}


# ------------------------------------------------------------------- exact --
# The definition in numpy: radial derivatives of the basic integral by
# composite Gauss-Legendre quadrature of the kernel's derivatives, Hermite
# integrals by the recursion, and the Hermite expansion of each pair.

def _kernel(factor, cls):
    """Terms {(a, b, g): c} of k(r) = sum c r^a e^{br - gr^2}."""
    if factor == "geminal":
        f = {(a, b, g): c for c, a, b, g in GEMINAL}
    else:
        p = FACTORS[factor]
        f = {(0.0, 0.0, p["mu"]): 1.0, (1.0, 0.0, p["mu"]): 0.5, (p["rho"], p["B"], 0.0): p["c0"]}
        for k in range(p["n"] + 1):
            f[(p["rho"] + 2 * k, p["B"], p["mu"])] = -p["c0"] * p["mu"] ** k / math.factorial(k)

    def prod(x, y):
        out = {}
        for (a, b, g), c in x.items():
            for (a2, b2, g2), c2 in y.items():
                key = (a + a2, b + b2, g + g2)
                out[key] = out.get(key, 0.0) + c * c2
        return out

    if cls == 1:
        return {(-1.0, 0.0, 0.0): 1.0}
    if cls == 2:
        return {(a - 1, b, g): c for (a, b, g), c in f.items()}
    if cls in (3, 5):
        return f
    if cls == 4:
        return prod(f, f)
    d = {}
    for (a, b, g), c in f.items():
        for key, v in (((a - 1, b, g), c * a), ((a, b, g), c * b), ((a + 1, b, g), -2 * c * g)):
            d[key] = d.get(key, 0.0) + v
    return prod(d, d)


def _radial(terms, L, x):
    """x^{2l+2} (D_r^l k)(x), l <= L, D_r = x^-1 d/dx: [L+1, len(x)]."""
    out = np.zeros((L + 1,) + x.shape)
    extra = {}
    for (a, b, g), c in terms.items():
        poly = {0: np.longdouble(c)}              # powers a + j - 2l
        for l in range(L + 1):
            extra.setdefault(l, []).append((a, b, g, dict(poly)))
            nxt = {}
            for j, v in poly.items():
                p = np.longdouble(a) + j - 2 * l
                for dj, w in ((0, v * p), (1, v * b), (2, -2 * v * g)):
                    if w != 0:
                        nxt[j + dj] = nxt.get(j + dj, np.longdouble(0)) + w
            poly = nxt
    for l, fams in extra.items():
        for a, b, g, poly in fams:
            q = np.zeros_like(x)
            for j in range(max(poly, default=0), -1, -1):
                q = q * x + float(poly.get(j, 0))
            out[l] += q * x ** (a + 2) * np.exp(b * x - g * x * x)
    return out


def _scaled_j(L, z):
    """e^{-z} (z^-1 d/dz)^l (sinh z / z), l <= L."""
    j = np.empty((L + 1,) + z.shape)
    big = z > 2.0 * L + 30.0
    zb = np.where(big, z, 1.0)
    iz = 1.0 / zb
    up = [0.5 * iz, 0.5 * (1.0 - iz) * iz * iz]
    for m in range(1, L):
        up.append((up[m - 1] - (2 * m + 1) * up[m]) * iz * iz)
    zs = np.where(big, 0.0, z)
    low = {}
    for m in range(L, max(L - 2, -1), -1):
        t = np.full(z.shape, 1.0 / math.prod(range(1, 2 * m + 2, 2)))
        s = t.copy()
        for k in range(200):
            t = t * zs * zs * (k + m + 1) / ((k + 1) * (2.0 * k + 2 * m + 2) * (2.0 * k + 2 * m + 3))
            s += t
        low[m] = s * np.exp(-zs)
    for m in range(L - 1, 0, -1):
        low[m - 1] = zs * zs * low[m + 1] + (2 * m + 1) * low[m]
    for m in range(L + 1):
        j[m] = np.where(big, up[m], low[m])
    return j


def _hat_g(factor, cls, xi, D, L):
    """hat g_l(xi, D), l <= L, for arrays xi and D: [len, L+1]."""
    terms = _kernel(factor, cls)
    gmax = max(g for _, _, g in terms)
    t, w = np.polynomial.legendre.leggauss(20)
    res = np.empty((len(xi), L + 1))
    order = np.argsort(xi, kind="stable")
    for i0 in range(0, len(xi), 1024):
        idx = order[i0:i0 + 1024]
        x1, d1 = xi[idx], D[idx]
        # panels about the peak in units of each point's width; 40 panels from
        # the lower end, the first in x = h u^4 when it starts at the origin
        wid = 1.0 / np.sqrt(x1 + (gmax if gmax else 0.0))
        lo = np.maximum(0.0, d1 - 9.0 / np.sqrt(x1))
        hi = d1 + 9.0 / np.sqrt(x1)
        npan = max(12, int(np.max((hi - lo) / (1.2 * wid))) + 1)
        npan = min(npan, 60)
        h = (hi - lo) / npan
        acc = np.zeros((L + 1, len(idx)))
        for p in range(npan):
            u = 0.5 * (t[None, :] + 1.0)
            if p == 0:
                x = lo[:, None] + h[:, None] * u ** 4
                wt = h[:, None] * 2.0 * u ** 3 * w[None, :]
            else:
                x = lo[:, None] + h[:, None] * (p + u)
                wt = h[:, None] * 0.5 * w[None, :]
            Fl = _radial(terms, L, x)
            jl = _scaled_j(L, 2.0 * x1[:, None] * d1[:, None] * x)
            e = wt * np.exp(-x1[:, None] * (x - d1[:, None]) ** 2)
            acc += np.sum(Fl * jl * e[None], axis=2)
        for l in range(L + 1):
            res[idx, l] = 4.0 * x1 * (2.0 * x1) ** l * acc[l]
    return res


def _cart(l):
    return [(i, j, l - i - j) for i in range(l, -1, -1) for j in range(l - i, -1, -1)]


def _hermite(i, j, a, b, x):
    """E_t^{ij}, t <= i + j, along one axis with separation x = A - B."""
    p = a + b
    e = {(0, 0): [math.exp(-a * b / p * x * x)]}

    def get(v, t):
        return v[t] if 0 <= t < len(v) else 0.0

    for n in range(1, i + 1):
        v = e[(n - 1, 0)]
        e[(n, 0)] = [get(v, t - 1) / (2 * p) - b / p * x * get(v, t) + (t + 1) * get(v, t + 1) for t in range(n + 1)]
    for m in range(1, j + 1):
        v = e[(i, m - 1)]
        e[(i, m)] = [get(v, t - 1) / (2 * p) + a / p * x * get(v, t) + (t + 1) * get(v, t + 1)
                     for t in range(i + m + 1)]
    return e[(i, j)]


def exact(case, seed):
    if case["kind"] == "aux":
        if case["n"] > 6000:   # the whole array would take minutes
            return None
        xi, D = _aux_points(case, seed)
        return _hat_g(case["factor"], int(case["classes"]), xi, D, AUX_NMAX)
    if case["kind"] != "class" or case["classes"] == "5" or case["d"] or case["f"] or case["n"] > 800:
        return None
    cls = int(case["classes"])
    basis = _molecule(case, seed)
    q = _quartets(case, seed, basis, None)
    po = basis.prim_off
    alpha = [basis.exps[po[s]] for s in range(basis.nshell)]     # one primitive per shell
    coef = [basis.coefs[po[s]] for s in range(basis.nshell)]
    geo = []
    for a, b, c, d in q:
        p, s = alpha[a] + alpha[b], alpha[c] + alpha[d]
        P = (alpha[a] * basis.centers[a] + alpha[b] * basis.centers[b]) / p
        Q = (alpha[c] * basis.centers[c] + alpha[d] * basis.centers[d]) / s
        geo.append((p, s, Q - P))
    xi = np.array([p * s / (p + s) for p, s, _ in geo])
    D = np.array([np.linalg.norm(x) for _, _, x in geo])
    gl = _hat_g(case["factor"], cls, xi, D, 4)
    out = []
    for (a, b, c, d), (p, s, X), g in zip(q, geo, gl):
        la, lb, lc, ld = (int(basis.l[k]) for k in (a, b, c, d))
        L = la + lb + lc + ld
        pre = math.pi ** 2.5 / (math.sqrt(p + s) * p * s) * coef[a] * coef[b] * coef[c] * coef[d]
        memo = {}

        def R(n, t, u, v):
            if t < 0 or u < 0 or v < 0:
                return 0.0
            key = (n, t, u, v)
            if key not in memo:
                if t:
                    r = (t - 1) * R(n + 1, t - 2, u, v) + X[0] * R(n + 1, t - 1, u, v)
                elif u:
                    r = (u - 1) * R(n + 1, t, u - 2, v) + X[1] * R(n + 1, t, u - 1, v)
                elif v:
                    r = (v - 1) * R(n + 1, t, u, v - 2) + X[2] * R(n + 1, t, u, v - 1)
                else:
                    r = g[n]
                memo[key] = r
            return memo[key]

        AB, CD = basis.centers[a] - basis.centers[b], basis.centers[c] - basis.centers[d]
        bra = [[_hermite(i[k], j[k], alpha[a], alpha[b], AB[k]) for k in range(3)] for i in _cart(la)
               for j in _cart(lb)]
        ket = [[_hermite(i[k], j[k], alpha[c], alpha[d], CD[k]) for k in range(3)] for i in _cart(lc)
               for j in _cart(ld)]
        for ex, ey, ez in bra:
            for fx, fy, fz in ket:
                tot = 0.0
                for t, et in enumerate(ex):
                    for u, eu in enumerate(ey):
                        for v, ev in enumerate(ez):
                            sgn = -1.0 if (t + u + v) & 1 else 1.0
                            for t2, ft in enumerate(fx):
                                for u2, fu in enumerate(fy):
                                    for v2, fv in enumerate(fz):
                                        tot += sgn * et * eu * ev * ft * fu * fv * R(0, t + t2, u + u2, v + v2)
                out.append(pre * tot)
        assert L <= 4
    return np.array(out)
