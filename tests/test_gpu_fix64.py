"""The limiter and the coupling terms with their divisions, roots and differences in mixed integer,
FP32 and FP64 arithmetic (csrc/fix64.cuh), against extended precision cell by cell: smooth fields,
neighbours many binades apart, constant fields (zero gradient), signed

Tolerances (u = 2^-53): kappa rho takes at most 9 roundings, a = kappa rho E one more, |grad E|
3, the limiter's numerator and denominator 4, the quotient and the products by c E 3: below
25 u = 2.8e-15 in D, plus the difference's own rounding, 18 units of 2^-57 of its largest operand
per axis, which enters D with a weight of at most one relative to |grad E|. The coupling terms
add products and a sum of 9 signed terms, bounded against the sum of their magnitudes."""
import numpy as np
import pytest

from oracle import fld as O
from paper_2503_02764_gb300 import inputs as I
from gpu_util import torch_cuda, library, dev, host

pytestmark = pytest.mark.gpu
L = np.longdouble
BC = [((0, 0), (1, 2), (2, 1)), ((2, 2), (0, 0), (1, 1))]


def _fields(kind, shape, seed):
    rng = np.random.default_rng(seed)
    if kind == "constant":
        return np.full(shape, 3.0), np.full(shape, 0.7), np.full(shape, 2.0)
    if kind == "binades":
        return tuple(10.0 ** rng.uniform(-e, e, shape) for e in (7, 3, 2))
    if kind == "far":                         # outside the FP32 range
        return tuple(10.0 ** rng.uniform(-e, e, shape) for e in (40, 25, 3))
    return (1.0 + 0.1 * rng.uniform(-1, 1, shape), 1.0 + rng.uniform(0, 1, shape),
            1.0 + rng.uniform(0, 1, shape))


def _grad(E, h, bc, Eb):
    """gradient in extended precision and the size of its rounding"""
    g, err = [], []
    for d in range(E.ndim):
        a = E.ndim - 1 - d
        P = O.pad_ghosts(E.astype(L), d, bc, {k: v.astype(L) for k, v in Eb.items()}, 2)
        n = E.shape[a]
        v = [np.take(P, range(q, q + n), axis=a) for q in (0, 1, 3, 4)]
        g.append((v[0] - 8 * v[1] + 8 * v[2] - v[3]) / (12 * L(h[d])))
        # the ghost 2 E_b - E is itself rounded to FP64: one more unit of the operands
        err.append(sum(np.abs(q) for q in v) * L(8 * 2.0 ** -53 + 18 * 2.0 ** -57) / (12 * L(h[d])))
    return g, err


@pytest.mark.parametrize("op", [(0, 3.0, 0.0, 0.0), (1, 2.0, 1.0, -3.5)])
@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("kind", ["smooth", "binades", "constant", "far"])
@pytest.mark.parametrize("bc", BC)
def test_limiter_and_coupling_roundings(bc, kind, mode, op):
    torch = torch_cuda()
    fld = library()
    shape, h, c = (7, 10, 37), (0.5, 0.25, 1.0), 2.0
    E, rho, T = _fields(kind, shape, 3 + mode)
    Eb = {(d, s): np.take(E, 0 if s == 0 else -1, axis=2 - d).copy()
          for d in range(3) for s in (0, 1) if bc[d][s] == 2}
    rng = np.random.default_rng(9)
    v = rng.uniform(-1, 1, (3,) + shape) * 10.0 ** rng.uniform(-3, 3, (3,) + shape)
    v[:, 2] = 0.0
    hd = fld.Handle(shape, h, bc, limiter=mode)
    k = fld.make_consts(c, 1.0, 5.0 / 3.0, 1.0)
    out = {n: torch.empty(E.size * m, dtype=torch.float64, device="cuda")
           for n, m in (("D", 1), ("lam", 1), ("F", 3), ("fr", 3), ("f", 1), ("vfr", 1), ("pt", 1))}
    ebc = dev(torch, I.pack_dirichlet(shape, bc, Eb))
    ops = fld.make_opacity(op)
    hd.limiter(k, ops, dev(torch, E), dev(torch, rho), dev(torch, T), ebc, out["D"], out["lam"])
    hd.coupling(k, ops, dev(torch, E), dev(torch, rho), dev(torch, T), ebc, dev(torch, v),
                out["F"], out["fr"], out["f"], out["vfr"], out["pt"])
    assert hd.status() == 0
    got = {n: host(t).astype(L).reshape((-1,) + shape) for n, t in out.items()}
    El, rl, Tl = E.astype(L), rho.astype(L), T.astype(L)
    kr = L(op[1]) * rl if op[0] == 0 else L(op[1]) * rl * rl / (Tl ** 3 * np.sqrt(Tl))
    g, ge = _grad(E, h, bc, Eb)
    gn = np.sqrt(sum(x * x for x in g))
    ga = np.sqrt(sum(x * x for x in ge))                 # rounding of |grad E|
    R = gn / (kr * El)
    lam = (2 + R) / (6 + 3 * R + R * R) if mode == 0 else np.full(shape, L(1) / 3) if mode == 1 \
        else np.where(R <= 1.5, 2 / (3 + np.sqrt(9 + 12 * R * R)), 1 / (1 + R + np.sqrt(1 + 2 * R)))
    rel = L(25 * 2.0 ** -53) + (0 if mode == 1 else ga / np.maximum(gn, ga + L(1e-300)))
    D = c * lam / kr
    assert np.all(np.abs(got["D"][0] - D) <= rel * D)
    assert np.all(np.abs(got["lam"][0] - lam) <= rel * lam)
    f = lam + lam * lam * R * R
    rel = L(30 * 2.0 ** -53) + 2 * ga / np.maximum(gn, ga + L(1e-300))
    assert np.all(np.abs(got["f"][0] - f) <= rel * f)
    vf = L(0)
    for d in range(3):
        assert np.all(np.abs(got["F"][d] + D * g[d]) <= D * (rel * np.abs(g[d]) + ge[d]))
        assert np.all(np.abs(got["fr"][d] + lam * g[d]) <= lam * (rel * np.abs(g[d]) + ge[d]))
        vf = vf - v[d].astype(L) * lam * g[d]
    size = sum(np.abs(v[d]) * lam * (np.abs(g[d]) * rel + ge[d]) for d in range(3))
    assert np.all(np.abs(got["vfr"][0] - vf) <= size + L(1e-300))
    if kind in ("smooth", "constant"):
        vbc = tuple((0, 0) if b[0] == 0 else (1, 1) for b in bc)
        n = [np.where(gn > 0, x / np.where(gn > 0, gn, 1), 0) for x in g]
        pt, size = L(0), L(0)
        for a in range(3):
            gv, gve = _grad(v[a], h, vbc, {})
            for b in range(3):
                Pab = ((0.5 * (1 - f) if a == b else 0) + 0.5 * (3 * f - 1) * n[a] * n[b]) * El
                pt = pt + Pab * gv[b]
                size = size + El * (np.abs(gv[b]) * rel * 4 + gve[b])
        assert np.all(np.abs(got["pt"][0] - pt) <= size)
    hd.close()
