"""log10 and 10^v of the opacity tables (csrc/logtab.cuh) through fld_limiter in the diffusion limit,
D = c / (3 kappa rho), where their table-driven reductions can go wrong: arguments at the edges of
the tables' rows and binades, next to one, subnormal, and powers where the library's functions
take over.

Tolerances, in the reference's extended precision. 10^v from a table of one value is v itself, so D
carries one unit of the last place of 10^v (2.3e-16), kappa0 times it, c/3, and the division (1.2e-16
each): 6e-16; the library's 10^v has two units (8e-16). log10: with log10 kappa = log10 T on one
interval from -1 to 1, kappa = T up to ln 10 times the absolute errors of log10 T (below 1.2e-16),
of the fraction and of the interpolation (1.2e-16 each), 8.3e-16, and the 6e-16 above. Subnormal T on
a table of slope 1/100 from -330 to 330: ln 10 / 100 times the 1.2e-13 of a library log10 near -320
(two units), of the coordinate (2.3e-16 of 660) and of its product, 3.5e-15, and the 6e-16."""
import numpy as np
import pytest

from gpu_util import torch_cuda, library, dev, host

pytestmark = pytest.mark.gpu
X = np.longdouble


def _kappa(torch, fld, T, kappa0, table, grid):
    """kappa of every T (rho = 1) from D = c / (3 kappa), c = 3."""
    n = T.size
    one = dev(torch, np.ones(n))
    hd = fld.Handle((n,), (1.0,), ((0, 0),), limiter=fld.LIMITER_DIFFUSION)
    D = torch.zeros(n, dtype=torch.float64, device="cuda")
    t = np.asarray(table, dtype=np.float64)
    hd.limiter(fld.make_consts(3.0, 1.0, 5.0 / 3.0, 1.0),
               fld.make_opacity((fld.OPACITY_TABLE, kappa0, t, grid), dev(torch, t)), one, one,
               dev(torch, T), None, D, None)
    assert hd.status() == fld.FLD_OK
    hd.close()
    return 1 / host(D).astype(X)


def _powers():
    step = np.log10(2.0) / 128
    v = [0.0, 1e-20, -1e-20, 1e-8, 0.5, -0.5, 1.0, 17.3, -123.4, 299.999, -299.999, 300.0, -300.0,
         301.7, -304.9]
    for k in (-40000, -129, -128, -1, 1, 63, 64, 127, 128, 12345, 127000):
        v += [k * step, (k + 0.5) * step, np.nextafter((k + 0.5) * step, 0.0)]
    return [x for x in v if abs(x) < 305]


def test_powers_of_ten():
    torch = torch_cuda()
    fld = library()
    for v in _powers():
        # kappa0 keeps kappa within the range
        kappa0 = 10.0 ** -round(v) if abs(v) > 100 else 1.0
        got = _kappa(torch, fld, np.ones(4), kappa0, np.full((2, 2), v), (-1.0, 1.0, -1.0, 1.0))
        want = X(kappa0) * X(10) ** X(v)
        assert np.max(np.abs(got / want - 1)) <= (8e-16 if abs(v) > 299.9 else 6e-16), v


def test_logarithms():
    torch = torch_cuda()
    fld = library()
    rng = np.random.default_rng(5)
    rows = np.concatenate([1.0 + np.arange(128) / 128.0, 1.0 + (np.arange(128) + 0.5) / 128.0])
    T = np.concatenate([rows, np.nextafter(rows, 0.0), np.nextafter(rows, 9.0), 1.0 + 2.0 ** -np.arange(1, 53),
                        1.0 - 2.0 ** -np.arange(1, 54), 2.0 ** np.arange(-3.0, 4.0),
                        np.nextafter(2.0 ** np.arange(-3.0, 4.0), 0.0), 10.0 ** rng.uniform(-1, 1, 20000)])
    T = T[(T > 0.1) & (T < 10.0)]
    table = [[-1.0, -1.0], [1.0, 1.0]]
    got = _kappa(torch, fld, T, 1.0, table, (-1.0, 1.0, -1.0, 2.0))
    assert np.max(np.abs(got / T - 1)) <= 1.5e-15


def test_subnormal_arguments_and_table_ends():
    torch = torch_cuda()
    fld = library()
    T = np.array([5e-324, 1e-323, 1e-320, 1e-310, 2.2250738585072014e-308, 2.3e-308, 1e-300])
    table = [[0.0, 0.0], [6.6, 6.6]]
    got = _kappa(torch, fld, T, 1.0, table, (-1.0, 1.0, -330.0, 660.0))
    lg = np.log2(T.astype(X)) * np.log10(X(2))
    assert np.max(np.abs(got / X(10) ** ((lg + 330) / 100) - 1)) <= 4.1e-15
    # beyond the table its edge values hold, exactly
    got = _kappa(torch, fld, np.array([1e-9, 0.1, 1e9, 1e300]), 1.0, [[0.0, 0.0], [1.0, 1.0]],
                 (-1.0, 1.0, -1.0, 2.0))
    assert np.max(np.abs(got / np.array([1.0, 1.0, 10.0, 10.0]) - 1)) <= 6e-16
