"""Quotients and square roots of the FP64 limiter (csrc/fix64.cuh) next to a power of two, where the
FP32 head of the approximation and the result may lie in different binades: through fld_limiter,
D = c / (3 kappa rho) in the diffusion limit, and D = c E (2 a + g) / (3 a (2 a + g) + g^2), a = kappa
rho E, g = |grad E|, where a is so small that D follows 1 / g.

Tolerance: c / 3 is 1 exactly (c = 3), kappa rho is rho, so that D is one quotient: half a unit of the
last place and the 2^-61 of the approximation, 1.2e-16. The other form rounds |grad E|^2 (exactly as
numpy does, which the reference takes), its root, 2 a + g, the denominator, the quotient and its
product with c E: six half units, 6.7e-16."""
import numpy as np
import pytest

from gpu_util import torch_cuda, library, dev, host

pytestmark = pytest.mark.gpu
X = np.longdouble


@pytest.mark.parametrize("e", [-30, -1, 0, 1, 20])
def test_quotients_next_to_powers_of_two(e):
    torch = torch_cuda()
    fld = library()
    i = np.arange(-2000, 2001)
    rho = np.concatenate([2.0 ** e * (1.0 + i * 2.0 ** -k) for k in (23, 24, 25, 27, 30, 40, 52)]
                         + [2.0 ** e * (1.0 + np.random.default_rng(1).uniform(-1, 1, 4000) * 2.0 ** -21)])
    n = rho.size
    one, D = dev(torch, np.ones(n)), torch.zeros(n, dtype=torch.float64, device="cuda")
    hd = fld.Handle((n,), (1.0,), ((0, 0),), limiter=fld.LIMITER_DIFFUSION)
    hd.limiter(fld.make_consts(3.0, 1.0, 5.0 / 3.0, 1.0), fld.make_opacity((0, 1.0, 0.0, 0.0)), one,
               dev(torch, rho), None, None, D, None)
    assert np.max(np.abs(host(D).astype(X) * rho.astype(X) - 1)) <= 1.2e-16
    hd.close()


@pytest.mark.parametrize("e", [-20, 0, 7])
def test_roots_next_to_powers_of_two(e):
    torch = torch_cuda()
    fld = library()
    n, kappa, c = 16, 1e-18, 1.0
    consts, op = fld.make_consts(c, 1.0, 5.0 / 3.0, 1.0), fld.make_opacity((0, kappa, 0.0, 0.0))
    one = dev(torch, np.ones(n))
    hd = fld.Handle((n,), (1.0,), ((1, 1),))
    D = torch.zeros(n, dtype=torch.float64, device="cuda")
    worst = 0.0
    for k in (22, 23, 24, 25, 26, 28, 34):
        for i in range(-12, 13):
            s = 2.0 ** e * (1.0 + i * 2.0 ** -k)         # E = s (q + 1): exact, and its differences
            E = s * np.arange(1, n + 1)
            hd.limiter(consts, op, dev(torch, E), one, None, None, D, None)
            g = (12.0 * s) * (1.0 / 12.0)
            g2 = X(np.float64(g * g))
            a = X(kappa) * E.astype(X)
            num = 2 * a + np.sqrt(g2)
            want = X(c) * E * num / (3 * a * num + g2)
            worst = max(worst, float(np.max(np.abs(host(D) / want - 1)[2:-2])))
    assert worst <= 6.7e-16
    hd.close()
