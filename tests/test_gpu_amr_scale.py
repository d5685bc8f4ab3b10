"""A composite solve does not depend on the units of E: the fields scaled by a power of two, down to
where FP32 holds no residual and up to where it overflows, take the same cycles to the same
fields, bit for bit after the scale, in every precision of the coarse correction (all operations
are linear in E and a power of two is exact, so that the tolerance is zero)."""
import numpy as np
import pytest

from paper_2503_02764_gb300 import inputs as I
from gpu_util import torch_cuda, library, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("shape", [(20, 24), (12, 14, 16)])
def test_scaled_fields_scale_the_solution(shape, precision):
    torch = torch_cuda()
    fld = library()
    nd = len(shape)
    rng = np.random.default_rng(nd)
    lo, hi = (3,) * nd, tuple(n - 4 for n in reversed(shape))
    fine = tuple(2 * (hi[nd - 1 - a] - lo[nd - 1 - a]) for a in range(nd))
    bc = ((1, 2),) + ((1, 1),) * (nd - 1)
    Dc, Df = (dev(torch, I.lognormal(rng, s, 0.6, 4.0)) for s in (shape, fine))
    Ec, Ef = 1.0 + rng.uniform(0, 1, shape), 1.0 + rng.uniform(0, 1, fine)
    face = 1.0 + rng.uniform(0, 1, shape[:-1])
    am = fld.Amr(shape, (1.0,) * nd, bc, lo, hi, precision=precision, tol=1e-12, max_cycles=100)

    def solve(scale):
        x, y = dev(torch, Ec * scale), dev(torch, Ef * scale)
        st = am.diffuse(20.0, Dc, Df, dev(torch, face * scale), x, y, raise_on_error=False)
        return st["status"], st["cycles"], host(x) / scale, host(y) / scale

    want = solve(1.0)
    assert want[0] == fld.FLD_OK
    for e in (-150, -110, 110, 200):
        got = solve(2.0 ** e)
        assert got[:2] == want[:2], e
        assert np.array_equal(got[2], want[2]) and np.array_equal(got[3], want[3]), e
    am.close()
