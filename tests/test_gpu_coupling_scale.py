"""The photon tiring term P : grad v at scales of E and v where |grad E|^2 or its products with
grad v leave the FP64 range or come near its ends: P is linear in E and in grad v, and n = grad E /
|grad E| has no scale, so the term divided by both scales is that of scale one.

Tolerance: two evaluations of |grad E|^2, f and n with FP64 roundings (1e-14 of the largest value),
but 2^-1074 / |grad E|^2 where that is subnormal (below 2^-1022), in n twice."""
import numpy as np
import pytest

from gpu_util import torch_cuda, library, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walls", [[(1, 1)] * 3, [(0, 0), (1, 1), (0, 0)]])
@pytest.mark.parametrize("shape", [(7, 9, 10), (11, 12), (40,)])
def test_tiring_term_has_the_scales_of_its_factors(shape, walls):
    torch = torch_cuda()
    fld = library()
    nd = len(shape)
    rng = np.random.default_rng(nd)
    E = 1.0 + 0.3 * rng.uniform(0, 1, shape)
    v = rng.uniform(-1, 1, (nd,) + shape)
    one = dev(torch, np.ones(shape))
    hd = fld.Handle(shape, (1.0,) * nd, tuple(walls[:nd]))
    consts, op = fld.make_consts(1.0, 1.0, 5.0 / 3.0, 1.0), fld.make_opacity((0, 1.0, 0.0, 0.0))

    def tiring(se, sv):
        pt = torch.zeros(shape, dtype=torch.float64, device="cuda")
        hd.coupling(consts, op, dev(torch, E * se), one, one, None, dev(torch, v * sv), None, None,
                    None, None, pt)
        assert hd.status() == fld.FLD_OK
        return host(pt) / se / sv

    want = tiring(1.0, 1.0)
    top = np.max(np.abs(want))
    # the smallest |grad E|^2 of these fields is above 2^-29
    for e in (-515, -511, -505, -400, -200, -100, 100, 200, 400, 500):
        tol = 1e-14 + (2.0 ** (-1074 - 2 * e + 30) if 2 * e - 29 < -1022 else 0.0)
        for u in (0, 60, -60):
            got = tiring(2.0 ** e, 2.0 ** u)
            assert np.all(np.isfinite(got)), (e, u)
            assert np.max(np.abs(got - want)) <= tol * top, (e, u)
    hd.close()
