"""2D levels with each side of the V-cycle in one launch (csrc/k_tile2d.cu) and the 2D FP64
residual (k_resid64.cu): extents around the tiles' (32 x 16, 64 x 32; 32 x 8 for the residual), odd
and even, every wall kind, sweep counts that give every halo width (an uneven split, none before or
none after the coarse correction), several cycles per refinement step, both prolongations.

The V-cycle must contract like the half-sweep one (smoother 1, out of place, the same updates in
another order of launches): at most one cycle more, and the same end where that one diverges or
stops at its limit (few sweeps on odd extents and a stiff step). A solve that converges stops at
1e-12 of ||b||_2; the fields vary by less than a factor 2 and ||A^-1|| <= 1, so with at most 6e4
cells the max norm is within 1e-12 * sqrt(6e4) < 3e-10."""
import numpy as np
import pytest

from oracle import fld as O
from paper_2503_02764_gb300 import inputs as I
from gpu_util import torch_cuda, library, dev, host, maxrel

pytestmark = pytest.mark.gpu

P, N, D, M = (0, 0), (1, 1), (2, 2), (1, 2)
SHAPES = [((64, 66), (P, P)), ((33, 65), (N, D)), ((31, 129), (M, N)), ((17, 34), (D, P)),
          ((200, 280), (P, M)), ((24, 1000), (N, N)), ((5, 40), (D, D)), ((40, 2), (P, P))]
OPTS = [dict(nu1=2, nu2=2), dict(nu1=1, nu2=0, inner=3), dict(nu1=0, nu2=3),
        dict(nu1=4, nu2=1, inner=2, prolong=1)]


@pytest.mark.parametrize("opts", OPTS)
@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("shape,bc", SHAPES)
def test_tile2d_solve_matches_oracle(shape, bc, precision, opts):
    torch = torch_cuda()
    fld = library()
    h = (1.0, 0.8)
    rng = np.random.default_rng(sum(shape))
    Dc = I.lognormal(rng, shape, 0.5, 4.0)
    E = 1.0 + rng.uniform(0, 1, shape)
    Eb = {(d, s): 1.0 + rng.uniform(0, 1, shape[0] if d == 0 else shape[1])
          for d in range(2) for s in (0, 1) if bc[d][s] == 2}
    packed = I.pack_dirichlet(shape, bc, Eb)
    ebc = dev(torch, packed) if packed.size else None
    hd = fld.Handle(shape, h, bc, precision=precision, tol=1e-12, max_cycles=80)
    for dt in (1.0, 40.0):
        xo = O.diffuse(E, Dc, h, bc, Eb, dt, method="splu")
        cyc, status = {}, {}
        for sm in (0, 1):
            hd.set_opts(precision=precision, tol=1e-12, max_cycles=80, smoother=sm, **opts)
            x = dev(torch, E)
            st = hd.diffuse(dt, dev(torch, Dc), ebc, x, raise_on_error=False)
            cyc[sm], status[sm] = st["cycles"], st["status"]
            if st["status"] == 0:
                assert maxrel(host(x).reshape(shape), xo) < 3e-10, (sm, dt)
        assert status[0] == status[1] and cyc[0] <= cyc[1] + 1, (status, cyc)
    hd.close()
