"""3D FP32 smoothing and transfers at the edges of their tiles: rows of whole 16-byte chunks (the
z-marching sweep, its rows' values kept in registers: 32 x 16 tiles, chunks of planes) and others
(half sweeps, restriction with four lanes a coarse cell), extents one cell from a tile's, two planes
and fewer planes than the march keeps, every wall kind, equal and unequal cell sizes (the two forms
of the FP64 residual).

The default smoother must end as the out-of-place half sweeps (smoother 1) do, whose updates are
the same: at most one cycle more. The solve stops at 1e-12 of ||b||_2, the fields vary by less
than a factor 2 and ||A^-1|| <= 1: the max norm over at most 4e4 cells is within 1e-12 * 200."""
import numpy as np
import pytest

from oracle import fld as O
from paper_2503_02764_gb300 import inputs as I
from gpu_util import torch_cuda, library, dev, host, maxrel

pytestmark = pytest.mark.gpu

P, N, D, M = (0, 0), (1, 1), (2, 2), (1, 2)
CASES = [((12, 34, 64), (P, P, P)), ((2, 18, 36), (M, D, P)), ((3, 15, 32), (N, M, D)),
         ((40, 16, 28), (D, N, M)), ((9, 33, 16), (P, N, N)), ((11, 13, 19), (M, N, D)),
         ((7, 20, 30), (P, P, M)), ((2, 3, 50), (P, D, N))]


@pytest.mark.parametrize("h", [(1.0, 1.0, 1.0), (1.0, 0.8, 1.3)])
@pytest.mark.parametrize("shape,bc", CASES)
def test_default_smoother_matches_half_sweeps_and_oracle(shape, bc, h):
    torch = torch_cuda()
    fld = library()
    rng = np.random.default_rng(sum(shape))
    Dc = I.lognormal(rng, shape, 0.5, 3.0)
    E = 1.0 + rng.uniform(0, 1, shape)
    Eb = {(d, s): 1.0 + rng.uniform(0, 1, tuple(n for a, n in enumerate(shape) if a != 2 - d))
          for d in range(3) for s in (0, 1) if bc[d][s] == 2}
    packed = I.pack_dirichlet(shape, bc, Eb)
    ebc = dev(torch, packed) if packed.size else None
    hd = fld.Handle(shape, h, bc, precision=1, tol=1e-12, max_cycles=80)
    for dt in (0.5, 8.0):
        xo = O.diffuse(E, Dc, h, bc, Eb, dt, method="splu")
        for opts in (dict(nu1=2, nu2=2), dict(nu1=1, nu2=1, inner=3)):
            cyc = {}
            for sm in (0, 1):
                hd.set_opts(precision=1, tol=1e-12, max_cycles=80, smoother=sm, **opts)
                x = dev(torch, E)
                st = hd.diffuse(dt, dev(torch, Dc), ebc, x)
                cyc[sm] = st["cycles"]
                assert maxrel(host(x).reshape(shape), xo) < 2e-10, (sm, dt)
            assert cyc[0] <= cyc[1] + 1, cyc
    hd.close()
