"""The composite grid on stored rows (csrc/k_amr.cu) at the edges of its tiles and boxes: odd
block extents, boxes one cell from a wall and spanning axes of every wall kind, 1D to 3D, both
precisions of the coarse correction, and a stiff step whose corrections need several V-cycles.

Tolerance: the solve stops at 1e-13 of ||b||_2 in the volume-weighted norm up to the factor
2^nd between the grids' volumes; the fields vary by less than a factor 2, so with at most 2e4
unknowns the max norm stays within 1e-13 * sqrt(8 * 2e4) < 1e-10."""
import numpy as np
import pytest

from oracle import amr as A
from paper_2503_02764_gb300 import inputs as I
from gpu_util import torch_cuda, library, dev, host, maxrel

pytestmark = pytest.mark.gpu

P, N, D, M = (0, 0), (1, 1), (2, 2), (1, 2)
CASES = [
    ((70,), (M,), (1,), (69,), 4.0), ((40,), (P,), (0,), (40,), 4.0),
    ((19, 33), (N, D), (1, 1), (32, 18), 3.0), ((17, 66), (P, M), (0, 3), (66, 12), 3.0),
    ((12, 13, 17), (D, N, P), (1, 1, 1), (16, 12, 11), 2.0),
    ((10, 9, 34), (P, M, P), (0, 2, 3), (34, 7, 8), 2.0),
    ((10, 12, 16), (M, P, N), (4, 0, 2), (9, 12, 9), 500.0),
]


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("shape,bc,lo,hi,dt", CASES)
def test_amr_rows_match_oracle(shape, bc, lo, hi, dt, precision):
    torch = torch_cuda()
    fld = library()
    nd = len(shape)
    h = tuple(1.0 + 0.2 * d for d in range(nd))
    rng = np.random.default_rng(sum(shape) + nd)
    fine = tuple(2 * (hi[nd - 1 - a] - lo[nd - 1 - a]) for a in range(nd))
    Dc, Df = I.lognormal(rng, shape, 0.6, 3.0), I.lognormal(rng, fine, 0.6, 6.0)
    Ec, Ef = 1.0 + rng.uniform(0, 1, shape), 1.0 + rng.uniform(0, 1, fine)
    Eb = {(d, s): 1.0 + rng.uniform(0, 1, tuple(n for a, n in enumerate(shape) if a != nd - 1 - d))
          for d in range(nd) for s in (0, 1) if bc[d][s] == 2}
    G = A.Composite(shape, h, bc, lo, hi)
    xc, xf = A.diffuse(G, Ec, Ef, Dc, Df, Eb, dt)
    packed = I.pack_dirichlet(shape, bc, Eb)
    am = fld.Amr(shape, h, bc, lo, hi, precision=precision, tol=1e-13, max_cycles=100)
    Ecd, Efd = dev(torch, Ec), dev(torch, Ef)
    st = am.diffuse(dt, dev(torch, Dc), dev(torch, Df), dev(torch, packed) if packed.size else None,
                    Ecd, Efd, raise_on_error=False)
    assert st["status"] == 0, st
    assert maxrel(host(Efd).reshape(fine), xf) < 1e-10
    assert maxrel(host(Ecd).reshape(shape), xc) < 1e-10
    am.close()
