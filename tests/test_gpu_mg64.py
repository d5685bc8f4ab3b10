"""The FP64 V-cycle on stored coefficients (csrc/k_mg64.cu): the solve against the oracle at the
edges of the kernels' tiles (32 pairs x 8 rows; 32 or 16 cells a row), on odd and even extents,
every wall kind, out-of-place smoothing, both face means, and the double-size levels whose
coefficients share the mixed modes' buffers (an FP64 solve between two mixed ones).

Tolerance: at tol 1e-13 the relative residual bounds ||x - A^-1 b|| / ||b|| by 1e-13
(||A^-1||_2 <= 1), and the max norm over at most 4e4 cells by sqrt(4e4) = 200 times that of the
mean; the fields vary by less than a factor 2, so 1e-10 holds with margin and 1e-11 is used."""
import numpy as np
import pytest

from oracle import fld as O
from paper_2503_02764_gb300 import inputs as I
from gpu_util import torch_cuda, library, dev, host, maxrel

pytestmark = pytest.mark.gpu

P, N, D = (0, 0), (1, 1), (2, 2)
CASES = [
    ((64, 66), (P, P)), ((33, 31), (N, D)), ((17, 130), ((1, 2), (2, 1))), ((9, 34), (P, N)),
    ((16, 18, 66), (P, P, P)), ((9, 15, 33), (P, N, D)), ((12, 17, 64), ((2, 1), (1, 2), P)),
    ((31, 8, 16), (D, D, D)), ((5, 40, 35), (N, P, N)), ((2, 2, 50), (P, D, N)),
]


def _case(shape, bc, seed):
    rng = np.random.default_rng(seed)
    Dc = I.lognormal(rng, shape, 0.7, 3.0)
    E = 1.0 + rng.uniform(0, 1, shape)
    Eb = {}
    for d in range(len(shape)):
        for s in (0, 1):
            if bc[d][s] == 2:
                fs = tuple(n for a, n in enumerate(shape) if a != len(shape) - 1 - d)
                Eb[(d, s)] = 1.0 + rng.uniform(0, 1, fs)
    return Dc, E, Eb


@pytest.mark.parametrize("smoother", [0, 1])
@pytest.mark.parametrize("shape,bc", CASES)
def test_fp64_solve_matches_oracle(shape, bc, smoother):
    torch = torch_cuda()
    fld = library()
    h = tuple(1.0 + 0.25 * d for d in range(len(shape)))
    Dc, E, Eb = _case(shape, bc, sum(shape))
    packed = I.pack_dirichlet(shape, bc, Eb)
    ebc = dev(torch, packed) if packed.size else None
    hd = fld.Handle(shape, h, bc, tol=1e-13, max_cycles=100, smoother=smoother)
    for dt, mean, name in ((3.0, fld.FACE_ARITH, "arith"), (20.0, fld.FACE_HARM, "harm")):
        xo = O.diffuse(E, Dc, h, bc, Eb, dt, face_mean=name, method="splu")
        for prec in (fld.PREC_FP64, fld.PREC_MIXED, fld.PREC_FP64):
            hd.set_opts(precision=prec, tol=1e-13, max_cycles=100, smoother=smoother,
                        face_mean=mean)
            x = dev(torch, E)
            st = hd.diffuse(dt, dev(torch, Dc), ebc, x)
            assert st["rel_resid"] <= 1e-13
            assert maxrel(host(x).reshape(shape), xo) < 1e-11, (prec, dt)
    hd.close()
