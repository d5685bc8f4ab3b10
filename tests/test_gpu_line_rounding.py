"""The rounding of the one-launch 1D solve (csrc/k_line.cu) on stiff lines with walls, where nothing
in its reduction cancels: against the system solved in extended precision (Thomas algorithm with
two steps of refinement).

Tolerance: the kernel's operations restated on the CPU differ from 113-bit solutions by at most
1.04e-15 relative in any cell, over lines of 32 to 4096 cells, K from 0.03 to 3e4 and every kind of
wall; four times that. The solve's own stopping rule is not what is tested: one reduction."""
import numpy as np
import pytest

from paper_2503_02764_gb300 import inputs as I
from gpu_util import torch_cuda, library, dev, host

pytestmark = pytest.mark.gpu
X = np.longdouble


def _solve(w, diag, b):
    n = b.size
    x = np.zeros(n, dtype=X)
    for _ in range(3):
        r = b - diag * x
        r[:-1] += w * x[1:]
        r[1:] += w * x[:-1]
        c, y = np.zeros(n, dtype=X), np.zeros(n, dtype=X)
        m = diag[0]
        y[0] = r[0] / m
        for i in range(1, n):
            c[i] = w[i - 1] / m
            m = diag[i] - w[i - 1] * c[i]
            y[i] = (r[i] + w[i - 1] * y[i - 1]) / m
        for i in range(n - 2, -1, -1):
            y[i] += c[i + 1] * y[i + 1]
        x = x + y
    return x


@pytest.mark.parametrize("bc", [(1, 1), (2, 2), (1, 2)])
@pytest.mark.parametrize("K", [32.0, 32768.0])
@pytest.mark.parametrize("n", [33, 257, 1000, 4096])
def test_stiff_line_is_solved_to_rounding(n, K, bc):
    torch = torch_cuda()
    fld = library()
    rng = np.random.default_rng(n + bc[0])
    D, E = 0.5 + rng.uniform(0, 1, n), 1.0 + 0.5 * rng.uniform(0, 1, n)
    Eb = {(0, s): np.array(1.25 + 0.25 * s) for s in (0, 1) if bc[s] == 2}
    packed = I.pack_dirichlet((n,), (bc,), Eb)
    k = X(K) * D.astype(X)
    w = (k[1:] + k[:-1]) / 2
    diag, b = np.ones(n, dtype=X), E.astype(X)
    diag[:-1] += w
    diag[1:] += w
    for (_, s), v in Eb.items():
        i = 0 if s == 0 else n - 1
        diag[i] += 2 * k[i]
        b[i] += 2 * k[i] * X(float(v))
    x = _solve(w, diag, b)
    hd = fld.Handle((n,), (1.0,), (bc,), tol=1e-9, max_cycles=1)
    Ed = dev(torch, E)
    st = hd.diffuse(K, dev(torch, D), dev(torch, packed) if packed.size else None, Ed)
    assert st["cycles"] == 1
    assert float(np.max(np.abs((host(Ed) - x) / x))) <= 4.2e-15
    hd.close()
