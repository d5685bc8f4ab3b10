"""The one-launch 1D substep, solve and wave stage (csrc/k_line.cu, k_wave1d.cu) at the edges of
their blocks: lines shorter than the cluster, one cell more and less than its blocks hold, the
longest line it takes and the first one past it, every wall kind.

Tolerance: FP64 arithmetic throughout; the solve stops at 1e-13 of ||b||_2, and with fields
that vary by less than a factor 2 and ||A^-1|| <= 1 the max norm stays within sqrt(n) of that:
1e-13 * sqrt(8193) < 1e-11. T carries E's error over the heat capacity, here of order one."""
import numpy as np
import pytest

from oracle import fld as O
from oracle import rmhd1d as W
from paper_2503_02764_gb300 import inputs as I
from gpu_util import torch_cuda, library, dev, host, maxrel

pytestmark = pytest.mark.gpu

SIZES = [2, 3, 7, 8, 9, 31, 32, 33, 255, 257, 1000, 8191, 8192, 8193]
WALLS = [(0, 0), (1, 1), (2, 2), (1, 2)]


@pytest.mark.parametrize("bc", WALLS)
@pytest.mark.parametrize("n", SIZES)
def test_line_matches_oracle(n, bc):
    torch = torch_cuda()
    fld = library()
    rng = np.random.default_rng(n + 10 * bc[0] + bc[1])
    h, c, a_r, kappa, dt = (1.0,), 1.0, 1.0, 2.0, 3.0
    rho, T, E = (1.0 + rng.uniform(0, 1, n) for _ in range(3))
    Eb = {(0, s): np.array(1.5 + 0.1 * s) for s in (0, 1) if bc[s] == 2}
    packed = I.pack_dirichlet((n,), (bc,), Eb)
    ebc = dev(torch, packed) if packed.size else None
    hd = fld.Handle((n,), h, (bc,), tol=1e-13, max_cycles=20)
    op = (0, kappa, 0.0, 0.0)
    To, Eo, Do = O.step(rho, T, E, h, (bc,), Eb, dt, c, a_r, 5.0 / 3.0, 1.0, op, method="splu")
    Td, Ed = dev(torch, T), dev(torch, E)
    st = hd.step(fld.make_consts(c, a_r, 5.0 / 3.0, 1.0), fld.make_opacity(op), dt,
                 dev(torch, rho), Td, Ed, ebc)
    assert st["rel_resid"] <= 1e-13 and st["levels"] == 1 and st["resid_hist"][0] > 1e-3
    assert maxrel(host(Ed), Eo) < 1e-11 and maxrel(host(Td), To) < 1e-11
    xo = O.diffuse(E, Do, h, (bc,), Eb, dt, method="splu")
    x = dev(torch, E)
    st = hd.diffuse(dt, dev(torch, Do), ebc, x)
    assert st["rel_resid"] <= 1e-13 and maxrel(host(x), xo) < 1e-11
    # a bad cell is reported, clears, and leaves the fields as they were
    bad = T.copy()
    bad[n // 2] = -1.0
    rho_bad = rho.copy()
    rho_bad[n // 2] = np.nan
    Td, Ed = dev(torch, bad), dev(torch, E)
    st = hd.step(fld.make_consts(c, a_r, 5.0 / 3.0, 1.0), fld.make_opacity(op), dt,
                 dev(torch, rho_bad), Td, Ed, ebc, raise_on_error=False)
    assert st["status"] == fld.FLD_ERR_DOMAIN
    assert np.array_equal(host(Td), bad) and np.array_equal(host(Ed), E)
    assert hd.status() == fld.FLD_OK
    hd.close()


@pytest.mark.parametrize("scheme", ["split", "ars3"])
@pytest.mark.parametrize("n", [8, 15, 16, 29, 31, 61])
def test_wave_step_at_block_edges(n, scheme):
    """Steps of the driven wave on lines around multiples of the advance kernel's 15 cells;
    1e-11 of each variable's scale, the tolerance of the wave step's other tests."""
    torch = torch_cuda()
    fld = library()
    P = I.wave1d(I.WAVE_BACKGROUNDS["strong"], n, 2)
    P.n_driven = min(P.n_driven, n - 4)
    w = W.Wave(P, scheme=scheme)
    w.driven = np.arange(n) < P.n_driven
    U = w.initial()
    gpu = fld.Wave1D(P, scheme=1 if scheme == "ars3" else 0, tol=1e-13, max_cycles=60)
    Ud = dev(torch, U)
    t = 0.0
    for _ in range(3):
        dt = w.dt_max(U)
        assert abs(gpu.max_dt(Ud, 0.8) - dt) <= 1e-12 * dt
        U = w.step(U, t, dt)
        assert gpu.step(Ud, t, dt)["status"] in (0, 3)
        t += dt
    got = host(Ud).reshape(8, n)
    for v in range(8):
        scale = max(np.max(np.abs(U[v])), abs(P.W0[0]) * P.phase_speed if 1 <= v <= 3 else 0.0)
        assert np.max(np.abs(got[v] - U[v])) <= 1e-11 * max(scale, 1e-300), v
    gpu.close()
