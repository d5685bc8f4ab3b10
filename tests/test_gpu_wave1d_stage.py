"""An ARS3 step whose first implicit stage fails reports a domain error and leaves the state as it
was, on the one-launch path and on the separate launches (lines above 8192 cells), on a fresh
handle and after good steps; the next step from a good state is that of a fresh handle.

The step is one that is too long for a strong expansion: the state is physical everywhere, but
the first predictor's gas pressure is negative in a few cells. Its density and E stay positive and
the opacity is constant, so nothing before the first stage's exchange can refuse it; and the
second predictor would be physical again, were it formed from an earlier step's stage."""
import numpy as np
import pytest

from oracle import rmhd1d as R
from paper_2503_02764_gb300 import inputs as I
from gpu_util import torch_cuda, library, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [280, 8200])
def test_failed_first_stage_leaves_the_state(n):
    torch = torch_cuda()
    fld = library()
    P = I.wave1d(I.WAVE_BACKGROUNDS["strong"], n, 7)
    orc = R.Wave(P, scheme="ars3")
    good = np.array(orc.initial(), dtype=np.float64).reshape(8, n)
    short = orc.dt_max(good)
    cf = float(R.fast_speed(P.W0[:, None], P.Bx, P.gamma)[0])
    W = R.primitive(good, P.Bx, P.gamma).copy()
    W[1, n - 60:] += 1.4 * cf * np.exp(-(np.arange(60) / 10.0) ** 2)
    bad = R.conserved(W, P.Bx, P.gamma)
    dt = 2.0 * P.dx / (np.max(np.abs(W[1])) + cf)
    ga = (3.0 + np.sqrt(3.0)) / 6.0
    L1 = orc.rhs(bad, 0.0)
    p1 = R.primitive(bad + ga * dt * L1, P.Bx, P.gamma)
    assert np.min(p1[6]) < -1e3 and np.min(p1[0] / P.W0[0]) > 0.1 and np.min(p1[7] / P.E0) > 0.1
    p2 = bad + dt * ((ga - 1.0) * L1 + 2.0 * (1.0 - ga) * orc.rhs(good, 0.0))
    p2 = R.primitive(p2, P.Bx, P.gamma)
    assert np.min(p2[6]) > 0.0 and np.min(p2[0]) > 0.0 and np.min(p2[7]) > 0.0

    def make():
        return fld.Wave1D(P, scheme=1, tol=1e-13, max_cycles=60)

    gpu = make()
    for good_before in (False, True):
        if good_before:
            assert gpu.step(dev(torch, good), 0.0, short)["status"] in (0, 3)
        Ud = dev(torch, bad)
        st = gpu.step(Ud, 0.0, dt, raise_on_error=False)
        assert st["status"] == fld.FLD_ERR_DOMAIN
        assert np.array_equal(host(Ud).reshape(8, n), bad)
    Ud, Vd, other = dev(torch, good), dev(torch, good), make()
    assert gpu.step(Ud, 0.0, short)["status"] in (0, 3)
    assert other.step(Vd, 0.0, short)["status"] in (0, 3)
    assert np.array_equal(host(Ud), host(Vd))
    gpu.close()
    other.close()
