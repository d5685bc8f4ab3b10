"""The captured V-cycles that a handle keeps (csrc/fld_api.cu): more option sets than it holds, each
asked for again after the others, give the fields of directly launched V-cycles bit for bit."""
import numpy as np
import pytest

from gpu_util import torch_cuda, library, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("shape", [(40, 48), (24, 20, 32)])
def test_more_option_sets_than_graphs(shape, precision):
    torch = torch_cuda()
    fld = library()
    nd = len(shape)
    rng = np.random.default_rng(nd)
    D, E = dev(torch, 0.5 + rng.uniform(0, 1, shape)), 1.0 + rng.uniform(0, 1, shape)
    hd = fld.Handle(shape, (1.0,) * nd, ((0, 0),) * nd)
    opts = [dict(nu1=1 + q % 2, nu2=1, inner=1 + q // 2) for q in range(8)]
    want = {}
    for graph, order in ((0, range(8)), (1, [0, 1, 2, 0, 3, 4, 5, 6, 7, 0, 7, 2, 1])):
        for q in order:
            hd.set_opts(precision=precision, tol=1e-12, max_cycles=60, graph=graph, **opts[q])
            x = dev(torch, E)
            st = hd.diffuse(8.0, D, None, x)
            if graph == 0:
                want[q] = host(x)
            assert st["status"] == 0 and np.array_equal(host(x), want[q]), (graph, q)
    hd.close()
