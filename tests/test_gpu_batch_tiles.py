"""2D problems of the batched step on both sides of the rule that picks tiles or half sweeps
(csrc/fld_batch.cuh, batch_tiled), and the last tiles of a problem, which load only the rows that
are left: sides of a whole number of tiles, one pair of rows and one row more, odd extents with
walls (tiles) and periodic ones (half sweeps below 65536 cells, tiles above), beside problems too
small for tiles. Each is compared with the FP64 solve of a handle of its own.

Tolerance: the handle solves to 1e-13 of ||b||_2, the batch to 2e-13 (the double-FP32 residual's
rounding may end it above 1e-13), with ||A^-1|| <= 1 and fields of order one; in the max norm at
most sqrt(66000) of each, 8e-11 together. T carries E's error over a heat capacity of order one."""
import numpy as np
import pytest

from paper_2503_02764_gb300 import inputs as I
from gpu_util import torch_cuda, library, dev, host, maxrel

pytestmark = pytest.mark.gpu

PER, NEU, DIR = (0, 0), (1, 1), (2, 2)
# (nx, ny, walls along x and y)
PROBLEMS = [(116, 84, PER, PER), (116, 86, PER, NEU), (116, 85, DIR, NEU), (117, 127, NEU, DIR),
            (97, 97, PER, PER), (257, 256, PER, PER), (112, 112, PER, PER), (64, 64, PER, PER),
            (16, 17, NEU, DIR), (160, 108, PER, (1, 2))]


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("nu", [1, 2])
@pytest.mark.parametrize("block,cluster", [(512, 1), (256, 1), (512, 2)])
def test_both_sides_of_the_tile_rule(block, cluster, nu, precision):
    torch = torch_cuda()
    fld = library()
    rng = np.random.default_rng(7)
    consts = fld.make_consts(1.0, 1.0, 5.0 / 3.0, 1.0)
    grids, fields, faces, ops, dts, want = [], [], [], [], [], []
    for nx, ny, bx, by in PROBLEMS:
        shape, bc = (ny, nx), (bx, by)
        rho, T, E = (1.0 + rng.uniform(0, 1, shape) for _ in range(3))
        Eb = {(d, s): 1.5 + 0.1 * rng.uniform(0, 1, shape[d]) for d in (0, 1) for s in (0, 1)
              if bc[d][s] == 2}
        packed = I.pack_dirichlet(shape, bc, Eb)
        op, dt = fld.make_opacity((0, 0.5 + rng.uniform(), 0.0, 0.0)), 4.0
        hd = fld.Handle(shape, (1.0, 1.0), bc, tol=1e-13, max_cycles=60)
        Td, Ed = dev(torch, T), dev(torch, E)
        assert hd.step(consts, op, dt, dev(torch, rho), Td, Ed,
                       dev(torch, packed) if packed.size else None)["status"] == 0
        want.append((host(Td), host(Ed)))
        hd.close()
        grids.append((shape, (1.0, 1.0), bc))
        fields.append((rho.ravel(), T.ravel(), E.ravel()))
        faces.append(packed)
        ops.append(op)
        dts.append(dt)
    rho, T, E = (dev(torch, np.concatenate([f[q] for f in fields])) for q in range(3))
    b = fld.Batch(grids, tol=1e-13, max_cycles=60, block=block, cluster=cluster, nu1=nu, nu2=nu,
                  precision=precision)
    rc, st = b.step(consts, ops, dts, rho, T, E, dev(torch, np.concatenate(faces)),
                    raise_on_error=False)
    assert rc in (0, 3) and max(q["rel_resid"] for q in st) <= 2e-13, st
    got, at = (host(T), host(E)), 0
    for (shape, _, _), w in zip(grids, want):
        n = shape[0] * shape[1]
        for q in (0, 1):
            assert maxrel(got[q][at:at + n], w[q].ravel()) < 1e-10, (shape, q)
        at += n
    b.close()
