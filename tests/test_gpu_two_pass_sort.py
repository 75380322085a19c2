"""The electrons' cell order is made in two passes when a tile has 64 to 4096 cells
(by tile, then by cell inside each tile, up to 8192 particles through a
permutation in shared memory).  Against the order by tile only, which takes one
pass: particles, charge and grain counts bit for bit after sorts with the electron
count of a one-tile mesh at and beside the permutation's limit, and for tiles at
and beside both ends of the range, cut off at the mesh's far sides, and empty."""
import dataclasses

import numpy as np
import pytest

import paper_1801_00972_gb300 as P
from paper_1801_00972_gb300 import build as B
from paper_1801_00972_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh,tile,halo,n_e", [
    ((16, 16, 16), (16, 16, 16), 0, 8191), ((16, 16, 16), (16, 16, 16), 0, 8192), ((16, 16, 16), (16, 16, 16), 0, 8193),
    ((16, 16, 16), (16, 16, 16), 0, 40000), ((16, 16, 32), (16, 16, 17), 0, 20000), ((16, 16, 16), (4, 4, 4), 1, 20000),
    ((16, 16, 16), (7, 3, 3), 1, 20000), ((20, 12, 28), (8, 8, 8), 2, 9000), ((20, 12, 28), (6, 5, 9), 0, 37)])
def test_two_pass_cell_order_keeps_every_particle(mesh, tile, halo, n_e):
    import torch
    B.build()
    torch.cuda.set_device(0)
    wl = I.small(nx=mesh[0], ny=mesh[1], nz=mesh[2], n_e=n_e, n_i=n_e, grains=0, v_dc=-40.0)
    pos = np.array([[0.2, 0.3, 8.5], [8.01, 7.99, 4.02]]) * wl.dx
    wl = dataclasses.replace(wl, grain_pos=pos, grain_r=np.full(2, 0.2 * wl.dx))
    parts = I.sample_particles(wl)
    runs = []
    for order in (0, 1):
        r = P.Run(wl, parts, prec=P.PIC_MIXED, stream=torch.cuda.current_stream().cuda_stream, sort_every=2)
        r.set_tuning(dict(sort_every=2, tile=list(tile), halo=halo, order=order))
        r.step(5)
        runs.append(r)
    a, b = runs
    for sp in range(2):
        xa, va, ia = a.particles(sp)
        xb, vb, ib = b.particles(sp)
        assert np.array_equal(ia, ib) and np.array_equal(xa, xb) and np.array_equal(va, vb)
    assert np.array_equal(a.rho(), b.rho())
    assert np.array_equal(a.grains()[0], b.grains()[0])
    a.close()
    b.close()
