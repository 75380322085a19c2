"""The push looks up the grain count of a particle's cell only in tiles whose
deposit window holds an MD cell.  A mesh that is one tile (its window holds every
grain, so every particle is looked up) against tiles of few cells, with grains at
the tiles' edges and across the periodic sides: particles, charge and grain
counts bit for bit, over steps between sorts in which particles leave their
tile's window."""
import dataclasses

import numpy as np
import pytest

import paper_1801_00972_gb300 as P
from paper_1801_00972_gb300 import build as B
from paper_1801_00972_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _run(wl, parts, tile, halo, order):
    import torch
    r = P.Run(wl, parts, prec=P.PIC_MIXED, stream=torch.cuda.current_stream().cuda_stream, sort_every=4)
    r.set_tuning(dict(sort_every=4, tile=list(tile), halo=halo, order=order))
    r.step(7)
    return r


@pytest.mark.parametrize("tile,halo,order", [((4, 4, 4), 0, 0), ((4, 4, 4), 2, 1), ((5, 3, 7), 1, 2), ((16, 2, 1), 3, 0),
                                             ((1, 1, 1), 0, 0), ((6, 6, 6), 8, 0)])
def test_tiles_without_md_cells_match_the_looked_up_mesh(tile, halo, order):
    import torch
    B.build()
    torch.cuda.set_device(0)
    wl = I.small(nx=16, ny=16, nz=16, n_e=30000, n_i=30000, grains=0, v_dc=-40.0)
    dx = wl.dx
    # in the corner cell (its region wraps in x and y), on a tile edge, next to the lower electrode's rim
    pos = np.array([[0.2, 0.3, 8.5], [8.01, 7.99, 4.02], [15.9, 4.5, 1.5]]) * dx
    wl = dataclasses.replace(wl, grain_pos=pos, grain_r=np.full(3, 0.2 * dx))
    parts = I.sample_particles(wl)
    a, b = _run(wl, parts, (16, 16, 16), 0, 0), _run(wl, parts, tile, halo, order)
    for sp in range(2):
        xa, va, ia = a.particles(sp)
        xb, vb, ib = b.particles(sp)
        assert np.array_equal(ia, ib) and np.array_equal(xa, xb) and np.array_equal(va, vb)
    assert np.array_equal(a.rho(), b.rho())
    na, nb = a.grains()[0], b.grains()[0]
    assert np.array_equal(na, nb) and na.sum() > 0
    a.close()
    b.close()
