"""What a sort by cell is for: right after one, the slots of both species run through
the tiles in order and through the cells of each tile in order, whichever way they got
there (in two passes for the electrons of tiles of 64 to 4096 cells, with up to 8192
particles through a permutation; in one pass otherwise)."""
import numpy as np
import pytest

import paper_1801_00972_gb300 as P
from paper_1801_00972_gb300 import build as B
from paper_1801_00972_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _keys(run, sp, tile):
    """Tile index * cells per tile + row-major cell inside the tile, in slot order."""
    wl = run.wl
    x, _, _ = run.particles(sp, sort=False)
    c = np.minimum(np.floor(x / wl.dx + 1e-9).astype(np.int64), [wl.nx - 1, wl.ny - 1, wl.nz - 1])
    t = np.array(tile)
    nt = -(-np.array([wl.nx, wl.ny, wl.nz]) // t)
    q, r = c // t, c % t
    return ((q[:, 2] * nt[1] + q[:, 1]) * nt[0] + q[:, 0]) * t.prod() + (r[:, 2] * t[1] + r[:, 1]) * t[0] + r[:, 0]


@pytest.mark.parametrize("mesh,tile,n", [
    ((16, 16, 16), (16, 16, 16), 8191), ((16, 16, 16), (16, 16, 16), 8192), ((16, 16, 16), (16, 16, 16), 8193),
    ((16, 16, 16), (16, 16, 16), 60000), ((16, 16, 32), (16, 16, 17), 20000), ((16, 16, 16), (7, 3, 3), 20000),
    ((16, 16, 16), (4, 4, 4), 20000), ((20, 12, 28), (8, 8, 8), 9000), ((64, 64, 64), (8, 8, 8), 300000),
    ((64, 64, 64), (4, 4, 4), 300000), ((64, 64, 64), (16, 16, 16), 300000)])
def test_slots_are_in_cell_order_after_a_sort(mesh, tile, n):
    import torch
    B.build()
    torch.cuda.set_device(0)
    wl = I.small(nx=mesh[0], ny=mesh[1], nz=mesh[2], n_e=n, n_i=n, grains=2, v_dc=-40.0)
    run = P.Run(wl, I.sample_particles(wl), prec=P.PIC_MIXED, stream=torch.cuda.current_stream().cuda_stream, sort_every=2)
    run.set_tuning(dict(sort_every=2, tile=list(tile), halo=0, order=0))   # (sorts at once)
    for steps in (0, 2, 4):   # each ends with a sort
        if steps:
            run.step(steps)
        for sp in range(2):
            k = _keys(run, sp, tile)
            assert len(k) > 0.5 * n and np.all(np.diff(k) >= 0), (sp, steps)
    run.close()
