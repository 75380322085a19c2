"""A warp of the substepping kernel takes 4 MD-region particles while they are few and 32
beyond 9728 of a species: every particle's step is the same bits whichever it was, and
however many others there are."""
import numpy as np
import pytest

import paper_1801_00972_gb300 as P
from paper_1801_00972_gb300 import build as B
from paper_1801_00972_gb300 import inputs as I

pytestmark = pytest.mark.gpu
FEW = 3000


@pytest.mark.parametrize("n", [9727, 9728, 9729, 40000])
def test_particles_do_not_depend_on_the_lanes_of_their_warp(n):
    import torch
    B.build()
    torch.cuda.set_device(0)
    wl = I.small(nx=8, ny=8, nz=16, n_e=n, n_i=n, grains=1, weight=1.0, dt=2e-11)
    cell = np.floor(wl.grain_pos[0] / wl.dx)
    rng = np.random.default_rng(3)
    parts = []
    for sp, v in ((0, 7.3e5), (1, 269.0)):   # all in the 27 cells around the grain's; the few first
        x = (cell - 1 + 3 * rng.random((n, 3)) * 0.999999) * wl.dx
        parts.append((x, rng.standard_normal((n, 3)) * v, np.arange(n, dtype=np.uint32) + sp * n))
    phi = np.random.default_rng(4).standard_normal(wl.nodes)
    out = []
    for m in (FEW, n):
        run = P.Run(wl, [tuple(a[:m] for a in p) for p in parts], prec=P.PIC_MIXED,
                    stream=torch.cuda.current_stream().cuda_stream)
        run.set_grain_counts([[40000, 0]])   # a charge that bends every path near it
        run.set_phi(phi)
        run.advance()   # (one step: what is absorbed changes the grain's charge for the next)
        res = []
        for sp in range(2):
            x, v, i = run.particles(sp)
            keep = (i >= sp * n) & (i < sp * n + FEW)   # (ionization products have other ids)
            res.append((x[keep], v[keep], i[keep]))
        out.append(res)
        run.close()
    for a, b in zip(*out):
        assert len(a[2]) > 0.5 * FEW
        for p, q in zip(a, b):
            assert np.array_equal(p, q)
