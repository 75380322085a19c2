"""The grain lists of the MD cells, built on the device: a ninth grain in a cell is
refused, eight are not, at the box's periodic corner and inside it; with many grains
in few cells a step in FP64 is the oracle's bit for bit (each particle sums the
grains of its cell in the list's order)."""
import dataclasses

import numpy as np
import pytest

import oracle as O
import paper_1801_00972_gb300 as P
from paper_1801_00972_gb300 import build as B
from paper_1801_00972_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _workload(pos):
    wl = I.small(nx=8, ny=8, nz=16, n_e=4000, n_i=4000, grains=0, v_dc=-20.0)
    return dataclasses.replace(wl, grain_pos=np.asarray(pos) * wl.dx, grain_r=np.full(len(pos), 0.04 * wl.dx))


def _cluster(n, at, seed):
    g = np.random.default_rng(seed)
    return np.concatenate([(at + 0.5 + 2 * (g.random((n, 3)) - 0.5) * [1.4, 1.4, 0.4]) % [8, 8, 16]])


@pytest.mark.parametrize("at", [(0.0, 0.0, 5.0), (7.0, 3.0, 9.0), (4.0, 4.0, 1.0)])
def test_nine_grains_in_a_cell_are_refused(at):
    import torch
    B.build()
    torch.cuda.set_device(0)
    st = torch.cuda.current_stream().cuda_stream
    pos = [np.array(at) + 0.1 + 0.09 * q for q in range(9)]
    for prec in (P.PIC_MIXED, P.PIC_FP64):
        P.Run(_workload(pos[:8]), None, prec=prec, stream=st).close()
        with pytest.raises(P.PicError):
            P.Run(_workload(pos), None, prec=prec, stream=st)


@pytest.mark.parametrize("n,at,seed", [(1, (0.0, 0.0, 5.0), 1), (8, (0.0, 0.0, 5.0), 2), (8, (3.0, 7.0, 8.0), 3)])
def test_a_step_sums_the_grains_in_order(n, at, seed):
    import torch
    B.build()
    torch.cuda.set_device(0)
    pos = np.concatenate([_cluster(n, np.array(at), seed), [[4.5, 3.5, 12.5], [0.5, 7.5, 12.5]]])
    wl = _workload(pos)
    ref = O.Sim(wl, None)
    run = P.Run(wl, None, prec=P.PIC_FP64, stream=torch.cuda.current_stream().cuda_stream)
    run.set_gtab(ref.gtab())
    run.set_phi(ref.phi())
    run.advance()
    ref.advance()
    for sp in range(2):
        xg, vg, ig = run.particles(sp)
        xo, vo, io = ref.particles(sp)
        assert np.array_equal(ig, io) and np.array_equal(xg, xo) and np.array_equal(vg, vo)
    assert np.array_equal(run.rho(), ref.rho())
    run.close()
