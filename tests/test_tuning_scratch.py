"""A run whose tiling is changed again and again, to fewer and more sort keys and tiles
in any order: no level of a sort's scan reaches into another of its buffers, and the
particles, the charge and the grain counts stay those of a run that was left alone."""
import numpy as np
import pytest

import paper_1801_00972_gb300 as P
from paper_1801_00972_gb300 import build as B
from paper_1801_00972_gb300 import inputs as I
from recording import STREAM, recorder  # noqa: F401

# on 64 x 64 x 64 cells: 343000 keys, 262144, 270336 in more tiles than before, 343000 again
TILES = [(7, 7, 7), (8, 8, 8), (3, 4, 4), (7, 7, 7), (1, 1, 1), (7, 7, 7), (16, 8, 4), (5, 5, 5)]


def _tuning(tile, order):
    return dict(sort_every=2, tile=list(tile), halo=1, order=order)


@pytest.mark.parametrize("order", [0, 1, 2])
def test_scan_buffers_do_not_overlap(recorder, order):  # noqa: F811
    with recorder.in_place():
        run = P.Run(I.small(nx=64, ny=64, nz=64), None, stream=STREAM)
        for tile in TILES:
            recorder.lib.rec_clear()
            run.set_tuning(_tuning(tile, order))
            ext = {}   # buffer -> bytes a scan writes there
            for c in recorder.calls():
                if c[0] == "launch" and "k_scan_block" in c[2]:
                    grid, _, out, sums, n = map(int, c[3:8])
                    ext[out] = max(ext.get(out, 0), 4 * n)
                    ext[sums] = max(ext.get(sums, 0), 4 * grid)
            spans = sorted(ext.items())
            assert len(spans) >= 2
            for (a, la), (b, _) in zip(spans, spans[1:]):
                assert a + la <= b, (tile, spans)
        run.close()


@pytest.mark.gpu
@pytest.mark.parametrize("order", [0, 2])
def test_tuning_back_and_forth_keeps_every_particle(order):
    import torch
    B.build()
    torch.cuda.set_device(0)
    st = torch.cuda.current_stream().cuda_stream
    wl = I.small(nx=64, ny=64, nz=64, n_e=200_000, n_i=200_000, grains=2)
    a, b = (P.Run(wl, None, stream=st, sort_every=2) for _ in range(2))
    for tile in TILES:
        b.set_tuning(_tuning(tile, order))
        a.step(3)
        b.step(3)
    for sp in range(2):
        for x, y in zip(a.particles(sp), b.particles(sp)):
            assert np.array_equal(x, y)
    assert np.array_equal(a.rho(), b.rho())
    assert np.array_equal(a.grains()[0], b.grains()[0])
    a.close()
    b.close()
