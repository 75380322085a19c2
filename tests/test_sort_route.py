"""Which runs sort their electrons in two passes, by the host's launches: many tiles with
some hundreds to some thousands of electrons each, that have crossed about a cell since
the last sort; everything else takes one pass.  On the GPU: tiles with as many particles
as the second pass's permutation holds and beside it come out in cell order with every
record in place, and a run whose interval goes in and out of the range keeps the bits of
one that was left alone."""
import dataclasses

import numpy as np
import pytest

import paper_1801_00972_gb300 as P
from paper_1801_00972_gb300 import build as B
from paper_1801_00972_gb300 import inputs as I
from recording import STREAM, recorder  # noqa: F401
from test_gpu_cell_order import _keys

T8 = (8, 8, 8)


@pytest.mark.parametrize("mesh,tile,n,every,dt,order,two", [
    ((16, 16, 32), T8, 1_000_000, 5, 1e-10, 0, False), ((16, 16, 32), T8, 1_000_000, 1, 1e-10, 0, False),
    ((64, 64, 256), T8, 5_000_000, 5, 1e-10, 0, False), ((64, 64, 512), T8, 10_000_000, 5, 1e-10, 0, True),
    ((64, 64, 512), T8, 20_000_000, 5, 1e-10, 0, False), ((128, 128, 256), T8, 8_000_000, 5, 1e-10, 0, True),
    ((128, 128, 256), T8, 8_000_000, 1, 1e-10, 0, False), ((128, 128, 256), T8, 8_000_000, 20, 1e-10, 0, False),
    ((128, 128, 256), T8, 8_000_000, 5, 1e-11, 0, False), ((128, 128, 256), T8, 8_000_000, 5, 1e-10, 1, False),
    ((128, 128, 256), T8, 70_000_000, 5, 1e-10, 0, False), ((64, 64, 64), (4, 4, 4), 2_000_000, 5, 1e-10, 0, True),
    ((64, 64, 64), (4, 4, 4), 300_000, 5, 1e-10, 0, False), ((64, 64, 100), (5, 4, 5), 2_300_000, 3, 1e-10, 0, True), ((128, 128, 256), (16, 16, 4), 8_000_000, 5, 1e-10, 0, True),
    ((128, 128, 256), (16, 16, 16), 500_000, 5, 1e-10, 0, False)])
def test_two_passes_where_they_pay(recorder, mesh, tile, n, every, dt, order, two):  # noqa: F811
    wl = I.small(nx=mesh[0], ny=mesh[1], nz=mesh[2], n_e=n, n_i=n, grains=0, dt=dt)
    with recorder.in_place():
        run = P.Run(wl, None, stream=STREAM, sort_every=every, capacity=(n, n))
        if (tile, order) != (T8, 0):
            recorder.lib.rec_clear()
            run.set_tuning(dict(sort_every=every, tile=list(tile), halo=1, order=order))
        calls = recorder.calls()
        run.close()
    assert sum("k_order_cells" in " ".join(c) for c in calls) == int(two)


def test_a_new_interval_changes_the_route(recorder):  # noqa: F811
    with recorder.in_place():
        run = P.Run(I.small(nx=64, ny=64, nz=64, n_e=2_000_000, n_i=1000, grains=0), None, stream=STREAM,
                    flags=P.PIC_F_NO_GRAPH)
        for every, two in ((4, 1), (1, 0), (2, 1), (20, 0), (3, 1)):
            run.set_tuning(dict(sort_every=every, tile=[4, 4, 4], halo=1, order=0))
            while run.step_index % every != every - 1:
                run.step(1)
            recorder.lib.rec_clear()
            run.step(1)
            assert sum("k_order_cells" in " ".join(c) for c in recorder.calls()) == two, every
        run.close()


@pytest.mark.gpu
@pytest.mark.parametrize("mesh,tile", [((64, 64, 64), (4, 4, 4)), ((64, 64, 100), (5, 4, 5)), ((128, 128, 256), (16, 16, 4))])
def test_full_and_overfull_tiles_keep_their_records(mesh, tile):
    import torch
    B.build()
    torch.cuda.set_device(0)
    n = 2_300_000
    wl = I.small(nx=mesh[0], ny=mesh[1], nz=mesh[2], n_e=n, n_i=100, grains=0, v_dc=0.0, weight=1e-3)
    rng = np.random.default_rng(8)
    t, m = np.array(tile), np.array(mesh)
    x = rng.random((n, 3)) * (m - [0, 0, t[2]]) + [0, 0, t[2]]   # the tiles of the first layer stay empty
    at = 0
    for q, count in enumerate((8191, 8192, 8193, 20000, 1)):     # but for these
        x[at:at + count] = (rng.random((count, 3)) * 0.999 + [q + 1, 1, 0]) * t
        at += count
    x *= wl.dx
    v = rng.standard_normal((n, 3)) * 7.3e5
    order = rng.permutation(n)
    ion = np.full((100, 3), 0.5 * wl.dx), np.zeros((100, 3)), np.arange(n, n + 100, dtype=np.uint32)
    parts = [(x[order], v[order], order.astype(np.uint32)), ion]
    run = P.Run(wl, parts, prec=P.PIC_MIXED, stream=torch.cuda.current_stream().cuda_stream, sort_every=3,
                flags=P.PIC_F_NO_MCC)
    before = run.particles(0)
    run.set_tuning(dict(sort_every=3, tile=list(tile), halo=1, order=0))   # (sorts at once)
    k = _keys(run, 0, tile)
    per = int(t.prod())
    nt0 = -(-mesh[0] // tile[0])
    assert np.bincount(k // per)[nt0 + 1:nt0 + 6].tolist() == [8191, 8192, 8193, 20000, 1]
    for _ in range(2):
        assert np.all(np.diff(k) >= 0)
        run.step(3)
        k = _keys(run, 0, tile)
    run.close()
    # the records themselves, by id
    run = P.Run(wl, parts, prec=P.PIC_MIXED, stream=torch.cuda.current_stream().cuda_stream, sort_every=3)
    run.set_tuning(dict(sort_every=3, tile=list(tile), halo=1, order=0))
    for a, b in zip(before, run.particles(0)):
        assert np.array_equal(a, b)
    run.close()


@pytest.mark.gpu
def test_intervals_in_and_out_of_the_range_keep_every_particle():
    import torch
    B.build()
    torch.cuda.set_device(0)
    st = torch.cuda.current_stream().cuda_stream
    wl = I.small(nx=64, ny=64, nz=64, n_e=2_000_000, n_i=2_000_000, grains=0, v_dc=-40.0)
    pos = np.array([[0.2, 0.3, 8.5], [8.01, 7.99, 4.02], [31.0, 40.5, 30.5]]) * wl.dx
    wl = dataclasses.replace(wl, grain_pos=pos, grain_r=np.full(3, 0.2 * wl.dx))
    a, b = (P.Run(wl, None, prec=P.PIC_MIXED, stream=st, sort_every=4) for _ in range(2))
    for every in (4, 1, 2, 20, 3):
        b.set_tuning(dict(sort_every=every, tile=[4, 4, 4], halo=1, order=0))
        a.step(5)
        b.step(5)
    b.tune_sort(1)
    a.step(b.step_index - a.step_index)
    for sp in range(2):
        for p, q in zip(a.particles(sp), b.particles(sp)):
            assert np.array_equal(p, q)
    assert np.array_equal(a.rho(), b.rho())
    assert np.array_equal(a.grains()[0], b.grains()[0]) and a.grains()[0].sum() > 0
    a.close()
    b.close()
