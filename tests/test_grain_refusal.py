"""More than 8 grains in one MD cell are an invalid argument, found before any device
memory is asked for: a run for which there is no memory at all is refused for its
grains, and one with grains that fit for the memory."""
import dataclasses

import numpy as np
import pytest

import paper_1801_00972_gb300 as P
from paper_1801_00972_gb300 import inputs as I
from recording import STREAM, recorder  # noqa: F401


def _status(rec, pos, shape=(8, 8, 16)):
    wl = I.small(nx=shape[0], ny=shape[1], nz=shape[2], grains=0)
    wl = dataclasses.replace(wl, grain_pos=np.asarray(pos) * wl.dx, grain_r=np.full(len(pos), 0.04 * wl.dx))
    with rec.in_place(limit=0), pytest.raises(P.PicError) as e:
        P.Run(wl, None, stream=STREAM)
    return e.value.status


@pytest.mark.parametrize("at", [(0.0, 0.0, 5.0), (7.0, 3.0, 9.0), (4.0, 4.0, 1.0)])
def test_a_ninth_grain_is_invalid_where_memory_is_short(recorder, at):  # noqa: F811
    pos = [np.array(at) + 0.1 + 0.09 * q for q in range(9)]
    assert _status(recorder, pos) == P.PIC_EINVAL
    assert _status(recorder, pos[:8]) == P.PIC_ENOMEM


@pytest.mark.parametrize("shape,most", [((4, 4, 8), 30), ((8, 4, 16), 60), ((16, 16, 16), 400)])
def test_clusters_are_refused_by_their_fullest_cell(recorder, shape, most):  # noqa: F811
    rng = np.random.default_rng(11)
    seen = set()
    for _ in range(100):
        n = int(rng.integers(1, most))
        pos = rng.random((n, 3)) * shape
        pos[:, 2] = 1.0 + rng.random(n) * (shape[2] - 2.001)
        count = {}
        for p in np.floor(pos).astype(int):
            for q in range(27):
                c = ((p[0] + q % 3 - 1) % shape[0], (p[1] + q // 3 % 3 - 1) % shape[1], p[2] + q // 9 - 1)
                count[c] = count.get(c, 0) + 1
        full = max(count.values())
        seen.add(full)
        assert _status(recorder, pos, shape) == (P.PIC_EINVAL if full > 8 else P.PIC_ENOMEM), (n, full)
    assert {8, 9} <= seen   # both sides of the limit came up


@pytest.mark.parametrize("shape,refused", [((8, 8, 301), True), ((8, 8, 401), True), ((10, 6, 331), True), ((8, 8, 221), False),
                                           ((8, 8, 151), False), ((8, 8, 450), False), ((16, 16, 49), False),
                                           ((16, 16, 32), False), ((80, 48, 100), False), ((4, 4, 63), False)])
def test_meshes_whose_solve_barely_converges_take_no_grains(recorder, shape, refused):  # noqa: F811
    # 8 x 8 x 301: a unit charge's solve on the device stood above 1e-12 after 200 cycles; 8 x 8 x 221
    # reached it, 8 x 8 x 450 halves to a level that is solved exactly
    wl = I.small(nx=shape[0], ny=shape[1], nz=shape[2], grains=1)
    bare = dataclasses.replace(wl, grain_pos=np.zeros((0, 3)), grain_r=np.zeros(0))
    with recorder.in_place():
        P.Run(bare, None, stream=STREAM).close()
        if refused:
            with pytest.raises(P.PicError) as e:
                P.Run(wl, None, stream=STREAM)
            assert e.value.status == P.PIC_ENOTCONV
        else:
            P.Run(wl, None, stream=STREAM).close()
