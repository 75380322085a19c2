"""Device memory of a large run: the particles' records, twice (a sort goes from one
copy to the other), the room for new particles of a step, and little more."""
import pytest

import paper_1801_00972_gb300 as P
from paper_1801_00972_gb300 import inputs as I
from recording import STREAM, recorder  # noqa: F401


@pytest.mark.parametrize("prec,slot", [(P.PIC_FP64, 2 * 64), (P.PIC_MIXED, 2 * 32 + 3 * 4 + 4)])
def test_bytes_per_particle_slot(recorder, prec, slot):  # noqa: F811
    # mixed: three lists of slots, and results of the substeps for an eighth of the slots (32 bytes each)
    cap = 32_000_000
    with recorder.in_place():
        run = P.Run(I.small(), None, prec=prec, stream=STREAM, capacity=(cap, cap))
        held = recorder.held()
        run.close()
    children = cap // 64 * 80
    assert held <= 2 * cap * slot + children + (128 << 20)   # two slabs for all the rest
    assert recorder.held() == 0
