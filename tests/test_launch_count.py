"""The count of kernels launched since the start of a run (pic_profile_read) against
the launches that the host code makes, with and without grains."""
import pytest

import paper_1801_00972_gb300 as P
from paper_1801_00972_gb300 import inputs as I
from recording import STREAM, recorder  # noqa: F401


@pytest.mark.parametrize("prec", [P.PIC_MIXED, P.PIC_FP64])
@pytest.mark.parametrize("grains", [0, 1, 12])
def test_launches_of_a_start_are_counted(recorder, prec, grains):  # noqa: F811
    with recorder.in_place():
        run = P.Run(I.small(nx=16, ny=16, nz=32, grains=grains), None, prec=prec, stream=STREAM)
        made = sum(c[0] == "launch" for c in recorder.calls())
        said = run.profile_read()["kernels"]
        run.close()
    assert made > 10 and said == made
