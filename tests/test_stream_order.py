"""A run on a stream that the legacy default stream does not wait for (a batch's, a
framework's side stream): no kernel, copy or clear of the run's stream comes after a
legacy-stream clear or copy to the device that nothing has waited for."""
import pytest

import paper_1801_00972_gb300 as P
from paper_1801_00972_gb300 import inputs as I
from recording import STREAM, recorder, unordered  # noqa: F401


def test_a_missing_wait_is_seen():
    copy = ["copy", "0", "1", "1", "2", "8"]
    assert unordered([copy, ["launch", "5", "k", "1"]])
    assert unordered([["memset", "0", "1", "8"], ["memset", "5", "1", "8"]])
    assert not unordered([copy, ["sync", "0"], ["launch", "5", "k", "1"]])
    assert not unordered([["copy", "5", "1", "1", "2", "8"], ["launch", "5", "k", "1"]])


@pytest.mark.parametrize("prec", [P.PIC_MIXED, P.PIC_FP64])
@pytest.mark.parametrize("kw", [dict(), dict(flags=P.PIC_F_MOMENTS | P.PIC_F_COULOMB, mom_phases=4, eepf_bins=20, eepf_de_ev=0.5)])
@pytest.mark.parametrize("drawn", [False, True])
def test_start_of_a_run_is_ordered(recorder, prec, kw, drawn):  # noqa: F811
    wl = I.small(nx=16, ny=16, nz=32, grains=12)
    with recorder.in_place():
        run = P.Run(wl, None if drawn else I.sample_particles(wl), prec=prec, stream=STREAM, **kw)
        calls = recorder.calls()
        run.close()
    assert sum(c[0] == "launch" and c[1] == str(STREAM) for c in calls) > 10
    assert not unordered(calls)


@pytest.mark.parametrize("prec", [P.PIC_MIXED, P.PIC_FP64])
def test_calls_on_a_run_are_ordered(recorder, prec):  # noqa: F811
    wl = I.small(nx=16, ny=16, nz=32, grains=3)
    with recorder.in_place():
        run = P.Run(wl, None, prec=prec, stream=STREAM, flags=P.PIC_F_MOMENTS | P.PIC_F_NO_GRAPH)
        calls = {"phi": lambda: run.set_phi(run.phi()), "tables": lambda: run.set_gtab(run.gtab()),
                 "counts": lambda: run.set_grain_counts([[1, 2], [3, 4], [5, 6]]), "step": lambda: run.step(2),
                 "moments": lambda: run.moments(1, reset=True), "counters": run.counts,
                 "tuning": lambda: run.set_tuning(dict(sort_every=3, tile=[4, 4, 4], halo=1, order=0))}
        for name, call in calls.items():
            recorder.lib.rec_clear()
            call()
            run.advance()   # the run's next kernels
            assert not unordered(recorder.calls()), name
        run.close()
