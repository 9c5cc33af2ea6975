"""Tube teams on a stream that cannot hold all their CTAs at once: the launch is refused,
and the tubes are marched without teams, with the same result."""
import numpy as np
import pytest

from paper_2401_15233_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,sizes", [("fp64", [16000]), ("fp64", [9000, 40, 8000]),
                                             ("mixed", [90000]), ("mixed", [50000, 40, 60000])])
@pytest.mark.parametrize("how", ["steps", "time", "dts"])
def test_refused_teams(precision, sizes, how):
    import ctypes as C

    import paper_2401_15233_gb300 as mx
    b = mx.Batch(sizes, [1.0] * len(sizes), precision=precision)
    state = b.pack([wl.smooth_field14(np.random.default_rng(n), n, 1)[0].T for n in sizes])

    def march():
        b.set_state(state)
        for _ in range(2):
            if how == "dts":
                mx.mxe_step_dt(b.ctx, [1e-7, 2e-7])
            else:
                b.run(3, float("inf") if how == "steps" else 4e-6)
        return b.get_moments("conserved"), b.clock()

    want, (t, n) = march()
    # more CTAs than the device holds: 31 (FP64) or 120 cells each
    assert mx.lib().mxe_test_team_slots(C.c_void_p(b.ctx.value), 1 << 20) == mx.OK
    got, (t1, n1) = march()
    assert np.array_equal(got, want) and np.array_equal(t, t1) and np.array_equal(n, n1)
    if precision == "mixed":
        assert b.layout()[0] > 0
    b.set_stream(0)                             # another stream: the teams are tried again
    got, _ = march()
    assert np.array_equal(got, want)
