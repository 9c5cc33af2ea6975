"""The bounded wait of the CTAs that march a tube together: one that counts on a CTA which
was never launched runs out, says so, and leaves the context usable."""
import numpy as np
import pytest

from paper_2401_15233_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SPIN = 2000                     # polls, under a millisecond


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("sizes", [[20], [500], [500, 64, 130]])
@pytest.mark.parametrize("how", ["step", "step_dt", "later"])
def test_wait_runs_out(precision, sizes, how):
    import ctypes as C

    import paper_2401_15233_gb300 as mx
    prims = [wl.smooth_field14(np.random.default_rng(n), n, 1)[0].T for n in sizes]
    one = len(sizes) == 1
    s = mx.Solver(nx=sizes[0], precision=precision) if one else mx.Batch(
        sizes, [1.0] * len(sizes), precision=precision)
    state = prims[0][:, None, :].copy() if one else s.pack(prims)
    march = lambda: mx.mxe_step(s.ctx, 3, float("inf"))  # noqa: E731
    s.set_state(state)
    march()
    want = s.get_moments("conserved")

    s.set_state(state)
    assert mx.lib().mxe_test_team_wait(C.c_void_p(s.ctx.value), SPIN, 1) == mx.OK
    with pytest.raises(mx.MaxentError) as e:
        if how == "step_dt":
            mx.mxe_step_dt(s.ctx, [1e-4, 1e-4])
        else:
            if how == "later":
                mx.mxe_step(s.ctx, 3, float("inf"), sync=False)
            march()
    assert e.value.status == mx.ETIMEOUT
    for call in (march, s.get_moments):         # nothing goes on from there
        with pytest.raises(mx.MaxentError) as e:
            call()
        assert e.value.status == mx.ESTATE

    assert mx.lib().mxe_test_team_wait(C.c_void_p(s.ctx.value), 0, 0) == mx.OK
    s.set_state(state)
    march()
    assert np.array_equal(s.get_moments("conserved"), want)
