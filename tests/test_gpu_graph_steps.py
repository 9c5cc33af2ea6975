"""Steps reported by synchronous calls between replays of a caller's CUDA graph that
holds a run of the same context: each call counts its own steps only."""
import numpy as np
import pytest

from paper_2401_15233_gb300 import workloads as wl
from tests._util import aos_to_soa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny,precision", [(1, "fp64"), (24, "fp64"), (24, "mixed")])
def test_steps_after_a_replay(ny, precision):
    torch = pytest.importorskip("torch")
    import paper_2401_15233_gb300 as mx
    nx = 40
    prim = aos_to_soa(wl.smooth_field14(np.random.default_rng(1), nx, ny))
    s, ref = (mx.Solver(nx=nx, ny=ny, precision=precision) for _ in range(2))
    st = torch.cuda.Stream()
    s.set_stream(st.cuda_stream)
    s.set_state(prim)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        s.step(3, sync=False)
    s.set_state(prim)
    ref.set_state(prim)
    # 3 replayed steps, then some of a call (a grid's clock has three slots, which come round
    # every three steps: a graph of it is replayed where it was captured)
    for extra in (2, 1, 5) if ny == 1 else (3, 6):
        with torch.cuda.stream(st):
            g.replay()
        t, n = s.step(extra)
        t_ref, _ = ref.step(3 + extra)
        assert n == extra
        assert s.diagnostics()["steps"] == ref.diagnostics()["steps"]
        if precision == "fp64":                 # mixed grids: the periodic re-sync of W is the caller's
            assert t == t_ref
            assert np.array_equal(s.get_moments("conserved"), ref.get_moments("conserved"))
