"""A context's first uploads are not overtaken by the clearing of its buffers."""
import numpy as np
import pytest

from paper_2401_15233_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def test_boundary_states_survive_creation():
    """A large context clears gigabytes while it is created; boundary states set
    right after it have to be there when it steps (inflow at the background's
    state leaves a uniform gas at rest as it is)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2401_15233_gb300 as mx
    n = 3000
    bg = wl.maxwellian14(1.0, 0.0, 0.0, 1.0)
    prim = torch.tensor(bg, device="cuda").reshape(14, 1, 1).expand(14, n, n).contiguous()
    torch.cuda.synchronize()
    for _ in range(3):
        s = mx.Solver(system=14, nx=n, ny=n, precision="mixed")
        s.set_bc(mx.XLO, mx.BC_DIRICHLET, 0.4, 0.6, bg)
        s.set_bc(mx.YLO, mx.BC_DIRICHLET, 0.4, 0.6, bg)
        s.set_state(prim)
        s.step(2)
        d = s.diagnostics()
        assert d["n_nonfinite"] == 0 and np.isfinite(d["max_rate"])
        s.close()
