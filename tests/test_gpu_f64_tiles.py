"""FP64 2D stage at the sizes where it changes its tile (5 x 5, 7 x 8,
15 x 16) and at their edges: one step against the oracle, to the 1e-12 of
one step from identical input."""
import numpy as np
import pytest

from paper_2401_15233_gb300 import workloads as wl
from tests._util import aos_to_soa, field_rel_err, jets_gpu_solver, jets_oracle_cfg, soa_to_aos

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module")
def mx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2401_15233_gb300 as mx
    return mx


# 5 x 5 up to about 100 x 80 and again near 160 x 160, 7 x 8 at 120 x 130 and
# 200 x 200, 15 x 16 from about 250 x 250
@pytest.mark.parametrize("nx,ny", [(4, 5), (5, 6), (11, 4), (61, 47), (120, 130), (160, 161),
                                   (203, 200), (255, 257)])
@pytest.mark.parametrize("planar", [True, False])
def test_one_step(mx, orc, nx, ny, planar):
    setup = wl.jets_setup(Kn=0.1)
    prim = wl.smooth_field14(np.random.default_rng(nx), nx, ny, planar=planar)
    U = orc.prim2cons_field(prim)
    cfg = jets_oracle_cfg(orc, nx, ny, setup)
    s = jets_gpu_solver(mx, nx, ny, setup)
    s.set_state(aos_to_soa(U), kind="conserved")
    dt = orc.dt(cfg, U, 0.0, 10.0)
    s.step_dt([dt])               # compared whether or not the step keeps positivity (4 x 5 does not)
    assert field_rel_err(soa_to_aos(s.get_moments("conserved")), orc.step(cfg, U, dt)).max() <= TOL
