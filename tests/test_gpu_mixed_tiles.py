"""Packed mixed 2D stage at the sizes where it changes its tile (15 x 7,
31 x 7, 31 x 18 planar or 31 x 15 general) and at their edges, over both fluxes and
limiters: two steps against the all-FP64 GPU path with the same step sizes,
within the 1e-4 per step that bounds the mixed path's steps elsewhere."""
import numpy as np
import pytest

from paper_2401_15233_gb300 import workloads as wl
from tests._util import aos_to_soa, field_rel_err, jets_gpu_solver, soa_to_aos

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2401_15233_gb300 as mx
    return mx


SIZES = [(4, 5), (15, 7), (16, 8), (31, 18), (33, 19), (97, 65), (230, 200), (310, 290), (520, 505)]


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("planar", [True, False])
@pytest.mark.parametrize("flux,limiter", [("hll", "minmod"), ("rusanov", "vanalbada")])
def test_two_steps(mx, nx, ny, planar, flux, limiter):
    setup = wl.jets_setup(Kn=0.1)
    prim = aos_to_soa(wl.smooth_field14(np.random.default_rng(nx), nx, ny, planar=planar))
    res = {}
    for precision in ("fp64", "mixed"):
        s = jets_gpu_solver(mx, nx, ny, setup, precision=precision, flux=flux, limiter=limiter)
        h = 0.1 / max(nx, ny)
        s.set_state(prim)
        s.step_dt([0.1 * h, 0.1 * h])
        assert s.diagnostics()["planar"] == int(planar)
        res[precision] = soa_to_aos(s.get_moments("conserved"))
    assert field_rel_err(res["mixed"], res["fp64"]).max() <= 2e-4
