"""FP64 face reverse over the schemes and sizes it takes (both fluxes and
limiters, first order, relaxation models; faces that do not fill a warp or a
block): <V, L' x> against the oracle's forward-mode tangent to 1e-10, the
bound of one residual."""
import numpy as np
import pytest

from paper_2401_15233_gb300 import workloads as wl
from tests._util import aos_to_soa, jets_gpu_solver, jets_oracle_cfg, soa_to_aos

pytestmark = pytest.mark.gpu
Z_ODD = [3, 6, 8, 12]


@pytest.fixture(scope="module")
def mx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2401_15233_gb300 as mx
    return mx


@pytest.mark.parametrize("nx,ny", [(4, 4), (17, 5), (32, 31)])
@pytest.mark.parametrize("kw", [dict(), dict(flux="rusanov"), dict(limiter="vanalbada"),
                                dict(flux="rusanov", limiter="vanalbada"), dict(order=1)])
@pytest.mark.parametrize("model", [0, 1, 2])
def test_residual_dot_product(mx, orc, nx, ny, kw, model):
    setup = wl.jets_setup(Kn=0.1)
    rng = np.random.default_rng(nx + 100 * model)
    U = orc.prim2cons_field(wl.smooth_field14(rng, nx, ny, planar=True))
    num = dict(flux={"hll": 0, "rusanov": 1}[kw.get("flux", "hll")],
               limiter={"minmod": 0, "vanalbada": 1}[kw.get("limiter", "minmod")],
               order=kw.get("order", 2))
    cfg = jets_oracle_cfg(orc, nx, ny, setup, **num)
    cfg.tau_model = model
    s = jets_gpu_solver(mx, nx, ny, setup, **kw)
    s.set_relaxation(model, setup["tau_ref"], setup["rho_ref"], setup["T_ref"])
    s.set_state(aos_to_soa(U), kind="conserved")
    V = rng.standard_normal(U.shape)
    V[..., Z_ODD] = 0.0
    V[: ny // 2, : nx // 2] = 0.0                 # faces without an adjoint
    out, gb, tb = s.adjoint_residual(aos_to_soa(U), aos_to_soa(V))
    x = U * rng.standard_normal(U.shape) * 1e-2
    x[..., Z_ODD] = 0.0
    g = np.zeros((4, 5, 14))
    g[0, 1, [0, 1, 2, 4, 5, 7, 9, 10, 11, 13]] = rng.standard_normal(10)
    for name, (xd, gd, td) in {"state": (x, g * 0, 0.0), "inflow": (x * 0, g, 0.0),
                               "tau": (x * 0, g * 0, 1.0)}.items():
        _, dL = orc.tangent_residual(orc.tangent_cfg(cfg, d_states=gd, d_tau_ref=td), U, xd)
        lhs = float((V * dL).sum())
        rhs = float((soa_to_aos(out) * xd).sum() + (gb * gd).sum() + tb * td)
        # the sum's own size: its terms cancel
        scale = float(np.abs(V * dL).sum()) + 1e-300
        assert abs(lhs - rhs) <= 1e-10 * scale, (name, lhs, rhs)
