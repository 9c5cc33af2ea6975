"""set_state: what the FP32 screen of the realizability check must leave to the
FP64 one, and a mixed grid's state given as primitives or as conserved moments."""
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


def _cell(P, rho=1.0, scale=1.0):
    """rho, P as given (xx, xy, xz, yy, yz, zz), q = 0, a fourth moment above every
    bound of it"""
    P = np.asarray(P) * scale
    p = abs(P[0] + P[3] + P[5]) / 3 + scale * 1e-3
    return np.array([rho, 0.3, -0.2, 0.0, *P, 0.0, 0.0, 0.0, 40.0 * p * p / rho])


GOOD = [([1, 0, 0, 1, 0, 1], 1.0, 1.0), ([1, 0, 0, 1, 0, 1e-9], 1.0, 1.0),
        ([1e-7, 0, 0, 1, 0, 1], 1.0, 1.0), ([1, 0.9999999, 0, 1, 0, 1], 1.0, 1.0),
        ([1, 0.2, 0.1, 2, 0.1, 1], 1e-25, 1e-30), ([1, 0, 0, 1, 0, 1], 1.0, 1e-35),
        ([1, 0, 0, 1, 0, 1], 1e20, 1e35)]
BAD = [([1, 0, 0, 1, 0, -1e-9], 1.0, 1.0), ([-1, 0, 0, -1, 0, -1], 1.0, 1.0),
       ([-1e-9, 0, 0, 1, 0, 1], 1.0, 1.0), ([1, 1.0000001, 0, 1, 0, 1], 1.0, 1.0),
       ([1, 0, 0, 1, 0, 0], 1.0, 1.0), ([1, 0, 0, 1, 0, 1], 0.0, 1.0),
       ([1, 0, 0, 1, 0, 1], -1.0, 1.0), ([1, 0, 0, np.nan, 0, 1], 1.0, 1.0),
       ([1, 0, 0, 1, 0, np.inf], 1.0, 1.0), ([0.1, 0, 0, -1, 0, -1], 1.0, 1.0)]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("ok,spec", [(True, s) for s in GOOD] + [(False, s) for s in BAD])
def test_realizability(mx, precision, ok, spec):
    P, rho, scale = spec
    prim = np.repeat(_cell([1, 0, 0, 1, 0, 1])[:, None], 40, 1).reshape(14, 5, 8).copy()
    with np.errstate(all="ignore"):
        prim[:, 3, 6] = _cell(P, rho, scale)
    s = mx.Solver(nx=8, ny=5, precision=precision)
    if ok:
        s.set_state(prim)
    else:
        with pytest.raises(mx.MaxentError):
            s.set_state(prim)


@pytest.mark.parametrize("planar", [True, False])
def test_primitive_and_conserved_input(mx, orc, planar):
    """The conserved state is the oracle's (1e-14: a few roundings); two steps of the mixed
    path from either input differ by the FP32 rounding of W (1e-4 a step, the
    bound of its steps)."""
    nx, ny = 37, 29
    setup = wl.jets_setup(Kn=0.1)
    prim = wl.smooth_field14(np.random.default_rng(5), nx, ny, planar=planar)
    U = orc.prim2cons_field(prim)
    out = []
    for kind, x in (("primitive", prim), ("conserved", U)):
        s = jets_gpu_solver(mx, nx, ny, setup, precision="mixed")
        s.set_state(aos_to_soa(x), kind=kind)
        got = soa_to_aos(s.get_moments("conserved"))
        assert field_rel_err(got, U).max() <= 1e-14
        s.step_dt([1e-4, 1e-4])
        out.append(soa_to_aos(s.get_moments("conserved")))
    assert field_rel_err(out[0], out[1]).max() <= 2e-4


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("size", [[300], [97, 1200], (37, 29), (900, 700)])
def test_device_array_is_free_after_the_call(mx, precision, size):
    """A device array may be overwritten, on a stream that the solver's does not wait for,
    as soon as set_state has returned (900 x 700 cells: more than the checks copy)."""
    import torch
    rng = np.random.default_rng(3)
    if isinstance(size, tuple):
        s = mx.Solver(nx=size[0], ny=size[1], precision=precision)
        prim = aos_to_soa(wl.smooth_field14(rng, size[0], size[1], planar=False))
    else:
        s = mx.Batch(size, [1.0] * len(size), precision=precision)
        prim = s.pack([wl.smooth_field14(rng, n, 1, planar=False)[0].T for n in size])
    s.set_state(prim)
    want = s.get_moments("conserved")
    keep = torch.from_numpy(prim).cuda()
    junk = torch.full_like(keep, float("nan"))
    x = torch.empty_like(keep)
    torch.cuda.synchronize()
    for _ in range(20):
        x.copy_(keep)
        torch.cuda.synchronize()
        s.set_state(x)
        x.copy_(junk)                       # on torch's stream, at once
        assert np.array_equal(s.get_moments("conserved"), want)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("size,off", [(3e2, 0.0), (3e2, 1e-4), (3e3, 0.0), (3e3, 1e-2)])
def test_cancelling_pressures_are_refused(mx, precision, size, off):
    """A negative P_zz beside large P_xx, P_yy that cancel it in the trace, and P_xy near
    sqrt(P_xx P_yy): in FP32 the minors are noise of any sign, in FP64 they are not."""
    rng = np.random.default_rng(int(size) + int(1e6 * off))
    good = _cell([1, 0, 0, 1, 0, 1])
    s = mx.Solver(nx=8, ny=5, precision=precision)
    prim = np.repeat(good[:, None], 40, 1).reshape(14, 5, 8).copy()
    s.set_state(prim)
    want = s.get_moments("conserved")
    for _ in range(300):
        a, d = size * rng.uniform(0.2, 1.0, 2)
        b = np.sqrt(a * d) * (1.0 + rng.uniform(-1, 1) * 10.0 ** rng.uniform(-9, -6))
        xz, yz = size * off * rng.uniform(-1, 1, 2)
        prim[:, 3, 6] = good
        prim[4:10, 3, 6] = a, b, xz, d, yz, 3.0 - a - d        # tr P = 3
        prim[13, 3, 6] = 1e6                                   # sigma far below 1
        with pytest.raises(mx.MaxentError, match="input cell 30"):
            s.set_state(prim)
    assert np.array_equal(s.get_moments("conserved"), want)    # and the state is kept
