"""FP64 tubes on teams of CTAs: the split of a tube over CTAs and chunk sizes,
the planar kernel and the place of the launch (alone, batched, captured in a
graph, on several streams) change nothing in the result."""
import ctypes as C

import numpy as np
import pytest

from paper_2401_15233_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2401_15233_gb300 as mx
    return mx


def _prim(system, n, seed):
    """smooth varying states in every moment of the 1D problem"""
    g = np.random.default_rng(seed)
    x = (np.arange(n) + 0.5) / n
    f = lambda a: a * np.sin(2 * np.pi * x * g.integers(1, 3) + g.uniform(0, 6))  # noqa: E731
    rho, T, u = 1 + f(0.3), 1 + f(0.2), f(0.4)
    P = rho * T
    if system == 5:
        return np.stack([rho, u, P, P * np.sqrt(T) * f(0.1), 3 * P * T * (1.1 + f(0.02))])
    z = 0 * x
    return np.stack([rho, u, f(0.2), z, P * (1 + f(0.05)), P * f(0.04), z, P * (1 + f(0.03)), z, P,
                     P * np.sqrt(T) * f(0.1), P * np.sqrt(T) * f(0.1), z, 15 * P * T * (1.1 + f(0.02))])


def _run(mx, system, n, prim, bc, integ, steps, order=2):
    s = mx.Solver(system=system, nx=n, ny=1, integrator=integ, order=order)
    if bc == "periodic":
        s.set_bc(mx.XLO, mx.BC_PERIODIC)
        s.set_bc(mx.XHI, mx.BC_PERIODIC)
    elif bc == "dirichlet":
        s.set_bc(mx.XLO, mx.BC_DIRICHLET, state=prim[:, 0])
    s.set_relaxation(mx.TAU_HARDSPHERE, 0.1, 1.0, 1.0)
    s.set_state(prim[:, None, :])
    s.step(steps)
    return s.get_moments("conserved")[:, 0, :]


SIZES = [4, 5, 30, 31, 32, 62, 63, 64, 125, 126, 127, 700]


@pytest.mark.parametrize("system,integ", [(5, "fe"), (5, "rk2"), (14, "fe"), (14, "rk2")])
@pytest.mark.parametrize("bc", ["transmissive", "periodic", "dirichlet"])
def test_alone_and_in_a_full_batch_are_the_same(mx, system, integ, bc):
    """Alone a tube is spread over CTAs of 31 cells; among more tubes than CTA
    slots it has one CTA and chunks of 63.  Same operations per cell: bitwise."""
    steps = 3                                   # odd: forward Euler ends in the stage buffer
    prims = [_prim(system, n, 7 + n) for n in SIZES]
    if bc == "dirichlet":                       # one boundary state for all tubes of a batch
        for p in prims:
            p[:, 0] = prims[-1][:, 0]
    alone = [_run(mx, system, n, p, bc, integ, steps) for n, p in zip(SIZES, prims)]
    ncells = SIZES + [40] * 700
    b = mx.Batch(ncells, [1.0] * len(ncells), system=system, integrator=integ)
    if bc == "periodic":
        b.set_bc(mx.XLO, mx.BC_PERIODIC)
        b.set_bc(mx.XHI, mx.BC_PERIODIC)
    elif bc == "dirichlet":
        b.set_bc(mx.XLO, mx.BC_DIRICHLET, state=prims[-1][:, 0])
    b.set_relaxation(mx.TAU_HARDSPHERE, 0.1, 1.0, 1.0)
    fill = _prim(system, 40, 3)
    b.set_state(b.pack(prims + [fill] * 700))
    b.run(steps, float("inf"))
    got = b.unpack(b.get_moments("conserved"))
    for n, x, y in zip(SIZES, alone, got):
        assert np.array_equal(x, y), n


def test_one_long_tube_several_passes(mx):
    """More chunks than CTA slots (several passes a stage) against the same
    tube as a member of a full batch."""
    n = 40000
    p = _prim(14, n, 1)
    x = _run(mx, 14, n, p, "transmissive", "rk2", 2)
    ncells = [n] + [40] * 700
    b = mx.Batch(ncells, [1.0] * len(ncells), system=14)
    b.set_relaxation(mx.TAU_HARDSPHERE, 0.1, 1.0, 1.0)
    b.set_state(b.pack([p] + [_prim(14, 40, 3)] * 700))
    b.run(2, float("inf"))
    assert np.array_equal(x, b.unpack(b.get_moments("conserved"))[0])


def test_planar_and_general_agree(mx):
    """The same flow with a z velocity in the whole tube is a Galilean shift: the
    ten moments of the planar kernel against the general one."""
    n = 200
    p = _prim(14, n, 5)
    q = p.copy()
    q[3] = 1e-30                                # not planar: all 14 moments are carried
    x = _run(mx, 14, n, p, "transmissive", "rk2", 4)
    y = _run(mx, 14, n, q, "transmissive", "rk2", 4)
    nx = np.linalg.norm(x, axis=1)
    err = np.linalg.norm(x - y, axis=1) / np.where(nx > 0, nx, nx.max())
    # 4 steps of a few thousand roundings of 1.1e-16, amplified by less than 1e2 a
    # step on this smooth flow (measured by the oracle's own sensitivity)
    assert err.max() <= 1e-10


def test_two_streams_at_once_and_in_a_graph(mx):
    import torch
    n, steps = 1000, 3
    p = _prim(14, n, 2)
    want = _run(mx, 14, n, p, "transmissive", "rk2", 2 * steps)
    sol = []
    for _ in range(3):
        s = mx.Solver(system=14, nx=n, ny=1)
        torch.cuda.synchronize()
        s.set_relaxation(mx.TAU_HARDSPHERE, 0.1, 1.0, 1.0)
        s.set_state(p[:, None, :])
        sol.append(s)
    for _ in range(2):
        for s in sol:
            s.step(steps, sync=False)           # nothing waits between the contexts
    for s in sol:
        assert np.array_equal(s.get_moments("conserved")[:, 0, :], want)
    # captured: the launch and its reset are stream-ordered
    s = sol[0]
    s.set_state(p[:, None, :])
    st = torch.cuda.Stream()
    s.set_stream(st.cuda_stream)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        s.step(steps, sync=False)
    g.replay()
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(s.get_moments("conserved")[:, 0, :], want)
    # the fixed-scratch entry point, first called outside a capture
    cfg = mx.make_config(system=14, nx=n, ny=1)
    s.set_state(p[:, None, :])
    U0 = torch.from_numpy(s.get_moments("conserved").reshape(14, n)).cuda()
    U = U0.clone()
    arg = dict(tau_model=mx.TAU_HARDSPHERE, tau_ref=0.1)
    mx.mxe_tube_run_noalloc(cfg, U, 0.0, 1e9, 2 * steps, **arg)
    assert np.array_equal(U.cpu().numpy(), want)
    U.copy_(U0)
    torch.cuda.synchronize()
    g2 = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g2, stream=st):
        rc = mx.lib().mxe_tube_run_noalloc(C.byref(cfg), 0, 0, mx.TAU_HARDSPHERE, 0.1, 1.0, 1.0,
                                           C.c_void_p(U.data_ptr()), 0.0, 1e9, 2 * steps, None,
                                           None, C.c_void_p(st.cuda_stream))
    assert rc == 0
    g2.replay()
    torch.cuda.synchronize()
    assert np.array_equal(U.cpu().numpy(), want)


@pytest.mark.parametrize("shape", ["tube5", "tube14", "planar", "general"])
@pytest.mark.parametrize("limiter", ["minmod", "vanalbada"])
def test_units_scale_exactly(mx, shape, limiter):
    """Powers of two as units of density and speed scale every FP64 result
    exactly: the FP32 screening of the limiter, the seeds and the integer
    comparisons must not see the units, far outside FP32's range too."""
    system = 5 if shape == "tube5" else 14
    ny = 1 if shape.startswith("tube") else 20
    n = 150 if ny == 1 else 37

    def run(a, b):
        if ny == 1:
            p = _prim(system, n, 11)[:, None, :]
        else:
            p = np.moveaxis(wl.smooth_field14(np.random.default_rng(4), n, ny,
                                              planar=shape == "planar"), -1, 0).copy()
        # flat stretches and opposite differences too
        p[:, :, n // 3:n // 2] = p[:, :, n // 3:n // 3 + 1]
        w = [0, 1, 2, 3, 4] if system == 5 else [0, 1, 1, 1] + [2] * 6 + [3] * 3 + [4]
        for k in range(system):
            p[k] *= 2.0 ** (a + b * w[k]) if k == 0 or w[k] != 1 else 2.0 ** b
        s = mx.Solver(system=system, nx=n, ny=ny, limiter=limiter)
        s.set_state(p)
        t, _ = s.step(2)
        U = s.get_moments("conserved")
        return t * 2.0 ** b, np.stack([U[k] / 2.0 ** (a + b * w[k]) for k in range(system)])

    t0, U0 = run(0, 0)
    for a, b in ((-100, 0), (90, 10), (-150, 40), (20, -60)):
        t, U = run(a, b)
        assert t == t0
        assert np.array_equal(U, U0)
