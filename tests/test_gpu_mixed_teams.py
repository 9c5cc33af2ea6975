"""Mixed tubes on teams of CTAs across the chip (the launch the library picks
for few tubes): the split over CTAs changes nothing in the result, which is
bitwise that of one CTA a tube."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2401_15233_gb300 as mx
    return mx


def _prim(n, seed, planar):
    """smooth varying states in every moment (or every planar one)"""
    g = np.random.default_rng(seed)
    x = (np.arange(n) + 0.5) / n
    f = lambda a: a * np.sin(2 * np.pi * x * g.integers(1, 3) + g.uniform(0, 6))  # noqa: E731
    rho, T, u = 1 + f(0.3), 1 + f(0.2), f(0.4)
    P = rho * T
    z = 0 * x if planar else 1.0
    h = P * np.sqrt(T)
    return np.stack([rho, u, f(0.2), z * f(0.1), P * (1 + f(0.05)), P * f(0.04), z * P * f(0.03),
                     P * (1 + f(0.03)), z * P * f(0.02), P, h * f(0.1), h * f(0.1), z * h * f(0.1),
                     15 * P * T * (1.1 + f(0.02))])


def _march(b, prims, bc, steps, mx, dts=None):
    if bc == "periodic":
        b.set_bc(mx.XLO, mx.BC_PERIODIC)
        b.set_bc(mx.XHI, mx.BC_PERIODIC)
    b.set_relaxation(mx.TAU_HARDSPHERE, 0.1, 1.0, 1.0)
    b.set_state(b.pack(prims))
    for s in steps:                             # several runs: clocks and graph carry over
        b.run(s, float("inf"))
    return b.unpack(b.get_moments("conserved"))


# one chunk is 126 cells; 90000 cells are more chunks than CTA slots
@pytest.mark.parametrize("sizes", [[4], [125], [126], [127], [252, 253, 4, 700], [90000, 5]])
@pytest.mark.parametrize("planar", [True, False])
@pytest.mark.parametrize("integ,bc", [("rk2", "transmissive"), ("fe", "periodic")])
def test_teams_match_one_cta_a_tube(mx, sizes, planar, integ, bc):
    prims = [_prim(n, n, planar) for n in sizes]
    out = []
    for shape in (None, (128, 1)):
        b = mx.Batch(sizes, [1.0] * len(sizes), precision="mixed", integrator=integ)
        if shape:
            b.set_shape(*shape)
        out.append(_march(b, prims, bc, (17, 2), mx))
        assert b.layout()[0] <= len(sizes)
    for n, x, y in zip(sizes, *out):
        assert np.array_equal(x, y), n


def test_single_tube_to_a_time_and_prescribed_steps(mx):
    n = 1000
    p = _prim(n, 3, True)
    got = []
    for make in (lambda: mx.Solver(nx=n, ny=1, precision="mixed"),
                 lambda: mx.Batch([n], [1.0], precision="mixed")):
        s = make()
        if isinstance(s, mx.Batch):
            s.set_shape(128, 1)
        s.set_relaxation(mx.TAU_HARDSPHERE, 0.1, 1.0, 1.0)
        s.set_state(s.pack([p]) if isinstance(s, mx.Batch) else p[:, None, :])
        if isinstance(s, mx.Batch):
            s.run(10**6, 0.01)
        else:
            t, k = s.step(10**6, 0.01)
            assert t == 0.01 and k > 10
        s.step_dt([1e-5, 2e-5, 1e-5])
        got.append(s.get_moments("conserved").reshape(-1))
    assert np.array_equal(*got)


@pytest.mark.parametrize("sizes", [[8192], [700] * 9])
def test_autotune_keeps_the_teams_where_they_are_faster(mx, sizes):
    """A tuned batch of few tubes is no slower than an untuned one (measured: the teams of one
    8192-cell tube take under a tenth of the best shape's time)."""
    import time
    b = mx.Batch(sizes, [1.0] * len(sizes), precision="mixed")
    prims = [_prim(n, n, True) for n in sizes]
    state = b.pack(prims)

    def ms():
        best = np.inf
        for _ in range(5):
            b.set_state(state)
            t = time.perf_counter()
            b.run(400, float("inf"))
            b.clock()
            best = min(best, time.perf_counter() - t)
        return 1e3 * best

    own = ms()
    b.set_state(state)
    nt, cl, kept = b.autotune(1e-3)
    tuned = ms()
    assert nt in (128, 256) and cl in (1, 2, 4, 8) and kept > 0
    assert tuned <= 1.5 * own
    b.set_shape(nt, cl)                         # and a chosen shape still counts
    assert ms() > 1.5 * own or len(sizes) > 1


# a warp's chunk is 30 cells, a CTA's pass 120: the edges of both, and of one CTA and two
@pytest.mark.parametrize("sizes", [[29], [30], [31], [60, 61], [119], [120], [121], [240, 241, 59]])
@pytest.mark.parametrize("planar", [True, False])
@pytest.mark.parametrize("integ,bc", [("rk2", "transmissive"), ("fe", "periodic")])
def test_chunk_edges(mx, sizes, planar, integ, bc):
    prims = [_prim(n, n, planar) for n in sizes]
    out = []
    for shape in (None, (128, 1), (256, 2)):
        b = mx.Batch(sizes, [1.0] * len(sizes), precision="mixed", integrator=integ)
        if shape:
            b.set_shape(*shape)
        out.append(_march(b, prims, bc, (17, 2), mx))
    for got in out[1:]:
        for n, x, y in zip(sizes, out[0], got):
            assert np.array_equal(x, y), n
