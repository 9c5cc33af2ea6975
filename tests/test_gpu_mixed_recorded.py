"""The mixed path's results on record: planar runs of the packed 2D stage, and tubes.

Where a field passes an extremum, the shared limiter turns on the last bits of the
FP32 primitives, and two roundings of the same formulas end up as far from one
another as either is from an FP64 march (1e-3 of a value in a cell of some
tubes).  So the roundings of the mixed stages are part of their results:
tests/golden/mixed_recorded.txt holds, for each run below, the time and a
checksum of the final state rounded to FP32, from the stages as they were
first written, and a change of arithmetic shows here.  Equality is exact: the
same operations on one kind of GPU give the same bits, whatever the tile, the
team or the order of the blocks.

Inputs are formed with +, -, * and / alone, which every host rounds alike.
"""
import os
import zlib

import numpy as np
import pytest

import paper_2401_15233_gb300 as mx

pytestmark = pytest.mark.gpu

RECORD = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "mixed_recorded.txt")

# name: (grid (nx, ny) or tube lengths, flux, limiter, steps, relaxation model)
RUNS = {
    "grid_97x65_hll_minmod": ((97, 65), "hll", "minmod", 8, mx.TAU_HARDSPHERE),
    "grid_331x260_hll_minmod": ((331, 260), "hll", "minmod", 20, mx.TAU_HARDSPHERE),
    "grid_450x440_hll_minmod": ((450, 440), "hll", "minmod", 6, mx.TAU_HARDSPHERE),
    "grid_640x600_hll_minmod": ((640, 600), "hll", "minmod", 6, mx.TAU_HARDSPHERE),
    "grid_450x450_rusanov_vanalbada": ((450, 450), "rusanov", "vanalbada", 6, mx.TAU_HARDSPHERE),
    "grid_700x690_rusanov_minmod": ((700, 690), "rusanov", "minmod", 6, mx.TAU_CONST),
    "grid_61x50_hll_vanalbada": ((61, 50), "hll", "vanalbada", 8, mx.TAU_CONST),
    "grid_120x83_rusanov_minmod": ((120, 83), "rusanov", "minmod", 8, mx.TAU_NONE),
    "tubes_hll_minmod": ([97, 240, 241, 700, 1531], "hll", "minmod", 40, mx.TAU_HARDSPHERE),
    "tubes_hll_vanalbada": ([64, 391], "hll", "vanalbada", 40, mx.TAU_NONE),
    "tubes_rusanov_minmod": ([119, 620], "rusanov", "minmod", 40, mx.TAU_CONST),
    "general_tubes_hll_minmod": ([97, 240, 1531], "hll", "minmod", 40, mx.TAU_HARDSPHERE),
    "general_tubes_rusanov_vanalbada": ([119, 620], "rusanov", "vanalbada", 40, mx.TAU_NONE),
}
TUBE_SHAPES = {"teams": None, "128x1": (128, 1), "256x8": (256, 8)}


def _conserved(rho, ux, uy, p, a, b, q, k):
    """Conserved fields of a planar state with pressures p(1+a), p(1+b), p(1-a-b), P_xy = 0,
    heat flux (q, -q/2) and fourth moment 15 k p^2 / rho."""
    Pxx, Pyy, Pzz = p * (1.0 + a), p * (1.0 + b), p * (1.0 - a - b)
    qx, qy, R = q, -0.5 * q, 15.0 * k * p * p / rho
    u2, tr = ux * ux + uy * uy, Pxx + Pyy + Pzz
    z = 0.0 * rho
    Pux, Puy = Pxx * ux, Pyy * uy
    return np.stack([
        rho, rho * ux, rho * uy, z, rho * ux * ux + Pxx, rho * ux * uy, z, rho * uy * uy + Pyy, z,
        Pzz, ux * (rho * u2 + tr) + 2.0 * Pux + qx, uy * (rho * u2 + tr) + 2.0 * Puy + qy, z,
        rho * u2 * u2 + 2.0 * u2 * tr + 4.0 * (ux * Pux + uy * Puy) + 4.0 * (ux * qx + uy * qy)
        + R])


def _state(x, y):
    """A gas expanding along x and y, out of equilibrium, with a swell in every field."""
    s = 16.0 * x * (1.0 - x) * (0.5 - x) * (1.0 + 0.3 * y)
    rho = 1.0 / (1.0 + 1.3 * x + 0.9 * y) + 0.05 * s
    ux, uy = 0.4 + 0.6 * x + 0.2 * y, 0.3 + 0.2 * x + 0.5 * y - 0.05 * s
    p = rho * (1.0 - 0.25 * x - 0.2 * y)
    return _conserved(rho, ux, uy, p, 0.1 + 0.05 * x, -0.05 - 0.04 * y, 0.12 * p * (1.0 + 0.4 * s),
                      1.12 + 0.1 * x)


def _general(x):
    """Primitives with all 14 moments along a tube."""
    s = 16.0 * x * (1.0 - x) * (0.5 - x)
    rho = 1.0 / (1.0 + 1.3 * x) + 0.05 * s
    p = rho * (1.0 - 0.25 * x)
    return np.stack([rho, 0.4 + 0.6 * x, 0.3 - 0.2 * x, 0.1 + 0.2 * x + 0.04 * s, p * (1.1 + 0.05 * x),
                     p * (0.06 - 0.03 * x), p * (0.04 + 0.02 * s), p * 0.95, p * (0.03 + 0.02 * x),
                     p * (0.95 - 0.05 * x), 0.12 * p * (1.0 + 0.4 * s), 0.1 * p * (1.0 - 0.3 * x),
                     0.08 * p * (1.0 + x), 15.0 * p * p / rho * (1.12 + 0.1 * x)])


def march(name, shape=None):
    """Times (one a tube) and the final conserved state in FP32."""
    size, flux, limiter, steps, tau = RUNS[name]
    general = name.startswith("general")
    kw = dict(system=14, precision="mixed", flux=flux, limiter=limiter)
    if isinstance(size, tuple):
        nx, ny = size
        s = mx.Solver(nx=nx, ny=ny, **kw)
        x, y = ((np.arange(n) + 0.5) / n for n in (nx, ny))
        U = _state(*np.broadcast_arrays(x[None, :], y[:, None]))
    else:
        s = mx.Batch(size, [1.0] * len(size), **kw)
        if shape:
            s.set_shape(*shape)
        x = [(np.arange(n) + 0.5) / n for n in size]
        U = np.concatenate([(_general(v) if general else _state(v, 0.0 * v)).reshape(-1) for v in x])
    s.set_relaxation(tau, 0.05, 1.0, 1.0)
    s.set_state(np.ascontiguousarray(U), kind="primitive" if general else "conserved")
    if isinstance(size, tuple):
        t = [s.step(steps)[0]]
    else:
        s.run(steps, float("inf"))
        t = list(s.clock()[0])
    V = np.asarray(s.get_moments("conserved"))
    s.close()
    return [float(v) for v in t], V.astype(np.float32)


def line(name, t, V):
    return " ".join([name, "%08x" % zlib.crc32(np.ascontiguousarray(V).tobytes())]
                    + [v.hex() for v in t])


def _recorded():
    with open(RECORD) as f:
        return {ln.split()[0]: ln.strip() for ln in f if ln.strip() and not ln.startswith("#")}


@pytest.mark.parametrize("name,shape", [(n, s) for n, r in RUNS.items()
                                        for s in (TUBE_SHAPES if isinstance(r[0], list) else [None])])
def test_as_recorded(name, shape):
    t, V = march(name, TUBE_SHAPES.get(shape))
    assert np.isfinite(V).all()
    assert line(name, t, V) == _recorded()[name]
