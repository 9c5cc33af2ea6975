"""Performance cases: what programs have this solver do, through its Python entry points.

A case is one simulation segment as a driver program runs it: primitive
moments on the device go in (``set_state``), the solver marches a number of
steps, the conserved moments come back on the device (``get_moments``).  The
context, its boundary conditions, relaxation and mixed-precision settings are
prepared once, as such a program does.  Kinds:

  grid     one 2D grid (or, with ny == 1, one 1D problem) in a Solver
  batch    independent uneven tubes in one Batch
  adjoint  a recorded segment and its reverse sweep on a 2D grid

The flows are smooth over the steps of a pass: the scheme's shared limiter
makes rough ones sensitive to the last bit.  Runs of the mixed path and of the
FP32 face-state reverse hand their results on as float32, the precision of
those stages; FP64 runs as float64.
"""
import math

import numpy as np
import torch

import paper_2401_15233_gb300 as mx

SIGMA_LIM = 1e-4
GAMMA = 5.0 / 3.0


# ------------------------------------------------------------------ the cases
def _case(name, kind, **kw):
    c = dict(name=name, kind=kind, system=14, nx=64, ny=1, precision="fp64", flow="sod",
             flux="hll", limiter="minmod", order=2, integrator="rk2", source="explicit",
             reverse="fp64", kn=0.1, steps=4)
    c.update(kw)
    return c


def listed():
    return [
        # The 1D1V Sod tube of the repository's first configuration: 1000 cells,
        # first order, forward Euler.  A single small 1D problem: latency.
        _case("sod5_1000", "grid", system=5, nx=1000, order=1, integrator="fe", kn=0.01,
              steps=100),
        # The 14-moment Sod tube at its stated 4096 cells, all-FP64 (second configuration).
        _case("sod14_4096_fp64", "grid", nx=4096, kn=0.01, steps=10),
        # The same tube in mixed precision, with the launch the library picks by itself.
        _case("sod14_4096_mixed", "grid", nx=4096, precision="mixed", kn=1.0, steps=50),
        # A parameter study: 256 uneven tubes, log-uniform lengths and Knudsen numbers
        # (fourth configuration), at the block shape the autotuner settles on.
        _case("batch256_mixed", "batch", precision="mixed", tubes=256, nmin=512, nmax=8192,
              nt=256, cl=8, steps=40),
        # A small FP64 study: fewer tubes than SMs, short and ragged.
        _case("batch24_fp64", "batch", tubes=24, nmin=100, nmax=700, nt=0, cl=0, steps=4),
        # Crossed jets at the benchmark's size: 4096 x 4096, mixed precision.
        _case("jets_4096_mixed", "grid", nx=4096, ny=4096, precision="mixed", flow="plume",
              steps=6),
        # Crossed jets of the third configuration: 1024 x 1024, mixed precision.
        _case("jets_1024_mixed", "grid", nx=1024, ny=1024, precision="mixed", flow="plume",
              steps=20),
        # A coarse set-up run of the same, ragged: launches and latency count.
        _case("jets_97x65_mixed", "grid", nx=97, ny=65, precision="mixed", flow="plume", steps=4),
        # A flow with all 14 moments, with the paper's own flux and limiter choice (Rusanov,
        # van Albada), mixed precision, odd sizes.
        _case("general_mixed", "grid", nx=777, ny=1001, precision="mixed", flow="plume3",
              flux="rusanov", limiter="vanalbada", steps=6),
        # All-FP64 crossed jets at the adjoint configuration's size: the reference the
        # mixed path is checked against.
        _case("jets_512_fp64", "grid", nx=512, ny=512, flow="jets", steps=2),
        # All 14 moments in FP64 on a small ragged grid, periodic, point-implicit source.
        _case("general_61x47_fp64", "grid", nx=61, ny=47, flow="periodic",
              source="point_implicit", kn=1e-3, steps=3),
        # Gradients: a recorded segment of the jets and its reverse sweep, FP64.
        _case("adjoint_128_fp64", "adjoint", nx=128, ny=128, flow="plume", steps=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges; the largest cost no more than jets_4096_mixed."""
    kind = rng.choice(["tube5", "tube14", "tube14m", "batch", "batchm", "grid", "grid", "gridm",
                       "gridm", "gridm", "adjoint"])
    kn = math.exp(rng.uniform(math.log(1e-2), math.log(3.0)))
    common = dict(kn=kn, flux=rng.choice(["hll", "hll", "rusanov"]),
                  limiter=rng.choice(["minmod", "minmod", "vanalbada"]))
    if kind == "tube5":
        second = rng.random() < 0.5
        c = _case("", "grid", system=5, nx=_log_int(rng, 200 if second else 40, 16000),
                  order=2 if second else 1, integrator="rk2" if second else "fe",
                  steps=rng.randint(3, 12) if second else rng.randint(10, 60), **common)
    elif kind == "tube14":
        c = _case("", "grid", nx=_log_int(rng, 200, 9000), steps=rng.randint(2, 5), **common)
    elif kind == "tube14m":
        c = _case("", "grid", nx=_log_int(rng, 400, 30000), precision="mixed",
                  steps=rng.randint(8, 24), **common)
    elif kind == "batch":
        c = _case("", "batch", system=rng.choice([5, 14]), tubes=_log_int(rng, 2, 200), nmin=100,
                  nmax=900, nt=0, cl=0, steps=rng.randint(2, 4), **common)
    elif kind == "batchm":
        c = _case("", "batch", precision="mixed", tubes=_log_int(rng, 4, 300), nmin=400,
                  nmax=_log_int(rng, 1000, 8192), nt=rng.choice([128, 256]),
                  cl=rng.choice([1, 2, 4, 8]), steps=rng.randint(8, 24), **common)
    elif kind == "grid":
        flow = rng.choice(["jets", "plume", "plume3", "periodic"])
        c = _case("", "grid", nx=_log_int(rng, 24, 700), ny=_log_int(rng, 24, 700), flow=flow,
                  steps=rng.randint(1, 2), **common)
    elif kind == "gridm":
        flow = rng.choice(["plume", "plume", "plume3"])
        top = 3500 if flow == "plume" else 2000
        c = _case("", "grid", nx=_log_int(rng, 48, top), ny=_log_int(rng, 48, top), flow=flow,
                  precision="mixed", steps=rng.randint(1, 4), **common)
    else:
        c = _case("", "adjoint", nx=_log_int(rng, 32, 200), ny=_log_int(rng, 32, 200),
                  flow="plume", steps=rng.randint(2, 3), kn=kn, order=rng.choice([1, 2, 2]),
                  reverse=rng.choice(["fp64", "fp64", "mixed"]))
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _mixture14(comps):
    """Primitive moments (14, ...) of a sum of Maxwellians [(rho, (ux, uy, uz), T), ...]:
    realizable, with pressure anisotropy, heat flux and excess kurtosis where they overlap."""
    rho = sum(c[0] for c in comps)
    u = [sum(c[0] * c[1][d] for c in comps) / rho for d in range(3)]
    P = [[0.0] * 3 for _ in range(3)]
    q, R = [0.0] * 3, 0.0
    for ra, ua, T in comps:
        c = [ua[d] - u[d] for d in range(3)]
        c2 = c[0] * c[0] + c[1] * c[1] + c[2] * c[2]
        for i in range(3):
            for j in range(i, 3):
                P[i][j] = P[i][j] + ra * ((T if i == j else 0.0) + c[i] * c[j])
            q[i] = q[i] + ra * c[i] * (c2 + 5.0 * T)
        R = R + ra * (c2 * c2 + 10.0 * T * c2 + 15.0 * T * T)
    return torch.stack([rho, u[0], u[1], u[2], P[0][0], P[0][1], P[0][2], P[1][1], P[1][2],
                        P[2][2], q[0], q[1], q[2], R])


def _centres(n, dev):
    return (torch.arange(n, dtype=torch.float64, device=dev) + 0.5) / n


def _tube(system, n, gen, dev):
    """The expansion side of a burst shock tube: density falling by a factor of 4 to 20, the gas
    accelerating and cooling along the tube, out of equilibrium throughout."""
    x = _centres(n, dev)
    rho = torch.exp(-gen.uniform(math.log(4.0), math.log(20.0)) * x)
    u = gen.uniform(0.1, 0.3) + gen.uniform(0.5, 0.9) * x
    T = 1.0 - gen.uniform(0.2, 0.4) * x
    P = rho * T
    th = P / rho
    heat = rho * th ** 1.5 * gen.uniform(0.1, 0.3) * (1.0 + 0.5 * x)
    if system == 5:
        return torch.stack([rho, u, P, heat, 3.0 * P * P / rho * (1.1 + 0.2 * x)])
    a = gen.uniform(0.1, 0.2) * (1.0 + x)
    zero = 0.0 * x
    return torch.stack([rho, u, zero, zero, P * (1.0 + a), zero, zero, P * (1.0 - 0.5 * a), zero,
                        P * (1.0 - 0.5 * a), heat, zero, zero,
                        15.0 * P * P / rho * (1.1 + 0.2 * x)])


def _jet_states(gen):
    """The imposed inflow states: Maxwellians at rho = T = 1 and Mach 2.5 to 3.5."""
    a = math.sqrt(GAMMA)
    m1, m2 = gen.uniform(2.5, 3.5), gen.uniform(2.5, 3.5)
    one = [0.0] * 14
    one[0] = one[4] = one[7] = one[9] = 1.0
    one[13] = 15.0
    left, bottom = list(one), list(one)
    left[1], bottom[2] = m1 * a, m2 * a
    return np.array(left), np.array(bottom)


def _jets(nx, ny, left, bottom, gen, dev):
    """Developed crossed jets on [0, 1]^2: background gas and two spreading beams, bimodal where
    they cross."""
    X, Y = _centres(nx, dev)[None, :], _centres(ny, dev)[:, None]
    reach = gen.uniform(0.7, 0.9)

    def beam(s, n):
        w = 0.05 + 0.35 * s
        return (0.5 * (1.0 - torch.tanh((n.abs() - w) / (0.02 + 0.05 * s))) * (0.05 / w) * 0.5
                * (1.0 - torch.tanh((s - reach) / 0.05)))

    zero = torch.zeros((ny, nx), dtype=torch.float64, device=dev)
    return _mixture14([(zero + 1e-3, (zero, zero, zero), 1.0),
                       (beam(X, Y - 0.5) + 1e-12 + zero, (float(left[1]), zero, zero), 1.0),
                       (beam(Y, X - 0.5) + 1e-12 + zero, (zero, float(bottom[2]), zero), 1.0)])


def _plume(nx, ny, gen, dev, planar):
    """The expanding gas behind the jets' crossing: density falling towards the far corner, the
    gas accelerating and cooling, sheared and out of equilibrium throughout (planar or with all
    14 moments).  Returns the cells' states and two upstream ones for the inflow slots."""
    c = [gen.uniform(0.8, 1.2, size=3) for _ in range(16)]

    def at(X, Y):
        def f(n, c0, cx, cy):
            return c0 * c[n][0] + cx * c[n][1] * X + cy * c[n][2] * Y

        rho = torch.exp(-f(0, 0.0, 1.1, 1.1))
        ux, uy = f(1, 1.2, 0.7, 0.3), f(2, 1.2, 0.3, 0.7)
        T = f(3, 1.0, -0.2, -0.2)
        P = rho * T
        a, b = f(4, 0.08, 0.08, 0.04), -f(5, 0.08, 0.04, 0.08)
        h = P * torch.sqrt(T)
        zero = 0.0 * P
        uz, Pxz, Pyz, qz = zero, zero, zero, zero
        if not planar:
            uz, Pxz, Pyz = f(6, 0.3, 0.2, 0.3), P * f(7, 0.05, 0.04, 0.05), P * f(8, 0.04, 0.05, 0.04)
            qz = h * f(9, 0.1, 0.1, 0.12)
        R = 15.0 * P * P / rho * (1.15 + f(10, 0.0, 0.1, 0.12))
        return torch.stack([rho, ux, uy, uz, P * (1.0 + a), P * f(11, 0.06, 0.06, 0.06), Pxz,
                            P * (1.0 + b), Pyz, P * (1.0 - a - b), h * f(12, 0.15, 0.15, 0.12),
                            h * f(13, 0.15, 0.12, 0.2), qz, R])

    X = _centres(nx, dev)[None, :].expand(ny, nx)
    Y = _centres(ny, dev)[:, None].expand(ny, nx)
    up = [torch.tensor(v, dtype=torch.float64) for v in ((-0.03, 0.5), (0.5, -0.03))]
    return at(X, Y), at(*up[0]).numpy(), at(*up[1]).numpy()


def _waves(nx, ny, gen, dev):
    """Smooth periodic overlap of three streaming gases."""
    X, Y = _centres(nx, dev)[None, :], _centres(ny, dev)[:, None]
    w = []
    for _ in range(3):
        k, l, ph = gen.integers(1, 3), gen.integers(1, 3), gen.uniform(0, 2 * math.pi)
        w.append(1.0 + 0.3 * torch.sin(2 * math.pi * (int(k) * X + int(l) * Y) + float(ph)))
    v = gen.uniform(-0.8, 0.8, size=(3, 3))
    T = gen.uniform(0.7, 1.3, size=3)
    zero = torch.zeros((ny, nx), dtype=torch.float64, device=dev)
    return _mixture14([(w[n] + zero, tuple(float(v[n, d]) + zero for d in range(3)), float(T[n]))
                       for n in range(3)])


def _lengths(case):
    """Cells of a batch's tubes, log-uniform: the study's parameter list, whatever the seed."""
    gen = np.random.default_rng(case["tubes"])
    n = gen.uniform(math.log(case["nmin"]), math.log(case["nmax"]), case["tubes"])
    return [int(round(x)) for x in np.exp(n)]


def _tau_ref(kn, length):
    return kn * length / math.sqrt(8.0 / math.pi)


SLOT = (0.45, 0.55)


def _setup(case, seed):
    """Everything a case is made of, from the seed alone: primitive states and boundary and
    relaxation parameters (shared by the program under test and by exact())."""
    dev = _device()
    gen = np.random.default_rng(seed)
    d = {}
    if case["kind"] == "batch":
        d["ncells"] = _lengths(case)
        d["prims"] = [_tube(case["system"], n, gen, dev) for n in d["ncells"]]
        d["taus"] = [_tau_ref(case["kn"] * math.exp(gen.uniform(-1, 1)), 1.0)
                     for _ in d["ncells"]]
        return d
    if case["ny"] == 1:
        d["prim"] = _tube(case["system"], case["nx"], gen, dev)[:, None, :].contiguous()
        d["tau"] = _tau_ref(case["kn"], 1.0)
        return d
    if case["flow"] == "periodic":
        d["prim"] = _waves(case["nx"], case["ny"], gen, dev)
        d["tau"] = _tau_ref(case["kn"], 1.0)
        return d
    d["tau"] = _tau_ref(case["kn"], 0.1)
    if case["flow"] == "jets":
        d["left"], d["bottom"] = _jet_states(gen)
        d["prim"] = _jets(case["nx"], case["ny"], d["left"], d["bottom"], gen, dev)
    else:
        d["prim"], left, bottom = _plume(case["nx"], case["ny"], gen, dev,
                                         case["flow"] != "plume3")
        if case["precision"] == "fp64":      # a slot's edge is where FP32 rounding shows first
            d["left"], d["bottom"] = left, bottom
    if case["kind"] == "adjoint":
        # step sizes of an earlier forward run, and the sensitivity of the output to the final
        # state (a smooth weight on every field)
        h = 1.0 / max(case["nx"], case["ny"])
        d["dts"] = [0.03 * h * (1.0 + 0.1 * gen.uniform()) for _ in range(case["steps"])]
        X, Y = _centres(case["nx"], dev)[None, :], _centres(case["ny"], dev)[:, None]
        ub = torch.zeros_like(d["prim"])
        for k in (0, 1, 2, 4, 5, 7, 9, 10, 11, 13):
            a, b = gen.uniform(0.5, 2.0, size=2)
            ub[k] = torch.cos(float(a) * 3 * X + float(b) * 2 * Y + k)
        d["ubar"] = ub
    return d


# ------------------------------------------------------------------ the program under test
def prepare(case, seed):
    d = _setup(case, seed)
    wait = torch.cuda.synchronize       # set-up on several streams: one thing after another
    st = {"case": case, "stream": torch.cuda.Stream()}
    kw = dict(system=case["system"], precision=case["precision"], flux=case["flux"],
              limiter=case["limiter"], order=case["order"], integrator=case["integrator"],
              cfl=0.5, sigma_lim=SIGMA_LIM)
    if case["kind"] == "batch":
        s = mx.Batch(d["ncells"], [1.0] * case["tubes"], **kw)
        wait()
        for b, tau in enumerate(d["taus"]):
            s.set_tube_relaxation(b, mx.TAU_HARDSPHERE, tau, 1.0, 1.0)
        if case["nt"]:
            s.set_shape(case["nt"], case["cl"])
        st["prim"] = torch.cat([p.reshape(-1) for p in d["prims"]])
        st["out"] = torch.empty_like(st["prim"])
    else:
        s = mx.Solver(nx=case["nx"], ny=case["ny"], **kw)
        wait()
        if case["ny"] > 1 and case["flow"] == "periodic":
            for side in (mx.XLO, mx.XHI, mx.YLO, mx.YHI):
                s.set_bc(side, mx.BC_PERIODIC)
        elif "left" in d:
            s.set_bc(mx.XLO, mx.BC_DIRICHLET, SLOT[0], SLOT[1], d["left"])
            s.set_bc(mx.YLO, mx.BC_DIRICHLET, SLOT[0], SLOT[1], d["bottom"])
        s.set_relaxation(mx.TAU_HARDSPHERE, d["tau"], 1.0, 1.0)
        s.set_source_scheme(case["source"])
        st["prim"] = d["prim"].contiguous()
        st["out"] = torch.empty_like(st["prim"])
        if case["kind"] == "adjoint":
            s.set_adjoint_precision(case["reverse"])
            s.set_adjoint_limiter("frozen")      # the common linearisation of limited schemes
            st["dts"], st["ubar"] = d["dts"], d["ubar"].contiguous()
            st["work"] = torch.empty_like(st["ubar"])
    # the solver's work on the program's own stream, beside its torch work
    s.set_stream(st["stream"].cuda_stream)
    wait()
    st["solver"] = s
    return st


def run(st):
    case, s = st["case"], st["solver"]
    with torch.cuda.stream(st["stream"]):
        s.set_state(st["prim"])
        if case["kind"] == "adjoint":
            s.adjoint_record(st["dts"])
            st["work"].copy_(st["ubar"])
            gbar, taubar = s.adjoint_run(st["work"])
            taubar = np.array([taubar])
            if case["reverse"] == "mixed":
                return {"ubar": st["work"].float(), "gbar": gbar.astype(np.float32),
                        "taubar": taubar.astype(np.float32)}
            return {"ubar": st["work"], "gbar": gbar, "taubar": taubar}
        if case["kind"] == "batch":
            s.run(case["steps"], float("inf"))
            t, n = s.clock()
        else:
            t, n = s.step(case["steps"])
            t, n = np.array([t]), np.array([n])
        s.get_moments("conserved", out=st["out"])
        if case["precision"] == "mixed":
            return {"U": st["out"].float(), "t": t.astype(np.float32), "steps": n}
        return {"U": st["out"], "t": t, "steps": n}


def work(case):
    """Bytes: the given and the returned state once, and the active moments of every cell read
    and written once a step.  Operations: per cell and stage, two face states a direction
    (closure, flux, wave speeds) and one limiter, with the update; a reverse stage three times."""
    if case["kind"] == "batch":
        cells = sum(_lengths(case))
    else:
        cells = case["nx"] * case["ny"]
    nf = case["system"]
    planar = nf == 14 and case["flow"] not in ("periodic", "plume3")
    active = 10 if planar else nf
    dims = 2 if case["ny"] > 1 else 1
    face = 110 if nf == 5 else 330 if planar else 620       # a face state's operations
    stage = dims * (2 * face + 8 * active) + 12 * active
    stages = case["steps"] * (2 if case["integrator"] == "rk2" else 1)
    flops = cells * stages * stage * (4 if case["kind"] == "adjoint" else 1)
    move = cells * 8 * (2 * nf + 2 * active * case["steps"])
    return {"bytes": float(move), "flops": float(flops)}


# ------------------------------------------------------------------ the same in plain torch, FP64
def _sqrt(x):
    """sqrt with derivative 0 at 0."""
    ok = x > 0
    return torch.where(ok, torch.sqrt(torch.where(ok, x, torch.ones_like(x))), 0.0 * x)


def _flat_scales(Q, nf):
    """Squared natural scales of the fields at the centre cell: rho, sqrt(p/rho), p,
    p sqrt(p/rho), p^2/rho."""
    rho = Q[0]
    p = Q[2] if nf == 5 else (Q[4] + Q[7] + Q[9]) / 3.0
    by = [rho * rho, p / rho, p * p, p ** 3 / rho, (p * p / rho) ** 2]
    kinds = [0, 1, 2, 3, 4] if nf == 5 else [0, 1, 1, 1, 2, 2, 2, 2, 2, 2, 3, 3, 3, 4]
    return [by[k] for k in kinds]


def _phi(Qm, Q0, Qp, limiter, nf):
    """The shared most-stringent limiter of the cells Q0 with neighbours Qm and Qp; a field
    whose two differences are both within 1e-10 of its natural scale does not limit."""
    phis, scales = [], _flat_scales(Q0, nf)
    for k in range(nf):
        a, b = Q0[k] - Qm[k], Qp[k] - Q0[k]
        up = a * b > 0
        if limiter == "vanalbada":
            den = a * a + b * b
            v = 2.0 * a * b / torch.where(up, den, torch.ones_like(den))
        else:
            den = 0.5 * (a.abs() + b.abs())
            v = torch.minimum(a.abs(), b.abs()) / torch.where(up, den, torch.ones_like(den))
        m = torch.maximum(a.abs(), b.abs())
        flat = (m * m <= 1e-20 * scales[k]) | (m == 0)
        phis.append(torch.where(flat, torch.ones_like(v), torch.where(up, v, torch.zeros_like(v))))
    s = torch.stack(phis)
    return torch.gather(s, 0, s.detach().argmin(0, keepdim=True))[0]


def _sig(a, b):
    return [[0, 1, 2], [1, 3, 4], [2, 4, 5]][a][b]


def _mm(A, B):
    """Product of commuting symmetric 3 x 3 fields, packed (xx, xy, xz, yy, yz, zz)."""
    return [sum(A[_sig(i, k)] * B[_sig(k, j)] for k in range(3))
            for i, j in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))]


def _solve3(A, v):
    c = [A[3] * A[5] - A[4] * A[4], A[2] * A[4] - A[1] * A[5], A[1] * A[4] - A[2] * A[3],
         A[0] * A[5] - A[2] * A[2], A[1] * A[2] - A[0] * A[4], A[0] * A[3] - A[1] * A[1]]
    det = A[0] * c[0] + A[1] * c[1] + A[2] * c[2]
    return [sum(c[_sig(i, j)] * v[j] for j in range(3)) / det for i in range(3)]


def _sigma_bar(A, X, T):
    rt = _sqrt(A * A + X)
    pos = A >= 0
    s = torch.where(pos, A + rt, X) / (4.0 * T * torch.where(pos, torch.ones_like(A), rt - A))
    return s.clamp(SIGMA_LIM, 1.0)


def _bracket(z, D0):
    D = z * z + D0
    ok = D > 0
    rt = torch.where(ok, _sqrt(D), z.abs() + 1.0)
    v = torch.where(z >= 0, z + rt, D0 / torch.where(z >= 0, torch.ones_like(z), rt - z))
    return torch.where(ok, v, z)


def _speed_terms(sb, Pkk):
    r = _sqrt(sb)
    C = _sqrt((3.0 - 3.0 * sb) * Pkk)
    E = 0.8 * C
    B = 5.0 - 4.0 * r + _sqrt((10.0 - 16.0 * r + 6.0 * sb).clamp(min=0.0))
    return C, E, (_sqrt(B) - E) ** 2


def _speeds14(Q, d, K):
    Pkk, sb = d["P"][_sig(K, K)], d["sb"]
    E1, E2 = (K + 1) % 3, (K + 2) % 3
    qp2 = d["q"][E1] ** 2 + d["q"][E2] ** 2
    qp = _sqrt(qp2)
    lP = torch.log(Pkk)
    a = 1.4 * torch.exp(1.1 * lP - Pkk * Pkk)
    b = 0.9 * Pkk * torch.exp(-0.5 * torch.exp(1.4 * lP))
    C, E, Y = _speed_terms(sb, Pkk)
    al = qp * (0.6 * Pkk * Pkk - 0.38 * Pkk + 0.35)
    base = 4.0 * sb * sb * Y + 0.1 * qp2
    pre = (a * sb + b) / (2.0 * sb)
    out = []
    for z in (d["q"][K] + al, -d["q"][K] + al):
        out.append(pre * _bracket(z, -0.8 * z * sb * C + base) + E)
    sq = _sqrt(d["th"])
    return Q[1 + K] - out[1] * sq, Q[1 + K] + out[0] * sq


def _dimless14(Q):
    rho = Q[0]
    p = (Q[4] + Q[7] + Q[9]) / 3.0
    th = p / rho
    P = [Q[4 + n] / p for n in range(6)]
    q = [Q[10 + n] / (p * _sqrt(th)) for n in range(3)]
    t = P[0] + P[3] + P[5]
    T2 = P[0] ** 2 + P[3] ** 2 + P[5] ** 2 + 2.0 * (P[1] ** 2 + P[2] ** 2 + P[4] ** 2)
    y = _solve3(P, q)
    A = 2.0 * T2 + t * t - Q[13] / (p * th)
    X = 8.0 * T2 * sum(q[n] * y[n] for n in range(3))
    return dict(p=p, th=th, P=P, q=q, t=t, T2=T2, y=y, sb=_sigma_bar(A, X, T2))


def _cons14(Q):
    rho, u, P, q = Q[0], [Q[1], Q[2], Q[3]], [Q[4 + n] for n in range(6)], [Q[10 + n] for n in range(3)]
    u2 = sum(x * x for x in u)
    t = P[0] + P[3] + P[5]
    Pu = [sum(P[_sig(i, j)] * u[j] for j in range(3)) for i in range(3)]
    E = [rho * u[i] * u[j] + P[_sig(i, j)] for i, j in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))]
    H = [u[i] * (rho * u2 + t) + 2.0 * Pu[i] + q[i] for i in range(3)]
    E4 = (rho * u2 * u2 + 2.0 * u2 * t + 4.0 * sum(u[i] * Pu[i] for i in range(3))
          + 4.0 * sum(u[i] * q[i] for i in range(3)) + Q[13])
    return [rho, rho * u[0], rho * u[1], rho * u[2]] + E + H + [E4]


def _prim14(U):
    rho = U[0]
    u = [U[1 + i] / rho for i in range(3)]
    idx = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))
    P = [U[4 + n] - rho * u[i] * u[j] for n, (i, j) in enumerate(idx)]
    u2 = sum(x * x for x in u)
    t = P[0] + P[3] + P[5]
    Pu = [sum(P[_sig(i, j)] * u[j] for j in range(3)) for i in range(3)]
    q = [U[10 + i] - u[i] * (rho * u2 + t) - 2.0 * Pu[i] for i in range(3)]
    R = (U[13] - rho * u2 * u2 - 2.0 * u2 * t - 4.0 * sum(u[i] * Pu[i] for i in range(3))
         - 4.0 * sum(u[i] * q[i] for i in range(3)))
    return [rho] + u + P + q + [R]


def _face14(Q, K):
    """Conserved state, K-flux and wave speeds of a face state."""
    d = _dimless14(Q)
    Ps, T2, t, y, sb = d["P"], d["T2"], d["t"], d["y"], d["sb"]
    P2 = _mm(Ps, Ps)
    P3 = _mm(P2, Ps)
    P4 = _mm(P2, P2)
    tr3 = P3[0] + P3[3] + P3[5]
    v = _solve3([2.0 * Ps[n] * T2 + 4.0 * P3[n] for n in range(6)], d["q"])
    w = [sum(Ps[_sig(i, j)] * v[j] for j in range(3)) for i in range(3)]
    Qs = [[2.0 * (w[K] * P2[_sig(a, b)] + w[a] * P2[_sig(K, b)] + w[b] * P2[_sig(K, a)])
           for b in range(3)] for a in range(3)]
    Rs = [sum(Qs[a][b] * y[b] for b in range(3)) / sb + 2.0 * (1.0 - sb) * P2[_sig(a, K)]
          + Ps[_sig(a, K)] * t for a in range(3)]
    yQy = sum(y[a] * y[b] * Qs[a][b] for a in range(3) for b in range(3))
    c1 = 2.0 * t ** 3 + 12.0 * tr3 - 2.0 * T2 * t
    c2 = 14.0 * T2 - 6.0 * t * t
    Wq = sum((c1 * Ps[_sig(K, a)] + c2 * P2[_sig(K, a)] + 20.0 * t * P3[_sig(K, a)]
              + 20.0 * P4[_sig(K, a)]) * v[a] for a in range(3))
    r = _sqrt(sb)
    Ss = yQy / (sb * sb) + 2.0 * r * t * d["q"][K] + (1.0 - r) * Wq
    s3 = d["p"] * _sqrt(d["th"])
    s4 = d["p"] * d["th"]
    Qk = [[Qs[a][b] * s3 for b in range(3)] for a in range(3)]
    Rk = [Rs[a] * s4 for a in range(3)]
    Sk = Ss * s4 * _sqrt(d["th"])
    U = _cons14(Q)
    u, q = [Q[1], Q[2], Q[3]], [Q[10], Q[11], Q[12]]
    P = [Q[4 + n] for n in range(6)]
    u2 = sum(x * x for x in u)
    PuK = sum(P[_sig(K, j)] * u[j] for j in range(3))
    Qu = [sum(Qk[a][b] * u[b] for b in range(3)) for a in range(3)]
    F = [u[K] * x for x in U]
    for i in range(3):
        F[1 + i] = F[1 + i] + P[_sig(i, K)]
        F[10 + i] = F[10 + i] + u[i] * (2.0 * PuK + q[K]) + u2 * P[_sig(i, K)] + 2.0 * Qu[i] + Rk[i]
    for n, (i, j) in enumerate(((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))):
        F[4 + n] = F[4 + n] + u[i] * P[_sig(j, K)] + u[j] * P[_sig(i, K)] + Qk[i][j]
    F[13] = F[13] + (4.0 * u2 * PuK + 2.0 * u2 * q[K] + 4.0 * sum(u[a] * Qu[a] for a in range(3))
                     + 4.0 * sum(u[a] * Rk[a] for a in range(3)) + Sk)
    lo, hi = _speeds14(Q, d, K)
    return U, F, lo, hi


def _sigma5(Q):
    th = Q[2] / Q[0]
    qs = Q[3] / (Q[2] * _sqrt(th))
    return th, qs, _sigma_bar(3.0 - Q[4] / (Q[2] * th), 8.0 * qs * qs, torch.ones_like(th))


def _speeds5(Q):
    th, qs, sb = _sigma5(Q)
    C, E, Y = _speed_terms(sb, torch.ones_like(sb))
    l = [_bracket(z, -0.8 * z * sb * C + 4.0 * sb * sb * Y) / (2.0 * sb) + E for z in (qs, -qs)]
    sq = _sqrt(th)
    return Q[1] - l[1] * sq, Q[1] + l[0] * sq


def _cons5(Q):
    rho, u, P, q, r = Q
    return [rho, rho * u, rho * u * u + P, rho * u ** 3 + 3.0 * u * P + q,
            rho * u ** 4 + 6.0 * u * u * P + 4.0 * u * q + r]


def _prim5(U):
    rho = U[0]
    u = U[1] / rho
    P = U[2] - rho * u * u
    q = U[3] - rho * u ** 3 - 3.0 * u * P
    return [rho, u, P, q, U[4] - rho * u ** 4 - 6.0 * u * u * P - 4.0 * u * q]


def _face5(Q, K):
    rho, u, P, q, r = Q
    th, qs, sb = _sigma5(Q)
    s = (qs ** 3 / (sb * sb) + (10.0 - 8.0 * _sqrt(sb)) * qs) * P * th * _sqrt(th)
    U = _cons5(Q)
    F = [U[1], U[2], U[3], U[4],
         rho * u ** 5 + 10.0 * u ** 3 * P + 10.0 * u * u * q + 5.0 * u * r + s]
    lo, hi = _speeds5(Q)
    return U, F, lo, hi


def _riemann(L, R, flux):
    (UL, FL, l0, l1), (UR, FR, r0, r1) = L, R
    if flux == "rusanov":
        s = torch.stack([l0.abs(), l1.abs(), r0.abs(), r1.abs()])
        s = torch.gather(s, 0, s.detach().argmax(0, keepdim=True))[0]
        return [0.5 * (FL[k] + FR[k]) - 0.5 * s * (UR[k] - UL[k]) for k in range(len(UL))]
    SL, SR = torch.where(l0 < r0, l0, r0), torch.where(l1 > r1, l1, r1)
    left, right = SL >= 0, (SL < 0) & (SR <= 0)
    inv = 1.0 / torch.where(left | right, torch.ones_like(SL), SR - SL)
    return [torch.where(left, FL[k], torch.where(
        right, FR[k], (SR * FL[k] - SL * FR[k] + SL * SR * (UR[k] - UL[k])) * inv))
        for k in range(len(UL))]


def _relaxed(Q, nf):
    """The conserved moments and those of the Maxwellian they relax to."""
    if nf == 5:
        M = _cons5([Q[0], Q[1], Q[2], 0.0 * Q[0], 3.0 * Q[2] * Q[2] / Q[0]])
        U = _cons5(Q)
    else:
        p = (Q[4] + Q[7] + Q[9]) / 3.0
        z = 0.0 * p
        M = _cons14([Q[0], Q[1], Q[2], Q[3], p, z, z, p, z, p, z, z, z, 15.0 * p * p / Q[0]])
        U = _cons14(Q)
    return U, M


class _Scheme:
    """The finite-volume scheme on cells with neighbour tables (ghost cells appended after the
    interior ones), every operation in FP64."""

    def __init__(self, case, nf, n, tables, h, ghosts, tau, tube=None):
        self.case, self.nf, self.n, self.tables, self.h = case, nf, n, tables, h
        self.ghosts, self.tau, self.tube = ghosts, tau, tube
        self.prim = _prim5 if nf == 5 else _prim14
        self.face = _face5 if nf == 5 else _face14

    def tau_of(self, Q):
        T = Q[2] / Q[0] if self.nf == 5 else (Q[4] + Q[7] + Q[9]) / (3.0 * Q[0])
        return self.tau / Q[0] / _sqrt(T)

    def rate(self, U):
        Q = self.prim(U)
        r = 0.0
        for K in range(len(self.tables)):
            lo, hi = _speeds5(Q) if self.nf == 5 else _speeds14(Q, _dimless14(Q), K)
            r = r + torch.maximum(lo.abs(), hi.abs()) / self.h[K]
        if self.tube is None:
            return r.max()
        m = torch.zeros(int(self.tube.max()) + 1, dtype=r.dtype, device=r.device)
        return m.scatter_reduce(0, self.tube, r, "amax")

    def residual(self, U):
        """-div F (and the source where it is explicit) of the conserved state."""
        Q = self.prim(U)
        # the ghost cells' states after the interior ones
        ext = [q if self.ghosts is None else torch.cat([q, self.ghosts[k]]) for k, q in enumerate(Q)]
        L = [0.0] * self.nf
        second = self.case["order"] == 2
        for K, (a2, a1, b1, b2) in enumerate(self.tables):
            s = [[q[i] for q in ext] for i in (a2, a1)] + [Q] + [[q[i] for q in ext] for i in (b1, b2)]
            phi = [None] + [_phi(s[m - 1], s[m], s[m + 1], self.case["limiter"], self.nf) if second
                            else None for m in (1, 2, 3)] + [None]
            # the limiter is held constant in derivatives
            phi = [f if f is None else f.detach() for f in phi]

            def state(m, sgn):
                if not second:
                    return s[m]
                return [s[m][k] + sgn * 0.25 * phi[m] * (s[m + 1][k] - s[m - 1][k])
                        for k in range(self.nf)]

            flux = self.case["flux"]
            lo = _riemann(self.face(state(1, 1.0), K), self.face(state(2, -1.0), K), flux)
            hi = _riemann(self.face(state(2, 1.0), K), self.face(state(3, -1.0), K), flux)
            L = [L[k] - (hi[k] - lo[k]) / self.h[K] for k in range(self.nf)]
        if self.case["source"] == "explicit":
            V, M = _relaxed(Q, self.nf)
            tau = self.tau_of(Q)
            L = [L[k] - (V[k] - M[k]) / tau if k > self.first() else L[k] for k in range(self.nf)]
        return L

    def first(self):
        return 2 if self.nf == 5 else 3        # fields up to this one are conserved exactly

    def stage(self, base, U, h):
        L = self.residual(U)
        V = [base[k] + h * L[k] for k in range(self.nf)]
        if self.case["source"] == "point_implicit":
            Q = self.prim(V)
            _, M = _relaxed(Q, self.nf)
            g = 1.0 / (1.0 + h / self.tau_of(Q))
            V = [V[k] if k < (2 if self.nf == 5 else 4) else M[k] + g * (V[k] - M[k])
                 for k in range(self.nf)]
        return V

    def step(self, U, dt):
        if self.case["integrator"] == "fe":
            return self.stage(U, U, dt)
        return self.stage(U, self.stage(U, U, 0.5 * dt), dt)

    def march(self, U):
        t = 0.0
        for _ in range(self.case["steps"]):
            dt = 0.5 / self.rate(U)
            t = t + dt
            U = self.step(U, dt if self.tube is None else dt[self.tube])
        return U, t


def _line_tables(start, n, dev):
    """Neighbours at -2, -1, +1, +2 of the cells of a tube [start, start + n), ends copied."""
    i = torch.arange(n, device=dev)
    return [start + (i + o).clamp(0, n - 1) for o in (-2, -1, 1, 2)]


def _grid_scheme(case, d, dev, ghosts=None):
    nx, ny, nf = case["nx"], case["ny"], case["system"]
    j, i = torch.meshgrid(torch.arange(ny, device=dev), torch.arange(nx, device=dev), indexing="ij")
    n = nx * ny
    periodic = ny > 1 and case["flow"] == "periodic"
    slots = "left" in d
    tables = []
    for K in range(2 if ny > 1 else 1):
        t = []
        for o in (-2, -1, 1, 2):
            a, m = (i, nx) if K == 0 else (j, ny)
            x = a + o
            y = x % m if periodic else x.clamp(0, m - 1)
            idx = j * nx + y if K == 0 else y * nx + i
            if slots:            # the inflow slot's ghost cells: state n (left) or n + 1 (bottom)
                tang = (j + 0.5) / ny if K == 0 else (i + 0.5) / nx
                idx = torch.where((x < 0) & (tang >= SLOT[0]) & (tang <= SLOT[1]), n + K, idx)
            t.append(idx.reshape(-1))
        tables.append(t)
    if slots and ghosts is None:
        ghosts = [torch.tensor([d["left"][k], d["bottom"][k]], dtype=torch.float64, device=dev)
                  for k in range(nf)]
    return _Scheme(case, nf, n, tables, [1.0 / nx, 1.0 / ny], ghosts, d["tau"])


def exact(case, seed):
    d = _setup(case, seed)
    dev = _device()
    nf = case["system"]
    cons = _cons5 if nf == 5 else _cons14
    if case["kind"] == "batch":
        ncells = d["ncells"]
        starts = np.concatenate([[0], np.cumsum(ncells)[:-1]])
        per = [_line_tables(int(s), n, dev) for s, n in zip(starts, ncells)]
        tables = [[torch.cat([p[m] for p in per]) for m in range(4)]]
        tube = torch.cat([torch.full((n,), b, device=dev) for b, n in enumerate(ncells)])
        sch = _Scheme(case, nf, sum(ncells), tables, [1.0 / torch.tensor(ncells, dtype=torch.float64, device=dev)[tube]],
                      None, torch.tensor(d["taus"], dtype=torch.float64, device=dev)[tube], tube)
        U, t = sch.march(cons(list(torch.cat(d["prims"], 1))))
        U = torch.stack(U)
        flat = torch.cat([U[:, int(s):int(s) + n].reshape(-1) for s, n in zip(starts, ncells)])
        return {"U": flat, "t": t.cpu().numpy(), "steps": None}
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, d, dev)
    sch = _grid_scheme(case, d, dev)
    U, t = sch.march(cons([q.reshape(-1) for q in d["prim"]]))
    U = torch.stack(U).reshape(nf, case["ny"], case["nx"])
    return {"U": U, "t": t.reshape(1).cpu().numpy(), "steps": None}


def _exact_adjoint(case, d, dev):
    """The reverse sweep by automatic differentiation of the same scheme at the given steps."""
    ghosts = [torch.tensor([d["left"][k], d["bottom"][k]], dtype=torch.float64, device=dev,
                           requires_grad=True) for k in range(14)]
    sch = _grid_scheme(case, d, dev, ghosts)
    sch.tau = torch.tensor(d["tau"], dtype=torch.float64, device=dev, requires_grad=True)
    U0 = [u.detach().clone().requires_grad_(True) for u in _cons14([q.reshape(-1) for q in d["prim"]])]
    U = U0
    for dt in d["dts"]:
        U = sch.step(U, dt)
    J = sum((U[k] * d["ubar"][k].reshape(-1)).sum() for k in range(14))
    leaves = U0 + ghosts + [sch.tau]
    g = torch.autograd.grad(J, leaves, allow_unused=True)
    g = [torch.zeros_like(x) if y is None else y for x, y in zip(leaves, g)]
    # the solver carries the ten moments of a planar state
    act = (0, 1, 2, 4, 5, 7, 9, 10, 11, 13)
    ubar = torch.stack([g[k] if k in act else torch.zeros_like(g[k]) for k in range(14)])
    gbar = np.zeros((4, mx.GHOST_SLOTS, 14))
    for k in act:
        gbar[mx.XLO, 1, k], gbar[mx.YLO, 1, k] = g[14 + k].cpu().numpy()
    return {"ubar": ubar.reshape(14, case["ny"], case["nx"]), "gbar": gbar,
            "taubar": np.array([float(g[28])])}
