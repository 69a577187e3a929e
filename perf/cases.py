"""What a user of this framework has it do, as cases that can be timed and compared.

A case is one call sequence of a user's program on one simulation, batch or
request stream: the initial state from page-locked host memory, some time
steps, the final state back to page-locked host memory (the library's
boundary is host data).  Kinds:

  channel   scalar advection in the inclined channel, one instance (FP64)
  cylinder  a moving cylinder meeting a shock, one instance
  naca      the pitching NACA 0012 aerofoil, one instance (rotating body)
  tube      the axisymmetric open-ended tube, one instance
  batch     many uneven grids advancing together (cylinder, triangle, piston)
  serve     requests of several bodies, sizes and run lengths through the
            request loop
  cone      the three-dimensional Schardin cone, FP64 or the FP32 flux option
  flow3     a three-dimensional flow without a body, FP64 or the FP32 option

prepare() makes the simulation handle and the host buffers, which a program
keeps; run() writes the state, steps and reads the state, so every pass does
the same work.
"""
import math

import numpy as np
import torch

from paper_1711_11361_gb300 import inputs, mb, mb3

TWO_PI = 2.0 * math.pi


def listed():
    return [
        # the paper's channel validation: a small grid over its whole run, so
        # launches and latency count
        {"name": "channel_100", "kind": "channel", "n": 100, "steps": 200, "fp32": False},
        # one simulation of the size of the paper's cylinder test, in the
        # fast precision and in the one that parity is held in
        {"name": "cylinder_400_fp32", "kind": "cylinder", "n": 400, "steps": 40, "fp32": True},
        {"name": "cylinder_399_fp64", "kind": "cylinder", "n": 399, "steps": 40, "fp32": False},
        # the aerofoil: a rotating body of many vertices
        {"name": "naca_1024_fp32", "kind": "naca", "n": 1024, "steps": 40, "fp32": True},
        # the paper's open tube on its coarsest mesh, axisymmetric, FP64
        {"name": "tube_94_fp64", "kind": "tube", "n": 94, "steps": 40, "fp32": False},
        # the main workload: 64 uneven grids, FP32 bulk, a stretch of steps
        {"name": "batch_64_fp32", "kind": "batch", "count": 64, "nmin": 128, "nmax": 1024, "mix": 1, "steps": 20,
         "fp32": True},
        # a batch held in plain FP64
        {"name": "batch_16_fp64", "kind": "batch", "count": 16, "nmin": 128, "nmax": 1024, "mix": 2, "steps": 8,
         "fp32": False},
        # step by step with the host: states in, one step, states out
        {"name": "batch_16_io_fp32", "kind": "batch", "count": 16, "nmin": 128, "nmax": 1024, "mix": 3, "steps": 1,
         "fp32": True},
        # a served stream: requests admitted, stepped together and retired
        {"name": "serve_16_fp32", "kind": "serve", "count": 16, "nmin": 256, "nmax": 1024, "mix": 4, "smin": 20,
         "smax": 60, "fp32": True},
        # the Schardin cone at the middle and the finest mesh of the paper
        {"name": "cone_20_fp64", "kind": "cone", "n": 20, "steps": 4, "fp32": False},
        {"name": "cone_40_fp32", "kind": "cone", "n": 40, "steps": 4, "fp32": True},
        # a flow without a body, whose fluxes plain 64-bit arithmetic gives
        {"name": "flow3_97x64x50_fp64", "kind": "flow3", "nx": 97, "ny": 64, "nz": 50, "steps": 4, "fp32": False},
    ]


def _log_int(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["channel", "cylinder", "naca", "tube", "batch", "batch", "serve", "cone", "cone", "flow3"])
    fp32 = rng.random() < 0.5
    if kind == "channel":
        return {"kind": kind, "n": _log_int(rng, 64, 400), "steps": rng.randint(50, 200), "fp32": False}
    if kind in ("cylinder", "naca"):
        return {"kind": kind, "n": _log_int(rng, 96, 2048 if fp32 else 1024), "steps": rng.randint(4, 20), "fp32": fp32}
    if kind == "tube":
        return {"kind": kind, "n": rng.randint(32, 189), "steps": rng.randint(4, 20), "fp32": False}
    if kind == "batch":
        nmin = _log_int(rng, 96, 512)
        return {"kind": kind, "count": _log_int(rng, 2, 48 if fp32 else 16), "nmin": nmin,
                "nmax": rng.randint(nmin, 1024), "mix": rng.randint(0, 999), "steps": rng.randint(1, 12 if fp32 else 6),
                "fp32": fp32}
    if kind == "serve":
        return {"kind": kind, "count": rng.randint(4, 16), "nmin": 256, "nmax": rng.randint(400, 1024),
                "mix": rng.randint(0, 999), "smin": 10, "smax": rng.randint(20, 60), "fp32": True}
    if kind == "cone":
        return {"kind": kind, "n": rng.randint(6, 36) if fp32 else rng.randint(6, 22), "steps": rng.randint(1, 4),
                "fp32": fp32}
    return {"kind": kind, "nx": _log_int(rng, 24, 160), "ny": _log_int(rng, 24, 160), "nz": _log_int(rng, 24, 96),
            "steps": rng.randint(1, 3), "fp32": fp32}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _waves(rng, sizes, amplitude):
    """Per axis (last first) a smooth factor 1 + amplitude sin(...) of one to three waves: scaling a conserved
    state by their product keeps its velocity and varies density and pressure, so that every cell has slopes."""
    return [1.0 + amplitude * np.sin(TWO_PI * rng.integers(1, 4) * (np.arange(n) + 0.5) / n + rng.uniform(0, TWO_PI))
            for n in sizes]


def _vary(prob, rng, amplitude=0.01):
    wy, wx = _waves(rng, (prob.ny, prob.nx), amplitude)
    prob.Q0 = prob.Q0 * wy[:, None] * wx[None, :]
    return prob


def _batch_specs(case):
    """Body and size of each instance: from the case alone."""
    rng = np.random.default_rng(case["mix"])
    return [(("cylinder", "triangle", "piston")[int(rng.integers(0, 3))],
             int(rng.integers(case["nmin"], case["nmax"] + 1))) for _ in range(case["count"])]


def _request_specs(case):
    rng = np.random.default_rng(case["mix"])
    lo, hi = math.log(case["nmin"]), math.log(case["nmax"])
    return [dict(k=k, kind=("cylinder", "triangle", "piston", "naca")[int(rng.integers(0, 4))],
                 N=int(round(math.exp(rng.uniform(lo, hi)))), steps=int(rng.integers(case["smin"], case["smax"] + 1)))
            for k in range(case["count"])]


def _problems2(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "channel":
        probs = [inputs.c1_advection(case["n"])]
    elif kind == "cylinder":
        probs = [inputs.c2_cylinder(case["n"], M=float(rng.uniform(1.5, 2.5)))]
    elif kind == "naca":
        probs = [inputs.c3_naca(case["n"])]
    elif kind == "tube":
        probs = [inputs.n2_open_tube(case["n"])]
    elif kind == "batch":
        probs = [inputs.small_case(body, n, float(rng.uniform(1.2, 3.0))) for body, n in _batch_specs(case)]
    else:
        probs = [inputs.make_request(dict(s, M=float(rng.uniform(1.2, 3.0)))) for s in _request_specs(case)]
    return [_vary(p, rng) for p in probs]


def _problem3(case, seed):
    """The three-dimensional problem and its state as planes (torch, FP64)."""
    rng = np.random.default_rng(seed)
    if case["kind"] == "cone":
        # inputs.n3_schardin_cone's set-up, the state made by broadcasting
        k = case["n"]
        h, c1 = 1.0 / k, math.sqrt(inputs.GAMMA)
        g, M = inputs.GAMMA, inputs.N3_MACH
        u1 = M * c1
        r2 = (g + 1.0) * M * M / ((g - 1.0) * M * M + 2.0)
        p2 = 1.0 + 2.0 * g / (g + 1.0) * (M * M - 1.0)
        xs = 4.0 + 0.3183 * h
        apex = (xs - 2.0 * h, 0.2718 * h, 0.0)
        nrm, off, bb = inputs.cone_planes(apex, math.sqrt(3.0) / 2.0, 0.5, 24, phase=0.5)
        prob = inputs.Problem3("cone", 10 * k, 10 * k, 5 * k, lo=(0.0, -5.0, 0.0), hi=(10.0, 5.0, 5.0),
                               bc=(inputs.TRANSMISSIVE,) * 4 + (inputs.REFLECTIVE, inputs.TRANSMISSIVE),
                               normals=nrm, offsets=off, bbox=bb, U=(u1, 0.0, 0.0))
        x = (np.arange(prob.nx) + 0.5) * h
        rho, u, p = np.where(x > xs, r2, 1.0), np.where(x > xs, u1 / r2, u1), np.where(x > xs, p2, 1.0)
    else:
        prob = inputs.Problem3("flow", case["nx"], case["ny"], case["nz"], hi=(1.5, 1.0, 0.8),
                               bc=(inputs.TRANSMISSIVE, inputs.TRANSMISSIVE, inputs.PERIODIC, inputs.PERIODIC,
                                   inputs.REFLECTIVE, inputs.TRANSMISSIVE))
        x = (np.arange(prob.nx) + 0.5) / prob.nx
        left = x < 0.4
        rho, u, p = np.where(left, 1.0, 0.25), np.where(left, 0.3, -0.1), np.where(left, 1.0, 0.2)
    wz, wy, wx = _waves(rng, (prob.nz, prob.ny, prob.nx), 0.01)
    v, w = (float(rng.uniform(-0.02, 0.02)) for _ in range(2))
    line = inputs.conserved3(rho, u, v, w, p) * wx                      # (5, nx)
    cross = torch.from_numpy(wz[:, None] * wy[None, :])                 # (nz, ny)
    return prob, torch.from_numpy(line)[:, None, None, :] * cross[None, :, :, None]


def _pinned(n, dtype):
    return torch.empty(n, dtype=dtype, pin_memory=torch.cuda.is_available())


def prepare(case, seed):
    if case["kind"] in ("cone", "flow3"):
        prob, Q = _problem3(case, seed)
        q_in, q_out = _pinned(Q.numel(), torch.float64), _pinned(Q.numel(), torch.float64)
        q_in.copy_(Q.reshape(-1))
        sim = mb3.Sim3(prob, write_initial=False, precision=mb.FP32 if case["fp32"] else mb.FP64)
        return {"case": case, "sim": sim, "q_in": q_in, "q_out": q_out}
    probs = _problems2(case, seed)
    if case["kind"] == "serve":
        return {"case": case, "probs": probs, "steps": [p.steps for p in probs]}
    dtype = torch.float32 if case["fp32"] else torch.float64
    sizes = [p.Q0.size for p in probs]
    q_in, q_out = _pinned(sum(sizes), dtype), _pinned(sum(sizes), dtype)
    at = np.cumsum([0] + sizes)
    for k, p in enumerate(probs):
        q_in[at[k]:at[k + 1]].copy_(torch.from_numpy(p.Q0).reshape(-1))
        p.Q0 = None
    sim = mb.Sim(probs, mb.FP32 if case["fp32"] else mb.FP64, write_initial=False)
    width = q_in.element_size()
    return {"case": case, "sim": sim, "q_in": q_in, "q_out": q_out,
            "p_in": [q_in.data_ptr() + width * int(a) for a in at[:-1]],
            "p_out": [q_out.data_ptr() + width * int(a) for a in at[:-1]]}


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def _address(t):
    return mb.ctypes.cast(t.data_ptr(), mb.ctypes.POINTER(mb.ctypes.c_double))


def run(state):
    case = state["case"]
    if case["kind"] in ("cone", "flow3"):
        sim = state["sim"]
        origin = np.zeros(3)
        clock = np.empty(5)
        sim._check(mb3.lib.mb3_write_state(sim._h, _address(state["q_in"]), 0.0,
                                           origin.ctypes.data_as(mb.ctypes.POINTER(mb.ctypes.c_double))))
        for _ in range(case["steps"]):
            sim.step()
        sim._check(mb3.lib.mb3_read_state(sim._h, _address(state["q_out"]), None,
                                          clock.ctypes.data_as(mb.ctypes.POINTER(mb.ctypes.c_double))))
        return {"Q": state["q_out"], "clock": clock}
    if case["kind"] == "serve":
        srv = mb.Server(mb.FP32, inputs.EULER, budget_bytes=32 * 2 ** 30, max_active=12)
        ids = [srv.submit(p, n) for p, n in zip(state["probs"], state["steps"])]
        while srv.tick()[2] < len(ids):
            pass
        # the final states hold FP32 values in FP64 arrays
        out = [torch.from_numpy(srv.result(i)).float() for i in ids]
        done = [srv.query(i)["state"] for i in ids]
        srv.close()
        return {"Q": out, "done": np.array(done)}
    sim = state["sim"]
    dtype = np.float32 if case["fp32"] else np.float64
    sim.write_states(state["p_in"], dtype=dtype)
    sim.run(case["steps"])
    _, clocks, _ = sim.read_states(out=state["p_out"], dtype=dtype)
    return {"Q": state["q_out"], "clocks": clocks}


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def work(case):
    """Each sweep reads every cell's state once and writes it once; about 250 floating-point operations per cell and
    sweep in two dimensions, 300 in three, 10 for advection (reconstruction, Riemann problem, update)."""
    kind = case["kind"]
    width = 4 if case["fp32"] else 8
    if kind in ("cone", "flow3"):
        cells = (10 * case["n"]) ** 2 * 5 * case["n"] if kind == "cone" else case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 3 * case["steps"] * cells * 2 * 5 * 8, "flops": 3 * case["steps"] * cells * 300}
    if kind == "channel":
        cells = case["n"] ** 2
        return {"bytes": 2 * case["steps"] * cells * 2 * width, "flops": 2 * case["steps"] * cells * 10}
    if kind == "tube":
        cell_steps = 40 * case["n"] ** 2 * case["steps"]
    elif kind == "batch":
        cell_steps = sum(n * n for _, n in _batch_specs(case)) * case["steps"]
    elif kind == "serve":
        cell_steps = sum(s["N"] ** 2 * s["steps"] for s in _request_specs(case))
    else:
        cell_steps = case["n"] ** 2 * case["steps"]
    return {"bytes": 2 * cell_steps * 2 * 4 * width, "flops": 2 * cell_steps * 250}


# --------------------------------------------------------------------------
# the flow without a body in plain 64-bit arithmetic
# --------------------------------------------------------------------------
def _flux(q, d, g):
    u = q[1 + d] / q[0]
    p = (g - 1.0) * (q[4] - 0.5 * (q[1] ** 2 + q[2] ** 2 + q[3] ** 2) / q[0])
    f = q * u
    f[1 + d] += p
    f[4] += p * u
    return f, u, p


def _hllc(ql, qr, d, g):
    fl, ul, pl = _flux(ql, d, g)
    fr, ur, pr = _flux(qr, d, g)
    cl, cr = torch.sqrt(g * pl / ql[0]), torch.sqrt(g * pr / qr[0])
    sl, sr = torch.minimum(ul - cl, ur - cr), torch.maximum(ul + cl, ur + cr)
    ss = (pr - pl + ql[0] * ul * (sl - ul) - qr[0] * ur * (sr - ur)) / (ql[0] * (sl - ul) - qr[0] * (sr - ur))

    def star(q, f, u, p, s):
        fac = q[0] * (s - u) / (s - ss)
        qs = fac * q / q[0]
        qs[1 + d] = fac * ss
        qs[4] = fac * (q[4] / q[0] + (ss - u) * (ss + p / (q[0] * (s - u))))
        return f + s * (qs - q)

    f = torch.where(ss >= 0, star(ql, fl, ul, pl, sl), star(qr, fr, ur, pr, sr))
    return torch.where(sl >= 0, fl, torch.where(sr <= 0, fr, f))


def _pad(q, axis, d, bc):
    """Two ghost cells on each side of an axis: periodic, mirrored, or mirrored with the normal velocity reversed."""
    n = q.shape[axis]
    index = torch.arange(-2, n + 2)
    if bc[0] == inputs.PERIODIC:
        return q.index_select(axis, index % n)
    mirrored = torch.where(index < 0, -1 - index, torch.where(index >= n, 2 * n - 1 - index, index))
    out = q.index_select(axis, mirrored)
    for side, kind in enumerate(bc):
        if kind == inputs.REFLECTIVE:
            out[1 + d].narrow(axis - 1, 0 if side == 0 else n + 2, 2).neg_()
    return out


def _sweep(q, d, lam, bc, g):
    axis = 3 - d                                   # planes are (5, nz, ny, nx)
    n = q.shape[axis]
    big = _pad(q, axis, d, bc)
    qm, q0, qp = (big.narrow(axis, s, n + 2) for s in (0, 1, 2))
    dm, dp = q0 - qm, qp - q0
    pr = dm * dp
    slope = torch.where(pr > 0, 2.0 * pr / torch.where(pr > 0, dm + dp, torch.ones_like(dm)), torch.zeros_like(dm))
    lo, hi = q0 - 0.5 * slope, q0 + 0.5 * slope
    change = 0.5 * lam * (_flux(lo, d, g)[0] - _flux(hi, d, g)[0])
    lo, hi = lo + change, hi + change

    def physical(x):
        return (x[0] > 0) & (2.0 * x[0] * x[4] > x[1] ** 2 + x[2] ** 2 + x[3] ** 2)

    ok = physical(lo) & physical(hi)
    lo, hi = torch.where(ok, lo, q0), torch.where(ok, hi, q0)
    f = _hllc(hi.narrow(axis, 0, n + 1), lo.narrow(axis, 1, n + 1), d, g)
    return q + lam * (f.narrow(axis, 0, n) - f.narrow(axis, 1, n))


def exact(case, seed):
    """The flow without a body: MUSCL-Hancock and HLLC sweeps in 64 bits.  The other kinds need the cut-cell
    geometry, wall states and redistribution of a whole simulation, which plain array code does not give within
    the time allowed."""
    if case["kind"] != "flow3":
        return None
    prob, q = _problem3(case, seed)
    g, t = prob.gamma, 0.0
    for step in range(case["steps"]):
        p = (g - 1.0) * (q[4] - 0.5 * (q[1] ** 2 + q[2] ** 2 + q[3] ** 2) / q[0])
        c = torch.sqrt(g * p / q[0])
        dt = prob.cfl * min(prob.h[a] / float((torch.abs(q[1 + a] / q[0]) + c).max()) for a in range(3))
        for d in ((0, 1, 2) if step % 2 == 0 else (2, 1, 0)):
            q = _sweep(q, d, dt / prob.h[d], prob.bc[2 * d:2 * d + 2], g)
        t += dt
    return {"Q": q.reshape(-1), "clock": np.array([t, 0.0, 0.0, 0.0, float(case["steps"])])}
