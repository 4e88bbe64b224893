"""Performance cases of the DGSEM library: what a program built on it calls, over the sizes it is used at.

A case is one of four calls of the public API on one mesh:

* ``run``       Solver.run: LSERK4(5) steps of the flow (the time loop of a simulation);
* ``rhs``       Solver.rhs: one semi-discrete right-hand side (an own time integrator, a steady residual);
* ``gradient``  adjoint.final_state and backward: the gradient of the final kinetic energy with respect
                to the initial state (optimisation, sensitivity);
* ``adjoint``   Solver.rhs_adjoint: one transposed right-hand side (an own adjoint integrator);
* ``reduce``    Solver.reduce: conserved totals, kinetic energy and its rate, admissible time step (monitoring).

Meshes are boxes of hexahedra handed over as unstructured meshes: ``box`` (Cartesian), ``sine`` (curved by
x_i = xi_i + 0.1 prod_j sin(pi xi_j)), ``mortar`` (two blocks, the second refined 2:1).  ``exact`` evaluates
the same discretisation with plain torch operations in 64 bits.
"""
from __future__ import annotations

import functools
import itertools
import math

import numpy as np
import torch

from paper_1910_02858_gb300 import Solver, SolverConfig
from paper_1910_02858_gb300 import flexi as F
from paper_1910_02858_gb300.adjoint import final_state

GAMMA, PR = 1.4, 0.72
RIEMANN = {"roe": F.RIEMANN_ROE, "hllc": F.RIEMANN_HLLC, "roe_smooth": F.RIEMANN_ROE_SMOOTH,
           "rusanov": F.RIEMANN_RUSANOV, "ec": F.RIEMANN_EC}
PRECISION = {"fp64": F.FP64, "fp32": F.FP32, "tf32": F.FP32_TF32, "bf16": F.FP32_BF16}
SPLIT = {"standard": F.SPLIT_STANDARD, "kep": F.SPLIT_KEP, "ec": F.SPLIT_EC}
FLOW = {"tgv": F.EXACT_TGV, "freestream": F.EXACT_FREESTREAM, "mms": F.EXACT_MANUFACTURED}
DEFAULTS = dict(call="run", mesh="box", turned=False, nodes="gauss", precision="fp64", riemann="hllc",
                split="standard", lifting="br1", flow="tgv", boundary="periodic", Ma=0.1, Re=1600.0, steps=1,
                own_stream=False, checkpoint_every=2)


def _case(**kw):
    return {**DEFAULTS, **kw}


def listed():
    return [
        # a short run of the smallest Taylor-Green configuration, on a stream of the program's own: launch latency
        _case(name="tgv_tiny_run", nx=4, ny=4, nz=4, N=3, nodes="lobatto", riemann="roe", steps=10, own_stream=True),
        # one right-hand side of a small box with rotated element frames and inflow, outflow and wall sides
        _case(name="bounded_small_rhs", call="rhs", nx=5, ny=3, nz=4, N=4, turned=True, flow="freestream",
              boundary="mixed", Ma=0.3, Re=400.0),
        # one step of the headline Taylor-Green configuration: 16^3 elements, N = 7, Gauss nodes, HLLC, 64 bits
        _case(name="tgv_n7_run", nx=16, ny=16, nz=16, N=7),
        # the same flow in kinetic-energy-preserving split form (under-resolved turbulence), a ragged box
        _case(name="split_n7_run", nx=11, ny=9, nz=10, N=7, nodes="lobatto", split="kep", riemann="roe"),
        # curved mesh with the manufactured solution, its source term and time-dependent exact boundaries
        _case(name="curved_mms_n7_run", nx=24, ny=24, nz=24, N=7, mesh="sine", flow="mms", boundary="exact", Re=100.0),
        # curved mesh, 32-bit form, free stream with exact-state sides
        _case(name="curved_fp32_n7_run", nx=24, ny=24, nz=24, N=7, mesh="sine", flow="freestream", boundary="exact",
              precision="fp32", steps=2),
        # the precision form's configuration: 32^3 elements, N = 5, 32 bits, line sweeps on the FP32 pipes
        _case(name="tgv_fp32_n5_run", nx=32, ny=32, nz=32, N=5, precision="fp32", steps=2),
        # the same form with the line sweeps on tensor cores (TF32 in three terms), a ragged box
        _case(name="tgv_tf32_n5_run", nx=19, ny=23, nz=17, N=5, precision="tf32", steps=2),
        # gradient of the final kinetic energy by the checkpointed discrete adjoint: 8^3 elements, N = 5
        _case(name="gradient_n5", call="gradient", nx=8, ny=8, nz=8, N=5, riemann="roe_smooth", Re=400.0, steps=4),
        # one transposed right-hand side on a curved periodic mesh of odd sizes
        _case(name="adjoint_curved_n6", call="adjoint", nx=7, ny=9, nz=8, N=6, mesh="sine", Re=400.0),
        # a 2:1 refined block behind a coarse one (mortar sides), odd polynomial count
        _case(name="mortar_n4_run", nx=4, ny=8, nz=8, N=4, mesh="mortar", riemann="rusanov"),
        # the monitoring sums of the headline configuration
        _case(name="monitor_n7_reduce", call="reduce", nx=16, ny=16, nz=16, N=7),
    ]


def draw(rng):
    c = _case(name=None)
    del c["name"]
    c["call"] = rng.choices(["run", "rhs", "gradient", "adjoint", "reduce"], [10, 3, 2, 2, 1])[0]
    c["precision"] = rng.choices(["fp64", "fp32", "tf32", "bf16"], [10, 6, 2, 2])[0] if c["call"] == "run" else "fp64"
    c["mesh"] = rng.choices(["box", "sine", "mortar"], [5, 4, 1])[0]
    c["nodes"] = rng.choices(["gauss", "lobatto"], [3, 2])[0]
    c["N"] = rng.choice([1, 2, 3, 4, 5, 5, 6, 7, 7, 7]) if c["mesh"] == "box" else rng.choice([2, 3, 4, 5, 6, 7, 7])
    if c["nodes"] == "lobatto" and c["precision"] in ("fp64", "fp32"):
        c["split"] = rng.choices(["standard", "kep", "ec"], [4, 3, 1])[0]
    if c["split"] == "standard" and c["precision"] in ("fp64", "fp32") and rng.random() < 0.15:
        c["lifting"] = "br2"
    c["riemann"] = rng.choice(["roe", "hllc", "roe_smooth", "rusanov"] + (["ec"] if c["split"] == "ec" else []))
    if c["call"] in ("gradient", "adjoint") and c["riemann"] == "roe":
        c["riemann"] = "roe_smooth"
    # degrees of freedom: spread over the logarithm of the range, the dearer calls not as far
    top = {"gradient": 2e5, "adjoint": 5e5}.get(c["call"], 5e5 if c["split"] == "ec" else 3e6)
    dof = math.exp(rng.uniform(math.log(1500.0), math.log(top)))
    elements = max(4.0, dof / (c["N"] + 1) ** 3)
    side = elements ** (1.0 / 3.0)
    c["nx"] = max(2, round(side * rng.uniform(0.6, 1.5)))
    c["ny"] = max(2, round(side * rng.uniform(0.7, 1.4)))
    c["nz"] = max(2, round(elements / (c["nx"] * c["ny"])))
    if c["mesh"] == "mortar":  # 1 + 8 elements per coarse one
        c["nx"], c["ny"], c["nz"] = max(1, c["nx"] // 2), max(1, c["ny"] // 2), max(1, c["nz"] // 2)
    c["turned"] = c["mesh"] != "mortar" and rng.random() < 0.3
    c["boundary"] = "periodic" if c["mesh"] == "mortar" or c["call"] == "gradient" else \
        rng.choices(["periodic", "exact", "mixed"], [5, 2, 1])[0]
    if c["boundary"] == "exact":
        c["flow"] = rng.choice(["freestream", "mms"])
    elif c["boundary"] == "mixed":
        c["flow"] = "freestream"
    c["Ma"] = rng.choice([0.1, 0.2, 0.3])
    c["Re"] = rng.choice([100.0, 400.0, 1600.0])
    c["steps"] = rng.choice([1, 2, 3]) if c["call"] == "run" else 2 if c["call"] == "gradient" else 1
    c["own_stream"] = c["call"] == "run" and rng.random() < 0.5
    return c


# ---------------------------------------------------------------- nodes, meshes and states


@functools.lru_cache(maxsize=None)
def _nodes(N, nodes):
    """Nodes and weights on [-1, 1]."""
    leg = np.polynomial.legendre
    if nodes == "gauss":
        return leg.leggauss(N + 1)
    c = np.zeros(N + 1)
    c[N] = 1.0
    x = np.sort(np.real(leg.legroots(leg.legder(c)))) if N > 1 else np.zeros(0)
    for _ in range(4):  # Newton on P_N' from the eigenvalues
        d1, d2 = leg.legval(x, leg.legder(c)), leg.legval(x, leg.legder(c, 2))
        x = x - d1 / d2
    x = np.concatenate([[-1.0], x, [1.0]])
    return x, 2.0 / (N * (N + 1) * leg.legval(x, c) ** 2)


@functools.lru_cache(maxsize=1)
def _frames():
    """The 24 proper rotations of the cube, as signed permutation matrices."""
    out = []
    for perm in itertools.permutations(range(3)):
        for signs in itertools.product((1, -1), repeat=3):
            R = np.zeros((3, 3), dtype=np.int64)
            R[range(3), perm] = signs
            if round(np.linalg.det(R)) == 1:
                out.append(R)
    return np.stack(out)


def _corner(s, p, q):
    xi = np.zeros(3, dtype=np.int64)
    a, b = [d for d in range(3) if d != s // 2]
    xi[s // 2], xi[a], xi[b] = 2 * (s % 2) - 1, 2 * p - 1, 2 * q - 1
    return xi


@functools.lru_cache(maxsize=None)
def _joint(a, b, s):
    """Neighbour side and orientation code across side s, for element frames number a and b."""
    Ra, Rb = _frames()[a], _frames()[b]
    out = Ra[:, s // 2] * (2 * (s % 2) - 1)
    inner = Rb.T @ -out  # the neighbour's outward direction in its own frame
    t = 2 * int(np.argmax(np.abs(inner))) + (1 if inner.sum() > 0 else 0)
    ax = [d for d in range(3) if d != t // 2]

    def image(p, q):
        xi = Rb.T @ (Ra @ _corner(s, p, q) - 2 * out)
        return (xi[ax[0]] + 1) // 2, (xi[ax[1]] + 1) // 2

    for o in range(8):
        def code(p, q):
            u, v = (q, p) if o & 1 else (p, q)
            return (1 - u if o & 2 else u), (1 - v if o & 4 else v)
        if all(image(p, q) == code(p, q) for p in (0, 1) for q in (0, 1)):
            return t, o
    raise ValueError("not a face map")


def _extent(case):
    """Lower corner and edge lengths of the domain."""
    return (0.0, 2 * math.pi) if case["flow"] == "tgv" else (-1.0, 2.0)


def _layout(case):
    """Elements as boxes in units of the finest cells (lower corners, sizes, domain), frames, connectivity, mortars."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["mesh"] == "mortar":
        def block(mx, my, mz, x0, size):
            k, j, i = np.meshgrid(np.arange(mz), np.arange(my), np.arange(mx), indexing="ij")
            lo = np.stack([i.ravel(), j.ravel(), k.ravel()], 1) * size
            lo[:, 0] += x0
            return lo, k * 0 + np.arange(k.size).reshape(k.shape)
        lo1, id1 = block(nx, ny, nz, 0, 2)
        lo2, id2 = block(2 * nx, 2 * ny, 2 * nz, 2 * nx, 1)
        id2 = id2 + len(lo1)
        conn = []
        for ids in (id1, id2):
            c = np.zeros(ids.shape + (6, 3), dtype=np.int32)
            for s in range(6):
                c[..., s, 0] = np.roll(ids, 1 if s % 2 == 0 else -1, axis=2 - s // 2)
                c[..., s, 1] = s ^ 1
            conn.append(c)
        rows = []
        for side, col in ((1, nx - 1), (0, 0)):  # coarse +x faces against fine -x faces, and across the period
            for k in range(nz):
                for j in range(ny):
                    m = len(rows)
                    conn[0][k, j, col, side] = (F.CONN_MORTAR, m, -1)
                    row = [id1[k, j, col], side, 3]
                    for pos in range(4):
                        at = (2 * k + pos // 2, 2 * j + pos % 2, 0 if side else 2 * nx - 1)
                        conn[1][at][side ^ 1] = (F.CONN_MORTAR, m, pos)
                        row += [id2[at], side ^ 1, 0]
                    rows.append(row)
        lo = np.concatenate([lo1, lo2])
        size = np.concatenate([np.full(len(lo1), 2), np.full(len(lo2), 1)])
        return (lo, size, np.array([4 * nx, 2 * ny, 2 * nz]), np.zeros(len(lo), dtype=np.int64),
                np.concatenate([c.reshape(-1, 6, 3) for c in conn]), np.array(rows, dtype=np.int32))
    dims = np.array([nx, ny, nz])
    k, j, i = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    lo = np.stack([i.ravel(), j.ravel(), k.ravel()], 1)
    K = len(lo)
    ident = int(np.argmax([np.array_equal(R, np.eye(3)) for R in _frames()]))
    frame = np.random.default_rng(K).integers(24, size=K) if case["turned"] else np.full(K, ident)
    conn = np.zeros((K, 6, 3), dtype=np.int32)
    table = np.zeros((24, 24, 2), dtype=np.int32)
    for s in range(6):
        out = _frames()[frame][:, :, s // 2] * (2 * (s % 2) - 1)
        to = lo + out
        nb = (to % dims) @ np.array([1, nx, nx * ny])
        for a, b in set(zip(frame.tolist(), frame[nb].tolist())):
            table[a, b] = _joint(a, b, s)
        conn[:, s, 0] = nb
        conn[:, s, 1:] = table[frame, frame[nb]]
        if case["boundary"] != "periodic":  # boundary ids 0..5 for -x, +x, -y, +y, -z, +z; "mixed" is periodic in z
            gone = ((to < 0) | (to >= dims)) & np.array([True, True, case["boundary"] == "exact"])
            face = 2 * np.argmax(np.abs(out), 1) + (out.sum(1) > 0)
            e = np.flatnonzero(gone.any(1))
            conn[e, s] = np.stack([-1 - face[e], -1 + 0 * e, 0 * e], 1)
    return lo, np.ones(K, dtype=np.int64), dims, frame, conn, None


def _points(case, layout, r, device):
    """Physical coordinates [K, m, m, m, 3] at the tensor product of the reference points r."""
    lo, size, dims, frame, _, _ = layout
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=device)
    m, x = len(r), t(r)
    xi = torch.stack([x.view(1, 1, m).expand(m, m, m), x.view(1, m, 1).expand(m, m, m), x.view(m, 1, 1).expand(m, m, m)], -1)
    eta = torch.einsum("kab,...b->k...a", t(_frames()[frame]), xi)
    K = len(lo)
    u = (t(lo).view(K, 1, 1, 1, 3) + (eta + 1) / 2 * t(size).view(K, 1, 1, 1, 1)) / t(dims)  # [0, 1]^3
    if case["mesh"] == "sine":
        u = u + 0.05 * torch.sin(math.pi * (2 * u - 1)).prod(-1, keepdim=True)
    x0, length = _extent(case)
    return x0 + length * u


def _reference(case, x, t):
    """Exact state of the case's flow at x [..., 3], conserved variables last."""
    X, Y, Z = x.unbind(-1)
    if case["flow"] == "mms":
        rho = 2.0 + 0.1 * torch.sin(math.pi * (X + Y + Z - 2.0 * t))
        return torch.stack([rho, rho, rho, rho, rho * rho], -1)
    if case["flow"] == "freestream":
        one = torch.ones_like(X)
        return _cons(one, 0.3 * one, 0.2 * one, 0.1 * one, one / GAMMA)
    u = torch.sin(X) * torch.cos(Y) * torch.cos(Z)
    v = -torch.cos(X) * torch.sin(Y) * torch.cos(Z)
    p = 1.0 / (GAMMA * case["Ma"] ** 2) + (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2.0) / 16.0
    return _cons(torch.ones_like(u), u, v, torch.zeros_like(u), p)


def _cons(rho, u, v, w, p):
    return torch.stack([rho, rho * u, rho * v, rho * w, p / (GAMMA - 1) + 0.5 * rho * (u * u + v * v + w * w)], -1)


def _start(case, layout, seed, device):
    """Initial state [K, 5, n, n, n] in 64 bits: the flow, where it is periodic shifted at random and carried by a
    slow mean wind, with smooth small-scale disturbances of 2 per cent."""
    rng = np.random.default_rng(seed)
    x = _points(case, layout, _nodes(case["N"], case["nodes"])[0], device)
    shift = torch.as_tensor(rng.uniform(0, 2 * math.pi, 3) if case["flow"] == "tgv" else np.zeros(3), device=device)
    W = _prim(_reference(case, x + shift, 0.0).movedim(-1, 1))
    k0 = 2 * math.pi / _extent(case)[1]

    def field():
        f = 0.0
        for _ in range(3):
            k = k0 * rng.integers(-2, 3, 3)
            f = f + rng.normal() * torch.sin(k[0] * x[..., 0] + k[1] * x[..., 1] + k[2] * x[..., 2] + rng.uniform(0, 6.28))
        return 0.02 * f

    wind = (0.1, 0.07, 0.05) if case["flow"] == "tgv" else (0.0, 0.0, 0.0)
    return _cons(W[:, 0] * (1 + field()), W[:, 1] + wind[0] + field(), W[:, 2] + wind[1] + field(), W[:, 3] + wind[2] + field(),
                 W[:, 4] * (1 + 0.1 * field())).movedim(-1, 1).contiguous()


def _dt(case):
    """Time step from the convective and viscous limits at about half of the admissible size."""
    dims = np.array([2 * case["nx"] + 2 * case["nx"], 2 * case["ny"], 2 * case["nz"]]) if case["mesh"] == "mortar" \
        else np.array([case["nx"], case["ny"], case["nz"]])
    rate = 2.0 / (_extent(case)[1] / dims) * (1.6 if case["mesh"] == "sine" else 1.0)
    speed = 1.2 + {"tgv": 1.0 / case["Ma"], "mms": 1.2, "freestream": 1.0}[case["flow"]]
    n = 2 * case["N"] + 1
    return float(0.5 * min(2.0 / (n * speed * rate.sum()), 4.0 / (n * 2.0 / case["Re"] * (rate ** 2).sum())))


def _kinetic_weights(case, layout, device):
    """Quadrature weights times the Jacobian of a Cartesian mesh, [K, n, n, n]."""
    w = torch.as_tensor(_nodes(case["N"], case["nodes"])[1], device=device)
    vol = np.prod(_extent(case)[1] / layout[2]) / 8.0 * layout[1] ** 3.0
    return torch.as_tensor(vol, device=device).view(-1, 1, 1, 1) * w.view(-1, 1, 1) * w.view(1, -1, 1) * w.view(1, 1, -1)


def _cotangent(U, seed):
    g = torch.Generator(device=U.device).manual_seed(int(seed))
    return torch.randn(U.shape, dtype=U.dtype, device=U.device, generator=g)


# ---------------------------------------------------------------- the calls


def prepare(case, seed):
    layout = _layout(case)
    geo = case["N"] if case["mesh"] == "sine" else 1
    coords = _points(case, layout, _nodes(geo, "lobatto")[0], "cuda").cpu().numpy()
    cfg = SolverConfig(N=case["N"], Ngeo=geo, node_type=F.NODES_GAUSS if case["nodes"] == "gauss" else F.NODES_LOBATTO,
                       riemann=RIEMANN[case["riemann"]], precision=PRECISION[case["precision"]],
                       bc_exact=FLOW[case["flow"]], source=case["flow"] == "mms", split_form=SPLIT[case["split"]],
                       adjoint=case["call"] in ("gradient", "adjoint"),
                       lifting=F.LIFTING_BR2 if case["lifting"] == "br2" else F.LIFTING_BR1,
                       gamma=GAMMA, Pr=PR, mu=1.0 / case["Re"], Ma=case["Ma"])
    solver = Solver(cfg, coords, layout[4], mortars=layout[5])
    if case["boundary"] == "mixed":
        solver.set_bc(1, F.BC_OUTFLOW)
        solver.set_bc(2, F.BC_SLIP_WALL)
        solver.set_bc(3, F.BC_SLIP_WALL)
    s = {"case": case, "solver": solver, "dt": _dt(case)}
    s["U0"] = _start(case, layout, seed, "cuda").to(solver.dtype)
    s["U"] = torch.empty_like(s["U0"])
    s["Ut"] = torch.empty_like(s["U0"]) if case["call"] != "reduce" else solver.rhs(s["U0"])
    s["stream"] = torch.cuda.Stream() if case["own_stream"] else torch.cuda.current_stream()
    if case["call"] == "gradient":
        s["weights"] = _kinetic_weights(case, layout, "cuda") if case["mesh"] != "sine" else 1.0
    if case["call"] == "adjoint":
        s["lam"] = _cotangent(s["U0"], seed)
    return s


def run(state):
    case, solver = state["case"], state["solver"]
    with torch.cuda.stream(state["stream"]):
        if case["call"] == "run":
            state["U"].copy_(state["U0"])  # the run advances its state in place
            return solver.run(state["U"], case["steps"], state["dt"])
        if case["call"] == "rhs":
            return solver.rhs(state["U0"], 0.0, out=state["Ut"])
        if case["call"] == "adjoint":
            return solver.rhs_adjoint(state["U0"], state["lam"], 0.0, out=state["Ut"])
        if case["call"] == "reduce":
            return solver.reduce(state["U0"], state["Ut"])
        U0 = state["U0"].clone().requires_grad_(True)
        U = final_state(U0, solver, case["steps"], state["dt"], checkpoint_every=case["checkpoint_every"])
        _energy(U, state["weights"]).backward()
        return U.detach(), U0.grad


def _energy(U, weights):
    return (weights * 0.5 * (U[:, 1] ** 2 + U[:, 2] ** 2 + U[:, 3] ** 2) / U[:, 0]).sum()


def work(case):
    """Per right-hand side and node: the state, its register and the geometry (9 metric terms, 1/J) read once,
    state and register written once; the line contractions of 45 lifting and 15 flux fields, the transforms and
    pointwise fluxes; the faces' share.  A run has five right-hand sides a step; a gradient recomputes the forward
    run once but for the last segment and adds one reverse pass at twice the arithmetic."""
    n = case["N"] + 1
    elements = case["nx"] * case["ny"] * case["nz"] * (9 if case["mesh"] == "mortar" else 1)
    nodes, word = elements * n ** 3, 8 if case["precision"] == "fp64" else 4
    f = 3.0 / n
    flops = 120.0 * n + 280 + 300 * f + (480 if case["nodes"] == "gauss" else 480.0 / n)
    if case["split"] != "standard":
        flops += (n + 1) / 2 * 3 * (40 if case["split"] == "kep" else 110)
    if case["call"] == "reduce":
        return {"bytes": 8.0 * nodes * 21, "flops": 100.0 * nodes}
    if case["call"] == "rhs":
        return {"bytes": (20.0 + 4 * f) * nodes * word, "flops": flops * nodes}
    if case["call"] == "adjoint":
        return {"bytes": (25.0 + 4 * f) * nodes * word, "flops": 3 * flops * nodes}
    stages = 5.0 * case["steps"]
    if case["call"] == "gradient":
        return {"bytes": (3 * 30.0 + 4 * f) * nodes * word * stages, "flops": 4 * flops * nodes * stages}
    return {"bytes": (30.0 + 4 * f) * nodes * word * stages, "flops": flops * nodes * stages}


# ---------------------------------------------------------------- the same in plain torch, 64 bits


def _prim(U):
    rho, u, v, w = U[:, 0], U[:, 1] / U[:, 0], U[:, 2] / U[:, 0], U[:, 3] / U[:, 0]
    return torch.stack([rho, u, v, w, (GAMMA - 1) * (U[:, 4] - 0.5 * rho * (u * u + v * v + w * w))], 1)


def _cons1(W):
    return _cons(W[:, 0], W[:, 1], W[:, 2], W[:, 3], W[:, 4]).movedim(-1, 1)


def _lagrange(x, at):
    """l_j(at_r), [len(at), len(x)]."""
    V = np.ones((len(at), len(x)))
    for j in range(len(x)):
        for i in range(len(x)):
            if i != j:
                V[:, j] *= (at - x[i]) / (x[j] - x[i])
    return V


def _derivative(x):
    n = len(x)
    w = np.array([1.0 / np.prod([x[j] - x[k] for k in range(n) if k != j]) for j in range(n)])
    D = np.array([[0.0 if r == s else w[s] / w[r] / (x[r] - x[s]) for s in range(n)] for r in range(n)])
    return D - np.diag(D.sum(1))


def _along(M, f, l):
    """Applies M along reference direction l of f[..., k, j, i]."""
    ax = f.dim() - 1 - l
    return torch.tensordot(f.movedim(ax, -1), M, dims=([-1], [1])).movedim(-1, ax)


def _dot(a, b):
    return (a * b).sum(1, keepdim=True)


def _conv(U, W, n):
    """Convective flux along n (any length), variables and components on axis 1."""
    un = _dot(W[:, 1:4], n)
    return torch.cat([U[:, :1] * un, U[:, 1:4] * un + W[:, 4:] * n, (U[:, 4:] + W[:, 4:]) * un], 1)


def _visc(W, G, n, mu):
    """Viscous flux along n; G [B, 3, 5, ...] holds d W_v / d x_d."""
    v, g = W[:, 1:4], G[:, :, 1:4]  # g[:, d, c] = d u_c / d x_d
    div = g[:, 0, 0] + g[:, 1, 1] + g[:, 2, 2]
    tn = mu * ((g * n.unsqueeze(2)).sum(1) + (g * n.unsqueeze(1)).sum(2) - 2.0 / 3.0 * div.unsqueeze(1) * n)
    gT = (G[:, :, 4] - (W[:, 4:] / W[:, :1]) * G[:, :, 0]) / W[:, :1]
    return torch.cat([torch.zeros_like(tn[:, :1]), tn, _dot(tn, v) + mu * GAMMA / ((GAMMA - 1) * PR) * _dot(gT, n)], 1)


def _log_mean(a, b):
    z = a / b
    f = (z - 1) / (z + 1)
    u = f * f
    series = sum(u ** k / (2 * k + 1) for k in range(9))
    near = u < 1e-2
    return (a + b) / (2 * torch.where(near, series, torch.log(z) / (2 * torch.where(near, torch.ones_like(f), f))))


def _pair(kind, Ua, Wa, Ub, Wb, n):
    """Two-point flux along n: kinetic energy preserving (Pirozzoli) or entropy conservative (Chandrashekar)."""
    v = 0.5 * (Wa[:, 1:4] + Wb[:, 1:4])
    un = _dot(v, n)
    if kind == "kep":
        m = 0.5 * (Wa[:, :1] + Wb[:, :1]) * un
        H = 0.5 * ((Ua[:, 4:] + Wa[:, 4:]) / Wa[:, :1] + (Ub[:, 4:] + Wb[:, 4:]) / Wb[:, :1])
        return torch.cat([m, m * v + 0.5 * (Wa[:, 4:] + Wb[:, 4:]) * n, m * H], 1)
    ba, bb = Wa[:, :1] / (2 * Wa[:, 4:]), Wb[:, :1] / (2 * Wb[:, 4:])
    q2 = 0.5 * (_dot(Wa[:, 1:4], Wa[:, 1:4]) + _dot(Wb[:, 1:4], Wb[:, 1:4]))
    m = _log_mean(Wa[:, :1], Wb[:, :1]) * un
    fm = m * v + 0.5 * (Wa[:, :1] + Wb[:, :1]) / (ba + bb) * n
    return torch.cat([m, fm, m * (1 / (2 * (GAMMA - 1) * _log_mean(ba, bb)) - 0.5 * q2) + _dot(v, fm)], 1)


def _riemann(kind, UL, UR, n):
    WL, WR = _prim(UL), _prim(UR)
    if kind == "ec":
        return _pair("ec", UL, WL, UR, WR, n)
    FL, FR = _conv(UL, WL, n), _conv(UR, WR, n)
    uL, uR = _dot(WL[:, 1:4], n), _dot(WR[:, 1:4], n)
    cL, cR = torch.sqrt(GAMMA * WL[:, 4:] / WL[:, :1]), torch.sqrt(GAMMA * WR[:, 4:] / WR[:, :1])
    if kind == "rusanov":
        return 0.5 * (FL + FR) - 0.5 * torch.maximum(uL.abs() + cL, uR.abs() + cR) * (UR - UL)
    sL, sR = torch.sqrt(WL[:, :1]), torch.sqrt(WR[:, :1])
    v = (sL * WL[:, 1:4] + sR * WR[:, 1:4]) / (sL + sR)
    H = (sL * (UL[:, 4:] + WL[:, 4:]) / WL[:, :1] + sR * (UR[:, 4:] + WR[:, 4:]) / WR[:, :1]) / (sL + sR)
    q2, un = _dot(v, v), _dot(v, n)
    c = torch.sqrt((GAMMA - 1) * (H - 0.5 * q2))
    if kind == "hllc":
        SL, SR = torch.minimum(uL - cL, un - c), torch.maximum(uR + cR, un + c)
        mL, mR = WL[:, :1] * (SL - uL), WR[:, :1] * (SR - uR)
        S = (WR[:, 4:] - WL[:, 4:] + uL * mL - uR * mR) / (mL - mR)

        def star(U, W, Sk, uk, mk, Fk):
            fac = mk / (Sk - S)
            E = fac * (U[:, 4:] / W[:, :1] + (S - uk) * (S + W[:, 4:] / mk))
            return Fk + Sk * (torch.cat([fac, fac * (W[:, 1:4] + (S - uk) * n), E], 1) - U)

        return torch.where(SL >= 0, FL, torch.where(S >= 0, star(UL, WL, SL, uL, mL, FL),
                                                    torch.where(SR >= 0, star(UR, WR, SR, uR, mR, FR), FR)))
    d = WR - WL
    dun = _dot(d[:, 1:4], n)

    def size(lam):
        if kind == "roe":
            return lam.abs()
        dl = 0.1 * c
        return torch.where(lam.abs() < dl, (lam * lam + dl * dl) / (2 * dl), lam.abs())

    rho = sL * sR
    w1, w5 = size(un - c) * (d[:, 4:] - rho * c * dun) / (2 * c * c), size(un + c) * (d[:, 4:] + rho * c * dun) / (2 * c * c)
    l2 = size(un)
    one, dt = torch.ones_like(un), d[:, 1:4] - dun * n
    diss = w1 * torch.cat([one, v - c * n, H - un * c], 1) + w5 * torch.cat([one, v + c * n, H + un * c], 1) \
        + l2 * (d[:, :1] - d[:, 4:] / (c * c)) * torch.cat([one, v, 0.5 * q2], 1) \
        + l2 * rho * torch.cat([0 * one, dt, _dot(v, dt)], 1)
    return 0.5 * (FL + FR) - 0.5 * diss


class _Plain:
    """The semi-discrete operator, equation by equation."""

    def __init__(self, case, device):
        self.case, self.device = case, device
        N, n = case["N"], case["N"] + 1
        self.layout = _layout(case)
        lo, size, dims, frame, conn, mortars = self.layout
        self.K, self.n = len(lo), n
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=device)
        x, w = _nodes(N, case["nodes"])
        D = _derivative(x)
        self.D, self.Dhat = t(D), t(-(w[None, :] / w[:, None]) * D.T)
        self.l = [t(_lagrange(x, np.array([e]))[0]) for e in (-1.0, 1.0)]
        self.lhat = [v / t(w) for v in self.l]
        halves = [_lagrange(x, (x + 2 * a - 1) / 2) for a in (0, 1)]
        self.I = [t(V) for V in halves]
        self.P = [t(V.T * w[None, :] / w[:, None]) for V in halves]
        # mapping, curl-form metrics collocated on the Gauss-Lobatto points of degree N
        geo = N if case["mesh"] == "sine" else 1
        xg, xl = _nodes(geo, "lobatto")[0], _nodes(N, "lobatto")[0]
        X = _points(case, self.layout, xg, device).movedim(-1, 1)

        def to(f, a, b):
            V = t(_lagrange(a, b))
            for l in range(3):
                f = _along(V, f, l)
            return f

        self.x = to(X, xg, x)
        X = X - X[:, :, :1, :1, :1]
        Xs = to(X, xg, x)
        self.J = torch.linalg.det(torch.stack([_along(self.D, Xs, l) for l in range(3)], 2).permute(0, 3, 4, 5, 1, 2))
        Dl, Xl = t(_derivative(xl)), to(X, xg, xl)
        dX = [_along(Dl, Xl, l) for l in range(3)]
        Ja = torch.empty(self.K, 3, 3, n, n, n, dtype=torch.float64, device=device)
        for d in range(3):
            m, p = (d + 1) % 3, (d + 2) % 3
            for i in range(3):
                i1, i2 = (i + 1) % 3, (i + 2) % 3
                Ja[:, i, d] = _along(Dl, Xl[:, p] * dX[i1][:, m], i2) - _along(Dl, Xl[:, p] * dX[i2][:, m], i1)
        self.Ja = to(Ja.flatten(1, 2), xl, x).view(self.K, 3, 3, n, n, n)
        # faces: outward normal times surface element, neighbour's element-side and node
        self.nF = torch.stack([(2 * (s % 2) - 1) * self.face(self.Ja[:, s // 2], s) for s in range(6)], 1)
        self.sF = (self.nF ** 2).sum(2, keepdim=True).sqrt()
        c = t(conn.astype(np.int64))
        p, q = np.meshgrid(np.arange(n), np.arange(n))
        maps = []
        for o in range(8):
            a, b = (q, p) if o & 1 else (p, q)
            maps.append(((N - b if o & 4 else b) * n + (N - a if o & 2 else a)).ravel())
        self.bnd = (c[..., 0] < 0) & (c[..., 0] != F.CONN_MORTAR)
        inner = c[..., 0] >= 0
        own = torch.arange(self.K * 6, device=device).view(self.K, 6)
        self.nb = torch.where(inner, c[..., 0] * 6 + c[..., 1], own)
        self.at = t(np.stack(maps))[torch.where(inner, c[..., 2], torch.zeros_like(own))]  # [K, 6, n^2]
        self.bc = (-1 - c[..., 0]) * self.bnd
        if mortars is not None:
            r = t(mortars.astype(np.int64))
            self.big = r[:, 0] * 6 + r[:, 1]
            self.small = torch.stack([r[:, 3 + 3 * k] * 6 + r[:, 4 + 3 * k] for k in range(4)], 1)
        else:
            self.big = None
        if self.bnd.any():
            xf = torch.stack([self.face(self.x, s) for s in range(6)], 1)  # [K, 6, 3, n^2]
            self.xb = xf[self.bnd].movedim(1, -1)
        if case["flow"] == "mms":
            self.s = self.x.sum(1)

    def face(self, f, s):
        """Values of f [K, C, n, n, n] on side s, [K, C, n^2] with the first free index fastest."""
        return torch.tensordot(f, self.l[s % 2], dims=([f.dim() - 1 - s // 2], [0])).flatten(-2)

    def faces(self, f):
        return torch.stack([self.face(f, s) for s in range(6)], 1)

    def spread(self, q, s):
        """l_hat_s times the face values q [K, C, n^2]."""
        n = self.n
        q = q.view(q.shape[0], q.shape[1], n, n)
        return q.unsqueeze(4 - s // 2) * self.lhat[s % 2].view([n if a == s // 2 else 1 for a in (2, 1, 0)])

    def halved(self, M, f, pos):
        n = self.n
        f = f.view(f.shape[0], f.shape[1], n, n)
        return torch.einsum("ab,cd,mvdb->mvac", M[pos % 2], M[pos // 2], f).transpose(2, 3).flatten(2)

    def across(self, f):
        """The neighbour's values of the face array f [K, 6, C, n^2] in this element's face frame."""
        K, _, C, n2 = f.shape
        flat = f.reshape(K * 6, C, n2)
        g = torch.gather(flat[self.nb.reshape(-1)], 2, self.at.reshape(K * 6, 1, n2).expand(-1, C, -1))
        if self.big is not None:
            for pos in range(4):
                g = g.index_copy(0, self.small[:, pos], self.halved(self.I, flat[self.big], pos))
        return g.view(K, 6, C, n2)

    def projected(self, f):
        """f [K, 6, C, n^2] with the big sides' values minus the projection of their small sides'."""
        if self.big is None:
            return f
        flat = f.reshape(-1, f.shape[2], f.shape[3])
        return flat.index_copy(0, self.big, -sum(self.halved(self.P, flat[self.small[:, p]], p) for p in range(4))).view(f.shape)

    def outer(self, UF, t):
        """Boundary states at the boundary sides' nodes, [B, 5, n^2]."""
        case = self.case
        exact = _reference(case, self.xb, t).movedim(-1, 1)
        if case["boundary"] != "mixed":
            return exact
        inner, n = UF[self.bnd], (self.nF / self.sF)[self.bnd]
        wall = torch.cat([inner[:, :1], inner[:, 1:4] - 2 * _dot(inner[:, 1:4], n) * n, inner[:, 4:]], 1)
        b = self.bc[self.bnd].view(-1, 1, 1)
        return torch.where(b == 1, inner, torch.where((b == 2) | (b == 3), wall, exact))

    def rhs(self, U, t):
        case, K, n, n2, mu = self.case, self.K, self.n, self.n ** 2, 1.0 / self.case["Re"]
        W, J = _prim(U), self.J.unsqueeze(1)
        UF = self.faces(U)
        UN = self.across(UF)
        if self.bnd.any():
            UN = UN.index_put((self.bnd,), self.outer(UF, t))
        flat = lambda f: f.reshape(K * 6, -1, n2)
        WF, WN = _prim(flat(UF)), _prim(flat(UN))
        nF = flat(self.nF)
        Q = self.projected((0.5 * (WF + WN).unsqueeze(1) * nF.unsqueeze(2)).reshape(K, 6, 15, n2))  # (d, v)
        G, lift = [], [[] for _ in range(6)]
        for d in range(3):
            acc = sum(_along(self.Dhat, self.Ja[:, l, d].unsqueeze(1) * W, l) for l in range(3))
            G.append((acc + sum(self.spread(Q[:, s, 5 * d:5 * d + 5], s) for s in range(6))) / J)
        G = torch.stack(G, 1)  # [K, 3, 5, n, n, n]
        if case["lifting"] == "br2":
            jump = Q - (WF.unsqueeze(1) * nF.unsqueeze(2)).reshape(K, 6, 15, n2)
            r = [self.spread(jump[:, s], s) / J for s in range(6)]
            broken = G.flatten(1, 2) - sum(r)
            GF = torch.stack([self.face(broken + 2.0 * r[s], s) for s in range(6)], 1)
        else:
            GF = self.faces(G.flatten(1, 2))
        GN = self.across(GF)
        if self.bnd.any():
            GN = torch.where(self.bnd.view(K, 6, 1, 1), GF, GN)
        s_ = flat(self.sF)
        nv = nF / s_
        g5 = lambda g: g.reshape(K * 6, 3, 5, n2)
        f = _riemann(case["riemann"], flat(UF), flat(UN), nv) - 0.5 * (_visc(WF, g5(GF), nv, mu) + _visc(WN, g5(GN), nv, mu))
        f = self.projected((f * s_).view(K, 6, 5, n2))
        out = 0.0
        for l in range(3):
            Jl = self.Ja[:, l]
            fc, fv = _conv(U, W, Jl), _visc(W, G, Jl, mu)
            if case["split"] == "standard":
                out = out + _along(self.Dhat, fc - fv, l)
                inner = None
            else:
                ax = 4 - l
                a = lambda q: q.unsqueeze(ax + 1)
                b = lambda q: q.unsqueeze(ax)
                Fs = _pair(case["split"], a(U), a(W), b(U), b(W), 0.5 * (a(Jl) + b(Jl)))
                shape = [1] * 6
                shape[ax], shape[ax + 1] = n, n
                out = out + 2 * (Fs * self.D.view(shape)).sum(ax + 1) - _along(self.D, fv, l)
                inner = fc - fv
            for s in (2 * l, 2 * l + 1):
                q = f[:, s] if inner is None else f[:, s] - (2 * (s % 2) - 1) * self.face(inner, s)
                out = out + self.spread(q, s)
        Ut = -out / J
        if case["flow"] == "mms":
            ph = math.pi * (self.s - 2 * t)
            r, r1, r2 = 2 + 0.1 * torch.sin(ph), 0.1 * math.pi * torch.cos(ph), -0.1 * math.pi ** 2 * torch.sin(ph)
            p1 = (GAMMA - 1) * (2 * r - 1.5) * r1
            Sm = r1 + p1
            Ut = Ut + torch.stack([r1, Sm, Sm, Sm, 2 * r * r1 + 3 * p1 - 3 * mu * GAMMA / PR * r2], 1)
        return Ut

    def steps(self, U, steps, dt, kept=None):
        A = [0.0, -567301805773 / 1357537059087, -2404267990393 / 2016746695238, -3550918686646 / 2091501179385,
             -1275806237668 / 842570457699]
        B = [1432997174477 / 9575080441755, 5161836677717 / 13612068292357, 1720146321549 / 2090206949498,
             3134564353537 / 4481467310338, 2277821191437 / 14882151754819]
        C = [0.0, 1432997174477 / 9575080441755, 2526269341429 / 6820363962896, 2006345519317 / 3224310063776,
             2802321613138 / 2924317926251]
        dU = torch.zeros_like(U)
        for k in range(steps):
            for a, b, c in zip(A, B, C):
                if kept is not None:
                    kept.append((U, a, b))
                dU = a * dU + dt * self.rhs(U, (k + c) * dt)
                U = U + b * dU
        return U

    def transposed(self, U, lam):
        with torch.enable_grad():
            x = U.detach().requires_grad_(True)
            return torch.autograd.grad(self.rhs(x, 0.0), x, lam)[0]


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    op = _Plain(case, device)
    U0 = _start(case, op.layout, seed, device)
    U = U0 if case["precision"] == "fp64" else U0.float().double()
    with torch.no_grad():
        if case["call"] == "run":
            return op.steps(U, case["steps"], _dt(case))
        if case["call"] == "rhs":
            return op.rhs(U, 0.0)
        if case["call"] == "adjoint":
            return op.transposed(U, _cotangent(U, seed))
        if case["call"] == "gradient":
            kept, dt = [], _dt(case)
            UT = op.steps(U, case["steps"], dt, kept)
            wts = _kinetic_weights(case, op.layout, device) if case["mesh"] != "sine" else 1.0
            with torch.enable_grad():
                x = UT.detach().requires_grad_(True)
                lam = torch.autograd.grad(_energy(x, wts), x)[0]
            mu = torch.zeros_like(lam)
            for Uk, a, b in reversed(kept):
                mu = mu + b * lam
                lam = lam + dt * op.transposed(Uk, mu)
                mu = a * mu
            return UT, lam
        # reduce: sums with the quadrature weights, and the time step limits summed over the reference directions
        w = torch.as_tensor(_nodes(case["N"], case["nodes"])[1], device=device)
        wJ = op.J * w.view(-1, 1, 1) * w.view(1, -1, 1) * w.view(1, 1, -1)
        Ut, W = op.rhs(U, 0.0), _prim(U)
        v2 = (W[:, 1:4] ** 2).sum(1)
        tot = [float((wJ * U[:, v]).sum()) for v in range(5)]
        rate = (W[:, 1:4] * Ut[:, 1:4]).sum(1) - 0.5 * v2 * Ut[:, 0]
        c = torch.sqrt(GAMMA * W[:, 4] / W[:, 0])
        conv = visc = 0.0
        for l in range(3):
            length = (op.Ja[:, l] ** 2).sum(1).sqrt()
            conv = conv + ((op.Ja[:, l] * W[:, 1:4]).sum(1).abs() + c * length) / op.J
            visc = visc + max(4 / 3, GAMMA / PR) / case["Re"] / W[:, 0] * (length / op.J) ** 2
        n = 2 * case["N"] + 1
        return {"mass": tot[0], "mom_x": tot[1], "mom_y": tot[2], "mom_z": tot[3], "energy": tot[4],
                "kinetic_energy": float((wJ * 0.5 * U[:, 0] * v2).sum()), "dkedt": float((wJ * rate).sum()),
                "dt_max": 0.9 * min(2.0 / (n * float(conv.max())), 4.0 / (n * float(visc.max()))), "status": 0}
