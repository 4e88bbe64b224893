"""The stable time step of flexi_reduce: FP32 bounds choose the nodes whose rates are evaluated
in FP64, so the value is the one of evaluating every node.

Scaling the units by 2^b (velocity and viscosity by 2^b, pressure by 2^2b) scales every FP64
operation exactly; at b = -70 the pressure is below the FP32 range and every node is evaluated
in FP64.  The two time steps are therefore equal to the bit, whichever rate sets them.  With a
NaN the allocation-free form, which evaluates every node, is the other side: about 40 roundings
of 2^-53 lie between the two.
"""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


def _solver(N, mapping, mu):
    from paper_1910_02858_gb300 import Solver, SolverConfig

    mesh = wl.box_mesh((3, 2, 4), lo=(0.0,) * 3, hi=(2 * np.pi,) * 3, Ngeo=N if mapping == "sine" else 1, mapping=mapping,
                       reorient_seed=N)
    return Solver(SolverConfig(N=N, Ngeo=mesh.Ngeo, mu=mu), mesh.coords, mesh.conn), mesh


def _dt(N, mapping, state, mu, b):
    import torch

    s, mesh = _solver(N, mapping, mu * 2.0 ** b)
    U = wl.perturbed(mesh.node_coords(N, 0), seed=N)
    if state == "uniform":  # every node of an affine element ties
        U[:] = np.array([1.0, 0.3, 0.2, 0.1, 2.0]).reshape(1, 5, 1, 1, 1)
    f = 2.0 ** b
    U = U * np.array([1.0, f, f, f, f * f]).reshape(1, 5, 1, 1, 1)
    dt = s.reduce(torch.tensor(U, device="cuda:0"))["dt_max"]
    s.close()
    return dt * f


@pytest.mark.parametrize("mu", [1e-4, 10.0], ids=["convective", "viscous"])
@pytest.mark.parametrize("state", ["uniform", "perturbed"])
@pytest.mark.parametrize("N,mapping", [(1, "cartesian"), (4, "cartesian"), (2, "sine"), (7, "sine")])
def test_bounds_keep_the_largest_rate(N, mapping, state, mu):
    assert _dt(N, mapping, state, mu, 0) == _dt(N, mapping, state, mu, -70)


@pytest.mark.parametrize("N", [3, 7])
def test_nan_node_changes_no_other(N):
    import torch

    from paper_1910_02858_gb300 import flexi as F

    s, mesh = _solver(N, "cartesian", 1e-3)
    U = wl.perturbed(mesh.node_coords(N, 0), seed=N)
    U[2, 1, 0, 1, 1] = np.nan
    Ud = torch.tensor(U, device="cuda:0")
    got = s.reduce(Ud, allow_nonphysical=True)["dt_max"]
    ref = F.flexi_reduce_noalloc(s.ctx, Ud, None, 0.9, torch.cuda.current_stream())[0][7]
    s.close()
    assert np.isfinite(ref) and abs(got - ref) <= 40 * 2.0 ** -53 * ref
