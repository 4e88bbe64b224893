"""Flat elements: the FP64 form's fixed-point contractions keep the accuracy of FP64 sums in every
variable where the metric terms of one direction exceed the others by the aspect ratio.

A box of elements of thickness 2^-20 in z carries a flow that is constant in z, with the velocity
w of the order of the thickness, so that the large metric term Ja_z meets small fluxes only.  The
other side is the FP64 body of the same kernels, reached by scaling the units by powers of two
(as in test_gpu_fixed_point.py), which scales every FP64 operation exactly.

Tolerance, derived: a node's value is a sum over the three directions of line contractions; with
mu = 0 each term of direction d is at most max|F_d,v| max|Ja_d| rowsum(|Dhat| + |lhat|) / min J =
T_d,v.  Each side rounds at most 2 * 3 (N + 3) times, relative to sum_d T_d,v; the same again for
products and pointwise fluxes.  A quantum relative to max|F| max|Ja| would be larger by the aspect ratio.
"""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu
THIN = 2.0 ** -20
SHAPE = (4, 3, 2)


def _mesh(mapping, seed):
    hi = (2 * np.pi, 2 * np.pi, 2 * np.pi * THIN)
    if mapping == "box":
        return wl.box_mesh(SHAPE, lo=(0.0,) * 3, hi=hi, Ngeo=1, reorient_seed=seed)
    mesh = wl.box_mesh(SHAPE, lo=(0.0,) * 3, hi=hi, Ngeo=2, reorient_seed=seed)
    mesh.coords[..., 0] += 0.1 * np.sin(mesh.coords[..., 0]) * np.sin(mesh.coords[..., 1])  # columns along z
    return mesh


def _state(mesh, N, nodes):
    x = mesh.node_coords(N, nodes)
    X, Y = x[:, 0], x[:, 1]
    rho = 1.0 + 0.1 * np.sin(X) * np.cos(Y)
    return np.stack([rho, np.sin(X) * np.cos(Y), -0.7 * np.cos(X) * np.sin(Y), np.cos(X + Y) * THIN,
                     2.0 + 0.1 * np.sin(X + Y)], axis=1)


def _bound(W, N, nodes):
    """sum_d T_d,v by variable, and the T_d without fluxes."""
    from oracle.basis import Basis

    b = Basis(N, nodes)
    R = float((b.Dhat.abs().sum(1) + b.lhat_minus.abs() + b.lhat_plus.abs()).max())
    h = np.array([2 * np.pi, 2 * np.pi, 2 * np.pi * THIN]) / np.array(SHAPE) / 2
    g = 1.6 * R / h  # rowsum * max|Ja_d| / min J, the distortion included
    rho, vel, p = np.abs(W[:, 0]).max(), [np.abs(W[:, 1 + d]).max() for d in range(3)], W[:, 4].max()
    E = p / 0.4 + 0.5 * rho * sum(v * v for v in vel)
    T = np.zeros(5)
    for d in range(3):
        F = np.array([rho * vel[d]] + [rho * vel[d] * vel[c] + (p if c == d else 0.0) for c in range(3)] + [vel[d] * (E + p)])
        T += g[d] * F
    return T, g


def _solver(mesh, N, nodes, **kw):
    from paper_1910_02858_gb300 import Solver, SolverConfig
    from paper_1910_02858_gb300 import flexi as F

    return Solver(SolverConfig(N=N, Ngeo=mesh.Ngeo, node_type=nodes, riemann=F.RIEMANN_HLLC, mu=0.0, **kw), mesh.coords, mesh.conn)


def _rhs(mesh, N, nodes, W, b, split):
    import torch

    f = 2.0 ** b
    scale = np.array([1.0, f, f, f, f * f]).reshape(1, 5, 1, 1, 1)
    U = wl.prim_to_cons_np(*np.moveaxis(W, 1, 0), 1.4)
    s = _solver(mesh, N, nodes, split_form=split)
    Ut = s.rhs(torch.tensor(np.ascontiguousarray(U * scale), device="cuda:0"), 0.0).cpu().numpy()
    s.close()
    return Ut / (scale * f)


@pytest.mark.parametrize("mapping", ["box", "columns"])
@pytest.mark.parametrize("nodes,split", [(0, 0), (1, 0), (1, 1)], ids=["gauss", "lobatto", "kep"])
@pytest.mark.parametrize("N", [4, 5, 6, 7])
def test_thin_elements(N, nodes, split, mapping):
    mesh = _mesh(mapping, N)
    W = _state(mesh, N, nodes)
    T, _ = _bound(W, N, nodes)
    a, c = _rhs(mesh, N, nodes, W, 0, split), _rhs(mesh, N, nodes, W, 120, split)
    tol = 4 * 2 * 3 * (N + 3) * 2.0 ** -53 * T * (4 if split else 1)  # pairs: as in test_gpu_fixed_point.py
    for v in range(5):
        assert np.abs(a[:, v] - c[:, v]).max() <= tol[v], v


@pytest.mark.parametrize("mapping", ["box", "columns"])
@pytest.mark.parametrize("N", [4, 5, 6, 7])
def test_adjoint_of_thin_elements(N, mapping):
    """The reverse kernel: adjoints of the y momentum, constant in z (Gauss-Lobatto: no jumps there).  The x and y
    momentum receive from direction d at most g_d |dF_d,v / d(rho u, rho v)| |lam|, with F_z,v = rho w v.  The FP64
    body is reached by lam 2^220, in which every operation is linear."""
    import torch

    mesh = _mesh(mapping, N)
    W = _state(mesh, N, 1)
    _, g = _bound(W, N, 1)
    x = mesh.node_coords(N, 1)
    lam = np.zeros_like(W)
    lam[:, 2] = np.sin(x[:, 0] + 0.3) * np.cos(2 * x[:, 1])
    U = torch.tensor(wl.prim_to_cons_np(*np.moveaxis(W, 1, 0), 1.4), device="cuda:0")
    s = _solver(mesh, N, 1, adjoint=True)
    a, c = (s.rhs_adjoint(U, torch.tensor(lam * f, device="cuda:0"), 0.0).cpu().numpy() / f for f in (1.0, 2.0 ** 220))
    s.close()
    u, v, w = (np.abs(W[:, d]).max() for d in (1, 2, 3))
    T = {1: g[0] * v + g[1] * 0.4 * u, 2: g[0] * u + g[1] * 1.6 * v + g[2] * w}
    for k in T:
        assert np.abs(a[:, k] - c[:, k]).max() <= 4 * 2 * 3 * (N + 3) * 2.0 ** -53 * T[k], k
