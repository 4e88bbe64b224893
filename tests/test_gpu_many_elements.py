"""The element kernels of ordinary meshes (not those of the smallest, which have kernels of their own) where a CTA
holds several elements and the last one is not full, and meshes of parallelepipeds and bent elements large enough
that each kind has its own launch.

Fixed-point contractions against the FP64 body of the same kernels by scaling the units, with the tolerance of
test_gpu_fixed_point.py; the Runge-Kutta surface kernel against stages put together from right-hand sides.
"""
import numpy as np
import pytest

import workloads as wl

from test_gpu_fixed_point import _adjoint, _rhs

pytestmark = pytest.mark.gpu
SHAPE = {1: (11, 11, 11), 2: (8, 8, 8), 3: (6, 6, 5)}  # 8, 3 and 1 elements per CTA; 3 and 2 left over


def _case(N, nodes, mapping, shape):
    from oracle.basis import Basis

    mesh = wl.box_mesh(shape, lo=(0.0,) * 3, hi=(2 * np.pi,) * 3, Ngeo=N if mapping == "sine" else min(N, 2),
                       mapping="sine" if mapping == "sine" else "cartesian", reorient_seed=N)
    h = 2 * np.pi / np.array(shape) / 2
    if mapping == "mixed":  # the last elements bent: displaced inner points (degree 2: the faces stay flat)
        k = len(mesh.coords) // 6
        mesh.coords[-k::2, 1, 1, 1] += 0.1 * h.min()
    U = wl.perturbed(mesh.node_coords(N, nodes), seed=N)
    b = Basis(N, nodes)
    D = float((b.Dhat.abs().sum(1) + b.lhat_minus.abs() + b.lhat_plus.abs()).max())
    p = np.abs(U[:, 4]).max()
    # largest flux of each variable and metric ratio as in test_gpu_fixed_point.py
    T = np.array([1.0, 2.0 * p, 2.0 * p, 2.0 * p, 2.0 * p]) * D * 1.4 / (0.3 * h.min())
    return mesh, U, 4 * 2 * 3 * (N + 3) * 2.0 ** -53 * T


@pytest.mark.parametrize("mapping", ["cartesian", "mixed", "sine"])
@pytest.mark.parametrize("nodes,split", [(0, 0), (1, 0), (1, 1)], ids=["gauss", "lobatto", "kep"])
@pytest.mark.parametrize("N", [1, 2, 3])
def test_several_elements_per_cta(N, nodes, split, mapping):
    if N == 1 and mapping == "mixed":
        pytest.skip("straight at degree 1")
    mesh, U, tol = _case(N, nodes, mapping, SHAPE[N])
    a, c = _rhs(mesh, N, nodes, U, 0, split=split), _rhs(mesh, N, nodes, U, 120, split=split)
    for v in range(5):
        assert np.abs(a[:, v] - c[:, v]).max() <= (4 if split else 1) * tol[v], v


@pytest.mark.parametrize("N,shape", [(2, (29, 29, 29)), (3, (22, 22, 22)), (4, (18, 18, 17)), (7, (11, 11, 13))])
def test_mixed_meshes_in_two_launches(N, shape):
    mesh, U, tol = _case(N, 0, "mixed", shape)
    a, c = _rhs(mesh, N, 0, U, 0), _rhs(mesh, N, 0, U, 120)
    for v in range(5):
        assert np.abs(a[:, v] - c[:, v]).max() <= tol[v], v


@pytest.mark.parametrize("N,shape", [(3, (22, 22, 22)), (4, (18, 18, 17)), (7, (11, 11, 13))])
@pytest.mark.parametrize("precision", ["FP32", "FP32_TF32", "FP32_BF16"])
def test_mixed_meshes_fp32(N, shape, precision):
    """Against the FP64 form: the bar is the FP64 tolerance with 2^-24 for 2^-53."""
    import torch

    from paper_1910_02858_gb300 import Solver, SolverConfig
    from paper_1910_02858_gb300 import flexi as F

    mesh, U, tol = _case(N, 0, "mixed", shape)
    out = []
    for p in (F.FP64, getattr(F, precision)):
        s = Solver(SolverConfig(N=N, Ngeo=mesh.Ngeo, riemann=F.RIEMANN_RUSANOV, mu=0.01, precision=p), mesh.coords, mesh.conn)
        out.append(s.rhs(torch.tensor(U, device="cuda:0", dtype=s.dtype), 0.0).double().cpu().numpy())
        s.close()
    for v in range(5):
        assert np.abs(out[0][:, v] - out[1][:, v]).max() <= tol[v] * 2.0 ** 29, v


@pytest.mark.parametrize("mapping", ["cartesian", "sine"])
@pytest.mark.parametrize("N", [1, 2, 3])
def test_adjoint_of_several_elements_per_cta(N, mapping):
    """lam 2^220 takes the reverse kernel's FP64 body, in which every operation is linear.  Bound: as in
    test_gpu_fixed_point.py, the forward one with the largest flux derivative for the largest flux."""
    from paper_1910_02858_gb300 import flexi as F

    mesh, U, tol = _case(N, 0, mapping, SHAPE[N])
    lam = np.random.default_rng(N).standard_normal(U.shape)
    a, c = (_adjoint(mesh, N, 0, U, lam * f, 0, F.RIEMANN_RUSANOV) / f for f in (1.0, 2.0 ** 220))
    assert np.abs(a - c).max() <= 4 * tol.max() * np.abs(lam).max() * np.abs(U).max()


@pytest.mark.parametrize("nodes", [0, 1])
@pytest.mark.parametrize("N", [1, 2, 3])
def test_step_is_its_stages(N, nodes):
    """dU = A dU + dt U_t, U = U + B dU, five times: the stage kernel forms the same sums with fused multiply-adds and
    hands on the face states; each stage differs by at most four roundings of 2^-53 of |U| and of |dU|, carried on
    through dt |dU_t / dU| < 1."""
    import torch

    from oracle.dgsem import RK_A, RK_B, RK_C
    from paper_1910_02858_gb300 import Solver, SolverConfig
    from paper_1910_02858_gb300 import flexi as F

    mesh, U0, tol = _case(N, nodes, "sine", SHAPE[N])
    s = Solver(SolverConfig(N=N, Ngeo=mesh.Ngeo, node_type=nodes, riemann=F.RIEMANN_HLLC, mu=0.01), mesh.coords, mesh.conn)
    U = torch.tensor(U0, device="cuda:0")
    dt = 0.5 * s.reduce(U)["dt_max"]
    V, dV, dU = U.clone(), torch.zeros_like(U), torch.zeros_like(U)
    s.step(V, dV, 0.0, dt)
    for k in range(5):
        dU = RK_A[k] * dU + dt * s.rhs(U, RK_C[k] * dt)
        U = U + RK_B[k] * dU
    s.close()
    scale = U.abs().amax(dim=(0, 2, 3, 4))
    bound = 5 * (4 * 2.0 ** -53 * 2 * scale.cpu().numpy() + dt * tol)
    assert ((V - U).abs().amax(dim=(0, 2, 3, 4)).cpu().numpy() <= bound).all()


@pytest.mark.parametrize("mapping", ["cartesian", "sine"])
@pytest.mark.parametrize("N", [2, 3, 4, 5, 6, 7])
def test_surface_kernel_matches_its_fp64_branch(N, mapping):
    """The surface kernel takes its FP64 expressions from 2^900 on, which finite data reach with a gas at rest (no
    product of two such values): dm/dt = -grad p scales with p exactly.  Gauss-Lobatto nodes: no jumps, so no
    dissipation.  Bound: that of the volume sums, twice, for the surface's products under the same row sums."""
    import torch

    from paper_1910_02858_gb300 import Solver, SolverConfig
    from paper_1910_02858_gb300 import flexi as F

    mesh, _, tol = _case(N, 1, mapping, SHAPE.get(N, (6, 6, 5)))
    x = mesh.node_coords(N, 1)
    U = np.zeros((x.shape[0], 5) + x.shape[2:])
    U[:, 0] = 1.0
    U[:, 4] = (1.0 + 0.1 * np.sin(x[:, 0]) * np.cos(x[:, 1] + x[:, 2])) / 0.4
    out = []
    for f in (1.0, 2.0 ** 910):
        s = Solver(SolverConfig(N=N, Ngeo=mesh.Ngeo, node_type=1, riemann=F.RIEMANN_RUSANOV, mu=0.0), mesh.coords, mesh.conn)
        V = U.copy()
        V[:, 4] *= f
        out.append(s.rhs(torch.tensor(V, device="cuda:0"), 0.0).cpu().numpy() / f)
        s.close()
    for v in (1, 2, 3):
        assert np.abs(out[0][:, v]).max() > 1e-3
        assert np.abs(out[0][:, v] - out[1][:, v]).max() <= 2 * tol[v], v
