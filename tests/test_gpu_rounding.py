"""Rounding noise of the FP64 form's fixed-point contractions against that of FP64 sums.

Velocity scaled by f, pressure by f^2 and viscosity by f scale every term of the right-hand side,
so U_t of the scaled state, scaled back, is U_t up to rounding.  The state is rounded to 40 bits:
f = 1.5 and f = 2^b scale it without error, and the difference of two evaluations whose factors
are not a power of two apart is sqrt(2) times the rounding noise of one.  At f = 1 and 1.5 the
elements go through the fixed-point contractions, at 2^120 and 1.5 * 2^120 through the FP64 body of
the same kernels.  Nodes inside the elements of Gauss-Lobatto meshes receive no face terms, so the
two differ in these sums only.

Bar: the fixed-point sums are as accurate as the FP64 ones, rms by rms; 1.25 covers the spread of
the pseudo-random roundings (8,000 values and more) and of the last conversion to FP64 on either side.
"""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu
SHAPE = (6, 6, 5)  # more elements than SMs: none of the small-mesh kernels


def _rhs(mesh, N, U, f, split):
    import torch

    from paper_1910_02858_gb300 import Solver, SolverConfig
    from paper_1910_02858_gb300 import flexi as F

    s = Solver(SolverConfig(N=N, Ngeo=mesh.Ngeo, node_type=F.NODES_LOBATTO, riemann=F.RIEMANN_HLLC, mu=f / 128.0,
                            split_form=split), mesh.coords, mesh.conn)
    scale = np.array([1.0, f, f, f, f * f]).reshape(1, 5, 1, 1, 1)
    Ut = s.rhs(torch.tensor(U * scale, device="cuda:0"), 0.0).cpu().numpy()
    s.close()
    return Ut[..., 1:-1, 1:-1, 1:-1] / (scale * f)


def _noise(N, mapping, split):
    mesh = wl.box_mesh(SHAPE, lo=(0.0,) * 3, hi=(2 * np.pi,) * 3, Ngeo=N if mapping == "sine" else 1, mapping=mapping)
    U = np.round(wl.perturbed(mesh.node_coords(N, 1), seed=N) * 2.0 ** 40) / 2.0 ** 40
    a, a2, b, b2 = (_rhs(mesh, N, U, f, split) for f in (1.0, 1.5, 2.0 ** 120, 1.5 * 2.0 ** 120))
    rms = lambda x: np.sqrt((x ** 2).mean(axis=(0, 2, 3, 4)))
    return rms(a - a2), rms(b - b2)


@pytest.mark.parametrize("mapping", ["cartesian", "sine"])
@pytest.mark.parametrize("N", [3, 4, 5, 6, 7])
def test_split_form(N, mapping):
    fixed, fp64 = _noise(N, mapping, 1)
    assert (fixed <= 1.25 * fp64).all(), fixed / fp64


@pytest.mark.parametrize("mapping", ["cartesian", "sine"])
@pytest.mark.parametrize("N", [3, 4, 5, 6, 7])
def test_standard_form(N, mapping):
    fixed, fp64 = _noise(N, mapping, 0)
    assert (fixed <= 1.25 * fp64).all(), fixed / fp64
