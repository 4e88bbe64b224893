"""Which elements count as parallelepipeds: those whose coordinates are affine to within their own
rounding, coordinate by coordinate."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bent", [1, 2])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("N", [4, 7])
def test_far_offset_in_one_direction(N, precision, bent):
    """Elements bent by 10^-9 in y or z, with x near 0 and x near 2^20.  The metric terms are formed from coordinates
    relative to the element's first node, and x is a multiple of 2^-30, so that the offset changes none of them: U_t
    is equal to the bit."""
    import torch

    from paper_1910_02858_gb300 import Solver, SolverConfig
    from paper_1910_02858_gb300 import flexi as F

    mesh = wl.box_mesh((3, 2, 4), lo=(0.0,) * 3, hi=(6.0, 4.0, 8.0), Ngeo=2, reorient_seed=N)
    x = mesh.coords.copy()
    x[..., 0] = np.round(x[..., 0] * 2.0 ** 30) / 2.0 ** 30
    x[:, 1, 1, 1, bent] += 1e-9
    U = wl.perturbed(mesh.node_coords(N, 0), seed=N)
    out = []
    for offset in (0.0, 2.0 ** 20):
        y = x.copy()
        y[..., 0] += offset
        s = Solver(SolverConfig(N=N, Ngeo=2, mu=0.01, precision=F.FP64 if precision == "fp64" else F.FP32), y, mesh.conn)
        out.append(s.rhs(torch.tensor(U, device="cuda:0", dtype=s.dtype), 0.0).cpu())
        s.close()
    assert torch.equal(out[0], out[1])


def test_parallelepipeds_far_away_still_count():
    """Boxes at x near 2^20, whose x is rounded there, keep the constant metric terms: a free stream stays exact in
    the other two directions' terms, to the rounding of x over the element's width."""
    import torch

    from paper_1910_02858_gb300 import Solver, SolverConfig

    mesh = wl.box_mesh((6, 5, 6), lo=(2.0 ** 20, 0.0, 0.0), hi=(2.0 ** 20 + 6.0, 5.0, 6.0), Ngeo=1)
    s = Solver(SolverConfig(N=7, mu=0.01), mesh.coords, mesh.conn)
    U = torch.tensor(wl.freestream(mesh.node_coords(7, 0)), device="cuda:0")
    Ut = s.rhs(U, 0.0)
    s.close()
    # sums of n + 2 terms up to rowsum(|Dhat| + |lhat|) 2 / h = 60 times the flux (3 at most), each rounded to 2^-53
    assert Ut.abs().max().item() <= 3 * 10 * 2.0 ** -53 * 3 * 60


@pytest.mark.parametrize("N", [1, 4])
def test_algorithmic_bytes_count_what_affine_elements_read(N):
    """46 + 117 (3 / n) words per DOF and stage; affine elements read ten metric words per element, not per node."""
    from paper_1910_02858_gb300 import Solver, SolverConfig
    from paper_1910_02858_gb300 import flexi as F

    n, shape = N + 1, (11, 12, 10)
    words = {}
    for mapping in ("cartesian", "bent"):
        mesh = wl.box_mesh(shape, lo=(0.0,) * 3, hi=(6.0, 6.0, 6.0), Ngeo=1)
        if mapping == "bent":
            mesh.coords[:, 0, 0, 0] += 1e-3  # no element keeps its parallel edges
        s = Solver(SolverConfig(N=N, mu=0.01), mesh.coords, mesh.conn)
        words[mapping] = s.query(F.Q_BYTES_PER_STAGE) / 8
        s.close()
    K = np.prod(shape)
    assert words["cartesian"] == (46 + 351 / n) * K * n ** 3 - 10 * K * (n ** 3 - 1)
    assert words["bent"] == (46 + 351 / n) * K * n ** 3
