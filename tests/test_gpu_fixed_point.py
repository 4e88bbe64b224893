"""Fixed-point line contractions of the FP64 form against the FP64 body of the same kernel
(which reads the metric terms per node, also where the fixed-point kernel takes the
constants of affine elements).

Scaling the units by powers of two (velocity by 2^b, pressure by 2^2b, viscosity by 2^b)
scales every FP64 operation of the right-hand side exactly, so U_t of the scaled state is
the scaled U_t.  At b = 120 the pressure leaves the fixed-point range and the element goes
through the FP64 body; unscaled it goes through the fixed-point contractions.

Tolerance, derived: both evaluations round each term of the sums of Eq. semiDiscrete.  A
line's n + 2 terms in each of 3 directions, through the lifting and the volume sweep, give
at most 2 * 3 (n + 2) roundings of 2^-53 relative to |terms|, bounded by
T_v = max|F_v| * rowsum(|Dhat| + |lhat|) * max|Ja| / min J per variable, with the same again
for the products and the pointwise fluxes.
"""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


def _rhs(mesh, N, nodes, U, b, poke=None, split=0):
    import torch

    from paper_1910_02858_gb300 import Solver, SolverConfig
    from paper_1910_02858_gb300 import flexi as F

    f = 2.0 ** b
    s = Solver(SolverConfig(N=N, Ngeo=mesh.Ngeo, node_type=nodes, riemann=F.RIEMANN_RUSANOV, mu=0.01 * f,
                            split_form=split), mesh.coords, mesh.conn)
    scale = np.array([1.0, f, f, f, f * f]).reshape(1, 5, 1, 1, 1)
    V = U * scale
    if poke is not None:
        V[poke[:-1]] = poke[-1]
    Ut = s.rhs(torch.tensor(V, device="cuda:0"), 0.0).cpu().numpy()
    s.close()
    return Ut / (scale * f)


def _mixed(N):
    """Parallelepipeds next to elements with displaced inner points (degree 2: the faces stay flat)."""
    mesh = wl.box_mesh((3, 2, 4), lo=(0.0,) * 3, hi=(2 * np.pi,) * 3, Ngeo=2, reorient_seed=N)
    mesh.coords[3::5, 1, 1, 1] += 0.05
    return mesh


def _case(N, nodes, mapping):
    from oracle.basis import Basis

    mesh = wl.box_mesh((3, 2, 4), lo=(0.0,) * 3, hi=(2 * np.pi,) * 3, Ngeo=N if mapping == "sine" else 1, mapping=mapping,
                       reorient_seed=N) if mapping != "mixed" else _mixed(N)
    U = wl.perturbed(mesh.node_coords(N, nodes), seed=N)
    b = Basis(N, nodes)
    D = b.Dhat.abs().sum(1) + b.lhat_minus.abs() + b.lhat_plus.abs()
    h = 2 * np.pi / np.array([3, 2, 4]) / 2
    ja = 1.4 * max(h[0] * h[1], h[1] * h[2], h[0] * h[2])
    J = 0.3 * h.prod()
    p = np.abs(U[:, 4]).max()
    F = np.array([1.0, 2.0 * p, 2.0 * p, 2.0 * p, 2.0 * p])  # largest flux of each variable, generously
    T = F * float(D.max()) * ja / J
    return mesh, U, 4 * 2 * 3 * (N + 3) * 2.0 ** -53 * T


@pytest.mark.parametrize("mapping", ["cartesian", "sine", "mixed"])
@pytest.mark.parametrize("nodes", [0, 1])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7])
def test_matches_fp64_body(N, nodes, mapping):
    if mapping != "cartesian" and N == 1:
        pytest.skip("straight at degree 1")
    mesh, U, tol = _case(N, nodes, mapping)
    a, c = _rhs(mesh, N, nodes, U, 0), _rhs(mesh, N, nodes, U, 120)
    for v in range(5):
        assert np.abs(a[:, v] - c[:, v]).max() <= tol[v], v


@pytest.mark.parametrize("mapping", ["cartesian", "sine", "mixed"])
@pytest.mark.parametrize("N", [2, 3, 4, 5, 6, 7])
def test_split_form_matches_fp64_body(N, mapping):
    """Kinetic-energy-preserving pairs: two line sums of n - 1 terms per direction in place of one of n + 2, each
    pair flux of four more roundings; at low speed too, where p outweighs the momentum flux."""
    mesh, U, tol = _case(N, 1, mapping)
    for slow in (1.0, 2.0 ** -12):
        V = U.copy()
        V[:, 1:4] *= slow
        V[:, 4] -= 0.5 * ((U[:, 1:4] ** 2).sum(1) * (1 - slow ** 2)) / U[:, 0]
        a, c = _rhs(mesh, N, 1, V, 0, split=1), _rhs(mesh, N, 1, V, 120, split=1)
        for v in range(5):
            assert np.abs(a[:, v] - c[:, v]).max() <= 4 * tol[v], (v, slow)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("N", [2, 5, 7])
def test_non_finite_values_spread_alike(N, bad):
    mesh, U, _ = _case(N, 0, "cartesian")
    poke = (5, 2, N, 1, 0, bad)
    a, c = _rhs(mesh, N, 0, U, 0, poke), _rhs(mesh, N, 0, U, 120, poke)
    assert not np.isfinite(a).all()
    assert np.array_equal(np.isfinite(a), np.isfinite(c))


def test_wide_ranges_within_an_element():
    """A field that falls by 2^40 across each element: the error stays that of FP64 relative to the largest terms."""
    mesh, U, tol = _case(7, 0, "cartesian")
    ramp = 2.0 ** (-40.0 * np.linspace(0.0, 1.0, 8)).reshape(1, 1, 1, 8)
    U[:, 1:4] *= ramp[:, None]
    a, c = _rhs(mesh, 7, 0, U, 0), _rhs(mesh, 7, 0, U, 120)
    for v in range(5):
        assert np.abs(a[:, v] - c[:, v]).max() <= tol[v], v


def _adjoint(mesh, N, nodes, U, lam, b, riemann, mu=0.01):
    import torch

    from paper_1910_02858_gb300 import Solver, SolverConfig

    f = 2.0 ** b
    s = Solver(SolverConfig(N=N, Ngeo=mesh.Ngeo, node_type=nodes, riemann=riemann, mu=mu * f, adjoint=True), mesh.coords,
               mesh.conn)
    scale = np.array([1.0, f, f, f, f * f]).reshape(1, 5, 1, 1, 1)
    t = lambda a: torch.tensor(a, device="cuda:0")
    # U_t' = f S L(U) for U' = S U, so the transpose maps S^-1 lam to f S^-1 (dL/dU)^T lam
    out = s.rhs_adjoint(t(U * scale), t(lam / scale), 0.0).cpu().numpy()
    s.close()
    return out * scale / f


@pytest.mark.parametrize("mapping", ["cartesian", "mixed"])
@pytest.mark.parametrize("N", [2, 4, 5, 6, 7])
def test_adjoint_matches_fp64_body(N, mapping):
    """The reverse kernel's fixed-point contractions against its FP64 body.  The transposed sums have the terms of
    the forward ones, at most 4 (N + 3) roundings deeper (the pointwise derivatives), on random unit-size adjoints:
    the same bound with max|F| replaced by the largest flux derivative, |u| + c times the largest column."""
    from paper_1910_02858_gb300 import flexi as F

    mesh, U, tol = _case(N, 0, mapping)
    lam = np.random.default_rng(N).standard_normal(U.shape)
    a, c = (_adjoint(mesh, N, 0, U, lam, b, F.RIEMANN_RUSANOV) for b in (0, 120))
    assert np.abs(a - c).max() <= 4 * tol.max() * np.abs(lam).max() * np.abs(U).max()


@pytest.mark.parametrize("riemann", ["hllc", "rusanov"])
@pytest.mark.parametrize("speed", [0.4, 3.0])
def test_flux_reverses_match_oracle(riemann, speed):
    """Hand-written HLLC and Rusanov reverses on subsonic and supersonic faces of both directions (1e-10, the bar of
    the adjoint against the oracle's reverse mode)."""
    import torch

    from oracle.dgsem import DGSEM, HLLC, RUSANOV, Params
    from paper_1910_02858_gb300 import flexi as F

    mesh = wl.box_mesh((2, 2, 2), reorient_seed=7)
    U = wl.perturbed(mesh.node_coords(3, 0), seed=11, Ma=1.0)
    rho = U[:, :1]
    m = U[:, 1:4] + speed * rho * np.array([1.0, -0.7, 0.5]).reshape(1, 3, 1, 1, 1)
    U = np.concatenate([rho, m, U[:, 4:] + 0.5 * (m ** 2 - U[:, 1:4] ** 2).sum(1, keepdims=True) / rho], axis=1)
    lam = np.random.default_rng(5).standard_normal(U.shape)
    out = _adjoint(mesh, 3, 0, U, lam, 0, F.RIEMANN_HLLC if riemann == "hllc" else F.RIEMANN_RUSANOV)
    dg = DGSEM(Params(N=3, node_type=0, riemann=HLLC if riemann == "hllc" else RUSANOV, mu=0.01), mesh.coords, mesh.conn)
    ref = dg.rhs_vjp(torch.tensor(U), 0.0, torch.tensor(lam)).numpy()
    assert np.linalg.norm(out - ref) <= 1e-10 * np.linalg.norm(ref)
