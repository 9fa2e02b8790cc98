"""Phases of the field maps at the limits of their series: bodies whose
farthest centroid (and point) lies just inside the range of the short series for
the centroid's phase, directions that are not unit vectors (the maps are defined
for any vector), and the order of the sums, which belongs to the body and not to
the other directions or points of the call."""
import numpy as np
import pytest

import pie_inputs as pi

pytestmark = pytest.mark.gpu


def _problem(k, offset=0.0, n=8, side=0.05, precision="PIE_MIXED"):
    from oracle.mesh import build_topology
    from tests._lib import ensure_built
    ensure_built()
    import paper_1806_04164_gb300 as pg
    xyz, tri = pi.square_patch(n, side)
    h = side / n * 2 ** 0.5
    u = np.array([0.48, -0.6, 0.64])
    xyz = xyz + offset * u
    return build_topology(xyz, tri), pg.Problem(pg.Mesh(xyz, tri), k, 3, root_side=max(1.01 * side, 6.01 * h),
                                                precision=getattr(pg, precision)), u


@pytest.mark.parametrize("kr", [0.0899, 0.15, 0.1999, 0.21])
def test_phase_series_at_its_limit(kr):
    """Every triangle's phase is kr to a few per cent, the largest kr itself, so
    that a series cut short shows in full.  Rounding: the phase to an ulp or two of
    0.2, sine and cosine to an ulp each, a dozen multiply-adds a term: below 5e-15
    of the norm."""
    import torch
    from oracle.farfield import far_field
    from oracle.nearzone import scattered_field
    top, _, u = _problem(0.1, offset=1.0)
    far = np.linalg.norm(top.centroid, axis=1).max()
    k = kr / far
    top, pr, u = _problem(k, offset=1.0)
    x = pi.complex_normal(pr.N, 3)
    d = np.stack([u, -u])
    xd = torch.from_numpy(x).cuda()
    E, Eo = pr.farfield(xd, d).cpu().numpy(), far_field(top, k, x, d)
    for i in range(2):
        assert np.linalg.norm(E[i] - Eo[i]) <= 5e-15 * np.linalg.norm(Eo[i])
    g = np.cross(u, pi.complex_normal(3, 4))[None]
    v = pr.farfield_adjoint(torch.from_numpy(g).cuda(), d[:1]).cpu().numpy()
    F = np.stack([far_field(top, k, e, d[:1])[0] for e in np.eye(pr.N)[:pr.E]])
    vo = np.concatenate([F.conj() @ g[0], np.zeros(pr.T)])
    assert np.linalg.norm(v - vo) <= 5e-15 * np.linalg.norm(vo)
    # centroids 1 m to one side, a point 1 m to the other: the distance is the sum
    k = kr / (far + 1.0)
    top, pr, u = _problem(k, offset=1.0)
    rho = pi.complex_normal(pr.T, 6) * 8.8e-12
    p = -u[None]
    E = pr.nearfield(xd, torch.from_numpy(rho).cuda(), p).cpu().numpy()
    Eo = scattered_field(top, k, x, rho, p)
    assert np.linalg.norm(E - Eo) <= 5e-15 * np.linalg.norm(Eo)


@pytest.mark.parametrize("length", [1e-3, 1.5, 4.0, 40.0, 1e4])
@pytest.mark.parametrize("kh", [1e-3, 0.1, 0.5])
def test_directions_of_any_length(length, kh):
    """F(rhat) for |rhat| != 1: the phases are k rhat . r whatever its length
    (rounding: 1e-16 of the largest phase, and 1e-12 as for unit vectors)."""
    import torch
    from oracle.farfield import far_field
    h = 0.05 / 8 * 2 ** 0.5
    k = kh / h
    top, pr, _ = _problem(k, offset=0.02)
    tol = 1e-12 + 4e-16 * k * length * 0.08
    x = pi.complex_normal(pr.N, 3)
    rng = np.random.default_rng(1)
    d = rng.normal(size=(5, 3))
    d *= length / np.linalg.norm(d, axis=1, keepdims=True)
    d[3] /= 7
    E, Eo = pr.farfield(torch.from_numpy(x).cuda(), d).cpu().numpy(), far_field(top, k, x, d)
    assert np.linalg.norm(E - Eo) <= tol * np.linalg.norm(Eo)
    g = pi.complex_normal(15, 4).reshape(5, 3)
    v = pr.farfield_adjoint(torch.from_numpy(g).cuda(), d).cpu().numpy()
    F = np.stack([far_field(top, k, e, d) for e in np.eye(pr.N)[:pr.E]])
    vo = np.concatenate([np.einsum("end,nd->e", F.conj(), g), np.zeros(pr.T)])
    assert np.linalg.norm(v - vo) <= tol * np.linalg.norm(vo)


@pytest.mark.parametrize("n,most", [(4, 90001), (25, 3000), (60, 700)])
def test_a_field_does_not_depend_on_its_neighbours(n, most):
    """One direction or point gives the same bits alone and among many (more of
    them than one launch's scratch holds in the first case)."""
    import torch
    _, pr, _ = _problem(0.3, offset=0.1, n=n)
    rng = np.random.default_rng(2)
    x = torch.from_numpy(pi.complex_normal(pr.N, 3)).cuda()
    rho = torch.from_numpy(pi.complex_normal(pr.T, 6)).cuda()
    d = rng.normal(size=(most, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    E, H = pr.farfield(x, d), pr.nearfield(x, rho, d)
    for i, j in ((0, 1), (1, 182), (most - 1, most), (most // 2, most // 2 + 33)):
        assert torch.equal(pr.farfield(x, d[i:j]), E[i:j]), (i, j)
        assert torch.equal(pr.nearfield(x, rho, d[i:j]), H[i:j]), (i, j)
