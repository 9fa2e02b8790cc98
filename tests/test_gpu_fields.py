"""The field maps (far field, its adjoint, near-zone field) against the
oracle's plain sums over the same quadrature points, in each range of the
phase series (k h below 6e-3, 0.13 and 0.52, h the longest edge; pie_problem_create
admits no larger one)
and at the counts where the split over chunks, warps and directions can go
wrong.  The maps are sums of about 7 T terms of one size with FP64 phases up
to a few radians: equal to 1e-12 of the result's norm (complex float
solutions: the input's rounding, 1e-6)."""
import numpy as np
import pytest

import pie_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kh", [1e-3, 0.1, 0.5])
@pytest.mark.parametrize("shape", ["octasphere", "patch"])
def test_field_maps_match_oracle(kh, shape):
    import torch
    from oracle.farfield import far_field
    from oracle.mesh import build_topology
    from oracle.nearzone import scattered_field
    from tests._lib import ensure_built
    ensure_built()
    import paper_1806_04164_gb300 as pg
    xyz, tri = pi.octasphere(2, axes=(1.0, 0.6, 0.5)) if shape == "octasphere" else pi.square_patch(9)
    h = max(np.linalg.norm(xyz[tri] - np.roll(xyz[tri], -1, 1), axis=2).ravel())
    k = kh / h
    top = build_topology(xyz, tri)
    rng = np.random.default_rng(5)
    for precision, tol in ((pg.PIE_MIXED, 1e-12), (pg.PIE_FP32, 1e-6)):
        pr = pg.Problem(pg.Mesh(xyz, tri), k, 3, root_side=6.01 * h, precision=precision)
        x = torch.from_numpy(pi.complex_normal(pr.N, 3)).cuda().to(pr.torch_dtype)
        xo = x.cpu().numpy().astype(np.complex128)
        for n in (1, 3, 33, 257):
            d = rng.normal(size=(n, 3))
            d /= np.linalg.norm(d, axis=1, keepdims=True)
            E = pr.farfield(x, d).cpu().numpy()
            Eo = far_field(top, k, xo, d)
            assert np.linalg.norm(E - Eo) <= tol * np.linalg.norm(Eo), (precision, n)
            if n > 33:
                continue
            g = pi.complex_normal(3 * n, n).reshape(n, 3)
            u = pr.farfield_adjoint(torch.from_numpy(g).cuda(), d).cpu().numpy()
            F = np.stack([far_field(top, k, e, d) for e in np.eye(pr.N)[:pr.E]])
            uo = np.concatenate([np.einsum("end,nd->e", F.conj(), g), np.zeros(pr.T)])
            assert np.linalg.norm(u - uo) <= tol * np.linalg.norm(uo), (precision, n)
        if precision == pg.PIE_FP32:
            continue
        rho = pi.complex_normal(pr.T, 6) * 8.8e-12
        for n in (1, 2, 65):
            p = rng.normal(size=(n, 3))
            p *= rng.uniform(1.5, 4.0, (n, 1)) / np.linalg.norm(p, axis=1, keepdims=True)
            E = pr.nearfield(x, torch.from_numpy(rho).cuda(), p).cpu().numpy()
            Eo = scattered_field(top, k, xo, rho, p)
            assert np.linalg.norm(E - Eo) <= tol * np.linalg.norm(Eo), n
