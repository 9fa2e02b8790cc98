"""The fixed-point near part of PIE_FP64 problems against the oracle's near
product: rows shorter and longer than a stage of 384 sources, several columns,
coefficients of very different sizes in different places (each leaf box has
its own scale), and inputs that are not finite."""
import numpy as np
import pytest

import pie_inputs as pi

pytestmark = pytest.mark.gpu


def _case(shape):
    from oracle.mlfma import MLFMA
    from tests._lib import ensure_built
    ensure_built()
    import paper_1806_04164_gb300 as pg
    if shape == "patch":      # about 200 sources a row
        xyz, tri, L, side = *pi.square_patch(20), 4, 0.6
    else:                     # rows of 600 to 1152 sources: two and three stages
        xyz, tri, L, side = *pi.cube(6), 3, 1.2
    k = 0.3
    M = MLFMA(xyz, tri, k, L, side=side)
    return M, pg.Problem(pg.Mesh(xyz, tri), k, L, root_side=side, max_nrhs=3)


@pytest.mark.parametrize("shape", ["patch", "cube"])
def test_near_fixed_matches_oracle(shape):
    """The sums are exact and each factor is rounded to 2^-54 of the largest
    of its row or leaf box, or better; the oracle's FP64 sums of up to 1152 terms are
    within 1e-13 of the exact ones."""
    import torch
    M, pr = _case(shape)
    rng = np.random.default_rng(2)
    x = np.stack([pi.complex_normal(pr.N, s) for s in (1, 2, 3)])
    x[1] *= 1e-200                                    # one scale for the whole column
    x[2, : pr.E] *= 10.0 ** rng.uniform(-3, 3, pr.E)  # scales mixed within a box
    y = pr.apply(torch.from_numpy(x).cuda(), near_only=True).cpu().numpy()
    for c in range(3):
        yo = M.apply(x[c], far=False)
        for part in (slice(0, pr.E), slice(pr.E, None)):
            assert np.linalg.norm(y[c][part] - yo[part]) <= 1e-13 * np.linalg.norm(yo[part]), (c, part)


def test_near_fixed_is_local():
    """Pulses 1e-30 in one half of the patch, 1 in the other: rows whose
    sources all lie in the small half keep their relative accuracy."""
    import torch
    M, pr = _case("patch")
    x = pi.complex_normal(pr.N, 5)
    x[: pr.E] = 0
    small = M.geo.cent[:, 0] < 0
    x[pr.E:][small] *= 1e-30
    y = pr.apply(torch.from_numpy(x).cuda(), near_only=True).cpu().numpy()[pr.E:]
    yo = M.apply(x, far=False)[pr.E:]
    rows = np.abs(yo) < 1e-20 * np.abs(yo).max()
    assert rows.sum() > 50
    assert np.linalg.norm(y[rows] - yo[rows]) <= 1e-13 * np.linalg.norm(yo[rows])


@pytest.mark.parametrize("bad", [np.nan, np.inf, complex(1e308, 0)])
@pytest.mark.parametrize("shape", ["patch", "cube"])
def test_near_fixed_keeps_non_finite_inputs(shape, bad):
    """A pulse that is not finite, or whose w^2 eps0 sigma overflows, reaches
    exactly the rows it is near to, as in floating point."""
    import torch
    M, pr = _case(shape)
    x = pi.complex_normal(pr.N, 7)
    x[pr.E + 11] = bad
    y = pr.apply(torch.from_numpy(x).cuda(), near_only=True).cpu().numpy()[pr.E:]
    near = np.zeros(pr.T, bool)
    inv = np.argsort(M.tree.perm)
    near[M.tree.perm[M.near_t[M.near_s == inv[11]]]] = True
    assert near.sum() < pr.T and near[11]
    x[pr.E + 11] = 0
    rest = pr.apply(torch.from_numpy(x).cuda(), near_only=True).cpu().numpy()[pr.E:]
    assert not np.any(np.isfinite(y[near]))
    assert np.array_equal(y[~near], rest[~near])
