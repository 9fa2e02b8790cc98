"""Near pair moments against the oracle's (FP64 sums of 49 or 2 x 64 x 7
terms: 1e-12 of each plane's largest), in every range of the series that the
set-up chooses by wavenumber (4.4 k0 leaf below 0.028, 0.59 and above; 2.9 k0 h
below 0.04 and above), on a closed and an open surface, with the tree and
lists bit for bit."""
import numpy as np
import pytest

import pie_inputs as pi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,L", [("ellipsoid", 3), ("patch", 4), ("cube", 3)])
@pytest.mark.parametrize("ka", [1e-3, 0.05, 0.7])
def test_pair_moments_match_oracle(shape, L, ka):
    from oracle.mlfma import MLFMA
    from tests._lib import ensure_built
    ensure_built()
    import paper_1806_04164_gb300 as pg
    xyz, tri = {"ellipsoid": lambda: pi.octasphere(2, axes=(1.0, 0.5, 0.5)), "patch": lambda: pi.square_patch(8),
                "cube": lambda: pi.cube(3)}[shape]()
    h = max(np.linalg.norm(xyz[tri] - np.roll(xyz[tri], -1, 1), axis=2).ravel())
    side = max(1.51 * h * 2 ** (L - 1), (xyz.max(0) - xyz.min(0)).max())
    k = ka / (side / 4)
    M = MLFMA(xyz, tri, k, L, side=side)
    pr = pg.Problem(pg.Mesh(xyz, tri), k, L, root_side=side)
    for l in range(3, L + 1):
        keys, ptr, idx, off = pr.level(l)
        assert np.array_equal(keys, M.tree.keys[l]) and np.array_equal(ptr, M.tree.il_ptr[l])
        assert np.array_equal(idx, M.tree.il_idx[l]) and np.array_equal(off, M.tree.il_off[l])
    ptr, idx = pr.near()
    assert np.array_equal(ptr, M.tree.near_ptr) and np.array_equal(idx, M.tree.near_idx)
    m0, mt, ms, mts = M.near_m
    om = [m0, mt[:, 0], mt[:, 1], mt[:, 2], ms[:, 0], ms[:, 1], ms[:, 2], mts]
    mom = pr.stage(4)
    for q in range(8):
        assert np.max(np.abs(mom[q] - om[q])) <= 1e-12 * np.max(np.abs(om[q])), q
