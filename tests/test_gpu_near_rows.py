"""One-column float near part where rows are long: rows the block stages, rows it
reads from global memory, and both in one launch, against the warp kernel bit
for bit.  Where all rows are within it, float moments stage up to 1344 sources
(2400 where one box has more than 1.5 times an SM's share of the pairs) and half
records up to 4480 (227 KB less the 16 KB ring, 48 bytes each); else
the rows of at most 448 where those hold half of the pairs."""
import numpy as np
import pytest

import pie_inputs as pi

pytestmark = pytest.mark.gpu


def _spot(base, spot, size):
    """A body and a small fine one inside it (two closed surfaces)."""
    (a, b), (c, d) = base, spot
    c = c * (size / np.abs(c).max()) + np.array([0.05, 0.04, 0.3])
    return np.concatenate([a, c]), np.concatenate([b, d + len(a)])


CASES = {  # mesh, levels, bounds of the longest row, bounds of the share of pairs in short rows
    "staged": (lambda: pi.icosphere(5), 4, (512, 1344), (0.0, 0.0)),
    "staged for the critical path": (lambda: pi.cylinder(nseg=64, nrings=10, nrows=55), 4, (1345, 2400), (0.0, 0.0)),
    "staged by half records, none in float": (lambda: _spot(pi.icosphere(5), pi.icosphere(4), 0.08), 6, (2401, 4480), (0.0, 0.4)),
    "staged by half records, short rows in float": (lambda: _spot(pi.icosphere(6), pi.cube(11), 0.03), 6, (2401, 4480), (0.5, 0.9)),
    "not staged": (lambda: pi.icosphere(5), 3, (4481, 9999), (0.0, 0.0)),
    "short rows only": (lambda: _spot(pi.icosphere(6), pi.cylinder(nseg=32, nrings=10, nrows=51), 0.03), 6, (4481, 9999), (0.5, 0.9)),
}


@pytest.mark.parametrize("case", list(CASES))
def test_long_rows_equal_the_warp_kernel(case):
    import torch
    from oracle.tree import build_tree
    from tests._lib import ensure_built
    ensure_built()
    import paper_1806_04164_gb300 as pg
    mk, levels, (lo, hi), (s0, s1) = CASES[case]
    xyz, tri = mk()
    tri = np.ascontiguousarray(tri, np.int32)
    tr = build_tree(xyz[tri].mean(1), xyz, levels, side=2.0)
    count = np.diff(tr.leaf_start)
    row = np.array([count[tr.near_idx[tr.near_ptr[b]:tr.near_ptr[b + 1]]].sum() for b in range(len(count))])
    pairs = row * count
    assert lo <= row.max() <= hi and s0 <= pairs[row <= 448].sum() / pairs.sum() <= s1
    for precision in (pg.PIE_MIXED, pg.PIE_FP32, pg.PIE_FP32H):
        pr = pg.Problem(pg.Mesh(xyz, tri), 0.01, levels, root_side=2.0, precision=precision, ntheta=4, tau=3, kappa_a=0.15)
        assert pr.near_pairs == pairs.sum()
        x = torch.from_numpy(pi.complex_normal(pr.N, 5)).cuda().to(pr.torch_dtype)
        y, n = pr.apply(x), pr.apply(x, near_only=True)
        pr.tuning = dict(near_kernel=1)
        assert torch.equal(pr.apply(x), y), precision
        assert torch.equal(pr.apply(x, near_only=True), n), precision
