"""Block sizes of the per-box far kernels at their limits: angular grids whose
one row of samples fills a block (16, 20 and 22 theta rows) and far_rows
settings whose rows would not fit a block's registers.  Every form keeps the order of
every sum, so the results are the same to the last bit; the wide grids also
stand against the oracle (rounding its tables to float alone moves the far
part by up to 1.2e-5 of its norm; eight times that for the rounded sums)."""
import numpy as np
import pytest

import pie_inputs as pi

pytestmark = pytest.mark.gpu

K, L = 0.01, 4


@pytest.fixture(scope="module")
def pg():
    from tests._lib import ensure_built
    ensure_built()
    import paper_1806_04164_gb300 as pg
    return pg


@pytest.mark.parametrize("ntheta", [16, 20, 22])
@pytest.mark.parametrize("precision", ["PIE_FP32", "PIE_FP32H"])
def test_wide_grids_in_float(pg, precision, ntheta):
    import torch
    from oracle.mlfma import MLFMA
    xyz, tri = pi.icosphere(2)
    pr = pg.Problem(pg.Mesh(xyz, tri), K, L, root_side=4.0, precision=getattr(pg, precision), tau=3,
                    kappa_a=0.15, ntheta=ntheta, max_nrhs=2)
    x = torch.from_numpy(np.stack([pi.complex_normal(pr.N, s) for s in (1, 2)])).cuda().to(torch.complex64)
    y = pr.apply(x)
    M = MLFMA(xyz, tri, K, L, tau=3, x=0.15, ntheta=ntheta, side=4.0)
    xo = x[0].cpu().numpy().astype(np.complex128)
    far, faro = pr.apply_levels(x[0].contiguous(), range(3, L + 1), near=False).cpu().numpy(), M.apply(xo, near=False)
    for part in (slice(0, pr.E), slice(pr.E, None)):
        assert np.linalg.norm(far[part] - faro[part]) <= 1e-4 * np.linalg.norm(faro[part])
    best, _ = pr.autotune(nrhs=2, reps=1)  # tries far_rows 1 .. 16
    assert best == pr.tuning
    assert torch.equal(pr.apply(x), y)


@pytest.mark.parametrize("precision,ntheta,cols,levels", [
    ("PIE_FP32", 4, 130, 4), ("PIE_FP32", 6, 130, 4), ("PIE_FP32H", 10, 40, 4), ("PIE_FP32", 14, 20, 4),
    ("PIE_FP64", 6, 130, 4), ("PIE_MIXED", 10, 40, 4), ("PIE_MIXED", 20, 12, 3)])
def test_far_rows_beyond_what_a_block_holds(pg, precision, ntheta, cols, levels):
    """Enough columns that every level leaves the forms for few boxes."""
    import torch
    pr = pg.Problem(pg.Mesh(*pi.icosphere(3)), K, levels, root_side=2.0, precision=getattr(pg, precision), tau=3,
                    kappa_a=0.15, ntheta=ntheta, max_nrhs=cols)
    gen = torch.Generator(device="cuda").manual_seed(4)
    x = torch.randn((cols, pr.N), generator=gen, device="cuda", dtype=torch.complex128).to(pr.torch_dtype)
    tuning = pr.tuning
    pr.tuning = dict(tuning, far_rows=1)
    y = pr.apply(x)
    for rows in (2, 4, 8, 16, 32):
        pr.tuning = dict(tuning, far_rows=rows)
        assert torch.equal(pr.apply(x), y), rows
    pr.tuning = tuning
    pr.autotune(nrhs=cols, reps=1)
    assert torch.equal(pr.apply(x), y)
