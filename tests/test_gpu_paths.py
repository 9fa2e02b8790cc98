"""The launch shapes of the product's kernels against one another.  A pass of
one column on a small tree takes the forms for few boxes (sums and components
over more threads, one warp per filter block, blocks sharing a leaf box), a
pass of 130 columns the forms for full grids (whole sums per thread, four
columns per near block), and two or three columns the near part's other
groupings; every form keeps the order of every sum, so the columns are the
same to the last bit.  Sizes leave remainders everywhere: rows that are no
multiple of 32 or 128, units that do not fill a warp, 130 = 32 x 4 + 2
columns, angular grids of 32, 72 and 128 samples."""
import pytest

import pie_inputs as pi

pytestmark = pytest.mark.gpu

POINTS = {4: (3, 0.15, 4), 6: (4, 0.1, 6), 8: (7, 0.08, 8)}


@pytest.mark.parametrize("ntheta", [4, 6, 8])
@pytest.mark.parametrize("precision", ["PIE_FP64", "PIE_FP32", "PIE_MIXED", "PIE_FP32H"])
def test_columns_do_not_depend_on_the_launch_shape(precision, ntheta):
    import torch
    from tests._lib import ensure_built
    ensure_built()
    import paper_1806_04164_gb300 as pg
    tau, kappa_a, nt = POINTS[ntheta]
    for mesh, L, side in ((pi.icosphere(3), 4, 2.0), (pi.square_patch(26), 4, 0.0)):
        m = pg.Mesh(*mesh)
        wide = pg.Problem(m, 0.01, L, root_side=side, precision=getattr(pg, precision), tau=tau, kappa_a=kappa_a,
                          ntheta=nt, max_nrhs=130)
        gen = torch.Generator(device="cuda").manual_seed(3)
        x = torch.randn((130, wide.N), generator=gen, device="cuda", dtype=torch.complex128).to(wide.torch_dtype)
        y = wide.apply(x)
        for cols in (1, 2, 3):
            for j in (0, 65, 130 - cols):
                z = wide.apply(x[j:j + cols].contiguous())
                assert torch.equal(z, y[j:j + cols]), (cols, j)
        # the near part alone: one column by the box-staged kernel in the near product
        n = wide.apply(x[129].contiguous(), near_only=True)
        wide.tuning = dict(near_kernel=1)
        assert torch.equal(wide.apply(x[129].contiguous()), y[129])
        assert torch.equal(wide.apply(x[129].contiguous(), near_only=True), n)
