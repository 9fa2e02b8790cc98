"""The radiated part of the near product in complex double.  At low frequency
the imaginary parts of the pair moments are k h / 4 of the real ones and less;
for real x they alone make Im(Z_near x), which is held to its own norm: 1e-13,
as the whole product (the oracle's FP64 sums of up to 1152 terms)."""
import numpy as np
import pytest

import pie_inputs as pi

pytestmark = pytest.mark.gpu

CASES = {"patch": lambda: (*pi.square_patch(20), 4, 0.6), "cube": lambda: (*pi.cube(6), 3, 1.2)}


@pytest.mark.parametrize("k", [1e-2, 1e-5, 1e-8])
@pytest.mark.parametrize("shape", ["patch", "cube"])
def test_parts_of_the_near_product_keep_their_own_accuracy(shape, k):
    import torch
    from oracle.mlfma import MLFMA
    from tests._lib import ensure_built
    ensure_built()
    import paper_1806_04164_gb300 as pg
    xyz, tri, L, side = CASES[shape]()
    M = MLFMA(xyz, tri, k, L, side=side)
    pr = pg.Problem(pg.Mesh(xyz, tri), k, L, root_side=side)
    m0, om0 = pr.stage(4)[0], M.near_m[0]
    assert np.abs(m0.imag - om0.imag).max() <= 1e-13 * np.abs(om0.imag).max()
    x = pi.complex_normal(pr.N, 1)
    # real, imaginary, and parts of very different sizes
    for z in (x.real + 0j, 1j * x.real, x.real + 1e-9j * x.imag, 1e-9 * x.real + 1j * x.imag):
        z = z.astype(np.complex128)
        y = pr.apply(torch.from_numpy(z).cuda(), near_only=True).cpu().numpy()
        yo = M.apply(z, far=False)
        for part in (slice(0, pr.E), slice(pr.E, None)):
            for f in (np.real, np.imag):
                a, b = f(y[part]), f(yo[part])
                assert np.linalg.norm(a - b) <= 1e-13 * np.linalg.norm(b), (part, f)


@pytest.mark.parametrize("mesh,levels,side", [("sphere", 4, 2.0), ("cube", 3, 1.2)])
def test_both_kernels_give_the_same_bits(mesh, levels, side):
    """Beside a far part of its own length the near part runs in two passes over a
    row, alone (overlap off) and beside a short far part in one: exact sums, so the
    order and the pass make no difference."""
    import torch
    from tests._lib import ensure_built
    ensure_built()
    import paper_1806_04164_gb300 as pg
    pr = pg.Problem(pg.Mesh(*(pi.icosphere(3) if mesh == "sphere" else pi.cube(6))), 1e-3, levels, root_side=side,
                    max_nrhs=3)
    x = torch.from_numpy(np.stack([pi.complex_normal(pr.N, s) for s in (1, 2, 3)])).cuda()
    y = pr.apply(x)
    pr.tuning = dict(overlap=0)
    assert torch.equal(pr.apply(x), y)
    pr.tuning = dict(overlap=1, near_ctas_per_sm=0)
    assert torch.equal(pr.apply(x), y)
