"""The transfer of several right-hand sides, whose blocks take two targets at a
time, against the one-target transfer of single products.

The sizes: levels with an odd number of targets (the last pair has one), 2 L^2
directions that 32 does not divide, a duct whose lists are short and uneven,
and block counts on both sides of the line between four and two warps per
block.

The two forms sum the same FP32 products in another order.  A target's sum has
at most a few hundred terms, n say, of comparable magnitude, and rounding
differences between two orders grow as sqrt(n) 2^-24 of their norm: 1.3e-6 for
n = 450, and less after the sum over levels and the near field, which are not
reordered.  The bounds are 4e-6 in the 2-norm and 2e-4 per element (against
at least 1e-3 of the largest).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2312_00005_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bem():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2312_00005_gb300 import bemfmm

    return bemfmm


def _sphere(nu):
    nodes, tris = inputs.geodesic_sphere(nu)
    return 0.1 * nodes, tris


@pytest.mark.parametrize("mesh,freq,kw", [
    (lambda: inputs.icosphere(3, 0.1), 1500.0, {}),
    (lambda: _sphere(11), 2500.0, dict(trunc_factor=4.0)),
    (lambda: inputs.duct(3.4, 0.2, 0.2 / 6), 400.0, {}),
    (lambda: inputs.bumpy_ellipsoid(23), 6000.0, dict(trunc_factor=8.0)),
    (lambda: inputs.bumpy_ellipsoid(45), 10000.0, dict(trunc_factor=8.0)),
])
def test_products_of_several_sides_match_single_products(bem, mesh, freq, kw):
    nodes, tris = mesh()
    n = len(tris)
    m = bem.Mesh(nodes, tris, **kw)
    x = torch.from_numpy(inputs.random_complex(n, 3, (7, n)).astype(np.complex64)).cuda()
    one = torch.stack([m.matvec(freq, x[r].contiguous()) for r in range(7)])
    assert sum(m.stats(freq)["n_interactions"]) > 0
    # 2, 4, 4 + 2 and 4 + 3 at once, and 2 again on the buffers of 4
    for nr in (2, 4, 6, 7, 2):
        y = m.matvec(freq, x[:nr].contiguous())
        for r in range(nr):
            d = (y[r] - one[r]).abs()
            l2 = float(torch.linalg.norm(y[r] - one[r]) / torch.linalg.norm(one[r]))
            el = float((d / one[r].abs().clamp(min=1e-3 * float(one[r].abs().max()))).max())
            print("%d elements, %d of %d: %.2e, per element %.2e" % (n, r, nr, l2, el))
            assert l2 < 4e-6 and el < 2e-4
