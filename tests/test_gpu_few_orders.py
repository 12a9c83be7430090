"""Rule sets of one to three orders (m_max): the recomputed and transposed
products and the direct field against the oracle, on meshes below and above
one tile of columns; and, since they need fewer quadrature points than the
default set, in no more time than it takes (a fifth for noise).

Bounds: 2e-5 relative l2 and 2e-4 per element for the products, 2e-5 of the
largest value for the field (FP32 entries and sums, as with the default rules)."""
import numpy as np
import pytest

import oracle
from paper_2312_00005_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

C, RHO, F = 343.0, 1.21, 900.0


@pytest.fixture(scope="module")
def bem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_00005_gb300 import bemfmm
    bemfmm.lib()
    return bemfmm


def _mesh(nu):
    nodes, tris = inputs.geodesic_sphere(nu)
    return 0.1 * nodes, tris


@pytest.mark.parametrize("m_max", [1, 2, 3])
@pytest.mark.parametrize("nu", [2, 5])
def test_products_and_field_of_few_orders_match_oracle(bem, nu, m_max):
    nodes, tris = _mesh(nu)
    n = tris.shape[0]
    x = inputs.random_complex(n, 5, (3, n))
    xt = torch.tensor(x, dtype=torch.complex64, device="cuda")
    A = oracle.assemble(nodes, tris, 2 * np.pi * F / C, np.ones(n, complex), np.zeros(n, complex), {"m_max": m_max})
    m = bem.Mesh(nodes, tris, mode=bem.MODE_DIRECT, m_max=m_max)
    y = m.matvec(F, xt, c=C, rho=RHO).cpu().numpy()
    yt = m.matvec_transpose(F, xt[0].contiguous(), c=C, rho=RHO).cpu().numpy()
    pts = inputs.fibonacci_sphere(50, 1.0) * np.linspace(0.101, 0.5, 50)[:, None]
    f = m.evaluate(F, xt[0].contiguous(), xt[1].contiguous(), pts, c=C, rho=RHO).cpu().numpy()
    m.close()
    for a, b in ((y, x @ A.T), (yt, x[0] @ A)):
        el = np.max(np.abs(a - b) / np.maximum(np.abs(b), 1e-3 * np.abs(b).max()))
        assert np.linalg.norm(a - b) < 2e-5 * np.linalg.norm(b) and el < 2e-4
    p, q = (t.cpu().numpy().astype(np.complex128) for t in xt[:2])
    fo = oracle.field(nodes, tris, F, p, q, pts, c=C, params={"m_max": m_max})
    assert np.abs(f - fo).max() < 2e-5 * np.abs(fo).max()


@pytest.mark.parametrize("nu", [8, 16])
def test_few_orders_take_no_longer_than_the_default(bem, nu):
    nodes, tris = _mesh(nu)
    n = tris.shape[0]
    x = torch.tensor(inputs.random_complex(n, 5), dtype=torch.complex64, device="cuda")
    times = {}
    for m_max in (6, 3, 2, 1):
        m = bem.Mesh(nodes, tris, mode=bem.MODE_DIRECT, m_max=m_max)
        for _ in range(5):
            m.matvec(F, x)
        t = []
        for _ in range(15):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(5):
                m.matvec(F, x)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b) / 5)
        m.close()
        times[m_max] = float(np.median(t))
    print("%d elements: ms by m_max %s" % (n, times))
    for m_max in (3, 2, 1):
        assert times[m_max] < 1.2 * times[6], times
