"""The direct field and particle velocity at points (bem_evaluate with
field_mode 1, bem_evaluate_velocity) against the oracle, for point counts
around the kernels' 32 points per block and for points within a fraction of an
element of the surface, whose nearby elements go through the queued general
rules (subdivided and high-order), on one tile of elements and on several.

Bounds: 2e-5 of the largest value for every point (FP32 entries and sums, as
the direct products; a point's field can be a cancelling sum)."""
import numpy as np
import pytest

import oracle
from paper_2312_00005_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

C, RHO = 343.0, 1.21


@pytest.fixture(scope="module")
def bem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_00005_gb300 import bemfmm
    bemfmm.lib()
    return bemfmm


@pytest.mark.parametrize("nu,m", [(3, 1), (3, 33), (8, 31), (8, 64), (8, 7), (11, 300)])
def test_direct_field_and_velocity_match_oracle(bem, nu, m):
    nodes, tris = inputs.geodesic_sphere(nu)
    nodes = 0.1 * nodes
    n, f = tris.shape[0], 1200.0
    edge = 0.115 / nu
    pts = inputs.fibonacci_sphere(m, 1.0)
    # every third point a third of an edge off the surface, the others 0.15 to 1 m out
    r = np.where(np.arange(m) % 3 == 0, 0.1 + edge / 3, np.linspace(0.15, 1.0, m))
    pts = pts * r[:, None]
    p, q = inputs.random_complex(n, 1), inputs.random_complex(n, 2) * 20
    pt, qt = (torch.tensor(v, dtype=torch.complex64, device="cuda") for v in (p, q))
    p, q = (t.cpu().numpy().astype(np.complex128) for t in (pt, qt))
    src = [("plane", (0.0, 0.0, 1.0), 1.0 + 0.5j)]
    gsrc = [bem.plane_wave((0.0, 0.0, 1.0), 1.0 + 0.5j)]
    mesh = bem.Mesh(nodes, tris, field_mode=1)
    fl = mesh.evaluate(f, pt, qt, pts, gsrc, c=C, rho=RHO).cpu().numpy()
    v = mesh.evaluate_velocity(f, pt, qt, pts, gsrc, c=C, rho=RHO).cpu().numpy()
    mesh.close()
    fo = oracle.field(nodes, tris, f, p, q, pts, c=C, sources=src)
    vo = oracle.field_velocity(nodes, tris, f, p, q, pts, c=C, rho=RHO, sources=src)
    assert np.abs(fl - fo).max() < 2e-5 * np.abs(fo).max()
    assert np.abs(v - vo).max() < 2e-5 * np.abs(vo).max()
