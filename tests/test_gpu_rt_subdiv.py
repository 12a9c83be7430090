"""rt_subdiv above the distances from which the orders 3, 2 and 1 would serve
(R_3 = 1.82, R_2 = 2.40, R_1 = 5.11 with the loose tolerance used here, with
which whole and subdivided elements differ visibly): such elements are
subdivided whatever order their distance would give, in the recomputed, the
transposed and the stored product and in the direct field and velocity.  With
8 and 20 elements are cut into more parts than a block's list holds.

Bounds: 2e-5 relative l2 and 2e-4 per element for the products, 2e-5 of the
largest value for the fields (FP32 entries and sums, as with the default
rules); taking the elements whole misses the products by more than 1e-4."""
import numpy as np
import pytest

import oracle
from paper_2312_00005_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

C, RHO, F = 343.0, 1.21, 900.0
TOL = 3e-2


@pytest.fixture(scope="module")
def bem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_00005_gb300 import bemfmm
    bemfmm.lib()
    return bemfmm


def _check(y, yo, what):
    l2 = np.linalg.norm(y - yo) / np.linalg.norm(yo)
    el = np.max(np.abs(y - yo) / np.maximum(np.abs(yo), 1e-3 * np.abs(yo).max()))
    assert l2 < 2e-5 and el < 2e-4, (what, l2, el)


@pytest.mark.parametrize("rt", [2.4, 4.0, 8.0, 20.0])
def test_subdivision_distance_above_the_order_distances(bem, rt):
    nodes, tris = inputs.geodesic_sphere(6)
    nodes, n, k = 0.1 * nodes, tris.shape[0], 2 * np.pi * F / C
    params = {"rt_subdiv": rt, "quad_tol": TOL}
    one, zero = np.ones(n, complex), np.zeros(n, complex)
    A = oracle.assemble(nodes, tris, k, one, zero, params)
    whole = oracle.assemble(nodes, tris, k, one, zero, {"quad_tol": TOL})
    x = inputs.random_complex(n, 5, (2, n))
    assert np.linalg.norm(x @ (A - whole).T) > 1e-4 * np.linalg.norm(x @ A.T)
    xt = torch.tensor(x, dtype=torch.complex64, device="cuda")
    for kw in ({"mode": bem.MODE_DIRECT}, {"mode": bem.MODE_FMM, "trunc_factor": 6.0}):
        m = bem.Mesh(nodes, tris, rt_subdiv=rt, quad_tol=TOL, field_mode=1, **kw)
        _check(m.matvec(F, xt, c=C, rho=RHO).cpu().numpy(), x @ A.T, ("product", kw))
        if kw["mode"] == bem.MODE_DIRECT:
            _check(m.matvec_transpose(F, xt[0].contiguous(), c=C, rho=RHO).cpu().numpy(), x[0] @ A, "transposed")
            pts = inputs.fibonacci_sphere(40, 1.0) * np.linspace(0.11, 0.3, 40)[:, None]
            p, q = (t.cpu().numpy().astype(np.complex128) for t in xt)
            fo = oracle.field(nodes, tris, F, p, q, pts, c=C, params=params)
            vo = oracle.field_velocity(nodes, tris, F, p, q, pts, c=C, rho=RHO, params=params)
            f = m.evaluate(F, xt[0].contiguous(), xt[1].contiguous(), pts, c=C, rho=RHO).cpu().numpy()
            v = m.evaluate_velocity(F, xt[0].contiguous(), xt[1].contiguous(), pts, c=C, rho=RHO).cpu().numpy()
            assert np.abs(f - fo).max() < 2e-5 * np.abs(fo).max()
            assert np.abs(v - vo).max() < 2e-5 * np.abs(vo).max()
        m.close()
