"""The field through the expansions (field_mode 2) at points close to the surface,
whose near lists hold expensive pairs: many of them in one list (a tight
quad_tol, a coarse surface), none, and few points, against the oracle; the
same call gives the same bits; and points at the surface take less than twice
the direct sum's time (three and a half times when a lane worked off a pair).

Bounds: 1e-4 of the largest value at expansion factor 6 on the coarse surfaces
(the FMM field's bound)."""
import numpy as np
import pytest

import oracle
from paper_2312_00005_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

C, RHO, F = 343.0, 1.21, 1200.0


@pytest.fixture(scope="module")
def bem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_00005_gb300 import bemfmm
    bemfmm.lib()
    return bemfmm


def _state(bem, nu, m, radius, **kw):
    nodes, tris = inputs.geodesic_sphere(nu)
    n = tris.shape[0]
    p, q = (torch.tensor(v, dtype=torch.complex64, device="cuda")
            for v in (inputs.random_complex(n, 1), inputs.random_complex(n, 2) * 20))
    pts = inputs.fibonacci_sphere(m, radius) if m > 1 else np.array([[0.0, 0.0, radius]])
    return 0.1 * nodes, tris, p, q, pts, bem.Mesh(0.1 * nodes, tris, field_mode=2, trunc_factor=6.0, autotune=0, **kw)


@pytest.mark.parametrize("nu,m,radius,kw", [
    (4, 1, 0.101, {}), (4, 500, 0.1005, {}), (8, 300, 0.101, {}), (8, 300, 0.3, {}), (12, 800, 0.1002, {}),
    (8, 300, 0.12, {"quad_tol": 1e-6}), (12, 300, 0.12, {"quad_tol": 1e-7}), (8, 200, 0.102, {"m_max": 2}),
    (8, 200, 0.102, {"rt_subdiv": 4.0}),
])
def test_expansion_field_near_the_surface(bem, nu, m, radius, kw):
    nodes, tris, p, q, pts, mesh = _state(bem, nu, m, radius, **kw)
    f = mesh.evaluate(F, p, q, pts, c=C, rho=RHO)
    for _ in range(4):
        assert torch.equal(mesh.evaluate(F, p, q, pts, c=C, rho=RHO), f)
    mesh.close()
    ph, qh = (t.cpu().numpy().astype(np.complex128) for t in (p, q))
    fo = oracle.field(nodes, tris, F, ph, qh, pts, c=C, params=kw)
    err = np.abs(f.cpu().numpy() - fo).max() / np.abs(fo).max()
    print("%d elements, %d points: %.2e of the largest value" % (tris.shape[0], m, err))
    assert err < 1e-4


def test_points_at_the_surface_cost_about_the_direct_sum(bem):
    t = {}
    for mode in (1, 2):
        nodes, tris = inputs.geodesic_sphere(8)
        n = tris.shape[0]
        p, q = (torch.tensor(inputs.random_complex(n, s), dtype=torch.complex64, device="cuda") for s in (1, 2))
        pts = inputs.fibonacci_sphere(5000, 0.101)
        mesh = bem.Mesh(0.1 * nodes, tris, field_mode=mode, autotune=0)
        for _ in range(3):
            mesh.evaluate(F, p, q, pts)
        ev = []
        for _ in range(10):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            mesh.evaluate(F, p, q, pts)
            b.record()
            b.synchronize()
            ev.append(a.elapsed_time(b))
        t[mode] = float(np.median(ev))
        mesh.close()
    print("ms direct %.3f, expansions %.3f" % (t[1], t[2]))
    assert t[2] < 2.0 * t[1], t
