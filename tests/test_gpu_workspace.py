"""Device memory of a solve: the Krylov workspace and the right-hand sides, and
no column parts of a recomputed product where the near field is stored; where
it is recomputed they are there before the Arnoldi steps are captured (a
capture may not allocate), for one and four right-hand sides and the adjoint."""
import numpy as np
import pytest

from paper_2312_00005_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

C, RHO, FREQ, RESTART = 343.0, 1.21, 2000.0, 20


@pytest.fixture(scope="module")
def bem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_00005_gb300 import bemfmm
    bemfmm.lib()
    bemfmm.test_hooks()
    return bemfmm


def test_stored_solve_holds_no_parts(bem):
    nodes, tris = inputs.icosphere(4, 0.1)
    n, nr = tris.shape[0], 4
    mesh = bem.Mesh(nodes, tris, restart=RESTART, autotune=0)
    src = [bem.plane_wave(d) for d in inputs.tetrahedral_directions()]
    x = torch.tensor(inputs.random_complex(n, 1, (nr, n)), dtype=torch.complex64, device="cuda")
    mesh.matvec(FREQ, x, c=C, rho=RHO)                 # the product's own buffers for four sides
    before = bem.test_hooks()
    mesh.solve_multi(FREQ, src, tol=1e-5, max_iter=40, c=C, rho=RHO)
    grown = bem.test_hooks() - before
    mesh.close()
    # basis (restart + 1), product, right-hand sides and solutions; the small
    # matrices and sums stay below 100 kB
    need = nr * n * 8 * (RESTART + 1 + 1 + 2)
    print("%d bytes for a basis and vectors of %d" % (grown, need))
    assert grown < need + 100_000


@pytest.mark.parametrize("kw", [{"near_store": 0}, {"mode": 1}])
def test_recomputed_solves_run_in_graphs(bem, kw):
    nodes, tris = inputs.icosphere(2, 0.1)
    n = tris.shape[0]
    bct = np.full(n, bem.ADMI, np.int32)
    adm = np.array([0.3 / (RHO * C)])
    mesh = bem.Mesh(nodes, tris, bc_type=bct, region=np.zeros(n, np.int32), restart=RESTART, **kw)
    src = [bem.point_source((0.0, 0.0, 0.3 + 0.1 * i)) for i in range(4)]
    P, _, infos = mesh.solve_multi(FREQ, src, admittance=adm, tol=1e-6, c=C, rho=RHO)
    p, _, info = mesh.solve(FREQ, src[:1], admittance=adm, tol=1e-6, c=C, rho=RHO)
    assert info["converged"] and all(i["converged"] for i in infos)
    assert float(torch.linalg.norm(P[0] - p) / torch.linalg.norm(p)) < 1e-4
    pts = inputs.fibonacci_sphere(10, 0.5)
    out = mesh.admittance_gradient(FREQ, src[:1], adm, pts, tol=1e-6, c=C, rho=RHO)
    mesh.close()
    assert np.all(np.isfinite(np.asarray(out[1], dtype=np.complex128)))
