"""Restarted GMRES of several right-hand sides solved together: cycles whose
length is and is not a multiple of the four steps of a graph body (the body
then runs past the end of the cycle, and what it skips must not reach the
next one), with the steps in graphs and one at a time, against the oracle.

Bounds: 1e-4 relative l2 and 1e-3 per element, as the restarted solve of one
right-hand side; iterations within 2 of the stepwise loop's (its FP64 sums are
added in another order)."""
import numpy as np
import pytest

import oracle
from paper_2312_00005_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

C, RHO, FREQ = 343.0, 1.21, 1000.0
DIRS = [(0.0, 0.0, 1.0), (1.0, 0.0, 0.0), (0.0, -0.6, 0.8), (0.6, 0.8, 0.0)]


@pytest.fixture(scope="module")
def bem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_00005_gb300 import bemfmm
    bemfmm.lib()
    return bemfmm


@pytest.fixture(scope="module")
def reference():
    nodes, tris = inputs.icosphere(3, 0.1)
    return nodes, tris, [oracle.solve(nodes, tris, FREQ, c=C, rho=RHO, sources=[("plane", d, 1.0)])[0] for d in DIRS]


@pytest.mark.parametrize("restart,nr", [(5, 4), (6, 2), (6, 3), (7, 4), (8, 4)])
def test_restarted_solves_of_several_sides_match_oracle(bem, reference, restart, nr):
    nodes, tris, po = reference
    src = [bem.plane_wave(d) for d in DIRS[:nr]]
    runs = []
    for graphs in (1, 0):
        mesh = bem.Mesh(nodes, tris, restart=restart, graphs=graphs)
        P, _, infos = mesh.solve_multi(FREQ, src, tol=1e-7, c=C, rho=RHO)
        mesh.close()
        runs.append([i["iterations"] for i in infos])
        for r in range(nr):
            assert infos[r]["converged"] and infos[r]["restarts"] >= 1, infos[r]
            d = np.abs(P[r].cpu().numpy() - po[r])
            l2 = np.linalg.norm(d) / np.linalg.norm(po[r])
            el = np.max(d / np.maximum(np.abs(po[r]), 1e-3 * np.abs(po[r]).max()))
            print("restart %d, side %d of %d, graphs %d: %.2e, per element %.2e" % (restart, r, nr, graphs, l2, el))
            assert l2 < 1e-4 and el < 1e-3
    assert all(abs(a - b) <= 2 for a, b in zip(*runs)), runs
