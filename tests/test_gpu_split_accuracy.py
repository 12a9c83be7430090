"""Cutting a recomputed product into more blocks costs no accuracy: the mean
relative l2 error of four random vectors stays below 1.2e-7 at sizes that are
cut into 3 to 20 parts.  The entries alone, to FP32 rounding (2^-24 / sqrt(3)
per operation, some dozen operations), account for about 1e-7; a plain FP32 sum
of the parts gave 1.27e-7, 1.40e-7 and 1.49e-7."""
import numpy as np
import pytest

import oracle
from paper_2312_00005_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

C, RHO, F = 343.0, 1.21, 900.0


@pytest.mark.parametrize("nu", [2, 4, 8])
def test_split_product_keeps_the_accuracy(nu):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_00005_gb300 import bemfmm as bem
    nodes, tris = inputs.geodesic_sphere(nu)
    nodes, n = 0.1 * nodes, tris.shape[0]
    A = oracle.assemble(nodes, tris, 2 * np.pi * F / C, np.ones(n, complex), np.zeros(n, complex))
    mesh = bem.Mesh(nodes, tris, mode=bem.MODE_DIRECT)
    err = []
    for seed in range(4):
        x = torch.tensor(inputs.random_complex(n, seed), dtype=torch.complex64, device="cuda")
        xh = x.cpu().numpy().astype(np.complex128)
        y, yt = (f(F, x, c=C, rho=RHO).cpu().numpy() for f in (mesh.matvec, mesh.matvec_transpose))
        err.append([np.linalg.norm(a - b) / np.linalg.norm(b) for a, b in ((y, A @ xh), (yt, A.T @ xh))])
    mesh.close()
    print("%d elements: product and transposed product %s" % (n, np.mean(err, axis=0)))
    assert np.mean(err, axis=0).max() < 1.2e-7
