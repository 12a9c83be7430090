"""The products whose near-field entries are recomputed by quadrature (direct
mode, near_store = 0, and the transposed product of both), for 1 to 5 right-
hand sides in one call, against the oracle's dense operator: meshes of less
than a warp of rows, less than a tile of columns, just over a tile, and
several tiles, and a rule set without the orders 4 to 6 (m_max = 3), where
every pair but the farthest takes the general rule.

Bounds: 2e-5 relative l2 and 2e-4 per element (FP32 entries and sums), as the
other direct products."""
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


def _mesh(name):
    if name == "tetrahedron":
        nodes = 0.1 * np.array([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]], float)
        return nodes, np.array([[0, 1, 2], [0, 3, 1], [0, 2, 3], [1, 3, 2]], np.int32)
    if name == "duct":
        return inputs.duct(0.6, 0.2, 0.1)
    nodes, tris = inputs.geodesic_sphere(int(name))
    return 0.1 * nodes, tris


def _check(y, yo, what):
    l2 = np.linalg.norm(y - yo) / np.linalg.norm(yo)
    el = np.max(np.abs(y - yo) / np.maximum(np.abs(yo), 1e-3 * np.abs(yo).max()))
    assert l2 < 2e-5 and el < 2e-4, (what, l2, el)


@pytest.mark.parametrize("mesh,nrhs,kw", [
    ("tetrahedron", 1, {}), ("2", 3, {}), ("duct", 2, {}), ("4", 4, {}), ("6", 5, {}), ("9", 1, {}),
    ("6", 2, {"m_max": 3}), ("6", 1, {"m_max": 1}), ("6", 1, {"near_store": 0, "fmm": 1}),
])
def test_recomputed_products_match_oracle(bem, mesh, nrhs, kw):
    nodes, tris = _mesh(mesh)
    n, f = tris.shape[0], 900.0
    kw = dict(kw)
    kw["mode"] = bem.MODE_FMM if kw.pop("fmm", 0) else bem.MODE_DIRECT
    rng = np.random.default_rng(n + nrhs)
    bct = rng.integers(0, 3, n).astype(np.int32)
    region = rng.integers(0, 3, n).astype(np.int32)
    adm = rng.uniform(0, 0.5, 3) * np.exp(1j * rng.uniform(-1.5, 1.5, 3)) / (RHO * C)
    cp, cq, _, _ = oracle.column_coeffs(bct, 2 * np.pi * f / C, C, RHO, (RHO * C * adm)[region])
    params = {"m_max": kw["m_max"]} if "m_max" in kw else None
    A = oracle.assemble(nodes, tris, 2 * np.pi * f / C, cp, cq, params)
    x = inputs.random_complex(n, 5, (nrhs, n))
    m = bem.Mesh(nodes, tris, bc_type=bct, region=region, trunc_factor=6.0, **kw)
    xt = torch.tensor(x, dtype=torch.complex64, device="cuda")
    y = m.matvec(f, xt, admittance=adm, c=C, rho=RHO).cpu().numpy()
    _check(y, x @ A.T, "product")
    yt = m.matvec_transpose(f, xt[0].contiguous(), admittance=adm, c=C, rho=RHO).cpu().numpy()
    _check(yt, x[0] @ A, "transposed product")
    m.close()
