"""The same product of recomputed entries gives the same bits in every call,
also where a block has more expensive pairs than its queue holds and chance
decides which of them find room: rule sets that queue far more pairs than the
default one (a tight quad_tol, few orders), blocks that hold a whole near
list, 1, 2 and 4 right-hand sides and the transposed product."""
import pytest

from paper_2312_00005_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2312_00005_gb300 import bemfmm
    bemfmm.lib()
    return bemfmm


@pytest.mark.parametrize("nu,fmm,kw", [
    (4, 0, {"quad_tol": 1e-4}), (8, 0, {"m_max": 3}), (8, 0, {"m_max": 1}), (8, 0, {"quad_tol": 1e-6}),
    (16, 1, {"quad_tol": 1e-4}), (16, 1, {"quad_tol": 1e-6}), (16, 0, {}),
])
def test_recomputed_product_repeats_bit_for_bit(bem, nu, fmm, kw):
    nodes, tris = inputs.geodesic_sphere(nu)
    n = tris.shape[0]
    mode = {"mode": bem.MODE_FMM, "near_store": 0} if fmm else {"mode": bem.MODE_DIRECT}
    m = bem.Mesh(0.1 * nodes, tris, **mode, **kw)
    x = torch.tensor(inputs.random_complex(n, 7, (4, n)), dtype=torch.complex64, device="cuda")
    for nr in (1, 2, 4):
        y = m.matvec(2000.0, x[:nr].contiguous()).clone()
        for _ in range(8):
            assert torch.equal(m.matvec(2000.0, x[:nr].contiguous()), y), (nr, "product")
    x0 = x[0].contiguous()
    y = m.matvec_transpose(2000.0, x0).clone()
    for _ in range(8):
        assert torch.equal(m.matvec_transpose(2000.0, x0), y), "transposed product"
    m.close()
